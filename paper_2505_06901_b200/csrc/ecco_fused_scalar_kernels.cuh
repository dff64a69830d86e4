// ecco_fused_scalar_kernels.cuh -- K2 / K3: fused GEMV (one to five rows of x) and attention scores (one or two heads)
// Part of the one translation unit ecco_kernels.cu; included from there only.
#pragma once

namespace {

// ---------------------------------------------------------------------------------------------
// K2/K3: fused consumers.  kV = number of dot products per group (batch rows of x, or query
// heads per KV head).  The vector slice [kV][128] fp16 lives in shared memory; every lane reads the same eight
// elements at the same time (one broadcast wavefront per eight symbols and vector) and adds the products with the
// mixed-precision multiply-add (fp16 x fp16 + fp32, one rounding): no operand is ever converted.
// Bound by the decode.  Two symbols per lookup and values in registers against one symbol per lookup and a value table in
// shared memory: the seven products of a 7B-shaped layer at batch 1 193.5 -> 149.2 us, a 4096 x 4096 matrix alone 20.4 -> 17.0 us.
// ---------------------------------------------------------------------------------------------
// Shared memory of a warp that keeps the decoded ranks of its groups: [27][32] words.  Rows 8..23 are the block's words, rows
// 24..26 are scratch; the ranks of step i go to row i.  By then the stream has been read past that row: step i leaves the position
// at bit 11 + 16 (i + 1) at least (eleven header bits, two bits per symbol), so the next window, which starts one bit early, starts in
// row 8 + (26 + 16 i) / 32 > i or later, and the outlier fields (bits 272 and up) sit in rows 16 and up.
constexpr uint32_t kRankRows = 8;
constexpr uint32_t kRankedBytes = (kRankRows + kBitRows) * 128;      // 3456

// acc += w . x over the two fp16 numbers of each word
__device__ __forceinline__ void fma_half2(float& acc, uint32_t w, uint32_t x)
{
    asm("{\n\t.reg .f16 a, b, c, d;\n\tmov.b32 {a, b}, %1;\n\tmov.b32 {c, d}, %2;\n\t"
        "fma.rn.f32.f16 %0, a, c, %0;\n\tfma.rn.f32.f16 %0, b, d, %0;\n\t}"
        : "+f"(acc)
        : "r"(w), "r"(x));
}
// the value of one rank of the group that begins with stream word hdr (see open_lane_group), for a lane that has not opened it
__device__ __forceinline__ float value_of(uint32_t hdr, uint32_t rank, const DecodeTables& tb, float T)
{
    const uint32_t kpe = lds_u16(tb.kp + ((hdr >> (kHeaderBits - 1)) & 0x1ffeu));
    const uint32_t cb = (kpe & (kMaxPatterns - 1u)) * kCodebooks + ((hdr >> 8) & 3u);
    const uint32_t top = lds_u32(tb.base + kSmemRec + cb * 16 + 12);
    const float c = __half2float(__ushort_as_half(static_cast<unsigned short>(lds_u16(cent_row(tb, cb) ^ (rank * 2)))));
    const float v = __half2float(__float2half_rn(c * (fp8_to_float(hdr & 0x7fu) * T)));
    return rank == top && (hdr & 0x80u) ? -v : v;
}

// the value of one rank of the lane's group
__device__ __forceinline__ float rank_value(const LaneGroup& g, uint32_t rank)
{
    const uint32_t s = rank & 7u, k = (rank >> 1) & 4u;
    const uint32_t lo = prmt(prmt(g.vlo[0], g.vlo[1], s), prmt(g.vlo[2], g.vlo[3], s), k);
    const uint32_t hi = prmt(prmt(g.vhi[0], g.vhi[1], s), prmt(g.vhi[2], g.vhi[3], s), k);
    return __half2float(__ushort_as_half(static_cast<unsigned short>(prmt(lo, hi, 0x0040u))));
}

// Partial sums per product.  One chain over a group's 128 products is less exact than the tensor cores' shorter ones where a warp has
// a single unit: 513 x 512 by three rows, error 2.06e-7 of the result against 1.97e-7, and 1.38e-7 with two chains.  At three to
// five rows the second chain costs 1.5 to 4 % (two 11008 x 4096 matrices 65.7 -> 66.8, 71.5 -> 74.4 and 79.4 -> 81.0 us), some of it by
// spills: 12 bytes per thread at four rows (none with one chain), 28 at five (16).
constexpr int kChains = 2;
__device__ __forceinline__ float sum_of(const float (&a)[kChains]) { return a[0] + a[1]; }

// kDeal: deal_outliers (caches) or every lane its own (weights)
// decode one group and accumulate its kV dot products against the slice at shared address xs
// keep = false: the products are not wanted.  The lanes past the end of a row decode its last group again; with 23 copies of a
// group of many outliers to deal, one warp held up a whole call (scores of 2 x 8 x 777 tokens 14.6 instead of 9.0 us).
template <int kV, bool kDeal>
__device__ __forceinline__ void fused_group(const Block& blk, const DecodeTables& tb, uint32_t bits, float T, uint32_t xs, bool keep, float (&acc)[kV][kChains])
{
    LaneGroup g = open_block(blk, bits, tb, T);
    if (kDeal) sts_u32(bits + 18 * 128, blk.w[0]);                    // the ranks will lie over the block's first words
    const uint32_t ranks_at = bits - kRankRows * 128;
    const uint32_t end = decode_group<kBlockBits, kBlockFreeSteps>(g, bits, tb.pairs, [&](int i, uint32_t ranks, bool cutting, int n_ok) {
        uint32_t v[4];
        map_ranks(g, ranks, v);
        if (cutting) cut_values(v, n_ok);
        sts_u32(ranks_at + i * 128, ranks);
#pragma unroll
        for (int b = 0; b < kV; ++b) {
            uint32_t x[4];
            asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]) : "r"(xs + b * (kGroup * 2) + i * 16));
            fma_half2(acc[b][0], v[0], x[0]);
            fma_half2(acc[b][1], v[1], x[1]);
            fma_half2(acc[b][0], v[2], x[2]);
            fma_half2(acc[b][1], v[3], x[3]);
        }
    });
    // outliers replace the mapped value at their location: add (outlier - mapped) * x.  Rows 24 and 25 behind the block hold the
    // list and the products.
    const int n_pad = keep ? pads_of(end) : 0;
    if (!kDeal) {
        uint32_t seen = 0;                                 // location mod 32 of the outliers so far
        for (int j = n_pad - 1; j >= 0; --j) {             // the last pad wins on a duplicate location (only corrupt blocks have one)
            const uint32_t f = pad_field(bits, j);
            const uint32_t loc = f & 127u, bit = 1u << (loc & 31u);
            if (seen & bit) {
                bool replaced = false;
                for (int k = j + 1; k < n_pad; ++k) replaced = replaced || (pad_field(bits, k) & 127u) == loc;
                if (replaced) continue;
            }
            seen |= bit;
            const float mapped = rank_value(g, (lds_u32(ranks_at + (loc >> 3) * 128) >> ((loc & 7u) * 4)) & 15u);
            const float outlier = __half2float(__float2half_rn(fp8_to_float(f >> 7) * T));
#pragma unroll
            for (int b = 0; b < kV; ++b) {
                const float x = __half2float(__ushort_as_half(static_cast<unsigned short>(lds_u16(xs + b * (kGroup * 2) + loc * 2))));
                acc[b][0] = fmaf(outlier - mapped, x, acc[b][0]);
            }
        }
    } else if (warp_any(n_pad > 0)) {
        const uint32_t lane4 = (threadIdx.x & 31u) * 4, bits0 = bits - lane4, list = bits0 + 16 * 128;
        deal_outliers(bits, list, n_pad, [&](uint32_t slot, uint32_t owner, uint32_t f, bool valid) {
            const uint32_t loc = f & 127u;
            const uint32_t rank = (lds_u32(ranks_at - lane4 + owner * 4 + (loc >> 3) * 128) >> ((loc & 7u) * 4)) & 15u;
            const float mapped = value_of(lds_u32(bits0 + 18 * 128 + owner * 4), rank, tb, T);
            const float outlier = __half2float(__float2half_rn(fp8_to_float(f >> 7) * T));
#pragma unroll
            for (int b = 0; b < kV; ++b) {
                const float x = __half2float(__ushort_as_half(static_cast<unsigned short>(lds_u16(xs + b * (kGroup * 2) + loc * 2))));
                const float p = valid ? (outlier - mapped) * x : 0.0f;
                sts_u32(list + (b ? 0 : 128) + slot * 4, __float_as_uint(p));     // the list has been read
            }
        }, [&](uint32_t first, int count) {
            for (int j = 0; j < count; ++j)
#pragma unroll
                for (int b = 0; b < kV; ++b) acc[b][0] += __uint_as_float(lds_u32(list + (b ? 0 : 128) + (first + j) * 4));
        });
    }
}

// Contiguous split of U work units over G workers: worker c owns [begin(c), begin(c + 1)), the first U mod G of them one unit more
// than the others.  (Boundaries at U * c / G took four 64-bit divisions to find a unit's owner, which every split sum does twice at its end.)
struct UnitSplit {
    int64_t per;
    int more;                                              // workers with per + 1 units
    __device__ __forceinline__ UnitSplit(int64_t U, int G)
    {
        per = static_cast<int64_t>(divide(static_cast<uint64_t>(U), static_cast<uint64_t>(G)));
        more = static_cast<int>(U - per * G);
    }
    __device__ __forceinline__ int64_t begin(int c) const { return per * c + min(c, more); }
    __device__ __forceinline__ int owner(int64_t u) const
    {
        const int64_t cut = (per + 1) * more;
        return u < cut ? static_cast<int>(divide(static_cast<uint64_t>(u), static_cast<uint64_t>(per + 1)))
                       : more + static_cast<int>(divide(static_cast<uint64_t>(u - cut), static_cast<uint64_t>(per)));
    }
};

// Ticket words of a workspace.  They need no clearing before the call, which would be a launch of its own (2 us of a small call's
// 10): a word counts from zero once it carries the call's tag, 48 bits that the host draws at random once and advances for every
// call (stale contents carry it with probability 2^-48).  Everyone who will take a ticket first claims the word, early, while its
// block is on the way: if the word does not carry the tag, an exchange against what was seen installs it, and it fails exactly
// when another has done so.  Taking is then one addition.  (Counting up by exchanges alone serialises the arrivals: 39 us instead of
// 17 for a 4096 x 4096 product.)  The last to arrive clears the word, so a captured call that is replayed with its tag finds none of
// its own counts.  For that everyone has to arrive: a CTA whose table fetch timed out passes its tickets (and its call's output is
// undefined, but the next replay's is not).
using Ticket = unsigned long long;
constexpr int kTicketStride = 4;                           // words from one ticket to the next: each in a sector of its own
__device__ __forceinline__ Ticket look_at_ticket(const Ticket* word) { return *reinterpret_cast<const volatile Ticket*>(word); }
__device__ __forceinline__ void claim_ticket(Ticket* word, Ticket seen, Ticket tag)
{
    if ((seen >> 16) != tag) atomicCAS(word, seen, tag << 16);
}
__device__ __forceinline__ unsigned int take_ticket(Ticket* word) { return static_cast<unsigned int>(atomicAdd(word, 1ull) & 0xffffu); }
// takes a ticket for nothing; the last of them has number `last`
__device__ __forceinline__ void pass_ticket(Ticket* word, int last, Ticket tag)
{
    claim_ticket(word, look_at_ticket(word), tag);
    if (take_ticket(word) == static_cast<unsigned int>(last)) *word = 0;
}

// One call of the fused GEMV may cover several matrices (ecco_gemv_batch): the units of all of them form one unit
// space, dealt out to the working warps as one, so that a group of small matrices pays one launch, one table fetch and
// one tail.  All matrices of a call share the decode tables (equal table hash; only the exponent differs).
constexpr int kMaxGemvJobs = 8;
struct GemvJob {
    const uint8_t* meta;       // metadata image of this matrix (its exponent factor T is read from here)
    const uint8_t* blocks;
    const __half* x;           // [kV or batch][k]
    float* y;                  // [batch][n_out]
    int32_t n_out, kblocks;
    int32_t tile_first;        // first 32-row tile of this matrix in the call's tile space (tickets and slots)
    int32_t reserved;
    int64_t unit_first;        // first unit of this matrix in the call's unit space
};
struct GemvBatch {
    int32_t n, reserved;
    int64_t units;             // of all matrices
    GemvJob job[kMaxGemvJobs];
};
// true (uniformly over the grid) if every matrix of the call carries the tables of the first
__device__ __forceinline__ bool same_tables(const GemvBatch& batch, const DecodeTables& tb)
{
    bool same = true;
    for (int t = 1; t < batch.n; ++t) {
        const DevHeader* hd = reinterpret_cast<const DevHeader*>(batch.job[t].meta);
        same = same && __ldg(&hd->hash_lo) == tb.hash_lo && __ldg(&hd->hash_hi) == tb.hash_hi;
    }
    if (!same && threadIdx.x == 0) atomicExch(&g_device_status, ECCO_ERR_INVALID_ARG);
    return same;
}

// Where a unit sits: matrix, 32-row tile and k-block.  Units are visited in order, so the position is advanced by one
// instead of being divided out of the unit number every time.
struct GemvPos { int j, tile, kb; };
__device__ __forceinline__ GemvPos gemv_pos_of(const GemvBatch& batch, int64_t u)
{
    GemvPos p = {0, 0, 0};
    while (p.j + 1 < batch.n && u >= batch.job[p.j + 1].unit_first) ++p.j;
    const int64_t lu = u - batch.job[p.j].unit_first;
    p.tile = static_cast<int>(divide(static_cast<uint64_t>(lu), static_cast<uint64_t>(batch.job[p.j].kblocks)));
    p.kb = static_cast<int>(lu - static_cast<int64_t>(p.tile) * batch.job[p.j].kblocks);
    return p;
}
__device__ __forceinline__ GemvPos gemv_pos_next(const GemvBatch& batch, GemvPos p)
{
    if (++p.kb == batch.job[p.j].kblocks) {
        p.kb = 0;
        if (++p.tile == (batch.job[p.j].n_out + 31) / 32) { p.tile = 0; ++p.j; }
    }
    return p;
}
// place of a row tile in the call's tile space (tickets and slots)
__device__ __forceinline__ int gemv_tile_of(const GemvBatch& batch, const GemvPos& p) { return batch.job[p.j].tile_first + p.tile; }
__device__ __forceinline__ const uint8_t* gemv_block_ptr(const GemvBatch& batch, const GemvPos& p, int lane)
{
    const GemvJob& jb = batch.job[p.j];
    const int row = min(p.tile * 32 + lane, jb.n_out - 1);                         // rows past the end: repeat the last
    return jb.blocks + (static_cast<uint64_t>(row) * jb.kblocks + p.kb) * kBlockBytes;
}

// A warp that gives up units u0 .. u1 - 1 passes the tickets of the row tiles it shares: at most the first and the last.
__device__ __forceinline__ void pass_gemv_tickets(const GemvBatch& batch, const UnitSplit& split, int64_t u0, int64_t u1, Ticket* d_tickets, Ticket tag)
{
    if (u0 >= u1 || (threadIdx.x & 31u)) return;
    int done = -1;
    for (int end = 0; end < 2; ++end) {
        const GemvPos pos = gemv_pos_of(batch, end ? u1 - 1 : u0);
        const GemvJob& jb = batch.job[pos.j];
        const int64_t g0 = jb.unit_first + static_cast<int64_t>(pos.tile) * jb.kblocks;
        const int gtile = gemv_tile_of(batch, pos), last = split.owner(g0 + jb.kblocks - 1) - split.owner(g0);
        if (last && gtile != done) pass_ticket(d_tickets + gtile * kTicketStride, last, tag);
        done = gtile;
    }
}

__host__ __device__ constexpr uint32_t scalar_warp_bytes(int v) { return v * kGroup * 2 + kRankedBytes; }

// K2 for one to five rows of x: the slice is small enough (256 B a row) for every warp to keep
// its own, so warps never meet at a barrier.  A work unit is (32 consecutive rows, one k-block),
// numbered matrix by matrix, row-tile major; every working warp owns a contiguous run of units and keeps its
// rows' partial sums in registers along k.  When a row tile is shared by several warps each writes its
// partial sums to its own workspace slot (slot = global warp id + row tile: unique along the
// staircase of (warp, tile) pairs) and the last to arrive (ticket counter) adds the slots in warp
// order: the result does not depend on scheduling.  Workspace: partial[slot][kV][32] floats, then
// one ticket per 32-row tile.
template <int kV, int kMaxWarps, bool kGiveUp>
__global__ void __launch_bounds__(kMaxWarps * 32, 1)
ecco_gemv_warp_kernel(const __grid_constant__ GemvBatch batch, float* __restrict__ d_partial, Ticket* d_tickets, Ticket tag)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    release_dependents();
    const uint8_t* d_meta = batch.job[0].meta;
    const DecodeTables tb = plan_decode_tables(smem_u32(smem), d_meta, true);
    const int nw = static_cast<int>(decode_warps(tb, scalar_warp_bytes(kV)));
    const int lane = static_cast<int>(threadIdx.x & 31u), warp = static_cast<int>(threadIdx.x >> 5);
    const uint32_t xs = tb.warp_base + warp * scalar_warp_bytes(kV);             // this warp's slice [kV][128] fp16
    const uint32_t bits = xs + kV * kGroup * 2 + kRankRows * 128 + lane * 4;

    // W working warps (chosen so that they all get the same number of units, and never more than there are
    // units); warp ids interleave over the CTAs; the other warps idle
    const int wg = warp < nw ? warp * static_cast<int>(gridDim.x) + static_cast<int>(blockIdx.x) : INT_MAX;
    const int64_t U = batch.units;
    const int W = static_cast<int>(balanced_warps(static_cast<uint64_t>(U), gridDim.x * static_cast<uint32_t>(nw)));
    const UnitSplit split(U, W);
    const int64_t u0 = wg < W ? split.begin(wg) : 0, u1 = wg < W ? split.begin(wg + 1) : 0;
    issue_decode_tables(tb, d_meta);
    if (!same_tables(batch, tb)) {                         // images are host-written: readable before the wait
        bounded_wait(tb.base, 0, kWaitLimit);              // the table copies into this CTA's shared memory must land first
        dependency_wait();                                 // and the next kernel relies on this one for the previous one's completion
        return;
    }
    GemvPos pos = {0, 0, 0};
    if (u0 < u1) { pos = gemv_pos_of(batch, u0); prefetch_block_l2(gemv_block_ptr(batch, pos, lane)); }
    if (!finish_decode_tables<kGiveUp>(tb)) { pass_gemv_tickets(batch, split, u0, u1, d_tickets, tag); return; }
    dependency_wait();                                     // everything but the host-written tables: after the previous kernel of the stream

    float acc[kV][kChains];                             // partial sums, added when the row tile is left
    auto clear_acc = [&]() {
#pragma unroll
        for (int b = 0; b < kV; ++b)
#pragma unroll
            for (int i = 0; i < kChains; ++i) acc[b][i] = 0.0f;
    };
    clear_acc();
    auto flush = [&](int jf, int tile) {
        const GemvJob& jb = batch.job[jf];
        const int n_out = jb.n_out, kblocks = jb.kblocks, gtile = jb.tile_first + tile;
        float* d_y = jb.y;
        const int row = tile * 32 + lane;
        const bool row_ok = row < n_out;
        const int64_t g0 = jb.unit_first + static_cast<int64_t>(tile) * kblocks;
        const UnitSplit split(U, W);                       // again: not held in registers through the decode
        const int w_lo = split.owner(g0);
        const int w_hi = split.owner(g0 + kblocks - 1);
        if (w_lo == w_hi) {
            if (row_ok) {
#pragma unroll
                for (int b = 0; b < kV; ++b) d_y[static_cast<size_t>(b) * n_out + row] = sum_of(acc[b]);
            }
            return;
        }
        float* mine = d_partial + static_cast<size_t>(wg + gtile) * kV * 32;
#pragma unroll
        for (int b = 0; b < kV; ++b) mine[b * 32 + lane] = sum_of(acc[b]);
        __threadfence();
        __syncwarp();
        unsigned int t = 0;
        if (lane == 0) t = take_ticket(&d_tickets[gtile * kTicketStride]);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t == static_cast<unsigned int>(w_hi - w_lo)) {  // last of the warps that share this tile
            __threadfence();
            if (row_ok) {
#pragma unroll
                for (int b = 0; b < kV; ++b) {
                    // slots are added in warp order whatever the arrival order; loads go out thirty-two at a time (a
                    // 4096-wide row is 32 k-blocks: one round trip to L2 instead of two at the end of the kernel)
                    const float* slot = d_partial + (static_cast<size_t>(w_lo + gtile) * kV + b) * 32 + lane;
                    float sum = 0.0f;
                    int ww = w_lo;
                    for (; ww + 32 <= w_hi + 1; ww += 32, slot += 32 * kV * 32) {
                        float v[32];
#pragma unroll
                        for (int i = 0; i < 32; ++i) v[i] = __ldcg(slot + i * kV * 32);
#pragma unroll
                        for (int i = 0; i < 32; ++i) sum += v[i];
                    }
                    for (; ww + 8 <= w_hi + 1; ww += 8, slot += 8 * kV * 32) {
                        float v[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) v[i] = __ldcg(slot + i * kV * 32);
#pragma unroll
                        for (int i = 0; i < 8; ++i) sum += v[i];
                    }
                    for (; ww <= w_hi; ++ww, slot += kV * 32) sum += __ldcg(slot);
                    d_y[static_cast<size_t>(b) * n_out + row] = sum;
                }
            }
            if (lane == 0) d_tickets[gtile * kTicketStride] = 0;
        }
    };

    // x for a unit is fetched one unit ahead, like the block
    uint2 xraw[kV];
    auto load_x = [&](const GemvPos& p) {
        const GemvJob& jb = batch.job[p.j];
        const size_t k = static_cast<size_t>(jb.kblocks) * kGroup;
#pragma unroll
        for (int b = 0; b < kV; ++b)
            xraw[b] = __ldcg(reinterpret_cast<const uint2*>(jb.x + static_cast<size_t>(b) * k + p.kb * kGroup + lane * 4));
    };
    if (u0 >= u1) return;
    load_x(pos);
    Ticket* const my_ticket[2] = {d_tickets + gemv_tile_of(batch, pos) * kTicketStride, d_tickets + gemv_tile_of(batch, gemv_pos_of(batch, u1 - 1)) * kTicketStride};
    const Ticket seen[2] = {look_at_ticket(my_ticket[0]), look_at_ticket(my_ticket[1])};
    int cur_j = pos.j, cur_tile = pos.tile;
    float T = __ldg(&reinterpret_cast<const DevHeader*>(batch.job[pos.j].meta)->T);
    const int n_units = static_cast<int>(u1 - u0);
    for (int left = n_units; left > 0; --left) {
        if (pos.j != cur_j || pos.tile != cur_tile) {
            flush(cur_j, cur_tile);
            clear_acc();
            if (pos.j != cur_j) T = __ldg(&reinterpret_cast<const DevHeader*>(batch.job[pos.j].meta)->T);
            cur_j = pos.j;
            cur_tile = pos.tile;
        }
        // this warp's slice: lane l holds x[b][kb*128 + 4l .. 4l+3]
        __syncwarp();
#pragma unroll
        for (int b = 0; b < kV; ++b) sts_v2(xs + b * (kGroup * 2) + lane * 8, xraw[b].x, xraw[b].y);
        __syncwarp();
        // the block is fetched when its turn comes (it was prefetched into L2 one unit earlier): holding the next
        // one in sixteen registers through a whole group costs more in resident warps than the fetch costs here
        Block cur;
        ldg_block(cur, gemv_block_ptr(batch, pos, lane));
        if (left == n_units && lane == 0) {                        // lane 0 is the one that takes
            claim_ticket(my_ticket[0], seen[0], tag);
            if (my_ticket[1] != my_ticket[0]) claim_ticket(my_ticket[1], seen[1], tag);
        }
        if (left > 1) {
            pos = gemv_pos_next(batch, pos);
            prefetch_block_l2(gemv_block_ptr(batch, pos, lane));
            load_x(pos);
        }
        fused_group<kV, false>(cur, tb, bits, T, xs, true, acc);
    }
    flush(cur_j, cur_tile);
}

// K3: scores[b][hq][t] = scale * q[b][hq] . K~[b][hq / kV][t] for one or two (kV) query heads per KV head.
// Built like K2: a work unit is (one (batch, kv head) pair, 32 consecutive tokens), a lane owns one token, every
// working warp owns a contiguous run of units and keeps its own query slice (restaged
// when the head changes), so warps never meet at a barrier and a ragged sequence length costs at most one
// partly filled unit per head.
template <int kV, int kMaxWarps>
__global__ void __launch_bounds__(kMaxWarps * 32, 1)
ecco_attn_scores_kernel(const uint8_t* __restrict__ d_meta, const uint8_t* __restrict__ d_kblocks, int heads, int seq,
                        const __half* d_q, float scale, float* __restrict__ d_scores)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    release_dependents();
    const DecodeTables tb = plan_decode_tables(smem_u32(smem), d_meta, true);
    const int nw = static_cast<int>(decode_warps(tb, scalar_warp_bytes(kV)));
    const int lane = static_cast<int>(threadIdx.x & 31u), warp = static_cast<int>(threadIdx.x >> 5);
    const uint32_t xs = tb.warp_base + warp * scalar_warp_bytes(kV);             // this warp's slice [kV][128] fp16
    const uint32_t bits = xs + kV * kGroup * 2 + kRankRows * 128 + lane * 4;

    const int wg = warp < nw ? warp * static_cast<int>(gridDim.x) + static_cast<int>(blockIdx.x) : INT_MAX;
    const int tiles = (seq + 31) / 32;
    const int64_t U = static_cast<int64_t>(heads) * tiles;
    const int W = static_cast<int>(balanced_warps(static_cast<uint64_t>(U), gridDim.x * static_cast<uint32_t>(nw)));
    const UnitSplit split(U, W);
    const int64_t u0 = wg < W ? split.begin(wg) : 0, u1 = wg < W ? split.begin(wg + 1) : 0;
    // lanes past the end of the sequence decode its last token again and store nothing; (head, tile) of a unit is
    // advanced by one per unit instead of divided out of the unit number
    auto block_ptr = [&](int bh, int tile) {
        return d_kblocks + (static_cast<uint64_t>(bh) * seq + min(tile * 32 + lane, seq - 1)) * kBlockBytes;
    };
    int bh = static_cast<int>(divide(static_cast<uint64_t>(u0), static_cast<uint64_t>(tiles))), tile = static_cast<int>(u0 - static_cast<int64_t>(bh) * tiles);
    issue_decode_tables(tb, d_meta);
    if (u0 < u1) prefetch_block_l2(block_ptr(bh, tile));
    if (!finish_decode_tables(tb)) return;
    dependency_wait();                                     // everything but the host-written tables: after the previous kernel of the stream
    const float T = tb.T;

    int cur_bh = -1;
    for (int64_t u = u0; u < u1; ++u) {
        const int t = tile * 32 + lane;
        if (bh != cur_bh) {
            // lane l stages q[b][h * kV + r][4l .. 4l+3]
            __syncwarp();                                  // every lane is done with the previous head's slice
#pragma unroll
            for (int r = 0; r < kV; ++r) {
                const uint2 raw = __ldcg(reinterpret_cast<const uint2*>(d_q + (static_cast<size_t>(bh) * kV + r) * kGroup) + lane);
                sts_v2(xs + r * (kGroup * 2) + lane * 8, raw.x, raw.y);
            }
            __syncwarp();
            cur_bh = bh;
        }
        Block cur;
        ldg_block(cur, block_ptr(bh, tile));
        const int out_bh = bh;
        if (++tile == tiles) { tile = 0; ++bh; }
        if (u + 1 < u1) prefetch_block_l2(block_ptr(bh, tile));
        float acc[kV][kChains];
#pragma unroll
        for (int r = 0; r < kV; ++r)
#pragma unroll
            for (int i = 0; i < kChains; ++i) acc[r][i] = 0.0f;
        fused_group<kV, true>(cur, tb, bits, T, xs, t < seq, acc);
        if (t < seq) {
#pragma unroll
            for (int r = 0; r < kV; ++r)
                d_scores[(static_cast<size_t>(out_bh) * kV + r) * seq + t] = scale * sum_of(acc[r]);
        }
    }
}


}  // namespace
