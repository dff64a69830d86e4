// ecco_fused_mma_kernels.cuh -- K2m / K3m: fused GEMV (six to eight rows) and attention scores (three to eight heads) on the tensor cores
// Part of the one translation unit ecco_kernels.cu; included from there only.
#pragma once

namespace {

// ---------------------------------------------------------------------------------------------
// K2m / K3m: the fused consumers for six to eight rows of x and three to eight query heads on the
// tensor cores: with eight products per weight the per-warp path spends eight FMAs per symbol.  Here the groups are
// decoded into tiles and each tile is contracted against the fp16
// vector fragments: C[32 rows][8] += tile[32 x 16] * V[16 x 8], two mma.m16n8k16 per tile, fp32
// accumulate (fp16 x fp16 products are exact in fp32).  A warp is independent of the others: no
// vector slice in shared memory, no block barrier.
// ---------------------------------------------------------------------------------------------
// vfrag[2c], vfrag[2c+1]: B fragments of chunk c (tile columns (lane%4)*2 + {0,1}, and + 8), vector lane/4
// acc[0] / acc[1]: C fragments of rows 0..15 / 16..31 of the warp's 32 groups
// fetch_vectors(vfrag) is called after the decode: a caller whose vectors change with every group (the GEMV)
// loads them there, so that they do not occupy sixteen registers during the decode; one whose vectors stay
// (the scores) copies them.
__device__ __forceinline__ void load_vfrag(uint32_t (&vfrag)[16], const __half* base, size_t col_stride, int n_cols);

// kDeal, keep: see decode_to_tiles (the scores of lanes past the end of a row are not wanted)
template <bool kDeal, class FetchVectors>
__device__ __forceinline__ void row_dot_mma(const Block& blk, const DecodeTables& tb, uint32_t tiles, float T, bool keep,
                                            FetchVectors&& fetch_vectors, float (&acc)[2][4])
{
    const uint32_t lane = threadIdx.x & 31u;
    decode_to_tiles<true, kDeal>(blk, tb, tiles, T, keep);
    uint32_t vfrag[16];
    fetch_vectors(vfrag);
    const uint32_t a_at = tiles + tile_byte(((lane >> 3) & 1u) * 8 + (lane & 7u), (lane >> 4) * 8);
#pragma unroll
    for (int ch = 0; ch < 8; ++ch) {
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
            uint32_t a[4];
            ldmatrix_x4(a, a_at + ch * kTileBytes + mt * 512);                 // rows + 16: the same swizzle
            mma_16816(acc[mt], a, vfrag[2 * ch], vfrag[2 * ch + 1]);
        }
    }
}

// fragments of eight fp16 vectors v[col][k0 .. k0+127] (col = lane/4; columns >= n_cols are zero)
__device__ __forceinline__ void load_vfrag(uint32_t (&vfrag)[16], const __half* base, size_t col_stride, int n_cols)
{
    const int lane = static_cast<int>(threadIdx.x & 31u), col = lane >> 2;
    const uint2* p = reinterpret_cast<const uint2*>(base + static_cast<size_t>(min(col, n_cols - 1)) * col_stride) + (lane & 3);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const uint2 v = col < n_cols ? __ldcg(p + c * 4) : make_uint2(0u, 0u);     // k = 16c + 4 (lane%4) .. + 3
        vfrag[2 * c] = v.x;                                // tile columns 2q, 2q+1
        vfrag[2 * c + 1] = v.y;                            // tile columns 2q+8, 2q+9
    }
}

// K2m: y[b][n] = sum_k W~[n][k] x[b][k] for six to eight rows of x.  Units (over all matrices of the call), ownership and the
// slot-and-ticket reduction are those of the per-warp kernel (unit = 32 rows x one k-block).
template <int kMaxWarps, bool kGiveUp>
__global__ void __launch_bounds__(kMaxWarps * 32, 1)
ecco_gemv_mma_kernel(const __grid_constant__ GemvBatch batch, int n_cols, float* __restrict__ d_partial,
                     Ticket* d_tickets, Ticket tag)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const int lane = static_cast<int>(threadIdx.x & 31u), warp = static_cast<int>(threadIdx.x >> 5);
    release_dependents();
    const uint8_t* d_meta = batch.job[0].meta;
    const DecodeTables tb = plan_decode_tables(smem_u32(smem), d_meta, false);       // one symbol per lookup: the tiles need the room
    const int nw = static_cast<int>(decode_warps(tb, kTiledWarpBytes));
    const uint32_t tiles_at = tb.warp_base + warp * kTiledWarpBytes;

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
    if (u0 >= u1) return;

    float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    // C fragment element (mt, i): row = 16 mt + lane/4 + 8 (i >= 2), column b = (lane%4)*2 + (i & 1)
    auto flush = [&](int jf, int tile) {
        const GemvJob& jb = batch.job[jf];
        const int n_out = jb.n_out, kblocks = jb.kblocks, gtile = jb.tile_first + tile;
        float* d_y = jb.y;
        const int64_t g0 = jb.unit_first + static_cast<int64_t>(tile) * kblocks;
        const UnitSplit split(U, W);                       // again: not held in registers through the decode
        const int w_lo = split.owner(g0);
        const int w_hi = split.owner(g0 + kblocks - 1);
        float* mine = d_partial + static_cast<size_t>(wg + gtile) * 8 * 32;
        if (w_lo != w_hi) {
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    mine[((lane & 3) * 2 + (i & 1)) * 32 + 16 * mt + (lane >> 2) + (i >= 2 ? 8 : 0)] = acc[mt][i];
            __threadfence();
            __syncwarp();
            unsigned int t = 0;
            if (lane == 0) t = take_ticket(&d_tickets[gtile * kTicketStride]);
            t = __shfl_sync(0xffffffffu, t, 0);
            if (t != static_cast<unsigned int>(w_hi - w_lo)) return;
            __threadfence();
        }
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = 16 * mt + (lane >> 2) + (i >= 2 ? 8 : 0), b = (lane & 3) * 2 + (i & 1);
                const int row = tile * 32 + r;
                float sum = acc[mt][i];
                if (w_lo != w_hi) {                        // slots in warp order, whatever the arrival order
                    sum = 0.0f;
                    for (int ww = w_lo; ww <= w_hi; ++ww) sum += __ldcg(d_partial + (static_cast<size_t>(ww + gtile) * 8 + b) * 32 + r);
                }
                if (row < n_out && b < n_cols) d_y[static_cast<size_t>(b) * n_out + row] = sum;
            }
        if (w_lo != w_hi && lane == 0) d_tickets[gtile * kTicketStride] = 0;
    };

    Ticket* const my_ticket[2] = {d_tickets + gemv_tile_of(batch, pos) * kTicketStride, d_tickets + gemv_tile_of(batch, gemv_pos_of(batch, u1 - 1)) * kTicketStride};
    const Ticket seen[2] = {look_at_ticket(my_ticket[0]), look_at_ticket(my_ticket[1])};
    int cur_j = pos.j, cur_tile = pos.tile;
    float T = __ldg(&reinterpret_cast<const DevHeader*>(batch.job[pos.j].meta)->T);
    const int n_units = static_cast<int>(u1 - u0);
    for (int left = n_units; left > 0; --left) {
        const GemvJob& jb = batch.job[pos.j];
        const int tile = pos.tile;
        if (pos.j != cur_j || tile != cur_tile) {
            flush(cur_j, cur_tile);
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[mt][i] = 0.0f;
            if (pos.j != cur_j) T = __ldg(&reinterpret_cast<const DevHeader*>(jb.meta)->T);
            cur_j = pos.j;
            cur_tile = tile;
        }
        Block cur;                                         // fetched now, prefetched into L2 one unit earlier (see the scalar kernels)
        ldg_block(cur, gemv_block_ptr(batch, pos, lane));
        if (left == n_units && lane == 0) {                        // lane 0 is the one that takes
            claim_ticket(my_ticket[0], seen[0], tag);
            if (my_ticket[1] != my_ticket[0]) claim_ticket(my_ticket[1], seen[1], tag);
        }
        const __half* xk = jb.x + pos.kb * kGroup;
        const size_t k = static_cast<size_t>(jb.kblocks) * kGroup;
        if (left > 1) { pos = gemv_pos_next(batch, pos); prefetch_block_l2(gemv_block_ptr(batch, pos, lane)); }
        row_dot_mma<false>(cur, tb, tiles_at, T, true, [&](uint32_t (&v)[16]) { load_vfrag(v, xk, k, n_cols); }, acc);
    }
    flush(cur_j, cur_tile);
}

// K3m: scores[b][hq][t] = scale * q[b][hq] . K~[b][hq / q_per_kv][t] for 3..8 query heads per KV head.
// Unit = (one (batch, kv head), 32 tokens); every working warp owns a contiguous run of units.
template <int kMaxWarps>
__global__ void __launch_bounds__(kMaxWarps * 32, 1)
ecco_attn_scores_mma_kernel(const uint8_t* __restrict__ d_meta, const uint8_t* __restrict__ d_kblocks, int heads, int seq,
                            int q_per_kv, const __half* d_q, float scale, float* __restrict__ d_scores)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const int lane = static_cast<int>(threadIdx.x & 31u), warp = static_cast<int>(threadIdx.x >> 5);
    release_dependents();
    const DecodeTables tb = plan_decode_tables(smem_u32(smem), d_meta, false);       // one symbol per lookup: the tiles need the room
    const int nw = static_cast<int>(decode_warps(tb, kTiledWarpBytes));
    const uint32_t tiles_at = tb.warp_base + warp * kTiledWarpBytes;

    const int wg = warp < nw ? warp * static_cast<int>(gridDim.x) + static_cast<int>(blockIdx.x) : INT_MAX;
    const int tiles = (seq + 31) / 32;
    const int64_t U = static_cast<int64_t>(heads) * tiles;
    const int W = static_cast<int>(balanced_warps(static_cast<uint64_t>(U), gridDim.x * static_cast<uint32_t>(nw)));
    const UnitSplit split(U, W);
    const int64_t u0 = wg < W ? split.begin(wg) : 0, u1 = wg < W ? split.begin(wg + 1) : 0;
    auto block_ptr = [&](int bh, int tile) {
        return d_kblocks + (static_cast<uint64_t>(bh) * seq + min(tile * 32 + lane, seq - 1)) * kBlockBytes;
    };
    int nbh = static_cast<int>(divide(static_cast<uint64_t>(u0), static_cast<uint64_t>(tiles))), ntile = static_cast<int>(u0 - static_cast<int64_t>(nbh) * tiles);     // advanced by one per unit
    issue_decode_tables(tb, d_meta);
    if (u0 < u1) prefetch_block_l2(block_ptr(nbh, ntile));
    if (!finish_decode_tables(tb)) return;
    dependency_wait();                                     // everything but the host-written tables: after the previous kernel of the stream
    const float T = tb.T;

    uint32_t vfrag[16];
    int cur_bh = -1;
    for (int64_t u = u0; u < u1; ++u) {
        const int bh = nbh, t0 = ntile * 32;
        if (bh != cur_bh) { load_vfrag(vfrag, d_q + static_cast<size_t>(bh) * q_per_kv * kGroup, kGroup, q_per_kv); cur_bh = bh; }
        Block cur;
        ldg_block(cur, block_ptr(nbh, ntile));
        if (++ntile == tiles) { ntile = 0; ++nbh; }
        if (u + 1 < u1) prefetch_block_l2(block_ptr(nbh, ntile));
        float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
        row_dot_mma<true>(cur, tb, tiles_at, T, t0 + lane < seq,
                    [&](uint32_t (&v)[16]) {
#pragma unroll
                        for (int i = 0; i < 16; ++i) v[i] = vfrag[i];
                    }, acc);
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int t = t0 + 16 * mt + (lane >> 2) + (i >= 2 ? 8 : 0), r = (lane & 3) * 2 + (i & 1);
                if (t < seq && r < q_per_kv) d_scores[(static_cast<size_t>(bh) * q_per_kv + r) * seq + t] = scale * acc[mt][i];
            }
    }
}


}  // namespace
