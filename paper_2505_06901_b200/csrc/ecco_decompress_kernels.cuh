// ecco_decompress_kernels.cuh -- K1 / K1v: ecco_decompress and ecco_var_decompress kernels
// Part of the one translation unit ecco_kernels.cu; included from there only.
#pragma once

namespace {

// ---------------------------------------------------------------------------------------------
// K1: ecco_decompress
// ---------------------------------------------------------------------------------------------
// number of working warps <= w_max such that `units` split evenly: all get ceil(units / w_max) or one less
__host__ __device__ __forceinline__ uint32_t balanced_warps(uint64_t units, uint32_t w_max)
{
    if (units <= w_max) return static_cast<uint32_t>(units);
    const uint64_t per_warp = divide(units + w_max - 1, w_max);
    return static_cast<uint32_t>(divide(units + per_warp - 1, per_warp));
}

// Work is dealt out in warp tiles of 32 consecutive groups, tile i to warp (i mod working warps):
// every SM then gets the same number of tiles to within one, whatever the tensor size.
constexpr uint32_t kSmallWarpBytes = kBitBytes;
template <int kMaxWarps>
__global__ void __launch_bounds__(kMaxWarps * 32, 1)
ecco_decompress_kernel(const uint8_t* __restrict__ d_meta, const uint8_t* __restrict__ d_blocks, uint64_t n_groups,
                       uint16_t* __restrict__ d_out)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const DecodeTables tb = plan_decode_tables(smem_u32(smem), d_meta, true);
    const uint32_t nw = decode_warps(tb, kSmallWarpBytes);
    const uint32_t bits = tb.warp_base + warp * kSmallWarpBytes + lane * 4;
    const uint64_t n_tiles = (n_groups + 31) / 32;
    // every working warp gets the same number of tiles (+-1 over the whole grid); warp ids interleave over
    // the CTAs, so every SM keeps the same number busy
    const uint64_t tile_stride = balanced_warps(n_tiles, gridDim.x * nw);
    uint64_t tile = static_cast<uint64_t>(warp) * gridDim.x + blockIdx.x;
    if (warp >= nw || tile >= tile_stride) tile = n_tiles;               // this warp sits the launch out (after the table barrier)
    issue_decode_tables(tb, d_meta);
    if (!finish_decode_tables(tb)) return;
    const float T = tb.T;

    for (; tile < n_tiles; tile += tile_stride) {
        const uint64_t g = tile * 32 + lane;
        const bool store = g < n_groups;                   // lanes past the end of the tensor decode the last group again and store nothing
        Block blk;
        ldg_block(blk, d_blocks + min(g, n_groups - 1) * kBlockBytes);
        LaneGroup lg = open_block(blk, bits, tb, T);
        uint16_t* out = d_out + min(g, n_groups - 1) * kGroup;
        const uint32_t end = decode_group<kBlockBits, kBlockFreeSteps>(lg, bits, tb.pairs, [&](int i, uint32_t ranks, bool cutting, int n_ok) {
            uint32_t v[4];
            map_ranks(lg, ranks, v);
            if (cutting) cut_values(v, n_ok);
            if (store) *reinterpret_cast<uint4*>(out + i * 8) = make_uint4(v[0], v[1], v[2], v[3]);
        });
        if (store) {
            const int n_pad = pads_of(end);
            for (int j = 0; j < n_pad; ++j) {
                const uint32_t f = pad_field(bits, j);
                // same thread, same address as the vector store above: program order holds
                out[f & 127u] = static_cast<uint16_t>(f2h_bits(fp8_to_float(f >> 7) * T));
            }
        }
    }
}

// K1, bulk-store variant.  Per-lane 32-byte stores land in 32 different 128-byte lines and cost the
// load/store pipe one pass per sector.  Here every 16 decoded values per lane go to a 1 KB
// staging tile in shared memory ([32 groups][32 bytes], 16-byte halves swizzled the way the
// tensor map's 32-byte swizzle expects, so the 128-bit shared stores are conflict-free) and one
// lane hands the tile to the TMA engine, which writes the 32 rows of the [n_groups][128] fp16
// tensor and drops rows past its end.  Outliers: those in the last tile (positions >= 112) are
// patched in shared memory before that tile leaves; the others are 2-byte global stores issued
// after the group's earlier tiles have been written (bulk wait + warp barrier), so they land last.
//
// The kernel takes up to kMaxJobs tensors.  Consecutive tensors whose images carry the same tables (equal table
// hash: the matrices of a layer calibrated together differ in the exponent only) form a run: the tables are
// staged once per run and the warp tiles of all its tensors are dealt out as one tile space, so a run pays one
// table fetch and one tail.  Between two runs only the CTA's own warps meet (the tables are the CTA's), so an SM
// that is done with one run starts the next while others still finish.
constexpr int kMaxJobs = 8;
struct alignas(64) DecompressJob {
    const uint8_t* meta;
    const uint8_t* blocks;
    uint64_t n_groups;
    uint16_t* out;
    uint32_t reserved[8];
    CUtensorMap map;           // [n_groups][128] fp16, box 32 x 16, 32-byte swizzle
};
struct DecompressBatch {
    int32_t n;
    int32_t reserved[15];
    DecompressJob job[kMaxJobs];
};
constexpr uint32_t kTmaWarpBytes = 1024 + kBitBytes;                 // staging tile, bit-stream array

template <int kMaxWarps>
__global__ void __launch_bounds__(kMaxWarps * 32, 1)
ecco_decompress_tma_kernel(const __grid_constant__ DecompressBatch batch)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t smem_base = smem_u32(smem);
    const uint32_t swz = ((lane >> 2) & 1u) << 4;                               // 32-byte swizzle: bit 4 ^= bit 7

    // The metadata images are written by the host only, never by a kernel of this library, and this kernel can
    // start early only behind a kernel that releases its dependents, i.e. one of this library: the tables of the
    // first run are fetched before the wait on the previous kernel, everything else after it.
    release_dependents();
    auto hash_of = [&](int t) {
        const DevHeader* hd = reinterpret_cast<const DevHeader*>(batch.job[t].meta);
        return make_uint2(__ldg(&hd->hash_lo), __ldg(&hd->hash_hi));
    };
    auto tiles_of = [&](int t) { return static_cast<uint32_t>((batch.job[t].n_groups + 31) / 32); };   // at most 2^26, eight jobs 2^29
    int run = 0;
    for (int t0 = 0; t0 < batch.n; ++run) {
        const DecodeTables tb = plan_decode_tables(smem_base, batch.job[t0].meta, true);
        int t1 = t0 + 1;
        uint32_t run_tiles = tiles_of(t0);
        for (; t1 < batch.n; ++t1) {
            const uint2 hh = hash_of(t1);
            if (hh.x != tb.hash_lo || hh.y != tb.hash_hi) break;
            run_tiles += tiles_of(t1);
        }
        if (run > 0) {
            // Every warp is done with the previous run's tables.  The copies below write where ordinary stores have written (the records
            // that build_rank_tables rewrote, warps' arrays of another layout): every thread orders its stores before them.
            fence_async_smem();
            __syncthreads();
        }
        issue_decode_tables(tb, batch.job[t0].meta, run == 0);
        const uint32_t tiles_base = (tb.warp_base + 1023u) & ~1023u;
        const uint32_t nw = decode_warps(tb, kTmaWarpBytes, tiles_base - tb.warp_base);
        const uint32_t stage = tiles_base + warp * 1024;                       // this warp's staging tile
        const uint32_t bits = tiles_base + nw * 1024 + warp * kBitBytes + lane * 4;
        const uint32_t my_row = stage + lane * 32;
        const uint32_t tile_stride = balanced_warps(run_tiles, gridDim.x * nw);
        uint32_t gt = warp * gridDim.x + blockIdx.x;                           // tile in the run's tile space
        if (warp >= nw || gt >= tile_stride) gt = run_tiles;
        // the job that holds tile gt, and the first tile of that job in the run's tile space
        int job_at = t0;
        uint32_t job_first = 0, job_tiles = tiles_of(t0);
        auto seek = [&](uint32_t g) {
            while (g >= job_first + job_tiles && job_at + 1 < t1) { job_first += job_tiles; ++job_at; job_tiles = tiles_of(job_at); }
        };
        auto block_ptr = [&](uint32_t g) {
            const DecompressJob& job = batch.job[job_at];
            return job.blocks + static_cast<uint64_t>(min((g - job_first) * 32 + lane, static_cast<uint32_t>(job.n_groups) - 1u)) * kBlockBytes;
        };
        if (gt < run_tiles) { seek(gt); prefetch_block_l2(block_ptr(gt)); }
        if (!finish_decode_tables(tb, static_cast<uint32_t>(run & 1))) return;
        if (run == 0) dependency_wait();                   // blocks and output: only after the previous kernel has completed

        while (gt < run_tiles) {
            const DecompressJob& job = batch.job[job_at];
            const float T = __ldg(&reinterpret_cast<const DevHeader*>(job.meta)->T);
            const uint32_t row0 = (gt - job_first) * 32, g = row0 + lane;
            const bool store = g < static_cast<uint32_t>(job.n_groups);
            uint16_t* out = job.out + static_cast<uint64_t>(g) * kGroup;
            const CUtensorMap* out_map = &job.map;
            // The block is fetched when its turn comes, after a prefetch into L2 one tile earlier: holding the next
            // block in sixteen registers through a whole group would cost four of the 32 warps.
            Block blk;
            ldg_block(blk, block_ptr(gt));
            LaneGroup lg = open_block(blk, bits, tb, T);
            gt += tile_stride;
            if (gt < run_tiles) { seek(gt); prefetch_block_l2(block_ptr(gt)); }
            auto send_tile = [&](int x) {
                fence_async_smem();                            // generic-proxy writes -> visible to the engine
                __syncwarp();
                if (lane == 0) { tma_store_2d(out_map, stage, x, static_cast<int>(row0)); bulk_commit(); }
            };
            const uint32_t end = decode_group<kBlockBits, kBlockFreeSteps>(lg, bits, tb.pairs, [&](int i, uint32_t ranks, bool cutting, int n_ok) {
                uint32_t v[4];
                map_ranks(lg, ranks, v);
                if (cutting) cut_values(v, n_ok);
                if (!(i & 1)) {
                    if (lane == 0) bulk_wait_read0();          // the engine has read the previous tile
                    __syncwarp();
                    sts_v4(my_row + swz, v[0], v[1], v[2], v[3]);
                } else {
                    sts_v4(my_row + (swz ^ 16u), v[0], v[1], v[2], v[3]);
                    if (i != 15) send_tile(i * 8 - 8);
                }
            });
            const int n_pad = pads_of(end);
            const int n_max = __reduce_max_sync(0xffffffffu, n_pad);
            if (n_max > 0) {
                if (lane == 0) bulk_wait_all();                // tiles 0..6 of this group are in memory
                __syncwarp();
#pragma unroll 1
                for (int j = 0; j < n_max; ++j) {              // ascending: a later pad overrides an earlier one
                    if (j < n_pad) {
                        const uint32_t f = pad_field(bits, j);
                        const uint32_t loc = f & 127u;
                        const unsigned short val = static_cast<unsigned short>(f2h_bits(fp8_to_float(f >> 7) * T));
                        if (loc >= 112u) {
                            const uint32_t byte = (loc - 112u) * 2;
                            asm volatile("st.shared.u16 [%0], %1;" ::"r"(my_row + ((byte & 16u) ^ swz) + (byte & 15u)), "h"(val) : "memory");
                        } else if (store) {
                            out[loc] = val;
                        }
                    }
                }
            }
            send_tile(112);
        }
        if (lane == 0) bulk_wait_all();                    // the staging tile may move with the next run's layout
        t0 = t1;
    }
}

// ---------------------------------------------------------------------------------------------
// K1v: decompress of the variable-length container (groups back to back in one bit stream, start
// index on the side; nothing clipped, nothing padded).  Same thread-per-group decode and the same
// TMA tile store as K1; the difference is the front end: a lane copies twenty words of the stream, from the 64-bit word in which
// its group begins, into its column of a transposed array, masks the bits that belong to the next group, and starts
// decoding at bit (start mod 64).  Groups of weights take 503 bits, and one in ten thousand does not fit; such a lane
// fetches again from where it has got to, in the middle of the group, and so does one that has run past its group's end
// (a corrupt index), for zeros.  A column of 24 rows instead of the 40 that the longest group covers is what leaves
// room for 28 warps beside the pair tables, hence one round of tiles where 19 warps would need two.  Against one symbol per lookup
// and a value table in shared memory: 131 072 groups of weights 19.9 -> 14.8 us, of which the memory traffic is 6.5.
// ---------------------------------------------------------------------------------------------
constexpr uint32_t kVarBits = 640;                       // of the stream at a time
constexpr uint32_t kVarRows = kVarBits / 32 + 4;         // and four zero rows: how far a step that starts inside the data may read
constexpr uint32_t kVarBitsBytes = kVarRows * 128;
constexpr uint32_t kVarWarpBytes = 1024 + kVarBitsBytes;

template <int kMaxWarps>
__global__ void __launch_bounds__(kMaxWarps * 32, 1)
ecco_var_decompress_kernel(const uint8_t* __restrict__ d_meta, const uint4* __restrict__ d_stream,
                           const uint64_t* __restrict__ d_index, uint64_t n_groups,
                           const __grid_constant__ CUtensorMap out_map)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;

    release_dependents();
    const DecodeTables tb = plan_decode_tables(smem_u32(smem), d_meta, true);
    const uint32_t tiles_base = (tb.warp_base + 1023u) & ~1023u;
    const uint32_t nw = decode_warps(tb, kVarWarpBytes, tiles_base - tb.warp_base);
    const uint32_t stage = tiles_base + warp * 1024;
    const uint32_t bits = tiles_base + nw * 1024 + warp * kVarBitsBytes + lane * 4;
    if (warp < nw)
        for (uint32_t r = kVarBits / 32; r < kVarRows; ++r) sts_u32(bits + r * 128, 0u);
    const uint32_t swz = ((lane >> 2) & 1u) << 4;
    const uint32_t my_row = stage + lane * 32;
    issue_decode_tables(tb, d_meta);
    dependency_wait();                                     // everything but the host-written tables: after the previous kernel of the stream
    const uint64_t total_bits = d_index[0];
    const uint64_t* chunk_base = d_index + 1;
    const uint32_t* off32 = reinterpret_cast<const uint32_t*>(d_index + 1 + var_chunks(n_groups));
    auto start_of = [&](uint64_t g) { return g < n_groups ? chunk_base[g >> kVarChunkShift] + off32[g] : total_bits; };

    const uint64_t n_tiles = (n_groups + 31) / 32;
    const uint64_t tile_stride = balanced_warps(n_tiles, gridDim.x * nw);
    uint64_t tile = static_cast<uint64_t>(warp) * gridDim.x + blockIdx.x;
    if (warp >= nw || tile >= tile_stride) tile = n_tiles;

    // The span of a group comes from the index and its chunks from the stream: two dependent trips to memory.
    // The span is fetched one tile ahead and its chunks are sent for, into L2.
    struct Span { const uint2* at; uint32_t first, end; };               // first 64-bit word; bits in it before the group, and up to its end
    auto span_of = [&](uint64_t t) {
        const uint64_t g = min(t * 32 + lane, n_groups - 1);
        const uint64_t from = min(start_of(g), total_bits);
        const uint64_t to = max(min(start_of(g + 1), total_bits), from);   // the group sees [from, to), zeros after
        const uint64_t w0 = from >> 6;
        Span sp;
        sp.at = reinterpret_cast<const uint2*>(d_stream) + w0;
        sp.first = static_cast<uint32_t>(from & 63u);
        sp.end = static_cast<uint32_t>(min(to - (w0 << 6), static_cast<uint64_t>(2048)));      // the longest group ends by 63 + 1046
        // groups lie back to back: the lanes' two sectors each cover the stream but for single sectors of long groups
        if (sp.end) {
            asm volatile("prefetch.global.L2 [%0];" ::"l"(sp.at));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(sp.at + ((sp.end - 1u) >> 7)));
        }
        return sp;
    };
    Span cur = {nullptr, 0, 0};
    if (tile < n_tiles) cur = span_of(tile);
    if (!finish_decode_tables(tb)) return;
    const float T = tb.T;

    for (; tile < n_tiles; tile += tile_stride) {
        Span sp = cur;
        uint32_t limit = 0;                                // a lane that starts a step behind this bit fetches first
        auto fill = [&]() {
            // whole 16-byte chunks are loaded: from half a chunk earlier, and half a chunk more, if the first word is a chunk's second
            const uint32_t odd = (reinterpret_cast<uintptr_t>(sp.at) >> 3) & 1u, end = sp.end ? sp.end + odd * 64u : 0u;
            const uint2* from = sp.at - odd;
            const uint32_t to = bits - odd * 256u;
            uint4 ch[kVarBits / 128 + 1];
#pragma unroll
            for (uint32_t c = 0; c <= kVarBits / 128; ++c) {
                ch[c] = make_uint4(0, 0, 0, 0);
                if (c * 128 < end && (c < kVarBits / 128 || odd))
                    asm volatile("ld.global.cg.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(ch[c].x), "=r"(ch[c].y), "=r"(ch[c].z), "=r"(ch[c].w) : "l"(from + 2 * c));
            }
#pragma unroll
            for (uint32_t c = 0; c <= kVarBits / 128; ++c) {
                uint32_t w[4] = {ch[c].x, ch[c].y, ch[c].z, ch[c].w};
                if (end < c * 128 + 128) {                 // bits of the next group read as zero
#pragma unroll
                    for (uint32_t k = 0; k < 4; ++k) {
                        uint32_t drop;                     // shl: amounts above 31 give zero
                        asm("shl.b32 %0, -1, %1;" : "=r"(drop) : "r"(static_cast<uint32_t>(max(static_cast<int>(end) - static_cast<int>(c * 128 + 32 * k), 0))));
                        w[k] &= ~drop;
                    }
                }
#pragma unroll
                for (uint32_t k = 0; k < 4; ++k) {
                    const uint32_t r = 4 * c + k;
                    if (r < 2 ? !odd : r < kVarBits / 32 || (odd && r < kVarBits / 32 + 2)) sts_u32(to + r * 128, w[k]);
                }
            }
            // a step takes 64 bits at most, from the position p + 1 on
            limit = sp.end > kVarBits ? kVarBits - 65u : sp.end;
        };
        fill();
        const uint32_t first = sp.first;
        if (tile + tile_stride < n_tiles) cur = span_of(tile + tile_stride);
        const uint32_t hdr = __funnelshift_r(lds_u32(bits + (first >> 5) * 128), lds_u32(bits + (first >> 5) * 128 + 128), first);
        LaneGroup lg = open_lane_group(hdr, first, tb, T);
        const int row0 = static_cast<int>(tile * 32);
        decode_group<kVarRows * 32, 16>(lg, bits, tb.pairs, [&](int i, uint32_t ranks, bool, int) {
            uint32_t v[4];
            map_ranks(lg, ranks, v);
            if (!(i & 1)) {
                if (lane == 0) bulk_wait_read0();          // the engine has read the previous tile
                __syncwarp();
                sts_v4(my_row + swz, v[0], v[1], v[2], v[3]);
            } else {
                sts_v4(my_row + (swz ^ 16u), v[0], v[1], v[2], v[3]);
                fence_async_smem();
                __syncwarp();
                if (lane == 0) { tma_store_2d(&out_map, stage, i * 8 - 8, row0); bulk_commit(); }
            }
        }, [&](uint32_t& p) {
            if (p > limit) {
                sp.at += p >> 6;
                sp.end -= min(sp.end, p & ~63u);
                p &= 63u;
                fill();
            }
        });
    }
    if (lane == 0) bulk_wait_all();
}


}  // namespace
