// ecco_group_tiles.cuh -- a warp's 32 decoded groups as fp16 tiles in shared memory, for the tensor cores
// Part of the one translation unit ecco_kernels.cu; included from there only.
#pragma once

namespace {

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&a)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&a)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                 : "r"(addr));
}
__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// the same with nothing to add to
__device__ __forceinline__ void mma_16816_first(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
                 : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.0f));
}

// What bounds the kernels on tiles is the shared-memory pipe: 3.4 of some 5 wavefronts per symbol of a warp are lookups in the shape
// tables.  The pair tables would halve these, but beside 80 KB of them twelve warps find room, and with the ranks kept
// instead of the values (2 KB, twenty warps or more) the second pass cost more than it saved: [16][8][32768][128] scores and
// values 1067 against 986 us, [8][32][4096][128] 269 against 233.  With the values in registers against a value table in shared
// memory: two 11008 x 4096 matrices by eight rows 91.5 -> 83.7 us, 1000 x 4096 18.3 -> 18.0, the caches above 1040 -> 986 and 234 -> 233.
//
// Eight [32 groups][16 positions] fp16 tiles per warp, the last of which lies over rows 0..7 of the warp's bit-stream array: it
// is written when the whole warp has decoded symbol 127, and by then every lane is past stream bit 256 (ten header bits at
// least and two bits per symbol), while the outlier fields sit in bits 272..511, rows 8..15.
constexpr uint32_t kTileBytes = 1024;
constexpr uint32_t kTiledWarpBytes = 7 * kTileBytes + kBitBytes;

// Position i (0..15) of a tile is staged in column 2q + (j & 1) + 8 (j >> 1) with i = 4q + j where the positions are the
// contraction index (kSpread).  The contraction index of an MMA may be permuted freely as long as both operands agree, and with this
// order the four vector elements a lane needs per tile (columns 2q, 2q+1, 2q+8, 2q+9) are the
// contiguous k = 4q .. 4q+3: one 8-byte load instead of two 4-byte ones.
__host__ __device__ constexpr uint32_t tile_column(uint32_t i) { return 2 * (i >> 2) + (i & 1) + 8 * ((i >> 1) & 1); }

// byte of tile column c in the row of group r: 16-byte halves swapped in every second block of four rows, which makes
// 16-byte stores and ldmatrix conflict-free
__device__ __forceinline__ uint32_t tile_byte(uint32_t r, uint32_t c) { return r * 32 + ((c * 2) ^ (((r >> 2) & 1u) << 4)); }

// One group per lane, outliers in place; a lane with keep = false contributes zeros.  The tiles are complete when this returns.
// kDeal: deal_outliers (caches) or every lane its own (weights).
template <bool kSpread, bool kDeal>
__device__ __forceinline__ void decode_to_tiles(const Block& blk, const DecodeTables& tb, uint32_t tiles, float T, bool keep)
{
    const uint32_t lane = threadIdx.x & 31u, bits = tiles + 7 * kTileBytes + lane * 4;
    const uint32_t my_row = tiles + lane * 32, swz = ((lane >> 2) & 1u) << 4;
    __syncwarp();                                          // the tiles of the previous groups have been read
    LaneGroup g = open_block(blk, bits, tb, T);
    uint32_t even[4] = {0, 0, 0, 0};
    const uint32_t end = decode_group_by_one<kBlockBits, kBlockFreeSteps>(g, bits, [&](int i, uint32_t ranks, bool cutting, int n_ok) {
        uint32_t v[4];
        map_ranks(g, ranks, v);
        if (cutting) cut_values(v, n_ok);
        const uint32_t row = my_row + (i >> 1) * kTileBytes;
        if (i & 1) {                                       // both halves now: the last tile may not be touched before symbol 127
            if (kSpread) {
                sts_v4(row + swz, even[0], even[2], v[0], v[2]);
                sts_v4(row + (swz ^ 16u), even[1], even[3], v[1], v[3]);
            } else {
                sts_v4(row + swz, even[0], even[1], even[2], even[3]);
                sts_v4(row + (swz ^ 16u), v[0], v[1], v[2], v[3]);
            }
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) even[k] = v[k];
        }
    });
    // outliers of a complete group replace the mapped values in the tiles
    auto put = [&](uint32_t owner, uint32_t f) {
        const uint32_t loc = f & 127u, i = loc & 15u;
        sts_u16(tiles + (loc >> 4) * kTileBytes + tile_byte(owner, kSpread ? tile_column(i) : i), f2h_bits(fp8_to_float(f >> 7) * T));
    };
    const int n_pad = keep ? pads_of(end) : 0;
    if (!kDeal) {
        for (int j = 0; j < n_pad; ++j) put(lane, pad_field(bits, j));         // ascending: a later pad overrides an earlier one
    } else if (warp_any(n_pad > 0)) {
        deal_outliers(bits, bits - lane * 4 + 16 * 128, n_pad, [&](uint32_t, uint32_t owner, uint32_t f, bool valid) { if (valid) put(owner, f); },
                      [](uint32_t, int) {});
    }
    if (warp_any(!keep)) {
        if (!keep) {
#pragma unroll
            for (int ch = 0; ch < 8; ++ch) {
                sts_v4(my_row + ch * kTileBytes, 0u, 0u, 0u, 0u);
                sts_v4(my_row + ch * kTileBytes + 16, 0u, 0u, 0u, 0u);
            }
        }
    }
    __syncwarp();
}

}  // namespace
