// ecco_kv_compress_kernel.cuh -- online 4x compressor kernel
// Part of the one translation unit ecco_kernels.cu; included from there only.
#pragma once

// ---------------------------------------------------------------------------------------------
// Online 4x compressor for the KV cache (Sec. 4.3, "High Compression Ratio (4x) Compressor"):
// one warp encodes one group of 128 fp16 values into its 64-byte block, four values per lane.
//   sorter stage      abs-max (first on ties) -> FP8 scale byte; min / max of the normalised rest
//   pattern selector  fitness = (pattern min - group min)^2 + (pattern max - group max)^2, S scores
//                     spread over the lanes, arg-min with ties to the lower id
//   encoders          nearest centroid per value, the four codebooks' total lengths, the shortest
//                     wins (ID_HF); bit positions by a warp prefix sum
//   pack / clip       codewords OR-ed into the block image in shared memory; the first codeword
//                     that crosses bit 512 is truncated and the rest dropped; a complete group is
//                     padded with its next-largest values (15-bit outliers from the tail)
// Every comparison that decides an index is made in the same precision and order as the host
// encoder (fp32 division by the scale, fp64 squared distances, no fused multiply-add), so the
// blocks are byte-identical to ecco_encode_host with ECCO_SELECT_MINMAX | ECCO_KEEP_EXPONENT.
// ---------------------------------------------------------------------------------------------
namespace {

constexpr int kKvWarps = 8;

__global__ void __launch_bounds__(kKvWarps * 32)
ecco_kv_compress_kernel(const uint8_t* __restrict__ d_meta, const __half* __restrict__ d_x, uint64_t n_groups,
                        uint8_t* __restrict__ d_blocks)
{
    __shared__ __align__(16) uint16_t pat_s[kMaxPatterns * 16];
    __shared__ __align__(16) uint16_t enc_s[kMaxPatterns * kCodebooks * kSymbols];
    __shared__ __align__(16) uint16_t kp_s[kMaxPatterns];
    __shared__ uint32_t blk_s[kKvWarps][16];
    const int tid = static_cast<int>(threadIdx.x), lane = tid & 31, warp = tid >> 5;
    release_dependents();
    {                                                      // the image is host-written: read before the wait on the previous kernel
        const uint4* src_p = reinterpret_cast<const uint4*>(d_meta + kOffPattern);
        for (int i = tid; i < static_cast<int>(kPatternBytes / 16); i += kKvWarps * 32) reinterpret_cast<uint4*>(pat_s)[i] = src_p[i];
        const uint4* src_e = reinterpret_cast<const uint4*>(d_meta + kOffEncCb);
        for (int i = tid; i < static_cast<int>(kEncCbBytes / 16); i += kKvWarps * 32) reinterpret_cast<uint4*>(enc_s)[i] = src_e[i];
        const uint4* src_k = reinterpret_cast<const uint4*>(d_meta + kOffEncKp);
        for (int i = tid; i < static_cast<int>(kEncKpBytes / 16); i += kKvWarps * 32) reinterpret_cast<uint4*>(kp_s)[i] = src_k[i];
    }
    dependency_wait();                                     // x and the blocks: after the previous kernel of the stream
    __syncthreads();
    const DevHeader* hdr = reinterpret_cast<const DevHeader*>(d_meta);
    const int S = hdr->S;
    const float T = hdr->T, invT = 1.0f / T;             // both exact powers of two
    const unsigned full = 0xffffffffu;
    uint32_t* blk = blk_s[warp];
    auto fp8 = [&](float v) { return static_cast<uint32_t>(__nv_cvt_float_to_fp8(v * invT, __NV_SATFINITE, __NV_E4M3)); };

    for (uint64_t g = static_cast<uint64_t>(blockIdx.x) * kKvWarps + warp; g < n_groups; g += static_cast<uint64_t>(gridDim.x) * kKvWarps) {
        const uint2 raw = __ldcg(reinterpret_cast<const uint2*>(d_x + g * kGroup) + lane);
        const uint32_t h16[4] = {raw.x & 0xffffu, raw.x >> 16, raw.y & 0xffffu, raw.y >> 16};
        float x[4];
        uint32_t key[4];                                   // |x| then low index first
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            x[j] = __half2float(__ushort_as_half(static_cast<unsigned short>(h16[j])));
            key[j] = ((h16[j] & 0x7fffu) << 7) | static_cast<uint32_t>(127 - (lane * 4 + j));
        }
        // sorter: abs-max, first index on ties
        const uint32_t best = __reduce_max_sync(full, max(max(key[0], key[1]), max(key[2], key[3])));
        const int pstar = 127 - static_cast<int>(best & 127u);
        const float xsel = (pstar & 3) == 0 ? x[0] : (pstar & 3) == 1 ? x[1] : (pstar & 3) == 2 ? x[2] : x[3];
        const float xp = __shfl_sync(full, xsel, pstar >> 2);
        const uint32_t qs = fp8(xp);
        const float scale = fabsf(fp8_to_float(qs) * T);
        float u[4], lo = INFINITY, hi = -INFINITY;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const bool is_max = lane * 4 + j == pstar;
            u[j] = (is_max || scale == 0.0f) ? 0.0f : __fdiv_rn(x[j], scale);
            if (!is_max) { lo = fminf(lo, u[j]); hi = fmaxf(hi, u[j]); }
        }
        // warp min / max through the order-preserving integer image of a float (the sign of a zero result is
        // irrelevant below: it only enters differences)
        auto ordered = [](float f) { const uint32_t b = __float_as_uint(f); return b ^ (static_cast<uint32_t>(static_cast<int32_t>(b) >> 31) | 0x80000000u); };
        auto unordered = [](uint32_t o) { return __uint_as_float(o ^ ((o >> 31) ? 0x80000000u : 0xffffffffu)); };
        lo = unordered(__reduce_min_sync(full, ordered(lo)));
        hi = unordered(__reduce_max_sync(full, ordered(hi)));
        // pattern selector: min/max fitness, two patterns per lane
        double score = INFINITY;
        int kp = lane;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int k = lane + 32 * r;
            if (k < S) {
                const double a = static_cast<double>(__half2float(__ushort_as_half(pat_s[k * 16]))) - static_cast<double>(lo);
                const double b = static_cast<double>(__half2float(__ushort_as_half(pat_s[k * 16 + 14]))) - static_cast<double>(hi);
                const double sc = __dadd_rn(__dmul_rn(a, a), __dmul_rn(b, b));
                if (sc < score) { score = sc; kp = k; }
            }
        }
        {   // arg-min over the lanes, ties to the lower id: a non-negative double orders like its bit pattern
            const uint64_t sb = static_cast<uint64_t>(__double_as_longlong(score));
            const uint32_t s_hi = static_cast<uint32_t>(sb >> 32), s_lo = static_cast<uint32_t>(sb);
            const uint32_t m_hi = __reduce_min_sync(full, s_hi);
            const uint32_t m_lo = __reduce_min_sync(full, s_hi == m_hi ? s_lo : 0xffffffffu);
            kp = static_cast<int>(__reduce_min_sync(full, (s_hi == m_hi && s_lo == m_lo) ? static_cast<uint32_t>(kp) : 0xffffffffu));
        }
        // value mappers: nearest centroid, ties to the lower index
        // The pattern is ascending, so the nearest centroid is one of the two that bracket the value
        // (exact fp32 comparisons find them); the fp64 squared distances of those two decide, as in the
        // definition, and equal centroids resolve to the lowest index.
        // A centroid is an fp16 number, so c <= u exactly when c <= u rounded down to fp16: the fifteen
        // comparisons are eight packed fp16 ones (entry 15 of the row is replaced by +inf).
        uint4 c_lo = reinterpret_cast<const uint4*>(pat_s)[kp * 2], c_hi = reinterpret_cast<const uint4*>(pat_s)[kp * 2 + 1];
        c_hi.w = (c_hi.w & 0xffffu) | 0x7c000000u;
        const uint32_t crow[8] = {c_lo.x, c_lo.y, c_lo.z, c_lo.w, c_hi.x, c_hi.y, c_hi.z, c_hi.w};
        uint32_t sym[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const __half2 uu = __half2half2(__float2half_rd(u[j]));
            __half2 cnt = __floats2half2_rn(0.0f, 0.0f);
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                __half2 c2;
                asm("mov.b32 %0, %1;" : "=r"(*reinterpret_cast<uint32_t*>(&c2)) : "r"(crow[m]));
                cnt = __hadd2(cnt, __hle2(c2, uu));
            }
            const int below = __half2int_rn(__hadd(__low2half(cnt), __high2half(cnt)));     // centroids <= u
            const int a = max(below - 1, 0), b = min(below, kCentroids - 1);
            const float ca = __half2float(__ushort_as_half(pat_s[kp * 16 + a])), cb = __half2float(__ushort_as_half(pat_s[kp * 16 + b]));
            const double da = static_cast<double>(u[j]) - static_cast<double>(ca), db = static_cast<double>(u[j]) - static_cast<double>(cb);
            int bi = __dmul_rn(db, db) < __dmul_rn(da, da) ? b : a;
            while (bi > 0 && pat_s[kp * 16 + bi - 1] == pat_s[kp * 16 + bi]) --bi;      // duplicates: first entry
            sym[j] = (lane * 4 + j == pstar) ? 15u : static_cast<uint32_t>(bi);
        }
        // four encoders: total length per codebook, the shortest wins (ties to the lower id)
        uint32_t t01 = 0, t23 = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint16_t* e = enc_s + (kp * kCodebooks) * kSymbols + sym[j];
            t01 += (e[0] >> 8) | (static_cast<uint32_t>(e[kSymbols] >> 8) << 16);
            t23 += (e[2 * kSymbols] >> 8) | (static_cast<uint32_t>(e[3 * kSymbols] >> 8) << 16);
        }
        t01 = __reduce_add_sync(full, t01);
        t23 = __reduce_add_sync(full, t23);
        const uint32_t tot[4] = {t01 & 0xffffu, t01 >> 16, t23 & 0xffffu, t23 >> 16};
        int hf = 0;
        uint32_t shortest = tot[0];
#pragma unroll
        for (int hh = 1; hh < 4; ++hh)
            if (tot[hh] < shortest) { shortest = tot[hh]; hf = hh; }
        // bit positions: header, ID_KP codeword, then a prefix sum over the 128 code lengths
        const uint32_t kpe = kp_s[kp];
        const uint32_t kp_len = kpe >> 12;
        uint32_t code[4], len[4], lane_bits = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t e = enc_s[(kp * kCodebooks + hf) * kSymbols + sym[j]];
            code[j] = e & 0xffu;
            len[j] = e >> 8;
            lane_bits += len[j];
        }
        uint32_t incl = lane_bits;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(full, incl, o);
            if (lane >= o) incl += v;
        }
        const uint32_t end_bit = kHeaderBits + kp_len + __shfl_sync(full, incl, 31);
        uint32_t pos = kHeaderBits + kp_len + incl - lane_bits;
        // pack / clip
        if (lane < 16) blk[lane] = 0;
        __syncwarp();
        if (lane == 0) atomicOr(&blk[0], qs | (static_cast<uint32_t>(hf) << 8) | ((kpe & 0xfffu) << kHeaderBits));
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (pos < static_cast<uint32_t>(kBlockBits)) {
                const uint32_t nbits = min(len[j], static_cast<uint32_t>(kBlockBits) - pos);   // truncated at bit 512
                const uint32_t v = code[j] & ((1u << nbits) - 1u);
                const uint32_t w = pos >> 5, off = pos & 31u;
                atomicOr(&blk[w], v << off);
                if (off + nbits > 32u) atomicOr(&blk[w + 1], v >> (32u - off));
            }
            pos += len[j];
        }
        if (end_bit <= static_cast<uint32_t>(kBlockBits)) {
            // outliers: the next-largest |x| (ties: lower index), as many 15-bit slots as fit, at most 16
            const int n_pad = min(kMaxPads, static_cast<int>((kBlockBits - end_bit) / kPadBits));
            // Every lane sorts its four keys (the abs-max itself left out); n_pad times the warp takes the largest
            // head and its owner advances.  A lane then knows which of its values are outliers and with which
            // slot numbers, and all lanes write their fields at once.
            uint32_t k0 = key[0] + 1u, k1 = key[1] + 1u, k2 = key[2] + 1u, k3 = key[3] + 1u;      // +1: zero means "nothing left"
            if ((pstar >> 2) == lane) {
                if ((pstar & 3) == 0) k0 = 0; else if ((pstar & 3) == 1) k1 = 0; else if ((pstar & 3) == 2) k2 = 0; else k3 = 0;
            }
            auto order = [](uint32_t& a, uint32_t& b) { const uint32_t hi_ = max(a, b), lo_ = min(a, b); a = hi_; b = lo_; };
            order(k0, k1); order(k2, k3); order(k0, k2); order(k1, k3); order(k1, k2);            // descending
            const uint32_t s0 = k0, s1 = k1, s2 = k2, s3 = k3;
            uint32_t slots = 0;                            // slot numbers of this lane's outliers, the latest in the low byte
            int mine = 0;
            for (int p = 0; p < n_pad; ++p) {
                const uint32_t top = __reduce_max_sync(full, k0);
                if (k0 == top) {                           // keys are distinct: exactly one lane
                    k0 = k1; k1 = k2; k2 = k3; k3 = 0;
                    slots = (slots << 8) | static_cast<uint32_t>(p);
                    ++mine;
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (i < mine) {
                    const int idx = 127 - static_cast<int>(((i == 0 ? s0 : i == 1 ? s1 : i == 2 ? s2 : s3) - 1u) & 127u);
                    const int p = static_cast<int>((slots >> (8 * (mine - 1 - i))) & 0xffu);
                    const int j = idx & 3;
                    const float xv = j == 0 ? x[0] : j == 1 ? x[1] : j == 2 ? x[2] : x[3];
                    const uint32_t field = static_cast<uint32_t>(idx) | (fp8(xv) << 7);
                    const uint32_t bp = kBlockBits - kPadBits * (p + 1), w = bp >> 5, off = bp & 31u;
                    atomicOr(&blk[w], field << off);
                    if (off + kPadBits > 32u) atomicOr(&blk[w + 1], field >> (32u - off));
                }
            }
        }
        __syncwarp();
        if (lane < 16) reinterpret_cast<uint32_t*>(d_blocks + g * kBlockBytes)[lane] = blk[lane];
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------------------------
// The same encoder for many groups: eight lanes per group, sixteen values per lane, four groups per warp, so that what is
// done once per group or once per reduction costs a quarter of the instructions.  Decisions are those of the kernel above;
// what makes them cheap:
//  * min / max of the normalised values = normalised min / max (division by the scale is monotone): packed fp16 extremes,
//    two divisions per group.
//  * the pattern with the least fp32 fitness wins unless another comes within 2^-20 of it; only then are the fp64 scores formed.
//  * nearest centroid = number of midpoints below the value.  A table per pattern holds for 256 cells of [-1, 1) how many
//    midpoints lie below the cell and, in the same word, the next one, so a value costs one lookup and one comparison; the value is x times
//    the scale's reciprocal, and where that comes within 2.4e-6 of a midpoint the exact division and fp64 distances decide.
//    (Count and midpoint in tables of their own: two calls of 131 072 groups 106.3 us, in one word 102.2.)
//  * the four codebooks' lengths are bytes of one word, summed together.
//  * a lane joins its sixteen codewords into one string of at most 128 bits in registers and ORs five words into the block.
// Bound by the issue slots (82 % busy, ncu): 304 warp instructions per group against 735 of the kernel above; two calls of
// 131 072 groups take 102 us against 213.6.  Making the tables costs a call 3 us, which is what the smaller instruction count
// saves at about 14 500 groups (two calls of 8192 24.4 against 17.8 us, of 12 288 26.4 / 24.3, of 14 336 27.6 / 27.7, of 16 383 28.9 / 29.6):
// fewer than 16 384, where it is 2 % faster, go to the kernel above.
// ---------------------------------------------------------------------------------------------
constexpr int kKvManyWarps = 32;
constexpr int kKvCells = 256;
constexpr float kCellWidth = 1.0f / 127.5f;
struct KvManySmem {
    // per cell the first midpoint not below it, as a float whose low five bits hold the number of those below; if the cell holds several,
    // that number | 16 and no midpoint: its values are decided exactly
    uint32_t cell[kMaxPatterns * kKvCells];
    uint16_t pat[kMaxPatterns * 16];
    uint16_t enc[kMaxPatterns * kCodebooks * kSymbols];    // length | codeword in stream order << 8
    uint16_t kp[kMaxPatterns];
    uint32_t len4[kMaxPatterns * kSymbols];                // code lengths of a symbol in the four codebooks, one per byte
    float mid[kMaxPatterns * 16];                          // midpoints of neighbouring centroids (14 per pattern), then infinity
    float2 ends[kMaxPatterns];                             // first and last centroid
    uint4 x[kKvManyWarps][64];                             // the warp's four groups, fp16 [4][128]
    uint32_t blk[kKvManyWarps][64];                        // their blocks
};

__device__ __forceinline__ uint32_t kv_key(uint32_t half, int pos) { return ((half & 0x7fffu) << 7) | static_cast<uint32_t>(127 - pos); }

__global__ void __launch_bounds__(kKvManyWarps * 32, 1)
ecco_kv_compress_many_kernel(const uint8_t* __restrict__ d_meta, const __half* __restrict__ d_x, uint64_t n_groups, uint8_t* __restrict__ d_blocks)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    KvManySmem& sm = *reinterpret_cast<KvManySmem*>(smem);
    const int tid = static_cast<int>(threadIdx.x), lane = tid & 31, warp = tid >> 5, sub = lane & 7, grp = lane >> 3;
    constexpr unsigned full = 0xffffffffu;
    release_dependents();
    const DevHeader* hdr = reinterpret_cast<const DevHeader*>(d_meta);
    const int S = min(max(__ldg(&hdr->S), 1), kMaxPatterns);
    const float T = __ldg(&hdr->T), invT = 1.0f / T;     // both exact powers of two
    // tables: from the image, which is host-written and may be read before the wait on the previous kernel
    for (int i = tid; i < static_cast<int>(kPatternBytes / 16); i += kKvManyWarps * 32) reinterpret_cast<uint4*>(sm.pat)[i] = __ldg(reinterpret_cast<const uint4*>(d_meta + kOffPattern) + i);
    for (int i = tid; i < static_cast<int>(kEncCbBytes / 16); i += kKvManyWarps * 32) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(d_meta + kOffEncCb) + i);   // bytes of every entry swapped
        reinterpret_cast<uint4*>(sm.enc)[i] = make_uint4(prmt(v.x, 0, 0x2301u), prmt(v.y, 0, 0x2301u), prmt(v.z, 0, 0x2301u), prmt(v.w, 0, 0x2301u));
    }
    for (int i = tid; i < static_cast<int>(kEncKpBytes / 16); i += kKvManyWarps * 32) reinterpret_cast<uint4*>(sm.kp)[i] = __ldg(reinterpret_cast<const uint4*>(d_meta + kOffEncKp) + i);
    __syncthreads();
    auto centroid = [&](int k, int j) { return __half2float(__ushort_as_half(sm.pat[k * 16 + j])); };
    for (int i = tid; i < kMaxPatterns * kSymbols; i += kKvManyWarps * 32) {
        const int k = i >> 4, s = i & 15;
        uint32_t v = 0;
#pragma unroll
        for (int h = 0; h < kCodebooks; ++h) v |= static_cast<uint32_t>(sm.enc[(k * kCodebooks + h) * kSymbols + s] & 0xffu) << (8 * h);
        // a centroid equal to the one before it never wins: its symbol stands for the first of them
        int f = s;
        while (f > 0 && f < kCentroids && centroid(k, f - 1) == centroid(k, f)) --f;
        if (f != s) {
            v = 0;
#pragma unroll
            for (int h = 0; h < kCodebooks; ++h) {
                const uint16_t e = sm.enc[(k * kCodebooks + h) * kSymbols + f];
                v |= static_cast<uint32_t>(e & 0xffu) << (8 * h);
                sm.enc[(k * kCodebooks + h) * kSymbols + s] = e;
            }
        }
        sm.len4[i] = v;
        sm.mid[i] = s < kCentroids - 1 ? 0.5f * (centroid(k, s) + centroid(k, s + 1)) : INFINITY;
        if (s == 0) sm.ends[k] = make_float2(centroid(k, 0), centroid(k, kCentroids - 1));
    }
    __syncthreads();
    // cell c holds the values with |127.5 (u + 1) - c| <= 1/2 and a little more on both sides (the edge cells all that is beyond);
    // a thread fills sixteen cells of a row, advancing through the ascending midpoints
    for (int i = tid; i < kMaxPatterns * kKvCells / 16; i += kKvManyWarps * 32) {
        const float* const m = sm.mid + (i / (kKvCells / 16)) * 16;
        int c = (i % (kKvCells / 16)) * 16, below = 0, upto = 0;
        uint32_t out[16];
#pragma unroll
        for (int q = 0; q < 16; ++q, ++c) {
            if (c > 0) while (below < kCentroids - 1 && m[below] < (static_cast<float>(c) - 0.51f) * kCellWidth - 1.0f) ++below;
            while (upto < kCentroids - 1 && (c == kKvCells - 1 || m[upto] <= (static_cast<float>(c) + 0.51f) * kCellWidth - 1.0f)) ++upto;
            // the nearest float that ends in those five bits: at most sixteen places off.  Infinity becomes a NaN, which nothing is above
            const uint32_t low = static_cast<uint32_t>(below);
            out[q] = upto - below > 1 ? low | 16u : ((__float_as_uint(m[below]) + 16u - low) & ~31u) | low;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) reinterpret_cast<uint4*>(sm.cell)[i * 4 + q] = make_uint4(out[4 * q], out[4 * q + 1], out[4 * q + 2], out[4 * q + 3]);
    }
    __syncthreads();
    dependency_wait();                                     // x and the blocks: after the previous kernel of the stream

    auto fp8 = [&](float v) { return static_cast<uint32_t>(__nv_cvt_float_to_fp8(v * invT, __NV_SATFINITE, __NV_E4M3)); };
    uint16_t* const xs = reinterpret_cast<uint16_t*>(sm.x[warp]) + grp * kGroup;          // this group's values
    uint32_t* const blk = sm.blk[warp] + grp * 16;
    const uint64_t n_units = (n_groups + 3) / 4;
    for (uint64_t unit = static_cast<uint64_t>(warp) * gridDim.x + blockIdx.x; unit < n_units; unit += static_cast<uint64_t>(gridDim.x) * kKvManyWarps) {
        const uint64_t g = min(unit * 4 + grp, n_groups - 1);            // past the end: the last group again, not stored
        uint32_t h[8];                                     // x is 16-byte aligned: two loads
        {
            const uint4* const src = reinterpret_cast<const uint4*>(d_x + g * kGroup + sub * 16);
            const uint4 a = __ldcg(src), b = __ldcg(src + 1);
            h[0] = a.x; h[1] = a.y; h[2] = a.z; h[3] = a.w; h[4] = b.x; h[5] = b.y; h[6] = b.z; h[7] = b.w;
        }
        uint4* const mine = reinterpret_cast<uint4*>(xs) + sub * 2;
        mine[0] = make_uint4(h[0], h[1], h[2], h[3]);
        mine[1] = make_uint4(h[4], h[5], h[6], h[7]);
        blk[sub * 2] = 0;
        blk[sub * 2 + 1] = 0;
        auto group_max = [&](uint32_t v) {
            v = max(v, __shfl_xor_sync(full, v, 1));
            v = max(v, __shfl_xor_sync(full, v, 2));
            return max(v, __shfl_xor_sync(full, v, 4));
        };
        // sorter: abs-max, first index on ties (key: |x|, then low index first)
        uint32_t best = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) best = max(best, max(kv_key(h[i], sub * 16 + 2 * i), kv_key(h[i] >> 16, sub * 16 + 2 * i + 1)));
        best = group_max(best);
        const int pstar = 127 - static_cast<int>(best & 127u);
        __syncwarp();
        const float xp = __half2float(__ushort_as_half(xs[pstar]));
        __syncwarp();
        if (sub == 0) xs[pstar] = 0x7e00u;                 // NaN: out of the extremes and, at the end, the largest key
        __syncwarp();
        {
            const uint4 a = mine[0], b = mine[1];
            h[0] = a.x; h[1] = a.y; h[2] = a.z; h[3] = a.w; h[4] = b.x; h[5] = b.y; h[6] = b.z; h[7] = b.w;
        }
        const uint32_t qs = fp8(xp);
        const float scale = fabsf(fp8_to_float(qs) * T);
        // extremes of the rest: (min, -max) in one packed number; a lane whose sixteen values are fine gives no NaN
        auto as_h2 = [](uint32_t v) { return *reinterpret_cast<const __half2*>(&v); };
        __half2 mn = as_h2(h[0]), mx = as_h2(h[0]);
#pragma unroll
        for (int i = 1; i < 8; ++i) { mn = __hmin2(mn, as_h2(h[i])); mx = __hmax2(mx, as_h2(h[i])); }
        __half2 ext = __halves2half2(__hmin(__low2half(mn), __high2half(mn)), __hneg(__hmax(__low2half(mx), __high2half(mx))));
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) ext = __hmin2(ext, __shfl_xor_sync(full, ext, o));
        const float lo = scale == 0.0f ? 0.0f : __fdiv_rn(__low2float(ext), scale), hi = scale == 0.0f ? 0.0f : __fdiv_rn(-__high2float(ext), scale);
        // pattern selector: min/max fitness, eight patterns per lane
        float low = INFINITY, sc[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int k = sub + 8 * r;
            const float2 e = sm.ends[k];
            const float a = e.x - lo, b = e.y - hi;
            sc[r] = k < S ? a * a + b * b : INFINITY;
            low = fminf(low, sc[r]);
        }
        low = fminf(low, __shfl_xor_sync(full, low, 1));
        low = fminf(low, __shfl_xor_sync(full, low, 2));
        low = fminf(low, __shfl_xor_sync(full, low, 4));
        uint32_t cand = 0;                                 // patterns of this lane that may be the best
        const float limit = fmaf(low, 1.00000095367431640625f, 1e-30f);      // 1 + 2^-20
#pragma unroll
        for (int r = 0; r < 8; ++r) cand |= (sc[r] <= limit && sub + 8 * r < S ? 1u : 0u) << r;
        int kp;
        {
            const uint32_t with = (__ballot_sync(full, cand != 0) >> (grp * 8)) & 0xffu;
            const bool clear = __popc(with) == 1 && (__popc(cand) <= 1);
            if (__all_sync(full, clear)) {
                kp = __shfl_sync(full, sub + 8 * (__ffs(cand) - 1), grp * 8 + __ffs(with) - 1);
            } else {                                       // fp64 scores of the candidates; a non-negative double orders like its bits
                uint64_t sb = ~0ull;
                uint32_t id = kMaxPatterns - 1;
                for (uint32_t c = cand; c; c &= c - 1u) {
                    const int k = sub + 8 * (__ffs(c) - 1);
                    const float2 e = sm.ends[k];
                    const double a = static_cast<double>(e.x) - static_cast<double>(lo), b = static_cast<double>(e.y) - static_cast<double>(hi);
                    const uint64_t v = static_cast<uint64_t>(__double_as_longlong(__dadd_rn(__dmul_rn(a, a), __dmul_rn(b, b))));
                    if (v < sb) { sb = v; id = static_cast<uint32_t>(k); }
                }
#pragma unroll
                for (int o = 1; o < 8; o <<= 1) {
                    const uint64_t v = __shfl_xor_sync(full, sb, o);
                    const uint32_t k = __shfl_xor_sync(full, id, o);
                    if (v < sb || (v == sb && k < id)) { sb = v; id = k; }
                }
                kp = static_cast<int>(id);
            }
        }
        // value mappers
        const float inv = scale == 0.0f ? 0.0f : __fdiv_rn(1.0f, scale);
        const uint32_t cells = smem_u32(sm.cell) + kp * (kKvCells * 4) - (0x4b400000u << 2), lens = smem_u32(sm.len4) + kp * 64;
        auto shared_word = [](uint32_t a) { uint32_t v; asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a)); return v; };
        auto cell_of = [&](float u) {                      // NaN: cell 0.  The sum's bits are those of 1.5 * 2^23 plus the cell's number
            return shared_word(__float_as_uint(fmaf(__saturatef(fmaf(u, 0.5f, 0.5f)), 255.0f, 12582912.0f)) * 4u + cells);
        };
        // more than x * (1 / scale) is off by for values up to 1.5 (2^-21) and a midpoint up to there by the bits in its last places (2^-19)
        constexpr float kBand = 2.4e-6f;
        uint32_t syms[2] = {0, 0}, l4 = 0, flags = 0;      // nibbles of values 0..7 and 8..15, the first one highest
        bool near = lo < -1.5f || hi > 1.5f;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const float u = (j & 1 ? __high2float(as_h2(h[j >> 1])) : __low2float(as_h2(h[j >> 1]))) * inv;
            const uint32_t e = cell_of(u);
            flags |= e;
            uint32_t s = e & 15u;
            const float d = u - __uint_as_float(e);        // without a midpoint in the cell this is the next one above: no step
            near = near || fabsf(d) <= kBand;
            if (d > 0.0f) ++s;
            syms[j >> 3] = syms[j >> 3] * 16u + s;
            l4 += shared_word(lens + s * 4);
        }
        if (warp_any(near || (flags & 16u))) {
            // the values in question as defined: exact quotient, fp64 distances, ties to the first centroid
            for (int j = 0; j < 16; ++j) {
                const float x = __half2float(__ushort_as_half(xs[sub * 16 + j]));
                const uint32_t e = cell_of(x * inv);
                if (!(fabsf(x) <= 65504.0f)) continue;     // the abs-max itself
                if (!(e & 16u) && fabsf(x * inv) <= 1.5f && !(fabsf(x * inv - __uint_as_float(e)) <= kBand)) continue;
                const float u = scale == 0.0f ? 0.0f : __fdiv_rn(x, scale);
                int below = 0;
                for (int i = 0; i < kCentroids; ++i) below += centroid(kp, i) <= u;
                const int a = max(below - 1, 0), b = min(below, kCentroids - 1);
                const double da = static_cast<double>(u) - static_cast<double>(centroid(kp, a)), db = static_cast<double>(u) - static_cast<double>(centroid(kp, b));
                const uint32_t s = static_cast<uint32_t>(__dmul_rn(db, db) < __dmul_rn(da, da) ? b : a), sh = 28u - 4u * (j & 7);
                uint32_t& w = j < 8 ? syms[0] : syms[1];
                l4 += sm.len4[kp * 16 + s] - sm.len4[kp * 16 + ((w >> sh) & 15u)];
                w = (w & ~(15u << sh)) | (s << sh);
            }
        }
        if ((pstar >> 4) == sub) {                         // the NaN has counted as symbol 0
            l4 += sm.len4[kp * 16 + 15] - sm.len4[kp * 16];
            const uint32_t w = 15u << (28u - 4u * (pstar & 7));
            if (pstar & 8) syms[1] |= w; else syms[0] |= w;
        }
        // four encoders: total length per codebook, the shortest wins (ties to the lower id)
        uint32_t t02 = l4 & 0x00ff00ffu, t13 = (l4 >> 8) & 0x00ff00ffu;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) { t02 += __shfl_xor_sync(full, t02, o); t13 += __shfl_xor_sync(full, t13, o); }
        const uint32_t tot[4] = {t02 & 0xffffu, t13 & 0xffffu, t02 >> 16, t13 >> 16};
        int hf = 0;
        uint32_t shortest = tot[0];
#pragma unroll
        for (int hh = 1; hh < 4; ++hh)
            if (tot[hh] < shortest) { shortest = tot[hh]; hf = hh; }
        // the lane's sixteen codewords as one bit string
        const uint16_t* const enc = sm.enc + (kp * kCodebooks + hf) * kSymbols;
        uint64_t half_bits[2];
        uint32_t half_len[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            uint32_t bits4[2], len4[2];
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                uint32_t e[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) e[j] = enc[(syms[q] >> (28 - 4 * (p * 4 + j))) & 15u];
                // an entry's low five bits are its length: it is the shift of what follows
                const uint32_t b01 = (e[0] >> 8) | __funnelshift_l(0u, e[1] >> 8, e[0]), b23 = (e[2] >> 8) | __funnelshift_l(0u, e[3] >> 8, e[2]);
                const uint32_t l01 = (e[0] + e[1]) & 0xffu;
                bits4[p] = b01 | __funnelshift_l(0u, b23, l01);
                len4[p] = l01 + ((e[2] + e[3]) & 0xffu);
            }
            half_bits[q] = static_cast<uint64_t>(bits4[0]) | (static_cast<uint64_t>(bits4[1]) << len4[0]);
            half_len[q] = len4[0] + len4[1];
        }
        // at most 64 bits each: the second string begins at half_len[0]
        uint64_t s0 = half_bits[0], s1 = 0;
        if (half_len[0] < 64) { s0 |= half_bits[1] << half_len[0]; s1 = half_len[0] ? half_bits[1] >> (64 - half_len[0]) : 0; }
        else s1 = half_bits[1];
        const uint32_t lane_bits = half_len[0] + half_len[1];
        uint32_t incl = lane_bits;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            const uint32_t v = __shfl_up_sync(full, incl, o, 8);
            if (sub >= o) incl += v;
        }
        const uint32_t kpe = sm.kp[kp], kp_len = kpe >> 12;
        const uint32_t end_bit = kHeaderBits + kp_len + shortest;
        const uint32_t pos = kHeaderBits + kp_len + incl - lane_bits, off = pos & 31u, w0 = pos >> 5;
        // pack / clip: what lies past bit 512 is dropped, so the first codeword that crosses it is truncated
        if (sub == 0) atomicOr(&blk[0], qs | (static_cast<uint32_t>(hf) << 8) | ((kpe & 0xfffu) << kHeaderBits));
        {
            const uint32_t q[4] = {static_cast<uint32_t>(s0), static_cast<uint32_t>(s0 >> 32), static_cast<uint32_t>(s1), static_cast<uint32_t>(s1 >> 32)};
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                const uint32_t v = __funnelshift_l(i ? q[i - 1] : 0u, i < 4 ? q[i] : 0u, off);
                if (w0 + i < 16u) atomicOr(&blk[w0 + i], v);
            }
        }
        // outliers: the next-largest |x| (ties: lower index), as many 15-bit slots as fit, at most 16
        const int n_pad = end_bit <= static_cast<uint32_t>(kBlockBits) ? min(kMaxPads, static_cast<int>((kBlockBits - end_bit) / kPadBits)) : 0;
        const int n_max = __reduce_max_sync(full, n_pad);
        if (n_max > 0) {
            uint32_t key[16];
#pragma unroll
            for (int i = 0; i < 8; ++i) { key[2 * i] = kv_key(h[i], sub * 16 + 2 * i); key[2 * i + 1] = kv_key(h[i] >> 16, sub * 16 + 2 * i + 1); }
            // keys are distinct and below 2^23: seen from `top` (mod 2^32) the largest smaller key is the largest number
            uint32_t top = kv_key(0x7e00u, pstar);         // the abs-max itself (its NaN) is out
            for (int p = 0; p < n_max; ++p) {
                uint32_t next = 0;
#pragma unroll
                for (int i = 0; i < 16; ++i) next = __viaddmax_u32(key[i], 0u - top, next);
                top += group_max(next);
                if (p < n_pad && sub == 0) {
                    const uint32_t loc = 127u - (top & 127u);
                    const uint32_t field = loc | (fp8(__half2float(__ushort_as_half(xs[loc]))) << 7);
                    const uint32_t bp = kBlockBits - kPadBits * (p + 1), w = bp >> 5, o = bp & 31u;
                    atomicOr(&blk[w], field << o);
                    if (o + kPadBits > 32u) atomicOr(&blk[w + 1], field >> (32u - o));
                }
            }
        }
        __syncwarp();
        if (unit * 4 + grp < n_groups) reinterpret_cast<uint2*>(d_blocks + g * kBlockBytes)[sub] = make_uint2(blk[sub * 2], blk[sub * 2 + 1]);
        __syncwarp();
    }
}

}  // namespace
