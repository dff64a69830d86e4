// ecco_act2x_kernels.cuh -- 2x activation codec kernels
// Part of the one translation unit ecco_kernels.cu; included from there only.
#pragma once

// ---------------------------------------------------------------------------------------------
// 2x activation format (Sec. 3.2 "Activation Compression"; Sec. 4.2 / 4.3 low-ratio units):
// 64 fp16 values <-> 64 bytes.  Byte i = 7-bit two's-complement value in bits 0..6 and one bit
// of metadata in bit 7: metadata bits 0..15 = fp16 scale, 16..31 = fp16 zero point, 32..63 = 0.
// Four lanes share a group (16 bytes / 16 values each), so a warp moves 512 B of blocks and
// 1 KB of fp16 per instruction, fully coalesced; both kernels are plain HBM streams.
// ---------------------------------------------------------------------------------------------
namespace {

// bit 7 of the four bytes of w, gathered into bits 0..3
__device__ __forceinline__ uint32_t top_bits(uint32_t w) { return ((w & 0x80808080u) * 0x00204081u) >> 28; }

// Both kernels are bound by HBM at large sizes.  A CTA takes one turn, and there are as many as the call needs: the scheduler starts one as
// soon as another is done, whatever number of them an SM has room for.  Eight CTAs per SM with equal numbers of turns did not all
// find room (40 or 64 registers) and left their last wave half empty.  Times are of calls one after the other in a graph: compressing 227 328
// groups 10.2 -> 9.1 us, 700 000 27.7 -> 23.2, decompressing 1 000 003 36.5 -> 29.5, there and back 1 000 003 66.5 -> 60.8.
// No conversion instruction between integers and floats is used (they issue at a quarter of the rate): a byte becomes a float by its place
// below the exponent of 2^23, and a float is rounded to an integer by adding 1.5 * 2^23.  262 144 groups there and back, the
// second kernel becoming resident while the first drains: 16.6 us (100 MB: 6.1 TB/s).
constexpr int kActThreads = 256;

__global__ void __launch_bounds__(kActThreads)
ecco_act_decompress_kernel(const uint4* __restrict__ d_blocks, uint64_t n_chunks, uint4* __restrict__ d_out)
{
    // one chunk = 16 bytes of a block = 16 values; chunk c belongs to group c / 4
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t c = static_cast<uint64_t>(blockIdx.x) * kActThreads + threadIdx.x;
    const bool mine = c < n_chunks;
    const uint4* const from = d_blocks + c;                // formed before the wait: 20 000 groups 2.1 -> 1.85 us
    release_dependents();
    dependency_wait();                                     // the blocks may come from the previous kernel of the stream
    uint4 b = make_uint4(0, 0, 0, 0);
    if (mine) asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w) : "l"(from));
    const uint32_t bits16 = top_bits(b.x) | (top_bits(b.y) << 4) | (top_bits(b.z) << 8) | (top_bits(b.w) << 12);
    const uint32_t scale_bits = __shfl_sync(0xffffffffu, bits16, lane & ~3u);          // chunk 0 of the group
    const uint32_t zero_bits = __shfl_sync(0xffffffffu, bits16, (lane & ~3u) | 1u);    // chunk 1
    const float scale = __half2float(__ushort_as_half(static_cast<unsigned short>(scale_bits)));
    const float zero = __half2float(__ushort_as_half(static_cast<unsigned short>(zero_bits)));
    const uint32_t w[4] = {b.x, b.y, b.z, b.w};
    uint32_t o[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t q = (w[i] ^ 0x40404040u) & 0x7f7f7f7fu;                         // 7-bit two's complement + 64
        float v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            v[j] = fmaf(__uint_as_float(prmt(q, 0x4b000000u, 0x7540u + j)) - (8388608.0f + 64.0f), scale, zero);
        o[2 * i] = f2h_bits(v[0]) | (f2h_bits(v[1]) << 16);
        o[2 * i + 1] = f2h_bits(v[2]) | (f2h_bits(v[3]) << 16);
    }
    if (mine) stg_v8(d_out + c * 2, o);
}

// kLoads chunks per thread, their loads in flight before any is used: see act_compress_loads
template <int kLoads>
__global__ void __launch_bounds__(kActThreads)
ecco_act_compress_kernel(const uint4* __restrict__ d_x, uint64_t n_chunks, uint4* __restrict__ d_blocks)
{
    const uint64_t base = static_cast<uint64_t>(blockIdx.x) * (kLoads * kActThreads);
    // of a single chunk bound and address are formed before the wait (20 000 groups 2.75 -> 2.4 us); of two that is slower (262 144: 10.3 -> 11.1)
    const bool mine = base + threadIdx.x < n_chunks;
    const uint4* const from = d_x + (base + threadIdx.x) * 2;
    release_dependents();
    dependency_wait();                                     // x may come from the previous kernel of the stream
    uint32_t in[kLoads][8];
#pragma unroll
    for (int k = 0; k < kLoads; ++k) {
        const uint64_t c = base + k * kActThreads + threadIdx.x;
#pragma unroll
        for (int i = 0; i < 8; ++i) in[k][i] = 0;
        if (kLoads == 1 ? mine : c < n_chunks)
            asm volatile("ld.global.L1::no_allocate.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                         : "=r"(in[k][0]), "=r"(in[k][1]), "=r"(in[k][2]), "=r"(in[k][3]), "=r"(in[k][4]), "=r"(in[k][5]), "=r"(in[k][6]), "=r"(in[k][7])
                         : "l"(kLoads == 1 ? from : d_x + c * 2));
    }
#pragma unroll
    for (int k = 0; k < kLoads; ++k) {
        const uint64_t c = base + k * kActThreads + threadIdx.x;
        const __half2* h = reinterpret_cast<const __half2*>(in[k]);
        // min / max over the four lanes of the group (the compressor's sorter stage, Sec. 4.3), as (min, -max) in one number
        __half2 mn = h[0], mx = h[0];
#pragma unroll
        for (int i = 1; i < 8; ++i) { mn = __hmin2(mn, h[i]); mx = __hmax2(mx, h[i]); }
        __half2 ext = __halves2half2(__hmin(__low2half(mn), __high2half(mn)), __hneg(__hmax(__low2half(mx), __high2half(mx))));
        ext = __hmin2(ext, __shfl_xor_sync(0xffffffffu, ext, 1));
        ext = __hmin2(ext, __shfl_xor_sync(0xffffffffu, ext, 2));
        const float lo = __low2float(ext), hi = -__high2float(ext);
        const uint32_t scale16 = f2h_bits(__fdiv_rn(hi - lo, 127.0f));
        const float scale = __half2float(__ushort_as_half(static_cast<unsigned short>(scale16)));
        const uint32_t zero16 = f2h_bits(fmaf(64.0f, scale, lo));      // 64 * scale is exact, so this is lo + 64 * scale rounded once
        const float zero = __half2float(__ushort_as_half(static_cast<unsigned short>(zero16)));
        const bool usable = scale > 0.0f && scale < __int_as_float(0x7f800000);
        const float inv = __fdiv_rn(1.0f, scale);      // multiply-and-round (Sec. 4.3): one division per group
        const uint32_t part = (threadIdx.x & 3u);
        const uint32_t meta16 = part == 0 ? scale16 : part == 1 ? zero16 : 0u;   // this chunk's 16 metadata bits
        uint32_t out[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            // clamping before the rounding gives what clamping after it gives (the bounds are integers, rounding is
            // monotone); the sum with 1.5 * 2^23 is rounded to nearest even and holds the integer in its low byte
            uint32_t q[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float x = j & 1 ? __high2float(h[2 * i + (j >> 1)]) : __low2float(h[2 * i + (j >> 1)]);
                const float p = fminf(fmaxf(__fmul_rn(x - zero, inv), -64.0f), 63.0f);
                q[j] = __float_as_uint(p + 12582912.0f);
            }
            const uint32_t w = prmt(prmt(q[0], q[1], 0x0040u), prmt(q[2], q[3], 0x0040u), 0x5410u);
            // bits 4i .. 4i+3 of the metadata go to bit 7 of bytes 0..3
            const uint32_t m4 = (meta16 >> (4 * i)) & 15u;
            out[i] = (usable ? w & 0x7f7f7f7fu : 0u) | (((m4 * 0x00204081u) & 0x01010101u) << 7);
        }
        if (c < n_chunks) d_blocks[c] = make_uint4(out[0], out[1], out[2], out[3]);
    }
}

// CTAs for n_chunks chunks, `loads` of them to a thread
inline unsigned act_ctas(uint64_t n_chunks, int loads) { return static_cast<unsigned>((n_chunks + loads * kActThreads - 1) / (loads * kActThreads)); }

// Chunks per thread of the compressor: one as long as an SM holds all its CTAs at a time (eight of 256 threads and 32 registers), beyond that
// two.  One against two, us: 8192 groups 1.5 / 1.9, 37 888 2.3 / 2.6, 75 776 (the line on 148 SMs) 3.4 / 3.4, 94 720 4.3 / 4.0,
// 227 328 9.7 / 9.1, 700 000 25.4 / 23.2, 2 000 000 73.5 / 66.4.  Four are slower than two up to 1 000 000 groups and within the noise above.  A
// thread of the decompressor takes one: one against two 3.0 / 3.8 us for 85 000 groups, 6.9 / 7.3 for 196 608, 29.7 / 30.3 for 1 000 003.
inline int act_compress_loads(uint64_t n_chunks, const DeviceInfo& di) { return n_chunks <= static_cast<uint64_t>(di.sms) * 8 * kActThreads ? 1 : 2; }

}  // namespace
