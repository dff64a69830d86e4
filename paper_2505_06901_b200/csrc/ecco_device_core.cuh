// ecco_device_core.cuh -- PTX helpers, bounded waits, overlapped launches
// Part of the one translation unit ecco_kernels.cu; included from there only.
#pragma once

#include <cuda.h>
#include <cuda/std/type_traits>
#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>

#include <sys/random.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <climits>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <mutex>

#include "../../include/ecco.h"
#include "ecco_format.h"

using namespace ecco;

namespace {


__device__ int g_device_status = 0;            // sticky: ECCO_ERR_DEVICE_TIMEOUT if a bounded wait expired
thread_local int t_last_cuda_error = 0;
std::atomic<uint64_t> g_launches{0};

constexpr uint32_t kSmemCtaBytes = 232448;                           // 227 KB: what every decoding kernel asks for
constexpr int kWaitLimit = 1 << 22;                                  // bounded mbarrier polling

// Quotient of numbers that are rarely beyond 32 bits: a 64-bit division takes some hundred instructions, one after the other
// (eight of them stood at the end of every split sum: see UnitSplit).
__host__ __device__ __forceinline__ uint64_t divide(uint64_t a, uint64_t b)
{
    return (a | b) >> 32 ? a / b : static_cast<uint32_t>(a) / static_cast<uint32_t>(b);
}

// ---------------------------------------------------------------------------------------------
// small PTX helpers
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// 1-D bulk copy global -> shared (TMA engine, no tensor map, no multicast); both addresses and
// the size are multiples of 16 bytes
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}
__device__ __forceinline__ uint32_t lds_u8(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint32_t lds_u16(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts_u16(uint32_t addr, uint32_t v) { asm volatile("st.shared.u16 [%0], %1;" ::"r"(addr), "h"(static_cast<unsigned short>(v)) : "memory"); }
__device__ __forceinline__ uint32_t lds_u32(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts_u32(uint32_t addr, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
// one 64-byte block = two 32-byte loads per lane: every load instruction asks for whole sectors.  Plain (coherent)
// loads that bypass L1: under the overlapped launches the blocks may have been written by the previous kernel of the
// stream (the online compressor), and the non-coherent path is only for data that nobody writes while a kernel lives.
struct Block { uint32_t w[16]; };
__device__ __forceinline__ void ldg_block(Block& b, const uint8_t* p)
{
    asm volatile("ld.global.L1::no_allocate.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(b.w[0]), "=r"(b.w[1]), "=r"(b.w[2]), "=r"(b.w[3]), "=r"(b.w[4]), "=r"(b.w[5]), "=r"(b.w[6]), "=r"(b.w[7])
                 : "l"(p));
    asm volatile("ld.global.L1::no_allocate.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(b.w[8]), "=r"(b.w[9]), "=r"(b.w[10]), "=r"(b.w[11]), "=r"(b.w[12]), "=r"(b.w[13]), "=r"(b.w[14]), "=r"(b.w[15])
                 : "l"(p + 32));
}
__device__ __forceinline__ void prefetch_block_l2(const uint8_t* p)
{
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p + 32));
}
__device__ __forceinline__ void stg_v8(void* p, const uint32_t (&r)[8])
{
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]),
                 "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}

__device__ __forceinline__ void sts_v2(uint32_t addr, uint32_t a, uint32_t b)
{
    asm volatile("st.shared.v2.u32 [%0], {%1,%2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ void sts_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
// 2-D tiled bulk store shared -> global through a tensor map (TMA); rows outside the tensor are dropped
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int x, int y)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(map), "r"(src), "r"(x),
                 "r"(y)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read0() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// OCP E4M3 byte -> fp32, exactly (the all-ones exponent/mantissa code reads as 480): exponent and mantissa lie as in an fp32 number
// whose exponent is 120 too small; the subnormals come out right because fp32 has subnormals, too
__device__ __forceinline__ float fp8_to_float(uint32_t b)
{
    const float mag = __uint_as_float((b & 0x7fu) << 20) * 1.329227995784916e36f;        // 2^120
    return __uint_as_float(__float_as_uint(mag) | ((b & 0x80u) << 24));
}
__device__ __forceinline__ uint32_t f2h_bits(float f) { return static_cast<uint32_t>(__half_as_ushort(__float2half_rn(f))); }

// Bounded wait of the whole CTA on a barrier word: at most 2 * limit polls per thread (the second round is a last
// chance for a copy in flight), then the CTA gives up together, records ECCO_ERR_DEVICE_TIMEOUT and returns false.
__device__ __forceinline__ bool bounded_wait(uint32_t bar, uint32_t parity, int limit)
{
    __syncthreads();                             // the barrier word is initialised
    bool done = false;
    for (int i = 0; i < limit && !done; ++i) done = mbar_try_wait(bar, parity);
    if (!done)
        for (int i = 0; i < limit && !done; ++i) done = mbar_try_wait(bar, parity);
    const bool all = __syncthreads_and(done);
    if (!all && threadIdx.x == 0) atomicExch(&g_device_status, ECCO_ERR_DEVICE_TIMEOUT);
    return all;
}
// Programmatic dependent launch: a kernel launched with the stream-serialisation attribute may become resident
// while the previous kernel in the stream is still draining.  dependency_wait() returns once that kernel has
// completed and its writes are visible (at once if there is no such overlap); every kernel executes it before
// its first access to global memory other than the metadata image (a prefetch into L2, where every write arrives, is no
// access), so stream order is what it is without the
// attribute and only launch, table fetch and prologue overlap.  The image is the exception because no kernel writes
// it: it reaches the device by a copy, which is a stream operation of its own (a kernel behind a copy starts after
// it), and a kernel can start early only behind one that releases its dependents, i.e. one of this file.
// A grid that ends without having waited breaks the chain: the kernel behind it waits for this grid only and could start on data that
// the one before it is still writing.  So a way out that every CTA may take leads through dependency_wait(), too.
// release_dependents() lets the next kernel of the stream do the same with respect to this one.
__device__ __forceinline__ void dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void release_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

}  // namespace
