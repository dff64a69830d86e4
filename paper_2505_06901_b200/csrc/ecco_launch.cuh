// ecco_launch.cuh -- host-side launch helpers: device query, overlapped launches, work plans
// Part of the one translation unit ecco_kernels.cu; included from there only.
#pragma once

namespace {

// ---------------------------------------------------------------------------------------------
// host-side launch helpers
// ---------------------------------------------------------------------------------------------
struct DeviceInfo {
    int device = -1, sms = 0, cc_major = 0;
    bool ok = false;
};

int device_info(DeviceInfo* out)
{
    static thread_local DeviceInfo cache[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) { t_last_cuda_error = static_cast<int>(e); return ECCO_ERR_CUDA; }
    if (dev < 0 || dev >= 64) return ECCO_ERR_INVALID_ARG;
    DeviceInfo& c = cache[dev];
    if (!c.ok) {
        cudaDeviceProp prop;
        e = cudaGetDeviceProperties(&prop, dev);
        if (e != cudaSuccess) { t_last_cuda_error = static_cast<int>(e); return ECCO_ERR_CUDA; }
        c.device = dev; c.sms = prop.multiProcessorCount; c.cc_major = prop.major; c.ok = true;
    }
    *out = c;
    return c.cc_major == 10 ? ECCO_OK : ECCO_ERR_UNSUPPORTED_ARCH;
}

int check_launch();
// Launch with the programmatic stream-serialisation attribute (see dependency_wait in the kernels):
// the kernel must call dependency_wait() before its first access to global memory.
template <class... Params, class... Args>
int launch_overlapped(void (*kernel)(Params...), unsigned grid, unsigned block, size_t smem, cudaStream_t stream, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
    if (e != cudaSuccess) { t_last_cuda_error = static_cast<int>(e); return ECCO_ERR_CUDA; }
    return check_launch();
}

// the tag of a call's ticket words (see take_ticket): 48 bits, never zero, another one for every call of the process
inline Ticket next_ticket_tag() noexcept
{
    static std::atomic<uint64_t> next{[] {
        // without exceptions: none may leave a C entry (std::random_device throws where it finds no source)
        uint64_t start = 0;
        if (getrandom(&start, sizeof start, GRND_NONBLOCK) != static_cast<ssize_t>(sizeof start))
            start = static_cast<uint64_t>(std::chrono::steady_clock::now().time_since_epoch().count()) * 0x9e3779b97f4a7c15ull ^ reinterpret_cast<uintptr_t>(&start);
        return start;
    }()};
    for (;;) {
        const Ticket tag = next.fetch_add(1, std::memory_order_relaxed) & ((1ull << 48) - 1);
        if (tag) return tag;
    }
}

template <class K>
int set_smem(K kernel, size_t bytes)
{
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
    if (e != cudaSuccess) { t_last_cuda_error = static_cast<int>(e); return ECCO_ERR_CUDA; }
    return ECCO_OK;
}

int check_launch()
{
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { t_last_cuda_error = static_cast<int>(e); return ECCO_ERR_CUDA; }
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return ECCO_OK;
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Warps per CTA the decoding kernels are launched with (their register budget); how many of them work is decided on
// the device, from the size of the image's tables.
constexpr int kDecompressWarps = 28;
constexpr int fused_warps(int v) { return v == 1 ? 32 : 28; }
constexpr int gemv_warp_warps(int v) { return v == 1 ? 32 : v <= 3 ? 28 : v == 4 ? 26 : 22; }

// CTAs for `units` warp-sized pieces of work: one per SM as soon as there are that many.  The kernels number their warps
// across the CTAs first, so a call with fewer pieces than the machine has warp slots puts a few on every SM instead of
// filling some SMs and leaving the others idle (decode attention over 2 x 8 x 777 tokens, 400 pieces: 37.6 -> 30.4 us).  The price is paid by
// small calls on several streams at once, which find no SM free: eight such calls side by side 20.4 us each, 6.5 with SMs filled first.
inline int spread_ctas(int64_t units, int ctas_max) { return static_cast<int>(units < ctas_max ? units : ctas_max); }

// Threads of such a CTA: a warp per piece it can get, but no more than the kernel is made for, and at least eight (they share the
// work of laying out the tables).  Warps without work are not free: they take part in every barrier of the set-up.
inline unsigned spread_threads(int64_t units, int grid, int max_warps)
{
    const int64_t per_cta = (units + grid - 1) / grid;
    const int64_t warps = per_cta < 8 ? 8 : per_cta < max_warps ? per_cta : max_warps;
    return static_cast<unsigned>((warps < max_warps ? warps : max_warps) * 32);
}

struct GemvPlan { int row_tiles, grid; size_t partial_bytes, ticket_bytes; };

// plan of a fused GEMV call over `units` units in `row_tiles` 32-row tiles (all matrices of the call together):
// persistent CTAs of `warps` warps, one slot of cols x 32 partial sums per (warp, tile) step of the staircase, one
// ticket per tile
inline GemvPlan gemv_plan(int64_t units, int row_tiles, int warps, int cols, int ctas_max)
{
    GemvPlan p;
    p.row_tiles = row_tiles;
    p.grid = spread_ctas(units, ctas_max);
    const int64_t workers = static_cast<int64_t>(p.grid) * warps < units ? static_cast<int64_t>(p.grid) * warps : units;
    p.partial_bytes = (static_cast<size_t>(workers + row_tiles) * cols * 32 * sizeof(float) + 255) & ~static_cast<size_t>(255);
    p.ticket_bytes = (static_cast<size_t>(row_tiles) * kTicketStride * sizeof(Ticket) + 255) & ~static_cast<size_t>(255);
    return p;
}

constexpr int kMmaWarps = 20;      // all find room beside the tables of an image of up to 66 code shapes (9.4 KB of shared memory per warp)

// the per-warp kernel (one to five rows of x: vpad columns) or the tensor-core kernel (6..8 rows: eight columns)
// Per-warp against tensor-core kernel, two 11008 x 4096 matrices in a call: 67 against 81 us at three rows, 81 against 81 at five,
// 85 against 81 at six, 104 against 81 at eight; 1000 x 4096: 14.2 against 18.1 at five, 15.3 against 17.9 at six.
inline GemvPlan gemv_plan_for(int64_t units, int row_tiles, int vpad, int ctas_max)
{
    return vpad <= 5 ? gemv_plan(units, row_tiles, gemv_warp_warps(vpad), vpad, ctas_max) : gemv_plan(units, row_tiles, kMmaWarps, 8, ctas_max);
}

inline int pad_v(int v) { return v <= 5 ? v : 8; }


}  // namespace
