// ecco_kernels.cu -- sm_100a kernels and the device half of the C ABI.
//
// One thread owns one group: a 64-byte block is independent of every other block (Sec. 3.2,
// "all group-wise information ... compressed to a fixed compressed block size"), so the decoder
// runs the serial Huffman chain (Sec. 4.2) once per thread and takes its parallelism across
// groups, not inside a group.  The lanes of a warp advance symbol by symbol in lock step, which
// keeps every per-symbol index (output position, activation element) uniform across the warp.
//
// Shared memory per CTA (sizes from the image's header, see ecco_decode_core.cuh):
//   tables   pattern[64][16] fp16 | codebook records [256] x 16 B | pair tables | centroids in rank order [256][16] fp16 | shape tables
//            [n_shapes][256] u8, and behind the warps' arrays, at the end of shared memory, ID_KP table [4096] u16; all but the centroids
//            are brought in by bulk copies (cp.async.bulk + mbarrier)
//   per warp bits[19][32] u32   the warp's 32 blocks, word-transposed: lane L's word w at
//                               [w][L] -> bank L whatever w is (conflict-free refills);
//                               rows 16 to 18 are scratch: what a lane reads past stream bit 512 does not matter (decode_group).  The
//                               scalar fused kernels keep the decoded ranks over its consumed rows, for the outlier fix-up
//            tiles              ecco_decompress: one [32 groups][16 values] fp16 staging tile for the tensor stores;
//                               tensor-core kernels: eight of them, the whole decoded group, as MMA operands
//
// Layout of the sources (one translation unit; the .cuh files are included here and nowhere else):
//   ecco_device_core.cuh            PTX helpers, bounded waits, overlapped launches
//   ecco_decode_core.cuh            the group decoder with the value table in registers
//   ecco_decompress_kernels.cuh     ecco_decompress (tile-store and small-tensor kernels), ecco_var_decompress
//   ecco_fused_scalar_kernels.cuh   fused GEMV (one to five rows) / attention scores (one or two heads)
//   ecco_group_tiles.cuh            decoded groups as fp16 tiles in shared memory
//   ecco_fused_mma_kernels.cuh      the same for more rows and heads, on the tensor cores
//   ecco_attn_values_kernels.cuh    softmax(scores) . V over a compressed V cache
//   ecco_act2x_kernels.cuh          2x activation codec
//   ecco_kv_compress_kernel.cuh     online 4x compressor
//   ecco_launch.cuh                 device query, overlapped launches, work plans
//   this file                       the C ABI: argument checks and launches
#include "ecco_device_core.cuh"
#include "ecco_decode_core.cuh"
#include "ecco_decompress_kernels.cuh"
#include "ecco_fused_scalar_kernels.cuh"
#include "ecco_group_tiles.cuh"
#include "ecco_attn_values_kernels.cuh"
#include "ecco_fused_mma_kernels.cuh"
#include "ecco_launch.cuh"
#include "ecco_act2x_kernels.cuh"
#include "ecco_kv_compress_kernel.cuh"


// ---------------------------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------------------------
extern "C" int ecco_last_cuda_error(void) { return t_last_cuda_error; }
extern "C" uint64_t ecco_kernel_launch_count(void) { return g_launches.load(); }

extern "C" int ecco_device_status(void)
{
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) { t_last_cuda_error = static_cast<int>(e); return ECCO_ERR_CUDA; }
    int st = 0, zero = 0;
    e = cudaMemcpyFromSymbol(&st, g_device_status, sizeof st);
    if (e == cudaSuccess && st) e = cudaMemcpyToSymbol(g_device_status, &zero, sizeof zero);
    if (e != cudaSuccess) { t_last_cuda_error = static_cast<int>(e); return ECCO_ERR_CUDA; }
    return st;
}

// Diagnostics: the give-up path of the bounded wait, exercised without anything that could hang.  The kernel arms a
// barrier with a byte count that no copy will ever deliver (nothing is in flight, so the CTA may exit at any time),
// polls it a few hundred times, gives up, records the time-out and returns normally.
namespace {
__global__ void ecco_wait_timeout_probe_kernel()
{
    __shared__ __align__(8) uint64_t bar;
    const uint32_t b = smem_u32(&bar);
    if (threadIdx.x == 0) {
        mbar_init(b, 1);
        mbar_expect_tx(b, 64);
    }
    (void)bounded_wait(b, 0, 256);
}
}  // namespace
extern "C" int ecco_test_wait_timeout(void* stream)
{
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc) return rc;
    ecco_wait_timeout_probe_kernel<<<1, 64, 0, static_cast<cudaStream_t>(stream)>>>();
    return check_launch();
}

// cuTensorMapEncodeTiled through the runtime's driver entry point query (no link against libcuda)
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_tiled_fn()
{
    static std::once_flag once;
    static EncodeTiledFn fn = nullptr;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

// tensor map of the output seen as [n_groups][128] fp16, box = 32 rows x 16 values, 32-byte swizzle
static bool make_out_map(CUtensorMap* map, void* d_out, uint64_t n_groups)
{
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {kGroup, n_groups};
    const cuuint64_t strides[1] = {kGroup * 2};
    const cuuint32_t box[2] = {16, 32};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, d_out, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

constexpr int kDecompressTmaWarps = 32;

// every decoding kernel asks for all the shared memory of an SM and lays itself out on the device
template <class K>
static int want_all_smem(K kernel, bool* configured)
{
    if (*configured) return ECCO_OK;
    const int rc = set_smem(kernel, kSmemCtaBytes);
    if (rc == ECCO_OK) *configured = true;
    return rc;
}

// tensors of fewer than 32 groups (the tile store's box is 32 rows tall), or when no tensor map can be made
static int launch_decompress_small(const DeviceInfo& di, const void* d_meta, const uint8_t* d_blocks, uint64_t n_groups, void* d_out,
                                   cudaStream_t stream)
{
    static thread_local bool configured[64] = {};
    auto kernel = ecco_decompress_kernel<kDecompressWarps>;
    int rc = want_all_smem(kernel, &configured[di.device]);
    if (rc) return rc;
    const unsigned grid = static_cast<unsigned>(spread_ctas(static_cast<int64_t>((n_groups + 31) / 32), di.sms));
    kernel<<<grid, kDecompressWarps * 32, kSmemCtaBytes, stream>>>(static_cast<const uint8_t*>(d_meta), d_blocks, n_groups,
                                                                   static_cast<uint16_t*>(d_out));
    return check_launch();
}

// one launch of the tile-store kernel over batch.n tensors (maps already made)
static int launch_decompress_batch(const DeviceInfo& di, DecompressBatch& batch, cudaStream_t stream)
{
    static thread_local bool configured[64] = {};
    auto kernel = ecco_decompress_tma_kernel<kDecompressTmaWarps>;
    int rc = want_all_smem(kernel, &configured[di.device]);
    if (rc) return rc;
    uint64_t tiles = 0;
    for (int t = 0; t < batch.n; ++t) tiles += (batch.job[t].n_groups + 31) / 32;
    const unsigned grid = static_cast<unsigned>(spread_ctas(static_cast<int64_t>(tiles), di.sms));
    return launch_overlapped(kernel, grid, spread_threads(static_cast<int64_t>(tiles), static_cast<int>(grid), kDecompressTmaWarps), kSmemCtaBytes, stream, batch);
}

// The tile-store kernel addresses output rows with the 32-bit signed coordinates of the TMA unit: tensors of 2^31 groups
// (256 GiB of fp16) or more are refused.
constexpr uint64_t kMaxGroups = (1ull << 31) - 32;

static int check_decompress_args(const void* d_meta, const uint8_t* d_blocks, uint64_t n_groups, const void* d_out)
{
    if (!d_meta || !d_blocks || !d_out) return ECCO_ERR_INVALID_ARG;
    if (!aligned16(d_meta) || !aligned16(d_blocks) || !aligned16(d_out)) return ECCO_ERR_ALIGNMENT;
    if (n_groups > kMaxGroups) return ECCO_ERR_INVALID_ARG;
    return ECCO_OK;
}

extern "C" int ecco_decompress_batch(const ecco_decompress_item* items, int32_t n_items, void* stream)
{
    if (n_items < 0 || (n_items > 0 && !items)) return ECCO_ERR_INVALID_ARG;
    for (int i = 0; i < n_items; ++i) {                    // nothing is launched unless every item is acceptable
        if (items[i].n_groups == 0) continue;
        const int rc = check_decompress_args(items[i].d_meta, items[i].d_blocks, items[i].n_groups, items[i].d_out_fp16);
        if (rc) return rc;
    }
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    DecompressBatch batch;
    std::memset(&batch, 0, sizeof batch);
    for (int i = 0; i < n_items; ++i) {
        const ecco_decompress_item& it = items[i];
        if (it.n_groups == 0) continue;
        DecompressJob& job = batch.job[batch.n];
        if (it.n_groups >= 32 && make_out_map(&job.map, it.d_out_fp16, it.n_groups)) {
            job.meta = static_cast<const uint8_t*>(it.d_meta);
            job.blocks = it.d_blocks;
            job.n_groups = it.n_groups;
            job.out = static_cast<uint16_t*>(it.d_out_fp16);
            if (++batch.n == kMaxJobs) {
                rc = launch_decompress_batch(di, batch, s);
                if (rc) return rc;
                batch.n = 0;
            }
        } else {                                           // items keep their order in the stream
            if (batch.n) {
                rc = launch_decompress_batch(di, batch, s);
                if (rc) return rc;
                batch.n = 0;
            }
            rc = launch_decompress_small(di, it.d_meta, it.d_blocks, it.n_groups, it.d_out_fp16, s);
            if (rc) return rc;
        }
    }
    return batch.n ? launch_decompress_batch(di, batch, s) : ECCO_OK;
}

extern "C" int ecco_decompress(const void* d_meta, const uint8_t* d_blocks, uint64_t n_groups, void* d_out, void* stream)
{
    if (n_groups == 0) return ECCO_OK;
    const ecco_decompress_item item = {d_meta, d_blocks, n_groups, d_out};
    return ecco_decompress_batch(&item, 1, stream);
}

constexpr int kVarWarps = 28;

extern "C" int ecco_var_decompress(const void* d_meta, const uint8_t* d_stream, const void* d_index, uint64_t n_groups, void* d_out,
                                   void* stream)
{
    if (n_groups == 0) return ECCO_OK;
    if (!d_meta || !d_stream || !d_index || !d_out) return ECCO_ERR_INVALID_ARG;
    if (!aligned16(d_meta) || !aligned16(d_stream) || !aligned16(d_out) || (reinterpret_cast<uintptr_t>(d_index) & 7u)) return ECCO_ERR_ALIGNMENT;
    if (n_groups > kMaxGroups) return ECCO_ERR_INVALID_ARG;
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc) return rc;
    // rows past the end of the tensor are dropped by the tile store, so any n_groups >= 1 works
    CUtensorMap map;
    if (!make_out_map(&map, d_out, n_groups)) return ECCO_ERR_CUDA;
    auto kernel = ecco_var_decompress_kernel<kVarWarps>;
    static thread_local bool configured[64] = {};
    rc = want_all_smem(kernel, &configured[di.device]);
    if (rc) return rc;
    const unsigned grid = static_cast<unsigned>(spread_ctas(static_cast<int64_t>((n_groups + 31) / 32), di.sms));
    return launch_overlapped(kernel, grid, spread_threads(static_cast<int64_t>((n_groups + 31) / 32), static_cast<int>(grid), kVarWarps), kSmemCtaBytes, static_cast<cudaStream_t>(stream),
                             static_cast<const uint8_t*>(d_meta), reinterpret_cast<const uint4*>(d_stream),
                             static_cast<const uint64_t*>(d_index), n_groups, map);
}

extern "C" size_t ecco_gemv_workspace_bytes(int32_t n_out, int32_t k, int32_t batch)
{
    if (n_out <= 0 || k <= 0 || k % kGroup || batch < 1 || batch > ECCO_MAX_BATCH) return 0;
    // sized for the largest plan any supported device can ask for (at most 256 persistent CTAs)
    const int row_tiles = (n_out + 31) / 32;
    const GemvPlan p = gemv_plan_for(static_cast<int64_t>(row_tiles) * (k / kGroup), row_tiles, pad_v(batch), 256);
    return p.partial_bytes + p.ticket_bytes;
}

// the matrices of one call with their places in the call's unit and tile spaces
struct GemvCall {
    GemvBatch b;
    int row_tiles;
};
static void gemv_call_begin(GemvCall* c)
{
    std::memset(c, 0, sizeof *c);
}
static void gemv_call_add(GemvCall* c, const void* d_meta, const uint8_t* d_blocks, int n_out, int kblocks, const void* d_x, float* d_y)
{
    GemvJob& j = c->b.job[c->b.n++];
    j.meta = static_cast<const uint8_t*>(d_meta);
    j.blocks = d_blocks;
    j.x = static_cast<const __half*>(d_x);
    j.y = d_y;
    j.n_out = n_out;
    j.kblocks = kblocks;
    j.tile_first = c->row_tiles;
    j.unit_first = c->b.units;
    const int tiles = (n_out + 31) / 32;
    c->row_tiles += tiles;
    c->b.units += static_cast<int64_t>(tiles) * kblocks;
}

// six to eight rows of x: the tensor-core kernel
template <bool kGiveUp = false>
static int launch_gemv_mma_call(const DeviceInfo& di, const GemvCall& c, int batch, void* d_ws, size_t ws_bytes, cudaStream_t stream)
{
    auto kernel = ecco_gemv_mma_kernel<kMmaWarps, kGiveUp>;
    static thread_local bool configured[64] = {};
    int rc = want_all_smem(kernel, &configured[di.device]);
    if (rc) return rc;
    const GemvPlan p = gemv_plan_for(c.b.units, c.row_tiles, 8, di.sms < 256 ? di.sms : 256);
    if (!d_ws || !aligned16(d_ws)) return d_ws ? ECCO_ERR_ALIGNMENT : ECCO_ERR_WORKSPACE;
    if (ws_bytes < p.partial_bytes + p.ticket_bytes) return ECCO_ERR_WORKSPACE;
    float* partial = static_cast<float*>(d_ws);
    Ticket* tickets = reinterpret_cast<Ticket*>(static_cast<uint8_t*>(d_ws) + p.partial_bytes);
    return launch_overlapped(kernel, static_cast<unsigned>(p.grid), spread_threads(c.b.units, p.grid, kMmaWarps), kSmemCtaBytes, stream, c.b, batch,
                             partial, tickets, next_ticket_tag());
}
static int launch_gemv_mma(const DeviceInfo& di, const void* d_meta, const uint8_t* d_blocks, int n_out, int kblocks,
                           const void* d_x, int batch, float* d_y, void* d_ws, size_t ws_bytes, cudaStream_t stream)
{
    GemvCall c;
    gemv_call_begin(&c);
    gemv_call_add(&c, d_meta, d_blocks, n_out, kblocks, d_x, d_y);
    return launch_gemv_mma_call(di, c, batch, d_ws, ws_bytes, stream);
}

// one to five rows of x (batch == kV): the per-warp kernel
template <int kV, bool kGiveUp = false>
static int launch_gemv_warp_call(const DeviceInfo& di, const GemvCall& c, void* d_ws, size_t ws_bytes, cudaStream_t stream)
{
    constexpr int kFusedWarps = gemv_warp_warps(kV);
    auto kernel = ecco_gemv_warp_kernel<kV, kFusedWarps, kGiveUp>;
    static thread_local bool configured[64] = {};
    int rc = want_all_smem(kernel, &configured[di.device]);
    if (rc) return rc;
    const GemvPlan p = gemv_plan_for(c.b.units, c.row_tiles, kV, di.sms < 256 ? di.sms : 256);
    if (!d_ws || !aligned16(d_ws)) return d_ws ? ECCO_ERR_ALIGNMENT : ECCO_ERR_WORKSPACE;
    if (ws_bytes < p.partial_bytes + p.ticket_bytes) return ECCO_ERR_WORKSPACE;
    float* partial = static_cast<float*>(d_ws);
    Ticket* tickets = reinterpret_cast<Ticket*>(static_cast<uint8_t*>(d_ws) + p.partial_bytes);
    return launch_overlapped(kernel, static_cast<unsigned>(p.grid), spread_threads(c.b.units, p.grid, kFusedWarps), kSmemCtaBytes, stream, c.b,
                             partial, tickets, next_ticket_tag());
}
template <int kV>
static int launch_gemv_warp(const DeviceInfo& di, const void* d_meta, const uint8_t* d_blocks, int n_out, int kblocks,
                            const void* d_x, float* d_y, void* d_ws, size_t ws_bytes, cudaStream_t stream)
{
    GemvCall c;
    gemv_call_begin(&c);
    gemv_call_add(&c, d_meta, d_blocks, n_out, kblocks, d_x, d_y);
    return launch_gemv_warp_call<kV>(di, c, d_ws, ws_bytes, stream);
}

extern "C" int ecco_gemv(const void* d_meta, const uint8_t* d_blocks, int32_t n_out, int32_t k, const void* d_x,
                         int32_t batch, float* d_y, void* d_workspace, size_t workspace_bytes, void* stream)
{
    if (!d_meta || !d_blocks || !d_x || !d_y) return ECCO_ERR_INVALID_ARG;
    if (n_out <= 0 || k <= 0 || k % kGroup || batch < 1 || batch > ECCO_MAX_BATCH) return ECCO_ERR_INVALID_ARG;
    if (!aligned16(d_meta) || !aligned16(d_blocks) || !aligned16(d_x) || !aligned16(d_y)) return ECCO_ERR_ALIGNMENT;
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int kblocks = k / kGroup;
    switch (pad_v(batch)) {
        case 1: return launch_gemv_warp<1>(di, d_meta, d_blocks, n_out, kblocks, d_x, d_y, d_workspace, workspace_bytes, s);
        case 2: return launch_gemv_warp<2>(di, d_meta, d_blocks, n_out, kblocks, d_x, d_y, d_workspace, workspace_bytes, s);
        case 3: return launch_gemv_warp<3>(di, d_meta, d_blocks, n_out, kblocks, d_x, d_y, d_workspace, workspace_bytes, s);
        case 4: return launch_gemv_warp<4>(di, d_meta, d_blocks, n_out, kblocks, d_x, d_y, d_workspace, workspace_bytes, s);
        case 5: return launch_gemv_warp<5>(di, d_meta, d_blocks, n_out, kblocks, d_x, d_y, d_workspace, workspace_bytes, s);
        default: return launch_gemv_mma(di, d_meta, d_blocks, n_out, kblocks, d_x, batch, d_y, d_workspace, workspace_bytes, s);
    }
}

// several matrices in one call: one unit space, one launch
static int check_gemv_items(const ecco_gemv_item* items, int32_t n_items, int32_t batch)
{
    if (!items || n_items < 1 || n_items > ECCO_MAX_GEMV_ITEMS || batch < 1 || batch > ECCO_MAX_BATCH) return ECCO_ERR_INVALID_ARG;
    for (int i = 0; i < n_items; ++i) {
        const ecco_gemv_item& it = items[i];
        if (!it.d_meta || !it.d_blocks || !it.d_x_fp16 || !it.d_y) return ECCO_ERR_INVALID_ARG;
        if (it.n_out <= 0 || it.k <= 0 || it.k % kGroup) return ECCO_ERR_INVALID_ARG;
        if (!aligned16(it.d_meta) || !aligned16(it.d_blocks) || !aligned16(it.d_x_fp16) || !aligned16(it.d_y)) return ECCO_ERR_ALIGNMENT;
    }
    return ECCO_OK;
}
static void gemv_call_from_items(GemvCall* c, const ecco_gemv_item* items, int32_t n_items)
{
    gemv_call_begin(c);
    for (int i = 0; i < n_items; ++i)
        gemv_call_add(c, items[i].d_meta, items[i].d_blocks, items[i].n_out, items[i].k / kGroup, items[i].d_x_fp16, items[i].d_y);
}

extern "C" size_t ecco_gemv_batch_workspace_bytes(const ecco_gemv_item* items, int32_t n_items, int32_t batch)
{
    if (!items || n_items < 1 || n_items > ECCO_MAX_GEMV_ITEMS || batch < 1 || batch > ECCO_MAX_BATCH) return 0;
    int64_t units = 0, tiles = 0;
    for (int i = 0; i < n_items; ++i) {
        if (items[i].n_out <= 0 || items[i].k <= 0 || items[i].k % kGroup) return 0;
        const int64_t t = (items[i].n_out + 31) / 32;
        tiles += t;
        units += t * (items[i].k / kGroup);
    }
    if (tiles > INT32_MAX) return 0;
    const GemvPlan p = gemv_plan_for(units, static_cast<int>(tiles), pad_v(batch), 256);
    return p.partial_bytes + p.ticket_bytes;
}

extern "C" int ecco_gemv_batch(const ecco_gemv_item* items, int32_t n_items, int32_t batch, void* d_workspace,
                               size_t workspace_bytes, void* stream)
{
    int rc = check_gemv_items(items, n_items, batch);
    if (rc) return rc;
    DeviceInfo di;
    rc = device_info(&di);
    if (rc) return rc;
    GemvCall c;
    gemv_call_from_items(&c, items, n_items);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    switch (pad_v(batch)) {
        case 1: return launch_gemv_warp_call<1>(di, c, d_workspace, workspace_bytes, s);
        case 2: return launch_gemv_warp_call<2>(di, c, d_workspace, workspace_bytes, s);
        case 3: return launch_gemv_warp_call<3>(di, c, d_workspace, workspace_bytes, s);
        case 4: return launch_gemv_warp_call<4>(di, c, d_workspace, workspace_bytes, s);
        case 5: return launch_gemv_warp_call<5>(di, c, d_workspace, workspace_bytes, s);
        default: return launch_gemv_mma_call(di, c, batch, d_workspace, workspace_bytes, s);
    }
}

extern "C" int ecco_test_gemv_give_up(const ecco_gemv_item* items, int32_t n_items, int32_t batch, void* d_workspace,
                                      size_t workspace_bytes, void* stream)
{
    int rc = check_gemv_items(items, n_items, batch);
    if (rc) return rc;
    if (batch > 1 && pad_v(batch) < 8) return ECCO_ERR_INVALID_ARG;
    DeviceInfo di;
    rc = device_info(&di);
    if (rc) return rc;
    GemvCall c;
    gemv_call_from_items(&c, items, n_items);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    return batch == 1 ? launch_gemv_warp_call<1, true>(di, c, d_workspace, workspace_bytes, s)
                      : launch_gemv_mma_call<true>(di, c, batch, d_workspace, workspace_bytes, s);
}

// ---------------------------------------------------------------------------------------------
// ecco_gemv_static_ws: ecco_gemv for callers that cannot allocate.  The split-k scratch is this
// fixed array in the library's device image.  In host code the name below is only a handle for
// the runtime, not a device address: the address comes from cudaGetSymbolAddress, once per
// device, and that pointer is what the kernel receives.
// ---------------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_static_workspace[ECCO_STATIC_WORKSPACE_BYTES];

extern "C" int ecco_gemv_static_ws(const void* d_meta, const uint8_t* d_blocks, int32_t n_out, int32_t k, const void* d_x,
                                   int32_t batch, float* d_y, void* stream)
{
    if (!d_meta || !d_blocks || !d_x || !d_y) return ECCO_ERR_INVALID_ARG;
    if (n_out <= 0 || k <= 0 || k % kGroup || batch < 1 || batch > ECCO_MAX_BATCH) return ECCO_ERR_INVALID_ARG;
    if (!aligned16(d_meta) || !aligned16(d_blocks) || !aligned16(d_x) || !aligned16(d_y)) return ECCO_ERR_ALIGNMENT;
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc) return rc;
    const int kblocks = k / kGroup, vpad = pad_v(batch);
    // refuse, before any launch, a shape whose plan does not fit the fixed array
    const int ctas = di.sms < 256 ? di.sms : 256;
    const int row_tiles = (n_out + 31) / 32;
    const GemvPlan p = gemv_plan_for(static_cast<int64_t>(row_tiles) * kblocks, row_tiles, vpad, ctas);
    if (p.partial_bytes + p.ticket_bytes > ECCO_STATIC_WORKSPACE_BYTES) return ECCO_ERR_WORKSPACE;
    // one-time set-up per device (the current device is di.device): resolve the array's address
    static std::mutex mu;
    static void* address[64] = {};
    void* ws = nullptr;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!address[di.device]) {
            void* ptr = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&ptr, g_static_workspace);
            if (e != cudaSuccess || !ptr) { t_last_cuda_error = static_cast<int>(e); return ECCO_ERR_CUDA; }
            address[di.device] = ptr;
        }
        ws = address[di.device];
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    switch (vpad) {
        case 1: return launch_gemv_warp<1>(di, d_meta, d_blocks, n_out, kblocks, d_x, d_y, ws, ECCO_STATIC_WORKSPACE_BYTES, s);
        case 2: return launch_gemv_warp<2>(di, d_meta, d_blocks, n_out, kblocks, d_x, d_y, ws, ECCO_STATIC_WORKSPACE_BYTES, s);
        case 3: return launch_gemv_warp<3>(di, d_meta, d_blocks, n_out, kblocks, d_x, d_y, ws, ECCO_STATIC_WORKSPACE_BYTES, s);
        case 4: return launch_gemv_warp<4>(di, d_meta, d_blocks, n_out, kblocks, d_x, d_y, ws, ECCO_STATIC_WORKSPACE_BYTES, s);
        case 5: return launch_gemv_warp<5>(di, d_meta, d_blocks, n_out, kblocks, d_x, d_y, ws, ECCO_STATIC_WORKSPACE_BYTES, s);
        default: return launch_gemv_mma(di, d_meta, d_blocks, n_out, kblocks, d_x, batch, d_y, ws, ECCO_STATIC_WORKSPACE_BYTES, s);
    }
}

template <int kV>
static int launch_attn(const DeviceInfo& di, const void* d_meta, const uint8_t* d_kblocks, int batch, int n_kv_heads,
                       int seq, const void* d_q, float scale, float* d_scores, cudaStream_t stream)
{
    constexpr int kFusedWarps = fused_warps(kV);
    auto kernel = ecco_attn_scores_kernel<kV, kFusedWarps>;
    static thread_local bool configured[64] = {};
    int rc = want_all_smem(kernel, &configured[di.device]);
    if (rc) return rc;
    const int heads = batch * n_kv_heads;
    // persistent CTAs; the units (32 tokens of a head) are split evenly over the working warps on the device
    const int64_t units = static_cast<int64_t>(heads) * ((seq + 31) / 32);
    const unsigned grid = static_cast<unsigned>(spread_ctas(units, di.sms));
    return launch_overlapped(kernel, grid, spread_threads(units, static_cast<int>(grid), kFusedWarps), kSmemCtaBytes, stream, static_cast<const uint8_t*>(d_meta),
                             d_kblocks, heads, seq, static_cast<const __half*>(d_q), scale, d_scores);
}

extern "C" int ecco_attn_scores(const void* d_meta, const uint8_t* d_kblocks, int32_t batch, int32_t n_kv_heads, int32_t seq,
                                int32_t q_per_kv, const void* d_q, float scale, float* d_scores, void* stream)
{
    if (batch == 0 || n_kv_heads == 0 || seq == 0) return (batch < 0 || n_kv_heads < 0 || seq < 0) ? ECCO_ERR_INVALID_ARG : ECCO_OK;
    if (!d_meta || !d_kblocks || !d_q || !d_scores) return ECCO_ERR_INVALID_ARG;
    if (batch < 0 || n_kv_heads < 0 || seq < 0 || q_per_kv < 1 || q_per_kv > 8) return ECCO_ERR_INVALID_ARG;
    if (static_cast<int64_t>(batch) * n_kv_heads > (1 << 24)) return ECCO_ERR_INVALID_ARG;
    if (!aligned16(d_meta) || !aligned16(d_kblocks) || !aligned16(d_q) || !aligned16(d_scores)) return ECCO_ERR_ALIGNMENT;
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    switch (pad_v(q_per_kv)) {
        case 1: return launch_attn<1>(di, d_meta, d_kblocks, batch, n_kv_heads, seq, d_q, scale, d_scores, s);
        case 2: return launch_attn<2>(di, d_meta, d_kblocks, batch, n_kv_heads, seq, d_q, scale, d_scores, s);
        default: {
            auto kernel = ecco_attn_scores_mma_kernel<kMmaWarps>;
            static thread_local bool configured[64] = {};
            rc = want_all_smem(kernel, &configured[di.device]);
            if (rc) return rc;
            const uint64_t units = static_cast<uint64_t>(batch) * n_kv_heads * ((seq + 31) / 32);
            const unsigned grid = static_cast<unsigned>(spread_ctas(static_cast<int64_t>(units), di.sms));
            return launch_overlapped(kernel, grid, spread_threads(static_cast<int64_t>(units), static_cast<int>(grid), kMmaWarps), kSmemCtaBytes, s, static_cast<const uint8_t*>(d_meta),
                                     d_kblocks, batch * n_kv_heads, seq, q_per_kv, static_cast<const __half*>(d_q), scale, d_scores);
        }
    }
}

// ---------------------------------------------------------------------------------------------
// ecco_attn_values
// ---------------------------------------------------------------------------------------------
namespace {
// Warps of a CTA of ecco_attn_values that decode.  20 find room (9.4 KB of shared memory per warp), but with more than 16 a thread has 96
// registers and the kernel spills a little and takes a few percent more per tile: two kernels, and units of 17 to 19 tiles only where
// they save turns (a [16][8][32768][128] cache, eight heads, 534 us with 16 and 518 with 19; [8][32][4096][128] 162 and 166, by an earlier
// state of the kernel).  20, which takes the same registers, has not been measured.
constexpr int kAvWarps = 16, kAvManyWarps = 19;
struct AvPlan { int grid, unit_warps, teams; size_t partial_bytes, ticket_bytes; };
// How a CTA's warps share the work.  A unit is unit_warps tiles (of 32 tokens) of one head.
// One team: the units of all heads are split evenly over the CTAs, and all SMs should be busy for the same number of turns.  A turn
// costs about the time of six tiles' decoding however few tiles it has (6, 16 and 40 measured alike), so long rows take the
// largest units (16 x 8 x 32768 tokens: 19 warps) and short ones are cut until every SM has some.  Against 16 warps throughout:
// 8 x 32 x 64 tokens 27.1 -> 22.2 us, 2 x 8 x 777 17.4 -> 15.9, 1 x 1 x 32768 39.9 -> 25.5.
// Several teams of warps, each with heads of its own, for many short rows: one team spends 5 us on every head's reduction, most of it
// waiting, and the warps beyond the row's few tiles have nothing to do.  Against one team: 32 x 32 x 40 tokens 69.7 -> 17.6 us, 8 x 32 x 64
// 22.2 -> 14.4, 16 x 32 x 300 48.8 -> 34.5, 32 x 8 x 700 49.9 -> 33.9; from 4 x 32 x 1500 on one team is as fast (49.2 against 50.0).
void av_teams(AvPlan* p, int heads, int seq)
{
    constexpr int64_t kTurn = 6, kReduce = 10;             // a turn's fixed cost, and that of the reduction of a head, in tiles' decoding
    const int64_t tiles = (seq + 31) / 32, ctas = p->grid;
    int64_t best = INT64_MAX;
    p->teams = 1;
    for (int w = kAvManyWarps; w >= 1; --w) {
        const int64_t units = heads * ((tiles + w - 1) / w), turns = (units + ctas - 1) / ctas;
        int64_t cost = turns * (kTurn + w) + std::max<int64_t>(1, (heads + ctas - 1) / ctas - 1) * kReduce;
        if (w > kAvWarps) cost += cost / 32 + 1;
        if (cost < best) { best = cost; p->unit_warps = w; }
    }
    for (int t = 2; t <= kAvWarps; ++t) {
        const int64_t per_team = (heads + ctas * t - 1) / (ctas * t), active = std::min<int64_t>(t, (heads + ctas - 1) / ctas);
        for (int w = 1; w * t <= kAvWarps; ++w) {
            const int64_t cost = per_team * ((tiles + w - 1) / w * (kTurn + w * active) + kReduce);
            if (cost < best) { best = cost; p->unit_warps = w; p->teams = t; }
        }
    }
}
AvPlan av_plan(int batch, int n_kv_heads, int seq, int ctas_max)
{
    AvPlan p;
    const int heads = batch * n_kv_heads;
    // at most this many units; the device splits what there is evenly
    p.grid = spread_ctas(static_cast<int64_t>(heads) * ((seq + 31) / 32), ctas_max);
    av_teams(&p, heads, seq);
    auto up = [](size_t v) { return (v + 255) & ~static_cast<size_t>(255); };
    p.partial_bytes = up(static_cast<size_t>(p.grid + heads) * kPieceFloats * sizeof(float));
    p.ticket_bytes = up(static_cast<size_t>(heads) * sizeof(Ticket));
    return p;
}

template <int kWarps, bool kGiveUp = false>
int launch_attn_values(const DeviceInfo& di, const AvPlan& p, const void* d_meta, const uint8_t* d_vblocks, int heads, int seq,
                       int q_per_kv, const float* d_scores, float* d_out, float* partial, Ticket* tickets, cudaStream_t s)
{
    auto kernel = ecco_attn_values_kernel<kWarps, kGiveUp>;
    static thread_local bool configured[64] = {};
    const int rc = want_all_smem(kernel, &configured[di.device]);
    if (rc) return rc;
    // at least eight warps: those beyond the unit's help with the reductions
    const int warps = p.unit_warps * p.teams < 8 ? 8 : p.unit_warps * p.teams;
    return launch_overlapped(kernel, static_cast<unsigned>(p.grid), static_cast<unsigned>(warps * 32), kSmemCtaBytes, s,
                             static_cast<const uint8_t*>(d_meta), d_vblocks, heads, seq, q_per_kv, p.unit_warps, p.teams, d_scores, d_out, partial, tickets, next_ticket_tag());
}
}  // namespace

extern "C" size_t ecco_attn_values_workspace_bytes(int32_t batch, int32_t n_kv_heads, int32_t seq, int32_t q_per_kv)
{
    if (batch <= 0 || n_kv_heads <= 0 || seq <= 0 || q_per_kv < 1 || q_per_kv > 8) return 0;
    if (static_cast<int64_t>(batch) * n_kv_heads > (1 << 24)) return 0;
    const AvPlan p = av_plan(batch, n_kv_heads, seq, 256);
    return p.partial_bytes + p.ticket_bytes;
}

template <bool kGiveUp>
static int attn_values(const void* d_meta, const uint8_t* d_vblocks, int32_t batch, int32_t n_kv_heads, int32_t seq,
                       int32_t q_per_kv, const float* d_scores, float* d_out, void* d_workspace, size_t workspace_bytes,
                       void* stream)
{
    if (batch == 0 || n_kv_heads == 0) return (batch < 0 || n_kv_heads < 0) ? ECCO_ERR_INVALID_ARG : ECCO_OK;
    if (!d_meta || !d_vblocks || !d_scores || !d_out) return ECCO_ERR_INVALID_ARG;
    if (batch < 0 || n_kv_heads < 0 || seq <= 0 || q_per_kv < 1 || q_per_kv > 8) return ECCO_ERR_INVALID_ARG;
    if (static_cast<int64_t>(batch) * n_kv_heads > (1 << 24)) return ECCO_ERR_INVALID_ARG;
    if (!aligned16(d_meta) || !aligned16(d_vblocks) || !aligned16(d_scores) || !aligned16(d_out)) return ECCO_ERR_ALIGNMENT;
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc) return rc;
    const AvPlan p = av_plan(batch, n_kv_heads, seq, di.sms < 256 ? di.sms : 256);
    if (!d_workspace || !aligned16(d_workspace)) return d_workspace ? ECCO_ERR_ALIGNMENT : ECCO_ERR_WORKSPACE;
    if (workspace_bytes < p.partial_bytes + p.ticket_bytes) return ECCO_ERR_WORKSPACE;
    if (kGiveUp && p.unit_warps > kAvWarps) return ECCO_ERR_INVALID_ARG;       // no kernel for it
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint8_t* wsb = static_cast<uint8_t*>(d_workspace);
    float* partial = reinterpret_cast<float*>(wsb);
    Ticket* tickets = reinterpret_cast<Ticket*>(wsb + p.partial_bytes);
    auto launch = p.unit_warps > kAvWarps ? launch_attn_values<kAvManyWarps> : launch_attn_values<kAvWarps, kGiveUp>;
    return launch(di, p, d_meta, d_vblocks, batch * n_kv_heads, seq, q_per_kv, d_scores, d_out, partial, tickets, s);
}

extern "C" int ecco_attn_values(const void* d_meta, const uint8_t* d_vblocks, int32_t batch, int32_t n_kv_heads, int32_t seq,
                                int32_t q_per_kv, const float* d_scores, float* d_out, void* d_workspace, size_t workspace_bytes,
                                void* stream)
{
    return attn_values<false>(d_meta, d_vblocks, batch, n_kv_heads, seq, q_per_kv, d_scores, d_out, d_workspace, workspace_bytes, stream);
}

extern "C" int ecco_test_attn_values_give_up(const void* d_meta, const uint8_t* d_vblocks, int32_t batch, int32_t n_kv_heads, int32_t seq,
                                             int32_t q_per_kv, const float* d_scores, float* d_out, void* d_workspace, size_t workspace_bytes,
                                             void* stream)
{
    return attn_values<true>(d_meta, d_vblocks, batch, n_kv_heads, seq, q_per_kv, d_scores, d_out, d_workspace, workspace_bytes, stream);
}


extern "C" int ecco_act_decompress(const uint8_t* d_blocks, uint64_t n_groups, void* d_out_fp16, void* stream)
{
    if (n_groups == 0) return ECCO_OK;
    if (!d_blocks || !d_out_fp16) return ECCO_ERR_INVALID_ARG;
    if (!aligned16(d_blocks) || (reinterpret_cast<uintptr_t>(d_out_fp16) & 31u)) return ECCO_ERR_ALIGNMENT;
    if (n_groups > kMaxGroups) return ECCO_ERR_INVALID_ARG;
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc) return rc;
    const uint64_t n_chunks = n_groups * 4;
    return launch_overlapped(ecco_act_decompress_kernel, act_ctas(n_chunks, 1), static_cast<unsigned>(kActThreads), 0, static_cast<cudaStream_t>(stream),
                             reinterpret_cast<const uint4*>(d_blocks), n_chunks, static_cast<uint4*>(d_out_fp16));
}

extern "C" int ecco_act_compress(const void* d_x_fp16, uint64_t n_groups, uint8_t* d_blocks, void* stream)
{
    if (n_groups == 0) return ECCO_OK;
    if (!d_blocks || !d_x_fp16) return ECCO_ERR_INVALID_ARG;
    if (!aligned16(d_blocks) || (reinterpret_cast<uintptr_t>(d_x_fp16) & 31u)) return ECCO_ERR_ALIGNMENT;
    if (n_groups > kMaxGroups) return ECCO_ERR_INVALID_ARG;
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc) return rc;
    const uint64_t n_chunks = n_groups * 4;
    const int loads = act_compress_loads(n_chunks, di);
    return launch_overlapped(loads == 1 ? ecco_act_compress_kernel<1> : ecco_act_compress_kernel<2>, act_ctas(n_chunks, loads), static_cast<unsigned>(kActThreads), 0,
                             static_cast<cudaStream_t>(stream), static_cast<const uint4*>(d_x_fp16), n_chunks, reinterpret_cast<uint4*>(d_blocks));
}


// calls of at least this many groups: eight lanes per group and tables in shared memory (see the kernel)
constexpr uint64_t kKvManyGroups = 16384;

extern "C" int ecco_kv_compress(const void* d_meta, const void* d_x_fp16, uint64_t n_groups, uint8_t* d_blocks, void* stream)
{
    if (n_groups == 0) return ECCO_OK;
    if (!d_meta || !d_x_fp16 || !d_blocks) return ECCO_ERR_INVALID_ARG;
    if (!aligned16(d_meta) || !aligned16(d_x_fp16) || !aligned16(d_blocks)) return ECCO_ERR_ALIGNMENT;
    if (n_groups > kMaxGroups) return ECCO_ERR_INVALID_ARG;
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (n_groups >= kKvManyGroups) {
        static thread_local bool configured[64] = {};
        if (!configured[di.device]) {
            rc = set_smem(ecco_kv_compress_many_kernel, sizeof(KvManySmem));
            if (rc) return rc;
            configured[di.device] = true;
        }
        return launch_overlapped(ecco_kv_compress_many_kernel, static_cast<unsigned>(spread_ctas(static_cast<int64_t>((n_groups + 3) / 4), di.sms)),
                                 static_cast<unsigned>(kKvManyWarps * 32), sizeof(KvManySmem), s, static_cast<const uint8_t*>(d_meta),
                                 static_cast<const __half*>(d_x_fp16), n_groups, d_blocks);
    }
    const uint64_t ctas = (n_groups + kKvWarps - 1) / kKvWarps;
    const uint64_t cap = static_cast<uint64_t>(di.sms) * 8;
    return launch_overlapped(ecco_kv_compress_kernel, static_cast<unsigned>(ctas < cap ? ctas : cap), static_cast<unsigned>(kKvWarps * 32), 0,
                             s, static_cast<const uint8_t*>(d_meta), static_cast<const __half*>(d_x_fp16), n_groups, d_blocks);
}
