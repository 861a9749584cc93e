// C ABI of the MXInt linear-layer library: argument validation and kernel launches.
// Everything here is host code; the arithmetic lives in the kernels of the included headers.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <map>
#include <mutex>
#include <new>
#include <tuple>
#include <type_traits>
#include <vector>

#include "../../include/mxint.h"
#include "mx_alt.cuh"
#include "mx_attention.cuh"
#include "mx_gemm_dec.cuh"
#include "mx_gemm_simt.cuh"
#include "mx_gemm_splitk.cuh"
#include "mx_gemm_tc.cuh"
#include "mx_gemm_tc2.cuh"
#include "mx_gemm_rec.cuh"
#include "mx_gemm_tc8.cuh"
#include "mx_gemm_tcw.cuh"
#include "mx_gemm_tcx.cuh"
#include "mx_gemm_tmw.cuh"
#include "mx_gemv_mma.cuh"
#include "mx_gemv_stream.cuh"
#include "mx_glue.cuh"
#include "mx_quantize.cuh"
#include "mx_records.cuh"

namespace {

constexpr int MAX_DEVICES = 64;
constexpr int SM_COUNT_FALLBACK = 148;

__device__ uint32_t g_status_word;      // per device: bit 0 = a bounded wait expired

thread_local char t_cuda_error[512] = "";

struct DeviceInfo {
    bool probed = false;
    bool is_sm100 = false;
    int sm_count = SM_COUNT_FALLBACK;
    uint32_t *status = nullptr;
    bool tc_attr_set[2][4] = {{false, false, false, false}, {false, false, false, false}};
    bool tc_tail_attr_set[2] = {false, false};
    bool stream_attr_set[2][2] = {};
    bool mma_attr_set[2][2] = {};
    bool gemv_attr_set[12] = {};
    int gemv_clusters[12][4][2] = {};          // resident clusters by kernel, log2 of the cluster size, two CTAs per SM
    bool stream32_attr_set[2][2] = {};
    bool tc2_attr_set[2] = {false, false};
    bool tcw_attr_set[4] = {};
    bool tcx_attr_set = false;
    bool tc8_attr_set = false;
    bool rec_attr_set[4] = {};
    bool splitk_attr_set[4] = {};
    int splitk_clusters[mx::SplitKCfg::MAX_SPLIT + 1] = {-1, -1, -1, -1, -1};
    bool attn_attr_set[2] = {false, false};
    bool tmw_attr_set[8] = {};
    int tmw_clusters[8][mx::TmwCfg::MAX_SPLIT + 1] = {};       // resident clusters by kernel and pairs per cluster
    bool dec_attr_set[12] = {};
    int dec_clusters[12][mx::DecCfg::MAX_SPLIT + 1] = {};      // resident clusters by kernel and cluster size
};
DeviceInfo g_dev[MAX_DEVICES];
std::mutex g_init_mu;        // guards every lazily initialised field above and below (calls may come from several host threads)

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode_tiled = nullptr;

// ---- launch profile: CUDA events around every kernel launch, summed per kernel kind ----------
enum KernelKind { KIND_QUANTIZE = 0, KIND_DEQUANTIZE = 1, KIND_GEMM_TC = 2, KIND_GEMM_SIMT = 3,
                  KIND_GEMM_STREAM = 4, KIND_PREP = 5, KIND_GLUE = 6, KIND_COUNT = MX_KERNEL_KINDS };
struct ProfEntry { cudaEvent_t a, b; int kind; };
struct Profiler {
    bool on = false;
    std::vector<ProfEntry> entries;      // events in use since mx_profile_begin
    std::vector<ProfEntry> pool;         // events kept for reuse
    std::mutex mu;
};
Profiler g_prof;

struct ProfScope {
    cudaStream_t st;
    ProfEntry e{};
    bool live = false;
    ProfScope(int kind, cudaStream_t s) : st(s)
    {
        if (!g_prof.on) return;
        std::lock_guard<std::mutex> lk(g_prof.mu);
        if (!g_prof.pool.empty()) {
            e = g_prof.pool.back();
            g_prof.pool.pop_back();
        } else if (cudaEventCreate(&e.a) != cudaSuccess || cudaEventCreate(&e.b) != cudaSuccess) {
            return;
        }
        e.kind = kind;
        live = cudaEventRecord(e.a, st) == cudaSuccess;
    }
    ~ProfScope()
    {
        if (!live) return;
        cudaEventRecord(e.b, st);
        std::lock_guard<std::mutex> lk(g_prof.mu);
        g_prof.entries.push_back(e);
    }
};

mx_status_t cuda_fail(cudaError_t e, const char *what)
{
    snprintf(t_cuda_error, sizeof(t_cuda_error), "%s: %s", what, cudaGetErrorString(e));
    return MX_ERR_CUDA;
}

#define MX_CUDA(call)                                            \
    do {                                                         \
        cudaError_t e_ = (call);                                 \
        if (e_ != cudaSuccess) return cuda_fail(e_, #call);      \
    } while (0)

mx_status_t device_info(DeviceInfo **out)
{
    int dev = 0;
    MX_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= MAX_DEVICES) return MX_ERR_CUDA;
    DeviceInfo &d = g_dev[dev];
    std::lock_guard<std::mutex> lk(g_init_mu);
    if (!d.probed) {
        int major = 0, sms = 0;
        MX_CUDA(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev));
        MX_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        d.is_sm100 = (major == 10);
        d.sm_count = sms > 0 ? sms : SM_COUNT_FALLBACK;
        if (d.is_sm100) {
            void *p = nullptr;
            MX_CUDA(cudaGetSymbolAddress(&p, g_status_word));
            d.status = static_cast<uint32_t *>(p);
        }
        d.probed = true;
    }
    *out = &d;
    return d.is_sm100 ? MX_OK : MX_ERR_ARCH;
}

// block_rows == 2: two adjacent rows share the exponents (the paper's (16,2) block shape).
// Either storage form of the mantissas ...
bool format_ok_any(const mx_format_t &f)
{
    return (f.block == 16 || f.block == 32) && f.elem_bits >= 2 && f.elem_bits <= 8 &&
           f.exp_bits == 8 && (f.block_rows == 1 || f.block_rows == 2) && (f.packing == 0 || f.packing == 1);
}
// ... the container form only (what most kernels read and every kernel writes).
bool format_ok(const mx_format_t &f) { return format_ok_any(f) && f.packing == 0; }
size_t mant_row_bytes(int64_t K, const mx_format_t &f)
{
    return f.packing ? (size_t)(K * f.elem_bits / 8) : (f.elem_bits <= 4 ? (size_t)(K / 2) : (size_t)K);
}
bool format_1d(const mx_format_t &f) { return format_ok(f) && f.block_rows == 1; }
bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
size_t round256(size_t n) { return (n + 255u) & ~size_t(255); }

// CTAs of `kernel` (256 threads, no dynamic shared memory) that are resident per SM; looked up once.
template <typename K> int resident_ctas(K kernel)
{
    static std::mutex mu;
    static std::map<const void *, int> cache;
    std::lock_guard<std::mutex> lk(mu);
    const void *key = reinterpret_cast<const void *>(kernel);
    auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, 256, 0) != cudaSuccess || n < 1) n = 4;
    cache[key] = n;
    return n;
}

int grid_for(int64_t work_items, int threads, int sm_count, int ctas_per_sm)
{
    int64_t g = (work_items + threads - 1) / threads;
    const int64_t cap = (int64_t)sm_count * ctas_per_sm;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (int)g;
}

// Launch that may overlap the tail of the previous kernel in the stream (programmatic dependent
// launch): the kernel becomes resident early, sets up, and blocks in ptx::dep_wait() until its
// predecessor has completed.  Only for kernels that keep the rule beside dep_wait(): no global memory
// before it but what the kernel right in front leaves alone, and dep_wait() before dep_trigger().
template <typename... KArgs, typename... Args>
cudaError_t launch_dep(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                       Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    // the launch profile records events between kernels, which serialises them anyway: launch plainly
    cfg.numAttrs = g_prof.on ? 0 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

// ---- quantize launchers ---------------------------------------------------------------------
template <typename InT>
mx_status_t launch_quantize_rows(const InT *x, int64_t rows, int64_t K, int64_t ldx,
                                 const mx_format_t &f, mx::QuantOut out, const DeviceInfo &d,
                                 cudaStream_t st)
{
    const int64_t chunks = rows * (K / 8);
    if (chunks == 0) return MX_OK;
    if (f.block_rows == 2) {
        const int grid = grid_for((chunks + 1) / 2, 256, d.sm_count, 4);
        ProfScope prof(KIND_QUANTIZE, st);
        if (f.block == 16)
            MX_CUDA(launch_dep(mx::quantize_rows2_kernel<InT, 16>, dim3(grid), dim3(256), 0, st, x, rows, K, ldx, f.elem_bits, out));
        else
            MX_CUDA(launch_dep(mx::quantize_rows2_kernel<InT, 32>, dim3(grid), dim3(256), 0, st, x, rows, K, ldx, f.elem_bits, out));
        return MX_OK;
    }
    // few items: one per warp, in CTAs of two warps on all SMs (CTAs of eight warps with two items each / these, us: 128 x 768 fp32 to
    // MXInt4 2.0 / 1.7, 352 x 2048 2.6 / 2.5, 1024 x 768 2.5 / 2.5: the line is where they are even).  Short rows are an item each: more
    // items than are resident at once only while the others' CTAs, counted by elements, are few as well (16384 x 16 14.2 / 8.9,
    // but 16384 x 32 7.8 / 8.9, 32768 x 16 14.2 / 17.5)
    const int64_t items = rows * ((K / 8 + 31) / 32);
    if (chunks <= (int64_t)d.sm_count * (items <= (int64_t)d.sm_count * 48 ? 512 : 352)) {
        const unsigned g = (unsigned)((items + 1) / 2);
        ProfScope prof(KIND_QUANTIZE, st);
        if (f.block == 16)
            MX_CUDA(launch_dep(mx::quantize_rows_kernel<InT, 16, 1>, dim3(g), dim3(64), 0, st, x, rows, K, ldx, (int)f.elem_bits, out));
        else
            MX_CUDA(launch_dep(mx::quantize_rows_kernel<InT, 32, 1>, dim3(g), dim3(64), 0, st, x, rows, K, ldx, (int)f.elem_bits, out));
        MX_CUDA(cudaGetLastError());
        return MX_OK;
    }
    constexpr int UNROLL = 2;
    // at most one resident wave of CTAs: the grid-stride loop does the rest without a ragged second wave
    const int per_sm = f.block == 16 ? resident_ctas(mx::quantize_rows_kernel<InT, 16, UNROLL>)
                                     : resident_ctas(mx::quantize_rows_kernel<InT, 32, UNROLL>);
    const int grid = grid_for((chunks + UNROLL - 1) / UNROLL, 256, d.sm_count, per_sm);
    ProfScope prof(KIND_QUANTIZE, st);
    if (f.block == 16)
        MX_CUDA(launch_dep(mx::quantize_rows_kernel<InT, 16, UNROLL>, dim3(grid), dim3(256), 0, st, x, rows, K, ldx, f.elem_bits, out));
    else
        MX_CUDA(launch_dep(mx::quantize_rows_kernel<InT, 32, UNROLL>, dim3(grid), dim3(256), 0, st, x, rows, K, ldx, f.elem_bits, out));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

template <typename InT>
mx_status_t launch_quantize_columns(const InT *x, int64_t rows, int64_t K, int64_t stride_k, const mx_format_t &f, const mx::QuantOut &out,
                                    const DeviceInfo &d, cudaStream_t st)
{
    const int64_t ctas = (((rows + 31) / 32) * (K / 32) + 1) / 2;
    ProfScope prof(KIND_QUANTIZE, st);
    MX_CUDA(launch_dep(mx::quantize_columns_kernel<InT>, dim3((unsigned)(ctas < INT32_MAX ? ctas : INT32_MAX)), dim3(64), 0, st, x, rows, K, stride_k,
                       (int)f.block, (int)f.elem_bits, out));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

mx_status_t quantize_rows_any(const void *x, mx_dtype_t dt, int64_t rows, int64_t K, int64_t ldx,
                              const mx_format_t &f, mx::QuantOut out, const DeviceInfo &d,
                              cudaStream_t st)
{
    if (dt == MX_F32)
        return launch_quantize_rows(static_cast<const float *>(x), rows, K, ldx, f, out, d, st);
    return launch_quantize_rows(static_cast<const __nv_bfloat16 *>(x), rows, K, ldx, f, out, d, st);
}

mx::PackedStrides dense_strides(int64_t K, const mx_format_t &f)
{
    mx::PackedStrides ps;
    ps.mant_ld = f.elem_bits <= 4 ? K / 2 : K;
    ps.exp_ld = K / f.block;
    ps.mant_batch = ps.exp_batch = ps.out_batch = 0;
    ps.exp_row_shift = f.block_rows == 2 ? 1 : 0;
    ps.perm = 0;
    return ps;
}

// (mant, exps) -> bf16 [rows, ld] for `batch` items laid out by `ps`.
mx_status_t launch_dequant_bf16(const void *mant, const uint8_t *exps, int64_t rows, int64_t K,
                                const mx_format_t &f, __nv_bfloat16 *out, int64_t ld,
                                const mx::PackedStrides &ps, int64_t batch, const DeviceInfo &d,
                                cudaStream_t st)
{
    const int64_t chunks = rows * (K / 8);
    if (chunks == 0 || batch == 0) return MX_OK;
    const uint8_t *m = static_cast<const uint8_t *>(mant);
    const bool wide_ok = (K % 32) == 0 && (ps.mant_ld % 16) == 0 && (ps.mant_batch % 16) == 0;
    const bool nib = f.elem_bits <= 4;
    if (wide_ok && batch == 1 && (K % 1024) != 0 && ld == K && ps.mant_ld == (nib ? K / 2 : K) && ps.exp_ld == K / f.block && !ps.exp_row_shift &&
        rows > 1 && rows * K / 32 <= INT32_MAX / 2) {
        // a dense tensor is one long row: warps of rows that are no whole segments would have idle lanes (352 columns: 21 of 32)
        mx::PackedStrides flat = ps;
        flat.mant_ld *= rows;
        flat.exp_ld *= rows;
        return launch_dequant_bf16(mant, exps, 1, rows * K, f, out, rows * K, flat, 1, d, st);
    }
    ProfScope prof(KIND_DEQUANTIZE, st);
    // few items: one per warp, in CTAs of two warps on all SMs (CTAs of eight warps with two items each / these, us: 352 x 2048 MXInt8
    // to bf16 2.7 / 1.9, 2048 x 768 3.0 / 2.6, 1024 x 4096 4.0 / 4.0)
    if (wide_ok && rows * (K / 32) * batch <= (int64_t)d.sm_count * 256) {
        const dim3 grid((unsigned)(rows * ((K / 32 + 31) / 32) + 1) / 2, (unsigned)batch);
        if (nib) MX_CUDA(launch_dep(mx::decode_bf16_kernel<true, 1>, dim3(grid), dim3(64), 0, st, m, exps, rows, K, f.block, f.elem_bits, out, ld, ps));
        else MX_CUDA(launch_dep(mx::decode_bf16_kernel<false, 1>, dim3(grid), dim3(64), 0, st, m, exps, rows, K, f.block, f.elem_bits, out, ld, ps));
    } else if (wide_ok) {                   // 32 elements per thread, 16-byte loads and stores
        constexpr int UNROLL = 2;
        const int64_t items = rows * (K / 32);
        const int per_sm = f.elem_bits <= 4 ? resident_ctas(mx::decode_bf16_kernel<true, UNROLL>)
                                            : resident_ctas(mx::decode_bf16_kernel<false, UNROLL>);
        const dim3 grid((unsigned)grid_for((items + UNROLL - 1) / UNROLL, 256, d.sm_count, per_sm), (unsigned)batch);
        if (f.elem_bits <= 4)
            MX_CUDA(launch_dep(mx::decode_bf16_kernel<true, UNROLL>, dim3(grid), dim3(256), 0, st, m, exps, rows, K, f.block, f.elem_bits, out, ld, ps));
        else
            MX_CUDA(launch_dep(mx::decode_bf16_kernel<false, UNROLL>, dim3(grid), dim3(256), 0, st, m, exps, rows, K, f.block, f.elem_bits, out, ld, ps));
    } else {
        const dim3 grid((unsigned)grid_for(chunks, 256, d.sm_count, 16), (unsigned)batch);
        mx::dequantize_kernel<__nv_bfloat16><<<grid, 256, 0, st>>>(m, exps, rows, K, f.block, f.elem_bits, out, ld, ps);
    }
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

mx_status_t launch_dequant_bf16(const void *mant, const uint8_t *exps, int64_t rows, int64_t K,
                                const mx_format_t &f, __nv_bfloat16 *out, int64_t ld,
                                const DeviceInfo &d, cudaStream_t st, bool perm = false)
{
    if (f.packing) {                    // dense storage: w bits per element
        if (rows == 0 || K == 0) return MX_OK;
        ProfScope prof(KIND_DEQUANTIZE, st);
        MX_CUDA(launch_dep(mx::dequantize_dense_kernel<__nv_bfloat16>, dim3(grid_for(rows * (K / 8), 256, d.sm_count, 8)),
                           dim3(256), 0, st, static_cast<const uint8_t *>(mant), exps, rows, K, (int)f.block,
                           (int)f.elem_bits, f.block_rows == 2 ? 1 : 0, out, ld, perm ? 1 : 0));
        MX_CUDA(cudaGetLastError());
        return MX_OK;
    }
    mx::PackedStrides ps = dense_strides(K, f);
    ps.perm = perm ? 1 : 0;
    return launch_dequant_bf16(mant, exps, rows, K, f, out, ld, ps, 1, d, st);
}

// Both operands of a product, (mant, exps) -> bf16 [rows, K]: one launch when both are in container form with
// whole 32-element items per row, else one launch each.
mx_status_t launch_dequant_pair(const void *a_mant, const uint8_t *a_exp, const mx_format_t &fa, int64_t M,
                                const void *w_mant, const uint8_t *w_exp, const mx_format_t &fw, int64_t N, int64_t K,
                                __nv_bfloat16 *a_hat, __nv_bfloat16 *w_hat, const DeviceInfo &d, cudaStream_t st)
{
    if (fa.packing || fw.packing || (K % 32) != 0) {
        const mx_status_t s = launch_dequant_bf16(a_mant, a_exp, M, K, fa, a_hat, K, d, st);
        if (s != MX_OK) return s;
        return launch_dequant_bf16(w_mant, w_exp, N, K, fw, w_hat, K, d, st);
    }
    mx::DecodePairJob j;
    j.a_mant = static_cast<const uint8_t *>(a_mant); j.a_exp = a_exp;
    j.w_mant = static_cast<const uint8_t *>(w_mant); j.w_exp = w_exp;
    j.M = M; j.N = N; j.K = K;
    j.block = fa.block; j.wa = fa.elem_bits; j.ww = fw.elem_bits;
    j.a_row_shift = fa.block_rows == 2 ? 1 : 0;
    j.w_row_shift = fw.block_rows == 2 ? 1 : 0;
    j.a_hat = a_hat; j.w_hat = w_hat;
    const bool na = fa.elem_bits <= 4, nw = fw.elem_bits <= 4;
    const int64_t items = (M + N) * (K / 32);
    ProfScope prof(KIND_DEQUANTIZE, st);
    static void (*const kernels[2][2])(mx::DecodePairJob) = {{mx::decode_pair_kernel<false, false>, mx::decode_pair_kernel<false, true>},
                                                              {mx::decode_pair_kernel<true, false>, mx::decode_pair_kernel<true, true>}};
    const auto kernel = kernels[na][nw];
    const dim3 grid((unsigned)grid_for((items + 1) / 2, 256, d.sm_count, resident_ctas(kernel)));
    MX_CUDA(launch_dep(kernel, dim3(grid), dim3(256), 0, st, j));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

// ---- tensor-core GEMM launcher ----------------------------------------------------------------
// Encoded tensor maps by (kind, base, extents): pure functions of their key, so entries never go stale.
typedef std::tuple<int, const void *, int64_t, int64_t, int64_t, int64_t, int64_t> MapKey;
std::map<MapKey, CUtensorMap> g_map_cache;
std::mutex g_map_mu;
bool cached_map(const MapKey &key, CUtensorMap *out)
{
    std::lock_guard<std::mutex> lk(g_map_mu);
    auto it = g_map_cache.find(key);
    if (it == g_map_cache.end()) return false;
    *out = it->second;
    return true;
}
// (without host memory for the entry the map is encoded again next time: no C++ exception leaves a C function)
void remember_map(const MapKey &key, const CUtensorMap &tm)
try {
    std::lock_guard<std::mutex> lk(g_map_mu);
    if (g_map_cache.size() > 8192) g_map_cache.clear();
    g_map_cache[key] = tm;
} catch (const std::bad_alloc &) {
}

// The driver's tensor-map encoder, looked up once.
mx_status_t ensure_encoder()
{
    std::lock_guard<std::mutex> lk(g_init_mu);
    if (g_encode_tiled) return MX_OK;
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    MX_CUDA(cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q));
    if (q != cudaDriverEntryPointSuccess || !fn) {
        snprintf(t_cuda_error, sizeof(t_cuda_error), "cuTensorMapEncodeTiled not available");
        return MX_ERR_CUDA;
    }
    g_encode_tiled = reinterpret_cast<EncodeTiledFn>(fn);
    return MX_OK;
}

// Sets a kernel's dynamic shared-memory limit the first time the kernel is used on a device.
template <typename K> mx_status_t smem_attr_once(bool &done, K kernel, int bytes)
{
    std::lock_guard<std::mutex> lk(g_init_mu);
    if (done) return MX_OK;
    MX_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    done = true;
    return MX_OK;
}

// bf16 [rows, K] (dense rows); batch > 1: `batch` such items `item_bytes` apart, as a rank-3 map.
mx_status_t encode_bf16_rows(CUtensorMap *tm, const void *base, int64_t rows, int64_t K, int box_rows,
                             int64_t batch = 1, size_t item_bytes = 0)
{
    {
        const mx_status_t es = ensure_encoder();
        if (es != MX_OK) return es;
    }
    // A map depends only on these seven numbers; a layer called again with the same workspace finds
    // its maps here instead of paying a driver call each (a few microseconds per product for small layers).
    const MapKey key = std::make_tuple(0, base, rows, K, (int64_t)box_rows, batch, (int64_t)item_bytes);
    if (cached_map(key, tm)) return MX_OK;
    const cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)batch};
    const cuuint64_t strides[2] = {(cuuint64_t)K * 2, (cuuint64_t)item_bytes};
    const cuuint32_t box[3] = {(cuuint32_t)mx::TC_BK, (cuuint32_t)box_rows, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    const CUresult r = g_encode_tiled(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, batch > 1 ? 3 : 2, const_cast<void *>(base),
                                      dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                      CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        snprintf(t_cuda_error, sizeof(t_cuda_error), "cuTensorMapEncodeTiled failed (%d)", (int)r);
        return MX_ERR_CUDA;
    }
    remember_map(key, *tm);
    return MX_OK;
}

size_t tc_workspace(int64_t M, int64_t N, int64_t K);

struct QuantizedOut {            // MXInt result of the tensor-core product (see TcParams::yq_mant)
    uint8_t *mant = nullptr;
    uint8_t *exps = nullptr;
    uint32_t *nonfinite = nullptr;
    mx_format_t f{};
};

struct TcBatch {                 // several products of one shape in one launch (W_BF16 kernels)
    int64_t count = 1;
    size_t a_item = 0, w_item = 0;   // bytes between the items' bf16 operands
    int64_t y_batch = 0;             // floats between the items' outputs
    bool no_events = false;          // never bracket the launch with profile events (mx_gemm_static)
};

struct EpiTail {                 // element-wise tail fused into the product's epilogue (see TcParams::relu)
    int relu = 0;
    const float *residual = nullptr;
    int64_t ldr = 0;
    bool any() const { return relu != 0 || residual != nullptr; }
};

struct PackedW {                 // weight operand of the fused kernels (unused for W_BF16)
    const uint8_t *mant = nullptr;
    const uint8_t *exps = nullptr;
    int bits = 0, block = 0;
};

mx_status_t encode_f32_out(CUtensorMap *tm, float *y, int64_t M, int64_t N, int64_t ldy, int64_t batch = 1,
                           int64_t y_batch = 0)
{
    const MapKey key = std::make_tuple(1, static_cast<const void *>(y), M, N, ldy, batch, y_batch);
    if (cached_map(key, tm)) return MX_OK;
    const cuuint64_t dims[3] = {(cuuint64_t)N, (cuuint64_t)M, (cuuint64_t)batch};
    const cuuint64_t strides[2] = {(cuuint64_t)ldy * 4, (cuuint64_t)y_batch * 4};
    const cuuint32_t box[3] = {32, 32, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    const CUresult r = g_encode_tiled(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, batch > 1 ? 3 : 2, y, dims, strides, box, estr,
                                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                      CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        snprintf(t_cuda_error, sizeof(t_cuda_error), "cuTensorMapEncodeTiled (output) failed (%d)", (int)r);
        return MX_ERR_CUDA;
    }
    remember_map(key, *tm);
    return MX_OK;
}

// fp32 result, no fused tail, rows of y and the items of a batch 8-byte aligned: the epilogue may store from registers
// in the accumulator-fragment shape (TcParams::frag_store)
bool frag_store_ok(bool quantized, bool tail, const float *y, int64_t ldy, int64_t y_batch)
{
    return !quantized && !tail && y && (ldy % 2) == 0 && (y_batch % 2) == 0 && (reinterpret_cast<uintptr_t>(y) & 7u) == 0;
}

template <int BN, int WMODE>
mx_status_t launch_tc(const __nv_bfloat16 *a_hat, const __nv_bfloat16 *w_hat, const PackedW &pw,
                      int64_t M, int64_t N, int64_t K, const float *bias, float *y, int64_t ldy,
                      const QuantizedOut *yq, DeviceInfo &d, cudaStream_t st, const TcBatch &tb = TcBatch(),
                      const EpiTail &et = EpiTail())
{
    using Cfg = mx::TcCfg<BN>;
    CUtensorMap tm_a, tm_w;
    mx_status_t s = encode_bf16_rows(&tm_a, a_hat, M, K, mx::TC_BM, tb.count, tb.a_item);
    if (s != MX_OK) return s;
    if (WMODE == mx::W_BF16) {
        s = encode_bf16_rows(&tm_w, w_hat, N, K, BN, tb.count, tb.w_item);
        if (s != MX_OK) return s;
    } else {
        tm_w = tm_a;                     // not read by the fused kernels
    }
    CUtensorMap tm_y = tm_a;             // placeholder when the epilogue stores directly
    // the tiled store clips at the tensor's extent in units of 16 bytes: with N % 4 != 0 it would write up to three
    // floats past column N - 1 of every row (into the caller's row padding), so such shapes take the direct stores
    const bool tma_store = !yq && (ldy % 4) == 0 && (N % 4) == 0 && (tb.y_batch % 4) == 0;
    if (tma_store) {
        s = encode_f32_out(&tm_y, y, M, N, ldy, tb.count, tb.y_batch);
        if (s != MX_OK) return s;
    }
    constexpr int slot = BN == 256 ? 0 : 1;
    const bool tail = WMODE == mx::W_BF16 && et.any();
    s = tail ? smem_attr_once(d.tc_tail_attr_set[slot], mx::gemm_tc_kernel<BN, mx::W_BF16, true>, (int)Cfg::SMEM_BYTES)
             : smem_attr_once(d.tc_attr_set[slot][WMODE], mx::gemm_tc_kernel<BN, WMODE>, (int)Cfg::SMEM_BYTES);
    if (s != MX_OK) return s;
    if (et.any() && !tail) return MX_ERR_FORMAT;          // the in-kernel decode variants have no tail
    mx::TcParams p;
    p.y = y;
    p.bias = et.any() ? nullptr : bias;
    p.ex_bias = et.any() ? bias : nullptr;
    p.relu = et.relu;
    p.residual = et.residual;
    p.ldr = et.ldr;
    p.ldy = ldy;
    p.M = (int)M;
    p.N = (int)N;
    p.K = (int)K;
    p.tiles_m = (int)((M + mx::TC_BM - 1) / mx::TC_BM);
    p.tiles_n = (int)((N + BN - 1) / BN);
    p.status = d.status;
    p.tma_store = tma_store ? 1 : 0;
    p.frag_store = frag_store_ok(yq != nullptr, et.any(), y, ldy, tb.y_batch) && WMODE == mx::W_BF16 ? 1 : 0;
    p.w_mant = pw.mant;
    p.w_exp = pw.exps;
    p.w_bits = pw.bits;
    p.block = pw.block;
    p.yq_mant = yq ? yq->mant : nullptr;
    p.yq_exp = yq ? yq->exps : nullptr;
    p.yq_nonfinite = yq ? yq->nonfinite : nullptr;
    p.yq_bits = yq ? yq->f.elem_bits : 0;
    p.yq_block = yq ? yq->f.block : 0;
    p.yq_rows2 = yq && yq->f.block_rows == 2 ? 1 : 0;
    p.batch = (int)tb.count;
    p.y_batch = tb.y_batch;
    const int64_t tiles64 = (int64_t)p.tiles_m * p.tiles_n * tb.count;
    if (tiles64 > INT32_MAX / 2) return MX_ERR_SHAPE;
    const int tiles = (int)tiles64;
    const int grid = tiles < d.sm_count ? tiles : d.sm_count;
    const int threads = mx::tc_threads(BN, WMODE);
    if (tb.no_events) {
        mx::gemm_tc_kernel<BN, WMODE><<<grid, threads, Cfg::SMEM_BYTES, st>>>(tm_a, tm_w, tm_y, p);
        MX_CUDA(cudaGetLastError());
        return MX_OK;
    }
    ProfScope prof(KIND_GEMM_TC, st);
    if (tail) MX_CUDA(launch_dep(mx::gemm_tc_kernel<BN, mx::W_BF16, true>, dim3(grid), dim3(threads), Cfg::SMEM_BYTES, st, tm_a, tm_w, tm_y, p));
    else MX_CUDA(launch_dep(mx::gemm_tc_kernel<BN, WMODE>, dim3(grid), dim3(threads), Cfg::SMEM_BYTES, st, tm_a, tm_w, tm_y, p));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

// The CTA-pair kernel: 256 x 256 tiles, one product per launch.
mx_status_t launch_tc2(const __nv_bfloat16 *a_hat, const __nv_bfloat16 *w_hat, int64_t M, int64_t N, int64_t K,
                       const float *bias, float *y, int64_t ldy, const QuantizedOut *yq, DeviceInfo &d, cudaStream_t st,
                       const EpiTail &et = EpiTail())
{
    using Cfg = mx::Tc2Cfg;
    CUtensorMap tm_a, tm_w;
    mx_status_t s = encode_bf16_rows(&tm_a, a_hat, M, K, mx::TC_BM);
    if (s != MX_OK) return s;
    s = encode_bf16_rows(&tm_w, w_hat, N, K, Cfg::BN / 2);
    if (s != MX_OK) return s;
    CUtensorMap tm_y = tm_a;
    const bool tma_store = !yq && (ldy % 4) == 0 && (N % 4) == 0;       // see launch_tc
    if (tma_store) {
        s = encode_f32_out(&tm_y, y, M, N, ldy);
        if (s != MX_OK) return s;
    }
    s = et.any() ? smem_attr_once(d.tc2_attr_set[1], mx::gemm_tc2_kernel<true>, (int)Cfg::SMEM_BYTES)
                 : smem_attr_once(d.tc2_attr_set[0], mx::gemm_tc2_kernel<false>, (int)Cfg::SMEM_BYTES);
    if (s != MX_OK) return s;
    mx::TcParams p{};
    p.y = y;
    p.bias = et.any() ? nullptr : bias;
    p.ex_bias = et.any() ? bias : nullptr;
    p.relu = et.relu;
    p.residual = et.residual;
    p.ldr = et.ldr;
    p.ldy = ldy;
    p.M = (int)M;
    p.N = (int)N;
    p.K = (int)K;
    p.tiles_m = (int)((M + 255) / 256);
    p.tiles_n = (int)((N + Cfg::BN - 1) / Cfg::BN);
    p.status = d.status;
    p.tma_store = tma_store ? 1 : 0;
    p.frag_store = frag_store_ok(yq != nullptr, et.any(), y, ldy, 0) ? 1 : 0;
    p.batch = 1;
    p.yq_mant = yq ? yq->mant : nullptr;
    p.yq_exp = yq ? yq->exps : nullptr;
    p.yq_nonfinite = yq ? yq->nonfinite : nullptr;
    p.yq_bits = yq ? yq->f.elem_bits : 0;
    p.yq_block = yq ? yq->f.block : 0;
    p.yq_rows2 = yq && yq->f.block_rows == 2 ? 1 : 0;
    const int tiles = p.tiles_m * p.tiles_n;
    const int pairs = tiles < d.sm_count / 2 ? tiles : d.sm_count / 2;
    ProfScope prof(KIND_GEMM_TC, st);
    if (et.any()) MX_CUDA(launch_dep(mx::gemm_tc2_kernel<true>, dim3(2 * pairs), dim3(Cfg::THREADS), Cfg::SMEM_BYTES, st, tm_a, tm_w, tm_y, p));
    else MX_CUDA(launch_dep(mx::gemm_tc2_kernel<false>, dim3(2 * pairs), dim3(Cfg::THREADS), Cfg::SMEM_BYTES, st, tm_a, tm_w, tm_y, p));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

// CTA pairs with 256 x width tiles (mx_gemm_tcw.cuh).
mx_status_t launch_tcw(const __nv_bfloat16 *a_hat, const __nv_bfloat16 *w_hat, int64_t M, int64_t N, int64_t K, int width,
                       const float *bias, float *y, int64_t ldy, const QuantizedOut *yq, DeviceInfo &d, cudaStream_t st,
                       const EpiTail &et)
{
    using Cfg = mx::TcwCfg;
    CUtensorMap tm_a, tm_w;
    mx_status_t s = encode_bf16_rows(&tm_a, a_hat, M, K, mx::TC_BM);
    if (s != MX_OK) return s;
    s = encode_bf16_rows(&tm_w, w_hat, N, K, width / 4);
    if (s != MX_OK) return s;
    const bool tail = et.any(), q = yq != nullptr;
    typedef void (*Kernel)(CUtensorMap, CUtensorMap, mx::TcParams, int, int);
    static const Kernel kernels[4] = {mx::gemm_tcw_kernel<false, false>, mx::gemm_tcw_kernel<false, true>,
                                      mx::gemm_tcw_kernel<true, false>, mx::gemm_tcw_kernel<true, true>};
    const int which = (tail ? 2 : 0) + (q ? 1 : 0);
    s = smem_attr_once(d.tcw_attr_set[which], kernels[which], 227 * 1024);
    if (s != MX_OK) return s;
    int stages = Cfg::MAX_STAGES;
    while (Cfg::smem_bytes(width, stages) > 227u * 1024u) --stages;
    mx::TcParams p{};
    p.y = y;
    p.bias = tail ? nullptr : bias;
    p.ex_bias = tail ? bias : nullptr;
    p.relu = et.relu;
    p.residual = et.residual;
    p.ldr = et.ldr;
    p.ldy = ldy;
    p.M = (int)M;
    p.N = (int)N;
    p.K = (int)K;
    p.tiles_m = (int)((M + 255) / 256);
    p.tiles_n = (int)((N + width - 1) / width);
    p.status = d.status;
    p.frag_store = frag_store_ok(q, false, y, ldy, 0) ? 1 : 0;
    p.batch = 1;
    p.yq_mant = yq ? yq->mant : nullptr;
    p.yq_exp = yq ? yq->exps : nullptr;
    p.yq_nonfinite = yq ? yq->nonfinite : nullptr;
    p.yq_bits = yq ? yq->f.elem_bits : 0;
    p.yq_block = yq ? yq->f.block : 0;
    p.yq_rows2 = yq && yq->f.block_rows == 2 ? 1 : 0;
    const int tiles = p.tiles_m * p.tiles_n;
    const int pairs = tiles < d.sm_count / 2 ? tiles : d.sm_count / 2;
    ProfScope prof(KIND_GEMM_TC, st);
    MX_CUDA(launch_dep(kernels[which], dim3(2 * pairs), dim3(Cfg::THREADS), Cfg::smem_bytes(width, stages), st, tm_a, tm_w, p, width, stages));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

// The block-wise kernel (one tensor-memory accumulator per block, blocks added in fp32 registers):
// 128 x 128 tiles, fp32 result, one product per launch.
mx_status_t launch_tcx(const __nv_bfloat16 *a_hat, const __nv_bfloat16 *w_hat, int64_t M, int64_t N, int64_t K,
                       int block, const float *bias, float *y, int64_t ldy, DeviceInfo &d, cudaStream_t st)
{
    using Cfg = mx::TcxCfg;
    CUtensorMap tm_a, tm_w;
    mx_status_t s = encode_bf16_rows(&tm_a, a_hat, M, K, mx::TC_BM);
    if (s != MX_OK) return s;
    s = encode_bf16_rows(&tm_w, w_hat, N, K, Cfg::BN);
    if (s != MX_OK) return s;
    CUtensorMap tm_y = tm_a;
    const bool tma_store = (ldy % 4) == 0 && (N % 4) == 0;              // see launch_tc
    if (tma_store) {
        s = encode_f32_out(&tm_y, y, M, N, ldy);
        if (s != MX_OK) return s;
    }
    s = smem_attr_once(d.tcx_attr_set, mx::gemm_tcx_kernel, (int)Cfg::SMEM_BYTES);
    if (s != MX_OK) return s;
    mx::TcParams p{};
    p.y = y;
    p.bias = bias;
    p.ldy = ldy;
    p.M = (int)M;
    p.N = (int)N;
    p.K = (int)K;
    p.tiles_m = (int)((M + mx::TC_BM - 1) / mx::TC_BM);
    p.tiles_n = (int)((N + Cfg::BN - 1) / Cfg::BN);
    p.status = d.status;
    p.tma_store = tma_store ? 1 : 0;
    p.batch = 1;
    p.block = block;
    const int64_t tiles64 = (int64_t)p.tiles_m * p.tiles_n;
    if (tiles64 > INT32_MAX / 2) return MX_ERR_SHAPE;
    const int grid = tiles64 < d.sm_count ? (int)tiles64 : d.sm_count;
    ProfScope prof(KIND_GEMM_TC, st);
    MX_CUDA(launch_dep(mx::gemm_tcx_kernel, dim3(grid), dim3(Cfg::THREADS), Cfg::SMEM_BYTES, st, tm_a, tm_w, tm_y, p));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

// ---- hardware block-scaled path (kind::mxf8f6f4): blocks of 32, widths <= 5 on both operands --------
bool mxf8_fits(const mx_format_t &fa, const mx_format_t &fw, int64_t K)
{
    return fa.block == 32 && fw.block == 32 && fa.elem_bits <= 5 && fw.elem_bits <= 5 && (K % 128) == 0 &&
           fa.packing == 0 && fw.packing == 0;
}
size_t mxf8_sf_bytes(int64_t rows, int64_t K) { return round256((size_t)((rows + 127) / 128) * (size_t)(K / 128) * 512); }
// E4M3 elements and scale chunks of both operands
size_t mxf8_operand_bytes(int64_t M, int64_t N, int64_t K)
{
    return round256((size_t)M * K) + mxf8_sf_bytes(M, K) + round256((size_t)N * K) + mxf8_sf_bytes(N, K);
}

mx_status_t encode_u8_sw128(CUtensorMap *tm, const void *base, int64_t rows, int64_t row_bytes, int box_rows)
{
    mx_status_t s = ensure_encoder();
    if (s != MX_OK) return s;
    const MapKey key = std::make_tuple(3, base, rows, row_bytes, (int64_t)box_rows, (int64_t)0, (int64_t)0);
    if (cached_map(key, tm)) return MX_OK;
    const cuuint64_t dims[2] = {(cuuint64_t)row_bytes, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)row_bytes};
    const cuuint32_t box[2] = {128, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = g_encode_tiled(tm, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void *>(base), dims, strides, box, estr,
                                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                      CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        snprintf(t_cuda_error, sizeof(t_cuda_error), "cuTensorMapEncodeTiled (8-bit operand) failed (%d)", (int)r);
        return MX_ERR_CUDA;
    }
    remember_map(key, *tm);
    return MX_OK;
}

// Packed MXInt operands -> E4M3 + scale chunks in `ws` (mxf8_operand_bytes), then the block-scaled product.
mx_status_t run_tc8(const void *a_mant, const uint8_t *a_exp, const mx_format_t &fa, const void *w_mant, const uint8_t *w_exp,
                    const mx_format_t &fw, int64_t M, int64_t N, int64_t K, const float *bias, float *y, int64_t ldy,
                    uint8_t *ws, DeviceInfo &d, cudaStream_t st)
{
    using Cfg = mx::Tc8Cfg;
    uint8_t *a8 = ws;
    uint8_t *sfa = a8 + round256((size_t)M * K);
    uint8_t *w8 = sfa + mxf8_sf_bytes(M, K);
    uint8_t *sfw = w8 + round256((size_t)N * K);
    const int64_t chunks_a = (M + 127) / 128, chunks_w = (N + 127) / 128;
    {
        ProfScope prof(KIND_DEQUANTIZE, st);
        MX_CUDA(launch_dep(mx::pack_e4m3_kernel, dim3(grid_for(M * (K / 8), 256, d.sm_count, 8)), dim3(256), 0, st,
                           static_cast<const uint8_t *>(a_mant), a_exp, M, K, (int)fa.elem_bits, fa.block_rows == 2 ? 1 : 0,
                           a8, sfa, chunks_a));
    }
    {
        ProfScope prof(KIND_DEQUANTIZE, st);
        MX_CUDA(launch_dep(mx::pack_e4m3_kernel, dim3(grid_for(N * (K / 8), 256, d.sm_count, 8)), dim3(256), 0, st,
                           static_cast<const uint8_t *>(w_mant), w_exp, N, K, (int)fw.elem_bits, fw.block_rows == 2 ? 1 : 0,
                           w8, sfw, chunks_w));
    }
    CUtensorMap tm_a, tm_w;
    mx_status_t s = encode_u8_sw128(&tm_a, a8, M, K, mx::TC_BM);
    if (s != MX_OK) return s;
    s = encode_u8_sw128(&tm_w, w8, N, K, Cfg::BN);
    if (s != MX_OK) return s;
    CUtensorMap tm_y = tm_a;
    const bool tma_store = (ldy % 4) == 0 && (N % 4) == 0;              // see launch_tc
    if (tma_store) {
        s = encode_f32_out(&tm_y, y, M, N, ldy);
        if (s != MX_OK) return s;
    }
    s = smem_attr_once(d.tc8_attr_set, mx::gemm_tc8_kernel, (int)Cfg::SMEM_BYTES);
    if (s != MX_OK) return s;
    mx::TcParams p{};
    p.y = y;
    p.bias = bias;
    p.ldy = ldy;
    p.M = (int)M;
    p.N = (int)N;
    p.K = (int)K;
    p.tiles_m = (int)chunks_a;
    p.tiles_n = (int)chunks_w;
    p.status = d.status;
    p.tma_store = tma_store ? 1 : 0;
    p.batch = 1;
    const int64_t tiles64 = chunks_a * chunks_w;
    if (tiles64 > INT32_MAX / 2) return MX_ERR_SHAPE;
    const int grid = tiles64 < d.sm_count ? (int)tiles64 : d.sm_count;
    ProfScope prof(KIND_GEMM_TC, st);
    MX_CUDA(launch_dep(mx::gemm_tc8_kernel, dim3(grid), dim3(mx::TC_THREADS), Cfg::SMEM_BYTES, st, tm_a, tm_w, tm_y, p,
                       (const uint8_t *)sfa, (const uint8_t *)sfw, (int)chunks_a, (int)chunks_w));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

// ---- block-scaled product on records (mx_records.cuh, mx_gemm_rec.cuh) ------------------------------
struct RecLayout {
    int panels_a, panels_w, kblocks, kgroups;
    size_t a_elems, a_sf, a_sfw, a_flags, w_elems, w_sf, w_sfw, w_flags, bytes;      // offsets into the workspace, total size
};
int even_up(int v) { return (v + 1) & ~1; }
RecLayout rec_layout(int64_t M, int64_t N, int64_t K)
{
    RecLayout l;
    l.panels_a = (int)((M + mx::REC_ROWS - 1) / mx::REC_ROWS);
    l.panels_w = (int)((N + mx::REC_ROWS - 1) / mx::REC_ROWS);
    l.kblocks = (int)((K + mx::REC_K - 1) / mx::REC_K);
    l.kgroups = (l.kblocks + 3) / 4;
    size_t off = 0;
    auto take = [&](size_t n) { const size_t at = off; off += round256(n); return at; };
    const size_t pa = (size_t)l.panels_a, pw = (size_t)l.panels_w, kb = (size_t)l.kblocks, kg = (size_t)l.kgroups;
    const size_t sa = (size_t)even_up(l.panels_a), sw = (size_t)even_up(l.panels_w);
    l.a_elems = take(pa * kb * mx::REC_BYTES);
    l.a_sf = take(sa * kg * mx::REC_SF_BYTES);
    l.a_sfw = take(sa * kb * mx::REC_SFW_BYTES);
    l.a_flags = take(pa * kb * 16);
    l.w_elems = take(pw * kb * mx::REC_BYTES);
    l.w_sf = take(sw * kg * mx::REC_SF_BYTES);
    l.w_sfw = take(sw * kb * mx::REC_SFW_BYTES);
    l.w_flags = take(pw * kb * 16);
    l.bytes = off;
    return l;
}

// Calls that the block-scaled product can take: mantissas that E4M3 holds, container form on both sides, whole groups of 32
// along K, within the workspace the caller was told to bring.
bool rec_fits(const mx_format_t &fa, const mx_format_t &fw, int64_t M, int64_t N, int64_t K)
{
    if (fa.elem_bits > 5 || fw.elem_bits > 5 || fa.packing || fw.packing || (K % 32) != 0) return false;
    const RecLayout l = rec_layout(M, N, K);
    if ((int64_t)l.panels_a * l.kblocks * 16 > INT32_MAX / 2 || (int64_t)l.panels_w * l.kblocks * 16 > INT32_MAX / 2)
        return false;
    return l.bytes <= tc_workspace(M, N, K);
}

mx::RecOut rec_out(const RecLayout &l, uint8_t *ws, bool weights)
{
    mx::RecOut o;
    o.elems = ws + (weights ? l.w_elems : l.a_elems);
    o.sf = ws + (weights ? l.w_sf : l.a_sf);
    o.sf_wide = ws + (weights ? l.w_sfw : l.a_sfw);
    o.flags = ws + (weights ? l.w_flags : l.a_flags);
    o.panels = weights ? l.panels_w : l.panels_a;
    o.panels_sf = even_up(o.panels);
    o.kblocks = l.kblocks;
    return o;
}

mx::RecPacked rec_packed(const void *mant, const uint8_t *exps, const mx_format_t &f, int64_t rows, int64_t K)
{
    mx::RecPacked p;
    p.mant = static_cast<const uint8_t *>(mant); p.exps = exps;
    p.rows = rows; p.K = K;
    p.block = f.block; p.w = f.elem_bits; p.row_shift = f.block_rows == 2 ? 1 : 0;
    return p;
}

// `rows` rows of `words` (at most 256) 32-bit words, box of `box_rows` of them (contiguous in shared memory).
mx_status_t encode_words(CUtensorMap *tm, const void *base, int words, int64_t rows, int box_rows)
{
    mx_status_t s = ensure_encoder();
    if (s != MX_OK) return s;
    const MapKey key = std::make_tuple(4, base, rows, (int64_t)box_rows, (int64_t)words, (int64_t)0, (int64_t)0);
    if (cached_map(key, tm)) return MX_OK;
    const cuuint64_t dims[2] = {(cuuint64_t)words, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)words * 4};
    const cuuint32_t box[2] = {(cuuint32_t)words, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = g_encode_tiled(tm, CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, const_cast<void *>(base), dims, strides, box, estr,
                                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                      CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        snprintf(t_cuda_error, sizeof(t_cuda_error), "cuTensorMapEncodeTiled (records) failed (%d)", (int)r);
        return MX_ERR_CUDA;
    }
    remember_map(key, *tm);
    return MX_OK;
}

template <bool TAIL, bool QOUT>
mx_status_t launch_rec_as(const mx::RecMaps &tm, const mx::TcParams &p, const mx::RecParams &rp, int pairs, DeviceInfo &d, cudaStream_t st)
{
    using Cfg = mx::RecCfg;
    const mx_status_t s = smem_attr_once(d.rec_attr_set[(TAIL ? 2 : 0) + (QOUT ? 1 : 0)],
                                         mx::gemm_rec_kernel<TAIL, QOUT>, (int)Cfg::SMEM_BYTES);
    if (s != MX_OK) return s;
    ProfScope prof(KIND_GEMM_TC, st);
    MX_CUDA(launch_dep(mx::gemm_rec_kernel<TAIL, QOUT>, dim3(2 * pairs), dim3(Cfg::THREADS), Cfg::SMEM_BYTES, st, tm, p, rp));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

mx_status_t launch_rec(const RecLayout &l, uint8_t *ws, int64_t M, int64_t N, int64_t K, const float *bias,
                       float *y, int64_t ldy, const QuantizedOut *yq, DeviceInfo &d, cudaStream_t st, const EpiTail &et)
{
    mx::RecMaps tm;
    const int sa = even_up(l.panels_a), sw = even_up(l.panels_w);
    constexpr int SF_WORDS = (int)mx::REC_SF_BYTES / 4, SFW_WORDS = (int)mx::REC_SFW_BYTES / 4;
    const struct { CUtensorMap *map; size_t at; int words; int64_t rows; int box; } maps[] = {
        {&tm.a, l.a_elems, 256, (int64_t)l.panels_a * l.kblocks * 16, 16},
        {&tm.w, l.w_elems, 256, (int64_t)l.panels_w * l.kblocks * 16, 16},
        {&tm.sa, l.a_sf, SF_WORDS, (int64_t)sa * l.kgroups, 1},
        {&tm.sw, l.w_sf, SF_WORDS, (int64_t)sw * l.kgroups, 2},
        {&tm.sa_wide, l.a_sfw, SFW_WORDS, (int64_t)sa * l.kblocks, 1},
        {&tm.sw_wide, l.w_sfw, SFW_WORDS, (int64_t)sw * l.kblocks, 2},
    };
    for (const auto &m : maps) {
        const mx_status_t s = encode_words(m.map, ws + m.at, m.words, m.rows, m.box);
        if (s != MX_OK) return s;
    }
    mx::TcParams p{};
    p.y = y;
    p.bias = et.any() ? nullptr : bias;
    p.ex_bias = et.any() ? bias : nullptr;
    p.relu = et.relu;
    p.residual = et.residual;
    p.ldr = et.ldr;
    p.ldy = ldy;
    p.M = (int)M;
    p.N = (int)N;
    p.K = (int)K;
    p.tiles_m = (l.panels_a + 1) / 2;
    p.tiles_n = (l.panels_w + 1) / 2;
    p.status = d.status;
    p.frag_store = frag_store_ok(yq != nullptr, false, y, ldy, 0) ? 1 : 0;
    p.batch = 1;
    p.yq_mant = yq ? yq->mant : nullptr;
    p.yq_exp = yq ? yq->exps : nullptr;
    p.yq_nonfinite = yq ? yq->nonfinite : nullptr;
    p.yq_bits = yq ? yq->f.elem_bits : 0;
    p.yq_block = yq ? yq->f.block : 0;
    p.yq_rows2 = yq && yq->f.block_rows == 2 ? 1 : 0;
    const mx::RecParams rp{ws + l.a_flags, ws + l.w_flags, l.panels_a, l.panels_w, sa, sw};
    const int64_t tiles = (int64_t)p.tiles_m * p.tiles_n;
    if (tiles > INT32_MAX / 2) return MX_ERR_SHAPE;
    const int pairs = tiles < d.sm_count / 2 ? (int)tiles : d.sm_count / 2;
    const bool tail = et.any(), q = yq != nullptr;
    if (tail) return q ? launch_rec_as<true, true>(tm, p, rp, pairs, d, st) : launch_rec_as<true, false>(tm, p, rp, pairs, d, st);
    return q ? launch_rec_as<false, true>(tm, p, rp, pairs, d, st) : launch_rec_as<false, false>(tm, p, rp, pairs, d, st);
}

template <typename Job>
mx_status_t launch_rec_prep(void (*kernel)(Job), const Job &job, int64_t items, int threads, int kind, const DeviceInfo &d, cudaStream_t st)
{
    const int per_sm = resident_ctas(kernel) * (256 / threads);
    ProfScope prof(kind, st);
    MX_CUDA(launch_dep(kernel, dim3((unsigned)grid_for(items, threads / 32, d.sm_count, per_sm)), dim3((unsigned)threads), 0, st, job));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

// A layer on records: activations quantized and weights re-laid in one launch, then the product.
mx_status_t run_rec_linear(const mx_linear_args_t &a, const float *bias, float *y, int64_t ldy, const QuantizedOut *yq,
                           uint8_t *ws, DeviceInfo &d, cudaStream_t st, const EpiTail &et)
{
    const RecLayout l = rec_layout(a.M, a.N, a.K);
    mx::RecPrepJob job;
    job.x = a.x; job.M = a.M; job.K = a.K; job.ldx = a.ldx;
    job.wa = a.fa.elem_bits; job.block = a.fa.block; job.a_rows2 = a.fa.block_rows == 2 ? 1 : 0;
    job.a = rec_out(l, ws, false);
    job.pw = rec_packed(a.w_mant, a.w_exp, a.fw, a.N, a.K);
    job.w = rec_out(l, ws, true);
    typedef __nv_bfloat16 bf16;
    static void (*const kernels[2][2])(mx::RecPrepJob) = {         // [fp32][nibble weights]
        {mx::rec_prep_kernel<bf16, false>, mx::rec_prep_kernel<bf16, true>},
        {mx::rec_prep_kernel<float, false>, mx::rec_prep_kernel<float, true>}};
    const int64_t items = (int64_t)l.panels_a * 16 * l.kblocks + (int64_t)l.panels_w * 16 * ((l.kblocks + 1) / 2);
    const mx_status_t s = launch_rec_prep(kernels[a.dt == MX_F32][a.fw.elem_bits <= 4], job, items, 128, KIND_PREP, d, st);
    if (s != MX_OK) return s;
    return launch_rec(l, ws, a.M, a.N, a.K, bias, y, ldy, yq, d, st, et);
}

// A product of two packed operands on records.
mx_status_t run_rec_gemm(const void *a_mant, const uint8_t *a_exp, const mx_format_t &fa, const void *w_mant,
                         const uint8_t *w_exp, const mx_format_t &fw, int64_t M, int64_t N, int64_t K, const float *bias,
                         float *y, int64_t ldy, const QuantizedOut *yq, uint8_t *ws, DeviceInfo &d, cudaStream_t st,
                         const EpiTail &et)
{
    const RecLayout l = rec_layout(M, N, K);
    mx::RecPairJob j;
    j.pa = rec_packed(a_mant, a_exp, fa, M, K);
    j.pw = rec_packed(w_mant, w_exp, fw, N, K);
    j.a = rec_out(l, ws, false);
    j.w = rec_out(l, ws, true);
    static void (*const kernels[2][2])(mx::RecPairJob) = {         // [nibble A][nibble W]
        {mx::rec_pair_kernel<false, false>, mx::rec_pair_kernel<false, true>},
        {mx::rec_pair_kernel<true, false>, mx::rec_pair_kernel<true, true>}};
    const int64_t items = (int64_t)(l.panels_a + l.panels_w) * 16 * ((l.kblocks + 1) / 2);
    const mx_status_t s = launch_rec_prep(kernels[fa.elem_bits <= 4][fw.elem_bits <= 4], j, items, 256, KIND_DEQUANTIZE, d, st);
    if (s != MX_OK) return s;
    return launch_rec(l, ws, M, N, K, bias, y, ldy, yq, d, st, et);
}

bool wide_tile(int64_t M, int64_t N, const DeviceInfo &d)
{
    const int64_t tiles256 = ((M + 127) / 128) * ((N + 255) / 256);
    return tiles256 >= (int64_t)d.sm_count * 3 / 4;
}

// Clusters of `split` CTAs of the split-K kernel that are resident at once (a cluster does not cross a GPC: 48 clusters of
// three do not fit on 148 SMs); looked up once.
mx_status_t splitk_clusters(DeviceInfo &d, int split, int *out)
{
    std::lock_guard<std::mutex> lk(g_init_mu);
    int &known = d.splitk_clusters[split];
    if (known < 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(split * d.sm_count));
        cfg.blockDim = dim3(mx::SplitKCfg::THREADS);
        cfg.dynamicSmemBytes = mx::SplitKCfg::SMEM_BYTES;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)split;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        MX_CUDA(cudaFuncSetAttribute(mx::gemm_splitk_kernel<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mx::SplitKCfg::SMEM_BYTES));
        int n = 0;
        MX_CUDA(cudaOccupancyMaxActiveClusters(&n, mx::gemm_splitk_kernel<false, false>, &cfg));
        known = n;
    }
    *out = known;
    return MX_OK;
}

// Few tiles, long reduction: into how many pieces K is cut over a cluster (see mx_gemm_splitk.cuh); 0 for the one-CTA
// kernels.  The most pieces whose clusters all fit at once, where the K steps that a CTA is spared are worth the two
// cluster barriers and the exchange (about 2.5 us against 0.2 us per step: at least 12 steps spared).  Whole calls, split /
// not (us): 352 x 2048 x 8192 in two 34.4 / 51.5, 352 x 2048 x 2048 14.7 / 17.3, 64 x 768 x 3072 in four 12.7 / 20.2,
// 512 x 1024 x 4096 18.4 / 27.5, 200 x 1024 x 1024 10.7 / 11.2; but 352 x 2048 x 1024 in two 13.2 / 12.2 and
// 128 x 768 x 768 in four 10.9 / 10.2.  More than 64 CTAs take longer to exchange and need 16 steps spared: at 12 and 14 the
// cut of 17 to 33 tiles in four is 0.5 us slower to 1.2 us slower (42 x 4096 x 1024, 42 x 3872 x 1024), at 18 it is 1 to 2 us
// faster, of 48 to 72 tiles in two within 0.3 us at 12 and 1 to 2 us faster at 16.
mx_status_t splitk_ways(int64_t M, int64_t N, int64_t K, DeviceInfo &d, int *out)
{
    *out = 0;
    const int64_t tiles = ((M + mx::TC_BM - 1) / mx::TC_BM) * ((N + mx::SplitKCfg::BN - 1) / mx::SplitKCfg::BN);
    const int64_t kblocks = (K + mx::TC_BK - 1) / mx::TC_BK;
    for (int s = mx::SplitKCfg::MAX_SPLIT; s > 1 && !*out; --s) {
        const int64_t spared = tiles * s > 64 ? 16 : 12;
        if (tiles * s > d.sm_count || kblocks * (s - 1) < spared * s) continue;
        int fit = 0;
        const mx_status_t st = splitk_clusters(d, s, &fit);
        if (st != MX_OK) return st;
        if (tiles <= fit) *out = s;
    }
    return MX_OK;
}

// Whether the block-scaled product is the faster one where it fits.  Measured on 550 shapes (1 to 4096 tokens, N 256 to
// 16384, K 512 to 16384; 4-bit, block 16, device time of whole calls, us, records / bf16):
// - Where run_tc would cut K, a pair tile's 0.36 us per 128 of K, one tile after another, stand against the split's 0.2 us
//   per 64 of a piece and its exchange, and against its operand form, which is twice as large.  The estimate below picks the
//   faster side but for 4 % at most: 1 x 256 x 16384 55.5 / 27.3, 64 x 768 x 3072 18.1 / 12.9, 352 x 2048 x 8192 40.2 / 37.6,
//   but 16 x 8192 x 8192 56.2 / 60.0 and 128 x 8192 x 16384 113 / 118.  (0.28 and 0.15 us since whole warps issue: the ratio, and
//   the line, are the same.  Over 280 shapes of 17 to 1237 rows measured since, the side taken is 0.5 % off the faster one on average.)
// - Otherwise records win from K = 2048 on (352 x 4096 x 4096 29.1 / 33.6, 768 x 2048 x 2048 19.1 / 19.3), and below that
//   where the operands are large enough to pay for the pair tile's longer start and drain: 4096 x 2048 x 768 20.8 / 22.1,
//   24 x 8192 x 512 11.7 / 12.5, but 1024 x 4096 x 768 15.9 / 14.7, 512 x 2048 x 1024 13.5 / 12.9.  Around the line the two
//   differ by up to 12 % either way (128 x 12288 x 768 16.7 / 14.8); short rows of wide layers are left on the slower side (448 x
//   9536 x 256 11.8 / 17.3: their pass deals an item per row).
mx_status_t rec_is_faster(int64_t M, int64_t N, int64_t K, DeviceInfo &d, bool *out)
{
    int split = 0;
    const mx_status_t s = splitk_ways(M, N, K, d, &split);
    if (s != MX_OK) return s;
    const int64_t operands = (M + N) * K;
    if (split) {
        const int64_t rec_ns = 360 * ((K + mx::REC_K - 1) / mx::REC_K);
        const int64_t steps = ((K + mx::TC_BK - 1) / mx::TC_BK + split - 1) / split;
        *out = rec_ns < 200 * steps + 1000 + operands * 17 / 100000;
    } else {
        *out = K >= 2048 || operands >= (4 << 20);
    }
    return MX_OK;
}

mx_status_t launch_splitk(const __nv_bfloat16 *a_hat, const __nv_bfloat16 *w_hat, int64_t M, int64_t N, int64_t K, int split,
                          const float *bias, float *y, int64_t ldy, const QuantizedOut *yq, DeviceInfo &d, cudaStream_t st,
                          const EpiTail &et)
{
    using Cfg = mx::SplitKCfg;
    CUtensorMap tm_a, tm_w;
    mx_status_t s = encode_bf16_rows(&tm_a, a_hat, M, K, mx::TC_BM);
    if (s != MX_OK) return s;
    s = encode_bf16_rows(&tm_w, w_hat, N, K, Cfg::BN);
    if (s != MX_OK) return s;
    const bool tail = et.any(), q = yq != nullptr;
    typedef void (*Kernel)(CUtensorMap, CUtensorMap, mx::TcParams, int);
    static const Kernel kernels[4] = {mx::gemm_splitk_kernel<false, false>, mx::gemm_splitk_kernel<false, true>,
                                      mx::gemm_splitk_kernel<true, false>, mx::gemm_splitk_kernel<true, true>};
    const int which = (tail ? 2 : 0) + (q ? 1 : 0);
    s = smem_attr_once(d.splitk_attr_set[which], kernels[which], (int)Cfg::SMEM_BYTES);
    if (s != MX_OK) return s;
    mx::TcParams p{};
    p.y = y;
    p.bias = tail ? nullptr : bias;
    p.ex_bias = tail ? bias : nullptr;
    p.relu = et.relu;
    p.residual = et.residual;
    p.ldr = et.ldr;
    p.ldy = ldy;
    p.M = (int)M;
    p.N = (int)N;
    p.K = (int)K;
    p.tiles_m = (int)((M + mx::TC_BM - 1) / mx::TC_BM);
    p.tiles_n = (int)((N + Cfg::BN - 1) / Cfg::BN);
    p.status = d.status;
    p.batch = 1;
    p.yq_mant = yq ? yq->mant : nullptr;
    p.yq_exp = yq ? yq->exps : nullptr;
    p.yq_nonfinite = yq ? yq->nonfinite : nullptr;
    p.yq_bits = yq ? yq->f.elem_bits : 0;
    p.yq_block = yq ? yq->f.block : 0;
    p.yq_rows2 = yq && yq->f.block_rows == 2 ? 1 : 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(p.tiles_m * p.tiles_n * split));
    cfg.blockDim = dim3(Cfg::THREADS);
    cfg.dynamicSmemBytes = Cfg::SMEM_BYTES;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)split;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g_prof.on ? 1 : 2;                     // see launch_dep
    ProfScope prof(KIND_GEMM_TC, st);
    MX_CUDA(cudaLaunchKernelEx(&cfg, kernels[which], tm_a, tm_w, p, split));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

// Width of the pair tiles where one wider than 256 columns fills the chip's pairs in so many fewer rounds that it is the faster
// one, else 0.  A round of 256 x 256 tiles takes about 5.8 ns per k, its epilogue under the next round's MMAs; a wide one takes
// 0.9 of that per column -- no less than for 384 columns, whose A operand alone keeps the loads busy -- and its epilogue is
// exposed.  Products, 256 / wide (us): 512 x 11008 x 4096 61.1 / 45.0 (320: 70 tiles on 74 pairs for 86 in two rounds),
// 2048 x 4096 x 16384 177 / 165 (480: 72 for 128), 4096 x 4096 x 11008 259 / 227, 384 x 16384 x 8192 102 / 89 (by name: AUTO decodes these
// weights in the product), 768 x 8192 x 2048
// 33.2 / 29.6; even or worse, and left alone: 2048 x 4096 x 4096 54.4 / 54.7, 2048 x 12288 x 4096 141 / 145,
// 4096 x 11008 x 4096 228 / 258 (five exposed epilogues of 38 MB).
int wide_pair_tile(int64_t M, int64_t N, int64_t K, const DeviceInfo &d)
{
    const int64_t rows = (M + 255) / 256, pairs = d.sm_count / 2;
    auto rounds = [&](int64_t w) { return (rows * ((N + w - 1) / w) + pairs - 1) / pairs; };
    const int64_t tile_ns = K * 29 / 5;
    int64_t best = (6000 + rounds(256) * tile_ns) * 93 / 100;
    int width = 0;
    for (int w = 288; w <= mx::TcwCfg::MAX_W; w += 32) {
        const int64_t ns = 2000 + rounds(w) * (tile_ns * (w > 384 ? w : 384) * 9 / 2560 + w * 75 / 4);
        if (ns < best) {
            best = ns;
            width = w;
        }
    }
    return width;
}

// Width of the pair tiles that fill one round, where the tiles of one CTA would fill one too, else 0.  An SM takes in 58 bytes per
// clock, and a 128 x 256 tile of one CTA needs 48 KB per K step of 64, half a 256 x W pair tile (128 + W / 2) * 128 bytes: from 160 to
// 224 columns the pair tiles are the faster ones by 5 to 15 %.  Whole calls (us): 1237 x 2048 x 2048 (M x K x N) 21.2 / 18.2, 1024 x 2048
// x 3002 23.1 / 20.6, 1536 x 4096 x 2048 37.0 / 33.1, 768 x 4096 x 4096 37.5 / 33.4, 512 x 2048 x 6144 25.3 / 22.3.  Narrower ones are as
// many as the 128 x 128 tiles and gain nothing (1024 x 2048 x 2048, 128 columns, 16.1 / 16.9), 256 columns neither (24.1 / 24.6).
// Not where tiles of 128 x 128 make one wave, which need 32 KB per step (19.6 / 22.1 at 384 x 2048 x 6144, 31.8 / 35.6 at 384 x 4096 x
// 6144, 35.3 / 38.1 at 384 x 5120 x 5120), and not for fewer than five K steps, whose results leave in one burst at the end (640 x 256 x
// 4096 12.4 / 13.6, 300 x 96 x 6464 17.0 / 23.8; of 300 shapes from K = 320 on none is more than 4 % slower), four of 160 columns
// (2048 x 256 x 1408 11.5 / 10.0).  Behind a pass that decodes both operands only from
// K = 512 on (of 224 shapes none slower by more than 1 %; 1490 x 256 x 1632 12.6 / 14.8, 1099 x 320 x 2240 12.4 / 14.2, 582 x 384 x 4160
// 13.0 / 13.6).
int one_round_width(int64_t M, int64_t N, int64_t K, const DeviceInfo &d)
{
    const int64_t rows = (M + 255) / 256, cols = d.sm_count / 2 / rows;
    if (!cols) return 0;
    const int64_t w = ((N + cols - 1) / cols + 31) / 32 * 32;
    return w >= 160 && w <= (K < 320 ? 160 : 224) ? (int)w : 0;
}

// Which product on bf16 operands a call takes (`count` products of one shape in one launch).  may_split: K may be cut (the sum is
// then not one chain).
// One wave of the smallest tile that gives one: a wave of 128 x 256 tiles takes 1.1 to 1.2 times as long as one of
// 128 x 128, not twice (352 x 8192 x 2048, 192 or 96 tiles: 33.3 against 25.7 us per call; 352 x 6144 x 2048, 144 or 72:
// 22.9 against 24.4).  Beyond that CTA pairs (a third less shared-memory traffic per flop: 512 x 11008 x 4096 74.3 against
// 83.3 us, +14 % on 8192^3), but a ragged half pair is not worth a second wave (300 x 12288 x 4096: 144 tiles of
// 128 x 256 62.1, 96 pair tiles 75.0).  Pairs also for one nearly full wave of long tiles (2048 x 2048 x 8192 product
// 49.5 against 56.5 us); a short single wave starts faster on the one-CTA kernel (2048^3 call 23.8 against 24.7).
enum TcKernel { TC_ONE = 5, TC_PAIR = 6, TC_PAIR_WIDE = 7, TC_CUT = 4 };     // (numbers: mx_selftest_route)
struct TcRoute { TcKernel kernel; int width, split; };                      // columns of a tile; pieces of K

// packed: the pass in front decodes both operands (launch_dequant_pair).
mx_status_t tc_route(int64_t M, int64_t N, int64_t K, int count, bool may_split, DeviceInfo &d, TcRoute *out, bool packed = false)
{
    const int64_t panels = (M + 127) / 128;
    const int64_t pair_tiles = ((M + 255) / 256) * ((N + 255) / 256);
    const int64_t tiles128 = panels * ((N + 127) / 128) * count, tiles256 = panels * ((N + 255) / 256) * count;
    const int pairs = d.sm_count / 2;
    const bool long_wave = K >= 4096 && pair_tiles <= pairs && 4 * pair_tiles >= 3 * pairs && (panels & 1) == 0;
    *out = {TC_ONE, N > 128 && tiles128 > d.sm_count ? 256 : 128, 1};
    if (count > 1) return MX_OK;
    if (M > 128 && (tiles256 > d.sm_count || long_wave)) {
        const int width = wide_pair_tile(M, N, K, d);
        *out = {width ? TC_PAIR_WIDE : TC_PAIR, width ? width : 256, 1};
        return MX_OK;
    }
    const int width = M > 128 && K >= (packed ? 512 : 256) && tiles128 > d.sm_count ? one_round_width(M, N, K, d) : 0;
    if (width) {
        *out = {TC_PAIR_WIDE, width, 1};
        return MX_OK;
    }
    int split = 0;
    const mx_status_t s = may_split ? splitk_ways(M, N, K, d, &split) : MX_OK;
    if (s == MX_OK && split) *out = {TC_CUT, 128, split};
    return s;
}

// Pre-decoded bf16 weights (both operands fetched by TMA).
mx_status_t run_tc(const __nv_bfloat16 *a_hat, const __nv_bfloat16 *w_hat, int64_t M, int64_t N,
                   int64_t K, const float *bias, float *y, int64_t ldy, DeviceInfo &d, cudaStream_t st,
                   const QuantizedOut *yq = nullptr, const TcBatch &tb = TcBatch(), const EpiTail &et = EpiTail(), bool may_split = true, bool packed = false)
{
    const PackedW none;
    TcRoute r;
    const mx_status_t s = tc_route(M, N, K, tb.count, may_split, d, &r, packed);
    if (s != MX_OK) return s;
    if (r.kernel == TC_PAIR_WIDE) return launch_tcw(a_hat, w_hat, M, N, K, r.width, bias, y, ldy, yq, d, st, et);
    if (r.kernel == TC_PAIR) return launch_tc2(a_hat, w_hat, M, N, K, bias, y, ldy, yq, d, st, et);
    if (r.kernel == TC_CUT) return launch_splitk(a_hat, w_hat, M, N, K, r.split, bias, y, ldy, yq, d, st, et);
    if (r.width == 256) return launch_tc<256, mx::W_BF16>(a_hat, w_hat, none, M, N, K, bias, y, ldy, yq, d, st, tb, et);
    return launch_tc<128, mx::W_BF16>(a_hat, w_hat, none, M, N, K, bias, y, ldy, yq, d, st, tb, et);
}

// Packed weights decoded inside the kernel.
mx_status_t run_tc_fused(const __nv_bfloat16 *a_hat, const void *w_mant, const uint8_t *w_exp,
                         const mx_format_t &fw, int64_t M, int64_t N, int64_t K, const float *bias,
                         float *y, int64_t ldy, DeviceInfo &d, cudaStream_t st, bool perm_a = false)
{
    PackedW pw;
    pw.mant = static_cast<const uint8_t *>(w_mant);
    pw.exps = w_exp;
    pw.bits = fw.elem_bits;
    pw.block = fw.block;
    const bool wide = wide_tile(M, N, d);
    if (perm_a) {                       // a_hat was written in the permuted K order: nibbles, K % 64 == 0
        if (wide) return launch_tc<256, mx::W_NIBBLE_PERM>(a_hat, nullptr, pw, M, N, K, bias, y, ldy, nullptr, d, st);
        return launch_tc<128, mx::W_NIBBLE_PERM>(a_hat, nullptr, pw, M, N, K, bias, y, ldy, nullptr, d, st);
    }
    if (fw.elem_bits <= 4) {
        if (wide) return launch_tc<256, mx::W_NIBBLE>(a_hat, nullptr, pw, M, N, K, bias, y, ldy, nullptr, d, st);
        return launch_tc<128, mx::W_NIBBLE>(a_hat, nullptr, pw, M, N, K, bias, y, ldy, nullptr, d, st);
    }
    if (wide) return launch_tc<256, mx::W_INT8>(a_hat, nullptr, pw, M, N, K, bias, y, ldy, nullptr, d, st);
    return launch_tc<128, mx::W_INT8>(a_hat, nullptr, pw, M, N, K, bias, y, ldy, nullptr, d, st);
}

// The fused kernels read weight rows with 16-byte loads and exponent pairs with 2-byte loads.
bool fused_ok(int64_t K, const uint8_t *w_exp)
{
    return (K % 32) == 0 && (reinterpret_cast<uintptr_t>(w_exp) & 1u) == 0;
}

size_t tc_operand_bytes(int64_t M, int64_t N, int64_t K)
{
    return round256((size_t)M * K * 2) + round256((size_t)N * K * 2);
}
size_t tc_workspace(int64_t M, int64_t N, int64_t K) { return tc_operand_bytes(M, N, K); }

size_t fused_workspace(int64_t M, int64_t K) { return round256((size_t)M * K * 2); }
size_t packed_workspace(int64_t M, int64_t K, const mx_format_t &fa)
{
    return round256(mx_mant_bytes(M, K, fa)) + round256(mx_exp_bytes(M, K, fa));
}

mx_status_t check_gemm_args(const void *a, const void *a_exp, const mx_format_t &fa, const void *w,
                            const void *w_exp, const mx_format_t &fw, int64_t M, int64_t N, int64_t K,
                            const float *bias, const float *y, int64_t ldy)
{
    if (!a || !w || !w_exp || !y) return MX_ERR_NULL;
    (void)a_exp;
    if (!format_ok_any(fa) || !format_ok_any(fw) || fa.block != fw.block) return MX_ERR_FORMAT;
    if (M <= 0 || N <= 0 || K <= 0 || (K % fa.block) != 0 || ldy < N) return MX_ERR_SHAPE;
    if ((M % fa.block_rows) != 0 || (N % fw.block_rows) != 0) return MX_ERR_SHAPE;     // whole two-row blocks
    if (M > INT32_MAX / 2 || N > INT32_MAX / 2 || K > INT32_MAX / 2) return MX_ERR_SHAPE;
    if (!aligned16(a) || !aligned16(w) || !aligned16(y) || (bias && !aligned16(bias))) return MX_ERR_ALIGN;
    return MX_OK;
}

// ---- decode: few tokens, weights streamed once ------------------------------------------------
// Tensor maps over packed weight matrices are cached: weights are static, so after the first
// call a layer costs a map lookup instead of a driver call.
struct WeightMaps { CUtensorMap mant, exps; };
std::map<std::tuple<const void *, const void *, int64_t, int64_t>, WeightMaps> g_wmap_cache;
std::mutex g_wmap_mu;

mx_status_t encode_u8_rows(CUtensorMap *out, const void *base, int64_t rows, int64_t row_bytes, int box_bytes,
                           CUtensorMapSwizzle swz)
{
    const cuuint64_t dims[2] = {(cuuint64_t)row_bytes, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)row_bytes};
    const cuuint32_t box[2] = {(cuuint32_t)box_bytes, 16};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = g_encode_tiled(out, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void *>(base), dims, strides,
                                      box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
                                      CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        snprintf(t_cuda_error, sizeof(t_cuda_error), "cuTensorMapEncodeTiled (packed weights) failed (%d)", (int)r);
        return MX_ERR_CUDA;
    }
    return MX_OK;
}

// out2[0]: over the packed mantissas (rows of row_bytes); out2[1], when nb is not 0: over the exponent bytes (rows of nb).
// (the caller holds g_wmap_mu)
mx_status_t packed_weight_maps(const void *w_mant, const void *w_exp, int64_t N, int64_t row_bytes, int64_t nb, CUtensorMap *out2)
{
    const auto key = std::make_tuple(w_mant, nb ? w_exp : nullptr, N, row_bytes);
    auto it = g_wmap_cache.find(key);
    if (it == g_wmap_cache.end()) {
        const mx_status_t es = ensure_encoder();
        if (es != MX_OK) return es;
        WeightMaps wm{};
        mx_status_t s = encode_u8_rows(&wm.mant, w_mant, N, row_bytes, 128, CU_TENSOR_MAP_SWIZZLE_128B);
        if (s != MX_OK) return s;
        if (nb) s = encode_u8_rows(&wm.exps, w_exp, N, nb, 16, CU_TENSOR_MAP_SWIZZLE_NONE);
        if (s != MX_OK) return s;
        out2[0] = wm.mant;
        if (nb) out2[1] = wm.exps;
        try {                            // without host memory for the entry they are encoded again next time
            if (g_wmap_cache.size() > 4096) g_wmap_cache.clear();
            g_wmap_cache.emplace(key, wm);
        } catch (const std::bad_alloc &) {
        }
        return MX_OK;
    }
    out2[0] = it->second.mant;
    if (nb) out2[1] = it->second.exps;
    return MX_OK;
}

size_t stream_table_bytes(int32_t n_layers)
{
    return round256((size_t)n_layers * sizeof(mx::StreamLayer)) + round256((size_t)n_layers * 2 * sizeof(CUtensorMap)) +
           round256((size_t)n_layers * sizeof(mx::QuantJob));
}

bool stream_layer_ok(const mx_linear_args_t &a)
{
    return a.M >= 1 && a.M <= 16 && a.fw.block == 32 && a.fa.block == 32 && a.fw.elem_bits <= 4 &&
           (a.K % 128) == 0 && a.fa.packing == 0 && a.fw.packing == 0;
}

size_t stream_act_bytes(const mx_linear_args_t &a)
{
    return round256(mx_mant_bytes(a.M, a.K, a.fa)) + round256(mx_exp_bytes(a.M, a.K, a.fa));
}

bool same_activation(const mx_linear_args_t &a, const mx_linear_args_t &b)
{
    return a.x == b.x && a.dt == b.dt && a.M == b.M && a.K == b.K && a.ldx == b.ldx &&
           a.fa.block == b.fa.block && a.fa.elem_bits == b.fa.elem_bits && a.fa.block_rows == b.fa.block_rows;
}

// owner[i]: the first layer with layer i's activation.  Layers that share one usually follow each other.
void activation_owners(const mx_linear_args_t *layers, int32_t n, std::vector<int> &owner)
{
    owner.resize((size_t)n);
    std::multimap<const void *, int> firsts;
    for (int i = 0; i < n; ++i) {
        owner[i] = i;
        if (i > 0 && same_activation(layers[i], layers[owner[i - 1]])) {
            owner[i] = owner[i - 1];
            continue;
        }
        const auto range = firsts.equal_range(layers[i].x);
        for (auto it = range.first; it != range.second && owner[i] == i; ++it)
            if (same_activation(layers[i], layers[it->second])) owner[i] = it->second;
        if (owner[i] == i) firsts.emplace(layers[i].x, i);
    }
}

size_t grouped_workspace(const mx_linear_args_t *layers, int32_t n, const std::vector<int> &owner)
{
    size_t total = stream_table_bytes(n);
    for (int i = 0; i < n; ++i)
        if (owner[i] == i) total += stream_act_bytes(layers[i]);
    return total;
}

template <int NT, typename Params>
mx_status_t launch_stream_as(const Params &sp, size_t smem, int grid, DeviceInfo &d, cudaStream_t st)
{
    constexpr bool INLINE = std::is_same<Params, mx::StreamInlineParams>::value;
    const mx_status_t as = smem_attr_once(d.stream_attr_set[INLINE ? 1 : 0][NT - 1], mx::gemv_stream_kernel<NT, Params>, 227 * 1024);
    if (as != MX_OK) return as;
    ProfScope prof(KIND_GEMM_STREAM, st);
    MX_CUDA(launch_dep(mx::gemv_stream_kernel<NT, Params>, dim3(grid), dim3(mx::StreamCfg<NT>::THREADS), smem, st, sp));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

template <int NT, typename Params>
mx_status_t launch_mma_as(const Params &sp, int warps, int stages, int early, size_t smem, int grid, DeviceInfo &d, cudaStream_t st)
{
    constexpr bool INLINE = std::is_same<Params, mx::StreamInlineParams>::value;
    const mx_status_t as = smem_attr_once(d.mma_attr_set[INLINE ? 1 : 0][NT - 1], mx::gemv_mma_kernel<NT, Params>, 227 * 1024);
    if (as != MX_OK) return as;
    ProfScope prof(KIND_GEMM_STREAM, st);
    MX_CUDA(launch_dep(mx::gemv_mma_kernel<NT, Params>, dim3(grid), dim3(32 * warps), smem, st, sp, stages, early));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

template <int TOK, typename Params>
mx_status_t launch_stream32_as(const Params &sp, int stages, int early, size_t smem, int grid, DeviceInfo &d, cudaStream_t st)
{
    constexpr bool INLINE = std::is_same<Params, mx::StreamInlineParams>::value;
    const mx_status_t as = smem_attr_once(d.stream32_attr_set[INLINE ? 1 : 0][TOK - 1], mx::gemv_stream32_kernel<TOK, Params>, 227 * 1024);
    if (as != MX_OK) return as;
    ProfScope prof(KIND_GEMM_STREAM, st);
    MX_CUDA(launch_dep(mx::gemv_stream32_kernel<TOK, Params>, dim3(grid), dim3(mx::Stream32Cfg<TOK>::THREADS), smem, st, sp, stages, early));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

// How a grouped call runs: one or two tokens a weight row per lane; else 16 rows per warp on the integer MMA, 16 warps or 8,
// whatever fits beside the tokens; else the register variant, which stages the tokens only.
struct StreamPlan {
    enum Kind { ROWS32, MMA, REGS } kind = REGS;
    int warps = 8, stages = 0, rows = 16, unit = 4;      // unit: blocks of 32 that a piece of a cut K is a multiple of
    size_t smem = 0;
};

template <typename Params>
mx_status_t launch_stream(const StreamPlan &sp, int tok, int early, const Params &p, int grid, DeviceInfo &d, cudaStream_t st)
{
    if (sp.kind == StreamPlan::ROWS32)
        return tok == 1 ? launch_stream32_as<1>(p, sp.stages, early, sp.smem, grid, d, st)
                        : launch_stream32_as<2>(p, sp.stages, early, sp.smem, grid, d, st);
    if (sp.kind == StreamPlan::MMA)
        return tok > 8 ? launch_mma_as<2>(p, sp.warps, sp.stages, early, sp.smem, grid, d, st)
                       : launch_mma_as<1>(p, sp.warps, sp.stages, early, sp.smem, grid, d, st);
    return tok > 8 ? launch_stream_as<2>(p, sp.smem, grid, d, st) : launch_stream_as<1>(p, sp.smem, grid, d, st);
}

// ---- one layer of few tokens in one launch (gemv_single_kernel) ----------------------------------------
// Whether the result is written over the activations (y = x in place, say).  Rows of one pitch: by their columns, so that two
// column ranges of one tensor are apart; else by the ranges of addresses, gaps between the rows included.
bool result_over_activations(const mx_linear_args_t &a)
{
    const int64_t size = a.dt == MX_F32 ? 4 : 2, px = a.ldx * size, py = a.ldy * 4, nx = a.K * size, ny = a.N * 4;
    const uintptr_t x0 = reinterpret_cast<uintptr_t>(a.x), y0 = reinterpret_cast<uintptr_t>(a.y);
    if (y0 >= x0 + (uintptr_t)((a.M - 1) * px + nx) || x0 >= y0 + (uintptr_t)((a.M - 1) * py + ny)) return false;
    if (px != py || a.M == 1) return true;
    const int64_t d = (int64_t)((y0 > x0 ? y0 - x0 : x0 - y0) % (uintptr_t)px), at = y0 > x0 || d == 0 ? d : px - d;
    return at < nx || at + ny > px;
}

// Container formats whose weight rows are whole 16-byte units (the TMA boxes), one-row activation blocks.  Its CTAs read the
// activations while others already write results, so those must not share memory; the routes with a pass over the activations
// in front allow it.
bool gemv_layer_ok(const mx_linear_args_t &a)
{
    const int64_t row_bytes = a.fw.elem_bits <= 4 ? a.K / 2 : a.K;
    return a.M >= 1 && a.M <= 32 && format_1d(a.fa) && format_ok(a.fw) && a.fa.block == a.fw.block && (row_bytes % 16) == 0 &&
           !result_over_activations(a);
}

struct GemvPlan { int cluster, rounds, stages, max_groups, exp_words; size_t smem; };

template <int NT, bool NIB, int BLOCK>
mx_status_t launch_gemv_as(int slot, const GemvPlan &g, const CUtensorMap &tm, const mx::GemvArgs &args, DeviceInfo &d, cudaStream_t st)
{
    const auto kernel = mx::gemv_single_kernel<NT, NIB, BLOCK>;
    const mx_status_t s = smem_attr_once(d.gemv_attr_set[slot], kernel, 227 * 1024);
    if (s != MX_OK) return s;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((args.row_groups + g.rounds - 1) / g.rounds * g.cluster));
    cfg.blockDim = dim3(mx::GemvCfg::THREADS);
    cfg.dynamicSmemBytes = g.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)g.cluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g_prof.on ? 1 : 2;                     // see launch_dep
    ProfScope prof(KIND_GEMM_STREAM, st);
    MX_CUDA(cudaLaunchKernelEx(&cfg, kernel, tm, args, g.stages));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

template <int NT, bool NIB, int BLOCK>
mx_status_t gemv_resident_as(int slot, int cluster, size_t smem, DeviceInfo &d, int *out)
{
    const auto kernel = mx::gemv_single_kernel<NT, NIB, BLOCK>;
    const mx_status_t s = smem_attr_once(d.gemv_attr_set[slot], kernel, 227 * 1024);
    if (s != MX_OK) return s;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(cluster * d.sm_count));
    cfg.blockDim = dim3(mx::GemvCfg::THREADS);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    MX_CUDA(cudaOccupancyMaxActiveClusters(out, kernel, &cfg));
    return MX_OK;
}

template <int NT, bool NIB, int BLOCK> size_t gemv_smem(const GemvPlan &g)
{
    return mx::GemvCfg::smem_bytes<NT, NIB, BLOCK>(g.max_groups, g.stages, g.rounds, g.cluster);
}
typedef mx_status_t (*GemvLaunch)(int, const GemvPlan &, const CUtensorMap &, const mx::GemvArgs &, DeviceInfo &, cudaStream_t);
struct GemvVariant {
    size_t (*smem)(const GemvPlan &);
    GemvLaunch launch;
    mx_status_t (*resident)(int, int, size_t, DeviceInfo &, int *);
};
#define MX_GEMV_ONE(NT, NIB, B) {gemv_smem<NT, NIB, B>, launch_gemv_as<NT, NIB, B>, gemv_resident_as<NT, NIB, B>}
#define MX_GEMV(NT) MX_GEMV_ONE(NT, false, 16), MX_GEMV_ONE(NT, false, 32), MX_GEMV_ONE(NT, true, 16), MX_GEMV_ONE(NT, true, 32)
const GemvVariant g_gemv[12] = {MX_GEMV(1), MX_GEMV(2), MX_GEMV(4)};      // nibbles, block 32: bits 1, 0
#undef MX_GEMV
#undef MX_GEMV_ONE
int gemv_slot(const mx_linear_args_t &a)
{
    const int nt = a.M <= 8 ? 0 : a.M <= 16 ? 1 : 2;
    return 4 * nt + (a.fw.elem_bits <= 4 ? 2 : 0) + (a.fw.block == 32 ? 1 : 0);
}

// Clusters of `cluster` CTAs that are resident at once; asked once per kernel, cluster size and number of CTAs that fit an SM.
mx_status_t gemv_resident(int slot, int cluster, bool two, DeviceInfo &d, int64_t *out)
{
    int log2c = 0;
    while ((1 << log2c) < cluster) ++log2c;
    int known;
    {
        std::lock_guard<std::mutex> lk(g_init_mu);
        known = d.gemv_clusters[slot][log2c][two];
    }
    if (known == 0) {
        // (asked with the most shared memory of the class)
        const mx_status_t s = g_gemv[slot].resident(slot, cluster, two ? 112u * 1024u : 227u * 1024u, d, &known);
        if (s != MX_OK) return s;
        std::lock_guard<std::mutex> lk(g_init_mu);
        d.gemv_clusters[slot][log2c][two] = known;
    }
    *out = known;
    return MX_OK;
}

// The cut of K depends on N and K alone, so among the calls that come here a token's bits do not depend on how many others share
// it (one or two tokens of a large layer of 4-bit weights in blocks of 32 go elsewhere: see grouped_impl).  Where the row groups
// alone fill the chip twice over K is not cut (one chain of ascending blocks); else it is cut as often as a cluster allows while
// the slices are whole steps or the CTAs fit at once (a step fetches 256 bytes of a row whatever its slice needs: 512 x 16384,
// 8 bits, in eight slices of 64 bytes 35 us).  A CTA then quantizes the smallest slice of the tokens and the most weight bytes
// are in flight.  Row groups beyond what is resident go to the same clusters, so that a staged slice is used again.
bool gemv_plan(const mx_linear_args_t &a, DeviceInfo &d, GemvPlan *out)
{
    if (!gemv_layer_ok(a)) return false;
    const bool nib = a.fw.elem_bits <= 4;
    const int64_t row_bytes = nib ? a.K / 2 : a.K, ng = (row_bytes + 63) / 64, groups = (a.N + mx::GemvCfg::ROWS - 1) / mx::GemvCfg::ROWS;
    if (ng > INT32_MAX / 64 || groups > INT32_MAX / 64) return false;
    const int slot = gemv_slot(a);
    GemvPlan g;
    g.cluster = 1;
    if (groups < 2 * d.sm_count)
        for (int c = 2; c <= mx::GemvCfg::MAX_CLUSTER && c <= ng && (groups * c <= 2 * d.sm_count || ng / c >= 4); c *= 2) g.cluster = c;
    g.max_groups = 0;
    const int gb = (nib ? 128 : 64) / a.fw.block;
    bool words = ((a.K / a.fw.block) % 4) == 0 && (reinterpret_cast<uintptr_t>(a.w_exp) & 3u) == 0;
    for (int r = 0; r < g.cluster; ++r) {
        const int lo = (int)(ng * r / g.cluster), hi = (int)(ng * (r + 1) / g.cluster);
        g.max_groups = hi - lo > g.max_groups ? hi - lo : g.max_groups;
        words = words && (lo * gb) % 4 == 0;
    }
    g.exp_words = words ? 1 : 0;
    // Two CTAs per SM where that leaves a stage, else one (32 x 8192 x 2048 at one CTA per SM: the clusters do not all fit, two
    // waves, 34 instead of 25 us).  Row groups beyond what is resident at once go to the same clusters, where a staged slice is
    // used again; the partial tiles of those rounds come before a third and second stage (5 x 4096 x 11008 with three stages and
    // three waves 19.5, two stages and three rounds 11.9).
    constexpr size_t HALF = 112u * 1024u, FULL = 227u * 1024u;
    const int steps = (g.max_groups + 3) / 4;
    for (const size_t cap : {HALF, FULL}) {
        g.stages = 1;
        g.rounds = 1;
        g.smem = g_gemv[slot].smem(g);
        if (g.smem > cap) continue;
        int64_t resident = 0;
        const mx_status_t s = gemv_resident(slot, g.cluster, cap == HALF, d, &resident);
        if (s != MX_OK || resident < 1) return false;
        const int64_t rounds = (groups + resident - 1) / resident;
        const int want = (int)(rounds < 8 ? rounds : 8);
        for (int st = 3; st >= 1; --st) {
            g.stages = st < steps * want ? st : steps * want;
            g.rounds = want;
            g.smem = g_gemv[slot].smem(g);
            for (; g.smem > cap && st == 1 && g.rounds > 1; g.smem = g_gemv[slot].smem(g)) --g.rounds;
            if (g.smem <= cap) break;
        }
        *out = g;
        return true;
    }
    return false;
}

// Up to 16 tokens always (operand pass and tensor-core product / this, us: 1 x 4096 x 4096 in blocks of 16 21.5 / 6.8,
// 16 x 16384 x 16384 in 8 bits 238 / 85, 1 x 768 x 768 9.8 / 4.4).  Up to 32 the arithmetic counts, two rescales per 32 k and
// token in blocks of 16: 32 x 4096 x 4096 20.2 / 17.3, 1024 x 1024 10.8 / 7.2, 640 x 5120 15.6 / 13.7, but 4096 x 11008
// 36.1 / 42.1 (three rounds of row groups) and 24 tokens of 8192 x 2048 in 8 bits 24.6 / 25.9; in blocks of 32 4096 x 11008
// 42.9 / 24.5, 8192 x 2048 24.3 / 19.8, 11008 x 4096 40.9 / 30.5.
bool gemv_is_faster(const mx_linear_args_t &a)
{
    return a.M <= 16 || (a.M <= 32 && (a.fw.block == 32 || (a.N * a.K <= (1 << 24) && a.K <= 6144)));
}

mx_status_t launch_gemv(const mx_linear_args_t &a, const GemvPlan &g, DeviceInfo &d, cudaStream_t st)
{
    CUtensorMap tm;
    const bool nib = a.fw.elem_bits <= 4;
    {
        std::lock_guard<std::mutex> lk(g_wmap_mu);
        const mx_status_t s = packed_weight_maps(a.w_mant, a.w_exp, a.N, nib ? a.K / 2 : a.K, 0, &tm);
        if (s != MX_OK) return s;
    }
    mx::GemvArgs p;
    p.x = a.x; p.ldx = a.ldx; p.w_exp = a.w_exp; p.bias = a.bias; p.y = a.y; p.ldy = a.ldy;
    p.T = (int)a.M; p.N = (int)a.N; p.K = (int)a.K;
    p.a_bits = a.fa.elem_bits; p.w_bits = a.fw.elem_bits; p.w_rows2 = a.fw.block_rows == 2 ? 1 : 0;
    p.rounds = g.rounds;
    p.row_groups = (int)((a.N + mx::GemvCfg::ROWS - 1) / mx::GemvCfg::ROWS);
    p.exp_words = g.exp_words;
    p.max_groups = g.max_groups;
    p.status = d.status;
    p.bf16 = a.dt == MX_BF16 ? 1 : 0;
    const int slot = gemv_slot(a);
    return g_gemv[slot].launch(slot, g, tm, p, d, st);
}

// ---- up to 384 rows: weights decoded inside the product (gemm_dec_kernel) --------------------------------
typedef void (*DecKernel)(CUtensorMap, CUtensorMap, mx::TcParams, mx::DecParams);
const DecKernel g_dec[12] = {                             // panels - 1, nibbles, MXInt result: 4 * , 2 * , 1 *
    mx::gemm_dec_kernel<1, false, false>, mx::gemm_dec_kernel<1, false, true>, mx::gemm_dec_kernel<1, true, false>, mx::gemm_dec_kernel<1, true, true>,
    mx::gemm_dec_kernel<2, false, false>, mx::gemm_dec_kernel<2, false, true>, mx::gemm_dec_kernel<2, true, false>, mx::gemm_dec_kernel<2, true, true>,
    mx::gemm_dec_kernel<3, false, false>, mx::gemm_dec_kernel<3, false, true>, mx::gemm_dec_kernel<3, true, false>, mx::gemm_dec_kernel<3, true, true>};

struct DecPlan { int which, panels, split, exp_words, tokens; };     // tokens: of gemm_tmw_kernel's tile, 0: gemm_dec_kernel

mx_status_t dec_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *attr, int panels, int grid, int split, cudaStream_t st)
{
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(mx::DecCfg::THREADS);
    cfg.dynamicSmemBytes = mx::DecCfg::smem_bytes(panels);
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)split;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return MX_OK;
}

bool dec_is_faster(int64_t M, int64_t N, int64_t K, int split, bool rec, int sm_count);

typedef void (*TmwKernel)(CUtensorMap, CUtensorMap, mx::TcParams, mx::TmwParams);
const TmwKernel g_tmw[8] = {                              // nibbles, MXInt result, K cut: 4 * , 2 * , 1 *
    mx::gemm_tmw_kernel<false, false, false>, mx::gemm_tmw_kernel<false, false, true>, mx::gemm_tmw_kernel<false, true, false>,
    mx::gemm_tmw_kernel<false, true, true>, mx::gemm_tmw_kernel<true, false, false>, mx::gemm_tmw_kernel<true, false, true>,
    mx::gemm_tmw_kernel<true, true, false>, mx::gemm_tmw_kernel<true, true, true>};

void tmw_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *attr, int split, int clusters, cudaStream_t st)
{
    cfg.gridDim = dim3((unsigned)(2 * split * clusters));
    cfg.blockDim = dim3(mx::TmwCfg::THREADS);
    cfg.dynamicSmemBytes = 227 * 1024;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)(2 * split);
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
}

// Clusters of 2 .. MAX_SPLIT pairs that are resident at once; looked up once.
mx_status_t tmw_clusters(DeviceInfo &d, int which, int (&out)[mx::TmwCfg::MAX_SPLIT + 1])
{
    const mx_status_t s = smem_attr_once(d.tmw_attr_set[which], g_tmw[which], 227 * 1024);
    if (s != MX_OK) return s;
    std::lock_guard<std::mutex> lk(g_init_mu);
    for (int split = 2; split <= mx::TmwCfg::MAX_SPLIT; ++split) {
        int &known = d.tmw_clusters[which][split];
        if (known == 0) {
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute attr[2];
            tmw_config(cfg, attr, split, d.sm_count, nullptr);
            MX_CUDA(cudaOccupancyMaxActiveClusters(&known, g_tmw[which], &cfg));
        }
        out[split] = known;
    }
    return MX_OK;
}

enum ExpRows { EXP_WIDE, EXP_WORDS, EXP_BYTES };            // exponent rows: see tmw_us
double tc_us(const TcRoute &r, int64_t M, int64_t N, int64_t K, bool quantized, int sm_count);
double rec_us(int64_t M, int64_t N, int64_t K, bool quantized, int sm_count);
double dec_us(int64_t M, int64_t N, int64_t K, int split, bool nib, bool words, bool quantized, int sm_count);
int tmw_tokens(int64_t M, int64_t N, int64_t K, bool nib, int block, ExpRows rows, bool quantized, double other, int sm_count, const int *clusters,
               int *pieces);

// Whether the product decodes its weights itself, in which kernel, and for gemm_dec_kernel into how many pieces K is cut: the most
// whose clusters all fit at once, of at least four K steps each.
mx_status_t dec_plan(int64_t M, int64_t N, int64_t K, const mx_format_t &fa, const mx_format_t &fw, const uint8_t *w_exp, bool quantized,
                     DeviceInfo &d, DecPlan *out, bool *use)
{
    *use = false;
    const bool nib = fw.elem_bits <= 4;
    const int64_t row_bytes = nib ? K / 2 : K, panels = (M + mx::TC_BM - 1) / mx::TC_BM, tiles = (N + mx::DecCfg::BN - 1) / mx::DecCfg::BN;
    if (!format_ok(fw) || (row_bytes % 16) != 0 || tiles > INT32_MAX / 16) return MX_OK;
    out->exp_words = ((K / fw.block) % 4) == 0 && (reinterpret_cast<uintptr_t>(w_exp) & 3u) == 0 ? 1 : 0;
    out->tokens = 0;
    bool rec = false;
    if (rec_fits(fa, fw, M, N, K)) {
        const mx_status_t rs = rec_is_faster(M, N, K, d, &rec);
        if (rs != MX_OK) return rs;
    }
    if (panels <= mx::DecCfg::MAX_P) {
        out->panels = (int)panels;
        out->which = 4 * ((int)panels - 1) + (nib ? 2 : 0) + (quantized ? 1 : 0);
        out->split = 1;
        const mx_status_t as = smem_attr_once(d.dec_attr_set[out->which], g_dec[out->which], 227 * 1024);
        if (as != MX_OK) return as;
        const int64_t kblocks = (K + mx::TC_BK - 1) / mx::TC_BK;
        for (int s = mx::DecCfg::MAX_SPLIT; s > 1 && out->split == 1; --s) {
            if (tiles * s > d.sm_count || kblocks < 4 * s) continue;
            std::lock_guard<std::mutex> lk(g_init_mu);
            int &known = d.dec_clusters[out->which][s];
            if (known == 0) {
                cudaLaunchConfig_t cfg = {};
                cudaLaunchAttribute attr[2];
                dec_config(cfg, attr, (int)panels, s * d.sm_count, s, nullptr);
                MX_CUDA(cudaOccupancyMaxActiveClusters(&known, g_dec[out->which], &cfg));
            }
            if (tiles <= known) out->split = s;
        }
        *use = dec_is_faster(M, N, K, out->split, rec, d.sm_count);
    }
    if (M > 1536) return MX_OK;                                          // (see tmw_tokens)
    double other = 0;                                                    // us of the route that is taken else
    if (*use) {
        other = dec_us(M, N, K, out->split, nib, out->exp_words != 0, quantized, d.sm_count);
    } else if (rec) {
        other = rec_us(M, N, K, quantized, d.sm_count);
    } else {
        TcRoute r;
        const mx_status_t ts = tc_route(M, N, K, 1, true, d, &r);
        if (ts != MX_OK) return ts;
        other = tc_us(r, M, N, K, quantized, d.sm_count);
    }
    const int which = (nib ? 4 : 0) + (quantized ? 2 : 0);
    int clusters[mx::TmwCfg::MAX_SPLIT + 1] = {}, pieces = 1;
    const mx_status_t cs = tmw_clusters(d, which + 1, clusters);
    if (cs != MX_OK) return cs;
    const bool pairs_of_words = (((uint64_t)(K / fw.block) | reinterpret_cast<uintptr_t>(w_exp)) & 7u) == 0;
    const ExpRows rows = !out->exp_words ? EXP_BYTES : pairs_of_words ? EXP_WIDE : EXP_WORDS;
    out->tokens = tmw_tokens(M, N, K, nib, fw.block, rows, quantized, other, d.sm_count, clusters, &pieces);
    if (out->tokens) {
        out->which = which + (pieces > 1 ? 1 : 0);
        out->split = pieces;
        *use = true;
    }
    return MX_OK;
}

mx_status_t launch_tmw(const DecPlan &g, const __nv_bfloat16 *a_hat, const void *w_mant, const mx_format_t &fw, mx::TcParams &p,
                       const uint8_t *w_exp, DeviceInfo &d, cudaStream_t st)
{
    using Cfg = mx::TmwCfg;
    const int T = g.tokens;
    CUtensorMap tm_x, tm_r;
    mx_status_t s = encode_bf16_rows(&tm_x, a_hat, p.M, p.K, T / 2);
    if (s != MX_OK) return s;
    s = encode_u8_sw128(&tm_r, w_mant, p.N, fw.elem_bits <= 4 ? p.K / 2 : p.K, Cfg::BN);
    if (s != MX_OK) return s;
    s = smem_attr_once(d.tmw_attr_set[g.which], g_tmw[g.which], 227 * 1024);
    if (s != MX_OK) return s;
    p.tiles_m = (p.M + T - 1) / T;
    p.tiles_n = (p.N + 2 * Cfg::BN - 1) / (2 * Cfg::BN);
    const int64_t tiles = (int64_t)p.tiles_m * p.tiles_n;
    if (tiles > INT32_MAX / 2) return MX_ERR_SHAPE;
    const int pairs = (int)(tiles < d.sm_count / 2 ? tiles : d.sm_count / 2);
    const mx::TmwParams wp{w_exp, fw.elem_bits, fw.block_rows == 2 ? 1 : 0, fw.block, T, Cfg::stages(T, p.yq_mant), 1, g.exp_words, g.split};
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    tmw_config(cfg, attr, g.split, g.split > 1 ? (int)tiles : pairs, st);
    cfg.dynamicSmemBytes = Cfg::smem_bytes(T, p.yq_mant);
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = g_prof.on ? 1 : 2;                     // see launch_dep
    ProfScope prof(KIND_GEMM_TC, st);
    MX_CUDA(cudaLaunchKernelEx(&cfg, g_tmw[g.which], tm_x, tm_r, p, wp));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

mx_status_t launch_dec(const DecPlan &g, const __nv_bfloat16 *a_hat, const void *w_mant, const uint8_t *w_exp, const mx_format_t &fw, int64_t M,
                       int64_t N, int64_t K, const float *bias, float *y, int64_t ldy, const QuantizedOut *yq, DeviceInfo &d, cudaStream_t st,
                       const EpiTail &et)
{
    mx::TcParams p{};
    p.y = y;
    p.ex_bias = bias;
    p.relu = et.relu;
    p.residual = et.residual;
    p.ldr = et.ldr;
    p.ldy = ldy;
    p.M = (int)M;
    p.N = (int)N;
    p.K = (int)K;
    p.tiles_m = 1;
    p.tiles_n = (int)((N + mx::DecCfg::BN - 1) / mx::DecCfg::BN);
    p.status = d.status;
    p.batch = 1;
    p.yq_mant = yq ? yq->mant : nullptr;
    p.yq_exp = yq ? yq->exps : nullptr;
    p.yq_nonfinite = yq ? yq->nonfinite : nullptr;
    p.yq_bits = yq ? yq->f.elem_bits : 0;
    p.yq_block = yq ? yq->f.block : 0;
    p.yq_rows2 = yq && yq->f.block_rows == 2 ? 1 : 0;
    if (g.tokens) return launch_tmw(g, a_hat, w_mant, fw, p, w_exp, d, st);
    CUtensorMap tm_a, tm_r;
    mx_status_t s = encode_bf16_rows(&tm_a, a_hat, M, K, mx::TC_BM);
    if (s != MX_OK) return s;
    s = encode_u8_sw128(&tm_r, w_mant, N, fw.elem_bits <= 4 ? K / 2 : K, mx::DecCfg::BN);
    if (s != MX_OK) return s;
    const mx::DecParams dp{w_exp, fw.elem_bits, fw.block_rows == 2 ? 1 : 0, fw.block, g.split, 1, g.exp_words};
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    dec_config(cfg, attr, g.panels, p.tiles_n * g.split, g.split, st);
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = g_prof.on ? 1 : 2;                     // see launch_dep
    ProfScope prof(KIND_GEMM_TC, st);
    MX_CUDA(cudaLaunchKernelEx(&cfg, g_dec[g.which], tm_a, tm_r, p, dp));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

// Estimates in us of whole calls on 148 SMs, pass over the activations included: what dec_plan compares gemm_tmw_kernel with the other
// routes by.  Fitted to 5600 shapes -- 17 .. 2048 rows, K 32 .. 16384, N 2 .. 16384, widths 8/4, 4/4, 6/6 and 8/8, blocks of 16 and 32 --
// with every route timed (tmw_tokens: up to eleven tiles and cuts each), 1900 of them with an MXInt result too.  One sigma of their
// errors: tmw_us and dec_us 4.9 %, tc_us 5.9 %, rec_us 4.6 %; with an MXInt result (`quantized`) 4.4, 6.5, 5.5 and 11 %.
double up(double x) { return (double)(int64_t)(x + 0.999999); }

// gemm_tmw_kernel on tiles of T tokens, K in `pieces`.  Rounds of 74 pairs, each 0.253 us per K step of 64 up to 160 tokens (its
// decoding warps), 0.263 at 192, 0.272 and 0.301 at 224 and 256 (its MMAs), for weights in bytes 0.342 and 0.349; a tenth less on few
// pairs.  The exponent rows have to be copied in as well: by words (EXP_WORDS), of two pieces per K step of bytes in blocks of 16, they
// take longer than the step, and so they do where they are no whole words (EXP_BYTES) and come by the words that hold them.  An odd
// number of steps costs two.  An epilogue behind the last round, with one accumulator behind each; that of an MXInt result is long
// enough to show under the next round's steps.
double tmw_us(double M, double N, double K, bool nib, int block, ExpRows rows, bool quantized, int T, int pieces, double pairs)
{
    const double steps = up(K / 64), mk = M * K * 1e-6, mn = M * N * 1e-6, unit = nib ? 4 : 2;   // unit: steps per stage of packed weights
    const double tiles = up(M / T) * up(N / 256), load = tiles * pieces < pairs ? tiles * pieces / pairs : 1;
    double step = nib ? T <= 160 ? 0.253 : T <= 192 ? 0.263 : T <= 224 ? 0.272 : 0.301 : T <= 192 ? 0.342 : 0.349;
    if (rows == EXP_BYTES) step = nib ? block == 16 ? 0.332 : 0.31 : block == 16 ? 0.46 : 0.415;
    else if (rows == EXP_WORDS && !nib && block == 16) step = 0.4;
    step *= 0.9 + 0.1 * load;
    if (pieces > 1)                                                      // (2 % on top: what the fit lacks where the clusters fill the chip)
        return 1.02 * (5.21 + 0.6 * pieces + 1.12 * load + 0.916 * mk + 0.753 * mn + up(up(steps / unit) / pieces) * unit * step + 0.021 * T) +
               (quantized ? 0.35 + 0.75 * mn + 0.006 * T : 0);
    const bool one = mx::TmwCfg::accs(T) == 1;
    const double rounds = up(tiles / pairs), odd = 2 * (steps - 2 * (double)(int64_t)(steps / 2));
    const double us = 6.32 + 0.916 * mk + 0.472 * mn + rounds * (steps + odd) * step + 0.009 * T * (one ? rounds : 1);
    if (!quantized) return us;
    const double epilogue = 0.0131 * T, shows = one ? epilogue - 2.36 : 0.42 * (epilogue + 1.57 - steps * (nib ? 0.26 : 0.345));
    return us - 0.27 + 0.315 * mn + epilogue + (one || shows > 0 ? (rounds - 1) * shows : 0);
}

// A pass that writes both operands out in bf16, and the product.  The pass deals items of 256 activations and 1024 weights of one row
// -- short rows leave lanes idle -- to CTAs that are counted by elements (prep_operands_kernel).
double tc_us(const TcRoute &r, int64_t M, int64_t N, int64_t K, bool quantized, int sm_count)
{
    const double m = (double)M, n = (double)N, k = (double)K, steps = up(k / 64), pairs = sm_count / 2;
    const double mk = m * k * 1e-6, mn = m * n * 1e-6, nk = n * k * 1e-6;
    const double ctas = mk * 1e6 / 2048 + nk * 1e6 / 8192, most = 16.0 * sm_count;
    const double turns = (m * up(k / 256) + n * up(k / 1024)) / (4 * (ctas < most ? ctas : most)) - 2;
    double us = 0.44 * n * up(k / 1024) * 1024e-6 + (nk > 40 ? 0.2 * (nk - 40) : 0) + 0.93 * mk + (turns > 0 ? 0.4 * turns : 0);
    us += (0.47 + (N % 4 ? 0.42 : 0)) * mn + (K % 32 ? 2 : 0);           // rows of y without whole 16 bytes; two launches
    if (quantized) us += (r.kernel == TC_CUT ? 1.45 : r.kernel == TC_PAIR ? 0.6 : r.kernel == TC_PAIR_WIDE ? 0.003 * r.width : 0.25) - 0.055 * mn;
    const double tiles = up(m / 256) * up(n / r.width);
    switch (r.kernel) {
    case TC_CUT: return us + 7.7 + 0.154 * up(steps / r.split);
    case TC_PAIR: return us + 8.05 + 0.283 * steps * 0.5 * (tiles / pairs + up(tiles / pairs));      // (the epilogue runs under the next round)
    case TC_PAIR_WIDE: return us + 7.1 + 0.286 * steps * up(tiles / pairs) * r.width / 256;
    default: break;
    }
    const double waves = up(up(m / 128) * up(n / r.width) / sm_count);
    return us + (r.width == 128 ? 6.35 + 0.182 * steps * waves : 7.0 + 0.302 * steps * waves);
}

// The same on block-scaled records.
double rec_us(int64_t M, int64_t N, int64_t K, bool quantized, int sm_count)
{
    const double m = (double)M, n = (double)N, k = (double)K, nk = n * k * 1e-6, t = up(m / 256) * up(n / 256) / (sm_count / 2);
    return 8.2 + 0.278 * up(k / 128) * (t > 1 ? 0.5 * (t + up(t)) : 1) + 0.424 * nk + (nk > 40 ? 0.19 * (nk - 40) : 0) + 1.22 * m * k * 1e-6 +
           (0.57 + (N % 4 ? 0.67 : 0)) * m * n * 1e-6 + (quantized ? 1.6 - 0.2 * m * n * 1e-6 : 0);
}

// gemm_dec_kernel: waves of clusters.
double dec_us(int64_t M, int64_t N, int64_t K, int split, bool nib, bool words, bool quantized, int sm_count)
{
    const double m = (double)M, k = (double)K, panels = up(m / 128), ctas = up((double)N / 128) * split, waves = up(ctas / sm_count);
    const double load = ctas < sm_count ? ctas / sm_count : 1;
    double step = (panels <= 1 ? 0.332 : panels <= 2 ? 0.449 : 0.634) * (nib ? 1 : 1.13);
    if (!words && step < 0.4) step = 0.4;
    return 5.85 + 1.8 * panels + 2.0 * m * k * 1e-6 + 0.51 * m * (double)N * 1e-6 + 0.02 * (split - 1) + 0.67 * load + 5 * (waves - 1) +
           waves * up(up(k / 64) / split) * step * (0.9 + 0.1 * load) + (quantized ? 1.14 + 0.46 * panels - 0.07 * m * (double)N * 1e-6 : 0);
}

// Tokens per tile and pieces of K with which gemm_tmw_kernel is expected to take at most 0.98 of `other` (0.97 with an MXInt result,
// whose estimates are off by more), else 0.  Over the shapes measured the route taken is then 0.925 (0.952) of the other one on average
// and 1.008 (1.010) of the best; in 50 of 5300 (31 of 1900) it is more than 2 % slower than the other one, in nine (four) by 8 to 15 %.  Whole calls without / with it: 160 x 4096 x 11008 (M x K x N)
// 40.4 / 25.0, 128 x 4096 x 11008 30.0 / 25.0, 256 x 2048 x 12288 26.8 / 21.3, 256 x 1024 x 16384 20.1 / 16.7, 512 x 8192 x 8192
// 80.5 / 53.0, 768 x 16384 x 4096 105 / 86, 1024 x 4096 x 4096 38.4 / 35.1; K cut in two 448 x 16384 x 4096 100 / 54.6, in three
// 352 x 8192 x 2048 29.6 / 27.6; left alone 1237 x 2048 x 2048 18.8 / 20.1.  Above 1536 rows the passes cost too little beside the product
// (2048 x 4096 x 4096 62.6 / 61.0, 3072 x 1344 x 11008 74 / 82).
int tmw_tokens(int64_t M, int64_t N, int64_t K, bool nib, int block, ExpRows rows, bool quantized, double other, int sm_count, const int *clusters,
               int *pieces)
{
    const double m = (double)M, n = (double)N, k = (double)K;
    double best = (quantized ? 0.97 : 0.98) * other;
    int tokens = 0;
    if (N < 32) return 0;                                                // an eighth of a tile (1400 x 64 x 4 7.6 / 7.9)
    for (int T = 64; T <= mx::TmwCfg::MAX_T && T < M + 64; T += 32) {
        const double tiles = up(m / T) * up(n / 256);
        for (int s = 1; s <= mx::TmwCfg::MAX_SPLIT; ++s) {
            if (s > 1 && (tiles > clusters[s] || up(k / 64) < s * (nib ? 4 : 2))) break;
            const double us = tmw_us(m, n, k, nib, block, rows, quantized, T, s, sm_count / 2);
            if (us < best) {
                best = us;
                tokens = T;
                *pieces = s;
            }
        }
    }
    return tokens;
}

// Whether gemm_dec_kernel beats a pass over the weights and then a product (`rec`: of block-scaled records, where that one would run,
// else of bf16); tmw_tokens decides after it.  Whole calls in a graph, us, 8-bit activations (records: 4 bits), 4-bit weights, blocks
// of 16; bf16 / records / gemm_dec_kernel / the best of gemm_tmw_kernel:
//   rows     K x N        bf16    rec    dec    tmw      rows     K x N        bf16    rec    dec    tmw
//   128   1024 x 4096    10.8   11.9    9.8   10.5      128   4096 x 22528   83.6   70.1   57.5   41.7
//   128   2048 x 6144    16.5   18.7   13.9   14.5      128   2048 x 28672   51.8   45.4   37.9   26.4
//   128   8192 x 2048    22.0   33.3   16.1   19.4      128   4096 x 32000  109.9   91.7   58.2   41.6
//   128   4096 x 4096    19.6   24.2   14.6   17.2      256   2048 x 2560    12.4   15.9   14.1   14.1
//   128   1024 x 9600    14.0   15.5   13.6   11.7      256   4096 x 4096    22.8   24.8   19.1   20.3
//   64    1024 x 9600    13.6   14.4   12.8   10.7      256  11008 x 4096    50.6   58.2   34.7   35.7
//   128    256 x 9600    12.7   10.4    9.5    8.7      256   1024 x 16384   20.1   18.9   20.7   16.7
//   128   4096 x 9600    37.8   35.6   29.9   24.8      256   3072 x 14336   41.8   36.2   35.3   26.1
//   128   1024 x 16384   17.1   18.0   14.0   12.4      256   4096 x 16384   63.3   48.8   43.3   31.8
//   128   4096 x 16384   58.2   48.0   31.1   26.1      384   4096 x 3072    21.7   24.7   23.5   22.5
//   128   1024 x 19072   21.5   22.8   25.7   16.2      384   4096 x 4096    26.7   26.2   25.2   23.6
//   128   4096 x 19072   74.8   62.2   57.2   40.6      384   4096 x 6144    31.2   31.2   34.6   26.9
//   128   1024 x 28672   26.7   27.6   27.5   17.9      384   6144 x 6144    46.2   43.6   46.5   34.9
//   128   1344 x 28672   37.4   35.8   31.0   22.9      384   8192 x 8192    76.0   61.0   58.6   45.7
// Up to 128 rows: while its CTAs make one wave that leaves at most three SMs in ten idle, wherever the weights are large.  A
// second wave repeats ramp and exchange, which the other product overlaps with its loads: from K = 1344 on where it is full, from
// 4096 on where not.  A single wave that is not full and not cut is worth it against bf16 only, for very short K or long.
// Below 2 M weights the other product is not cut under 16 K steps of 64; this one, cut in three pieces from 12 steps on, is the
// faster one then (without / with, 8/4: 64 x 768 x 256 9.6 / 8.9, 64 x 896 x 1024 10.4 / 10.2, 96 x 960 x 512 10.6 / 10.3; in two
// pieces 64 x 704 x 512 9.5 / 10.5; against a cut one 64 x 992 x 512 8.6 / 9.4), beyond 96 rows while a piece has four steps
// (128 x 768: N = 256 9.5 / 9.7, 512 9.9 / 9.8, 2048 10.2 / 9.9; 128 x 896 x 512 10.7 / 10.8).
// With more rows a CTA's steps cost more of what decoding them once saves, so there the weights have to be larger, or K long.
bool dec_is_faster(int64_t M, int64_t N, int64_t K, int split, bool rec, int sm_count)
{
    const int64_t size = N * K, ctas = (N + mx::DecCfg::BN - 1) / mx::DecCfg::BN * split, waves = (ctas + sm_count - 1) / sm_count;
    const bool full = 10 * ctas >= 7 * waves * sm_count;
    if (M <= 128) {
        const int64_t steps = (K + mx::TC_BK - 1) / mx::TC_BK;
        if (size <= (1 << 21)) return steps >= 12 && steps < 16 && (M <= 96 || (steps == 12 && N >= 512));
        if (full) return waves == 1 || K >= 1280;
        if (rec) return false;
        return split >= 2 || (waves == 1 ? K < 512 || K >= 3072 : K >= 4096);
    }
    if (M <= 256) return size >= 3 << 22 && N >= 2560 && full && (split >= 2 || (!rec && K >= 3072));
    return size >= 1 << 24 && K >= (split == 3 ? 6144 : 4096) && full && (split >= 4 || !rec);
}

// Both operands of one layer in the tensor-core form: activations quantized straight to exact
// bf16, packed weights decoded to bf16.  One launch when K % 32 == 0, else two.
mx_status_t tc_prepare(const mx_linear_args_t &a, __nv_bfloat16 *a_hat, __nv_bfloat16 *w_hat, DeviceInfo &d,
                       cudaStream_t st)
{
    const int64_t M = a.M, N = a.N, K = a.K;
    mx::QuantOut out{nullptr, nullptr, a_hat, K, nullptr};
    if ((K % 32) != 0 || a.fw.packing) {
        mx_status_t s = quantize_rows_any(a.x, a.dt, M, K, a.ldx, a.fa, out, d, st);
        if (s != MX_OK) return s;
        return launch_dequant_bf16(a.w_mant, a.w_exp, N, K, a.fw, w_hat, K, d, st);
    }
    // one launch for both sides; every warp takes its share of each (see the kernel)
    mx::PrepJob job;
    job.x = a.x; job.M = M; job.K = K; job.ldx = a.ldx; job.wa = a.fa.elem_bits; job.block = a.fa.block;
    job.a_hat = a_hat;
    job.w_mant = static_cast<const uint8_t *>(a.w_mant); job.w_exp = a.w_exp; job.N = N; job.ww = a.fw.elem_bits;
    job.w_hat = w_hat;
    job.w_row_shift = a.fw.block_rows == 2 ? 1 : 0;
    job.a_rows2 = a.fa.block_rows == 2 ? 1 : 0;
    const bool f32 = a.dt == MX_F32, nib = a.fw.elem_bits <= 4;
    // CTAs of 128 threads (8 K registers): small enough to become resident beside a persistent product CTA of the
    // previous call, where they wait in griddepcontrol.wait and start the moment that grid completes
    constexpr int PT = 128;
    const int need_q = grid_for((M * (K / 8) + 1) / 2, PT, 1 << 20, 1);
    const int need_d = grid_for((N * (K / 32) + 1) / 2, PT, 1 << 20, 1);
    const int per_sm = (256 / PT) * (f32 ? (nib ? resident_ctas(mx::prep_operands_kernel<float, true>)
                                            : resident_ctas(mx::prep_operands_kernel<float, false>))
                                     : (nib ? resident_ctas(mx::prep_operands_kernel<__nv_bfloat16, true>)
                                            : resident_ctas(mx::prep_operands_kernel<__nv_bfloat16, false>)));
    const int total = d.sm_count * per_sm;            // at most one resident wave
    const int grid = need_q + need_d < total ? need_q + need_d : total;
    ProfScope prof(KIND_PREP, st);
    if (f32) {
        if (nib) MX_CUDA(launch_dep(mx::prep_operands_kernel<float, true>, dim3(grid), dim3(PT), 0, st, job));
        else MX_CUDA(launch_dep(mx::prep_operands_kernel<float, false>, dim3(grid), dim3(PT), 0, st, job));
    } else {
        if (nib) MX_CUDA(launch_dep(mx::prep_operands_kernel<__nv_bfloat16, true>, dim3(grid), dim3(PT), 0, st, job));
        else MX_CUDA(launch_dep(mx::prep_operands_kernel<__nv_bfloat16, false>, dim3(grid), dim3(PT), 0, st, job));
    }
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

}  // namespace

// =================================================================================================
extern "C" {

static mx_status_t grouped_impl(const mx_linear_args_t *layers, int32_t n_layers,
                                const uint8_t *const *packed_exps, bool any_order, void *workspace, size_t workspace_bytes,
                                void *stream);

size_t mx_mant_bytes(int64_t rows, int64_t K, mx_format_t f)
{
    if (!format_ok_any(f) || rows < 0 || K < 0 || (K % f.block) != 0) return 0;
    return (size_t)rows * mant_row_bytes(K, f);
}

size_t mx_exp_bytes(int64_t rows, int64_t K, mx_format_t f)
{
    if (!format_ok_any(f) || rows < 0 || K < 0 || (K % f.block) != 0 || (rows % f.block_rows) != 0) return 0;
    return (size_t)(rows / f.block_rows) * (size_t)(K / f.block);
}

double mx_format_bits(mx_format_t f)
{
    if (f.block <= 0 || f.block_rows <= 0 || f.exp_bits <= 0 || f.elem_bits < 2) return 0.0;
    return (double)f.exp_bits / ((double)f.block * (double)f.block_rows) + (double)(f.elem_bits - 1) + 1.0;
}

size_t mx_workspace_bytes_ex(int64_t M, int64_t N, int64_t K, mx_format_t fa, mx_format_t fw,
                             mx_algo_t algo)
{
    if (!format_ok_any(fa) || !format_ok_any(fw) || M <= 0 || N <= 0 || K <= 0) return 0;
    const size_t pk = packed_workspace(M, K, fa);          // mx_linear with the CUDA-core kernel
    switch (algo) {
    case MX_ALGO_SIMT: return pk;
    case MX_ALGO_STREAM: return stream_table_bytes(1) + round256(mx_mant_bytes(M, K, fa)) +
                                round256(mx_exp_bytes(M, K, fa));
    case MX_ALGO_AUTO: {            // mx_linear may stream (M <= 16), mx_gemm uses the tensor cores
        const size_t st = mx_workspace_bytes_ex(M, N, K, fa, fw, MX_ALGO_STREAM);
        const size_t tc = tc_workspace(M, N, K);
        return st > tc ? st : tc;
    }
    case MX_ALGO_TCGEN05:
    case MX_ALGO_TCGEN05_BLOCKWISE: return tc_workspace(M, N, K);
    case MX_ALGO_TCGEN05_FUSED: return (K % 32) == 0 ? fused_workspace(M, K) : tc_workspace(M, N, K);
    case MX_ALGO_TCGEN05_MXF8:      // E4M3 operands + scale chunks; mx_linear also keeps the packed activations
        return mxf8_fits(fa, fw, K) ? mxf8_operand_bytes(M, N, K) + pk : 0;
    default: return 0;
    }
}

size_t mx_workspace_bytes(int64_t M, int64_t N, int64_t K, mx_format_t fa, mx_format_t fw)
{
    return mx_workspace_bytes_ex(M, N, K, fa, fw, MX_ALGO_AUTO);
}

const char *mx_status_string(mx_status_t s)
{
    switch (s) {
    case MX_OK: return "ok";
    case MX_ERR_NULL: return "null pointer";
    case MX_ERR_SHAPE: return "bad shape";
    case MX_ERR_FORMAT: return "unsupported MXInt format";
    case MX_ERR_ALIGN: return "misaligned pointer or stride";
    case MX_ERR_WORKSPACE: return "workspace missing or too small";
    case MX_ERR_CUDA: return "CUDA error";
    case MX_ERR_TIMEOUT: return "device-side wait timed out";
    case MX_ERR_ARCH: return "device is not sm_100";
    }
    return "unknown status";
}

const char *mx_last_cuda_error(void) { return t_cuda_error; }

mx_status_t mx_quantize(const void *x, mx_dtype_t dt, int64_t rows, int64_t K, int64_t stride_row,
                        int64_t stride_k, mx_format_t f, void *mant_out, uint8_t *exp_out,
                        uint32_t *nonfinite_count, void *stream)
{
    if (!format_ok(f) || (dt != MX_F32 && dt != MX_BF16)) return MX_ERR_FORMAT;
    if (rows < 0 || K < 0 || (K % f.block) != 0 || (rows % f.block_rows) != 0) return MX_ERR_SHAPE;
    if (rows == 0 || K == 0) return MX_OK;               // empty tensor: nothing to do
    if (f.block_rows != 1 && stride_k != 1) return MX_ERR_FORMAT;   // two-row blocks: rows contiguous along K only
    if (!x || !mant_out || !exp_out) return MX_ERR_NULL;
    if (stride_k == 0 || (stride_k == 1 && stride_row < K)) return MX_ERR_SHAPE;
    if (!aligned16(x) || !aligned16(mant_out)) return MX_ERR_ALIGN;
    if (stride_k == 1 && (stride_row % 8) != 0) return MX_ERR_ALIGN;
    DeviceInfo *d = nullptr;
    mx_status_t s = device_info(&d);
    if (s != MX_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    mx::QuantOut out{static_cast<uint8_t *>(mant_out), exp_out, nullptr, 0, nonfinite_count};
    if (stride_k == 1) return quantize_rows_any(x, dt, rows, K, stride_row, f, out, *d, st);
    if (stride_row == 1 && (K % 32) == 0 && (reinterpret_cast<uintptr_t>(mant_out) & 15u) == 0) {
        // a transposed view: blocks along the slow axis of a row-major tensor
        if (dt == MX_F32) return launch_quantize_columns(static_cast<const float *>(x), rows, K, stride_k, f, out, *d, st);
        return launch_quantize_columns(static_cast<const __nv_bfloat16 *>(x), rows, K, stride_k, f, out, *d, st);
    }
    const int grid = grid_for(rows * (K / f.block), 256, d->sm_count, 8);
    ProfScope prof(KIND_QUANTIZE, st);
    if (dt == MX_F32)
        mx::quantize_strided_kernel<float><<<grid, 256, 0, st>>>(
            static_cast<const float *>(x), rows, K, stride_row, stride_k, f.block, f.elem_bits, out);
    else
        mx::quantize_strided_kernel<__nv_bfloat16><<<grid, 256, 0, st>>>(
            static_cast<const __nv_bfloat16 *>(x), rows, K, stride_row, stride_k, f.block, f.elem_bits, out);
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

static mx_status_t repack_impl(const void *src, int64_t rows, int64_t K, mx_format_t f, void *dst, bool to_dense, void *stream)
{
    f.packing = 0;
    if (!format_ok(f)) return MX_ERR_FORMAT;
    if (rows < 0 || K < 0 || (K % f.block) != 0) return MX_ERR_SHAPE;
    if (rows == 0 || K == 0) return MX_OK;
    if (!src || !dst) return MX_ERR_NULL;
    if (!aligned16(to_dense ? src : dst)) return MX_ERR_ALIGN;
    DeviceInfo *d = nullptr;
    mx_status_t s = device_info(&d);
    if (s != MX_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int grid = grid_for(rows * (K / 8), 256, d->sm_count, 8);
    ProfScope prof(KIND_QUANTIZE, st);
    if (to_dense)
        MX_CUDA(launch_dep(mx::dense_pack_kernel, dim3(grid), dim3(256), 0, st, static_cast<const uint8_t *>(src), rows, K,
                           (int)f.elem_bits, static_cast<uint8_t *>(dst)));
    else
        MX_CUDA(launch_dep(mx::dense_unpack_kernel, dim3(grid), dim3(256), 0, st, static_cast<const uint8_t *>(src), rows, K,
                           (int)f.elem_bits, static_cast<uint8_t *>(dst)));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

mx_status_t mx_pack_dense(const void *mant, int64_t rows, int64_t K, mx_format_t f, void *dense_out, void *stream)
{
    return repack_impl(mant, rows, K, f, dense_out, true, stream);
}

mx_status_t mx_unpack_dense(const void *dense, int64_t rows, int64_t K, mx_format_t f, void *mant_out, void *stream)
{
    return repack_impl(dense, rows, K, f, mant_out, false, stream);
}

mx_status_t mx_cast(const void *mant_in, const uint8_t *exp_in, mx_format_t f_in, int64_t rows, int64_t K,
                    mx_format_t f_out, void *mant_out, uint8_t *exp_out, uint32_t *nonfinite_count, void *stream)
{
    if (!format_1d(f_in) || !format_1d(f_out)) return MX_ERR_FORMAT;
    if (rows < 0 || K < 0 || (K % f_in.block) != 0 || (K % f_out.block) != 0) return MX_ERR_SHAPE;
    if (rows == 0 || K == 0) return MX_OK;
    if (!mant_in || !exp_in || !mant_out || !exp_out) return MX_ERR_NULL;
    if (!aligned16(mant_in) || !aligned16(mant_out)) return MX_ERR_ALIGN;
    DeviceInfo *d = nullptr;
    mx_status_t s = device_info(&d);
    if (s != MX_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    mx::QuantOut out{static_cast<uint8_t *>(mant_out), exp_out, nullptr, 0, nonfinite_count};
    const int grid = grid_for(rows * (K / 8), 256, d->sm_count, 8);
    const uint8_t *mi = static_cast<const uint8_t *>(mant_in);
    ProfScope prof(KIND_QUANTIZE, st);
    if (f_out.block == 16)
        MX_CUDA(launch_dep(mx::cast_rows_kernel<16>, dim3(grid), dim3(256), 0, st, mi, exp_in, (int)f_in.block,
                           (int)f_in.elem_bits, rows, K, (int)f_out.elem_bits, out));
    else
        MX_CUDA(launch_dep(mx::cast_rows_kernel<32>, dim3(grid), dim3(256), 0, st, mi, exp_in, (int)f_in.block,
                           (int)f_in.elem_bits, rows, K, (int)f_out.elem_bits, out));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

mx_status_t mx_dequantize(const void *mant, const uint8_t *exps, int64_t rows, int64_t K,
                          mx_format_t f, void *out, mx_dtype_t dt, int64_t ld_out, void *stream)
{
    if (!mant || !exps || !out) return MX_ERR_NULL;
    if (!format_ok_any(f) || (dt != MX_F32 && dt != MX_BF16)) return MX_ERR_FORMAT;
    if (rows < 0 || K < 0 || (K % f.block) != 0 || ld_out < K || (rows % f.block_rows) != 0) return MX_ERR_SHAPE;
    if (!aligned16(mant) || !aligned16(out) || (ld_out % 8) != 0) return MX_ERR_ALIGN;
    if (rows == 0 || K == 0) return MX_OK;
    DeviceInfo *d = nullptr;
    mx_status_t s = device_info(&d);
    if (s != MX_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (f.packing && dt == MX_F32) {
        ProfScope prof(KIND_DEQUANTIZE, st);
        MX_CUDA(launch_dep(mx::dequantize_dense_kernel<float>, dim3(grid_for(rows * (K / 8), 256, d->sm_count, 8)), dim3(256), 0,
                           st, static_cast<const uint8_t *>(mant), exps, rows, K, (int)f.block, (int)f.elem_bits,
                           f.block_rows == 2 ? 1 : 0, static_cast<float *>(out), ld_out, 0));
        MX_CUDA(cudaGetLastError());
        return MX_OK;
    }
    if (dt == MX_BF16)
        return launch_dequant_bf16(mant, exps, rows, K, f, static_cast<__nv_bfloat16 *>(out), ld_out, *d, st);
    ProfScope prof(KIND_DEQUANTIZE, st);
    mx::dequantize_kernel<float><<<grid_for(rows * (K / 8), 256, d->sm_count, 16), 256, 0, st>>>(
        static_cast<const uint8_t *>(mant), exps, rows, K, f.block, f.elem_bits,
        static_cast<float *>(out), ld_out, dense_strides(K, f));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

mx_status_t mx_gemm_ex(const void *a_mant, const uint8_t *a_exp, mx_format_t fa, const void *w_mant,
                       const uint8_t *w_exp, mx_format_t fw, int64_t M, int64_t N, int64_t K,
                       const float *bias, float *y, int64_t ldy, void *workspace,
                       size_t workspace_bytes, mx_algo_t algo, void *stream)
{
    mx_status_t s = check_gemm_args(a_mant, a_exp, fa, w_mant, w_exp, fw, M, N, K, bias, y, ldy);
    if (s != MX_OK) return s;
    if (!a_exp) return MX_ERR_NULL;
    const bool any_algo = algo == MX_ALGO_AUTO;
    {
        mx_linear_args_t one;
        one.x = a_mant; one.dt = MX_F32; one.M = M; one.K = K; one.ldx = K; one.fa = fa;
        one.w_mant = w_mant; one.w_exp = w_exp; one.fw = fw; one.N = N; one.bias = bias; one.y = y; one.ldy = ldy;
        const bool can_stream = stream_layer_ok(one) && (reinterpret_cast<uintptr_t>(w_exp) & 3u) == 0 &&
                                workspace && workspace_bytes >= stream_table_bytes(1);
        if (algo == MX_ALGO_AUTO && !can_stream) {
            DeviceInfo *dd = nullptr;
            s = device_info(&dd);
            if (s != MX_OK) return s;
            bool dec = false;
            DecPlan plan;
            s = dec_plan(M, N, K, fa, fw, w_exp, false, *dd, &plan, &dec);
            if (s != MX_OK) return s;
            if (dec) {
                if (!workspace || workspace_bytes < tc_workspace(M, N, K)) return MX_ERR_WORKSPACE;
                if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return MX_ERR_ALIGN;
                __nv_bfloat16 *a_dec = static_cast<__nv_bfloat16 *>(workspace);
                cudaStream_t sd = static_cast<cudaStream_t>(stream);
                s = launch_dequant_bf16(a_mant, a_exp, M, K, fa, a_dec, K, *dd, sd, true);
                if (s != MX_OK) return s;
                return launch_dec(plan, a_dec, w_mant, w_exp, fw, M, N, K, bias, y, ldy, nullptr, *dd, sd, EpiTail());
            }
        }
        if (algo == MX_ALGO_AUTO && !can_stream && rec_fits(fa, fw, M, N, K)) {
            if (!workspace || workspace_bytes < tc_workspace(M, N, K)) return MX_ERR_WORKSPACE;
            if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return MX_ERR_ALIGN;
            DeviceInfo *dr = nullptr;
            s = device_info(&dr);
            if (s != MX_OK) return s;
            bool rec = false;
            s = rec_is_faster(M, N, K, *dr, &rec);
            if (s != MX_OK) return s;
            if (rec)
                return run_rec_gemm(a_mant, a_exp, fa, w_mant, w_exp, fw, M, N, K, bias, y, ldy, nullptr,
                                    static_cast<uint8_t *>(workspace), *dr, static_cast<cudaStream_t>(stream), EpiTail());
        }
        if (algo == MX_ALGO_AUTO) algo = can_stream ? MX_ALGO_STREAM : MX_ALGO_TCGEN05;
        if (algo == MX_ALGO_STREAM) return grouped_impl(&one, 1, &a_exp, false, workspace, workspace_bytes, stream);
    }
    if (algo == MX_ALGO_TCGEN05_MXF8) {
        if (!mxf8_fits(fa, fw, K)) return MX_ERR_FORMAT;
        if (!workspace || workspace_bytes < mxf8_operand_bytes(M, N, K)) return MX_ERR_WORKSPACE;
        if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return MX_ERR_ALIGN;
        DeviceInfo *d8 = nullptr;
        s = device_info(&d8);
        if (s != MX_OK) return s;
        return run_tc8(a_mant, a_exp, fa, w_mant, w_exp, fw, M, N, K, bias, y, ldy, static_cast<uint8_t *>(workspace), *d8,
                       static_cast<cudaStream_t>(stream));
    }
    if (algo != MX_ALGO_SIMT && algo != MX_ALGO_TCGEN05_FUSED && algo != MX_ALGO_TCGEN05 &&
        algo != MX_ALGO_TCGEN05_BLOCKWISE)
        return MX_ERR_FORMAT;
    // dense storage is read by the decode pass in front of the tensor-core kernels only
    if ((fa.packing || fw.packing) && algo != MX_ALGO_TCGEN05 && algo != MX_ALGO_TCGEN05_BLOCKWISE) return MX_ERR_FORMAT;
    DeviceInfo *d = nullptr;
    s = device_info(&d);
    if (s != MX_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (algo == MX_ALGO_SIMT) {
        dim3 grid((unsigned)((N + 15) / 16), (unsigned)((M + 15) / 16));
        ProfScope prof(KIND_GEMM_SIMT, st);
        mx::gemm_simt_kernel<<<grid, 256, 0, st>>>(static_cast<const uint8_t *>(a_mant), a_exp,
                                                   fa.elem_bits, static_cast<const uint8_t *>(w_mant),
                                                   w_exp, fw.elem_bits, M, N, K, fa.block, bias, y, ldy,
                                                   fa.block_rows == 2 ? 1 : 0, fw.block_rows == 2 ? 1 : 0);
        MX_CUDA(cudaGetLastError());
        return MX_OK;
    }
    const bool fused = algo == MX_ALGO_TCGEN05_FUSED && (K % 32) == 0 && fw.block_rows == 1;
    if (fused && !fused_ok(K, w_exp)) return MX_ERR_ALIGN;
    if (!workspace || workspace_bytes < (fused ? fused_workspace(M, K) : tc_workspace(M, N, K)))
        return MX_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return MX_ERR_ALIGN;
    __nv_bfloat16 *a_hat = static_cast<__nv_bfloat16 *>(workspace);
    if (fused) {
        s = launch_dequant_bf16(a_mant, a_exp, M, K, fa, a_hat, K, *d, st);
        if (s != MX_OK) return s;
        return run_tc_fused(a_hat, w_mant, w_exp, fw, M, N, K, bias, y, ldy, *d, st);
    }
    __nv_bfloat16 *w_hat = reinterpret_cast<__nv_bfloat16 *>(static_cast<uint8_t *>(workspace) +
                                                             round256((size_t)M * K * 2));
    s = launch_dequant_pair(a_mant, a_exp, fa, M, w_mant, w_exp, fw, N, K, a_hat, w_hat, *d, st);
    if (s != MX_OK) return s;
    if (algo == MX_ALGO_TCGEN05_BLOCKWISE) return launch_tcx(a_hat, w_hat, M, N, K, fa.block, bias, y, ldy, *d, st);
    return run_tc(a_hat, w_hat, M, N, K, bias, y, ldy, *d, st, nullptr, TcBatch(), EpiTail(), any_algo, true);
}

mx_status_t mx_gemm(const void *a_mant, const uint8_t *a_exp, mx_format_t fa, const void *w_mant,
                    const uint8_t *w_exp, mx_format_t fw, int64_t M, int64_t N, int64_t K,
                    const float *bias, float *y, int64_t ldy, void *workspace, size_t workspace_bytes,
                    void *stream)
{
    return mx_gemm_ex(a_mant, a_exp, fa, w_mant, w_exp, fw, M, N, K, bias, y, ldy, workspace,
                      workspace_bytes, MX_ALGO_AUTO, stream);
}

mx_status_t mx_linear_ex(const void *x, mx_dtype_t dt, int64_t M, int64_t K, int64_t ldx,
                         mx_format_t fa, const void *w_mant, const uint8_t *w_exp, mx_format_t fw,
                         int64_t N, const float *bias, float *y, int64_t ldy, void *workspace,
                         size_t workspace_bytes, mx_algo_t algo, void *stream)
{
    mx_status_t s = check_gemm_args(x, nullptr, fa, w_mant, w_exp, fw, M, N, K, bias, y, ldy);
    if (s != MX_OK) return s;
    if (dt != MX_F32 && dt != MX_BF16) return MX_ERR_FORMAT;
    if (fa.packing) return MX_ERR_FORMAT;                 // the activations are produced here: container form
    if (ldx < K) return MX_ERR_SHAPE;
    if ((ldx % 8) != 0) return MX_ERR_ALIGN;
    mx_linear_args_t one;
    one.x = x; one.dt = dt; one.M = M; one.K = K; one.ldx = ldx; one.fa = fa;
    one.w_mant = w_mant; one.w_exp = w_exp; one.fw = fw; one.N = N; one.bias = bias; one.y = y; one.ldy = ldy;
    if (fw.packing && algo != MX_ALGO_AUTO && algo != MX_ALGO_TCGEN05 && algo != MX_ALGO_TCGEN05_BLOCKWISE)
        return MX_ERR_FORMAT;
    const bool any_algo = algo == MX_ALGO_AUTO;
    if (algo == MX_ALGO_AUTO)
        algo = (stream_layer_ok(one) && (reinterpret_cast<uintptr_t>(w_exp) & 3u) == 0) ? MX_ALGO_STREAM
                                                                                     : MX_ALGO_TCGEN05;
    if (algo == MX_ALGO_STREAM) return grouped_impl(&one, 1, nullptr, any_algo, workspace, workspace_bytes, stream);
    if (algo != MX_ALGO_SIMT && algo != MX_ALGO_TCGEN05_FUSED && algo != MX_ALGO_TCGEN05 &&
        algo != MX_ALGO_TCGEN05_BLOCKWISE && algo != MX_ALGO_TCGEN05_MXF8)
        return MX_ERR_FORMAT;
    DeviceInfo *d = nullptr;
    s = device_info(&d);
    if (s != MX_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (!workspace) return MX_ERR_WORKSPACE;
    if (algo == MX_ALGO_TCGEN05_MXF8) {
        if (!mxf8_fits(fa, fw, K)) return MX_ERR_FORMAT;
        if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return MX_ERR_ALIGN;
        if (workspace_bytes < mxf8_operand_bytes(M, N, K) + packed_workspace(M, K, fa)) return MX_ERR_WORKSPACE;
        uint8_t *ws8 = static_cast<uint8_t *>(workspace);
        uint8_t *a_mant = ws8 + mxf8_operand_bytes(M, N, K);
        uint8_t *a_exp = a_mant + round256(mx_mant_bytes(M, K, fa));
        mx::QuantOut qo{a_mant, a_exp, nullptr, 0, nullptr};
        s = quantize_rows_any(x, dt, M, K, ldx, fa, qo, *d, st);
        if (s != MX_OK) return s;
        return run_tc8(a_mant, a_exp, fa, w_mant, w_exp, fw, M, N, K, bias, y, ldy, ws8, *d, st);
    }
    if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return MX_ERR_ALIGN;
    uint8_t *ws = static_cast<uint8_t *>(workspace);
    if (algo == MX_ALGO_SIMT) {
        if (workspace_bytes < packed_workspace(M, K, fa)) return MX_ERR_WORKSPACE;
        uint8_t *a_mant = ws;
        uint8_t *a_exp = ws + round256(mx_mant_bytes(M, K, fa));
        mx::QuantOut out{a_mant, a_exp, nullptr, 0, nullptr};
        s = quantize_rows_any(x, dt, M, K, ldx, fa, out, *d, st);
        if (s != MX_OK) return s;
        return mx_gemm_ex(a_mant, a_exp, fa, w_mant, w_exp, fw, M, N, K, bias, y, ldy, nullptr, 0,
                          MX_ALGO_SIMT, stream);
    }
    const bool fused = algo == MX_ALGO_TCGEN05_FUSED && (K % 32) == 0 && fw.block_rows == 1;
    if (fused && !fused_ok(K, w_exp)) return MX_ERR_ALIGN;
    if (workspace_bytes < (fused ? fused_workspace(M, K) : tc_workspace(M, N, K))) return MX_ERR_WORKSPACE;
    GemvPlan gemv;
    if (any_algo && gemv_is_faster(one) && gemv_plan(one, *d, &gemv)) return launch_gemv(one, gemv, *d, st);
    __nv_bfloat16 *a_hat = reinterpret_cast<__nv_bfloat16 *>(ws);
    // the activations' mantissas and exponents go straight to the MMA operand form (exact bf16)
    mx::QuantOut out{nullptr, nullptr, a_hat, K, nullptr};
    bool dec = false;
    DecPlan plan;
    if (any_algo) {
        s = dec_plan(M, N, K, fa, fw, w_exp, false, *d, &plan, &dec);
        if (s != MX_OK) return s;
    }
    if (dec) {
        out.xhat_perm = 1;
        s = quantize_rows_any(x, dt, M, K, ldx, fa, out, *d, st);
        if (s != MX_OK) return s;
        return launch_dec(plan, a_hat, w_mant, w_exp, fw, M, N, K, bias, y, ldy, nullptr, *d, st, EpiTail());
    }
    bool rec = false;
    if (any_algo && rec_fits(fa, fw, M, N, K)) {
        s = rec_is_faster(M, N, K, *d, &rec);
        if (s != MX_OK) return s;
    }
    if (rec) return run_rec_linear(one, bias, y, ldy, nullptr, ws, *d, st, EpiTail());
    if (fused) {
        // 4-bit weights and whole K steps: the lean in-kernel decode, which wants both operands in
        // its own K order inside every group of 8
        const bool perm = fw.elem_bits <= 4 && (K % 64) == 0;
        out.xhat_perm = perm ? 1 : 0;
        s = quantize_rows_any(x, dt, M, K, ldx, fa, out, *d, st);
        if (s != MX_OK) return s;
        return run_tc_fused(a_hat, w_mant, w_exp, fw, M, N, K, bias, y, ldy, *d, st, perm);
    }
    __nv_bfloat16 *w_hat = reinterpret_cast<__nv_bfloat16 *>(ws + round256((size_t)M * K * 2));
    s = tc_prepare(one, a_hat, w_hat, *d, st);
    if (s != MX_OK) return s;
    if (algo == MX_ALGO_TCGEN05_BLOCKWISE) return launch_tcx(a_hat, w_hat, M, N, K, fa.block, bias, y, ldy, *d, st);
    return run_tc(a_hat, w_hat, M, N, K, bias, y, ldy, *d, st, nullptr, TcBatch(), EpiTail(), any_algo);
}

mx_status_t mx_linear(const void *x, mx_dtype_t dt, int64_t M, int64_t K, int64_t ldx, mx_format_t fa,
                      const void *w_mant, const uint8_t *w_exp, mx_format_t fw, int64_t N,
                      const float *bias, float *y, int64_t ldy, void *workspace, size_t workspace_bytes,
                      void *stream)
{
    return mx_linear_ex(x, dt, M, K, ldx, fa, w_mant, w_exp, fw, N, bias, y, ldy, workspace,
                        workspace_bytes, MX_ALGO_AUTO, stream);
}

// ---- the layer with an MXInt result -------------------------------------------------------------
static mx_status_t check_quantized_out(mx_format_t fy, int64_t M, int64_t N, const void *y_mant, const uint8_t *y_exp)
{
    if (!y_mant || !y_exp) return MX_ERR_NULL;
    if (!format_ok(fy)) return MX_ERR_FORMAT;
    if ((N % fy.block) != 0 || (M % fy.block_rows) != 0) return MX_ERR_SHAPE;
    if (!aligned16(y_mant)) return MX_ERR_ALIGN;
    return MX_OK;
}

// Tensor-core product of packed operands with an fp32 (y) or MXInt (fy, y_mant, y_exp) result and an
// optional element-wise tail.
static mx_status_t gemm_tc_impl(const void *a_mant, const uint8_t *a_exp, mx_format_t fa, const void *w_mant,
                                const uint8_t *w_exp, mx_format_t fw, int64_t M, int64_t N, int64_t K,
                                const float *bias, const EpiTail &et, float *y, int64_t ldy, mx_format_t fy,
                                void *y_mant, uint8_t *y_exp, uint32_t *nonfinite_count, void *workspace,
                                size_t workspace_bytes, void *stream)
{
    // the output pointer checks (non-null, 16-byte aligned) apply to the mantissa array of an MXInt result
    mx_status_t s = check_gemm_args(a_mant, a_exp, fa, w_mant, w_exp, fw, M, N, K, bias,
                                    y ? y : static_cast<const float *>(y_mant), y ? ldy : N);
    if (s != MX_OK) return s;
    if (!a_exp) return MX_ERR_NULL;
    if (!y) {
        s = check_quantized_out(fy, M, N, y_mant, y_exp);
        if (s != MX_OK) return s;
    }
    DeviceInfo *d = nullptr;
    s = device_info(&d);
    if (s != MX_OK) return s;
    if (!workspace || workspace_bytes < tc_workspace(M, N, K)) return MX_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return MX_ERR_ALIGN;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    __nv_bfloat16 *a_hat = static_cast<__nv_bfloat16 *>(workspace);
    __nv_bfloat16 *w_hat = reinterpret_cast<__nv_bfloat16 *>(static_cast<uint8_t *>(workspace) +
                                                             round256((size_t)M * K * 2));
    QuantizedOut yq;
    yq.mant = static_cast<uint8_t *>(y_mant);
    yq.exps = y_exp;
    yq.nonfinite = nonfinite_count;
    yq.f = fy;
    bool dec = false;
    DecPlan plan;
    s = dec_plan(M, N, K, fa, fw, w_exp, !y, *d, &plan, &dec);
    if (s != MX_OK) return s;
    if (dec) {
        s = launch_dequant_bf16(a_mant, a_exp, M, K, fa, a_hat, K, *d, st, true);
        if (s != MX_OK) return s;
        return launch_dec(plan, a_hat, w_mant, w_exp, fw, M, N, K, bias, y, y ? ldy : N, y ? nullptr : &yq, *d, st, et);
    }
    bool rec = false;
    if (rec_fits(fa, fw, M, N, K)) {
        s = rec_is_faster(M, N, K, *d, &rec);
        if (s != MX_OK) return s;
    }
    if (rec)
        return run_rec_gemm(a_mant, a_exp, fa, w_mant, w_exp, fw, M, N, K, bias, y, y ? ldy : N, y ? nullptr : &yq,
                            static_cast<uint8_t *>(workspace), *d, st, et);
    s = launch_dequant_pair(a_mant, a_exp, fa, M, w_mant, w_exp, fw, N, K, a_hat, w_hat, *d, st);
    if (s != MX_OK) return s;
    if (y) return run_tc(a_hat, w_hat, M, N, K, bias, y, ldy, *d, st, nullptr, TcBatch(), et, true, true);
    return run_tc(a_hat, w_hat, M, N, K, bias, nullptr, N, *d, st, &yq, TcBatch(), et, true, true);
}

// The same for the layer: activations quantized on the fly.
// The operand pass with LayerNorm in front of the activation quantizer (see prep_ln_operands_kernel).
static mx_status_t tc_prepare_ln(const mx_linear_args_t &a, const mx_prologue_t &ln, __nv_bfloat16 *a_hat,
                                 __nv_bfloat16 *w_hat, DeviceInfo &d, cudaStream_t st, bool perm = false)
{
    mx::PrepLnJob j;
    j.x = static_cast<const float *>(a.x); j.M = a.M; j.K = a.K; j.ldx = a.ldx;
    j.gamma = ln.ln_gamma; j.beta = ln.ln_beta; j.eps = ln.ln_eps;
    j.wa = a.fa.elem_bits; j.block = a.fa.block; j.a_hat = a_hat;
    j.w_mant = static_cast<const uint8_t *>(a.w_mant); j.w_exp = a.w_exp; j.N = a.N; j.ww = a.fw.elem_bits;
    j.w_hat = w_hat; j.w_row_shift = a.fw.block_rows == 2 ? 1 : 0;
    j.perm = perm ? 1 : 0;
    const int per = (int)((a.K + mx::GLUE_THREADS - 1) / mx::GLUE_THREADS);
    const bool nib = a.fw.elem_bits <= 4;
    // a CTA per row, but a resident wave where the weights have that much work: a grid of few rows decodes them on few SMs, and
    // started beside a product that leaves some SMs free, several of its CTAs share one (64 tokens, hidden 4096, FFN 16384,
    // 8 x 8 bits, the whole block 640 -> 267 us)
    const int64_t rows = a.M < (int64_t)d.sm_count * 8 ? a.M : (int64_t)d.sm_count * 8;
    const int64_t decode = grid_for((a.N * (a.K / 32) + 1) / 2, mx::GLUE_THREADS, d.sm_count, 4);
    const unsigned g = (unsigned)(rows > decode ? rows : decode);
    ProfScope prof(KIND_PREP, st);
#define MX_LAUNCH_LN(P)                                                                                                  \
    do {                                                                                                                 \
        if (nib) MX_CUDA(launch_dep(mx::prep_ln_operands_kernel<P, true>, dim3(g), dim3(mx::GLUE_THREADS), 0, st, j));   \
        else MX_CUDA(launch_dep(mx::prep_ln_operands_kernel<P, false>, dim3(g), dim3(mx::GLUE_THREADS), 0, st, j));      \
    } while (0)
    if (per <= 4) MX_LAUNCH_LN(4);
    else if (per <= 8) MX_LAUNCH_LN(8);
    else if (per <= 16) MX_LAUNCH_LN(16);
    else MX_LAUNCH_LN(32);
#undef MX_LAUNCH_LN
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

static mx_status_t linear_tc_impl(const void *x, mx_dtype_t dt, int64_t M, int64_t K, int64_t ldx, mx_format_t fa,
                                  const void *w_mant, const uint8_t *w_exp, mx_format_t fw, int64_t N,
                                  const float *bias, const EpiTail &et, float *y, int64_t ldy, mx_format_t fy,
                                  void *y_mant, uint8_t *y_exp, uint32_t *nonfinite_count, void *workspace,
                                  size_t workspace_bytes, void *stream, const mx_prologue_t *ln = nullptr)
{
    mx_status_t s = check_gemm_args(x, nullptr, fa, w_mant, w_exp, fw, M, N, K, bias,
                                    y ? y : static_cast<const float *>(y_mant), y ? ldy : N);
    if (s != MX_OK) return s;
    if (dt != MX_F32 && dt != MX_BF16) return MX_ERR_FORMAT;
    if (fa.packing) return MX_ERR_FORMAT;
    if (ldx < K) return MX_ERR_SHAPE;
    if ((ldx % 8) != 0) return MX_ERR_ALIGN;
    if (!y) {
        s = check_quantized_out(fy, M, N, y_mant, y_exp);
        if (s != MX_OK) return s;
    }
    const bool with_ln = ln && ln->layernorm;
    if (with_ln) {
        // rows normalised in registers: fp32 input, rows of at most 8192 values, one-row container formats
        if (dt != MX_F32 || fa.block_rows != 1 || fw.packing) return MX_ERR_FORMAT;
        if ((K % 32) != 0 || K > mx::GLUE_THREADS * mx::GLUE_MAX_PER_THREAD) return MX_ERR_SHAPE;
    }
    DeviceInfo *d = nullptr;
    s = device_info(&d);
    if (s != MX_OK) return s;
    if (!workspace || workspace_bytes < tc_workspace(M, N, K)) return MX_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return MX_ERR_ALIGN;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    uint8_t *ws = static_cast<uint8_t *>(workspace);
    __nv_bfloat16 *a_hat = reinterpret_cast<__nv_bfloat16 *>(ws);
    __nv_bfloat16 *w_hat = reinterpret_cast<__nv_bfloat16 *>(ws + round256((size_t)M * K * 2));
    mx_linear_args_t one;
    one.x = x; one.dt = dt; one.M = M; one.K = K; one.ldx = ldx; one.fa = fa;
    one.w_mant = w_mant; one.w_exp = w_exp; one.fw = fw; one.N = N; one.bias = bias; one.y = y; one.ldy = y ? ldy : N;
    QuantizedOut yq;
    yq.mant = static_cast<uint8_t *>(y_mant);
    yq.exps = y_exp;
    yq.nonfinite = nonfinite_count;
    yq.f = fy;
    bool dec = false;
    DecPlan plan;
    s = dec_plan(M, N, K, fa, fw, w_exp, !y, *d, &plan, &dec);
    if (s != MX_OK) return s;
    if (dec) {
        if (with_ln) {
            mx_linear_args_t rows = one;
            rows.N = 0;                                   // the activations alone
            s = tc_prepare_ln(rows, *ln, a_hat, w_hat, *d, st, true);
        } else {
            s = quantize_rows_any(x, dt, M, K, ldx, fa, mx::QuantOut{nullptr, nullptr, a_hat, K, nullptr, 1}, *d, st);
        }
        if (s != MX_OK) return s;
        return launch_dec(plan, a_hat, w_mant, w_exp, fw, M, N, K, bias, y, y ? ldy : N, y ? nullptr : &yq, *d, st, et);
    }
    bool rec = false;
    if (!with_ln && rec_fits(fa, fw, M, N, K)) {
        s = rec_is_faster(M, N, K, *d, &rec);
        if (s != MX_OK) return s;
    }
    if (rec)
        return run_rec_linear(one, bias, y, y ? ldy : N, y ? nullptr : &yq, ws, *d, st, et);
    if (with_ln) {
        s = tc_prepare_ln(one, *ln, a_hat, w_hat, *d, st);
    } else {
        s = tc_prepare(one, a_hat, w_hat, *d, st);
    }
    if (s != MX_OK) return s;
    if (y) return run_tc(a_hat, w_hat, M, N, K, bias, y, ldy, *d, st, nullptr, TcBatch(), et);
    return run_tc(a_hat, w_hat, M, N, K, bias, nullptr, N, *d, st, &yq, TcBatch(), et);
}

mx_status_t mx_gemm_q(const void *a_mant, const uint8_t *a_exp, mx_format_t fa, const void *w_mant,
                      const uint8_t *w_exp, mx_format_t fw, int64_t M, int64_t N, int64_t K,
                      const float *bias, mx_format_t fy, void *y_mant, uint8_t *y_exp,
                      uint32_t *nonfinite_count, void *workspace, size_t workspace_bytes, void *stream)
{
    if (!y_mant) return MX_ERR_NULL;
    return gemm_tc_impl(a_mant, a_exp, fa, w_mant, w_exp, fw, M, N, K, bias, EpiTail(), nullptr, 0, fy, y_mant, y_exp,
                        nonfinite_count, workspace, workspace_bytes, stream);
}

mx_status_t mx_linear_q(const void *x, mx_dtype_t dt, int64_t M, int64_t K, int64_t ldx, mx_format_t fa,
                        const void *w_mant, const uint8_t *w_exp, mx_format_t fw, int64_t N,
                        const float *bias, mx_format_t fy, void *y_mant, uint8_t *y_exp,
                        uint32_t *nonfinite_count, void *workspace, size_t workspace_bytes, void *stream)
{
    if (!y_mant) return MX_ERR_NULL;
    return linear_tc_impl(x, dt, M, K, ldx, fa, w_mant, w_exp, fw, N, bias, EpiTail(), nullptr, 0, fy, y_mant, y_exp,
                          nonfinite_count, workspace, workspace_bytes, stream);
}

// ---- the product with a fused element-wise tail ---------------------------------------------------
static mx_status_t tail_of(const mx_epilogue_t *ep, int64_t N, const float *y, const void *y_mant, const float **bias,
                           EpiTail *et)
{
    if ((y != nullptr) == (y_mant != nullptr)) return MX_ERR_NULL;        // exactly one kind of result
    *bias = nullptr;
    *et = EpiTail();
    if (!ep) return MX_OK;
    *bias = ep->bias;
    et->relu = ep->relu ? 1 : 0;
    et->residual = ep->residual;
    et->ldr = ep->ldr;
    if (ep->residual && ep->ldr < N) return MX_ERR_SHAPE;
    if (ep->residual && (reinterpret_cast<uintptr_t>(ep->residual) & 3u) != 0) return MX_ERR_ALIGN;
    return MX_OK;
}

mx_status_t mx_gemm_fused(const void *a_mant, const uint8_t *a_exp, mx_format_t fa, const void *w_mant,
                          const uint8_t *w_exp, mx_format_t fw, int64_t M, int64_t N, int64_t K,
                          const mx_epilogue_t *ep, float *y, int64_t ldy, mx_format_t fy, void *y_mant,
                          uint8_t *y_exp, void *workspace, size_t workspace_bytes, void *stream)
{
    const float *bias;
    EpiTail et;
    const mx_status_t s = tail_of(ep, N, y, y_mant, &bias, &et);
    if (s != MX_OK) return s;
    return gemm_tc_impl(a_mant, a_exp, fa, w_mant, w_exp, fw, M, N, K, bias, et, y, ldy, fy, y_mant, y_exp, nullptr,
                        workspace, workspace_bytes, stream);
}

mx_status_t mx_linear_fused(const void *x, mx_dtype_t dt, int64_t M, int64_t K, int64_t ldx, mx_format_t fa,
                            const mx_prologue_t *pro, const void *w_mant, const uint8_t *w_exp, mx_format_t fw,
                            int64_t N, const mx_epilogue_t *ep, float *y, int64_t ldy, mx_format_t fy, void *y_mant,
                            uint8_t *y_exp, void *workspace, size_t workspace_bytes, void *stream)
{
    const float *bias;
    EpiTail et;
    const mx_status_t s = tail_of(ep, N, y, y_mant, &bias, &et);
    if (s != MX_OK) return s;
    return linear_tc_impl(x, dt, M, K, ldx, fa, w_mant, w_exp, fw, N, bias, et, y, ldy, fy, y_mant, y_exp, nullptr,
                          workspace, workspace_bytes, stream, pro);
}

// ---- decode: few tokens, weights streamed once ------------------------------------------------
size_t mx_linear_grouped_workspace_bytes(const mx_linear_args_t *layers, int32_t n_layers)
{
    if (!layers || n_layers <= 0) return 0;
    for (int i = 0; i < n_layers; ++i)
        if (!format_ok(layers[i].fa) || !format_ok(layers[i].fw)) return 0;
    try {
        std::vector<int> owner;
        activation_owners(layers, n_layers, owner);
        return grouped_workspace(layers, n_layers, owner);
    } catch (const std::bad_alloc &) {                  // no C++ exception leaves a C function
        return 0;
    }
}

// packed_exps == nullptr: layers[i].x are floating-point activations, quantized here.
// packed_exps != nullptr: layers[i].x are mantissas already in format fa, packed_exps[i] their exponents.
// any_order: the algorithm was left open (MX_ALGO_AUTO), K may be cut over a cluster.
static mx_status_t grouped_impl(const mx_linear_args_t *layers, int32_t n_layers,
                                const uint8_t *const *packed_exps, bool any_order, void *workspace, size_t workspace_bytes,
                                void *stream)
try {
    if (!layers) return MX_ERR_NULL;
    if (n_layers <= 0) return MX_ERR_SHAPE;
    int max_t = 0, max_nb = 0;
    for (int i = 0; i < n_layers; ++i) {
        const mx_linear_args_t &a = layers[i];
        mx_status_t s = check_gemm_args(a.x, nullptr, a.fa, a.w_mant, a.w_exp, a.fw, a.M, a.N, a.K, a.bias,
                                        a.y, a.ldy);
        if (s != MX_OK) return s;
        if (!packed_exps && a.dt != MX_F32 && a.dt != MX_BF16) return MX_ERR_FORMAT;
        if (packed_exps && !packed_exps[i]) return MX_ERR_NULL;
        if (!packed_exps && a.ldx < a.K) return MX_ERR_SHAPE;
        if ((!packed_exps && (a.ldx % 8) != 0) || (reinterpret_cast<uintptr_t>(a.w_exp) & 3u) != 0) return MX_ERR_ALIGN;
        if (!stream_layer_ok(a)) return a.M > 16 || (a.K % 128) != 0 ? MX_ERR_SHAPE : MX_ERR_FORMAT;
        max_t = a.M > max_t ? (int)a.M : max_t;
        const int nb = (int)(a.K / 32);
        max_nb = nb > max_nb ? nb : max_nb;
    }
    std::vector<int> owner;
    if (!packed_exps) activation_owners(layers, n_layers, owner);
    const size_t need = packed_exps ? stream_table_bytes(n_layers) : grouped_workspace(layers, n_layers, owner);
    if (!workspace || workspace_bytes < need) return MX_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return MX_ERR_ALIGN;
    const int nt = max_t > 8 ? 2 : 1;
    constexpr size_t SMEM = 227u * 1024u;
    StreamPlan plan;
    plan.smem = nt == 2 ? mx::StreamCfg<2>::smem_bytes(max_nb) : mx::StreamCfg<1>::smem_bytes(max_nb);
    if (plan.smem > SMEM) return MX_ERR_SHAPE;                     // tokens x K too large to stage
    DeviceInfo *d = nullptr;
    mx_status_t s = device_info(&d);
    if (s != MX_OK) return s;
    // K is cut over the warps of a CTA only when the row tiles alone cannot fill the GPU; the pieces are whole units in every layer
    auto choose_split = [&](int64_t tiles, int64_t warp_slots, int unit, int least) {      // least: blocks in a piece
        for (int cand = 8; tiles < warp_slots && cand > 1; cand >>= 1) {
            bool fits = cand <= 4 || tiles * 4 < warp_slots;
            for (int i = 0; i < n_layers && fits; ++i) fits = (layers[i].K / 32) % (unit * cand) == 0 && layers[i].K / 32 >= least * cand;
            if (fits) return cand;
        }
        return 1;
    };
    // whole steps of the TMA kernels with exponent bytes of one row per weight row at 16-byte offsets
    bool whole = true;
    int64_t sum_weights = 0;
    for (int i = 0; i < n_layers; ++i) {
        whole = whole && (layers[i].K % 512) == 0 && (reinterpret_cast<uintptr_t>(layers[i].w_exp) & 15u) == 0 && layers[i].fw.block_rows == 1;
        sum_weights += layers[i].N * layers[i].K;
    }
    const bool boxes = whole && max_t <= 2;              // exponents in boxes as well (gemv_stream32_kernel)
    // one layer, algorithm open: one launch -- but for one token of a large one and two of one with very many rows, where the row-per-lane
    // kernel's loads run ahead over more rows (K x N, one token: 4096 x 11008 8.9 against 10.2 us, 8192 x 16384 15.6 / 19.0,
    // 4096 x 32000 14.6 / 20.0, but 4096 x 4096 5.5 / 5.7 and on the host one launch less; two: 4096 x 32000 18.6 / 22.0,
    // 8192 x 16384 20.8 / 21.4, 4096 x 11008 11.0 / 10.3, 8192 x 8192 14.6 / 11.9)
    if (any_order && n_layers == 1 && !packed_exps) {
        GemvPlan g;
        const int64_t n = layers[0].N, weights = n * layers[0].K;
        const bool rows = boxes && (max_t == 1 ? weights >= (1 << 25) : n >= 24576 && weights >= (1 << 26));
        if (!rows && gemv_plan(layers[0], *d, &g)) return launch_gemv(layers[0], g, *d, static_cast<cudaStream_t>(stream));
    }
    auto take = [&](StreamPlan::Kind kind, int warps, int stages, int rows, int unit, size_t smem) {
        if (plan.kind != StreamPlan::REGS || smem > SMEM) return;
        plan.kind = kind; plan.warps = warps; plan.stages = stages; plan.rows = rows; plan.unit = unit; plan.smem = smem;
    };
    for (int n = mx::Stream32Cfg<1>::MAX_STAGES; boxes && n >= 2; --n)       // with as many stages as fit beside the tokens
        take(StreamPlan::ROWS32, mx::Stream32Cfg<1>::WARPS, n, 32, 16,
             max_t == 1 ? mx::Stream32Cfg<1>::smem_bytes(max_nb, n) : mx::Stream32Cfg<2>::smem_bytes(max_nb, n));
    auto mma_smem = [&](int warps, int stages) {                             // (8: any cut)
        return nt == 2 ? mx::MmaStreamCfg::smem_bytes<2>(max_nb / 4, warps, stages, 8) : mx::MmaStreamCfg::smem_bytes<1>(max_nb / 4, warps, stages, 8);
    };
    // Few weights in rows of partial steps: the register variant, whose CTAs of eight warps spread the tiles over more of the chip
    // and start without barriers (registers / MMA, us, B200, K x N: packed tokens, one layer, 4 tokens of 1152 x 3072 7.7 / 9.5,
    // 2176 x 8192 12.4 / 13.0, 4224 x 4096 21.3 / 20.3, 16 of 640 x 640 6.9 / 10.5, of 1152 x 3072 10.3 / 11.3; twelve layers of
    // 640 x 640 14.4 / 15.7, four of 1152 x 3072 11.0 / 11.2, twelve 18.5 / 17.6; beyond 8 tokens 15.4 / 16.6, 13.9 / 13.0, 26.8 / 18.5)
    const bool few = !whole && (max_t <= 8 ? sum_weights < (1 << 23) : sum_weights < (max_nb < 768 / 32 ? 1 << 23 : packed_exps ? 1 << 22 : 0));
    for (int warps = 16; warps >= 8 && !few; warps -= 8)
        for (int n = mx::MmaStreamCfg::MAX_STAGES; n >= 2; --n) take(StreamPlan::MMA, warps, n, 16, 16, mma_smem(warps, n));
    const bool tma = plan.kind != StreamPlan::REGS;
    cudaStream_t st = static_cast<cudaStream_t>(stream);

    // quantize every distinct activation tensor once, build the device layer table
    uint8_t *ws = static_cast<uint8_t *>(workspace);
    size_t off = stream_table_bytes(n_layers);
    const size_t tmap_off = round256((size_t)n_layers * sizeof(mx::StreamLayer));
    const size_t job_off = tmap_off + round256((size_t)n_layers * 2 * sizeof(CUtensorMap));
    // one image of the three tables (layers, tensor maps, quantization jobs), laid out as in the workspace; a call of few
    // layers passes the first two as launch parameters instead
    const bool in_params = n_layers <= mx::STREAM_INLINE_LAYERS;
    mx::StreamInlineParams sp;
    // (in units that are aligned as its strictest member is: a vector of bytes starts on 16 bytes only)
    struct alignas(64) ImageLine { uint8_t bytes[64]; };
    static_assert(alignof(ImageLine) >= alignof(CUtensorMap) && alignof(ImageLine) >= alignof(mx::StreamLayer) &&
                  alignof(ImageLine) >= alignof(mx::QuantJob), "the tables are written in place");
    std::vector<ImageLine> image_lines(in_params ? 0 : off / sizeof(ImageLine));       // off: a multiple of 256
    uint8_t *image = reinterpret_cast<uint8_t *>(image_lines.data());
    mx::StreamLayer *table = in_params ? sp.inline_layers : reinterpret_cast<mx::StreamLayer *>(image);
    CUtensorMap *tmaps = in_params ? sp.inline_maps : reinterpret_cast<CUtensorMap *>(image + tmap_off);
    std::vector<mx::QuantJob> jobs, pair_jobs;          // (pair_jobs: pairs of tokens share their exponents)
    bool any_dt[2] = {false, false};
    int64_t max_chunks = 0;
    std::vector<uint8_t *> act_ptr((size_t)n_layers, nullptr);
    std::unique_lock<std::mutex> map_lock(g_wmap_mu, std::defer_lock);
    if (tma) map_lock.lock();
    int total_tiles = 0;
    for (int i = 0; i < n_layers; ++i) {
        const mx_linear_args_t &a = layers[i];
        if (!packed_exps) act_ptr[i] = act_ptr[owner[i]];
        if (!act_ptr[i] && !packed_exps) {
            act_ptr[i] = ws + off;
            off += stream_act_bytes(a);
            mx::QuantJob job;
            job.x = a.x;
            job.rows = a.M;
            job.K = a.K;
            job.ldx = a.ldx;
            job.w = a.fa.elem_bits;
            job.block = a.fa.block;
            job.dt = a.dt == MX_F32 ? 0 : 1;
            job.out = mx::QuantOut{act_ptr[i], act_ptr[i] + round256(mx_mant_bytes(a.M, a.K, a.fa)), nullptr, 0, nullptr};
            if (a.fa.block_rows == 2) {
                pair_jobs.push_back(job);
            } else {
                jobs.push_back(job);
                any_dt[job.dt] = true;
                const int64_t chunks = a.M * (a.K / 8);
                max_chunks = chunks > max_chunks ? chunks : max_chunks;
            }
        }
        mx::StreamLayer &L = table[i];
        L.w_mant = static_cast<const uint8_t *>(a.w_mant);
        L.w_exp = a.w_exp;
        L.a_mant = packed_exps ? static_cast<const uint8_t *>(a.x) : act_ptr[i];
        L.a_exp = packed_exps ? packed_exps[i] : act_ptr[i] + round256(mx_mant_bytes(a.M, a.K, a.fa));
        L.bias = a.bias;
        L.y = a.y;
        L.ldy = a.ldy;
        L.N = (int)a.N;
        L.K = (int)a.K;
        L.T = (int)a.M;
        L.a_bits = a.fa.elem_bits;
        L.w_bits = a.fw.elem_bits;
        L.w_rows2 = a.fw.block_rows == 2 ? 1 : 0;
        L.a_rows2 = a.fa.block_rows == 2 ? 1 : 0;
        L.tile_begin = total_tiles;
        L.n_tiles = (int)((a.N + plan.rows - 1) / plan.rows);
        total_tiles += L.n_tiles;
        if (tma) {
            s = packed_weight_maps(a.w_mant, a.w_exp, a.N, a.K / 2, plan.kind == StreamPlan::ROWS32 ? a.K / 32 : 0, &tmaps[(size_t)i * 2]);
            if (s != MX_OK) return s;
        }
    }
    // nothing is launched under the lock: a launch may wait for room in its stream, and other threads' calls with it
    if (tma) map_lock.unlock();
    auto quantize_one = [&](const mx::QuantJob &q, int block_rows) {
        mx_format_t f{};
        f.block = q.block; f.elem_bits = q.w; f.exp_bits = 8; f.block_rows = block_rows;
        return quantize_rows_any(q.x, q.dt == 0 ? MX_F32 : MX_BF16, q.rows, q.K, q.ldx, f, q.out, *d, st);
    };
    // the activations: one tensor, with its sizes as launch parameters; several, by one launch per input type over a table
    const size_t n_jobs = jobs.size() > 1 ? jobs.size() : 0;
    if (!in_params || n_jobs) {          // a captured copy would read this call's tables at every replay, long after they are gone
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) {
            (void)cudaGetLastError();
        } else if (cap != cudaStreamCaptureStatusNone) {
            snprintf(t_cuda_error, sizeof(t_cuda_error), "grouped call: its tables are copied from host memory of the call, which a stream capture cannot hold "
                     "(capture calls of up to %d layers with one activation tensor)", mx::STREAM_INLINE_LAYERS);
            return MX_ERR_CUDA;
        }
    }
    for (const mx::QuantJob &q : pair_jobs) {            // the two-row quantizer, one launch per tensor
        s = quantize_one(q, 2);
        if (s != MX_OK) return s;
    }
    if (!in_params) {
        if (n_jobs) memcpy(image + job_off, jobs.data(), n_jobs * sizeof(mx::QuantJob));
        // in pieces of at most 64 KB: those travel with the commands, a larger pageable copy goes through the copy engine and
        // its staging buffer (192 matrices, 66 KB: the call 531 instead of 522 us)
        const size_t total = job_off + n_jobs * sizeof(mx::QuantJob), piece = 64 * 1024;
        for (size_t at = 0; at < total; at += piece)
            MX_CUDA(cudaMemcpyAsync(ws + at, image + at, total - at < piece ? total - at : piece, cudaMemcpyHostToDevice, st));
    } else if (n_jobs) {
        MX_CUDA(cudaMemcpyAsync(ws + job_off, jobs.data(), n_jobs * sizeof(mx::QuantJob), cudaMemcpyHostToDevice, st));
    }
    if (jobs.size() == 1) {
        s = quantize_one(jobs[0], 1);
        if (s != MX_OK) return s;
    }
    if (n_jobs) {
        const mx::QuantJob *dj = reinterpret_cast<const mx::QuantJob *>(ws + job_off);
        const dim3 qgrid((unsigned)grid_for((max_chunks + 1) / 2, 256, d->sm_count, 8), (unsigned)n_jobs);
        if (any_dt[0]) {
            ProfScope prof(KIND_QUANTIZE, st);
            MX_CUDA(launch_dep(mx::quantize_multi_kernel<float, 0>, dim3(qgrid), dim3(256), 0, st, dj));
        }
        if (any_dt[1]) {
            ProfScope prof(KIND_QUANTIZE, st);
            MX_CUDA(launch_dep(mx::quantize_multi_kernel<__nv_bfloat16, 1>, dim3(qgrid), dim3(256), 0, st, dj));
        }
        MX_CUDA(cudaGetLastError());
    }

    const int fit = (int)(SMEM / (plan.smem + 1024));
    const int ctas_per_sm = plan.kind == StreamPlan::MMA || fit < 1 ? 1 : fit < 4 ? fit : 4;
    const int max_ctas = d->sm_count * ctas_per_sm;
    int split = choose_split(total_tiles, (int64_t)max_ctas * plan.warps, plan.unit, plan.unit);
    // (a piece of less than a step costs a step: four layers of 512 x 4096, 3 tokens, in four pieces 10.0 us, not cut 7.9)
    if (split == 1 && plan.kind == StreamPlan::MMA) split = choose_split(total_tiles, (int64_t)max_ctas * plan.warps, 4, 16);
    const int tpr = plan.warps / split;
    const int rounds = (total_tiles + tpr - 1) / tpr;
    const int grid = rounds < max_ctas ? rounds : max_ctas;
    const int early = packed_exps ? 0 : 1;      // the launch in front is the quantizer above: weights may be fetched meanwhile
    sp.layers = reinterpret_cast<const mx::StreamLayer *>(ws);          // (unused by a call that brings them along)
    sp.n_layers = n_layers;
    sp.total_tiles = total_tiles;
    sp.split = split;
    sp.max_nb = max_nb;
    sp.status = d->status;
    sp.tmaps = reinterpret_cast<const CUtensorMap *>(ws + tmap_off);
    if (in_params) return launch_stream(plan, max_t, early, sp, grid, *d, st);
    mx::StreamTableParams tp;
    static_cast<mx::StreamParams &>(tp) = sp;
    return launch_stream(plan, max_t, early, tp, grid, *d, st);
} catch (const std::bad_alloc &) {                      // (the tables of the call are kept in host memory)
    snprintf(t_cuda_error, sizeof(t_cuda_error), "grouped call: out of host memory for the tables of %d layers", (int)n_layers);
    return MX_ERR_CUDA;
}

mx_status_t mx_linear_grouped(const mx_linear_args_t *layers, int32_t n_layers, void *workspace,
                              size_t workspace_bytes, void *stream)
{
    return grouped_impl(layers, n_layers, nullptr, false, workspace, workspace_bytes, stream);
}

// ---- batched product (per-head attention matmuls) ------------------------------------------------
size_t mx_gemm_batched_workspace_bytes(int64_t M, int64_t N, int64_t K, int64_t batch)
{
    if (M <= 0 || N <= 0 || K <= 0 || batch <= 0) return 0;
    return (size_t)batch * (round256((size_t)M * K * 2) + round256((size_t)N * K * 2));
}

mx_status_t mx_gemm_batched(const void *a_mant, const uint8_t *a_exp, mx_format_t fa, int64_t lda,
                            int64_t stride_a, const void *w_mant, const uint8_t *w_exp, mx_format_t fw,
                            int64_t ldw, int64_t stride_w, int64_t M, int64_t N, int64_t K, int64_t batch,
                            float *y, int64_t ldy, int64_t stride_y, void *workspace,
                            size_t workspace_bytes, void *stream)
{
    mx_status_t s = check_gemm_args(a_mant, a_exp, fa, w_mant, w_exp, fw, M, N, K, nullptr, y, ldy);
    if (s != MX_OK) return s;
    if (!a_exp) return MX_ERR_NULL;
    if (fa.packing || fw.packing) return MX_ERR_FORMAT;
    if (batch <= 0 || lda < K || ldw < K || stride_a < 0 || stride_w < 0 || stride_y < 0) return MX_ERR_SHAPE;
    // row and batch strides must keep whole blocks and whole container bytes together
    if ((lda % fa.block) || (ldw % fw.block) || (stride_a % fa.block) || (stride_w % fw.block) ||
        (lda % 8) || (ldw % 8) || (stride_a % 8) || (stride_w % 8) || (stride_y % 4))
        return MX_ERR_ALIGN;
    if (!workspace || workspace_bytes < mx_gemm_batched_workspace_bytes(M, N, K, batch)) return MX_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return MX_ERR_ALIGN;
    DeviceInfo *d = nullptr;
    s = device_info(&d);
    if (s != MX_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t a_item = round256((size_t)M * K * 2), w_item = round256((size_t)N * K * 2);
    __nv_bfloat16 *a_hat = static_cast<__nv_bfloat16 *>(workspace);
    __nv_bfloat16 *w_hat = reinterpret_cast<__nv_bfloat16 *>(static_cast<uint8_t *>(workspace) + (size_t)batch * a_item);
    // two-row blocks: an item must start on an even row of the packed tensor
    if ((fa.block_rows == 2 && ((stride_a / lda) & 1)) || (fw.block_rows == 2 && ((stride_w / ldw) & 1))) return MX_ERR_ALIGN;
    auto strides = [](const mx_format_t &f, int64_t ld, int64_t bstride, size_t out_item) {
        mx::PackedStrides ps;
        ps.mant_ld = f.elem_bits <= 4 ? ld / 2 : ld;
        ps.exp_ld = ld / f.block;
        ps.mant_batch = f.elem_bits <= 4 ? bstride / 2 : bstride;
        ps.perm = 0;
        ps.exp_row_shift = f.block_rows == 2 ? 1 : 0;   // rows 2i, 2i+1 read one row of exponent bytes
        // an item starts (bstride / ld) rows down and (bstride % ld) elements into the row
        ps.exp_batch = ((bstride / ld) >> ps.exp_row_shift) * (ld / f.block) + (bstride % ld) / f.block;
        ps.out_batch = (int64_t)(out_item / 2);
        return ps;
    };
    // one decode launch per operand and one product launch cover every batch item
    s = launch_dequant_bf16(a_mant, a_exp, M, K, fa, a_hat, K, strides(fa, lda, stride_a, a_item), batch, *d, st);
    if (s != MX_OK) return s;
    s = launch_dequant_bf16(w_mant, w_exp, N, K, fw, w_hat, K, strides(fw, ldw, stride_w, w_item), batch, *d, st);
    if (s != MX_OK) return s;
    TcBatch tb;
    tb.count = batch;
    tb.a_item = a_item;
    tb.w_item = w_item;
    tb.y_batch = stride_y;
    // one chain of K steps per output, however many items the call has
    return run_tc(a_hat, w_hat, M, N, K, nullptr, y, ldy, *d, st, nullptr, tb, EpiTail(), false);
}

// ---- fused attention ---------------------------------------------------------------------------
extern "C++" {
// The fused attention kernel on operands already in bf16 operand form: q_hat, k_hat [seq, hid], v_hat [hid, seq].
template <int D>
static mx_status_t launch_attention_d(const __nv_bfloat16 *q_hat, const __nv_bfloat16 *k_hat, const __nv_bfloat16 *v_hat,
                                      int64_t seq, int64_t heads, float scale, int causal, mx_format_t fp, float *ctx,
                                      int64_t ldc, void *p_mant_out, uint8_t *p_exp_out, DeviceInfo *d, cudaStream_t st)
{
    using Cfg = mx::AttnCfgT<D>;
    const int64_t hid = heads * D;
    CUtensorMap tm_q, tm_k, tm_v;
    mx_status_t s = encode_bf16_rows(&tm_q, q_hat, seq, hid, 128);
    if (s != MX_OK) return s;
    s = encode_bf16_rows(&tm_k, k_hat, seq, hid, 128);
    if (s != MX_OK) return s;
    s = encode_bf16_rows(&tm_v, v_hat, hid, seq, D);
    if (s != MX_OK) return s;
    s = smem_attr_once(d->attn_attr_set[D == 128 ? 0 : 1], mx::attention_kernel<D>, (int)Cfg::SMEM_BYTES);
    if (s != MX_OK) return s;
    mx::AttnParams ap;
    ap.ctx = ctx;
    ap.ldc = ldc;
    ap.seq = (int)seq;
    ap.heads = (int)heads;
    ap.scale = scale;
    ap.causal = causal ? 1 : 0;
    ap.p_bits = fp.elem_bits;
    ap.p_block = fp.block;
    ap.p_mant = static_cast<uint8_t *>(p_mant_out);
    ap.p_exp = p_exp_out;
    ap.status = d->status;
    const int64_t items = ((seq + Cfg::BQ - 1) / Cfg::BQ) * heads;
    const int grid = items < d->sm_count ? (int)items : d->sm_count;
    ProfScope prof(KIND_GEMM_TC, st);
    MX_CUDA(launch_dep(mx::attention_kernel<D>, dim3(grid), dim3(Cfg::THREADS), Cfg::SMEM_BYTES, st, tm_q, tm_k, tm_v, ap));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

static mx_status_t launch_attention(const __nv_bfloat16 *q_hat, const __nv_bfloat16 *k_hat, const __nv_bfloat16 *v_hat,
                                    int64_t seq, int64_t heads, int64_t head_dim, float scale, int causal, mx_format_t fp,
                                    float *ctx, int64_t ldc, void *p_mant_out, uint8_t *p_exp_out, DeviceInfo *d,
                                    cudaStream_t st)
{
    if (head_dim == 64)
        return launch_attention_d<64>(q_hat, k_hat, v_hat, seq, heads, scale, causal, fp, ctx, ldc, p_mant_out, p_exp_out, d, st);
    return launch_attention_d<128>(q_hat, k_hat, v_hat, seq, heads, scale, causal, fp, ctx, ldc, p_mant_out, p_exp_out, d, st);
}

}  // extern "C++"

size_t mx_attention_workspace_bytes(int64_t seq, int64_t heads, int64_t head_dim)
{
    if (seq <= 0 || heads <= 0 || head_dim <= 0) return 0;
    return 3 * round256((size_t)seq * heads * head_dim * 2);
}

mx_status_t mx_attention(const void *q_mant, const uint8_t *q_exp, const void *k_mant, const uint8_t *k_exp, mx_format_t fqk,
                         const void *vt_mant, const uint8_t *vt_exp, mx_format_t fv, int64_t seq, int64_t heads,
                         int64_t head_dim, float scale, int causal, mx_format_t fp, float *ctx, int64_t ldc,
                         void *p_mant_out, uint8_t *p_exp_out, void *workspace, size_t workspace_bytes, void *stream)
{
    if (!q_mant || !q_exp || !k_mant || !k_exp || !vt_mant || !vt_exp || !ctx) return MX_ERR_NULL;
    if ((p_mant_out == nullptr) != (p_exp_out == nullptr)) return MX_ERR_NULL;
    if (!format_1d(fqk) || !format_1d(fv) || !format_1d(fp)) return MX_ERR_FORMAT;
    const int64_t hid = heads * head_dim;
    if (seq <= 0 || heads <= 0 || (head_dim != 128 && head_dim != 64) || (seq % 32) != 0 || ldc < hid ||
        seq > INT32_MAX / 4 || hid > INT32_MAX / 4 || !(scale > 0.f))
        return MX_ERR_SHAPE;
    if (!aligned16(q_mant) || !aligned16(k_mant) || !aligned16(vt_mant) || !aligned16(ctx) || (ldc % 4) != 0 ||
        (p_mant_out && !aligned16(p_mant_out)))
        return MX_ERR_ALIGN;
    if (!workspace || workspace_bytes < mx_attention_workspace_bytes(seq, heads, head_dim)) return MX_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return MX_ERR_ALIGN;
    DeviceInfo *d = nullptr;
    mx_status_t s = device_info(&d);
    if (s != MX_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t one = round256((size_t)seq * hid * 2);
    uint8_t *ws = static_cast<uint8_t *>(workspace);
    __nv_bfloat16 *q_hat = reinterpret_cast<__nv_bfloat16 *>(ws), *k_hat = reinterpret_cast<__nv_bfloat16 *>(ws + one),
                  *v_hat = reinterpret_cast<__nv_bfloat16 *>(ws + 2 * one);
    s = launch_dequant_bf16(q_mant, q_exp, seq, hid, fqk, q_hat, hid, *d, st);
    if (s != MX_OK) return s;
    s = launch_dequant_bf16(k_mant, k_exp, seq, hid, fqk, k_hat, hid, *d, st);
    if (s != MX_OK) return s;
    s = launch_dequant_bf16(vt_mant, vt_exp, hid, seq, fv, v_hat, seq, *d, st);
    if (s != MX_OK) return s;
    return launch_attention(q_hat, k_hat, v_hat, seq, heads, head_dim, scale, causal, fp, ctx, ldc, p_mant_out, p_exp_out, d, st);
}

mx_status_t mx_attention_fp(const void *q, const void *k, const void *v, mx_dtype_t dt, int64_t ldq, int64_t ldk,
                            int64_t ldv, mx_format_t fqk, mx_format_t fv, int64_t seq, int64_t heads, int64_t head_dim,
                            float scale, int causal, mx_format_t fp, float *ctx, int64_t ldc, void *workspace,
                            size_t workspace_bytes, void *stream)
{
    if (!q || !k || !v || !ctx) return MX_ERR_NULL;
    if (dt != MX_F32 && dt != MX_BF16) return MX_ERR_FORMAT;
    if (!format_1d(fqk) || !format_1d(fv) || !format_1d(fp) || fqk.packing || fv.packing) return MX_ERR_FORMAT;
    const int64_t hid = heads * head_dim;
    if (seq <= 0 || heads <= 0 || (head_dim != 128 && head_dim != 64) || (seq % 32) != 0 || ldc < hid || ldq < hid ||
        ldk < hid || ldv < hid || seq > INT32_MAX / 4 || hid > INT32_MAX / 4 || !(scale > 0.f))
        return MX_ERR_SHAPE;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(ctx) || (ldc % 4) != 0 || (ldq % 8) != 0 ||
        (ldk % 8) != 0 || (ldv % 8) != 0)
        return MX_ERR_ALIGN;
    if (!workspace || workspace_bytes < mx_attention_workspace_bytes(seq, heads, head_dim)) return MX_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return MX_ERR_ALIGN;
    DeviceInfo *d = nullptr;
    mx_status_t s = device_info(&d);
    if (s != MX_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t one = round256((size_t)seq * hid * 2);
    uint8_t *ws = static_cast<uint8_t *>(workspace);
    __nv_bfloat16 *q_hat = reinterpret_cast<__nv_bfloat16 *>(ws), *k_hat = reinterpret_cast<__nv_bfloat16 *>(ws + one),
                  *v_hat = reinterpret_cast<__nv_bfloat16 *>(ws + 2 * one);
    // one launch for the three operands: q and k in blocks along the head dimension, v in blocks along the tokens
    // (the slow axis of v) and written transposed, [hid, seq]; all straight to the operand form
    {
        mx::AttnOperandsJob j;
        j.q = q; j.k = k; j.v = v;
        j.seq = seq; j.hid = hid; j.ldq = ldq; j.ldk = ldk; j.ldv = ldv;
        j.block_qk = fqk.block; j.w_qk = fqk.elem_bits; j.block_v = fv.block; j.w_v = fv.elem_bits;
        j.q_hat = q_hat; j.k_hat = k_hat; j.v_hat = v_hat;
        const int64_t items = 2 * seq * ((hid + 255) / 256) + ((hid + 31) / 32) * (seq / 32);
        const int64_t want = (items + 7) / 8;                                                // 8 warps per CTA
        const int per_sm = dt == MX_F32 ? resident_ctas(mx::attention_operands_kernel<float>)
                                        : resident_ctas(mx::attention_operands_kernel<__nv_bfloat16>);
        const int64_t cap = (int64_t)d->sm_count * per_sm;
        const int grid = (int)(want < cap ? want : cap);
        ProfScope prof(KIND_QUANTIZE, st);
        if (dt == MX_F32) MX_CUDA(launch_dep(mx::attention_operands_kernel<float>, dim3(grid), dim3(256), 0, st, j));
        else MX_CUDA(launch_dep(mx::attention_operands_kernel<__nv_bfloat16>, dim3(grid), dim3(256), 0, st, j));
        MX_CUDA(cudaGetLastError());
    }
    return launch_attention(q_hat, k_hat, v_hat, seq, heads, head_dim, scale, causal, fp, ctx, ldc, nullptr, nullptr, d, st);
}

// ---- fp32 glue of the transformer block ---------------------------------------------------------
mx_status_t mx_layernorm(const float *x, int64_t ldx, const float *gamma, const float *beta, float eps,
                         int64_t rows, int64_t cols, float *y, int64_t ldy, void *stream)
{
    if (!x || !y) return MX_ERR_NULL;
    if (rows < 0 || cols <= 0 || ldx < cols || ldy < cols || cols > mx::GLUE_THREADS * mx::GLUE_MAX_PER_THREAD)
        return MX_ERR_SHAPE;
    if (rows == 0) return MX_OK;
    DeviceInfo *d = nullptr;
    mx_status_t s = device_info(&d);
    if (s != MX_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int per = (int)((cols + mx::GLUE_THREADS - 1) / mx::GLUE_THREADS);
    const unsigned g = (unsigned)rows;
    ProfScope prof(KIND_GLUE, st);
    if (per <= 4) mx::layernorm_kernel<4><<<g, mx::GLUE_THREADS, 0, st>>>(x, ldx, gamma, beta, eps, (int)cols, y, ldy);
    else if (per <= 8) mx::layernorm_kernel<8><<<g, mx::GLUE_THREADS, 0, st>>>(x, ldx, gamma, beta, eps, (int)cols, y, ldy);
    else if (per <= 16) mx::layernorm_kernel<16><<<g, mx::GLUE_THREADS, 0, st>>>(x, ldx, gamma, beta, eps, (int)cols, y, ldy);
    else mx::layernorm_kernel<32><<<g, mx::GLUE_THREADS, 0, st>>>(x, ldx, gamma, beta, eps, (int)cols, y, ldy);
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

mx_status_t mx_softmax(float *s_inout, int64_t ld, int64_t rows, int64_t cols, float scale, int causal,
                       int64_t rows_per_batch, void *stream)
{
    if (!s_inout) return MX_ERR_NULL;
    if (rows < 0 || cols <= 0 || ld < cols || cols > mx::GLUE_THREADS * mx::GLUE_MAX_PER_THREAD ||
        (causal && rows_per_batch <= 0))
        return MX_ERR_SHAPE;
    if (rows == 0) return MX_OK;
    DeviceInfo *d = nullptr;
    mx_status_t s = device_info(&d);
    if (s != MX_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int per = (int)((cols + mx::GLUE_THREADS - 1) / mx::GLUE_THREADS);
    const unsigned g = (unsigned)rows;
    ProfScope prof(KIND_GLUE, st);
    if (per <= 4) mx::softmax_kernel<4><<<g, mx::GLUE_THREADS, 0, st>>>(s_inout, ld, (int)cols, scale, causal, rows_per_batch);
    else if (per <= 8) mx::softmax_kernel<8><<<g, mx::GLUE_THREADS, 0, st>>>(s_inout, ld, (int)cols, scale, causal, rows_per_batch);
    else if (per <= 16) mx::softmax_kernel<16><<<g, mx::GLUE_THREADS, 0, st>>>(s_inout, ld, (int)cols, scale, causal, rows_per_batch);
    else mx::softmax_kernel<32><<<g, mx::GLUE_THREADS, 0, st>>>(s_inout, ld, (int)cols, scale, causal, rows_per_batch);
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

mx_status_t mx_softmax_q(const float *s_in, int64_t ld, int64_t rows, int64_t cols, float scale, int causal,
                         int64_t rows_per_batch, mx_format_t fp, void *p_mant, uint8_t *p_exp, void *stream)
{
    if (!s_in || !p_mant || !p_exp) return MX_ERR_NULL;
    if (!format_1d(fp)) return MX_ERR_FORMAT;
    if (rows < 0 || cols <= 0 || ld < cols || cols > mx::GLUE_THREADS * mx::GLUE_MAX_PER_THREAD ||
        (cols % fp.block) != 0 || (causal && rows_per_batch <= 0))
        return MX_ERR_SHAPE;
    if (!aligned16(s_in) || !aligned16(p_mant) || (ld % 4) != 0) return MX_ERR_ALIGN;
    if (rows == 0) return MX_OK;
    DeviceInfo *d = nullptr;
    mx_status_t st_ = device_info(&d);
    if (st_ != MX_OK) return st_;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int per8 = (int)((cols / 8 + mx::GLUE_THREADS - 1) / mx::GLUE_THREADS);      // 1..4
    const unsigned g = (unsigned)rows;
    uint8_t *pm = static_cast<uint8_t *>(p_mant);
    ProfScope prof(KIND_GLUE, st);
#define MX_SOFTMAX_Q(P8)                                                                                         \
    do {                                                                                                         \
        if (fp.block == 16)                                                                                      \
            mx::softmax_q_kernel<P8, 16><<<g, mx::GLUE_THREADS, 0, st>>>(s_in, ld, (int)cols, scale, causal,     \
                                                                         rows_per_batch, fp.elem_bits, pm, p_exp); \
        else                                                                                                     \
            mx::softmax_q_kernel<P8, 32><<<g, mx::GLUE_THREADS, 0, st>>>(s_in, ld, (int)cols, scale, causal,     \
                                                                         rows_per_batch, fp.elem_bits, pm, p_exp); \
    } while (0)
    if (per8 <= 1) MX_SOFTMAX_Q(1);
    else if (per8 <= 2) MX_SOFTMAX_Q(2);
    else MX_SOFTMAX_Q(4);
#undef MX_SOFTMAX_Q
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

mx_status_t mx_relu_add(const float *a, const float *b, float *y, int64_t n, int relu, void *stream)
{
    if (!a || !y) return MX_ERR_NULL;
    if (n < 0) return MX_ERR_SHAPE;
    if (!aligned16(a) || !aligned16(y) || (b && !aligned16(b))) return MX_ERR_ALIGN;
    if (n == 0) return MX_OK;
    DeviceInfo *d = nullptr;
    mx_status_t s = device_info(&d);
    if (s != MX_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    ProfScope prof(KIND_GLUE, st);
    mx::relu_add_kernel<<<grid_for((n + 3) / 4, mx::GLUE_THREADS, d->sm_count, 8), mx::GLUE_THREADS, 0, st>>>(a, b, y, n, relu);
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

// ---- Block Minifloat / Block Logarithm ---------------------------------------------------------
static bool alt_format_ok(const mx_alt_format_t &f)
{
    if (f.block != 16 && f.block != 32) return false;
    if (f.kind == MX_ELEM_BMF)
        return f.elem_exp_bits >= 1 && f.elem_exp_bits <= 5 && f.elem_man_bits >= 1 &&
               1 + f.elem_exp_bits + f.elem_man_bits <= 8;
    if (f.kind == MX_ELEM_BL) return f.elem_exp_bits >= 1 && f.elem_exp_bits <= 5 && f.elem_man_bits == 0;
    return false;
}
static mx::AltFormat alt_of(const mx_alt_format_t &f)
{
    return mx::AltFormat{f.kind, f.block, f.elem_exp_bits, f.elem_man_bits};
}

mx_status_t mx_alt_quantize(const void *x, mx_dtype_t dt, int64_t rows, int64_t K, int64_t ldx, mx_alt_format_t f,
                            uint8_t *codes, uint8_t *shared, uint32_t *nonfinite_count, void *stream)
{
    if (!alt_format_ok(f) || (dt != MX_F32 && dt != MX_BF16)) return MX_ERR_FORMAT;
    if (rows < 0 || K < 0 || (K % f.block) != 0 || ldx < K) return MX_ERR_SHAPE;
    if (rows == 0 || K == 0) return MX_OK;
    if (!x || !codes || !shared) return MX_ERR_NULL;
    if (!aligned16(x) || !aligned16(codes) || (ldx % 8) != 0) return MX_ERR_ALIGN;
    DeviceInfo *d = nullptr;
    mx_status_t s = device_info(&d);
    if (s != MX_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int64_t items = rows * ((K / 8 + 31) / 32);
    const int grid = grid_for(items * 32, 256, d->sm_count, 8);
    const mx::AltFormat af = alt_of(f);
    ProfScope prof(KIND_QUANTIZE, st);
    if (dt == MX_F32) {
        const float *xf = static_cast<const float *>(x);
        if (f.block == 16) MX_CUDA(launch_dep(mx::alt_quantize_kernel<float, 16>, dim3(grid), dim3(256), 0, st, xf, rows, K, ldx, af, codes, shared, nonfinite_count));
        else MX_CUDA(launch_dep(mx::alt_quantize_kernel<float, 32>, dim3(grid), dim3(256), 0, st, xf, rows, K, ldx, af, codes, shared, nonfinite_count));
    } else {
        const __nv_bfloat16 *xb = static_cast<const __nv_bfloat16 *>(x);
        if (f.block == 16) MX_CUDA(launch_dep(mx::alt_quantize_kernel<__nv_bfloat16, 16>, dim3(grid), dim3(256), 0, st, xb, rows, K, ldx, af, codes, shared, nonfinite_count));
        else MX_CUDA(launch_dep(mx::alt_quantize_kernel<__nv_bfloat16, 32>, dim3(grid), dim3(256), 0, st, xb, rows, K, ldx, af, codes, shared, nonfinite_count));
    }
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

static mx_status_t alt_decode_any(const uint8_t *codes, const uint8_t *shared, int64_t rows, int64_t K,
                                  const mx_alt_format_t &f, void *out, mx_dtype_t dt, int64_t ld_out, DeviceInfo &d,
                                  cudaStream_t st)
{
    const int grid = grid_for(rows * (K / 8), 256, d.sm_count, 8);
    const mx::AltFormat af = alt_of(f);
    ProfScope prof(KIND_DEQUANTIZE, st);
    if (dt == MX_F32)
        MX_CUDA(launch_dep(mx::alt_decode_kernel<float>, dim3(grid), dim3(256), 0, st, codes, shared, rows, K, af,
                           static_cast<float *>(out), ld_out));
    else
        MX_CUDA(launch_dep(mx::alt_decode_kernel<__nv_bfloat16>, dim3(grid), dim3(256), 0, st, codes, shared, rows, K, af,
                           static_cast<__nv_bfloat16 *>(out), ld_out));
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

mx_status_t mx_alt_dequantize(const uint8_t *codes, const uint8_t *shared, int64_t rows, int64_t K, mx_alt_format_t f,
                              void *out, mx_dtype_t dt, int64_t ld_out, void *stream)
{
    if (!codes || !shared || !out) return MX_ERR_NULL;
    if (!alt_format_ok(f) || (dt != MX_F32 && dt != MX_BF16)) return MX_ERR_FORMAT;
    if (rows < 0 || K < 0 || (K % f.block) != 0 || ld_out < K) return MX_ERR_SHAPE;
    if (!aligned16(codes) || !aligned16(out) || (ld_out % 8) != 0) return MX_ERR_ALIGN;
    if (rows == 0 || K == 0) return MX_OK;
    DeviceInfo *d = nullptr;
    mx_status_t s = device_info(&d);
    if (s != MX_OK) return s;
    return alt_decode_any(codes, shared, rows, K, f, out, dt, ld_out, *d, static_cast<cudaStream_t>(stream));
}

size_t mx_alt_gemm_workspace_bytes(int64_t M, int64_t N, int64_t K)
{
    if (M <= 0 || N <= 0 || K <= 0) return 0;
    return tc_operand_bytes(M, N, K);
}

mx_status_t mx_alt_gemm(const uint8_t *a_codes, const uint8_t *a_shared, mx_alt_format_t fa, const uint8_t *w_codes,
                        const uint8_t *w_shared, mx_alt_format_t fw, int64_t M, int64_t N, int64_t K, const float *bias,
                        float *y, int64_t ldy, void *workspace, size_t workspace_bytes, void *stream)
{
    if (!a_codes || !a_shared || !w_codes || !w_shared || !y) return MX_ERR_NULL;
    if (!alt_format_ok(fa) || !alt_format_ok(fw) || fa.block != fw.block) return MX_ERR_FORMAT;
    if (M <= 0 || N <= 0 || K <= 0 || (K % fa.block) != 0 || ldy < N) return MX_ERR_SHAPE;
    if (M > INT32_MAX / 2 || N > INT32_MAX / 2 || K > INT32_MAX / 2) return MX_ERR_SHAPE;
    if (!aligned16(a_codes) || !aligned16(w_codes) || !aligned16(y) || (bias && !aligned16(bias))) return MX_ERR_ALIGN;
    if (!workspace || workspace_bytes < tc_operand_bytes(M, N, K)) return MX_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return MX_ERR_ALIGN;
    DeviceInfo *d = nullptr;
    mx_status_t s = device_info(&d);
    if (s != MX_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    __nv_bfloat16 *a_hat = static_cast<__nv_bfloat16 *>(workspace);
    __nv_bfloat16 *w_hat = reinterpret_cast<__nv_bfloat16 *>(static_cast<uint8_t *>(workspace) + round256((size_t)M * K * 2));
    s = alt_decode_any(a_codes, a_shared, M, K, fa, a_hat, MX_BF16, K, *d, st);
    if (s != MX_OK) return s;
    s = alt_decode_any(w_codes, w_shared, N, K, fw, w_hat, MX_BF16, K, *d, st);
    if (s != MX_OK) return s;
    return run_tc(a_hat, w_hat, M, N, K, bias, y, ldy, *d, st, nullptr, TcBatch(), EpiTail(), true, true);
}

// ---- product without any allocation ---------------------------------------------------------
// Scratch for mx_gemm_static: a fixed array in the library's device image.  In host code the
// name below is only a handle for the runtime, never a device address; the address a kernel can
// use comes from cudaGetSymbolAddress, looked up once per device with that device current.
static __device__ __align__(256) unsigned char g_static_scratch[MX_STATIC_SCRATCH_BYTES];
static void *g_static_scratch_addr[MAX_DEVICES] = {nullptr};

mx_status_t mx_gemm_static(const void *a_mant, const uint8_t *a_exp, mx_format_t fa,
                           const void *w_mant, const uint8_t *w_exp, mx_format_t fw, int64_t M,
                           int64_t N, int64_t K, const float *bias, float *y, int64_t ldy,
                           void *stream)
{
    mx_status_t s = check_gemm_args(a_mant, a_exp, fa, w_mant, w_exp, fw, M, N, K, bias, y, ldy);
    if (s != MX_OK) return s;
    if (!a_exp) return MX_ERR_NULL;
    if (fa.block_rows != 1 || fw.block_rows != 1 || fa.packing || fw.packing) return MX_ERR_FORMAT;
    const size_t need = tc_operand_bytes(M, N, K);
    if (need > (size_t)MX_STATIC_SCRATCH_BYTES) {
        snprintf(t_cuda_error, sizeof(t_cuda_error),
                 "mx_gemm_static: M=%lld N=%lld K=%lld needs %zu bytes of scratch, the built-in array holds %zu",
                 (long long)M, (long long)N, (long long)K, need, (size_t)MX_STATIC_SCRATCH_BYTES);
        return MX_ERR_WORKSPACE;
    }
    DeviceInfo *d = nullptr;
    s = device_info(&d);
    if (s != MX_OK) return s;
    int dev = 0;
    MX_CUDA(cudaGetDevice(&dev));
    {
        std::lock_guard<std::mutex> lk(g_init_mu);
        if (!g_static_scratch_addr[dev]) {          // set-up: first call on this device
            void *p = nullptr;
            MX_CUDA(cudaGetSymbolAddress(&p, g_static_scratch));
            g_static_scratch_addr[dev] = p;
        }
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    uint8_t *scratch = static_cast<uint8_t *>(g_static_scratch_addr[dev]);
    __nv_bfloat16 *a_hat = reinterpret_cast<__nv_bfloat16 *>(scratch);
    __nv_bfloat16 *w_hat = reinterpret_cast<__nv_bfloat16 *>(scratch + round256((size_t)M * K * 2));
    // Decode both operands into the scratch (every byte the product reads is written here first,
    // so nothing left by an earlier call is ever observed), then the tensor-core product.
    // Launches are issued directly: no event, no buffer and no handle is created on this path.
    mx::dequantize_kernel<__nv_bfloat16><<<grid_for(M * (K / 8), 256, d->sm_count, 16), 256, 0, st>>>(
        static_cast<const uint8_t *>(a_mant), a_exp, M, K, fa.block, fa.elem_bits, a_hat, K, dense_strides(K, fa));
    MX_CUDA(cudaGetLastError());
    mx::dequantize_kernel<__nv_bfloat16><<<grid_for(N * (K / 8), 256, d->sm_count, 16), 256, 0, st>>>(
        static_cast<const uint8_t *>(w_mant), w_exp, N, K, fw.block, fw.elem_bits, w_hat, K, dense_strides(K, fw));
    MX_CUDA(cudaGetLastError());
    TcBatch opt;
    opt.no_events = true;
    return launch_tc<128, mx::W_BF16>(a_hat, w_hat, PackedW(), M, N, K, bias, y, ldy, nullptr, *d, st, opt);
}

mx_status_t mx_profile_begin(void)
{
    std::lock_guard<std::mutex> lk(g_prof.mu);
    for (const ProfEntry &e : g_prof.entries) g_prof.pool.push_back(e);
    g_prof.entries.clear();
    g_prof.on = true;
    return MX_OK;
}

mx_status_t mx_profile_end(double *ms_per_kind, int64_t *launches_per_kind)
{
    if (!ms_per_kind || !launches_per_kind) return MX_ERR_NULL;
    std::lock_guard<std::mutex> lk(g_prof.mu);
    g_prof.on = false;
    for (int k = 0; k < MX_KERNEL_KINDS; ++k) {
        ms_per_kind[k] = 0.0;
        launches_per_kind[k] = 0;
    }
    mx_status_t rc = MX_OK;
    for (const ProfEntry &e : g_prof.entries) {
        float ms = 0.f;
        cudaError_t err = cudaEventSynchronize(e.b);
        if (err == cudaSuccess) err = cudaEventElapsedTime(&ms, e.a, e.b);
        if (err != cudaSuccess) rc = cuda_fail(err, "mx_profile_end");
        if (e.kind >= 0 && e.kind < MX_KERNEL_KINDS) {
            ms_per_kind[e.kind] += ms;
            launches_per_kind[e.kind] += 1;
        }
        g_prof.pool.push_back(e);
    }
    g_prof.entries.clear();
    return rc;
}

// One warp waits, with the library's bounded wait, on a barrier that nothing ever arrives on.
__global__ void wait_probe_kernel(uint32_t *status, uint64_t limit_ns)
{
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t abort_flag;
    if (threadIdx.x == 0) {
        mx::ptx::mbar_init(mx::ptx::smem_u32(&bar), 1);
        abort_flag = 0;
        mx::ptx::fence_mbar_init();
    }
    __syncthreads();
    const bool ok = mx::ptx::mbar_wait_bounded(mx::ptx::smem_u32(&bar), 0u, &abort_flag, limit_ns);
    if (!ok && threadIdx.x == 0) atomicOr(status, mx::STATUS_TIMEOUT_BIT);
}

mx_status_t mx_selftest_wait_expiry(uint32_t limit_us, void *stream)
{
    if (limit_us == 0 || limit_us > 100000u) return MX_ERR_SHAPE;       // at most 0.1 s
    DeviceInfo *d = nullptr;
    mx_status_t s = device_info(&d);
    if (s != MX_OK) return s;
    wait_probe_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(d->status, (uint64_t)limit_us * 1000ull);
    MX_CUDA(cudaGetLastError());
    return MX_OK;
}

mx_status_t mx_selftest_route(int64_t M, int64_t N, int64_t K, mx_format_t fa, mx_format_t fw, int32_t quantized, mx_algo_t algo,
                               int32_t *route)
{
    if (!route) return MX_ERR_NULL;
    if (!format_ok_any(fa) || !format_ok_any(fw) || fa.block != fw.block || (algo != MX_ALGO_AUTO && algo != MX_ALGO_TCGEN05)) return MX_ERR_FORMAT;
    if (M <= 32 || N <= 0 || K <= 0 || (K % fa.block) != 0 || M > INT32_MAX / 2 || N > INT32_MAX / 2 || K > INT32_MAX / 2) return MX_ERR_SHAPE;
    DeviceInfo *d = nullptr;
    mx_status_t s = device_info(&d);
    if (s != MX_OK) return s;
    bool dec = false, rec = false;
    DecPlan plan;
    const bool any = algo == MX_ALGO_AUTO;
    if (any) s = dec_plan(M, N, K, fa, fw, nullptr, quantized != 0, *d, &plan, &dec);
    if (s != MX_OK) return s;
    if (dec) {
        route[0] = plan.tokens ? 2 : 1;
        route[1] = plan.tokens ? plan.tokens : mx::DecCfg::BN;
        route[2] = plan.split;
        return MX_OK;
    }
    if (any && rec_fits(fa, fw, M, N, K)) {
        s = rec_is_faster(M, N, K, *d, &rec);
        if (s != MX_OK) return s;
    }
    TcRoute r;
    s = tc_route(M, N, K, 1, any, *d, &r);
    if (s != MX_OK) return s;
    route[0] = rec ? 3 : (int)r.kernel;
    route[1] = rec ? 256 : r.width;
    route[2] = rec ? 1 : r.split;
    return MX_OK;
}

mx_status_t mx_poll_status(void *stream)
{
    DeviceInfo *d = nullptr;
    mx_status_t s = device_info(&d);
    if (s != MX_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    MX_CUDA(cudaStreamSynchronize(st));
    uint32_t word = 0;
    MX_CUDA(cudaMemcpy(&word, d->status, sizeof(word), cudaMemcpyDeviceToHost));
    if (word != 0) {
        const uint32_t zero = 0;
        MX_CUDA(cudaMemcpy(d->status, &zero, sizeof(zero), cudaMemcpyHostToDevice));
    }
    return (word & mx::STATUS_TIMEOUT_BIT) ? MX_ERR_TIMEOUT : MX_OK;
}

}  // extern "C"
