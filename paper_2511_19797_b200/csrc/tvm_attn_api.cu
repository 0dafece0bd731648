// C-ABI entry points of the attention-JVP library (see include/tvm_attn.h): argument checks, TMA
// tensor-map construction and kernel launches.  No device memory is allocated here.
#include "tvm_attn.h"

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cmath>
#include <cstring>
#include <mutex>
#include <utility>

#include "jvp_sm100.cuh"
#include "qk_rmsnorm.cuh"
#include "rowsums.cuh"
#include "simt_kernels.cuh"

namespace tvm_attn {

static std::atomic<uint64_t> g_launches{0};

__device__ int g_status_word = 0;  // raised by a tensor-core kernel whose bounded wait ran out

// What a call needs to know about the current device, looked up once per thread and CUDA context (the lookups cost a
// small call as much as a launch): a context's id is never used again in a process, so a device reset or a switch of
// devices is a new lookup.
struct DeviceFacts {
    unsigned long long ctx = 0;
    int sms = 0, major = 0;
    int* status = nullptr;   // device address of g_status_word
};

// Driver functions, by the runtime's entry-point lookup (the library does not link the driver).
template <typename F>
static F driver_function(const char* name) {
    void* sym = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint(name, &sym, cudaEnableDefault, &qres) != cudaSuccess || qres != cudaDriverEntryPointSuccess) return nullptr;
    return reinterpret_cast<F>(sym);
}

// Id of the calling thread's CUDA context, initialising the device if it has none yet; 0 on error.
static unsigned long long context_id() {
    static const auto get_current = driver_function<CUresult (*)(CUcontext*)>("cuCtxGetCurrent");
    static const auto get_id = driver_function<CUresult (*)(CUcontext, unsigned long long*)>("cuCtxGetId");
    if (!get_current || !get_id) return 0;
    CUcontext ctx = nullptr;
    if (get_current(&ctx) != CUDA_SUCCESS) return 0;
    if (!ctx) {
        // A thread's first CUDA call: the device it is on becomes current.  Not by cudaFree(nullptr), which invalidates the stream
        // captures under way, of other threads too.
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaSetDevice(dev) != cudaSuccess || get_current(&ctx) != CUDA_SUCCESS || !ctx) return 0;
    }
    unsigned long long id = 0;
    return get_id(ctx, &id) == CUDA_SUCCESS ? id : 0;
}

static const DeviceFacts* device_facts() {
    thread_local DeviceFacts facts;
    const unsigned long long ctx = context_id();
    if (ctx == 0) return nullptr;
    if (facts.ctx == ctx) return &facts;
    DeviceFacts f;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&f.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&f.major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess || f.sms <= 0 ||
        cudaGetSymbolAddress(reinterpret_cast<void**>(&f.status), g_status_word) != cudaSuccess || !f.status)
        return nullptr;
    f.ctx = ctx;
    facts = f;
    return &facts;
}

// The facts of a device that runs the tensor-core kernels.
static int tensor_core_device(const DeviceFacts** f) {
    *f = device_facts();
    return !*f ? TVM_ATTN_CUDA_ERROR : (*f)->major == 10 ? TVM_ATTN_OK : TVM_ATTN_UNSUPPORTED;
}

// Prepares a tensor-core kernel for launches, once per thread and context (KERN is its identity): its dynamic shared
// memory, and a check that it was compiled to the registers its warpgroups redistribute (fewer would make them wait for
// registers that do not exist).
template <auto KERN>
static bool prepare_kernel(const DeviceFacts& f, int smem_bytes) {
    thread_local unsigned long long done = 0;
    if (done == f.ctx) return true;
    cudaFuncAttributes attr;
    if (cudaFuncGetAttributes(&attr, KERN) != cudaSuccess || attr.numRegs != JVP_REGS || attr.sharedSizeBytes != 0) return false;
    if (cudaFuncSetAttribute(KERN, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes) != cudaSuccess) return false;
    done = f.ctx;
    return true;
}

// Optional per-kernel timing: events recorded around each launch of the most recent call.  While it is
// disabled (the normal state) a call only reads the atomic flag, so concurrent calls from several host
// threads do not touch shared state; while it is enabled the library is to be driven by one thread.
struct Profiler {
    std::atomic<bool> enabled{false};
    std::atomic<int> count{0};  // kernels recorded by the last call
    cudaEvent_t ev[8] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
    void begin_call() { if (enabled.load(std::memory_order_relaxed)) count.store(0); }
    void mark(cudaStream_t st, int idx) {
        if (idx >= 8) return;
        if (!ev[idx] && cudaEventCreate(&ev[idx]) != cudaSuccess) { ev[idx] = nullptr; return; }
        cudaEventRecord(ev[idx], st);
    }
    void before(cudaStream_t st) { if (enabled.load(std::memory_order_relaxed) && count.load() == 0) mark(st, 0); }
    void after(cudaStream_t st) { if (enabled.load(std::memory_order_relaxed)) { mark(st, count.load() + 1); count.fetch_add(1); } }
};
static Profiler g_prof;

struct Shape {
    int B, H, N, M, d, dp;   // N keys, M queries per head
    long long BH;
    float alpha;
    bool fp32, simt;
    Geom q, k;               // query side (M rows) and key side (N rows)
    bool plain;              // self-attention on packed (B, H, N, d) tensors
};

// Strides of one side: all zero selects the packed (B, H, rows, d) layout.
static int side_geometry(const int64_t st[3], int rows, int H, int d, Geom* g) {
    g->rows = rows;
    if (st[0] == 0 && st[1] == 0 && st[2] == 0) {
        g->rs = d; g->hs = (long long)rows * d; g->bs = (long long)H * rows * d;
        return TVM_ATTN_OK;
    }
    // rows must not overlap inside themselves and every row must start on a 16-byte boundary (TMA, vector loads)
    if (st[0] < d || st[1] <= 0 || st[2] <= 0 || st[0] % 8 || st[1] % 8 || st[2] % 8) return TVM_ATTN_INVALID_ARG;
    if (st[0] > (1LL << 36) || st[1] > (1LL << 36) || st[2] > (1LL << 36)) return TVM_ATTN_UNSUPPORTED;  // TMA strides < 2^40 bytes
    g->rs = st[0]; g->hs = st[1]; g->bs = st[2];
    return TVM_ATTN_OK;
}

static int check_params(const tvm_attn_params* p, Shape* s) {
    if (!p) return TVM_ATTN_INVALID_ARG;
    if (p->B <= 0 || p->H <= 0 || p->N <= 0 || p->d <= 0 || p->M < 0) return TVM_ATTN_INVALID_ARG;
    if (p->dtype != TVM_ATTN_BF16 && p->dtype != TVM_ATTN_FP32) return TVM_ATTN_INVALID_ARG;
    if (p->flags & ~TVM_ATTN_FLAG_CUDA_CORES) return TVM_ATTN_INVALID_ARG;
    if (!(p->scale >= 0.0f) || !std::isfinite(p->scale)) return TVM_ATTN_INVALID_ARG;
    if (p->d > 128 || p->d % 8 != 0) return TVM_ATTN_UNSUPPORTED;
    s->B = p->B; s->H = p->H; s->N = p->N; s->d = p->d;
    s->M = p->M > 0 ? p->M : p->N;
    int rg = side_geometry(p->q_strides, s->M, p->H, p->d, &s->q);
    if (rg != TVM_ATTN_OK) return rg;
    rg = side_geometry(p->k_strides, s->N, p->H, p->d, &s->k);
    if (rg != TVM_ATTN_OK) return rg;
    s->plain = s->M == s->N && s->q.rs == s->d && s->k.rs == s->d && s->q.hs == (long long)s->N * s->d && s->k.hs == s->q.hs &&
               s->q.bs == (long long)s->H * s->N * s->d && s->k.bs == s->q.bs;
    s->dp = (p->d + 15) / 16 * 16;
    s->BH = (long long)p->B * p->H;
    s->alpha = p->scale == 0.0f ? 1.0f / std::sqrt((float)p->d) : p->scale;
    s->fp32 = p->dtype == TVM_ATTN_FP32;
    s->simt = s->fp32 || (p->flags & TVM_ATTN_FLAG_CUDA_CORES);
    // every kernel flattens (head, row tile) into blockIdx.x
    const long long longer = s->M > s->N ? s->M : s->N;
    const long long tiles16 = (longer + 15LL) / 16;
    if (s->BH * tiles16 > 2147483647LL) return TVM_ATTN_UNSUPPORTED;
    if (s->BH > 2147483647LL / longer) return TVM_ATTN_UNSUPPORTED;  // B*H*rows indexable as int
    return TVM_ATTN_OK;
}

static bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

static int cuda_status(cudaError_t e) { return e == cudaSuccess ? TVM_ATTN_OK : TVM_ATTN_CUDA_ERROR; }

// ------------------------------------------------------------------------------------------------
// CUDA-core path
template <typename T>
static int simt_fwd(const Shape& s, const void* Q, const void* K, const void* V, const void* tQ, const void* tK,
                    const void* tV, void* O, void* tO, float* lse, float* mu, cudaStream_t st) {
    const size_t smem = simt_smem_bytes(s.d, 2);
    cudaError_t e = cudaFuncSetAttribute(simt_fwd_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return TVM_ATTN_CUDA_ERROR;
    const unsigned grid = (unsigned)(s.BH * ((s.M + SIMT_ROWS - 1) / SIMT_ROWS));
    g_prof.before(st);
    simt_fwd_kernel<T><<<grid, SIMT_THREADS, smem, st>>>((const T*)Q, (const T*)K, (const T*)V, (const T*)tQ,
                                                         (const T*)tK, (const T*)tV, (T*)O, (T*)tO, lse, mu, s.q, s.k, s.H,
                                                         s.d, s.alpha);
    g_prof.after(st);
    g_launches += 1;
    return cuda_status(cudaGetLastError());
}

static bool q_packed(const Shape& s) {
    return s.q.rs == s.d && s.q.hs == (long long)s.M * s.d && s.q.bs == (long long)s.H * s.M * s.d;
}

// launch(chunks a lane, whether a last lane has one less, lanes a row) for the split of rows of d elements, the first two as
// types: the streaming kernels exist for the splits that a head dim has.
template <typename T, int CMAX, int C = CMAX, typename F>
static int with_split(int d, const F& launch) {
    if constexpr (C == 0) {
        return TVM_ATTN_UNSUPPORTED;
    } else {
        const int cpr = d * (int)sizeof(T) / 16;   // 16-byte chunks per row (d % 8 == 0)
        const RmsSplit split = rms_split(cpr, CMAX);
        const bool ragged = split.C * split.P > cpr;
        if constexpr (rms_split_exists<T>(CMAX, C, false))
            if (split.C == C && !ragged) return launch(std::integral_constant<int, C>(), std::false_type(), split.P);
        if constexpr (rms_split_exists<T>(CMAX, C, true))
            if (split.C == C && ragged) return launch(std::integral_constant<int, C>(), std::true_type(), split.P);
        return with_split<T, CMAX, C - 1>(d, launch);
    }
}

template <typename T>
static int launch_rowsums(const Shape& s, const void* G, const void* Hc, const void* O, const void* tO, const float* lse,
                          float* sig1, float* cvec, float* lse2, float sign, cudaStream_t st) {
    const long long rows = s.BH * s.M;           // fit 31 bits
    return with_split<T, 4>(s.d, [&](auto C, auto ragged, int P) {
        const long long rows_per_block = (ROWSUM_THREADS / 32) * (32 / P), blocks = (rows + rows_per_block - 1) / rows_per_block;
        g_prof.before(st);
        bwd_rowsums_kernel<T, C(), ragged()><<<(unsigned)(blocks < ROWSUM_BLOCKS ? blocks : ROWSUM_BLOCKS), ROWSUM_THREADS, 0, st>>>(
            (const T*)G, (const T*)Hc, (const T*)O, (const T*)tO, lse, sig1, cvec, lse2, (unsigned)rows, s.q, q_packed(s) ? 0 : s.H, s.d, P, sign);
        g_prof.after(st);
        g_launches += 1;
        return cuda_status(cudaGetLastError());
    });
}

template <typename T>
static int simt_bwd(const Shape& s, const void* Q, const void* K, const void* V, const void* tQ, const void* tK,
                    const void* tV, const float* lse, const float* mu, const void* G, const void* Hc,
                    const float* sig1, const float* cvec, void* dQ, void* dK, void* dV, void* dtQ, void* dtK, void* dtV,
                    cudaStream_t st) {
    const size_t smem = simt_smem_bytes(s.d, 4);
    if (cudaFuncSetAttribute(simt_bwd_dq_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaFuncSetAttribute(simt_bwd_dkv_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return TVM_ATTN_CUDA_ERROR;
    const unsigned grid_q = (unsigned)(s.BH * ((s.M + SIMT_ROWS - 1) / SIMT_ROWS));
    const unsigned grid_k = (unsigned)(s.BH * ((s.N + SIMT_ROWS - 1) / SIMT_ROWS));
    simt_bwd_dq_kernel<T><<<grid_q, SIMT_THREADS, smem, st>>>((const T*)Q, (const T*)K, (const T*)V, (const T*)tQ,
                                                              (const T*)tK, (const T*)tV, (const T*)G, (const T*)Hc, lse,
                                                              mu, sig1, cvec, (T*)dQ, (T*)dtQ, s.q, s.k, s.H, s.d, s.alpha);
    g_prof.after(st);
    simt_bwd_dkv_kernel<T><<<grid_k, SIMT_THREADS, smem, st>>>((const T*)Q, (const T*)K, (const T*)V, (const T*)tQ,
                                                               (const T*)tK, (const T*)tV, (const T*)G, (const T*)Hc,
                                                               lse, mu, sig1, cvec, (T*)dK, (T*)dV, (T*)dtK, (T*)dtV,
                                                               s.q, s.k, s.H, s.d, s.alpha);
    g_prof.after(st);
    g_launches += 2;
    return cuda_status(cudaGetLastError());
}

// ------------------------------------------------------------------------------------------------
// Tensor-core path
typedef CUresult (*encode_tiled_fn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                    const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                    CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static encode_tiled_fn get_encode_fn() {
    static const encode_tiled_fn fn = driver_function<encode_tiled_fn>("cuTensorMapEncodeTiled");
    return fn;
}

// A bf16 tensor of one side viewed as a 4-D tensor (d, rows, H, B) with that side's strides; a box is 64 columns x
// `box_rows` rows of one head with the 128-byte swizzle; columns or rows beyond the tensor read as zero.
static int make_tmap(CUtensorMap* m, const void* ptr, const Shape& s, const Geom& g, int box_rows = JVP_BC) {
    encode_tiled_fn fn = get_encode_fn();
    if (!fn) return TVM_ATTN_CUDA_ERROR;
    cuuint64_t dims[4] = {(cuuint64_t)s.d, (cuuint64_t)g.rows, (cuuint64_t)s.H, (cuuint64_t)s.B};
    cuuint64_t strides[3] = {(cuuint64_t)g.rs * 2, (cuuint64_t)g.hs * 2, (cuuint64_t)g.bs * 2};
    cuuint32_t box[4] = {64, (cuuint32_t)box_rows, 1, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(ptr), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? TVM_ATTN_OK : TVM_ATTN_CUDA_ERROR;
}

// A tensor of a call and its map (with boxes of 64 rows one map serves a tensor in every role it has in the passes of a
// call, except as a stream of shorter tiles).  An absent cotangent is never loaded: its map is that of a present tensor and unused.
struct Operand {
    const __nv_bfloat16* ptr;
    const CUtensorMap* map;
};

template <int MODE, int DP>
static int launch_pass(const Shape& s, const Operand (&own)[4], const Operand (&strm)[4], JvpParams prm, const DeviceFacts& dev, cudaStream_t st) {
    using C = JvpCfg<MODE, DP>;
    constexpr auto kern = jvp_kernel<MODE, DP>;
    if (!prepare_kernel<kern>(dev, C::SMEM_BYTES)) return TVM_ATTN_CUDA_ERROR;
    // DV, DK: keys own, queries stream; FWD, DQ: queries own, keys stream
    prm.o = C::TRANSPOSED ? s.k : s.q;
    prm.s = C::TRANSPOSED ? s.q : s.k;
    for (int t = 0; t < 4; ++t) {
        prm.own[t] = own[t].ptr;
        prm.strm[t] = strm[t].ptr;
    }
    // one CTA per SM (each needs the whole tensor memory and most of the shared memory of one); the work
    // items go round-robin over them
    prm.row_tiles = (prm.o.rows + JVP_ROWS - 1) / JVP_ROWS;
    prm.items = (int)(s.BH * prm.row_tiles);
    prm.T = (prm.s.rows + C::BC - 1) / C::BC;
    prm.item_wait_ns = JVP_WAIT_LIMIT_NS + (uint64_t)prm.T * JVP_TILE_LIMIT_NS;
    g_prof.before(st);
    // DK and DQ read nothing that the pass before them writes (all passes depend on the row-sums pre-pass only, which has
    // completed before the first of them starts), so their CTAs may fill the SMs that the last, partial wave of the pass
    // before leaves idle: programmatic dependent launch, with every CTA of these kernels releasing its dependents at
    // once.  None waits for its primary before it works; each waits for it once at the very end (griddepcontrol.wait in
    // the teardown), so that no pass can complete before the one in front of it: work enqueued behind the call still sees all
    // six gradients.  Not while per-kernel events are being recorded: they would time overlapping kernels.
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(prm.items < dev.sms ? prm.items : dev.sms));
    cfg.blockDim = dim3(JVP_THREADS);
    cfg.dynamicSmemBytes = C::SMEM_BYTES;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = ((MODE == PASS_DK || MODE == PASS_DQ || MODE == PASS_DQ_G) && !g_prof.enabled.load(std::memory_order_relaxed)) ? 1 : 0;
    if (cudaLaunchKernelEx(&cfg, kern, *strm[0].map, *strm[1].map, *strm[2].map, *strm[3].map, *own[0].map, *own[1].map, *own[2].map,
                           *own[3].map, prm) != cudaSuccess)
        return cuda_status(cudaGetLastError());
    g_prof.after(st);
    g_launches += 1;
    return cuda_status(cudaGetLastError());
}

// The passes there are: FWD and DQ for every head dim; DKV where its four accumulators fit into tensor memory next to the
// scores, DV and DK where they do not; DKV_G and DQ_G, the backward without dtO, up to the same head dim.
static constexpr bool pass_exists(int mode, int dp) {
    return mode == PASS_DKV || mode == PASS_DKV_G || mode == PASS_DQ_G ? dp <= 80 : mode == PASS_DV || mode == PASS_DK ? dp > 80 : true;
}

template <int MODE, int DP = 16>
static int launch_pass_dp(const Shape& s, const Operand (&own)[4], const Operand (&strm)[4], const JvpParams& prm, const DeviceFacts& dev, cudaStream_t st) {
    if constexpr (DP > 128) {
        return TVM_ATTN_UNSUPPORTED;
    } else {
        if constexpr (pass_exists(MODE, DP))
            if (s.dp == DP) return launch_pass<MODE, DP>(s, own, strm, prm, dev, st);
        return launch_pass_dp<MODE, DP + 16>(s, own, strm, prm, dev, st);
    }
}

// Scratch of tvm_attn_jvp_bwd_noalloc: three floats per row, for callers that cannot allocate.  In host code
// this name is only a handle for cudaGetSymbolAddress, never a device pointer.
static __device__ __align__(256) float g_noalloc_scratch[3 * TVM_ATTN_NOALLOC_MAX_ROWS];
static constexpr int kMaxDevices = 64;
static float* g_noalloc_addr[kMaxDevices] = {};  // device address of the array, per device
static std::mutex g_noalloc_mutex;

// Device address of the scratch array on the current device, looked up on first use.
static int noalloc_scratch_address(float** out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return TVM_ATTN_CUDA_ERROR;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_addr[dev]) {
        float* ptr = nullptr;
        if (cudaGetSymbolAddress(reinterpret_cast<void**>(&ptr), g_noalloc_scratch) != cudaSuccess || !ptr)
            return TVM_ATTN_CUDA_ERROR;
        g_noalloc_addr[dev] = ptr;
    }
    *out = g_noalloc_addr[dev];
    return TVM_ATTN_OK;
}

// One warp waits, with a limit, on an mbarrier that nobody arrives at: the same bounded wait the tensor-core
// kernels use, made to run out on purpose so that the time-out reporting can be exercised without disturbing
// a real kernel.  Raises the device status word like they do.
__global__ void selftest_timeout_kernel(int* status, unsigned long long limit_ns) {
    __shared__ __align__(8) unsigned long long barrier;
    __shared__ int abort_flag;
    if (*reinterpret_cast<volatile int*>(status) != 0) return;
    const uint32_t bar = ptx::smem_u32(&barrier);
    if (threadIdx.x == 0) {
        abort_flag = 0;
        ptx::mbar_init(bar, 1);
        ptx::fence_mbar_init();
    }
    __syncwarp();
    const bool ok = ptx::mbar_wait_warp(bar, 0, &abort_flag, limit_ns);
    if (!ok && threadIdx.x == 0 && abort_flag) atomicExch(status, 1);
}

// ------------------------------------------------------------------------------------------------
// RMSNorm QK-normalisation prologue
// The rows of a side in memory order.  Dimensions of one element drop out, and two that are dense in one another
// merge: both tensor layouts of a transformer, packed and (B, rows, H, d), end as one dimension.
static RmsRows rms_rows(const Shape& s, const Geom& g) {
    struct Dim { long long n, st; } dim[3] = {{g.rows, g.rs}, {s.H, g.hs}, {s.B, g.bs}};
    for (int i = 0; i < 2; ++i)   // by stride, innermost first
        for (int j = 0; j < 2 - i; ++j)
            if (dim[j].n == 1 || (dim[j + 1].n > 1 && dim[j + 1].st < dim[j].st)) std::swap(dim[j], dim[j + 1]);
    RmsRows r;
    r.total = (unsigned)(s.BH * g.rows);
    int n = 0;
    Dim out[3] = {{1, s.d}, {1, 0}, {1, 0}};
    for (int i = 0; i < 3; ++i) {
        if (dim[i].n == 1) continue;
        if (n > 0 && dim[i].st == out[n - 1].n * out[n - 1].st) out[n - 1].n *= dim[i].n;
        else out[n++] = dim[i];
    }
    r.n0 = (unsigned)out[0].n; r.n1 = (unsigned)out[1].n;
    r.s0 = out[0].st; r.s1 = out[1].st; r.s2 = out[2].st;
    return r;
}

// Blocks of both sides, at most `most` of them: in proportion to the rows, at least one each.
static void rms_blocks(long long rows_q, long long rows_k, int rows_per_block, int most, int* nbq, int* nbk) {
    const long long need_q = (rows_q + rows_per_block - 1) / rows_per_block, need_k = (rows_k + rows_per_block - 1) / rows_per_block;
    if (need_q + need_k <= most) { *nbq = (int)need_q; *nbk = (int)need_k; return; }
    long long q = (most * rows_q + (rows_q + rows_k) / 2) / (rows_q + rows_k);
    q = q < 1 ? 1 : q > most - 1 ? most - 1 : q;
    *nbq = (int)(q < need_q ? q : need_q);
    *nbk = (int)(most - q < need_k ? most - q : need_k);
}

template <typename T, int C, bool RAGGED>
static int rms_fwd_c(const Shape& s, float eps, const RmsFwdSide<T>& q, const RmsFwdSide<T>& k, int P, cudaStream_t st) {
    int nbq, nbk;
    rms_blocks(q.rows.total, k.rows.total, (RMS_THREADS / 32) * rms_fwd_groups(C) * (32 / P), RMS_FWD_BLOCKS, &nbq, &nbk);
    qk_rmsnorm_jvp_fwd_kernel<T, C, RAGGED><<<nbq + nbk, RMS_THREADS, 0, st>>>(q, k, nbq, s.d, P, eps);
    g_launches += 1;
    return cuda_status(cudaGetLastError());
}

template <typename T>
static int rms_fwd(const Shape& s, float eps, const void* Q, const void* tQ, const void* K, const void* tK, const float* gQ,
                   const float* gK, void* Qn, void* tQn, void* Kn, void* tKn, cudaStream_t st) {
    const RmsFwdSide<T> q{(const T*)Q, (const T*)tQ, gQ, (T*)Qn, (T*)tQn, rms_rows(s, s.q)};
    const RmsFwdSide<T> k{(const T*)K, (const T*)tK, gK, (T*)Kn, (T*)tKn, rms_rows(s, s.k)};
    return with_split<T, 4>(s.d, [&](auto C, auto ragged, int P) { return rms_fwd_c<T, C(), ragged()>(s, eps, q, k, P, st); });
}

template <typename T, int C, bool RAGGED>
static int rms_bwd_c(const Shape& s, float eps, RmsBwdSide<T> q, RmsBwdSide<T> k, int P, float* dgQ, float* dgK, cudaStream_t st) {
    int nbq, nbk;
    rms_blocks(q.rows.total, k.rows.total, (RMS_BWD_THREADS / 32) * (32 / P), RMS_BWD_BLOCKS, &nbq, &nbk);
    k.partial = q.partial + (size_t)nbq * s.d;
    qk_rmsnorm_jvp_bwd_kernel<T, C, RAGGED><<<nbq + nbk, RMS_BWD_THREADS, 0, st>>>(q, k, nbq, s.d, P, eps);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return TVM_ATTN_CUDA_ERROR;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)s.d / 4, 2);
    cfg.blockDim = dim3(RMS_REDUCE_THREADS);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, qk_rmsnorm_dg_reduce_kernel, (const float*)q.partial, (const float*)k.partial, dgQ, dgK, nbq, nbk, s.d);
    g_launches += 2;
    return cuda_status(e);
}

template <typename T>
static int rms_bwd(const Shape& s, float eps, const void* Q, const void* tQ, const void* K, const void* tK, const float* gQ,
                   const float* gK, const void* dQn, const void* dtQn, const void* dKn, const void* dtKn, void* dQ, void* dtQ,
                   void* dK, void* dtK, float* dgQ, float* dgK, float* partial, cudaStream_t st) {
    const RmsBwdSide<T> q{(const T*)Q, (const T*)tQ, gQ, (const T*)dQn, (const T*)dtQn, (T*)dQ, (T*)dtQ, partial, rms_rows(s, s.q)};
    const RmsBwdSide<T> k{(const T*)K, (const T*)tK, gK, (const T*)dKn, (const T*)dtKn, (T*)dK, (T*)dtK, nullptr, rms_rows(s, s.k)};
    return with_split<T, 3>(s.d, [&](auto C, auto ragged, int P) { return rms_bwd_c<T, C(), ragged()>(s, eps, q, k, P, dgQ, dgK, st); });
}

static bool rms_eps_ok(float eps) { return eps >= 0.0f && std::isfinite(eps); }

}  // namespace tvm_attn

using namespace tvm_attn;

extern "C" {

size_t tvm_attn_jvp_workspace_bytes(const tvm_attn_params* p, int is_bwd) {
    Shape s;
    if (check_params(p, &s) != TVM_ATTN_OK) return 0;
    if (!is_bwd) return 0;
    return (size_t)3 * sizeof(float) * (size_t)s.BH * (size_t)s.M;   // per query row
}

int tvm_attn_jvp_fwd(const tvm_attn_params* p, const void* Q, const void* K, const void* V, const void* tQ,
                     const void* tK, const void* tV, void* O, void* tO, float* lse, float* mu, void* workspace,
                     size_t workspace_bytes, void* cuda_stream) {
    (void)workspace; (void)workspace_bytes;
    Shape s;
    int rc = check_params(p, &s);
    if (rc != TVM_ATTN_OK) return rc;
    const void* ptrs[] = {Q, K, V, tQ, tK, tV, O, tO, lse, mu};
    for (const void* x : ptrs)
        if (!x || !aligned16(x)) return TVM_ATTN_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    g_prof.begin_call();
    if (s.simt) {
        return s.fp32 ? simt_fwd<float>(s, Q, K, V, tQ, tK, tV, O, tO, lse, mu, st)
                      : simt_fwd<__nv_bfloat16>(s, Q, K, V, tQ, tK, tV, O, tO, lse, mu, st);
    }
    const DeviceFacts* dev;
    rc = tensor_core_device(&dev);
    if (rc != TVM_ATTN_OK) return rc;
    if (s.dp > 80 && !s.plain) return TVM_ATTN_UNSUPPORTED;  // head dims above 80: self-attention on packed tensors only
    CUtensorMap maps[6];
    const void* in[6] = {Q, tQ, K, tK, V, tV};
    Operand x[6];
    for (int t = 0; t < 6; ++t) {
        rc = make_tmap(&maps[t], in[t], s, t < 2 ? s.q : s.k);
        if (rc != TVM_ATTN_OK) return rc;
        x[t] = {static_cast<const __nv_bfloat16*>(in[t]), &maps[t]};
    }
    JvpParams f;
    std::memset(&f, 0, sizeof f);
    f.d = s.d; f.H = s.H;
    f.alpha = s.alpha; f.c2 = s.alpha * 1.4426950408889634f;
    f.out0 = static_cast<__nv_bfloat16*>(O); f.out1 = static_cast<__nv_bfloat16*>(tO);
    f.lse = lse; f.mu_out = mu; f.status = dev->status;
    return launch_pass_dp<PASS_FWD>(s, {x[0], x[1], x[0], x[1]}, {x[2], x[3], x[4], x[5]}, f, *dev, st);
}

int tvm_attn_jvp_bwd(const tvm_attn_params* p, const void* Q, const void* K, const void* V, const void* tQ,
                     const void* tK, const void* tV, const void* O, const void* tO, const float* lse, const float* mu,
                     const void* dO, const void* dtO, void* dQ, void* dK, void* dV, void* dtQ, void* dtK, void* dtV,
                     void* workspace, size_t workspace_bytes, void* cuda_stream) {
    Shape s;
    int rc = check_params(p, &s);
    if (rc != TVM_ATTN_OK) return rc;
    const void* ptrs[] = {Q, K, V, tQ, tK, tV, O, tO, lse, mu, dQ, dK, dV, workspace};
    for (const void* x : ptrs)
        if (!x || !aligned16(x)) return TVM_ATTN_INVALID_ARG;
    // A null cotangent means zero (dtO null = the "detach JVP" setting: no gradient through tO).  With dtO null the
    // tangent gradients are identically zero and their outputs may be null too.
    if (!dO && !dtO) return TVM_ATTN_INVALID_ARG;
    const void* opt[] = {dO, dtO, dtQ, dtK, dtV};
    for (const void* x : opt)
        if (x && !aligned16(x)) return TVM_ATTN_INVALID_ARG;
    if (dtO && (!dtQ || !dtK || !dtV)) return TVM_ATTN_INVALID_ARG;
    // DKV takes its statistics divided by the scale, which overflows where that is next to nothing (lse / 1e-36 does at 340):
    // such a call, all of whose weights are equal, goes to the CUDA-core kernels.
    if (s.alpha < 1e-36f && pass_exists(PASS_DKV, s.dp)) s.simt = true;
    if ((!dO || !dtO || !s.plain) && !s.simt && s.dp > 80) return TVM_ATTN_UNSUPPORTED;  // head dims above 80: both cotangents, packed self-attention
    const size_t rows = (size_t)s.BH * (size_t)s.M;   // query rows: what the workspace and the statistics are sized by
    if (workspace_bytes < 3 * sizeof(float) * rows) return TVM_ATTN_WORKSPACE_TOO_SMALL;
    float* sig1 = static_cast<float*>(workspace);
    float* cvec = sig1 + rows;
    float* lse2 = cvec + rows;  // lse * log2(e)
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    g_prof.begin_call();
    if (!dtO) {  // the tangent gradients of a call without dtO are zero: written here, by none of the passes
        void* zero_out[] = {dtQ, dtK, dtV};
        const int esz = s.fp32 ? 4 : 2, cpr = s.d * esz / 16;
        for (int i = 0; i < 3; ++i) {
            if (!zero_out[i]) continue;
            const Geom& g = i == 0 ? s.q : s.k;
            const long long zr = s.BH * g.rows, n = zr * cpr;
            zero_rows_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(static_cast<uint4*>(zero_out[i]), g, s.H, zr, cpr, 16 / esz);
            g_launches += 1;
            if (cudaGetLastError() != cudaSuccess) return TVM_ATTN_CUDA_ERROR;
        }
    }
    if (s.simt) {
        if (s.fp32) {
            rc = launch_rowsums<float>(s, dO, dtO, O, tO, lse, sig1, cvec, lse2, 1.0f, st);
            if (rc != TVM_ATTN_OK) return rc;
            return simt_bwd<float>(s, Q, K, V, tQ, tK, tV, lse, mu, dO, dtO, sig1, cvec, dQ, dK, dV, dtQ, dtK, dtV, st);
        }
        rc = launch_rowsums<__nv_bfloat16>(s, dO, dtO, O, tO, lse, sig1, cvec, lse2, 1.0f, st);
        if (rc != TVM_ATTN_OK) return rc;
        return simt_bwd<__nv_bfloat16>(s, Q, K, V, tQ, tK, tV, lse, mu, dO, dtO, sig1, cvec, dQ, dK, dV, dtQ, dtK, dtV, st);
    }
    const DeviceFacts* dev;
    rc = tensor_core_device(&dev);
    if (rc != TVM_ATTN_OK) return rc;
    rc = launch_rowsums<__nv_bfloat16>(s, dO, dtO, O, tO, lse, sig1, cvec, lse2, -1.0f, st);
    if (rc != TVM_ATTN_OK) return rc;
    CUtensorMap maps[12];
    const void* in[8] = {Q, tQ, dtO, dO, K, tK, V, tV};
    Operand x[12];
    for (int t = 0; t < 8; ++t) {
        x[t] = {static_cast<const __nv_bfloat16*>(in[t]), in[t] ? &maps[t] : &maps[0]};
        rc = in[t] ? make_tmap(&maps[t], in[t], s, t < 4 ? s.q : s.k) : TVM_ATTN_OK;
        if (rc != TVM_ATTN_OK) return rc;
    }
    // the query side as DKV streams it
    const int short_rows = s.dp == 80 ? JvpCfg<PASS_DKV, 80>::BC : JVP_BC;
    for (int t = 0; t < 4; ++t) {
        x[8 + t] = x[t];
        if (short_rows == JVP_BC || !in[t] || !dtO) continue;
        x[8 + t].map = &maps[8 + t];
        rc = make_tmap(&maps[8 + t], in[t], s, s.q, short_rows);
        if (rc != TVM_ATTN_OK) return rc;
    }
    const Operand &xQ = x[0], &xtQ = x[1], &xH = x[2], &xG = x[3], &xK = x[4], &xtK = x[5], &xV = x[6], &xtV = x[7];
    JvpParams b;
    std::memset(&b, 0, sizeof b);
    b.d = s.d; b.H = s.H;
    b.alpha = s.alpha; b.c2 = s.alpha * 1.4426950408889634f;
    b.nlse2 = lse2; b.mu = mu; b.nsig1 = sig1; b.ncvec = cvec; b.status = dev->status; b.no_g = !dO;
    auto bf16 = [](void* ptr) { return static_cast<__nv_bfloat16*>(ptr); };
    if (!dtO) {   // owner keys (K, V), stream queries (Q, G); owner queries (Q, G), stream keys (K, V)
        b.out0 = bf16(dV);
        b.out1 = bf16(dK);
        b.out_scale = s.alpha;
        rc = launch_pass_dp<PASS_DKV_G>(s, {xK, xV, xK, xV}, {xQ, xG, xQ, xG}, b, *dev, st);
        if (rc != TVM_ATTN_OK) return rc;
        b.out0 = nullptr;
        b.out1 = bf16(dQ);
        return launch_pass_dp<PASS_DQ_G>(s, {xQ, xG, xQ, xG}, {xK, xV, xK, xV}, b, *dev, st);
    }
    auto outputs = [&](void* tangent, void* primal, float scale) {
        b.out0 = bf16(tangent);
        b.out1 = bf16(primal);
        b.out_scale = scale;
    };
    // dtV = P^T Hc, dV = P^T G + (P*Nn)^T Hc; dtK = alpha W^T Q, dK = alpha (dA^T Q + W^T tQ) : owner keys, stream queries
    if (pass_exists(PASS_DKV, s.dp)) {
        outputs(dtV, dV, s.alpha);
        b.out2 = bf16(dtK);
        b.out3 = bf16(dK);
        rc = launch_pass_dp<PASS_DKV>(s, {xK, xtK, xV, xtV}, {x[10], x[11], x[8], x[9]}, b, *dev, st);
    } else {
        outputs(dtV, dV, 1.0f);
        rc = launch_pass_dp<PASS_DV>(s, {xK, xtK, xK, xtK}, {xQ, xtQ, xH, xG}, b, *dev, st);
        if (rc != TVM_ATTN_OK) return rc;
        outputs(dtK, dK, s.alpha);
        rc = launch_pass_dp<PASS_DK>(s, {xK, xtK, xV, xtV}, {xH, xG, xQ, xtQ}, b, *dev, st);
    }
    if (rc != TVM_ATTN_OK) return rc;
    // dtQ = alpha W K, dQ = alpha (dA K + W tK) : owner queries (Q, tQ, Hc, G); stream (V, tV | K, tK)
    outputs(dtQ, dQ, s.alpha);
    return launch_pass_dp<PASS_DQ>(s, {xQ, xtQ, xH, xG}, {xV, xtV, xK, xtK}, b, *dev, st);
}

int tvm_attn_jvp_bwd_noalloc(const tvm_attn_params* p, const void* Q, const void* K, const void* V, const void* tQ,
                             const void* tK, const void* tV, const void* O, const void* tO, const float* lse,
                             const float* mu, const void* dO, const void* dtO, void* dQ, void* dK, void* dV, void* dtQ,
                             void* dtK, void* dtV, void* cuda_stream) {
    Shape s;
    const int rc = check_params(p, &s);
    if (rc != TVM_ATTN_OK) return rc;
    if (s.BH * (long long)s.M > (long long)TVM_ATTN_NOALLOC_MAX_ROWS) return TVM_ATTN_TOO_LARGE;
    float* scratch = nullptr;
    const int rs = noalloc_scratch_address(&scratch);
    if (rs != TVM_ATTN_OK) return rs;
    return tvm_attn_jvp_bwd(p, Q, K, V, tQ, tK, tV, O, tO, lse, mu, dO, dtO, dQ, dK, dV, dtQ, dtK, dtV, scratch,
                            sizeof(float) * 3 * (size_t)TVM_ATTN_NOALLOC_MAX_ROWS, cuda_stream);
}

int tvm_attn_check_status(void* cuda_stream) {
    if (cudaStreamSynchronize(static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess) return TVM_ATTN_CUDA_ERROR;
    int host = 0;
    if (cudaMemcpyFromSymbol(&host, g_status_word, sizeof(int)) != cudaSuccess) return TVM_ATTN_CUDA_ERROR;
    if (host != 0) {
        const int zero = 0;
        if (cudaMemcpyToSymbol(g_status_word, &zero, sizeof(int)) != cudaSuccess) return TVM_ATTN_CUDA_ERROR;
        return TVM_ATTN_DEVICE_TIMEOUT;
    }
    return TVM_ATTN_OK;
}

size_t tvm_qk_rmsnorm_jvp_workspace_bytes(const tvm_attn_params* p) {
    Shape s;
    if (check_params(p, &s) != TVM_ATTN_OK) return 0;
    return (size_t)RMS_PARTIAL_ROWS * (size_t)s.d * sizeof(float);
}

int tvm_qk_rmsnorm_jvp_fwd(const tvm_attn_params* p, float eps, const void* Q, const void* tQ, const void* K, const void* tK,
                           const float* gQ, const float* gK, void* Qn, void* tQn, void* Kn, void* tKn, void* cuda_stream) {
    Shape s;
    const int rc = check_params(p, &s);
    if (rc != TVM_ATTN_OK) return rc;
    if (!rms_eps_ok(eps)) return TVM_ATTN_INVALID_ARG;
    const void* ptrs[] = {Q, tQ, K, tK, gQ, gK, Qn, tQn, Kn, tKn};
    for (const void* x : ptrs)
        if (!x || !aligned16(x)) return TVM_ATTN_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    return s.fp32 ? rms_fwd<float>(s, eps, Q, tQ, K, tK, gQ, gK, Qn, tQn, Kn, tKn, st)
                  : rms_fwd<__nv_bfloat16>(s, eps, Q, tQ, K, tK, gQ, gK, Qn, tQn, Kn, tKn, st);
}

int tvm_qk_rmsnorm_jvp_bwd(const tvm_attn_params* p, float eps, const void* Q, const void* tQ, const void* K, const void* tK,
                           const float* gQ, const float* gK, const void* dQn, const void* dtQn, const void* dKn,
                           const void* dtKn, void* dQ, void* dtQ, void* dK, void* dtK, float* dgQ, float* dgK, void* workspace,
                           size_t workspace_bytes, void* cuda_stream) {
    Shape s;
    const int rc = check_params(p, &s);
    if (rc != TVM_ATTN_OK) return rc;
    if (!rms_eps_ok(eps)) return TVM_ATTN_INVALID_ARG;
    const void* ptrs[] = {Q, tQ, K, tK, gQ, gK, dQn, dtQn, dKn, dtKn, dQ, dtQ, dK, dtK, dgQ, dgK, workspace};
    for (const void* x : ptrs)
        if (!x || !aligned16(x)) return TVM_ATTN_INVALID_ARG;
    if (workspace_bytes < (size_t)RMS_PARTIAL_ROWS * (size_t)s.d * sizeof(float)) return TVM_ATTN_WORKSPACE_TOO_SMALL;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    float* part = static_cast<float*>(workspace);
    return s.fp32 ? rms_bwd<float>(s, eps, Q, tQ, K, tK, gQ, gK, dQn, dtQn, dKn, dtKn, dQ, dtQ, dK, dtK, dgQ, dgK, part, st)
                  : rms_bwd<__nv_bfloat16>(s, eps, Q, tQ, K, tK, gQ, gK, dQn, dtQn, dKn, dtKn, dQ, dtQ, dK, dtK, dgQ, dgK, part, st);
}

int tvm_attn_selftest_timeout(uint64_t limit_ns, void* cuda_stream) {
    if (limit_ns == 0 || limit_ns > 100ull * 1000ull * 1000ull) return TVM_ATTN_INVALID_ARG;
    const DeviceFacts* dev = device_facts();
    if (!dev) return TVM_ATTN_CUDA_ERROR;
    selftest_timeout_kernel<<<1, 32, 0, static_cast<cudaStream_t>(cuda_stream)>>>(dev->status, limit_ns);
    g_launches += 1;
    return cuda_status(cudaGetLastError());
}

int tvm_attn_set_profiling(int enable) {
    g_prof.enabled.store(enable != 0);
    g_prof.count.store(0);
    return TVM_ATTN_OK;
}

int tvm_attn_get_profile(float* ms, int capacity) {
    if (!ms || capacity < 0) return TVM_ATTN_INVALID_ARG;
    const int recorded = g_prof.count.load();
    int n = recorded < capacity ? recorded : capacity;
    if (n > 7) n = 7;
    if (n > 0 && cudaEventSynchronize(g_prof.ev[n]) != cudaSuccess) return TVM_ATTN_CUDA_ERROR;
    for (int k = 0; k < n; ++k)
        if (cudaEventElapsedTime(&ms[k], g_prof.ev[k], g_prof.ev[k + 1]) != cudaSuccess) return TVM_ATTN_CUDA_ERROR;
    return n;
}

uint64_t tvm_attn_launch_count(void) { return g_launches.load(); }

const char* tvm_attn_strerror(int code) {
    switch (code) {
        case TVM_ATTN_OK: return "ok";
        case TVM_ATTN_INVALID_ARG: return "invalid argument (null or misaligned pointer, bad dimension, dtype, flags or scale)";
        case TVM_ATTN_UNSUPPORTED: return "unsupported shape or device (need 8 <= d <= 128, d % 8 == 0, an sm_100 GPU)";
        case TVM_ATTN_WORKSPACE_TOO_SMALL: return "workspace smaller than tvm_attn_jvp_workspace_bytes()";
        case TVM_ATTN_CUDA_ERROR: return "a CUDA call or kernel launch failed";
        case TVM_ATTN_DEVICE_TIMEOUT: return "a bounded wait inside a kernel ran out; outputs are unspecified";
        case TVM_ATTN_TOO_LARGE: return "B*H*N exceeds TVM_ATTN_NOALLOC_MAX_ROWS, the built-in scratch of tvm_attn_jvp_bwd_noalloc; "
                                        "call tvm_attn_jvp_bwd with a workspace instead";
        default: return "unknown status";
    }
}

int tvm_attn_version(void) { return 100; }

}  // extern "C"
