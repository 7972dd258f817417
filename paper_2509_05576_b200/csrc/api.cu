// C-ABI entry points (see include/ptq.h): argument checks, workspace carving, kernel sequencing.
#include "common.cuh"
#include "dgemm.cuh"
#include "chol.cuh"
#include "order.cuh"
#include "colloop.cuh"
#include "gram.cuh"
#include "dynamic.cuh"
#include "perrow.cuh"
#include "i8gemm.cuh"
#include "cholpanel.cuh"

using namespace ptq;

namespace {

__global__ void convert_f32_f64_kernel(const float* __restrict__ X, int rows, int n, int64_t ldx,
                                       double* __restrict__ Xd) {
    const int i = blockIdx.y;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x)
        Xd[(int64_t)i * n + k] = (double)X[(int64_t)i * ldx + k];
}

inline int grid_x_for(int n, int threads) {
    int g = cdiv(n, threads);
    return g < 1 ? 1 : (g > 1024 ? 1024 : g);
}

constexpr int kMaxGridY = 65535;
constexpr int kSlicedMinCols = 3072;      // from here on the large float64 products run on the int8 tensor path
// The loss product goes there too where it is large enough to pay for slicing H and for a second product, and where the
// slices (7 bytes a value, both sizes rounded up to multiples of 128) and the two sets of partial sums fit into the pieces of
// the workspace that are free by then: dW's into E, H's into U (8 bytes a value each).  So a size whose padding takes more
// than an eighth of it keeps the float64 product: 560 x 2304 and 2561 x 1025 do, 512 x 2304 and 1000 x 1791 do not.
// Both sides measured, float64 -> sliced, by rows cols^2 / 2^30: 512 x 1536 (1.1) 69 -> 81 us, 256 x 3008 (2.2) 130 -> 141,
// 1024 x 1536 (2.3) 123 -> 136, 512 x 2304 (2.5) 126 -> 118, 768 x 1920 (2.6) 157 -> 155, 768 x 2304 (3.8) 174 -> 167,
// 1000 x 2048 (3.9) 209 -> 151, 512 x 4608 (10) 418 -> 316, 2000 x 4608 (40) 1599 -> 844.  Its error against extended
// precision is no larger, also where the channels differ in scale (the operands are equilibrated, i8gemm.cuh).  Median and
// largest relative error over ten kinds of activations at three calibration lengths, float64 library sums / this: 512 x 2304
// 1.1e-16, 8.9e-13 / 9.8e-17, 2.1e-12; 1000 x 2048 1.1e-16, 2.1e-13 / 1.7e-16, 1.6e-13; 512 x 4608 1.3e-16, 6.0e-13 /
// 1.3e-16, 2.8e-13 (the largest are those of inputs that share one component, where most of the sum cancels).  W^T W stays
// where it is below kSlicedMinCols: sliced it is 8 % faster there (164 -> 151 us at 2304 columns), but the error of the inverse
// up to three times larger.
constexpr double kSlicedLossMinWork = 2.5 * (1 << 30);
constexpr int kSlicedLossMinCols = 1024;
constexpr int kLossMaxSplit = 8;
size_t loss_partials_count(int rows, int cols) {
    return (size_t)kLossMaxSplit * cdiv(rows, 64) * cdiv(cols, 64);
}
bool sliced_loss(int rows, int cols) {
    return cols >= kSlicedLossMinCols && cols <= kXMaxK && (double)rows * cols * cols >= kSlicedLossMinWork &&
           x_operand_bytes(rows, cols) <= (size_t)rows * cols * sizeof(double) &&
           x_operand_bytes(cols, cols) <= (size_t)cols * cols * sizeof(double) &&
           2 * (size_t)x_num_tiles(rows, cols) <= loss_partials_count(rows, cols);
}
// Digits of E and U in the deferred part of Eq. 11 of layers that are swept panel by panel.  With eight the product is more
// exact than the float64 MMA steps of the sweep for every kind of input measured, with seven it is less exact where the input
// channels differ in scale (i8gemm.cuh).  Layers this tall and wide had no float64 steps to match and keep seven: eight
// would take 7.19 -> 7.32 ms at 4096 x 4096 and 53.6 -> 54.8 at 4096 x 11008.  Below, seven -> eight: 512 x 4608 6.18 -> 6.22 ms,
// 2000 x 4608 7.63 -> 7.73, 512 x 8192 19.2 -> 19.3, 2000 x 8000 21.7 -> 22.1.
inline int deferred_digits(int rows, int cols) { return rows >= 2048 && cols >= 4096 ? kXSlices : kXMoreSlices; }
// The float64 loss product is cut along k into as many slices as it takes to put about two CTAs on every SM.
int loss_ksplit(int rows, int cols) {
    const long ctas = (long)cdiv(rows, 64) * ((cdiv(cols, 64) + 1) / 2);
    const long want = (2 * 148 + ctas - 1) / ctas;
    return (int)(want < 1 ? 1 : (want > kLossMaxSplit ? kLossMaxSplit : want));
}

// Built-in scratch of ptq_sensitivity_order_static: lives in every device that loads the library, until exit.
constexpr size_t kStaticScratchDoubles = PTQ_STATIC_SCRATCH_BYTES / sizeof(double);
static __device__ __align__(256) double g_static_score_scratch[kStaticScratchDoubles];

// Device address of the array on the current device.  In host code the symbol's name is only a handle, so the
// address is asked of the runtime, with the caller's device current, on every call: the lookup is cheap after the
// first one, and an address remembered across a cudaDeviceReset or under another context would be stale.
int static_scratch_address(double** out) {
    double* p = nullptr;
    if (cudaGetSymbolAddress((void**)&p, g_static_score_scratch) != cudaSuccess || !p) {
        cudaGetLastError();
        return PTQ_ERR_CUDA;
    }
    *out = p;
    return PTQ_OK;
}

// Scores and order (Sec. 4.2 steps 1-3) with the per-row-chunk partial sums in `partial`.
int order_launch(const float* W, int rows, int cols, int64_t ldw, const double* Hinv_diag, const float* scale,
                 const float* zero, int bits, int mode, int ascending, double* S, int32_t* perm, double* partial,
                 int32_t* status, cudaStream_t stream) {
    const int chunks = cdiv(rows, kScoreRowChunk);
    if (chunks > 65535) return PTQ_ERR_UNSUPPORTED;
    if (mode != PTQ_SCORE_NONE) {
        Launch l(K_SCORE_PARTIAL, stream);
        launch_chained(score_partial_kernel<float>, dim3(cdiv(cols, kScoreCols), chunks), 256, 0, stream, W, rows, cols, ldw,
                       scale, zero, bits, mode, partial);
    }
    {
        Launch l(K_SCORE_FINAL, stream);
        launch_chained(score_final_kernel, cdiv(cols, 128), 128, 0, stream, partial, chunks, cols, Hinv_diag, (int64_t)1,
                       mode, S, status);
    }
    {
        Launch l(K_RANK_SORT, stream);
        launch_chained(rank_sort_kernel, cdiv(cols, kRankCols), 256, 0, stream, S, cols, ascending, perm, nullptr);
    }
    return launch_status();
}

int order_args_check(const float* W, int rows, int cols, int64_t ldw, const double* Hinv_diag, const float* scale,
                     const float* zero, int bits, int score_mode, const double* S, const int32_t* perm) {
    if (!W || !S || !perm || rows < 1 || cols < 1 || ldw < cols || bits < 2 || bits > 8) return PTQ_ERR_INVALID_ARG;
    if (score_mode & ~(PTQ_SCORE_ASCENDING | 7)) return PTQ_ERR_INVALID_ARG;
    const int mode = score_mode & ~PTQ_SCORE_ASCENDING;
    if (mode < PTQ_SCORE_QERR || mode > PTQ_SCORE_NONE) return PTQ_ERR_INVALID_ARG;
    if ((mode == PTQ_SCORE_QERR || mode == PTQ_SCORE_PRUNE) && !Hinv_diag) return PTQ_ERR_INVALID_ARG;
    if ((mode == PTQ_SCORE_QERR || mode == PTQ_SCORE_ERR) && (!scale || !zero)) return PTQ_ERR_INVALID_ARG;
    return PTQ_OK;
}

// Self-test kernels: they call the very wait routines of the factorisation and of the sweep on a target that nothing
// will ever reach, so that the wait must run out, report PTQ_ERR_TIMEOUT and return.
__global__ void __launch_bounds__(kCholThreads) selftest_barrier_kernel(unsigned* bar, int32_t* status, long long spin_limit) {
    __shared__ int s_flag;
    const bool ok = grid_barrier(bar, gridDim.x + 1u, &s_flag, spin_limit);      // one arrival more than the grid has
    if (!ok && threadIdx.x == 0) report(status, PTQ_ERR_TIMEOUT, blockIdx.x, 1);
}
__global__ void selftest_counter_kernel(unsigned* words, int32_t* status, long long spin_limit) {
    if (threadIdx.x == 0 && !bounded_counter_wait(&words[0], 1u, &words[1], spin_limit))
        report(status, PTQ_ERR_TIMEOUT, blockIdx.x, 2);
}

// What ptq_selftest_abandoned_sweep starts from: one block row, two row groups.
constexpr int kAbandonedRows = 2 * kSweepRows;
static_assert(kAbandonedRows == kNB, "one launch fills the matrix and the rows");
__global__ void __launch_bounds__(kNB) selftest_unit_layer_kernel(double* __restrict__ U, double* __restrict__ Wp, double* __restrict__ E,
                                                                   float* __restrict__ scale, float* __restrict__ zero) {
    const int i = blockIdx.x, j = threadIdx.x;
    U[i * kNB + j] = i == j ? 1.0 : 0.0;
    Wp[i * kNB + j] = 0.0;
    E[i * kNB + j] = __longlong_as_double(-1ll);
    if (j == 0) { scale[i] = 1.0f; zero[i] = 0.0f; }
}

// What the factorisations make of a pivot, one value per thread.
__global__ void __launch_bounds__(256) selftest_reciprocal_kernel(const double* __restrict__ x, int n, double* __restrict__ rcp,
                                                                   double* __restrict__ rsq) {
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    rcp[i] = pivot_reciprocal(x[i]);
    rsq[i] = pivot_rsqrt(x[i]);
}

// Float64 throughput probes: eight independent chains per thread, nothing but the arithmetic instruction in the loop.
constexpr int kProbeThreads = 256, kProbeCtasPerSm = 4, kProbeChains = 8;
__global__ void __launch_bounds__(kProbeThreads) fp64_probe_fma_kernel(int iters, double* sink) {
    double acc[kProbeChains];
    const double a = 1.0 + 1e-9 * threadIdx.x, b = 1e-12 * (blockIdx.x + 1);
#pragma unroll
    for (int c = 0; c < kProbeChains; ++c) acc[c] = (double)c;
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int c = 0; c < kProbeChains; ++c) acc[c] = fma(acc[c], a, b);
    }
    double s = 0.0;
#pragma unroll
    for (int c = 0; c < kProbeChains; ++c) s += acc[c];
    if (s == 123.456) sink[0] = s;          // never true: keeps the loop alive without a store per thread
}
__global__ void __launch_bounds__(kProbeThreads) fp64_probe_mma_kernel(int iters, double* sink) {
    double acc[kProbeChains][2];
    const double a = 1.0 + 1e-9 * threadIdx.x, b = 1e-3 * ((threadIdx.x & 3) + 1);
#pragma unroll
    for (int c = 0; c < kProbeChains; ++c) acc[c][0] = acc[c][1] = 1e-12 * c;
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int c = 0; c < kProbeChains; ++c) dmma_884(acc[c][0], acc[c][1], a, b);
    }
    double s = 0.0;
#pragma unroll
    for (int c = 0; c < kProbeChains; ++c) s += acc[c][0] + acc[c][1];
    if (s == 123.456) sink[0] = s;
}

}  // namespace

extern "C" {

int ptq_version(void) { return 1; }

int ptq_kernel_count(void) { return K_COUNT; }

const char* ptq_kernel_name(int kernel_id) { return kernel_name(kernel_id); }

long long ptq_launch_count(int kernel_id) {
    const Profiler& p = profiler();
    if (kernel_id >= 0 && kernel_id < K_COUNT) return p.launches[kernel_id];
    long long total = 0;
    for (int k = 0; k < K_COUNT; ++k) total += p.launches[k];
    return total;
}

int ptq_set_cta_limit(int limit) {
    if (limit < 0) return PTQ_ERR_INVALID_ARG;
    DeviceState* dev = nullptr;
    const int st = current_device_state(&dev);
    if (st) return st;
    std::lock_guard<std::mutex> lock(host_state_mutex());
    dev->cta_limit = limit;
    return PTQ_OK;
}

int ptq_profile_enable(int on) {
    Profiler& p = profiler();
    p.clear();
    p.on = on != 0;
    return PTQ_OK;
}

int ptq_profile_read(int kernel_id, double* total_ms, long long* launches) {
    Profiler& p = profiler();
    if (kernel_id < 0 || kernel_id >= K_COUNT || !total_ms || !launches) return PTQ_ERR_INVALID_ARG;
    double ms = 0.0;
    long long cnt = 0;
    for (const auto& r : p.recs) {
        if (r.id != kernel_id) continue;
        if (cudaEventSynchronize(r.b) != cudaSuccess) return PTQ_ERR_CUDA;
        float t = 0.f;
        if (cudaEventElapsedTime(&t, r.a, r.b) != cudaSuccess) return PTQ_ERR_CUDA;
        ms += (double)t;
        ++cnt;
    }
    *total_ms = ms;
    *launches = cnt;
    return PTQ_OK;
}

const char* ptq_status_string(int code) {
    switch (code) {
        case PTQ_OK: return "ok";
        case PTQ_ERR_INVALID_ARG: return "invalid argument";
        case PTQ_ERR_ALIGNMENT: return "pointer or leading dimension not aligned";
        case PTQ_ERR_WORKSPACE: return "workspace too small";
        case PTQ_ERR_NOT_SPD: return "matrix not positive definite";
        case PTQ_ERR_NONFINITE: return "non-finite value";
        case PTQ_ERR_TIMEOUT: return "bounded device wait expired";
        case PTQ_ERR_CUDA: return "CUDA runtime error";
        case PTQ_ERR_UNSUPPORTED: return "unsupported configuration";
        case PTQ_ERR_STATIC_SCRATCH: return "problem too large for the built-in scratch array";
        default: return "unknown status";
    }
}

size_t ptq_workspace_bytes(int call_id, int rows, int cols, int n) {
    if (cols < 1) return 0;
    const size_t c = (size_t)cols;
    size_t total = 0;
    auto add = [&](size_t bytes) { total += align_up(bytes); };
    switch (call_id) {
        case PTQ_CALL_HESSIAN_ACCUMULATE:
            if (n < 1) return 0;
            return gram_workspace_bytes(cols, n);
        case PTQ_CALL_HESSIAN_ACCUMULATE_F64:
            if (n < 1) return 0;
            add(c * (size_t)n * sizeof(double));
            break;
        case PTQ_CALL_PREPARE_HINV:
            add(c * c * sizeof(double));
            add(c * c * sizeof(double));
            add(2 * sizeof(unsigned));                      // grid barrier of the factorisation kernel
            add(chol_scratch_doubles(cols) * sizeof(double));
            add(chol_panel_workspace_bytes(cols));          // operand slices of the panel updates (large matrices)
            break;
        case PTQ_CALL_SENSITIVITY_ORDER:
            if (rows < 1) return 0;
            add((size_t)cdiv(rows, kScoreRowChunk) * c * sizeof(double));
            break;
        case PTQ_CALL_QUANTIZE_LAYER:
            if (rows < 1) return 0;
            add(c * c * sizeof(double));                    // permuted inverse Hessian -> its factor U
            add((size_t)rows * c * sizeof(double));         // permuted W (float64), later dW
            add((size_t)rows * c * sizeof(double));         // scaled errors E
            add((size_t)rows * c);                          // codes in permuted order
            add(c * sizeof(int32_t));                       // inverse permutation
            add(loss_partials_count(rows, cols) * sizeof(double));
            add(2 * sizeof(unsigned));                      // grid barrier of the factorisation kernel
            add(((size_t)cdiv(rows, kSweepRows) + 1) * sizeof(unsigned));   // per-row-group progress counters of the sweep
            add(chol_scratch_doubles(cols) * sizeof(double));
            if (cols >= kPanelMinCols) {
                // slices of U[panel, later] and of E[:, panel]; always for the most digits, so that what suffices for one
                // layer suffices for every smaller one
                add(x_operand_bytes(cols, kPanelBlocks * kNB, kXMoreSlices));
                add(x_operand_bytes(rows, kPanelBlocks * kNB, kXMoreSlices));
            }
            break;
        case PTQ_CALL_QUANTIZE_LAYER_PER_ROW:
            if (rows < 1) return 0;
            add((size_t)rows * sizeof(double));             // per-row losses
            break;
        case PTQ_CALL_QUANTIZE_LAYER_DYNAMIC:
            if (rows < 1) return 0;
            add(c * c * sizeof(double));                    // current matrix and the gathered one (ping-pong)
            add(c * c * sizeof(double));
            add((size_t)rows * c * sizeof(double));         // current weights and the gathered ones (ping-pong)
            add((size_t)rows * c * sizeof(double));
            add((size_t)rows * c * sizeof(double));         // scaled errors E
            add((size_t)rows * c * sizeof(double));         // dW
            add((size_t)rows * c);                          // codes of the block being swept
            add(c * sizeof(double));                        // scores
            add((size_t)cdiv(rows, kScoreRowChunk) * c * sizeof(double));
            add(c * sizeof(int32_t));                       // order of the round
            add(c * sizeof(int32_t));                       // original column of every position (ping-pong)
            add(c * sizeof(int32_t));
            add(loss_partials_count(rows, cols) * sizeof(double));
            add(2 * sizeof(unsigned));
            add(((size_t)cdiv(rows, kSweepRows) + 1) * sizeof(unsigned));
            add(chol_scratch_doubles(cols) * sizeof(double));
            break;
        default:
            return 0;
    }
    return total;
}

int ptq_hessian_accumulate_f64(double* H, const float* X, int cols, int n, int64_t ldx, void* ws, size_t ws_bytes,
                               int32_t* status, void* stream_) {
    (void)status;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (!H || !X || cols < 1 || n < 1 || ldx < n) return PTQ_ERR_INVALID_ARG;
    if (cols > kMaxGridY) return PTQ_ERR_UNSUPPORTED;
    if (!aligned16(H) || !aligned16(ws)) return PTQ_ERR_ALIGNMENT;
    if (!ws || ws_bytes < ptq_workspace_bytes(PTQ_CALL_HESSIAN_ACCUMULATE_F64, 0, cols, n)) return PTQ_ERR_WORKSPACE;
    Carver cv(ws);
    double* Xd = cv.take<double>((size_t)cols * n);
    { Launch l(K_CONVERT_F64, stream); convert_f32_f64_kernel<<<dim3(grid_x_for(n, 256), cols), 256, 0, stream>>>(X, cols, n, ldx, Xd); }
    GemmParams g = gemm_defaults();
    g.A = Xd; g.lda = n; g.a_trans = 0;
    g.B = Xd; g.ldb = n; g.b_trans = 1;
    g.C = H; g.ldc = cols;
    g.M = cols; g.N = cols; g.K = n;
    g.alpha = 2.0; g.beta = 1.0; g.upper_only = 1; g.mirror = 1;
    return launch_dgemm(K_DGEMM_GRAM, g, 1, stream);
}

int ptq_hessian_accumulate(double* H, const float* X, int cols, int n, int64_t ldx, void* ws, size_t ws_bytes,
                           int32_t* status, void* stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (!H || !X || cols < 1 || n < 1 || ldx < n) return PTQ_ERR_INVALID_ARG;
    if (!aligned16(H) || !aligned16(ws)) return PTQ_ERR_ALIGNMENT;
    if (!ws || ws_bytes < ptq_workspace_bytes(PTQ_CALL_HESSIAN_ACCUMULATE, 0, cols, n)) return PTQ_ERR_WORKSPACE;
    GramSource src{};
    src.base = X; src.ldx = ldx;
    return gram_accumulate(H, src, cols, n, ws, status, stream);
}

int ptq_hessian_accumulate_conv(double* H, const float* act, int batch, int channels, int height, int width, int kh,
                                int kw, int stride, int pad, void* ws, size_t ws_bytes, int32_t* status,
                                void* stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (!H || !act || batch < 1 || channels < 1 || height < 1 || width < 1 || kh < 1 || kw < 1 || stride < 1 || pad < 0)
        return PTQ_ERR_INVALID_ARG;
    if (height + 2 * pad < kh || width + 2 * pad < kw) return PTQ_ERR_INVALID_ARG;
    const int64_t oh = (height + 2 * pad - kh) / stride + 1, ow = (width + 2 * pad - kw) / stride + 1;
    const int64_t cols64 = (int64_t)channels * kh * kw, n64 = (int64_t)batch * oh * ow;
    if (cols64 > (1 << 20) || n64 > (int64_t)1 << 30) return PTQ_ERR_UNSUPPORTED;
    const int cols = (int)cols64, n = (int)n64;
    if (!aligned16(H) || !aligned16(ws)) return PTQ_ERR_ALIGNMENT;
    if (!ws || ws_bytes < ptq_workspace_bytes(PTQ_CALL_HESSIAN_ACCUMULATE, 0, cols, n)) return PTQ_ERR_WORKSPACE;
    GramSource src{};
    src.base = act; src.conv = 1;
    src.channels = channels; src.height = height; src.width = width;
    src.kh = kh; src.kw = kw; src.stride = stride; src.pad = pad; src.oh = (int)oh; src.ow = (int)ow;
    return gram_accumulate(H, src, cols, n, ws, status, stream);
}

int ptq_prepare_hinv(const double* H, int cols, int damp_mode, double damp, double* Hinv, double* Hinv_diag,
                     double* lambda_out, void* ws, size_t ws_bytes, int32_t* status, void* stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (!H || !Hinv || !Hinv_diag || !lambda_out || cols < 1 || !(damp >= 0.0)) return PTQ_ERR_INVALID_ARG;
    if (damp_mode != PTQ_DAMP_REL_MEAN_DIAG && damp_mode != PTQ_DAMP_ABS) return PTQ_ERR_INVALID_ARG;
    if (cols > kMaxGridY) return PTQ_ERR_UNSUPPORTED;                          // rows index the grid's y dimension
    if (!aligned16(H) || !aligned16(Hinv) || !aligned16(ws)) return PTQ_ERR_ALIGNMENT;
    if (!ws || ws_bytes < ptq_workspace_bytes(PTQ_CALL_PREPARE_HINV, 0, cols, 0)) return PTQ_ERR_WORKSPACE;
    const int n = cols;
    Carver cv(ws);
    double* R = cv.take<double>((size_t)n * n);
    double* V = cv.take<double>((size_t)n * n);
    unsigned* bar = cv.take<unsigned>(2);
    double* Dbuf = cv.take<double>(chol_scratch_doubles(n));
    void* pws = chol_panel_workspace_bytes(n) ? static_cast<void*>(cv.take<char>(chol_panel_workspace_bytes(n))) : nullptr;
    {
        Launch l(K_LAMBDA, stream);
        launch_chained(lambda_kernel, 1, 256, 0, stream, H, n, damp_mode, damp, lambda_out, status);
    }
    {
        Launch l(K_DAMP_COPY, stream);
        launch_chained(damp_copy_kernel, dim3(cdiv(n, 1024), n), 256, 0, stream, H, R, V, n, lambda_out, bar);
    }
    // W = U^-T comes out of the factorisation sweep itself (V must start as zero)
    int st = cholesky_inverse_upper(R, n, V, Dbuf, bar, pws, status, stream);
    if (st) return st;
    if (n >= kSlicedMinCols && n <= kXMaxK && x_operand_bytes(n, n) <= (size_t)n * n * sizeof(double)) {
        // Hinv = W^T W on the int8 tensor path: the columns of the lower-triangular W are sliced once (into R, which is
        // free now) and serve as both operands; only k >= max(i, j) contributes, upper tiles computed and mirrored
        Carver rv(R);
        const XOperand w = x_slice_operand(rv, V, n, 1, n, n, status, stream);
        XGemmParams prm{};
        prm.C = Hinv; prm.ldc = n; prm.alpha = 1.0; prm.status = status; prm.diag = Hinv_diag;
        prm.out_mode = X_OUT_SYM; prm.k_mode = X_K_FROM_MAX;
        st = x_product(w, w, prm, stream);
    } else {
        st = lauum_lower(V, Hinv, Hinv_diag, n, stream);
    }
    return st ? st : launch_status();
}

int ptq_minmax_grid(const float* W, int rows, int cols, int64_t ldw, int bits, float* scale, float* zero,
                    int32_t* status, void* stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (!W || !scale || !zero || rows < 1 || cols < 1 || ldw < cols || bits < 2 || bits > 8)
        return PTQ_ERR_INVALID_ARG;
    {
        Launch l(K_MINMAX_GRID, stream);
        launch_chained(minmax_grid_kernel, rows, 256, 0, stream, W, rows, cols, ldw, bits, scale, zero, status);
    }
    return launch_status();
}

int ptq_sensitivity_order(const float* W, int rows, int cols, int64_t ldw, const double* Hinv_diag, const float* scale,
                          const float* zero, int bits, int score_mode, double* S, int32_t* perm, void* ws,
                          size_t ws_bytes, int32_t* status, void* stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    const int bad = order_args_check(W, rows, cols, ldw, Hinv_diag, scale, zero, bits, score_mode, S, perm);
    if (bad) return bad;
    if (!ws || ws_bytes < ptq_workspace_bytes(PTQ_CALL_SENSITIVITY_ORDER, rows, cols, 0)) return PTQ_ERR_WORKSPACE;
    if (!aligned16(ws)) return PTQ_ERR_ALIGNMENT;
    Carver cv(ws);
    double* partial = cv.take<double>((size_t)cdiv(rows, kScoreRowChunk) * cols);
    return order_launch(W, rows, cols, ldw, Hinv_diag, scale, zero, bits, score_mode & ~PTQ_SCORE_ASCENDING,
                        (score_mode & PTQ_SCORE_ASCENDING) ? 1 : 0, S, perm, partial, status, stream);
}

int ptq_sensitivity_order_static(const float* W, int rows, int cols, int64_t ldw, const double* Hinv_diag,
                                 const float* scale, const float* zero, int bits, int score_mode, double* S,
                                 int32_t* perm, int32_t* status, void* stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    const int bad = order_args_check(W, rows, cols, ldw, Hinv_diag, scale, zero, bits, score_mode, S, perm);
    if (bad) return bad;
    if ((size_t)cdiv(rows, kScoreRowChunk) * (size_t)cols > kStaticScratchDoubles) return PTQ_ERR_STATIC_SCRATCH;
    double* partial = nullptr;
    const int st = static_scratch_address(&partial);
    if (st) return st;
    // Every partial[ch][j] that score_final_kernel reads is written first by score_partial_kernel, so nothing
    // left in the array by an earlier call is ever used and nothing needs clearing.
    return order_launch(W, rows, cols, ldw, Hinv_diag, scale, zero, bits, score_mode & ~PTQ_SCORE_ASCENDING,
                        (score_mode & PTQ_SCORE_ASCENDING) ? 1 : 0, S, perm, partial, status, stream);
}

int ptq_quantize_layer_dynamic(const float* W, int rows, int cols, int64_t ldw, const double* Hinv, const float* scale,
                               const float* zero, int bits, int score_mode, int block, uint8_t* codes, float* What,
                               int32_t* order_out, const double* H_undamped, double* loss_out, void* ws,
                               size_t ws_bytes, int32_t* status, void* stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (!W || !Hinv || !scale || !zero || !codes || !order_out || rows < 1 || cols < 1 || ldw < cols || bits < 2 ||
        bits > 8 || block < 1)
        return PTQ_ERR_INVALID_ARG;
    if (score_mode & ~(PTQ_SCORE_ASCENDING | 7)) return PTQ_ERR_INVALID_ARG;
    const int mode = score_mode & ~PTQ_SCORE_ASCENDING, ascending = (score_mode & PTQ_SCORE_ASCENDING) ? 1 : 0;
    if (mode < PTQ_SCORE_QERR || mode > PTQ_SCORE_NONE) return PTQ_ERR_INVALID_ARG;
    if (block < cols && (block % kNB) != 0) return PTQ_ERR_UNSUPPORTED;     // rounds end on the 64-column block grid
    if (rows > kMaxGridY || cols > kMaxGridY || cdiv(rows, kScoreRowChunk) > kMaxGridY) return PTQ_ERR_UNSUPPORTED;
    if (!aligned16(Hinv) || !aligned16(ws)) return PTQ_ERR_ALIGNMENT;
    if (!ws || ws_bytes < ptq_workspace_bytes(PTQ_CALL_QUANTIZE_LAYER_DYNAMIC, rows, cols, 0)) return PTQ_ERR_WORKSPACE;
    const size_t c = (size_t)cols;
    Carver cv(ws);
    double* Abuf[2] = {cv.take<double>(c * c), nullptr};
    Abuf[1] = cv.take<double>(c * c);
    double* Wbuf[2] = {cv.take<double>((size_t)rows * c), nullptr};
    Wbuf[1] = cv.take<double>((size_t)rows * c);
    double* E = cv.take<double>((size_t)rows * c);
    double* dW = cv.take<double>((size_t)rows * c);
    uint8_t* codes_p = cv.take<uint8_t>((size_t)rows * c);
    double* S = cv.take<double>(c);
    const int chunks = cdiv(rows, kScoreRowChunk);
    double* partial = cv.take<double>((size_t)chunks * c);
    int32_t* ordr = cv.take<int32_t>(c);
    int32_t* obuf[2] = {cv.take<int32_t>(c), nullptr};
    obuf[1] = cv.take<int32_t>(c);
    double* partials = cv.take<double>(loss_partials_count(rows, cols));
    unsigned* bar = cv.take<unsigned>(2);
    unsigned* sweep_flags = cv.take<unsigned>((size_t)cdiv(rows, kSweepRows) + 1);
    double* Dbuf = cv.take<double>(chol_scratch_doubles(cols));
    const bool want_loss = H_undamped && loss_out;
    DeviceState* dev = nullptr;
    {
        const int dst = current_device_state(&dev);
        if (dst) return dst;
    }

    const int32_t* ocur = nullptr;           // original column index of every current position; none yet: itself
    // current state: the m columns still to do, their matrix (upper triangle valid) and their weights
    const double* Acur = Hinv;
    int64_t lda = cols;
    const double* Wcur = nullptr;            // round 0 reads the float32 weights
    int64_t ldc = 0;
    int m = cols, done = 0, cur = 0;
    while (m > 0) {
        const int b = block < m ? block : m;
        if (mode != PTQ_SCORE_NONE) {
            Launch l(K_SCORE_PARTIAL, stream);
            if (Wcur)
                launch_chained(score_partial_kernel<double>, dim3(cdiv(m, kScoreCols), chunks), 256, 0, stream, Wcur, rows, m,
                               ldc, scale, zero, bits, mode, partial);
            else
                launch_chained(score_partial_kernel<float>, dim3(cdiv(m, kScoreCols), chunks), 256, 0, stream, W, rows, m,
                               ldw, scale, zero, bits, mode, partial);
        }
        {
            Launch l(K_SCORE_FINAL, stream);
            launch_chained(score_final_kernel, cdiv(m, 128), 128, 0, stream, partial, chunks, m, Acur, lda + 1, mode, S,
                           status);
        }
        {
            Launch l(K_RANK_SORT, stream);
            launch_chained(rank_sort_kernel, cdiv(m, kRankCols), 256, 0, stream, S, m, ascending, ordr, ocur);
        }
        double* An = Abuf[cur];
        double* Wn = Wbuf[cur];
        int32_t* onew = obuf[cur ^ 1];
        {
            Launch l(K_DYN_GATHER, stream);
            const dim3 grid(grid_x_for(m, 256), m + rows < 8192 ? m + rows : 8192);
            const int n_flags = cdiv(rows, kSweepRows) + 1;
            if (Wcur)
                launch_chained(round_gather_kernel<double>, grid, 256, 0, stream, Acur, lda, Wcur, ldc, rows, ordr, ocur, m,
                               b, An, Wn, E, onew, order_out + done, bar, sweep_flags, n_flags);
            else
                launch_chained(round_gather_kernel<float>, grid, 256, 0, stream, Acur, lda, W, ldw, rows, ordr, ocur, m, b,
                               An, Wn, E, onew, order_out + done, bar, sweep_flags, n_flags);
        }
        int st = PTQ_OK;
        const CholRange range = {0, b < m ? b / kNB : cdiv(m, kNB), cdiv(m, kNB)};
        const int budget = coop_cta_budget(dev), behind = sweep_ctas_behind(rows, b, m, range, budget);
        if (behind > 0) {
            st = factor_sweep_launch(An, m, range, Dbuf, bar, behind, Wn, E, codes_p, scale, zero, rows, b, bits, sweep_flags, status,
                                     stream, budget, true);
        } else {
            st = cholesky_upper(An, m, nullptr, Dbuf, bar, status, stream, range.stop, 0, 0, true);
            if (st) return st;
            st = sweep_launch(Wn, An, E, codes_p, scale, zero, rows, b, bits, sweep_flags, status, stream, m, true);
        }
        if (st) return st;
        if (b < m) {
            // Eq. 11 for the columns still to come, all b columns at once: Wn[:, b:] -= E[:, :b] U[:b, b:]
            GemmParams g = gemm_defaults();
            g.A = E; g.lda = m; g.a_trans = 0;
            g.B = An + b; g.ldb = m; g.b_trans = 0;
            g.C = Wn + b; g.ldc = m;
            g.M = rows; g.N = m - b; g.K = b;
            g.alpha = -1.0; g.beta = 1.0;
            st = launch_dgemm(K_DGEMM_DYN, g, 1, stream);
            if (st) return st;
        }
        {
            Launch l(K_DYN_AUX, stream);
            const int gr = rows < 4096 ? rows : 4096;
            launch_chained(emit_block_kernel, dim3(grid_x_for(b, 256), gr), 256, 0, stream, codes_p, m, onew, b, W, rows,
                           cols, ldw, scale, zero, codes, What, want_loss ? dW : nullptr);
        }
        Acur = An + (size_t)b * m + b; lda = m;
        Wcur = Wn + b; ldc = m;
        // what is left of the gathered arrays is the next round's state; the next round gathers into the other buffers
        ocur = onew + b;
        done += b;
        m -= b;
        cur ^= 1;
    }
    if (want_loss) {
        GemmParams g = gemm_defaults();
        g.kend_mode = 1; g.sym_double = 1;
        g.A = dW; g.lda = cols; g.a_trans = 0;
        g.B = H_undamped; g.ldb = cols; g.b_trans = 0;
        g.M = rows; g.N = cols; g.K = cols;
        g.D = dW; g.ldd = cols; g.partials = partials;
        g.ksplit = loss_ksplit(rows, cols);
        dim3 grid;
        const int st = launch_dgemm(K_DGEMM_LOSS, g, 1, stream, 64, &grid);
        if (st) return st;
        {
            Launch l(K_SUM_PARTIALS, stream);
            launch_chained(sum_partials_kernel, 1, 256, 0, stream, partials, (int)(grid.x * grid.y * grid.z), 0.5, loss_out);
        }
    }
    return launch_status();
}

int ptq_quantize_layer_per_row(const float* W, int rows, int cols, int64_t ldw, const double* Hinv, const float* scale,
                               const float* zero, int bits, int score_mode, uint8_t* codes, float* What,
                               int32_t* perm_rows, const double* H_undamped, double* loss_out, void* ws,
                               size_t ws_bytes, int32_t* status, void* stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (!W || !Hinv || !scale || !zero || !codes || !perm_rows || rows < 1 || cols < 1 || ldw < cols || bits < 2 ||
        bits > 8)
        return PTQ_ERR_INVALID_ARG;
    if (score_mode & ~(PTQ_SCORE_ASCENDING | 7)) return PTQ_ERR_INVALID_ARG;
    const int mode = score_mode & ~PTQ_SCORE_ASCENDING, ascending = (score_mode & PTQ_SCORE_ASCENDING) ? 1 : 0;
    if (mode < PTQ_SCORE_QERR || mode > PTQ_SCORE_NONE) return PTQ_ERR_INVALID_ARG;
    if (cols > kPerRowMaxCols) return PTQ_ERR_UNSUPPORTED;       // one private inverse Hessian per CTA, in shared memory
    if (!ws || ws_bytes < ptq_workspace_bytes(PTQ_CALL_QUANTIZE_LAYER_PER_ROW, rows, cols, 0)) return PTQ_ERR_WORKSPACE;
    if (!aligned16(ws)) return PTQ_ERR_ALIGNMENT;
    DeviceState* dev = nullptr;
    int st = current_device_state(&dev);
    if (st) return st;
    st = ensure_smem_attr(dev, SA_SMALL, [] {
        return cudaFuncSetAttribute(per_row_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)per_row_smem_bytes(kPerRowMaxCols));
    });
    if (st) return st;
    Carver cv(ws);
    double* row_loss = cv.take<double>(rows);
    const bool want_loss = H_undamped && loss_out;
    {
        Launch l(K_PER_ROW, stream);
        launch_chained(per_row_kernel, rows, kPerRowThreads, per_row_smem_bytes(cols), stream, W, rows, cols, ldw, Hinv,
                       scale, zero, bits, mode, ascending, codes, What, perm_rows, want_loss ? H_undamped : nullptr,
                       want_loss ? row_loss : nullptr, status);
    }
    if (want_loss) {
        Launch l(K_SUM_PARTIALS, stream);
        launch_chained(sum_partials_kernel, 1, 256, 0, stream, row_loss, rows, 1.0, loss_out);
    }
    return launch_status();
}

size_t ptq_gemm_nt_sliced_workspace_bytes(int m, int n, int k) {
    if (m < 1 || n < 1 || k < 1) return 0;
    return i8gemm_workspace_bytes(m, n, k);
}

int ptq_gemm_nt_sliced(double* C, int64_t ldc, const double* A, int64_t lda, const double* B, int64_t ldb, int b_is_kn,
                       int m, int n, int k, double alpha, void* ws, size_t ws_bytes, int32_t* status, void* stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (!C || !A || !B || m < 1 || n < 1 || k < 1 || ldc < n || lda < k || ldb < (b_is_kn ? n : k))
        return PTQ_ERR_INVALID_ARG;
    if (k > kXMaxK) return PTQ_ERR_UNSUPPORTED;
    if (!ws || ws_bytes < i8gemm_workspace_bytes(m, n, k)) return PTQ_ERR_WORKSPACE;
    if (!aligned16(ws)) return PTQ_ERR_ALIGNMENT;
    return i8gemm_nt(C, ldc, A, lda, B, ldb, b_is_kn ? 1 : 0, m, n, k, alpha, ws, status, stream);
}

int ptq_sort_scores(const double* S, int cols, int ascending, int32_t* perm, void* stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (!S || !perm || cols < 1) return PTQ_ERR_INVALID_ARG;
    {
        Launch l(K_RANK_SORT, stream);
        launch_chained(rank_sort_kernel, cdiv(cols, kRankCols), 256, 0, stream, S, cols, ascending ? 1 : 0, perm, nullptr);
    }
    return launch_status();
}

int ptq_selftest_wait_timeout(int which, long long limit_cycles, void* ws, size_t ws_bytes, int32_t* status,
                              void* stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if ((which != 0 && which != 1) || limit_cycles < 1 || limit_cycles > kSpinLimitCycles || !status)
        return PTQ_ERR_INVALID_ARG;
    if (!ws || ws_bytes < 4 * sizeof(unsigned)) return PTQ_ERR_WORKSPACE;
    if (!aligned16(ws)) return PTQ_ERR_ALIGNMENT;
    unsigned* words = static_cast<unsigned*>(ws);
    if (cudaMemsetAsync(words, 0, 4 * sizeof(unsigned), stream) != cudaSuccess) return PTQ_ERR_CUDA;
    if (which == 1) {
        Launch l(K_SELFTEST, stream);
        selftest_counter_kernel<<<1, 32, 0, stream>>>(words, status, limit_cycles);
        return launch_status();
    }
    DeviceState* dev = nullptr;
    const int st = current_device_state(&dev);
    if (st) return st;
    if (!dev->coop) return PTQ_ERR_UNSUPPORTED;
    void* args[] = {&words, &status, &limit_cycles};
    Launch l(K_SELFTEST, stream);
    if (cudaLaunchCooperativeKernel((const void*)selftest_barrier_kernel, dim3(dev->sms), dim3(kCholThreads), args, 0,
                                    stream) != cudaSuccess) {
        cudaGetLastError();
        return PTQ_ERR_CUDA;
    }
    return PTQ_OK;
}

int ptq_selftest_abandoned_sweep(long long limit_cycles, void* ws, size_t ws_bytes, int32_t* abort_word, int32_t* status,
                                 void* stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (limit_cycles < 1 || limit_cycles > kSpinLimitCycles || !abort_word || !status) return PTQ_ERR_INVALID_ARG;
    if (!ws || ws_bytes < PTQ_ABANDONED_SWEEP_BYTES) return PTQ_ERR_WORKSPACE;
    if (!aligned16(ws)) return PTQ_ERR_ALIGNMENT;
    constexpr int groups = kAbandonedRows / kSweepRows;
    Carver cv(ws);
    double* U = cv.take<double>(kNB * kNB);
    double* Wp = cv.take<double>(kAbandonedRows * kNB);
    double* E = cv.take<double>(kAbandonedRows * kNB);
    double* Dbuf = cv.take<double>(chol_scratch_doubles(kNB));
    float* scale = cv.take<float>(kAbandonedRows);
    float* zero = cv.take<float>(kAbandonedRows);
    uint8_t* codes = cv.take<uint8_t>(kAbandonedRows * kNB);
    unsigned* bar = cv.take<unsigned>(2);
    unsigned* flags = cv.take<unsigned>(groups + 1);
    static_assert(4 * kNB * kNB * 8 + 2 * kNB * 4 + kNB * kNB + 2 * 256 <= PTQ_ABANDONED_SWEEP_BYTES, "the pieces above");
    { Launch l(K_SELFTEST, stream); selftest_unit_layer_kernel<<<kNB, kNB, 0, stream>>>(U, Wp, E, scale, zero); }
    // one CTA per row group, so that nothing but the wait for the factorisation can raise the sweep's abort word
    const int st = factor_sweep_launch(U, kNB, chol_all_rows(kNB), Dbuf, bar, groups, Wp, E, codes, scale, zero, kAbandonedRows, kNB, 4,
                                       flags, status, stream, groups + 1, false, limit_cycles, 1u);
    if (st) return st;
    if (cudaMemcpyAsync(abort_word, flags + groups, sizeof(int32_t), cudaMemcpyDeviceToDevice, stream) != cudaSuccess)
        return PTQ_ERR_CUDA;
    return launch_status();
}

int ptq_selftest_reciprocal(const double* x, int n, double* rcp, double* rsq, void* stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (!x || !rcp || !rsq || n < 1) return PTQ_ERR_INVALID_ARG;
    { Launch l(K_SELFTEST, stream); selftest_reciprocal_kernel<<<cdiv(n, 256), 256, 0, stream>>>(x, n, rcp, rsq); }
    return launch_status();
}

int ptq_fp64_probe(int kind, int iters, double* sink, double* flops_out, void* stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if ((kind != 0 && kind != 1) || iters < 1 || iters > (1 << 24) || !sink || !flops_out) return PTQ_ERR_INVALID_ARG;
    DeviceState* dev = nullptr;
    const int st = current_device_state(&dev);
    if (st) return st;
    const int grid = dev->sms * kProbeCtasPerSm;
    const double threads = (double)grid * kProbeThreads;
    Launch l(K_FP64_PROBE, stream);
    if (kind == 0) {
        fp64_probe_fma_kernel<<<grid, kProbeThreads, 0, stream>>>(iters, sink);
        *flops_out = threads * kProbeChains * (double)iters * 2.0;
    } else {
        fp64_probe_mma_kernel<<<grid, kProbeThreads, 0, stream>>>(iters, sink);
        *flops_out = (threads / 32.0) * kProbeChains * (double)iters * (8.0 * 8.0 * 4.0 * 2.0);
    }
    return launch_status();
}

int ptq_quantize_layer(const float* W, int rows, int cols, int64_t ldw, const double* Hinv, const int32_t* perm,
                       const float* scale, const float* zero, int bits, uint8_t* codes, float* What,
                       const double* H_undamped, double* loss_out, void* ws, size_t ws_bytes, int32_t* status,
                       void* stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (!W || !Hinv || !perm || !scale || !zero || !codes || rows < 1 || cols < 1 || ldw < cols || bits < 2 ||
        bits > 8)
        return PTQ_ERR_INVALID_ARG;
    if (rows > kMaxGridY || cols > kMaxGridY) return PTQ_ERR_UNSUPPORTED;     // rows / columns index the grid's y dimension
    if (!aligned16(Hinv) || !aligned16(ws)) return PTQ_ERR_ALIGNMENT;
    if (!ws || ws_bytes < ptq_workspace_bytes(PTQ_CALL_QUANTIZE_LAYER, rows, cols, 0)) return PTQ_ERR_WORKSPACE;
    const int n = cols;
    Carver cv(ws);
    double* U = cv.take<double>((size_t)n * n);
    double* Wp = cv.take<double>((size_t)rows * n);
    double* E = cv.take<double>((size_t)rows * n);
    uint8_t* codes_p = cv.take<uint8_t>((size_t)rows * n);
    int32_t* invperm = cv.take<int32_t>(n);
    double* partials = cv.take<double>(loss_partials_count(rows, cols));
    unsigned* bar = cv.take<unsigned>(2);
    unsigned* sweep_flags = cv.take<unsigned>((size_t)cdiv(rows, kSweepRows) + 1);
    double* Dbuf = cv.take<double>(chol_scratch_doubles(n));
    const int digits = deferred_digits(rows, n);
    auto panel_operand = [&](int r) {
        return n >= kPanelMinCols ? static_cast<void*>(cv.take<char>(x_operand_bytes(r, kPanelBlocks * kNB, digits))) : nullptr;
    };
    void* uws = panel_operand(n);
    void* ews = panel_operand(rows);

    DeviceState* dev = nullptr;
    int st = current_device_state(&dev);
    if (st) return st;
    st = ensure_smem_attr(dev, SA_GATHER, [] {
        return cudaFuncSetAttribute(sweep_gather_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    kGatherMaxCols * (int)sizeof(double));
    });
    if (st) return st;
    const int n_flags = cdiv(rows, kSweepRows) + 1;
    {
        Launch l(K_PERM_CHECK, stream);
        launch_chained(perm_check_kernel, cdiv(n, 256), 256, 0, stream, perm, n, invperm, bar, sweep_flags, n_flags, status);
    }
    {
        Launch l(K_SWEEP_GATHER, stream);
        if (n <= kGatherMaxCols)
            launch_chained(sweep_gather_kernel<true>, n + rows, kGatherThreads, (size_t)n * sizeof(double), stream, Hinv, W,
                           rows, n, ldw, perm, invperm, U, Wp, E, status);
        else
            launch_chained(sweep_gather_kernel<false>, n + rows, kGatherThreads, 0, stream, Hinv, W, rows, n, ldw, perm,
                           invperm, U, Wp, E, status);
    }
    // Blocked Eq. 12 and the sweep: of everything at once, or, on wide layers, panel by panel (cholpanel.cuh).  There the part of
    // Eq. 11 that a panel's columns owe to all later ones, W[:, later] -= E[:, panel] U[panel, later], is one large product on
    // the int8 tensor path, as the panel's share of Eq. 12 is; both take the same slices of U.  (4096 x 11008 with the
    // updates inside the sweep kernel instead, 32 x 64 x 64 tiles: 30 ms in place of 11.)
    const int budget = coop_cta_budget(dev), panel = n >= kPanelMinCols ? kPanelBlocks : cdiv(n, kNB);
    for (int kf = 0; kf < cdiv(n, kNB); kf += panel) {
        const int off = kf * kNB, cols_now = n - off < panel * kNB ? n - off : panel * kNB, rest = n - off - cols_now;
        const CholRange range = {kf, kf + cdiv(cols_now, kNB), kf + cdiv(cols_now, kNB)};
        const int behind = sweep_ctas_behind(rows, cols_now, n, range, budget);
        if (behind > 0) {
            st = factor_sweep_launch(U, n, range, Dbuf, bar, behind, Wp + off, E + off, codes_p + off, scale, zero, rows, cols_now, bits,
                                     sweep_flags, status, stream, budget, kf == 0);
        } else {
            st = cholesky_upper(U, n, nullptr, Dbuf, bar, status, stream, range.stop, range.first, range.row_limit, kf == 0);
            if (st) return st;
            st = sweep_launch(Wp + off, U + (size_t)off * (n + 1), E + off, codes_p + off, scale, zero, rows, cols_now, bits, sweep_flags,
                              status, stream, n, kf == 0);
        }
        if (st) return st;
        if (rest > 0) {
            Carver uv(uws), ev(ews);
            double* below = U + (size_t)off * n + off + cols_now;                 // U[panel, later]
            const XOperand u = x_slice_operand(uv, below, n, 1, rest, cols_now, status, stream, nullptr, 1, digits);
            st = chol_apply_panel(U, n, off + cols_now, u, status, stream);
            if (st) return st;
            const XOperand e = x_slice_operand(ev, E + off, n, 0, rows, cols_now, status, stream, nullptr, 1, digits);
            XGemmParams prm{};
            prm.C = Wp + off + cols_now; prm.ldc = n; prm.alpha = -1.0; prm.status = status;
            prm.out_mode = X_OUT_ADD; prm.k_mode = X_K_ALL;
            st = x_product(e, u, prm, stream, digits);
            if (st) return st;
        }
    }

    const bool want_loss = H_undamped && loss_out;
    double* dW = want_loss ? Wp : nullptr;
    const bool sliced = want_loss && sliced_loss(rows, n);
    int8_t* kexp = sliced ? reinterpret_cast<int8_t*>(Dbuf) : nullptr;      // the factorisation is done with Dbuf
    {
        Launch l(K_FINALIZE, stream);
        launch_chained(finalize_kernel, dim3(cdiv(n, 1024), rows), 256, 0, stream, codes_p, invperm, W, rows, n, ldw, scale,
                       zero, codes, What, dW, H_undamped, kexp);
    }
    if (sliced) {
        // 1/2 sum_ij dW_ij (dW H)_ij on the int8 tensor path.  H is symmetric: per 64-column block j the column blocks
        // k < j count twice (they stand in for the blocks k > j as well) and the block k = j once, so two products
        // with reduction epilogues, k before the tile's own block (weight 2 * 1/2) and k in it (weight 1/2).
        // The slices of dW go where E was, those of H where U was: both are free now.
        Carver ev(E), uv(U);
        const XOperand a = x_slice_operand(ev, dW, n, 0, rows, n, status, stream, kexp, 1);
        const XOperand b = x_slice_operand(uv, H_undamped, n, 0, n, n, status, stream, kexp, -1);
        const int tiles = x_num_tiles(rows, n);
        XGemmParams prm{};
        prm.status = status; prm.out_mode = X_OUT_REDUCE; prm.D = dW; prm.ldd = n;
        prm.k_mode = X_K_BEFORE_J; prm.alpha = 1.0; prm.partials = partials;
        st = x_product(a, b, prm, stream);
        if (st) return st;
        prm.k_mode = X_K_OWN_J; prm.alpha = 0.5; prm.partials = partials + tiles;
        st = x_product(a, b, prm, stream);
        if (st) return st;
        {
            Launch l(K_SUM_PARTIALS, stream);
            launch_chained(sum_partials_kernel, 1, 256, 0, stream, partials, 2 * tiles, 1.0, loss_out);
        }
    } else if (want_loss) {
        // sum_ic dW_ic (dW H)_ic; H is symmetric, so for the 64-column block of c only k up to the end of that block is
        // summed and the blocks before it are doubled
        GemmParams g = gemm_defaults();
        g.kend_mode = 1; g.sym_double = 1;
        g.A = dW; g.lda = n; g.a_trans = 0;
        g.B = H_undamped; g.ldb = n; g.b_trans = 0;
        g.M = rows; g.N = n; g.K = n;
        g.D = dW; g.ldd = n; g.partials = partials;
        g.ksplit = loss_ksplit(rows, n);
        dim3 grid;
        st = launch_dgemm(K_DGEMM_LOSS, g, 1, stream, 64, &grid);
        if (st) return st;
        {
            Launch l(K_SUM_PARTIALS, stream);
            launch_chained(sum_partials_kernel, 1, 256, 0, stream, partials, (int)(grid.x * grid.y * grid.z), 0.5, loss_out);
        }
    }
    return launch_status();
}

}  // extern "C"
