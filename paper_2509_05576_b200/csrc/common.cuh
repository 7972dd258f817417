// Shared host/device helpers of the quantizer library (status word, launch checks, workspace carving).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>
#include <mutex>
#include <vector>

#include "../../include/ptq.h"

namespace ptq {

constexpr int kNB = 64;  // block size of the factorisations and of the column loop

// Pivots of a factorisation are accepted from the smallest normal number up to 10^300: the hardware approximations that the
// chains refine take a subnormal for zero, and the reciprocal of what lies above is (nearly) subnormal itself.
constexpr double kMinPivot = 2.2250738585072014e-308, kMaxPivot = 1.0e300;

// 1 / d and 1 / sqrt(d) of an accepted pivot without a branch: what a chain of eight pivots waits for.  Both take the
// hardware's approximation (a documented instruction, about 20 bits) as the start of one step of third order:
//   1 / d:        y (1 + e + e^2), e = 1 - d y: the hyperpower iteration of order three (M. Altman, Pacific J. Math. 10, 1960),
//                 i.e. the geometric series of 1 / (1 - e) cut off before e^3;
//   1 / sqrt(d):  z (1 + g / 2 + 3 g^2 / 8), g = 1 - d z^2: Newton's binomial series of (1 - g)^(-1/2) cut off before g^3.
// What is cut off is below 2^-56.  Left are the rounding of the result and, for the root, that of z^2, whose half enters:
// at most 0.6 and 1.1 units in the last place (ptq_selftest_reciprocal).
__device__ __forceinline__ double pivot_reciprocal(double d) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
    const double e = fma(-d, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double pivot_rsqrt(double d) {
    double z;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(z) : "d"(d));
    const double g = fma(-(z * z), d, 1.0);
    return fma(z, g * fma(0.375, g, 0.5), z);
}

// First statement of a kernel launched by launch_chained.  chained_wait: waits until the kernel before it in the stream is done
// and its writes are there.  chained_begin: and then lets the next kernel be put in place, whose CTAs wait here in turn.
// The long kernels (Gram, products) do without the latter: CTAs that wait beside them cost more than the launch they hide
// (a 256 x 2304 layer 1783 us without, 1840 us with).
__device__ __forceinline__ void chained_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chained_begin() {
    chained_wait();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// First error wins; later kernels keep running on whatever numbers they find (no traps, no faults).
__device__ __forceinline__ void report(int32_t* status, int code, int index, int aux = 0) {
    if (status && atomicCAS(status, 0, code) == 0) {
        status[1] = index;
        status[2] = aux;
    }
}

// ---------------------------------------------------------------------------------------------------------
// Shared-memory barriers and tensor-map (TMA) tile copies used by the tile pipelines.
// ---------------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn get_encode_tiled() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

inline size_t align_up(size_t x, size_t a = 256) { return (x + a - 1) / a * a; }

// Carves aligned pieces out of the caller's workspace.
struct Carver {
    char* base;
    size_t off = 0;
    explicit Carver(void* p) : base(static_cast<char*>(p)) {}
    template <typename T>
    T* take(size_t count) {
        T* p = reinterpret_cast<T*>(base + off);
        off = align_up(off + count * sizeof(T));
        return p;
    }
};

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Launches a kernel that begins with chained_begin() or chained_wait(): its launch overlaps the kernel before it in the stream
// instead of following its end.  A layer is some twenty launches, most of them of a few microseconds: 64 x 128 148 -> 130 us,
// 64 x 147 as a graph 161 -> 154, 128 x 1152 with dynamic re-ranking (some 120 launches) 1235 -> 1060, 256 x 2304 1810 -> 1783.
// (The cooperative kernels keep their ordinary launch: the same times with it and without.)
template <typename... Params, typename... Args>
inline void launch_chained(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, Args... args) {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = stream;
    cfg.attrs = attr; cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);       // an error stays for launch_status()
}

inline int launch_status() { return cudaGetLastError() == cudaSuccess ? PTQ_OK : PTQ_ERR_CUDA; }

inline int cdiv(int a, int b) { return (a + b - 1) / b; }

// Bounded device-side waits give up after this many SM clock cycles (about two seconds).
constexpr long long kSpinLimitCycles = 4000000000LL;

// ---------------------------------------------------------------------------------------------------------
// Host-side state that belongs to a DEVICE, not to the process: the SM count that sizes the persistent grids, the
// cooperative-launch capability and which kernels already carry their dynamic shared-memory attribute there
// (cudaFuncSetAttribute is per device).  One table, one mutex; looked up with the caller's device current.
// ---------------------------------------------------------------------------------------------------------
constexpr int kMaxDevices = 64;
enum SmemAttrSlot { SA_CHOL = 0, SA_SWEEP, SA_GRAM, SA_DGEMM, SA_SMALL, SA_XGEMM, SA_FACTOR_SWEEP, SA_GATHER, SA_COUNT };
struct DeviceState {
    int sms = 0;
    int coop = 0;
    int cta_limit = 0;            // > 0: the persistent cooperative kernels launch at most this many CTAs (ptq_set_cta_limit)
    bool attr[SA_COUNT] = {};
};
inline std::mutex& host_state_mutex() { static std::mutex mu; return mu; }
inline int current_device_state(DeviceState** out) {
    static DeviceState table[kMaxDevices];
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return PTQ_ERR_CUDA;
    std::lock_guard<std::mutex> lock(host_state_mutex());
    DeviceState& d = table[dev];
    if (d.sms == 0) {
        int sms = 0, coop = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return PTQ_ERR_CUDA;
        if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess) return PTQ_ERR_CUDA;
        d.coop = coop;
        d.sms = sms;
    }
    *out = &d;
    return PTQ_OK;
}
// CTAs a persistent cooperative kernel may launch on this device: one per SM, or the caller's limit if that is lower.
inline int coop_cta_budget(const DeviceState* d) {
    std::lock_guard<std::mutex> lock(host_state_mutex());
    return (d->cta_limit > 0 && d->cta_limit < d->sms) ? d->cta_limit : d->sms;
}
// Runs `set` (the cudaFuncSetAttribute calls of one kernel family) once per device.
template <typename F>
inline int ensure_smem_attr(DeviceState* d, SmemAttrSlot slot, F set) {
    std::lock_guard<std::mutex> lock(host_state_mutex());
    if (!d->attr[slot]) {
        if (set() != cudaSuccess) { cudaGetLastError(); return PTQ_ERR_CUDA; }
        d->attr[slot] = true;
    }
    return PTQ_OK;
}

// ---------------------------------------------------------------------------------------------------------
// Launch accounting.  Every kernel launch of the library goes through a Launch scope: it always counts the
// launch, and, while profiling is enabled, brackets it with CUDA events on the launching stream so that the
// bench can read per-kernel device time live.  Profiling adds event records between kernels, so it is used on
// separate, untimed passes.
// ---------------------------------------------------------------------------------------------------------
enum KernelId {
    K_GRAM_SPLIT = 0, K_GRAM_I8, K_GRAM_FINISH, K_CONVERT_F64, K_DGEMM_GRAM, K_LAMBDA, K_DAMP_COPY, K_CHOL_COOP,
    K_DGEMM_LAUUM, K_MINMAX_GRID, K_SCORE_PARTIAL,
    K_SCORE_FINAL, K_RANK_SORT, K_PERM_CHECK, K_SWEEP_GATHER, K_SWEEP_COOP, K_FINALIZE,
    K_DGEMM_LOSS, K_SUM_PARTIALS, K_SELFTEST, K_FP64_PROBE, K_DYN_AUX, K_DYN_GATHER,
    K_DGEMM_DYN, K_PER_ROW, K_DGEMM_EQ11, K_X_SLICE, K_X_GEMM, K_FACTOR_SWEEP, K_COUNT
};

inline const char* kernel_name(int id) {
    static const char* names[K_COUNT] = {
        "gram_split", "gram_i8_tcgen05", "gram_finish", "convert_f64", "dgemm_gram_f64", "lambda", "damp_copy", "chol_coop",
        "dgemm_lauum",
        "minmax_grid", "score_partial", "score_final", "rank_sort", "perm_check", "sweep_gather",
        "sweep_coop", "finalize", "dgemm_loss", "sum_partials", "selftest", "fp64_probe", "dyn_aux", "dyn_gather",
        "dgemm_dyn", "per_row", "dgemm_eq11", "x_slice", "i8gemm_tcgen05", "factor_sweep"};
    return (id >= 0 && id < K_COUNT) ? names[id] : "unknown";
}

struct Profiler {
    bool on = false;
    long long launches[K_COUNT] = {};
    struct Rec { int id; cudaEvent_t a, b; };
    std::vector<Rec> recs;
    std::vector<cudaEvent_t> pool;
    cudaEvent_t get() {
        if (!pool.empty()) { cudaEvent_t e = pool.back(); pool.pop_back(); return e; }
        cudaEvent_t e = nullptr;
        cudaEventCreate(&e);
        return e;
    }
    void clear() {
        for (auto& r : recs) { pool.push_back(r.a); pool.push_back(r.b); }
        recs.clear();
    }
};
inline Profiler& profiler() { static Profiler p; return p; }

inline std::mutex& profiler_mutex() { static std::mutex mu; return mu; }

struct Launch {
    int id; cudaStream_t s; cudaEvent_t a = nullptr, b = nullptr;
    Launch(int id_, cudaStream_t s_) : id(id_), s(s_) {
        std::lock_guard<std::mutex> lock(profiler_mutex());
        Profiler& p = profiler();
        ++p.launches[id];
        if (p.on) { a = p.get(); b = p.get(); if (a) cudaEventRecord(a, s); }
    }
    ~Launch() {
        if (a && b) {
            cudaEventRecord(b, s);
            std::lock_guard<std::mutex> lock(profiler_mutex());
            profiler().recs.push_back({id, a, b});
        }
    }
};

}  // namespace ptq
