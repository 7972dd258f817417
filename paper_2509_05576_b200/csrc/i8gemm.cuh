// C += alpha * A * B^T for float64 operands on the 5th-generation tensor cores, to float64 accuracy: the deferred part
// of Eq. 11 (W[:, later] -= E[:, block] U[block, later]) and the other large float64 products of the path.
//
// tcgen05 has no float64 kind, so the product is formed the way the Hessian is (gram.cuh): every row a_i of A and
// every row b_j of B is scaled by a power of two 2^sh so that |x| 2^sh < 2^54, rounded to an integer (exact for the
// entries within 2^-54 of the row maximum, an absolute error of at most 2^-55 of the row maximum for the others) and
// written as seven balanced base-256 digits, most significant first.  Then
//     sum_k va_ik vb_jk = sum_{s,t} 256^(12-s-t) (Da_s Db_t^T)_ij ,
// every Da_s Db_t^T is an exact int8 x int8 -> int32 tensor-core product, pairs with s + t = g share one int32 TMEM
// accumulator, groups g <= 6 are kept (28 products; the dropped ones weigh 2^-56 and less), the groups are combined
// exactly in int64, rounded to float64 and scaled by 2^(48 - sh_i - sh_j).  The error of an entry is of the order of
// 2^-54 max|a_i| max|b_j| per term, i.e. that of a float64 dot product whose terms are of one size; the result is
// deterministic.
//
// The loss 1/2 tr(dW H dW^T) is a sum of terms of very different sizes where the input channels differ in scale, and much
// of it cancels where they are correlated.  Its operands are therefore equilibrated first, dW_ij 2^e_j and H_jk 2^-e_j with
// e_j half the exponent of H_jj (powers of two: nothing is rounded, and dW H does not change), which makes the entries of a
// row of H as alike as those of a correlation matrix, and group 7 is kept as well (34 products).  Relative error of the loss
// against 80-bit sums, 128 x 1152 layers quantized by the oracle, largest of five draws (float64 MMA / these products /
// without either measure): channel scales log-normal with sigma 2: 5e-15 / 1e-15 / 3e-14; four channels 10^4 times larger whose
// weights are zero: 3e-16 / 4e-16 / 4e-13; one component shared by all channels: 7e-13 / 7e-13 / 6e-12.
//
// The deferred part of Eq. 11 adds terms E_ir U_rj to weights of any size, and where the input channels differ in scale
// neither a row of E nor a column of U is of one size.  Where it stands in for float64 MMA steps of 64 columns (deferred_digits
// in api.cu) its operands have eight digits (|x| 2^sh < 2^62) and the groups up to 7 are kept (36 products).  Error of the updated
// weights against extended precision over that of the float64 steps, root mean square / worst column of 2048, behind 1024
// of 3072 columns (eight digits / seven digits / seven digits with group 7): channels of one scale 0.25 / 0.8, 0.4 / 1.7,
// 0.26 / 0.8; channel scales log-normal with sigma 2 0.25 / 0.8, 7.2 / 41, 0.5 / 2.6; those with a small absolute damping
// 0.19 / 0.7, 17 / 88, 1.25 / 4.3; four channels 10^4 times larger, the same damping 0.12 / 0.6, 15 / 66, 0.9 / 3.9.
//
// Kernel: one 128 x 64 output tile per CTA iteration.  A TMA producer warp streams 64-wide K blocks of the seven (eight)
// slices of both operands (SWIZZLE_64B, 2 stages of 84 (96) KB); one thread issues the 20 tcgen05.mma.kind::i8 of a stage
// into seven TMEM accumulators (7 x 64 columns; the loss: 22 into eight; eight digits: 24 into eight); four epilogue warps read them back with tcgen05.ld, combine, hand TMEM
// back (the next tile's products then overlap the rest of the epilogue) and add into C through a shared-memory
// transpose, so that the read-modify-write of C is coalesced.  Every mbarrier wait is bounded.
#pragma once
#include "common.cuh"
#include "dgemm.cuh"
#include "gram.cuh"

namespace ptq {

constexpr int kXSlices = 7;
constexpr int kXMoreSlices = 8;              // the digits of the seven, and one below them
constexpr int kXGroups = 7;                  // groups g = s + t = 0..6
constexpr int kXMoreGroups = 8;              // and 7: all of TMEM (8 x 64 columns)
constexpr int kXTM = 128, kXTN = 64, kXKB = 64;
constexpr int kXStages = 2;
constexpr int kXABytes = kXTM * kXKB;        // 8 KB per slice
constexpr int kXBBytes = kXTN * kXKB;        // 4 KB per slice
__host__ __device__ constexpr int x_stage_bytes(int slices) { return slices * (kXABytes + kXBBytes); }     // 84 KB, 96 KB
static_assert(kXABytes == kGramABytes && kXBBytes == kGramBBytes && kXTN == kGramTN, "tc_slice_products relies on them");
constexpr int kXEpiDoubles = 4 * 32 * 17;    // per epilogue warp: 32 rows x 16 columns (+1 padding)
constexpr int x_smem_bytes(int slices) { return kXStages * x_stage_bytes(slices) + 1024 /*align*/ + 256 /*barriers*/ + kXEpiDoubles * 8; }
static_assert(x_smem_bytes(kXMoreSlices) <= 227 * 1024, "shared memory of a CTA");
constexpr int kXThreads = 192;               // warp 0: TMA, warp 1: MMA + TMEM, warps 2..5: epilogue
constexpr int kXShiftTarget = 54;
constexpr int kXMaxK = 16384;                // 7 * 2^14 * 16384 < 2^31
constexpr int kXMoreMaxK = 8192;             // 8 * 2^14 * 8192 < 2^31

inline size_t i8gemm_plane_bytes(int rows, int k, int slices = kXSlices) {
    return (size_t)slices * (size_t)(cdiv(rows, 128) * 128) * (size_t)(cdiv(k, 128) * 128);
}
inline size_t i8gemm_workspace_bytes(int m, int n, int k) {
    return align_up(i8gemm_plane_bytes(m, k)) + align_up(i8gemm_plane_bytes(n, k)) +
           align_up((size_t)(cdiv(m, 128) * 128) * 12) + align_up((size_t)(cdiv(n, 128) * 128) * 12) + 1024;
}
// Output / K-range modes and the slicing of one operand at a time: see XGemmParams, x_slice_operand, x_product below.

// Integers have no NaN and no infinity.  A row with one (or with a magnitude of 2^900 and more, whose power of two would
// leave the double range) is recorded in the status word, gets zero digits and this shift: the epilogue's factor
// 2^(24 - shift) is then infinite and its sums zero, so every entry formed from the row is 0 * inf = NaN, as the float64
// products have it.
constexpr double kXMaxMagnitude = 8.452712498170644e270;     // 2^900
constexpr int kXShiftBad = -1000;
static_assert(1023 + 24 - kXShiftBad == 2047, "exponent field of an infinity");
// Shift of a row whose largest magnitude is m: |x| 2^sh < 2^54 (0 for an all-zero row); at most `most`.  With eight digits the
// integer is x 2^(sh + 8) and its first seven digits stand for x 2^sh, so the shift is the same for both.
__device__ __forceinline__ int x_row_shift(double m, int most = 900) {
    if (!(m < kXMaxMagnitude)) return kXShiftBad;
    if (!(m > 0.0)) return 0;
    const int sh = kXShiftTarget - (ilogb(m) + 1);
    return sh > most ? most : sh;
}

// Slices of the rows of X [rows x k] (row stride ld): Q[s][row][kk], one CTA per (padded) row.  KEXP: the columns are
// multiplied by 2^(ksign kexp[kk]) first; kexp is 4-byte aligned and may be read up to its next multiple of four.  (One byte
// an exponent: what is read beside a row is an eighth of it.  4608 x 4608: 59 us without, 60 us with exponents.)
template <bool KEXP, int SLICES>
__global__ void __launch_bounds__(256, SLICES == kXSlices ? 6 : 5) x_slice_rows_kernel(const double* __restrict__ X, int rows, int k, int64_t ld,
                                                              int rows_pad, int k_pad, int8_t* __restrict__ Q,
                                                              int32_t* __restrict__ shifts, int32_t* status,
                                                              const int8_t* __restrict__ kexp, int ksign) {
    chained_begin();
    __shared__ unsigned long long smax[256];
    const int row = blockIdx.x;
    const size_t plane = (size_t)rows_pad * k_pad;
    int8_t* q0 = Q + (size_t)row * k_pad;
    if (row >= rows) {
        for (int kk = threadIdx.x * 4; kk < k_pad; kk += 1024)
#pragma unroll
            for (int s = 0; s < SLICES; ++s) *reinterpret_cast<uint32_t*>(q0 + s * plane + kk) = 0u;
        if (threadIdx.x == 0) shifts[row] = 0;
        return;
    }
    const double* x = X + (int64_t)row * ld;
    // the largest magnitude by its bit pattern: non-negative doubles are ordered as integers, a NaN above all of them (a
    // floating-point maximum would drop it)
    unsigned long long m = 0ull;
    for (int kk = threadIdx.x; kk < k; kk += 256) {
        const double v = KEXP ? x[kk] * power_of_two(ksign * (int)kexp[kk]) : x[kk];
        const unsigned long long a = (unsigned long long)__double_as_longlong(fabs(v));
        m = a > m ? a : m;
    }
    smax[threadIdx.x] = m;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w && smax[threadIdx.x + w] > smax[threadIdx.x]) smax[threadIdx.x] = smax[threadIdx.x + w];
        __syncthreads();
    }
    // with an exponent on top: within power_of_two's range
    const int sh = x_row_shift(__longlong_as_double((long long)smax[0]), KEXP ? 850 : 900);
    const bool bad = sh == kXShiftBad;
    if (threadIdx.x == 0) {
        shifts[row] = sh;
        if (bad) report(status, PTQ_ERR_NONFINITE, row, 5);
    }
    const int sh0 = bad ? 0 : sh, kx = bad ? 0 : k;
    for (int kk = threadIdx.x * 4; kk < k_pad; kk += 1024) {
        long long v[4];
        char4 e4 = make_char4(0, 0, 0, 0);
        if (KEXP && kk < k) e4 = *reinterpret_cast<const char4*>(kexp + kk);
        const int e[4] = {e4.x, e4.y, e4.z, e4.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const double xv = kk + u < kx ? x[kk + u] : 0.0;
            v[u] = __double2ll_rn(xv * power_of_two((KEXP ? sh0 + ksign * e[u] : sh0) + 8 * (SLICES - kXSlices)));
        }
        uint32_t packed[SLICES];
        pack_digits4<SLICES>(v, packed);
#pragma unroll
        for (int s = 0; s < SLICES; ++s) *reinterpret_cast<uint32_t*>(q0 + s * plane + kk) = packed[s];
    }
}

// Slices of the COLUMNS of X [k x cols] (row stride ld): Q[s][col][kk] -- the operand B of C += A B^T when the matrix
// at hand is stored as [k][j].  Two passes, both over a grid of (32-column groups) x (256-row chunks of k), so that a
// deep operand is spread over many CTAs: x_colmax_kernel takes the column maxima (reads along rows are coalesced; the
// maxima of the chunks meet by an integer atomic maximum on the bit patterns, which orders non-negative doubles as it
// orders integers and does not depend on the order of arrival); x_slice_cols_kernel reads 32 x 32 tiles row-wise, cuts
// them into digits and writes them out transposed through shared memory.
constexpr int kXColChunk = 256;
__global__ void __launch_bounds__(256) x_colmax_kernel(const double* __restrict__ X, int k, int cols, int64_t ld,
                                                        unsigned long long* __restrict__ colmax) {
    chained_begin();
    __shared__ double smax[8][33];
    const int c0 = blockIdx.x * 32, k0 = blockIdx.y * kXColChunk;
    const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
    const int col = c0 + lane;
    const int k1 = k0 + kXColChunk < k ? k0 + kXColChunk : k;
    double m = 0.0;
    if (col < cols)
        for (int kk = k0 + wy; kk < k1; kk += 8) {
            const double a = fabs(X[(int64_t)kk * ld + col]);
            m = a > m || !(a == a) ? a : m;                   // a NaN sticks
        }
    smax[wy][lane] = m;
    __syncthreads();
    if (wy == 0 && col < cols) {
        double mm = smax[0][lane];
#pragma unroll
        for (int w = 1; w < 8; ++w) mm = (smax[w][lane] > mm || !(smax[w][lane] == smax[w][lane])) ? smax[w][lane] : mm;
        // NaN and infinity have bit patterns above every finite double: they win the maximum as well
        atomicMax(colmax + col, (unsigned long long)__double_as_longlong(mm));
    }
}
__global__ void __launch_bounds__(256) x_slice_cols_kernel(const double* __restrict__ X, int k, int cols, int64_t ld,
                                                            int cols_pad, int k_pad,
                                                            const unsigned long long* __restrict__ colmax,
                                                            int8_t* __restrict__ Q, int32_t* __restrict__ shifts,
                                                            int32_t* status) {
    chained_begin();
    __shared__ uint8_t dig[kXSlices][32][36];          // [slice][column][kk within the tile]
    const int c0 = blockIdx.x * 32, kbeg = blockIdx.y * kXColChunk;
    const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;          // 8 row slices x 32 columns
    const size_t plane = (size_t)cols_pad * k_pad;
    const int col = c0 + lane;
    const double mm = col < cols ? __longlong_as_double((long long)colmax[col]) : 0.0;
    const int sh = x_row_shift(mm);
    const bool bad = sh == kXShiftBad;
    if (blockIdx.y == 0 && wy == 0 && col < cols_pad) {
        shifts[col] = sh;
        if (bad) report(status, PTQ_ERR_NONFINITE, col, 5);
    }
    const double scale = power_of_two(bad ? 0 : sh);
    const int kx = mm > 0.0 && !bad ? k : 0;           // nothing is read of a column of zeros, nor beyond the last column
    const int kend = kbeg + kXColChunk < k_pad ? kbeg + kXColChunk : k_pad;
    for (int k0 = kbeg; k0 < kend; k0 += 32) {
        // thread (wy, lane): rows k0 + wy, + 8, + 16, + 24 of column `col`
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int kk = k0 + wy + 8 * r;
            const double xv = kk < kx ? X[(int64_t)kk * ld + col] : 0.0;
            const unsigned long long d = balanced_digits<kXSlices>(__double2ll_rn(xv * scale));
#pragma unroll
            for (int s = 0; s < kXSlices; ++s) dig[kXSlices - 1 - s][lane][wy + 8 * r] = (uint8_t)(d >> (8 * s));
        }
        __syncthreads();
        // out: for every slice and column, 32 consecutive bytes; thread -> (column = threadIdx / 8, 4 bytes = threadIdx % 8)
        const int oc = threadIdx.x >> 3, ob = (threadIdx.x & 7) * 4;
        if (c0 + oc < cols_pad) {
#pragma unroll
            for (int s = 0; s < kXSlices; ++s)
                *reinterpret_cast<uint32_t*>(Q + s * plane + (size_t)(c0 + oc) * k_pad + k0 + ob) =
                    *reinterpret_cast<const uint32_t*>(&dig[s][oc][ob]);
        }
        __syncthreads();
    }
}

// The same in one pass where the columns are at most kXOnceMaxK long (the panels): a CTA holds eight of them in shared memory,
// so the matrix is read once and there is neither a maximum to be cleared nor a kernel between.  Bound by memory: 8 bytes in
// and 7 out per value instead of 16 and 7; three CTAs per SM, so that one loads while another cuts digits.  A panel of 4608
// columns 34 -> 26 us; 512 x 4608 6967 -> 6843 us, 4096 x 4096 7892 -> 7798.
constexpr int kXOnceMaxK = 1024, kXOnceCols = 8, kXOnceLd = kXOnceCols + 1;       // odd: four rows on are eight banks on
inline size_t x_once_smem_bytes(int k_pad) { return (size_t)k_pad * kXOnceLd * sizeof(double); }
template <int SLICES>
__global__ void __launch_bounds__(256, 3) x_slice_cols_once_kernel(const double* __restrict__ X, int k, int cols, int64_t ld, int cols_pad,
                                                                   int k_pad, int8_t* __restrict__ Q, int32_t* __restrict__ shifts,
                                                                   int32_t* status) {
    chained_begin();
    extern __shared__ __align__(16) double x_once_tile[];            // [k_pad][kXOnceLd]
    __shared__ unsigned long long smax[32][kXOnceCols];
    const int c0 = blockIdx.x * kXOnceCols, tid = threadIdx.x, c = tid & 7;
    const size_t plane = (size_t)cols_pad * k_pad;
    const bool col_in = c0 + c < cols;
    for (int kk = tid >> 3; kk < k_pad; kk += 32) {
        const bool in = col_in && kk < k;
        cp_async8(x_once_tile + kk * kXOnceLd + c, in ? X + (int64_t)kk * ld + c0 + c : X, in);
    }
    cp_async_commit();
    cp_async_wait<0>();
    // the column maxima as bit patterns: non-negative doubles are ordered as integers, a NaN above all of them (every thread
    // takes the values it has copied itself)
    unsigned long long m = 0ull;
    for (int kk = tid >> 3; kk < k_pad; kk += 32) {
        const unsigned long long a = (unsigned long long)__double_as_longlong(fabs(x_once_tile[kk * kXOnceLd + c]));
        m = a > m ? a : m;
    }
    smax[tid >> 3][c] = m;
    __syncthreads();
    for (int w = 16; w > 0; w >>= 1) {
        if ((tid >> 3) < w && smax[(tid >> 3) + w][c] > smax[tid >> 3][c]) smax[tid >> 3][c] = smax[(tid >> 3) + w][c];
        __syncthreads();
    }
    if (tid < kXOnceCols) {
        const int sh = x_row_shift(__longlong_as_double((long long)smax[0][tid]));
        shifts[c0 + tid] = sh;
        if (sh == kXShiftBad) report(status, PTQ_ERR_NONFINITE, c0 + tid, 5);
    }
    // a warp: four columns, eight groups of four consecutive values each, 32 bytes of a slice's row side by side
    const int lane = tid & 31, warp = tid >> 5, oc = (warp & 1) * 4 + (lane & 3);
    const int sh = x_row_shift(__longlong_as_double((long long)smax[0][oc]));
    const bool bad = sh == kXShiftBad;
    const double scale = power_of_two(bad ? 0 : sh + 8 * (SLICES - kXSlices));
    int8_t* q = Q + (size_t)(c0 + oc) * k_pad;
    for (int k0 = (warp >> 1) * 32 + (lane >> 2) * 4; k0 < k_pad; k0 += 128) {
        long long v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = bad ? 0ll : __double2ll_rn(x_once_tile[(k0 + u) * kXOnceLd + oc] * scale);
        uint32_t packed[SLICES];
        pack_digits4<SLICES>(v, packed);
#pragma unroll
        for (int s = 0; s < SLICES; ++s) *reinterpret_cast<uint32_t*>(q + s * plane + k0) = packed[s];
    }
}

// Output modes: what the epilogue does with P = A B^T.
enum { X_OUT_ADD_UPPER = 3,  // C += alpha P on the tiles that touch the upper triangle only (A = B, C symmetric, upper kept)
       X_OUT_ADD = 0,        // C += alpha P
       X_OUT_SYM = 1,        // C = alpha P on the tiles that touch the upper triangle, and C[j][i] = C[i][j] (A = B)
       X_OUT_REDUCE = 2 };   // partials[tile] = alpha * sum_ij P_ij D_ij ; C is not touched
// K ranges per tile (operands known to be zero outside them, or terms accounted for elsewhere).
enum { X_K_ALL = 0,
       X_K_FROM_MAX = 1,     // k >= max(i0, j0): A[i][k] = 0 for k < i and B[j][k] = 0 for k < j (a triangular factor)
       X_K_BEFORE_J = 2,     // k < j0: the column blocks before the tile's own
       X_K_OWN_J = 3 };      // j0 <= k < j0 + 64: the tile's own column block
struct XGemmParams {
    double* C;              // [m x n], row stride ldc
    int64_t ldc;
    int m, n, k_pad;
    double alpha;
    const int32_t* sh_a;    // per row of A
    const int32_t* sh_b;    // per row of B
    int32_t* status;
    int out_mode, k_mode;
    const double* D;        // X_OUT_REDUCE: [m x n], row stride ldd
    int64_t ldd;
    double* partials;       // X_OUT_REDUCE: one per tile (0 for tiles without work)
    double* diag;           // X_OUT_SYM: diag[i] = C[i][i] as well, unless null
};

// K blocks [kb0, kb1) of tile (bi, bj); an empty range or a tile below the diagonal (X_OUT_SYM) has no work at all.
__device__ __forceinline__ bool x_tile_range(const XGemmParams& prm, int bi, int bj, int nkb, int& kb0, int& kb1) {
    const int i0 = bi * kXTM, j0 = bj * kXTN;
    kb0 = 0;
    kb1 = nkb;
    if ((prm.out_mode == X_OUT_SYM || prm.out_mode == X_OUT_ADD_UPPER) && i0 > j0 + kXTN - 1) return false;
    if (prm.k_mode == X_K_FROM_MAX) kb0 = (i0 > j0 ? i0 : j0) / kXKB;
    else if (prm.k_mode == X_K_BEFORE_J) kb1 = j0 / kXKB;
    else if (prm.k_mode == X_K_OWN_J) { kb0 = j0 / kXKB; kb1 = kb0 + 1; }
    if (kb1 > nkb) kb1 = nkb;
    return kb0 < kb1;
}

template <int GROUPS, int SLICES>
__global__ void __launch_bounds__(kXThreads, 1)
i8gemm_kernel(const __grid_constant__ CUtensorMap tmapA, const __grid_constant__ CUtensorMap tmapB, XGemmParams prm) {
    chained_wait();
    constexpr int kStageBytes = x_stage_bytes(SLICES);
    extern __shared__ unsigned char xg_smem_raw[];
    const uint32_t raw = smem_u32(xg_smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    unsigned char* base_ptr = xg_smem_raw + (base - raw);
    uint64_t* bars = reinterpret_cast<uint64_t*>(base_ptr + kXStages * kStageBytes);
    const uint32_t bar0 = base + kXStages * kStageBytes;
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (kXStages + s); };
    const uint32_t acc_full = bar0 + 8u * (2 * kXStages);
    const uint32_t acc_empty = bar0 + 8u * (2 * kXStages + 1);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kXStages + 2);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    double* epi = reinterpret_cast<double*>(base_ptr + kXStages * kStageBytes + 256);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nkb = prm.k_pad / kXKB;
    const int tiles_n = (prm.n + kXTN - 1) / kXTN, tiles_m = (prm.m + kXTM - 1) / kXTM;
    const int num_tiles = tiles_m * tiles_n;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kXStages; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        mbar_init(acc_full, 1);
        mbar_init(acc_empty, 128);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        // ---------------------------------------------------------------- TMA producer
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            int armed[kXStages];
#pragma unroll
            for (int s = 0; s < kXStages; ++s) armed[s] = -1;
            bool ok = true;
            for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
                const int bi = tile / tiles_n, bj = tile - bi * tiles_n;
                int kb0, kb1;
                if (!x_tile_range(prm, bi, bj, nkb, kb0, kb1)) continue;
                for (int kb = kb0; kb < kb1 && ok; ++kb) {
                    ok = mbar_wait_bounded(empty_bar(stage), phase ^ 1u, abort_flag);
                    if (!ok) break;
                    const uint32_t sbase = base + stage * kStageBytes;
                    mbar_arrive_expect_tx(full_bar(stage), kStageBytes);
                    armed[stage] = (int)phase;
#pragma unroll
                    for (int s = 0; s < SLICES; ++s) {
                        tma_load_3d(sbase + s * kXABytes, &tmapA, kb * kXKB, bi * kXTM, s, full_bar(stage));
                        tma_load_3d(sbase + SLICES * kXABytes + s * kXBBytes, &tmapB, kb * kXKB, bj * kXTN, s,
                                    full_bar(stage));
                    }
                    if (++stage == kXStages) { stage = 0; phase ^= 1u; }
                }
            }
            if (!ok) {
                // drain: wait (bounded) until the copies already issued have landed
                for (int s = 0; s < kXStages; ++s)
                    if (armed[s] >= 0) {
                        const long long t0 = clock64();
                        while (!mbar_try_wait(full_bar(s), (uint32_t)armed[s]) && clock64() - t0 < 200000000LL) {}
                    }
            }
        }
    } else if (warp == 1) {
        // ---------------------------------------------------------------- MMA issuer
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0, acc_phase = 0;
            bool ok = true;
            for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
                const int bi = tile / tiles_n, bj = tile - bi * tiles_n;
                int kb0, kb1;
                if (!x_tile_range(prm, bi, bj, nkb, kb0, kb1)) continue;
                ok = mbar_wait_bounded(acc_empty, acc_phase ^ 1u, abort_flag);   // epilogue has drained TMEM
                if (!ok) break;
                tc_fence_after();
                for (int kb = kb0; kb < kb1 && ok; ++kb) {
                    ok = mbar_wait_bounded(full_bar(stage), phase, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t sb = kDescLo + ((base + stage * kStageBytes) >> 4);
                    const uint32_t first = kb > kb0 ? 1u : 0u;    // the first product of a group overwrites
#pragma unroll
                    for (int ks = 0; ks < kXKB / 32; ++ks)
                        tc_slice_products<GROUPS>(tmem_base, sb + ks * 2, sb + ks * 2 + ((SLICES * kXABytes) >> 4),
                                                  ks > 0 ? 1u : first, std::make_integer_sequence<int, SLICES>());
                    tc_commit(empty_bar(stage));     // the stage may be refilled once these MMAs have read it
                    if (++stage == kXStages) { stage = 0; phase ^= 1u; }
                }
                if (ok) tc_commit(acc_full);         // accumulators complete
                acc_phase ^= 1u;
            }
        }
    } else {
        // ---------------------------------------------------------------- epilogue (warps 2..5)
        const int quarter = warp & 3;                 // TMEM lanes this warp may read
        const int r_in_tile = quarter * 32 + lane;
        double* my = epi + quarter * 32 * 17;
        uint32_t acc_phase = 0;
        bool ok = true;
        for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
            const int bi = tile / tiles_n, bj = tile - bi * tiles_n;
            int kb0, kb1;
            if (!x_tile_range(prm, bi, bj, nkb, kb0, kb1)) {
                if (prm.out_mode == X_OUT_REDUCE && threadIdx.x == 64) prm.partials[tile] = 0.0;
                continue;
            }
            ok = mbar_wait_bounded(acc_full, acc_phase, abort_flag);
            if (!ok) break;
            tc_fence_after();
            const int row = bi * kXTM + r_in_tile;
            // 1. drain: v = hi 2^32 + lo with lo = 2^-8 G7 + G6 + 2^8 G5 + 2^16 G4 + 2^24 G3, hi = G2 + 2^8 G1 + 2^16 G0,
            //    both exact (lo times 2^8 where there is a group 7: below 2^63, as |G3| < 4 2^14 kXMaxK)
            double v[kXTN];
#pragma unroll
            for (int ch = 0; ch < kXTN / 16; ++ch) {
                long long lo[16], hi[16];
                uint32_t r[16];
                const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + ch * 16;
#pragma unroll
                for (int g = GROUPS - 1; g >= 3; --g) {
                    tc_ld16(taddr + g * kXTN, r); tc_wait_ld();
#pragma unroll
                    for (int c = 0; c < 16; ++c)
                        lo[c] = (g == GROUPS - 1 ? 0ll : lo[c]) + ((long long)(int)r[c] << (8 * (GROUPS - 1 - g)));
                }
                tc_ld16(taddr + 2 * kXTN, r); tc_wait_ld();
#pragma unroll
                for (int c = 0; c < 16; ++c) hi[c] = (long long)(int)r[c];
                tc_ld16(taddr + 1 * kXTN, r); tc_wait_ld();
#pragma unroll
                for (int c = 0; c < 16; ++c) hi[c] += (long long)(int)r[c] << 8;
                tc_ld16(taddr + 0 * kXTN, r); tc_wait_ld();
#pragma unroll
                for (int c = 0; c < 16; ++c) hi[c] += (long long)(int)r[c] << 16;
#pragma unroll
                for (int c = 0; c < 16; ++c) 
                    v[ch * 16 + c] = fma((double)hi[c], 4294967296.0,
                                         GROUPS == kXGroups ? (double)lo[c] : (double)lo[c] * 0.00390625);
            }
            tc_fence_before();
            mbar_arrive(acc_empty);
            acc_phase ^= 1u;
            // 2. C += alpha v 2^(48 - sh_i - sh_j), sixteen columns at a time through a transpose in shared memory:
            //    lane r writes its row's sixteen values, then half a warp reads one row's sixteen columns (128 bytes)
            const int sh_i = row < prm.m ? prm.sh_a[row] : 0;
            const double fi = prm.alpha * __longlong_as_double((long long)(1023 + 24 - sh_i) << 52);
            const int orow = lane >> 4, ocol = lane & 15;
            if (prm.out_mode == X_OUT_REDUCE) {
                // sum_ij P_ij D_ij over the tile, in a fixed order: along the row in this lane, then over the lanes of
                // the warp by a shuffle tree, then over the four warps in ascending order
                double s = 0.0;
                if (row < prm.m) {
                    const double* drow = prm.D + (int64_t)row * prm.ldd + bj * kXTN;
#pragma unroll
                    for (int c = 0; c < kXTN; ++c) {
                        const int col = bj * kXTN + c;
                        if (col < prm.n) {
                            const double fj = __longlong_as_double((long long)(1023 + 24 - prm.sh_b[col]) << 52);
                            s = fma((v[c] * fi) * fj, drow[c], s);
                        }
                    }
                }
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
                if (lane == 0) my[0] = s;
                asm volatile("bar.sync 1, 128;" ::: "memory");           // the four epilogue warps
                if (quarter == 0 && lane == 0)
                    prm.partials[tile] = ((epi[0] + epi[32 * 17]) + epi[2 * 32 * 17]) + epi[3 * 32 * 17];
                asm volatile("bar.sync 1, 128;" ::: "memory");
                continue;
            }
            if (prm.out_mode == X_OUT_SYM) {
                // mirrored entries C[col][row]: consecutive lanes are consecutive rows, i.e. contiguous there
                if (row < prm.m) {
#pragma unroll
                    for (int c = 0; c < kXTN; ++c) {
                        const int col = bj * kXTN + c;
                        if (col < prm.n) {
                            const double fj = __longlong_as_double((long long)(1023 + 24 - prm.sh_b[col]) << 52);
                            prm.C[(int64_t)col * prm.ldc + row] = (v[c] * fi) * fj;
                            if (col == row && prm.diag != nullptr) prm.diag[row] = (v[c] * fi) * fj;
                        }
                    }
                }
            }
#pragma unroll
            for (int ch = 0; ch < kXTN / 16; ++ch) {
                const int col0 = bj * kXTN + ch * 16;
#pragma unroll
                for (int c = 0; c < 16; ++c) my[lane * 17 + c] = v[ch * 16 + c] * fi;
                __syncwarp();
                const int col = col0 + ocol;
                if (col < prm.n) {
                    const double fj = __longlong_as_double((long long)(1023 + 24 - prm.sh_b[col]) << 52);
                    double* dst0 = prm.C + (int64_t)(bi * kXTM + quarter * 32 + orow) * prm.ldc + col;
                    const int rows_left = prm.m - (bi * kXTM + quarter * 32 + orow);      // rows rr with rr < rows_left exist
                    // all sixteen old values are requested before the first is used: one memory latency per chunk
                    double oldv[16];
#pragma unroll
                    for (int q = 0; q < 16; ++q)
                        oldv[q] = (prm.out_mode != X_OUT_SYM && 2 * q < rows_left)
                                      ? __ldcg(dst0 + (int64_t)(2 * q) * prm.ldc) : 0.0;
#pragma unroll
                    for (int q = 0; q < 16; ++q)
                        if (2 * q < rows_left)
                            __stcg(dst0 + (int64_t)(2 * q) * prm.ldc, oldv[q] + my[(2 * q + orow) * 17 + ocol] * fj);
                }
                __syncwarp();
            }
        }
    }

    // ---------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
    if (threadIdx.x == 0 && *abort_flag) report(prm.status, PTQ_ERR_TIMEOUT, blockIdx.x, 4);
}

// ------------------------------------------------------------------------------------------------------------
// Host side
// ------------------------------------------------------------------------------------------------------------
inline int x_make_map(CUtensorMap* m, int8_t* Q, int rows_pad, int k_pad, int slices, int box_rows) {
    EncodeTiledFn enc = get_encode_tiled();
    if (!enc) return PTQ_ERR_CUDA;
    const cuuint64_t dims[3] = {(cuuint64_t)k_pad, (cuuint64_t)rows_pad, (cuuint64_t)slices};
    const cuuint64_t strides[2] = {(cuuint64_t)k_pad, (cuuint64_t)rows_pad * (cuuint64_t)k_pad};
    const cuuint32_t box[3] = {(cuuint32_t)kXKB, (cuuint32_t)box_rows, 1u};
    const cuuint32_t estr[3] = {1u, 1u, 1u};
    const CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, Q, dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? PTQ_OK : PTQ_ERR_CUDA;
}

// Slices of one operand in the workspace: planes [slices][rows_pad][k_pad] and the per-row shifts.
struct XOperand {
    int8_t* Q;
    int32_t* sh;
    int rows, k, slices;
};
inline size_t x_operand_bytes(int rows, int k, int slices = kXSlices) {
    return align_up(i8gemm_plane_bytes(rows, k, slices)) + align_up((size_t)(cdiv(rows, 128) * 128) * sizeof(int32_t)) +
           align_up((size_t)(cdiv(rows, 128) * 128) * sizeof(unsigned long long));
}
inline int x_attributes(DeviceState* dev) {
    return ensure_smem_attr(dev, SA_XGEMM, [] {
        cudaError_t e = cudaSuccess;
        auto smem = [&](const void* kernel, size_t bytes) {
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        };
        smem((const void*)i8gemm_kernel<kXGroups, kXSlices>, x_smem_bytes(kXSlices));
        smem((const void*)i8gemm_kernel<kXMoreGroups, kXSlices>, x_smem_bytes(kXSlices));
        smem((const void*)i8gemm_kernel<kXMoreGroups, kXMoreSlices>, x_smem_bytes(kXMoreSlices));
        smem((const void*)x_slice_cols_once_kernel<kXSlices>, x_once_smem_bytes(kXOnceMaxK));
        smem((const void*)x_slice_cols_once_kernel<kXMoreSlices>, x_once_smem_bytes(kXOnceMaxK));
        return e;
    });
}
// X is [rows x k] (transposed = 0, row stride ld) or [k x rows] (transposed = 1: the operand's rows are X's columns).
// kexp (with transposed = 0): column kk is multiplied by 2^(ksign kexp[kk]), see x_slice_rows_kernel.  slices: digits per value,
// seven, or eight without kexp and with at most kXOnceMaxK columns' length where transposed (x_product refuses what is neither).
inline XOperand x_slice_operand(Carver& cv, const double* X, int64_t ld, int transposed, int rows, int k, int32_t* status,
                                cudaStream_t stream, const int8_t* kexp = nullptr, int ksign = 1, int slices = kXSlices) {
    const int rows_pad = cdiv(rows, 128) * 128, k_pad = cdiv(k, 128) * 128;
    XOperand op;
    op.Q = cv.take<int8_t>(i8gemm_plane_bytes(rows, k, slices));
    op.sh = cv.take<int32_t>(rows_pad);
    unsigned long long* colmax = cv.take<unsigned long long>(rows_pad);
    op.rows = rows; op.k = k; op.slices = slices;
    DeviceState* dev = nullptr;
    if (current_device_state(&dev) == PTQ_OK) x_attributes(dev);          // an error shows at the launch
    Launch l(K_X_SLICE, stream);
    if (transposed && k <= kXOnceMaxK) {
        launch_chained(slices == kXMoreSlices ? x_slice_cols_once_kernel<kXMoreSlices> : x_slice_cols_once_kernel<kXSlices>,
                       rows_pad / kXOnceCols, 256, x_once_smem_bytes(k_pad), stream, X, k, rows, ld, rows_pad, k_pad, op.Q,
                       op.sh, status);
    } else if (transposed && slices == kXSlices) {
        cudaMemsetAsync(colmax, 0, (size_t)rows_pad * sizeof(unsigned long long), stream);
        launch_chained(x_colmax_kernel, dim3(rows_pad / 32, cdiv(k, kXColChunk)), 256, 0, stream, X, k, rows, ld, colmax);
        launch_chained(x_slice_cols_kernel, dim3(rows_pad / 32, cdiv(k_pad, kXColChunk)), 256, 0, stream, X, k, rows, ld,
                       rows_pad, k_pad, colmax, op.Q, op.sh, status);
    } else if (!transposed && kexp && slices == kXSlices) {
        launch_chained(x_slice_rows_kernel<true, kXSlices>, rows_pad, 256, 0, stream, X, rows, k, ld, rows_pad, k_pad, op.Q,
                       op.sh, status, kexp, ksign);
    } else if (!transposed && !kexp) {
        launch_chained(slices == kXMoreSlices ? x_slice_rows_kernel<false, kXMoreSlices> : x_slice_rows_kernel<false, kXSlices>,
                       rows_pad, 256, 0, stream, X, rows, k, ld, rows_pad, k_pad, op.Q, op.sh, status, nullptr, 1);
    } else {
        op.slices = 0;
    }
    return op;
}

// The product of two sliced operands (A: m rows, B: n rows, same k <= kXMaxK) in the given output / K-range modes, of the first
// `digits` digits of both: seven (X_OUT_REDUCE: with group 7), or eight (k <= kXMoreMaxK).
inline int x_product(const XOperand& a, const XOperand& b, XGemmParams prm, cudaStream_t stream, int digits = kXSlices) {
    if (a.k != b.k || a.k > kXMaxK || digits > a.slices || digits > b.slices) return PTQ_ERR_UNSUPPORTED;
    if (digits == kXMoreSlices && (a.k > kXMoreMaxK || prm.out_mode == X_OUT_REDUCE)) return PTQ_ERR_UNSUPPORTED;
    DeviceState* dev = nullptr;
    int st = current_device_state(&dev);
    if (st) return st;
    st = x_attributes(dev);
    if (st) return st;
    const int k_pad = cdiv(a.k, 128) * 128;
    CUtensorMap mapA, mapB;
    st = x_make_map(&mapA, a.Q, cdiv(a.rows, 128) * 128, k_pad, a.slices, kXTM);
    if (st) return st;
    st = x_make_map(&mapB, b.Q, cdiv(b.rows, 128) * 128, k_pad, b.slices, kXTN);
    if (st) return st;
    prm.m = a.rows; prm.n = b.rows; prm.k_pad = k_pad;
    prm.sh_a = a.sh; prm.sh_b = b.sh;
    const int tiles = cdiv(prm.m, kXTM) * cdiv(prm.n, kXTN);
    const int grid = tiles < dev->sms ? tiles : dev->sms;
    {
        Launch l(K_X_GEMM, stream);
        auto kernel = digits == kXMoreSlices ? i8gemm_kernel<kXMoreGroups, kXMoreSlices>
                                             : (prm.out_mode == X_OUT_REDUCE ? i8gemm_kernel<kXMoreGroups, kXSlices>
                                                                             : i8gemm_kernel<kXGroups, kXSlices>);
        launch_chained(kernel, grid, kXThreads, (size_t)x_smem_bytes(digits), stream, mapA, mapB, prm);
    }
    return launch_status();
}
inline int x_num_tiles(int m, int n) { return cdiv(m, kXTM) * cdiv(n, kXTN); }

// C[m x n] += alpha * A B^T with A [m x k] (rows contiguous in k, stride lda) and B given either as [n x k]
// (b_is_kn = 0, stride ldb) or as [k x n] (b_is_kn = 1: B^T is what is stored, stride ldb).  k <= kXMaxK.
inline int i8gemm_nt(double* C, int64_t ldc, const double* A, int64_t lda, const double* B, int64_t ldb, int b_is_kn,
                     int m, int n, int k, double alpha, void* ws, int32_t* status, cudaStream_t stream) {
    if (m <= 0 || n <= 0 || k <= 0) return PTQ_OK;
    if (k > kXMaxK) return PTQ_ERR_UNSUPPORTED;
    Carver cv(ws);
    const XOperand a = x_slice_operand(cv, A, lda, 0, m, k, status, stream);
    const XOperand b = x_slice_operand(cv, B, ldb, b_is_kn, n, k, status, stream);
    XGemmParams prm{};
    prm.C = C; prm.ldc = ldc; prm.alpha = alpha; prm.status = status;
    prm.out_mode = X_OUT_ADD; prm.k_mode = X_K_ALL;
    return x_product(a, b, prm, stream);
}

}  // namespace ptq
