// Float64 blocked factorisation pieces: A = U^T U (upper Cholesky, in place, row-major), the inverse of the
// factor W = U^-T from the same sweep, and Hinv = W^T W.  Sec. 5 item 1 of the paper (Cholesky, then the inverse of
// the factor); the same Cholesky applied to the permuted inverse Hessian is the blocked form of Eq. 12:
// step p of a right-looking Cholesky subtracts (row p)^T (row p) / pivot from the trailing matrix.
#pragma once
#include "common.cuh"
#include "dgemm.cuh"
#include <type_traits>
#include <utility>

namespace ptq {

// lambda = damp * mean(diag H) or damp; one CTA, fixed summation order.  Flags non-finite diagonals.
__global__ void __launch_bounds__(256) lambda_kernel(const double* __restrict__ H, int n, int mode, double damp,
                                                      double* __restrict__ lambda_out, int32_t* status) {
    chained_begin();
    __shared__ double red[256];
    double s = 0.0;
    bool bad = false;
    for (int j = threadIdx.x; j < n; j += 256) {
        const double d = H[(int64_t)j * n + j];
        if (!isfinite(d)) bad = true;
        s += d;
    }
    if (bad) report(status, PTQ_ERR_NONFINITE, -1);
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *lambda_out = mode == PTQ_DAMP_REL_MEAN_DIAG ? damp * (red[0] / (double)n) : damp;
}

// A = H + lambda I, from each row's 64-column diagonal tile on (the factorisation reads the upper triangle only, whole
// tiles on the diagonal), and V = 0 (where the inverse of the factor will be built); one grid row per matrix row.  Also
// clears the factorisation's grid barrier.  Up to four columns a thread: with one, the CTAs come and go faster than the memory
// (27 -> 17 us at 2304 columns, 556 -> 305 at 11008).
__global__ void damp_copy_kernel(const double* __restrict__ H, double* __restrict__ A, double* __restrict__ V, int n,
                                 const double* __restrict__ lambda, unsigned* __restrict__ bar) {
    chained_begin();
    const int i = blockIdx.y;
    const double lam = *lambda;
    const int64_t row = (int64_t)i * n;
    const int first = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
    if (i == 0 && first < 2) bar[first] = 0u;
    for (int j = (i & ~(kNB - 1)) + first; j < n; j += step) A[row + j] = H[row + j] + (j == i ? lam : 0.0);
    for (int j = first; j < n; j += step) V[row + j] = 0.0;
}

// ------------------------------------------------------------------------------------------------------------
// Blocked upper Cholesky A = U^T U as ONE persistent cooperative kernel (one CTA per SM, 512 threads).
// For each 64-row block k:
//   strip phase    every CTA that owns a panel chunk of 8 to 40 columns factorises the 64 x 64 diagonal block itself (all
//                  CTAs do the same arithmetic on it, so no broadcast is needed) and applies the same row
//                  operations to its chunk: the unblocked algorithm on a strip of 64 rows, eight pivots at a time
//                  (see chol_strip).  That replaces "factor the block, then solve the panel against it".
//   trailing phase A[i][j] -= U[k][i]^T U[k][j] on the upper 64 x 64 tiles, float64 tensor-core MMA, operands
//                  double-buffered through shared memory with cp.async.
// When the next block row has few strip work items, a few CTAs update and factorise it (look-ahead) while the others
// are still applying the current one to the rows below, which takes the strip off the critical path.
// The phases are separated by a grid-wide barrier whose wait is bounded: when it expires the CTA records
// PTQ_ERR_TIMEOUT, raises the abort word and leaves; the other CTAs see the abort word and leave too.
// A pivot that is not positive, normal and finite is reported (PTQ_ERR_NOT_SPD, pivot index) and replaced by 1.
// ------------------------------------------------------------------------------------------------------------
constexpr int kCholThreads = 512;
constexpr int kCholLd = kNB + 4;                               // operand row stride (68 = 4 mod 16: conflict-free)
constexpr int kCholBlock = kNB * kCholLd;                      // doubles of a 64 x 64 operand block
constexpr int kCholOpndDoubles = 2 /*operands*/ * 2 /*slots*/ * kCholBlock;
constexpr int kCholMaxBlockRows = 1024;                         // 65535 columns
constexpr unsigned kStripsOnly = 8u;
constexpr size_t kCholSmemBytes = sizeof(double) * kCholOpndDoubles + 16 + kCholMaxBlockRows * sizeof(unsigned);

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void red_release_add_u32(unsigned* p, unsigned v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// bar[0]: arrival counter (monotonic, zero at launch), bar[1]: abort word.  Returns false when the CTA must leave.
// spin_limit: SM clock cycles after which the wait gives up.
// One thread arrives with a release and waits with an acquire; with the block's own barriers on both sides they order what
// every thread of the grid wrote before against what every thread reads after.  Full fences around a plain atomic instead
// cost about 600 clocks per barrier: both factorisations at 1152 columns 248 + 242 -> 242 + 236 us, at 2304 662 + 535 ->
// 648 + 523.
__device__ __forceinline__ bool grid_barrier(unsigned* bar, unsigned target, int* s_flag, long long spin_limit) {
    __syncthreads();
    if (threadIdx.x == 0) {
        red_release_add_u32(&bar[0], 1u);
        const long long t0 = clock64();
        int ok = 1;
        unsigned it = 0;
        while (ld_acquire_u32(&bar[0]) < target) {
            if ((++it & 63u) == 0u) {
                if (ld_acquire_u32(&bar[1]) != 0u) { ok = 0; break; }
                if (clock64() - t0 > spin_limit) { atomicExch(&bar[1], 1u); ok = 0; break; }
            }
        }
        *s_flag = ok;
    }
    __syncthreads();
    return *s_flag != 0;
}

__device__ __forceinline__ void cp_async16_cg(void* smem_dst, const void* gsrc, bool valid) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_dst);
    const int sz = valid ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(gsrc), "r"(sz) : "memory");
}

// -x by its sign bit: an arithmetic negation would queue for the float64 pipe behind the MMAs it is an operand of.
__device__ __forceinline__ double flip_sign(double x) {
    return __hiloint2double(__double2hiint(x) ^ (int)0x80000000, __double2loint(x));
}

// Loads the 64 x ncols block A[r0 .. r0+63][c0 .. c0+ncols-1] into dst[64][kCholLd], ncols = 1 << lg in {16, 32, 64};
// entries beyond n are zero.  Every one of the NT threads (tid = 0 .. NT - 1) copies a fixed column (pair) of successive row
// groups, so a block that lies inside the matrix needs one pointer increment per copy and no bounds test.
template <int NT>
__device__ __forceinline__ void chol_load_block(double* dst, const double* __restrict__ A, int64_t ld, int n, int r0,
                                                int c0, int lg, int vec16, int tid) {
    const bool interior = r0 + kNB <= n && c0 + (1 << lg) <= n;
    if (vec16) {
        const int sh = lg - 1;                           // pairs per row = 1 << sh
        const int c = (tid & ((1 << sh) - 1)) * 2;
        const int rstep = NT >> sh;
        int r = tid >> sh;
        const double* src = A + (int64_t)(r0 + r) * ld + c0 + c;
        double* d = dst + r * kCholLd + c;
        if (interior) {
            for (; r < kNB; r += rstep, src += (int64_t)rstep * ld, d += rstep * kCholLd) cp_async16_cg(d, src, true);
        } else {
            for (; r < kNB; r += rstep, src += (int64_t)rstep * ld, d += rstep * kCholLd) {
                const bool ok = r0 + r < n && c0 + c < n;  // n is even on this path: a pair never straddles n
                cp_async16_cg(d, ok ? src : A, ok);
            }
        }
    } else {
        const int c = tid & ((1 << lg) - 1);
        const int rstep = NT >> lg;
        int r = tid >> lg;
        const double* src = A + (int64_t)(r0 + r) * ld + c0 + c;
        double* d = dst + r * kCholLd + c;
        for (; r < kNB; r += rstep, src += (int64_t)rstep * ld, d += rstep * kCholLd) {
            const bool ok = interior || (r0 + r < n && c0 + c < n);
            cp_async8(d, ok ? src : A, ok);
        }
    }
}

// ------------------------------------------------------------------------------------------------------------
// Strip factorisation: the strip [diagonal block | 8 pg panel columns], pg = 1, 2, 3 or 5, is held in registers as 8 x 8 MMA
// accumulator fragments, eight strip columns (one column group, all 64 rows) per warp.  Pivots are taken eight at a time.  For pivot
// block b:
//   1. warp 0 factorises the 8 x 8 diagonal mini-block M = U_M^T U_M (all of M in every lane, so the serial chain of
//      eight pivots has no data exchange in it) and carries the identity along to obtain W = U_M^-T;
//   2. it makes the next mini-block itself, M' = T - (W R)^T (W R), from what the owner of those columns has put out
//      before: the rows R of this pivot block and T, the next diagonal tile without this pivot block's update;
//   3. meanwhile every other warp forms the new rows U[8 b .. 8 b + 7][own columns] = W R and, when all of them are out,
//      subtracts them from its rows further down, A[i][c] -= U[p][i] U[p][c], by MMA, and brings the rows of the next
//      pivot block up to date with the block row above (look-ahead).
// Named barriers, by the parity of b: 1 / 2 (owner, warp 0) hand over R and T, 3 / 4 (all) hand out W; 5 (all but warp 0)
// makes the new rows visible.  Owners only arrive at 1 / 2 and warp 0 only arrives at 3 / 4, so warp 0 may be one pivot
// block ahead of or behind the other warps, hence two of each.  It is never two ahead: R and T of block b + 1 leave their
// owner after the barriers 3 / 4 and 5 of block b; nor two behind: they wait for it at 3 / 4.
//
// What bounds a strip: scalar float64 instructions queue behind the float64 MMAs of their scheduler (measured: 9 clocks per
// dependent FMA alone, 137 next to one warp that streams MMAs on the same scheduler, 9 again when the MMAs are on the other
// three).  So warp 0 has its scheduler to itself: warps 4, 8 and 12 take no part in a strip, and the updates are dealt to the
// other three schedulers.  With 40 panel columns (twelve warps with one column group each) they have 1800 MMAs, 9.8 k clocks at
// the full rate, and between two hand-outs of W their own sequence (new rows, barrier, update, look-ahead) takes longer than
// warp 0's.  Narrower strips have fewer (1400 with 24 columns, 1200 with 16, 1000 with 8), but more CTAs factorise the
// diagonal block, so the width is chosen per block row, by how much trailing work waits (chol_coop_kernel).
// ------------------------------------------------------------------------------------------------------------
constexpr int kStripMaxPanel = 40;                                       // most panel columns of a strip
constexpr int kStripLd = kNB + kStripMaxPanel + 12;                      // row stride of the 8-row panels (116 = 4 mod 16)
// Column groups (0 .. 7 diagonal, from 8 on panel; 15: the warp takes no part) of the sixteen warps, four bits a warp.  Warps
// w, w + 4, w + 8 and w + 12 share a scheduler: scheduler 0 holds the chain (group 0) alone, the others about equal shares of
// the MMAs (a panel group 200, a diagonal group g 38 to 200).
__device__ __forceinline__ unsigned long long strip_warps(int pg) {
    return pg == 5 ? 0x231F645F7B9FCA80ull : (pg == 3 ? 0xAFFF142F398F5670ull : (pg == 2 ? 0x2FFF31FF498F5670ull : 0x1FFF2FFF345F6780ull));
}
// What a strip counts for when the trailing tiles are dealt, in eighths of a tile: with 40 panel columns, with fewer.  (Both
// factorisations of a layer with 24 / 32 / 40 for the former: 2048 columns 1030 / 1007 / 1016 us, 2304 1273 / 1228 / 1241.)
constexpr int kStripCost = 32, kNarrowStripCost = 28;
// Narrow strips are taken where the trailing tiles are at most this many eighths of a tile for every CTA without a strip.
// Both factorisations with 12 / 20 / 28: 1600 columns 328 + 307 / 323 + 304 / 344 + 310 us, 2304 663 + 506 / 661 + 503 /
// 666 + 508, no difference up to 1152.
constexpr int kNarrowStripWork = 20;
constexpr int kStripSmemDoubles = 2 * 8 * kStripLd + 64 /*M*/ + 64 /*W R*/ + 2 * 64 /*W*/ + 2 * 2 * 64 /*R, T*/;
static_assert(kStripSmemDoubles + 2 * kCholBlock <= kCholOpndDoubles,
              "the strip panels and the look-ahead operands alias the trailing-phase operand buffers");

template <int ID>
__device__ __forceinline__ void named_bar_sync(int count) { asm volatile("bar.sync %0, %1;" ::"n"(ID), "r"(count) : "memory"); }
template <int ID>
__device__ __forceinline__ void named_bar_arrive(int count) { asm volatile("bar.arrive %0, %1;" ::"n"(ID), "r"(count) : "memory"); }

struct StripSmem {
    double* R;       // [8][kStripLd] rows of the pivot block (every warp reads back its own columns only)
    double* U;       // [8][kStripLd] new rows
    double* M;       // [8][8] mini-block (warp 0 only)
    double* V;       // [8][8] W R of the next eight columns (warp 0 only)
    double* W;       // [2][8][8] by parity of the pivot block: a warp may read W late, while warp 0 is in its next chain
    double* X;       // [2][2][8][8] by the same parity: R and T of the next eight columns
    __device__ __forceinline__ explicit StripSmem(double* p)
        : R(p), U(R + 8 * kStripLd), M(U + 8 * kStripLd), V(M + 64), W(V + 64), X(W + 128) {}
};

// acc[r] -= U[:, 8 r .. 8 r + 7]^T U[:, own columns] for the fragment rows R0 <= r < R1 (U: the eight rows in Ubuf).
template <int R0, int R1>
__device__ __forceinline__ void chol_strip_update(double (&acc)[8][2], const double* Ubuf, int grp, int lq, int lr) {
    if constexpr (R0 < R1) {
        const double b0 = Ubuf[lr * kStripLd + 8 * grp + lq], b1 = Ubuf[(4 + lr) * kStripLd + 8 * grp + lq];
#pragma unroll
        for (int r = R0; r < R1; ++r) {
            if (grp < 8 && r > grp) continue;                            // entirely below the diagonal: never used
            dmma_884(acc[r][0], acc[r][1], flip_sign(Ubuf[lr * kStripLd + 8 * r + lq]), b0);
            dmma_884(acc[r][0], acc[r][1], flip_sign(Ubuf[(4 + lr) * kStripLd + 8 * r + lq]), b1);
        }
    }
}

// Look-ahead update of fragment row RB of this warp's strip columns with the block row above (see chol_strip):
//     acc[RB] -= ua[:, 8 RB .. 8 RB + 7]^T bsrc[:, own 8 columns]        (ua, bsrc: 64 rows in shared memory)
// Applied one fragment row at a time, shortly before the row is needed, by the warps that wait for warp 0's chain.
template <int RB>
__device__ __forceinline__ void chol_strip_lookahead(double (&acc)[8][2], const double* ua, const double* bsrc, int grp,
                                                     int lq, int lr) {
    if (grp < 8 && RB > grp) return;            // fragments that lie entirely below the diagonal are never used
    // summed apart and subtracted once: added one by one to the old value they would be rounded to its size sixteen times.
    // Two sums, because an MMA waits for the one before on the same accumulator (both factorisations at 1152 columns: 228 +
    // 217 -> 220 + 209 us; the error of the inverse becomes 1 to 8 % smaller).
    double p0 = 0.0, p1 = 0.0, q0 = 0.0, q1 = 0.0;
#pragma unroll 4
    for (int kk = 0; kk < kNB; kk += 8) {
        dmma_884(p0, p1, ua[(kk + lr) * kCholLd + 8 * RB + lq], bsrc[(kk + lr) * kCholLd + lq]);
        dmma_884(q0, q1, ua[(kk + 4 + lr) * kCholLd + 8 * RB + lq], bsrc[(kk + 4 + lr) * kCholLd + lq]);
    }
    acc[RB][0] -= p0 + q0;
    acc[RB][1] -= p1 + q1;
}

// Step 1 above.  mb: the mini-block M (row-major, 8 x 8, upper part); leaves W in Wbuf.  Returns the first pivot that is not
// accepted (it is replaced by 1) or -1.  This is the general form; chol_chain8 comes here when a pivot is not accepted.
__device__ __noinline__ int chol_chain8_general(const double* mb, double* Wbuf, int lane) {
    double m[8][8];
#pragma unroll
    for (int p = 0; p < 8; ++p)
#pragma unroll
        for (int j = p; j < 8; ++j) m[p][j] = mb[p * 8 + j];
    // lane j carries column j of the identity along, which becomes column j of W = U_M^-T
    const int jc = lane & 7;
    double x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = i == jc ? 1.0 : 0.0;
    int bad = -1;
#pragma unroll
    for (int p = 0; p < 8; ++p) {
        // A bad pivot is replaced by 1 and remembered; the report is made after the chain, so that the eight steps
        // stay one straight line of code.
        const double d0 = m[p][p];
        const bool ok = d0 >= kMinPivot && d0 < kMaxPivot;
        bad = (!ok && bad < 0) ? p : bad;
        const double d = ok ? d0 : 1.0;
        const double inv = pivot_reciprocal(d);            // what the chain waits for
        const double rs = pivot_rsqrt(d);                  // beside the chain
        const double tx = x[p] * inv;
        x[p] *= rs;
#pragma unroll
        for (int i = p + 1; i < 8; ++i) {
            const double f = m[p][i] * inv;
#pragma unroll
            for (int j = i; j < 8; ++j) m[i][j] = fma(-f, m[p][j], m[i][j]);
            x[i] = fma(-m[p][i], tx, x[i]);
        }
    }
    if (lane < 8) {
#pragma unroll
        for (int p = 0; p < 8; ++p) Wbuf[p * 8 + lane] = x[p];    // W[p][j] = (U_M^-T)[p][j]
    }
    return bad;
}

// The same for accepted pivots.  One warp issues a float64 instruction every four clocks or so, and that is what a chain takes,
// so only what the next pivot needs is done by every lane: the elimination of the mini-block and of a column of the identity.
// The square roots, the scaling of the rows of W and the tests of the pivots are dealt to the four groups of eight lanes,
// which all hold the same columns: group q takes the rows 2 q and 2 q + 1.  861 -> 758 clocks
// by itself, 1210 -> 800 in a strip; both factorisations at 576 columns 105 + 101 -> 101 + 97 us, at 2304 637 + 477 -> 634 + 470.
__device__ __forceinline__ int chol_chain8(const double* mb, double* Wbuf, int lane) {
    double m[8][8];
#pragma unroll
    for (int p = 0; p < 8; ++p)
#pragma unroll
        for (int j = p & ~1; j < 8; j += 2) {
            const double2 v = *reinterpret_cast<const double2*>(mb + p * 8 + j);
            m[p][j] = v.x;
            m[p][j + 1] = v.y;
        }
    // lane j carries column j mod 8 of the identity along, which becomes column j of L^-1, M = L D L^T
    double x[8], d[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = i == (lane & 7) ? 1.0 : 0.0;
#pragma unroll
    for (int p = 0; p < 8; ++p) {
        d[p] = m[p][p];
        if (p == 7) break;
        const double inv = pivot_reciprocal(d[p]);         // what the chain waits for
#pragma unroll
        for (int i = p + 1; i < 8; ++i) {
            const double f = m[p][i] * inv;
#pragma unroll
            for (int j = i; j < 8; ++j) m[i][j] = fma(-f, m[p][j], m[i][j]);
            x[i] = fma(-f, x[p], x[i]);
        }
    }
    const int q = lane >> 3;
    double d0 = d[0], d1 = d[1], x0 = x[0], x1 = x[1];
#pragma unroll
    for (int r = 1; r < 4; ++r) {
        d0 = q == r ? d[2 * r] : d0;
        d1 = q == r ? d[2 * r + 1] : d1;
        x0 = q == r ? x[2 * r] : x0;
        x1 = q == r ? x[2 * r + 1] : x1;
    }
    double* w = Wbuf + 16 * q + (lane & 7);                // W[p][j] = (U_M^-T)[p][j]
    w[0] = x0 * pivot_rsqrt(d0);
    w[8] = x1 * pivot_rsqrt(d1);
    const bool ok = d0 >= kMinPivot && d0 < kMaxPivot && d1 >= kMinPivot && d1 < kMaxPivot;
    if (__all_sync(0xffffffffu, ok)) return -1;
    __syncwarp();                                          // a vote orders no memory: what W holds by now is written again
    return chol_chain8_general(mb, Wbuf, lane);
}

// Two MMAs: the 8 x 8 product W R in accumulator layout, W row-major in Wbuf, R with row stride ldr.
__device__ __forceinline__ double2 chol_new_rows(const double* Wbuf, const double* R, int ldr, int lq, int lr) {
    double2 v = make_double2(0.0, 0.0);
    dmma_884(v.x, v.y, Wbuf[lq * 8 + lr], R[lr * ldr + lq]);
    dmma_884(v.x, v.y, Wbuf[lq * 8 + 4 + lr], R[(4 + lr) * ldr + lq]);
    return v;
}

// Warp 0: the chains of all eight pivot blocks and the mini-blocks in between.  first: the first mini-block in accumulator
// layout (group 0's only fragment in use).  Returns the first eight rows of the factor in those columns.
__device__ __forceinline__ double2 chol_strip_chain(double2 first, const StripSmem& sm, int lane, int k0, bool reporter,
                                                    int32_t* status, int threads) {
    const int lq = lane >> 2, lr = lane & 3;
    *reinterpret_cast<double2*>(sm.M + lq * 8 + 2 * lr) = first;
    *reinterpret_cast<double2*>(sm.R + lq * kStripLd + 2 * lr) = first;
    __syncwarp();
#pragma unroll 1
    for (int b = 0; b < 8; ++b) {
        double* Wb = sm.W + (b & 1) * 64;
        const int bad = chol_chain8(sm.M, Wb, lane);
        if (b & 1) named_bar_arrive<4>(threads); else named_bar_arrive<3>(threads);
        if (bad >= 0 && reporter) report(status, PTQ_ERR_NOT_SPD, k0 + 8 * b + bad);
        __syncwarp();
        if (b < 7) {
            const double* X = sm.X + (b & 1) * 128;
            if (b & 1) named_bar_sync<2>(64); else named_bar_sync<1>(64);      // R and T of the next eight columns are out
            const double2 v = chol_new_rows(Wb, X, 8, lq, lr);
            *reinterpret_cast<double2*>(sm.V + lq * 8 + 2 * lr) = v;
            double2 t = *reinterpret_cast<const double2*>(X + 64 + lq * 8 + 2 * lr);
            __syncwarp();
            const double u0 = sm.V[lr * 8 + lq], u1 = sm.V[(4 + lr) * 8 + lq];
            dmma_884(t.x, t.y, flip_sign(u0), u0);
            dmma_884(t.x, t.y, flip_sign(u1), u1);
            *reinterpret_cast<double2*>(sm.M + lq * 8 + 2 * lr) = t;
            __syncwarp();
        }
        if (b == 0) first = chol_new_rows(Wb, sm.R, kStripLd, lq, lr);
    }
    return first;
}

// Every other warp: pivot block B.
template <int B>
__device__ __forceinline__ void chol_strip_block(double (&acc)[8][2], const StripSmem& sm, int grp, int lane, bool update,
                                                 const double* ua, const double* bsrc, int threads) {
    const int lq = lane >> 2, lr = lane & 3;
    // While warp 0 is in its chain: the update by the pivot block before, and the look-ahead update of the rows of the next
    // pivot block.  The owner of the next eight columns puts out what warp 0 is going to need first; it has brought its next
    // diagonal fragment up to date one pivot block early, so that only the update by the pivot block before stands in between.
    const bool owner = B < 7 && grp == B + 1;
    if constexpr (B > 0) chol_strip_update<B, (B < 7 ? B + 2 : 8)>(acc, sm.U, grp, lq, lr);
    if (owner) {
        if constexpr (B == 0) {
            if (update) chol_strip_lookahead<1>(acc, ua, bsrc, grp, lq, lr);
        }
        double* X = sm.X + (B & 1) * 128 + lq * 8 + 2 * lr;
        *reinterpret_cast<double2*>(X) = make_double2(acc[B][0], acc[B][1]);
        if constexpr (B < 7) *reinterpret_cast<double2*>(X + 64) = make_double2(acc[B + 1][0], acc[B + 1][1]);
        named_bar_arrive<1 + (B & 1)>(64);
    }
    if constexpr (B > 0 && B < 6) chol_strip_update<B + 2, 8>(acc, sm.U, grp, lq, lr);
    if constexpr (B < 7) {
        if (update && !owner) chol_strip_lookahead<B + 1>(acc, ua, bsrc, grp, lq, lr);
    }
    if constexpr (B < 6) {
        if (update && grp == B + 2) chol_strip_lookahead<B + 2>(acc, ua, bsrc, grp, lq, lr);
    }
    // the rows of this pivot block as an MMA operand (read back by this warp only)
    *reinterpret_cast<double2*>(sm.R + lq * kStripLd + 8 * grp + 2 * lr) = make_double2(acc[B][0], acc[B][1]);
    named_bar_sync<3 + (B & 1)>(threads);             // W is there; nobody reads the previous new rows any more
    if (grp >= B) {
        const double2 v = chol_new_rows(sm.W + (B & 1) * 64, sm.R + 8 * grp, kStripLd, lq, lr);
        acc[B][0] = v.x;
        acc[B][1] = v.y;
        *reinterpret_cast<double2*>(sm.U + lq * kStripLd + 8 * grp + 2 * lr) = v;
    }
    if constexpr (B < 7) named_bar_sync<5>(threads - 32);             // the new rows are out
}
template <int... Bs>
__device__ __forceinline__ void chol_strip_blocks(double (&acc)[8][2], const StripSmem& sm, int grp, int lane, bool update,
                                                  const double* ua, const double* bsrc, int threads, std::integer_sequence<int, Bs...>) {
    (chol_strip_block<Bs>(acc, sm, grp, lane, update, ua, bsrc, threads), ...);
}

// Factorises the diagonal block of A at k0 and applies the same row operations to 8 pg panel columns with it: columns
// pc0 .. pc0 + 8 pg - 1 of rows k0 .. k0 + 63 of the matrix P (row stride ld); with add_identity the entries on P's diagonal are
// taken as 1 (P = W, zero there in memory: the transform of the identity block is the inverse of the transposed diagonal
// factor).  P == nullptr: diagonal block only.
// Every CTA working on this block row reads the diagonal block of A, at a time of its own, so the factor of that
// block is NOT written in place: the CTA with write_diag set stores it to D (64 x 64, row stride 64), and the kernel
// copies all diagonal factors into A at its very end.
// look_ahead: the strip is first brought up to date with the previous block row, which is final by then:
//     strip -= upd_a^T [upd_a | upd_b],   upd_a[kk][r] = U[k0 - 64 + kk][k0 + r],  upd_b[kk][c] = P[k0 - 64 + kk][pc0 + c]
// (64 rows in shared memory, row stride kCholLd).
// Not inlined: the chain alone needs nearly all of the 128 registers, and what the kernel keeps across a strip is saved
// once around the call instead of inside the chain.
__device__ __noinline__ void chol_strip(double* __restrict__ A, int64_t ld, int n, int k0, double* __restrict__ P,
                                        int pc0, int pg, bool add_identity, bool write_diag, double* __restrict__ D, int vec16,
                                        int32_t* status, bool look_ahead) {
    extern __shared__ __align__(16) unsigned char chol_smem_raw[];
    double* smem = reinterpret_cast<double*>(chol_smem_raw);
    // operands of the look-ahead update, beyond the strip's own panel buffers
    double* upd_a = smem + kStripSmemDoubles;
    double* upd_b = upd_a + kCholBlock;
    const bool has_b = look_ahead && P != nullptr;
    if (look_ahead) {
        chol_load_block<kCholThreads>(upd_a, A, ld, n, k0 - kNB, k0, 6, vec16, threadIdx.x);
        if (has_b) chol_load_block<kCholThreads>(upd_b, P, ld, n, k0 - kNB, pc0, pg == 5 ? 6 : (pg == 3 ? 5 : 4), vec16, threadIdx.x);
        cp_async_commit();
    }
    const int lane = threadIdx.x & 31, grp = (int)((strip_warps(pg) >> (4 * (threadIdx.x >> 5))) & 15u);
    const int threads = 32 * (8 + pg);                                       // of the warps that take part
    const int lq = lane >> 2, lr = lane & 3;
    const StripSmem sm(smem);
    const bool is_diag = grp < 8;
    const int gc0 = is_diag ? k0 + 8 * grp : pc0 + 8 * (grp - 8);           // first global column of this warp
    const int sc0 = 8 * grp;                                                 // first strip column
    double acc[8][2];
    if (grp < 15) {
        // columns that lie inside the matrix: plain vector loads (of the diagonal block only the fragments from the
        // diagonal up; what lies below the diagonal in the diagonal fragment itself is never used)
        const bool fast = vec16 && k0 + kNB <= n && (is_diag || (P != nullptr && pc0 + 8 * pg <= n));
        if (fast) {
            const double* src = (is_diag ? A : P) + (int64_t)(k0 + lq) * ld + gc0 + 2 * lr;
#pragma unroll
            for (int rb = 0; rb < 8; ++rb) {
                if (is_diag && rb > grp) { acc[rb][0] = acc[rb][1] = 0.0; continue; }
                const double2 v = __ldcg(reinterpret_cast<const double2*>(src + (int64_t)(8 * rb) * ld));
                acc[rb][0] = v.x;
                acc[rb][1] = v.y;
            }
        } else {
#pragma unroll
            for (int rb = 0; rb < 8; ++rb) {
                const int row = 8 * rb + lq, grow = k0 + row;
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int sc = sc0 + 2 * lr + e, gc = gc0 + 2 * lr + e;
                    double val = 0.0;
                    if (is_diag) {
                        if (sc >= row) {
                            if (grow < n && gc < n) val = __ldcg(A + (int64_t)grow * ld + gc);
                            else if (sc == row) val = 1.0;                   // identity padding below n
                        }
                    } else if (P != nullptr && grow < n && gc < n) {
                        val = __ldcg(P + (int64_t)grow * ld + gc);
                    }
                    acc[rb][e] = val;
                }
            }
        }
        if (add_identity && !is_diag) {
#pragma unroll
            for (int rb = 0; rb < 8; ++rb)
#pragma unroll
                for (int e = 0; e < 2; ++e)
                    if (gc0 + 2 * lr + e == k0 + 8 * rb + lq) acc[rb][e] = 1.0;
        }
    }
    // Look-ahead update with the block row above: only the first fragment row is brought up to date here; the others
    // follow inside the strip, each while warp 0 works on the mini-block before it.
    const double* bsrc = is_diag ? upd_a + 8 * grp : upd_b + 8 * (grp - 8);
    const bool update = look_ahead && (is_diag || has_b);
    if (look_ahead) {
        cp_async_wait<0>();
        __syncthreads();
        if (update && grp < 15) chol_strip_lookahead<0>(acc, upd_a, bsrc, grp, lq, lr);
    }
    if (grp == 15) return;
    if (grp == 0) {
        const double2 v = chol_strip_chain(make_double2(acc[0][0], acc[0][1]), sm, lane, k0, write_diag && lane == 0, status, threads);
        if (write_diag) {
            if (2 * lr >= lq) D[lq * kNB + 2 * lr] = v.x;
            if (2 * lr + 1 >= lq) D[lq * kNB + 2 * lr + 1] = v.y;
        }
        return;
    }
    chol_strip_blocks(acc, sm, grp, lane, update, upd_a, bsrc, threads, std::make_integer_sequence<int, 8>());
    if (is_diag) {
        if (write_diag) {
#pragma unroll
            for (int rb = 0; rb < 8; ++rb) {
                const int row = 8 * rb + lq, sc = sc0 + 2 * lr;
                if (sc >= row) D[row * kNB + sc] = acc[rb][0];
                if (sc + 1 >= row) D[row * kNB + sc + 1] = acc[rb][1];
            }
        }
    } else if (P != nullptr) {
#pragma unroll
        for (int rb = 0; rb < 8; ++rb) {
            const int grow = k0 + 8 * rb + lq, gc = gc0 + 2 * lr;
            if (grow >= n || gc >= n) continue;
            double* dst = P + (int64_t)grow * ld + gc;
            if (vec16) {
                __stcg(reinterpret_cast<double2*>(dst), make_double2(acc[rb][0], acc[rb][1]));
            } else {
                __stcg(dst, acc[rb][0]);
                if (gc + 1 < n) __stcg(dst + 1, acc[rb][1]);
            }
        }
    }
}

// One H x 64 piece of a trailing tile, C[i0 .. i0 + H)[j0 .. j0 + 64); the 16 warps as 4 x 4 (H = 16: 2 x 8).
// tri >= 0: the piece lies in a diagonal tile, tri rows below its top, and only entries with c >= tri + r are touched.
struct CholPiece {
    double* C;
    const double* Bsrc;
    int i0, j0, tri;
};
template <int H>
struct CholPieceShape {
    static constexpr int WN = H == 16 ? 8 : 4;                 // warps side by side
    static constexpr int FM = H * WN / 128, FN = 8 / WN;       // 8 x 8 fragments of a warp
};
__device__ __forceinline__ bool chol_piece_has(const CholPiece& pc, int n, int r, int c) {
    return pc.i0 + r < n && pc.j0 + c < n && (pc.tri < 0 || c >= pc.tri + r);
}
// a piece inside the matrix and off the diagonal needs no bounds or triangle tests at all
template <int H>
__device__ __forceinline__ bool chol_piece_plain(const CholPiece& pc, int n, int vec16) {
    return vec16 && pc.tri < 0 && pc.i0 + H <= n && pc.j0 + kNB <= n;
}
// The two entries of the piece at (r, c), (r, c + 1); zero where the piece has none.
__device__ __forceinline__ double2 chol_pair_load(const CholPiece& pc, const double* src, int n, int r, int c, bool plain,
                                                  int vec16) {
    const bool k0 = plain || chol_piece_has(pc, n, r, c);
    if (plain || (vec16 && k0)) return __ldcg(reinterpret_cast<const double2*>(src));       // n even: the pair is inside
    return make_double2(k0 ? __ldcg(src) : 0.0, chol_piece_has(pc, n, r, c + 1) ? __ldcg(src + 1) : 0.0);
}
__device__ __forceinline__ void chol_pair_store(const CholPiece& pc, double* dst, int n, int r, int c, bool plain, int vec16,
                                                double2 v) {
    const bool k0 = plain || chol_piece_has(pc, n, r, c);
    if (plain || (vec16 && k0)) {
        __stcg(reinterpret_cast<double2*>(dst), v);
    } else {
        if (k0) __stcg(dst, v.x);
        if (chol_piece_has(pc, n, r, c + 1)) __stcg(dst + 1, v.y);
    }
}

// Trailing tiles of block row k restricted to the target block rows row_base <= i < row_limit.
//   tiles of A: (i, j), row_base <= i <= j: A[i][j] -= U[k][i]^T U[k][j]
//   tiles of W: (i, c), row_base <= i, c <= k:  W[i][c] -= U[k][i]^T W[k][c]       (row-major lists, A first)
// In look-ahead mode the CTAs come here after `strips_b` strips of the next block row, the CTAs 0 .. n_more - 1 after
// one more; a strip costs strip_cost eighths of a tile, so they take correspondingly fewer pieces (the busier CTAs from the
// end of the list) and all CTAs finish at about the same time.
// Not inlined, for the sake of the registers, like chol_strip.
__device__ __noinline__ void chol_trailing_phase(double* __restrict__ A, double* __restrict__ Wm, int n, int64_t ld, int vec16,
                                                 int G, int k, int row_base, int row_limit, int n_more, int strips_b, int strip_cost) {
    extern __shared__ __align__(16) unsigned char chol_smem_raw[];
    const int nb = (n + kNB - 1) / kNB;
    const int k0 = k * kNB;
    const int m = nb - row_base;                                        // tiles in the first target row
    const int R = (row_limit < nb ? row_limit : nb) - row_base;         // target block rows
    if (R <= 0) return;
    const int TA = R * m - R * (R - 1) / 2;
    const int TW = Wm != nullptr ? R * (k + 1) : 0;
    const int T = TA + TW;
    if (T <= 0) return;
    // Tiles are cut into 64 / H row pieces so that a short tile list still spreads over the grid: in two where there are no
    // more of them than CTAs (against half as many: 2304 columns 1228.5 -> 1228.0 us, 2816: 1825.8 -> 1824.4, no difference
    // below), in four where the pieces are still no more than CTAs.
    const int lgH = 4 * T <= G ? 4 : (T <= G ? 5 : 6);
    const int lgP = 6 - lgH;
    const int TP = T << lgP;
    const int S = n_more < G ? n_more : G, N = G - S;
    const int cs = strip_cost << lgP;                                   // in eighths of a piece
    const int cost_a = (strips_b + 1) * cs, cost_b = strips_b * cs;
    const int all = 8 * TP + S * cost_a + N * cost_b;
    int ps = 0;
    if (S > 0) {
        // what a strip CTA is short of the average, in whole pieces
        ps = all > G * cost_a ? (int)((unsigned)(all - G * cost_a + 8 * G - 1) / (unsigned)(8 * G)) : 0;
        if (N == 0) ps = (int)((unsigned)(TP + S - 1) / (unsigned)S);
    }
    const int TPn = TP - S * ps > 0 ? TP - S * ps : 0;
    const int pn = N > 0 ? (int)((unsigned)(TPn + N - 1) / (unsigned)N) : 0;
    int tp_beg, tp_end;
    if ((int)blockIdx.x >= S) {
        tp_beg = ((int)blockIdx.x - S) * pn;
        tp_end = tp_beg + pn < TPn ? tp_beg + pn : TPn;
    } else {
        tp_beg = TPn + (int)blockIdx.x * ps;
        tp_end = tp_beg + ps < TP ? tp_beg + ps : TP;
    }
    if (tp_beg >= tp_end) return;
    // pieces are asked for in ascending order, so the row of the triangular list is found by walking on from the
    // row of the previous piece
    int cur_r = 0, cur_start = 0;                       // row cur_r of the A list starts at tile cur_start
    auto piece_of = [&](int tp) {
        CholPiece pc;
        const int t = tp >> lgP;
        const int h0 = (tp & ((1 << lgP) - 1)) << lgH;
        if (t < TA) {
            while (t >= cur_start + (m - cur_r)) { cur_start += m - cur_r; ++cur_r; }
            const int r = cur_r;
            const int bi = row_base + r, bj = bi + (t - cur_start);
            pc.C = A; pc.Bsrc = A; pc.i0 = bi * kNB + h0; pc.j0 = bj * kNB;
            pc.tri = bi == bj ? h0 : -1;
        } else {
            const int tw = t - TA;
            const int r = (int)((unsigned)tw / (unsigned)(k + 1)), c = tw - r * (k + 1);
            pc.C = Wm; pc.Bsrc = Wm; pc.i0 = (row_base + r) * kNB + h0; pc.j0 = c * kNB;
            pc.tri = -1;
        }
        return pc;
    };
    // Operand blocks: a slot of abuf holds U[k][i-block] (as[kk][r]), a slot of bbuf U or W [k][j-block] (bs[kk][c]).
    // Every CTA takes a contiguous run of the list, in which consecutive tiles mostly share their row block: the A
    // operand then stays where it is and only B is fetched.  The next piece's operands and this one's old values are
    // requested at the start of the piece; the products are summed apart and subtracted from the old values once (added one
    // by one to them they would be rounded to their size sixteen times).  One barrier per piece.
    double* abuf = reinterpret_cast<double*>(chol_smem_raw);      // [2][64][kCholLd]
    double* bbuf = abuf + 2 * kCholBlock;                         // [2][64][kCholLd]
    auto run = [&](auto height) {
        constexpr int H = decltype(height)::value, FM = CholPieceShape<H>::FM, FN = CholPieceShape<H>::FN;
        constexpr int WN = CholPieceShape<H>::WN, LGH = H == 64 ? 6 : (H == 32 ? 5 : 4);
        const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, lq = lane >> 2, lr = lane & 3;
        const int wm0 = (warp / WN) * 8 * FM, wn0 = (warp % WN) * 8 * FN;
        const int pr = wm0 + lq, pq = wn0 + 2 * lr;       // this lane's entries: (pr + 8 a, pq + 8 b), and one further
        int stage = 0, a_slot = 0;
        CholPiece cur = piece_of(tp_beg), nxt = cur;
        chol_load_block<kCholThreads>(abuf, A, ld, n, k0, cur.i0, LGH, vec16, tid);
        chol_load_block<kCholThreads>(bbuf, cur.Bsrc, ld, n, k0, cur.j0, 6, vec16, tid);
        cp_async_commit();
        for (int tp = tp_beg; tp < tp_end; ++tp) {
            const bool more = tp + 1 < tp_end;
            if (more) nxt = piece_of(tp + 1);
            const bool new_a = more && nxt.i0 != cur.i0, plain = chol_piece_plain<H>(cur, n, vec16);
            const int a_next = a_slot ^ (new_a ? 1 : 0);
            const double* as = abuf + a_slot * kCholBlock;
            const double* bs = bbuf + stage * kCholBlock;
            cp_async_wait<0>();
            __syncthreads();         // this piece's operands have landed; the slots of the piece before are free
            double2 acc[FM][FN], old[FM][FN];
#pragma unroll
            for (int a = 0; a < FM; ++a)
#pragma unroll
                for (int b = 0; b < FN; ++b) acc[a][b] = make_double2(0.0, 0.0);
            // all k steps unrolled, addresses as constants (four at a time: 3 % slower)
            auto k_step = [&](int k4) {
                const int kk = 4 * k4 + lr;
                double af[FM], bf[FN];
#pragma unroll
                for (int a = 0; a < FM; ++a) af[a] = as[kk * kCholLd + wm0 + a * 8 + lq];
#pragma unroll
                for (int b = 0; b < FN; ++b) bf[b] = bs[kk * kCholLd + wn0 + b * 8 + lq];
#pragma unroll
                for (int a = 0; a < FM; ++a)
#pragma unroll
                    for (int b = 0; b < FN; ++b) dmma_884(acc[a][b].x, acc[a][b].y, af[a], bf[b]);
            };
            // The loads of a warp queue in order, so the products go first: the next operands are requested after two k steps, the
            // old values in the middle.  With both in front, both factorisations took 636 + 520 us at 2304 columns (the second
            // with the sweep behind it) and 1590 + 1241 at 4608; with the operands alone in front 601 + 508 and 1530 + 1213;
            // now 591 + 507 and 1509 + 1207.
            k_step(0);
            k_step(1);
            if (more) {
                // half of the warps request the next operands: the copies keep the issuing warps busy for several
                // hundred cycles, during which the others already feed the tensor pipe
                if (warp < 8) {
                    chol_load_block<kCholThreads / 2>(bbuf + (stage ^ 1) * kCholBlock, nxt.Bsrc, ld, n, k0, nxt.j0, 6, vec16, tid);
                    if (new_a)
                        chol_load_block<kCholThreads / 2>(abuf + a_next * kCholBlock, A, ld, n, k0, nxt.i0, LGH, vec16, tid);
                }
            }
#pragma unroll
            for (int k4 = 2; k4 < 8; ++k4) k_step(k4);
            // the old values
#pragma unroll
            for (int a = 0; a < FM; ++a)
#pragma unroll
                for (int b = 0; b < FN; ++b)
                    old[a][b] = chol_pair_load(cur, cur.C + (int64_t)(cur.i0 + pr + 8 * a) * ld + cur.j0 + pq + 8 * b, n,
                                               pr + 8 * a, pq + 8 * b, plain, vec16);
#pragma unroll
            for (int k4 = 8; k4 < kNB / 4; ++k4) k_step(k4);
            cp_async_commit();
#pragma unroll
            for (int a = 0; a < FM; ++a)
#pragma unroll
                for (int b = 0; b < FN; ++b)
                    chol_pair_store(cur, cur.C + (int64_t)(cur.i0 + pr + 8 * a) * ld + cur.j0 + pq + 8 * b, n, pr + 8 * a,
                                    pq + 8 * b, plain, vec16,
                                    make_double2(old[a][b].x - acc[a][b].x, old[a][b].y - acc[a][b].y));
            stage ^= 1;
            a_slot = a_next;
            cur = nxt;
        }
    };
    if (lgH == 6) run(std::integral_constant<int, 64>());
    else if (lgH == 5) run(std::integral_constant<int, 32>());
    else run(std::integral_constant<int, 16>());
}

// The whole of it, by the CTAs 0 .. G - 1 of the grid.
__device__ __forceinline__ void chol_factorise(double* __restrict__ A, double* __restrict__ Wm, double* __restrict__ Dbuf, int n,
                                               int64_t ld, int vec16, unsigned* bar, int32_t* status, long long spin_limit,
                                               int k_first, int nb_stop, int row_limit, const int G) {
    extern __shared__ __align__(16) unsigned char chol_smem_raw[];
    int* s_flag = reinterpret_cast<int*>(chol_smem_raw + sizeof(double) * kCholOpndDoubles);
    unsigned* s_plan = reinterpret_cast<unsigned*>(s_flag + 4);                    // [block rows], see below
    const int tid = threadIdx.x;
    const int nb = (n + kNB - 1) / kNB, nbs = nb_stop < nb ? nb_stop : nb;
    unsigned epoch = 0;

    // Strip work items of block row k: the chunks of 8 pg columns of A right of the block, then (with Wm) those of row block k
    // of W up to the end of the block's own columns, which start as the identity.
    auto chunks = [&](int k, int pg, int& ca, int& all) {
        const int wa = n - (k + 1) * kNB, ww = Wm != nullptr ? ((k + 1) * kNB < n ? (k + 1) * kNB : n) : 0;
        ca = wa > 0 ? (int)((unsigned)(wa + 8 * pg - 1) / (unsigned)(8 * pg)) : 0;
        all = ca + (int)((unsigned)(ww + 8 * pg - 1) / (unsigned)(8 * pg));
        if (all < 1) all = 1;                                                // last block without Wm: diagonal only
    };
    // The strips of every block row, worked out once per launch by a thread per block row: a few integer divisions on the way
    // from one grid barrier to the next cost as much as the whole barrier (both factorisations at 1152 columns: 222 + 209
    // -> 209 + 195 us without them).  Packed: panel groups, chunks of A << 4, chunks << 17, and whether the strips are all that
    // their CTAs are due (kStripsOnly).
    for (int k = k_first + tid; k < nbs; k += kCholThreads) {
        const int R = (row_limit < nb ? row_limit : nb) - (k + 1), m = nb - (k + 1);
        const int T = k > k_first && R > 0 ? R * m - R * (R - 1) / 2 + (Wm != nullptr ? R * k : 0) : 0;
        int pg = 5, ca, all;
        chunks(k, 5, ca, all);
        for (int c = 1; c < 5; c += c == 3 ? 2 : 1) {
            int ca_c, all_c;
            chunks(k, c, ca_c, all_c);
            if (all_c <= G && 8 * T <= (G - all_c) * kNarrowStripWork) { pg = c; ca = ca_c; all = all_c; break; }
        }
        const bool only = all < G && 8 * T <= (G - all) * (pg == 5 ? kStripCost : kNarrowStripCost);
        s_plan[k - k_first] = (unsigned)pg | (only ? kStripsOnly : 0u) | (unsigned)ca << 4 | (unsigned)all << 17;
    }
    __syncthreads();
    auto strips = [&](int k, int pg, int ca, int all, bool look_ahead) {
        for (int g = blockIdx.x; g < all; g += G) {
            double* P = nullptr;
            int pc0 = 0;
            if (g < ca) { P = A; pc0 = (k + 1) * kNB + g * 8 * pg; }
            else if (Wm != nullptr) { P = Wm; pc0 = (g - ca) * 8 * pg; }
            __syncthreads();     // the panel buffers are those of the repetition before and of the trailing phase
            chol_strip(A, ld, n, k * kNB, P, pc0, pg, P == Wm, g == 0, Dbuf + (size_t)k * kNB * kNB, vec16, status, look_ahead);
            __syncthreads();
        }
    };
    // The block rows k_first .. nb_stop - 1 are factorised (block row k_first must already carry the updates of all rows
    // above it); their updates are applied to the target rows below row_limit.
    //   k_first = 0, nb_stop = nb, row_limit = nb : the whole factorisation;
    //   nb_stop < nb, row_limit = nb : a partial factorisation that leaves the Schur complement of the leading block in
    //       the upper triangle of A[64 nb_stop :, 64 nb_stop :] (what Eq. 12 leaves after that many columns);
    //   row_limit = nb_stop : a panel -- only its own block rows are touched; the caller applies the panel to the rows
    //       below it in one product of depth 64 (nb_stop - k_first).
    const int steps = nbs < nb ? (row_limit > nbs ? nbs : nbs - 1) : nb - 1;
    {
        const unsigned plan = s_plan[0];
        strips(k_first, (int)(plan & 7u), (int)(plan >> 4 & 0x1fffu), (int)(plan >> 17), false);
    }
    for (int k = k_first; k < steps; ++k) {
        ++epoch;
        if (!grid_barrier(bar, epoch * (unsigned)G, s_flag, spin_limit)) break;
        // Block row k is final; the updates of block rows < k have been applied everywhere.
        if (k + 1 >= nbs) {                  // last factorised block row of a partial run: its update only
            chol_trailing_phase(A, Wm, n, ld, vec16, G, k, k + 1, row_limit, 0, 0, 0);
            continue;
        }
        // Look-ahead: the CTAs factorise the strips of block row k + 1 first (item g by CTA g mod G; each brings its
        // strip up to date with block row k itself) and then join the trailing tiles of block row k below row k + 1 with
        // a share reduced by what their strips cost, so nobody idles and there is one grid barrier per block row.
        const unsigned plan = s_plan[k + 1 - k_first];
        const int pg = (int)(plan & 7u), all = (int)(plan >> 17);
        strips(k + 1, pg, (int)(plan >> 4 & 0x1fffu), all, true);
        if (!(plan & kStripsOnly) || (int)blockIdx.x >= all)
            chol_trailing_phase(A, Wm, n, ld, vec16, G, k, k + 2, row_limit, all < G ? all : all % G, all < G ? 0 : all / G,
                                pg == 5 ? kStripCost : kNarrowStripCost);
    }
    cp_async_wait<0>();
    // the diagonal factors move from the side buffer into A once nobody reads the original diagonal blocks any more
    ++epoch;
    if (grid_barrier(bar, epoch * (unsigned)G, s_flag, spin_limit)) {
        for (int b = k_first + blockIdx.x; b < nbs; b += G)
            for (int idx = tid; idx < kNB * kNB; idx += kCholThreads) {
                const int r = idx >> 6, c = idx & 63;
                if (c >= r && b * kNB + c < n)
                    A[(int64_t)(b * kNB + r) * ld + b * kNB + c] = __ldcg(Dbuf + (size_t)b * kNB * kNB + idx);
            }
    }
    if (tid == 0 && ld_acquire_u32(&bar[1]) != 0u) report(status, PTQ_ERR_TIMEOUT, blockIdx.x, 1);
}

__global__ void __launch_bounds__(kCholThreads, 1)
chol_coop_kernel(double* __restrict__ A, double* __restrict__ Wm, double* __restrict__ Dbuf, int n, int64_t ld,
                 int vec16, unsigned* bar, int32_t* status, long long spin_limit, int k_first, int nb_stop,
                 int row_limit) {
    chol_factorise(A, Wm, Dbuf, n, ld, vec16, bar, status, spin_limit, k_first, nb_stop, row_limit, gridDim.x);
}

// In-place blocked upper Cholesky A = U^T U of the n x n matrix A (row stride n).  Only the upper triangle is read or
// written.  With Wm (n x n, zero on entry) the same sweep also leaves W = U^-T there (lower triangular): the row
// operations of the factorisation are applied to the identity, which gives the inverse of the Cholesky factor that
// Sec. 5 item 1 asks for.
// `bar` is 2 x uint32 of device scratch, Dbuf holds chol_scratch_doubles(n) doubles (the diagonal factors on their way).
inline size_t chol_scratch_doubles(int n) { return (size_t)((n + kNB - 1) / kNB) * kNB * kNB; }
// One CTA per SM (the cooperative launch guarantees that all of them are resident); a matrix of a few block rows
// gets no more CTAs than it has work for, which makes its grid barriers cheaper and leaves SMs to kernels of other
// streams.  Twice the 64 x 64 tiles of A and W, and at least a CTA per eight columns: never fewer than the narrowest strips
// of a block row, and with W never fewer than the pieces of its trailing tiles (without W there are up to a third more
// pieces than CTAs at 7 to 11 block rows).
inline int chol_grid(int n, bool with_w, int budget) {
    const int nbr = cdiv(n, kNB);
    const long tiles2 = 2L * ((long)nbr * (nbr + 1) / 2 + (with_w ? (long)nbr * nbr : 0));
    const long items = tiles2 > (n + 7) / 8 ? tiles2 : (n + 7) / 8;
    return items < budget ? (int)(items < 1 ? 1 : items) : budget;
}
// Which block rows of a factorisation: first .. stop - 1, their updates applied to the rows below row_limit (chol_factorise).
struct CholRange {
    int first, stop, row_limit;
};
inline CholRange chol_all_rows(int n) { return {0, cdiv(n, kNB), cdiv(n, kNB)}; }
// nb_stop > 0: factorise the block rows k_first .. nb_stop - 1 only (see the kernel for what row_limit selects;
// row_limit <= 0: all rows below are updated).  A partial run that updates everything below must not ask for Wm.
// bar_ready: the caller has cleared `bar`.
inline int cholesky_upper(double* A, int n, double* Wm, double* Dbuf, unsigned* bar, int32_t* status,
                          cudaStream_t stream, int nb_stop = 0, int k_first = 0, int row_limit = 0,
                          bool bar_ready = false) {
    const int nb_all = (n + kNB - 1) / kNB;
    if (nb_stop <= 0) nb_stop = nb_all;
    if (row_limit <= 0) row_limit = nb_all;
    if (nb_stop < nb_all && row_limit > nb_stop && Wm != nullptr) return PTQ_ERR_INVALID_ARG;
    if (k_first < 0 || k_first >= nb_stop) return PTQ_ERR_INVALID_ARG;
    DeviceState* dev = nullptr;
    int st = current_device_state(&dev);
    if (st) return st;
    if (!dev->coop) return PTQ_ERR_UNSUPPORTED;
    st = ensure_smem_attr(dev, SA_CHOL, [] {
        cudaError_t e = cudaFuncSetAttribute(chol_coop_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kCholSmemBytes);
        int per_sm = 0;
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, chol_coop_kernel, kCholThreads, kCholSmemBytes);
        return (e == cudaSuccess && per_sm < 1) ? cudaErrorLaunchOutOfResources : e;
    });
    if (st) return st;
    const int grid = chol_grid(n, Wm != nullptr, coop_cta_budget(dev));
    if (!bar_ready && cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned), stream) != cudaSuccess) return PTQ_ERR_CUDA;
    int64_t ld = n;
    int vec16 = ((n & 1) == 0 && aligned16(A) && aligned16(Wm)) ? 1 : 0;
    long long spin_limit = kSpinLimitCycles;
    void* args[] = {&A, &Wm, &Dbuf, &n, &ld, &vec16, &bar, &status, &spin_limit, &k_first, &nb_stop, &row_limit};
    Launch l(K_CHOL_COOP, stream);
    if (cudaLaunchCooperativeKernel((const void*)chol_coop_kernel, dim3(grid), dim3(kCholThreads), args,
                                    kCholSmemBytes, stream) != cudaSuccess) {
        cudaGetLastError();
        return PTQ_ERR_CUDA;
    }
    return PTQ_OK;
}

// Hinv = W^T W for the lower-triangular W = U^-T: Hinv[i][j] = sum over k >= max(i, j) of W[k][i] W[k][j]; upper tiles
// computed, mirrored below; its diagonal also goes to diag.
inline int lauum_lower(const double* W, double* Hinv, double* diag, int n, cudaStream_t stream) {
    GemmParams g = gemm_defaults();
    g.A = W; g.lda = n; g.a_trans = 1;
    g.B = W; g.ldb = n; g.b_trans = 0;
    g.C = Hinv; g.ldc = n; g.diag = diag;
    g.M = n; g.N = n; g.K = n;
    g.kbeg_mode = 1; g.upper_only = 1; g.mirror = 1;
    return launch_dgemm(K_DGEMM_LAUUM, g, 1, stream);
}

}  // namespace ptq
