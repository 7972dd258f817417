// Dynamic re-ranking (Sec. 5 places the sort inside the per-column loop): the columns still to be quantized are ranked
// again every `block` columns, from the compensated weights and the diagonal of the Eq.-12-updated inverse Hessian.
//
// One round, with m columns left, A the current m x m matrix (what Eq. 12 has left of the inverse Hessian) and Wc the
// current weights: scores and order of the m columns; both are gathered into that order; the first b = min(block, m)
// block rows of the Cholesky factor of A are computed, which leaves the Schur complement of the leading b x b block --
// the matrix Eq. 12 leaves after those b columns -- in the rest; the first b columns are swept with those rows of the
// factor; the remaining columns absorb the b columns' errors in one product, Wc[:, b:] -= E U[:b, b:] (Eq. 11, deferred).
// The rest of A and Wc are the next round's inputs.  Only the upper triangle of A is kept up to date.
#pragma once
#include "common.cuh"
#include "order.cuh"

namespace ptq {

// Everything a round starts from, in the new order, one grid row per row of the matrix and then of the weights:
//   Anew[a][c] = A[lo][hi] with {lo, hi} = {ordr[a], ordr[c]} sorted, for c from row a's diagonal tile on (only the upper triangle
//   of A is read, and only that of Anew, whole tiles on the diagonal, is read later);
//   orig_new[a] = orig[ordr[a]], the original column at position a (orig == nullptr: ordr[a]); the first b go to order_out;
//   Wnew[i][p] = (double) Wc[i][ordr[p]];  E[i][p] = NaN for the first b columns, "not published yet" for the sweep;
//   and the counters of the factorisation (two words) and of the sweep are cleared.
// One launch for what were three kernels and three clears, 13 operations a round -> 7 (128 x 1152 with rounds of 128 columns,
// whole layer: 1035 -> 949 us).
template <typename T>
__global__ void __launch_bounds__(256) round_gather_kernel(const double* __restrict__ A, int64_t lda, const T* __restrict__ Wc,
                                                           int64_t ldw, int rows, const int32_t* __restrict__ ordr,
                                                           const int32_t* __restrict__ orig, int m, int b, double* __restrict__ Anew,
                                                           double* __restrict__ Wnew, double* __restrict__ E,
                                                           int32_t* __restrict__ orig_new, int32_t* __restrict__ order_out,
                                                           unsigned* __restrict__ bar, unsigned* __restrict__ flags, int n_flags) {
    chained_begin();
    const int step = gridDim.x * 256, first = blockIdx.x * 256 + threadIdx.x;
    if (blockIdx.y == 0) {
        if (first < 2) bar[first] = 0u;
        for (int f = first; f < n_flags; f += step) flags[f] = 0u;
    }
    for (int y = blockIdx.y; y < m + rows; y += gridDim.y) {
        if (y < m) {
            const int oa = ordr[y];
            if (first == 0) {
                const int o = orig != nullptr ? orig[oa] : oa;
                orig_new[y] = o;
                if (y < b) order_out[y] = o;
            }
            for (int c = (y & ~(kNB - 1)) + first; c < m; c += step) {
                const int oc = ordr[c];
                const int lo = oa < oc ? oa : oc, hi = oa < oc ? oc : oa;
                Anew[(int64_t)y * m + c] = A[(int64_t)lo * lda + hi];
            }
        } else {
            const int i = y - m;
            for (int p = first; p < m; p += step) {
                Wnew[(int64_t)i * m + p] = (double)Wc[(int64_t)i * ldw + ordr[p]];
                if (p < b) E[(int64_t)i * m + p] = __longlong_as_double(-1ll);
            }
        }
    }
}

// The b columns just swept go out in the ORIGINAL column order: codes, What = float32(scale (code - zero)), dW = W - What.
__global__ void emit_block_kernel(const uint8_t* __restrict__ codes_p, int64_t ld, const int32_t* __restrict__ orig, int b,
                                  const float* __restrict__ W, int rows, int cols, int64_t ldw,
                                  const float* __restrict__ scale, const float* __restrict__ zero,
                                  uint8_t* __restrict__ codes, float* __restrict__ What, double* __restrict__ dW) {
    chained_begin();
    for (int i = blockIdx.y; i < rows; i += gridDim.y) {
        const double sc = (double)scale[i], zp = (double)zero[i];
        for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < b; p += gridDim.x * blockDim.x) {
            const int j = orig[p];
            const uint8_t c = codes_p[(int64_t)i * ld + p];
            codes[(int64_t)i * cols + j] = c;
            const float q = (float)(sc * ((double)c - zp));
            if (What) What[(int64_t)i * cols + j] = q;
            if (dW) dW[(int64_t)i * cols + j] = (double)W[(int64_t)i * ldw + j] - (double)q;
        }
    }
}

}  // namespace ptq
