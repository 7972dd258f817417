// The non-parallel arm of the paper's ablation (Sec. 4.2, the paragraph on the per-row inverse Hessians; the rows of
// Table 3 without the parallel tick): every row ranks ITS weights by their own sensitivities (Sec. 4.1) and is quantized
// in that order against a private copy of the inverse Hessian -- the [d_row, d_col, d_col] tensor, one slice per CTA,
// held in shared memory.  Cost rows * cols^3 / 3, which is what the row-parallel method saves; narrow layers only.
#pragma once
#include "common.cuh"
#include "order.cuh"
#include "colloop.cuh"

namespace ptq {

constexpr int kPerRowMaxCols = 128;
constexpr int kPerRowWarps = 5;              // chain, column loop, three for the trailing tiles
constexpr int kPerRowThreads = 32 * kPerRowWarps;
// Shared memory: the upper 8 x 8 tiles of the row's matrix, then [n8] weights, differences and reciprocal pivots,
// W (8 x 8), the scaled diagonal tile (8 x 8), the order and its inverse.
inline size_t per_row_smem_bytes(int cols) {
    const size_t nf = (size_t)(cols + 7) / 8;
    return sizeof(double) * (nf * (nf + 1) / 2 * 64 + 3 * 8 * nf + 128) + 2 * sizeof(int32_t) * 8 * nf;
}

// The eight pivots of the diagonal tile `m` (row-major 8 x 8, symmetric): m = L D L^T.  All of the tile sits in every
// lane, so the serial chain has no data exchange in it; lane j carries column j of the identity along, which becomes
// column j of L^-1.  Leaves L^-1 in Wb and the reciprocal pivots in dinv.  A pivot that is not accepted is replaced by 1;
// returns the first such pivot or -1.
// DIVIDE = false accepts normal pivots only.  DIVIDE = true, for the repetition of a tile with some other pivot, divides, and
// so takes subnormal pivots as well, down to those whose reciprocal overflows.
template <bool DIVIDE>
__device__ __forceinline__ int per_row_chain(const double* tile, double* Wb, double* dinv, int lane) {
    double m[8][8], x[8];
#pragma unroll
    for (int p = 0; p < 8; ++p)
#pragma unroll
        for (int j = p; j < 8; ++j) m[p][j] = tile[8 * p + j];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = i == (lane & 7) ? 1.0 : 0.0;
    int bad = -1;
#pragma unroll
    for (int p = 0; p < 8; ++p) {
        const double d0 = m[p][p];
        const bool ok = DIVIDE ? d0 > 0.0 && d0 < kMaxPivot && isfinite(1.0 / d0) : d0 >= kMinPivot && d0 < kMaxPivot;
        bad = (!ok && bad < 0) ? p : bad;
        const double d = ok ? d0 : 1.0;
        const double inv = DIVIDE ? 1.0 / d : pivot_reciprocal(d);
        if (lane == 0) dinv[p] = inv;
#pragma unroll
        for (int i = p + 1; i < 8; ++i) {
            const double f = m[p][i] * inv;
            x[i] = fma(-f, x[p], x[i]);
#pragma unroll
            for (int j = i; j < 8; ++j) m[i][j] = fma(-f, m[p][j], m[i][j]);
        }
    }
    if (lane < 8) {
#pragma unroll
        for (int p = 0; p < 8; ++p) Wb[8 * p + lane] = x[p];
    }
    return bad;
}

// One CTA per row i.
//   1. L_j = score of w_ij (the keys of ptq_sensitivity_order on this single row); perm = stable sort of the columns
//   2. A = Hinv[perm][:, perm] in shared memory, upper 8 x 8 tiles only; A = L D L^T, eight pivots at a time: warp 0
//      factorises the diagonal tile, the new rows are L_bb^-1 R and the trailing tiles C -= (D^-1 R_i)^T R_c, both on
//      the float64 MMA.  The rows of the next pivots are updated first; the other trailing tiles then run (warps 2..4)
//      under the next tile's chain.
//   3. under the same chain warp 1 runs the column loop on the eight columns just finished: q = quant(w_p),
//      w_j -= (w_p - q) A_pj / A_pp, A_p the row of the Eq.-12-updated matrix (Eq. 11).
//   4. codes, What and the order go out; row_loss[i] = 1/2 dw H dw^T
// Bound by latency: the chains of pivots (about 1200 clocks per eight) and the barriers between their steps, with three
// CTAs per SM to fill each other's gaps, which the packed triangle (70 KB at 128 columns, 132 KB as a square) and 128
// registers allow.  Reading Hinv as it lies, sixteen loads of a lane in flight, matters as much: an element at a time it
// was 163 us.  512 x 128: 977 us with one barrier and one rank-1 update of the whole triangle per pivot -> 140 us.
__global__ void __launch_bounds__(kPerRowThreads, 3) per_row_kernel(const float* __restrict__ W, int rows, int cols, int64_t ldw,
                                                                 const double* __restrict__ Hinv,
                                                                 const float* __restrict__ scale,
                                                                 const float* __restrict__ zero, int bits, int mode,
                                                                 int ascending, uint8_t* __restrict__ codes,
                                                                 float* __restrict__ What, int32_t* __restrict__ perm_rows,
                                                                 const double* __restrict__ H, double* __restrict__ row_loss,
                                                                 int32_t* status) {
    chained_begin();
    extern __shared__ __align__(16) unsigned char per_row_smem[];
    __shared__ double red[kPerRowWarps];
    const int n = cols, nf = (n + 7) >> 3, n8 = 8 * nf;
    double* tiles = reinterpret_cast<double*>(per_row_smem);
    double* w = tiles + (nf * (nf + 1) / 2) * 64;                  // [n8] weights in the row's own order
    double* dw = w + n8;                                           // [n8] scores, later w - What in original order
    double* dinv = dw + n8;                                        // [n8] 1 / pivot
    double* Wb = dinv + n8;                                        // [8][8] L_bb^-1
    double* us = Wb + 64;                                          // [8][8] rows of the diagonal tile / their pivots
    int32_t* perm = reinterpret_cast<int32_t*>(us + 64);           // [n8]
    int32_t* rank_of = perm + n8;                                  // [n8]
    auto tile = [&](int r, int c) { return tiles + ((c * (c + 1) >> 1) + r) * 64; };       // r <= c
    const int i = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int lq = lane >> 2, lr = lane & 3;
    const double maxq = (double)((1 << bits) - 1);
    const RowGrid rg = make_row_grid((double)scale[i], (double)zero[i], maxq);

    // 1. scores and order
    unsigned long long* key = reinterpret_cast<unsigned long long*>(dw);
    for (int j = tid; j < n; j += kPerRowThreads) {
        const double x = (double)W[(int64_t)i * ldw + j];
        double num = 0.0;
        if (mode == PTQ_SCORE_QERR || mode == PTQ_SCORE_ERR) {
            const double d = x - rg.sc * (quant_code_d(x, rg.sc, rg.zp, maxq) - rg.zp);
            num = d * d;
        } else if (mode == PTQ_SCORE_PRUNE || mode == PTQ_SCORE_W) {
            num = x * x;
        }
        if (mode == PTQ_SCORE_QERR || mode == PTQ_SCORE_PRUNE) num = num / (2.0 * Hinv[(int64_t)j * n + j]);
        key[j] = sortable_key(num) ^ (ascending ? ~0ull : 0ull);
    }
    __syncthreads();
    for (int j = tid; j < n; j += kPerRowThreads) {
        const unsigned long long kj = key[j];
        int rank = 0;
#pragma unroll 8
        for (int t = 0; t < n; ++t) rank += (key[t] > kj || (key[t] == kj && t < j)) ? 1 : 0;
        perm[rank] = j;
        rank_of[j] = rank;
        w[rank] = (double)W[(int64_t)i * ldw + j];
    }
    // padding up to a whole tile: identity, weight zero
    for (int p = n + tid; p < n8; p += kPerRowThreads) w[p] = 0.0;
    if (n < n8)
        for (int idx = tid; idx < nf * 64; idx += kPerRowThreads)
            tile(0, nf - 1)[idx] = (idx >> 6) == nf - 1 && ((idx >> 3) & 7) == (idx & 7) ? 1.0 : 0.0;
    __syncthreads();
    // 2. the row's own permuted inverse Hessian: rows of Hinv are read as they lie and scattered to their places
    // (up to sixteen loads of a lane in flight: four rows of four)
    for (int j0 = warp; j0 < n; j0 += 4 * kPerRowWarps) {
        double v[4][4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int j = j0 + u * kPerRowWarps, k = lane + 32 * q;
                v[u][q] = j < n && k < n ? __ldg(Hinv + (int64_t)j * n + k) : 0.0;
            }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = j0 + u * kPerRowWarps;
            const int a = j < n ? rank_of[j] : n;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int k = lane + 32 * q;
                const int c = k < n ? rank_of[k] : -1;
                if (c < a) continue;
                double* t = tile(a >> 3, c >> 3);
                t[(a & 7) * 8 + (c & 7)] = v[u][q];
                if ((a >> 3) == (c >> 3)) t[(c & 7) * 8 + (a & 7)] = v[u][q];
            }
        }
    }
    __syncthreads();
    // C -= (D^-1 R_r)^T R_c with the rows of pivot block b
    auto update_tile = [&](int b, int r, int c) {
        const double* tr = tile(b, r);
        const double* tc = tile(b, c);
        const double a0 = -(dinv[8 * b + lr] * tr[lr * 8 + lq]), a1 = -(dinv[8 * b + 4 + lr] * tr[(4 + lr) * 8 + lq]);
        double2* dst = reinterpret_cast<double2*>(tile(r, c)) + lane;
        double2 v = *dst;
        dmma_884(v.x, v.y, a0, tc[lr * 8 + lq]);
        dmma_884(v.x, v.y, a1, tc[(4 + lr) * 8 + lq]);
        *dst = v;
    };
    // 3. the column loop on columns 8 b .. 8 b + 7 (one warp; every lane takes the same decisions)
    auto column_loop = [&](int b) {
        const double* td = tile(b, b);
        us[lane] = td[lane] * dinv[8 * b + (lane >> 3)];
        us[lane + 32] = td[lane + 32] * dinv[8 * b + 4 + (lane >> 3)];
        __syncwarp();
        double v[8], lev[8];
#pragma unroll
        for (int p = 0; p < 8; ++p) v[p] = w[8 * b + p];
        double my_lev = 0.0, my_code = 0.0;
        if (sweep_chain8<false, 8>(v, lev, us, rg)) {
            // by the definition: code = clamp(rint(w / s) + z), level = code - z.  (For a zero-point that is no integer of
            // ordinary size, code and level cannot be had from one another.)
#pragma unroll
            for (int p = 0; p < 8; ++p) v[p] = w[8 * b + p];
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                const double code = quant_code_d(v[p], rg.sc, rg.zp, maxq), level = code - rg.zp;
                const double d = v[p] - rg.sc * level;
#pragma unroll
                for (int j = p + 1; j < 8; ++j) v[j] = fma(-d, us[p * 8 + j], v[j]);
                v[p] = d;
                my_lev = lane == p ? level : my_lev;
                my_code = lane == p ? code : my_code;
            }
        } else {
#pragma unroll
            for (int p = 0; p < 8; ++p) my_lev = lane == p ? lev[p] : my_lev;
            my_code = my_lev + rg.zp;
        }
#pragma unroll
        for (int p = 0; p < 8; ++p) v[p] *= dinv[8 * b + p];
        for (int c = 8 * (b + 1) + lane; c < n8; c += 32) {
            const double* tc = tile(b, c >> 3) + (c & 7);
            double acc = w[c];
#pragma unroll
            for (int p = 0; p < 8; ++p) acc = fma(-v[p], tc[8 * p], acc);
            w[c] = acc;
        }
        if (lane < 8 && 8 * b + lane < n) {
            const int j = perm[8 * b + lane];
            codes[(int64_t)i * n + j] = (uint8_t)(int)my_code;
            const float qf = (float)(rg.sc * my_lev);
            if (What) What[(int64_t)i * n + j] = qf;
            dw[j] = (double)W[(int64_t)i * ldw + j] - (double)qf;
            perm_rows[(int64_t)i * n + 8 * b + lane] = j;
        }
        __syncwarp();
    };

    for (int b = 0; b < nf; ++b) {
        if (warp == 0) {
            int bad = per_row_chain<false>(tile(b, b), Wb, dinv + 8 * b, lane);
            if (bad >= 0) bad = per_row_chain<true>(tile(b, b), Wb, dinv + 8 * b, lane);
            if (bad >= 0 && lane == 0) report(status, PTQ_ERR_NOT_SPD, 8 * b + bad, i);
        } else if (b > 0) {
            if (warp == 1) {
                column_loop(b - 1);
            } else {
                int t = warp - 2;                      // tiles (r, c), b < r <= c, dealt round-robin
                for (int c = b + 1; c < nf; ++c) {
                    for (; t < c - b; t += kPerRowWarps - 2) update_tile(b - 1, b + 1 + t, c);
                    t -= c - b;
                }
            }
        }
        __syncthreads();
        // new rows of this block
        const double a0 = Wb[lq * 8 + lr], a1 = Wb[lq * 8 + 4 + lr];
        for (int c = b + warp; c < nf; c += kPerRowWarps) {
            double* tc = tile(b, c);
            const double b0 = tc[lr * 8 + lq], b1 = tc[(4 + lr) * 8 + lq];
            double2 v = make_double2(0.0, 0.0);
            dmma_884(v.x, v.y, a0, b0);
            dmma_884(v.x, v.y, a1, b1);
            __syncwarp();
            reinterpret_cast<double2*>(tc)[lane] = v;
        }
        __syncthreads();
        // the rows of the next block first
        for (int c = b + 1 + warp; c < nf; c += kPerRowWarps) update_tile(b, b + 1, c);
        __syncthreads();
    }
    if (warp == 1) column_loop(nf - 1);
    __syncthreads();
    // 4. 1/2 dw H dw^T for this row: a warp per row of H, every lane keeps its columns' share
    if (H != nullptr && row_loss != nullptr) {
        double s = 0.0, dk[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) dk[q] = lane + 32 * q < n ? dw[lane + 32 * q] : 0.0;
#pragma unroll 4
        for (int a = warp; a < n; a += kPerRowWarps) {
            double t = 0.0;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                t = fma(lane + 32 * q < n ? __ldg(H + (int64_t)a * n + lane + 32 * q) : 0.0, dk[q], t);
            s = fma(dw[a], t, s);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if (lane == 0) red[warp] = s;
        __syncthreads();
        if (tid == 0) {
            double t = red[0];
#pragma unroll
            for (int k = 1; k < kPerRowWarps; ++k) t += red[k];
            row_loss[i] = 0.5 * t;
        }
    }
}

}  // namespace ptq
