// inv_diag.cuh -- W = L^-1 of a 128 x 128 diagonal block in double, for the
// gradient (k_grad.cu) and the kriging variance (k_var_tc.cu).  File-local (an
// anonymous namespace) to each including translation unit.
#pragma once

#include "gp_internal.cuh"

namespace gp {

namespace {

// W = L^-1 (lower; zeros above the diagonal), a CTA per 32 columns of it (their
// rows above are zero): lane = column, warp w holds rows
// c0 + w + 4 i of acc_ij = sum_{m<k} L_im W_mj in registers.  Step k finishes row
// k (W_kj = -acc_kj / L_kk, W_kk = 1 / L_kk), one barrier, and adds its term to the
// rows after it.  Four rows are one iteration of a loop (the rows move down
// one register as they finish), in forms for up to 31, 23, 15 and 7 rows left.
// 0.13 ms for every block of n = 4064 at once (0.45 ms with one CTA a block
// and a dependent sum per entry).
constexpr int kPackedTri = GP_NB * (GP_NB + 1) / 2;
constexpr int kInvThreads = 128;
constexpr int kInvWarps = kInvThreads / 32;
constexpr int kInvCols = 32;
constexpr int kInvRows = GP_NB / kInvWarps;            // rows of a warp
__device__ __forceinline__ int prow(int r) { return r * (r + 1) / 2; }

// Rows k = k0 .. k0 + 31, or up to row 127 where LEFT rows of a warp are left.
template <int LEFT>
__device__ __forceinline__ void inv_rows(double (&acc)[kInvRows], const double* Lp, const double* dinv,
                                         double (*Wk)[kInvCols], double* Xt, int k0, int c0, int warp, int lane) {
#pragma unroll 1
    for (int g = 0; g < 8; ++g) {
#pragma unroll
        for (int q = 0; q < kInvWarps; ++q) {
            const int k = k0 + kInvWarps * g + q;
            if (warp == q) {
                const double w = c0 + lane == k ? dinv[k] : -dinv[k] * acc[0];
                Wk[k & 1][lane] = w;
                Xt[(size_t)(c0 + lane) * GP_NB + k] = w;
            }
            __syncthreads();
            const double w = Wk[k & 1][lane];
            if (warp > q) acc[0] = fma(Lp[prow(k - q + warp) + k], w, acc[0]);
#pragma unroll
            for (int i = 1; i <= LEFT; ++i) {
                const int r = k - q + warp + kInvWarps * i;
                if (i <= LEFT - 7 || r < GP_NB) acc[i] = fma(Lp[prow(r) + k], w, acc[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < LEFT; ++i) acc[i] = acc[i + 1];
    }
}

// Columns c0 .. c0 + 31 of W, rows c0 .. 127, into the column-major tile Xt.
// Lp: L's packed lower triangle, dinv: 1 / L_kk (both from row c0 on).
__device__ __forceinline__ void inv_columns(const double* Lp, const double* dinv, double (*Wk)[kInvCols], double* Xt,
                                            int c0, int warp, int lane) {
    double acc[kInvRows];
#pragma unroll
    for (int i = 0; i < kInvRows; ++i) acc[i] = 0.0;
    if (c0 <= 0) inv_rows<31>(acc, Lp, dinv, Wk, Xt, 0, c0, warp, lane);
    if (c0 <= 32) inv_rows<23>(acc, Lp, dinv, Wk, Xt, 32, c0, warp, lane);
    if (c0 <= 64) inv_rows<15>(acc, Lp, dinv, Wk, Xt, 64, c0, warp, lane);
    inv_rows<7>(acc, Lp, dinv, Wk, Xt, 96, c0, warp, lane);
}

}  // namespace

}  // namespace gp
