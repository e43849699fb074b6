// k_grad.cu -- gradient of -2 log L (eq. 4) with respect to theta for a
// batch of candidates factored by the FP64 path.
//
//   d(-2logL)/dtheta_k = tr(R^-1 dR_k) - (n / Q) w' dR_k w
//                      = sum_{i != j} M_ij R_ij dlog rho_k(x_i, x_j),
//   M = R^-1 - (n / Q) w w',  w = R^-1 (Y - 1 mu_hat),
//
// from d log|R| = tr(R^-1 dR) and dQ = -w' dR w (mu_hat minimises Q); dR_k
// is zero on the diagonal (the nugget and the unit diagonal do not depend on
// theta).  -2logL and w come from the IEEE-double factor, and so do X = L^-1
// and R^-1 = X'X, formed on the tensor cores by rows of X (twice the
// factorisation's n^3/6 multiply-adds):
//   X_JJ = W_J = L_JJ^-1 (double, in shared memory, all J at once), then for
//   J = 0, 1, ...
//     X_JK = -W_J S_JK                       K < J   (S_IK = sum_{M<I} L_IM X_MK)
//     S_IK += L_IJ X_JK (I > J),  (R^-1)_IK += X_JI' X_JK (I <= J),   K <= J
// as exact digit products added in double (k_update_tc.cu; a tile of S turns
// into the tile of R^-1 once its row is consumed).  Every step updates every
// tile it can, so a single candidate fills the GPU.  One pass over the lower
// tiles then recomputes R_ij (powers in double-float, as the assembly takes
// them) and dlog rho, reducing d partial sums per tile that a last kernel
// adds in a fixed order.
//
// The inverse in double-float multiply-adds on the FP32 pipes, along the tile
// diagonals of X, took 36.6 ms of the gradient's 49 at n = 4064, T = 1.
#include "corr.cuh"
#include "gp_internal.cuh"

namespace gp {

namespace {

constexpr int kThreads = 256;

template <typename T>
__device__ __forceinline__ T* tile_at(T* base, size_t stride, int t, int I, int J, int nt) {
    return base + (size_t)t * stride + (size_t)tile_index(I, J, nt) * GP_TILE_ELEMS;
}

// X_JJ = L_JJ^-1 (lower; zeros above the diagonal), one CTA per (J, instance),
// in double: row i of W from rows j < i, W_ij = -(1/L_ii) sum_{k=j}^{i-1} L_ik W_kj.
// Dynamic smem: L and W as packed lower triangles (row r at r (r + 1) / 2).
constexpr int kPackedTri = GP_NB * (GP_NB + 1) / 2;
__device__ __forceinline__ int prow(int r) { return r * (r + 1) / 2; }

__global__ void __launch_bounds__(kThreads) k_inv_diag(Batch b, double* X) {
    extern __shared__ double sm[];
    double* Lp = sm;
    double* Wp = sm + kPackedTri;
    __shared__ double dinv[GP_NB];
    const int J = blockIdx.x, t = blockIdx.y;
    if (b.st[t].status != GP_OK) return;
    const double* L = tile_at(b.A, b.inst_stride, t, J, J, b.nt);
    for (int q = threadIdx.x; q < GP_TILE_ELEMS; q += kThreads) {
        const int r = q % GP_NB, c = q / GP_NB;
        if (r >= c) {
            const double l = L[q];
            Lp[prow(r) + c] = l;
            Wp[prow(r) + c] = 0.0;
            if (r == c) dinv[r] = 1.0 / l;    // one division per pivot
        }
    }
    __syncthreads();
    for (int i = 0; i < GP_NB; ++i) {
        const double inv = dinv[i];
        for (int j = threadIdx.x; j < i; j += kThreads) {
            double s = 0.0;
            for (int k = j; k < i; ++k) s = fma(Lp[prow(i) + k], Wp[prow(k) + j], s);
            Wp[prow(i) + j] = -inv * s;
        }
        if (threadIdx.x == 0) Wp[prow(i) + i] = inv;
        __syncthreads();
    }
    double* Xt = tile_at(X, b.inst_stride, t, J, J, b.nt);
    for (int q = threadIdx.x; q < GP_TILE_ELEMS; q += kThreads) {
        const int r = q % GP_NB, c = q / GP_NB;
        Xt[q] = (r >= c) ? Wp[prow(r) + c] : 0.0;
    }
    // the exponents of W's rows, |W_rc| < 2^E, into the factor's diagonal tile
    // (its slot 2; the factor's own diagonal block is not needed any more)
    if (threadIdx.x < GP_NB) {
        const int r = threadIdx.x;
        unsigned m = 0;
        for (int c = 0; c <= r; ++c) m = max(m, (unsigned)__double2hiint(Wp[prow(r) + c]) & 0x7fffffffu);
        reinterpret_cast<int*>(tile_at(b.A, b.inst_stride, t, J, J, b.nt))[2 * GP_NB + r] = (int)(m >> 20) - 1022;
    }
}

// Exponents of the columns of tiles (J, K), K = blockIdx.x, of `src`: |entry| <
// 2^E, into slot `slot` of the factor's diagonal tile (K, K).  A warp per
// column, its 128 entries in one coalesced kilobyte.
__global__ void __launch_bounds__(kThreads) k_col_exponents(Batch b, const double* src, int J, int slot) {
    const int K = blockIdx.x, t = blockIdx.y;
    if (b.st[t].status != GP_OK) return;
    const double* T = tile_at(src, b.inst_stride, t, J, K, b.nt);
    int* out = reinterpret_cast<int*>(tile_at(b.A, b.inst_stride, t, K, K, b.nt)) + slot * GP_NB;
    const int lane = threadIdx.x & 31;
#pragma unroll 4
    for (int c = threadIdx.x >> 5; c < GP_NB; c += kThreads / 32) {
        unsigned m = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            m = max(m, (unsigned)__double2hiint(T[(size_t)c * GP_NB + 32 * u + lane]) & 0x7fffffffu);
        m = __reduce_max_sync(0xffffffffu, m);
        if (lane == 0) out[c] = (int)(m >> 20) - 1022;
    }
}

// e = b - mu_hat a in column 1 of Z (w = L^-T e follows by the backward solve)
__global__ void k_residual_vec(Batch b, double* Z, size_t zs) {
    const int t = blockIdx.x;
    const InstState st = b.st[t];
    if (st.status != GP_OK) return;
    const int npad = b.nt * GP_NB;
    double* z0 = Z + (size_t)t * zs;
    double* z1 = z0 + npad;
    for (int i = threadIdx.x; i < npad; i += blockDim.x) z1[i] = fma(-st.mu, z0[i], z1[i]);
}

// Partial sums of sum_{i != j} M_ij R_ij dlog rho_k over lower tile
// q = blockIdx.x (both (i, j) and (j, i): twice the strictly lower part).
// D_k = |dx_k|^p (power-exponential) or |dx_k| (Matern) is taken once per
// element and serves both R_ij and its derivative:
//   dlog rho_k / dtheta_k = -D_k                       (eq. 2, Matern 1/2)
//                         = -h / (1 + h) c D_k          (3/2, h = c theta_k D_k)
//                         = -h (1 + h) / (3 + 3h + h^2) c D_k   (5/2)
template <int DB>
__global__ void __launch_bounds__(kThreads) k_grad_tiles(Batch b, const double* Ri, const double* Z, size_t zs,
                                                         double* partial, int ntiles) {
    __shared__ double red[kThreads / 32][DB];
    __shared__ dfl tab[kExpTab];
    fill_exp2_table(tab);
    __syncthreads();
    const int t = blockIdx.y, nt = b.nt, n = b.n, d = b.d;
    const InstState st = b.st[t];
    if (st.status != GP_OK) return;
    int J = 0;
    {
        long long rem = blockIdx.x;
        while (rem >= nt - J) { rem -= nt - J; ++J; }
    }
    const int I = J + (int)(blockIdx.x - tile_index(J, J, nt));
    const double* R1 = tile_at(Ri, b.inst_stride, t, I, J, nt);
    const int pmode = pow_mode(b.p);
    const dfl pd = df_from_double(b.p);
    const double* w = Z + (size_t)t * zs + (size_t)nt * GP_NB;
    const double* th = b.theta + (size_t)t * d;
    const double nq = n / st.Q;
    const int corr = b.corr;
    const bool matern = corr_is_matern(corr);
    const double cm = corr_theta_scale(corr);
    double acc[DB];
#pragma unroll
    for (int k = 0; k < DB; ++k) acc[k] = 0.0;
    for (int q = threadIdx.x; q < GP_TILE_ELEMS; q += kThreads) {
        const int r = q % GP_NB, c = q / GP_NB;
        const int gi = I * GP_NB + r, gj = J * GP_NB + c;
        if (gi >= n || gj >= n || gi <= gj) continue;
        const double m = R1[q] - nq * w[gi] * w[gj];
        double D[DB], h[DB];
        double s = 0.0, qp = 1.0;
#pragma unroll
        for (int k = 0; k < DB; ++k) {
            D[k] = 0.0;
            h[k] = 0.0;
            if (k < d) {
                const double a = fabs(b.x[(size_t)gi * d + k] - b.x[(size_t)gj * d + k]);
                // |dx|^p for general p in double-float (FP64 pow is scarce here)
                D[k] = (matern || pmode == kPowOne) ? a
                                                    : (pmode == kPowTwo ? a * a
                                                                        : df_to_double(df_powabs(df_from_double(a), pmode, b.p, pd, tab)));
                h[k] = cm * th[k] * D[k];
                s += h[k];
                if (matern) qp *= matern_q(h[k], corr);
            }
        }
        const double mr = 2.0 * m * qp * exp(-s);
#pragma unroll
        for (int k = 0; k < DB; ++k) {
            if (k < d) {
                double dl = -D[k];
                if (corr == GP_CORR_MATERN32) dl = -h[k] / (1.0 + h[k]) * cm * D[k];
                if (corr == GP_CORR_MATERN52) dl = -h[k] * (1.0 + h[k]) / (3.0 + 3.0 * h[k] + h[k] * h[k]) * cm * D[k];
                acc[k] = fma(mr, dl, acc[k]);
            }
        }
    }
    // fixed-order block reduction of the d sums
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < DB; ++k) {
        double v = acc[k];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) red[wp][k] = v;
    }
    __syncthreads();
    if (threadIdx.x < d) {
        double v = 0.0;
        for (int i = 0; i < kThreads / 32; ++i) v += red[i][threadIdx.x];
        partial[((size_t)t * ntiles + blockIdx.x) * d + threadIdx.x] = v;
    }
}

// grad[t][k] = sum over tiles, in tile order; NaN where the likelihood
// itself failed (status: the finalize kernel's, which also flags Q = 0)
__global__ void k_grad_reduce(Batch b, const double* partial, int ntiles, const int* status, double* grad) {
    const int t = blockIdx.x, d = b.d;
    const int k = threadIdx.x;
    if (k >= d) return;
    if (b.st[t].status != GP_OK || status[t] != GP_OK) {
        grad[(size_t)t * d + k] = __longlong_as_double(0x7ff8000000000000LL);
        return;
    }
    double v = 0.0;
    for (int q = 0; q < ntiles; ++q) v += partial[((size_t)t * ntiles + q) * d + k];
    grad[(size_t)t * d + k] = v;
}

}  // namespace

cudaError_t launch_grad(const Batch& b, double* Z, size_t zs, double* X, double* Ri, double* partial,
                        const int* status, double* grad, cudaStream_t s, int* kernels) {
    const int nt = b.nt;
    int k = 0;
    k_residual_vec<<<b.count, kThreads, 0, s>>>(b, Z, zs);
    ++k;
    cudaError_t e = launch_backward_solve(b, Z, zs, 1, s);   // w = L^-T (b - mu a), double factor
    if (e != cudaSuccess) return e;
    k += solve_f64_launches(nt, true);
    {
        const size_t smem = (size_t)2 * kPackedTri * sizeof(double);
        static std::atomic<size_t> attr[kMaxDevices];
        e = raise_smem_limit(k_inv_diag, smem, attr);
        if (e != cudaSuccess) return e;
        k_inv_diag<<<dim3(nt, b.count), kThreads, smem, s>>>(b, X);
        ++k;
    }
    for (int J = 0; J < nt; ++J) {
        if (J > 0) {
            k_col_exponents<<<dim3(J, b.count), kThreads, 0, s>>>(b, Ri, J, 1);
            e = launch_inverse_apply(b, J, X, Ri, s);
            if (e != cudaSuccess) return e;
            k += 2;
        }
        k_col_exponents<<<dim3(J + 1, b.count), kThreads, 0, s>>>(b, X, J, 0);
        e = launch_inverse_update(b, J, X, Ri, s);
        if (e != cudaSuccess) return e;
        k += 2;
    }
    const int ntiles = (int)packed_tiles(nt);
    if (b.d <= 4)
        k_grad_tiles<4><<<dim3(ntiles, b.count), kThreads, 0, s>>>(b, Ri, Z, zs, partial, ntiles);
    else if (b.d <= 8)
        k_grad_tiles<8><<<dim3(ntiles, b.count), kThreads, 0, s>>>(b, Ri, Z, zs, partial, ntiles);
    else
        k_grad_tiles<16><<<dim3(ntiles, b.count), kThreads, 0, s>>>(b, Ri, Z, zs, partial, ntiles);
    ++k;
    k_grad_reduce<<<b.count, 64, 0, s>>>(b, partial, ntiles, status, grad);
    ++k;
    if (kernels) *kernels = k;
    return cudaGetLastError();
}

}  // namespace gp
