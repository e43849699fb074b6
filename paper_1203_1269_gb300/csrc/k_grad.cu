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
#include "inv_diag.cuh"
#include "mixed_common.cuh"

namespace gp {

namespace {

constexpr int kThreads = 256;

template <typename T>
__device__ __forceinline__ T* tile_at(T* base, size_t stride, int t, int I, int J, int nt) {
    return base + (size_t)t * stride + (size_t)tile_index(I, J, nt) * GP_TILE_ELEMS;
}

// X_JJ = W_J = L_JJ^-1 in double (inv_diag.cuh), a CTA per 32 columns of it.
__global__ void __launch_bounds__(kInvThreads) k_inv_diag(Batch b, double* X) {
    grid_dependency();
    extern __shared__ double Lp[];                     // packed lower triangle, row r at r (r + 1) / 2
    __shared__ double dinv[GP_NB];
    __shared__ double Wk[2][kInvCols];
    const int J = blockIdx.x, t = blockIdx.y, c0 = kInvCols * blockIdx.z;
    if (b.st[t].status != GP_OK) return;
    const double* L = tile_at(b.A, b.inst_stride, t, J, J, b.nt);
    double* Xt = tile_at(X, b.inst_stride, t, J, J, b.nt);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int q = threadIdx.x; q < GP_TILE_ELEMS; q += kInvThreads) {
        const int r = q % GP_NB, c = q / GP_NB;
        if (r >= c && c >= c0) cp_async8(Lp + prow(r) + c, L + q);
        if (r < c0 && c >= c0 && c < c0 + kInvCols) Xt[q] = 0.0;
    }
    if ((int)threadIdx.x >= c0) dinv[threadIdx.x] = 1.0 / L[threadIdx.x * (GP_NB + 1)];
    cp_async_wait_all();
    __syncthreads();
    inv_columns(Lp, dinv, Wk, Xt, c0, warp, lane);
}

// Exponents of W_J's rows, |W_rc| < 2^E, into slot 2 of the factor's diagonal
// tile (the factor's own diagonal block is not needed any more).
__global__ void __launch_bounds__(GP_NB) k_row_exponents(Batch b, const double* X) {
    grid_dependency();
    const int J = blockIdx.x, t = blockIdx.y, r = threadIdx.x;
    if (b.st[t].status != GP_OK) return;
    const double* T = tile_at(X, b.inst_stride, t, J, J, b.nt) + r;
    unsigned m = 0;
#pragma unroll 16
    for (int c = 0; c < GP_NB; ++c) m = max(m, (unsigned)__double2hiint(T[(size_t)c * GP_NB]) & 0x7fffffffu);
    reinterpret_cast<int*>(tile_at(b.A, b.inst_stride, t, J, J, b.nt))[2 * GP_NB + r] = (int)(m >> 20) - 1022;
}

// Exponents of the columns of tiles (J, K), K = blockIdx.x, of `src`: |entry| <
// 2^E, into slot `slot` of the factor's diagonal tile (K, K).  A warp per four
// columns, 128 entries in a coalesced kilobyte each.
constexpr int kExpSplit = 4;
__global__ void __launch_bounds__(kThreads) k_col_exponents(Batch b, const double* src, int J, int slot) {
    grid_dependency();
    const int K = blockIdx.x, t = blockIdx.y;
    if (b.st[t].status != GP_OK) return;
    const double* T = tile_at(src, b.inst_stride, t, J, K, b.nt);
    int* out = reinterpret_cast<int*>(tile_at(b.A, b.inst_stride, t, K, K, b.nt)) + slot * GP_NB;
    const int lane = threadIdx.x & 31;
    constexpr int kCols = GP_NB / kExpSplit / (kThreads / 32);
    const int c0 = (GP_NB / kExpSplit) * blockIdx.z + kCols * (threadIdx.x >> 5);
    unsigned m[kCols];
#pragma unroll
    for (int c = 0; c < kCols; ++c) {
        m[c] = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            m[c] = max(m[c], (unsigned)__double2hiint(T[(size_t)(c0 + c) * GP_NB + 32 * u + lane]) & 0x7fffffffu);
    }
#pragma unroll
    for (int c = 0; c < kCols; ++c) {
        m[c] = __reduce_max_sync(0xffffffffu, m[c]);
        if (lane == 0) out[c0 + c] = (int)(m[c] >> 20) - 1022;
    }
}

// e = b - mu_hat a in column 1 of Z (w = L^-T e follows by the backward solve)
__global__ void k_residual_vec(Batch b, double* Z, size_t zs) {
    grid_dependency();
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
//
// A CTA takes a quarter of a tile (whole tiles left a last wave of 72 CTAs to
// themselves at n = 4064: FP64 pipes 85% busy on average, 54% of the time), and
// its sums go to the factor's memory, which nothing needs any more.
// G candidates share an element's powers, whose double-float logarithms and
// conversions are half of its cost; theta comes scaled from shared memory and
// exp(-S) from the assembly's table (11 double operations): FP64-bound, about
// d + 25 + (7 d + 14) / G double operations per element and candidate (16 d + 2 d
// + 30 each with CUDA's exp and a candidate at a time).  n = 1024, d = 6, T = 16:
// 2.12 -> 0.94 ms; n = 4064, T = 1: 2.11 -> 1.72 ms.
constexpr int kGradSplit = 4;

template <int DB, int G>
__global__ void __launch_bounds__(kThreads) k_grad_tiles(Batch b, const double* Ri, const double* Z, size_t zs,
                                                         ExpTab64 etab, const float2* e2tab) {
    grid_dependency();
    __shared__ double red[kThreads / 32][DB];
    __shared__ dfl tab[kExpTab];
    __shared__ ExpTab64 et;
    __shared__ double th[G][DB], nq[G];
    __shared__ int live[G];
    const int t0 = blockIdx.y * G, nt = b.nt, n = b.n, d = b.d;
    const int corr = b.corr;
    const bool matern = corr_is_matern(corr);
    const double cm = corr_theta_scale(corr);
    load_exp2_table(tab, e2tab);
    for (int q = threadIdx.x; q < (int)(sizeof(ExpTab64) / sizeof(double)); q += kThreads)
        reinterpret_cast<double*>(&et)[q] = reinterpret_cast<const double*>(&etab)[q];
    for (int q = threadIdx.x; q < G * DB; q += kThreads) {
        const int g = q / DB, k = q % DB;
        th[g][k] = (t0 + g < b.count && k < d) ? cm * b.theta[(size_t)(t0 + g) * d + k] : 0.0;
    }
    if (threadIdx.x < G) {
        live[threadIdx.x] = t0 + (int)threadIdx.x < b.count && b.st[t0 + threadIdx.x].status == GP_OK;
        if (live[threadIdx.x]) nq[threadIdx.x] = n / b.st[t0 + threadIdx.x].Q;
    }
    __syncthreads();
    int J = 0;
    {
        long long rem = blockIdx.x / kGradSplit;
        while (rem >= nt - J) { rem -= nt - J; ++J; }
    }
    const int I = J + (int)(blockIdx.x / kGradSplit - tile_index(J, J, nt));
    const int pmode = pow_mode(b.p);
    const dfl pd = df_from_double(b.p);
    // a thread's elements all lie in one row
    static_assert(kThreads % GP_NB == 0, "rows per thread");
    const int r = threadIdx.x % GP_NB, gi = I * GP_NB + r;
    double acc[G][DB], wi[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        wi[g] = (live[g] && gi < n) ? nq[g] * Z[(size_t)(t0 + g) * zs + (size_t)nt * GP_NB + gi] : 0.0;
#pragma unroll
        for (int k = 0; k < DB; ++k) acc[g][k] = 0.0;
    }
    constexpr int kCols = GP_NB / kGradSplit;
    const int c0 = kCols * (blockIdx.x % kGradSplit);
    for (int c = c0 + threadIdx.x / GP_NB; c < c0 + kCols; c += kThreads / GP_NB) {
        const int gj = J * GP_NB + c;
        if (gi >= n || gj >= n || gi <= gj) continue;
        double D[DB];
#pragma unroll
        for (int k = 0; k < DB; ++k) {
            D[k] = 0.0;
            if (k < d) {
                const double a = fabs(b.x[(size_t)gi * d + k] - b.x[(size_t)gj * d + k]);
                // |dx|^p for general p in double-float (FP64 pow is scarce here)
                D[k] = (matern || pmode == kPowOne) ? a
                                                    : (pmode == kPowTwo ? a * a
                                                                        : df_to_double_positive(df_powabs(df_from_positive(a), pmode, b.p, pd, tab)));
            }
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
            if (!live[g]) continue;
            const int t = t0 + g;
            const double m = tile_at(Ri, b.inst_stride, t, I, J, nt)[c * GP_NB + r] -
                             wi[g] * Z[(size_t)t * zs + (size_t)nt * GP_NB + gj];
            double s = 0.0, qp = m;
#pragma unroll
            for (int k = 0; k < DB; ++k)
                if (k < d) {
                    s = fma(th[g][k], D[k], s);
                    if (matern) qp *= matern_q(th[g][k] * D[k], corr);
                }
            const double mr = qp * exp_neg_tab64(s, et);
#pragma unroll
            for (int k = 0; k < DB; ++k)
                if (k < d) {
                    double dl = D[k];
                    if (corr == GP_CORR_MATERN32 || corr == GP_CORR_MATERN52) {
                        const double h = th[g][k] * D[k];
                        dl *= corr == GP_CORR_MATERN32 ? h / (1.0 + h) * cm
                                                       : h * (1.0 + h) / (3.0 + 3.0 * h + h * h) * cm;
                    }
                    acc[g][k] = fma(mr, dl, acc[g][k]);
                }
        }
    }
    // fixed-order block reduction of each candidate's d sums; both (i, j) and
    // (j, i), and the derivative's sign
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        if (!live[g]) continue;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < DB; ++k) {
            double v = acc[g][k];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            if (lane == 0) red[wp][k] = v;
        }
        __syncthreads();
        if (threadIdx.x < d) {
            double v = 0.0;
            for (int i = 0; i < kThreads / 32; ++i) v += red[i][threadIdx.x];
            b.A[(size_t)(t0 + g) * b.inst_stride + (size_t)blockIdx.x * d + threadIdx.x] = -2.0 * v;
        }
    }
}

// grad[t][k] = the sum of the tile parts' sums, in a fixed order (a warp per k);
// NaN where the likelihood itself failed (status: the finalize kernel's, which
// also flags Q = 0).  A candidate that a kernel of the inverse gave up after
// finalize has its status and -2logL corrected here.
__global__ void k_grad_reduce(Batch b, int parts, int* status, double* nll, double* grad) {
    grid_dependency();
    const int t = blockIdx.x, d = b.d;
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (k >= d) return;
    if (b.st[t].status != GP_OK || status[t] != GP_OK) {
        const double nan = __longlong_as_double(0x7ff8000000000000LL);
        if (lane == 0) grad[(size_t)t * d + k] = nan;
        if (threadIdx.x == 0 && b.st[t].status == GP_ETIMEOUT && status[t] != GP_ETIMEOUT) {
            status[t] = GP_ETIMEOUT;
            nll[t] = nan;
        }
        return;
    }
    const double* partial = b.A + (size_t)t * b.inst_stride;
    double v = 0.0;
    for (int q = lane; q < parts; q += 32) v += partial[(size_t)q * d + k];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) grad[(size_t)t * d + k] = v;
}

}  // namespace

cudaError_t launch_grad(const Batch& b, double* Z, size_t zs, double* X, double* Ri, int* status, double* nll,
                        double* grad, cudaStream_t s, int* kernels) {
    const int nt = b.nt;
    int k = 0;
    launch_chained(ahead_f64(b), k_residual_vec, b.count, kThreads, 0, s, b, Z, zs);
    ++k;
    cudaError_t e = launch_backward_solve(b, Z, zs, 1, s);   // w = L^-T (b - mu a), double factor
    if (e != cudaSuccess) return e;
    k += solve_f64_launches(nt, true);
    {
        const size_t smem = (size_t)kPackedTri * sizeof(double);
        static std::atomic<size_t> attr[kMaxDevices];
        e = raise_smem_limit(k_inv_diag, smem, attr);
        if (e != cudaSuccess) return e;
        launch_chained(ahead_f64(b), k_inv_diag, dim3(nt, b.count, GP_NB / kInvCols), kInvThreads, smem, s, b, X);
        launch_chained(ahead_f64(b), k_row_exponents, dim3(nt, b.count), GP_NB, 0, s, b, X);
        k += 2;
    }
    for (int J = 0; J < nt; ++J) {
        if (J > 0) {
            launch_chained(ahead_f64(b), k_col_exponents, dim3(J, b.count, kExpSplit), kThreads, 0, s, b, Ri, J, 1);
            e = launch_inverse_apply(b, J, X, Ri, s);
            if (e != cudaSuccess) return e;
            k += 2;
        }
        launch_chained(ahead_f64(b), k_col_exponents, dim3(J + 1, b.count, kExpSplit), kThreads, 0, s, b, X, J, 0);
        e = launch_inverse_update(b, J, X, Ri, s);
        if (e != cudaSuccess) return e;
        k += 2;
    }
    const int ntiles = (int)packed_tiles(nt);
    ExpTab64 et;
    exp_tab64_fill(et);
    // four candidates an element where their CTAs fill most of the SMs
    const int parts = kGradSplit * ntiles;
    const int G = (long long)ntiles * ((b.count + 3) / 4) * 4 >= 3LL * device_sms() && b.count > 1 ? 4 : 1;
    const dim3 grid(parts, (b.count + G - 1) / G);
#define GP_GRAD_TILES(DB)                                                                                   \
    (G == 4 ? launch_chained(ahead_f64(b), k_grad_tiles<DB, 4>, grid, kThreads, 0, s, b, Ri, Z, zs, et, exp2_table()) \
            : launch_chained(ahead_f64(b), k_grad_tiles<DB, 1>, grid, kThreads, 0, s, b, Ri, Z, zs, et, exp2_table()))
    if (b.d <= 4)      GP_GRAD_TILES(4);
    else if (b.d <= 8) GP_GRAD_TILES(8);
    else               GP_GRAD_TILES(16);
#undef GP_GRAD_TILES
    ++k;
    launch_chained(ahead_f64(b), k_grad_reduce, b.count, 32 * 16, 0, s, b, parts, status, nll, grad);
    ++k;
    if (kernels) *kernels = k;
    return cudaGetLastError();
}

}  // namespace gp
