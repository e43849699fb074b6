// k_panel_f64.cu -- one block column of the double-precision Cholesky in
// four 32-column steps (matrices of three block columns and more):
//   inner  columns 32 s .. 32 s + 31 take the products of the steps before
//          them, on the tensor cores (k_update_tc.cu)           s > 0
//   diag   the 32 x 32 block is factored                         one CTA per instance
//   solve  X L_ss^T = A for every row below it                   eight rows a warp
// On this GPU a double multiply-add takes a warp 64 cycles, issue and latency
// alike, so what stays on the FP64 pipe is kept to the 32-wide triangles: a
// quarter of the panel's multiply-adds, spread over all SMs by rows.  A block
// column is bound by its chain: four 32-pivot sweeps of about 12 us, four
// solves of 168 dependent double operations (6 us) and three inner updates.
// Measured, one candidate at n = 4064: 190 us a block column (0.4 ms for the
// 128-pivot sweep and 0.35 ms for the tile solve on the FP64 pipe alone); the
// double fit 29.8 -> 13.6 ms, twelve candidates 55 -> 37.3 ms.
#include "gp_internal.cuh"

namespace gp {

namespace {

constexpr int kB = kPanelStep;                 // 32
constexpr int kThreads = 128;
constexpr int kWarps = kThreads / 32;
constexpr int kUnit = 8;                       // rows a warp solves at a time

__device__ __forceinline__ double* inst_tile(const Batch& b, int t, int I, int J) {
    return b.A + (size_t)t * b.inst_stride + (size_t)tile_index(I, J, b.nt) * GP_TILE_ELEMS;
}

// 1 / sqrt(a) for a normal a > 0: a float seed (2^-20), then y = y0 (1 + e/2 +
// 3 e^2 / 8), e = 1 - a y0^2 (the next term, 5 e^3 / 16, is below 2^-58): five
// double operations where sqrt and a division take 1360 cycles.
__device__ __forceinline__ double rsqrt_f64(double a) {
    const int hi = __double2hiint(a), lo = __double2loint(a);
    const int e = (hi >> 20) - 1023;
    const int h = e >> 1;                               // a = m 2^(2h), m in [1, 4)
    const unsigned fb = (unsigned)((e - 2 * h + 127) << 23) | ((unsigned)(hi & 0xfffff) << 3) | ((unsigned)lo >> 29);
    float s;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(__uint_as_float(fb)));
    const unsigned sb = __float_as_uint(s);              // in (1/2, 1]
    const int ye = (int)(sb >> 23) - 127 + 1023 - h;
    const double y0 = __hiloint2double((ye << 20) | (int)((sb & 0x7fffff) >> 3), (int)(sb << 29));
    const double t = a * y0;
    const double err = fma(-t, y0, 1.0);
    const double p = fma(err, 0.375, 0.5);
    return fma(y0 * err, p, y0);
}

// L_ss of sub-block s.  Thread (lane, warp) holds row lane, columns warp + 4 j;
// the warp that owns column c takes its pivot and publishes the finished
// column, one barrier a column.
__global__ void __launch_bounds__(kThreads) k_diag32_f64(Batch b, int J, int s) {
    __shared__ double Ls[kB][kB + 1];              // Ls[c][r]
    __shared__ int failed;
    const int t = blockIdx.x;
    if (b.st[t].status != GP_OK) return;
    double* T = inst_tile(b, t, J, J) + (size_t)(kB * s) * GP_NB + kB * s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double a[kB / kWarps];
#pragma unroll
    for (int j = 0; j < kB / kWarps; ++j) {
        const int k = warp + kWarps * j;
        a[j] = lane >= k ? T[(size_t)k * GP_NB + lane] : 0.0;
    }
    if (threadIdx.x == 0) failed = -1;
    __syncthreads();
    // pivot and finished column c, held in a[c / 4] of warp c % 4
    auto finish = [&](double& v, int c) {
        const double piv = __shfl_sync(0xffffffffu, v, c);
        double y = 0.0;
        if (!(piv > 0.0) || !isfinite(piv)) {
            if (lane == 0 && failed < 0) failed = c;   // the sweep goes on with zeros
        } else if (piv < 0x1p-1000) {
            y = 1.0 / sqrt(piv);
        } else {
            y = rsqrt_f64(piv);
        }
        v *= y;
        Ls[c][lane] = v;
    };
    if (warp == 0) finish(a[0], 0);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kB / kWarps; ++j)
#pragma unroll
        for (int q = 0; q < kWarps; ++q) {
            const int c = kWarps * j + q;
            const double lr = Ls[c][lane];
            // column c + 1 first, and its pivot
            constexpr int kLast = kB / kWarps - 1;
            const int jn = q == kWarps - 1 ? j + 1 : j, qn = (q + 1) % kWarps;
            if (warp == qn && jn <= kLast) {
                const int jc = jn <= kLast ? jn : kLast;
                a[jc] = fma(-lr, Ls[c][c + 1 < kB ? c + 1 : c], a[jc]);
                finish(a[jc], c + 1);
            }
#pragma unroll
            for (int i = j; i < kB / kWarps; ++i) {
                const int k = warp + kWarps * i;
                if (k > c && !(warp == qn && i == jn)) a[i] = fma(-lr, Ls[c][k], a[i]);
            }
            __syncthreads();
        }
    if (failed >= 0) {
        if (threadIdx.x == 0) {
            b.st[t].status = GP_ENOTPD;
            b.st[t].fail_col = J * GP_NB + kB * s + failed;
        }
        return;
    }
#pragma unroll
    for (int j = 0; j < kB / kWarps; ++j) {
        const int k = warp + kWarps * j;
        if (lane >= k) T[(size_t)k * GP_NB + lane] = a[j];
    }
}

// Rows below sub-block s, `per_warp` groups of eight rows a warp: lane (row
// rr, kq) holds columns kq + 4 j of its row; x_c goes from its owner to the
// row's other lanes by a shuffle, and column c leaves the columns after it in
// the order of c.
__global__ void __launch_bounds__(kThreads) k_solve32_f64(Batch b, int J, int s, int units, int per_warp) {
    __shared__ double Ls[kB][kB + 1];
    __shared__ double inv[kB];
    const int t = blockIdx.y;
    if (b.st[t].status != GP_OK) return;
    const double* T = inst_tile(b, t, J, J) + (size_t)(kB * s) * GP_NB + kB * s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rr = lane & 7, kq = lane >> 3;
    int u = (blockIdx.x * kWarps + warp) * per_warp;
    const int end = u + per_warp < units ? u + per_warp : units;
    auto rows = [&](int unit) {
        const int row = kB * (s + 1) + kUnit * unit;
        return inst_tile(b, t, J + (row >> 7), J) + (size_t)(kB * s) * GP_NB + (row & 127) + rr;
    };
    double a[kB / 4], nx[kB / 4];
    if (u < end) {
        const double* p = rows(u);
#pragma unroll
        for (int j = 0; j < kB / 4; ++j) nx[j] = p[(size_t)(kq + 4 * j) * GP_NB];
    }
    for (int q = threadIdx.x; q < kB * kB; q += kThreads) {
        const int r = q % kB, c = q / kB;
        if (r >= c) Ls[c][r] = T[(size_t)c * GP_NB + r];
    }
    __syncthreads();
    if (threadIdx.x < kB) inv[threadIdx.x] = 1.0 / Ls[threadIdx.x][threadIdx.x];
    __syncthreads();
    for (; u < end; ++u) {
        double* p = rows(u);
#pragma unroll
        for (int j = 0; j < kB / 4; ++j) a[j] = nx[j];
        if (u + 1 < end) {
            const double* pn = rows(u + 1);
#pragma unroll
            for (int j = 0; j < kB / 4; ++j) nx[j] = pn[(size_t)(kq + 4 * j) * GP_NB];
        }
#pragma unroll
        for (int c = 0; c < kB; ++c) {
            const int jc = c / 4, qc = c % 4;
            const double x = __shfl_sync(0xffffffffu, a[jc], 8 * qc + rr) * inv[c];
            if (qc < 3) {
                const double v = fma(-x, Ls[c][kq + 4 * jc], a[jc]);
                a[jc] = kq > qc ? v : (kq == qc ? x : a[jc]);
            } else if (kq == 3) {
                a[jc] = x;
            }
#pragma unroll
            for (int j = jc + 1; j < kB / 4; ++j) a[j] = fma(-x, Ls[c][kq + 4 * j], a[j]);
        }
#pragma unroll
        for (int j = 0; j < kB / 4; ++j) p[(size_t)(kq + 4 * j) * GP_NB] = a[j];
    }
}

// log|R| = 2 sum log L_ii over the factor's diagonal (padded rows give 0),
// one CTA per instance, in a fixed order.
__global__ void __launch_bounds__(256) k_logdet_f64(Batch b) {
    __shared__ double red[8];
    const int t = blockIdx.x;
    if (b.st[t].status != GP_OK) return;
    double v = 0.0;
    for (int i = threadIdx.x; i < b.nt * GP_NB; i += 256) {
        const int r = i & (GP_NB - 1);
        v += log(inst_tile(b, t, i >> 7, i >> 7)[r * GP_NB + r]);
    }
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double sum = 0.0;
        for (int w = 0; w < 8; ++w) sum += red[w];
        b.st[t].logdet = 2.0 * sum;
    }
}

}  // namespace

// Kernels of launch_panel_f64.
int panel_f64_launches(int nt, int J) { return J + 1 < nt ? 11 : 10; }

cudaError_t launch_panel_f64(const Batch& b, int J, cudaStream_t st) {
    const int sms = device_sms();
    for (int s = 0; s < GP_NB / kB; ++s) {
        if (s > 0) {
            cudaError_t e = launch_update_f64_inner(b, J, s, st);
            if (e != cudaSuccess) return e;
        }
        k_diag32_f64<<<b.count, kThreads, 0, st>>>(b, J, s);
        const int units = ((b.nt - J) * GP_NB - kB * (s + 1)) / kUnit;
        if (units > 0) {
            const long long warps = (long long)sms * 8;      // two CTAs an SM
            const int per_warp = (int)(((long long)units * b.count + warps - 1) / warps);
            const int grid = (units + kWarps * per_warp - 1) / (kWarps * per_warp);
            k_solve32_f64<<<dim3(grid, b.count), kThreads, 0, st>>>(b, J, s, units, per_warp);
        }
    }
    return cudaGetLastError();
}

cudaError_t launch_logdet_f64(const Batch& b, cudaStream_t st) {
    k_logdet_f64<<<b.count, 256, 0, st>>>(b);
    return cudaGetLastError();
}

}  // namespace gp
