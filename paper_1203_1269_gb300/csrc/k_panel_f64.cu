// k_panel_f64.cu -- one block column of the double-precision Cholesky in
// four 32-column steps:
//   inner  columns 32 s .. 32 s + 31 take the products of the steps before
//          them, on the tensor cores (k_update_tc.cu)           s > 0
//   diag   the 32 x 32 block is factored                         one CTA per instance
//   solve  X L_ss^T = A for every row below it                   a few rows a warp
// Matrices of up to two block columns keep IEEE operations throughout, in the
// order of the unblocked loops (below).
// On this GPU a double multiply-add takes a warp 64 cycles, issue and latency
// alike, so what stays on the FP64 pipe is kept to the 32-wide triangles: a
// quarter of the panel's multiply-adds, spread over all SMs by rows.  A block
// column is bound by its chain: four 32-pivot sweeps of about 12 us (17 us
// with a warp's terms all taken in the step of their column, 22 us as
// unrolled code), four solves of about 8 us and three inner updates of 8 to
// 13 us.  Measured, one candidate at n = 4064: 165 us a block column (0.4 ms
// for a 128-pivot sweep in one CTA and 0.35 ms for the tile solve, on the FP64
// pipe alone); the double fit 29.8 -> 10.5 ms with the solves after it.
#include "mixed_common.cuh"

namespace gp {

namespace {

constexpr int kB = kPanelStep;                 // 32
constexpr int kThreads = 128;
constexpr int kWarps = kThreads / 32;

__device__ __forceinline__ double* inst_tile(const Batch& b, int t, int I, int J) {
    return b.A + (size_t)t * b.inst_stride + (size_t)tile_index(I, J, b.nt) * GP_TILE_ELEMS;
}

// 1 / sqrt(a) to about 2^-20 for a normal a > 0, from the float instruction.
__device__ __forceinline__ double rsqrt_seed(double a) {
    const int hi = __double2hiint(a), lo = __double2loint(a);
    const int e = (hi >> 20) - 1023;
    const int h = e >> 1;                               // a = m 2^(2h), m in [1, 4)
    const unsigned fb = (unsigned)((e - 2 * h + 127) << 23) | ((unsigned)(hi & 0xfffff) << 3) | ((unsigned)lo >> 29);
    float s;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(__uint_as_float(fb)));
    const unsigned sb = __float_as_uint(s);              // in (1/2, 1]
    const int ye = (int)(sb >> 23) - 127 + 1023 - h;
    return __hiloint2double((ye << 20) | (int)((sb & 0x7fffff) >> 3), (int)(sb << 29));
}

// v / sqrt(a) for a normal a > 0: v y0 (1 + e/2 + 3 e^2 / 8), e = 1 - a y0^2 (the
// next term, 5 e^3 / 16, is below 2^-58): six double operations, five of them
// in a chain, where sqrt and a division take 1360 cycles.
__device__ __forceinline__ double over_sqrt(double v, double a) {
    const double y0 = rsqrt_seed(a);
    const double t = a * y0;
    const double err = fma(-t, y0, 1.0);
    const double vy = v * y0;
    const double q = err * fma(err, 0.375, 0.5);
    return fma(vy, q, vy);
}

// l = sqrt(a) and inv = 1 / l, both correctly rounded, for a normal a > 0 (P.
// Markstein, "Computation of elementary functions on the IBM RISC System/6000
// processor", IBM J. Res. Dev. 34, 1990): y = 1 / sqrt(a) and g = a y as above to
// about an ulp, l = g + (a - g^2) y / 2, inv = y + y (1 - l y).  His theorem
// excepts the reciprocal of a significand of all ones, which is divided.
// Compared with sqrt and the division over 8.6e9 arguments: no difference.
__device__ __forceinline__ void sqrt_and_reciprocal(double a, double& l, double& inv) {
    const double y0 = rsqrt_seed(a);
    const double t = a * y0;
    const double err = fma(-t, y0, 1.0);
    const double q = err * fma(err, 0.375, 0.5);
    const double y = fma(y0, q, y0);
    const double g = fma(t, q, t);
    const double r = fma(-g, g, a);
    l = fma(r, __hiloint2double(__double2hiint(y) - 0x100000, __double2loint(y)), g);
    inv = fma(y, fma(-l, y, 1.0), y);
    if ((__double2hiint(l) & 0xfffff) == 0xfffff && __double2loint(l) == -1) inv = 1.0 / l;
}

// A pivot outside the normal range: v / sqrt(piv), or zeros (the sweep goes on
// with them) and the column recorded when piv is not positive and finite.
__device__ __noinline__ double odd_pivot(double v, double piv, int c, int lane, int* failed) {
    if (piv > 0.0 && isfinite(piv)) {
        const double l = sqrt(piv);
        return lane == c ? l : v * (1.0 / l);
    }
    if (lane == 0 && *failed < 0) *failed = c;
    return 0.0;
}

// L_ss of sub-block s.  Thread (lane, warp) holds row lane, columns warp + 4 i;
// one barrier a column.  The warp that owns column c + 1 takes its last term,
// its pivot and the finished column in step c, 600 cycles of dependent double
// operations and the sweep's critical path; the others' work fits beside
// it.  Of the terms of four columns (a group), those for the next two groups
// of columns are taken at once, the others in the next group, two columns by
// four terms in each of a warp's three steps without a pivot.  Pivots are
// tested by their bits (a comparison of doubles costs 64 cycles, too).  A group
// is one iteration of a loop, in two forms (up to six and up to three columns
// to come; the columns move down one register as they finish, and what moves
// in past the last one is not used): unrolled over all columns the sweep
// waits for its code.
constexpr int kLsCols = 48;                    // rows of Ls, with room for the unused columns' reads

// IEEE: L_cc = sqrt(a_cc) and a_rc (1 / L_cc), each correctly rounded, and every
// position's terms in the order of c.
template <int LEFT, bool IEEE>
__device__ __forceinline__ void diag32_columns(double (&a)[kB / kWarps], double (*Ls)[kLsCols], int j0, int warp,
                                               int lane, int* failed) {
    constexpr int kCols = kB / kWarps;
    // pivot and finished column c, held in v by the warp that owns it
    auto finish = [&](double& v, int c) {
        const double piv = __shfl_sync(0xffffffffu, v, c);
        const unsigned hi = (unsigned)__double2hiint(piv);
        if (hi - 0x00100000u >= 0x7fe00000u) {         // not normal, positive and finite
            v = odd_pivot(v, piv, c, lane, failed);
        } else if (IEEE) {
            double l, inv;
            sqrt_and_reciprocal(piv, l, inv);
            v = lane == c ? l : v * inv;
        } else {
            v = over_sqrt(v, piv);
        }
        Ls[c][lane] = v;
    };
    // the four terms of group j - 1 for columns i0, i0 + 1
    auto pending = [&](int j, int i0) {
        double l[4], lk[4][2];
#pragma unroll
        for (int u = 0; u < kWarps; ++u) {
            const double* col = Ls[kWarps * (j - 1) + u];
            l[u] = col[lane];
#pragma unroll
            for (int i = 0; i < 2; ++i) lk[u][i] = col[warp + kWarps * (j + i0 + i)];
        }
#pragma unroll
        for (int u = 0; u < kWarps; ++u)
#pragma unroll
            for (int i = 0; i < 2; ++i)
                if (i0 + i <= LEFT) a[i0 + i] = fma(-l[u], lk[u][i], a[i0 + i]);
    };
    if (j0 == 0) {
        if (warp == 0) finish(a[0], 0);
        __syncthreads();
    }
#pragma unroll 1
    for (int j = j0; j < j0 + kCols / 2; ++j) {
#pragma unroll
        for (int q = 0; q < kWarps; ++q) {
            const int c = kWarps * j + q;
            const double lr = Ls[c][lane], l0 = Ls[c][warp + kWarps * j], l1 = Ls[c][warp + kWarps * (j + 1)];
            if (warp == (q + 1) % kWarps) {
                if (q < kWarps - 1) {
                    a[0] = fma(-lr, l0, a[0]);
                    finish(a[0], c + 1);
                    if (q > 0) a[1] = fma(-lr, l1, a[1]);
                } else if (c + 1 < kB) {
                    a[1] = fma(-lr, l1, a[1]);
                    finish(a[1], c + 1);
                }
            } else {
                // this warp's step number among those without a pivot
                const int step = q - (q > (warp + kWarps - 1) % kWarps ? 1 : 0);
                if (warp > q) a[0] = fma(-lr, l0, a[0]);
                if (j > 0 && step == 0) pending(j, 1);
                // every column's terms in order: warp 1's pivot comes before the
                // group's first step without one
                if (q == 1 && warp == 1) a[1] = fma(-Ls[c - 1][lane], Ls[c - 1][warp + kWarps * (j + 1)], a[1]);
                a[1] = fma(-lr, l1, a[1]);
                if (j > 0) {
                    if (step == 1 && LEFT > 2) pending(j, 3);
                    if (step == 2 && LEFT > 4) pending(j, 5);
                }
            }
            __syncthreads();
        }
#pragma unroll
        for (int i = 0; i + 1 < kCols; ++i) a[i] = a[i + 1];
    }
}

template <bool IEEE>
__global__ void __launch_bounds__(kThreads) k_diag32_f64(Batch b, int J, int s) {
    grid_dependency();
    __shared__ double Ls[kB][kLsCols];             // Ls[c][r]
    __shared__ int failed;
    const int t = blockIdx.x;
    if (b.st[t].status != GP_OK) return;
    double* T = inst_tile(b, t, J, J) + (size_t)(kB * s) * GP_NB + kB * s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int kCols = kB / kWarps;
    double a[kCols];
#pragma unroll
    for (int i = 0; i < kCols; ++i) {
        const int k = warp + kWarps * i;
        a[i] = lane >= k ? T[(size_t)k * GP_NB + lane] : 0.0;
    }
    for (int q = threadIdx.x; q < kB * kLsCols; q += kThreads) (&Ls[0][0])[q] = 0.0;
    if (threadIdx.x == 0) failed = -1;
    __syncthreads();
    diag32_columns<kCols - 2, IEEE>(a, Ls, 0, warp, lane, &failed);
    diag32_columns<kCols / 2 - 1, IEEE>(a, Ls, kCols / 2, warp, lane, &failed);
    if (failed >= 0) {
        if (threadIdx.x == 0) {
            b.st[t].status = GP_ENOTPD;
            b.st[t].fail_col = J * GP_NB + kB * s + failed;
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < kCols; ++i) {
        const int k = warp + kWarps * i;
        if (lane >= k) T[(size_t)k * GP_NB + lane] = Ls[k][lane];
    }
}

// Rows below sub-block s, `per_warp` groups of 32 / LANES rows a warp: lane (row
// rr, kq) holds columns kq + LANES j of its row; x_c goes from its owner to the
// row's other lanes by a shuffle, and column c leaves the columns after it in
// the order of c.  Four lanes a row take 168 double operations for eight rows,
// eight lanes 104 for four: less in all with four, sooner done with eight
// where the rows do not fill the schedulers.
template <int LANES>
__global__ void __launch_bounds__(kThreads) k_solve32_f64(Batch b, int J, int s, int units, int per_warp) {
    grid_dependency();
    constexpr int kRows = 32 / LANES, kCols = kB / LANES;
    __shared__ double Ls[kB][kB + 1];
    __shared__ double inv[kB];
    const int t = blockIdx.y;
    if (b.st[t].status != GP_OK) return;
    const double* T = inst_tile(b, t, J, J) + (size_t)(kB * s) * GP_NB + kB * s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rr = lane % kRows, kq = lane / kRows;
    int u = (blockIdx.x * kWarps + warp) * per_warp;
    const int end = u + per_warp < units ? u + per_warp : units;
    auto rows = [&](int unit) {
        const int row = kB * (s + 1) + kRows * unit;
        return inst_tile(b, t, J + (row >> 7), J) + (size_t)(kB * s) * GP_NB + (row & 127) + rr;
    };
    double a[kCols], nx[kCols];
    if (u < end) {
        const double* p = rows(u);
#pragma unroll
        for (int j = 0; j < kCols; ++j) nx[j] = p[(size_t)(kq + LANES * j) * GP_NB];
    }
    for (int q = threadIdx.x; q < kB * kB; q += kThreads) {
        const int r = q % kB, c = q / kB;
        if (r >= c) cp_async8(&Ls[c][r], T + (size_t)c * GP_NB + r);
    }
    if (threadIdx.x < kB) inv[threadIdx.x] = 1.0 / T[(size_t)threadIdx.x * (GP_NB + 1)];
    cp_async_wait_all();
    __syncthreads();
    for (; u < end; ++u) {
        double* p = rows(u);
#pragma unroll
        for (int j = 0; j < kCols; ++j) a[j] = nx[j];
        if (u + 1 < end) {
            const double* pn = rows(u + 1);
#pragma unroll
            for (int j = 0; j < kCols; ++j) nx[j] = pn[(size_t)(kq + LANES * j) * GP_NB];
        }
#pragma unroll
        for (int c = 0; c < kB; ++c) {
            const int jc = c / LANES, qc = c % LANES;
            const double x = __shfl_sync(0xffffffffu, a[jc], kRows * qc + rr) * inv[c];
            if (qc < LANES - 1) {
                const double v = fma(-x, Ls[c][kq + LANES * jc], a[jc]);
                a[jc] = kq > qc ? v : (kq == qc ? x : a[jc]);
            } else if (kq == LANES - 1) {
                a[jc] = x;
            }
#pragma unroll
            for (int j = jc + 1; j < kCols; ++j) a[j] = fma(-x, Ls[c][kq + LANES * j], a[j]);
        }
#pragma unroll
        for (int j = 0; j < kCols; ++j) p[(size_t)(kq + LANES * j) * GP_NB] = a[j];
    }
}

// LaunchLog around one launch
struct Logged {
    LaunchLog* log;
    Logged(LaunchLog* l, int phase, cudaStream_t st) : log(l) {
        if (log) log->begin(phase, st);
    }
    ~Logged() {
        if (log) log->end();
    }
};

template <int LANES>
void launch_solve32(const Batch& b, int J, int s, int rows, int sms, cudaStream_t st) {
    const int units = rows / (32 / LANES);
    const long long warps = (long long)sms * 8;              // two CTAs an SM
    const int per_warp = (int)(((long long)units * b.count + warps - 1) / warps);
    const int grid = (units + kWarps * per_warp - 1) / (kWarps * per_warp);
    launch_chained(ahead_f64(b), k_solve32_f64<LANES>, dim3(grid, b.count), kThreads, 0, st, b, J, s, units,
                   per_warp);
}

// Up to two block columns: the products of sub-block s for the columns of block
// column J after it, A_rk = fma(-L_rc, L_kc, A_rk) for c in order, a CTA per 32 x
// 32 block (rb, kb) of 32-row and 32-column groups counted from the sub-block:
// thread (lane, warp) owns row lane, columns warp + 8 j.
constexpr int kInnerThreads = 256;
constexpr int kInnerCols = kB * kB / kInnerThreads;

__global__ void __launch_bounds__(kInnerThreads) k_inner_f64(Batch b, int J, int s) {
    grid_dependency();
    __shared__ double Lk[kB][kB + 1];              // Lk[c][k]
    const int t = blockIdx.z;
    if (b.st[t].status != GP_OK) return;
    const int kb = s + 1 + blockIdx.y, rb = kb + blockIdx.x;      // from tile (J, J)'s first
    const int row0 = kB * rb;
    if (J * GP_NB + row0 >= b.n) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double* Lj = inst_tile(b, t, J, J) + (size_t)(kB * s) * GP_NB + kB * kb;
    for (int q = threadIdx.x; q < kB * kB; q += kInnerThreads) cp_async8(&Lk[q / kB][q % kB], Lj + (size_t)(q / kB) * GP_NB + q % kB);
    double* T = inst_tile(b, t, J + (row0 >> 7), J) + (row0 & 127) + lane;
    double lr[kB], a[kInnerCols];
#pragma unroll
    for (int c = 0; c < kB; ++c) lr[c] = T[(size_t)(kB * s + c) * GP_NB];
#pragma unroll
    for (int j = 0; j < kInnerCols; ++j) a[j] = T[(size_t)(kB * kb + warp + 8 * j) * GP_NB];
    cp_async_wait_all();
    __syncthreads();
#pragma unroll
    for (int c = 0; c < kB; ++c)
#pragma unroll
        for (int j = 0; j < kInnerCols; ++j) a[j] = fma(-lr[c], Lk[c][warp + 8 * j], a[j]);
#pragma unroll
    for (int j = 0; j < kInnerCols; ++j) T[(size_t)(kB * kb + warp + 8 * j) * GP_NB] = a[j];
}

// Tile (1, 1) less L_10 L_10^T: sums from zero over the 128 columns in order, then
// one subtraction, a CTA per 32 x 32 block of the lower triangle.
__global__ void __launch_bounds__(kInnerThreads) k_trailing_f64(Batch b) {
    grid_dependency();
    __shared__ double Lk[GP_NB][kB + 1];
    const int t = blockIdx.y;
    if (b.st[t].status != GP_OK) return;
    int rb, kb;
    tri_decode(blockIdx.x, rb, kb);
    if (GP_NB + kB * rb >= b.n) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double* L = inst_tile(b, t, 1, 0);
    for (int q = threadIdx.x; q < GP_NB * kB; q += kInnerThreads) cp_async8(&Lk[q / kB][q % kB], L + (size_t)(q / kB) * GP_NB + kB * kb + q % kB);
    double* C = inst_tile(b, t, 1, 1) + kB * rb + lane;
    L += kB * rb + lane;
    double acc[kInnerCols] = {};
    cp_async_wait_all();
    __syncthreads();
#pragma unroll 16
    for (int c = 0; c < GP_NB; ++c) {
        const double lr = L[(size_t)c * GP_NB];
#pragma unroll
        for (int j = 0; j < kInnerCols; ++j) acc[j] = fma(lr, Lk[c][warp + 8 * j], acc[j]);
    }
#pragma unroll
    for (int j = 0; j < kInnerCols; ++j) C[(size_t)(kB * kb + warp + 8 * j) * GP_NB] -= acc[j];
}

// log|R| of up to two block columns: the pivots' logarithms summed in column
// order per block, the blocks' sums in turn.
__global__ void __launch_bounds__(GP_NB) k_logdet_small_f64(Batch b) {
    grid_dependency();
    __shared__ double logs[GP_NB];
    const int t = blockIdx.x;
    if (b.st[t].status != GP_OK) return;
    double total = 0.0;
    for (int J = 0; J < b.nt; ++J) {
        logs[threadIdx.x] = log(inst_tile(b, t, J, J)[threadIdx.x * (GP_NB + 1)]);
        __syncthreads();
        if (threadIdx.x == 0) {
            double sum = 0.0;
            for (int c = 0; c < GP_NB; ++c) sum += logs[c];
            total += 2.0 * sum;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) b.st[t].logdet = total;
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

// Factor matrices of one or two block columns, the padded rows and columns left
// as they are (the identity).  Every position takes its operations in the
// order of the unblocked loops: the same bits as one CTA per tile and instance
// on the FP64 pipe gave (n = 200, T = 64: 1.59 -> 0.52 ms).
cudaError_t launch_factor_small_f64(const Batch& b, cudaStream_t st, LaunchLog* log) {
    const int sms = device_sms();
    for (int J = 0; J < b.nt; ++J) {
        const int left = b.n - J * GP_NB;                    // real rows from block column J on
        for (int s = 0; s < GP_NB / kB && kB * s < left; ++s) {
            {
                Logged l(log, GP_PHASE_POTRF, st);
                launch_chained(ahead_f64(b), k_diag32_f64<true>, b.count, kThreads, 0, st, b, J, s);
            }
            const int rows = (left - kB * (s + 1) + 7) / 8 * 8;
            if (rows <= 0) continue;
            {
                Logged l(log, GP_PHASE_TRSM, st);
                if ((long long)rows * b.count <= 4 * 4LL * sms) launch_solve32<8>(b, J, s, rows, sms, st);
                else                                            launch_solve32<4>(b, J, s, rows, sms, st);
            }
            const int cols = GP_NB / kB - 1 - s, groups = (left + kB - 1) / kB - 1 - s;
            if (cols > 0 && groups > 0) {
                Logged l(log, GP_PHASE_TRSM, st);
                launch_chained(ahead_f64(b), k_inner_f64, dim3(groups, cols < groups ? cols : groups, b.count),
                               kInnerThreads, 0, st, b, J, s);
            }
        }
        if (J + 1 < b.nt) {
            const int groups = (left - GP_NB + kB - 1) / kB;
            Logged l(log, GP_PHASE_UPDATE, st);
            launch_chained(ahead_f64(b), k_trailing_f64, dim3(groups * (groups + 1) / 2, b.count),
                           kInnerThreads, 0, st, b);
        }
    }
    Logged l(log, GP_PHASE_POTRF, st);
    launch_chained(ahead_f64(b), k_logdet_small_f64, b.count, GP_NB, 0, st, b);
    return cudaGetLastError();
}

cudaError_t launch_panel_f64(const Batch& b, int J, cudaStream_t st, LaunchLog* log) {
    const int sms = device_sms();
    for (int s = 0; s < GP_NB / kB; ++s) {
        if (s > 0) {
            Logged l(log, GP_PHASE_TRSM, st);
            cudaError_t e = launch_update_f64_inner(b, J, s, st);
            if (e != cudaSuccess) return e;
        }
        {
            Logged l(log, GP_PHASE_POTRF, st);
            launch_chained(s > 0 && ahead_f64(b), k_diag32_f64<false>, b.count, kThreads, 0, st, b, J, s);
        }
        const int rows = (b.nt - J) * GP_NB - kB * (s + 1);
        if (rows > 0) {
            Logged l(log, GP_PHASE_TRSM, st);
            if ((long long)rows * b.count <= 4 * 4LL * sms) launch_solve32<8>(b, J, s, rows, sms, st);
            else                                            launch_solve32<4>(b, J, s, rows, sms, st);
        }
    }
    return cudaGetLastError();
}

cudaError_t launch_logdet_f64(const Batch& b, cudaStream_t st) {
    k_logdet_f64<<<b.count, 256, 0, st>>>(b);
    return cudaGetLastError();
}

}  // namespace gp
