// gp_internal.cuh -- shared definitions of libgp's CUDA sources.
//
// Storage of R and of its Cholesky factor (per instance): the lower
// triangle in NB x NB tiles.  Tile (I, J), I >= J, starts at tile index
// J*nt - J*(J-1)/2 + (I - J) (tile columns packed one after another), and
// is column-major inside (element (r, c) at r + NB*c).  Rows/columns >= n
// hold the identity so that the padded factor is block-diag(L, I).
// Diagonal tiles hold both triangles of R; after factorisation their
// lower triangle holds L.
#pragma once

#include <atomic>
#include <mutex>

#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>
#include <cuda_bf16.h>

#include "../../include/gp.h"

#define GP_NB 128
#define GP_TILE_ELEMS (GP_NB * GP_NB)
#define GP_MAX_D 64
#define GP_MAX_SLICES 7
#define GP_PANEL_SLICES 7

namespace gp {

// Candidates one call takes: the chunk loops over them stay in int.
constexpr int kMaxCandidates = 1 << 30;

__host__ __device__ inline int num_tiles(int n) { return (n + GP_NB - 1) / GP_NB; }

__host__ __device__ inline long long tile_index(int I, int J, int nt) {
    return (long long)J * nt - (long long)J * (J - 1) / 2 + (I - J);
}

__host__ __device__ inline long long packed_tiles(int nt) {
    return (long long)nt * (nt + 1) / 2;
}

__host__ __device__ inline size_t packed_elems(int n) {
    int nt = num_tiles(n);
    return (size_t)packed_tiles(nt) * GP_TILE_ELEMS;
}

// lower-triangle linear index q -> (i, k), k <= i, over an m x m triangle
// (a float square root seeds r, the integer loops make it exact: FP64 is
// scarce on this GPU and this runs once per work item in every warp role)
__device__ inline void tri_decode(int q, int& i, int& k) {
    int r = (int)((sqrtf(8.f * (float)q + 1.f) - 1.f) * 0.5f);
    while ((long long)(r + 1) * (r + 2) / 2 <= q) ++r;
    while ((long long)r * (r + 1) / 2 > q) --r;
    i = r;
    k = q - r * (r + 1) / 2;
}

// Per-instance record written by the factorisation and solve kernels.
struct InstState {
    double logdet;
    double aa;      // 1'R^-1 1
    double ab;      // 1'R^-1 Y
    double mu;
    double Q;
    double bb;
    int status;
    int fail_col;
    // 1-norm condition estimate (split path, k_cond.cu): ||R||_1, Hager's
    // estimate of ||R^-1||_1 and the iteration's state
    double anorm;
    double est;
    int hager_iter;
    int hager_jprev;
    int hager_done;   // 1: the estimate has stopped; the solve kernels skip the instance
    // iterative refinement of the split path (k_mixed.cu)
    double piv_inv;   // sum_i 1 / L_ii^2 over the factor's pivots
    double dq_prev;   // change of n log Q made by the previous refinement step
    int refine_done;  // 1: the refinement has stopped; the solve kernels skip the instance
};

// Batched problem description handed to the kernels (by value).
struct Batch {
    int n, d, nt, count;          // count = instances in this launch chunk
    double p, delta;
    const double* x;              // n x d
    const double* y;              // n
    const double* theta;          // count x d (already offset to the chunk)
    double* A;                    // count * packed_elems(n)   (double tiles), or
    float2* Adf;                  // double-float tiles (split path; A unused then)
    float2* Rdf;                  // double-float copy of R (split path)
    size_t inst_stride;           // elements between instances in A / Adf / Rdf
    InstState* st;                // count
    int asm_cols;                 // double-float assembly: tile columns per CTA (16 or 32)
    int corr;                     // gp_correlation
    int inject_timeout;           // test hook: one tensor-core CTA waits on a barrier nothing signals
};

// Split-precision path: per-instance buffers (double-float tiles, bf16
// slice images of the current panel and of W = L_JJ^-1, solve vectors).
struct MixedBatch {
    int n, d, nt, count;
    double delta;                 // the nugget (the refinement's log-det error estimate)
    int s;                        // slices of the trailing update operands
    int ps;                       // slices of the panel solve operands (GP_PANEL_SLICES)
    int ug;                       // accumulator groups of the trailing update (3, 4 or 7)
    int inject_timeout;           // test hook: one split-GEMM CTA waits on a barrier nothing signals
    int update_tile;              // columns of a trailing-update output tile (128 or 64)
    int sp;                       // slice slots per row block in PS (max(s, ps))
    float2* A;                    // working matrix -> factor (double-float tiles)
    float2* Rc;                   // copy of R (double-float tiles), for residuals
    size_t inst_stride;
    __nv_bfloat16* PS;            // panel slices: [row block][slice][4 chunks][128 x 32]
    int* PE;                      // panel row exponents: [row block][128]
    __nv_bfloat16* WS;            // slices of W's rows: [slice][4 chunks][128 x 32]
    int* WE;                      // [128]
    __nv_bfloat16* PF;            // two-panel slices for the fused update: [row block][slice][8 chunks][128 x 32]
    int* FE;                      // their row exponents: [row block][128]
    size_t pf_stride, fe_stride;
    int fuse;                     // 1: trailing updates of panel pairs fused (K = 256)
    int fwd;                      // 1: the forward solve L [x_1 x_y] = [1 Y] runs inside the
                                  // factorisation (diagonal blocks and panel slicing)
    float2* WT;                   // L_JJ^-1 per diagonal block, double-float tiles: [J][128 x 128]
    float2* WR;                   // the same, row-major (its transpose column-major), stride wt_stride
    size_t wt_stride;
    size_t ps_stride, pe_stride, ws_stride, we_stride;
    float2* Z;                    // 10 columns of npad double-float values: x_1, x_y, two
                                  // residual / correction columns, 1 / L_ii, two
                                  // condition-estimate columns, |R| row sums, and
                                  // a = L^-1 1, b = L^-1 Y (kept from the forward solve)
    size_t z_stride;
    float2* RP;                   // per-tile partial sums of the tile-parallel solves and residual
    size_t rp_stride;
    int lookahead;                // SMs that the rest of an update leaves to the next block columns (0: none)
    int* SC;                      // per-block counters of the tile-parallel substitutions
    size_t sc_stride;
    const double* y;
    InstState* st;
    int* err;                     // set when a bounded device wait gave up
};

constexpr int kZCols = 10;
// kernel launches of one forward or backward substitution pass (the first
// block's diagonal step, then a tile step per further block column that
// also finishes the next block)
inline int subst_launches(int nt) { return nt; }
// partial sums of the tile-parallel residual per lower tile: row products
// [2 column halves][2 right-hand sides][128], then column products [2][2][64]
constexpr int kRpTile = 2 * 2 * GP_NB + 2 * 2 * (GP_NB / 2);

// A kernel's dynamic shared-memory limit is a per-device attribute: each
// launcher keeps the largest size it has set on every device ordinal and
// raises the limit once per device (and again when it needs more).  Threads
// that launch the same kernel with different sizes (contexts on several
// streams) take a lock around the check and the attribute call, so the
// attribute only ever grows: without it, a thread setting a smaller size
// after another set a larger one would leave the larger launches refused.
constexpr int kMaxDevices = 64;
inline std::mutex& smem_limit_mutex() {
    static std::mutex m;
    return m;
}
template <typename Kernel>
inline cudaError_t raise_smem_limit(Kernel* kernel, size_t bytes, std::atomic<size_t> (&done)[kMaxDevices]) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool cached = dev >= 0 && dev < kMaxDevices;
    if (cached && bytes <= done[dev].load(std::memory_order_acquire)) return cudaSuccess;
    std::lock_guard<std::mutex> lock(smem_limit_mutex());
    if (cached && bytes <= done[dev].load(std::memory_order_acquire)) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess && cached) done[dev].store(bytes, std::memory_order_release);
    return e;
}

// SMs of the current device (looked up once per device ordinal)
inline int device_sms() {
    static std::atomic<int> cache[kMaxDevices];
    int dev = 0;
    cudaGetDevice(&dev);
    const bool cached = dev >= 0 && dev < kMaxDevices;
    int n = cached ? cache[dev].load(std::memory_order_relaxed) : 0;
    if (n == 0) {
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 1;
        if (cached) cache[dev].store(n, std::memory_order_relaxed);
    }
    return n;
}

// The current device's table of 2^(-j/1024) as double-float (k_assemble.cu),
// filled once per device by init_exp2_table (gp_create; it synchronises).
cudaError_t init_exp2_table();
const float2* exp2_table();

// ---- context accessors (gp_capi.cu) ----------------------------------------
int ctx_fail(gp_ctx* ctx, int code, const char* fmt, ...);
int ctx_device(const gp_ctx* ctx);
// the argument checks every entry point shares: n, d, p (for eq. 2's family), delta
int ctx_check_common(gp_ctx* ctx, int n, int d, double p, double delta);
int ctx_correlation(const gp_ctx* ctx);
cudaStream_t ctx_stream(const gp_ctx* ctx);

// ---- kernels (launch helpers, all on `stream`) ----------------------------
cudaError_t launch_validate_theta(const Batch& b, cudaStream_t s);
cudaError_t launch_assemble_tiles(const Batch& b, cudaStream_t s);
cudaError_t launch_assemble_dense(int n, int d, const double* x, const double* theta, double p, int corr,
                                  double delta, double* R, cudaStream_t s);
// the tiles of a trailing update: all, column J + 1 only, or the others
enum : int { kUpdateAll = 0, kUpdateColumn = 1, kUpdateRest = 2 };
cudaError_t launch_update_f64_tc(const Batch& b, int J, cudaStream_t s, int which = kUpdateAll);
// columns 32 step .. 32 step + 31 of block column J, less the products of its columns before them
cudaError_t launch_update_f64_inner(const Batch& b, int J, int step, cudaStream_t s);
// steps of X = L^-1 and R^-1 = X'X by rows of X (k_grad.cu, k_update_tc.cu)
cudaError_t launch_inverse_apply(const Batch& b, int J, double* X, double* S, cudaStream_t s);
cudaError_t launch_inverse_update(const Batch& b, int J, double* X, double* S, cudaStream_t s);
// What a caller that accounts for phases (GP_PHASE_*) is told around each launch
// of the functions that mix them
struct LaunchLog {
    virtual void begin(int phase, cudaStream_t s) = 0;
    virtual void end() = 0;
};
constexpr int kPanelStep = 32;
// block column J factored and solved (kUpdateTcTiles block columns and more), and the
// log-determinant once they all are
cudaError_t launch_panel_f64(const Batch& b, int J, cudaStream_t s, LaunchLog* log = nullptr);
cudaError_t launch_logdet_f64(const Batch& b, cudaStream_t s);
// the whole factorisation and log-determinant of fewer block columns
cudaError_t launch_factor_small_f64(const Batch& b, cudaStream_t s, LaunchLog* log = nullptr);
// Block columns from which the double path's products run on the tensor cores
// (k_update_tc.cu), whatever the batch.  They are faster from the first tile on
// (a tile's update is 0.55 ms of one SM's FP64 pipe, 22 us as digits); up to 256 points the factor keeps IEEE operations
// throughout, so the small designs that are fitted with p = 2 next to
// singularity (cond(R) 1e11, where any change of rounding shows in the eighth
// digit of mu_hat) keep their bits.
constexpr int kUpdateTcTiles = 3;
// The split path looks ahead with at most so many candidates and at least so
// many block columns (ms, without -> with; candidates x n): 32x1448 3.63 ->
// 3.52, 16x2048 4.36 -> 4.10, 8x4000 9.76 -> 8.90, 32x4000 20.2 -> 19.1, 4x8192
// 24.4 -> 21.3, 1x12000 29.4 -> 26.6, 8x16384 175.4 -> 170.9.  With fewer block
// columns the launches set up ahead give more (1x512 .76 against .78), and with
// more candidates the diagonal steps themselves fill the SMs (64x2048 8.30 ->
// 8.15 but 64x4000 34.2 -> 34.5, 100x1024 3.24 -> 3.28, 128x2047 14.04 -> 14.11).
constexpr int kLookaheadMixedMax = 48;
constexpr int kLookaheadMixedTiles = 12;

// Launches of a chain of kernels in one stream.  With `ahead`, the kernel is set
// up on the GPU while the one before it still runs (programmatic stream
// serialization); its first statement, grid_dependency(), waits until that one
// has completed with its writes visible, so no result depends on the flag.  Only
// for kernels that begin with grid_dependency().
//
// Where few blocks run it saves 1 to 1.5 us a launch, and a block column of the
// factor is a dozen launches (ms, without -> with; candidates x n):
//   double factor: 1x200 .577 -> .518, 16x300 1.11 -> 1.03, 16x1024 3.06 -> 2.88,
//     8x2048 6.43 -> 6.13, 1x4064 9.06 -> 8.28, 1x8192 27.9 -> 27.1;
//   split factor: 100x64 .286 -> .263, 32x256 .501 -> .467, 8x1024 1.86 -> 1.80,
//     1x4000 7.43 -> 7.19.
// Where many do it costs: a block that waits takes its place beside one that
// runs, so that several blocks of the next kernel share an SM (and its FP64 or
// shared-memory rate) while others idle, and the second stream's slicing finds
// no room: 16x200 .750 -> .760, 64x200 1.11 -> 1.22, 128x300 2.17 -> 2.55, 32x1024 4.28 -> 4.83 (all
// double), 8x4064 the same either way, split 8x16384 188 -> 190 to 193.
// kAhead* are the lines between the two.  The first launch after a wait for the
// other stream is a plain one.
constexpr int kAheadSmallF64 = 8;      // candidates, double, up to two block columns
constexpr int kAheadCountF64 = 16;     // the same, more block columns
constexpr int kAheadColumnsF64 = 128;  // candidates x block columns, double
constexpr int kAheadColumnsMixed = 256;

inline bool ahead_f64(const Batch& b) {
    return b.count <= (b.nt < kUpdateTcTiles ? kAheadSmallF64 : kAheadCountF64) &&
           (long long)b.count * b.nt <= kAheadColumnsF64;
}

inline bool ahead_mixed(const MixedBatch& b) {
    return !b.lookahead && (long long)b.count * b.nt <= kAheadColumnsMixed;
}

inline bool ahead_assemble(const Batch& b) {
    return b.Adf ? (long long)b.count * b.nt <= kAheadColumnsMixed : ahead_f64(b);
}

template <typename T>
struct NotDeduced {
    using type = T;
};
template <typename... P>
inline cudaError_t launch_chained(bool ahead, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                                  cudaStream_t s, typename NotDeduced<P>::type... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = ahead ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// What the launch directly before has written is read by ordinary loads, after
// this: that kernel may still run when this one starts, and __ldg wants data that
// nothing writes while the kernel lives.  Older data may go through __ldg: the
// launch before lets this one start only after its own wait.
__device__ __forceinline__ void grid_dependency() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

cudaError_t launch_forward_solve(const Batch& b, double* Z, size_t z_stride, cudaStream_t s);
cudaError_t launch_finalize(const Batch& b, const double* Z, size_t z_stride, double* nll,
                            double* mu, double* sigma2, double* logdet, int* status,
                            cudaStream_t s);
cudaError_t launch_fit_finish(const Batch& b, double* Z, size_t z_stride, double* scalars,
                              cudaStream_t s);
cudaError_t launch_backward_solve(const Batch& b, double* Z, size_t z_stride, int col,
                                  cudaStream_t s);
// kernels that launch_forward_solve (backward = false) or launch_backward_solve launch
int solve_f64_launches(int nt, bool backward);
// Kriging with the variance's solve on the tensor cores (k_var_tc.cu).
struct VarTables {
    __nv_bfloat16* LS;            // slices of the rows of L left of the diagonal blocks
    __nv_bfloat16* WS;            // slices of the rows of W_J = L_JJ^-1
    int* LE;                      // npad row exponents of LS
    int* WE;                      // npad row exponents of WS
    int* lbits;                   // npad scratch: row maxima as float bits
};
struct VarCall {
    int n, d, nt, N, corr;
    double p, c0;
    int ev;                       // fixed exponent of the slices of v = L^-1 r
    int inject_timeout;
    const float2* x;              // n x d design points (double-float)
    const double* theta;
    const float2* w;              // npad: R^-1 (Y - 1 mu_hat)
    const float2* a;              // npad: L^-1 1
    const double* sc;             // model scalars
    const double* xs;             // N x d
    double* yhat;
    double* s2;                   // null: means only
    VarTables t;
    int* err;
    float2* rtab;                 // var_rhs_tab_bytes(): the r kernel's tables
};
size_t var_table_bytes(int nt);
size_t var_rx_bytes(int nt);      // per point block
size_t var_mp_bytes(int nt);      // per point block
size_t var_vs_bytes(int nt);      // per CTA: the slices of V
size_t var_cta_bytes(int nt);     // per CTA of the tensor-core pass: V's and C_J's slices
size_t var_rhs_tab_bytes();
VarTables var_tables_at(void* base, int nt);
cudaError_t launch_var_rhs_tables(const VarCall& c, cudaStream_t s, int* kernels);
cudaError_t launch_var_tables(const float2* L, int nt, const VarTables& t, cudaStream_t s, int* kernels);
cudaError_t launch_var_points(const VarCall& c, int m0, int npb, float2* RX, float2* MP, cudaStream_t s,
                              int* kernels);
cudaError_t launch_var_pass(const VarCall& c, int m0, int npb, const float2* RX, __nv_bfloat16* VS,
                            __nv_bfloat16* CS, int grid, cudaStream_t s, int* kernels);
cudaError_t launch_predict(int n, int d, int nt, const float2* x, const double* theta, double p, int corr, double c0,
                           const float2* L, const float2* w, const float2* a, const double* scalars, int N,
                           const double* xs, double* yhat, double* s2, float2* work, int chunk, int nr,
                           cudaStream_t s);
cudaError_t launch_to_df_inplace(double* p, size_t count, cudaStream_t s);
size_t predict_work_per_cta(int nt, int nr);
// test points per CTA for N points on a device of `sms` SMs (8 or 16)
int predict_points_per_cta(int N, int sms);

cudaError_t launch_diag_mixed(const MixedBatch& b, int J, cudaStream_t s);
cudaError_t launch_split_panel(const MixedBatch& b, int J, int ns, int gemv, cudaStream_t s);
cudaError_t launch_gemm_panel(const MixedBatch& b, int J, cudaStream_t s);
cudaError_t launch_gemm_update(const MixedBatch& b, int J, cudaStream_t s);
cudaError_t launch_gemm_update_column(const MixedBatch& b, int J, cudaStream_t s);
cudaError_t launch_gemm_update_fused(const MixedBatch& b, int J, int which, cudaStream_t s);
cudaError_t launch_split_fused(const MixedBatch& b, int J, cudaStream_t s);
cudaError_t launch_df_forward(const MixedBatch& b, int c0, int init, cudaStream_t s);
cudaError_t launch_rhs_init(const MixedBatch& b, cudaStream_t s);
cudaError_t launch_df_backward(const MixedBatch& b, int c0, int add_to, cudaStream_t s);
cudaError_t launch_df_residual(const MixedBatch& b, cudaStream_t s);
cudaError_t launch_grad(const Batch& b, double* Z, size_t zs, double* X, double* Ri, int* status, double* nll,
                        double* grad, cudaStream_t s, int* kernels);
cudaError_t launch_norm1(const MixedBatch& b, cudaStream_t s);
cudaError_t launch_hager(const MixedBatch& b, int phase, double* cond, cudaStream_t s);
cudaError_t launch_fill_int(int* dst, int count, int value, cudaStream_t s);
cudaError_t launch_scatter(int m, const int* idx, const double* src, double* dst, cudaStream_t s);
cudaError_t launch_scatter_int(int m, const int* idx, const int* src, int* dst, cudaStream_t s);
cudaError_t launch_df_finalize(const MixedBatch& b, double* nll, double* mu, double* sigma2,
                               double* logdet, int* status, cudaStream_t s);
cudaError_t launch_keep_forward(const MixedBatch& b, cudaStream_t s);
cudaError_t launch_refine_check(const MixedBatch& b, int step, cudaStream_t s);
cudaError_t launch_split_model(const MixedBatch& v, float2* Zm, double* scalars, const double* nll,
                               const int* status, int* status_out, cudaStream_t s);
cudaError_t launch_df_to_double(const float2* src, double* dst, size_t count, cudaStream_t s);

}  // namespace gp
