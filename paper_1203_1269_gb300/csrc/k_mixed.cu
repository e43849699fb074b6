// k_mixed.cu -- the split-precision (GP_MIXED) factorisation around its
// tensor-core GEMMs (k_gemm.cu), and the solves.
//
// Blocked right-looking Cholesky of R(theta) + delta I (Section 3 of the
// paper factors R by Cholesky for the determinant and the solves) with the
// off-diagonal work on the tensor cores:
//
//   diag   L_JJ = chol(A_JJ), W_J = L_JJ^-1        double-float (k_diag_mixed)
//   panel  L_IJ = A_IJ W_J^T            I > J      split GEMM (k_gemm.cu)
//   update A_IK -= L_IJ L_KJ^T      J < K <= I     split GEMM (k_gemm.cu)
//
// Split GEMM (after Ozaki, Ogita, Oishi & Rump, "Error-free transformations
// of matrix multiplication by using fast routines of matrix multiplication",
// Numer. Algorithms 59, 2012): each row i of an operand is scaled by 2^(7-E_i)
// (|row| < 2^E_i) and cut into s slices q_a 2^(-8a) with integers |q_a| <= 128,
//     row = 2^(E_i - 7) sum_a q_a 2^(-8a),
// which bf16 holds exactly; this file's slicing kernels write them as the
// pre-swizzled images the MMA descriptors read (mixed_common.cuh).  The
// first forward solve L [x_1 x_y] = [1 Y] is carried out inside the
// factorisation (the diagonal kernel and the slicing of each solved panel).
//
// Solves: the backward substitution with the double-float factor, two
// right-hand sides, then iterative refinement against the double-float copy
// of R (residual r = b - R x, forward correction z = L^-1 r), all
// tile-parallel, with the sums of eq. 3 taken from forward-only identities
// (k_refine_check) and a per-candidate stopping rule; then the profile
// likelihood.
#include "slices.cuh"

namespace gp {

namespace {

// ----------------------------------------------------------- kernels -------

// The next slice of a double-float x (scaled so |x| < 2^7 before the first
// one): the integer q nearest x.hi, |q| <= 128, times the slice's weight w =
// 2^(-8a), so that x = sum_a slice_a and every product of slices carries its
// own weight 2^(-8(a+b)) into the tensor-core accumulators; x moves on to
// 256 (x - q).  q comes from the float 1.5 2^23, whose unit is 1: rintf's
// instruction has a longer latency, which shows here, where eight warps' rows
// are all there is to run (the panels' slicing, next_slice8, has warps enough
// and too many additions: the kriging pass lost 0.8% to this form).
__device__ __forceinline__ float cut_one(float& xh, float& xl, float w) {
    constexpr float kRound = 12582912.f;
    const float q = __fsub_rn(__fadd_rn(xh, kRound), kRound);
    two_sum(__fsub_rn(xh, q), xl, xh, xl);       // xh - q is exact
    xh = __fmul_rn(xh, 256.f);
    xl = __fmul_rn(xl, 256.f);
    return __fmul_rn(q, w);
}

// Diagonal block of column J in double-float on the FP32 pipes (an FP64
// instruction costs about 64 FP32 ones here): L_JJ = chol(A_JJ), log-det,
// the reciprocal diagonal, and W = L_JJ^-1 with the slices of W's rows.
//
// Factor and inverse run in one right-looking sweep over c = 0 .. 127.
// Before step c, position (i, p) of the lower triangle holds, for rows i >= c,
//   p <  c:  acc_ip = sum_{k<c} L_ik W_kp   (the inverse's partial sums)
//   p >= c:  a_ip, the Cholesky trailing matrix.
// Step c finishes row c of W (W_cp = -acc_cp / L_cc, W_cc = 1 / L_cc) and
// column c of L (L_pc = a_pc / L_cc), giving
//   V_p = W_cp (p <= c),   V_p = -L_pc (p > c),
// and adds L_ic V_p to every position of the rows i > c: the Cholesky update
// for p > c, the inverse's for p < c, and at p = c acc_ic = L_ic V_c restarts
// the position from zero.
//
// The steps are taken kDiagB = 8 at a time, every position receiving its
// terms in the order of c (so the block size does not show in the results):
//   diag   one warp factors the 8 x 8 block, rows across lanes, the pivots
//          passed by shuffles;
//   panel  one thread per column p <= c0 + 7 finishes the 8 rows of W, one
//          thread per row i > c0 + 7 the 8 columns of L (28 multiply-adds
//          each), giving the 8 vectors V in shared memory;
//   update the rows below take the 8 terms.
// The triangle lives in the registers of 16 warps: lane l of warp w holds
// columns l + 32 j of rows w + 16 k (j <= k / 2: 20 double-float values a
// thread), rows k = 2 m and 2 m + 1 as pairs, so that one paired FP32
// instruction serves both: the update is 15 of them per pair and term, and
// little else (per term and warp four loads of V shared by its rows, one
// load per pair of rows).  It first reaches the next block's columns and
// rows, which go to shared memory; a 17th warp then factors the next 8 x 8
// block while the others finish the update.  Three more warps write the
// finished rows and columns out and take what follows from a finished row of
// W -- its slices, the tiles the solves read, the forward solve's x_J, the
// pivots' logarithms -- beside the sweep.  Three barriers per eight columns.
//
// Bound by FP32 issue: the 128^3 / 3 multiply-adds of 15 instructions are
// 0.10 M cycles on an SM's four schedulers at the measured 1.04 cycles each;
// the sweep takes about twice that, the rest being the panels and the 8 x 8
// blocks of the last columns.  Measured, a block column at up to 152
// candidates: 254 us with the triangle in shared memory and two barriers a
// column (loads, stores and index arithmetic took three of four issue slots),
// 160 us with registers but a barrier pair per column, 131 us with the rows'
// slices and copies after the sweep, 126 us now.  n = 1024, T = 100: 4.46 -> 3.46
// ms a batch; n = 64, T = 100: 0.363 -> 0.247 ms; n = 4000, T = 256: 130.0 -> 127.2
// ms.
constexpr int kDiagWarps = 16;                         // warps that hold the triangle
constexpr int kDiagHelpers = 4;                        // one for the 8 x 8 blocks, three for finished rows
constexpr int kDiagThreads = 32 * (kDiagWarps + kDiagHelpers);
constexpr int kDiagRows = GP_NB / kDiagWarps;          // rows per warp
constexpr int kDiagB = 8;
constexpr int kDiagBlocks = GP_NB / kDiagB;
static_assert(kDiagWarps == 16, "the row-to-warp map assumes two row groups per 32-column block");
constexpr int kPacked = GP_NB * (GP_NB + 1) / 2;

__device__ __forceinline__ int prow(int r) { return r * (r + 1) / 2; }

struct DiagShared {
    // the block's vectors V (zero at p > c inside the block): each value
    // twice (hi, hi, lo, lo), and the rows below in pairs (hi of rows w + 32 m
    // and w + 32 m + 16, then their lo)
    float4 vdup[kDiagB][GP_NB];
    float4 vrow[kDiagB][kDiagWarps][kDiagRows / 2];
    dfl col[kDiagB][GP_NB];     // the block's columns of the trailing matrix
    dfl row[kDiagB][GP_NB];     // the block's rows of the inverse's sums
    float4 ld[kDiagB][kDiagB / 2];   // the block's L: column c, rows 2 u and 2 u + 1 in pairs
    dfl dinv[GP_NB];            // 1 / L_cc
    dfl lcc[GP_NB];             // L_cc
    dfl bj[2][GP_NB];           // the forward solve's right-hand sides
    double lsum[GP_NB / 32], psum[GP_NB / 32];
    int failed;
};

__device__ __forceinline__ df2 df2_load(const float4* p) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
    return {v.x, v.y};
}

__device__ __forceinline__ void ld_store(DiagShared& sh, int r, int c, dfl v) {
    float* p = reinterpret_cast<float*>(&sh.ld[c][r >> 1]) + (r & 1);
    p[0] = v.hi;
    p[2] = v.lo;
}

__device__ __forceinline__ dfl df_shfl(dfl a, int src) {
    return {__shfl_sync(0xffffffffu, a.hi, src), __shfl_sync(0xffffffffu, a.lo, src)};
}

// Pivots in [2^-100, 2^100] (the float seed's comfortable range): 1 / sqrt(a)
// from the hardware seed (about 22 correct bits), one float Newton step to y1
// (about 24 bits), then y = y1 (1 + e/2 + 3 e^2/8) with e = 1 - a y1^2:
// Newton's step with its second-order term, the next term (5 e^3 / 16) being
// below 2^-65.  e is about 2^-23 and needed to float precision only, so it
// comes from the exact products a.hi y1 and (a.hi y1) y1 (1 - q_h is exact,
// q_h lying within 2^-22 of 1), and y is the exact sum y1 + corr: about 2^-46
// relative, as two double-float Newton steps give, in a quarter of their
// dependent chain.
__device__ __forceinline__ bool pivot_in_range(dfl a) { return a.hi > 7.9e-31f && a.hi < 1.26e30f; }

__device__ __forceinline__ dfl pivot_rsqrt(dfl a) {
    float y0;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"(a.hi));
    const float p0 = __fmul_rn(a.hi, y0);
    const float y1 = __fmaf_rn(__fmul_rn(y0, 0.5f), __fmaf_rn(-p0, y0, 1.f), y0);
    const float ph = __fmul_rn(a.hi, y1);
    const float pl = __fmaf_rn(a.hi, y1, -ph);
    const float qh = __fmul_rn(ph, y1);
    const float ql = __fmaf_rn(pl, y1, __fmaf_rn(ph, y1, -qh));
    const float rl = __fmul_rn(__fmul_rn(a.lo, y1), y1);
    const float e = __fsub_rn(__fsub_rn(__fsub_rn(1.f, qh), ql), rl);
    const float h = __fmul_rn(y1, 0.5f);
    const float corr = __fmaf_rn(h, e, __fmul_rn(__fmul_rn(h, __fmul_rn(e, e)), 0.75f));
    dfl y;
    fast_two_sum(y1, corr, y.hi, y.lo);
    return y;
}

// The 8 x 8 block at c0 with a pivot outside pivot_in_range: those take the
// double square root; the first that is not positive and finite is recorded
// in sh.failed.
__device__ __noinline__ void diag_block8_slow(DiagShared& sh, int c0, int lane) {
    const int r = lane & 7;
    dfl a[kDiagB];
#pragma unroll
    for (int q = 0; q < kDiagB; ++q) a[q] = sh.col[q][c0 + r];
    bool ok = true;
#pragma unroll
    for (int cc = 0; cc < kDiagB; ++cc) {
        const dfl piv = df_shfl(a[cc], cc);
        const bool good = piv.hi > 0.f && isfinite(piv.hi);
        dfl y = {1.f, 0.f}, d = {1.f, 0.f};
        if (pivot_in_range(piv)) {
            y = pivot_rsqrt(piv);
            d = df_mul(piv, y);
        } else if (good) {
            const double ld = sqrt(df_to_double(piv));
            y = df_from_double(1.0 / ld);
            d = df_from_double(ld);
        }
        if (ok && !good && lane == 0) sh.failed = c0 + cc;
        ok = ok && good;
        const dfl l = df_mul(a[cc], y);
        if (lane == cc) {
            sh.dinv[c0 + cc] = y;
            sh.lcc[c0 + cc] = d;
        }
        if (lane < kDiagB) ld_store(sh, lane, cc, lane == cc ? d : l);
#pragma unroll
        for (int q = cc + 1; q < kDiagB; ++q) a[q] = df_fma(l, df_neg(df_shfl(l, q)), a[q]);
    }
}

// The 8 x 8 block at c0 (one warp): lane r + 8 u holds columns 2 u and 2 u + 1 of
// row r.  Every lane takes each pivot and the results go out at the end, so
// the eight columns are one straight-line chain: a pivot, the column, a
// shuffle and the next pivot's last term, the other terms beside it.
__device__ __forceinline__ void diag_block8(DiagShared& sh, int c0, int lane) {
    const int r = lane & 7, u = lane >> 3;
    df2 a = df2_pack(sh.col[2 * u][c0 + r], sh.col[2 * u + 1][c0 + r]);
    dfl l0 = {0.f, 0.f}, l1 = {0.f, 0.f}, yr = {0.f, 0.f};     // L_{r, 2u}, L_{r, 2u+1}, 1 / L_rr
    bool ok = true;
#pragma unroll
    for (int cc = 0; cc < kDiagB; ++cc) {
        const int from = 8 * (cc / 2);                          // lanes from + r hold column cc
        const dfl acc = (cc & 1) ? df2_second(a) : df2_first(a);
        const dfl piv = df_shfl(acc, from + cc);
        ok = ok && pivot_in_range(piv);
        const dfl y = pivot_rsqrt(piv);
        const dfl l = df_mul(acc, y);                           // at row cc: a y, the pivot's square root
        if (r == cc) yr = y;
        if (u == cc / 2) {
            if (cc & 1) l1 = l;
            else        l0 = l;
        }
        if (cc + 1 < kDiagB) {
            const df2 la = df2_dup(df_shfl(l, from + r));
            const df2 lq = df2_pack(df_shfl(l, from + 2 * u), df_shfl(l, from + 2 * u + 1));
            a = df2_fnma(f2_mul(f2_neg(la.hi), lq.hi), la, lq, a);
        }
    }
    if (ok) {
        ld_store(sh, r, 2 * u, l0);
        ld_store(sh, r, 2 * u + 1, l1);
        if (r / 2 == u) {
            sh.dinv[c0 + r] = yr;
            sh.lcc[c0 + r] = (r & 1) ? l1 : l0;
        }
    } else {
        diag_block8_slow(sh, c0, lane);
    }
}

// The panels of block c0: thread p <= c0 + 7 finishes column p of W's eight
// rows, thread i > c0 + 7 row i of L's eight columns.
__device__ __forceinline__ void diag_panels(DiagShared& sh, int c0, int warp, int lane) {
    df2 v[kDiagB / 2];
    if (warp < 4) {
        const int p = 32 * warp + lane, q0 = p - c0;       // q0 >= 0: a column of the block
        if (p >= c0 + kDiagB) return;
#pragma unroll
        for (int u = 0; u < kDiagB / 2; ++u)
            v[u] = q0 < 0 ? df2_pack(sh.row[2 * u][p], sh.row[2 * u + 1][p]) : df2{0, 0};
#pragma unroll
        for (int cc = 0; cc < kDiagB; ++cc) {
            const dfl di = sh.dinv[c0 + cc];
            const dfl m = df_mul(di, (cc & 1) ? df2_second(v[cc / 2]) : df2_first(v[cc / 2]));
            dfl w = df_neg(m);
            if (q0 == cc) w = di;
            if (q0 > cc) w = dfl{0.f, 0.f};
            sh.vdup[cc][p] = make_float4(w.hi, w.hi, w.lo, w.lo);
            const df2 wn = df2_dup(df_neg(w));
            const f32x2 wh = f2_pack(w.hi, w.hi);
#pragma unroll
            for (int u = (cc + 1) / 2; u < kDiagB / 2; ++u) {
                const df2 ld = df2_load(&sh.ld[cc][u]);
                v[u] = df2_fnma(f2_mul(ld.hi, wh), ld, wn, v[u]);
            }
        }
    } else if (warp < 8) {
        const int i = 32 * (warp - 4) + lane;
        if (i < c0 + kDiagB) return;
#pragma unroll
        for (int u = 0; u < kDiagB / 2; ++u) v[u] = df2_pack(sh.col[2 * u][i], sh.col[2 * u + 1][i]);
#pragma unroll
        for (int cc = 0; cc < kDiagB; ++cc) {
            const dfl l = df_mul((cc & 1) ? df2_second(v[cc / 2]) : df2_first(v[cc / 2]), sh.dinv[c0 + cc]);
            sh.vdup[cc][i] = make_float4(-l.hi, -l.hi, -l.lo, -l.lo);
            float* vr = reinterpret_cast<float*>(&sh.vrow[cc][i & 15][i >> 5]) + ((i >> 4) & 1);
            vr[0] = -l.hi;
            vr[2] = -l.lo;
            const df2 la = df2_dup(l);
            const f32x2 nl = f2_neg(la.hi);
#pragma unroll
            for (int u = (cc + 1) / 2; u < kDiagB / 2; ++u) {
                const df2 ld = df2_load(&sh.ld[cc][u]);
                v[u] = df2_fnma(f2_mul(nl, ld.hi), la, ld, v[u]);
            }
        }
    }
}

// Block c0's columns of L into the tile T and its rows of W into the packed
// triangle P, from the vectors V (the helper warps h = 0 .. 3, two columns and
// rows each).
__device__ __forceinline__ void diag_write(const DiagShared& sh, int c0, float2* T, dfl* P, int h, int lane) {
    if (h == 0 && lane < kDiagB) {
#pragma unroll
        for (int cc = 0; cc < kDiagB; ++cc) {
            const float* p = reinterpret_cast<const float*>(&sh.ld[cc][lane >> 1]) + (lane & 1);
            if (lane >= cc) T[(size_t)(c0 + cc) * GP_NB + c0 + lane] = make_float2(p[0], p[2]);
        }
    }
#pragma unroll
    for (int q = 0; q < kDiagB / kDiagHelpers; ++q) {
        const int cc = h + kDiagHelpers * q;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int p = lane + 32 * j;
            const float4 v = sh.vdup[cc][p];
            if (p <= c0 + cc)
                P[prow(c0 + cc) + p] = dfl{v.x, v.z};
            else if (p >= c0 + kDiagB)
                T[(size_t)(c0 + cc) * GP_NB + p] = make_float2(-v.x, -v.z);
        }
    }
}

// Row c of W: exponent (of the largest high word, as the panel slicing takes
// it) and slices; one warp, lane l columns 4 l .. 4 l + 3 (half of one 16-byte
// piece).
__device__ __forceinline__ void diag_slices(const dfl* P, uint8_t* WS, int* WE, int c, int lane) {
    const dfl* w = P + prow(c);
    const int k0 = 4 * lane;
    float xh[4], xl[4], mx = 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const dfl v = (k0 + e <= c) ? w[k0 + e] : dfl{0.f, 0.f};
        xh[e] = v.hi;
        xl[e] = v.lo;
        mx = fmaxf(mx, fabsf(v.hi));
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const int E = exponent_of(mx);
    if (lane == 0) WE[c] = E;
    float sa, sb;
    slice_scale(E, sa, sb);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        xh[e] = __fmul_rn(__fmul_rn(xh[e], sa), sb);
        xl[e] = __fmul_rn(__fmul_rn(xl[e], sa), sb);
    }
    uint8_t* dst = WS + (size_t)(k0 >> 5) * kChunkBytes + image_piece(c, k0 & ~7) + ((k0 & 4) ? 8u : 0u);
    float wt = 1.f;
#pragma unroll
    for (int a = 0; a < GP_PANEL_SLICES; ++a) {
        float m[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) m[e] = cut_one(xh[e], xl[e], wt);
        *reinterpret_cast<uint2*>(dst + (size_t)a * kChunks * kChunkBytes) =
            make_uint2(pack_bf16x2(m[0], m[1]), pack_bf16x2(m[2], m[3]));
        wt = __fmul_rn(wt, 0.00390625f);
    }
}

// Rows c0 .. c0 + 7 of W as parts of the double-float tiles that the solves read:
// column-major (forward) and row-major (backward), zeros above the diagonal;
// `parts` warps.
__device__ __forceinline__ void diag_tiles(const dfl* P, float2* Wt, float2* Wr, int c0, int part, int parts,
                                           int lane) {
    for (int c = part; c < kDiagB; c += parts)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int r = c0 + c, p = lane + 32 * j;
            const dfl v = p <= r ? P[prow(r) + p] : dfl{0.f, 0.f};
            Wr[(size_t)r * GP_NB + p] = make_float2(v.hi, v.lo);
        }
    const int r = c0 + (lane & 7);
#pragma unroll 4
    for (int p = (lane >> 3) + 4 * part; p < GP_NB; p += 4 * parts) {
        const dfl v = p <= r ? P[prow(r) + p] : dfl{0.f, 0.f};
        Wt[(size_t)p * GP_NB + r] = make_float2(v.hi, v.lo);
    }
}

// Rows c0 .. c0 + 7 of the forward solve x_J = W (b_J - sum_{K<J} L_JK x_K), the sum
// already subtracted by the slicing of panels K < J, in double-float (one
// warp): lane (row, right-hand side k, half h) sums the columns h, h + 2, ...
// of its row, then the two halves add.
__device__ __forceinline__ void diag_forward(const DiagShared& sh, const dfl* P, float2* zJ, size_t npad, int c0,
                                             int lane) {
    const int r = c0 + (lane & 7), k = (lane >> 3) & 1, h = lane >> 4;
    const dfl* w = P + prow(r);
    dfl sum = {0.f, 0.f};
#pragma unroll 4
    for (int c = h; c <= r; c += 2) sum = df_fma(w[c], sh.bj[k][c], sum);
    const dfl other = df_shfl(sum, (lane & 15) + 16);
    if (h == 0) df_store(zJ + (size_t)k * npad + r, df_add(sum, other));
}

// log L_cc and 1 / L_cc^2 over columns 32 q .. 32 q + 31 (one warp), and the
// reciprocal diagonal out: sums by a warp tree, the four quarters' in turn at
// the end of the kernel.  The squares (over real rows only) are the
// refinement's estimate of the log-det's own error (k_refine_check).
__device__ __forceinline__ void diag_logs(DiagShared& sh, float2* rinv, int q, int real_rows, int lane) {
    const int c = 32 * q + lane;
    double v = log(df_to_double(sh.lcc[c]));
    const double di = df_to_double(sh.dinv[c]);
    double s = c < real_rows ? di * di : 0.0;
    for (int o = 16; o > 0; o >>= 1) {
        v += __shfl_down_sync(0xffffffffu, v, o);
        s += __shfl_down_sync(0xffffffffu, s, o);
    }
    if (lane == 0) {
        sh.lsum[q] = v;
        sh.psum[q] = s;
    }
    df_store(rinv + c, sh.dinv[c]);
}

// A thread's part of the triangle: rows 2 m and 2 m + 1 of its warp in column
// block j <= m.
struct DiagRegs {
    df2 x[kDiagRows / 2][4];
};

// Term cc of the block's update for rows k >= K0 of the warp: in column block
// JN (REST: in all the others), row K0 of an owner in every one.
template <int JN, int K0, bool OWNER, bool REST>
__device__ __forceinline__ void diag_term(const DiagShared& sh, DiagRegs& R, int cc, int warp, int lane) {
    constexpr int M0 = K0 / 2;                 // pair of row K0
    df2 b[4];
    f32x2 nb[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (REST ? j != JN : (j == JN || (OWNER && j <= M0))) {
            b[j] = df2_load(&sh.vdup[cc][lane + 32 * j]);
            nb[j] = f2_neg(b[j].hi);
        }
#pragma unroll
    for (int m = M0; m < kDiagRows / 2; ++m) {
        const df2 a = df2_load(&sh.vrow[cc][warp][m]);
#pragma unroll
        for (int j = 0; j <= m; ++j) {
            const bool mine = REST ? j != JN : j == JN;
            const bool own = OWNER && m == M0 && !mine;      // row K0 alone
            if (mine && !((K0 & 1) && m == M0)) {
                R.x[m][j] = df2_fnma(f2_mul(a.hi, nb[j]), a, b[j], R.x[m][j]);
            } else if (mine || own) {
                // one row of the pair, on the scalar instructions
                const dfl bs = df2_first(b[j]);
                if (K0 & 1)
                    R.x[m][j] = df2_pack(df2_first(R.x[m][j]),
                                         df_fma(df_neg(df2_second(a)), bs, df2_second(R.x[m][j])));
                else
                    R.x[m][j] = df2_pack(df_fma(df_neg(df2_first(a)), bs, df2_first(R.x[m][j])),
                                         df2_second(R.x[m][j]));
            }
        }
    }
}

// The update by the block in sh.V, first part, and the export of block c0's
// columns (in column block JN, lanes q = 0 .. 7) and rows (owner: row K0 of
// this warp): rows k >= K0 take the eight terms in column block JN, and row
// K0 of an owner in the others too.  The exported columns restart at zero.
template <int JN, int K0, bool OWNER>
__device__ __forceinline__ void diag_update_first(DiagShared& sh, DiagRegs& R, int c0, int warp, int lane) {
    if constexpr (K0 < kDiagRows) {
#pragma unroll 1
        for (int cc = 0; cc < kDiagB; ++cc) diag_term<JN, K0, OWNER, false>(sh, R, cc, warp, lane);
        const int q = lane - (c0 & 31);
#pragma unroll
        for (int k = K0; k < kDiagRows; ++k)
            if (q >= 0 && q < kDiagB) {
                df2& v = R.x[k / 2][JN];
                sh.col[q][warp + kDiagWarps * k] = (k & 1) ? df2_second(v) : df2_first(v);
                if (k & 1) v = df2{0, 0};
            }
        if (OWNER) {
#pragma unroll
            for (int j = 0; j <= K0 / 2; ++j)
                if (lane + 32 * j < c0)
                    sh.row[warp + kDiagWarps * K0 - c0][lane + 32 * j] =
                        (K0 & 1) ? df2_second(R.x[K0 / 2][j]) : df2_first(R.x[K0 / 2][j]);
        }
    }
}

// Second part: rows k >= K0 in every column block but JN.
template <int JN, int K0>
__device__ __forceinline__ void diag_update_rest(const DiagShared& sh, DiagRegs& R, int warp, int lane) {
    if constexpr (K0 < kDiagRows) {
#pragma unroll 1
        for (int cc = 0; cc < kDiagB; ++cc) diag_term<JN, K0, false, true>(sh, R, cc, warp, lane);
    }
}

// The instance of diag_update_first / diag_update_rest for block nb = 4 JN ..
// 4 JN + 3 and a warp whose rows reach from k0 on.
template <int JN>
__device__ __forceinline__ void diag_dispatch_first(DiagShared& sh, DiagRegs& R, int c0, int k0, bool owner,
                                                    int warp, int lane) {
    if (owner) {
        if (k0 == 2 * JN) diag_update_first<JN, 2 * JN, true>(sh, R, c0, warp, lane);
        else              diag_update_first<JN, 2 * JN + 1, true>(sh, R, c0, warp, lane);
    } else {
        if (k0 == 2 * JN)          diag_update_first<JN, 2 * JN, false>(sh, R, c0, warp, lane);
        else if (k0 == 2 * JN + 1) diag_update_first<JN, 2 * JN + 1, false>(sh, R, c0, warp, lane);
        else                       diag_update_first<JN, 2 * JN + 2, false>(sh, R, c0, warp, lane);
    }
}

template <int JN>
__device__ __forceinline__ void diag_dispatch_rest(const DiagShared& sh, DiagRegs& R, int k0, int warp,
                                                   int lane) {
    if (k0 == 2 * JN)          diag_update_rest<JN, 2 * JN>(sh, R, warp, lane);
    else if (k0 == 2 * JN + 1) diag_update_rest<JN, 2 * JN + 1>(sh, R, warp, lane);
    else                       diag_update_rest<JN, 2 * JN + 2>(sh, R, warp, lane);
}

__global__ void __launch_bounds__(kDiagThreads, 1) k_diag_mixed(MixedBatch b, int J) {
    grid_dependency();
    extern __shared__ dfl P[];             // kPacked double-float values: A_JJ in, W out
    __shared__ DiagShared sh;
    const int t = blockIdx.x;
    if (b.st[t].status != GP_OK) return;
    float2* T = df_tile(b, b.A, t, J, J);
    for (int q = threadIdx.x; q < GP_TILE_ELEMS; q += kDiagThreads) {
        const int rr = q & 127, cc = q >> 7;
        if (rr >= cc) cp_async8(P + prow(rr) + cc, T + q);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int kWarps = kDiagWarps;
    const int helper = warp - kWarps;      // 0: the 8 x 8 blocks, 1 .. 3: finished rows
    const size_t npad = (size_t)b.nt * GP_NB;
    float2* zJ = b.Z + (size_t)t * b.z_stride + (size_t)J * GP_NB;
    uint8_t* WS = reinterpret_cast<uint8_t*>(b.WS + (size_t)t * b.ws_stride);
    int* WE = b.WE + (size_t)t * b.we_stride;
    float2* Wt = b.WT + (size_t)t * b.wt_stride + (size_t)J * GP_TILE_ELEMS;
    float2* Wr = b.WR + (size_t)t * b.wt_stride + (size_t)J * GP_TILE_ELEMS;
    if (b.fwd && threadIdx.x < 2 * GP_NB)
        sh.bj[threadIdx.x >> 7][threadIdx.x & 127] = df_load(zJ + (threadIdx.x >> 7) * npad + (threadIdx.x & 127));
    if (threadIdx.x == 0) sh.failed = -1;
    cp_async_wait_all();
    __syncthreads();
    DiagRegs R;
#pragma unroll
    for (int m = 0; m < kDiagRows / 2; ++m)
#pragma unroll
        for (int j = 0; j <= m; ++j) {
            const int i = warp + 32 * m, p = lane + 32 * j;
            const dfl u = (warp < kWarps && p <= i) ? P[prow(i) + p] : dfl{0.f, 0.f};
            const dfl v = (warp < kWarps && p <= i + 16) ? P[prow(i + 16) + p] : dfl{0.f, 0.f};
            R.x[m][j] = df2_pack(u, v);
        }
    // block 0's columns (no rows: it has no columns before it)
    if (lane < kDiagB && warp < kWarps)
#pragma unroll
        for (int m = 0; m < kDiagRows / 2; ++m) {
            sh.col[lane][warp + 32 * m] = df2_first(R.x[m][0]);
            sh.col[lane][warp + 32 * m + 16] = df2_second(R.x[m][0]);
            R.x[m][0] = df2{0, 0};
        }
    __syncthreads();
    // what follows from the finished rows of block nb, by helpers 1 .. 3
    auto finished = [&](int nb) {
        const int c0 = kDiagB * nb;
        if (helper == 3) {                 // a chain of up to 64 dependent multiply-adds
            if (b.fwd) diag_forward(sh, P, zJ, npad, c0, lane);
        } else {
#pragma unroll 2
            for (int q = 0; q < kDiagB / 2; ++q) diag_slices(P, WS, WE, c0 + 2 * q + helper - 1, lane);
            diag_tiles(P, Wt, Wr, c0, helper - 1, 2, lane);
            if (helper == 1 && (nb & 3) == 3) diag_logs(sh, zJ + 4 * npad, nb >> 2, b.n - J * GP_NB, lane);
        }
    };
    for (int nb = 0;; ++nb) {
        const int c0 = kDiagB * nb;
        // the warps of one half own a row each of block nb + 1; the warp's
        // rows below block nb reach from k0 on
        const bool owner = (warp >> 3) == ((nb + 1) & 1);
        const int k0 = (c0 + kDiagB - warp + kDiagWarps - 1) >> 4;
        if (helper == 0) {
            diag_block8(sh, c0, lane);
        } else if (nb > 0 && helper > 0) {
            finished(nb - 1);
        } else if (nb > 0) {               // the rest of block nb - 1's update
            const int k1 = (c0 - warp + kDiagWarps - 1) >> 4;
            const int kr = k1 + (owner ? 0 : 1);   // past the warp's row of block nb, exported with it
            switch (nb >> 2) {
                case 0: diag_dispatch_rest<0>(sh, R, kr, warp, lane); break;
                case 1: diag_dispatch_rest<1>(sh, R, kr, warp, lane); break;
                case 2: diag_dispatch_rest<2>(sh, R, kr, warp, lane); break;
                default: diag_dispatch_rest<3>(sh, R, kr, warp, lane); break;
            }
        }
        __syncthreads();
        if (sh.failed >= 0) break;         // uniform
        diag_panels(sh, c0, warp, lane);
        __syncthreads();
        if (helper >= 0) diag_write(sh, c0, T, P, helper, lane);
        if (helper < 0 && nb + 1 < kDiagBlocks) {
            switch ((nb + 1) >> 2) {
                case 0: diag_dispatch_first<0>(sh, R, c0 + kDiagB, k0, owner, warp, lane); break;
                case 1: diag_dispatch_first<1>(sh, R, c0 + kDiagB, k0, owner, warp, lane); break;
                case 2: diag_dispatch_first<2>(sh, R, c0 + kDiagB, k0, owner, warp, lane); break;
                default: diag_dispatch_first<3>(sh, R, c0 + kDiagB, k0, owner, warp, lane); break;
            }
        }
        __syncthreads();
        if (nb + 1 == kDiagBlocks) break;
    }
    if (sh.failed >= 0) {
        if (threadIdx.x == 0) {
            b.st[t].status = GP_ENOTPD;
            b.st[t].fail_col = J * GP_NB + sh.failed;
        }
        return;
    }
    // the last block's rows, by every warp
    constexpr int kLast = GP_NB - kDiagB;
    if (warp < kDiagB)           diag_slices(P, WS, WE, kLast + warp, lane);
    else if (warp == 8)        { if (b.fwd) diag_forward(sh, P, zJ, npad, kLast, lane); }
    else if (warp == 9)          diag_logs(sh, zJ + 4 * npad, 3, b.n - J * GP_NB, lane);
    else                         diag_tiles(P, Wt, Wr, kLast, warp - 10, kDiagThreads / 32 - 10, lane);
    __syncthreads();
    if (threadIdx.x == 0) {
        double ld = 0.0, pq = 0.0;
        for (int w = 0; w < GP_NB / 32; ++w) {
            ld += sh.lsum[w];
            pq += sh.psum[w];
        }
        b.st[t].logdet += 2.0 * ld;
        b.st[t].piv_inv += pq;
    }
}

// Slices of the panel tiles (I, J), I = J + 1 + blockIdx.x / 2, into row
// block I of PS.  A CTA of 512 threads takes one half (64 rows) of a tile:
// thread (r, q, u) owns row r's columns 32q + 16u .. 32q + 16u + 15, two of
// the 16-byte pieces of image chunk q, so it loads its values once
// (coalesced along r) and writes only its own pieces; 16 values per thread
// leave registers for four CTAs per SM, whose loads overlap each other's
// slicing.  The eight owners of a row agree on the row's exponent through
// shared memory.
constexpr int kSplitThreads = 512;
constexpr int kSplitParts = 8;                          // column parts of a row
constexpr int kSplitRows = kSplitThreads / kSplitParts; // rows of a tile per CTA
constexpr int kSplitCols = GP_NB / kSplitParts;         // 16 columns per thread
// k_split_fused: 16 columns of one of the two panels per thread, a quarter tile
constexpr int kFusedParts = 16;
constexpr int kFusedRows = kSplitThreads / kFusedParts;

// gemv (with b.fwd; the slicing of the solved panel for the update): the
// forward solve's panel step b_I -= L_IJ x_J for this CTA's rows, two
// right-hand sides, from the values already in registers.  c0: the first of
// the thread's 16 columns.
template <int NC, int ROWS>
__device__ __forceinline__ void fwd_partials(const float2 (&v)[NC], const dfl (*xs)[GP_NB], int c0,
                                             int part, int rl, dfl (*red)[2][ROWS]) {
    dfl p0 = {0.f, 0.f}, p1 = {0.f, 0.f};
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        const dfl l = {v[j].x, v[j].y};
        p0 = df_fma(l, xs[0][c0 + j], p0);
        p1 = df_fma(l, xs[1][c0 + j], p1);
    }
    red[part][0][rl] = p0;
    red[part][1][rl] = p1;
}

// b_I[r] -= the PARTS column parts' partial sums, pairwise in a fixed order
// (parts 0 and 1 take one right-hand side each); after a barrier that
// follows fwd_partials
template <int PARTS, int ROWS>
__device__ __forceinline__ void fwd_apply(const MixedBatch& b, int t, int I, int r, int part, int rl,
                                          const dfl (*red)[2][ROWS]) {
    if (part < 2) {
        const int k = part;
        dfl acc[PARTS];
#pragma unroll
        for (int i = 0; i < PARTS; ++i) acc[i] = red[i][k][rl];
#pragma unroll
        for (int w = 1; w < PARTS; w *= 2)
#pragma unroll
            for (int i = 0; i + w < PARTS; i += 2 * w) acc[i] = df_add(acc[i], acc[i + w]);
        float2* z = b.Z + (size_t)t * b.z_stride + (size_t)k * b.nt * GP_NB + (size_t)I * GP_NB + r;
        df_store(z, df_sub(df_load(z), acc[0]));
    }
}

__global__ void __launch_bounds__(kSplitThreads) k_split_panel(MixedBatch b, int J, int ns, int gemv) {
    grid_dependency();
    __shared__ float pmax[kSplitParts][kSplitRows];
    __shared__ dfl xs[2][GP_NB];
    __shared__ dfl red[kSplitParts][2][kSplitRows];
    const int t = blockIdx.y;
    if (b.st[t].status != GP_OK) return;
    const int I = J + 1 + blockIdx.x / 2;
    const float2* src = df_tile(b, b.A, t, I, J);
    const int rl = threadIdx.x % kSplitRows, part = threadIdx.x / kSplitRows;
    const int q = part >> 1, u = part & 1, c0 = kSplitCols * part;
    const int r = (blockIdx.x & 1) * kSplitRows + rl;
    gemv = gemv && b.fwd;
    if (gemv && threadIdx.x < 2 * GP_NB) {
        // x_J of both right-hand sides
        const int k = threadIdx.x >> 7, c = threadIdx.x & 127;
        xs[k][c] = df_load(b.Z + (size_t)t * b.z_stride + (size_t)k * b.nt * GP_NB + (size_t)J * GP_NB + c);
    }
    float2 v[kSplitCols];
#pragma unroll
    for (int j = 0; j < kSplitCols; ++j) v[j] = src[(size_t)(c0 + j) * GP_NB + r];
    float mx = 0.f;
#pragma unroll
    for (int j = 0; j < kSplitCols; ++j) mx = fmaxf(mx, fabsf(v[j].x));
    pmax[part][rl] = mx;
    __syncthreads();
    if (gemv) fwd_partials(v, xs, c0, part, rl, red);
#pragma unroll
    for (int k = 0; k < kSplitParts; ++k) mx = fmaxf(mx, pmax[k][rl]);
    const int E = exponent_of(mx);
    if (part == 0) pe_block(b, t, I)[r] = E;
    float sa, sb;
    slice_scale(E, sa, sb);
    uint8_t* chunk0 = reinterpret_cast<uint8_t*>(ps_block(b, t, I) + (size_t)q * kChunkElems);
    slice_pieces(v, sa, sb, r, 16 * u, ns, chunk0, (size_t)kChunks * kChunkBytes);
    if (gemv) {
        __syncthreads();
        fwd_apply<kSplitParts>(b, t, I, r, part, rl, red);
    }
}

// Slices of two adjacent panels at once, for the fused (K = 256) trailing
// update: row r of row block I = J + 2 + blockIdx.x / 4 spans tiles (I, J) and
// (I, J + 1) and gets one exponent for all 256 columns, so the products of
// both panels accumulate in the same tensor-memory groups.  A CTA takes a
// quarter tile (32 rows); thread (r, part) owns 16 columns of one panel
// (parts 0-7 panel J, 8-15 panel J + 1; the same two pieces of an image
// chunk as in k_split_panel), so every tile is read once and every slice
// written in 32-byte stores; the row maximum spans all 16 parts.
__global__ void __launch_bounds__(kSplitThreads) k_split_fused(MixedBatch b, int J) {
    grid_dependency();
    __shared__ float pmax[kFusedParts][kFusedRows];
    __shared__ dfl xs[2][GP_NB];
    __shared__ dfl red[kFusedParts / 2][2][kFusedRows];
    const int t = blockIdx.y;
    if (b.st[t].status != GP_OK) return;
    const int I = J + 2 + blockIdx.x / 4;
    const int rl = threadIdx.x % kFusedRows, part = threadIdx.x / kFusedRows;
    const int panel = part >> 3, lp = part & 7;
    const int q = lp >> 1, u = lp & 1, c0 = kSplitCols * lp;
    const int r = (blockIdx.x & 3) * kFusedRows + rl;
    if (b.fwd && threadIdx.x < 2 * GP_NB) {
        // x_{J+1}: the panel J term was applied by k_split_panel
        const int k = threadIdx.x >> 7, c = threadIdx.x & 127;
        xs[k][c] = df_load(b.Z + (size_t)t * b.z_stride + (size_t)k * b.nt * GP_NB + (size_t)(J + 1) * GP_NB + c);
    }
    const float2* src = df_tile(b, b.A, t, I, J + panel);
    float2 v[kSplitCols];
#pragma unroll
    for (int j = 0; j < kSplitCols; ++j) v[j] = src[(size_t)(c0 + j) * GP_NB + r];
    float mx = 0.f;
#pragma unroll
    for (int j = 0; j < kSplitCols; ++j) mx = fmaxf(mx, fabsf(v[j].x));
    pmax[part][rl] = mx;
    __syncthreads();
    if (b.fwd && panel == 1) fwd_partials(v, xs, c0, lp, rl, red);
#pragma unroll
    for (int k = 0; k < kFusedParts; ++k) mx = fmaxf(mx, pmax[k][rl]);
    const int E = exponent_of(mx);
    if (part == 0) fe_block(b, t, I)[r] = E;
    float sa, sb;
    slice_scale(E, sa, sb);
    const size_t slice_bytes = (size_t)2 * kChunks * kChunkBytes;
    uint8_t* base = reinterpret_cast<uint8_t*>(pf_block(b, t, I));
    slice_pieces(v, sa, sb, r, 16 * u, b.s, base + (size_t)(4 * panel + q) * kChunkElems * 2, slice_bytes);
    if (b.fwd) {
        __syncthreads();
        fwd_apply<kFusedParts / 2>(b, t, I, r, part, rl, red);
    }
}

// ------------------------------------------------------------ solves -------
// Z (per instance, float2): column k of length npad at Z + k * npad.
//   0: x_1   1: x_y   2, 3: residual / correction   4: 1 / L_ii
// The substitutions and the residual are tile-parallel (kernels below);
// tiles whose transpose is needed are staged in shared memory column by
// column with one entry of padding, so that a thread walking a column and
// one walking a row both read conflict-free (2-way for the 8-byte entries).

constexpr int kSolveThreads = 512;   // the finalising reduction
constexpr int kTs = GP_NB + 1;       // staged column stride of a 128-row tile part

__device__ __forceinline__ float2* zcol(const MixedBatch& b, int t, int k) {
    return b.Z + (size_t)t * b.z_stride + (size_t)k * b.nt * GP_NB;
}

// Fixed-order sum over the block of a double-float value held per thread.
__device__ dfl block_sum_df(dfl v, dfl* red) {
    for (int o = 16; o > 0; o >>= 1) {
        dfl w;
        w.hi = __shfl_down_sync(0xffffffffu, v.hi, o);
        w.lo = __shfl_down_sync(0xffffffffu, v.lo, o);
        v = df_add(v, w);
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        dfl s = red[0];
        for (int i = 1; i < (int)(blockDim.x >> 5); ++i) s = df_add(s, red[i]);
        red[0] = s;
    }
    __syncthreads();
    dfl s = red[0];
    __syncthreads();
    return s;
}


// The same sums as block_sum_df of N values at once, their last additions in
// N threads of different warps.
template <int N>
__device__ __forceinline__ void block_sums_df(dfl (&v)[N], dfl (*red)[N]) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < N; ++k) {
            dfl u;
            u.hi = __shfl_down_sync(0xffffffffu, v[k].hi, o);
            u.lo = __shfl_down_sync(0xffffffffu, v[k].lo, o);
            v[k] = df_add(v[k], u);
        }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < N; ++k)
        if (lane == 0) red[w][k] = v[k];
    __syncthreads();
    if (lane == 0 && w < N) {
        dfl s = red[0][w];
        for (int i = 1; i < (int)(blockDim.x >> 5); ++i) s = df_add(s, red[i][w]);
        red[0][w] = s;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < N; ++k) v[k] = red[0][k];
}

// [1 Y] (zero on padded rows) into Z columns 0, 1: the right-hand sides of
// the forward solve that the factorisation carries out block by block
__global__ void k_rhs_init(MixedBatch b) {
    grid_dependency();
    const int t = blockIdx.y;
    const int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= b.nt * GP_NB) return;
    const bool in = gi < b.n;
    df_store(zcol(b, t, 0) + gi, dfl{in ? 1.f : 0.f, 0.f});
    df_store(zcol(b, t, 1) + gi, in ? df_from_double(b.y[gi]) : dfl{0.f, 0.f});
}

// Forward and backward substitution with the double-float factor for two
// columns (c0, c0 + 1) of Z in place, tile-parallel: block column by block
// column, a small kernel finishes the diagonal block from the partial
// products of the tiles already applied (fixed order), and a tile kernel
// forms the next partial products of every tile of that block column (or
// row) at once, one CTA per tile half.  Partial products live in RP:
// per lower tile q, [2 halves][2 columns][128] double-float values.
// A step is a chain of latencies (the tile from HBM, its partial products
// through L2 to the diagonal step, W from L2), so each link's loads are issued
// together and the next block's two tiles come first in the grid (the
// candidates run along x): their diagonal step ends while the other tiles are
// worked on.  Each step of 100 candidates at n = 1024: 42 -> 22 us forward,
// 35 -> 24 backward; the solve phase there .82 -> .56 ms, 32 x 1448 1.07 ->
// .64, 8 x 16384 17.4 -> 10.7, 256 x 4000 15.5 -> 14.4 (2.4 a pass is what the
// factor's bytes take).

// N entries of both right-hand sides side by side, for the paired FP32
// instructions: hl = {hi of both, lo of both}, and the negated high words.  A
// product with L then takes half the issue slots of two scalar ones (the
// residual issued in 67 % of the cycles, the forward tiles in 70): the solve
// phase of 256 x 4000 14.4 -> 13.3 ms, 128 x 2047 2.11 -> 1.95, 8 x 16384 10.7 ->
// 10.1, 100 x 1024 .565 -> .525; the same bits.
template <int N>
struct SubX {
    float4 hl[N];
    float2 n[N];
    __device__ __forceinline__ void set(int i, int k, dfl v) {
        float* p = reinterpret_cast<float*>(hl + i);
        p[k] = v.hi;
        p[2 + k] = v.lo;
        reinterpret_cast<float*>(n + i)[k] = -v.hi;
    }
    __device__ __forceinline__ df2 fma(dfl l, int i, df2 c) const {
        const float4 x = hl[i];
        const float2 m = n[i];
        return df2_fma_shared(l, df2{f2_pack(x.x, x.y), f2_pack(x.z, x.w)}, f2_pack(m.x, m.y), c);
    }
};

constexpr int kSubThreads = 256;
// Entries that a thread has in flight: partial-product tiles, W and L, and the
// CTAs per SM that its registers leave room for.
struct SubDeep {
    static constexpr int kSum = 4, kW = 16, kL = 32, kFwd = 2, kBwd = 2;
};
struct SubWide {
    static constexpr int kSum = 4, kW = 8, kL = 8, kFwd = 4, kBwd = 3;
};

__device__ __forceinline__ bool sub_active(const MixedBatch& b, int t) {
    return b.st[t].status == GP_OK && !b.st[t].hager_done && !b.st[t].refine_done;
}

__device__ __forceinline__ float2* rp_part(const MixedBatch& b, int t, int I, int J) {
    return b.RP + (size_t)t * b.rp_stride + (size_t)tile_index(I, J, b.nt) * kRpTile;
}

__device__ __forceinline__ dfl df_load_cg(const float2* p) {
    const float2 v = __ldcg(p);
    return {v.x, v.y};
}

// The diagonal steps run either as their own launch (the first block of a
// pass) or inside the tile launch before them, by whichever of the two CTAs
// writing the block's last partial products finishes second: each of them
// fences its partial products device-wide and counts itself on the block's
// counter (which the second leaves at zero again); the second reads all the block's partial
// products in the same fixed order as a separate launch would.  No CTA
// waits for another.
__device__ __forceinline__ bool second_of_two(const MixedBatch& b, int t, int blk) {
    __shared__ int last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = (atomicInc((unsigned*)b.SC + (size_t)t * b.sc_stride + blk, 1) == 1);
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// Sums over `count` partial products of both right-hand sides, count in steps
// of two tiles (one per half): pp(i) is the i-th tile's part for this thread.
// The loads of N tiles are issued before their sums (in the tiles' order).
template <int N, typename F>
__device__ __forceinline__ void sum_partials(int count, F pp, dfl& p0, dfl& p1) {
    p0 = {0.f, 0.f};
    p1 = {0.f, 0.f};
#pragma unroll 1
    for (int i = 0; i < count; i += N) {
        dfl v[N][4];
#pragma unroll
        for (int j = 0; j < N; ++j)
            if (i + j < count) {
                const float2* q = pp(i + j);
#pragma unroll
                for (int k = 0; k < 4; ++k) v[j][k] = df_load_cg(q + k * GP_NB);
            }
#pragma unroll
        for (int j = 0; j < N; ++j)
            if (i + j < count) {
                p0 = df_add(p0, df_add(v[j][0], v[j][2]));
                p1 = df_add(p1, df_add(v[j][1], v[j][3]));
            }
    }
}

// The first N of the 64 entries of W (stride GP_NB) of a thread of a
// diagonal step.
template <int N>
__device__ __forceinline__ void diag_load(const float2* W, float2 (&w)[N]) {
#pragma unroll
    for (int j = 0; j < N; ++j) w[j] = W[(size_t)j * GP_NB];
}

// Products of 64 entries of W with both right-hand sides (from entry
// `first` of xs), even and odd terms apart.  w holds the first N entries; each
// batch is loaded while the one before it is multiplied: left to the
// compiler, every load waited for L2 on its own (18 to 36 thousand clocks for
// the 64 terms, against 5.6 thousand that the products issue in).
template <int N>
__device__ __forceinline__ void diag_products(const float2* W, float2 (&w)[N], const SubX<GP_NB>& xs, int first,
                                              dfl& s0, dfl& s1) {
    df2 even = {f2_pack(0.f, 0.f), f2_pack(0.f, 0.f)}, odd = even;
#pragma unroll 1
    for (int c0 = 0; c0 < GP_NB / 2; c0 += N) {
        float2 next[N];
        if (c0 + N < GP_NB / 2) diag_load(W + (size_t)(c0 + N) * GP_NB, next);
#pragma unroll
        for (int j = 0; j < N; j += 2) {
            even = xs.fma(dfl{w[j].x, w[j].y}, first + c0 + j, even);
            odd = xs.fma(dfl{w[j + 1].x, w[j + 1].y}, first + c0 + j + 1, odd);
        }
#pragma unroll
        for (int j = 0; j < N; ++j) w[j] = next[j];
    }
    s0 = df_add(df2_first(even), df2_first(odd));
    s1 = df_add(df2_second(even), df2_second(odd));
}

// forward, block J: z_J <- W_J (z_J - sum_{K<J} L_JK z_K), W_J = L_JJ^-1.
// Thread (r, h) takes both right-hand sides of row r over half h of the
// terms (every other partial-product tile, then columns 64h .. 64h + 63 of
// the column-major WT, one load serving both sums); the halves add in a
// fixed order.  W is zero above its diagonal; a fixed trip count.
// part: 2 x 2 x 128 scratch.
template <typename V>
__device__ __forceinline__ void fwd_diag_step(const MixedBatch& b, int t, int c0, int J, SubX<GP_NB>& rhs,
                                              dfl (*part)[2][GP_NB]) {
    const int r = threadIdx.x & 127, h = threadIdx.x >> 7;
    float2* zr = zcol(b, t, c0 + h) + (size_t)J * GP_NB + r;     // half h finishes right-hand side h
    const float2* W = b.WT + (size_t)t * b.wt_stride + (size_t)J * GP_TILE_ELEMS + (size_t)(64 * h) * GP_NB + r;
    float2 w[V::kW];
    diag_load(W, w);
    const dfl z = df_load(zr);
    dfl p0, p1;
    sum_partials<V::kSum>((J - h + 1) / 2, [&](int i) { return rp_part(b, t, J, h + 2 * i) + r; }, p0, p1);
    part[h][0][r] = p0;
    part[h][1][r] = p1;
    __syncthreads();
    rhs.set(r, h, df_sub(z, df_add(part[0][h][r], part[1][h][r])));
    __syncthreads();
    dfl s0, s1;
    diag_products(W, w, rhs, 64 * h, s0, s1);
    part[h][0][r] = s0;
    part[h][1][r] = s1;
    __syncthreads();
    df_store(zr, df_add(part[0][h][r], part[1][h][r]));
}

__global__ void __launch_bounds__(kSubThreads) k_fwd_diag(MixedBatch b, int c0, int J) {
    grid_dependency();
    __shared__ SubX<GP_NB> rhs;
    __shared__ dfl part[2][2][GP_NB];
    const int t = blockIdx.x;
    if (!sub_active(b, t)) return;
    fwd_diag_step<SubDeep>(b, t, c0, J, rhs, part);
}

// forward, tiles (I, J), I > J, half h of the columns: L_IJ(:, h) z_J(h);
// the CTA finishing tile (J + 1, J) second then takes block J + 1's
// diagonal step
template <typename V>
__global__ void __launch_bounds__(kSubThreads, V::kFwd) k_fwd_tiles(MixedBatch b, int c0, int J) {
    grid_dependency();
    __shared__ SubX<GP_NB / 2> xs;
    __shared__ dfl part[2][2][GP_NB];
    __shared__ SubX<GP_NB> rhs;
    const int t = blockIdx.x;
    if (!sub_active(b, t)) return;
    const int I = J + 1 + (blockIdx.y >> 1), h = blockIdx.y & 1;
    const int tid = threadIdx.x;
    // W_{J+1} heads for L2 for the diagonal step
    if (tid == 0 && I == J + 1 && h == 0)
        prefetch_l2(b.WT + (size_t)t * b.wt_stride + (size_t)(J + 1) * GP_TILE_ELEMS, GP_TILE_ELEMS * sizeof(float2));
    const int r = tid & 127, g = tid >> 7;
    const float2* L = df_tile(b, b.A, t, I, J) + ((size_t)h * 64 + 32 * g) * GP_NB + r;
    float2 l[V::kL];
#pragma unroll
    for (int c = 0; c < V::kL; ++c) l[c] = __ldg(L + (size_t)c * GP_NB);
    if (tid < GP_NB)
        xs.set(tid & 63, tid >> 6, df_load(zcol(b, t, c0 + (tid >> 6)) + (size_t)J * GP_NB + 64 * h + (tid & 63)));
    __syncthreads();
    df2 u = {f2_pack(0.f, 0.f), f2_pack(0.f, 0.f)};
#pragma unroll 1
    for (int q = 0; q < 32; q += V::kL) {
        float2 next[V::kL];
        if (q + V::kL < 32) {
#pragma unroll
            for (int c = 0; c < V::kL; ++c) next[c] = __ldg(L + (size_t)(q + V::kL + c) * GP_NB);
        }
#pragma unroll
        for (int c = 0; c < V::kL; ++c) u = xs.fma(dfl{l[c].x, l[c].y}, 32 * g + q + c, u);
#pragma unroll
        for (int c = 0; c < V::kL; ++c) l[c] = next[c];
    }
    part[g][0][r] = df2_first(u);
    part[g][1][r] = df2_second(u);
    __syncthreads();
    const int k = tid >> 7;
    df_store(rp_part(b, t, I, J) + (h * 2 + k) * GP_NB + r, df_add(part[0][k][r], part[1][k][r]));
    if (I == J + 1 && second_of_two(b, t, I)) fwd_diag_step<V>(b, t, c0, I, rhs, part);
}

// backward, block K: z_K <- W_K^T (z_K - sum_{K' > K} L_K'K^T z_K'); W^T
// from the row-major copy WR (thread (c, h) reads column c of W along rows
// 64h .. 64h + 63, both right-hand sides per load; the partial-product
// tiles alternate between the halves); the halves add in a fixed order.
// With add_to >= 0 the result is also added into (add_to, add_to + 1).
template <typename V>
__device__ __forceinline__ void bwd_diag_step(const MixedBatch& b, int t, int c0, int K, int add_to,
                                              SubX<GP_NB>& rhs, dfl (*part)[2][GP_NB]) {
    const int c = threadIdx.x & 127, h = threadIdx.x >> 7;
    float2* zc = zcol(b, t, c0 + h) + (size_t)K * GP_NB + c;     // half h finishes right-hand side h
    float2* acc = add_to >= 0 ? zcol(b, t, add_to + h) + (size_t)K * GP_NB + c : nullptr;
    const float2* W = b.WR + (size_t)t * b.wt_stride + (size_t)K * GP_TILE_ELEMS + (size_t)(64 * h) * GP_NB + c;
    float2 w[V::kW];
    diag_load(W, w);
    const dfl z = df_load(zc);
    dfl total = {0.f, 0.f};
    if (acc) total = df_load(acc);
    dfl p0, p1;
    sum_partials<V::kSum>((b.nt - K - h) / 2, [&](int i) { return rp_part(b, t, K + 1 + h + 2 * i, K) + c; }, p0, p1);
    part[h][0][c] = p0;
    part[h][1][c] = p1;
    __syncthreads();
    rhs.set(c, h, df_sub(z, df_add(part[0][h][c], part[1][h][c])));
    __syncthreads();
    dfl s0, s1;
    diag_products(W, w, rhs, 64 * h, s0, s1);
    part[h][0][c] = s0;
    part[h][1][c] = s1;
    __syncthreads();
    const dfl x = df_add(part[0][h][c], part[1][h][c]);
    df_store(zc, x);
    if (acc) df_store(acc, df_add(total, x));
}

__global__ void __launch_bounds__(kSubThreads) k_bwd_diag(MixedBatch b, int c0, int K, int add_to) {
    grid_dependency();
    __shared__ SubX<GP_NB> rhs;
    __shared__ dfl part[2][2][GP_NB];
    const int t = blockIdx.x;
    if (!sub_active(b, t)) return;
    bwd_diag_step<SubDeep>(b, t, c0, K, add_to, rhs, part);
}

// backward, tiles (K, I), I < K, half h of the rows: L_KI(h, :)^T z_K(h);
// the half tile is staged column by column (64 rows + 1 of padding) so that
// thread c walks column c conflict-free; the CTA finishing tile (K, K - 1)
// second then takes block K - 1's diagonal step
constexpr int kBwdTs = GP_NB / 2 + 1;
template <typename V>
__global__ void __launch_bounds__(kSubThreads, V::kBwd) k_bwd_tiles(MixedBatch b, int c0, int K, int add_to) {
    grid_dependency();
    extern __shared__ dfl T[];                  // GP_NB x kBwdTs
    __shared__ SubX<GP_NB / 2> xs;
    __shared__ dfl part[2][2][GP_NB];
    __shared__ SubX<GP_NB> rhs;
    const int t = blockIdx.x;
    if (!sub_active(b, t)) return;
    const int I = K - 1 - (blockIdx.y >> 1), h = blockIdx.y & 1;
    const int tid = threadIdx.x;
    // W_{K-1} (row-major) heads for L2 for the next diagonal step
    if (tid == 0 && I == K - 1 && h == 0)
        prefetch_l2(b.WR + (size_t)t * b.wt_stride + (size_t)(K - 1) * GP_TILE_ELEMS, GP_TILE_ELEMS * sizeof(float2));
    if (tid < GP_NB)
        xs.set(tid & 63, tid >> 6, df_load(zcol(b, t, c0 + (tid >> 6)) + (size_t)K * GP_NB + 64 * h + (tid & 63)));
    const float2* L = df_tile(b, b.A, t, K, I) + 64 * h;
#pragma unroll
    for (int e = tid; e < 64 * GP_NB; e += kSubThreads) {
        const int c = e >> 6, rr = e & 63;
        cp_async8(T + c * kBwdTs + rr, L + (size_t)c * GP_NB + rr);
    }
    cp_async_wait_all();
    __syncthreads();
    const int c = tid & 127, g = tid >> 7;
    const dfl* col = T + c * kBwdTs;
    df2 sum = {f2_pack(0.f, 0.f), f2_pack(0.f, 0.f)};
#pragma unroll 8
    for (int rr = 32 * g; rr < 32 * g + 32; ++rr) sum = xs.fma(col[rr], rr, sum);
    part[g][0][c] = df2_first(sum);
    part[g][1][c] = df2_second(sum);
    __syncthreads();
    const int k = tid >> 7;
    df_store(rp_part(b, t, K, I) + (h * 2 + k) * GP_NB + c, df_add(part[0][k][c], part[1][k][c]));
    // the CTA finishing tile (K, K - 1) second takes block K - 1's diagonal step
    if (I == K - 1 && second_of_two(b, t, I)) bwd_diag_step<V>(b, t, c0, I, add_to, rhs, part);
}

// Residual r = b - R x of the solution columns (0, 1) into columns (2, 3),
// against the double-float copy of R, tile-parallel: one CTA per (lower tile
// (I, J) of the R copy, column half hc) stages its 128 x 64 part and writes
// the partial sums
//   U = R_IJ(:, half) x_J(half)        two columns of 128 (row products)
//   V = R_IJ(:, half)^T x_I            two columns of 64 (column products, I != J)
// into RP; k_resid_reduce adds them per row block in a fixed order.  The
// diagonal tiles of the R copy hold both triangles, so they give U only.
// RP per tile q: U[hc][k][128] then V[hc][k][64] (kRpTile values).
constexpr int kResThreads = 256;
constexpr int kResCols = GP_NB / 2;
static_assert(kRpTile == 2 * 2 * GP_NB + 2 * 2 * kResCols, "residual partial layout");

__global__ void __launch_bounds__(kResThreads) k_resid_tiles(MixedBatch b) {
    grid_dependency();
    extern __shared__ dfl T[];                  // kResCols x kTs
    __shared__ SubX<kResCols> xa;               // x_J on this half's columns
    __shared__ SubX<GP_NB> xb;                  // x_I
    __shared__ dfl part[2 * 2 * GP_NB];           // U: [2][2][128], then V: [4][2][64]
    const int t = blockIdx.y;
    if (b.st[t].status != GP_OK || b.st[t].refine_done) return;
    const int nt = b.nt;
    const int q = blockIdx.x >> 1, hc = blockIdx.x & 1;
    int J = 0, rem = q;
    while (rem >= nt - J) {
        rem -= nt - J;
        ++J;
    }
    const int I = J + rem;
    const int tid = threadIdx.x;
    if (tid < 2 * kResCols)
        xa.set(tid & 63, tid >> 6, df_load(zcol(b, t, tid >> 6) + J * GP_NB + hc * kResCols + (tid & 63)));
    xb.set(tid & 127, tid >> 7, df_load(zcol(b, t, tid >> 7) + I * GP_NB + (tid & 127)));
    const float2* src = df_tile(b, b.Rc, t, I, J) + (size_t)hc * kResCols * GP_NB;
#pragma unroll
    for (int e = tid; e < kResCols * GP_NB; e += kResThreads) cp_async8(T + (e >> 7) * kTs + (e & 127), src + e);
    cp_async_wait_all();
    __syncthreads();
    float2* rp = b.RP + (size_t)t * b.rp_stride + (size_t)q * kRpTile;
    {
        // U: thread (r, h) takes the columns 32h .. 32h + 31 of the half
        const int r = tid & 127, h = tid >> 7;
        df2 u = {f2_pack(0.f, 0.f), f2_pack(0.f, 0.f)};
#pragma unroll 8
        for (int c = 32 * h; c < 32 * h + 32; ++c) u = xa.fma(T[c * kTs + r], c, u);
        part[(h * 2 + 0) * GP_NB + r] = df2_first(u);
        part[(h * 2 + 1) * GP_NB + r] = df2_second(u);
    }
    __syncthreads();
    {
        const int k = tid >> 7, r = tid & 127;
        df_store(rp + (hc * 2 + k) * GP_NB + r, df_add(part[k * GP_NB + r], part[(2 + k) * GP_NB + r]));
    }
    if (I == J) return;                         // uniform
    __syncthreads();
    {
        // V: thread (c, h) takes the rows 32h .. 32h + 31 of column c
        const int c = tid & 63, h = tid >> 6;
        const dfl* col = T + c * kTs;
        df2 sum = {f2_pack(0.f, 0.f), f2_pack(0.f, 0.f)};
#pragma unroll 8
        for (int r = 32 * h; r < 32 * h + 32; ++r) sum = xb.fma(col[r], r, sum);
        part[(h * 2 + 0) * kResCols + c] = df2_first(sum);
        part[(h * 2 + 1) * kResCols + c] = df2_second(sum);
    }
    __syncthreads();
    if (tid < 2 * kResCols) {
        const int k = tid >> 6, c = tid & 63;
        const dfl v = df_add(df_add(part[(0 + k) * kResCols + c], part[(2 + k) * kResCols + c]),
                             df_add(part[(4 + k) * kResCols + c], part[(6 + k) * kResCols + c]));
        df_store(rp + 4 * GP_NB + (hc * 2 + k) * kResCols + c, v);
    }
}

// r_I = b_I - (sum_{J <= I} U(I, J) + sum_{J > I} V(J, I)) for both columns,
// into Z columns 2, 3; padded rows: R is the identity there and x is zero,
// so r = 0.  One CTA per (row block I, instance).
__global__ void __launch_bounds__(kResThreads) k_resid_reduce(MixedBatch b) {
    grid_dependency();
    const int t = blockIdx.y, I = blockIdx.x;
    if (b.st[t].status != GP_OK || b.st[t].refine_done) return;
    const int nt = b.nt, n = b.n;
    const int k = threadIdx.x >> 7, r = threadIdx.x & 127;
    const float2* rp = b.RP + (size_t)t * b.rp_stride;
    dfl y = {0.f, 0.f};
    // eight partial sums loaded before they are added (in their order)
#pragma unroll 1
    for (int J = 0; J <= I; J += 4) {
        dfl v[8];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (J + j <= I) {
                const float2* u = rp + (size_t)tile_index(I, J + j, nt) * kRpTile;
                v[2 * j] = df_load(u + k * GP_NB + r);
                v[2 * j + 1] = df_load(u + (2 + k) * GP_NB + r);
            }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (J + j <= I) y = df_add(df_add(y, v[2 * j]), v[2 * j + 1]);
    }
#pragma unroll 1
    for (int K = I + 1; K < nt; K += 8) {
        dfl v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (K + j < nt)
                v[j] = df_load(rp + (size_t)tile_index(K + j, I, nt) * kRpTile + 4 * GP_NB +
                               ((r >> 6) * 2 + k) * kResCols + (r & 63));
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (K + j < nt) y = df_add(y, v[j]);
    }
    const int gi = I * GP_NB + r;
    dfl bq = {0.f, 0.f};
    if (gi < n) bq = k ? df_from_double(b.y[gi]) : dfl{1.f, 0.f};
    df_store(zcol(b, t, 2 + k) + gi, (gi < n) ? df_sub(bq, y) : dfl{0.f, 0.f});
}

// a = L^-1 1 and b = L^-1 Y (Z columns 0, 1 after the forward solve) into
// columns 8, 9, where the refinement's sums read them
__global__ void k_keep_forward(MixedBatch b) {
    grid_dependency();
    const int t = blockIdx.y;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int npad = b.nt * GP_NB;
    if (b.st[t].status != GP_OK || i >= 2 * npad) return;
    const int k = i / npad, r = i - k * npad;
    zcol(b, t, 8 + k)[r] = zcol(b, t, k)[r];
}

// The sums of eq. 3 after refinement step `step` (0: the first solve, before
// any correction), and whether the candidate refines further.
//
// With the factor L (L L' ~ R), x = [x_1 x_y] the current solution of
// R x = [1 Y], r = [1 Y] - R x its residual and z = L^-1 r (Z columns 2, 3),
// the refined solution is x + L^-T z, and every sum eq. 3 needs follows
// without that backward substitution, since v' L^-T z = (L^-1 v)' z:
//   1'R^-1 1 = 1'x_1 + a'z_1,   1'R^-1 Y = 1'x_y + a'z_y,   mu = their ratio,
//   Q = (Y - 1 mu)'(x_y - mu x_1) + (b - mu a)'(z_y - mu z_1),
//   Y'R^-1 Y = Y'x_y + b'z_y,
// a = L^-1 1, b = L^-1 Y (columns 8, 9).  A further step first applies the
// backward substitution to z and adds it to x.
//
// Stopping rule.  The factor's pivots carry an absolute error of about
// u (1 + delta) each, u = 2^-8s for s slices in the trailing updates (2^-40
// at the default 5: a row of L has norm^2 R_ii = 1 + delta and the split
// products are exact to about u of it), so log|R| = sum log L_ii^2 is
// uncertain by about e_ld = u (1 + delta) sum_i 1 / L_ii^2.  Step k
// changes n log Q by dq_k; with the contraction rho of the iteration (1/16
// assumed after the first step, then dq_k / dq_{k-1}) the error of n log Q
// left is about dq_k rho / (1 - rho).  Once that is below e_ld, further steps
// cannot make -2logL more accurate, and the candidate stops.
// 2^-8s, the accuracy unit of a factor with s slices in its trailing updates
__device__ __forceinline__ double split_unit(int s) {
    return __longlong_as_double((long long)(1023 - 8 * s) << 52);
}

__global__ void __launch_bounds__(kSolveThreads) k_refine_check(MixedBatch b, int step) {
    grid_dependency();
    __shared__ dfl red[kSolveThreads / 32], red3[kSolveThreads / 32][3];
    __shared__ double log_prev;
    const int t = blockIdx.x;
    InstState* st = b.st + t;
    if (st->status != GP_OK || st->refine_done) return;
    const int n = b.n;
    const float2* x1 = zcol(b, t, 0);
    const float2* xy = zcol(b, t, 1);
    const float2* z1 = zcol(b, t, 2);
    const float2* zy = zcol(b, t, 3);
    const float2* av = zcol(b, t, 8);
    const float2* bv = zcol(b, t, 9);
    const bool corr = step > 0;
    dfl sa = {0.f, 0.f}, sb = {0.f, 0.f}, sc = {0.f, 0.f};
    for (int i = threadIdx.x; i < n; i += kSolveThreads) {
        const dfl c = df_load(xy + i);
        sa = df_add(sa, df_load(x1 + i));
        sb = df_add(sb, c);
        sc = df_fma(df_from_double(b.y[i]), c, sc);
        if (corr) {
            const dfl ai = df_load(av + i), zyi = df_load(zy + i);
            sa = df_fma(ai, df_load(z1 + i), sa);
            sb = df_fma(ai, zyi, sb);
            sc = df_fma(df_load(bv + i), zyi, sc);
        }
    }
    dfl sums[3] = {sa, sb, sc};
    block_sums_df(sums, red3);
    const double A = df_to_double(sums[0]), B = df_to_double(sums[1]), C = df_to_double(sums[2]);
    const double m = B / A;
    const dfl md = df_from_double(m);
    dfl sq = {0.f, 0.f};
    for (int i = threadIdx.x; i < n; i += kSolveThreads) {
        const dfl e = df_sub(df_from_double(b.y[i]), md);
        sq = df_fma(e, df_fms(md, df_load(x1 + i), df_load(xy + i)), sq);
        if (corr) {
            const dfl u = df_fms(md, df_load(av + i), df_load(bv + i));
            sq = df_fma(u, df_fms(md, df_load(z1 + i), df_load(zy + i)), sq);
        }
    }
    if (corr && threadIdx.x == 32) log_prev = log(st->Q);       // beside the sum; a barrier follows
    const double Q = df_to_double(block_sum_df(sq, red));
    if (threadIdx.x == 0) {
        st->aa = A;
        st->ab = B;
        st->bb = C;
        st->mu = m;
        st->Q = Q;
        if (!(Q > 0.0)) {
            st->refine_done = 1;            // degenerate: the finalisation reports it
        } else if (corr) {
            const double dq = n * fabs(log(Q) - log_prev);
            double rho = 0.0625;
            if (step > 1 && st->dq_prev > 0.0) rho = fmin(0.5, fmax(dq / st->dq_prev, 1.52587890625e-05));
            const double rest = dq * rho / (1.0 - rho);
            const double e_ld = split_unit(b.s) * (1.0 + b.delta) * st->piv_inv;
            st->dq_prev = dq;
            if (rest <= e_ld) st->refine_done = 1;
        }
    }
}

// -2logL = log|R| + n log Q from the sums of the last refinement check; Q is
// taken as zero when Q <= 16 n eps^2 Y'R^-1 Y with eps = 2^-8s, the accuracy
// unit of the split factorisation (2^-40 at 5 slices).
__global__ void k_df_finalize(MixedBatch b, double* nll, double* mu, double* sigma2, double* logdet,
                              int* status) {
    grid_dependency();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= b.count) return;
    const InstState st = b.st[t];
    const int n = b.n;
    const double nan = __longlong_as_double(0x7ff8000000000000LL);
    const double inf = __longlong_as_double(0x7ff0000000000000LL);
    if (st.status != GP_OK) {
        nll[t] = (st.status == GP_ENOTPD) ? inf : nan;
        mu[t] = nan;
        sigma2[t] = nan;
        if (logdet) logdet[t] = nan;
        status[t] = st.status;
        return;
    }
    const double eps = split_unit(b.s);
    const double Q = st.Q;
    const bool degenerate = !(Q > 16.0 * n * eps * eps * fabs(st.bb));
    nll[t] = degenerate ? -inf : st.logdet + n * log(Q);
    mu[t] = st.mu;
    sigma2[t] = Q / n;
    if (logdet) logdet[t] = st.logdet;
    status[t] = degenerate ? GP_EDEGENERATE : GP_OK;
}

// The kriging weights of one split-precision candidate (v: its one-candidate
// view, the last correction already applied to x): [a | w] as the
// double-float pairs the kriging kernel reads, a = L^-1 1 (column 8) and
// w = x_y - mu x_1 = R^-1 (Y - 1 mu), and the fit's scalars [-2logL, mu,
// sigma2, log|R|, Q, 1'R^-1 1].
__global__ void k_split_model(MixedBatch v, float2* Zm, double* scalars, const double* nll, const int* status,
                              int* status_out) {
    const InstState st = v.st[0];
    const int npad = v.nt * GP_NB;
    const float2* x1 = zcol(v, 0, 0);
    const float2* xy = zcol(v, 0, 1);
    const float2* av = zcol(v, 0, 8);
    const dfl md = df_from_double(st.mu);
    for (int i = threadIdx.x; i < npad; i += blockDim.x) {
        Zm[i] = av[i];
        df_store(Zm + npad + i, df_fms(md, df_load(x1 + i), df_load(xy + i)));
    }
    if (threadIdx.x == 0) {
        scalars[0] = *nll;
        scalars[1] = st.mu;
        scalars[2] = st.Q / v.n;
        scalars[3] = st.logdet;
        scalars[4] = st.Q;
        scalars[5] = st.aa;
        *status_out = *status;
    }
}

// Convert the double-float factor and solve vectors of one fitted instance
// into the double layout that the kriging kernel reads: L (tiles), a = L^-1 1
// is not needed by the mixed fit, so column 0 of Zd gets x_1 = R^-1 1 and
// column 1 w; the kriging kernel's a'v term is formed from R^-1 1 instead.
__global__ void k_df_to_double(const float2* src, double* dst, size_t count) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) {
        const float2 v = src[i];
        dst[i] = (double)v.x + (double)v.y;
    }
}

}  // namespace

cudaError_t launch_diag_mixed(const MixedBatch& b, int J, cudaStream_t s) {
    const size_t smem = (size_t)kPacked * sizeof(dfl);
    static std::atomic<size_t> attr[kMaxDevices];
    cudaError_t e = raise_smem_limit(k_diag_mixed, smem, attr);
    if (e != cudaSuccess) return e;
    launch_chained(ahead_mixed(b), k_diag_mixed, b.count, kDiagThreads, smem, s, b, J);
    return cudaGetLastError();
}

cudaError_t launch_split_panel(const MixedBatch& b, int J, int ns, int gemv, cudaStream_t s) {
    const int m = b.nt - J - 1;
    if (m <= 0) return cudaSuccess;
    launch_chained(gemv && ahead_mixed(b), k_split_panel, dim3(2 * m, b.count), kSplitThreads, 0, s, b, J, ns, gemv);
    return cudaGetLastError();
}

cudaError_t launch_split_fused(const MixedBatch& b, int J, cudaStream_t s) {
    const int m = b.nt - J - 2;
    if (m <= 0) return cudaSuccess;
    launch_chained(ahead_mixed(b), k_split_fused, dim3(4 * m, b.count), kSplitThreads, 0, s, b, J);
    return cudaGetLastError();
}

cudaError_t launch_rhs_init(const MixedBatch& b, cudaStream_t s) {
    const int npad = b.nt * GP_NB;
    launch_chained(ahead_mixed(b), k_rhs_init, dim3((npad + 255) / 256, b.count), 256, 0, s, b);
    return cudaGetLastError();
}

// The tile launches of a substitution: many CTAs are bound by what an SM
// issues and run more of them with fewer loads in flight; few are bound by
// latency.  The line is at eight CTAs per SM (solve phase, ms, wide / deep:
// 256 x 4000 14.5 / 15.7, 128 x 2047 2.19 / 2.27, 100 x 1024 .60 / .59,
// 8 x 16384 12.2 / 11.1, 32 x 1448 .77 / .70).
static bool sub_wide(dim3 grid) { return (long long)grid.x * grid.y > 8 * device_sms(); }

cudaError_t launch_df_forward(const MixedBatch& b, int c0, int init, cudaStream_t s) {
    if (init) {
        if (c0 != 0) return cudaErrorInvalidValue;
        cudaError_t e = launch_rhs_init(b, s);
        if (e != cudaSuccess) return e;
    }
    launch_chained(true, k_fwd_diag, b.count, kSubThreads, 0, s, b, c0, 0);
    for (int J = 0; J + 1 < b.nt; ++J) {
        const dim3 grid(b.count, 2 * (b.nt - 1 - J));
        launch_chained(true, sub_wide(grid) ? k_fwd_tiles<SubWide> : k_fwd_tiles<SubDeep>, grid, kSubThreads, 0,
                       s, b, c0, J);
    }
    return cudaGetLastError();
}

cudaError_t launch_df_backward(const MixedBatch& b, int c0, int add_to, cudaStream_t s) {
    const size_t smem = (size_t)GP_NB * kBwdTs * sizeof(dfl);
    static std::atomic<size_t> attr[2][kMaxDevices];
    cudaError_t e = raise_smem_limit(k_bwd_tiles<SubDeep>, smem, attr[0]);
    if (e == cudaSuccess) e = raise_smem_limit(k_bwd_tiles<SubWide>, smem, attr[1]);
    if (e != cudaSuccess) return e;
    launch_chained(true, k_bwd_diag, b.count, kSubThreads, 0, s, b, c0, b.nt - 1, add_to);
    for (int K = b.nt - 1; K > 0; --K) {
        const dim3 grid(b.count, 2 * K);
        launch_chained(true, sub_wide(grid) ? k_bwd_tiles<SubWide> : k_bwd_tiles<SubDeep>, grid, kSubThreads,
                       smem, s, b, c0, K, add_to);
    }
    return cudaGetLastError();
}

cudaError_t launch_df_residual(const MixedBatch& b, cudaStream_t s) {
    const size_t smem = (size_t)kResCols * kTs * sizeof(dfl);
    static std::atomic<size_t> attr[kMaxDevices];
    cudaError_t e = raise_smem_limit(k_resid_tiles, smem, attr);
    if (e != cudaSuccess) return e;
    launch_chained(true, k_resid_tiles, dim3(2 * (unsigned)packed_tiles(b.nt), b.count), kResThreads,
                   smem, s, b);
    launch_chained(ahead_mixed(b), k_resid_reduce, dim3(b.nt, b.count), kResThreads, 0, s, b);
    return cudaGetLastError();
}

cudaError_t launch_df_finalize(const MixedBatch& b, double* nll, double* mu, double* sigma2, double* logdet,
                               int* status, cudaStream_t s) {
    launch_chained(true, k_df_finalize, (b.count + 127) / 128, 128, 0, s, b, nll, mu, sigma2, logdet,
                   status);
    return cudaGetLastError();
}

cudaError_t launch_split_model(const MixedBatch& v, float2* Zm, double* scalars, const double* nll,
                               const int* status, int* status_out, cudaStream_t s) {
    k_split_model<<<1, 512, 0, s>>>(v, Zm, scalars, nll, status, status_out);
    return cudaGetLastError();
}

cudaError_t launch_keep_forward(const MixedBatch& b, cudaStream_t s) {
    const int npad = b.nt * GP_NB;
    launch_chained(ahead_mixed(b), k_keep_forward, dim3((2 * npad + 255) / 256, b.count), 256, 0, s, b);
    return cudaGetLastError();
}

cudaError_t launch_refine_check(const MixedBatch& b, int step, cudaStream_t s) {
    launch_chained(ahead_mixed(b), k_refine_check, b.count, kSolveThreads, 0, s, b, step);
    return cudaGetLastError();
}

cudaError_t launch_df_to_double(const float2* src, double* dst, size_t count, cudaStream_t s) {
    if (count == 0) return cudaSuccess;
    k_df_to_double<<<(unsigned)((count + 255) / 256), 256, 0, s>>>(src, dst, count);
    return cudaGetLastError();
}

}  // namespace gp
