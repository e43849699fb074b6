// k_update_tc.cu -- the trailing update of the double-precision Cholesky,
// A_IK -= L_IJ L_KJ^T, as exact products of 8-bit digits on the tensor cores
// (after Ozaki, Ogita, Oishi & Rump, "Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication", Numer.
// Algorithms 59, 2012).
//
// An off-diagonal entry of L is at most 1 in magnitude, whatever the nugget:
// sum_{k<i} l_ik^2 = 1 + delta - l_ii^2 and l_ii^2 >= delta for a positive
// semidefinite R.  So every entry is cut at one fixed scale, with no row
// exponents:
//   X = round(l 2^56) = sum_{a=0..6} q_a 256^(6-a),  |q_a| <= 128 (a > 0), |q_0| <= 256
// (balanced digits), each digit exact in fp16.  The product groups S_g =
// sum_{a+b=g} q_a q_b', g = 0 .. 7, summed over the panel's 128 columns in fp32
// are integers below 2^24, hence exact (at most 2^21 for a pair of lower
// digits, of which a group has six at most, and less than 2^18.6 by
// Cauchy-Schwarz for a pair with q_0, since the rows of L have norm 1; the
// inverse's operands, which have no such norm: at combine() below); what
// is left out, a + b >= 8, is below 2^-66 of 1 per term.  Rounding moves l by at
// most 2^-57, so that all panels together leave sum_k (|l_ik| + |l_jk|) 2^-57 in an
// entry of A at most, and about 2^-57 as a root mean square, where IEEE
// multiply-adds leave up to 2^-53 of the entry per panel column.  The unit is
// absolute: entries of L below 2^-3 keep fewer than 53 bits in the products,
// so the bound holds for the matrix, not entry by entry.  R - L L' over 50
// matrices (n = 300 .. 5000, d = 2 .. 12, p = 1 .. 2, delta = 0 .. 1) against IEEE
// multiply-adds: its largest entry 0.08 to 0.67 times, its root mean square 0.10
// to 1.0 times in 46 of them and up to 1.5 times (1.0e-17) in the four whose
// entries of R are smallest.
//
// The digits are cut on the way into shared memory by eight converter
// warps, from the double tiles themselves: no workspace, so the callers'
// memory is the same on either path.
//
// Bound by the tensor pipe: an M = 128, N = 64 product of K = 16 takes 80
// cycles here (its operands' shared-memory reads), so a half tile's 272 take
// 22 k cycles, then the groups' sum in front of the next tile 3 k (5 k with
// every group through the conversion instruction).  The cutting runs beside
// it since it costs 15 integer instructions an entry and 2 a digit (38 in
// all, where it set the pace: 19.9 -> 15 us a half tile).
// Measured, max |R - L L'| at n = 900, d = 2: 1.3e-16 (1.6e-15 with double
// multiply-adds on the FP64 pipe).  Twelve candidates at n = 4064: 270 ms with
// the updates on the FP64 pipe (256 of them), 28.9 ms now (updates 19); the
// double fit at n = 4064 54.6 -> 10.5 ms (9.65 with its launches set up ahead).
#include "mixed_common.cuh"

namespace gp {

namespace {

constexpr int kNS = 7;                        // digits per entry
constexpr int kNG = 8;                        // accumulator groups a + b = g
constexpr uint32_t kABytes = kNS * kChunkBytes;           // 128 rows x 32 columns, every digit
// NT columns of an output tile (64: half tiles of the trailing update; 32: a
// panel's inner update)
constexpr uint32_t b_chunk(int nt) { return kChunkBytes / (GP_NB / nt); }
constexpr uint32_t stage_bytes(int nt) { return kABytes + kNS * b_chunk(nt); }
constexpr int kConvWarps = 8, kEpiWarps = 8;
constexpr int kConvBase = 4, kEpiBase = kConvBase + kConvWarps;
constexpr int kThreads = 32 * (kEpiBase + kEpiWarps);     // warpgroup 0: the MMA warp (and three idle ones)
constexpr int kPieces = 3;                                // most (32 rows x 8 columns) pieces of a stage per warp
// registers after the split; their sum fits the launch's 96 a thread
constexpr int kMmaRegs = 56, kConvRegs = 96, kEpiRegs = 112;
static_assert(128 * kMmaRegs + 32 * kConvWarps * kConvRegs + 32 * kEpiWarps * kEpiRegs <= kThreads * 96,
              "register split exceeds the launch's registers");

// X = l 2^(56 - E) rounded to the nearest integer, plus the digits' bias: byte 6 - a
// of the result is q_a + 128 (a >= 1), the 16 bits from 48 up q_0 + 512.  |l| >= 2^E
// (possible only on the way to a failed factorisation) is cut to its
// significand, in [1, 2) 2^E.  15 integer instructions, which this GPU issues at
// half the FP32 rate: the converters' rate is what they cost.  Two of them are the
// rounding's (cut down without it, the sums' errors had one sign: mean of R - L L'
// -3e-17 at n = 4064, d = 12, and a root mean square up to three times that of
// IEEE multiply-adds where the entries of R are small).
__device__ __forceinline__ uint2 biased_digits(double l, int E) {
    const unsigned hi = (unsigned)__double2hiint(l), lo = (unsigned)__double2loint(l);
    // r = 1023 + E - e in [0, 63]: l 2^(57 - E) = (m << 5) >> r for the 53-bit significand m
    const int r = __viaddmin_s32_relu((int)((~hi & 0x7ff00000u) >> 20), 1023 + E - 2047, 63);
    const unsigned long long m = (unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32 | lo;
    const unsigned long long w = (m << 5) >> r;
    // -1 - w for a negative l, so that what is cut off below the half lies on the
    // same side of it for either sign
    const unsigned s = (unsigned)((int)hi >> 31);
    const unsigned long long x = (unsigned long long)((unsigned)(w >> 32) ^ s) << 32 | ((unsigned)w ^ s);
    const unsigned long long y = (x + (2 * 0x0200808080808080ull + 1)) >> 1;
    return make_uint2((unsigned)y, (unsigned)(y >> 32));
}

// fp16 pair of two bytes' digits (y - 128 for byte k of u and of v): 0x6400 | y
// is 1024 + y, and the subtraction is exact
__device__ __forceinline__ uint32_t digit_pair(unsigned u, unsigned v, int k) {
    const unsigned p = __byte_perm(u, v, k | (k << 4) | ((4 + k) << 8) | ((4 + k) << 12));
    uint32_t r;
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"((p & 0x00ff00ffu) | 0x64006400u), "r"(0xe480e480u));   // - 1152
    return r;
}

__device__ __forceinline__ uint32_t top_pair(unsigned u, unsigned v) {
    uint32_t r;
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(__byte_perm(u, v, 0x7632) | 0x64006400u), "r"(0xe600e600u));   // - 1536
    return r;
}

// Eight columns of one row into the digit images: piece at `dst`, digit a at
// dst + a * stride.
__device__ __forceinline__ void store_digits(const double (&l)[8], int E, uint8_t* dst, uint32_t stride) {
    unsigned yl[8], yh[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const uint2 y = biased_digits(l[e], E);
        yl[e] = y.x;
        yh[e] = y.y;
    }
#pragma unroll
    for (int a = 0; a < kNS; ++a) {
        uint4 v;
        uint32_t* q = &v.x;
#pragma unroll
        for (int e = 0; e < 4; ++e)
            q[e] = a == 0 ? top_pair(yh[2 * e], yh[2 * e + 1])
                          : (a <= 2 ? digit_pair(yh[2 * e], yh[2 * e + 1], 2 - a)
                                    : digit_pair(yl[2 * e], yl[2 * e + 1], 6 - a));
        *reinterpret_cast<uint4*>(dst + a * stride) = v;
    }
}

// Instruction descriptor: fp16 x fp16 -> f32, both K-major, M = 128, N = n.
constexpr uint32_t idesc_f16(uint32_t n) { return (1u << 4) | ((n >> 3) << 17) | ((128u >> 4) << 24); }

// The MMAs of one stage (two K = 16 steps): every digit product with a + b <
// kNG into group a + b; the first stage of a tile overwrites the groups.
template <int kNT, bool FIRST>
__device__ __forceinline__ void issue(uint32_t tacc, uint64_t ad0, uint64_t bd0) {
    constexpr uint32_t idesc = idesc_f16(kNT), kBChunk = b_chunk(kNT);
#pragma unroll
    for (int a = 0; a < kNS; ++a)
#pragma unroll
        for (int bb = 0; bb < kNS && a + bb < kNG; ++bb)
#pragma unroll
            for (int kk = 0; kk < 2; ++kk) {
                const bool overwrite = FIRST && kk == 0 && (a == 0 || (a == 1 && bb == kNS - 1));
                mma_bf16(tacc + (a + bb) * kNT, ad0 + (uint64_t)((a * kChunkBytes + kk * 32) >> 4),
                         bd0 + (uint64_t)((bb * kBChunk + kk * 32) >> 4), idesc, overwrite ? 0u : 1u);
            }
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float* v) {
    uint32_t r[4];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(r[i]);
}

// sum_g S_g 256^(5 - g), groups 6 and 7 rounded: the product of the two rows
// in units of 2^-56 (below 2^63 for 128 terms under 1; the high word wraps on
// the way).  A group turns into an integer by the conversion instruction, or, an
// eighth of its cost, by adding 1.5 2^23, which is exact up to 2^22.  Groups 6 and 7
// go as one rounded float, |S_6 + S_7 / 256| 2^-8 < 2^17.  The others:
//
//   L L' (FACTOR)  both operands' rows have norm 1, so by Cauchy-Schwarz a pair
//                  with q_0 stays below 2^18.6 and a pair of lower digits below
//                  2^21: S_0 .. S_2 < 2^21.5, S_3 .. S_5 < 2^23.2.
//   W S, L X, X'X  (the inverse) only |q_0| <= 256, |q_a| <= 128 hold, and they
//                  are reached: a column of L^-1 next to a dominant nugget is
//                  nearly constant over a block, so that S_0 of X'X comes
//                  close to 128 2^16 = 2^23.  S_1 <= 2^23, S_2 <= 2^23.4,
//                  S_3 .. S_5 <= 2^24, so groups 0 .. 5 by the instruction; S_6 <=
//                  2^24.2, rounded in any case.
template <bool FACTOR>
__device__ __forceinline__ long long combine(const float (&s)[kNG]) {
    constexpr float kRound = 12582912.f;                  // 1.5 2^23, unit 1
    constexpr int kBits = 0x4b400000;
    auto whole = [](float v) { return FACTOR ? __float_as_int(__fadd_rn(v, kRound)) - kBits : __float2int_rn(v); };
    const unsigned t0 = whole(s[0]), t1 = whole(s[1]);
    const int t2 = whole(s[2]);
    const float low = __fmaf_rn(s[7], 0x1p-8f, s[6]);
    const int t6 = __float_as_int(__fmaf_rn(low, 0x1p-8f, kRound)) - kBits;
    long long v = (long long)((unsigned long long)(t0 * 256u + t1) << 32);
    v += (long long)t2 * (1 << 24);
    v += (long long)__float2int_rn(s[3]) * (1 << 16);
    v += (long long)__float2int_rn(s[4]) * (1 << 8);
    return v + (__float2int_rn(s[5]) + t6);
}

enum : int { kFactorMode = 0, kInnerMode = 1, kInvApply = 2, kInvUpdate = 3 };

// Persistent: one CTA per SM walks the half tiles w = blockIdx.x + k gridDim.x
// (instance-major).  The converter warps cut the operands of one 32-column
// stage into a two-slot ring that runs on across tiles (each warp loads its
// part of the next stage as it stores this one's), warp 0 issues the MMAs,
// the epilogue warps sum the groups into 64-bit integers, release tensor
// memory and then update C beside the next tile's MMAs.  Every wait is
// bounded; a timeout marks the instances GP_ETIMEOUT and stops the CTA after
// its MMAs have landed.
//
// MODE kInner (NT = 32, chunks = s): columns 32 s .. 32 s + 31 of block column J
// itself take the products of its columns before them, for the rows from
// 32 s of tile (J, J) down.
//
// MODE kInvApply, kInvUpdate: the same machine on the rows of X = L^-1
// (k_grad.cu), whose columns are cut at their own exponents:
//   apply   X_JK = -W_J S_JK                              K < J
//   update  S_IK += L_IJ X_JK (I > J),  (R^-1)_IK += X_JI' X_JK (I <= J),  K <= J,
// S and R^-1 sharing one set of tiles (row J of S is consumed by step J).
// The exponents lie in the factor's own diagonal tiles, which the inverse no
// longer needs: tile (K, K) holds those of X_JK's columns, of S_JK's columns
// and of W_K's rows.
template <int kNT, int MODE>
__global__ void __launch_bounds__(kThreads, 1)
    k_update_f64_tc(Batch b, int J, int which, int per_inst, int chunks, double* X, double* S) {
    grid_dependency();
    constexpr bool kInner = MODE == kInnerMode;
    constexpr bool kInv = MODE == kInvApply || MODE == kInvUpdate;
    constexpr uint32_t kBChunk = b_chunk(kNT), kStageBytes = stage_bytes(kNT);
    constexpr int kStagePieces = (GP_NB + kNT) / 32 * 4;
    constexpr int kEpiCols = kNT / 2;          // columns of an epilogue warp
    static_assert(kNG * kNT <= 512, "accumulators exceed tensor memory");
    static_assert(kStagePieces <= kPieces * kConvWarps, "pieces per stage");
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned* live = reinterpret_cast<unsigned*>(smem + 2 * kStageBytes);   // a bit per instance
    __shared__ __align__(8) uint64_t full_bar[2];
    __shared__ __align__(8) uint64_t empty_bar[2];
    __shared__ __align__(8) uint64_t tfull_bar, tempty_bar, drain_bar;
    __shared__ __align__(8) uint64_t never_bar;   // never signalled: the timeout test waits on it
    __shared__ uint32_t tmem_base;
    __shared__ volatile int abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int total = per_inst * b.count;
    // the statuses are read once: a look-ahead's diagonal step may set one
    // while this kernel runs, and the roles must agree on the tiles
    for (int t0 = 32 * warp; t0 < b.count; t0 += kThreads) {
        const bool ok = t0 + lane < b.count && *(volatile const int*)&b.st[t0 + lane].status == GP_OK;
        const unsigned m = __ballot_sync(0xffffffffu, ok);
        if (lane == 0) live[t0 >> 5] = m;
    }
    if (threadIdx.x == 0) {
        for (int u = 0; u < 2; ++u) {
            mbar_init(&full_bar[u], 32 * kConvWarps);
            mbar_init(&empty_bar[u], 1);
        }
        mbar_init(&tfull_bar, 1);
        mbar_init(&tempty_bar, 32 * kEpiWarps);
        mbar_init(&drain_bar, 1);
        mbar_init(&never_bar, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_base)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = tmem_base;

    // first live work item from w on (total when there is none)
    auto next_live = [&](int w) {
        while (w < total) {
            const int t = w / per_inst;
            if (live[t >> 5] >> (t & 31) & 1) return w;
            w += gridDim.x;
        }
        return total;
    };
    auto decode = [&](int w, int& t, int& I, int& K, int& col0) {
        t = w / per_inst;
        const int q = w - t * per_inst;
        if (kInner) {
            I = J + q;
            K = J;
            col0 = kNT * chunks;
            return;
        }
        constexpr int kParts = GP_NB / kNT;
        col0 = (q % kParts) * kNT;
        if (MODE == kInvApply) {
            I = J;
            K = q / kParts;
            return;
        }
        if (MODE == kInvUpdate) {
            const int lower = (b.nt - 1 - J) * (J + 1), v = q / kParts;
            if (v < lower) {
                I = J + 1 + v / (J + 1);
                K = v % (J + 1);
            } else {
                tri_decode(v - lower, I, K);
            }
            return;
        }
        int ii, kk;
        if (which == kUpdateColumn) {
            ii = q / kParts;
            kk = 0;
        } else {
            tri_decode(q / kParts, ii, kk);
            if (which == kUpdateRest) {
                ++ii;
                ++kk;
            }
        }
        I = J + 1 + ii;
        K = J + 1 + kk;
    };
    auto tile_of = [&](double* base, int t, int I, int K) {
        return base + (size_t)t * b.inst_stride + (size_t)tile_index(I, K, b.nt) * GP_TILE_ELEMS;
    };
    auto tile = [&](int t, int I, int K) { return tile_of(b.A, t, I, K); };
    auto exps = [&](int t, int K, int slot) { return reinterpret_cast<const int*>(tile(t, K, K)) + slot * GP_NB; };

    if (warp >= kEpiBase) {
        regs_inc<kEpiRegs>();
        const int q = warp & 3, half = (warp - kEpiBase) >> 2;
        const int r = q * 32 + lane, c0 = kEpiCols * half;
        const uint32_t lane_addr = tbase + ((uint32_t)(q * 32) << 16) + c0;
        int i = 0;
        for (int w = next_live(blockIdx.x); w < total && !abort_flag; w = next_live(w + gridDim.x), ++i) {
            int t, I, K, col0;
            decode(w, t, I, K, col0);
            double* C = (MODE == kInvApply    ? tile_of(X, t, I, K)
                         : MODE == kInvUpdate ? tile_of(S, t, I, K)
                                              : tile(t, I, K)) + (size_t)col0 * GP_NB;
            // what the products are added to: nothing the first time a tile of S
            // (K = J) or of R^-1 (I = J) is reached
            const bool fresh = MODE == kInvApply || (MODE == kInvUpdate && (I > J ? K == J : I == J));
            if (threadIdx.x == 32 * kEpiBase && !fresh) prefetch_l2(C, kNT * GP_NB * sizeof(double));
            if (!mbar_wait(&tfull_bar, i & 1, &abort_flag)) {
                abort_flag = 1;
                break;
            }
            tc_fence_after();
            long long v[kEpiCols];
#pragma unroll
            for (int c = 0; c < kEpiCols; c += 4) {
                float s[kNG][4];
#pragma unroll
                for (int g = 0; g < kNG; ++g) tmem_ld4(lane_addr + g * kNT + c, s[g]);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float u[kNG];
#pragma unroll
                    for (int g = 0; g < kNG; ++g) u[g] = s[g][j];
                    v[c + j] = combine<!kInv>(u);
                }
            }
            tc_fence_before();
            mbar_arrive(&tempty_bar);
            // the rows of the diagonal tile above the inner update's columns
            // are finished
            if (kInner && I == K && r < col0) continue;
            double* p = C + (size_t)c0 * GP_NB + r;
            // the rows' exponents (MODE kInvUpdate: of L_IJ none, of X_JI' its columns')
            int ea = 0;
            const int* eb = nullptr;
            if (kInv) {
                ea = MODE == kInvApply ? exps(t, J, 2)[r] : (I > J ? 0 : exps(t, I, 0)[r]);
                eb = exps(t, K, MODE == kInvApply ? 1 : 0) + col0 + c0;
            }
#pragma unroll
            for (int c = 0; c < kEpiCols; c += 8) {
                double cv[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) cv[j] = fresh ? 0.0 : p[(size_t)(c + j) * GP_NB];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    double scale = 0x1p-56;
                    if (kInv) {
                        const int e = 1023 - 56 + ea + eb[c + j];      // 0 below the normal range
                        scale = __hiloint2double(e > 0 ? e << 20 : 0, 0);
                    }
                    const double d = __ll2double_rn(v[c + j]);
                    p[(size_t)(c + j) * GP_NB] = fma(MODE == kInvUpdate ? d : -d, scale, cv[j]);
                }
            }
        }
    } else if (warp >= kConvBase) {
        regs_inc<kConvRegs>();
        const int cw = warp - kConvBase;
        // this warp's pieces of a stage: 32 rows (of the 128 of A, then the NT
        // of B) by 8 columns.  Operand rows run along a tile's columns for L and
        // W, along its rows (eight consecutive doubles a lane) for X and S.
        // A work item's pointers are formed once; a stage moves them on.
        struct Piece {
            const double* p;       // its first value
            int step;              // to the next of the eight columns
            int E;
        };
        auto source = [&](int w, int u) -> Piece {
            int t, I, K, col0;
            decode(w, t, I, K, col0);
            const int piece = min(cw + kConvWarps * u, kStagePieces - 1), rg = piece >> 2, oct = piece & 3;
            const bool isA = rg < 4;
            const int row = (isA ? 32 * rg : col0 + 32 * (rg - 4)) + lane;
            if (!kInv)
                return {(isA ? tile(t, I, J) : tile(t, K, J)) + (size_t)(8 * oct) * GP_NB + row, GP_NB, 0};
            const bool byRow = isA && (MODE == kInvApply || I > J);
            const double* src;
            int E = 0;
            if (MODE == kInvApply) {
                src = isA ? tile_of(X, t, J, J) : tile_of(S, t, J, K);
                E = isA ? exps(t, J, 2)[row] : exps(t, K, 1)[row];
            } else {
                src = byRow ? tile(t, I, J) : tile_of(X, t, J, isA ? I : K);
                if (!byRow) E = exps(t, isA ? I : K, 0)[row];
            }
            return byRow ? Piece{src + (size_t)(8 * oct) * GP_NB + row, GP_NB, E}
                         : Piece{src + (size_t)row * GP_NB + 8 * oct, 1, E};
        };
        double raw[kPieces][8];
        Piece at[kPieces];
        int w = next_live(blockIdx.x), kc = 0;
        if (w < total) {
#pragma unroll
            for (int u = 0; u < kPieces; ++u) {
                at[u] = source(w, u);
#pragma unroll
                for (int e = 0; e < 8; ++e) raw[u][e] = at[u].p[e * (kInv ? at[u].step : GP_NB)];
            }
        }
        for (int g = 0; w < total && !abort_flag; ++g) {
            const int st = g & 1;
            if (g >= 2 && !mbar_wait(&empty_bar[st], ((g >> 1) - 1) & 1, &abort_flag)) {
                abort_flag = 1;
                break;
            }
            const int kn = kc + 1 == chunks ? 0 : kc + 1;
            const int wn = kn == 0 ? next_live(w + gridDim.x) : w;
            uint8_t* stage = smem + st * kStageBytes;
#pragma unroll
            for (int u = 0; u < kPieces; ++u) {
                const int piece = cw + kConvWarps * u, rg = piece >> 2, oct = piece & 3;
                const bool isA = rg < 4;
                uint8_t* dst = stage + (isA ? 0u : kABytes) + image_piece((isA ? 32 * rg : 32 * (rg - 4)) + lane, 8 * oct);
                if (piece < kStagePieces) store_digits(raw[u], kInv ? at[u].E : 0, dst, isA ? kChunkBytes : kBChunk);
                if (wn < total) {
                    if (kn == 0) at[u] = source(wn, u);
                    else         at[u].p += 32 * (kInv ? at[u].step : GP_NB);
#pragma unroll
                    for (int e = 0; e < 8; ++e) raw[u][e] = at[u].p[e * (kInv ? at[u].step : GP_NB)];
                }
            }
            // the tensor core reads shared memory through the asynchronous proxy
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_arrive(&full_bar[st]);
            w = wn;
            kc = kn;
        }
    } else {
        regs_dec<kMmaRegs>();
        if (warp == 0 && lane == 0) {
            int g = 0, i = 0;
            for (int w = next_live(blockIdx.x); w < total && !abort_flag; w = next_live(w + gridDim.x), ++i) {
                if (i >= 1 && !mbar_wait(&tempty_bar, (i - 1) & 1, &abort_flag)) {
                    abort_flag = 1;
                    break;
                }
                // test hook: a wait that nothing ends, limited to 5 ms
                if ((MODE == kFactorMode || MODE == kInvUpdate) && b.inject_timeout && J == 0 && blockIdx.x == 0 &&
                    i == 0 && !mbar_wait(&never_bar, 0, &abort_flag, 5000000ull)) {
                    abort_flag = 1;
                    break;
                }
                tc_fence_after();
                for (int kc = 0; kc < chunks; ++kc, ++g) {
                    const int st = g & 1;
                    if (!mbar_wait(&full_bar[st], (g >> 1) & 1, &abort_flag)) {
                        abort_flag = 1;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t sa = smem_u32(smem + st * kStageBytes);
                    const uint64_t ad0 = smem_desc(sa, 16, 512, 4), bd0 = smem_desc(sa + kABytes, 16, 512, 4);
                    if (kc == 0) issue<kNT, true>(tbase, ad0, bd0);
                    else         issue<kNT, false>(tbase, ad0, bd0);
                    mma_commit(&empty_bar[st]);
                }
                if (abort_flag) break;
                mma_commit(&tfull_bar);
            }
            // every MMA issued has completed before tensor memory is released
            mma_commit(&drain_bar);
            mbar_wait(&drain_bar, 0);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (abort_flag && threadIdx.x == 0)
        for (int w = blockIdx.x; w < total; w += gridDim.x) b.st[w / per_inst].status = GP_ETIMEOUT;
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tbase));
}

template <int NT, int MODE>
cudaError_t launch(const Batch& b, int J, cudaStream_t s, int which, int per_inst, int chunks, double* X = nullptr,
                   double* S = nullptr) {
    const size_t smem = 2 * (size_t)stage_bytes(NT) + 1024 + (size_t)(b.count + 31) / 32 * 4;
    static std::atomic<size_t> attr[kMaxDevices];
    cudaError_t e = raise_smem_limit(k_update_f64_tc<NT, MODE>, smem, attr);
    if (e != cudaSuccess) return e;
    const long long total = (long long)per_inst * b.count;
    // the rest of an update runs beside the next block column's panel, whose
    // kernels cannot share an SM with this one: a third of the SMs stay free
    // for them (ms, without the look-ahead / every SM taken / a third free / half
    // free; candidates x n: 1x4064 8.59 / 9.08 / 8.23 / 8.23, 4x2048 4.79 / 5.13 / 4.72 /
    // 4.65, 16x1024 2.81 / 3.07 / 2.84 / 2.81, 12x4064 28.57 / 29.65 / 28.85 / 32.77)
    const int cap = which == kUpdateRest ? device_sms() - device_sms() / 3 : device_sms();
    const int grid = (int)(total < cap ? total : cap);
    launch_chained(which != kUpdateColumn && ahead_f64(b), k_update_f64_tc<NT, MODE>, grid, kThreads, smem, s, b, J,
                   which, per_inst, chunks, X, S);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_update_f64_tc(const Batch& b, int J, cudaStream_t s, int which) {
    const int m = b.nt - J - 1;
    const int tiles = which == kUpdateColumn ? m : (which == kUpdateRest ? m * (m - 1) / 2 : m * (m + 1) / 2);
    if (tiles <= 0) return cudaSuccess;
    // quarter tiles where the half tiles would leave half of the SMs idle (the
    // same bits; a tile's chain is 22 us in halves, about 15 in quarters)
    if ((long long)4 * tiles * b.count <= device_sms()) return launch<32, kFactorMode>(b, J, s, which, 4 * tiles, kChunks);
    return launch<64, kFactorMode>(b, J, s, which, 2 * tiles, kChunks);
}

cudaError_t launch_update_f64_inner(const Batch& b, int J, int step, cudaStream_t s) {
    return launch<32, kInnerMode>(b, J, s, kUpdateAll, b.nt - J, step);
}

cudaError_t launch_inverse_apply(const Batch& b, int J, double* X, double* S, cudaStream_t s) {
    if (J == 0) return cudaSuccess;
    return launch<64, kInvApply>(b, J, s, kUpdateAll, 2 * J, kChunks, X, S);
}

cudaError_t launch_inverse_update(const Batch& b, int J, double* X, double* S, cudaStream_t s) {
    const int tiles = (b.nt - 1 - J) * (J + 1) + (J + 1) * (J + 2) / 2;
    return launch<64, kInvUpdate>(b, J, s, kUpdateAll, 2 * tiles, kChunks, X, S);
}

}  // namespace gp
