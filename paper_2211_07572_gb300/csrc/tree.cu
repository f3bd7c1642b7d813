// Stage 1: elimination of the slab interiors (Sec. 3.1, Algorithm 3 first loop).
//
// Each slab's interior block A_JJ is eliminated by cyclic reduction along y:
// the rows form a binary "ruler" tree (row c has height ctz(c)), and a launch
// eliminates every node of one height in every slab at once.  Node c merges
// the condensed systems of its two child segments through its separator row:
//   S   = D_c + R_alpha[bot,bot] + R_beta[top,top]            (m x m, SPD)
//   B   = couplings of row c to {top row, bot row, interface nodes of the segment}
//   L L^T = S,   Z = L^{-1} B,   R_merged = R_others - Z^T Z.
// Only the rows of R that belong to the top/bot rows are kept (the interface x
// interface part is summed later by the fused T assembly), so the per-node work
// is O(m^2 w) and the storage O(m s log s) per slab.
#include "tree_args.cuh"

namespace {

constexpr int MAXM = SLAB_MAXM;
constexpr int SP = MAXM + 1;          // smem row stride of S: a lane reads its row without conflicts
constexpr int LP = MAXM + 4;          // smem row stride of the inverse: 16-byte rows
constexpr int ZP = 2 * MAXM + 4;      // smem row stride of the m x 2m blocks: top columns at 0, bottom at MAXM
constexpr int TB_THREADS = 128;

// Four consecutive shared-memory values, 16-byte aligned.
__device__ __forceinline__ void lds4(const float* p, float (&v)[4]) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void lds4(const double* p, double (&v)[4]) {
    const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ bool usable_square(float d) { return d > 0.0f && d <= 3.402823466e38f; }
__device__ __forceinline__ bool usable_square(double d) { return d > 0.0 && d <= 1.7976931348623157e308; }
__device__ __forceinline__ unsigned magnitude(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }
__device__ __forceinline__ bool usable_magnitude(double v) {
    return (magnitude(v) | (unsigned)__double2loint(v)) != 0u && magnitude(v) < 0x7ff00000u;
}

// The separator inverses are one warp's work with a row per lane in registers: m dependent steps without a
// block barrier.  (By the whole block in shared memory, with four barriers a step, they were most of an
// upper height's 130 us.)
//
// Li = L^{-1} (stride LP, zeros right of the diagonal and in the padding) of the Cholesky factor of the
// m x m matrix S (stride SP, lower triangle read).  Register a[j] of lane i is S_ij until column j is
// eliminated and X_ij of X = L^{-1} from then on; step k publishes in P the finished row k of X (entries
// up to k) and the column k of L (entries below), and every row below takes a -= l P.
template <typename T>
__device__ __forceinline__ void chol_inv_warp(const T* S, T* Li, T (*P)[MAXM], int m, unsigned* status) {
    const int lane = threadIdx.x & 31;
    T a[MAXM];
#pragma unroll
    for (int j = 0; j < MAXM; ++j) a[j] = (lane < m && j <= lane) ? S[lane * SP + j] : T(0);
#pragma unroll
    for (int k = 0; k < MAXM; ++k) {
        if (k < m) {                                              // (uniform; a break would keep the loop rolled)
            T* p = P[k & 1];
            T d = __shfl_sync(0xffffffffu, a[k], k);
            if (!usable_square(d)) {
                if (lane == 0) atomicOr(status, SLAB_DEV_NOTSPD);
                d = T(1);
            }
            const T r = rsqrt_newton(d);
            const T l = lane > k ? a[k] * r : T(0);
            if (lane == k) {
#pragma unroll
                for (int j = 0; j < k; ++j) a[j] *= r;
                a[k] = r;
#pragma unroll
                for (int j = 0; j <= k; ++j) p[j] = a[j];
            } else if (lane > k) {
                a[k] = T(0);
                p[lane] = l;
            }
            __syncwarp();
#pragma unroll
            for (int j = 0; j < MAXM; j += 4) {
                if (j < m) {
                    T v[4];
                    lds4(p + j, v);
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (lane > k) a[j + q] -= l * v[q];
                }
            }
        }
    }
#pragma unroll
    for (int j = 0; j < MAXM; ++j) Li[lane * LP + j] = (lane < m && j <= lane) ? a[j] : T(0);
}

// Si = S^{-1} (stride LP, zero padding) by Gauss-Jordan elimination in place with partial pivoting (largest
// |s_ik| among the rows not used yet): step k replaces the pivot row's entry k by 1 and clears column k of all
// other rows; the pivot rows are divided by their pivots at the end, all at once.  Row p(k), column j of the
// result is (S^{-1})[k][p(j)].  A zero or non-finite pivot sets SLAB_DEV_NOTSPD and continues with 1.
//   In FP64 for both types: its rounding is what the refinement's gain per pass hangs on where A is indefinite or
// nonsymmetric.  n = 2000 Helmholtz with FP32 trees: gain 0.51 a pass in FP32 (the iteration stops as stalled), 0.21 in
// FP64; n = 768 convection: residual after two passes 1.0e-9 and 1.5e-10, factor + solve + adjoint 41.0 and 42.5 ms.
template <typename T>
__device__ __forceinline__ void gj_inv_warp(const T* S, T* Si, double (*P)[MAXM], int* perm, int m, unsigned* status) {
    const int lane = threadIdx.x & 31;
    double a[MAXM];
#pragma unroll
    for (int j = 0; j < MAXM; ++j) a[j] = (lane < m && j < m) ? (double)S[lane * SP + j] : 0.0;
    bool open = lane < m;
    int mine = 0;
    double scale = 0.0;                                               // reciprocal of this row's pivot
#pragma unroll
    for (int k = 0; k < MAXM; ++k) {
        if (k < m) {                                              // (uniform; a break would keep the loop rolled)
            double* p = P[k & 1];
            const unsigned key = open ? magnitude(a[k]) + 1u : 0u;
            const unsigned best = __reduce_max_sync(0xffffffffu, key);
            const int src = __ffs(__ballot_sync(0xffffffffu, key == best)) - 1;
            double f = a[k], r = 1.0;
            if (lane == src) {
                if (usable_magnitude(f)) r = reciprocal_full(f);
                else atomicOr(status, SLAB_DEV_NOTSPD);
                a[k] = 1.0;
#pragma unroll
                for (int j = 0; j < MAXM; ++j) p[j] = a[j];
                open = false;
                mine = k;
                perm[k] = lane;
                scale = r;
            } else {
                a[k] = 0.0;
            }
            r = __shfl_sync(0xffffffffu, r, src);
            f = lane == src ? 0.0 : f * r;
            __syncwarp();
#pragma unroll
            for (int j = 0; j < MAXM; j += 4) {
                if (j < m) {
                    double v[4];
                    lds4(p + j, v);
#pragma unroll
                    for (int q = 0; q < 4; ++q) a[j + q] -= f * v[q];
                }
            }
        }
    }
#pragma unroll
    for (int j = 0; j < MAXM; ++j) {
        if (lane >= m) Si[lane * LP + j] = T(0);                  // padding rows and columns
        else if (j >= m) Si[mine * LP + j] = T(0);
        else Si[mine * LP + perm[j]] = (T)(a[j] * scale);
    }
}

// z = M b for an m x m block M in shared memory (stride LP, zero padding); TRI: lower triangular.
template <typename T, bool TRI>
__device__ __forceinline__ void block_times(const T* M, const T (&b)[MAXM], T (&z)[MAXM], int m) {
#pragma unroll
    for (int i = 0; i < MAXM; ++i) {
        z[i] = T(0);
        if (i < m) {
#pragma unroll
            for (int l = 0; l < MAXM; l += 4)
                if ((!TRI || l <= i) && l < m) {
                    T v[4];
                    lds4(M + i * LP + l, v);
#pragma unroll
                    for (int q = 0; q < 4; ++q) z[i] += v[q] * b[l + q];
                }
        }
    }
}
// z = M^T b
template <typename T>
__device__ __forceinline__ void block_transposed_times(const T* M, const T (&b)[MAXM], T (&z)[MAXM], int m) {
#pragma unroll
    for (int i = 0; i < MAXM; ++i) z[i] = T(0);
#pragma unroll
    for (int l = 0; l < MAXM; ++l)
        if (l < m) {
#pragma unroll
            for (int i = 0; i < MAXM; i += 4)
                if (i < m) {
                    T v[4];
                    lds4(M + l * LP + i, v);
#pragma unroll
                    for (int q = 0; q < 4; ++q) z[i + q] += v[q] * b[l];
                }
        }
}

// The condensed top and bottom entries of one interface column: dt[a] = ct[a] - sum_i Z[i][a] z[i] and likewise for the
// bottom rows (Z at column offset MAXM); ct / cb null: zero.  All with stride sp.
template <typename T>
__device__ __forceinline__ void condense_column(const T* Z, const T (&z)[MAXM], int m, int64_t sp, const T* ct, const T* cb,
                                                T* dt, T* db) {
#pragma unroll 1
    for (int a = 0; a < m; a += 4) {
        T vt[4], vb[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            vt[q] = (ct && a + q < m) ? ct[(a + q) * sp] : T(0);
            vb[q] = (cb && a + q < m) ? cb[(a + q) * sp] : T(0);
        }
#pragma unroll
        for (int i = 0; i < MAXM; ++i)
            if (i < m) {
                T x[4], y[4];
                lds4(Z + i * ZP + a, x);
                lds4(Z + i * ZP + MAXM + a, y);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    vt[q] -= x[q] * z[i];
                    vb[q] -= y[q] * z[i];
                }
            }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (a + q < m) {
                dt[(a + q) * sp] = vt[q];
                db[(a + q) * sp] = vb[q];
            }
    }
}

// R[2m][2m] = blockdiag(Ra[top,top], Rb[bot,bot]) - Zl^T Zr: thread (ag, bg) owns 4 x 8 entries.  SYM: the product is
// symmetric; 4 x 4 blocks on and below the diagonal, each stored twice (FP64, where multiply-adds are the
// bound; in FP32 the larger blocks are faster).
template <typename T, bool SYM>
__device__ __forceinline__ void condense_node(const T* Zl, const T* Zr, int m, const T* Ra, const T* Rb, T* Rg) {
    constexpr int NB = SYM ? 4 : 8, NT = SYM ? 136 : 128;
    const int m2 = 2 * m;
    for (int e = threadIdx.x; e < NT; e += TB_THREADS) {
        int ag = e >> 3, bg = e & 7;
        if (SYM) {                                              // e = ag (ag + 1) / 2 + bg
            ag = (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f);
            bg = e - ag * (ag + 1) / 2;
        }
        const int a0 = 4 * ag, b0 = NB * bg;                    // padded columns: top at 0, bottom at MAXM
        if ((a0 & (MAXM - 1)) >= m || (b0 & (MAXM - 1)) >= m) continue;
        T acc[4][NB];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < NB; ++j) acc[i][j] = T(0);
#pragma unroll 4
        for (int l = 0; l < m; ++l) {
            T x[4], y[NB];
            lds4(Zl + l * ZP + a0, x);
#pragma unroll
            for (int j = 0; j < NB; j += 4) {
                T v[4];
                lds4(Zr + l * ZP + b0 + j, v);
#pragma unroll
                for (int q = 0; q < 4; ++q) y[j + q] = v[q];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < NB; ++j) acc[i][j] -= x[i] * y[j];
        }
        const bool at = a0 < MAXM, bt = b0 < MAXM;
        const T* add = at && bt ? Ra : (!at && !bt ? Rb : nullptr);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                const int ai = (a0 & (MAXM - 1)) + i, bj = (b0 & (MAXM - 1)) + j;
                if (ai < m && bj < m && !(SYM && a0 == b0 && j > i)) {
                    const int r = at ? ai : m + ai, c = bt ? bj : m + bj;
                    const T v = acc[i][j] + (add ? add[r * m2 + c] : T(0));
                    Rg[r * m2 + c] = v;
                    if (SYM && r != c) Rg[c * m2 + r] = v;
                }
            }
    }
}

// One height of the cyclic reduction in every slab.
// grid = (node index a at this height, column chunk, slab t); block = TB_THREADS.
// SPD kinds: L L^T = S, Z = L^{-1} B; stored Linv, Z.  Indefinite kind: S^{-1} by pivoted
// Gauss-Jordan, W = S^{-1} B; stored S^{-1}, B (in the Z arrays) and W.  In both cases the
// condensed rows are R_merged = R_others - B^T S^{-1} B (= Z^T Z in the SPD form).
//   A thread owns a column (top, bottom or interface) with its m entries in registers and multiplies it by
// blocks read four entries at a time from shared memory.  At height 0 the couplings are diagonal, which
// leaves the inverse and, for the SPD kinds, Z^T Z.  Bound at low heights by the traffic (7 m^2
// entries written a node), above by the latency of the m elimination steps.  n = 2048, b = 32, FP32: 8.4 ms for the
// eleven heights (14.4 with the inverse and the products by the whole block in shared memory); n = 512
// Helmholtz, FP64: 5.1 ms (9.3), bound by the FP64 pipe.
template <typename T, bool INDEF>
__global__ void __launch_bounds__(TB_THREADS) tree_factor_kernel(TreeArgs<T> A, int k) {
    __shared__ __align__(16) T SW[MAXM * ZP];      // S (stride SP); indefinite kind: then W
    __shared__ __align__(16) T Li[MAXM * LP];
    __shared__ __align__(16) T Bt[MAXM * ZP];      // B; SPD kind: then Z = Li B in place
    __shared__ __align__(16) double Pd[2][MAXM];
    T(*P)[MAXM] = reinterpret_cast<T(*)[MAXM]>(Pd);
    __shared__ int perm[MAXM];
    constexpr bool FP64 = sizeof(T) == 8;
    const int tid = threadIdx.x, nth = blockDim.x;
    const int t = blockIdx.z;
    const int c = (2 * blockIdx.x + 1) << k;
    const int s = A.s, m = A.m;
    if (c > s) return;
    const int lo = c - (1 << k) + 1;
    const int hi = min(s, c + (1 << k) - 1);
    const int w = hi - lo + 1;
    const int ncols = 2 * w;
    const int q0 = blockIdx.y * TB_THREADS;
    if (blockIdx.y > 0 && q0 >= ncols) return;
    const int alpha = k > 0 ? c - (1 << (k - 1)) : 0;
    const int kb = tree_right_height(s, c, k);
    const int beta = kb >= 0 ? c + (1 << kb) : 0;
    const int x0 = t * A.b + 1;
    const int np1 = A.n + 1;
    const double* DGr = A.DG + (int64_t)c * np1;
    const double* AXr = A.AX + (int64_t)c * np1;
    const T* Ra = alpha ? A.rtb(t, alpha) : nullptr;
    const T* Rb = beta ? A.rtb(t, beta) : nullptr;
    const int m2 = 2 * m;
    const int lane = tid & 31, warp = tid >> 5;

    // S = D_c + R_alpha[bot,bot] + R_beta[top,top];  B = [top | bot] couplings (a warp a row)
    for (int i = warp; i < m; i += nth / 32) {
        const int j = lane;
        if (j < m) {
            double v = 0.0;
            if (i == j) v = DGr[x0 + i];
            else if (j == i + 1) v = -AXr[x0 + i];
            else if (j == i - 1) v = -AXr[x0 + j];
            T tv = (T)v;
            if (Ra) tv += Ra[(m + i) * m2 + (m + j)];
            if (Rb) tv += Rb[i * m2 + j];
            SW[i * SP + j] = tv;
        }
        T vt = T(0), vb = T(0);
        if (j < m) {
            if (Ra) vt = Ra[(m + i) * m2 + j];                      // alpha's bot row x its top column
            else if (i == j && c - 1 >= 1) vt = (T)(-A.AY[(int64_t)(c - 1) * np1 + x0 + i]);
            if (Rb) vb = Rb[i * m2 + m + j];                        // beta's top row x its bot column
            else if (i == j && c + 1 <= s) vb = (T)(-A.AY[(int64_t)c * np1 + x0 + i]);
        }
        Bt[i * ZP + j] = vt;
        Bt[i * ZP + MAXM + j] = vb;
    }
    __syncthreads();
    if (warp == 0) {
        if (INDEF) gj_inv_warp<T>(SW, Li, Pd, perm, m, A.status);    // Li = S^{-1}
        else chol_inv_warp<T>(SW, Li, P, m, A.status);
    }
    __syncthreads();
    T bvec[MAXM], z[MAXM];
    if (tid < 2 * MAXM && (tid & (MAXM - 1)) < m) {                 // Z = Li B (SPD, in place), W = S^{-1} B
#pragma unroll
        for (int i = 0; i < MAXM; ++i) bvec[i] = i < m ? Bt[i * ZP + tid] : T(0);
        if (k == 0) {                                               // B is diagonal
            const int d = tid & (MAXM - 1);
            const T b = Bt[d * ZP + tid];
#pragma unroll
            for (int i = 0; i < MAXM; ++i) z[i] = i < m ? Li[i * LP + d] * b : T(0);
        } else {
            block_times<T, !INDEF>(Li, bvec, z, m);
        }
        T* dst = INDEF ? SW : Bt;
#pragma unroll
        for (int i = 0; i < MAXM; ++i)
            if (i < m) dst[i * ZP + tid] = z[i];
    }
    __syncthreads();
    const T* Zl = Bt;                  // left factor of the update: Z (SPD) or B (indefinite)
    const T* Zr = INDEF ? SW : Bt;     // right factor: Z (SPD) or W (indefinite)
    if (blockIdx.y == 0) {
        T* Lg = A.linv(t, c);
        T* Zg = A.ztb(t, c);
        T* Wg = INDEF ? A.wtb(t, c) : nullptr;
        for (int i = warp; i < m; i += nth / 32)
            if (lane < m) {
                Lg[i * m + lane] = Li[i * LP + lane];
                Zg[i * m2 + lane] = Bt[i * ZP + lane];
                Zg[i * m2 + m + lane] = Bt[i * ZP + MAXM + lane];
                if (INDEF) {
                    Wg[i * m2 + lane] = SW[i * ZP + lane];
                    Wg[i * m2 + m + lane] = SW[i * ZP + MAXM + lane];
                }
            }
        if (INDEF && FP64 && k == 0) {                              // B diagonal: one term an entry
            T* Rg = A.rtb(t, c);
            for (int e = tid; e < 4 * MAXM * MAXM; e += nth) {
                const int a = e / (2 * MAXM), b = e % (2 * MAXM), ai = a & (MAXM - 1), bj = b & (MAXM - 1);
                if (ai < m && bj < m)
                    Rg[(a < MAXM ? ai : m + ai) * m2 + (b < MAXM ? bj : m + bj)] = -(Bt[ai * ZP + a] * SW[ai * ZP + b]);
            }
        } else {
            condense_node<T, FP64>(Zl, Zr, m, Ra, Rb, A.rtb(t, c));
        }
    }
    const int64_t sp = A.s_pad;
    if (k == 0) {
        // the node's two interface columns have one entry each: z is a column of Li; then a thread per condensed entry
        T* zc = P[0];                                               // [2][MAXM]
        if (tid < 2 * MAXM) {
            const int side = tid / MAXM, i = tid & (MAXM - 1), d = side ? m - 1 : 0;
            const bool has = side ? t <= A.NS - 2 : t >= 1;
            const T b = has ? (T)(-AXr[side ? x0 + m - 1 : x0 - 1]) : T(0);
            const T v = i < m ? Li[i * LP + d] * b : T(0);
            zc[tid] = v;
            if (i < m) {
                A.zi(t, 0, side)[i * sp + c - 1] = INDEF ? (i == d ? b : T(0)) : v;
                if (INDEF) A.wi(t, 0, side)[i * sp + c - 1] = v;
            }
        }
        __syncthreads();
        const int side = tid / (2 * MAXM), col = tid & (2 * MAXM - 1), a = col & (MAXM - 1);
        if (a < m) {
            T v = T(0);
#pragma unroll 4
            for (int i = 0; i < m; ++i) v -= Zl[i * ZP + col] * zc[side * MAXM + i];
            A.ri(t, 0, col / MAXM, side)[a * sp + c - 1] = v;
        }
        return;
    }
    // interface columns of the segment: one thread per column
    const int q = q0 + tid;
    if (q < ncols) {
        const int side = q >= w;
        const int j = lo + (side ? q - w : q);
        const int rr = j - 1;
#pragma unroll
        for (int i = 0; i < MAXM; ++i) bvec[i] = T(0);
        if (j == c) {
            if (side == 0) {
                if (t >= 1) bvec[0] = (T)(-AXr[x0 - 1]);
            } else if (t <= A.NS - 2) {
#pragma unroll
                for (int i = 0; i < MAXM; ++i) if (i == m - 1) bvec[i] = (T)(-AXr[x0 + m - 1]);
            }
        } else {
            const T* src = (j < c ? A.ri(t, k - 1, 1, side) : A.ri(t, kb, 0, side)) + rr;
#pragma unroll
            for (int i = 0; i < MAXM; ++i) if (i < m) bvec[i] = src[i * sp];
        }
        block_times<T, !INDEF>(Li, bvec, z, m);                     // SPD: z = Li b; indefinite: w = S^{-1} b
        T* zd = A.zi(t, k, side) + rr;
        T* wd = INDEF ? A.wi(t, k, side) + rr : nullptr;
#pragma unroll
        for (int i = 0; i < MAXM; ++i)
            if (i < m) {
                zd[i * sp] = INDEF ? bvec[i] : z[i];
                if (INDEF) wd[i * sp] = z[i];
            }
        // condensed top/bot rows for this interface column: R - Zl^T z  (Zl = Z or B)
        condense_column<T>(Zl, z, m, sp, j < c ? A.ri(t, k - 1, 0, side) + rr : nullptr,
                           j > c ? A.ri(t, kb, 1, side) + rr : nullptr, A.ri(t, k, 0, side) + rr,
                           A.ri(t, k, 1, side) + rr);
    }
}

// One height of the cyclic reduction for the nonsymmetric kind (the same elimination as the
// indefinite kind with both orientations of every coupling kept).  Node c's separator block S,
// its row couplings B (separator rows x {top, bot, interface} columns) and column couplings C
// ({top, bot, interface} rows x separator columns) give
//   R_merged = R_others - C S^{-1} B,
// with S^{-1} from pivoted Gauss-Jordan.  Stored for A: S^{-1}, C^T, W = S^{-1} B; for A^T (whose
// separator block is S^T, row couplings C^T, column couplings B^T): S^{-T}, B, V = S^{-T} C^T.
// The condensed couplings are kept in both orientations: RI (top/bot rows x interface columns)
// and RIc (interface rows x top/bot columns).  grid = (node, column chunk, slab), as above.
// n = 768, FP32: 3.6 ms for the ten heights (6.3 by the whole block in shared memory).
template <typename T>
__global__ void __launch_bounds__(TB_THREADS) tree_factor_ns_kernel(TreeArgs<T> A, int k) {
    __shared__ __align__(16) T SW[MAXM * ZP];      // S (stride SP), then W = S^{-1} B
    __shared__ __align__(16) T Li[MAXM * LP];      // S^{-1}
    __shared__ __align__(16) T Bt[MAXM * ZP];      // B, then C^T
    __shared__ __align__(16) double Pd[2][MAXM];
    __shared__ int perm[MAXM];
    const int tid = threadIdx.x, nth = blockDim.x;
    const int t = blockIdx.z;
    const int c = (2 * blockIdx.x + 1) << k;
    const int s = A.s, m = A.m;
    if (c > s) return;
    const int lo = c - (1 << k) + 1;
    const int hi = min(s, c + (1 << k) - 1);
    const int w = hi - lo + 1;
    const int ncols = 2 * w;
    const int q0 = blockIdx.y * TB_THREADS;
    if (blockIdx.y > 0 && q0 >= ncols) return;
    const int alpha = k > 0 ? c - (1 << (k - 1)) : 0;
    const int kb = tree_right_height(s, c, k);
    const int beta = kb >= 0 ? c + (1 << kb) : 0;
    const int x0 = t * A.b + 1;
    const int np1 = A.n + 1;
    const double* DGr = A.DG + (int64_t)c * np1;
    const double* AXr = A.AX + (int64_t)c * np1;       // -h^2 A[(x,c),(x+1,c)]
    const double* AXTr = A.AXT + (int64_t)c * np1;     // -h^2 A[(x+1,c),(x,c)]
    const T* Ra = alpha ? A.rtb(t, alpha) : nullptr;   // alpha's rows/cols: top 0..m-1, bot m..2m-1
    const T* Rb = beta ? A.rtb(t, beta) : nullptr;
    const int m2 = 2 * m;
    const int lane = tid & 31, warp = tid >> 5;

    // S = D_c + R_alpha[bot,bot] + R_beta[top,top];  B = couplings of row c to [top | bot]
    for (int i = warp; i < m; i += nth / 32) {
        const int j = lane;
        T vt = T(0), vb = T(0);
        if (j < m) {
            double v = 0.0;
            if (i == j) v = DGr[x0 + i];
            else if (j == i + 1) v = -AXr[x0 + i];
            else if (j == i - 1) v = -AXTr[x0 + j];
            T tv = (T)v;
            if (Ra) tv += Ra[(m + i) * m2 + (m + j)];
            if (Rb) tv += Rb[i * m2 + j];
            SW[i * SP + j] = tv;
            if (Ra) vt = Ra[(m + i) * m2 + j];                      // R_alpha[bot i][top j]
            else if (i == j && c - 1 >= 1) vt = (T)(-A.AYT[(int64_t)(c - 1) * np1 + x0 + i]);
            if (Rb) vb = Rb[i * m2 + m + j];                        // R_beta[top i][bot j]
            else if (i == j && c + 1 <= s) vb = (T)(-A.AY[(int64_t)c * np1 + x0 + i]);
        }
        Bt[i * ZP + j] = vt;
        Bt[i * ZP + MAXM + j] = vb;
    }
    __syncthreads();
    if (warp == 0) gj_inv_warp<T>(SW, Li, Pd, perm, m, A.status);    // Li = S^{-1}
    __syncthreads();
    T vec[MAXM], z[MAXM];
    const bool tbcol = tid < 2 * MAXM && (tid & (MAXM - 1)) < m;    // this thread's top / bottom column
    if (tbcol) {                                                    // W = S^{-1} B (into S's buffer)
#pragma unroll
        for (int i = 0; i < MAXM; ++i) vec[i] = i < m ? Bt[i * ZP + tid] : T(0);
        block_times<T, false>(Li, vec, z, m);
#pragma unroll
        for (int i = 0; i < MAXM; ++i)
            if (i < m) SW[i * ZP + tid] = z[i];
    }
    __syncthreads();
    if (blockIdx.y == 0) {
        T* Lg = A.linv(t, c);
        T* LTg = A.per_node(A.LinvT, t, c, m * m);
        T* Bg = A.per_node(A.ZtbT, t, c, m * m2);
        T* Wg = A.wtb(t, c);
        for (int i = warp; i < m; i += nth / 32)
            if (lane < m) {
                Lg[i * m + lane] = Li[i * LP + lane];
                LTg[i * m + lane] = Li[lane * LP + i];
                Bg[i * m2 + lane] = Bt[i * ZP + lane];
                Bg[i * m2 + m + lane] = Bt[i * ZP + MAXM + lane];
                Wg[i * m2 + lane] = SW[i * ZP + lane];
                Wg[i * m2 + m + lane] = SW[i * ZP + MAXM + lane];
            }
    }
    __syncthreads();
    // C^T: Ct[i][j] = coupling of top/bot node j into separator node i
    for (int j = warp; j < m; j += nth / 32) {                      // (lane = i: rows of the children's blocks)
        const int i = lane;
        if (i < m) {
            T vt = T(0), vb = T(0);
            if (Ra) vt = Ra[j * m2 + m + i];                        // R_alpha[top j][bot i]
            else if (i == j && c - 1 >= 1) vt = (T)(-A.AY[(int64_t)(c - 1) * np1 + x0 + i]);
            if (Rb) vb = Rb[(m + j) * m2 + i];                      // R_beta[bot j][top i]
            else if (i == j && c + 1 <= s) vb = (T)(-A.AYT[(int64_t)c * np1 + x0 + i]);
            Bt[i * ZP + j] = vt;
            Bt[i * ZP + MAXM + j] = vb;
        }
    }
    __syncthreads();
    const T* Ct = Bt;
    if (blockIdx.y == 0) {
        T* Cg = A.ztb(t, c);
        T* Vg = A.per_node(A.WtbT, t, c, m * m2);
        if (tbcol) {                                                // V = S^{-T} C^T
            const int col = tid < MAXM ? tid : m + tid - MAXM;
#pragma unroll
            for (int i = 0; i < MAXM; ++i) vec[i] = i < m ? Ct[i * ZP + tid] : T(0);
            block_transposed_times<T>(Li, vec, z, m);
#pragma unroll
            for (int i = 0; i < MAXM; ++i)
                if (i < m) {
                    Cg[i * m2 + col] = vec[i];
                    Vg[i * m2 + col] = z[i];
                }
        }
        condense_node<T, false>(Ct, SW, m, Ra, Rb, A.rtb(t, c));
    }
    // interface columns of the segment: one thread per column
    const int q = q0 + tid;
    if (q < ncols) {
        const int side = q >= w;
        const int j = lo + (side ? q - w : q);
        const int rr = j - 1;
        const int64_t sp = A.s_pad;
        // pass 0: b = coupling of the separator rows to interface node j, W column z = S^{-1} b, condensed rows
        // RI = R_child - C[tb, sep] z.  Pass 1: c = coupling of interface node j into the separator columns, V
        // column z = S^{-T} c, condensed columns RIc = R_child - c^T W[:, tb].
#pragma unroll
        for (int pass = 0; pass < 2; ++pass) {
#pragma unroll
            for (int i = 0; i < MAXM; ++i) vec[i] = T(0);
            if (j == c) {
                if (side == 0) {                                     // A[(x0,c),(x0-1,c)] and A[(x0-1,c),(x0,c)]
                    if (t >= 1) vec[0] = (T)(pass ? -AXr[x0 - 1] : -AXTr[x0 - 1]);
                } else if (t <= A.NS - 2) {
                    const T v = (T)(pass ? -AXTr[x0 + m - 1] : -AXr[x0 + m - 1]);
#pragma unroll
                    for (int i = 0; i < MAXM; ++i) if (i == m - 1) vec[i] = v;
                }
            } else {
                const T* src = (j < c ? (pass ? A.ric(t, k - 1, 1, side) : A.ri(t, k - 1, 1, side))
                                      : (pass ? A.ric(t, kb, 0, side) : A.ri(t, kb, 0, side))) + rr;
#pragma unroll
                for (int i = 0; i < MAXM; ++i) if (i < m) vec[i] = src[i * sp];
            }
            if (pass) block_transposed_times<T>(Li, vec, z, m);
            else block_times<T, false>(Li, vec, z, m);
            T* vd = (pass ? A.zi(t, k, side) : A.per_height(A.ZIT, t, k, side)) + rr;
            T* zd = A.per_height(pass ? A.WIT : A.WI, t, k, side) + rr;
#pragma unroll
            for (int i = 0; i < MAXM; ++i)
                if (i < m) {
                    vd[i * sp] = vec[i];
                    zd[i * sp] = z[i];
                }
            const T* ct = j < c ? (pass ? A.ric(t, k - 1, 0, side) : A.ri(t, k - 1, 0, side)) + rr : nullptr;
            const T* cb = j > c ? (pass ? A.ric(t, kb, 1, side) : A.ri(t, kb, 1, side)) + rr : nullptr;
            T* dt = (pass ? A.ric(t, k, 0, side) : A.ri(t, k, 0, side)) + rr;
            T* db = (pass ? A.ric(t, k, 1, side) : A.ri(t, k, 1, side)) + rr;
            if (pass) condense_column<T>(SW, vec, m, sp, ct, cb, dt, db);
            else condense_column<T>(Ct, z, m, sp, ct, cb, dt, db);
        }
    }
}

inline int chunks_at(int s, int k) {
    const int wmax = min(s, (1 << (k + 1)) - 1);
    return (2 * wmax + TB_THREADS - 1) / TB_THREADS;
}

}  // namespace

template <typename T>
slab_status tree_factor(slab_handle* h) {
    TreeArgs<T> a = make_tree_args<T>(h);
    const TreeDims& d = h->td;
    const bool indef = h->kind == SLAB_HELMHOLTZ;
    const bool nonsym = h->kind == SLAB_CONVECTION;
    for (int k = 0; k < d.H; ++k) {
        const int cnt = tree_nodes_at(d.s, k);
        if (!cnt) continue;
        dim3 grid(cnt, chunks_at(d.s, k), d.NS);
        SLAB_PROF(h, KC_TREE_FACTOR);
        if (nonsym) tree_factor_ns_kernel<T><<<grid, TB_THREADS, 0, h->stream>>>(a, k);
        else if (indef) tree_factor_kernel<T, true><<<grid, TB_THREADS, 0, h->stream>>>(a, k);
        else tree_factor_kernel<T, false><<<grid, TB_THREADS, 0, h->stream>>>(a, k);
        SLAB_CK_LAUNCH(h);
        if (slab_debug() && slab_debug_status(h, "slab tree factor (height, nodes)", k, cnt)) return SLAB_ESINGULAR;
    }
    return tree_node_major<T>(h);
}

template slab_status tree_factor<float>(slab_handle*);
template slab_status tree_factor<double>(slab_handle*);
