// Stage 2: factorisation of the block-tridiagonal reduced matrix T
// (Sec. 4, Algorithm 1) and the sweeping solve (Algorithm 2).
//
// T is symmetric positive definite for the SPD kinds, so Algorithm 1's
// S_1 = T_11, S_{j+1} = T_{j+1,j+1} - T_{j+1,j} S_j^{-1} T_{j,j+1} is carried out as a
// block Cholesky: S_j = L_j L_j^T, Y_j = L_j^{-1} T_{j,j+1}, S_{j+1} = T_{j+1,j+1} - Y_j^T Y_j.
//
// Per interface block j the tall matrix W_j = [S_j ; T_{j+1,j} ; I] (3 s_pad x s_pad, the
// middle block absent for the final interface) is eliminated column panel by column panel
// (64 columns): the panel kernel factors the 64 x 64 diagonal tile and multiplies every tile
// below it by L_kk^{-T}; one product C -= A B^T then updates everything right of the panel.
// Rows r of the identity block stay zero in columns < r, so panel kb only touches its first
// (kb+1)*64 rows.  Afterwards the lower blocks of W_j hold Y_j^T and L_j^{-T}, and
// S_{j+1} = T_{j+1,j+1} - Y_j^T (Y_j^T)^T is one more product.  In FP32 every product runs on
// the tensor cores (tcgen05, 3xTF32); the FP64 path uses the same structure on SIMT units.
//
// Algorithm 2 then needs products only (vectors stored right-hand-side major, [k][s_pad]):
//   forward   z_j = L_j^{-1} (f_j - Y_{j-1}^T z_{j-1})
//   backward  u_j = L_j^{-T} (z_j - Y_j u_{j+1}).
#include <algorithm>
#include <cstdio>
#include <vector>

#include "slab_internal.cuh"

namespace {

constexpr int TL = SLAB_TILE;   // 64
constexpr int TLP = TL + 1;
constexpr int PTP = TL + 4;      // row pitch of the panel kernels' tiles: 16-byte rows, rows four banks apart

// C(64x64) += op(A) op(B) over [k0, k1) (multiple of 16); 256 threads, 4x4 per thread.
// op(A)(i,k) = TA ? A[k*lda+i] : A[i*lda+k];  op(B)(k,j) = TB ? B[j*ldb+k] : B[k*ldb+j].
// Columns j >= ncols of B are treated as zero (and not loaded).
template <typename T, bool TA, bool TB>
__device__ inline void tile_gemm(T acc[4][4], const T* __restrict__ A, int64_t lda,
                                 const T* __restrict__ B, int64_t ldb, int k0, int k1, int ncols,
                                 T* sA, T* sB) {
    const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
    for (int kk0 = k0; kk0 < k1; kk0 += 16) {
        __syncthreads();
        for (int idx = tid; idx < 16 * TL; idx += 256) {
            int kk, i;
            if (TA) { kk = idx / TL; i = idx % TL; sA[kk * TLP + i] = A[(int64_t)(kk0 + kk) * lda + i]; }
            else { i = idx / 16; kk = idx % 16; sA[kk * TLP + i] = A[(int64_t)i * lda + kk0 + kk]; }
        }
        for (int idx = tid; idx < 16 * TL; idx += 256) {
            int kk, j;
            if (TB) { j = idx / 16; kk = idx % 16; sB[kk * TLP + j] = j < ncols ? B[(int64_t)j * ldb + kk0 + kk] : T(0); }
            else { kk = idx / TL; j = idx % TL; sB[kk * TLP + j] = j < ncols ? B[(int64_t)(kk0 + kk) * ldb + j] : T(0); }
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            T av[4], bv[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) av[a] = sA[kk * TLP + ty + 16 * a];
#pragma unroll
            for (int b = 0; b < 4; ++b) bv[b] = sB[kk * TLP + tx + 16 * b];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] += av[a] * bv[b];
        }
    }
}

// SIMT C = beta C + alpha A B^T (A [M][K], B [N][K] row-major), K multiple of 16.
// transC writes C^T; lower_only skips 64 x 64 output tiles above the diagonal; tiles of rows >= mcut and
// columns >= ncut are skipped.
template <typename T>
__global__ void __launch_bounds__(256) gemm_tn_kernel(int M, int N, int K, T alpha, const T* A, int64_t lda,
                                                      const T* B, int64_t ldb, T beta, T* C, int64_t ldc,
                                                      int transC, int lower_only, int64_t sA, int64_t sB,
                                                      int64_t sC, int mcut, int ncut) {
    __shared__ T sA_[16 * TLP];
    __shared__ T sB_[16 * TLP];
    T* sAm = sA_;
    T* sBm = sB_;
    const int bj = blockIdx.x, bi = blockIdx.y;
    A += (int64_t)blockIdx.z * sA;
    B += (int64_t)blockIdx.z * sB;
    C += (int64_t)blockIdx.z * sC;
    if (lower_only && bj > bi) return;
    if (bi * TL >= mcut && bj * TL >= ncut) return;
    const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
    T acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
    const int ncols = min(TL, N - bj * TL);
    tile_gemm<T, false, true>(acc, A + (int64_t)bi * TL * lda, lda, B + (int64_t)bj * TL * ldb, ldb, 0, K, ncols,
                              sAm, sBm);
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int r = bi * TL + ty + 16 * a, c = bj * TL + tx + 16 * b;
            if (r < M && c < N) {
                T* p = transC ? C + (int64_t)c * ldc + r : C + (int64_t)r * ldc + c;
                *p = (beta == T(0) ? T(0) : beta * *p) + alpha * acc[a][b];
            }
        }
}

// The same product on 16 x 16 tiles, one output per thread (K % 16 == 0).  An SM does two FP64 multiply-adds
// a cycle, so a product is bound by the number of SMs it runs on, not by operand reuse: taken where the
// 64 x 64 tiles would not fill the chip (128 x 128 x 128: 144 us on four CTAs, 10 us on 64).
template <typename T>
__global__ void __launch_bounds__(256) gemm_tn_spread_kernel(int M, int N, int K, T alpha, const T* A, int64_t lda,
                                                             const T* B, int64_t ldb, T beta, T* C, int64_t ldc,
                                                             int transC, int lower_only, int64_t sA, int64_t sB,
                                                             int64_t sC, int mcut, int ncut) {
    constexpr int KC = 64;
    __shared__ T sa[16][KC + 1], sb[16][KC + 1];
    pdl_wait();
    pdl_trigger();
    const int bj = blockIdx.x, bi = blockIdx.y;
    // the same tiles are left out as with 64 x 64 ones: the square part above its 64-wide diagonal tiles
    if (lower_only && bj / 4 > bi / 4) return;
    if (bi * 16 >= mcut && bj * 16 >= ncut) return;
    A += (int64_t)blockIdx.z * sA;
    B += (int64_t)blockIdx.z * sB;
    C += (int64_t)blockIdx.z * sC;
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const int r = bi * 16 + ty, c = bj * 16 + tx;
    T acc[2] = {T(0), T(0)};
    for (int k0 = 0; k0 < K; k0 += KC) {
        const int kn = min(KC, K - k0);
        T va[4], vb[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int e = tid + 256 * q, i = e / KC, k = e % KC;
            va[q] = (k < kn && bi * 16 + i < M) ? A[(int64_t)(bi * 16 + i) * lda + k0 + k] : T(0);
            vb[q] = (k < kn && bj * 16 + i < N) ? B[(int64_t)(bj * 16 + i) * ldb + k0 + k] : T(0);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int e = tid + 256 * q, i = e / KC, k = e % KC;
            sa[i][k] = va[q];
            sb[i][k] = vb[q];
        }
        __syncthreads();
#pragma unroll 8
        for (int k = 0; k < kn; k += 2) {
            acc[0] += sa[ty][k] * sb[tx][k];
            acc[1] += sa[ty][k + 1] * sb[tx][k + 1];
        }
    }
    if (r < M && c < N) {
        T* p = transC ? C + (int64_t)c * ldc + r : C + (int64_t)r * ldc + c;
        *p = (beta == T(0) ? T(0) : beta * *p) + alpha * (acc[0] + acc[1]);
    }
}

// SIMT skinny variant (N <= 64) of the same product, K split over gridDim.y CTAs per row tile;
// partial tiles go to ws and the last CTA of a tile (ticket) adds them in split order.
template <typename T>
__global__ void __launch_bounds__(256) gemm_tn_skinny_kernel(int M, int N, int K, T alpha, const T* A,
                                                             int64_t lda, const T* B, int64_t ldb, T beta, T* C,
                                                             int64_t ldc, int transC, T* ws, unsigned* tickets) {
    __shared__ T sA[16 * TLP];
    __shared__ T sB[16 * TLP];
    __shared__ bool last;
    const int bi = blockIdx.x, sp = blockIdx.y, KS = gridDim.y;
    const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
    const int kchunk = K / KS;
    const int k0 = sp * kchunk, k1 = k0 + kchunk;
    T acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
    tile_gemm<T, false, true>(acc, A + (int64_t)bi * TL * lda, lda, B, ldb, k0, k1, N, sA, sB);
    T* w = ws + ((int64_t)bi * KS + sp) * TL * TL;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) w[(ty + 16 * a) * TL + tx + 16 * b] = acc[a][b];
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(tickets + bi, 1u) == (unsigned)(KS - 1);
    __syncthreads();
    if (!last) return;
    __threadfence();
    const T* w0 = ws + (int64_t)bi * KS * TL * TL;
    for (int e = tid; e < TL * TL; e += 256) {
        const int r = e / TL, c = e % TL;
        T v = T(0);
        for (int q = 0; q < KS; ++q) v += __ldcg(w0 + (int64_t)q * TL * TL + e);
        const int gr = bi * TL + r;
        if (gr < M && c < N) {
            T* p = transC ? C + (int64_t)c * ldc + gr : C + (int64_t)gr * ldc + c;
            *p = (beta == T(0) ? T(0) : beta * *p) + alpha * v;
        }
    }
    if (tid == 0) tickets[bi] = 0;
}

// Cholesky L L^T = S of the 64 x 64 tile S (smem, stride PTP; lower triangle read) and
// Li = L^{-1} (written to smem, stride PTP), by 256 threads in 4 x 4 register blocks, as one sweep
// of right-looking elimination over [S | I] (16 block steps of 4 columns, two barriers each).
// Thread (ti, tj), tj <= ti, of the first 136 holds one block: A_ij while column block tj is not yet eliminated,
// then X_ij, the block of X = L^{-1} under construction (X starts as I).  Block step kt:
//   the diagonal thread factors its 4 x 4 block, L_kk L_kk^T = A_kk, inverts L_kk (reciprocal
//   square roots refined by one Newton step) and continues with X_kk = I;
//   the owners of block column kt publish L_ik = A_ik L_kk^{-T} and continue with X_ik = 0, the
//   owners of block row kt of X apply X_kj := L_kk^{-1} X_kj and publish it;
//   every thread below row kt applies B_ij -= L_ik R_j with R_j = L_jk^T (j > kt, its A block) or
//   R_j = X_kj (j <= kt, its X block).
// L's column block and X's row block share one staging buffer pb[p][4 j + c] (rows of L for
// j > kt, columns of X for j <= kt), so both updates are one product with no divergence, and the
// 16 column owners of a warp read 16 consecutive words per load.  A non-positive or non-finite
// pivot sets SLAB_DEV_NOTSPD and continues with 1.
// Bound by the chain of its 16 steps: in FP32 the two barriers, the 4 x 4 factor and the shared-memory round trips
// (four entries an access; a panel pair with two of these tiles 34.5 -> 30.4 us), in FP64 by the
// multiply-adds, one per sub-partition every 64 cycles (137 -> 125 us; the blocks packed into whole warps).
// A usable Cholesky pivot: positive and finite (NaN fails both comparisons), in T's own arithmetic.
__device__ __forceinline__ bool pivot_ok(float d) { return d > 0.0f && d <= 3.402823466e38f; }
__device__ __forceinline__ bool pivot_ok(double d) { return d > 0.0 && d <= 1.7976931348623157e308; }

// Four consecutive shared-memory values, 16-byte aligned: one 128-bit load (float), two (double).
__device__ __forceinline__ void ld4(const float* p, float v[4]) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void ld4(const double* p, double v[4]) {
    const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}

__device__ __forceinline__ void st4(float* p, const float v[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void st4(double* p, const double v[4]) {
    reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
}

template <typename T>
__device__ __forceinline__ void chol_inv_tile(const T* S, T* Li, unsigned* status) {
    __shared__ __align__(16) T dinv[16];          // L_kk^{-1} (4x4 lower, row-major)
    __shared__ __align__(16) T pb[4 * 64];        // column block kt of L / row block kt of X: [p][4 j + c]
    // threads 0 .. 135: the blocks on and below the diagonal, last row first, so that the warps that run out of work
    // are whole ones; the others: zeros above
    const int t = threadIdx.x, e = t < 136 ? 135 - t : t - 136;
    int bi = (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f), bj = e - bi * (bi + 1) / 2;
    if (t >= 136) { ++bi; bj = 15 - bj; bi = 15 - bi; }
    const int ti = t < 136 ? bi : -1, tj = t < 136 ? bj : -1;
    T blk[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r) ld4(S + (4 * bi + r) * PTP + 4 * bj, blk[r]);
    for (int kt = 0; kt < 16; ++kt) {
        if (ti == kt && tj == kt) {               // 4x4 Cholesky and inverse in registers
            T li[4][4];
            bool bad = false;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const T d = blk[c][c];
                T rd = rsqrt_tile(d);
                if (!pivot_ok(d)) { bad = true; rd = T(1); }
                li[c][c] = rd;
#pragma unroll
                for (int r = c + 1; r < 4; ++r) blk[r][c] *= rd;
#pragma unroll
                for (int r = c + 1; r < 4; ++r)
#pragma unroll
                    for (int q = c + 1; q <= r; ++q) blk[r][q] -= blk[r][c] * blk[q][c];
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
#pragma unroll
                for (int r = 0; r < c; ++r) li[r][c] = T(0);
#pragma unroll
                for (int r = c + 1; r < 4; ++r) {
                    T v = T(0);
#pragma unroll
                    for (int p = c; p < r; ++p) v -= blk[r][p] * li[p][c];
                    li[r][c] = v * li[r][r];
                }
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                st4(dinv + 4 * r, li[r]);
#pragma unroll
                for (int c = 0; c < 4; ++c) blk[r][c] = (r == c) ? T(1) : T(0);   // X_kk starts as I
            }
            if (bad) atomicOr(status, SLAB_DEV_NOTSPD);
        }
        __syncthreads();
        if ((tj == kt && ti > kt) || (ti == kt && tj <= kt)) {
            T di[4][4];
#pragma unroll
            for (int r = 0; r < 4; ++r) ld4(dinv + 4 * r, di[r]);
            if (ti > kt) {                        // publish L_ik = A_ik L_kk^{-T}; continue with X_ik = 0
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    T v[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        v[r] = T(0);
#pragma unroll
                        for (int p = 0; p <= c; ++p) v[r] += blk[r][p] * di[c][p];
                    }
                    st4(pb + c * 64 + 4 * ti, v);
                }
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int c = 0; c < 4; ++c) blk[r][c] = T(0);
            } else {                              // X_kt,j = L_kk^{-1} X_kt,j, published
                T o[4][4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        T v = T(0);
#pragma unroll
                        for (int p = 0; p <= r; ++p) v += di[r][p] * blk[p][c];
                        o[r][c] = v;
                    }
                    st4(pb + r * 64 + 4 * tj, o[r]);
                }
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int c = 0; c < 4; ++c) blk[r][c] = o[r][c];
            }
        }
        __syncthreads();
        if (ti > kt) {                            // B_ij -= L_ik R_j
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                T lk[4], rj[4];
                ld4(pb + p * 64 + 4 * ti, lk);
                ld4(pb + p * 64 + 4 * tj, rj);
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int c = 0; c < 4; ++c) blk[r][c] -= lk[r] * rj[c];
            }
        }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        if (ti < 0)
#pragma unroll
            for (int c = 0; c < 4; ++c) blk[r][c] = T(0);
        st4(Li + (4 * bi + r) * PTP + 4 * bj, blk[r]);
    }
    __syncthreads();
}

// Stage a 64 x 64 tile (row stride ld) in registers, then in shared memory (row stride PTP); 256
// threads.  Every global load of a thread is issued before its first shared store, so a tile costs
// one memory round trip instead of one per element the thread copies.
constexpr int TPT = TL * TL / 256;     // elements of a tile per thread
template <typename T>
__device__ __forceinline__ void tile_fetch(const T* src, int64_t ld, T (&v)[TPT]) {
#pragma unroll
    for (int q = 0; q < TPT; ++q) {
        const int i = threadIdx.x + 256 * q;
        v[q] = src[(int64_t)(i / TL) * ld + i % TL];
    }
}
template <typename T>
__device__ __forceinline__ void tile_stash(const T (&v)[TPT], T* dst) {
#pragma unroll
    for (int q = 0; q < TPT; ++q) {
        const int i = threadIdx.x + 256 * q;
        dst[(i / TL) * PTP + i % TL] = v[q];
    }
}

// acc[a][b] += sum_l X[ty + 16 a][l] Y[tx + 16 b][l] for 64 x 64 tiles X, Y in shared memory (row
// pitch PTP, 16-byte aligned), four l at a time: eight vector loads per 64 FMAs; the 16 rows
// tx + 16 b of a warp's loads are PTP = 68 words apart, so a phase of eight lanes hits eight
// distinct bank quads.
template <typename T>
__device__ __forceinline__ void tile_nt(const T* X, const T* Y, T acc[4][4], int ty, int tx) {
#pragma unroll 4
    for (int l = 0; l < TL; l += 4) {
        T av[4][4], bv[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a) ld4(X + (ty + 16 * a) * PTP + l, av[a]);
#pragma unroll
        for (int b = 0; b < 4; ++b) ld4(Y + (tx + 16 * b) * PTP + l, bv[b]);
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] += av[a][u] * bv[b][u];
    }
}

// Panel of tile column kb of the tall matrix Wt (leading dimension ld), in two launches.
// panel_diag_kernel (one CTA per matrix of the batch): Cholesky of the diagonal tile
// Wt[kb][kb] = L L^T and Linv = L^{-1} to Lw (64 x 64 per matrix, row-major).
template <typename T>
__global__ void __launch_bounds__(256) panel_diag_kernel(const T* Wt, int64_t ld, int kb, unsigned* status,
                                                         int64_t bstride, T* Lw) {
    pdl_wait();
    pdl_trigger();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* S = reinterpret_cast<T*>(smem_raw);
    T* Li = S + TL * PTP;
    const int tid = threadIdx.x;
    Wt += (int64_t)blockIdx.y * bstride;
    const T* D = Wt + (int64_t)kb * TL * ld + (int64_t)kb * TL;
    {
        T v[TPT];
        tile_fetch<T>(D, ld, v);
        tile_stash<T>(v, S);
    }
    __syncthreads();
    chol_inv_tile<T>(S, Li, status);
    T* out = Lw + (int64_t)blockIdx.y * TL * TL;
    for (int i = tid; i < TL * TL; i += 256) out[i] = Li[(i / TL) * PTP + i % TL];
}

// panel_apply_kernel: CTA x replaces the tile Wt[kb+1+x][kb] by itself times L^{-T}.  DIAG: every
// CTA factors the diagonal tile itself (the same arithmetic as panel_diag_kernel, so every CTA
// obtains the same L^{-1}) instead of reading Lw -- one launch per panel where the row tiles of the
// batch fit in one wave, so the redundant 64 x 64 factorisations cost no extra time.
template <typename T, bool DIAG>
__global__ void __launch_bounds__(256) panel_apply_kernel(T* Wt, int64_t ld, int kb, int64_t bstride,
                                                          const T* Lw, unsigned* status) {
    pdl_wait();
    pdl_trigger();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* Li = reinterpret_cast<T*>(smem_raw);
    T* X = Li + TL * PTP;
    T* S = X + TL * PTP;                          // DIAG only: the diagonal tile
    const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
    const int r = kb + 1 + blockIdx.x;
    Wt += (int64_t)blockIdx.y * bstride;
    T* src = Wt + (int64_t)r * TL * ld + (int64_t)kb * TL;
    {
        T vl[TPT], vx[TPT];
        if (DIAG) tile_fetch<T>(Wt + (int64_t)kb * TL * ld + (int64_t)kb * TL, ld, vl);
        else tile_fetch<T>(Lw + (int64_t)blockIdx.y * TL * TL, TL, vl);
        tile_fetch<T>(src, ld, vx);
        tile_stash<T>(vl, DIAG ? S : Li);
        tile_stash<T>(vx, X);
    }
    __syncthreads();
    if (DIAG) chol_inv_tile<T>(S, Li, status);
    T acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
    tile_nt<T>(X, Li, acc, ty, tx);       // out = X Li^T
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) src[(int64_t)(ty + 16 * a) * ld + tx + 16 * b] = acc[a][b];
}

// FP64 panel apply on slices of 8 rows: tile row x / 8 below the diagonal, rows 8 (x % 8) .. of it, times L^{-T}
// (each row depends on itself alone, so the tile is updated in place).  64 x 64 x 64 FP64 multiply-adds
// are 65 us of one SM.
template <typename T>
__global__ void __launch_bounds__(256) panel_apply_rows_kernel(T* Wt, int64_t ld, int kb, int64_t bstride, const T* Lw) {
    pdl_wait();
    pdl_trigger();
    __shared__ T Li[TL][TL + 1], X[8][TL];
    const int tid = threadIdx.x, c = tid & 63, r0 = (tid >> 6) * 2;
    const int rt = kb + 1 + blockIdx.x / 8, row = rt * TL + (blockIdx.x % 8) * 8;
    Wt += (int64_t)blockIdx.y * bstride;
    const T* L = Lw + (int64_t)blockIdx.y * TL * TL;
    T* src = Wt + (int64_t)row * ld + (int64_t)kb * TL;
    T v[TPT];
#pragma unroll
    for (int q = 0; q < TPT; ++q) v[q] = L[tid + 256 * q];
    for (int e = tid; e < 8 * TL; e += 256) X[e / TL][e % TL] = src[(int64_t)(e / TL) * ld + e % TL];
#pragma unroll
    for (int q = 0; q < TPT; ++q) Li[(tid + 256 * q) / TL][(tid + 256 * q) % TL] = v[q];
    __syncthreads();
    T a0 = T(0), a1 = T(0);
    const int ke = (c | 31) + 1;                  // Linv is lower triangular: a warp's columns need k < ke
#pragma unroll 8
    for (int k = 0; k < ke; ++k) {
        const T l = Li[c][k];
        a0 += X[r0][k] * l;
        a1 += X[r0 + 1][k] * l;
    }
    src[(int64_t)r0 * ld + c] = a0;
    src[(int64_t)(r0 + 1) * ld + c] = a1;
}

// Two panels kb, kb+1 of the tall Cholesky in one launch after panel_diag_kernel(kb): CTA x owns
// row tile r = kb+1+x and
//   scales its tile of panel kb, P_r = W[r][kb] L^{-T} (written back, except for r = kb+1),
//   recomputes P_{kb+1} = W[kb+1][kb] L^{-T} from the unscaled tile (every CTA reads it; its scaled
//   value is used only here, so it is never written),
//   applies panel kb to panel kb+1: W[r][kb+1] -= P_r P_{kb+1}^T,
// and the CTA of r = kb+1 then factors the updated diagonal tile of panel kb+1 (Cholesky and
// inverse, as panel_diag_kernel) into Lw2.  Panel kb+1 is finished by panel_apply_kernel(kb+1, Lw2).
// DIAG: every CTA factors panel kb's diagonal tile itself, as panel_apply_kernel<T, true>.
template <typename T, bool DIAG>
__global__ void __launch_bounds__(256) panel_pair_kernel(T* Wt, int64_t ld, int kb, int64_t bstride, const T* Lw,
                                                         T* Lw2, unsigned* status) {
    pdl_wait();
    pdl_trigger();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* Li = reinterpret_cast<T*>(smem_raw);
    T* X = Li + TL * PTP;
    T* Y = X + TL * PTP;
    T* C = Y + TL * PTP;
    T* S = C + TL * PTP;                          // DIAG only: panel kb's diagonal tile
    const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
    const int r = kb + 1 + blockIdx.x;
    Wt += (int64_t)blockIdx.y * bstride;
    T* src = Wt + (int64_t)r * TL * ld + (int64_t)kb * TL;
    const T* src1 = Wt + (int64_t)(kb + 1) * TL * ld + (int64_t)kb * TL;
    T* dst = Wt + (int64_t)r * TL * ld + (int64_t)(kb + 1) * TL;
    {
        T vl[TPT], vx[TPT], vy[TPT], vc[TPT];
        if (DIAG) tile_fetch<T>(Wt + (int64_t)kb * TL * ld + (int64_t)kb * TL, ld, vl);
        else tile_fetch<T>(Lw + (int64_t)blockIdx.y * TL * TL, TL, vl);
        tile_fetch<T>(src, ld, vx);
        tile_fetch<T>(src1, ld, vy);
        tile_fetch<T>(dst, ld, vc);
        tile_stash<T>(vl, DIAG ? S : Li);
        tile_stash<T>(vx, X);
        tile_stash<T>(vy, Y);
        tile_stash<T>(vc, C);
    }
    __syncthreads();
    if (DIAG) chol_inv_tile<T>(S, Li, status);
    T p[4][4], q[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) p[a][b] = q[a][b] = T(0);
    tile_nt<T>(X, Li, p, ty, tx);                  // P_r
    tile_nt<T>(Y, Li, q, ty, tx);                  // P_{kb+1}
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            X[(ty + 16 * a) * PTP + tx + 16 * b] = p[a][b];
            Y[(ty + 16 * a) * PTP + tx + 16 * b] = q[a][b];
            if (r != kb + 1) src[(int64_t)(ty + 16 * a) * ld + tx + 16 * b] = p[a][b];
        }
    __syncthreads();
    T u[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) u[a][b] = C[(ty + 16 * a) * PTP + tx + 16 * b];
    {
        T pq[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) pq[a][b] = T(0);
        tile_nt<T>(X, Y, pq, ty, tx);              // P_r P_{kb+1}^T
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) u[a][b] -= pq[a][b];
    }
    if (r != kb + 1) {
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) dst[(int64_t)(ty + 16 * a) * ld + tx + 16 * b] = u[a][b];
        return;
    }
    __syncthreads();                               // (uniform: this CTA alone) all reads of C done
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) C[(ty + 16 * a) * PTP + tx + 16 * b] = u[a][b];
    __syncthreads();
    chol_inv_tile<T>(C, X, status);                // X := L^{-1} of panel kb+1's diagonal tile
    T* out = Lw2 + (int64_t)blockIdx.y * TL * TL;
    for (int i = tid; i < TL * TL; i += 256) out[i] = X[(i / TL) * PTP + i % TL];
}

// Panels kb and kb+1 complete in one launch (every CTA factors both diagonal tiles itself): CTA x
// owns row tile r = kb+1+x, x = 0 .. nrt (one more than panel kb's row tiles: with the identity
// block starting on a tile boundary, the last one enters with panel kb+1, and its tile of panel kb
// is zero), and
//   factors W[kb][kb] = L L^T,  P_r = W[r][kb] L^{-T} (written back, except for r = kb+1),
//   P_{kb+1} = W[kb+1][kb] L^{-T} (recomputed from the unscaled tile, never written),
//   W[r][kb+1] -= P_r P_{kb+1}^T and the updated diagonal tile D = W[kb+1][kb+1] - P_{kb+1} P_{kb+1}^T,
//   factors D = L' L'^T and writes W[r][kb+1] L'^{-T} (except for r = kb+1, the diagonal tile).
// The same arithmetic in every CTA gives every CTA the same L^{-1} and L'^{-1}.
template <typename T>
__global__ void __launch_bounds__(256) panel_pair_full_kernel(T* Wt, int64_t ld, int kb, int64_t bstride,
                                                              unsigned* status) {
    pdl_wait();
    pdl_trigger();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* Li = reinterpret_cast<T*>(smem_raw);
    T* X = Li + TL * PTP;
    T* Y = X + TL * PTP;
    T* C = Y + TL * PTP;
    T* S = C + TL * PTP;
    const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
    const int r = kb + 1 + blockIdx.x;
    Wt += (int64_t)blockIdx.y * bstride;
    T* src = Wt + (int64_t)r * TL * ld + (int64_t)kb * TL;
    const T* src1 = Wt + (int64_t)(kb + 1) * TL * ld + (int64_t)kb * TL;
    T* dst = Wt + (int64_t)r * TL * ld + (int64_t)(kb + 1) * TL;
    T vd[TPT];
    {
        T vs[TPT], vx[TPT], vy[TPT], vc[TPT];
        tile_fetch<T>(Wt + (int64_t)kb * TL * ld + (int64_t)kb * TL, ld, vs);
        tile_fetch<T>(src, ld, vx);
        tile_fetch<T>(src1, ld, vy);
        tile_fetch<T>(dst, ld, vc);
        tile_fetch<T>(Wt + (int64_t)(kb + 1) * TL * ld + (int64_t)(kb + 1) * TL, ld, vd);
        tile_stash<T>(vs, S);
        tile_stash<T>(vx, X);
        tile_stash<T>(vy, Y);
        tile_stash<T>(vc, C);
    }
    __syncthreads();
    chol_inv_tile<T>(S, Li, status);               // ends with a barrier: S is free
    tile_stash<T>(vd, S);
    T p[4][4], q[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) p[a][b] = q[a][b] = T(0);
    tile_nt<T>(X, Li, p, ty, tx);                  // P_r
    tile_nt<T>(Y, Li, q, ty, tx);                  // P_{kb+1}
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            X[(ty + 16 * a) * PTP + tx + 16 * b] = p[a][b];
            Y[(ty + 16 * a) * PTP + tx + 16 * b] = q[a][b];
            if (r != kb + 1) src[(int64_t)(ty + 16 * a) * ld + tx + 16 * b] = p[a][b];
        }
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) p[a][b] = q[a][b] = T(0);
    tile_nt<T>(X, Y, p, ty, tx);                   // P_r P_{kb+1}^T
    tile_nt<T>(Y, Y, q, ty, tx);                   // P_{kb+1} P_{kb+1}^T
    T u[4][4], d[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            u[a][b] = C[(ty + 16 * a) * PTP + tx + 16 * b] - p[a][b];
            d[a][b] = S[(ty + 16 * a) * PTP + tx + 16 * b] - q[a][b];
        }
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            C[(ty + 16 * a) * PTP + tx + 16 * b] = u[a][b];
            S[(ty + 16 * a) * PTP + tx + 16 * b] = d[a][b];
        }
    __syncthreads();
    chol_inv_tile<T>(S, Li, status);               // L'^{-1}
    if (r == kb + 1) return;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) p[a][b] = T(0);
    tile_nt<T>(C, Li, p, ty, tx);
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) dst[(int64_t)(ty + 16 * a) * ld + tx + 16 * b] = p[a][b];
}

// The block S (n x n, n a multiple of 64) and the identity, ident elements after it, into the tall matrices W; blockIdx.y
// selects one of a batch, ss and sw elements apart.  One launch in the chain of dependent launches: a copy and a
// memset for each matrix and a launch for the ones took 3 us a matrix (n = 777: 75 copies,
// factor + solve 9.08 -> 8.86 ms; n = 512 factor + solve + adjoint 5.27 -> 5.03 ms).
template <typename T>
__global__ void __launch_bounds__(256) tall_fill_kernel(const T* S, int64_t ss, T* W, int64_t sw, int64_t ident, int n) {
    constexpr int V = 16 / sizeof(T);
    pdl_wait();
    pdl_trigger();
    S += (int64_t)blockIdx.y * ss;
    W += (int64_t)blockIdx.y * sw;
    for (int r = blockIdx.x; r < n; r += gridDim.x)
        for (int c = threadIdx.x; c < n / V; c += 256) {
            const int64_t e = (int64_t)r * (n / V) + c;
            alignas(16) T one[V];
#pragma unroll
            for (int q = 0; q < V; ++q) one[q] = c * V + q == r ? T(1) : T(0);
            reinterpret_cast<uint4*>(W)[e] = reinterpret_cast<const uint4*>(S)[e];
            reinterpret_cast<uint4*>(W + ident)[e] = *reinterpret_cast<const uint4*>(one);
        }
}
template <typename T>
slab_status tall_fill(slab_handle* h, const T* S, int64_t ss, T* W, int64_t sw, int64_t ident, int n, int batch) {
    SLAB_PROF(h, KC_OTHER);
    SLAB_CK(h, launch_pdl(tall_fill_kernel<T>, dim3(n, batch), dim3(256), 0, h->stream, S, ss, W, sw, ident, n));
    return SLAB_OK;
}

// out[c][r] = in[r][c] for the 64 x 64 tile (blockIdx.y, blockIdx.x) of a rows x cols block, 256
// threads: every thread issues its 16 loads (rows of in, coalesced) before its first shared store,
// then writes 16 elements (rows of out, coalesced).  tile[.][65]: column reads are conflict-free.
template <typename T>
__device__ __forceinline__ void transpose_tile64(const T* in, int64_t ldin, T* out, int64_t ldout, int rows, int cols,
                                                 T* copy = nullptr) {
    __shared__ T tile[64][65];
    const int c0 = blockIdx.x * 64, r0 = blockIdx.y * 64;
    const int tx = threadIdx.x & 63, ty = threadIdx.x >> 6;
    T v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        const int r = r0 + ty + 4 * q, c = c0 + tx;
        v[q] = (r < rows && c < cols) ? in[(int64_t)r * ldin + c] : T(0);
        if (copy && r < rows && c < cols) copy[(int64_t)r * ldin + c] = v[q];
    }
#pragma unroll
    for (int q = 0; q < 16; ++q) tile[ty + 4 * q][tx] = v[q];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        const int c = c0 + ty + 4 * q, r = r0 + tx;
        if (r < rows && c < cols) out[(int64_t)c * ldout + r] = tile[tx][ty + 4 * q];
    }
}

// out = in^T for an n x n block (both row-major, leading dimension n); blockIdx.z selects one of a
// batch of blocks sin / sout elements apart.  copy (optional, sout apart): in as it is.
template <typename T>
__global__ void __launch_bounds__(256) transpose_kernel(const T* in, T* out, int n, int64_t sin, int64_t sout, T* copy) {
    pdl_wait();
    pdl_trigger();
    transpose_tile64<T>(in + (int64_t)blockIdx.z * sin, n, out + (int64_t)blockIdx.z * sout, n, n, n,
                        copy ? copy + (int64_t)blockIdx.z * sout : nullptr);
}

template <typename T>
slab_status transpose_batched(slab_handle* h, const T* in, int64_t sin, T* out, int64_t sout, int n, int batch,
                              T* copy = nullptr) {
    if (batch <= 0) return SLAB_OK;
    dim3 grid((n + 63) / 64, (n + 63) / 64, batch);
    SLAB_PROF(h, KC_OTHER);
    SLAB_CK(h, launch_pdl(transpose_kernel<T>, grid, dim3(256), 0, h->stream, in, out, n, sin, sout, copy));
    return SLAB_OK;
}

template <typename T>
slab_status transpose(slab_handle* h, const T* in, T* out, int n) {
    return transpose_batched<T>(h, in, 0, out, 0, n, 1);
}

// The factor's Schur, trailing and (3-D) T-assembly products (FP32, 3xTF32 accuracy requested)
// run as three FP16 products of row-scaled hi/lo splits when the handle holds a large enough
// work buffer (it exists only while the factor runs).
inline bool use_f16x3(slab_handle* h, int cls, TcGemmArgs& g) {
    if (!h->w16 || g.split != 1 || (cls != KC_SYRK && cls != KC_TRAIL && cls != KC_ASSEMBLE) || g.K % 64)
        return false;
    if (f16x3_work_bytes(g.M, g.N, g.K, g.batch, f16x3_shared(g)) > h->w16_bytes) return false;
    g.split = 2;
    g.w16 = h->w16;
    g.w16_bytes = h->w16_bytes;
    return true;
}

// The solve phases' products with few loads (their A is a stored factor) have kernels of their own.
inline bool use_solve_product(int cls, int N, int K, const float* A, int64_t lda, int64_t sA, const float* B,
                              int64_t ldb, int64_t sB, int lower_only) {
    return (cls == KC_SOLVE_PROD || cls == KC_TREE_UP || cls == KC_TREE_DOWN) && !lower_only &&
           solve_product_ok(N, K, A, lda, sA, B, ldb, sB);
}

// C = beta C + alpha A B^T on the unit of this precision: tensor cores for FP32, SIMT for FP64.
// mcut > 0: rows from mcut on are wanted only in the columns below ncut (whole tiles beyond are skipped).
template <typename T>
slab_status gemm_tn(slab_handle* h, int cls, int M, int N, int K, T alpha, const T* A, int64_t lda, const T* B,
                    int64_t ldb, T beta, T* C, int64_t ldc, int transC, int lower_only, int triA = 0, int mcut = 0,
                    int ncut = 0);

template <>
slab_status gemm_tn<float>(slab_handle* h, int cls, int M, int N, int K, float alpha, const float* A, int64_t lda,
                           const float* B, int64_t ldb, float beta, float* C, int64_t ldc, int transC,
                           int lower_only, int triA, int mcut, int ncut) {
    SLAB_PROF(h, cls);
    if (use_solve_product(cls, N, K, A, lda, 0, B, ldb, 0, lower_only))
        return solve_product(h, M, N, K, alpha, A, lda, 0, B, ldb, 0, beta, C, ldc, 0, transC, triA, 1);
    TcGemmArgs g;
    g.M = M; g.N = N; g.K = K; g.alpha = alpha; g.beta = beta;
    g.A = A; g.lda = lda; g.B = B; g.ldb = ldb; g.C = C; g.ldc = ldc;
    g.transC = transC; g.split = h->tf32_now ? 0 : 1; g.lower_only = lower_only;
    g.batch = 1; g.sA = g.sB = g.sC = 0;
    g.ksplit = 1; g.part = nullptr;
    g.w16 = nullptr; g.w16_bytes = 0;
    g.triA = triA;
    if (mcut > 0) { g.mcut = mcut; g.ncut = ncut; }
    if (use_f16x3(h, cls, g)) {
        // FP16 three-product path (factor products)
    } else if (N <= 64 && !lower_only && h->wPart) {     // skinny: split K over CTAs
        const int64_t cap = (int64_t)splitk_part_bytes(h->td.s_pad) / sizeof(float);
        int ks = 1;
        while (2 * ks <= SLAB_SPLITK && (M + 127) / 128 * ks < 148 && K % (2 * ks * 32) == 0 &&
               (int64_t)2 * ks * M * N <= cap)
            ks *= 2;
        g.ksplit = ks;
        g.part = (float*)h->wPart;
    }
    const slab_status st = tc_gemm(h->stream, g, h->dstatus);
    if (st == SLAB_ECUDA && h->err == SLAB_OK) h->err = SLAB_ECUDA;
    prof_extra(h, cls, tc_gemm_extra_launches(g));
    return st;
}

template <typename T>
__global__ void scale_matrix_kernel(T* C, int64_t ldc, int M, int N, T beta) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)M * N) return;
    T* p = C + (e / N) * ldc + e % N;
    *p = beta == T(0) ? T(0) : beta * *p;
}

// C = beta C + alpha A B^T for N <= 8 (right-hand sides): one warp per row of A, lanes over K
// (coalesced), so the product streams A once at memory speed.
template <typename T, int NB>
__global__ void __launch_bounds__(256) gemv_rows_kernel(int M, int N, int K, T alpha, const T* __restrict__ A,
                                                        int64_t lda, const T* __restrict__ B, int64_t ldb, T beta,
                                                        T* C, int64_t ldc, int transC) {
    const int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (row >= M) return;
    T acc[NB];
#pragma unroll
    for (int r = 0; r < NB; ++r) acc[r] = T(0);
    const T* a = A + (int64_t)row * lda;
    for (int k = lane; k < K; k += 32) {
        const T av = a[k];
#pragma unroll
        for (int r = 0; r < NB; ++r)
            if (r < N) acc[r] += av * B[(int64_t)r * ldb + k];
    }
#pragma unroll
    for (int r = 0; r < NB; ++r) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
    }
    if (lane == 0) {
#pragma unroll
        for (int r = 0; r < NB; ++r) {
            if (r >= N) break;
            T* c = transC ? C + (int64_t)r * ldc + row : C + (int64_t)row * ldc + r;
            *c = (beta == T(0) ? T(0) : beta * *c) + alpha * acc[r];
        }
    }
}

// SIMT FP64 product, on 16 x 16 tiles where fewer than four 64 x 64 tiles an SM would run.
slab_status launch_fp64_product(slab_handle* h, int M, int N, int K, double alpha, const double* A, int64_t lda,
                                int64_t sA, const double* B, int64_t ldb, int64_t sB, double beta, double* C,
                                int64_t ldc, int64_t sC, int transC, int lower_only, int batch, int mcut, int ncut) {
    if (M <= 0 || N <= 0) return SLAB_OK;
    const dim3 big((N + TL - 1) / TL, (M + TL - 1) / TL, batch);
    if ((int64_t)big.x * big.y * batch < 4 * SMS && (M + 15) / 16 <= 65535)
        SLAB_CK(h, launch_pdl(gemm_tn_spread_kernel<double>, dim3((N + 15) / 16, (M + 15) / 16, batch), dim3(256), 0,
                              h->stream, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, transC, lower_only, sA, sB, sC,
                              mcut, ncut));
    else
        gemm_tn_kernel<double><<<big, 256, 0, h->stream>>>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, transC, lower_only,
                                                           sA, sB, sC, mcut, ncut);
    SLAB_CK_LAUNCH(h);
    return SLAB_OK;
}

template <>
slab_status gemm_tn<double>(slab_handle* h, int cls, int M, int N, int K, double alpha, const double* A,
                            int64_t lda, const double* B, int64_t ldb, double beta, double* C, int64_t ldc,
                            int transC, int lower_only, int /*triA: the FP64 products read all of A*/, int mcut,
                            int ncut) {
    if (N <= 8 && !lower_only && M > 0) {
        SLAB_PROF(h, cls);
        gemv_rows_kernel<double, 8><<<(M + 7) / 8, 256, 0, h->stream>>>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc,
                                                                       transC);
        SLAB_CK_LAUNCH(h);
        return SLAB_OK;
    }
    if (h->fp64tc_now && !transC && K % 32 == 0 && M > 0 && N > 0) {
        // FP64-accurate tensor-core product, K in chunks of 64
        SLAB_PROF(h, cls);
        if (beta != 1.0) {
            scale_matrix_kernel<double><<<(unsigned)(((int64_t)M * N + 255) / 256), 256, 0, h->stream>>>(C, ldc, M, N,
                                                                                                         beta);
            SLAB_CK_LAUNCH(h);
        }
        for (int k0 = 0; k0 < K; k0 += 64) {
            const int kc = std::min(64, K - k0);
            const slab_status st = ozaki_gemm(h->stream, M, N, kc, alpha, A + k0, lda, B + k0, ldb, C, ldc, lower_only,
                                              h->ozw, h->dstatus, mcut, ncut);
            if (st) {
                if (h->err == SLAB_OK) h->err = st;
                return st;
            }
        }
        // launches beyond the one counted: the scaling of C and two per K chunk (split, product)
        prof_extra(h, cls, (beta != 1.0 ? 1 : 0) + 2 * ((K + 63) / 64) - 1);
        return SLAB_OK;
    }
    SLAB_PROF(h, cls);
    if (N <= 64 && !lower_only && h->wTickets) {
        int KS = K / 256;
        if (KS < 1) KS = 1;
        if (KS > SLAB_SPLITK) KS = SLAB_SPLITK;
        while (K % (KS * 16)) --KS;
        dim3 grid((M + TL - 1) / TL, KS);
        gemm_tn_skinny_kernel<double><<<grid, 256, 0, h->stream>>>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc,
                                                                   transC, (double*)h->wPart, h->wTickets);
    } else {
        return launch_fp64_product(h, M, N, K, alpha, A, lda, 0, B, ldb, 0, beta, C, ldc, 0, transC, lower_only, 1,
                                   mcut > 0 ? mcut : M, ncut);
    }
    SLAB_CK_LAUNCH(h);
    return SLAB_OK;
}

// ---------------------------------------------------------------- general kinds (Helmholtz, convection)
// Blocked Gauss-Jordan elimination of the augmented system of interface j, one matrix G of 2 s_pad rows
// with leading dimension 3 s_pad:
//   top    [ S_j        | T_{j,j+1}    | I ]      (wt = 3 s_pad columns; [S | I], 2 s_pad, for the last j)
//   bottom [ T_{j+1,j}  | T_{j+1,j+1}      ]      (2 s_pad columns)
// eliminating the S_j columns in panels of 64.  At the end the top rows hold (in pivot order)
// [I | S_j^{-1} T_{j,j+1} | S_j^{-1}] and the bottom right block is S_{j+1} of Algorithm 1.
// Rows are never swapped: perm[c] records the physical top row that pivots on column c.
// Pivot rows of a panel are chosen by tournament pivoting: partial-pivoting elimination on 256-row
// groups of the not-yet-pivoted rows keeps 64 winners each, and up to four winner sets are merged
// (original row values) until one set of 64 is left.  Up to 512 rows are one group: 37 us in FP32 where two
// groups and their merge took 50 (256 rows: 26).  The panel step is then
//   A11 = G[piv, panel],  X = A11^{-1} G[piv, rest],  G[piv, rest] = X,  G[piv, panel] = 0,
//   G[all, rest] -= G[all, panel] X       (tensor-core rank-64 update of all rows).
// The s_pad / 64 panel steps of an interface are a serial chain, so their latency is what counts:
// three launches a step (tournament, which also delivers the LU of A11 in FP32, solve, update).  Measured:
// convection n = 768, b = 24 factor + solve + adjoint 230 -> 43 ms, Helmholtz n = 512, b = 32 (FP64) 103 -> 28 ms
// against one warp per 128-row group in shared memory, LU and solve with barriers every column, and two updates.
constexpr int GJ_LEAF = 256;          // rows per tournament group, one per thread
constexpr int GJ_WAY = 4;             // winner sets per merge: GJ_WAY * 64 = GJ_LEAF rows
constexpr int GJ_ONE = 512;           // more rows than a group's, up to these, are one group without a merge

// LU factors of A11 as the solve kernel reads them: L and U each as [step k][thread q][c], the
// multipliers of rows TPC (k / TPC + c) + q of step k (U with rows and steps counted from the end), zero
// where the row is not below (above) the step; then the reciprocals of U's diagonal.  TPC threads share a
// column of the solve: 4 in FP32; 16 in FP64, where an SM sub-partition starts a warp's multiply-add
// only every 64 cycles, so that a panel's solve has to be spread over all of them.
template <typename T>
struct LuLayout {
    static constexpr int TPC = sizeof(T) == 8 ? 16 : 4;
    static constexpr int C = 64 / TPC;
    static constexpr int PITCH = C + (sizeof(T) == 8 ? 2 : 4);   // 16-byte rows, the threads' rows on distinct banks
    static constexpr int TRI = 64 * TPC * PITCH;
    static constexpr int ELEMS = 2 * TRI + 64;
    // element e of 64 x 64: its step, row and place
    __device__ static void at(int e, int& k, int& i, int& place) {
        const int q = (e / C) % TPC, c = e % C;
        k = e >> 6;
        i = TPC * (k / TPC + c) + q;
        place = (k * TPC + q) * PITCH + c;
    }
};

struct GjWork {
    int* act;         // [2][s_pad] not-yet-pivoted top rows, double-buffered by panel parity
    int* perm;        // [s_pad] physical row pivoting on column c
    int* pflag;       // [s_pad] panel index + 1 at which the row pivoted (0: not yet)
    int* cand;        // tournament winner sets, [nodes][64]
    unsigned* tick;   // tournament tickets, [nodes]
    int* piv;         // [64] pivot rows of the current panel, in elimination order
};

__host__ __device__ inline int gj_level_count(int L, int l) {          // nodes at tournament level l
    int c = L;
    for (int i = 0; i < l; ++i) c = (c + GJ_WAY - 1) / GJ_WAY;
    return c;
}
__host__ __device__ inline int gj_level_off(int L, int l) {
    int o = 0, c = L;
    for (int i = 0; i < l; ++i) { o += c; c = (c + GJ_WAY - 1) / GJ_WAY; }
    return o;
}
__host__ __device__ inline int gj_nodes(int L) {                       // all nodes, leaves to root
    int o = 0, c = L;
    while (c > 1) { o += c; c = (c + GJ_WAY - 1) / GJ_WAY; }
    return o + 1;
}

// 64 values of a row, 16 bytes at a time (16-byte aligned rows), as floats.
__device__ __forceinline__ void load_row64(const float* p, float (&a)[64]) {
#pragma unroll
    for (int c = 0; c < 64; c += 4) {
        const float4 v = *reinterpret_cast<const float4*>(p + c);
        a[c] = v.x; a[c + 1] = v.y; a[c + 2] = v.z; a[c + 3] = v.w;
    }
}
__device__ __forceinline__ void load_row64(const double* p, float (&a)[64]) {
#pragma unroll
    for (int c = 0; c < 64; c += 2) {
        const double2 v = *reinterpret_cast<const double2*>(p + c);
        a[c] = (float)v.x; a[c + 1] = (float)v.y;
    }
}

template <int ROWS>
struct GeppSmem {
    float row[2][ROWS / 32][8];        // each warp's candidate: its columns of the current block
    unsigned key[2][ROWS / 32];
    int tid[2][ROWS / 32];
    float tail[8][64];                 // the block's pivot rows right of the block, then U there
    float mul[8][8];                   // the block's multipliers of its own pivot rows
    int order[64];                     // the chosen threads
    int rows[ROWS];                    // physical rows
    int base[ROWS / 32];
    int go;
};

// Partial-pivoting elimination of up to ROWS rows x 64 columns, thread t holding row t in registers
// (have: it holds one), in blocks of 8 columns.  In a block, each of the 8 steps has one barrier: every
// warp publishes its best row's 8 columns, and after the barrier every thread picks the best warp (first
// in row order among equals; a NaN counts as largest and is flagged when A11 is factored) and updates
// its own 8 columns.  Then the 8 pivot rows are finished right of the block by one thread a column, all
// other rows take the rank-8 update, and the registers move 8 columns left, so that every block runs
// the same code.  sm.order receives the 64 chosen threads.  With emit, Lm[k][t] = the multiplier of
// thread t's row in step k (pitch ROWS) and Us[k][j] = U (pitch 65).
// Bound by the latency of the 64 dependent steps: publishing and updating whole rows in every step
// took 300 instructions a step and twice the time.
template <int ROWS>
__device__ __forceinline__ void gj_gepp(float (&a)[64], bool have, GeppSmem<ROWS>& sm, bool emit, float* Lm, float* Us,
                                        unsigned* status) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    bool open = have;
#pragma unroll 1
    for (int jb = 0; jb < 64; jb += 8) {
        float lm[8];
        int mine = -1;                                   // step of this block that chose this row
#pragma unroll
        for (int jj = 0; jj < 8; ++jj) {
            const int buf = jj & 1;
            const unsigned key = open ? (__float_as_uint(a[jj]) & 0x7fffffffu) + 1u : 0u;
            const unsigned best = __reduce_max_sync(0xffffffffu, key);
            const int src = __ffs(__ballot_sync(0xffffffffu, key == best)) - 1;
            if (lane == src) {
                sm.key[buf][warp] = best;
                sm.tid[buf][warp] = t;
#pragma unroll
                for (int c = jj & ~3; c < 8; c += 4)
                    *reinterpret_cast<float4*>(&sm.row[buf][warp][c]) = make_float4(a[c], a[c + 1], a[c + 2], a[c + 3]);
            }
            __syncthreads();
            const unsigned kw = lane < ROWS / 32 ? sm.key[buf][lane] : 0u;
            const unsigned bk = __reduce_max_sync(0xffffffffu, kw);
            const int ww = __ffs(__ballot_sync(0xffffffffu, kw == bk)) - 1;
            float p[8];
#pragma unroll
            for (int c = jj & ~3; c < 8; c += 4) {
                const float4 v = *reinterpret_cast<const float4*>(&sm.row[buf][ww][c]);
                p[c] = v.x; p[c + 1] = v.y; p[c + 2] = v.z; p[c + 3] = v.w;
            }
            if (t == sm.tid[buf][ww]) {
                open = false;
                mine = jj;
                sm.order[jb + jj] = t;
            }
            const float l = bk > 1u ? pivot_quotient(a[jj], p[jj], bk - 1u) : 0.f;   // a pivot that is not zero
            lm[jj] = l;
            if (emit) {
                const bool ok = bk > 1u && bk <= 0x7f800000u;            // and finite
                if (t >= jj && t < 8) Us[(jb + jj) * 65 + jb + t] = (t == jj && !ok) ? 1.f : sm.row[buf][ww][t];
                if (t == 0 && !ok) atomicOr(status, SLAB_DEV_NOTSPD);
                Lm[(jb + jj) * ROWS + t] = l;
            }
#pragma unroll
            for (int c = jj + 1; c < 8; ++c) a[c] -= l * p[c];           // (a chosen row's are not used again)
        }
        const int left = 56 - jb;                        // columns right of the block
        if (left == 0) break;
        if (mine >= 0) {
#pragma unroll
            for (int c = 0; c < 56; c += 4)
                if (c < left)
                    *reinterpret_cast<float4*>(&sm.tail[mine][c]) = make_float4(a[c + 8], a[c + 9], a[c + 10], a[c + 11]);
            *reinterpret_cast<float4*>(&sm.mul[mine][0]) = make_float4(lm[0], lm[1], lm[2], lm[3]);
            *reinterpret_cast<float4*>(&sm.mul[mine][4]) = make_float4(lm[4], lm[5], lm[6], lm[7]);
        }
        __syncthreads();
        if (t < left) {                                  // U right of the block, one thread a column
            float u[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                u[k] = sm.tail[k][t];
#pragma unroll
                for (int i = 0; i < k; ++i) u[k] -= sm.mul[k][i] * u[i];
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                sm.tail[k][t] = u[k];
                if (emit) Us[(jb + k) * 65 + jb + 8 + t] = u[k];
            }
        }
        __syncthreads();
        if (open) {
#pragma unroll
            for (int c = 0; c < 56; c += 4)
                if (c < left) {
                    float v[4] = {a[c + 8], a[c + 9], a[c + 10], a[c + 11]};
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const float4 u = *reinterpret_cast<const float4*>(&sm.tail[k][c]);
                        v[0] -= lm[k] * u.x; v[1] -= lm[k] * u.y; v[2] -= lm[k] * u.z; v[3] -= lm[k] * u.w;
                    }
                    a[c] = v[0]; a[c + 1] = v[1]; a[c + 2] = v[2]; a[c + 3] = v[3];
                }
        }
    }
    __syncthreads();
}

// One launch per panel: leaves, merges (ticketed: the last child's CTA goes on; deterministic), and at the
// root the panel's pivot rows in elimination order, their flags and perm entries, the compacted list of
// remaining rows and, where lu is given (FP32), the LU factors of A11, which the root's elimination
// has just computed.  For FP64 storage the choice of rows runs in FP32 all the same (it only chooses);
// gj_a11_lu_kernel then factors A11 in FP64.
template <typename T, int ROWS>
__global__ void __launch_bounds__(ROWS) gj_tournament_kernel(const T* __restrict__ G, int64_t ld, int c0, int panel,
                                                                int nact, GjWork w, const int* act, int* act_next,
                                                                float* lu, unsigned* status) {
    extern __shared__ __align__(16) unsigned char gj_smem[];
    __shared__ GeppSmem<ROWS> sm;
    pdl_wait();
    pdl_trigger();
    float* Lm = reinterpret_cast<float*>(gj_smem);       // [64][ROWS], with lu only
    float* Us = Lm + 64 * ROWS;                       // [64][65]
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int L = (nact + ROWS - 1) / ROWS;
    int node = blockIdx.x, lvl = 0;
    int nr = min(ROWS, nact - node * ROWS);
    if (t < nr) sm.rows[t] = act[node * ROWS + t];
    while (true) {
        const bool root = gj_level_count(L, lvl) == 1;
        float a[64];
        __syncthreads();
        if (t < nr) load_row64(G + (int64_t)sm.rows[t] * ld + c0, a);
        else
#pragma unroll
            for (int c = 0; c < 64; ++c) a[c] = 0.f;
        gj_gepp<ROWS>(a, t < nr, sm, root && lu, Lm, Us, status);
        if (root) break;
        const int parent = node / GJ_WAY;
        const int nchild = min(GJ_WAY, gj_level_count(L, lvl) - GJ_WAY * parent);
        if (t < 64) w.cand[(gj_level_off(L, lvl) + node) * 64 + t] = sm.rows[sm.order[t]];
        __threadfence();
        __syncthreads();
        if (t == 0) sm.go = atomicAdd(w.tick + gj_level_off(L, lvl + 1) + parent, 1u) + 1u == (unsigned)nchild;
        __syncthreads();
        if (!sm.go) return;                              // another child's CTA finishes the merge
        __threadfence();
        nr = nchild * 64;
        if (t < nr) sm.rows[t] = __ldcg(w.cand + (gj_level_off(L, lvl) + GJ_WAY * parent) * 64 + t);
        node = parent;
        ++lvl;
    }
    if (t < 64) {
        const int r = sm.rows[sm.order[t]];
        w.piv[t] = r;
        w.perm[c0 + t] = r;
        w.pflag[r] = panel + 1;
    }
    // every other CTA has taken its ticket: reset them for the next panel
    for (int i = t; i < gj_nodes(L); i += ROWS) w.tick[i] = 0u;
    if (lu) {
        using Lay = LuLayout<float>;
        for (int e = t; e < 64 * 64; e += ROWS) {
            int k, i, pl;
            Lay::at(e, k, i, pl);
            const bool in = i > k && i < 64;
            lu[pl] = in ? Lm[k * ROWS + sm.order[i & 63]] : 0.f;
            lu[Lay::TRI + pl] = in ? Us[(63 - (i & 63)) * 65 + 63 - k] : 0.f;
        }
        if (t < 64) lu[2 * Lay::TRI + t] = 1.f / Us[t * 65 + t];
    }
    __threadfence_block();
    __syncthreads();
    // remaining rows, in order
    int done = 0;
    for (int i0 = 0; i0 < nact; i0 += ROWS) {
        const int r = i0 + t < nact ? act[i0 + t] : -1;
        const bool keep = r >= 0 && __ldcg(w.pflag + r) != panel + 1;
        const unsigned bal = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) sm.base[warp] = __popc(bal);
        __syncthreads();
        int off = done, tot = 0;
        for (int q = 0; q < ROWS / 32; ++q) {
            if (q < warp) off += sm.base[q];
            tot += sm.base[q];
        }
        if (keep) act_next[off + __popc(bal & ((1u << lane) - 1u))] = r;
        done += tot;
        __syncthreads();
    }
}

// Pivot rows restricted to the diagonal block: the panel's pivot rows are the first 64 rows not yet
// pivoted, in order (the rows c0 .. c0+63 when every earlier panel did the same); A11's own partial
// pivoting (gj_a11_lu_kernel) orders them.
__global__ void __launch_bounds__(256) gj_local_rows_kernel(int panel, int nact, GjWork w, const int* act,
                                                            int* act_next) {
    pdl_wait();
    pdl_trigger();
    for (int i = threadIdx.x; i < nact; i += 256) {
        const int r = act[i];
        if (i < 64) {
            w.piv[i] = r;
            w.pflag[r] = panel + 1;
        } else {
            act_next[i - 64] = r;
        }
    }
}

// LU of the panel's pivot block A11 = G[piv, panel] with partial pivoting in T, into the solve kernel's
// layout; reorders piv by the elimination and records it in perm.  One CTA; four threads a row, thread q
// holding columns 4 c + q, c < 16, moved one register left every four steps.  The four steps of a block touch
// its own columns only, with two barriers each: every warp publishes its best row, the winner its reciprocal.
// Then the four pivot rows are finished right of the block, a thread a column, and all other rows take
// the rank-4 update.  In FP64 a sub-partition starts a multiply-add every 64 cycles, so the chain of the steps
// must not wait for whole rows (93 us when each step updated all columns, 72 us now) and magnitudes are
// compared as integers (FP64: the upper words).  A zero or non-finite pivot sets SLAB_DEV_NOTSPD.
__device__ __forceinline__ unsigned magnitude_key(float v) { return __float_as_uint(v) & 0x7fffffffu; }
__device__ __forceinline__ unsigned magnitude_key(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }
__device__ __forceinline__ bool usable_pivot(float v) {
    const unsigned k = magnitude_key(v);
    return k != 0u && k < 0x7f800000u;
}
__device__ __forceinline__ bool usable_pivot(double v) {
    const unsigned k = magnitude_key(v);
    return (k | (unsigned)__double2loint(v)) != 0u && k < 0x7ff00000u;
}
template <typename T>
__global__ void __launch_bounds__(256) gj_a11_lu_kernel(const T* __restrict__ G, int64_t ld, int c0, int* piv, int* perm,
                                                        T* lu, unsigned* status) {
    extern __shared__ __align__(16) unsigned char gj_smem[];
    T* Lm = reinterpret_cast<T*>(gj_smem);               // [64 steps][64 rows]
    T* Us = Lm + 64 * 64;                                // [64][65]
    __shared__ T slot[2][8][4];                          // each warp's candidate: its columns of the block
    __shared__ T tail[4][64];                            // the block's pivot rows right of the block, then U there
    __shared__ T mul[4][4];                              // the block's multipliers of its own pivot rows
    __shared__ T rps[2];
    __shared__ unsigned bk[2][8];
    __shared__ int br[2][8], order[64], prow[64];
    pdl_wait();
    pdl_trigger();
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, r = t >> 2, q = t & 3;
    if (t < 64) prow[t] = piv[t];
    __syncthreads();
    T a[16];
    {
        const T* src = G + (int64_t)prow[r] * ld + c0 + q;
#pragma unroll
        for (int c = 0; c < 16; ++c) a[c] = src[4 * c];
    }
    bool open = true;
#pragma unroll 1
    for (int kc = 0; kc < 16; ++kc) {
        T lm[4];
        int mine = -1;                                   // step of this block that chose this row
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int k = 4 * kc + u, buf = k & 1;
            const T v = __shfl_sync(0xffffffffu, a[0], (lane & ~3) | u);     // this row's entry of column k
            const unsigned key = open ? magnitude_key(v) + 1u : 0u;
            const unsigned best = __reduce_max_sync(0xffffffffu, key);
            const int src = __ffs(__ballot_sync(0xffffffffu, key == best)) - 1;   // first lane of a row
            if ((lane & ~3) == src) {
                slot[buf][warp][q] = a[0];
                if (q == 0) { bk[buf][warp] = best; br[buf][warp] = r; }
            }
            __syncthreads();
            const unsigned kw = lane < 8 ? bk[buf][lane] : 0u;
            const unsigned wb = __reduce_max_sync(0xffffffffu, kw);
            const int ww = __ffs(__ballot_sync(0xffffffffu, kw == wb)) - 1;
            const T* p = slot[buf][ww];                  // the pivot row's columns of the block
            const bool ok = usable_pivot(p[u]);
            if (r == br[buf][ww]) {
                open = false;
                mine = u;
                if (q == 0) {
                    order[k] = r;
                    if (!ok) atomicOr(status, SLAB_DEV_NOTSPD);
                    rps[buf] = ok ? reciprocal_full(v) : T(1);
                }
            }
            if (t < 4) Us[k * 65 + 4 * kc + t] = (t == u && !ok) ? T(1) : p[t];
            __syncthreads();
            const T l = open ? v * rps[buf] : T(0);
            lm[u] = l;
            if (q == 0) Lm[k * 64 + r] = l;
            if (open && q > u) a[0] -= l * p[q];
        }
        const int left = 60 - 4 * kc;                    // columns right of the block
        if (left == 0) break;
        if (mine >= 0) {
#pragma unroll
            for (int c = 1; c < 16; ++c)
                if (c < 16 - kc) tail[mine][4 * (c - 1) + q] = a[c];
            if (q == 0)
#pragma unroll
                for (int i = 0; i < 4; ++i) mul[mine][i] = lm[i];
        }
        __syncthreads();
        if (t < left) {                                  // U right of the block, one thread a column
            T w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                w[k] = tail[k][t];
#pragma unroll
                for (int i = 0; i < k; ++i) w[k] -= mul[k][i] * w[i];
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                tail[k][t] = w[k];
                Us[(4 * kc + k) * 65 + 4 * kc + 4 + t] = w[k];
            }
        }
        __syncthreads();
        if (open) {
#pragma unroll
            for (int c = 1; c < 16; ++c)
                if (c < 16 - kc)
#pragma unroll
                    for (int i = 0; i < 4; ++i) a[c] -= lm[i] * tail[i][4 * (c - 1) + q];
        }
#pragma unroll
        for (int c = 0; c < 15; ++c) a[c] = a[c + 1];
        a[15] = T(0);
    }
    __syncthreads();
    using Lay = LuLayout<T>;
    for (int e = t; e < 64 * 64; e += 256) {
        int kk, i, pl;
        Lay::at(e, kk, i, pl);
        const bool in = i > kk && i < 64;
        lu[pl] = in ? Lm[kk * 64 + order[i & 63]] : T(0);
        lu[Lay::TRI + pl] = in ? Us[(63 - (i & 63)) * 65 + 63 - kk] : T(0);
    }
    if (t < 64) {
        lu[2 * Lay::TRI + t] = reciprocal_full(Us[t * 65 + t]);
        const int pr = prow[order[t]];
        piv[t] = pr;
        perm[c0 + t] = pr;
    }
}

__device__ __forceinline__ void copy16_async(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// X = U^{-1} L^{-1} G[piv, cb .. cb+NC-1] for the columns right of the panel, written to G[piv, cols] and
// to XT[col - (c0+64)][0..63]; the last block zeroes G[piv, panel], so that the update may multiply
// the panel columns of all rows.  TPC threads a column (LuLayout), thread q holding rows TPC c + q, 128 threads
// a CTA; the solves need only shuffles.
template <typename T>
constexpr int gj_cols() { return 128 / LuLayout<T>::TPC; }
template <typename T>
constexpr size_t gj_apply_smem() { return (LuLayout<T>::ELEMS + 64 * (gj_cols<T>() + 1)) * sizeof(T); }

template <typename T>
__global__ void __launch_bounds__(128) gj_panel_apply_kernel(T* G, int64_t ld, int wt, int c0,
                                                                          const int* __restrict__ piv,
                                                                          const T* __restrict__ lu, T* XT) {
    using Lay = LuLayout<T>;
    constexpr int NC = gj_cols<T>(), NT = 128, YP = NC + 1, TPC = Lay::TPC, C = Lay::C;
    extern __shared__ __align__(16) unsigned char gj_smem[];
    T* Ls = reinterpret_cast<T*>(gj_smem);
    T* Us = Ls + Lay::TRI;
    T* rd = Us + Lay::TRI;
    T* ys = rd + 64;                                     // [64][YP]
    pdl_wait();
    pdl_trigger();
    const int t = threadIdx.x, lane = t & 31;
    if (blockIdx.x == gridDim.x - 1) {
        for (int e = t; e < 64 * 64; e += NT) G[(int64_t)piv[e >> 6] * ld + c0 + (e & 63)] = T(0);
        return;
    }
    const int cb = c0 + 64 + blockIdx.x * NC;            // first column of this block
    const int nc = min(NC, wt - cb);
    for (int e = t; e < (int)(Lay::ELEMS * sizeof(T) / 16); e += NT)
        copy16_async(reinterpret_cast<char*>(Ls) + 16 * e, reinterpret_cast<const char*>(lu) + 16 * e);
#pragma unroll 8
    for (int e = t; e < 64 * NC; e += NT) {
        const int i = e / NC, j = e % NC;
        ys[i * YP + j] = j < nc ? G[(int64_t)piv[i] * ld + cb + j] : T(0);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    const int col = t / TPC, q = t % TPC;
    T x[C];
#pragma unroll
    for (int c = 0; c < C; ++c) x[c] = ys[(TPC * c + q) * YP + col];
#pragma unroll
    for (int pass = 0; pass < 2; ++pass) {               // L forward, then U backward (reversed indices)
        const T* tri = pass ? Us : Ls;
#pragma unroll 1
        for (int kc = 0; kc < C; ++kc) {
#pragma unroll
            for (int u = 0; u < TPC; ++u) {
                const int k = TPC * kc + u;
                T xk = __shfl_sync(0xffffffffu, x[0], (lane & ~(TPC - 1)) | u);
                if (pass) {
                    xk *= rd[63 - k];
                    if (q == u) x[0] = xk;
                }
                const T* m = tri + (k * TPC + q) * Lay::PITCH;
#pragma unroll
                for (int c = 0; c < C; c += 4)
                    if (c < C - kc) {
                        T mv[4];
                        ld4(m + c, mv);
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if (C > 4 || c + i < C - kc) x[c + i] -= mv[i] * xk;
                    }
            }
            ys[(pass ? 63 - (TPC * kc + q) : TPC * kc + q) * YP + col] = x[0];
#pragma unroll
            for (int c = 0; c < C - 1; ++c) x[c] = x[c + 1];
            x[C - 1] = T(0);
        }
        __syncwarp();
        if (!pass)
#pragma unroll
            for (int c = 0; c < C; ++c) x[c] = ys[(63 - (TPC * c + q)) * YP + col];
        __syncwarp();
    }
    __syncthreads();
    for (int e = t; e < 64 * NC; e += NT) {
        const int i = e / NC, j = e % NC;                // row of X, column in block
        if (j < nc) G[(int64_t)piv[i] * ld + cb + j] = ys[i * YP + j];
    }
    for (int e = t; e < 64 * NC; e += NT) {
        const int j = e >> 6, i = e & 63;                // XT row = column, 64 consecutive i
        if (j < nc) XT[(int64_t)(cb - c0 - 64 + j) * 64 + i] = ys[i * YP + j];
    }
}

// Build the augmented system of interface j (leading dimension ld).  S comes from Tb[0] (j = 0) or from
// the bottom right block of the previous elimination (copied before the bottom block is rebuilt).
template <typename T>
__global__ void gj_fill_top_kernel(T* Gt, int64_t ld, int sp, int wt, const T* __restrict__ S, int64_t lds,
                                   const T* __restrict__ T12) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, i = blockIdx.y;
    if (c >= wt) return;
    T v;
    if (c < sp) v = S[(int64_t)i * lds + c];
    else if (T12 && c < 2 * sp) v = T12[(int64_t)i * sp + (c - sp)];
    else v = (c - (wt - sp)) == i ? T(1) : T(0);
    Gt[i * ld + c] = v;
}

// Bottom rows [T_{j+1,j} | T_{j+1,j+1}]: T21 given (nonsymmetric kind), else T_{j,j+1}^T from T12.
template <typename T>
__global__ void gj_fill_bottom_kernel(T* Gb, int64_t ld, int sp, const T* __restrict__ T12, const T* __restrict__ T22,
                                      const T* __restrict__ T21) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, i = blockIdx.y;
    if (c >= 2 * sp) return;
    Gb[i * ld + c] = c < sp ? (T21 ? T21[(int64_t)i * sp + c] : T12[(int64_t)c * sp + i]) : T22[(int64_t)i * sp + (c - sp)];
}

// Sinv[i] = Gt[perm[i]][wt-sp ..], W[i] = Gt[perm[i]][sp .. 2sp) (W optional)
template <typename T>
__global__ void gj_gather_kernel(const T* __restrict__ Gt, int64_t ld, int sp, int wt, const int* perm, T* Sinv, T* W) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, i = blockIdx.y;
    if (c >= sp) return;
    const T* row = Gt + (int64_t)perm[i] * ld;
    Sinv[(int64_t)i * sp + c] = row[wt - sp + c];
    if (W) W[(int64_t)i * sp + c] = row[sp + c];
}

template <typename T>
__global__ void gj_init_rows_kernel(int* act, int* pflag, int sp) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < sp) { act[i] = i; pflag[i] = 0; }
}

// Batched C_b = beta C_b + alpha A_b B_b^T, b < batch, with element strides sA, sB, sC.
template <typename T>
slab_status gemm_tn_batched(slab_handle* h, int cls, int M, int N, int K, T alpha, const T* A, int64_t lda,
                            int64_t sA, const T* B, int64_t ldb, int64_t sB, T beta, T* C, int64_t ldc,
                            int64_t sC, int transC, int lower_only, int batch, int triA = 0);

template <>
slab_status gemm_tn_batched<float>(slab_handle* h, int cls, int M, int N, int K, float alpha, const float* A,
                                   int64_t lda, int64_t sA, const float* B, int64_t ldb, int64_t sB, float beta,
                                   float* C, int64_t ldc, int64_t sC, int transC, int lower_only, int batch, int triA) {
    // a factor product whose operand splits do not fit the FP16 work buffer runs on slices of the
    // batch that do, rather than falling back to the slower 3xTF32 product
    if (batch > 1 && h->w16 && !h->tf32_now && K % 64 == 0 &&
        (cls == KC_SYRK || cls == KC_TRAIL || cls == KC_ASSEMBLE)) {
        const bool shared = A == B && lda == ldb && sA == sB && N <= M;
        if (f16x3_work_bytes(M, N, K, batch, shared) > h->w16_bytes) {
            int bc = batch;
            while (bc > 1 && f16x3_work_bytes(M, N, K, bc, shared) > h->w16_bytes) bc = (bc + 1) / 2;
            if (f16x3_work_bytes(M, N, K, bc, shared) <= h->w16_bytes) {
                for (int b0 = 0; b0 < batch; b0 += bc) {
                    const int nb = std::min(bc, batch - b0);
                    const slab_status st = gemm_tn_batched<float>(h, cls, M, N, K, alpha, A + b0 * sA, lda, sA,
                                                                  B + b0 * sB, ldb, sB, beta, C + b0 * sC, ldc, sC,
                                                                  transC, lower_only, nb, triA);
                    if (st) return st;
                }
                return SLAB_OK;
            }
        }
    }
    SLAB_PROF(h, cls);
    if (use_solve_product(cls, N, K, A, lda, sA, B, ldb, sB, lower_only))
        return solve_product(h, M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, transC, triA, batch);
    TcGemmArgs g;
    g.M = M; g.N = N; g.K = K; g.alpha = alpha; g.beta = beta;
    g.A = A; g.lda = lda; g.B = B; g.ldb = ldb; g.C = C; g.ldc = ldc;
    g.transC = transC; g.split = h->tf32_now ? 0 : 1; g.lower_only = lower_only;
    g.batch = batch; g.sA = sA; g.sB = sB; g.sC = sC;
    g.ksplit = 1; g.part = nullptr;
    g.w16 = nullptr; g.w16_bytes = 0;
    g.triA = triA;
    if (use_f16x3(h, cls, g)) {
        // FP16 three-product path (factor products)
    } else if (N <= 64 && !lower_only && h->wPart) {     // skinny batches that leave SMs idle: split K as well
        const int64_t tiles = (int64_t)((M + 127) / 128) * ((N + 63) / 64) * batch;
        const int64_t cap = (int64_t)splitk_part_bytes(h->td.s_pad) / sizeof(float);
        int ks = 1;
        while (2 * ks <= SLAB_SPLITK && tiles * ks < 148 && K % (2 * ks * 32) == 0 &&
               (int64_t)2 * ks * batch * M * N <= cap)
            ks *= 2;
        g.ksplit = ks;
        g.part = (float*)h->wPart;
    }
    const slab_status st = tc_gemm(h->stream, g, h->dstatus);
    if (st == SLAB_ECUDA && h->err == SLAB_OK) h->err = SLAB_ECUDA;
    prof_extra(h, cls, tc_gemm_extra_launches(g));
    return st;
}

template <>
slab_status gemm_tn_batched<double>(slab_handle* h, int cls, int M, int N, int K, double alpha, const double* A,
                                    int64_t lda, int64_t sA, const double* B, int64_t ldb, int64_t sB,
                                    double beta, double* C, int64_t ldc, int64_t sC, int transC, int lower_only,
                                    int batch, int /*triA*/) {
    SLAB_PROF(h, cls);
    return launch_fp64_product(h, M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, transC, lower_only, batch, M, 0);
}

}  // namespace

// Indefinite kind: Algorithm 1 as printed, S_1 = T_11, S_{j+1} = T_{j+1,j+1} - T_{j+1,j} W_j with
// W_j = S_j^{-1} T_{j,j+1}, all three from one blocked Gauss-Jordan elimination of the augmented
// system (see above).  Stored: S_j^{-1} (in Linv), W_j (in Y) and T_{j+1,j} (in ToT).
// Work: G in Fct; XT, the LU of A11 and the pivot bookkeeping in gjw.
template <typename T>
slab_status sweep_factor_indef(slab_handle* h) {
    const int NI = h->td.NI, sp = h->td.s_pad, nt = h->nt;
    const int64_t blk = (int64_t)sp * sp;
    T* Tb = (T*)h->Tb;
    T* To = (T*)h->To;
    T* ToT = (T*)h->ToT;
    T* Tl = (T*)h->Tl;                   // nonsymmetric kind: T_{q+1,q} as assembled (else null)
    T* Sinv = (T*)h->Linv;
    T* Wn = (T*)h->Y;
    const int64_t ld = 3 * (int64_t)sp;
    T* Gt = (T*)h->Fct;                  // rows 0 .. sp-1 of G
    T* Gb = Gt + sp * ld;                // rows sp .. 2 sp-1
    char* wb = (char*)h->gjw;
    T* XT = (T*)wb;                      wb += (size_t)3 * sp * 64 * sizeof(T);
    T* lu = (T*)wb;                      wb += (size_t)LuLayout<T>::ELEMS * sizeof(T);
    GjWork w;
    int* act0 = (int*)wb;                wb += (size_t)2 * sp * sizeof(int);
    w.act = act0;
    w.perm = (int*)wb;                   wb += (size_t)sp * sizeof(int);
    w.pflag = (int*)wb;                  wb += (size_t)sp * sizeof(int);
    const int nodes = gj_nodes((sp + GJ_LEAF - 1) / GJ_LEAF);
    w.cand = (int*)wb;                   wb += (size_t)nodes * 64 * sizeof(int);
    w.tick = (unsigned*)wb;              wb += (size_t)nodes * sizeof(unsigned);
    w.piv = (int*)wb;
    const bool f32 = sizeof(T) == 4;     // the tournament delivers A11's LU
    auto tsmem = [&](int rows) { return f32 ? (size_t)(64 * rows + 64 * 65) * sizeof(float) : (size_t)0; };
    const size_t ismem = (size_t)(64 * 64 + 64 * 65) * sizeof(T);
    const size_t asmem = gj_apply_smem<T>();
    SLAB_CK(h, cudaFuncSetAttribute(gj_tournament_kernel<T, GJ_LEAF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)tsmem(GJ_LEAF)));
    SLAB_CK(h, cudaFuncSetAttribute(gj_tournament_kernel<T, GJ_ONE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)tsmem(GJ_ONE)));
    SLAB_CK(h, cudaFuncSetAttribute(gj_a11_lu_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)ismem));
    SLAB_CK(h, cudaFuncSetAttribute(gj_panel_apply_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)asmem));
    SLAB_CK(h, cudaMemsetAsync(w.tick, 0, (size_t)nodes * sizeof(unsigned), h->stream));
    slab_status st;
    for (int j = 0; j < NI; ++j) {
        const bool hasNext = j < NI - 1;
        const int wt = (hasNext ? 3 : 2) * sp;
        {
            SLAB_PROF(h, KC_OTHER);
            gj_fill_top_kernel<T><<<dim3((wt + 255) / 256, sp), 256, 0, h->stream>>>(
                Gt, ld, sp, wt, j == 0 ? Tb : Gb + sp, j == 0 ? (int64_t)sp : ld, hasNext ? To + j * blk : nullptr);
            SLAB_CK_LAUNCH(h);
            if (hasNext) {
                gj_fill_bottom_kernel<T><<<dim3((2 * sp + 255) / 256, sp), 256, 0, h->stream>>>(
                    Gb, ld, sp, To + j * blk, Tb + (j + 1) * blk, Tl ? Tl + j * blk : nullptr);
                SLAB_CK_LAUNCH(h);
            }
            gj_init_rows_kernel<T><<<(sp + 255) / 256, 256, 0, h->stream>>>(act0, w.pflag, sp);
            SLAB_CK_LAUNCH(h);
        }
        for (int kb = 0; kb < nt; ++kb) {
            const int c0 = kb * 64;
            const int nact = sp - c0;
            const int* act = act0 + (kb & 1) * sp;
            int* act_next = act0 + ((kb + 1) & 1) * sp;
            const int L = (nact + GJ_LEAF - 1) / GJ_LEAF;
            {
                SLAB_PROF(h, KC_PANEL);
                if (h->pivot_local)
                    SLAB_CK(h, launch_pdl(gj_local_rows_kernel, dim3(1), dim3(256), 0, h->stream, kb, nact, w, act,
                                          act_next));
                else if (nact > GJ_LEAF && nact <= GJ_ONE)
                    SLAB_CK(h, launch_pdl(gj_tournament_kernel<T, GJ_ONE>, dim3(1), dim3(GJ_ONE), tsmem(GJ_ONE), h->stream,
                                          (const T*)Gt, ld, c0, kb, nact, w, act, act_next, f32 ? (float*)lu : nullptr,
                                          h->dstatus));
                else
                    SLAB_CK(h, launch_pdl(gj_tournament_kernel<T, GJ_LEAF>, dim3(L), dim3(GJ_LEAF), tsmem(GJ_LEAF),
                                          h->stream, (const T*)Gt, ld, c0, kb, nact, w, act, act_next,
                                          f32 ? (float*)lu : nullptr, h->dstatus));
                if (h->pivot_local || !f32)
                    SLAB_CK(h, launch_pdl(gj_a11_lu_kernel<T>, dim3(1), dim3(256), ismem, h->stream, (const T*)Gt, ld, c0,
                                          w.piv, w.perm, lu, h->dstatus));
                const int ncol = wt - c0 - 64;
                SLAB_CK(h, launch_pdl(gj_panel_apply_kernel<T>, dim3((ncol + gj_cols<T>() - 1) / gj_cols<T>() + 1),
                                      dim3(128), asmem, h->stream, Gt, ld, wt, c0, (const int*)w.piv,
                                      (const T*)lu, XT));
                prof_extra(h, KC_PANEL, h->pivot_local || !f32 ? 2 : 1);
            }
            // G[all, rest] -= G[all, panel] X : top rows over all remaining columns, bottom rows up to 2 sp
            if ((st = gemm_tn<T>(h, KC_TRAIL, hasNext ? 2 * sp : sp, wt - c0 - 64, 64, T(-1), Gt + c0, ld, XT, 64, T(1),
                                 Gt + c0 + 64, ld, 0, 0, 0, sp, 2 * sp - c0 - 64)))
                return st;
            if (slab_debug()) {
                if (slab_debug_status(h, "interface elimination (interface, panel)", j, kb)) return SLAB_ESINGULAR;
                // pivot bookkeeping: distinct pivot rows drawn from the active list, act_next = act - piv
                std::vector<int> hp(64), ha(nact), hn(nact > 64 ? nact - 64 : 1);
                cudaMemcpy(hp.data(), w.piv, 64 * sizeof(int), cudaMemcpyDeviceToHost);
                cudaMemcpy(ha.data(), act, nact * sizeof(int), cudaMemcpyDeviceToHost);
                if (nact > 64) cudaMemcpy(hn.data(), act_next, (nact - 64) * sizeof(int), cudaMemcpyDeviceToHost);
                std::vector<char> inA(sp, 0), inP(sp, 0);
                bool bad = false;
                for (int r : ha) inA[r] = 1;
                for (int r : hp) { if (r < 0 || r >= sp || !inA[r] || inP[r]) bad = true; else inP[r] = 1; }
                size_t q = 0;
                for (int r : ha) if (!inP[r]) { if (q >= hn.size() || hn[q] != r) bad = true; ++q; }
                if (bad) {
                    std::fprintf(stderr, "slab: pivot bookkeeping inconsistent at (%d, %d)\n", j, kb);
                    return SLAB_ESINGULAR;
                }
            }
        }
        {
            SLAB_PROF(h, KC_OTHER);
            gj_gather_kernel<T><<<dim3((sp + 255) / 256, sp), 256, 0, h->stream>>>(Gt, ld, sp, wt, w.perm, Sinv + j * blk,
                                                                                   hasNext ? Wn + j * blk : nullptr);
            SLAB_CK_LAUNCH(h);
        }
        if (!Tl && hasNext && (st = transpose<T>(h, To + j * blk, ToT + j * blk, sp))) return st;   // T_{j+1,j}
        if (h->kind == SLAB_CONVECTION) {                 // factors of the transposed sweep (A^T solves; Tl is null for one interface)
            if ((st = transpose<T>(h, Sinv + j * blk, (T*)h->SinvT + j * blk, sp))) return st;
            if (hasNext && (st = transpose<T>(h, Wn + j * blk, (T*)h->WT + j * blk, sp))) return st;
            if (hasNext && (st = transpose<T>(h, Tl + j * blk, (T*)h->TlT + j * blk, sp))) return st;
        }
    }
    return SLAB_OK;
}

template <typename S, typename D>
__global__ void convert_kernel(const S* __restrict__ src, D* __restrict__ dst, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = (D)src[i];
}

slab_status widen_to_double(slab_handle* h, const float* src, double* dst, int64_t n) {
    if (n <= 0) return SLAB_OK;
    SLAB_PROF(h, KC_OTHER);
    convert_kernel<float, double><<<(unsigned)std::min<int64_t>((n + 255) / 256, SMS * 16), 256, 0, h->stream>>>(
        src, dst, n);
    SLAB_CK_LAUNCH(h);
    return SLAB_OK;
}

slab_status narrow_to_float(slab_handle* h, const double* src, float* dst, int64_t n) {
    if (n <= 0) return SLAB_OK;
    SLAB_PROF(h, KC_OTHER);
    convert_kernel<double, float><<<(unsigned)std::min<int64_t>((n + 255) / 256, SMS * 16), 256, 0, h->stream>>>(
        src, dst, n);
    SLAB_CK_LAUNCH(h);
    return SLAB_OK;
}

// Bytes of the indefinite-kind Stage-2 work area (gjw).
size_t gj_work_bytes(int sp, size_t rsz) {
    const int nodes = gj_nodes((sp + GJ_LEAF - 1) / GJ_LEAF);
    return ((size_t)3 * sp * 64 + std::max(LuLayout<float>::ELEMS, LuLayout<double>::ELEMS)) * rsz + (size_t)4 * sp * sizeof(int) +
           (size_t)nodes * 64 * sizeof(int) + (size_t)nodes * sizeof(unsigned) + 64 * sizeof(int) + 256;
}

// Algorithm 2 for the indefinite kind on X ([NI][kcap][s_pad]):
//   forward  z_j = S_j^{-1} f_j,  f_{j+1} -= T_{j+1,j} z_j;   backward  u_j = z_j - W_j u_{j+1}.
template <typename T>
slab_status sweep_solve_indef(slab_handle* h, int K) {
    const int NI = h->td.NI, sp = h->td.s_pad;
    const int64_t blk = (int64_t)sp * sp;
    const int64_t vb = (int64_t)sp * h->kcap;
    T* Sinv = (T*)h->Linv;
    T* Wn = (T*)h->Y;
    T* ToT = h->Tl ? (T*)h->Tl : (T*)h->ToT;     // T_{j+1,j}
    T* X = (T*)h->wX;
    T* Z = (T*)h->wZ;
    slab_status st;
    for (int j = 0; j < NI; ++j) {
        if ((st = gemm_tn<T>(h, KC_SOLVE_PROD, sp, K, sp, T(1), Sinv + j * blk, sp, X + j * vb, sp, T(0), Z + j * vb,
                             sp, 1, 0)))
            return st;
        if (j < NI - 1 && (st = gemm_tn<T>(h, KC_SOLVE_PROD, sp, K, sp, T(-1), ToT + j * blk, sp, Z + j * vb, sp,
                                           T(1), X + (j + 1) * vb, sp, 1, 0)))
            return st;
    }
    for (int j = NI - 1; j >= 0; --j) {
        SLAB_CK(h, cudaMemcpyAsync(X + j * vb, Z + j * vb, (size_t)K * sp * sizeof(T), cudaMemcpyDeviceToDevice,
                                   h->stream));
        if (j < NI - 1 && (st = gemm_tn<T>(h, KC_SOLVE_PROD, sp, K, sp, T(-1), Wn + j * blk, sp, X + (j + 1) * vb, sp,
                                           T(1), X + j * vb, sp, 1, 0)))
            return st;
    }
    return SLAB_OK;
}

// Algorithm 2 for T^T (the adjoint of the nonsymmetric kind) with the factors of T = L U, L block
// lower bidiagonal (S_j, T_{j+1,j}), U unit block upper bidiagonal (W_j): T^T = U^T L^T, so
//   forward  y_j = f_j - W_{j-1}^T y_{j-1};   backward  x_j = S_j^{-T} (y_j - T_{j+1,j}^T x_{j+1}),
// on X ([NI][kcap][s_pad]), result in X.
template <typename T>
slab_status sweep_solve_indef_transposed(slab_handle* h, int K) {
    const int NI = h->td.NI, sp = h->td.s_pad;
    const int64_t blk = (int64_t)sp * sp;
    const int64_t vb = (int64_t)sp * h->kcap;
    T* SinvT = (T*)h->SinvT;
    T* WT = (T*)h->WT;
    T* TlT = (T*)h->TlT;
    T* X = (T*)h->wX;
    T* Z = (T*)h->wZ;
    slab_status st;
    for (int j = 1; j < NI; ++j)
        if ((st = gemm_tn<T>(h, KC_SOLVE_PROD, sp, K, sp, T(-1), WT + (j - 1) * blk, sp, X + (j - 1) * vb, sp, T(1),
                             X + j * vb, sp, 1, 0)))
            return st;
    for (int j = NI - 1; j >= 0; --j) {
        if (j < NI - 1 && (st = gemm_tn<T>(h, KC_SOLVE_PROD, sp, K, sp, T(-1), TlT + j * blk, sp, Z + (j + 1) * vb, sp,
                                           T(1), X + j * vb, sp, 1, 0)))
            return st;
        if ((st = gemm_tn<T>(h, KC_SOLVE_PROD, sp, K, sp, T(1), SinvT + j * blk, sp, X + j * vb, sp, T(0), Z + j * vb,
                             sp, 1, 0)))
            return st;
    }
    for (int j = 0; j < NI; ++j)
        SLAB_CK(h, cudaMemcpyAsync(X + j * vb, Z + j * vb, (size_t)K * sp * sizeof(T), cudaMemcpyDeviceToDevice,
                                   h->stream));
    return SLAB_OK;
}

// Factor-phase layout: Fct[j] = [S_j ; Y_j^T ; L_j^{-T}] (3 s_pad x s_pad; for the last j the
// L^{-T} block sits right below S), plus the transposed copies Lin[j] = L_j^{-1} and Yn[j] = Y_j
// for the solve products.
template <typename T>
slab_status sweep_factor(slab_handle* h) {
    if (h->kind == SLAB_HELMHOLTZ || h->kind == SLAB_CONVECTION) return sweep_factor_indef<T>(h);
    if (h->stage2) return cr_factor<T>(h);
    const int NI = h->td.NI, sp = h->td.s_pad;
    const int64_t blk = (int64_t)sp * sp;
    T* Tb = (T*)h->Tb;
    T* To = (T*)h->To;
    T* F = (T*)h->Fct;
    T* Lin = (T*)h->Linv;
    T* Yn = (T*)h->Y;
    slab_status st;
    for (int j = 0; j < NI; ++j) {
        T* W = F + j * 3 * blk;
        const int hasY = j < NI - 1;
        T* S = W;
        T* Yt = W + blk;
        T* LT = W + (hasY ? 2 : 1) * blk;
        if ((st = tall_fill<T>(h, Tb + j * blk, 0, W, 0, LT - W, sp, 1))) return st;
        if (j > 0) {           // S_j = T_jj - Y_{j-1}^T Y_{j-1}  (lower tiles)
            const T* Yp = F + (j - 1) * 3 * blk + blk;
            if ((st = gemm_tn<T>(h, KC_SYRK, sp, sp, sp, T(-1), Yp, sp, Yp, sp, T(1), S, sp, 0, 1))) return st;
        }
        if (hasY && (st = transpose<T>(h, To + j * blk, Yt, sp))) return st;      // T_{j+1,j}
        const int lt0 = (hasY ? 2 : 1) * sp;         // first row of the identity block
        if ((st = dense_tall_cholesky<T>(h, W, sp, lt0, 1, 0))) return st;
        if ((st = transpose<T>(h, LT, Lin + j * blk, sp))) return st;
        if (hasY && (st = transpose<T>(h, Yt, Yn + j * blk, sp))) return st;
    }
    return SLAB_OK;
}

// Algorithm 2 on the interface workspace X ([NI][kcap][s_pad], right-hand sides 0..K-1), result in X.
template <typename T>
slab_status sweep_solve(slab_handle* h, int K) {
    if (h->kind == SLAB_CONVECTION && h->transposed) return sweep_solve_indef_transposed<T>(h, K);
    if (h->kind == SLAB_HELMHOLTZ || h->kind == SLAB_CONVECTION) return sweep_solve_indef<T>(h, K);
    if (h->stage2) return cr_solve<T>(h, K);
    const int NI = h->td.NI, sp = h->td.s_pad;
    const int64_t blk = (int64_t)sp * sp;
    const int64_t vb = (int64_t)sp * h->kcap;
    T* F = (T*)h->Fct;
    T* Lin = (T*)h->Linv;
    T* Yn = (T*)h->Y;
    T* X = (T*)h->wX;
    T* Z = (T*)h->wZ;
    slab_status st;
    for (int j = 0; j < NI; ++j) {        // forward: z_j = L_j^{-1} (f_j - Y_{j-1}^T z_{j-1})
        if (j > 0) {
            const T* Yt = F + (j - 1) * 3 * blk + blk;
            if ((st = gemm_tn<T>(h, KC_SOLVE_PROD, sp, K, sp, T(-1), Yt, sp, Z + (j - 1) * vb, sp, T(1), X + j * vb, sp, 1, 0)))
                return st;
        }
        if ((st = gemm_tn<T>(h, KC_SOLVE_PROD, sp, K, sp, T(1), Lin + j * blk, sp, X + j * vb, sp, T(0), Z + j * vb, sp, 1, 0,
                             1)))                 // L^{-1} is lower triangular
            return st;
    }
    for (int j = NI - 1; j >= 0; --j) {   // backward: u_j = L_j^{-T} (z_j - Y_j u_{j+1})
        if (j < NI - 1) {
            if ((st = gemm_tn<T>(h, KC_SOLVE_PROD, sp, K, sp, T(-1), Yn + j * blk, sp, X + (j + 1) * vb, sp, T(1), Z + j * vb, sp,
                                 1, 0)))
                return st;
        }
        const T* LT = F + j * 3 * blk + (j < NI - 1 ? 2 : 1) * blk;
        if ((st = gemm_tn<T>(h, KC_SOLVE_PROD, sp, K, sp, T(1), LT, sp, Z + j * vb, sp, T(0), X + j * vb, sp, 1, 0,
                             2)))                 // L^{-T} is upper triangular
            return st;
    }
    return SLAB_OK;
}

// ------------------------------------------------------------------ odd-even elimination order
// The odd-even order for eliminating the blocks of T (Sec. 4, remark on the elimination order;
// conclusion).  Each level eliminates the blocks at odd positions among the remaining ones; the
// remaining blocks of level l are the multiples of 2^l, so the eliminated ones o = 2^l (2i+1) and
// their neighbours a = o - 2^l, c = o + 2^l (absent past the last block) are uniformly strided,
// and every step of a level is one batched launch.  With D the current diagonal blocks and
// E_i the current block coupling i to its right remaining neighbour:
//   L_o L_o^T = D_o,  P_o = L_o^{-1} E_a^T,  Q_o = L_o^{-1} E_o,
//   D_a -= P_o^T P_o,  D_c -= Q_o^T Q_o,  E_a <- -P_o^T Q_o.
// Stored per eliminated block: L^{-1} (Linv), L^{-T}, P^T, P, Q^T, Q.  Solve: forward
// y_o = L_o^{-1} b_o, b_a -= P_o^T y_o, b_c -= Q_o^T y_o level by level; the last block
// x = L^{-T} L^{-1} b; backward x_o = L_o^{-T} (y_o - P_o x_a - Q_o x_c).
struct CrLevel {
    int o0, step, nb, nc;     // first eliminated block, its neighbour distance, #eliminated, #with a c
};

static std::vector<CrLevel> cr_levels(int NI, int* last) {
    std::vector<CrLevel> L;
    int step = 1;
    while (step < NI) {                          // remaining: 0, step, 2 step, ... < NI
        const int nrem = (NI - 1) / step + 1;
        if (nrem < 2) break;
        CrLevel lv;
        lv.o0 = step;
        lv.step = step;
        lv.nb = nrem / 2;                        // positions 1, 3, 5, ... < nrem
        lv.nc = (nrem - 1) / 2;                  // those with position + 1 < nrem
        L.push_back(lv);
        step *= 2;
    }
    *last = 0;
    return L;
}

int cr_max_batch(int NI) {
    int last = 0;
    std::vector<CrLevel> L = cr_levels(NI, &last);
    int b = 1;
    for (auto& lv : L) b = std::max(b, lv.nb);
    return b;
}

// Cholesky with L^{-1} and L^{-T} of nb blocks D[o0 + i st] as one batch of tall eliminations
// [D ; I] in the work buffer (2 s_pad x s_pad per block).
template <typename T>
static slab_status cr_potrf_batch(slab_handle* h, int o0, int st_blk, int nb) {
    const int sp = h->td.s_pad;
    const int64_t blk = (int64_t)sp * sp;
    T* D = (T*)h->crD;
    T* W = (T*)h->crW;
    T* LT = (T*)h->crLT;
    T* Lin = (T*)h->Linv;
    const int64_t sb = (int64_t)st_blk * blk;
    slab_status st;
    if ((st = tall_fill<T>(h, D + o0 * blk, sb, W, 2 * blk, blk, sp, nb))) return st;
    if ((st = dense_tall_cholesky<T>(h, W, sp, sp, nb, 2 * blk))) return st;
    return transpose_batched<T>(h, W + blk, 2 * blk, Lin + o0 * blk, sb, sp, nb, LT + o0 * blk);
}

template <typename T>
slab_status cr_factor(slab_handle* h) {
    const int NI = h->td.NI, sp = h->td.s_pad;
    const int64_t blk = (int64_t)sp * sp;
    T* D = (T*)h->crD;
    T* E = (T*)h->crE;
    T* Et = (T*)h->crW;                  // free between the batched Cholesky steps
    T* Lin = (T*)h->Linv;
    T* Pt = (T*)h->crPt;
    T* P = (T*)h->crP;
    T* Qt = (T*)h->crQt;
    T* Q = (T*)h->crQ;
    SLAB_CK(h, cudaMemcpyAsync(D, h->Tb, NI * blk * sizeof(T), cudaMemcpyDeviceToDevice, h->stream));
    if (NI > 1)
        SLAB_CK(h, cudaMemcpyAsync(E, h->To, (NI - 1) * blk * sizeof(T), cudaMemcpyDeviceToDevice, h->stream));
    int last = 0;
    const std::vector<CrLevel> levels = cr_levels(NI, &last);
    slab_status st;
    for (const CrLevel& lv : levels) {
        const int o0 = lv.o0, a0 = lv.o0 - lv.step, c0 = lv.o0 + lv.step, nb = lv.nb, nc = lv.nc;
        const int64_t sb = 2 * (int64_t)lv.step * blk;           // stride between consecutive o (and a, c)
        if ((st = cr_potrf_batch<T>(h, o0, 2 * lv.step, nb))) return st;
        // P_o^T = E_a L_o^{-T};  Q_o^T = E_o^T L_o^{-T}
        if ((st = gemm_tn_batched<T>(h, KC_SYRK, sp, sp, sp, T(1), E + a0 * blk, sp, sb, Lin + o0 * blk, sp, sb, T(0),
                                     Pt + o0 * blk, sp, sb, 0, 0, nb)))
            return st;
        if (nc > 0) {
            if ((st = transpose_batched<T>(h, E + o0 * blk, sb, Et, blk, sp, nc))) return st;
            if ((st = gemm_tn_batched<T>(h, KC_SYRK, sp, sp, sp, T(1), Et, sp, blk, Lin + o0 * blk, sp, sb, T(0),
                                         Qt + o0 * blk, sp, sb, 0, 0, nc)))
                return st;
        }
        // D_a -= P_o^T P_o (lower tiles)
        if ((st = gemm_tn_batched<T>(h, KC_SYRK, sp, sp, sp, T(-1), Pt + o0 * blk, sp, sb, Pt + o0 * blk, sp, sb, T(1),
                                     D + a0 * blk, sp, sb, 0, 1, nb)))
            return st;
        if (nc > 0) {
            // D_c -= Q_o^T Q_o (lower tiles);  E_a = -P_o^T Q_o
            if ((st = gemm_tn_batched<T>(h, KC_SYRK, sp, sp, sp, T(-1), Qt + o0 * blk, sp, sb, Qt + o0 * blk, sp, sb,
                                         T(1), D + c0 * blk, sp, sb, 0, 1, nc)))
                return st;
            if ((st = gemm_tn_batched<T>(h, KC_SYRK, sp, sp, sp, T(-1), Pt + o0 * blk, sp, sb, Qt + o0 * blk, sp, sb,
                                         T(0), E + a0 * blk, sp, sb, 0, 0, nc)))
                return st;
            if ((st = transpose_batched<T>(h, Qt + o0 * blk, sb, Q + o0 * blk, sb, sp, nc))) return st;
        }
        if ((st = transpose_batched<T>(h, Pt + o0 * blk, sb, P + o0 * blk, sb, sp, nb))) return st;
    }
    return cr_potrf_batch<T>(h, last, 1, 1);
}

// The two products of a step of the odd-even solve in one launch, where the streaming kernels take them: block
// w0 + i s2 of OUT gains -(M1_i v1_i + M2_i v2_i).  Returns false where they do not.
static bool cr_pair(slab_handle* h, int K, const ProdTerms& P, float* out, int s2, int batch, slab_status* st) {
    const int sp = h->td.s_pad;
    const int64_t blk = (int64_t)sp * sp, vb = (int64_t)sp * h->kcap;
    if (batch > 65535) return false;
    for (int q = 0; q < 2; ++q)
        if (!use_solve_product(KC_SOLVE_PROD, K, sp, P.A[q], sp, s2 * blk, P.B[q], sp, s2 * vb, 0)) return false;
    SLAB_PROF(h, KC_SOLVE_PROD);
    *st = solve_product_pair(h, sp, K, sp, -1.f, P, sp, s2 * blk, sp, s2 * vb, 1.f, out, sp, s2 * vb, 1, batch);
    return true;
}

template <typename T>
slab_status cr_solve(slab_handle* h, int K) {
    const int NI = h->td.NI, sp = h->td.s_pad;
    const int64_t blk = (int64_t)sp * sp;
    const int64_t vb = (int64_t)sp * h->kcap;
    T* Lin = (T*)h->Linv;
    T* LT = (T*)h->crLT;
    T* Pt = (T*)h->crPt;
    T* P = (T*)h->crP;
    T* Qt = (T*)h->crQt;
    T* Q = (T*)h->crQ;
    T* X = (T*)h->wX;
    T* Z = (T*)h->wZ;
    int last = 0;
    const std::vector<CrLevel> levels = cr_levels(NI, &last);
    slab_status st;
    // out_i (K x sp, RHS-major) = beta out_i + alpha M_i v_i for the nbat strided blocks i;
    // a single product takes the split-K path; L^{-1} (lower) and L^{-T} (upper) are triangular
#define TRI(Mx) ((Mx) == Lin ? 1 : ((Mx) == LT ? 2 : 0))
#define PROD(Mx, m0, V, v0, OUT, w0, alpha_, beta_, nbat, sm, sv)                                                   \
    if ((st = (nbat) == 1                                                                                          \
                  ? gemm_tn<T>(h, KC_SOLVE_PROD, sp, K, sp, T(alpha_), Mx + (m0) * blk, sp, V + (v0) * vb, sp,      \
                               T(beta_), OUT + (w0) * vb, sp, 1, 0, TRI(Mx))                                      \
                  : gemm_tn_batched<T>(h, KC_SOLVE_PROD, sp, K, sp, T(alpha_), Mx + (m0) * blk, sp, (sm) * blk,    \
                                       V + (v0) * vb, sp, (sv) * vb, T(beta_), OUT + (w0) * vb, sp, (sv) * vb, 1, \
                                       0, (nbat), TRI(Mx))))                                                       \
    return st
    for (const CrLevel& lv : levels) {
        const int o0 = lv.o0, a0 = lv.o0 - lv.step, c0 = lv.o0 + lv.step, s2 = 2 * lv.step;
        PROD(Lin, o0, X, o0, Z, o0, 1, 0, lv.nb, s2, s2);
        if constexpr (sizeof(T) == 4) {
            // remaining block a0 + i s2: P^T y of its right neighbour o_i (i < nb), Q^T y of its left one o_{i-1}
            if (lv.nc > 0) {
                const ProdTerms P2 = {{Pt + o0 * blk, Qt + (o0 - s2) * blk}, {Z + o0 * vb, Z + (o0 - s2) * vb}, {0, 1},
                                      {lv.nb, lv.nc + 1}};
                if (cr_pair(h, K, P2, X + a0 * vb, s2, std::max(lv.nb, lv.nc + 1), &st)) {
                    if (st) return st;
                    continue;
                }
            }
        }
        PROD(Pt, o0, Z, o0, X, a0, -1, 1, lv.nb, s2, s2);
        if (lv.nc > 0) PROD(Qt, o0, Z, o0, X, c0, -1, 1, lv.nc, s2, s2);
    }
    PROD(Lin, last, X, last, Z, last, 1, 0, 1, 1, 1);
    PROD(LT, last, Z, last, X, last, 1, 0, 1, 1, 1);
    for (size_t l = levels.size(); l-- > 0;) {
        const CrLevel& lv = levels[l];
        const int o0 = lv.o0, a0 = lv.o0 - lv.step, c0 = lv.o0 + lv.step, s2 = 2 * lv.step;
        bool paired = false;
        if constexpr (sizeof(T) == 4) {
            if (lv.nc > 0) {
                const ProdTerms P2 = {{P + o0 * blk, Q + o0 * blk}, {X + a0 * vb, X + c0 * vb}, {0, 0}, {lv.nb, lv.nc}};
                paired = cr_pair(h, K, P2, Z + o0 * vb, s2, lv.nb, &st);
                if (paired && st) return st;
            }
        }
        if (!paired) {
            PROD(P, o0, X, a0, Z, o0, -1, 1, lv.nb, s2, s2);
            if (lv.nc > 0) PROD(Q, o0, X, c0, Z, o0, -1, 1, lv.nc, s2, s2);
        }
        PROD(LT, o0, Z, o0, X, o0, 1, 0, lv.nb, s2, s2);
    }
#undef PROD
#undef TRI
    return SLAB_OK;
}

template slab_status sweep_factor<float>(slab_handle*);
template slab_status sweep_factor<double>(slab_handle*);
template slab_status sweep_solve<float>(slab_handle*, int);
template slab_status sweep_solve<double>(slab_handle*, int);
template slab_status cr_factor<float>(slab_handle*);
template slab_status cr_factor<double>(slab_handle*);
template slab_status cr_solve<float>(slab_handle*, int);
template slab_status cr_solve<double>(slab_handle*, int);

// ---------------------------------------------------------------- exported dense helpers
namespace {
// out[c][r] = in[r][c] for a rows x cols block (leading dimensions ldin, ldout), batched by blockIdx.z
template <typename T>
__global__ void __launch_bounds__(256) transpose_rect_kernel(const T* __restrict__ in, int64_t ldin, int64_t sin,
                                                             T* __restrict__ out, int64_t ldout, int64_t sout,
                                                             int rows, int cols) {
    transpose_tile64<T>(in + (int64_t)blockIdx.z * sin, ldin, out + (int64_t)blockIdx.z * sout, ldout, rows, cols);
}

template <typename T>
__global__ void copy_batched_kernel(const T* __restrict__ in, int64_t sin, T* __restrict__ out, int64_t sout,
                                    int64_t n) {
    in += (int64_t)blockIdx.y * sin;
    out += (int64_t)blockIdx.y * sout;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) out[i] = in[i];
}

// The same copy in 16-byte units (both blocks 16-byte aligned, strides and length multiples of 16
// bytes), four loads in flight per thread before their stores.
__global__ void copy16_batched_kernel(const uint4* __restrict__ in, int64_t sin, uint4* __restrict__ out, int64_t sout,
                                      int64_t n) {
    in += (int64_t)blockIdx.y * sin;
    out += (int64_t)blockIdx.y * sout;
    const int64_t stride = (int64_t)gridDim.x * 256;
    int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    for (; i + 3 * stride < n; i += 4 * stride) {
        uint4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = in[i + u * stride];
#pragma unroll
        for (int u = 0; u < 4; ++u) out[i + u * stride] = v[u];
    }
    for (; i < n; i += stride) out[i] = in[i];
}
}  // namespace

// Panel workspace (one 64 x 64 inverse per matrix of a batch); grown on demand during the factor.
// The factor allocates the panel inverses for its largest batch up front (factor_create); a
// larger request (direct use of the tall Cholesky) grows them.
static slab_status ensure_panel_work(slab_handle* h, size_t bytes) {
    if (h->pnl_bytes >= bytes) return SLAB_OK;
    slab_dfree(h, h->pnl);                             // in stream order, after the work that may still read it
    h->pnl = nullptr;
    h->pnl_bytes = 0;
    const slab_status st = slab_dalloc(h, &h->pnl, bytes);
    if (st) return st;
    h->pnl_bytes = bytes;
    return SLAB_OK;
}

template <typename T>
slab_status dense_gemm(slab_handle* h, int cls, int M, int N, int K, T alpha, const T* A, int64_t lda, int64_t sA,
                       const T* B, int64_t ldb, int64_t sB, T beta, T* C, int64_t ldc, int64_t sC, int transC,
                       int lower_only, int batch, int triA) {
    if (batch <= 0 || M <= 0 || N <= 0) return SLAB_OK;
    if (batch == 1) return gemm_tn<T>(h, cls, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, transC, lower_only, triA);
    return gemm_tn_batched<T>(h, cls, M, N, K, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, transC, lower_only,
                              batch, triA);
}

template <typename T>
slab_status dense_transpose(slab_handle* h, const T* in, int64_t ldin, int64_t sin, T* out, int64_t ldout,
                            int64_t sout, int rows, int cols, int batch) {
    if (batch <= 0 || rows <= 0 || cols <= 0) return SLAB_OK;
    for (int b0 = 0; b0 < batch; b0 += 65535) {
        const int nb = std::min(65535, batch - b0);
        dim3 grid((cols + 63) / 64, (rows + 63) / 64, nb);
        SLAB_PROF(h, KC_OTHER);
        transpose_rect_kernel<T><<<grid, 256, 0, h->stream>>>(in + b0 * sin, ldin, sin, out + b0 * sout, ldout, sout,
                                                              rows, cols);
        SLAB_CK_LAUNCH(h);
    }
    return SLAB_OK;
}

template <typename T>
slab_status dense_copy(slab_handle* h, const T* in, int64_t sin, T* out, int64_t sout, int64_t n, int batch) {
    if (batch <= 0 || n <= 0) return SLAB_OK;
    for (int b0 = 0; b0 < batch; b0 += 65535) {
        const int nb = std::min(65535, batch - b0);
        SLAB_PROF(h, KC_OTHER);
        const T* ib = in + b0 * sin;
        T* ob = out + b0 * sout;
        const bool v16 = ((uintptr_t)ib % 16 == 0) && ((uintptr_t)ob % 16 == 0) && (sin * sizeof(T)) % 16 == 0 &&
                         (sout * sizeof(T)) % 16 == 0 && (n * sizeof(T)) % 16 == 0;
        if (v16) {
            const int64_t n16 = n * (int64_t)sizeof(T) / 16;
            copy16_batched_kernel<<<dim3((unsigned)std::min<int64_t>((n16 + 1023) / 1024, 64), nb), 256, 0,
                                    h->stream>>>((const uint4*)ib, sin * (int64_t)sizeof(T) / 16, (uint4*)ob,
                                                 sout * (int64_t)sizeof(T) / 16, n16);
        } else {
            copy_batched_kernel<T><<<dim3((unsigned)std::min<int64_t>((n + 255) / 256, 64), nb), 256, 0,
                                     h->stream>>>(ib, sin, ob, sout, n);
        }
        SLAB_CK_LAUNCH(h);
    }
    return SLAB_OK;
}

// Cholesky of the leading ncols x ncols block of a batch of tall matrices (row-major, ld = ncols,
// bstride apart) whose rows below are eliminated with it: rows [ncols, ident0) receive B^T L^{-T},
// rows [ident0, ident0 + ncols), which must hold the identity, receive L^{-T}.
// Identity row ident0 + r is zero in the columns left of r until column r is eliminated, so the
// columns [0, c) only ever touch rows [0, ident0 + c).
//
// Recursive column bisection (right-looking at every level): factor the left half of a column
// range, apply its one update to the right half -- C[c0:, c0:c1] -= P P[:c1-c0]^T with P the left
// half's columns and K = the left half's width -- then factor the right half.  64-column panels
// are the leaves (panel_diag_kernel factors the diagonal tile once, panel_apply_kernel scales the
// tiles below by its inverse).  Each level reads and writes the trailing matrix once, so the
// trailing updates stream it about log2(ncols / 64) times in all, and most of their flops fall in
// products with a large K.
namespace {

// C[c0 : rows, c0 : c1] -= W[c0 : rows, k0 : k1] W[c0 : c1, k0 : k1]^T (lower tiles of the square
// part), for every matrix of the batch.  Where the FP16 three-product work buffer of the factor is
// too small for the whole batch, the product runs on slices of the batch, or of K for one matrix.
template <typename T>
slab_status tall_update(slab_handle* h, T* W, int ncols, int rows, int c0, int c1, int k0, int k1, int batch,
                        int64_t bstride) {
    const int M = rows - c0, N = c1 - c0;
    int bchunk = batch, kchunk = k1 - k0;
    if (sizeof(T) == 4 && h->w16 && !h->tf32_now) {
        while (bchunk > 1 && f16x3_work_bytes(M, N, kchunk, bchunk, true) > h->w16_bytes) bchunk = (bchunk + 1) / 2;
        while (kchunk > TL && f16x3_work_bytes(M, N, kchunk, bchunk, true) > h->w16_bytes)
            kchunk = (kchunk / TL + 1) / 2 * TL;
    }
    slab_status st;
    for (int b0 = 0; b0 < batch; b0 += bchunk) {
        const int nb = std::min(bchunk, batch - b0);
        T* Wb = W + (int64_t)b0 * bstride;
        for (int ka = k0; ka < k1; ka += kchunk) {
            const int kw = std::min(kchunk, k1 - ka);
            const T* P = Wb + (int64_t)c0 * ncols + ka;
            if ((st = dense_gemm<T>(h, KC_TRAIL, M, N, kw, T(-1), P, ncols, bstride, P, ncols, bstride, T(1),
                                    Wb + (int64_t)c0 * ncols + c0, ncols, bstride, 0, 1, nb)))
                return st;
        }
    }
    return SLAB_OK;
}

// Whether an FP32 panel launch of `ctas` CTAs with one extra 64 x 64 tile of shared memory runs in one wave
// on the 152 SMs (two CTAs per SM): then every CTA can factor the diagonal tile itself and the separate
// diagonal launch is saved.  FP64 panels factor it once and spread everything else over the SMs: the
// fused kernels' redundant products cost 65 us each there (n = 128, b = 16 Poisson solve 6.5 -> 3.7 ms).
inline bool one_wave(int64_t ctas) { return ctas <= 2 * SMS; }

template <typename T>
slab_status tall_panel(slab_handle* h, T* W, int ncols, int ident0, int kb, int batch, int64_t bstride, size_t smem) {
    const int rows = ident0 + (kb + 1) * TL;
    const int nrt = rows / TL - kb - 1;
    T* Lw = (T*)h->pnl;
    for (int b0 = 0; b0 < batch; b0 += 65535) {
        const int nb = std::min(65535, batch - b0);
        if constexpr (sizeof(T) == 4)
            if (nrt > 0 && one_wave((int64_t)nrt * nb)) {
                SLAB_PROF(h, KC_PANEL);
                SLAB_CK(h, launch_pdl(panel_apply_kernel<T, true>, dim3(nrt, nb), dim3(256), smem + TL * PTP * sizeof(T),
                                      h->stream, W + b0 * bstride, (int64_t)ncols, kb, bstride, (const T*)Lw,
                                      h->dstatus));
                SLAB_CK_LAUNCH(h);
                continue;
            }
        {
            SLAB_PROF(h, KC_PANEL);
            SLAB_CK(h, launch_pdl(panel_diag_kernel<T>, dim3(1, nb), dim3(256), smem, h->stream, W + b0 * bstride,
                                  (int64_t)ncols, kb, h->dstatus, bstride, Lw));
            SLAB_CK_LAUNCH(h);
        }
        if (nrt > 0) {
            SLAB_PROF(h, KC_PANEL);
            if constexpr (sizeof(T) == 8)
                SLAB_CK(h, launch_pdl(panel_apply_rows_kernel<T>, dim3(8 * nrt, nb), dim3(256), 0, h->stream,
                                      W + b0 * bstride, (int64_t)ncols, kb, bstride, (const T*)Lw));
            else
                SLAB_CK(h, launch_pdl(panel_apply_kernel<T, false>, dim3(nrt, nb), dim3(256), smem, h->stream,
                                      W + b0 * bstride, (int64_t)ncols, kb, bstride, (const T*)Lw, h->dstatus));
            SLAB_CK_LAUNCH(h);
        }
    }
    return SLAB_OK;
}

// Panels kb and kb+1 (kb+1 < ncols / 64), all updates from the columns left of kb applied: three
// launches -- panel_diag_kernel(kb), panel_pair_kernel(kb) (panel kb scaled, its update of panel
// kb+1, panel kb+1's diagonal factored), panel_apply_kernel(kb+1) -- instead of a panel, a product
// and a panel; one (panel_pair_full_kernel) where the row tiles fit in one wave.
template <typename T>
slab_status tall_pair(slab_handle* h, T* W, int ncols, int ident0, int kb, int batch, int64_t bstride, size_t smem) {
    const int nrt0 = (ident0 + (kb + 1) * TL) / TL - kb - 1;      // row tiles below the diagonal, panel kb
    const int nrt1 = (ident0 + (kb + 2) * TL) / TL - kb - 2;      // and panel kb+1
    const size_t psmem = 4 * TL * PTP * sizeof(T);
    T* Lw = (T*)h->pnl;
    for (int b0 = 0; b0 < batch; b0 += 65535) {
        const int nb = std::min(65535, batch - b0);
        T* Lw2 = Lw + (int64_t)nb * TL * TL;
        SLAB_PROF(h, KC_PANEL);
        if (ident0 % TL == 0 && nrt1 == nrt0 && one_wave((int64_t)(nrt0 + 1) * nb)) {
            SLAB_CK(h, launch_pdl(panel_pair_full_kernel<T>, dim3(nrt0 + 1, nb), dim3(256), psmem + TL * PTP * sizeof(T),
                                  h->stream, W + b0 * bstride, (int64_t)ncols, kb, bstride, h->dstatus));
            SLAB_CK_LAUNCH(h);
            continue;
        }
        if (one_wave((int64_t)nrt0 * nb)) {
            SLAB_CK(h, launch_pdl(panel_pair_kernel<T, true>, dim3(nrt0, nb), dim3(256), psmem + TL * PTP * sizeof(T),
                                  h->stream, W + b0 * bstride, (int64_t)ncols, kb, bstride, (const T*)Lw, Lw2,
                                  h->dstatus));
            SLAB_CK_LAUNCH(h);
        } else {
            SLAB_CK(h, launch_pdl(panel_diag_kernel<T>, dim3(1, nb), dim3(256), smem, h->stream, W + b0 * bstride,
                                  (int64_t)ncols, kb, h->dstatus, bstride, Lw));
            SLAB_CK_LAUNCH(h);
            SLAB_CK(h, launch_pdl(panel_pair_kernel<T, false>, dim3(nrt0, nb), dim3(256), psmem, h->stream,
                                  W + b0 * bstride, (int64_t)ncols, kb, bstride, (const T*)Lw, Lw2, h->dstatus));
            SLAB_CK_LAUNCH(h);
            prof_extra(h, KC_PANEL, 1);
        }
        if (nrt1 > 0) {
            SLAB_CK(h, launch_pdl(panel_apply_kernel<T, false>, dim3(nrt1, nb), dim3(256), smem, h->stream,
                                  W + b0 * bstride, (int64_t)ncols, kb + 1, bstride, (const T*)Lw2, h->dstatus));
            SLAB_CK_LAUNCH(h);
            prof_extra(h, KC_PANEL, 1);
        }
    }
    return SLAB_OK;
}

// Panels [kb0, kb1), all updates from the columns left of kb0 already applied.
template <typename T>
slab_status tall_chol_range(slab_handle* h, T* W, int ncols, int ident0, int kb0, int kb1, int batch,
                            int64_t bstride, size_t smem) {
    if (kb1 - kb0 == 1) return tall_panel<T>(h, W, ncols, ident0, kb0, batch, bstride, smem);
    // FP32: the fused pair saves launches on the latency-bound critical path of small batches; large batches
    // fill the GPU anyway, and there its redundant tile products cost more than the launches it saves
    const int64_t tiles = (int64_t)batch * ((ident0 + (kb0 + 1) * TL) / TL - kb0 - 1);
    if constexpr (sizeof(T) == 4)
        if (kb1 - kb0 == 2 && tiles <= 8 * SMS) return tall_pair<T>(h, W, ncols, ident0, kb0, batch, bstride, smem);
    const int kbm = kb0 + (kb1 - kb0) / 2;
    slab_status st;
    if ((st = tall_chol_range<T>(h, W, ncols, ident0, kb0, kbm, batch, bstride, smem))) return st;
    if ((st = tall_update<T>(h, W, ncols, ident0 + kbm * TL, kbm * TL, kb1 * TL, kb0 * TL, kbm * TL, batch, bstride)))
        return st;
    return tall_chol_range<T>(h, W, ncols, ident0, kbm, kb1, batch, bstride, smem);
}

}  // namespace

template <typename T>
slab_status dense_tall_cholesky(slab_handle* h, T* W, int ncols, int ident0, int batch, int64_t bstride) {
    const size_t smem = 2 * TL * PTP * sizeof(T);
    SLAB_CK(h, cudaFuncSetAttribute(panel_diag_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if constexpr (sizeof(T) == 4) {
        const int tile = (int)(TL * PTP * sizeof(T));
        SLAB_CK(h, cudaFuncSetAttribute(panel_apply_kernel<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)smem));
        SLAB_CK(h, cudaFuncSetAttribute(panel_apply_kernel<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)smem + tile));
        SLAB_CK(h, cudaFuncSetAttribute(panel_pair_kernel<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        4 * tile));
        SLAB_CK(h, cudaFuncSetAttribute(panel_pair_kernel<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        5 * tile));
        SLAB_CK(h, cudaFuncSetAttribute(panel_pair_full_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 5 * tile));
    }
    const int bchunk = std::min(batch, 65535);
    slab_status st;
    if ((st = ensure_panel_work(h, 2 * (size_t)bchunk * TL * TL * sizeof(T)))) return st;   // L^-1 of two panels
    const int nt = ncols / TL;
    if (nt <= 0) return SLAB_OK;
    return tall_chol_range<T>(h, W, ncols, ident0, 0, nt, batch, bstride, smem);
}

template slab_status dense_gemm<float>(slab_handle*, int, int, int, int, float, const float*, int64_t, int64_t,
                                       const float*, int64_t, int64_t, float, float*, int64_t, int64_t, int, int, int, int);
template slab_status dense_gemm<double>(slab_handle*, int, int, int, int, double, const double*, int64_t, int64_t,
                                        const double*, int64_t, int64_t, double, double*, int64_t, int64_t, int, int,
                                        int, int);
template slab_status dense_transpose<float>(slab_handle*, const float*, int64_t, int64_t, float*, int64_t, int64_t,
                                            int, int, int);
template slab_status dense_transpose<double>(slab_handle*, const double*, int64_t, int64_t, double*, int64_t,
                                             int64_t, int, int, int);
template slab_status dense_copy<float>(slab_handle*, const float*, int64_t, float*, int64_t, int64_t, int);
template slab_status dense_copy<double>(slab_handle*, const double*, int64_t, double*, int64_t, int64_t, int);
template slab_status dense_tall_cholesky<float>(slab_handle*, float*, int, int, int, int64_t);
template slab_status dense_tall_cholesky<double>(slab_handle*, double*, int, int, int, int64_t);
