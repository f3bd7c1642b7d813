// The parallel phases of Algorithm 4 in two dimensions for more than SOLVE_NARROW loads (treesolve.cu
// runs the others): one launch per tree height, the m x K products of a node in 4 x 4 register blocks
// over a 64-wide block of loads; in FP32 with up to 32 loads the low heights run a warp per node.
#include "tree_args.cuh"

namespace {

constexpr int MAXM = SLAB_MAXM;
constexpr int TB_THREADS = 128;

template <typename T>
struct SolveArgs {
    TreeArgs<T> tr;
    int K;            // right-hand sides in this call (<= kcap)
    int kcap;         // stride of the right-hand-side index
    T* Yv;            // [NS][s+1][m][kcap]
    T* Gtb;           // [NS][s+1][2][m][kcap]
    T* Xs;            // [NS][s+1][m][kcap]
    T* Fi;            // [NS][2][s_pad][kcap]
    T* X;             // [NI][kcap][s_pad]  right-hand-side major
    __device__ int64_t nodeoff(int t, int c) const { return (int64_t)t * (tr.s + 1) + c; }
    __device__ T* yv(int t, int c) const { return Yv + nodeoff(t, c) * tr.m * kcap; }
    __device__ T* gtb(int t, int c, int tb) const { return Gtb + (nodeoff(t, c) * 2 + tb) * tr.m * kcap; }
    __device__ T* xs(int t, int c) const { return Xs + nodeoff(t, c) * tr.m * kcap; }
    __device__ T* fi(int t, int side) const { return Fi + ((int64_t)t * 2 + side) * tr.s_pad * kcap; }
    __device__ T* xi(int q) const { return X + (int64_t)q * tr.s_pad * kcap; }   // [kcap][s_pad]
};

constexpr int KMAX = 64;   // right-hand sides handled per launch
constexpr int LP = 36;     // smem row stride of the 32-row blocks read 4 at a time (16-byte aligned)
constexpr int KP = KMAX + 4;   // smem row stride of the m x K blocks: 16-byte aligned, rows 4 banks apart

// Lane -> (row i, right-hand side r) inside a warp tile of 8 rows x 4 right-hand sides, for the
// copies between a [row][r] smem block of stride KP and global memory contiguous in the row
// index: the smem words (KP i + r) of a warp (a half-warp for double) fall in distinct banks,
// and the global side touches four (double: eight) 32-byte segments per warp.
template <typename T>
__device__ inline void lane_rows_rhs(int lane, int& i, int& r) {
    if (sizeof(T) == 8) { i = (lane & 3) | ((lane >> 4) << 2); r = (lane >> 2) & 3; }
    else { i = lane & 7; r = lane >> 3; }
}

// four consecutive smem values (16-byte aligned): one 128-bit store for float, two for double
__device__ inline void sts4(float* p, const float v[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ inline void sts4(double* p, const double v[4]) {
    reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
}

// four consecutive smem values (16-byte aligned): one 128-bit load for float, two for double
__device__ inline void lds4(const float* p, float v[4]) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ inline void lds4(const double* p, double v[4]) {
    const double2 a = *reinterpret_cast<const double2*>(p);
    const double2 b = *reinterpret_cast<const double2*>(p + 2);
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}

// Up pass of one height: y = Li (f_c + G_alpha[bot] + G_beta[top]); condensed top/bot load;
// interface load Fi -= Z_I^T y.  grid = (node, chunk, slab).  The m x K products use 4 x 4
// register blocks: thread (tA, tB) owns rows 4tA..4tA+3 and right-hand sides 4tB..4tB+3.
template <typename T>
__global__ void __launch_bounds__(TB_THREADS, sizeof(T) == 8 ? 5 : 8) tree_up_kernel(SolveArgs<T> P, int k, const double* F,
                                                             double fscale, int r0) {
    constexpr int ZP = 2 * MAXM + 4;   // Zt row stride: top half at 0, bottom half at MAXM
    __shared__ __align__(16) T Li[MAXM * LP];      // Li[l][i] = (L^{-1})[i][l], zero outside m x m
    __shared__ __align__(16) T Zt[MAXM * ZP];      // Zt[i][tb MAXM + a] = Z[i][tb m + a], zero for a >= m
    __shared__ __align__(16) T y[MAXM * KP];
    // 32 interface columns of Z_I, staged per pass; Zt is no longer read by then
    T* const zs = Zt;
    static_assert(ZP >= LP, "staging area must fit in Zt");
    const TreeArgs<T>& A = P.tr;
    const int tid = threadIdx.x, nth = blockDim.x;
    const int tA = tid >> 4, tB = tid & 15;
    const int t = blockIdx.z;
    const int c = (2 * blockIdx.x + 1) << k;
    const int s = A.s, m = A.m, K = P.K, kc = P.kcap;
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
    const int m2 = 2 * m;
    const T* Lg = A.linv(t, c);
    const T* Zg = A.ztb(t, c);
    // Zt: rows by warp, columns by lane.  Li transposed through tiles of JB columns x 32/JB rows
    // per warp (jl fast): smem words (LP l + i) of a wavefront fall in distinct banks.  Each
    // group of loads is issued into registers before its stores.
    constexpr int NW = TB_THREADS / 32;
    const int lane = tid & 31, warp = tid >> 5;
    {
        constexpr int JB = sizeof(T) == 8 ? 4 : 8;
        constexpr int LIT = (MAXM / JB) * (MAXM / (32 / JB)) / NW;
        const int jl = lane % JB, il = lane / JB;
        T z0[MAXM / NW], z1[MAXM / NW], lr[LIT];
#pragma unroll
        for (int it = 0; it < MAXM / NW; ++it) {
            const int i = warp + NW * it;
            const bool ok = i < m && lane < m;
            z0[it] = ok ? Zg[i * m2 + lane] : T(0);
            z1[it] = ok ? Zg[i * m2 + m + lane] : T(0);
        }
#pragma unroll
        for (int it = 0; it < LIT; ++it) {
            const int wb = warp + NW * it;
            const int l = JB * (wb % (MAXM / JB)) + jl, i = (32 / JB) * (wb / (MAXM / JB)) + il;
            lr[it] = (i < m && l < m) ? Lg[i * m + l] : T(0);
        }
#pragma unroll
        for (int it = 0; it < MAXM / NW; ++it) {
            const int i = warp + NW * it;
            Zt[i * ZP + lane] = z0[it];
            Zt[i * ZP + MAXM + lane] = z1[it];
        }
#pragma unroll
        for (int it = 0; it < LIT; ++it) {
            const int wb = warp + NW * it;
            const int l = JB * (wb % (MAXM / JB)) + jl, i = (32 / JB) * (wb / (MAXM / JB)) + il;
            Li[l * LP + i] = lr[it];
        }
    }
    const int64_t N = (int64_t)s * s;
    {
        constexpr int YIT = (MAXM / 8) * (KMAX / 4) / NW;
        int il, rl;
        lane_rows_rhs<T>(lane, il, rl);
        T g[YIT];
#pragma unroll
        for (int it = 0; it < YIT; ++it) {
            const int wb = warp + NW * it;
            const int i = 8 * (wb % (MAXM / 8)) + il, r = 4 * (wb / (MAXM / 8)) + rl;
            g[it] = (i < m && r < K)
                        ? (T)F[(int64_t)(r0 + r) * N + (int64_t)(c - 1) * s + (x0 - 1 + i)] * (T)fscale
                        : T(0);
        }
        if (alpha) {
            const T* ga = P.gtb(t, alpha, 1);
#pragma unroll
            for (int it = 0; it < YIT; ++it) {
                const int wb = warp + NW * it;
                const int i = 8 * (wb % (MAXM / 8)) + il, r = 4 * (wb / (MAXM / 8)) + rl;
                if (i < m && r < K) g[it] += ga[i * kc + r];
            }
        }
        if (beta) {
            const T* gb = P.gtb(t, beta, 0);
#pragma unroll
            for (int it = 0; it < YIT; ++it) {
                const int wb = warp + NW * it;
                const int i = 8 * (wb % (MAXM / 8)) + il, r = 4 * (wb / (MAXM / 8)) + rl;
                if (i < m && r < K) g[it] += gb[i * kc + r];
            }
        }
#pragma unroll
        for (int it = 0; it < YIT; ++it) {
            const int wb = warp + NW * it;
            y[(8 * (wb % (MAXM / 8)) + il) * KP + 4 * (wb / (MAXM / 8)) + rl] = g[it];
        }
    }
    __syncthreads();
    // y = Li g
    {
        T acc[4][4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int p = 0; p < 4; ++p) acc[q][p] = T(0);
        for (int l = 0; l < m; ++l) {
            T gv[4], lv[4];
            lds4(y + l * KP + 4 * tB, gv);
            lds4(Li + l * LP + 4 * tA, lv);
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int p = 0; p < 4; ++p) acc[q][p] += lv[q] * gv[p];
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 4; ++q) sts4(y + (4 * tA + q) * KP + 4 * tB, acc[q]);
    }
    __syncthreads();
    if (blockIdx.y == 0) {
        T* yd = P.yv(t, c);
        for (int i = tid >> 6; i < m; i += nth >> 6) {
            const int r = tid & 63;
            if (r < K) yd[i * kc + r] = y[i * KP + r];
        }
        // condensed top / bottom loads: G_tb[a][r] = G_child[a][r] - sum_i Z[i][tb*m + a] y[i][r]
        for (int tb = 0; tb < 2; ++tb) {
            const int child = tb == 0 ? alpha : beta;
            T acc[4][4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int p = 0; p < 4; ++p) acc[q][p] = T(0);
            for (int i = 0; i < m; ++i) {
                T yv[4], zv[4];
                lds4(y + i * KP + 4 * tB, yv);
                lds4(Zt + i * ZP + tb * MAXM + 4 * tA, zv);
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int p = 0; p < 4; ++p) acc[q][p] += zv[q] * yv[p];
            }
            const T* gc = child ? P.gtb(t, child, tb) : nullptr;
            T* gd = P.gtb(t, c, tb);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int a = 4 * tA + q;
                if (a >= m) continue;
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const int r = 4 * tB + p;
                    if (r < K) gd[a * kc + r] = (gc ? gc[a * kc + r] : T(0)) - acc[q][p];
                }
            }
        }
    }
    // interface load: Fi[side][rr][r] -= sum_i Z_I[i][rr] y[i][r]
    const int qend = min(ncols, q0 + TB_THREADS);
    if (qend - q0 <= 16) {
        // few columns (low heights): thread = (column, group of RB right-hand sides)
        const int nq = qend - q0;
        const int RB = nq <= 2 ? 1 : (nq <= 4 ? 2 : (nq <= 8 ? 4 : 8));
        const int groups = KMAX / RB;
        const int qq = tid / groups, r0b = (tid % groups) * RB;
        if (qq < nq && r0b < K) {
            const int col = q0 + qq;
            const int sd = col / w, rr = lo + col % w - 1;
            const T* zcol = A.zi(t, k, sd) + rr;
            T acc[8], zv[MAXM];
#pragma unroll
            for (int p = 0; p < 8; ++p) acc[p] = T(0);
#pragma unroll
            for (int i = 0; i < MAXM; ++i) zv[i] = i < m ? zcol[(int64_t)i * A.s_pad] : T(0);
#pragma unroll
            for (int i = 0; i < MAXM; ++i) {
                if (i >= m) break;
#pragma unroll
                for (int p = 0; p < 8; ++p)
                    if (p < RB) acc[p] += zv[i] * y[i * KP + r0b + p];
            }
            T* fo = P.fi(t, sd) + (int64_t)rr * kc;
#pragma unroll
            for (int p = 0; p < 8; ++p)
                if (p < RB && r0b + p < K) fo[r0b + p] -= acc[p];
        }
        return;
    }
    for (int qa = q0; qa < qend; qa += 32) {
        int sd[4], rr[4];
        bool ok[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int qq = qa + 4 * tA + q;
            ok[q] = qq < qend;
            sd[q] = ok[q] ? qq / w : 0;
            rr[q] = ok[q] ? lo + qq % w - 1 : 0;
        }
        // stage Z_I[i][columns qa .. qa+31] (rows by warp, columns by lane: coalesced)
        T zr[MAXM / NW];
        {
            const int qq = qa + lane;
            const int sdq = qq >= w, rq = lo + (sdq ? qq - w : qq) - 1;
            const T* zsrc = A.zi(t, k, sdq) + rq;
#pragma unroll
            for (int it = 0; it < MAXM / NW; ++it) {
                const int i = warp + NW * it;
                zr[it] = (i < m && qq < qend) ? zsrc[(int64_t)i * A.s_pad] : T(0);
            }
        }
        __syncthreads();
#pragma unroll
        for (int it = 0; it < MAXM / NW; ++it) zs[(warp + NW * it) * LP + lane] = zr[it];
        __syncthreads();
        T acc[4][4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int p = 0; p < 4; ++p) acc[q][p] = T(0);
        for (int i = 0; i < m; ++i) {
            T yv[4], zv[4];
            lds4(y + i * KP + 4 * tB, yv);
            lds4(zs + i * LP + 4 * tA, zv);
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int p = 0; p < 4; ++p) acc[q][p] += zv[q] * yv[p];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (!ok[q]) continue;
            T* fo = P.fi(t, sd[q]) + (int64_t)rr[q] * kc;
#pragma unroll
            for (int p = 0; p < 4; ++p)
                if (4 * tB + p < K) fo[4 * tB + p] -= acc[q][p];
        }
    }
}

// Down pass of one height: x_c = Li^T (y - Z_top x_top - Z_bot x_bot - Z_I u_I).
// grid = (node, chunk, slab).  A node's 2w interface columns are split into chunks of DCW; each
// CTA reduces its chunk (chunk 0 also the 2m top/bottom columns) into a partial V (m x K) held
// in 4 x 4 register blocks.  Nodes with one chunk finish in place; otherwise the partials go to
// ws and the last CTA of the node (ticket) adds them in chunk order and finishes the node.
constexpr int DCW = 256;      // largest chunk; heights with few nodes use smaller chunks (down_chunk)
constexpr int DCW_MIN = 32;

// Interface columns per CTA of the down pass at a height with `nodes` nodes of 2 wmax columns:
// enough CTAs to fill the GPU (about 4 per SM) without chunks narrower than DCW_MIN.
inline int down_chunk(int nodes, int wmax) {
    int c = DCW;
    while (c > DCW_MIN && (int64_t)nodes * ((2 * wmax + c - 1) / c) < 4 * SMS) c /= 2;
    return c;
}
template <typename T, bool INDEF>
__global__ void __launch_bounds__(TB_THREADS, sizeof(T) == 8 ? 5 : 8) tree_down_kernel(SolveArgs<T> P, int k, double* U,
                                                               int accumulate, int r0, T* ws,
                                                               unsigned* tickets, int dcw) {
    constexpr int CJ = sizeof(T) == 8 ? 16 : 32;   // columns per smem stage
    constexpr int NW = TB_THREADS / 32;
    // Staging tiles of 32 elements per warp: lane (jl, il) with jl fast.  zc[jj][i] and uc[jj][r]
    // rows are LP (KP) words apart = 4 banks, so 8 columns x 4 rows (double: 4 x 8, 16 lanes
    // per wavefront) hit distinct banks while the global side reads 32-byte segments along the
    // column index.  Stages made only of top/bottom columns read x_top / x_bot, which are
    // contiguous in r, with r on the lanes instead.  Each thread issues all loads of a stage
    // into registers before the barrier that frees the smem tiles.
    constexpr int JB = sizeof(T) == 8 ? 4 : 8;
    constexpr int ZIT = (CJ / JB) * (MAXM / (32 / JB)) / NW;   // zc tiles per warp
    constexpr int UIT = (CJ / JB) * (KMAX / (32 / JB)) / NW;   // uc tiles per warp
    static_assert(UIT == (CJ / NW) * (KMAX / 32), "top/bottom staging covers the same tile count");
    __shared__ __align__(16) T Li[MAXM * LP];          // Li[l][i], zero for i >= m
    __shared__ __align__(16) T V[MAXM * KP];
    __shared__ __align__(16) T zc[CJ * LP];            // zc[jj][i]: column jj of the stage, rows i
    __shared__ __align__(16) T uc[CJ * KP];            // uc[jj][r]: column jj of the stage, rhs r
    __shared__ bool last;
    const TreeArgs<T>& A = P.tr;
    const int tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    const int tA = tid >> 4, tB = tid & 15;
    const int t = blockIdx.z;
    const int c = (2 * blockIdx.x + 1) << k;
    const int s = A.s, m = A.m, K = P.K, kc = P.kcap;
    if (c > s) return;
    const int lo = c - (1 << k) + 1;
    const int hi = min(s, c + (1 << k) - 1);
    const int w = hi - lo + 1;
    const int nch = (2 * w + dcw - 1) / dcw;
    if ((int)blockIdx.y >= nch) return;
    const int qa = blockIdx.y * dcw, qb = min(2 * w, qa + dcw);
    const int x0 = t * A.b + 1;
    const int m2 = 2 * m;
    // acc accumulates -y + sum_j z_j u_j^T (y only in chunk 0), so that V = y - sum = -acc.
    // The y loads and the Li staging are issued first and overlap the first stage.
    T acc[4][4];
    if (blockIdx.y == 0) {
        const T* yv = P.yv(t, c);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const int row = 4 * tA + q, r = 4 * tB + p;
                acc[q][p] = (row < m && r < K) ? -yv[row * kc + r] : T(0);
            }
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int p = 0; p < 4; ++p) acc[q][p] = T(0);
    }
    if (!INDEF) {
        const T* Lg = A.linv(t, c);
        T lr[MAXM / NW];
#pragma unroll
        for (int it = 0; it < MAXM / NW; ++it) {
            const int i = warp + NW * it;
            lr[it] = (i < m && lane < m) ? Lg[i * m + lane] : T(0);
        }
#pragma unroll
        for (int it = 0; it < MAXM / NW; ++it) Li[(warp + NW * it) * LP + lane] = lr[it];
    }
    const T* Zg = INDEF ? A.wtb(t, c) : A.ztb(t, c);    // SPD: Z; indefinite: W = S^{-1} B
    const T* xt = (lo - 1 >= 1) ? P.xs(t, lo - 1) : nullptr;
    const T* xb = (hi + 1 <= s) ? P.xs(t, hi + 1) : nullptr;
    // one list of columns: the 2m top/bot columns (chunk 0 only), then this chunk's interface
    // columns of the left (ic < w) and right side; staged CJ at a time
    const int ntb = blockIdx.y == 0 ? m2 : 0;
    const int ntot = ntb + (qb - qa);
    const T* ZIl = (t >= 1) ? (INDEF ? A.wi(t, k, 0) : A.zi(t, k, 0)) + (lo - 1) : nullptr;
    const T* ZIr = (t < A.NS - 1) ? (INDEF ? A.wi(t, k, 1) : A.zi(t, k, 1)) + (lo - 1) : nullptr;
    const T* Ul = (t >= 1) ? P.xi(t - 1) + (lo - 1) : nullptr;
    const T* Ur = (t < A.NS - 1) ? P.xi(t) + (lo - 1) : nullptr;
    const int jl = lane % JB, il = lane / JB;
    for (int v0 = 0; v0 < ntot; v0 += CJ) {
        const int nj = min(CJ, ntot - v0);
        T zr[ZIT], ur[UIT];
#pragma unroll
        for (int it = 0; it < ZIT; ++it) {
            const int wb = warp + NW * it;
            const int jj = JB * (wb % (CJ / JB)) + jl, i = (32 / JB) * (wb / (CJ / JB)) + il;
            const int col = v0 + jj;
            T z = T(0);
            if (jj < nj && i < m) {
                if (col < ntb) {
                    z = Zg[(int64_t)i * m2 + col];
                } else {
                    const int ic = qa + col - ntb;
                    const bool right = ic >= w;
                    const T* zs = right ? ZIr : ZIl;
                    if (zs) z = zs[(int64_t)i * A.s_pad + (right ? ic - w : ic)];
                }
            }
            zr[it] = z;
        }
        const bool tb_only = v0 + CJ <= ntb;
        if (tb_only) {
#pragma unroll
            for (int it = 0; it < UIT; ++it) {
                const int jj = warp + NW * (it / (KMAX / 32)), r = lane + 32 * (it % (KMAX / 32));
                const int col = v0 + jj;
                const T* xv = col < m ? xt : xb;
                ur[it] = (xv && r < K) ? xv[(col < m ? col : col - m) * kc + r] : T(0);
            }
        } else {
#pragma unroll
            for (int it = 0; it < UIT; ++it) {
                const int wb = warp + NW * it;
                const int jj = JB * (wb % (CJ / JB)) + jl, r = (32 / JB) * (wb / (CJ / JB)) + il;
                const int col = v0 + jj;
                T v = T(0);
                if (jj < nj && r < K) {
                    if (col < ntb) {
                        const T* xv = col < m ? xt : xb;
                        if (xv) v = xv[(col < m ? col : col - m) * kc + r];
                    } else {
                        const int ic = qa + col - ntb;
                        const bool right = ic >= w;
                        const T* us = right ? Ur : Ul;
                        if (us) v = us[(int64_t)r * A.s_pad + (right ? ic - w : ic)];
                    }
                }
                ur[it] = v;
            }
        }
        __syncthreads();
#pragma unroll
        for (int it = 0; it < ZIT; ++it) {
            const int wb = warp + NW * it;
            const int jj = JB * (wb % (CJ / JB)) + jl, i = (32 / JB) * (wb / (CJ / JB)) + il;
            zc[jj * LP + i] = zr[it];
        }
        if (tb_only) {
#pragma unroll
            for (int it = 0; it < UIT; ++it)
                uc[(warp + NW * (it / (KMAX / 32))) * KP + lane + 32 * (it % (KMAX / 32))] = ur[it];
        } else {
#pragma unroll
            for (int it = 0; it < UIT; ++it) {
                const int wb = warp + NW * it;
                const int jj = JB * (wb % (CJ / JB)) + jl, r = (32 / JB) * (wb / (CJ / JB)) + il;
                uc[jj * KP + r] = ur[it];
            }
        }
        __syncthreads();
        for (int jj = 0; jj < nj; ++jj) {
            T zv[4], uv[4];
            lds4(zc + jj * LP + 4 * tA, zv);
            lds4(uc + jj * KP + 4 * tB, uv);
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int p = 0; p < 4; ++p) acc[q][p] += zv[q] * uv[p];
        }
    }
    if (nch > 1) {
        // partial of this chunk straight from the registers; the last CTA of the node adds the
        // partials in chunk order (deterministic), loading a thread's 16 elements together
        T* wsn = ws + ((int64_t)(t * gridDim.x + blockIdx.x) * gridDim.y) * MAXM * KMAX;
        T* wsc = wsn + (int64_t)blockIdx.y * MAXM * KMAX;
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int p = 0; p < 4; ++p) wsc[(4 * tA + q) * KMAX + 4 * tB + p] = acc[q][p];
        __threadfence();
        __syncthreads();
        unsigned* tk = tickets + (int64_t)t * gridDim.x + blockIdx.x;
        if (tid == 0) last = atomicAdd(tk, 1u) == (unsigned)(nch - 1);
        __syncthreads();
        if (!last) return;
        __threadfence();
        constexpr int PER = MAXM * KMAX / TB_THREADS;
        T v[PER];
#pragma unroll
        for (int j = 0; j < PER; ++j) v[j] = T(0);
        for (int ch = 0; ch < nch; ++ch) {
            const T* src = wsn + (int64_t)ch * MAXM * KMAX + tid;
            T ld[PER];
#pragma unroll
            for (int j = 0; j < PER; ++j) ld[j] = __ldcg(src + j * TB_THREADS);
#pragma unroll
            for (int j = 0; j < PER; ++j) v[j] += ld[j];
        }
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int idx = tid + j * TB_THREADS;
            V[(idx / KMAX) * KP + idx % KMAX] = -v[j];
        }
        if (tid == 0) *tk = 0;
    } else {
        __syncthreads();   // zc / uc reads of the last stage are not affected; V is free
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const T nv[4] = {-acc[q][0], -acc[q][1], -acc[q][2], -acc[q][3]};
            sts4(V + (4 * tA + q) * KP + 4 * tB, nv);
        }
    }
    __syncthreads();
    // finish the node: V = y - sum; SPD: x = Li^T V, indefinite: x = V (y already holds S^{-1} g)
    if (!INDEF) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int p = 0; p < 4; ++p) acc[q][p] = T(0);
        for (int l = 0; l < m; ++l) {                      // x[i] = sum_{l >= i} Li[l][i] V[l]
            T lv[4], vv[4];
            lds4(Li + l * LP + 4 * tA, lv);
            lds4(V + l * KP + 4 * tB, vv);
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int p = 0; p < 4; ++p) acc[q][p] += lv[q] * vv[p];
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 4; ++q) sts4(V + (4 * tA + q) * KP + 4 * tB, acc[q]);
        __syncthreads();
    }
    const int64_t N = (int64_t)s * s;
    if (k > 0) {                       // x of a height-0 row is read by no lower node
        T* xd = P.xs(t, c);
        for (int i = tid >> 6; i < m; i += TB_THREADS >> 6) {
            const int r = tid & 63;
            if (r < K) xd[i * kc + r] = V[i * KP + r];
        }
    }
    {
        int ul, rl;
        lane_rows_rhs<T>(lane, ul, rl);
        for (int wb = warp; wb < (MAXM / 8) * (KMAX / 4); wb += NW) {
            const int i = 8 * (wb % (MAXM / 8)) + ul, r = 4 * (wb / (MAXM / 8)) + rl;
            if (i < m && r < K) {
                const double v = (double)V[i * KP + r];
                double* up = U + (int64_t)(r0 + r) * N + (int64_t)(c - 1) * s + (x0 - 1 + i);
                if (accumulate) *up += v;
                else *up = v;
            }
        }
    }
}

// ---------------------------------------------------------------- low heights, FP32, up to 32 loads: a warp per node
// Lane r holds load r, a node's m entries of it in registers.  The m x m blocks are read four entries at a time from
// shared memory, one address a warp; nothing is exchanged between the lanes but the FP64 loads and
// solutions, whose memory runs along the row (a tile of shared memory).  The kernels above compute 64 loads
// whatever their number.  n = 2048, b = 32, 32 loads: reduced load 3.87 -> 2.80 ms, reduced load and interior
// solve 7.29 -> 5.10 ms (12 loads: 2.43, 4.36); n = 768, 16 loads, convection: 0.64 -> 0.58 and 1.08 -> 0.95 ms.  (Two loads a lane for up to 64:
// 4.54 and 8.60 ms, too few warps in flight.)
//   Heights above LANE_MAX_W rows a segment have too few nodes and more interface columns than a warp should
// walk alone: they stay on the kernels above, as FP64 does (its multiply-adds are the bound).
constexpr int LANES = 32;             // most loads
constexpr int LW = 4;                 // warps (nodes) per CTA
constexpr int LANE_MAX_W = 15;        // widest segment
constexpr int TP = MAXM + 1;          // row stride of the tile of 32 loads x m entries
struct LaneSmem {                     // per warp
    float Z[MAXM * 2 * MAXM];         // row i: top columns at 0, bottom at MAXM; down: then the tile
    float Li[MAXM * MAXM];            // row i: entries l; up: Li and zi first the tile
    float zi[MAXM * 4];               // four interface columns: [i][column]
};
static_assert(MAXM * MAXM + MAXM * 4 >= 32 * TP, "the tile fits");

__device__ __forceinline__ void copy4_async(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
// m rows of m entries, row stride pitch, into rows of stride DP; entries beyond m zero, rows up to the next
// multiple of 8.  Asynchronous.
template <int DP>
__device__ __forceinline__ void lane_fetch(float* dst, const float* src, int pitch, int m, int lane) {
#pragma unroll 4
    for (int i = 0; i < m; ++i) {
        if (lane < m) copy4_async(dst + i * DP + lane, src + i * pitch + lane);
        else dst[i * DP + lane] = 0.f;
    }
    for (int i = m; i < ((m + 7) & ~7); ++i) dst[i * DP + lane] = 0.f;
}
__device__ __forceinline__ void lane_fetch_z(LaneSmem& sm, const float* Zg, int m, int lane) {
    lane_fetch<2 * MAXM>(sm.Z, Zg, 2 * m, m, lane);
    lane_fetch<2 * MAXM>(sm.Z + MAXM, Zg + m, 2 * m, m, lane);
}
// Interface columns col0 .. col0 + 3 of 2 w (left, then right) into sm.zi: zd: the array with the interface node as
// the row (a column's m entries side by side), else zi / wi.
template <bool ROWS>
__device__ __forceinline__ void lane_columns(LaneSmem& sm, const TreeArgs<float>& A, int t, int k, int lo, int w, int col0,
                                             int lane) {
    float v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int col = col0 + e, side = col >= w, rr = lo + (side ? col - w : col) - 1;
        v[e] = 0.f;
        if (lane < A.m && col < 2 * w)
            v[e] = ROWS ? A.zd(t, k, side)[(int64_t)rr * A.m + lane] : A.zi(t, k, side)[(int64_t)lane * A.s_pad + rr];
    }
    __syncwarp();
    *reinterpret_cast<float4*>(&sm.zi[lane * 4]) = make_float4(v[0], v[1], v[2], v[3]);
    __syncwarp();
}

template <bool INDEF>
__global__ void __launch_bounds__(32 * LW, 4) tree_up_lanes_kernel(SolveArgs<float> P, int k, const double* F,
                                                                   float fscale, int r0) {
    extern __shared__ __align__(16) unsigned char lane_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    LaneSmem& sm = reinterpret_cast<LaneSmem*>(lane_smem)[warp];
    const TreeArgs<float>& A = P.tr;
    const int t = blockIdx.y, s = A.s, m = A.m, K = P.K;
    const int64_t kc = P.kcap;
    const int c = (2 * (blockIdx.x * LW + warp) + 1) << k;
    if (c > s) return;                                         // (whole warps: no block barrier below)
    const int lo = c - (1 << k) + 1, hi = min(s, c + (1 << k) - 1), w = hi - lo + 1;
    const int alpha = k > 0 ? c - (1 << (k - 1)) : 0;
    const int kb = tree_right_height(s, c, k);
    const int beta = kb >= 0 ? c + (1 << kb) : 0;
    lane_fetch_z(sm, A.ztb(t, c), m, lane);
    // g = f + the children's condensed loads
    float g[MAXM];
    const double* Fc = F + (int64_t)(c - 1) * s + (int64_t)t * A.b + lane;
    const int64_t N = (int64_t)s * s;
    float* tile = sm.Li;
    for (int q = 0; q < K; q += 8) {
        double v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = (lane < m && q + e < K) ? Fc[(int64_t)(r0 + q + e) * N] : 0.0;
#pragma unroll
        for (int e = 0; e < 8; ++e) tile[(q + e) * TP + lane] = (float)v[e] * fscale;
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < MAXM; ++i) g[i] = tile[lane * TP + i];        // (lanes beyond K: not used)
    __syncwarp();
    lane_fetch<MAXM>(sm.Li, A.linv(t, c), m, m, lane);
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const int child = side ? beta : alpha;
        if (!child) continue;
        const float* gc = P.gtb(t, child, side ? 0 : 1);
        if (lane < K) {
#pragma unroll
            for (int i = 0; i < MAXM; ++i)
                if (i < m) g[i] += gc[i * kc + lane];
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    // y = Li g: SPD, lower triangular, in place from the last row
    float y[MAXM];
#pragma unroll
    for (int ii = 0; ii < MAXM; ++ii) {
        const int i = INDEF ? ii : MAXM - 1 - ii;
        float acc = 0.f;
        if ((i & ~7) < m) {
#pragma unroll
            for (int l = 0; l < MAXM; l += 4)
                if (INDEF || l <= i) {
                    float v[4];
                    lds4(&sm.Li[i * MAXM + l], v);
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (INDEF || l + q <= i) acc += v[q] * g[l + q];
                }
        }
        (INDEF ? y[i] : g[i]) = acc;
    }
    if (!INDEF) {
#pragma unroll
        for (int i = 0; i < MAXM; ++i) y[i] = g[i];
    }
    if (lane < K) {
        float* yd = P.yv(t, c) + lane;
#pragma unroll
        for (int i = 0; i < MAXM; ++i)
            if (i < m) yd[i * kc] = y[i];
    }
    // condensed top / bottom loads, eight rows at a time
#pragma unroll 1
    for (int ch = 0; ch < MAXM / 4; ++ch) {
        const int tb = ch / (MAXM / 8), a0 = 8 * (ch % (MAXM / 8));
        if (a0 >= m) continue;
        float acc[8];
        const int child = tb ? beta : alpha;
        const float* gc = (child ? P.gtb(t, child, tb) : nullptr) + lane;
#pragma unroll
        for (int e = 0; e < 8; ++e)
            acc[e] = (child && a0 + e < m && lane < K) ? gc[(a0 + e) * kc] : 0.f;
#pragma unroll
        for (int i = 0; i < MAXM; ++i)
            if ((i & ~7) < m) {
                float v[8];
                lds4(&sm.Z[i * 2 * MAXM + tb * MAXM + a0], *reinterpret_cast<float(*)[4]>(&v[0]));
                lds4(&sm.Z[i * 2 * MAXM + tb * MAXM + a0 + 4], *reinterpret_cast<float(*)[4]>(&v[4]));
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[e] -= v[e] * y[i];
            }
        float* gd = P.gtb(t, c, tb) + lane;
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (a0 + e < m && lane < K) gd[(a0 + e) * kc] = acc[e];
    }
    // interface loads
#pragma unroll 1
    for (int col0 = 0; col0 < 2 * w; col0 += 4) {
        lane_columns<!INDEF>(sm, A, t, k, lo, w, col0, lane);
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 0; i < MAXM; ++i)
            if ((i & ~7) < m) {
                float v[4];
                lds4(&sm.zi[i * 4], v);
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[e] += v[e] * y[i];
            }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int col = col0 + e, side = col >= w, rr = lo + (side ? col - w : col) - 1;
            if (col < 2 * w && lane < K) P.fi(t, side)[rr * kc + lane] -= acc[e];
        }
    }
}

template <bool INDEF>
__global__ void __launch_bounds__(32 * LW, 4) tree_down_lanes_kernel(SolveArgs<float> P, int k, double* U, int accumulate,
                                                                     int r0) {
    extern __shared__ __align__(16) unsigned char lane_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    LaneSmem& sm = reinterpret_cast<LaneSmem*>(lane_smem)[warp];
    const TreeArgs<float>& A = P.tr;
    const int t = blockIdx.y, s = A.s, m = A.m, K = P.K;
    const int64_t kc = P.kcap;
    const int c = (2 * (blockIdx.x * LW + warp) + 1) << k;
    if (c > s) return;                                         // (whole warps: no block barrier below)
    const int lo = c - (1 << k) + 1, hi = min(s, c + (1 << k) - 1), w = hi - lo + 1;
    lane_fetch_z(sm, INDEF ? A.wtb(t, c) : A.ztb(t, c), m, lane);
    if (!INDEF) lane_fetch<MAXM>(sm.Li, A.linv(t, c), m, m, lane);
    // V = y - Z_top x_top - Z_bot x_bot - Z_I u_I
    float V[MAXM];
    {
        const float* yv = P.yv(t, c) + lane;
#pragma unroll
        for (int i = 0; i < MAXM; ++i) V[i] = (i < m && lane < K) ? yv[i * kc] : 0.f;
    }
#pragma unroll
    for (int tb = 0; tb < 2; ++tb) {
        const int cx = tb ? hi + 1 : lo - 1;
        float x[MAXM];
        if (cx >= 1 && cx <= s) {
            const float* xv = P.xs(t, cx) + lane;
#pragma unroll
            for (int i = 0; i < MAXM; ++i) x[i] = (i < m && lane < K) ? xv[i * kc] : 0.f;
        }
        if (tb == 0) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncwarp();
        }
        if (cx >= 1 && cx <= s) {
#pragma unroll
            for (int i = 0; i < MAXM; ++i)
                if ((i & ~7) < m) {
#pragma unroll
                    for (int l = 0; l < MAXM; l += 4)
                        if ((l & ~7) < m) {
                            float v[4];
                            lds4(&sm.Z[i * 2 * MAXM + tb * MAXM + l], v);
#pragma unroll
                            for (int q = 0; q < 4; ++q) V[i] -= v[q] * x[l + q];
                        }
                }
        }
    }
#pragma unroll 1
    for (int col0 = 0; col0 < 2 * w; col0 += 4) {
        float u[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int col = col0 + e, side = col >= w, rr = lo + (side ? col - w : col) - 1;
            const bool has = col < 2 * w && (side ? t < A.NS - 1 : t >= 1);
            const float* us = has ? P.xi(side ? t : t - 1) + rr : nullptr;
            u[e] = (has && lane < K) ? us[(int64_t)lane * A.s_pad] : 0.f;
        }
        lane_columns<true>(sm, A, t, k, lo, w, col0, lane);
#pragma unroll
        for (int i = 0; i < MAXM; ++i)
            if ((i & ~7) < m) {
                float v[4];
                lds4(&sm.zi[i * 4], v);
#pragma unroll
                for (int e = 0; e < 4; ++e) V[i] -= v[e] * u[e];
            }
    }
    if (!INDEF) {                                              // x = Li^T V in place, row l of Li at a time
#pragma unroll
        for (int l = 0; l < MAXM; ++l)
            if ((l & ~7) < m) {
                const float vl = V[l];
                V[l] = 0.f;
#pragma unroll
                for (int i = 0; i <= l; i += 4) {
                    float v[4];
                    lds4(&sm.Li[l * MAXM + i], v);
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (i + q <= l) V[i + q] += v[q] * vl;
                }
            }
    }
    if (k > 0 && lane < K) {           // x of a height-0 row is read by no lower node
        float* xd = P.xs(t, c) + lane;
#pragma unroll
        for (int i = 0; i < MAXM; ++i)
            if (i < m) xd[i * kc] = V[i];
    }
    double* Uc = U + (int64_t)(c - 1) * s + (int64_t)t * A.b + lane;
    const int64_t N = (int64_t)s * s;
    float* tile = sm.Z;
    __syncwarp();
#pragma unroll
    for (int i = 0; i < MAXM; ++i) tile[lane * TP + i] = V[i];
    __syncwarp();
    for (int q = 0; q < K; q += 8) {
        double o[8];
#pragma unroll
        for (int e = 0; e < 8; ++e)
            o[e] = (accumulate && lane < m && q + e < K) ? Uc[(int64_t)(r0 + q + e) * N] : 0.0;
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (lane < m && q + e < K) {
                const double v = (double)tile[(q + e) * TP + lane];
                Uc[(int64_t)(r0 + q + e) * N] = accumulate ? o[e] + v : v;
            }
    }
}

template <typename Kernel, typename... Args>
cudaError_t launch_lanes(Kernel kernel, int nodes, int NS, cudaStream_t st, Args... args) {
    const size_t smem = LW * sizeof(LaneSmem);
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kernel<<<dim3((nodes + LW - 1) / LW, NS), 32 * LW, smem, st>>>(args...);
    return cudaGetLastError();
}
inline bool on_lanes(int k, int K) { return K <= LANES && (1 << (k + 1)) - 1 <= LANE_MAX_W; }

// X[q][r][rr] = fscale f[r][rr][x_q] + Fi[q][R][rr][r] + Fi[q+1][L][rr][r]  (padding rows zero)
template <typename T>
__global__ void gather_ftilde_kernel(SolveArgs<T> P, const double* F, double fscale, int r0) {
    const TreeArgs<T>& A = P.tr;
    const int q = blockIdx.y;
    const int K = P.K, kc = P.kcap;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)A.s_pad * K) return;
    const int r = (int)(idx / A.s_pad), rr = (int)(idx % A.s_pad);
    T v = T(0);
    if (rr < A.s) {
        const int64_t N = (int64_t)A.s * A.s;
        const int xq = (q + 1) * A.b;
        v = (T)(fscale * F[(int64_t)(r0 + r) * N + (int64_t)rr * A.s + (xq - 1)]);
        v += P.fi(q, 1)[(int64_t)rr * kc + r] + P.fi(q + 1, 0)[(int64_t)rr * kc + r];
    }
    P.xi(q)[(int64_t)r * A.s_pad + rr] = v;
}

template <typename T>
__global__ void scatter_utilde_kernel(SolveArgs<T> P, double* U, int accumulate, int r0) {
    const TreeArgs<T>& A = P.tr;
    const int q = blockIdx.y;
    const int K = P.K, kc = P.kcap;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)A.s * K) return;
    const int rr = (int)(idx % A.s), r = (int)(idx / A.s);
    const int64_t N = (int64_t)A.s * A.s;
    const int xq = (q + 1) * A.b;
    double* up = U + (int64_t)(r0 + r) * N + (int64_t)rr * A.s + (xq - 1);
    const double v = (double)P.xi(q)[(int64_t)r * A.s_pad + rr];
    if (accumulate) *up += v;
    else *up = v;
}

template <typename T>
SolveArgs<T> make_solve_args(slab_handle* h, int K) {
    SolveArgs<T> p;
    p.tr = make_tree_args<T>(h);
    p.K = K; p.kcap = h->kcap;
    p.Yv = (T*)h->wYv; p.Gtb = (T*)h->wGtb; p.Xs = (T*)h->wXs; p.Fi = (T*)h->wFi; p.X = (T*)h->wX;
    return p;
}


inline int chunks_at(int s, int k) {
    const int wmax = min(s, (1 << (k + 1)) - 1);
    return (2 * wmax + TB_THREADS - 1) / TB_THREADS;
}

}  // namespace

// Up pass over all heights for right-hand sides [r0, r0+K) of F (FP64, [k][N]) scaled by fscale,
// then the reduced load f~ into X.
template <typename T>
slab_status tree_up_wide(slab_handle* h, const double* F, double fscale, int r0, int K) {
    SolveArgs<T> p = make_solve_args<T>(h, K);
    const TreeDims& d = h->td;
    SLAB_CK(h, cudaMemsetAsync(h->wFi, 0, (size_t)d.NS * 2 * d.s_pad * h->kcap * h->rsz, h->stream));
    for (int k = 0; k < d.H; ++k) {
        const int cnt = tree_nodes_at(d.s, k);
        if (!cnt) continue;
        dim3 grid(cnt, chunks_at(d.s, k), d.NS);
        SLAB_PROF(h, KC_TREE_UP);
        if constexpr (sizeof(T) == 4) {
            if (on_lanes(k, K)) {
                const bool general = h->kind == SLAB_HELMHOLTZ || h->kind == SLAB_CONVECTION;
                SLAB_CK(h, launch_lanes(general ? tree_up_lanes_kernel<true> : tree_up_lanes_kernel<false>, cnt, d.NS, h->stream,
                                        p, k, F, (float)fscale, r0));
                continue;
            }
        }
        tree_up_kernel<T><<<grid, TB_THREADS, 0, h->stream>>>(p, k, F, fscale, r0);
        SLAB_CK_LAUNCH(h);
    }
    dim3 g2((unsigned)(((int64_t)d.s_pad * K + 255) / 256), d.NI);
    SLAB_PROF(h, KC_TREE_UP);
    gather_ftilde_kernel<T><<<g2, 256, 0, h->stream>>>(p, F, fscale, r0);
    SLAB_CK_LAUNCH(h);
    return SLAB_OK;
}

template <typename T>
slab_status tree_down_wide(slab_handle* h, double* U, int accumulate, int r0, int K) {
    SolveArgs<T> p = make_solve_args<T>(h, K);
    const TreeDims& d = h->td;
    for (int k = d.H - 1; k >= 0; --k) {
        const int cnt = tree_nodes_at(d.s, k);
        if (!cnt) continue;
        const int wmax = min(d.s, (1 << (k + 1)) - 1);
        const int dcw = down_chunk(cnt * d.NS, wmax);
        dim3 grid(cnt, (2 * wmax + dcw - 1) / dcw, d.NS);
        SLAB_PROF(h, KC_TREE_DOWN);
        if constexpr (sizeof(T) == 4) {
            if (on_lanes(k, K)) {
                const bool general = h->kind == SLAB_HELMHOLTZ || h->kind == SLAB_CONVECTION;
                SLAB_CK(h, launch_lanes(general ? tree_down_lanes_kernel<true> : tree_down_lanes_kernel<false>, cnt, d.NS,
                                        h->stream, p, k, U, accumulate, r0));
                continue;
            }
        }
        if (h->kind == SLAB_HELMHOLTZ || h->kind == SLAB_CONVECTION)
            tree_down_kernel<T, true><<<grid, TB_THREADS, 0, h->stream>>>(p, k, U, accumulate, r0, (T*)h->wVp,
                                                                          (unsigned*)h->wVtk, dcw);
        else
            tree_down_kernel<T, false><<<grid, TB_THREADS, 0, h->stream>>>(p, k, U, accumulate, r0, (T*)h->wVp,
                                                                           (unsigned*)h->wVtk, dcw);
        SLAB_CK_LAUNCH(h);
    }
    dim3 g2((unsigned)(((int64_t)d.s * K + 255) / 256), d.NI);
    SLAB_PROF(h, KC_TREE_DOWN);
    scatter_utilde_kernel<T><<<g2, 256, 0, h->stream>>>(p, U, accumulate, r0);
    SLAB_CK_LAUNCH(h);
    return SLAB_OK;
}

// Scratch elements of the down-pass partial sums (largest height with split nodes) and tickets.
size_t tree_down_ws_elems(int s, int m, int NS) {
    size_t best = 0;
    const int H = tree_height_count(s);
    for (int k = 0; k < H; ++k) {
        const int wmax = min(s, (1 << (k + 1)) - 1);
        const int nch = (2 * wmax + DCW_MIN - 1) / DCW_MIN;
        if (nch <= 1) continue;
        const size_t e = (size_t)NS * tree_nodes_at(s, k) * nch * MAXM * KMAX;
        if (e > best) best = e;
    }
    return best;
}
size_t tree_down_tickets(int s, int NS) { return (size_t)NS * (s / 2 + 1); }
template slab_status tree_up_wide<float>(slab_handle*, const double*, double, int, int);
template slab_status tree_up_wide<double>(slab_handle*, const double*, double, int, int);
template slab_status tree_down_wide<float>(slab_handle*, double*, int, int, int);
template slab_status tree_down_wide<double>(slab_handle*, double*, int, int, int);
