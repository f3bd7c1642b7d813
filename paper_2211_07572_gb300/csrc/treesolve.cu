// The parallel phases of Algorithm 4 in two dimensions -- reduced load (eqs. f1-f5) and interior
// back-solve (eq. usol_even) -- on the slab trees factored by tree.cu, for up to SOLVE_NARROW loads
// (treesolve_wide.cu runs more).
//
// Up pass: the rows' condensed loads g start as f; node c of height k, whose segment lies between the
// rows c - 2^k and c + 2^k, does
//   y_c = L^{-1} g_c,   g_{c - 2^k} -= Z_top^T y_c,   g_{c + 2^k} -= Z_bot^T y_c,
// and the reduced load of an interface q is f_q - sum over both slabs and all heights of Z_I^T y.
// Down pass:  x_c = L^{-T} (y_c - Z_I u_I - Z_top x_{c - 2^k} - Z_bot x_{c + 2^k})   (SPD kinds)
//             x_c = y_c - W_I u_I - W_top x_{c - 2^k} - W_bot x_{c + 2^k}   (general kinds, y = S^{-1} g).
//
// Only g and x are recursive in the height; the interface products are not.  So a pass is a few
// launches of recursion, several heights each, and one launch for the interface products of all
// heights: gather_load_kernel reads every Z_I once and writes the reduced load, iface_sum_kernel forms
// Z_I u_I of every node of height >= KSUM (lower nodes have at most 14 columns, summed in place).
//   With one load a pass streams 1.5 m^2 + 2 m w entries a node and does one multiply-add with each:
// bound by HBM and, up the tree, by latency.  A CTA therefore owns a subtree of up to 2^L - 1 rows and
// copies all its matrices into shared memory at once, before it waits for the preceding launch;
// the recursion inside then runs at shared-memory latency.  The unit of work is a warp with one node:
// lane = row of the separator, the loads in registers, the other operand broadcast.
//   Measured (FP32, n = 1024, b = 32, one load, kernel times of a pass): up 0.76 -> 0.16 ms, down 0.67 ->
// 0.19 ms against the kernels of treesolve_wide.cu, which compute 64 loads whatever their number; the low
// launches move 4.1 / 3.0 TB/s through DRAM, 61 / 45 % of a plain copy's rate.  Up to SOLVE_NARROW = 8 loads (n = 777, 5 loads: up + down
// 2.7 -> 0.9 ms a pass) a thread holds them all in registers; beyond, the wide kernels' blocks are fuller.
#include <algorithm>
#include <atomic>

#include "tree_args.cuh"

namespace {

constexpr int MAXM = SLAB_MAXM;
constexpr int KSUM = 3;            // heights below do their own interface products in the down pass
constexpr int CW = 128;            // interface columns per partial sum of a higher node
constexpr int MAXH = 31;
constexpr int KMAX = 64;           // right-hand sides per pass
// Shared memory of a launch over low heights (several CTAs on an SM, their copies and their
// recursion overlap) and of the last one (a CTA per slab; as many heights as fit).
constexpr size_t LOW_SMEM = 72 * 1024, TOP_SMEM = 200 * 1024;

template <typename T>
struct SolveArgs {
    TreeArgs<T> tr;
    int K;            // right-hand sides in this call (<= kcap)
    int kcap;         // stride of the right-hand-side index
    T* Yv;            // [NS][s+1][kcap][m]
    T* Gtb;           // [NS][s+1][2][kcap][m]
    T* Xs;            // [NS][s+1][kcap][m]
    T* X;             // [NI][kcap][s_pad]  right-hand-side major
    T* Vp;            // [NS][vslots][SOLVE_NARROW][m] partial interface sums of the down pass
    int vslots;
    int voff[MAXH];   // first slot of a height
    int vch[MAXH];    // partial sums per node of a height
    __device__ int64_t nodeoff(int t, int c) const { return (int64_t)t * (tr.s + 1) + c; }
    __device__ T* yv(int t, int c, int r) const { return Yv + (nodeoff(t, c) * kcap + r) * tr.m; }
    __device__ T* gtb(int t, int c, int tb, int r) const { return Gtb + ((nodeoff(t, c) * 2 + tb) * kcap + r) * tr.m; }
    __device__ T* xs(int t, int c, int r) const { return Xs + (nodeoff(t, c) * kcap + r) * tr.m; }
    __device__ T* xi(int q, int r) const { return X + ((int64_t)q * kcap + r) * tr.s_pad; }
    __device__ T* vp(int t, int slot, int r) const { return Vp + (((int64_t)t * vslots + slot) * SOLVE_NARROW + r) * tr.m; }
};

// KB consecutive shared-memory values: 16-byte loads where they make up whole ones.
template <int KB>
__device__ __forceinline__ void ldk(const float* p, float (&v)[KB]) {
    if constexpr (KB % 4 == 0) {
#pragma unroll
        for (int q = 0; q < KB; q += 4) {
            const float4 t = *reinterpret_cast<const float4*>(p + q);
            v[q] = t.x; v[q + 1] = t.y; v[q + 2] = t.z; v[q + 3] = t.w;
        }
    } else {
#pragma unroll
        for (int q = 0; q < KB; ++q) v[q] = p[q];
    }
}
template <int KB>
__device__ __forceinline__ void ldk(const double* p, double (&v)[KB]) {
    if constexpr (KB % 2 == 0) {
#pragma unroll
        for (int q = 0; q < KB; q += 2) {
            const double2 t = *reinterpret_cast<const double2*>(p + q);
            v[q] = t.x; v[q + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int q = 0; q < KB; ++q) v[q] = p[q];
    }
}
template <int KB, typename T>
__device__ __forceinline__ void stk(T* p, const T (&v)[KB]) {
    if constexpr (sizeof(T) == 4 && KB % 4 == 0) {
#pragma unroll
        for (int q = 0; q < KB; q += 4)
            *reinterpret_cast<float4*>(p + q) = make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]);
    } else {
#pragma unroll
        for (int q = 0; q < KB; ++q) p[q] = v[q];
    }
}

__device__ __forceinline__ void copy_async(float* dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_async(double* dst, const double* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// A CTA's subtree: rows base + (i + 1) 2^k0, i < 2^L - 1, of slab t; row i has height k0 + ctz(i + 1).
// Shared memory: per row an m x ml block (Linv, ml = m | 1) and an m x mz block (the top and bottom
// columns, mz = 2 m | 1); the odd row strides let the lanes read a column without conflicts.
struct Subtree {
    int t, base, k0, L, n;
    __device__ int row(int i) const { return base + ((i + 1) << k0); }
};
__host__ __device__ inline int node_words(int m) { return m * ((m | 1) + (2 * m | 1)); }

// Start the copies of the subtree's matrices (Zg: [m][2m] per node; LIN: Linv too, its lower triangle
// where TRI).  Missing rows (c > s) are skipped; they are never read.
template <typename T, bool LIN, bool TRI>
__device__ __forceinline__ void fetch_subtree(const TreeArgs<T>& A, const T* Zbase, const Subtree& B, T* mats) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int m = A.m, ml = m | 1, mz = 2 * m | 1, nstr = node_words(m);
    for (int i = 0; i < B.n; ++i) {
        const int c = B.row(i);
        if (c > A.s) break;
        const T* Lg = A.linv(B.t, c);
        const T* Zg = Zbase + A.node(B.t, c) * 2 * m * m;
        T* Ls = mats + (size_t)i * nstr;
        T* Zs = Ls + m * ml;
        for (int r = warp; r < m; r += nw) {
            if (LIN && lane < (TRI ? r + 1 : m)) copy_async(Ls + r * ml + lane, Lg + r * m + lane);
            if (lane < 2 * m) copy_async(Zs + r * mz + lane, Zg + r * 2 * m + lane);
            if (lane + 32 < 2 * m) copy_async(Zs + r * mz + lane + 32, Zg + r * 2 * m + lane + 32);
        }
    }
}

// ---------------------------------------------------------------- up pass
// Heights k0 .. k0 + L - 1.  ga[dir][slot]: condensed loads of the subtree's rows that came from the
// segment above (dir 0) and below (dir 1), [slot][l][KB]; slot n is the row outside at the top (dir 1)
// and at the bottom (dir 0) of the subtree, handed to the next launch through Gtb[row][dir].  Two nodes
// of one height may feed the same row, but never the same direction of it.
template <typename T, bool TRI, int KB>
__global__ void __launch_bounds__(256) tree_up_kernel(SolveArgs<T> P, int k0, int L, const double* F, double fscale,
                                                      int r0) {
    extern __shared__ __align__(16) unsigned char ts_smem[];
    const TreeArgs<T>& A = P.tr;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int s = A.s, m = A.m, K = P.K;
    const Subtree B{(int)blockIdx.y, (int)blockIdx.x << (k0 + L), k0, L, (1 << L) - 1};
    const int SL = MAXM * KB;                               // words of one vector slot
    T* ga = reinterpret_cast<T*>(ts_smem);                  // [2][n + 1] slots
    T* vs = ga + (size_t)2 * (B.n + 1) * SL + (size_t)warp * SL;
    T* mats = ga + (size_t)(2 * (B.n + 1) + nw) * SL;
    fetch_subtree<T, true, TRI>(A, A.Ztb, B, mats);
    pdl_wait();
    pdl_trigger();
    const int64_t N = (int64_t)s * s;
    const int x0 = B.t * A.b + 1;
    for (int i = warp; i <= B.n; i += nw) {                 // loads of the rows; the outside slots start at 0
        const int c = i < B.n ? B.row(i) : s + 1;
        T g[KB], z[KB];
#pragma unroll
        for (int q = 0; q < KB; ++q) {
            T v = T(0);
            if (c <= s && lane < m && q < K) {
                v = (T)F[(int64_t)(r0 + q) * N + (int64_t)(c - 1) * s + (x0 - 1 + lane)] * (T)fscale;
                if (k0 > 0) {
                    v += P.gtb(B.t, c, 0, q)[lane];
                    if (c < s) v += P.gtb(B.t, c, 1, q)[lane];
                }
            }
            g[q] = v;
            z[q] = T(0);
        }
        stk<KB>(ga + (size_t)i * SL + lane * KB, g);
        stk<KB>(ga + (size_t)(B.n + 1 + i) * SL + lane * KB, z);
    }
    copy_async_wait();
    __syncthreads();
    const int ml = m | 1, mz = 2 * m | 1, nstr = node_words(m);
    for (int lv = 0; lv < L; ++lv) {
        const int k = k0 + lv;
        for (int i = ((2 * warp + 1) << lv) - 1; i < B.n; i += (2 * nw) << lv) {
            const int c = B.row(i);
            if (c > s) break;
            const T* Ls = mats + (size_t)i * nstr;
            const T* Zs = Ls + m * ml;
            {
                T a[KB], b[KB];
                ldk<KB>(ga + (size_t)i * SL + lane * KB, a);
                ldk<KB>(ga + (size_t)(B.n + 1 + i) * SL + lane * KB, b);
#pragma unroll
                for (int q = 0; q < KB; ++q) a[q] += b[q];
                __syncwarp();
                stk<KB>(vs + lane * KB, a);
                __syncwarp();
            }
            T y[KB];
#pragma unroll
            for (int q = 0; q < KB; ++q) y[q] = T(0);
            const int lr = lane < m ? lane : 0;
#pragma unroll 8
            for (int l = 0; l < m; ++l) {
                const T a = (!TRI || l <= lr) ? Ls[lr * ml + l] : T(0);
                T gv[KB];
                ldk<KB>(vs + l * KB, gv);
#pragma unroll
                for (int q = 0; q < KB; ++q) y[q] += a * gv[q];
            }
            __syncwarp();
            stk<KB>(vs + lane * KB, y);
#pragma unroll
            for (int q = 0; q < KB; ++q)
                if (lane < m && q < K) P.yv(B.t, c, q)[lane] = y[q];
            __syncwarp();
            const int ct = c - (1 << k), cb = c + (1 << k);
            if (ct <= 0 && cb > s) continue;                // the last node: nothing above or below
            T a0[KB], a1[KB];
#pragma unroll
            for (int q = 0; q < KB; ++q) a0[q] = a1[q] = T(0);
#pragma unroll 8
            for (int l = 0; l < m; ++l) {
                const T z0 = Zs[l * mz + lr], z1 = Zs[l * mz + m + lr];
                T yv[KB];
                ldk<KB>(vs + l * KB, yv);
#pragma unroll
                for (int q = 0; q < KB; ++q) {
                    a0[q] += z0 * yv[q];
                    a1[q] += z1 * yv[q];
                }
            }
            if (lane < m) {
                if (ct > 0) {
                    const int it = ct == B.base ? B.n : ((ct - B.base) >> k0) - 1;
                    T* p = ga + (size_t)(B.n + 1 + it) * SL + lane * KB;
#pragma unroll
                    for (int q = 0; q < KB; ++q) p[q] -= a0[q];
                }
                if (cb <= s) {
                    const int ib = ((cb - B.base) >> k0) - 1;    // n for the row outside
                    T* p = ga + (size_t)ib * SL + lane * KB;
#pragma unroll
                    for (int q = 0; q < KB; ++q) p[q] -= a1[q];
                }
            }
        }
        __syncthreads();
    }
    // the rows outside: above (dir 1) and below (dir 0), added to what lower heights left there
    for (int d = warp; d < 2; d += nw) {
        const int c = d ? B.base : B.base + (1 << (k0 + L));
        if (c < 1 || c > s || (d && B.row(0) > s)) continue;
        T a[KB];
        ldk<KB>(ga + (size_t)(d * (B.n + 1) + B.n) * SL + lane * KB, a);
#pragma unroll
        for (int q = 0; q < KB; ++q)
            if (lane < m && q < K) {
                T* p = P.gtb(B.t, c, d, q);
                p[lane] = (k0 > 0 ? p[lane] : T(0)) + a[q];
            }
    }
}

// Reduced load X[q][r][rr] = fscale f[r][rr][x_q] - sum over the slabs q (its right side) and q + 1 (its
// left side) and all heights of Z_I[:, rr]^T y(node of that height owning rr); padding rows zero.
// CTA = 32 interface nodes of one interface and KB loads; its 8 warps take the (slab, height) pairs in
// turn, lane = node, and add up in a fixed order at the end.  All loads of a pair are issued before its
// sums (bound by the bytes in flight).  KB > 1: the tile's nodes (16 / 2^k at height k < 4, else one) have
// their y staged in shared memory first.
constexpr int GL_WARPS = 8;
template <int KB>
__host__ __device__ constexpr int gl_buf() { return KB == 1 ? 32 : 16 * 33 * KB; }

template <typename T, int KB>
__global__ void __launch_bounds__(32 * GL_WARPS) gather_load_kernel(SolveArgs<T> P, const double* F, double fscale,
                                                                     int r0) {
    extern __shared__ __align__(16) unsigned char ts_smem[];
    constexpr int BUF = gl_buf<KB>();
    const TreeArgs<T>& A = P.tr;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T* ys = reinterpret_cast<T*>(ts_smem) + (size_t)warp * BUF;
    const int q0 = blockIdx.y, rg = blockIdx.z * KB;
    const int s = A.s, m = A.m, K = P.K;
    const int rr = blockIdx.x * 32 + lane, j = rr + 1;
    T acc[KB];
#pragma unroll
    for (int q = 0; q < KB; ++q) acc[q] = T(0);
    bool waited = false;
    for (int pr = warp; pr < 2 * A.H; pr += GL_WARPS) {
        const int k = pr >> 1, t = q0 + (pr & 1), side = (pr & 1) ? 0 : 1;
        const int c = (2 * (rr >> (k + 1)) + 1) << k;
        const bool own = rr < s && c <= s && (j & ((2 << k) - 1)) != 0;
        const T* zp = A.zi(t, k, side) + rr;
        T z[MAXM];                                         // of the factor: before the wait
#pragma unroll
        for (int i = 0; i < MAXM; ++i) z[i] = (own && i < m) ? zp[(int64_t)i * A.s_pad] : T(0);
        if (!waited) {
            pdl_wait();
            pdl_trigger();
            waited = true;
        }
        if constexpr (KB == 1) {
            const T* yp = P.yv(t, own ? c : 1, rg);
            T y[MAXM];
#pragma unroll
            for (int i = 0; i < MAXM; ++i) y[i] = (own && i < m) ? yp[i] : T(0);
#pragma unroll
            for (int i = 0; i < MAXM; ++i) acc[0] += z[i] * y[i];
        } else {
            const int nn = k < 4 ? 16 >> k : 1;            // nodes of this height in the tile
            const int a0 = (int)(blockIdx.x * 32) >> (k + 1);
            __syncwarp();
#pragma unroll 4
            for (int nd = 0; nd < nn; ++nd) {
                const int cn = (2 * (a0 + nd) + 1) << k;
                T v[KB];
#pragma unroll
                for (int q = 0; q < KB; ++q)
                    v[q] = (cn <= s && rg + q < K && lane < m) ? P.yv(t, cn, rg + q)[lane] : T(0);
                stk<KB>(ys + (nd * 33 + lane) * KB, v);
            }
            __syncwarp();
            const T* yl = ys + (nn > 1 ? (rr >> (k + 1)) - a0 : 0) * 33 * KB;
#pragma unroll
            for (int i = 0; i < MAXM; ++i) {
                T yv[KB];
                ldk<KB>(yl + i * KB, yv);
#pragma unroll
                for (int q = 0; q < KB; ++q) acc[q] += z[i] * yv[q];
            }
        }
    }
    if (!waited) {
        pdl_wait();
        pdl_trigger();
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < KB; ++q) ys[q * 32 + lane] = acc[q];
    __syncthreads();
    const int64_t N = (int64_t)s * s;
    const int xq = (q0 + 1) * A.b;
    for (int e = threadIdx.x; e < 32 * KB; e += 32 * GL_WARPS) {
        const int r = rg + (e >> 5), row = blockIdx.x * 32 + (e & 31);
        if (r >= K || row >= A.s_pad) continue;
        T v = T(0);
        if (row < s) {
            v = (T)(fscale * F[(int64_t)(r0 + r) * N + (int64_t)row * s + (xq - 1)]);
            T sum = T(0);
#pragma unroll
            for (int w = 0; w < GL_WARPS; ++w) sum += reinterpret_cast<const T*>(ts_smem)[(size_t)w * BUF + e];
            v -= sum;
        }
        P.xi(q0, r)[row] = v;
    }
}

// ---------------------------------------------------------------- down pass
// sum over interface columns [qa, qb) of one side (column index within the segment, rows lo..) of
// column * u, added to acc; u is staged 32 columns at a time.
template <typename T, int KB>
__device__ __forceinline__ void iface_cols(const SolveArgs<T>& P, const T* __restrict__ zd, int q, int rr0, int ncol,
                                           int rg, int lane, T* us, T (&acc)[KB]) {
    const int m = P.tr.m, K = P.K;
    for (int j0 = 0; j0 < ncol; j0 += 32) {
        const int nj = min(32, ncol - j0);
        __syncwarp();
        {
            T u[KB];
#pragma unroll
            for (int p = 0; p < KB; ++p) u[p] = (lane < nj && rg + p < K) ? P.xi(q, rg + p)[rr0 + j0 + lane] : T(0);
            stk<KB>(us + lane * KB, u);
        }
        __syncwarp();
        const T* z0 = zd + (int64_t)(rr0 + j0) * m + lane;
#pragma unroll
        for (int h = 0; h < 32; h += 16) {
            if (h >= nj) break;
            T z[16];
#pragma unroll
            for (int jj = 0; jj < 16; ++jj) z[jj] = (lane < m && h + jj < nj) ? z0[(h + jj) * m] : T(0);
#pragma unroll
            for (int jj = 0; jj < 16; ++jj) {
                T uv[KB];
                ldk<KB>(us + (h + jj) * KB, uv);
#pragma unroll
                for (int p = 0; p < KB; ++p) acc[p] += z[jj] * uv[p];
            }
        }
    }
}

// Partial interface sums of every node of height >= KSUM: one warp per (slab, slot, group of loads),
// slot = CW columns of one node's 2w (left side first).
template <typename T, int KB>
__global__ void __launch_bounds__(128) iface_sum_kernel(SolveArgs<T> P) {
    extern __shared__ __align__(16) unsigned char ts_smem[];
    const TreeArgs<T>& A = P.tr;
    pdl_wait();
    pdl_trigger();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T* us = reinterpret_cast<T*>(ts_smem) + warp * 32 * KB;
    const int slot = blockIdx.x * 4 + warp, t = blockIdx.y, rg = 0;
    if (slot >= P.vslots) return;
    int k = KSUM;
    while (k + 1 < A.H && slot >= P.voff[k + 1]) ++k;
    const int node = (slot - P.voff[k]) / P.vch[k], ch = (slot - P.voff[k]) % P.vch[k];
    const int c = (2 * node + 1) << k;
    const int lo = c - (1 << k) + 1, hi = min(A.s, c + (1 << k) - 1), w = hi - lo + 1;
    const int qa = ch * CW, qb = min(2 * w, qa + CW);
    T acc[KB];
#pragma unroll
    for (int p = 0; p < KB; ++p) acc[p] = T(0);
    if (t >= 1 && qa < w)
        iface_cols<T, KB>(P, A.zd(t, k, 0), t - 1, lo - 1 + qa, min(w, qb) - qa, rg, lane, us, acc);
    if (t < A.NS - 1 && qb > w)
        iface_cols<T, KB>(P, A.zd(t, k, 1), t, lo - 1 + max(qa - w, 0), qb - max(qa, w), rg, lane, us, acc);
#pragma unroll
    for (int p = 0; p < KB; ++p)
        if (lane < A.m && rg + p < P.K) P.vp(t, slot, rg + p)[lane] = acc[p];
}

// Heights k0 + L - 1 .. k0 (downwards) of one subtree, laid out as in tree_up_kernel.  First every node's
// y - (interface products), which need no x; then the recursion on the slots xv (slot n: the row outside
// at the top, n + 1: at the bottom).  Writes x of its rows into U -- with the row's node on the slab's right
// interface as entry m, so that a row's stores are one contiguous run -- and, for rows that later
// launches read (k0 > 0), into Xs.
template <typename T, bool INDEF, int KB>
__global__ void __launch_bounds__(256) tree_down_kernel(SolveArgs<T> P, int k0, int L, double* U, int accumulate,
                                                        int r0) {
    extern __shared__ __align__(16) unsigned char ts_smem[];
    const TreeArgs<T>& A = P.tr;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int s = A.s, m = A.m, K = P.K;
    const Subtree B{(int)blockIdx.y, (int)blockIdx.x << (k0 + L), k0, L, (1 << L) - 1};
    const int SL = MAXM * KB;
    T* xv = reinterpret_cast<T*>(ts_smem);                  // [n + 2] slots
    T* vs = xv + (size_t)(B.n + 2) * SL + (size_t)warp * SL;
    T* mats = xv + (size_t)(B.n + 2 + nw) * SL;
    fetch_subtree<T, !INDEF, true>(A, INDEF ? A.Wtb : A.Ztb, B, mats);
    pdl_wait();
    pdl_trigger();
    const int64_t N = (int64_t)s * s;
    const int t = B.t, x0 = t * A.b + 1;
    const int me = t < A.NS - 1 ? m + 1 : m;               // entries of a row written to U
    for (int i = warp; i < B.n + 2; i += nw) {
        const int c = i < B.n ? B.row(i) : (i == B.n ? B.base : B.base + (1 << (k0 + L)));
        T v[KB];
#pragma unroll
        for (int p = 0; p < KB; ++p) v[p] = T(0);
        if (i >= B.n) {
#pragma unroll
            for (int p = 0; p < KB; ++p)
                if (c >= 1 && c <= s && lane < m && p < K) v[p] = P.xs(t, c, p)[lane];
        } else if (c <= s) {
            const int k = k0 + __ffs(i + 1) - 1;
            const int lo = c - (1 << k) + 1, hi = min(s, c + (1 << k) - 1), w = hi - lo + 1;
            T y[KB];
#pragma unroll
            for (int p = 0; p < KB; ++p) y[p] = (lane < m && p < K) ? P.yv(t, c, p)[lane] : T(0);
            if (k < KSUM) {
                if (t >= 1) iface_cols<T, KB>(P, A.zd(t, k, 0), t - 1, lo - 1, w, 0, lane, vs, v);
                if (t < A.NS - 1) iface_cols<T, KB>(P, A.zd(t, k, 1), t, lo - 1, w, 0, lane, vs, v);
            } else {
                const int slot = P.voff[k] + (c >> (k + 1)) * P.vch[k], nch = (2 * w + CW - 1) / CW;
#pragma unroll 8
                for (int ch = 0; ch < nch; ++ch)
#pragma unroll
                    for (int p = 0; p < KB; ++p)
                        if (lane < m && p < K) v[p] += P.vp(t, slot + ch, p)[lane];
            }
#pragma unroll
            for (int p = 0; p < KB; ++p) v[p] = y[p] - v[p];
        }
        stk<KB>(xv + (size_t)i * SL + lane * KB, v);
    }
    copy_async_wait();
    __syncthreads();
    const int ml = m | 1, mz = 2 * m | 1, nstr = node_words(m);
    const int lr = lane < m ? lane : 0;
    for (int lv = L - 1; lv >= 0; --lv) {
        const int k = k0 + lv;
        for (int i = ((2 * warp + 1) << lv) - 1; i < B.n; i += (2 * nw) << lv) {
            const int c = B.row(i);
            if (c > s) break;
            const T* Ls = mats + (size_t)i * nstr;
            const T* Zs = Ls + m * ml;
            const int ct = c - (1 << k), cb = c + (1 << k);
            T v[KB];
            ldk<KB>(xv + (size_t)i * SL + lane * KB, v);
#pragma unroll
            for (int hb = 0; hb < 2; ++hb) {
                if (hb ? cb > s : ct <= 0) continue;
                const int ix = hb ? (cb == B.base + (1 << (k0 + L)) ? B.n + 1 : ((cb - B.base) >> k0) - 1)
                                  : (ct == B.base ? B.n : ((ct - B.base) >> k0) - 1);
                const T* xo = xv + (size_t)ix * SL;
                const T* zr = Zs + lr * mz + hb * m;
#pragma unroll 8
                for (int j = 0; j < m; ++j) {
                    const T z = zr[j];
                    T xj[KB];
                    ldk<KB>(xo + j * KB, xj);
#pragma unroll
                    for (int p = 0; p < KB; ++p) v[p] -= z * xj[p];
                }
            }
            if (!INDEF) {                                  // x_i = sum_{l >= i} Linv[l][i] v_l
                __syncwarp();
                stk<KB>(vs + lane * KB, v);
                __syncwarp();
#pragma unroll
                for (int p = 0; p < KB; ++p) v[p] = T(0);
#pragma unroll 8
                for (int l = 0; l < m; ++l) {
                    const T a = lr <= l ? Ls[l * ml + lr] : T(0);
                    T vv[KB];
                    ldk<KB>(vs + l * KB, vv);
#pragma unroll
                    for (int p = 0; p < KB; ++p) v[p] += a * vv[p];
                }
            }
            if (lane < m) stk<KB>(xv + (size_t)i * SL + lane * KB, v);
#pragma unroll
            for (int p = 0; p < KB; ++p) {
                if (p >= K) continue;
                if (k0 > 0 && lane < m) P.xs(t, c, p)[lane] = v[p];
                double* up = U + (int64_t)(r0 + p) * N + (int64_t)(c - 1) * s + (x0 - 1);
                if (lane < m) {
                    if (accumulate) up[lane] += (double)v[p];
                    else up[lane] = (double)v[p];
                }
                const int li = lane < m ? lane + 32 : lane;        // the interface entry: lane m (m = 32: lane 0)
                if (li == m && m < me) {
                    const double xi = (double)P.xi(t, p)[c - 1];
                    if (accumulate) up[m] += xi;
                    else up[m] = xi;
                }
            }
        }
        __syncthreads();
    }
}

// [i][rr] -> [rr][i] of every (slab, height, side) block; CTA = 32 interface nodes of one block
template <typename T>
__global__ void __launch_bounds__(128) node_major_kernel(const T* __restrict__ Z, T* __restrict__ ZD, int m, int s,
                                                         int s_pad) {
    __shared__ T tile[MAXM][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t blk = (int64_t)blockIdx.y * m * s_pad;
    const int rr0 = blockIdx.x * 32;
    for (int i = warp; i < m; i += 4) tile[i][lane] = Z[blk + (int64_t)i * s_pad + rr0 + lane];
    __syncthreads();
    for (int e = threadIdx.x; e < 32 * m; e += 128) {
        const int r = e / m, i = e % m;
        if (rr0 + r < s) ZD[blk + (int64_t)(rr0 + r) * m + i] = tile[i][r];
    }
}

// ftilde (FP64, [k][q][j]) <-> X (scalar, [q][j][r])
template <typename T>
__global__ void export_x_kernel(SolveArgs<T> P, double* out, double scale, int NI, int r0) {
    const TreeArgs<T>& A = P.tr;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t per = (int64_t)NI * A.s;
    if (idx >= per * P.K) return;
    const int r = (int)(idx / per);
    const int64_t rem = idx % per;
    const int q = (int)(rem / A.s), rr = (int)(rem % A.s);
    out[(int64_t)(r0 + r) * per + rem] = scale * (double)P.xi(q, r)[rr];
}
template <typename T>
__global__ void import_x_kernel(SolveArgs<T> P, const double* in, int NI, int r0) {
    const TreeArgs<T>& A = P.tr;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t per = (int64_t)NI * A.s_pad;
    if (idx >= per * P.K) return;
    const int r = (int)(idx / per);
    const int64_t rem = idx % per;
    const int q = (int)(rem / A.s_pad), rr = (int)(rem % A.s_pad);
    P.xi(q, r)[rr] = rr < A.s ? (T)in[(int64_t)(r0 + r) * NI * A.s + (int64_t)q * A.s + rr] : T(0);
}

// ---------------------------------------------------------------- host side

// Partial-sum slots of the down pass: heights KSUM.., ceil(2 w / CW) per node (w of a full segment).
int partial_slots(int s, int H, int* off, int* per) {
    int n = 0;
    for (int k = 0; k < H; ++k) {
        const int wmax = std::min(s, (1 << (k + 1)) - 1);
        const int nch = k < KSUM ? 0 : (2 * wmax + CW - 1) / CW;
        if (off) off[k] = n;
        if (per) per[k] = nch;
        n += nch * tree_nodes_at(s, k);
    }
    return n;
}

template <typename T>
SolveArgs<T> make_solve_args(slab_handle* h, int K) {
    SolveArgs<T> p{};
    p.tr = make_tree_args<T>(h);
    p.K = K; p.kcap = h->kcap;
    p.Yv = (T*)h->wYv; p.Gtb = (T*)h->wGtb; p.Xs = (T*)h->wXs; p.X = (T*)h->wX; p.Vp = (T*)h->wVp;
    p.vslots = partial_slots(p.tr.s, p.tr.H, p.voff, p.vch);
    return p;
}

// Heights [k0, k0 + L) of each launch, bottom up: the last one takes as many heights as fit in
// TOP_SMEM, those below as many as fit in LOW_SMEM, shared out evenly.
template <typename T>
size_t subtree_smem(int L, int m, int KB, int nw) {
    const int n = (1 << L) - 1;
    return ((size_t)(2 * (n + 1) + nw) * MAXM * KB + (size_t)n * node_words(m)) * sizeof(T);
}
inline int group_warps(int L) { return L >= 4 ? 8 : 4; }
template <typename T>
int height_groups(int H, int m, int KB, int (*grp)[2]) {
    int top = 1, low = 1;
    while (top < H && top < 7 && subtree_smem<T>(top + 1, m, KB, group_warps(top + 1)) <= TOP_SMEM) ++top;
    while (low < 6 && subtree_smem<T>(low + 1, m, KB, group_warps(low + 1)) <= LOW_SMEM) ++low;
    const int rest = H - top, ng = (rest + low - 1) / low;
    int n = 0, k = 0;
    for (int i = 0; i < ng; ++i) {
        const int len = (rest - k + (ng - i) - 1) / (ng - i);
        grp[n][0] = k;
        grp[n++][1] = len;
        k += len;
    }
    grp[n][0] = k;
    grp[n++][1] = H - k;
    return n;
}

// Opt a kernel in to the largest dynamic shared memory once per device (idempotent, any thread).
template <auto Kern>
slab_status opt_in_smem(slab_handle* h, size_t bytes) {
    static std::atomic<uint32_t> done(0);
    if (bytes <= 48 * 1024) return SLAB_OK;
    int dev = 0;
    SLAB_CK(h, cudaGetDevice(&dev));
    const uint32_t bit = 1u << (dev & 31);
    if (done.load(std::memory_order_acquire) & bit) return SLAB_OK;
    SLAB_CK(h, cudaFuncSetAttribute(Kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    done.fetch_or(bit, std::memory_order_acq_rel);
    return SLAB_OK;
}

template <typename T, bool INDEF, int KB>
slab_status up_gather_kb(slab_handle* h, const double* F, double fscale, int r0, int K) {
    const SolveArgs<T> p = make_solve_args<T>(h, K);
    const TreeDims& d = h->td;
    int grp[MAXH][2];
    const int ng = height_groups<T>(d.H, d.m, KB, grp);
    slab_status st;
    for (int i = 0; i < ng; ++i) {
        const int k0 = grp[i][0], L = grp[i][1], nw = group_warps(L);
        const size_t smem = subtree_smem<T>(L, d.m, KB, nw);
        if ((st = opt_in_smem<tree_up_kernel<T, !INDEF, KB>>(h, smem))) return st;
        const int ranges = (d.s + (1 << (k0 + L)) - 1) >> (k0 + L);
        SLAB_PROF(h, KC_TREE_UP);
        SLAB_CK(h, launch_pdl(tree_up_kernel<T, !INDEF, KB>, dim3(ranges, d.NS), dim3(32 * nw), smem, h->stream, p, k0,
                              L, F, fscale, r0));
    }
    constexpr int KG = KB < 4 ? KB : 4;                    // loads per CTA of the reduced load
    const size_t smem = (size_t)GL_WARPS * gl_buf<KG>() * sizeof(T);
    if ((st = opt_in_smem<gather_load_kernel<T, KG>>(h, smem))) return st;
    SLAB_PROF(h, KC_TREE_UP);
    SLAB_CK(h, launch_pdl(gather_load_kernel<T, KG>, dim3(d.s_pad / 32, d.NI, (K + KG - 1) / KG), dim3(32 * GL_WARPS),
                          smem, h->stream, p, F, fscale, r0));
    return SLAB_OK;
}

template <typename T, bool INDEF, int KB>
slab_status down_scatter_kb(slab_handle* h, double* U, int accumulate, int r0, int K) {
    const SolveArgs<T> p = make_solve_args<T>(h, K);
    const TreeDims& d = h->td;
    slab_status st;
    if (p.vslots > 0) {
        SLAB_PROF(h, KC_TREE_DOWN);
        SLAB_CK(h, launch_pdl(iface_sum_kernel<T, KB>, dim3((p.vslots + 3) / 4, d.NS), dim3(128),
                              4 * 32 * KB * sizeof(T), h->stream, p));
    }
    int grp[MAXH][2];
    for (int i = height_groups<T>(d.H, d.m, KB, grp) - 1; i >= 0; --i) {
        const int k0 = grp[i][0], L = grp[i][1], nw = group_warps(L);
        const size_t smem = subtree_smem<T>(L, d.m, KB, nw);
        if ((st = opt_in_smem<tree_down_kernel<T, INDEF, KB>>(h, smem))) return st;
        const int ranges = (d.s + (1 << (k0 + L)) - 1) >> (k0 + L);
        SLAB_PROF(h, KC_TREE_DOWN);
        SLAB_CK(h, launch_pdl(tree_down_kernel<T, INDEF, KB>, dim3(ranges, d.NS), dim3(32 * nw), smem, h->stream, p, k0,
                              L, U, accumulate, r0));
    }
    return SLAB_OK;
}

inline bool general_kind(const slab_handle* h) { return h->kind == SLAB_HELMHOLTZ || h->kind == SLAB_CONVECTION; }

}  // namespace

// Up pass over all heights for right-hand sides [r0, r0+K) of F (FP64, [k][N]) scaled by fscale,
// then the reduced load f~ into X.
template <typename T>
slab_status tree_up_gather(slab_handle* h, const double* F, double fscale, int r0, int K) {
    if (K > SOLVE_NARROW) return tree_up_wide<T>(h, F, fscale, r0, K);
#define UP(KB) (general_kind(h) ? up_gather_kb<T, true, KB>(h, F, fscale, r0, K) : up_gather_kb<T, false, KB>(h, F, fscale, r0, K))
    return K <= 1 ? UP(1) : (K <= 4 ? UP(4) : UP(8));
#undef UP
}

template <typename T>
slab_status tree_down_scatter(slab_handle* h, double* U, int accumulate, int r0, int K) {
    if (K > SOLVE_NARROW) return tree_down_wide<T>(h, U, accumulate, r0, K);
#define DOWN(KB) \
    (general_kind(h) ? down_scatter_kb<T, true, KB>(h, U, accumulate, r0, K) : down_scatter_kb<T, false, KB>(h, U, accumulate, r0, K))
    return K <= 1 ? DOWN(1) : (K <= 4 ? DOWN(4) : DOWN(8));
#undef DOWN
}

// The node-major copies of the interface columns that the down pass reads, at the end of the tree factor.
template <typename T>
slab_status tree_node_major(slab_handle* h) {
    const TreeDims& d = h->td;
    const dim3 grid(d.s_pad / 32, d.NS * d.H * 2);
    SLAB_PROF(h, KC_TREE_FACTOR);
    node_major_kernel<T><<<grid, 128, 0, h->stream>>>((const T*)(general_kind(h) ? h->tWI : h->tZI), (T*)h->tZD, d.m,
                                                      d.s, d.s_pad);
    SLAB_CK_LAUNCH(h);
    if (h->kind == SLAB_CONVECTION) {
        node_major_kernel<T><<<grid, 128, 0, h->stream>>>((const T*)h->tWIT, (T*)h->tZDT, d.m, d.s, d.s_pad);
        SLAB_CK_LAUNCH(h);
        prof_extra(h, KC_TREE_FACTOR, 1);
    }
    return SLAB_OK;
}

template <typename T>
slab_status export_ftilde_part(slab_handle* h, double* out, double scale, int r0, int K) {
    SolveArgs<T> p = make_solve_args<T>(h, K);
    const int64_t tot = (int64_t)h->td.NI * h->td.s * K;
    SLAB_PROF(h, KC_OTHER);
    export_x_kernel<T><<<(unsigned)((tot + 255) / 256), 256, 0, h->stream>>>(p, out, scale, h->td.NI, r0);
    SLAB_CK_LAUNCH(h);
    return SLAB_OK;
}

template <typename T>
slab_status import_utilde_part(slab_handle* h, const double* in, int r0, int K) {
    SolveArgs<T> p = make_solve_args<T>(h, K);
    const int64_t tot = (int64_t)h->td.NI * h->td.s_pad * K;
    SLAB_PROF(h, KC_OTHER);
    import_x_kernel<T><<<(unsigned)((tot + 255) / 256), 256, 0, h->stream>>>(p, in, h->td.NI, r0);
    SLAB_CK_LAUNCH(h);
    return SLAB_OK;
}

int tree_kmax() { return KMAX; }

// Elements of the down pass's partial interface sums.
size_t tree_partial_elems(int s, int m, int NS) {
    return (size_t)partial_slots(s, tree_height_count(s), nullptr, nullptr) * NS * SOLVE_NARROW * m;
}

#define INSTANTIATE(T)                                                                                 \
    template slab_status tree_up_gather<T>(slab_handle*, const double*, double, int, int);             \
    template slab_status tree_down_scatter<T>(slab_handle*, double*, int, int, int);                   \
    template slab_status tree_node_major<T>(slab_handle*);                                             \
    template slab_status export_ftilde_part<T>(slab_handle*, double*, double, int, int);               \
    template slab_status import_utilde_part<T>(slab_handle*, const double*, int, int);
INSTANTIATE(float)
INSTANTIATE(double)
