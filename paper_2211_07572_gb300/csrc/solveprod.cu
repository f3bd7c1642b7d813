// Products of the solve phases with few right-hand sides: C = alpha (A B^T + A' B'^T) + beta C, A (M x K) a stored factor
// block, B (N x K) the vectors, FP32, N <= 32, batched; the second term is optional.
//
// A product streams A once (up to 330 MB) and is otherwise one link in a chain of dependent products of
// a few microseconds each, so both the bytes in flight and the latency of a launch count.  Neither
// kernel has barriers or staging in its main loop: every warp loads its part of A straight into registers
// -- the first loads before the wait on the preceding launch, which A does not depend on -- and the K
// range is split over the warps of a CTA, whose sums meet in shared memory once.  A step of the odd-even solve
// multiplies by both neighbours' blocks in one launch: n = 777, 5 loads: 28 launches an interface solve instead of
// 36, factor + solve 9.31 -> 9.11 ms; n = 512 factor + solve + adjoint 5.37 -> 5.27 ms.
//   N <= 4: FP32 multiply-adds, a warp one to four whole rows.
//   N <= 32: 3xTF32 (hi hi + hi lo + lo hi, as the tcgen05 product) on warp-level MMAs, whose operands come from
// registers.  The tcgen05 path needs A in shared memory twice (hi and lo), a conversion pass and a TMEM round
// trip per 128-row tile: 3-D n = 64, b = 8, 16 loads 2.4 ms of products a pass for 4.8 GB (2 TB/s).
#include <algorithm>

#include "slab_internal.cuh"

namespace {

__device__ __forceinline__ float4 ld4g(const float* p) { return *reinterpret_cast<const float4*>(p); }
constexpr float4 ZERO4 = {0.f, 0.f, 0.f, 0.f};

// c + alpha v of every term the element has, rounded term by term: the same bits as one launch a term
template <int TERMS>
__device__ __forceinline__ float add_terms(float c, float alpha, const float (&v)[TERMS], const bool (&has)[TERMS]) {
#pragma unroll
    for (int q = 0; q < TERMS; ++q)
        if (has[q]) c = c + alpha * v[q];
    return c;
}

// ---------------------------------------------------------------- N <= 4
// Warp = R rows of A; lanes over K, U float4 a lane and row in flight.  triA: 1 lower, 2 upper triangular.
//   rows_ctas: CTAs that share an SM, whose loads in flight hide each other's latency.  Without the bound one term and
// four loads take 222 registers, one CTA; two terms with U = 8 spill.  Two refinement passes: 3-D n = 64, b = 8, 4 loads 5.39 ms,
// 6.19 without the bounds and with U = 8; n = 35, b = 7, 3 loads 1.71 and 2.09 ms.
constexpr int rows_ctas(int terms, int nb) { return terms == 2 ? 2 : (nb == 1 ? 4 : 3); }
template <int TERMS, int R, int U, int NB>
__global__ void __launch_bounds__(256, rows_ctas(TERMS, NB))
    rows_nt_kernel(int M, int N, int K, float alpha, ProdTerms P, int64_t lda, int64_t sA, int64_t ldb, int64_t sB,
                   float beta, float* C, int64_t ldc, int64_t sC, int transC, int triA) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row0 = (blockIdx.x * 8 + warp) * R, bt = blockIdx.y;
    C += (int64_t)bt * sC;
    const int last = min(row0 + R, M) - 1;                     // last row of the warp
    int k0 = 0, k1 = K;
    if (triA == 1) k1 = min(K, (last + 4) & ~3);
    if (triA == 2) k0 = min(row0, M - 1) & ~3;
    float acc[TERMS][R][NB];                                   // a sum per term: C takes them one after another
#pragma unroll
    for (int q = 0; q < TERMS; ++q)
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int n = 0; n < NB; ++n) acc[q][r][n] = 0.f;
    bool has[TERMS];                                           // (one term: every element has it)
#pragma unroll
    for (int q = 0; q < TERMS; ++q) has[q] = TERMS == 1 || (bt >= P.lo[q] && bt < P.hi[q]);
    const float* Am[TERMS];
#pragma unroll
    for (int q = 0; q < TERMS; ++q) Am[q] = P.A[q] + (int64_t)bt * sA;
    int64_t ro[R];
#pragma unroll
    for (int r = 0; r < R; ++r) ro[r] = (int64_t)min(row0 + r, M - 1) * lda;
    float4 a[TERMS][R][U];
    auto load = [&](int term, int kb) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int k = kb + 128 * u + 4 * lane;
#pragma unroll
            for (int r = 0; r < R; ++r) a[term][r][u] = k < k1 ? ld4g(Am[term] + ro[r] + k) : ZERO4;
        }
    };
#pragma unroll
    for (int term = 0; term < TERMS; ++term)
        if (has[term]) load(term, k0);
    pdl_wait();
    pdl_trigger();
#pragma unroll
    for (int term = 0; term < TERMS; ++term) {
        if (!has[term]) continue;
        const float* B = P.B[term] + (int64_t)bt * sB;
        for (int kb = k0; kb < k1; kb += 128 * U) {
            if (kb > k0) load(term, kb);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int k = kb + 128 * u + 4 * lane;
#pragma unroll
                for (int n = 0; n < NB; ++n) {
                    const float4 b = (n < N && k < k1) ? ld4g(B + (int64_t)n * ldb + k) : ZERO4;
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const float4 v = a[term][r][u];
                        float& s = acc[term][r][n];
                        s = fmaf(v.x, b.x, fmaf(v.y, b.y, fmaf(v.z, b.z, fmaf(v.w, b.w, s))));
                    }
                }
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int n = 0; n < NB; ++n) {
            float v[TERMS];
#pragma unroll
            for (int q = 0; q < TERMS; ++q) {
                v[q] = acc[q][r][n];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
            }
            const int row = row0 + r;
            if (lane == n && n < N && row < M) {
                float* c = transC ? C + (int64_t)n * ldc + row : C + (int64_t)row * ldc + n;
                *c = add_terms<TERMS>(beta == 0.f ? 0.f : beta * *c, alpha, v, has);
            }
        }
}

// ---------------------------------------------------------------- 5 <= N <= 32
// x rounded to TF32 (nearest, ties away) on the integer pipe: the conversion unit does 16 values a cycle, which
// would bound the whole product
__device__ __forceinline__ uint32_t tf32_hi(float x) { return (__float_as_uint(x) + 0x1000u) & 0xffffe000u; }
__device__ __forceinline__ void mma_m16n8k8(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// CTA = 16 MT rows, 8 warps; warp w takes the K chunks w, w + 8, ... of CK.  Thread (g, t) = (lane / 4, lane % 4)
// holds float4s A[g (+ 8)][k + 4 t ..] and B[g][k + 4 t ..] of 16 K values: .x, .y are its entries of one
// m16n8k8 step and .z, .w of the next (the order of K within a step is free as long as A and B agree).
template <int TERMS, int MT, int NT>
__global__ void __launch_bounds__(256, 2) stream_nt_kernel(int M, int N, int K, float alpha, ProdTerms P, int64_t lda,
                                                           int64_t sA, int64_t ldb, int64_t sB, float beta, float* C,
                                                           int64_t ldc, int64_t sC, int transC, int triA) {
    constexpr int S = MT == 1 && NT <= 2 ? 4 : 2;              // 16-wide steps of a chunk, loaded together
    constexpr int CK = 16 * S;
    constexpr int RP = 16 * MT + 1;
    __shared__ float red[8][8 * NT][RP];                       // [warp][n][row]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int row0 = blockIdx.x * 16 * MT, bt = blockIdx.y;
    C += (int64_t)bt * sC;
    int k0 = 0, k1 = K;
    if (triA == 1) k1 = min(K, row0 + 16 * MT);
    if (triA == 2) k0 = row0;                                  // (multiples of 16, as K)
    float acc[MT][NT][4];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[mt][nt][q] = 0.f;
    bool has[TERMS];                                           // (one term: every element has it)
#pragma unroll
    for (int q = 0; q < TERMS; ++q) has[q] = TERMS == 1 || (bt >= P.lo[q] && bt < P.hi[q]);
    const float* Am[TERMS];
#pragma unroll
    for (int q = 0; q < TERMS; ++q) Am[q] = P.A[q] + (int64_t)bt * sA + 4 * t;
    int64_t bo[NT];                                            // (rows beyond N repeat the last: not written)
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) bo[nt] = (int64_t)min(8 * nt + g, N - 1) * ldb;
    int64_t ro[MT][2];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) ro[mt][hf] = (int64_t)min(row0 + 16 * mt + 8 * hf + g, M - 1) * lda;
    float4 av[TERMS][S][MT][2];
    auto load_a = [&](int term, int kc) {
        const bool full = kc + CK <= k1;
#pragma unroll
        for (int s = 0; s < S; ++s)
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int hf = 0; hf < 2; ++hf)
                    av[term][s][mt][hf] = full || kc + 16 * s < k1 ? ld4g(Am[term] + ro[mt][hf] + kc + 16 * s) : ZERO4;
    };
    const int kfirst = k0 + warp * CK;
#pragma unroll
    for (int term = 0; term < TERMS; ++term)
        if (has[term] && kfirst < k1) load_a(term, kfirst);
    pdl_wait();
    pdl_trigger();
#pragma unroll
    for (int term = 0; term < TERMS; ++term) {
        if (!has[term]) continue;
        const float* bp = P.B[term] + (int64_t)bt * sB + 4 * t;
        for (int kc = kfirst; kc < k1; kc += 8 * CK) {
            float4 bv[S][NT];
#pragma unroll
            for (int s = 0; s < S; ++s)
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) bv[s][nt] = kc + 16 * s < k1 ? ld4g(bp + bo[nt] + kc + 16 * s) : ZERO4;
            if (kc > kfirst) load_a(term, kc);
#pragma unroll
            for (int s = 0; s < S; ++s)
#pragma unroll
                for (int st = 0; st < 2; ++st) {
                    uint32_t ah[MT][4], al[MT][4];
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt) {
                        const float4 lo = av[term][s][mt][0], hi = av[term][s][mt][1];
                        const float e[4] = {st ? lo.z : lo.x, st ? hi.z : hi.x, st ? lo.w : lo.y, st ? hi.w : hi.y};
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            ah[mt][q] = tf32_hi(e[q]);
                            al[mt][q] = __float_as_uint(e[q] - __uint_as_float(ah[mt][q]));
                        }
                    }
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) {
                        const float4 b = bv[s][nt];
                        const float x = st ? b.z : b.x, y = st ? b.w : b.y;
                        const uint32_t xh = tf32_hi(x), yh = tf32_hi(y);
                        const uint32_t xl = __float_as_uint(x - __uint_as_float(xh)), yl = __float_as_uint(y - __uint_as_float(yh));
#pragma unroll
                        for (int mt = 0; mt < MT; ++mt) {
                            mma_m16n8k8(acc[mt][nt], ah[mt], xh, yh);
                            mma_m16n8k8(acc[mt][nt], ah[mt], xl, yl);
                            mma_m16n8k8(acc[mt][nt], al[mt], xh, yh);
                        }
                    }
                }
        }
    }
    // sums of the warps' K ranges, in warp order
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                red[warp][8 * nt + 2 * t + (q & 1)][16 * mt + g + (q >= 2 ? 8 : 0)] = acc[mt][nt][q];
    __syncthreads();
    for (int e = threadIdx.x; e < 16 * MT * N; e += 256) {
        const int n = e / (16 * MT), r = e % (16 * MT), row = row0 + r;
        if (row >= M) continue;
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) v += red[w][n][r];
        float* c = transC ? C + (int64_t)n * ldc + row : C + (int64_t)row * ldc + n;
        *c = (beta == 0.f ? 0.f : beta * *c) + alpha * v;
    }
}

}  // namespace

bool solve_product_ok(int N, int K, const float* A, int64_t lda, int64_t sA, const float* B, int64_t ldb, int64_t sB) {
    return N >= 1 && N <= 32 && K > 0 && K % 16 == 0 && lda % 4 == 0 && ldb % 4 == 0 && sA % 4 == 0 && sB % 4 == 0 &&
           ((uintptr_t)A & 15) == 0 && ((uintptr_t)B & 15) == 0;
}

// The number of rows a warp (a CTA) takes grows with the work, as long as every SM keeps a few CTAs: more rows
// read B less often.  Two terms hold the first loads of both before the wait; the 32-row warps of 17 to 32
// loads have no registers for that.
template <int TERMS>
static slab_status launch_products(slab_handle* h, int M, int N, int K, float alpha, const ProdTerms& P, int64_t lda,
                                   int64_t sA, int64_t ldb, int64_t sB, float beta, float* C, int64_t ldc, int64_t sC,
                                   int transC, int triA, int batch) {
    auto go = [&](auto kernel, int rows_per_cta) -> cudaError_t {
        return launch_pdl(kernel, dim3((unsigned)((M + rows_per_cta - 1) / rows_per_cta), (unsigned)batch), dim3(256), 0,
                          h->stream, M, N, K, alpha, P, lda, sA, ldb, sB, beta, C, ldc, sC, transC, triA);
    };
    const int64_t rows = (int64_t)M * batch;
    cudaError_t e;
    if (N == 1) e = rows >= 32 * 4 * SMS ? go(rows_nt_kernel<TERMS, 4, 2, 1>, 32) : go(rows_nt_kernel<TERMS, 1, 8, 1>, 8);
    else if (N <= 4)
        e = rows >= 32 * 4 * SMS ? go(rows_nt_kernel<TERMS, 4, 2, 4>, 32)
                                 : go(rows_nt_kernel<TERMS, 1, TERMS == 2 ? 4 : 8, 4>, 8);
    else if (N <= 8) e = rows >= 32 * 2 * SMS ? go(stream_nt_kernel<TERMS, 2, 1>, 32) : go(stream_nt_kernel<TERMS, 1, 1>, 16);
    else if (N <= 16) e = rows >= 32 * 2 * SMS ? go(stream_nt_kernel<TERMS, 2, 2>, 32) : go(stream_nt_kernel<TERMS, 1, 2>, 16);
    else if (TERMS == 1 && rows >= 32 * 2 * SMS) e = go(stream_nt_kernel<1, 2, 4>, 32);
    else e = go(stream_nt_kernel<TERMS, 1, 4>, 16);
    SLAB_CK(h, e);
    return SLAB_OK;
}

slab_status solve_product(slab_handle* h, int M, int N, int K, float alpha, const float* A, int64_t lda, int64_t sA,
                          const float* B, int64_t ldb, int64_t sB, float beta, float* C, int64_t ldc, int64_t sC,
                          int transC, int triA, int batch) {
    if (M <= 0) return SLAB_OK;
    for (int b0 = 0; b0 < batch; b0 += 65535) {
        const int nb = std::min(65535, batch - b0);
        const ProdTerms P = {{A + b0 * sA, nullptr}, {B + b0 * sB, nullptr}, {0, 0}, {nb, 0}};
        const slab_status st =
            launch_products<1>(h, M, N, K, alpha, P, lda, sA, ldb, sB, beta, C + b0 * sC, ldc, sC, transC, triA, nb);
        if (st) return st;
    }
    return SLAB_OK;
}

slab_status solve_product_pair(slab_handle* h, int M, int N, int K, float alpha, const ProdTerms& P, int64_t lda, int64_t sA,
                               int64_t ldb, int64_t sB, float beta, float* C, int64_t ldc, int64_t sC, int transC,
                               int batch) {
    if (M <= 0 || batch <= 0) return SLAB_OK;
    if (batch > 65535) return SLAB_EINVAL;
    return launch_products<2>(h, M, N, K, alpha, P, lda, sA, ldb, sB, beta, C, ldc, sC, transC, 0, batch);
}
