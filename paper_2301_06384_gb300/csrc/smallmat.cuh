// Dense M x M matrices (M <= 128) in shared memory, one CTA: blocked Cholesky, blocked inverse
// of a triangular matrix, products of triangular matrices.
//
// One SM works on these, so their time is latency: barriers, dependent operations, and FP64
// operations above all (two FMAs per clock and SM on this part).  Blocks of 16: a diagonal block
// is factored by one warp in registers, with no barrier, and the same instructions give the
// inverse of its factor; everything else is products of 16 or more independent terms over all
// threads, in 2 x 2 register tiles, a warp's lanes along the columns.  Rows are lda elements
// apart, lda even (pairs of elements are loaded at once).
#pragma once
#include "kb_internal.cuh"

namespace kb {
namespace sm {

constexpr int NB = 16;   // block edge

template <typename S> struct Pair;
template <> struct Pair<float> { using type = float2; };
template <> struct Pair<double> { using type = double2; };
template <typename S>
__device__ __forceinline__ void ld2(const S *p, S (&v)[2]) {
    const typename Pair<S>::type t = *reinterpret_cast<const typename Pair<S>::type *>(p);
    v[0] = t.x;
    v[1] = t.y;
}

// 1/d for a positive double d by Newton's iteration for the reciprocal, r <- r + r (1 - d r),
// from the single-precision reciprocal: two steps take its 2^-23 relative error to the
// FP64 rounding level (the error squares at each step).  The FP64 division it replaces is
// a long dependent sequence on this part's FP64 unit; this is four FMAs.  Outside the
// normal single-precision range the division is used.
__device__ __forceinline__ double recip(double d) {
    if (!(d > 1e-36 && d < 1e36)) return 1.0 / d;
    double r = double(__frcp_rn(float(d)));
    double e = fma(-d, r, 1.0);
    r = fma(r, e, r);
    e = fma(-d, r, 1.0);
    return fma(r, e, r);
}
__device__ __forceinline__ float recip(float d) { return __frcp_rn(d); }

// 2 x 2 tiles (i0, j0) of the rows [0, R) and columns [0, C): a warp takes rows i0, i0 + 1 and
// its lanes the column pairs (several row pairs per warp when the columns are few).
template <typename F>
__device__ __forceinline__ void tiles2(int R, int C, const F &f) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int cp = (C + 1) / 2;
    int lpr = 32;                       // lanes per row pair
    while (lpr > 1 && lpr / 2 >= cp) lpr /= 2;
    const int rpw = 32 / lpr;
    for (int i = (warp * rpw + lane / lpr) * 2; i < R; i += nw * rpw * 2)
        for (int j = (lane % lpr) * 2; j < C; j += lpr * 2) f(i, j);
}

// Cholesky G = R^T R: the upper triangle of A holds G on entry and R on return.  Inv (ld lda,
// or nullptr) receives the inverses of R's NB x NB diagonal blocks (upper triangular, zeros
// below).  Returns false (all threads) on a pivot (diagonal entry of the Schur complement) not
// above thr.  scr: NB * NB elements.
template <typename S>
__device__ bool chol_blocked(S *A, S *Inv, int lda, int M, S thr, S *scr) {
    __shared__ int s_bad;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_bad = 0;
    __syncthreads();
    for (int j0 = 0; j0 < M; j0 += NB) {
        const int nb = min(NB, M - j0);
        if (warp == 0) {
            // lanes 0..15: the columns of the diagonal block; lanes 16..31: those of I, on which
            // the same row operations leave R^{-T}
            const int c = lane & (NB - 1);
            const bool inv = lane >= NB;
            S a[NB];
#pragma unroll
            for (int i = 0; i < NB; ++i)
                a[i] = (!inv && i < nb && c < nb) ? (i <= c ? A[(j0 + i) * lda + j0 + c] : S(0)) : S(i == c ? 1 : 0);
            bool bad = false;
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                S d = __shfl_sync(0xffffffffu, a[j], j);
                if (j < nb && !(d > thr)) {
                    bad = true;
                    d = S(1);
                }
                const S r = sqrt(d);
                const S ri = recip(r);
                a[j] = (!inv && c == j) ? r : a[j] * ri;
#pragma unroll
                for (int i = j + 1; i < NB; ++i) {
                    const S rji = __shfl_sync(0xffffffffu, a[j], i);
                    a[i] = fma(-rji, a[j], a[i]);
                }
            }
            if (bad && lane == 0) s_bad = 1;
#pragma unroll
            for (int i = 0; i < NB; ++i) {
                if (inv) scr[i * NB + c] = a[i];                  // R^{-T}, lower triangular
                if (i < nb && c < nb) {
                    if (!inv) A[(j0 + i) * lda + j0 + c] = i <= c ? a[i] : S(0);
                    else if (Inv) Inv[(j0 + c) * lda + j0 + i] = i >= c ? a[i] : S(0);
                }
            }
        }
        __syncthreads();
        if (s_bad) return false;
        const int c0 = j0 + nb, rest = M - c0;
        if (rest <= 0) break;
        // R_12 = R_11^{-T} A_12: four lanes per column, each every fourth row
        for (int g0 = 0; g0 < rest; g0 += int(blockDim.x) / 4) {
            const int g = g0 + int(threadIdx.x) / 4, q = threadIdx.x & 3;
            S x[NB], y[NB / 4];
#pragma unroll
            for (int k = 0; k < NB; ++k) x[k] = g < rest ? A[(j0 + k) * lda + c0 + g] : S(0);
            __syncwarp();
#pragma unroll
            for (int u = 0; u < NB / 4; ++u) {
                y[u] = S(0);
#pragma unroll
                for (int k = 0; k < 4 * u + 4; ++k) y[u] = fma(scr[(4 * u + q) * NB + k], x[k], y[u]);
            }
            if (g < rest)
#pragma unroll
                for (int u = 0; u < NB / 4; ++u) A[(j0 + 4 * u + q) * lda + c0 + g] = y[u];
        }
        __syncthreads();
        // A_22 -= R_12^T R_12 (upper triangle)
        tiles2(rest, rest, [&](int i, int j) {
            if (j + 1 < i) return;
            S *p = A + (c0 + i) * lda + c0 + j;
            const bool i1 = i + 1 < rest, j1 = j + 1 < rest;
            S s00 = p[0], s01 = j1 ? p[1] : S(0), s10 = i1 ? p[lda] : S(0), s11 = i1 && j1 ? p[lda + 1] : S(0);
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                S u[2], v[2];
                ld2(A + (j0 + k) * lda + c0 + i, u);
                ld2(A + (j0 + k) * lda + c0 + j, v);
                s00 = fma(-u[0], v[0], s00);
                s01 = fma(-u[0], v[1], s01);
                s10 = fma(-u[1], v[0], s10);
                s11 = fma(-u[1], v[1], s11);
            }
            p[0] = s00;
            if (j1) p[1] = s01;
            if (i1 && j > i) p[lda] = s10;
            if (i1 && j1) p[lda + 1] = s11;
        });
        __syncthreads();
    }
    return true;
}

// The inverses of the NB x NB diagonal blocks of the upper triangular A (ld lda), in place: a
// warp per block, a lane per column, back substitution in registers.
template <typename S>
__device__ void tri_inv_diag(S *A, int lda, int M) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int b = warp; b * NB < M; b += nw) {
        const int j0 = b * NB, nb = min(NB, M - j0), c = lane & (NB - 1);
        S *D = A + j0 * lda + j0;
        const S rd = lane < nb ? S(1) / D[lane * lda + lane] : S(1);
        S y[NB];
#pragma unroll
        for (int i = 0; i < NB; ++i) y[i] = S(i == c ? 1 : 0);
#pragma unroll
        for (int k = NB - 1; k >= 0; --k) {
            y[k] *= __shfl_sync(0xffffffffu, rd, k);
            if (k < nb) {
#pragma unroll
                for (int i = 0; i < k; ++i) y[i] = fma(-D[i * lda + k], y[k], y[i]);
            }
        }
        __syncwarp();
        if (lane < nb)
#pragma unroll
            for (int i = 0; i < NB; ++i)
                if (i < nb) D[i * lda + c] = i <= c ? y[i] : S(0);
    }
    __syncthreads();
}

// In-place inverse of an upper triangular matrix whose NB x NB diagonal blocks are inverted
// already: pairs [A B; 0 C] of inverted diagonal blocks become [A^-1, -A^-1 B C^-1; 0, C^-1],
// edge 16, 32, 64; two barriers per level.  tmp: (M / 2 rounded up to a power of two)^2 elements
// (tri_tmp_elems).
__host__ __device__ inline int tri_tmp_elems(int M) {
    int P = NB;
    while (P < M) P *= 2;
    return P / 2 * (P / 2);
}
template <typename S>
__device__ void tri_inv_merge(S *A, int lda, int M, S *tmp) {
    for (int bs = NB; bs < M; bs *= 2) {
        const int np = (M + 2 * bs - 1) / (2 * bs);
        for (int pass = 0; pass < 2; ++pass) {
            // all pairs' rows side by side: row index p * bs + i
            tiles2(np * bs, bs, [&](int ri, int j) {
                const int p = ri / bs, i = ri % bs, r0 = p * 2 * bs, c0 = r0 + bs;
                if (c0 + j >= M) return;
                const bool j1 = c0 + j + 1 < M;
                S s00 = 0, s01 = 0, s10 = 0, s11 = 0;
                S *T = tmp + p * bs * bs;
                if (pass == 0) {
                    // T = A^-1 B (A^-1 upper triangular: k >= i)
                    for (int k = i; k < bs; ++k) {
                        const S a0 = A[(r0 + i) * lda + r0 + k], a1 = A[(r0 + i + 1) * lda + r0 + k];
                        S v[2];
                        ld2(A + (r0 + k) * lda + c0 + j, v);
                        s00 = fma(a0, v[0], s00);
                        s01 = fma(a0, v[1], s01);
                        s10 = fma(a1, v[0], s10);
                        s11 = fma(a1, v[1], s11);
                    }
                    T[i * bs + j] = s00;
                    T[i * bs + j + 1] = j1 ? s01 : S(0);
                    T[(i + 1) * bs + j] = s10;
                    T[(i + 1) * bs + j + 1] = j1 ? s11 : S(0);
                } else {
                    // B <- -T C^-1 (C^-1 upper triangular: k <= j)
                    const int ke = min(j + 2, M - c0);
                    for (int k = 0; k < ke; ++k) {
                        const S a0 = T[i * bs + k], a1 = T[(i + 1) * bs + k];
                        S v[2];
                        ld2(A + (c0 + k) * lda + c0 + j, v);
                        s00 = fma(a0, v[0], s00);
                        s01 = fma(a0, v[1], s01);
                        s10 = fma(a1, v[0], s10);
                        s11 = fma(a1, v[1], s11);
                    }
                    S *q = A + (r0 + i) * lda + c0 + j;
                    q[0] = -s00;
                    q[lda] = -s10;
                    if (j1) {
                        q[1] = -s01;
                        q[lda + 1] = -s11;
                    }
                }
            });
            __syncthreads();
        }
    }
}

// epi(i, j, c) for the upper triangle of C = A B, A and B upper triangular (ld lda, zeros below
// the diagonal), in 2 x 2 tiles.
template <typename S, typename FE>
__device__ void tri_mm(const S *A, const S *B, int lda, int M, const FE &epi) {
    tiles2(M, M, [&](int i, int j) {
        if (j + 1 < i) return;
        const bool i1 = i + 1 < M;
        const S *pa = A + i * lda, *pb = pa + (i1 ? lda : 0);
        S s00 = 0, s01 = 0, s10 = 0, s11 = 0;
        const int ke = min(j + 2, M);
#pragma unroll 4
        for (int k = i; k < ke; ++k) {
            const S a0 = pa[k], a1 = pb[k];
            S v[2];
            ld2(B + k * lda + j, v);
            s00 = fma(a0, v[0], s00);
            s01 = fma(a0, v[1], s01);
            s10 = fma(a1, v[0], s10);
            s11 = fma(a1, v[1], s11);
        }
        const bool j1 = j + 1 < M;
        if (j >= i) epi(i, j, s00);
        if (j1) epi(i, j + 1, s01);
        if (i1 && j >= i + 1) epi(i + 1, j, s10);
        if (i1 && j1) epi(i + 1, j + 1, s11);
    });
}

// epi(i, j, e) for the upper triangle of E = I - S R (both upper triangular FP32, zeros below),
// each entry accumulated as an unevaluated pair of floats: every product s r is split exactly
// into p + pe (p the rounded product, pe = fma(s, r, -p)) and subtracted with Knuth's two-sum,
// so the residual, whose size is the FP32 rounding of the inverse, keeps about 48 bits while
// running on the FP32 pipe.
template <typename FE>
__device__ void tri_residual(const float *Sm, const float *R, int lda, int M, const FE &epi) {
    tiles2(M, M, [&](int i, int j) {
        if (j + 1 < i) return;
        const bool i1 = i + 1 < M;
        const float *pa = Sm + i * lda, *pb = pa + (i1 ? lda : 0);
        float hi[2][2], lo[2][2];
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                hi[r][q] = i + r == j + q ? 1.f : 0.f;
                lo[r][q] = 0.f;
            }
        const int ke = min(j + 2, M);
#pragma unroll 2
        for (int k = i; k < ke; ++k) {
            const float a[2] = {pa[k], pb[k]};
            float v[2];
            ld2(R + k * lda + j, v);
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const float p = __fmul_rn(a[r], v[q]);
                    const float pe = fmaf(a[r], v[q], -p);
                    float s, e;
                    two_sum(hi[r][q], -p, s, e);
                    hi[r][q] = s;
                    lo[r][q] += e - pe;
                }
        }
        const bool j1 = j + 1 < M;
        if (j >= i) epi(i, j, hi[0][0] + lo[0][0]);
        if (j1) epi(i, j + 1, hi[0][1] + lo[0][1]);
        if (i1 && j >= i + 1) epi(i + 1, j, hi[1][0] + lo[1][0]);
        if (i1 && j1) epi(i + 1, j + 1, hi[1][1] + lo[1][1]);
    });
}

// store(i, j, v) for the M x M entries of a row-major matrix in global memory (leading dimension
// ldg): rows by warp, columns by lane, eight loads in flight per lane.
template <typename FS>
__device__ __forceinline__ void load_square(const double *g, int ldg, int M, const FS &store) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int j = lane; j < M; j += 32)
        for (int i0 = warp; i0 < M; i0 += 8 * nw) {
            double v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = i0 + u * nw;
                v[u] = i < M ? __ldcg(g + i * ldg + j) : 0.0;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = i0 + u * nw;
                if (i < M) store(i, j, v[u]);
            }
        }
}
// f(i, j) for all i < R, j < C: rows by warp, columns by lane
template <typename F>
__device__ __forceinline__ void each(int R, int C, const F &f) {
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int i = threadIdx.x >> 5; i < R; i += nw)
        for (int j = lane; j < C; j += 32) f(i, j);
}

}  // namespace sm
}  // namespace kb
