// Dense M x M matrices (M <= 128) in shared memory, one CTA: blocked Cholesky, blocked inverse
// of a triangular matrix, products of triangular matrices.
//
// One SM works on these, so their time is latency: barriers, dependent operations, and FP64
// operations above all (two FMAs per clock and SM on this part).  Blocks of 16: a diagonal block
// is factored by four warps in registers, and the same instructions give the inverse of its
// factor; everything else is products of 16 or more independent terms, in tiles shared out
// over all threads.  Rows are lda elements apart, lda even (pairs of elements are loaded at
// once).  Cycles of the parts at M = 64 (FP32 / FP64), now and with the diagonal block in one
// warp and tiles by rows: Cholesky 25 k / 104 k and 33 k / 173 k, merges 7 k / 40 k and 9 k /
// 52 k, one product 6 k / 44 k and 6 k / 78 k.
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

template <int E, typename S>
__device__ __forceinline__ void ldE(const S *p, S (&v)[E]) {
    if constexpr (E == 2) ld2(p, v);
    else v[0] = p[0];
}

// 1/d for a positive double d by Newton's iteration for the reciprocal, r <- r + r (1 - d r),
// from the hardware approximation (relative error about 2^-20): two steps take it to the FP64
// rounding level (the error squares at each step).  The FP64 division it replaces is a long
// dependent sequence on this part's FP64 unit; this is four FMAs.
__device__ __forceinline__ double recip(double d) {
    if (!(d > 1e-290 && d < 1e290)) return 1.0 / d;
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    double e = fma(-d, r, 1.0);
    r = fma(r, e, r);
    e = fma(-d, r, 1.0);
    return fma(r, e, r);
}
__device__ __forceinline__ float recip(float d) { return __frcp_rn(d); }   // (rounded to nearest)

// Edge of the register tiles: 2 in FP32, where a shared load is the dearer part, 1 in FP64,
// whose FMA occupies a scheduler for some 64 cycles, so that only spreading the entries helps.
template <typename S> struct Tile { static constexpr int E = sizeof(S) == 8 ? 1 : 2; };

// E x E tiles (i0, j0) meeting the upper triangle of an M x M matrix, shared out evenly over
// the threads: consecutive threads along a row, or (DIAG) along a diagonal, where the sums over
// k = i0 .. j0 of triangular products are equally long.
template <int E, bool DIAG, typename F>
__device__ __forceinline__ void tri_tiles(int M, const F &f) {
    const int nt = (M + E - 1) / E, total = nt * (nt + 1) / 2;
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
        // rows above hold i nt - i (i - 1) / 2 tiles
        const float h = float(nt) + 0.5f;
        int i = int(h - sqrtf(fmaxf(h * h - 2.f * float(t), 0.f)));
        i = max(0, min(i, nt - 1));
        while (i > 0 && i * nt - i * (i - 1) / 2 > t) --i;
        while ((i + 1) * nt - (i + 1) * i / 2 <= t) ++i;
        const int j = i + t - (i * nt - i * (i - 1) / 2);
        if (DIAG) f((j - i) * E, j * E);   // (row i of the enumeration: the i-th diagonal)
        else f(i * E, j * E);
    }
}

// Cholesky G = R^T R: the upper triangle of A holds G on entry and R on return.  Inv (ld lda,
// or nullptr) receives the inverses of R's NB x NB diagonal blocks (upper triangular, zeros
// below).  Returns false (all threads) on a pivot (diagonal entry of the Schur complement) not
// above thr.  scr: NB * NB elements.
template <typename S>
__device__ bool chol_blocked(S *A, S *Inv, int lda, int M, S thr, S *scr) {
    __shared__ int s_bad;
    __shared__ S s_row[64];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_bad = 0;
    __syncthreads();
    for (int j0 = 0; j0 < M; j0 += NB) {
        const int nb = min(NB, M - j0);
        if (warp < 4) {
            // Four warps (one per scheduler), warp w the rows w, w + 4, ..; lanes 0..15 the columns
            // of the diagonal block, lanes 16..31 those of I, on which the same row operations
            // leave R^{-T}.  Square-root free: row j goes round unscaled through shared memory,
            // its multiple by 1 / d_j updates the rows below, so a step is one exchange, one
            // reciprocal, one product and up to four FMAs; the square roots of the pivots come
            // at the end, all at once.
            const int c = lane & (NB - 1);
            const bool inv = lane >= NB;
            S a[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = warp + 4 * u;
                a[u] = (!inv && i < nb && c < nb) ? (i <= c ? A[(j0 + i) * lda + j0 + c] : S(0)) : S(i == c ? 1 : 0);
            }
            bool bad = false;
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                S *rb = s_row + (j & 1) * 32;
                if (warp == j % 4) rb[lane] = a[j / 4];
                asm volatile("bar.sync 1, 128;" ::: "memory");
                S d = rb[j];
                if (j < nb && !(d > thr)) {
                    bad = true;
                    d = S(1);
                }
                const S sc = rb[lane] * recip(d);
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (4 * u + 3 > j && warp + 4 * u > j) a[u] = fma(-rb[warp + 4 * u], sc, a[u]);
            }
            if (bad && lane == 0) s_bad = 1;
            // row i times 1 / sqrt(d_i)
            S piv = S(1);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const S d = __shfl_sync(0xffffffffu, a[u], warp + 4 * u);
                if (lane == u && warp + 4 * u < nb) piv = d;
            }
            const S rt = sqrt(piv), ri = recip(rt);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = warp + 4 * u;
                const S r = __shfl_sync(0xffffffffu, rt, u), q = __shfl_sync(0xffffffffu, ri, u);
                const S v = (!inv && c == i) ? r : a[u] * q;
                if (inv) scr[i * NB + c] = v;                  // R^{-T}, lower triangular
                if (i < nb && c < nb) {
                    if (!inv) A[(j0 + i) * lda + j0 + c] = i <= c ? v : S(0);
                    else if (Inv) Inv[(j0 + c) * lda + j0 + i] = i >= c ? v : S(0);
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
        constexpr int E = Tile<S>::E;
        tri_tiles<E, false>(rest, [&](int i, int j) {
            S acc[E][E];
#pragma unroll
            for (int r = 0; r < E; ++r)
#pragma unroll
                for (int q = 0; q < E; ++q)
                    acc[r][q] = i + r < rest && j + q < rest ? A[(c0 + i + r) * lda + c0 + j + q] : S(0);
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                S u[E], v[E];
                ldE<E>(A + (j0 + k) * lda + c0 + i, u);
                ldE<E>(A + (j0 + k) * lda + c0 + j, v);
#pragma unroll
                for (int r = 0; r < E; ++r)
#pragma unroll
                    for (int q = 0; q < E; ++q) acc[r][q] = fma(-u[r], v[q], acc[r][q]);
            }
#pragma unroll
            for (int r = 0; r < E; ++r)
#pragma unroll
                for (int q = 0; q < E; ++q)
                    if (i + r <= j + q && j + q < rest) A[(c0 + i + r) * lda + c0 + j + q] = acc[r][q];
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
            constexpr int E = Tile<S>::E;
            const int per = bs / E;   // tiles of a row or column (a power of two)
            for (int t = threadIdx.x; t < np * per * per; t += blockDim.x) {
                const int j = (t % per) * E, ri = (t / per) * E;
                const int p = ri / bs, i = ri % bs, r0 = p * 2 * bs, c0 = r0 + bs;
                if (c0 + j >= M) continue;
                S acc[E][E];
#pragma unroll
                for (int r = 0; r < E; ++r)
#pragma unroll
                    for (int q = 0; q < E; ++q) acc[r][q] = S(0);
                S *T = tmp + p * bs * bs;
                // pass 0: T = A^-1 B (A^-1 upper triangular: k >= i); pass 1: B <- -T C^-1 (C^-1
                // upper triangular: k <= j)
                const S *L = pass == 0 ? A + (r0 + i) * lda + r0 : T + i * bs;
                const int ldl = pass == 0 ? lda : bs;
                const S *Rm = A + (pass == 0 ? r0 : c0) * lda + c0 + j;
                const int k0 = pass == 0 ? i : 0, k1 = pass == 0 ? bs : min(j + E, M - c0);
#pragma unroll 4
                for (int k = k0; k < k1; ++k) {
                    S v[E];
                    ldE<E>(Rm + k * lda, v);
#pragma unroll
                    for (int r = 0; r < E; ++r) {
                        const S a = L[r * ldl + k];
#pragma unroll
                        for (int q = 0; q < E; ++q) acc[r][q] = fma(a, v[q], acc[r][q]);
                    }
                }
#pragma unroll
                for (int r = 0; r < E; ++r)
#pragma unroll
                    for (int q = 0; q < E; ++q) {
                        const bool in = c0 + j + q < M;
                        if (pass == 0) T[(i + r) * bs + j + q] = in ? acc[r][q] : S(0);
                        else if (in) A[(r0 + i + r) * lda + c0 + j + q] = -acc[r][q];
                    }
            }
            __syncthreads();
        }
    }
}

// epi(i, j, c, x) for the upper triangle of C = A B, A and B upper triangular (ld lda, zeros
// below the diagonal); x = pre(i, j), asked for before the sums so that its load overlaps them.
template <typename S, typename FP, typename FE>
__device__ void tri_mm(const S *A, const S *B, int lda, int M, const FP &pre, const FE &epi) {
    constexpr int E = Tile<S>::E;
    tri_tiles<E, true>(M, [&](int i, int j) {
        S acc[E][E];
        decltype(pre(0, 0)) x[E][E];
#pragma unroll
        for (int r = 0; r < E; ++r)
#pragma unroll
            for (int q = 0; q < E; ++q) {
                acc[r][q] = S(0);
                x[r][q] = pre(min(i + r, M - 1), min(j + q, M - 1));
            }
        const int ke = min(j + E, M);
#pragma unroll 4
        for (int k = i; k < ke; ++k) {
            S v[E];
            ldE<E>(B + k * lda + j, v);
#pragma unroll
            for (int r = 0; r < E; ++r) {
                const S a = A[min(i + r, M - 1) * lda + k];
#pragma unroll
                for (int q = 0; q < E; ++q) acc[r][q] = fma(a, v[q], acc[r][q]);
            }
        }
#pragma unroll
        for (int r = 0; r < E; ++r)
#pragma unroll
            for (int q = 0; q < E; ++q)
                if (i + r <= j + q && j + q < M) epi(i + r, j + q, acc[r][q], x[r][q]);
    });
}

// epi(i, j, e) for the upper triangle of E = I - S R (both upper triangular FP32, zeros below),
// each entry accumulated as an unevaluated pair of floats: every product s r is split exactly
// into p + pe (p the rounded product, pe = fma(s, r, -p)) and subtracted with Knuth's two-sum,
// so the residual, whose size is the FP32 rounding of the inverse, keeps about 48 bits while
// running on the FP32 pipe.
template <typename FE>
__device__ void tri_residual(const float *Sm, const float *R, int lda, int M, const FE &epi) {
    tri_tiles<2, true>(M, [&](int i, int j) {
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
#pragma unroll 4
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
