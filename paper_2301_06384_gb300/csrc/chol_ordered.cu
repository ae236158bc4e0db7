// CholeskyQR of FP32 solves with full reorthogonalisation (the contract of k_chol in chol.cu): the
// factorisation column by column, so that the rounding of the basis is one and the same for
// such solves (rowblock.cuh, ordered form).
#include "kb_internal.cuh"
#include "kb_kernels.cuh"
#include "smallmat.cuh"

namespace kb {
namespace {

// In-place inverse of an upper triangular M x M matrix in shared memory (ld lda), column
// by column: with the leading j x j block already inverted, column j of the inverse is
// -(1/a_jj) X_{0:j,0:j} a_{0:j,j}.  The diagonal reciprocals do not depend on the other
// columns and are formed first, all in parallel; the original entries of column j+1 are
// copied into the second half of t while column j is formed, so each column costs one
// barrier.  Each row's dot product is split over TPR consecutive lanes (TPR = 1, 2, 4 or 8)
// and combined with shuffles.  t: shared scratch of 2 M values.
template <typename S>
__device__ void tri_inv_upper_inplace(S *A, int lda, int M, S *t) {
    int TPR = 1;
    while (TPR < 8 && TPR * 2 * M <= int(blockDim.x)) TPR *= 2;
    const int sub = threadIdx.x % TPR;
    const int row0 = threadIdx.x / TPR;
    const int rstride = blockDim.x / TPR;
    for (int j = threadIdx.x; j < M; j += blockDim.x) A[j * lda + j] = S(1) / A[j * lda + j];
    if (M > 1 && threadIdx.x == 0) t[M] = A[1];   // column 1, row 0
    __syncthreads();
    for (int j = 1; j < M; ++j) {
        const S *tc = (j & 1) ? t + M : t;   // original column j, rows < j
        S *tn = (j & 1) ? t : t + M;         // original column j+1, rows <= j
        if (j + 1 < M)
            for (int i = threadIdx.x; i <= j; i += blockDim.x) tn[i] = A[i * lda + j + 1];
        const S ajj = A[j * lda + j];        // already 1 / a_jj
        // rows i < j, all TPR lanes of a row iterate together (uniform loop bound per warp)
        for (int ib = 0; ib < j; ib += rstride) {
            const int i = ib + row0;
            S acc = S(0);
            if (i < j)
                for (int k = i + sub; k < j; k += TPR) acc = fma(A[i * lda + k], tc[k], acc);
            for (int off = 1; off < TPR; off <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
            if (i < j && sub == 0) A[i * lda + j] = -ajj * acc;
        }
        __syncthreads();
    }
}

// 1/d for a positive double d by Newton's iteration for the reciprocal, r <- r + r (1 - d r),
// from the single-precision reciprocal: two steps take its 2^-23 relative error to the
// FP64 rounding level (the error squares at each step).  The FP64 division it replaces is
// a long dependent sequence on this part's FP64 unit; this is four FMAs.  Outside the
// normal single-precision range the division is used.
__device__ __forceinline__ double recip_newton(double d) {
    if (!(d > 1e-36 && d < 1e36)) return 1.0 / d;
    double r = double(__frcp_rn(float(d)));
    double e = fma(-d, r, 1.0);
    r = fma(r, e, r);
    e = fma(-d, r, 1.0);
    return fma(r, e, r);
}

__device__ __forceinline__ double chol_recip(double d) { return recip_newton(d); }
// the correctly rounded reciprocal (the same value as 1.0f / d, without the division sequence)
__device__ __forceinline__ float chol_recip(float d) { return __frcp_rn(d); }
// 1 / d rounded to nearest in either precision
__device__ __forceinline__ float recip_rn(float d) { return __frcp_rn(d); }
__device__ __forceinline__ double recip_rn(double d) { return 1.0 / d; }

// Scratch of tri_inv_upper_blocked: (P/2)^2 values, P the power of two >= M.
__host__ __device__ inline int tri_inv_tmp_elems(int M) {
    int P = 1;
    while (P < M) P *= 2;
    return (P / 2) * (P / 2);
}

// Blocked in-place inverse of an upper triangular M x M matrix in shared memory (ld lda),
// with few barriers: the 8 x 8 diagonal blocks are inverted one per thread (column by
// column, rows ascending, so each row still reads the original column above the diagonal),
// then pairs of inverted diagonal blocks [A B; 0 C] are merged level by level into
// [A^-1, -A^-1 B C^-1; 0, C^-1] (block edge 8, 16, 32, 64): two barriers per level instead
// of one per column.  tmp: tri_inv_tmp_elems(M) values of shared scratch (the products
// A^-1 B of every pair at the widest level).
template <typename S>
__device__ void tri_inv_upper_blocked(S *A, int lda, int M, S *tmp) {
    const int nb = (M + 7) / 8;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        const int r0 = b * 8, r1 = min(r0 + 8, M);
        for (int j = r0; j < r1; ++j) {
            const S ajj = recip_rn(A[j * lda + j]);
            for (int i = r0; i < j; ++i) {
                S acc = S(0);
                for (int k = i; k < j; ++k) acc = fma(A[i * lda + k], A[k * lda + j], acc);
                A[i * lda + j] = -ajj * acc;
            }
            A[j * lda + j] = ajj;
        }
    }
    __syncthreads();
    for (int lg = 3, bs = 8; bs < M; ++lg, bs *= 2) {
        // T_p = A_p^-1 B_p for every pair p (rows r0.., columns r0 + bs..); each thread four
        // consecutive columns of one row (four independent FMA chains sharing the A loads)
        const int npairs = (M + 2 * bs - 1) / (2 * bs);
        const int per = bs * bs;
        const int lq = lg - 2;   // log2(bs / 4)
        for (int idx = threadIdx.x; idx < npairs * (per >> 2); idx += blockDim.x) {
            const int p = idx >> (2 * lg - 2), i = (idx >> lq) & (bs - 1), c = (idx & ((bs >> 2) - 1)) << 2;
            const int r0 = p * 2 * bs, cb = min(bs, M - r0 - bs);
            if (cb <= 0 || c >= cb) continue;
            S acc[4] = {S(0), S(0), S(0), S(0)};
            for (int k = i; k < bs; ++k) {
                const S a = A[(r0 + i) * lda + r0 + k];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (c + q < cb) acc[q] = fma(a, A[(r0 + k) * lda + r0 + bs + c + q], acc[q]);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) tmp[p * per + i * bs + c + q] = acc[q];
        }
        __syncthreads();
        // B_p <- -T_p C_p^-1 (C^-1 upper triangular: the terms k > c are exact zeros)
        for (int idx = threadIdx.x; idx < npairs * (per >> 2); idx += blockDim.x) {
            const int p = idx >> (2 * lg - 2), i = (idx >> lq) & (bs - 1), c = (idx & ((bs >> 2) - 1)) << 2;
            const int r0 = p * 2 * bs, cb = min(bs, M - r0 - bs);
            if (cb <= 0 || c >= cb) continue;
            const int c0 = r0 + bs;
            S acc[4] = {S(0), S(0), S(0), S(0)};
            const int kend = min(c + 4, cb);
            for (int k = 0; k < kend; ++k) {
                const S t = tmp[p * per + i * bs + k];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (c + q < cb) acc[q] = fma(t, A[(c0 + k) * lda + c0 + c + q], acc[q]);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (c + q < cb) A[(r0 + i) * lda + c0 + c + q] = -acc[q];
        }
        __syncthreads();
    }
}

// The upper triangle of an M x M matrix in 4 x 4 tiles: tile t (row-major over the tiles
// (bi, bj), bi <= bj, of the ceil(M/4) x ceil(M/4) grid) -> first row i0, first column j0.
__device__ __forceinline__ void upper_tile(int t, int nt, int &i0, int &j0) {
    int bi = 0;
    while (t >= nt - bi) {
        t -= nt - bi;
        ++bi;
    }
    i0 = 4 * bi;
    j0 = 4 * (bi + t);
}

// C = init + sum_k a(i, k) b(k, j) over the upper triangle i <= j < M of a product of two
// upper triangular M x M matrices, read through the accessors a and b (which must return
// exact zeros below the diagonal).  Each thread takes 4 x 4 tiles of C: 16 independent
// FMA chains over k = i0 .. j0 + 3, the only k where a term of the tile can be non-zero,
// in ascending order, so every entry is the FMA chain of the plain loop k = i .. j with
// exact zero terms added.  epi(i, j, c) receives the upper-triangle entries.
template <typename S, typename FA, typename FB, typename FI, typename FE>
__device__ void tri_mm_upper(int M, const FA &a, const FB &b, const FI &init, const FE &epi) {
    const int nt = (M + 3) / 4;
    const int ntiles = nt * (nt + 1) / 2;
    for (int t = threadIdx.x; t < ntiles; t += blockDim.x) {
        int i0, j0;
        upper_tile(t, nt, i0, j0);
        S acc[4][4];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                acc[r][q] = (i0 + r < M && j0 + q < M) ? init(i0 + r, j0 + q) : S(0);
        const int kend = min(j0 + 4, M);
        for (int k = i0; k < kend; ++k) {
            S av[4], bv[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) av[r] = (i0 + r < M) ? a(i0 + r, k) : S(0);
#pragma unroll
            for (int q = 0; q < 4; ++q) bv[q] = (j0 + q < M) ? b(k, j0 + q) : S(0);
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[r][q] = fma(av[r], bv[q], acc[r][q]);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = i0 + r, j = j0 + q;
                if (i < M && j < M && j >= i) epi(i, j, acc[r][q]);
            }
    }
}

// E = I - S R for upper triangular FP32 matrices S and R in shared memory (ld lda, zeros
// below the diagonal), each entry accumulated as an unevaluated pair of floats: every
// product s r is split exactly into p + pe (p the rounded product, pe = fma(s, r, -p)) and
// subtracted with Knuth's two-sum, so the residual, whose size is the FP32 rounding of the
// inverse, keeps about 48 bits while running on the FP32 pipe.  Returns E rounded to FP32
// through epi(i, j, e) for the upper triangle.
template <typename FE>
__device__ void tri_residual_df(const float *Sm, const float *Rm, int lda, int M, const FE &epi) {
    const int nt = (M + 3) / 4;
    const int ntiles = nt * (nt + 1) / 2;
    for (int t = threadIdx.x; t < ntiles; t += blockDim.x) {
        int i0, j0;
        upper_tile(t, nt, i0, j0);
        float hi[4][4], lo[4][4];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                hi[r][q] = (i0 + r == j0 + q) ? 1.f : 0.f;
                lo[r][q] = 0.f;
            }
        const int kend = min(j0 + 4, M);
        for (int k = i0; k < kend; ++k) {
            float sv[4], rv[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) sv[r] = (i0 + r < M) ? Sm[(i0 + r) * lda + k] : 0.f;
#pragma unroll
            for (int q = 0; q < 4; ++q) rv[q] = (j0 + q < M) ? Rm[k * lda + j0 + q] : 0.f;
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float p = __fmul_rn(sv[r], rv[q]);
                    const float pe = fmaf(sv[r], rv[q], -p);
                    float s, e;
                    two_sum(hi[r][q], -p, s, e);
                    hi[r][q] = s;
                    lo[r][q] += e - pe;
                }
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = i0 + r, j = j0 + q;
                if (i < M && j < M && j >= i) epi(i, j, hi[r][q] + lo[r][q]);
            }
    }
}

// Cholesky G = R^T R of an M x M symmetric matrix in shared memory, upper R overwriting A
// and the lower part zeroed.  Square-root-free form: step j needs the pivot d_j (the
// diagonal of the current Schur complement) and one reciprocal; the Schur complement update
// is A_ab -= u_ja u_jb / d_j with the unscaled pivot row u_j.  The square roots and the row
// scaling R_j = u_j / sqrt(d_j) are applied at the end, for all rows at once.  Look-ahead:
// during step j warp 0 updates only the next pivot row j+1, takes its pivot and the one
// FP64 division and forms the scaled row u_{j+1} / d_{j+1} (into the other half of a double
// buffer), while the other warps update rows j+2..; so each column costs one barrier and
// the division overlaps the bulk of the update.  Returns false (all threads) on a pivot
// <= piv_rel2 * max diag.  t: shared scratch of 3 M doubles.  Needs blockDim.x >= 64.
// bad: two shared flags, zero on entry.  The failure of pivot j is recorded in bad[j & 1]
// (by warp 0 during step j-1) and read by every thread at the top of step j, after the
// barrier that ends step j-1; the flag warp 0 writes during step j is the other one, so no
// thread can read a flag in the same barrier interval in which it is written (all threads
// leave at the same step).
template <typename S>
__device__ bool chol_upper_inplace(S *A, int lda, int M, S piv_rel2, S maxdiag, S *t, int *bad) {
    S *const srow0 = t, *const srow1 = t + M;   // u_j / d_j, double-buffered by the parity of j
    S *piv = t + 2 * M;        // d_j
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const S thr = piv_rel2 * maxdiag;
    // pivot row 0
    if (warp == 0) {
        const S d = A[0];
        if (!(d > thr)) {
            if (lane == 0) bad[0] = 1;
        } else {
            const S dinv = chol_recip(d);
            for (int c = 1 + lane; c < M; c += 32) srow0[c] = A[c] * dinv;
            if (lane == 0) piv[0] = d;
        }
    }
    __syncthreads();
    for (int j = 0; j < M; ++j) {
        if (bad[j & 1]) return false;
        const S *sr = (j & 1) ? srow1 : srow0;
        if (warp == 0) {
            if (j + 1 < M) {
                // the next pivot row: A[j+1][c] -= u_{j,j+1} u_{j,c} / d_j, c >= j+1, held in
                // registers (lane l: c = j+1+l+32q); its pivot comes from lane 0 by a shuffle
                const S ujn = A[j * lda + j + 1];
                S v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int c = j + 1 + lane + 32 * q;
                    v[q] = c < M ? fma(-ujn, sr[c], A[(j + 1) * lda + c]) : S(0);
                }
                const S d = __shfl_sync(0xffffffffu, v[0], 0);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int c = j + 1 + lane + 32 * q;
                    if (c < M) A[(j + 1) * lda + c] = v[q];
                }
                if (!(d > thr)) {
                    if (lane == 0) bad[(j + 1) & 1] = 1;
                } else {
                    const S dinv = chol_recip(d);
                    S *sn = ((j + 1) & 1) ? srow1 : srow0;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int c = j + 1 + lane + 32 * q;
                        if (c >= j + 2 && c < M) sn[c] = v[q] * dinv;
                    }
                    if (lane == 0) piv[j + 1] = d;
                }
            }
        } else {
            // rows j+2.. of the trailing upper triangle: rows by warp, columns by lane (c =
            // lane + 32q); four rows' loads are issued before any of their stores
            const int nw = (blockDim.x >> 5) - 1;
            S srv[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) srv[q] = lane + 32 * q < M ? sr[lane + 32 * q] : S(0);
            for (int ra0 = j + 1 + warp; ra0 < M; ra0 += 4 * nw) {
                S u[4], a[4][4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int ra = ra0 + r * nw;
                    u[r] = ra < M ? A[j * lda + ra] : S(0);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int c = lane + 32 * q;
                        a[r][q] = (ra < M && c >= ra && c < M) ? A[ra * lda + c] : S(0);
                    }
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int ra = ra0 + r * nw;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int c = lane + 32 * q;
                        if (ra < M && c >= ra && c < M) A[ra * lda + c] = fma(-u[r], srv[q], a[r][q]);
                    }
                }
            }
        }
        __syncthreads();
    }
    // (no pivot is examined during the last step: the flags are final here)
    if (bad[0] | bad[1]) return false;
    // R_jj = sqrt(d_j), R_jc = u_jc / sqrt(d_j)
    S *rinv = srow0;
    for (int j = threadIdx.x; j < M; j += blockDim.x) {
        const S r = sqrt(piv[j]);
        piv[j] = r;
        rinv[j] = recip_rn(r);
    }
    __syncthreads();
    for (int i = warp; i < M; i += blockDim.x >> 5)
        for (int j = lane; j < M; j += 32) {
            if (j < i) A[i * lda + j] = S(0);
            else if (j == i) A[i * lda + j] = piv[i];
            else A[i * lda + j] *= rinv[i];
        }
    __syncthreads();
    return true;
}

// Reduced QR of the new block by CholeskyQR (Algorithm 1), pass 1 or 2 of
// CholeskyQR2.  Outputs: Rinv (W x W, basis precision) applied by the row-block kernels;
// pass 1 records R1 = the FP64 inverse of the applied inverse; pass 2 records
// H_{k+1,k} = R2 R1 (rounded to the basis precision) and B = H^T.
//
// Pass 1 (G = X^T X, any conditioning): Cholesky in FP32, or in FP64 where a pivot is small; the
// inverse is formed in FP32 and R1 is then the inverse of that FP32 inverse, so that X = X1 R1
// holds for the applied matrices.
// Pass 2 (G = I + E, ||E|| of the order of the FP32 rounding of pass 1):
// to first order R2 = I + Phi(E) with Phi = strict upper part plus half the diagonal,
// R2^{-1} = I - Phi(E) (the orthogonality of Q = X1 (I - Phi(E)) is then I + O(||E||^2));
// the applied inverse I - F has the inverse I + F + F^2 + O(F^3), so H = R1 + F R1 + F (F R1),
// the corrections formed in FP32.  When ||E|| is not small (max |E_ij| >= 1e-4) pass 2 uses the
// pass-1 algorithm.
//
// The kernel runs on one SM, so its time is latency: the matrices are loaded with several
// loads in flight per thread, the triangular products run as 4 x 4 register tiles (16
// independent FMA chains per thread instead of one serial chain per entry), the residual of
// the FP32 inverse uses pairs of floats rather than FP64 (whose rate on this part is a small
// fraction of FP32), the statistics of G are reduced in parallel (max |E_ij| through the
// order-preserving bit patterns of non-negative doubles) and the Cholesky factorisation needs
// one division per column.
constexpr int CHOL_NEWTON_MAX = 64;   // widest block with the corrected-inverse scratch
__global__ void __launch_bounds__(256) k_chol_ordered(const double *G, int M, int W, int pass, int step,
                                              double inv_thresh2, double piv_rel2, double *R1,
                                              float *Rinv, double *Hs, float *Bout, Ctrl *ctrl) {
    if (ctrl->stop) return;
    // [M][M+1] FP64, then [M][M+1] FP32, then 3 M + 2 doubles of scratch
    extern __shared__ __align__(16) double A[];
    __shared__ int bad, small;
    __shared__ int pivot_bad[2];   // chol_upper_inplace's per-parity pivot failure flags
    __shared__ double maxdiag;
    __shared__ unsigned long long emax_bits;
    const int lda = M + 1;
    float *Sf = reinterpret_cast<float *>(A + M * lda);
    double *t = reinterpret_cast<double *>(Sf + M * lda + (M * lda) % 2);
    const bool try_small = pass == 2;
    if (threadIdx.x == 0) {
        emax_bits = 0ull;
        bad = 0;
        pivot_bad[0] = 0;
        pivot_bad[1] = 0;
    }
    __syncthreads();
    unsigned long long my_e = 0ull;
    sm::load_square(G, W, M, [&](int i, int j, double g) {
        A[i * lda + j] = g;
        if (try_small) {
            double e = g;
            if (i == j) e -= 1.0;
            const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(fabs(e)));
            my_e = b > my_e ? b : my_e;
        }
    });
    if (try_small) {
        for (int off = 16; off > 0; off >>= 1) {
            const unsigned long long o = __shfl_xor_sync(0xffffffffu, my_e, off);
            my_e = o > my_e ? o : my_e;
        }
        if ((threadIdx.x & 31) == 0) atomicMax(&emax_bits, my_e);
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        // trace and largest diagonal entry (non-negative for a Gram matrix: bit order)
        double tr = 0.0;
        unsigned long long mx = 0ull;
        for (int i = threadIdx.x; i < M; i += 32) {
            const double d = A[i * lda + i];
            tr += d;
            const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(fabs(d)));
            mx = b > mx ? b : mx;
        }
        for (int off = 16; off > 0; off >>= 1) {
            tr += __shfl_xor_sync(0xffffffffu, tr, off);
            const unsigned long long o = __shfl_xor_sync(0xffffffffu, mx, off);
            mx = o > mx ? o : mx;
        }
        if (threadIdx.x == 0) {
            maxdiag = __longlong_as_double(static_cast<long long>(mx));
            small = (try_small && __longlong_as_double(static_cast<long long>(emax_bits)) < 1e-4) ? 1 : 0;
            if (pass == 1 && !(tr > inv_thresh2)) {
                // X vanished: the block Krylov space is invariant; keep the blocks so far
                ctrl->stop = 1;
                ctrl->steps = step;
                bad = 2;
            }
        }
    }
    __syncthreads();
    if (bad) return;
    if (small) {
        // ---- pass 2, first order: S = I - Phi(E) applied; F = I - S exactly
        for (int i = threadIdx.x >> 5; i < W; i += blockDim.x >> 5)
            for (int j = threadIdx.x & 31; j < W; j += 32) {
                const int idx = i * W + j;
                // one FP64 subtraction per entry (E is small: the rest is exact or FP32-level)
                float v = 0.f;
                if (i < M && j < M && j >= i) {
                    const float e = float(A[i * lda + j] - (i == j ? 1.0 : 0.0));
                    v = (i == j) ? 1.f - 0.5f * e : -e;
                }
                Rinv[idx] = v;
                if (i < M && j < M) Sf[i * lda + j] = (j >= i) ? (i == j ? 1.f : 0.f) - v : 0.f;
            }
        __syncthreads();
        // A is free now: R1 rounded to FP32, and C = F R1 (both upper triangular, zeros below)
        float *R1t = reinterpret_cast<float *>(A);
        float *Ct = R1t + M * lda;
        sm::load_square(R1, M, M, [&](int i, int j, double v) {
            R1t[i * lda + j] = (j >= i) ? float(v) : 0.f;
            Ct[i * lda + j] = 0.f;
        });
        __syncthreads();
        auto sf = [&](int i, int k) { return Sf[i * lda + k]; };
        auto zero = [](int, int) { return 0.f; };
        tri_mm_upper<float>(M, sf, [&](int k, int j) { return R1t[k * lda + j]; }, zero,
                        [&](int i, int j, float c) { Ct[i * lda + j] = c; });
        // entries of Hs and B outside H's upper triangle are zero
        for (int i = threadIdx.x >> 5; i < W; i += blockDim.x >> 5)
            for (int j = threadIdx.x & 31; j < W; j += 32) {
                if (i < M && j < M && j >= i) continue;
                if (i < M && j < M) Hs[i * M + j] = 0.0;
                Bout[j * W + i] = 0.f;
            }
        __syncthreads();
        // H = (I + F + F^2) R1 = R1 + (C + F C), the corrections of relative size ||E||
        tri_mm_upper<float>(M, sf, [&](int k, int j) { return Ct[k * lda + j]; }, zero,
                        [&](int i, int j, float corr2) {
                            const double h = __ldg(R1 + i * M + j) + double(Ct[i * lda + j] + corr2);
                            const float ht = float(h);
                            Hs[i * M + j] = double(ht);
                            Bout[j * W + i] = ht;
                        });
        return;
    }
    // ---- general CholeskyQR pass
    // Pass 1 first factors G in FP32 (the FP32 pipe runs 64 times the FP64
    // rate): the first pass only has to bring X close to orthonormal, the second pass
    // corrects what is left (its first-order form when max |G2 - I| < 1e-4, a full
    // factorisation otherwise), and R1 below is the FP64 inverse of the applied inverse
    // whatever R it came from.  A pivot below 1e-5 of the largest diagonal entry is not
    // trusted in FP32: the factorisation is then redone in FP64 (which alone decides a
    // breakdown).
    bool factored = false;
    if (pass == 1) {
        float *Af = Sf;   // Sf is free until the inverse below
        float *tf = reinterpret_cast<float *>(t);
        for (int i = threadIdx.x >> 5; i < M; i += blockDim.x >> 5)
            for (int j = threadIdx.x & 31; j < M; j += 32) {
                Af[i * lda + j] = float(A[i * lda + j]);
            }
        __syncthreads();
        if (chol_upper_inplace<float>(Af, lda, M, 1e-5f, float(maxdiag), tf, pivot_bad)) {
            for (int i = threadIdx.x >> 5; i < M; i += blockDim.x >> 5)
                for (int j = threadIdx.x & 31; j < M; j += 32) {
                    A[i * lda + j] = (j >= i) ? double(Af[i * lda + j]) : 0.0;
                }
            factored = true;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            pivot_bad[0] = 0;
            pivot_bad[1] = 0;
        }
        __syncthreads();
    }
    if (!factored && !chol_upper_inplace<double>(A, lda, M, piv_rel2, maxdiag, t, pivot_bad)) {
        if (threadIdx.x == 0) {
            ctrl->status = KB_ERR_BREAKDOWN;
            ctrl->stop = 1;
            ctrl->steps = step;
            ctrl->breakdown_step = step;
        }
        return;
    }
    const bool newton = M <= CHOL_NEWTON_MAX;
    double *Sd = t + 3 * M + 2;                               // [M][M+1] (newton only)
    float *Rf = reinterpret_cast<float *>(Sd + M * lda);      // [M][M+1]
    float *C1 = Rf + M * lda;                                 // [M][M+1]
    for (int i = threadIdx.x >> 5; i < M; i += blockDim.x >> 5)
        for (int j = threadIdx.x & 31; j < M; j += 32) {
            Sf[i * lda + j] = float(A[i * lda + j]);
            if (newton) Rf[i * lda + j] = Sf[i * lda + j];
        }
    __syncthreads();
    {
        // scratch after the Newton region (launch_chol sizes it)
        unsigned char *after = reinterpret_cast<unsigned char *>(t + 3 * M + 2) + (newton ? 16 * size_t(M) * lda : 0);
        tri_inv_upper_blocked<float>(Sf, lda, M, reinterpret_cast<float *>(after));
    }
    for (int i = threadIdx.x >> 5; i < W; i += blockDim.x >> 5)
        for (int j = threadIdx.x & 31; j < W; j += 32) {
            const int idx = i * W + j;
            Rinv[idx] = (i < M && j < M && j >= i) ? Sf[i * lda + j] : 0.f;
        }
    // R := the FP64 inverse of the applied FP32 inverse S.
    bool exact = !newton;
    if (newton) {
        // With S R = I - E (E upper triangular, of the order of the FP32 rounding),
        // S^{-1} = R (I - E)^{-1} = R + R E + R E^2 + O(E^3): E is formed from S and R with
        // a residual more precise than FP32 (pairs of floats when R is the FP32 factor,
        // FP64 when the factorisation fell back to FP64), the corrections in FP32.  When
        // max |E_ij| >= 1e-3 the exact FP64 inverse below is used instead.
        __shared__ unsigned int emax_e;
        // E goes to the Sd region (pair residual; S stays in Sf) or, with the FP64
        // residual, which reads S from Sd, over S in Sf
        float *Ef = factored ? reinterpret_cast<float *>(Sd) : Sf;
        if (threadIdx.x == 0) emax_e = 0u;
        for (int i = threadIdx.x >> 5; i < M; i += blockDim.x >> 5)
            for (int j = threadIdx.x & 31; j < M; j += 32) {
                if (factored) {
                    if (j < i) Ef[i * lda + j] = 0.f;
                } else {
                    Sd[i * lda + j] = (j >= i) ? double(Sf[i * lda + j]) : 0.0;
                }
            }
        __syncthreads();
        unsigned int my = 0u;
        auto put_e = [&](int i, int j, float ef) {
            Ef[i * lda + j] = ef;
            const unsigned int bits = __float_as_uint(fabsf(ef));
            my = bits > my ? bits : my;
        };
        if (factored) {
            tri_residual_df(Sf, Rf, lda, M, put_e);
        } else {
            tri_mm_upper<double>(
                M, [&](int i, int k) { return -Sd[i * lda + k]; }, [&](int k, int j) { return A[k * lda + j]; },
                [](int i, int j) { return i == j ? 1.0 : 0.0; },
                [&](int i, int j, double e) { put_e(i, j, float(e)); });
        }
        atomicMax(&emax_e, my);
        __syncthreads();
        if (__uint_as_float(emax_e) < 1e-3f) {
            auto ef = [&](int k, int j) { return Ef[k * lda + j]; };
            auto zero = [](int, int) { return 0.f; };
            for (int i = threadIdx.x >> 5; i < M; i += blockDim.x >> 5)
                for (int j = threadIdx.x & 31; j < M; j += 32) {
                    if (j < i) C1[i * lda + j] = 0.f;
                }
            tri_mm_upper<float>(M, [&](int i, int k) { return Rf[i * lda + k]; }, ef, zero,
                                [&](int i, int j, float c) { C1[i * lda + j] = c; });
            __syncthreads();
            tri_mm_upper<float>(M, [&](int i, int k) { return C1[i * lda + k]; }, ef, zero,
                                [&](int i, int j, float c2) { A[i * lda + j] += double(C1[i * lda + j] + c2); });
            __syncthreads();
        } else {
            exact = true;
            for (int i = threadIdx.x >> 5; i < M; i += blockDim.x >> 5)
                for (int j = threadIdx.x & 31; j < M; j += 32) {
                    A[i * lda + j] = factored ? ((j >= i) ? double(Sf[i * lda + j]) : 0.0) : Sd[i * lda + j];
                }
            __syncthreads();
        }
    } else {
        for (int i = threadIdx.x >> 5; i < M; i += blockDim.x >> 5)
            for (int j = threadIdx.x & 31; j < M; j += 32) {
                A[i * lda + j] = (j >= i) ? double(Sf[i * lda + j]) : 0.0;
            }
        __syncthreads();
    }
    if (exact) tri_inv_upper_inplace<double>(A, lda, M, t);
    if (pass == 1) {
        for (int i = threadIdx.x >> 5; i < M; i += blockDim.x >> 5)
            for (int j = threadIdx.x & 31; j < M; j += 32) {
                const int idx = i * M + j;
                R1[idx] = (j >= i) ? A[i * lda + j] : 0.0;
            }
    } else {
        // H_{k+1,k} = R2 R1 (upper triangular); B = H^T for the next three-term step.  H is
        // recorded rounded to the basis precision, i.e. exactly as the next step subtracts it.
        for (int i = threadIdx.x >> 5; i < W; i += blockDim.x >> 5)
            for (int j = threadIdx.x & 31; j < W; j += 32) {
                if (i < M && j < M && j >= i) continue;
                if (i < M && j < M) Hs[i * M + j] = 0.0;
                Bout[j * W + i] = 0.f;
            }
        tri_mm_upper<double>(
            M, [&](int i, int k) { return A[i * lda + k]; }, [&](int k, int j) { return __ldg(R1 + k * M + j); },
            [](int, int) { return 0.0; },
            [&](int i, int j, double h) {
                const float ht = float(h);
                Hs[i * M + j] = double(ht);
                Bout[j * W + i] = ht;
            });
    }
}

}  // namespace

int launch_chol_ordered(const double *G, int M, int W, int pass, int step, double inv_thresh2,
                double piv_rel2, double *R1, float *Rinv, double *Hs, float *Bout, Ctrl *ctrl,
                cudaStream_t s) {
    auto bytes_for = [](int m) {
        const bool newton = m <= CHOL_NEWTON_MAX;
        return sizeof(double) * size_t(m) * (m + 1) + sizeof(float) * (size_t(m) * (m + 1) + 2) +
               sizeof(double) * size_t(3 * m + 2) +
               (newton ? (sizeof(double) + 2 * sizeof(float)) * size_t(m) * (m + 1) : 0) +
               sizeof(float) * size_t(tri_inv_tmp_elems(m));
    };
    const size_t smem = bytes_for(M);
    // function-local static: set once, thread-safe
    static const cudaError_t attr = cudaFuncSetAttribute(
        k_chol_ordered, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes_for(128)));
    (void)attr;
    prof_begin(KernelClass::SMALL, s);
    k_chol_ordered<<<1, 256, smem, s>>>(G, M, W, pass, step, inv_thresh2, piv_rel2, R1, Rinv, Hs, Bout, ctrl);
    KB_CUDA_TRY(cudaGetLastError());
    prof_end(KernelClass::SMALL, s, 0, 0);
    return 0;
}

}  // namespace kb
