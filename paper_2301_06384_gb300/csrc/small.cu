// Small dense FP64 kernels and element-wise kernels of the Krylov drivers.
//
//  * k_lanczos_*    scalar recurrences of the global (Algorithm 2) and sequential
//                   (Section 3.3) Lanczos methods: h_kk, h_{k+1,k}, 1/h.
//  * k_tridiag_phi  u = phi(H_m) f_1 for the tridiagonal Lanczos matrices (the projected
//                   step of Algorithm 2; Section 3.3 with phi applied, which its formula omits).
//  * element-wise   unit blocks E_W, node markers, column norms, scaled copies, the
//                   diagonal assembly sum_k u_k Q_k, NaN fill on breakdown.
#include <climits>
#include <type_traits>

#include <cooperative_groups.h>

#include "kb_internal.cuh"
#include "kb_kernels.cuh"

namespace cg = cooperative_groups;

namespace kb {

// ---------------------------------------------------------------- 16-byte vector access
__device__ __forceinline__ void ldv4(const float *p, float (&v)[4]) {
    const float4 t = *reinterpret_cast<const float4 *>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void ldv4(const double *p, double (&v)[4]) {
    const double2 a = reinterpret_cast<const double2 *>(p)[0];
    const double2 b = reinterpret_cast<const double2 *>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void stv4(float *p, const float (&v)[4]) {
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void stv4(double *p, const double (&v)[4]) {
    reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
}
__device__ __forceinline__ void ldv4(const __nv_bfloat16 *p, float (&v)[4]) {
    const uint2 raw = *reinterpret_cast<const uint2 *>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw.y));
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void stv4(__nv_bfloat16 *p, const float (&v)[4]) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]);
    const __nv_bfloat162 b = __floats2bfloat162_rn(v[2], v[3]);
    uint2 raw;
    raw.x = *reinterpret_cast<const unsigned int *>(&a);
    raw.y = *reinterpret_cast<const unsigned int *>(&b);
    *reinterpret_cast<uint2 *>(p) = raw;
}
template <typename T> __device__ __forceinline__ double to_double(T v) { return double(v); }
template <> __device__ __forceinline__ double to_double<__nv_bfloat16>(__nv_bfloat16 v) {
    return double(__bfloat162float(v));
}

// ---------------------------------------------------------------- control / init
__global__ void k_ctrl_init(Ctrl *c, int steps) {
    c->status = KB_OK;
    c->stop = 0;
    c->steps = steps;
    c->breakdown_step = -1;
    c->est_change = -1.0;
    c->from_check = -1;
}

template <typename T>
__global__ void k_scatter(T *block, int64_t ld, NodeChunk ch, T val) {
    const int j = threadIdx.x + blockIdx.x * blockDim.x;
    if (j < ch.cnt) block[int64_t(ch.idx[j]) * ld + ch.col0 + j] = val;
}

__global__ void k_marker(int32_t *marker, NodeChunk ch) {
    const int j = threadIdx.x + blockIdx.x * blockDim.x;
    if (j < ch.cnt) marker[ch.idx[j]] = ch.col0 + j;
}

// out = scale in on the listed 32-row tiles (all rows without a list), 16 bytes at a time
template <typename T>
__global__ void __launch_bounds__(256) k_scale_copy(T *out, const T *in, int64_t n, int W, double scale,
                                                    const int32_t *__restrict__ alist, const int32_t *acount) {
    constexpr int V = 16 / int(sizeof(T));
    const int64_t nt = (n + ACT_ROWS - 1) / ACT_ROWS;
    const int64_t cnt = alist ? int64_t(*acount) : nt;
    for (int64_t it = blockIdx.x; it < cnt; it += gridDim.x) {
        const int64_t r0 = (alist ? int64_t(__ldg(alist + it)) : it) * ACT_ROWS;
        const int64_t rows = n - r0 < ACT_ROWS ? n - r0 : ACT_ROWS;
        for (int64_t i = int64_t(threadIdx.x) * V; i < rows * W; i += 256 * V) {
            uint4 raw = *reinterpret_cast<const uint4 *>(in + r0 * W + i);
            T *v = reinterpret_cast<T *>(&raw);
#pragma unroll
            for (int q = 0; q < V; ++q) v[q] = T(scale * to_double(v[q]));
            *reinterpret_cast<uint4 *>(out + r0 * W + i) = raw;
        }
    }
}

__global__ void k_fill_nan(float *Y, int64_t n, int64_t ldy, int mo, const Ctrl *ctrl) {
    if (ctrl->status == KB_OK) return;
    const float nanv = __int_as_float(0x7fc00000);
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n * mo;
         i += int64_t(gridDim.x) * blockDim.x)
        Y[(i / mo) * ldy + (i % mo)] = nanv;
}

// ---------------------------------------------------------------- full reorthogonalisation
// "Twice is enough" (Kahan's criterion, as given in Parlett's The Symmetric Eigenvalue
// Problem): after one classical Gram-Schmidt pass x_1 = x_0 - Q Q^T x_0, x_1 is orthogonal to
// Q to working precision when ||x_1|| >= ||x_0|| / sqrt(2); otherwise a second pass is
// needed.  Applied column by column to the block: the squared column norms of X before the
// first pass (the diagonal of its Gram) are saved, and after the pass the second one is
// skipped (*skip = 1) when every column kept at least half of its squared norm.
__global__ void k_reorth_save(const double *G, int M, int W, double *d0) {
    for (int i = threadIdx.x; i < M; i += blockDim.x) d0[i] = G[int64_t(i) * W + i];
}
__global__ void k_reorth_decide(const double *G, const double *d0, int M, int W, int32_t *skip) {
    bool ok = true;
    for (int i = threadIdx.x; i < M; i += 32) ok = ok && G[int64_t(i) * W + i] >= 0.5 * d0[i];
    ok = __all_sync(0xffffffffu, ok);
    if (threadIdx.x == 0) *skip = ok ? 1 : 0;
}

int launch_reorth_save(const double *G, int M, int W, double *d0, cudaStream_t s) {
    k_reorth_save<<<1, 128, 0, s>>>(G, M, W, d0);
    count_launches(1);
    KB_CUDA_TRY(cudaGetLastError());
    return 0;
}
int launch_reorth_decide(const double *G, const double *d0, int M, int W, int32_t *skip, cudaStream_t s) {
    k_reorth_decide<<<1, 32, 0, s>>>(G, d0, M, W, skip);
    count_launches(1);
    KB_CUDA_TRY(cudaGetLastError());
    return 0;
}

// ---------------------------------------------------------------- gbl / sbl scalars
// The scalars of a step come from [nparts][W] partial column sums.  A cluster of W / 16 CTAs takes
// 16 columns each (one CTA reading all partials is bound by its SM's L2 bandwidth: alpha / beta at
// W = 64 15.9 / 16.3 us, now 12.3 / 15.1; at W = 128 27.1 / 19.5, now 11.2 / 14.1); the global method's totals meet in distributed shared
// memory.  df: the partials are double-float pairs (FP32 arithmetic), combined on the FP32
// pipe; else doubles.
constexpr int LZ_THREADS = 512;
constexpr int LZ_COLS = 16;

// Sum of the partials' column blockIdx.x * 16 + c into s[c], c < 16, in a fixed order: 32 strided
// subsets of the partials, eight loads in flight per thread, then a fixed-order combination.
__device__ void reduce_cols(const double *parts, int nparts, int W, double *s, int df) {
    __shared__ double tmp[LZ_THREADS / 32][LZ_COLS];
    constexpr int U = 8, NG = LZ_THREADS / LZ_COLS;
    const int c = threadIdx.x % LZ_COLS, g = threadIdx.x / LZ_COLS;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t col = int64_t(blockIdx.x) * LZ_COLS + c;
    if (df) {
        const DF *pp = reinterpret_cast<const DF *>(parts);
        DF a[U];
#pragma unroll
        for (int u = 0; u < U; ++u) a[u] = DF{0.f, 0.f};
        for (int p = g; p < nparts; p += U * NG) {
            DF v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) v[u] = p + u * NG < nparts ? pp[int64_t(p + u * NG) * W + col] : DF{0.f, 0.f};
#pragma unroll
            for (int u = 0; u < U; ++u) df_merge(a[u], v[u]);
        }
#pragma unroll
        for (int u = 1; u < U; ++u) df_merge(a[0], a[u]);
        // the warp's two subsets
        const DF o{__shfl_xor_sync(0xffffffffu, a[0].hi, 16), __shfl_xor_sync(0xffffffffu, a[0].lo, 16)};
        df_merge(a[0], o);
        if (lane < LZ_COLS) reinterpret_cast<DF &>(tmp[warp][c]) = a[0];
    } else {
        double a[U];
#pragma unroll
        for (int u = 0; u < U; ++u) a[u] = 0.0;
        for (int p = g; p < nparts; p += U * NG) {
            double v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) v[u] = p + u * NG < nparts ? parts[int64_t(p + u * NG) * W + col] : 0.0;
#pragma unroll
            for (int u = 0; u < U; ++u) a[u] += v[u];
        }
        double t = a[0];
#pragma unroll
        for (int u = 1; u < U; ++u) t += a[u];
        t += __shfl_xor_sync(0xffffffffu, t, 16);
        if (lane < LZ_COLS) tmp[warp][c] = t;
    }
    __syncthreads();
    if (threadIdx.x < LZ_COLS) {
        if (df) {
            DF t = reinterpret_cast<const DF &>(tmp[0][c]);
            for (int w = 1; w < LZ_THREADS / 32; ++w) df_merge(t, reinterpret_cast<const DF &>(tmp[w][c]));
            s[c] = df_value(t);
        } else {
            double t = 0.0;
            for (int w = 0; w < LZ_THREADS / 32; ++w) t += tmp[w][c];
            s[c] = t;
        }
    }
    __syncthreads();
}

// Sum of s over the columns of all CTAs of the cluster, in rank order, in every CTA (s holds zeros
// in padding columns).
__device__ double cluster_total(const double *s) {
    __shared__ double own, tot;
    cg::cluster_group cl = cg::this_cluster();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int c = 0; c < LZ_COLS; ++c) t += s[c];
        own = t;
    }
    cl.sync();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (unsigned r = 0; r < cl.num_blocks(); ++r) t += *cl.map_shared_rank(&own, r);
        tot = t;
    }
    cl.sync();   // (no CTA leaves while another reads its sum)
    return tot;
}

// Scale factors sigma (Q_k = sigma_k P_k) are rounded to the basis precision when the
// basis is FP32, so that the SpMM applies exactly the sigma the recurrence records.
__device__ __forceinline__ double round_to(double v, int round32) {
    return round32 ? double(float(v)) : v;
}

__global__ void k_lanczos_init(int W, int M, int gbl, int round32, double *sigma, int32_t *alive,
                               double *c1, double *c2) {
    for (int c = threadIdx.x; c < W; c += blockDim.x) {
        const bool live = c < M;
        const double s0 = live ? round_to(gbl ? 1.0 / sqrt(double(M)) : 1.0, round32) : 0.0;
        sigma[c] = s0;
        alive[c] = live ? 1 : 0;
        c1[c] = s0;
        c2[c] = 0.0;
    }
}

// alpha_k = <Q_k, X> (gbl: Frobenius, sbl: per column) from SpMM dot partials of P_k . X
__global__ void __launch_bounds__(LZ_THREADS)
k_lanczos_alpha(const double *parts, int nparts, int W, int M, int gbl, int k, int df, const double *sigma,
                double *alpha, double *a_upd, const Ctrl *ctrl) {
    pdl_wait();
    if (ctrl->stop) return;
    __shared__ double s[LZ_COLS];
    reduce_cols(parts, nparts, W, s, df);
    pdl_trigger();
    const double *sg = sigma + int64_t(k) * W;
    const double tot = gbl ? sg[0] * cluster_total(s) : 0.0;
    if (threadIdx.x < LZ_COLS) {
        const int c = blockIdx.x * LZ_COLS + threadIdx.x;
        const double al = c < M ? (gbl ? tot : sg[c] * s[threadIdx.x]) : 0.0;
        alpha[int64_t(k) * W + c] = al;
        a_upd[c] = al * (gbl ? sg[0] : sg[c]);
    }
}

// beta_{k+1} = ||X|| (gbl: Frobenius, sbl: per column), sigma_{k+1} = 1/beta, and the
// SpMM coefficients of the next step: X = sigma_{k+1} L P_{k+1} - beta_{k+1} sigma_k P_k.
// sigma_{k+1} is rounded to the basis precision and beta_{k+1} is recorded as its exact
// reciprocal, so Q_{k+1} = sigma_{k+1} P_{k+1} = X / beta_{k+1} holds for the stored values.
__global__ void __launch_bounds__(LZ_THREADS)
k_lanczos_beta(const double *parts, int nparts, int W, int M, int gbl, int k, int round32, double thresh,
               double *beta, double *sigma, int32_t *alive, double *c1, double *c2, Ctrl *ctrl) {
    pdl_wait();
    if (ctrl->stop) return;
    __shared__ double s[LZ_COLS];
    reduce_cols(parts, nparts, W, s, round32);
    pdl_trigger();
    const double *sk = sigma + int64_t(k) * W;
    double *sn = sigma + int64_t(k + 1) * W;
    double *bn = beta + int64_t(k + 1) * W;
    const double tot = gbl ? cluster_total(s) : 0.0;   // (a barrier: no CTA has stopped the process before all read stop)
    if (threadIdx.x < LZ_COLS) {
        const int c = blockIdx.x * LZ_COLS + threadIdx.x;
        const double b = sqrt(gbl ? tot : s[threadIdx.x]);
        bool live = c < M && b > thresh;
        if (gbl) {
            if (c == 0 && !(b > thresh)) {
                ctrl->stop = 1;
                ctrl->steps = k + 1;
            }
        } else {
            live = live && alive[c];
            if (!live) alive[c] = 0;
        }
        const double sg = live ? round_to(1.0 / b, round32) : 0.0;
        const double bt = live ? 1.0 / sg : 0.0;
        bn[c] = bt;
        sn[c] = sg;
        c1[c] = sg;
        c2[c] = live ? -bt * sk[c] : 0.0;
    }
}

// u = phi(T) e_1 for each column's tridiagonal T (diag alpha_k, off-diagonal beta_{k+1}),
// then assembly weights omega_k[c] = scale * u_k * sigma_k[c].
//   exp:    Chebyshev series of e^{-t lambda} on [0, Lambda] in T_j(I - 2T/Lambda)
//   spline: s_int solves with the SPD tridiagonal eps I + T (Thomas algorithm; the
//           factorisation is formed once and reused by the s_int solves)
// One CTA per tridiagonal (column c; a single one for the global method), its threads
// parallel over the rows of the three-term recurrence.  The vectors live in shared memory
// when 6 m doubles fit (m <= TRI_SMEM_M), else in the global scratch work (4 m per column).
constexpr int TRI_SMEM_M = 1024;
constexpr int TRI_THREADS = 128;

// Chebyshev series of e^{-t lambda} applied to e_1, terms [j0, j0 + cc.n) of it, for series
// longer than one ChebCoef: V_j (term j) lives in slot j % 3 of the column's global state
// (3 m doubles), the partial sum u in the fourth m doubles (the layout k_tridiag_phi reads
// with u_ready).  A = I - (2/lam) T; V_0 = e_1, V_1 = A e_1, V_j = 2 A V_{j-1} - V_{j-2}.
__global__ void __launch_bounds__(TRI_THREADS) k_tridiag_exp_chunk(int W, int M, int m, int gbl,
                                                                   const double *alpha,
                                                                   const double *beta, double lam,
                                                                   ChebCoef cc, int j0,
                                                                   double *work, const Ctrl *ctrl) {
    const int c = blockIdx.x;
    if (c >= (gbl ? 1 : M)) return;
    const int s = gbl ? ctrl->steps : m;
    double *slot[3] = {work + int64_t(c) * 4 * m, work + int64_t(c) * 4 * m + m, work + int64_t(c) * 4 * m + 2 * m};
    double *u = work + int64_t(c) * 4 * m + 3 * m;
    auto a_of = [&](int k) { return alpha[int64_t(k) * W + c]; };
    auto b_of = [&](int k) { return beta[int64_t(k) * W + c]; };
    const double g = 2.0 / lam;
    for (int q = 0; q < cc.n; ++q) {
        const int j = j0 + q;
        double *vn = slot[j % 3];
        if (j == 0) {
            for (int k = threadIdx.x; k < m; k += blockDim.x) {
                vn[k] = k == 0 ? 1.0 : 0.0;
                u[k] = k == 0 ? cc.d[q] : 0.0;
                slot[1][k] = 0.0;
                slot[2][k] = 0.0;
            }
        } else {
            const double *pc = slot[(j - 1) % 3];
            const double *pp = slot[(j + 1) % 3];   // V_{j-2} (slot (j - 2) % 3)
            for (int k = threadIdx.x; k < s; k += blockDim.x) {
                double tv = a_of(k) * pc[k];
                if (k > 0) tv += b_of(k) * pc[k - 1];
                if (k + 1 < s) tv += b_of(k + 1) * pc[k + 1];
                const double av = pc[k] - g * tv;
                const double v = j == 1 ? av : 2.0 * av - pp[k];
                vn[k] = v;
                u[k] += cc.d[q] * v;
            }
        }
        __syncthreads();
    }
}

// u_ready: the series part of e^{-t T} e_1 was formed by k_tridiag_exp_chunk in work; only
// the bound check and the scaling into omega run here.
__global__ void __launch_bounds__(TRI_THREADS) k_tridiag_phi(int W, int M, int m, int gbl,
                                                             const double *alpha,
                                                             const double *beta,
                                                             const double *sigma, int phi_kind,
                                                             double eps, int s_int, double lam,
                                                             TriCoef tc, double *omega,
                                                             double *work, double *qwork,
                                                             Ctrl *ctrl, double bound, int u_ready) {
    const ChebCoef &cc = tc.cc;
    const int c = blockIdx.x;
    const int ncol = gbl ? 1 : M;
    if (c >= ncol) {
        for (int k = threadIdx.x; k < m; k += blockDim.x) omega[int64_t(k) * W + c] = 0.0;
        return;
    }
    const int s = gbl ? ctrl->steps : m;
    extern __shared__ __align__(16) double tsm[];
    const bool in_smem = m <= TRI_SMEM_M && !u_ready;
    double *v0, *v1, *v2, *u;
    const double *av, *bv;
    int64_t st;   // stride of av / bv
    if (in_smem) {
        v0 = tsm; v1 = v0 + m; v2 = v1 + m; u = v2 + m;
        double *a_s = u + m, *b_s = a_s + m;
        for (int k = threadIdx.x; k < m; k += blockDim.x) {
            a_s[k] = alpha[int64_t(k) * W + c];
            b_s[k] = beta[int64_t(k) * W + c];
        }
        av = a_s; bv = b_s; st = 1;
    } else {
        v0 = work + int64_t(c) * 4 * m; v1 = v0 + m; v2 = v1 + m; u = v2 + m;
        av = alpha + c; bv = beta + c; st = W;
    }
    // b_of(k) couples rows k-1 and k
    auto a_of = [&](int k) { return av[int64_t(k) * st]; };
    auto b_of = [&](int k) { return bv[int64_t(k) * st]; };
    if (!u_ready)
        for (int k = threadIdx.x; k < m; k += blockDim.x) { v0[k] = 0.0; v1[k] = 0.0; v2[k] = 0.0; u[k] = 0.0; }
    __syncthreads();
    if (u_ready) {
        // (series formed in chunks)
    } else if (phi_kind == KB_PHI_EXP) {
        // v0 = e_1, v1 = A e_1, v_{j+1} = 2 A v_j - v_{j-1}, A = I - (2/lam) T
        const double g = 2.0 / lam;
        if (threadIdx.x == 0) { v0[0] = 1.0; u[0] = cc.d[0]; }
        __syncthreads();
        double *pp = v0, *pc = v1, *pn = v2;
        for (int k = threadIdx.x; k < s; k += blockDim.x) {
            double tv = a_of(k) * pp[k];
            if (k > 0) tv += b_of(k) * pp[k - 1];
            if (k + 1 < s) tv += b_of(k + 1) * pp[k + 1];
            pc[k] = pp[k] - g * tv;
            u[k] += cc.d[1] * pc[k];
        }
        __syncthreads();
        for (int j = 2; j < cc.n; ++j) {
            for (int k = threadIdx.x; k < s; k += blockDim.x) {
                double tv = a_of(k) * pc[k];
                if (k > 0) tv += b_of(k) * pc[k - 1];
                if (k + 1 < s) tv += b_of(k + 1) * pc[k + 1];
                pn[k] = 2.0 * (pc[k] - g * tv) - pp[k];
                u[k] += cc.d[j] * pn[k];
            }
            __syncthreads();
            double *t = pp; pp = pc; pc = pn; pn = t;
        }
    } else {
        const QuadRule &q = tc.q;
        if (q.n > 0) {
            // fractional factor: u = sum_j W_j (sigma_j I + T)^{-1} e_1, one node per thread
            // (Thomas algorithm: modified super-diagonal in cq, solution in xq), then the
            // weighted sum per row in a fixed order
            double *qw = qwork + int64_t(c) * 2 * m * q.n;
            for (int j = threadIdx.x; j < q.n; j += blockDim.x) {
                double *cq = qw + int64_t(j) * 2 * m, *xq = cq + m;
                const double sg = q.shift[j];
                double piv = 1.0 / (sg + a_of(0));
                cq[0] = (s > 1) ? b_of(1) * piv : 0.0;
                xq[0] = piv;
                for (int k = 1; k < s; ++k) {
                    piv = 1.0 / (sg + a_of(k) - b_of(k) * cq[k - 1]);
                    cq[k] = (k + 1 < s) ? b_of(k + 1) * piv : 0.0;
                    xq[k] = -b_of(k) * xq[k - 1] * piv;
                }
                for (int k = s - 2; k >= 0; --k) xq[k] -= cq[k] * xq[k + 1];
            }
            __syncthreads();
            for (int k = threadIdx.x; k < s; k += blockDim.x) {
                double acc = 0.0;
                for (int j = 0; j < q.n; ++j) acc = fma(q.weight[j], qw[int64_t(j) * 2 * m + m + k], acc);
                u[k] = acc;
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            // (eps I + T) = L U: v0 = modified super-diagonal, v2 = reciprocal pivots (once);
            // then s_int forward / backward sweeps from rhs = e_1 (or from the fractional factor)
            double den = eps + a_of(0);
            v2[0] = 1.0 / den;
            v0[0] = (s > 1) ? b_of(1) * v2[0] : 0.0;
            for (int k = 1; k < s; ++k) {
                den = eps + a_of(k) - b_of(k) * v0[k - 1];
                v2[k] = 1.0 / den;
                v0[k] = (k + 1 < s) ? b_of(k + 1) * v2[k] : 0.0;
            }
            if (q.n == 0) u[0] = 1.0;
            for (int rep = 0; rep < s_int; ++rep) {
                v1[0] = u[0] * v2[0];
                for (int k = 1; k < s; ++k) v1[k] = (u[k] - b_of(k) * v1[k - 1]) * v2[k];
                u[s - 1] = v1[s - 1];
                for (int k = s - 2; k >= 0; --k) u[k] = v1[k] - v0[k] * u[k + 1];
            }
        }
    }
    __syncthreads();
    // phi(T) e_1 within max phi on [0, Lambda] unless T left the interval (lost orthogonality)
    {
        bool bad = false;
        for (int k = threadIdx.x; k < s; k += blockDim.x)
            if (!(fabs(u[k]) <= bound)) bad = true;
        if (__syncthreads_or(bad) && threadIdx.x == 0)
            atomicCAS(reinterpret_cast<int *>(&ctrl->status), KB_OK, KB_ERR_ORTHOGONALITY);
    }
    // E_W = P_1 and Q_1 = sigma_1 P_1, so Y = (1/sigma_1) [Q_1..Q_m] phi(T) e_1
    // (the sqrt(N) factor of Algorithm 2's final step, for the global method)
    const double scale = 1.0 / sigma[c];
    if (gbl) {
        for (int idx = threadIdx.x; idx < m * W; idx += blockDim.x) {
            const int k = idx / W, c2 = idx % W;
            omega[idx] = (c2 < M && k < s) ? scale * u[k] * sigma[int64_t(k) * W] : 0.0;
        }
    } else {
        for (int k = threadIdx.x; k < m; k += blockDim.x)
            omega[int64_t(k) * W + c] = k < s ? scale * u[k] * sigma[int64_t(k) * W + c] : 0.0;
    }
}

// X[:, c] -= a[c] * P[:, c]; partial column sums of X^2 per CTA.  Rows of tiles beyond
// the frontier limit are zero in X and P and are skipped.
template <typename T, int W>
__global__ void __launch_bounds__(256) k_axpy_colnorm(T *X, const T *P, const double *a, int64_t n,
                                                       double *parts, const Ctrl *ctrl,
                                                       const int32_t *alist, const int32_t *acount,
                                                       ProfCount pc) {
    pdl_wait();
    if (ctrl->stop) return;
    using C = typename Cmp<T>::type;
    constexpr int CG = W / 4;
    constexpr int RPP = 256 / CG;   // rows per pass
    __shared__ double s[RPP][W];
    const int cg = threadIdx.x % CG, rr = threadIdx.x / CG;
    const int c4 = cg * 4;
    C ah[4], al[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        ah[q] = C(a[c4 + q]);
        al[q] = C(a[c4 + q] - double(ah[q]));
    }
    C acc[4] = {0, 0, 0, 0};
    unsigned long long my_rows = 0;
    if (alist) {
        // active 32-row tiles only: RPP rows per pass
        const int cnt = *acount;
        for (int it = blockIdx.x; it < cnt; it += gridDim.x) {
            const int64_t t0 = int64_t(__ldg(alist + it)) * ACT_ROWS;
            for (int sub = rr; sub < ACT_ROWS; sub += RPP) {
                const int64_t row = t0 + sub;
                if (row >= n) break;
                C xv[4], pv[4];
                ldv4(X + row * W + c4, xv);
                ldv4(P + row * W + c4, pv);
                if (cg == 0) ++my_rows;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    xv[q] = xv[q] - fma(ah[q], pv[q], al[q] * pv[q]);
                    if constexpr (!std::is_same<T, C>::value) xv[q] = C(T(xv[q]));
                    acc[q] = fma(xv[q], xv[q], acc[q]);
                }
                stv4(X + row * W + c4, xv);
            }
        }
    }
    // two rows per iteration, 16-byte vector accesses: four loads in flight per thread
    const int64_t stride = int64_t(gridDim.x) * RPP;
    for (int64_t row = int64_t(blockIdx.x) * RPP + rr; !alist && row < n; row += 2 * stride) {
        const int64_t row2 = row + stride;
        const bool second = row2 < n;
        C xv[2][4], pv[2][4];
        ldv4(X + row * W + c4, xv[0]);
        ldv4(P + row * W + c4, pv[0]);
        if (second) {
            ldv4(X + row2 * W + c4, xv[1]);
            ldv4(P + row2 * W + c4, pv[1]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (h && !second) continue;
            if (cg == 0) ++my_rows;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                xv[h][q] = xv[h][q] - fma(ah[q], pv[h][q], al[q] * pv[h][q]);
                // the norm is that of the stored (narrowed) value
                if constexpr (!std::is_same<T, C>::value) xv[h][q] = C(T(xv[h][q]));
                acc[q] = fma(xv[h][q], xv[h][q], acc[q]);
            }
            stv4(X + (h ? row2 : row) * W + c4, xv[h]);
        }
    }
    pdl_trigger();
    if (pc.rows && cg == 0 && my_rows) atomicAdd(pc.rows, my_rows);
    if constexpr (std::is_same<C, float>::value) {
        // double-float column sums on the FP32 pipe; partials written as DF pairs
        DF *sd = reinterpret_cast<DF *>(&s[0][0]);
#pragma unroll
        for (int q = 0; q < 4; ++q) sd[rr * W + c4 + q] = DF{acc[q], 0.f};
        __syncthreads();
        DF *out = reinterpret_cast<DF *>(parts);
        for (int c = threadIdx.x; c < W; c += 256) {
            DF t = sd[c];
            for (int r = 1; r < RPP; ++r) df_merge(t, sd[r * W + c]);
            out[int64_t(blockIdx.x) * W + c] = t;
        }
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) s[rr][c4 + q] = acc[q];
        __syncthreads();
        for (int c = threadIdx.x; c < W; c += 256) {
            double t = 0.0;
            for (int r = 0; r < RPP; ++r) t += s[r][c];
            parts[int64_t(blockIdx.x) * W + c] = t;
        }
    }
}

// Y[i, c] = sum_k omega_k[c] P_k[i, c]  (global / sequential Lanczos assembly); with a
// frontier, block kbase + k is zero in rows whose tile is more than kbase + k hops from W.
// accumulate: Y is added to (the FP32 accumulator starts from Y, so adding the blocks one
// launch at a time gives the same bits as one launch over all of them).
template <typename T, int W>
__global__ void __launch_bounds__(256) k_assemble_diag(const T *basis, int64_t stride, int nblk,
                                                        const double *omega, int64_t n, float *Y,
                                                        int64_t ldy, int mo, const int32_t *tgen,
                                                        int kbase, int accumulate, const Ctrl *ctrl,
                                                        ProfCount pc) {
    constexpr int CG = W / 4;
    constexpr int RPP = 256 / CG;
    using C = typename Cmp<T>::type;
    // blocks of steps after a stop were never written (their weights are zero)
    nblk = min(nblk, max(ctrl->steps - kbase, 0));
    extern __shared__ __align__(16) unsigned char sm_raw[];
    C *som = reinterpret_cast<C *>(sm_raw);     // [nblk][W]
    for (int i = threadIdx.x; i < nblk * W; i += blockDim.x) som[i] = C(omega[i]);
    __syncthreads();
    const int cg = threadIdx.x % CG, rr = threadIdx.x / CG;
    const int c4 = cg * 4;
    unsigned long long my_units = 0;
    for (int64_t row = int64_t(blockIdx.x) * RPP + rr; row < n; row += int64_t(gridDim.x) * RPP) {
        C acc[4] = {0, 0, 0, 0};
        if (accumulate)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (c4 + q < mo) acc[q] = Y[row * ldy + c4 + q];
        const int k0 = tgen ? min(max(__ldg(tgen + row / ACT_ROWS) - kbase, 0), nblk) : 0;
        if (cg == 0) my_units += nblk - k0;
        for (int k = k0; k < nblk; ++k) {
            C pv[4];
            ldv4(basis + int64_t(k) * stride + row * W + c4, pv);
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q] = fma(som[k * W + c4 + q], pv[q], acc[q]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (c4 + q < mo) Y[row * ldy + c4 + q] = acc[q];
    }
    if (pc.nnz && cg == 0 && my_units) atomicAdd(pc.nnz, my_units);
}

template <typename T>
__global__ void k_u_convert(const double *U, int M, int W, int m, T *Ut, const Ctrl *ctrl) {
    // U: (steps*M) x M row-major -> Ut: (m*W) x W, zero padded, zero beyond steps
    const int steps = ctrl->steps;
    for (int64_t idx = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; idx < int64_t(m) * W * W;
         idx += int64_t(gridDim.x) * blockDim.x) {
        const int blk = int(idx / (W * W));
        const int i = int((idx / W) % W), j = int(idx % W);
        double v = 0.0;
        if (blk < steps && i < M && j < M) v = U[(int64_t(blk) * M + i) * M + j];
        Ut[idx] = T(v);
    }
}

// phi(H) F_1 (or phi(T) e_1) must stay within the bound that holds when the projected
// matrix has its spectrum in [0, Lambda]; a NaN or a larger entry means the Lanczos basis
// lost orthogonality, and the solve is marked KB_ERR_ORTHOGONALITY (Y is then NaN-filled).
__global__ void k_check_projected(const double *U, int64_t count, double bound, Ctrl *ctrl) {
    if (ctrl->status != KB_OK) return;
    bool bad = false;
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < count;
         i += int64_t(gridDim.x) * blockDim.x)
        if (!(fabs(U[i]) <= bound)) bad = true;
    if (__syncthreads_or(bad) && threadIdx.x == 0)
        atomicCAS(reinterpret_cast<int *>(&ctrl->status), KB_OK, KB_ERR_ORTHOGONALITY);
}

// ---------------------------------------------------------------- launchers
int launch_check_projected(const double *U, int64_t count, double bound, Ctrl *ctrl, cudaStream_t s) {
    const int grid = int(std::max<int64_t>(1, std::min<int64_t>((count + 255) / 256, int64_t(num_sms()) * 2)));
    k_check_projected<<<grid, 256, 0, s>>>(U, count, bound, ctrl);
    count_launches(1);
    KB_CUDA_TRY(cudaGetLastError());
    return 0;
}

namespace {
__global__ void k_ctrl_snapshot(Ctrl *dst, const Ctrl *src, int k) {
    Ctrl c = *src;
    // once the process stopped (converged, invariant space, breakdown) later checks have
    // nothing to decide: zero steps make the projected kernels return at once
    c.steps = src->stop ? 0 : min(c.steps, k);
    c.stop = 0;
    *dst = c;
}

__global__ void __launch_bounds__(1024) k_conv_check(const double *U, const double *Up, int M,
                                                     const Ctrl *chk, int32_t *prev_steps,
                                                     double tol, Ctrl *ctrl, int buf) {
    if (ctrl->stop) return;   // already stopped (invariant space, breakdown or converged)
    __shared__ double sd[32], sn[32];
    const int steps = chk->steps, ps = *prev_steps;
    const int64_t cnt = int64_t(steps) * M * M, pcnt = int64_t(ps) * M * M;
    double d2 = 0.0, n2 = 0.0;
    for (int64_t i = threadIdx.x; i < cnt; i += blockDim.x) {
        const double u = U[i];
        const double e = u - (i < pcnt ? Up[i] : 0.0);
        d2 = fma(e, e, d2);
        n2 = fma(u, u, n2);
    }
    for (int off = 16; off > 0; off >>= 1) {
        d2 += __shfl_xor_sync(0xffffffffu, d2, off);
        n2 += __shfl_xor_sync(0xffffffffu, n2, off);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { sd[warp] = d2; sn[warp] = n2; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double D = 0.0, N = 0.0;
        for (int w = 0; w < int(blockDim.x >> 5); ++w) { D += sd[w]; N += sn[w]; }
        if (ps > 0) {
            // (a U with NaN or infinite entries has not converged: no change <= tol holds then)
            const double change = N == 0.0 ? 0.0 : isfinite(N) ? sqrt(D) / sqrt(N) : N - N;
            ctrl->est_change = change;
            if (change <= tol) {
                ctrl->stop = 1;
                ctrl->steps = steps;
                ctrl->from_check = buf;   // U of this check is the result: no second solve
            }
        }
        *prev_steps = steps;
    }
}
}  // namespace

int launch_ctrl_snapshot(Ctrl *dst, const Ctrl *src, int k, cudaStream_t s) {
    k_ctrl_snapshot<<<1, 1, 0, s>>>(dst, src, k);
    count_launches(1);
    KB_CUDA_TRY(cudaGetLastError());
    return 0;
}

// The control block the final projected solve runs on: a copy of ctrl with no steps when
// the stopping rule already formed U at its last check (then k_copy_check_u supplies it).
__global__ void k_ctrl_final(Ctrl *dst, const Ctrl *src) {
    Ctrl c = *src;
    if (c.from_check >= 0) c.steps = 0;
    *dst = c;
}
__global__ void k_copy_check_u(const double *Uc, int64_t per, double *U, const Ctrl *ctrl) {
    const int b = ctrl->from_check;
    if (b < 0) return;
    const int64_t cnt = per;   // the check zeroed its whole buffer: copy it all
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < cnt; i += int64_t(gridDim.x) * blockDim.x)
        U[i] = Uc[b * per + i];
}
int launch_ctrl_final(Ctrl *dst, const Ctrl *src, cudaStream_t s) {
    k_ctrl_final<<<1, 1, 0, s>>>(dst, src);
    count_launches(1);
    KB_CUDA_TRY(cudaGetLastError());
    return 0;
}
int launch_copy_check_u(const double *Uc, int64_t per, double *U, const Ctrl *ctrl, cudaStream_t s) {
    const int grid = int(std::max<int64_t>(1, std::min<int64_t>((per + 255) / 256, 4 * int64_t(num_sms()))));
    k_copy_check_u<<<grid, 256, 0, s>>>(Uc, per, U, ctrl);
    count_launches(1);
    KB_CUDA_TRY(cudaGetLastError());
    return 0;
}

int launch_conv_check(const double *U, const double *Up, int M, const Ctrl *chk, int32_t *prev_steps,
                      double tol, Ctrl *ctrl, cudaStream_t s, int buf) {
    prof_begin(KernelClass::SMALL, s);
    k_conv_check<<<1, 1024, 0, s>>>(U, Up, M, chk, prev_steps, tol, ctrl, buf);
    KB_CUDA_TRY(cudaGetLastError());
    prof_end(KernelClass::SMALL, s, 0, 0);
    return 0;
}

int launch_ctrl_init(Ctrl *c, int steps, cudaStream_t s) {
    k_ctrl_init<<<1, 1, 0, s>>>(c, steps);
    count_launches(1);
    return cudaGetLastError() == cudaSuccess ? 0 : cuda_fail(cudaGetLastError(), "k_ctrl_init");
}

template <typename T>
int launch_scatter(T *block, int64_t ld, const int32_t *nodes, int M, int col0, T val, cudaStream_t s) {
    for (int j0 = 0; j0 < M; j0 += NodeChunk::CAP) {
        NodeChunk ch;
        ch.cnt = std::min(NodeChunk::CAP, M - j0);
        ch.col0 = col0 + j0;
        for (int j = 0; j < ch.cnt; ++j) ch.idx[j] = nodes[j0 + j];
        k_scatter<T><<<1, NodeChunk::CAP, 0, s>>>(block, ld, ch, val);
        count_launches(1);
    }
    KB_CUDA_TRY(cudaGetLastError());
    return 0;
}

int launch_marker(int32_t *marker, const int32_t *nodes, int M, cudaStream_t s) {
    for (int j0 = 0; j0 < M; j0 += NodeChunk::CAP) {
        NodeChunk ch;
        ch.cnt = std::min(NodeChunk::CAP, M - j0);
        ch.col0 = j0;
        for (int j = 0; j < ch.cnt; ++j) ch.idx[j] = nodes[j0 + j];
        k_marker<<<1, NodeChunk::CAP, 0, s>>>(marker, ch);
        count_launches(1);
    }
    KB_CUDA_TRY(cudaGetLastError());
    return 0;
}

template <typename T>
int launch_scale_copy(T *out, const T *in, int64_t n, int W, double scale, const int32_t *alist,
                      const int32_t *acount, cudaStream_t s) {
    const int grid = int(std::min<int64_t>((n + ACT_ROWS - 1) / ACT_ROWS, int64_t(num_sms()) * 8));
    k_scale_copy<T><<<std::max(grid, 1), 256, 0, s>>>(out, in, n, W, scale, alist, acount);
    count_launches(1);
    KB_CUDA_TRY(cudaGetLastError());
    return 0;
}

int launch_fill_nan(float *Y, int64_t n, int64_t ldy, int mo, const Ctrl *ctrl, cudaStream_t s) {
    const int grid = int(std::min<int64_t>((n * mo + 255) / 256, int64_t(num_sms()) * 8));
    k_fill_nan<<<std::max(grid, 1), 256, 0, s>>>(Y, n, ldy, mo, ctrl);
    count_launches(1);
    KB_CUDA_TRY(cudaGetLastError());
    return 0;
}

int launch_lanczos_init(int W, int M, int gbl, int round32, double *sigma, int32_t *alive,
                        double *c1, double *c2, cudaStream_t s) {
    k_lanczos_init<<<1, 128, 0, s>>>(W, M, gbl, round32, sigma, alive, c1, c2);
    count_launches(1);
    KB_CUDA_TRY(cudaGetLastError());
    return 0;
}

int launch_lanczos_alpha(const double *parts, int nparts, int W, int M, int gbl, int k, int df,
                         const double *sigma, double *alpha, double *a_upd, const Ctrl *ctrl,
                         cudaStream_t s) {
    prof_begin(KernelClass::SMALL, s);
    KB_CUDA_TRY(launch_dep(k_lanczos_alpha, dim3(W / LZ_COLS), LZ_THREADS, 0, s, W / LZ_COLS, parts, nparts, W, M, gbl, k, df, sigma, alpha, a_upd,
                               ctrl));
    prof_end(KernelClass::SMALL, s, double(nparts) * W * 8, 0);
    return 0;
}

int launch_lanczos_beta(const double *parts, int nparts, int W, int M, int gbl, int k, int round32,
                        double thresh, double *beta, double *sigma, int32_t *alive, double *c1,
                        double *c2, Ctrl *ctrl, cudaStream_t s) {
    prof_begin(KernelClass::SMALL, s);
    KB_CUDA_TRY(launch_dep(k_lanczos_beta, dim3(W / LZ_COLS), LZ_THREADS, 0, s, W / LZ_COLS, parts, nparts, W, M, gbl, k, round32, thresh, beta, sigma,
                               alive, c1, c2, ctrl));
    prof_end(KernelClass::SMALL, s, double(nparts) * W * 8, 0);
    return 0;
}

int launch_tridiag_phi(int W, int M, int m, int gbl, const double *alpha, const double *beta,
                       const double *sigma, int phi_kind, double eps, int s_int, double lam,
                       const TriCoef &tc, double *omega, double *work, double *qwork, Ctrl *ctrl,
                       double bound, cudaStream_t s, const std::vector<double> *series) {
    prof_begin(KernelClass::PROJECTED, s);
    int launches = 1, u_ready = 0;
    if (phi_kind == KB_PHI_EXP && series && int(series->size()) > ChebCoef::CAP) {
        // a series longer than one parameter block: chunks of CAP terms, state in work
        for (size_t j0 = 0; j0 < series->size(); j0 += ChebCoef::CAP) {
            ChebCoef cc{};
            cc.n = int(std::min<size_t>(ChebCoef::CAP, series->size() - j0));
            for (int q = 0; q < cc.n; ++q) cc.d[q] = (*series)[j0 + q];
            k_tridiag_exp_chunk<<<gbl ? 1 : W, TRI_THREADS, 0, s>>>(W, M, m, gbl, alpha, beta, lam, cc,
                                                                    int(j0), work, ctrl);
            ++launches;
        }
        u_ready = 1;
    }
    const size_t smem = (m <= TRI_SMEM_M && !u_ready) ? sizeof(double) * 6 * size_t(m) : 0;
    static const cudaError_t attr = cudaFuncSetAttribute(
        k_tridiag_phi, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sizeof(double) * 6 * TRI_SMEM_M));
    (void)attr;
    k_tridiag_phi<<<gbl ? 1 : W, TRI_THREADS, smem, s>>>(W, M, m, gbl, alpha, beta, sigma,
                                                         phi_kind, eps, s_int, lam, tc, omega,
                                                         work, qwork, ctrl, bound, u_ready);
    KB_CUDA_TRY(cudaGetLastError());
    prof_end(KernelClass::PROJECTED, s, 0, 0, launches);
    return 0;
}

template <typename T>
int launch_axpy_colnorm(int W, T *X, const T *P, const double *a, int64_t n, double *parts,
                        int *grid_out, const Ctrl *ctrl, int64_t M_alg, cudaStream_t s,
                        const int32_t *alist, const int32_t *acount) {
    const int rpp = 256 / (W / 4);
    const int grid = int(std::min<int64_t>((n + rpp - 1) / rpp, int64_t(num_sms()) * 4));
    *grid_out = std::max(grid, 1);
    const ProfCount pc = prof_begin(KernelClass::ROWBLOCK, s);
    cudaError_t err = cudaSuccess;
    switch (W) {
        case 16: err = launch_dep(k_axpy_colnorm<T, 16>, dim3(*grid_out), 256, 0, s, 0, X, P, a, n, parts, ctrl, alist, acount, pc); break;
        case 32: err = launch_dep(k_axpy_colnorm<T, 32>, dim3(*grid_out), 256, 0, s, 0, X, P, a, n, parts, ctrl, alist, acount, pc); break;
        case 64: err = launch_dep(k_axpy_colnorm<T, 64>, dim3(*grid_out), 256, 0, s, 0, X, P, a, n, parts, ctrl, alist, acount, pc); break;
        case 128: err = launch_dep(k_axpy_colnorm<T, 128>, dim3(*grid_out), 256, 0, s, 0, X, P, a, n, parts, ctrl, alist, acount, pc); break;
        default: return fail(KB_ERR_ARG, "bad width");
    }
    KB_CUDA_TRY(err);
    const double row = double(M_alg) * sizeof(T);
    prof_end(KernelClass::ROWBLOCK, s, 3.0 * double(n) * row, 3.0 * double(n) * M_alg, 1, 3.0 * row,
             0.0, 3.0 * M_alg, 0.0);
    return 0;
}

int axpy_max_grid() { return num_sms() * 4; }

#define KB_ASM_DIAG(WW)                                                                       \
    do {                                                                                      \
        cudaFuncSetAttribute(k_assemble_diag<T, WW>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                             int(smem));                                                      \
        k_assemble_diag<T, WW><<<grid, 256, smem, s>>>(basis, stride, nblk, omega, n, Y, ldy, mo,  \
                                                       tgen, kbase, accumulate, ctrl, pc);    \
    } while (0)

template <typename T>
int launch_assemble_diag(int W, const T *basis, int64_t stride, int nblk, const double *omega,
                         int64_t n, float *Y, int64_t ldy, int mo, int64_t M_alg,
                         const int32_t *tgen, const Ctrl *ctrl, cudaStream_t s, int kbase, int accumulate) {
    const int rpp = 256 / (W / 4);
    const int grid = std::max(1, int(std::min<int64_t>((n + rpp - 1) / rpp, int64_t(num_sms()) * 8)));
    const size_t smem = sizeof(typename Cmp<T>::type) * size_t(nblk) * W;
    if (smem > 200 * 1024) return fail(KB_ERR_UNSUPPORTED, "too many blocks for the diagonal assembly");
    const ProfCount pc = prof_begin(KernelClass::ASSEMBLE, s);
    switch (W) {
        case 16: KB_ASM_DIAG(16); break;
        case 32: KB_ASM_DIAG(32); break;
        case 64: KB_ASM_DIAG(64); break;
        case 128: KB_ASM_DIAG(128); break;
        default: return fail(KB_ERR_ARG, "bad width");
    }
    KB_CUDA_TRY(cudaGetLastError());
    prof_end(KernelClass::ASSEMBLE, s, double(nblk) * n * M_alg * sizeof(T) + double(n) * M_alg * 4,
             2.0 * nblk * double(n) * M_alg, 1, 0.0, double(M_alg) * sizeof(T), 0.0,
             double(n) * M_alg * 4);
    return 0;
}

template <typename T>
int launch_u_convert(const double *U, int M, int W, int m, T *Ut, const Ctrl *ctrl, cudaStream_t s) {
    const int64_t cnt = int64_t(m) * W * W;
    const int grid = int(std::min<int64_t>((cnt + 255) / 256, 1024));
    k_u_convert<T><<<std::max(grid, 1), 256, 0, s>>>(U, M, W, m, Ut, ctrl);
    count_launches(1);
    KB_CUDA_TRY(cudaGetLastError());
    return 0;
}

#define KB_INST(T)                                                                              \
    template int launch_scatter<T>(T *, int64_t, const int32_t *, int, int, T, cudaStream_t);   \
    template int launch_scale_copy<T>(T *, const T *, int64_t, int, double, const int32_t *,    \
                                      const int32_t *, cudaStream_t);                           \
    template int launch_axpy_colnorm<T>(int, T *, const T *, const double *, int64_t, double *,  \
                                        int *, const Ctrl *, int64_t,                           \
                                        cudaStream_t, const int32_t *, const int32_t *);        \
    template int launch_assemble_diag<T>(int, const T *, int64_t, int, const double *, int64_t, \
                                         float *, int64_t, int, int64_t, const int32_t *,       \
                                         const Ctrl *, cudaStream_t, int, int);                             \
    template int launch_u_convert<T>(const double *, int, int, int, T *, const Ctrl *, cudaStream_t);
KB_INST(float)
KB_INST(double)
#undef KB_INST
// BF16 blocks: element-wise kernels on the stored type (small matrices stay FP32)
template int launch_scatter<__nv_bfloat16>(__nv_bfloat16 *, int64_t, const int32_t *, int, int,
                                           __nv_bfloat16, cudaStream_t);
template int launch_scale_copy<__nv_bfloat16>(__nv_bfloat16 *, const __nv_bfloat16 *, int64_t, int,
                                              double, const int32_t *, const int32_t *, cudaStream_t);
template int launch_axpy_colnorm<__nv_bfloat16>(int, __nv_bfloat16 *, const __nv_bfloat16 *,
                                                const double *, int64_t, double *, int *,
                                                const Ctrl *, int64_t,
                                                cudaStream_t, const int32_t *, const int32_t *);
template int launch_assemble_diag<__nv_bfloat16>(int, const __nv_bfloat16 *, int64_t, int,
                                                 const double *, int64_t, float *, int64_t, int,
                                                 int64_t, const int32_t *, const Ctrl *, cudaStream_t, int, int);

}  // namespace kb
