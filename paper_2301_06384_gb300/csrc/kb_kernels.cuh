// Launchers of the small / element-wise / projected-problem kernels (internal).
#pragma once

#include <algorithm>

#include "kb_internal.cuh"

namespace kb {

// Up to CAP node indices passed by value to a kernel (no host-to-device copy needed).
struct NodeChunk {
    static constexpr int CAP = 256;
    int32_t idx[CAP];
    int32_t cnt;
    int32_t col0;
};

// Chebyshev coefficients d_0..d_{n-1} passed by value (sum_j d_j T_j, no halving).
struct ChebCoef {
    static constexpr int CAP = 440;
    int32_t n;
    double d[CAP];
};

// Rational (quadrature) form of the fractional spline power, used for non-integer s:
//   (eps + lambda)^{-s} = (eps + lambda)^{-s_int} * sum_k weight_k / (shift_k + lambda),
// s_int = floor(s); the sum approximates (eps + lambda)^{-alpha}, alpha = s - s_int, on
// [0, lam] by Gauss-Jacobi quadrature of the Stieltjes integral of z^{-alpha}
// (quadrature.cu).  n = 0 when s is an integer.  Passed to kernels by value.
struct QuadRule {
    static constexpr int CAP = 240;   // keeps the struct under 4 KB of kernel parameters
    int32_t n;
    int32_t s_int;
    double shift[CAP];
    double weight[CAP];
};
// Fills q for (eps, s) on the spectral interval [0, lam] such that the relative error of the
// sum on [0, lam] is at most tol (checked on a grid); KB_ERR_UNSUPPORTED when CAP nodes do
// not reach tol, KB_ERR_ARG for bad arguments.  Host only.
int spline_quadrature(double eps, double s, double lam, double tol, QuadRule &q);

// Coefficients of the projected step of gbl / sbl passed to the tridiagonal kernel: the
// Chebyshev series of e^{-t lambda} (diffusion kernel) or, for the spline kernel with
// non-integer s, the quadrature rule of the fractional power.
struct TriCoef {
    union {
        ChebCoef cc;
        QuadRule q;
    };
};
static_assert(sizeof(TriCoef) <= 3900, "projected-step coefficients must fit the 4 KB kernel parameter space");

int launch_ctrl_init(Ctrl *c, int steps, cudaStream_t s);
// dst = src with steps = min(src->steps, k) (the projected problem of the first k steps),
// or 0 once src stopped
int launch_ctrl_snapshot(Ctrl *dst, const Ctrl *src, int k, cudaStream_t s);
// Stopping rule of the serving workload: with steps = chk->steps and p = *prev_steps,
// stops ctrl (stop = 1, steps) when p > 0 and ||U - [Up; 0]||_F <= tol ||U||_F (U, Up:
// (steps M) x M and (p M) x M row-major); then *prev_steps = steps.  No-op once ctrl stopped.
// buf: index of U among the alternating check buffers; recorded in ctrl->from_check when the
// check stops the process.
int launch_conv_check(const double *U, const double *Up, int M, const Ctrl *chk, int32_t *prev_steps,
                      double tol, Ctrl *ctrl, cudaStream_t s, int buf);
// dst = src, with steps = 0 when src->from_check >= 0 (the final projected solve is then
// skipped); launch_copy_check_u copies that check's U (buffers of per doubles) into U.
int launch_ctrl_final(Ctrl *dst, const Ctrl *src, cudaStream_t s);
int launch_copy_check_u(const double *Uc, int64_t per, double *U, const Ctrl *ctrl, cudaStream_t s);
template <typename T>
int launch_scatter(T *block, int64_t ld, const int32_t *nodes, int M, int col0, T val, cudaStream_t s);
int launch_marker(int32_t *marker, const int32_t *nodes, int M, cudaStream_t s);
template <typename T>
int launch_scale_copy(T *out, const T *in, int64_t n, int W, double scale, const int32_t *alist,
                      const int32_t *acount, cudaStream_t s);   // the listed tiles, or all rows
int launch_fill_nan(float *Y, int64_t n, int64_t ldy, int mo, const Ctrl *ctrl, cudaStream_t s);

template <typename T>
int launch_chol(const double *G, int M, int W, int pass, int step, double inv_thresh2,
                double piv_rel2, double *R1, T *Rinv, double *Hs, T *Bout, Ctrl *ctrl,
                cudaStream_t s);

// FP32 solves with full reorthogonalisation (chol_ordered.cu)
int launch_chol_ordered(const double *G, int M, int W, int pass, int step, double inv_thresh2,
                        double piv_rel2, double *R1, float *Rinv, double *Hs, float *Bout, Ctrl *ctrl,
                        cudaStream_t s);

int launch_lanczos_init(int W, int M, int gbl, int round32, double *sigma, int32_t *alive,
                        double *c1, double *c2, cudaStream_t s);
int launch_lanczos_alpha(const double *parts, int nparts, int W, int M, int gbl, int k, int df,
                         const double *sigma, double *alpha, double *a_upd, const Ctrl *ctrl,
                         cudaStream_t s);
int launch_lanczos_beta(const double *parts, int nparts, int W, int M, int gbl, int k, int round32,
                        double thresh, double *beta, double *sigma, int32_t *alive, double *c1,
                        double *c2, Ctrl *ctrl, cudaStream_t s);
// phi(T) e_1 per tridiagonal T (one for gbl, one per column for sbl).  Spline kernel:
// (eps I + T)^{-s_int} applied after the fractional factor sum_k W_k (sigma_k I + T)^{-1}
// when tc.q.n > 0; qwork: 2 m tc.q.n doubles per column (nullptr when tc.q.n == 0).
// series: the full Chebyshev series of e^{-t lambda} (diffusion kernel); when it is longer
// than one ChebCoef it is applied in chunks (state in work, 4 m doubles per column) and tc.cc
// is not used.
int launch_tridiag_phi(int W, int M, int m, int gbl, const double *alpha, const double *beta,
                       const double *sigma, int phi_kind, double eps, int s_int, double lam,
                       const TriCoef &tc, double *omega, double *work, double *qwork, Ctrl *ctrl,
                       double bound, cudaStream_t s, const std::vector<double> *series = nullptr);
template <typename T>
int launch_axpy_colnorm(int W, T *X, const T *P, const double *a, int64_t n, double *parts,
                        int *grid_out, const Ctrl *ctrl, int64_t M_alg, cudaStream_t s,
                        const int32_t *alist = nullptr, const int32_t *acount = nullptr);
int axpy_max_grid();
template <typename T>
int launch_assemble_diag(int W, const T *basis, int64_t stride, int nblk, const double *omega,
                         int64_t n, float *Y, int64_t ldy, int mo, int64_t M_alg,
                         const int32_t *tgen, const Ctrl *ctrl, cudaStream_t s, int kbase = 0,
                         int accumulate = 0);

// Frontier restriction (frontier.cu).  The arrays of one solve; see kb_internal.cuh for the
// meaning of gen, tgen, alist and acount.
struct FrontierBufs {
    uint8_t *gen = nullptr;
    int32_t *tgen = nullptr, *alist = nullptr, *acount = nullptr;
    int32_t *lists = nullptr;          // levels + 1 lists of nt tiles
    // of the search alone:
    unsigned char *zeroed = nullptr;   // qlev, tcnt (the barrier behind it) and vis: cleared first
    size_t zero_bytes = 0;
    int32_t *qlev = nullptr, *tcnt = nullptr, *queue = nullptr;
    int32_t *sync = nullptr;           // barrier count, error flag
    uint32_t *vis = nullptr;
    int levels = 0;
    int64_t nt = 0;
    // the tiles within k hops in index order, and their number (device)
    const int32_t *list(int k) const { return lists + (k < levels ? k : levels) * nt; }
    const int32_t *count(int k) const { return acount + (k < levels ? k : levels); }
};
// Lays the arrays out from base (nullptr: sizes only) for a search of `levels` hops; *bytes
// receives their size.  search: frontier_search_bytes(n) bytes that only launch_frontier uses (the
// solves give it block memory, which the steps write afterwards).
size_t frontier_search_bytes(int64_t n);
void plan_frontier(FrontierBufs &f, int64_t n, int levels, unsigned char *base, size_t *bytes, unsigned char *search);
// Hop distances up to f.levels from the nodes, and the tile lists; every row at distance 0 when a
// barrier of the search runs out of its polls.
int launch_frontier(const GraphDev &g, FrontierBufs &f, const int32_t *nodes, int M, cudaStream_t s,
                    int spins = GRID_BARRIER_SPINS);
// Zeros on the tiles within f.levels hops: see k_zero_tiles.
int launch_zero_tiles(void *blocks, int64_t block_bytes, int nblk, int row_bytes, int64_t n, bool ring,
                      const FrontierBufs &f, cudaStream_t s);
template <typename T>
int launch_u_convert(const double *U, int M, int W, int m, T *Ut, const Ctrl *ctrl, cudaStream_t s);

// Projected problem of the classical block Lanczos method (FP64, block tridiagonal H_m).
// Hdf: nullptr for the FP64 recurrence; else 2 m M (M + 1) doubles of scratch for H as floats, and
// the recurrence runs in double-float on the FP32 pipe (the FP32 and BF16 modes), with sync (two
// words of scratch) in one cooperative launch.  kmax: a host-side bound on ctrl->steps (0: m).
// proc: control block of the process, stopped with KB_ERR_CUDA when a barrier of that launch runs
// out of its polls.
int launch_cheb_bt(const double *Hd, const double *Hs, int M, int m, double lam,
                   const std::vector<double> &d, double *V0, double *V1, double *V2, double *U,
                   const Ctrl *ctrl, cudaStream_t s, double *Hdf = nullptr, int32_t *sync = nullptr,
                   int kmax = 0, Ctrl *proc = nullptr, int spins = GRID_BARRIER_SPINS);
// U = (eps I + H_m)^{-s} F_1.  Integer s: s_int block Cholesky solves (q == nullptr or
// q->n == 0).  Non-integer s: the quadrature rule q gives the fractional factor
// sum_k W_k (sigma_k I + H_m)^{-1} F_1, one block Cholesky factorisation and solve per node
// (qbatch nodes at a time, one CTA each, in qscr: qbatch * bt_quad_node_doubles(M, m)
// doubles), then s_int solves with eps I + H_m.
__host__ __device__ inline size_t bt_quad_node_doubles(int M, int m) {
    return 3 * size_t(m) * M * M + size_t(m) * M;   // Ld, Ls, Y blocks and reciprocal diagonals
}
// The factors of eps I + H, kept from one stopping-rule check to the next: m blocks of M x M each, Ls
// two.
struct SplineBufs {
    double *Ri, *RiT, *Y, *GT, *K, *Ls;
};
// Blocks r0 .. kmax - 1 are factored now (0: all m), those before r0 were by an earlier call with
// the same buffers; y0 likewise for the forward solutions of the first solve.  fc: the control
// block of the process (its steps bound the blocks); ctrl: that of this solve.
int launch_bt_spline(const double *Hd, const double *Hs, int M, int m, double eps, int s_int,
                     const SplineBufs &b, double *U, const Ctrl *fc, const Ctrl *ctrl, cudaStream_t s,
                     const QuadRule *q, double *qscr, int qbatch, int r0, int y0, int kmax);
// Blocks r0 .. kmax - 1 of that factorisation alone.
int launch_bt_factor(const double *Hd, const double *Hs, int M, double eps, const SplineBufs &b, const Ctrl *fc,
                     cudaStream_t s, int r0, int kmax);

// Full reorthogonalisation: save the diagonal of the Gram of X before the first pass; after
// it, *skip = 1 when every column kept at least half of its squared norm (the second pass is
// then not needed).
int launch_reorth_save(const double *G, int M, int W, double *d0, cudaStream_t s);
int launch_reorth_decide(const double *G, const double *d0, int M, int W, int32_t *skip, cudaStream_t s);

// Graph utilities.
int launch_gershgorin(const GraphDev &g, double *out, cudaStream_t s);

// Marks the solve KB_ERR_ORTHOGONALITY when |U| exceeds bound or is NaN.
int launch_check_projected(const double *U, int64_t count, double bound, Ctrl *ctrl, cudaStream_t s);

}  // namespace kb
