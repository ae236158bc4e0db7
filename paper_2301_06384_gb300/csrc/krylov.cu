// The five block Krylov drivers and the kb_krylov_apply entry points.
//
//   cbl   Algorithm 1 (classical block Lanczos) with CholeskyQR2 for the reduced QR of
//         each new block and the FP64 projected problem U = phi(H_m) F_1.
//   gbl   Algorithm 2 (global block Lanczos), Frobenius inner products.
//   sbl   Section 3.3 (one ordinary Lanczos per column), run for all columns at once.
//   cheb  Section 3.4: the degree-m Lobatto interpolant applied by Clenshaw's backward
//         recurrence (same polynomial as the forward three-term recurrence; 3 block
//         reads/writes per product instead of 5).
//   cheb2 Section 3.4.1: the interpolant of sqrt(phi) of degree floor(m/2) applied twice.
//
// Every step runs on the device; the host only enqueues work (breakdown and early stops travel
// through a device control block).  It waits for the device in the middle of a solve only where
// that has a stopping rule and reports to the caller (CheckWatch).
#include "kb_internal.cuh"
#include "kb_kernels.cuh"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <limits>
#include <memory>
#include <mutex>
#include <type_traits>

namespace kb {

// ---------------------------------------------------------------- host coefficient math
// e^{-t lambda} on [0, lam] as sum_k d_k T_k(1 - 2 lambda / lam):  with rho = t lam / 2,
// e^{-t lambda} = e^{-rho} e^{rho x} and e^{rho x} = I_0(rho) + 2 sum_k I_k(rho) T_k(x)
// (modified Bessel functions).  e^{-|rho|} I_k(|rho|) is computed by Miller's backward
// recurrence I_{k-1} = I_{k+1} + (2k/a) I_k, normalised by I_0 + 2 sum_k I_k = e^{a}.
std::vector<double> exp_series_coeffs(double t, double lam, double tol) {
    const double rho = 0.5 * t * lam;
    const double a = std::fabs(rho);
    if (a < 1e-300) return {1.0, 0.0};
    const int kmax = int(std::ceil(a + 12.0 * std::sqrt(a) + 60.0));
    std::vector<double> b(kmax + 2, 0.0);
    b[kmax + 1] = 0.0;
    b[kmax] = 1e-280;
    for (int k = kmax; k >= 1; --k) {
        b[k - 1] = b[k + 1] + (2.0 * k / a) * b[k];
        if (b[k - 1] > 1e250) {
            for (int q = k - 1; q <= kmax + 1; ++q) b[q] *= 1e-250;
        }
    }
    double S = b[0];
    for (int k = 1; k <= kmax; ++k) S += 2.0 * b[k];
    std::vector<double> d(kmax + 1);
    const double growth = rho < 0 ? std::exp(2.0 * a) : 1.0;
    double total = 0.0;
    for (int k = 0; k <= kmax; ++k) {
        double v = (k == 0 ? 1.0 : 2.0) * (b[k] / S) * growth;
        if (rho < 0 && (k & 1)) v = -v;
        d[k] = v;
        total += std::fabs(v);
    }
    int last = 1;
    for (int k = 0; k <= kmax; ++k)
        if (std::fabs(d[k]) > tol * total) last = std::max(last, k);
    d.resize(last + 1);
    return d;
}

// phi (or sqrt(phi)) at a point.
static double phi_value(kb_phi phi, const kb_params &p, double lam, bool sqrt_phi) {
    if (phi == KB_PHI_EXP) return std::exp(-(sqrt_phi ? 0.5 * p.t : p.t) * lam);
    return std::pow(p.eps + lam, -(sqrt_phi ? 0.5 * p.s : p.s));
}

// Eq. (chebcoeff) read as interpolation at the Chebyshev-Lobatto points:
//   c_k = (2/m) sum_{j=0..m}'' f(lambda_j) cos(pi j k / m),  lambda_j = lam/2 (1 - cos(pi j/m)),
// the double prime halving the j = 0 and j = m terms.  The series sum_k'' c_k T_k (c_0 and
// c_m halved) interpolates f on the grid.
// f and c: caller arrays of m + 1 doubles (f receives the samples); no allocation, so the
// fixed-scratch entry point shares it.
void lobatto_coeffs_into(kb_phi phi, const kb_params &p, int m, double lam, bool sqrt_phi, double *f,
                         double *c) {
    for (int j = 0; j <= m; ++j)
        f[j] = phi_value(phi, p, 0.5 * lam * (1.0 - std::cos(M_PI * j / m)), sqrt_phi);
    for (int k = 0; k <= m; ++k) {
        double s = 0.0;
        for (int j = 0; j <= m; ++j) {
            const double wj = (j == 0 || j == m) ? 0.5 : 1.0;
            // cos(pi j k / m) with the argument reduced mod 2m for accuracy
            const long r = (long(j) * k) % (2L * m);
            s += wj * f[j] * std::cos(M_PI * double(r) / m);
        }
        c[k] = 2.0 / m * s;
    }
}

std::vector<double> lobatto_coeffs(kb_phi phi, const kb_params &p, int m, double lam, bool sqrt_phi) {
    std::vector<double> f(m + 1), c(m + 1);
    lobatto_coeffs_into(phi, p, m, lam, sqrt_phi, f.data(), c.data());
    return c;
}

// The kernel choice and its parameters (Section 2.4): t finite for e^{-t lambda}; eps > 0 and
// s > 0, both finite, for (eps + lambda)^{-s}.
int validate_phi(kb_phi phi, const kb_params &p) {
    if (phi == KB_PHI_EXP) {
        if (!std::isfinite(p.t)) return fail(KB_ERR_ARG, "t not finite");
    } else if (phi == KB_PHI_SPLINE) {
        if (!(p.eps > 0) || !std::isfinite(p.eps)) return fail(KB_ERR_ARG, "eps must be > 0");
        if (!(p.s > 0) || !std::isfinite(p.s)) return fail(KB_ERR_ARG, "s must be > 0");
    } else {
        return fail(KB_ERR_ARG, "bad phi");
    }
    return KB_OK;
}

// ---------------------------------------------------------------- workspace
namespace {
struct Arena {
    char *base = nullptr;
    size_t off = 0;
    template <typename T>
    T *take(size_t count) {
        const size_t bytes = (count * sizeof(T) + 255) & ~size_t(255);
        T *p = reinterpret_cast<T *>(base ? base + off : nullptr);
        off += bytes;
        return p;
    }
    // `count` values of block memory, which also serves the search for reached rows
    template <typename T>
    T *take_blocks(size_t count, int64_t n, bool restricted) {
        blocks = base ? reinterpret_cast<unsigned char *>(base + off) : nullptr;
        return reinterpret_cast<T *>(take<char>(std::max(count * sizeof(T), restricted ? frontier_search_bytes(n) : 0)));
    }
    // hops: the last step whose products the search has to cover
    void frontier(FrontierBufs &f, int64_t n, int hops) {
        size_t bytes = 0;
        plan_frontier(f, n, hops + 1, base ? reinterpret_cast<unsigned char *>(base + off) : nullptr, &bytes, blocks);
        off += bytes;
    }
    unsigned char *blocks = nullptr;
};

void ensure_pool(int dev) {
    // once per device; callers may run on several host threads (the serving workers)
    static std::mutex mu;
    static std::vector<int> done;
    std::lock_guard<std::mutex> lk(mu);
    if (std::find(done.begin(), done.end(), dev) != done.end()) return;
    cudaMemPool_t pool;
    if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
        uint64_t thr = std::numeric_limits<uint64_t>::max();
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
    }
    done.push_back(dev);
}

// What a stopping-rule solve that reports to its caller (info) reads back while it runs: the
// control block after a check, in pinned host memory, so that the host stops enqueueing the
// steps of a process that has stopped (with m = 100 and a stop at step 24 three quarters of the
// launches did nothing; four requests on Barabasi-Albert graphs of 23535 rows 35.4 -> 31.6 ms,
// on a geometric graph of 55392 rows, which the GPU bounds, 69.2 -> 69.1 ms).  64 slots for the
// process, allocated once and returned after each solve; a solve that finds none free enqueues
// all steps.
class CheckWatch {
  public:
    explicit CheckWatch(bool wanted) {
        if (!wanted) return;
        {
            std::lock_guard<std::mutex> lk(mu());
            Pool &p = pool();
            if (!p.tried) {
                p.tried = true;
                void *mem = nullptr;
                // (an allocation must not disturb a capture that another thread has begun)
                cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
                cudaThreadExchangeStreamCaptureMode(&mode);
                if (cudaHostAlloc(&mem, sizeof(Ctrl) * 64, cudaHostAllocPortable) == cudaSuccess) p.base = static_cast<Ctrl *>(mem);
                else (void)cudaGetLastError();
                cudaThreadExchangeStreamCaptureMode(&mode);
            }
            for (int i = 0; p.base && i < 64 && slot_ < 0; ++i)
                if (!p.used[i]) {
                    p.used[i] = true;
                    slot_ = i;
                }
        }
        if (slot_ >= 0 && cudaEventCreateWithFlags(&ev_, cudaEventDisableTiming) != cudaSuccess) {
            (void)cudaGetLastError();
            ev_ = nullptr;
        }
    }
    ~CheckWatch() {
        if (pending_) cudaEventSynchronize(ev_);   // the copy into the slot must not outlive it
        if (ev_) cudaEventDestroy(ev_);
        if (slot_ >= 0) {
            std::lock_guard<std::mutex> lk(mu());
            pool().used[slot_] = false;
        }
    }
    CheckWatch(const CheckWatch &) = delete;
    CheckWatch &operator=(const CheckWatch &) = delete;
    // after the launches of a check
    void record(const Ctrl *ctrl, cudaStream_t s) {
        if (!ev_ || pending_) return;
        pending_ = cudaMemcpyAsync(&host(), ctrl, sizeof(Ctrl), cudaMemcpyDeviceToHost, s) == cudaSuccess &&
                   cudaEventRecord(ev_, s) == cudaSuccess;
    }
    // whether the process had stopped at the recorded check (waits for that)
    bool stopped() {
        if (!pending_) return false;
        pending_ = false;
        return cudaEventSynchronize(ev_) == cudaSuccess && host().stop != 0;
    }
    const Ctrl &seen() const { return pool().base[slot_]; }

  private:
    struct Pool {
        Ctrl *base = nullptr;
        bool used[64] = {};
        bool tried = false;
    };
    static std::mutex &mu() {
        static std::mutex m;
        return m;
    }
    static Pool &pool() {
        static Pool p;
        return p;
    }
    Ctrl &host() { return pool().base[slot_]; }
    int slot_ = -1;
    cudaEvent_t ev_ = nullptr;
    bool pending_ = false;
};

// A second stream of one solve, for work that the next steps do not need.  The destructor
// makes the solve's stream wait for what is left there, so that scratch freed on that stream
// afterwards is no longer in use.  Not used while the stream is being captured.
class SideStream {
  public:
    SideStream(bool wanted, cudaStream_t main) : main_(main) {
        if (!wanted) return;
        cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
        int prio = 0;
        if (cudaStreamIsCapturing(main, &st) != cudaSuccess || st != cudaStreamCaptureStatusNone ||
            cudaStreamGetPriority(main, &prio) != cudaSuccess ||
            cudaStreamCreateWithPriority(&side_, cudaStreamNonBlocking, prio) != cudaSuccess) {
            (void)cudaGetLastError();
            side_ = nullptr;
            return;
        }
        if (cudaEventCreateWithFlags(&ready_, cudaEventDisableTiming) != cudaSuccess ||
            cudaEventCreateWithFlags(&done_, cudaEventDisableTiming) != cudaSuccess) {
            (void)cudaGetLastError();
            release();
        }
    }
    ~SideStream() {
        if (pending_ && join() != KB_OK) cudaStreamSynchronize(side_);
        release();
    }
    SideStream(const SideStream &) = delete;
    SideStream &operator=(const SideStream &) = delete;
    explicit operator bool() const { return side_ != nullptr; }
    cudaStream_t stream() const { return side_; }
    // the work enqueued on the side stream from here on follows what the main one holds now
    int fork() {
        KB_CUDA_TRY(cudaEventRecord(ready_, main_));
        KB_CUDA_TRY(cudaStreamWaitEvent(side_, ready_, 0));
        pending_ = true;
        return KB_OK;
    }
    // the main stream waits for the side one
    int join() {
        if (!pending_) return KB_OK;
        KB_CUDA_TRY(cudaEventRecord(done_, side_));
        KB_CUDA_TRY(cudaStreamWaitEvent(main_, done_, 0));
        pending_ = false;
        return KB_OK;
    }

  private:
    void release() {
        if (ready_) cudaEventDestroy(ready_);
        if (done_) cudaEventDestroy(done_);
        if (side_) cudaStreamDestroy(side_);
        ready_ = done_ = nullptr;
        side_ = nullptr;
    }
    cudaStream_t main_, side_ = nullptr;
    cudaEvent_t ready_ = nullptr, done_ = nullptr;
    bool pending_ = false;
};

struct Common {
    kb_graph *g;
    kb_phi phi;
    kb_params p;
    int s_int;
    cudaStream_t s;
    int spmm = 0;
    Ctrl *hctrl = nullptr;   // host copy of the control block when the caller wants info
    bool frontier = true;    // restrict the per-step kernels to the reached rows
    int tc = 0;              // tensor-core row-block kernels allowed (asked once per solve)
    int ordered = 0;         // FP32 cbl with full reorthogonalisation: sums in a fixed order
    const QuadRule *quad = nullptr;   // spline kernel with non-integer s (Lanczos methods)
};

// The quadrature rule of the fractional spline power for the Lanczos methods (q->n = 0 when
// it is not needed: diffusion kernel, Chebyshev methods, integer s).  Relative accuracy
// 1e-14 on [0, Lambda], far below the FP64 rounding of the projected solves it feeds.
int quad_setup(const kb_graph *g, kb_method method, kb_phi phi, const kb_params &p, QuadRule &q) {
    q.n = 0;
    q.s_int = 0;
    if (phi != KB_PHI_SPLINE || method == KB_CHEB || method == KB_CHEB2) return KB_OK;
    return spline_quadrature(p.eps, p.s, g->lambda_proj, 1e-14, q);
}

// Quadrature nodes processed at once by the cbl projected step (one CTA and one scratch
// region of bt_quad_node_doubles(M, m) doubles each), at most 1 GiB of scratch.
int quad_batch(const QuadRule *q, int M, int m) {
    if (!q || q->n == 0) return 0;
    const size_t per = bt_quad_node_doubles(M, m) * sizeof(double);
    const size_t cap = std::max<size_t>(1, (size_t(1) << 30) / per);
    return int(std::min<size_t>({size_t(q->n), size_t(2 * num_sms()), cap}));
}
#define KB_TRY(x)                \
    do {                         \
        int _rc = (x);           \
        if (_rc) return _rc;     \
    } while (0)

// Largest |entry| of phi(H) F_1 when the spectrum of H lies in [0, Lambda] (F_1 = I on the
// first block): max phi on [0, Lambda]; infinity where no useful bound exists.
double projected_bound(const Common &c) {
    const double lam = c.g->lambda;
    if (c.phi == KB_PHI_EXP) {
        // slack 25 %: rounding of a slightly perturbed spectrum stays inside, a basis that
        // lost orthogonality (values growing like cosh(j acosh|x|), |x| > 1) does not
        if (c.p.t >= 0) return 1.25;
        const double e = -c.p.t * lam;
        return e < 700 ? std::exp(e) * 1.25 : std::numeric_limits<double>::infinity();
    }
    const double b = std::pow(c.p.eps, -c.p.s);
    return std::isfinite(b) ? b * 1.25 : std::numeric_limits<double>::infinity();
}

// ---------------------------------------------------------------- cbl
// W x W matrices kept per step (CblBufs)
static int step_mats(const Common &c) { return c.p.reorth == 2 ? 6 : 4; }

template <typename T>
struct CblBufs {
    using C = typename Cmp<T>::type;   // small matrices and Gram partials
    T *basis, *wbuf;
    C *parts, *Ut, *Cstk;
    // per-step small matrices (one W x W slot per step), kept for the two-pass replay:
    // H_kk as subtracted, H_{k,k+1} as subtracted at the next step, the two applied inverse
    // Cholesky factors, and the two local reorthogonalisation coefficient blocks
    C *Cbs, *Bs, *Rs1, *Rs2, *Cloc;
    double *Gsum, *Hd, *Hs, *R1, *V0, *V1, *V2, *U;
    double *Uc;          // stopping rule: two U_k of the checks (alternating)
    double *qscr;        // projected step with non-integer s: per-node block solves
    double *Hdf;         // projected e^{-tH} F_1 in double-float: H as floats, and transposed;
                         // spline kernel: two of the factor arrays
    double *bt_ls;
    int32_t *chk_prev;   // steps of the previous check (0: none yet)
    double *reo_d0;      // full reorthogonalisation: squared column norms before the first pass
    int32_t *reo_skip;   // ... and the flag that skips the second pass
    Ctrl *ctrl, *ctrl2, *ctrl_chk;
    FrontierBufs fr;
    unsigned *hcnt;   // CTA counter of the reduction that forms H_kk
    int32_t *csync;   // grid barrier of the projected series
};

template <typename T>
void plan_cbl(Arena &ar, CblBufs<T> &b, const Common &c, int64_t n, int M, int W, int m, int rb_grid, int qbatch) {
    b.basis = ar.take_blocks<T>(size_t(c.p.two_pass ? 3 : m) * n * W, n, c.frontier);
    b.wbuf = ar.take<T>(size_t(n) * W);
    using C = typename Cmp<T>::type;
    b.parts = ar.take<C>(size_t(rb_grid) * W * W);
    b.Cbs = ar.take<C>(size_t(m) * W * W * step_mats(c));   // Cbs | Bs | Rs1 | Rs2 | Cloc (2 per step)
    b.Bs = b.Cbs + size_t(m) * W * W;
    b.Rs1 = b.Bs + size_t(m) * W * W;
    b.Rs2 = b.Rs1 + size_t(m) * W * W;
    b.Cloc = b.Rs2 + size_t(m) * W * W;
    b.Ut = ar.take<C>(size_t(m) * W * W);
    b.Gsum = ar.take<double>(size_t(W) * W);
    b.Hd = ar.take<double>(size_t(m) * M * M);
    b.Hs = ar.take<double>(size_t(m) * M * M);
    b.R1 = ar.take<double>(size_t(M) * M);
    b.Cstk = c.p.reorth == 1 ? ar.take<C>(size_t(m) * W * W) : nullptr;
    b.V0 = ar.take<double>(size_t(m) * M * M);
    b.V1 = ar.take<double>(size_t(m) * M * M);
    b.V2 = ar.take<double>(size_t(m) * M * M);
    b.U = ar.take<double>(size_t(m) * M * M);
    b.Uc = c.p.tol > 0.0 ? ar.take<double>(size_t(2) * m * M * M) : nullptr;
    b.qscr = qbatch > 0 ? ar.take<double>(size_t(qbatch) * bt_quad_node_doubles(M, m)) : nullptr;
    const bool spline = c.phi == KB_PHI_SPLINE;
    b.Hdf = spline ? ar.take<double>(size_t(2) * m * M * M)
                   : sizeof(C) == 4 ? ar.take<double>(size_t(2) * m * M * (M + 1)) : nullptr;
    b.bt_ls = spline ? ar.take<double>(size_t(2) * M * M) : nullptr;
    b.chk_prev = ar.take<int32_t>(1);
    b.reo_d0 = ar.take<double>(size_t(W));
    b.reo_skip = ar.take<int32_t>(1);
    b.ctrl = ar.take<Ctrl>(1);
    b.ctrl2 = ar.take<Ctrl>(1);
    b.ctrl_chk = ar.take<Ctrl>(1);
    if (c.frontier) ar.frontier(b.fr, n, m);
    b.hcnt = ar.take<unsigned>(1);
    b.csync = ar.take<int32_t>(2);
}

template <typename T>
int cbl_grid(const Common &c, int W, int M, int64_t n) {
    return rowblock_max_grid<T>(W, M, n, c.ordered != 0, c.tc != 0);
}

template <typename T>
int run_cbl(Common &c, const int32_t *nodes, int M, int m, float *Y, int64_t ldy) {
    using C = typename Cmp<T>::type;
    const int64_t n = c.g->dev.n;
    const int W = width_for(M);
    const bool f64 = sizeof(C) == 8;
    const int rb_grid = cbl_grid<T>(c, W, M, n);
    const bool two = c.p.two_pass != 0;
    const int qbatch = quad_batch(c.quad, M, m);
    Arena dry;
    CblBufs<T> b{};
    plan_cbl<T>(dry, b, c, n, M, W, m, rb_grid, qbatch);
    Arena ar;
    KB_CUDA_TRY(cudaMallocAsync(reinterpret_cast<void **>(&ar.base), dry.off, c.s));
    plan_cbl<T>(ar, b, c, n, M, W, m, rb_grid, qbatch);
    auto body = [&]() -> int {
        const double lam = c.g->lambda;        // thresholds (scale of L)
        const double lam_p = c.g->lambda_proj; // interval of the projected series
        const double tau_inv = f64 ? 1e-12 : 1e-6;
        const double tau_piv = f64 ? 1e-12 : 1e-5;
        const double inv_thresh2 = (tau_inv * lam) * (tau_inv * lam) * M;
        const double piv2 = tau_piv * tau_piv;
        KB_TRY(launch_ctrl_init(b.ctrl, m, c.s));
        // with the frontier restriction a block is written on the tiles it reaches and zero on
        // those just beyond; otherwise each block is written in full
        const int nbuf = two ? 3 : m;
        const int64_t bs = n * W;
        const bool ord = c.ordered != 0;
        auto start_blocks = [&]() -> int {
            if (!c.frontier) {
                KB_CUDA_TRY(cudaMemsetAsync(b.basis, 0, sizeof(T) * size_t(bs), c.s));
            } else if (c.tc || ord) {
                // (kernels that walk whole tiles of 64 rows or more, or all tiles for every block,
                // read rows beyond a block's reach)
                KB_CUDA_TRY(cudaMemsetAsync(b.basis, 0, sizeof(T) * size_t(bs) * nbuf, c.s));
                KB_CUDA_TRY(cudaMemsetAsync(b.wbuf, 0, sizeof(T) * size_t(bs), c.s));
            } else {
                KB_TRY(launch_zero_tiles(b.basis, bs * sizeof(T), nbuf, W * int(sizeof(T)), n, !two, b.fr, c.s));
            }
            return launch_scatter<T>(b.basis, W, nodes, M, 0, T(1), c.s);
        };
        if (c.frontier) KB_TRY(launch_frontier(c.g->dev, b.fr, nodes, M, c.s));
        KB_TRY(start_blocks());
        // slots of steps after a stop are never written: keep them zero
        KB_CUDA_TRY(cudaMemsetAsync(b.Cbs, 0, sizeof(C) * size_t(m) * W * W * step_mats(c), c.s));
        // the frontier arguments of a row-block launch over the tiles within k hops
        const int32_t *tg = c.frontier ? b.fr.tgen : nullptr;
        auto within = [&](RowArgs<T> &ra, int k) {
            ra.max_grid = rb_grid;
            ra.tc = c.tc;
            ra.ordered = c.ordered;
            ra.tgen = tg;
            ra.limit = k;
            ra.alist = tg ? b.fr.list(k) : nullptr;
            ra.acount = tg ? b.fr.count(k) : nullptr;
        };
        // a launch with a Gram in an ordered solve: all tiles of step k
        auto in_order = [&](RowArgs<T> &ra, int k) {
            if (!ord || !tg) return;
            ra.limit = k;
            ra.alist = b.fr.list(k);
            ra.acount = b.fr.count(k);
        };
        const size_t WW = size_t(W) * W;
        auto blk = [&](int j) { return b.basis + int64_t(two ? j % 3 : j) * bs; };
        KB_CUDA_TRY(cudaMemsetAsync(b.hcnt, 0, sizeof(unsigned), c.s));
        int nchk = 0;
        int last_check = 0;
        CheckWatch watch(c.p.tol > 0.0 && c.hctrl);
        bool ended = false;   // the host knows that the process has stopped (watch.seen())
        int kfac = 0;   // blocks of the spline kernel's factorisation that are enqueued
        int kfwd = 0;   // blocks whose forward solutions earlier checks formed (s_int == 1)
        // The spline kernel's block factorisation needs H_kk and H_{k,k-1} only: block k - 1 is
        // factored beside the rest of step k and step k + 1 (at M = 64 a chain of 0.13 ms on few
        // SMs; four requests on a geometric graph of 55392 rows 69.1 -> 62.5 ms, full
        // reorthogonalisation with M = 128 on 5e5 rows 173.2 -> 167.6 ms).  The blocks before the process's steps are all factored: a process stops with
        // steps >= k at step k.
        SideStream side(c.phi == KB_PHI_SPLINE && c.s_int > 0 && m > 1, c.s);
        const SplineBufs sbufs{b.V0, b.V1, b.V2, b.Hdf, b.Hdf + size_t(m) * M * M, b.bt_ls};
        if (c.p.tol > 0.0) KB_CUDA_TRY(cudaMemsetAsync(b.chk_prev, 0, sizeof(int32_t), c.s));
        for (int k = 1; k <= m; ++k) {
            // two steps behind a check its outcome is asked for: the GPU has those steps to do
            // meanwhile
            if (last_check > 0 && k == last_check + 3 && watch.stopped()) {
                ended = true;
                c.spmm += m - k + 1;   // (reported are the products of m steps, as without info)
                break;
            }
            T *Qk = blk(k - 1);
            T *Qp = k >= 2 ? blk(k - 2) : nullptr;
            C *Cb = b.Cbs + (k - 1) * WW;                     // H_kk
            const C *Bp = k >= 2 ? b.Bs + (k - 2) * WW : nullptr;   // H_{k-1,k} (step k-1)
            C *Bk = b.Bs + (k - 1) * WW;
            C *S1 = b.Rs1 + (k - 1) * WW, *S2 = b.Rs2 + (k - 1) * WW;
            C *Cl = b.Cloc + 2 * (k - 1) * WW;
            // Q_k is supported on rows within k-1 hops of W; L Q_k within k hops
            // block SpMM: W = L Q_k
            LinEpi<T> e;
            e.s1 = 1.0;
            e.out = b.wbuf;
            e.one_group = c.ordered;
            e.ctrl = b.ctrl;
            e.tgen = tg;
            e.gen = tg ? b.fr.gen : nullptr;
            e.limit = k;
            e.alist = tg ? b.fr.list(k) : nullptr;
            e.acount = tg ? b.fr.count(k) : nullptr;
            KB_TRY(launch_spmm<T>(c.g->dev, W, Qk, e, c.s, nullptr, M, 0));
            ++c.spmm;
            // diagonal block: H_kk = Q_k^T L Q_k
            int grid = 0;
            RowArgs<T> pa;
            pa.n = n; pa.x = b.wbuf; pa.qa = Qk; pa.partials = b.parts; pa.ctrl = b.ctrl;
            within(pa, k - 1);   // (Q_k is zero elsewhere)
            in_order(pa, k);
            KB_TRY(launch_rowblock<T>(RB_PROJ, W, pa, c.s, &grid, M));
            KB_TRY(launch_reduce_hkk<C>(b.parts, grid, M, W, b.Gsum, b.Hd + size_t(k - 1) * M * M, Cb, b.hcnt, b.ctrl,
                                        c.s));
            if (side) {
                KB_TRY(side.fork());
                KB_TRY(launch_bt_factor(b.Hd, b.Hs, M, c.p.eps, sbufs, b.ctrl, side.stream(), k - 1, k));
                kfac = k;
            }
            if (k == m) break;   // Q_{m+1} is never used
            // three-term update: X = L Q_k - Q_{k-1} H_{k-1,k} - Q_k H_kk, then Gram X^T X
            T *X = blk(k);
            RowArgs<T> ua;
            ua.n = n; ua.x = b.wbuf; ua.qa = Qp; ua.ca = Bp; ua.qb = Qk; ua.cb = Cb;
            ua.out = X; ua.partials = b.parts; ua.ctrl = b.ctrl;
            within(ua, k);
            in_order(ua, k);
            ua.lim_a = k - 2; ua.lim_b = k - 1; ua.tri_a = 1;   // (H_{k-1,k} is lower triangular)
            KB_TRY(launch_rowblock<T>(RB_UPD, W, ua, c.s, &grid, M));
            KB_TRY(launch_reduce<C>(b.parts, grid, W * W, b.Gsum, c.s, b.ctrl));
            if (c.p.reorth == 2) {
                // local reorthogonalisation (not in the paper): a second
                // classical Gram-Schmidt pass against Q_k and Q_{k-1},
                // X -= Q_k (Q_k^T X) + Q_{k-1} (Q_{k-1}^T X); it keeps the three-term
                // orthogonality that FP32 rounding erodes when Ritz values converge
                const T *loc[2] = {Qk, Qp};
                for (int j = 0; j < 2; ++j) {
                    if (!loc[j]) continue;
                    RowArgs<T> ra;
                    ra.n = n; ra.x = X; ra.qa = loc[j]; ra.partials = b.parts; ra.ctrl = b.ctrl;
                    within(ra, k - 1 - j);
                    KB_TRY(launch_rowblock<T>(RB_PROJ, W, ra, c.s, &grid, M));
                    KB_TRY(launch_reduce<C>(b.parts, grid, W * W, b.Gsum, c.s, b.ctrl, Cl + j * WW));
                }
                RowArgs<T> la;
                la.n = n; la.x = X; la.qa = Qp; la.ca = Cl + WW; la.qb = Qk;
                la.cb = Cl; la.out = X; la.partials = b.parts; la.ctrl = b.ctrl;
                within(la, k);
                la.lim_a = k - 2; la.lim_b = k - 1;
                KB_TRY(launch_rowblock<T>(RB_UPD, W, la, c.s, &grid, M));
                KB_TRY(launch_reduce<C>(b.parts, grid, W * W, b.Gsum, c.s, b.ctrl));
            }
            if (c.p.reorth == 1) {
                // full reorthogonalisation (not in the paper): classical Gram-Schmidt against all
                // stored blocks, X -= Q_{1:k} (Q_{1:k}^T X); the second pass runs only when the
                // first removed more than half of some column's squared norm (Kahan's "twice
                // is enough"; the device decides, the host launches both passes); the last
                // subtraction that runs also forms the Gram X^T X for the QR
                KB_TRY(launch_reorth_save(b.Gsum, M, W, b.reo_d0, c.s));
                for (int pass = 0; pass < 2; ++pass) {
                    const int32_t *skip = pass == 1 ? b.reo_skip : nullptr;
                    for (int j = 0; j < k; ++j) {
                        RowArgs<T> ra;
                        ra.n = n; ra.x = X; ra.qa = b.basis + j * bs; ra.partials = b.parts;
                        ra.ctrl = b.ctrl; ra.skip = skip;
                        within(ra, j);
                        in_order(ra, k);
                        KB_TRY(launch_rowblock<T>(RB_PROJ, W, ra, c.s, &grid, M));
                        KB_TRY(launch_reduce<C>(b.parts, grid, W * W, b.Gsum, c.s, b.ctrl,
                                                b.Cstk + size_t(j) * W * W, skip));
                    }
                    RowArgs<T> sa;
                    sa.n = n; sa.x = X; sa.basis = b.basis; sa.block_stride = bs; sa.nblk = k;
                    sa.ca = b.Cstk; sa.out = X; sa.partials = b.parts; sa.ctrl = b.ctrl; sa.skip = skip;
                    within(sa, k);
                    in_order(sa, k);
                    KB_TRY(launch_rowblock<T>(RB_ASMSUB, W, sa, c.s, &grid, M));
                    KB_TRY(launch_reduce<C>(b.parts, grid, W * W, b.Gsum, c.s, b.ctrl, nullptr, skip));
                    if (pass == 0) KB_TRY(launch_reorth_decide(b.Gsum, b.reo_d0, M, W, b.reo_skip, c.s));
                }
            }
            // reduced QR: X = Q_{k+1} H_{k+1,k} by CholeskyQR2
            auto chol = [&](int pass, C *Rinv, double *Hs, C *B) -> int {
                if constexpr (std::is_same<T, float>::value) {
                    if (ord)
                        return launch_chol_ordered(b.Gsum, M, W, pass, k, inv_thresh2, piv2, b.R1, Rinv, Hs, B,
                                                   b.ctrl, c.s);
                }
                return launch_chol<C>(b.Gsum, M, W, pass, k, inv_thresh2, piv2, b.R1, Rinv, Hs, B, b.ctrl, c.s);
            };
            KB_TRY(chol(1, S1, nullptr, nullptr));
            RowArgs<T> ma;
            ma.n = n; ma.x = X; ma.ca = S1; ma.out = X; ma.partials = b.parts; ma.ctrl = b.ctrl;
            within(ma, k);
            in_order(ma, k);
            KB_TRY(launch_rowblock<T>(RB_MULGRAM, W, ma, c.s, &grid, M));
            KB_TRY(launch_reduce<C>(b.parts, grid, W * W, b.Gsum, c.s, b.ctrl));
            KB_TRY(chol(2, S2, b.Hs + size_t(k - 1) * M * M, Bk));
            RowArgs<T> qa;
            qa.n = n; qa.x = X; qa.ca = S2; qa.out = X; qa.ctrl = b.ctrl;
            within(qa, k);
            KB_TRY(launch_rowblock<T>(RB_MUL, W, qa, c.s, &grid, M));
            // stopping rule: U_k at the check steps, compared with the previous check's
            if (c.p.tol > 0.0 && k < m && (k == 8 || k == 12 || k == 16 || k == 24 || k == 32 ||
                                           k == 48 || k == 64 || k == 96)) {
                double *Ucur = b.Uc + size_t(nchk % 2) * m * M * M;
                const double *Uprev = b.Uc + size_t((nchk + 1) % 2) * m * M * M;
                KB_TRY(launch_ctrl_snapshot(b.ctrl_chk, b.ctrl, k, c.s));
                if (c.phi == KB_PHI_EXP) {
                    const std::vector<double> d = exp_series_coeffs(c.p.t, lam_p, 1e-17);
                    KB_TRY(launch_cheb_bt(b.Hd, b.Hs, M, m, lam_p, d, b.V0, b.V1, b.V2, Ucur, b.ctrl_chk, c.s, f64 ? nullptr : b.Hdf, b.csync, k, b.ctrl));
                } else {
                    KB_TRY(side.join());
                    KB_TRY(launch_bt_spline(b.Hd, b.Hs, M, m, c.p.eps, c.s_int, sbufs, Ucur, b.ctrl, b.ctrl_chk,
                                            c.s, c.quad, b.qscr, qbatch, kfac, c.s_int == 1 ? kfwd : 0, k));
                    kfac = kfwd = k;
                }
                KB_TRY(launch_conv_check(Ucur, Uprev, M, b.ctrl_chk, b.chk_prev, c.p.tol, b.ctrl, c.s, nchk % 2));
                ++nchk;
                last_check = k;
                watch.record(b.ctrl, c.s);
            }
        }
        // projected problem: U = phi(H_m) F_1 in FP64 (skipped when the stopping rule's last
        // check formed it: the check's U is copied instead)
        const Ctrl *cfin = b.ctrl;
        if (c.p.tol > 0.0) {
            KB_TRY(launch_ctrl_final(b.ctrl_chk, b.ctrl, c.s));
            cfin = b.ctrl_chk;
        }
        // (nothing is left to form when the host has seen a check stop the process; one that stopped by
        // itself has seen().steps blocks)
        const bool formed = ended && watch.seen().from_check >= 0;
        const int kend = ended && !formed ? std::max(1, std::min(m, int(watch.seen().steps))) : m;
        if (formed) {
        } else if (c.phi == KB_PHI_EXP) {
            const std::vector<double> d = exp_series_coeffs(c.p.t, lam_p, 1e-17);
            KB_TRY(launch_cheb_bt(b.Hd, b.Hs, M, m, lam_p, d, b.V0, b.V1, b.V2, b.U, cfin, c.s, f64 ? nullptr : b.Hdf, b.csync, kend, b.ctrl));
        } else {
            // (a process that stopped by itself skipped the later checks: their Y are formed now)
            KB_TRY(side.join());
            KB_TRY(launch_bt_spline(b.Hd, b.Hs, M, m, c.p.eps, c.s_int, sbufs, b.U, b.ctrl, cfin, c.s, c.quad,
                                    b.qscr, qbatch, std::min(kfac, kend), 0, kend));
        }
        if (c.p.tol > 0.0) KB_TRY(launch_copy_check_u(b.Uc, int64_t(m) * M * M, b.U, b.ctrl, c.s));
        KB_TRY(launch_check_projected(b.U, int64_t(m) * M * M, projected_bound(c), b.ctrl, c.s));
        KB_TRY(launch_u_convert<C>(b.U, M, W, m, b.Ut, b.ctrl, c.s));
        // assembly: Y = [Q_1 .. Q_m] U
        if (!two) {
            RowArgs<T> aa;
            aa.n = n; aa.basis = b.basis; aa.block_stride = bs; aa.nblk = m; aa.ca = b.Ut;
            aa.y = Y; aa.ldy = ldy; aa.mo = M; aa.ctrl = b.ctrl;
            within(aa, m);
            aa.alist = tg ? b.fr.alist : nullptr;   // all tiles, by rising distance
            int grid = 0;
            KB_TRY(launch_rowblock<T>(RB_ASM, W, aa, c.s, &grid, M));
        } else {
            // second pass: the same products and updates with the recorded matrices
            // (bit-identical blocks); Y += Q_k U_k as each block is recomputed
            KB_TRY(launch_ctrl_init(b.ctrl2, m, c.s));
            KB_TRY(start_blocks());
            for (int k = 1; k <= m; ++k) {
                T *Qk = blk(k - 1);
                T *Qp = k >= 2 ? blk(k - 2) : nullptr;
                RowArgs<T> aa;
                aa.n = n; aa.basis = Qk; aa.block_stride = bs; aa.nblk = 1;
                aa.ca = b.Ut + (k - 1) * WW; aa.y = Y; aa.ldy = ldy; aa.mo = M;
                within(aa, k - 1);
                if (k == 1) aa.alist = tg ? b.fr.alist : nullptr;   // (the first launch writes all of Y)
                aa.kbase = k - 1; aa.accumulate = k > 1 ? 1 : 0;
                int grid = 0;
                KB_TRY(launch_rowblock<T>(RB_ASM, W, aa, c.s, &grid, M));
                if (k == m) break;
                LinEpi<T> e;
                e.s1 = 1.0;
                e.out = b.wbuf;
                e.ctrl = b.ctrl2;
                e.tgen = tg;
                e.gen = tg ? b.fr.gen : nullptr;
                e.limit = k;
                e.alist = tg ? b.fr.list(k) : nullptr;
                e.acount = tg ? b.fr.count(k) : nullptr;
                KB_TRY(launch_spmm<T>(c.g->dev, W, Qk, e, c.s, nullptr, M, 0));
                ++c.spmm;
                T *X = blk(k);
                RowArgs<T> ua;
                ua.n = n; ua.x = b.wbuf; ua.qa = Qp; ua.ca = k >= 2 ? b.Bs + (k - 2) * WW : nullptr;
                ua.qb = Qk; ua.cb = b.Cbs + (k - 1) * WW;
                ua.out = X; ua.partials = b.parts; ua.ctrl = b.ctrl2; within(ua, k);
                ua.lim_a = k - 2; ua.lim_b = k - 1; ua.tri_a = 1;
                KB_TRY(launch_rowblock<T>(RB_UPD, W, ua, c.s, &grid, M));
                if (c.p.reorth == 2) {
                    RowArgs<T> la = ua;
                    la.tri_a = 0;
                    la.x = X; la.ca = b.Cloc + (2 * (k - 1) + 1) * WW; la.cb = b.Cloc + 2 * (k - 1) * WW;
                    KB_TRY(launch_rowblock<T>(RB_UPD, W, la, c.s, &grid, M));
                }
                for (int pass = 0; pass < 2; ++pass) {
                    RowArgs<T> qa;
                    qa.n = n; qa.x = X; qa.ca = (pass == 0 ? b.Rs1 : b.Rs2) + (k - 1) * WW;
                    qa.out = X; qa.ctrl = b.ctrl2; within(qa, k);
                    KB_TRY(launch_rowblock<T>(RB_MUL, W, qa, c.s, &grid, M));
                }
            }
        }
        KB_TRY(launch_fill_nan(Y, n, ldy, M, b.ctrl, c.s));
        return 0;
    };
    int rc = body();
    if (!rc && c.hctrl) {
        cudaError_t e = cudaMemcpyAsync(c.hctrl, b.ctrl, sizeof(Ctrl), cudaMemcpyDeviceToHost, c.s);
        if (e != cudaSuccess) rc = cuda_fail(e, "ctrl readback");
    }
    cudaFreeAsync(ar.base, c.s);
    return rc;
}

// ---------------------------------------------------------------- gbl / sbl
template <typename T>
struct LzBufs {
    T *basis;
    double *parts, *sigma, *alpha, *beta, *work;
    double *qwork;                    // fractional spline factor: 2 m nodes per column
    int32_t *alive;
    double *c1, *c2, *aupd, *omega;   // c1, c2, aupd: one row of W per step
    Ctrl *ctrl, *ctrl2;
    FrontierBufs fr;
};

template <typename T>
void plan_lz(Arena &ar, LzBufs<T> &b, const Common &c, int64_t n, int W, int m, int pgrid, int nquad) {
    // two-pass: three rotating blocks; the coefficients of every step are kept for the replay
    b.basis = ar.take_blocks<T>(size_t(c.p.two_pass ? 3 : m + 1) * n * W, n, c.frontier);
    b.parts = ar.take<double>(size_t(pgrid) * W);
    b.sigma = ar.take<double>(size_t(m + 1) * W);
    b.alpha = ar.take<double>(size_t(m + 1) * W);
    b.beta = ar.take<double>(size_t(m + 1) * W);
    b.work = ar.take<double>(size_t(W) * 4 * m);
    b.qwork = nquad > 0 ? ar.take<double>(size_t(W) * 2 * m * nquad) : nullptr;
    b.alive = ar.take<int32_t>(W);
    b.c1 = ar.take<double>(size_t(m + 1) * W);
    b.c2 = ar.take<double>(size_t(m + 1) * W);
    b.aupd = ar.take<double>(size_t(m + 1) * W);
    b.omega = ar.take<double>(size_t(m) * W);
    b.ctrl = ar.take<Ctrl>(1);
    b.ctrl2 = ar.take<Ctrl>(1);
    if (c.frontier) ar.frontier(b.fr, n, m);
}

template <typename T>
int run_lanczos_scalar(Common &c, bool gbl, const int32_t *nodes, int M, int m, float *Y,
                       int64_t ldy) {
    const int64_t n = c.g->dev.n;
    const int W = width_for(M);
    const bool f64 = sizeof(T) == 8;
    const int pgrid = std::max(spmm_max_grid<T>(W), axpy_max_grid());
    auto tc = std::make_unique<TriCoef>();
    int nquad = 0;
    std::vector<double> series;
    if (c.phi == KB_PHI_EXP) {
        series = exp_series_coeffs(c.p.t, c.g->lambda_proj, 1e-17);
        // longer series are applied in chunks by launch_tridiag_phi
        tc->cc.n = int(std::min<size_t>(series.size(), ChebCoef::CAP));
        for (int j = 0; j < tc->cc.n; ++j) tc->cc.d[j] = series[j];
    } else {
        tc->q.n = 0;
        tc->q.s_int = c.s_int;
        if (c.quad) {
            tc->q = *c.quad;
            nquad = c.quad->n;
        }
    }
    const bool two = c.p.two_pass != 0;
    Arena dry;
    LzBufs<T> b{};
    plan_lz<T>(dry, b, c, n, W, m, pgrid, nquad);
    Arena ar;
    KB_CUDA_TRY(cudaMallocAsync(reinterpret_cast<void **>(&ar.base), dry.off, c.s));
    plan_lz<T>(ar, b, c, n, W, m, pgrid, nquad);
    auto body = [&]() -> int {
        const double thresh = (f64 ? 1e-12 : 1e-6) * c.g->lambda;
        KB_TRY(launch_ctrl_init(b.ctrl, m, c.s));
        const int nbuf = two ? 3 : m + 1;
        const int64_t bs = n * W;
        const int32_t *tg = c.frontier ? b.fr.tgen : nullptr;
        auto start_blocks = [&]() -> int {
            if (!c.frontier) KB_CUDA_TRY(cudaMemsetAsync(b.basis, 0, sizeof(T) * size_t(bs), c.s));
            else KB_TRY(launch_zero_tiles(b.basis, bs * sizeof(T), nbuf, W * int(sizeof(T)), n, !two, b.fr, c.s));
            return launch_scatter<T>(b.basis, W, nodes, M, 0, T(1), c.s);
        };
        if (c.frontier) KB_TRY(launch_frontier(c.g->dev, b.fr, nodes, M, c.s));
        KB_TRY(start_blocks());
        // coefficients of steps after an invariant stop are never written: keep them zero
        KB_CUDA_TRY(cudaMemsetAsync(b.c1, 0, sizeof(double) * size_t(m + 1) * W, c.s));
        KB_CUDA_TRY(cudaMemsetAsync(b.c2, 0, sizeof(double) * size_t(m + 1) * W, c.s));
        KB_CUDA_TRY(cudaMemsetAsync(b.aupd, 0, sizeof(double) * size_t(m + 1) * W, c.s));
        KB_CUDA_TRY(cudaMemsetAsync(b.beta, 0, sizeof(double) * size_t(m + 1) * W, c.s));
        KB_CUDA_TRY(cudaMemsetAsync(b.alpha, 0, sizeof(double) * size_t(m + 1) * W, c.s));
        KB_CUDA_TRY(cudaMemsetAsync(b.sigma, 0, sizeof(double) * size_t(m + 1) * W, c.s));
        KB_TRY(launch_lanczos_init(W, M, gbl ? 1 : 0, f64 ? 0 : 1, b.sigma, b.alive, b.c1, b.c2, c.s));
        auto blk = [&](int j) { return b.basis + int64_t(two ? j % 3 : j) * bs; };
        for (int k = 1; k <= m; ++k) {
            T *Pk = blk(k - 1);
            T *Pp = k >= 2 ? blk(k - 2) : nullptr;
            T *X = blk(k);
            // X = L Q_k - h_{k,k-1} Q_{k-1}, with Q_k = sigma_k P_k; dots <P_k, X> per column
            LinEpi<T> e;
            e.tgen = tg;
            e.gen = tg ? b.fr.gen : nullptr;
            e.limit = k;
            e.alist = tg ? b.fr.list(k) : nullptr;
            e.acount = tg ? b.fr.count(k) : nullptr;
            e.a1 = b.c1 + int64_t(k - 1) * W;
            e.a2 = b.c2 + int64_t(k - 1) * W;
            e.s0 = 0.0;
            e.y = Pp;
            e.out = X;
            e.dot_partials = b.parts;
            e.ctrl = b.ctrl;
            int grid = 0;
            KB_TRY(launch_spmm<T>(c.g->dev, W, Pk, e, c.s, &grid, M, Pp ? 1 : 0));
            ++c.spmm;
            KB_TRY(launch_lanczos_alpha(b.parts, grid, W, M, gbl ? 1 : 0, k - 1, f64 ? 0 : 1, b.sigma, b.alpha,
                                        b.aupd + int64_t(k - 1) * W, b.ctrl, c.s));
            if (k == m) break;
            int grid2 = 0;
            KB_TRY(launch_axpy_colnorm<T>(W, X, Pk, b.aupd + int64_t(k - 1) * W, n, b.parts, &grid2,
                                          b.ctrl, M, c.s, tg ? b.fr.list(k) : nullptr, tg ? b.fr.count(k) : nullptr));
            KB_TRY(launch_lanczos_beta(b.parts, grid2, W, M, gbl ? 1 : 0, k - 1, f64 ? 0 : 1, thresh, b.beta,
                                       b.sigma, b.alive, b.c1 + int64_t(k) * W, b.c2 + int64_t(k) * W,
                                       b.ctrl, c.s));
        }
        KB_TRY(launch_tridiag_phi(W, M, m, gbl ? 1 : 0, b.alpha, b.beta, b.sigma, int(c.phi),
                                  c.p.eps, c.s_int, c.g->lambda_proj, *tc, b.omega, b.work, b.qwork, b.ctrl,
                                  projected_bound(c), c.s, c.phi == KB_PHI_EXP ? &series : nullptr));
        if (!two) {
            KB_TRY(launch_assemble_diag<T>(W, b.basis, bs, m, b.omega, n, Y, ldy, M, M, tg, b.ctrl, c.s));
        } else {
            // second pass: the same products and updates with the recorded coefficients
            // (bit-identical blocks), each block added to Y as soon as it exists
            KB_TRY(launch_ctrl_init(b.ctrl2, m, c.s));
            KB_TRY(start_blocks());
            KB_TRY(launch_assemble_diag<T>(W, blk(0), bs, 1, b.omega, n, Y, ldy, M, M, tg, b.ctrl, c.s, 0, 0));
            for (int k = 1; k < m; ++k) {
                T *Pk = blk(k - 1);
                T *Pp = k >= 2 ? blk(k - 2) : nullptr;
                T *X = blk(k);
                LinEpi<T> e;
                e.tgen = tg;
                e.gen = tg ? b.fr.gen : nullptr;
                e.limit = k;
                e.alist = tg ? b.fr.list(k) : nullptr;
                e.acount = tg ? b.fr.count(k) : nullptr;
                e.a1 = b.c1 + int64_t(k - 1) * W;
                e.a2 = b.c2 + int64_t(k - 1) * W;
                e.s0 = 0.0;
                e.y = Pp;
                e.out = X;
                e.dot_partials = b.parts;
                e.ctrl = b.ctrl2;
                int grid = 0;
                KB_TRY(launch_spmm<T>(c.g->dev, W, Pk, e, c.s, &grid, M, Pp ? 1 : 0));
                ++c.spmm;
                int grid2 = 0;
                KB_TRY(launch_axpy_colnorm<T>(W, X, Pk, b.aupd + int64_t(k - 1) * W, n, b.parts, &grid2,
                                              b.ctrl2, M, c.s, tg ? b.fr.list(k) : nullptr, tg ? b.fr.count(k) : nullptr));
                KB_TRY(launch_assemble_diag<T>(W, X, bs, 1, b.omega + int64_t(k) * W, n, Y, ldy, M, M,
                                               tg, b.ctrl, c.s, k, 1));
            }
        }
        KB_TRY(launch_fill_nan(Y, n, ldy, M, b.ctrl, c.s));
        return 0;
    };
    int rc = body();
    if (!rc && c.hctrl) {
        cudaError_t e = cudaMemcpyAsync(c.hctrl, b.ctrl, sizeof(Ctrl), cudaMemcpyDeviceToHost, c.s);
        if (e != cudaSuccess) rc = cuda_fail(e, "ctrl readback");
    }
    cudaFreeAsync(ar.base, c.s);
    return rc;
}

// ---------------------------------------------------------------- cheb / cheb2
template <typename T>
int cheb_pass(Common &c, const std::vector<double> &coef, double lam, int W, int64_t n,
              const int32_t *marker, const int32_t *nodes, int Mc, const T *Zsrc, T *bufs[3],
              T *out, float *yout, int64_t ldo, int mo, int64_t M_alg, const FrontierBufs *fr, int hop0) {
    // weights of sum_k'' c_k T_k (Lobatto interpolation: c_0 and c_m halved)
    const int h = int(coef.size()) - 1;
    std::vector<double> w(coef);
    w[0] *= 0.5;
    w[h] *= 0.5;
    // b_h = w_h S
    int cur_i = 0, prev_i = -1;
    if (Zsrc) {
        KB_TRY(launch_scale_copy<T>(bufs[0], Zsrc, n, W, w[h], fr ? fr->list(hop0) : nullptr,
                                    fr ? fr->count(hop0) : nullptr, c.s));
    } else {
        if (!fr) KB_CUDA_TRY(cudaMemsetAsync(bufs[0], 0, sizeof(T) * size_t(n) * W, c.s));
        KB_TRY(launch_scatter<T>(bufs[0], W, nodes, Mc, 0, T(w[h]), c.s));
    }
    // b_k = w_k S + 2 A b_{k+1} - b_{k+2} (k = h-1..1);  result = w_0 S + A b_1 - b_2,
    // A = I - (2/lam) L
    for (int k = h - 1; k >= 0; --k) {
        const bool last = k == 0;
        int dst_i = 0;
        while (dst_i == cur_i || dst_i == prev_i) ++dst_i;
        // b_k is supported on rows within hop0 + (h - k) hops of W
        const int hop = hop0 + (h - k);
        LinEpi<T> e;
        e.tgen = fr ? fr->tgen : nullptr;
        e.gen = fr ? fr->gen : nullptr;
        e.limit = hop;
        e.alist = fr ? (last && yout ? fr->alist : fr->list(hop)) : nullptr;
        e.acount = fr ? fr->count(hop) : nullptr;
        e.zero_inactive = last && yout ? 1 : 0;
        e.s1 = (last ? -2.0 : -4.0) / lam;
        e.s0 = last ? 1.0 : 2.0;
        e.s2 = -1.0;
        e.y = prev_i >= 0 ? bufs[prev_i] : nullptr;
        if (Zsrc) { e.z = Zsrc; e.s3 = w[k]; }
        else { e.marker = marker; e.wE = w[k]; }
        if (last) {
            if (yout) e.yout = yout;
            else e.out = out;
        } else {
            e.out = bufs[dst_i];
        }
        KB_TRY(launch_spmm<T>(c.g->dev, W, bufs[cur_i], e, c.s, nullptr, M_alg,
                              (prev_i >= 0 ? 1 : 0) + (Zsrc ? 1 : 0), (last && yout) ? ldo : 0,
                              (last && yout) ? mo : 0));
        ++c.spmm;
        prev_i = cur_i;
        cur_i = dst_i;
    }
    return 0;
}

template <typename T>
void plan_cheb(Arena &ar, const Common &c, int64_t n, int Mmax, bool squared, int hops, T **bufs, T **Z,
               int32_t **marker, FrontierBufs &fr) {
    // bufs and Z are consecutive blocks of n Wmax elements
    const int Wmax = width_for(Mmax);
    T *p = ar.take_blocks<T>(size_t(squared ? 4 : 3) * n * Wmax, n, c.frontier);
    for (int i = 0; i < 3; ++i) bufs[i] = p ? p + size_t(i) * n * Wmax : nullptr;
    *Z = squared && p ? p + size_t(3) * n * Wmax : nullptr;
    *marker = ar.take<int32_t>(size_t(n));
    if (c.frontier) ar.frontier(fr, n, hops);
}

template <typename T>
int run_cheb(Common &c, bool squared, const int32_t *nodes, int M, int m, float *Y, int64_t ldy) {
    const int64_t n = c.g->dev.n;
    const double lam = c.p.lambda_max > 0 ? c.p.lambda_max : c.g->lambda;
    const int h = squared ? m / 2 : m;
    const std::vector<double> coef = lobatto_coeffs(c.phi, c.p, h, lam, squared);
    const int Mmax = std::min(M, sizeof(T) == 8 ? 64 : 128);
    Arena dry;
    T *bufs[3], *Z;
    int32_t *marker;
    FrontierBufs fb;
    plan_cheb<T>(dry, c, n, Mmax, squared, squared ? 2 * h : h, bufs, &Z, &marker, fb);
    Arena ar;
    KB_CUDA_TRY(cudaMallocAsync(reinterpret_cast<void **>(&ar.base), dry.off, c.s));
    plan_cheb<T>(ar, c, n, Mmax, squared, squared ? 2 * h : h, bufs, &Z, &marker, fb);
    auto body = [&]() -> int {
        for (int col0 = 0; col0 < M; col0 += Mmax) {
            const int Mc = std::min(Mmax, M - col0);
            const int W = width_for(Mc);
            KB_CUDA_TRY(cudaMemsetAsync(marker, 0xFF, sizeof(int32_t) * size_t(n), c.s));
            KB_TRY(launch_marker(marker, nodes + col0, Mc, c.s));
            const FrontierBufs *fr = c.frontier ? &fb : nullptr;
            if (c.frontier) {
                // Clenshaw blocks rotate and are written on reached tiles only: zeros on all of those
                KB_TRY(launch_frontier(c.g->dev, fb, nodes + col0, Mc, c.s));
                KB_TRY(launch_zero_tiles(bufs[0], int64_t(sizeof(T)) * n * width_for(Mmax), squared ? 4 : 3,
                                         W * int(sizeof(T)), n, false, fb, c.s));
            }
            if (!squared) {
                KB_TRY(cheb_pass<T>(c, coef, lam, W, n, marker, nodes + col0, Mc, nullptr, bufs,
                                    nullptr, Y + col0, ldy, Mc, Mc, fr, 0));
            } else {
                KB_TRY(cheb_pass<T>(c, coef, lam, W, n, marker, nodes + col0, Mc, nullptr, bufs, Z,
                                    nullptr, 0, 0, Mc, fr, 0));
                KB_TRY(cheb_pass<T>(c, coef, lam, W, n, marker, nodes + col0, Mc, Z, bufs,
                                    nullptr, Y + col0, ldy, Mc, Mc, fr, h));
            }
        }
        return 0;
    };
    const int rc = body();
    cudaFreeAsync(ar.base, c.s);
    return rc;
}

// Scratch bytes of one solve (the same plans the runs allocate).
template <typename T>
size_t workspace_bytes_t(const Common &c, kb_method method, int M, int m) {
    Arena dry;
    const int64_t n = c.g->dev.n;
    const QuadRule *q = c.quad;
    const int W = width_for(M);
    switch (method) {
        case KB_CBL: {
            CblBufs<T> b{};
            plan_cbl<T>(dry, b, c, n, M, W, m, cbl_grid<T>(c, W, M, n), quad_batch(q, M, m));
            break;
        }
        case KB_GBL:
        case KB_SBL: {
            // sbl runs column groups one after the other; each group allocates its own scratch
            const int Mg = method == KB_SBL ? std::min(M, sizeof(T) == 8 ? 64 : 128) : M;
            const int Wg = width_for(Mg);
            LzBufs<T> b{};
            plan_lz<T>(dry, b, c, n, Wg, m, std::max(spmm_max_grid<T>(Wg), axpy_max_grid()), q ? q->n : 0);
            break;
        }
        case KB_CHEB:
        case KB_CHEB2: {
            T *bufs[3], *Z;
            int32_t *marker;
            FrontierBufs fb;
            plan_cheb<T>(dry, c, n, std::min(M, sizeof(T) == 8 ? 64 : 128), method == KB_CHEB2,
                         method == KB_CHEB2 ? 2 * (m / 2) : m, bufs, &Z, &marker, fb);
            break;
        }
    }
    return dry.off;
}

}  // namespace
}  // namespace kb

// ---------------------------------------------------------------- C ABI
using namespace kb;

namespace {

int validate(kb_graph *g, kb_method method, kb_phi phi, const kb_params *params,
             const int32_t *nodes, int32_t M, int32_t m, const void *Y, int *s_int) {
    if (!g) return fail(KB_ERR_ARG, "graph is NULL");
    if (!params) return fail(KB_ERR_ARG, "params is NULL");
    if (!nodes) return fail(KB_ERR_ARG, "nodes is NULL");
    if (!Y) return fail(KB_ERR_ARG, "Y is NULL");
    if (method < KB_CBL || method > KB_CHEB2) return fail(KB_ERR_ARG, "bad method");
    if (M < 1 || M > g->dev.n) return fail(KB_ERR_ARG, "M out of range");
    if (m < 1 || m > 100000) return fail(KB_ERR_ARG, "m out of range");
    if (method == KB_CHEB2 && m < 2) return fail(KB_ERR_ARG, "KB_CHEB2 needs m >= 2");
    if (params->basis != KB_F32 && params->basis != KB_F64 && params->basis != KB_BF16)
        return fail(KB_ERR_ARG, "bad basis dtype");
    if (params->reorth < 0 || params->reorth > 2) return fail(KB_ERR_ARG, "reorth must be 0, 1 or 2");
    if (params->two_pass != 0 && params->two_pass != 1) return fail(KB_ERR_ARG, "two_pass must be 0 or 1");
    if (params->two_pass && params->reorth == 1)
        return fail(KB_ERR_UNSUPPORTED, "full reorthogonalisation needs the stored basis (two_pass = 0)");
    if (params->reorth && method != KB_CBL)
        return fail(KB_ERR_UNSUPPORTED, "reorthogonalisation is implemented for KB_CBL only");
    if (!(params->tol >= 0.0) || !std::isfinite(params->tol)) return fail(KB_ERR_ARG, "tol must be finite and >= 0");
    if (params->tol > 0.0 && method != KB_CBL)
        return fail(KB_ERR_UNSUPPORTED, "the stopping rule (tol > 0) is implemented for KB_CBL only");
    if (params->tol > 0.0 && params->two_pass)
        return fail(KB_ERR_UNSUPPORTED, "the stopping rule (tol > 0) needs the stored basis (two_pass = 0)");
    const int wmax = params->basis == KB_F64 ? 64 : 128;
    if ((method == KB_CBL || method == KB_GBL) && M > wmax)
        return fail(KB_ERR_UNSUPPORTED, "block width too large for this method and dtype");
    if (int rc = validate_phi(phi, *params)) return rc;
    *s_int = 0;
    if (phi == KB_PHI_SPLINE && (method == KB_CBL || method == KB_GBL || method == KB_SBL)) {
        // floor(s) block solves with eps I + H_m, the fractional rest by quadrature
        if (params->s >= 65) return fail(KB_ERR_UNSUPPORTED, "Lanczos methods support s < 65");
        *s_int = int(std::floor(params->s));
    }
    if (method == KB_CBL && phi == KB_PHI_EXP && std::fabs(params->t) * g->lambda_proj > 2e5)
        return fail(KB_ERR_UNSUPPORTED, "t * Lambda too large for the Chebyshev projected solve");
    std::vector<int32_t> sorted(nodes, nodes + M);
    std::sort(sorted.begin(), sorted.end());
    if (sorted.front() < 0 || sorted.back() >= g->dev.n) return fail(KB_ERR_NODES, "node index out of range");
    for (int i = 1; i < M; ++i)
        if (sorted[i] == sorted[i - 1]) return fail(KB_ERR_NODES, "repeated node " + std::to_string(sorted[i]));
    return KB_OK;
}

// A solve's settings.  restricted: the per-step kernels may keep to the rows reached from W.
Common solve_of(kb_graph *g, kb_method method, kb_phi phi, const kb_params &params, int M, int m, int s_int,
                cudaStream_t s, const QuadRule &quad, bool restricted) {
    Common c{g, phi, params, s_int, s, 0, nullptr, true};
    if (quad.n > 0) c.quad = &quad;
    // exact restriction of the per-step kernels to rows reached from W (hop distances are kept
    // in 8 bits).  It costs a breadth-first search and a sort (about 5 us per hop), so blocks
    // below 16 MiB, which stay in L2, run on all rows: measured with 20 steps on random
    // geometric graphs, restricted / all rows (us): 16384 rows, M = 64, cheb 308 / 222, cbl
    // 5061 / 4975; 65536 rows, M = 64 (16 MiB), cheb 456 / 429, cbl 6290 / 7050; 262144 rows,
    // M = 16 (16 MiB), cheb 321 / 552, cbl 2558 / 3598.  FP64 products cost some 16 times as
    // much per row.
    const int64_t blk_bytes = g->dev.n * width_for(std::min(M, 128)) * (params.basis == KB_F64 ? 128 : 4);
    c.ordered = method == KB_CBL && params.reorth == 1 && params.basis == KB_F32 ? 1 : 0;
    c.frontier = restricted && !params.no_frontier && m <= FRONTIER_MAX_HOPS && (blk_bytes >= (int64_t(16) << 20) || c.ordered);
    c.tc = rowblock_tc_enabled() ? 1 : 0;
    return c;
}

int apply_once(kb_graph *g, kb_method method, kb_phi phi, const kb_params *params, const int32_t *nodes, int32_t M,
               int32_t m, float *Y, void *stream, kb_info *info, bool &restricted) {
    int s_int = 0;
    int rc = validate(g, method, phi, params, nodes, M, m, Y, &s_int);
    if (rc) return rc;
    DeviceGuard dg;
    KB_CUDA_TRY(dg.set(g->device));
    ensure_pool(g->device);
    auto quad = std::make_unique<QuadRule>();
    rc = quad_setup(g, method, phi, *params, *quad);
    if (rc) return rc;
    Common c = solve_of(g, method, phi, *params, M, m, s_int, static_cast<cudaStream_t>(stream), *quad, restricted);
    restricted = c.frontier;
    const bool f64 = params->basis == KB_F64;
    const bool bf16 = params->basis == KB_BF16;
    const int chunk = f64 ? 64 : 128;
    // one host control block per column group (sbl may run several groups)
    std::vector<Ctrl> hc;
    const int ngroups = method == KB_SBL ? (M + chunk - 1) / chunk : 1;
    if (info) hc.assign(ngroups, Ctrl{KB_OK, 0, m, -1, -1.0, -1, 0});
    switch (method) {
        case KB_CBL:
            c.hctrl = info ? &hc[0] : nullptr;
            rc = f64 ? run_cbl<double>(c, nodes, M, m, Y, M)
                 : bf16 ? run_cbl<__nv_bfloat16>(c, nodes, M, m, Y, M)
                        : run_cbl<float>(c, nodes, M, m, Y, M);
            break;
        case KB_GBL:
            c.hctrl = info ? &hc[0] : nullptr;
            rc = f64 ? run_lanczos_scalar<double>(c, true, nodes, M, m, Y, M)
                 : bf16 ? run_lanczos_scalar<__nv_bfloat16>(c, true, nodes, M, m, Y, M)
                        : run_lanczos_scalar<float>(c, true, nodes, M, m, Y, M);
            break;
        case KB_SBL:
            for (int col0 = 0, gi = 0; col0 < M && !rc; col0 += chunk, ++gi) {
                const int Mc = std::min(chunk, M - col0);
                c.hctrl = info ? &hc[gi] : nullptr;
                rc = f64 ? run_lanczos_scalar<double>(c, false, nodes + col0, Mc, m, Y + col0, M)
                     : bf16 ? run_lanczos_scalar<__nv_bfloat16>(c, false, nodes + col0, Mc, m, Y + col0, M)
                            : run_lanczos_scalar<float>(c, false, nodes + col0, Mc, m, Y + col0, M);
            }
            break;
        case KB_CHEB:
        case KB_CHEB2:
            rc = f64 ? run_cheb<double>(c, method == KB_CHEB2, nodes, M, m, Y, M)
                 : bf16 ? run_cheb<__nv_bfloat16>(c, method == KB_CHEB2, nodes, M, m, Y, M)
                        : run_cheb<float>(c, method == KB_CHEB2, nodes, M, m, Y, M);
            break;
    }
    if (rc) return rc;
    if (!info) return KB_OK;
    KB_CUDA_TRY(cudaStreamSynchronize(c.s));
    info->status = KB_OK;
    info->steps_done = m;
    info->breakdown_step = -1;
    info->est_change = -1.0;
    for (const Ctrl &h : hc) {
        if (h.status != KB_OK) info->status = h.status;
        if (h.breakdown_step >= 0) info->breakdown_step = h.breakdown_step;
        if (method != KB_SBL) info->steps_done = h.steps;
    }
    if (method == KB_CBL && params->tol > 0.0) info->est_change = hc[0].est_change;
    if (method == KB_CHEB2) info->steps_done = 2 * (m / 2);
    info->spmm_launches = c.spmm;
    info->lambda_used = (method == KB_CHEB || method == KB_CHEB2)
                            ? (params->lambda_max > 0 ? params->lambda_max : g->lambda)
                            : 0.0;
    if (info->status == KB_ERR_ORTHOGONALITY)
        return fail(info->status, "the projected matrix left the spectral interval [0, Lambda] "
                                  "(loss of orthogonality of the Lanczos basis); use reorth");
    if (info->status == KB_ERR_CUDA)
        return fail(info->status, "a kernel gave up waiting (grid barrier, or completion of a tensor-core product)");
    if (info->status != KB_OK) return fail(info->status, "Lanczos breakdown: rank-deficient block");
    return KB_OK;
}

// The restriction takes scratch of its own (the tile lists: n / 8 bytes per step), which memory that
// is nearly full may not hold: the solve then runs on all rows.
int apply_device(kb_graph *g, kb_method method, kb_phi phi, const kb_params *params, const int32_t *nodes, int32_t M,
                 int32_t m, float *Y, void *stream, kb_info *info) {
    bool restricted = true;
    int rc = apply_once(g, method, phi, params, nodes, M, m, Y, stream, info, restricted);
    if (rc == KB_ERR_NOMEM && restricted) {
        restricted = false;
        rc = apply_once(g, method, phi, params, nodes, M, m, Y, stream, info, restricted);
    }
    return rc;
}

}  // namespace

extern "C" int kb_krylov_apply(kb_graph *g, kb_method method, kb_phi phi, const kb_params *params,
                               const int32_t *nodes, int32_t M, int32_t m, float *Y, void *stream,
                               kb_info *info) {
    try {
        return apply_device(g, method, phi, params, nodes, M, m, Y, stream, info);
    } catch (const std::bad_alloc &) {
        return fail(KB_ERR_NOMEM, "host allocation failed");
    } catch (...) {
        return fail(KB_ERR_CUDA, "unexpected exception");
    }
}

extern "C" int kb_krylov_apply_host(kb_graph *g, kb_method method, kb_phi phi,
                                    const kb_params *params, const int32_t *nodes, int32_t M,
                                    int32_t m, float *Y_host, void *stream, kb_info *info) {
    try {
        if (!g || !Y_host) return fail(KB_ERR_ARG, "graph or Y_host is NULL");
        if (M < 1 || M > g->dev.n) return fail(KB_ERR_ARG, "M out of range");
        DeviceGuard dg;
        KB_CUDA_TRY(dg.set(g->device));
        cudaStream_t s = static_cast<cudaStream_t>(stream);
        float *dY = nullptr;
        const size_t bytes = sizeof(float) * size_t(g->dev.n) * size_t(M);
        KB_CUDA_TRY(cudaMallocAsync(reinterpret_cast<void **>(&dY), bytes, s));
        int rc = apply_device(g, method, phi, params, nodes, M, m, dY, stream, info);
        if (rc == KB_OK || rc == KB_ERR_BREAKDOWN) {
            cudaError_t e = cudaMemcpyAsync(Y_host, dY, bytes, cudaMemcpyDeviceToHost, s);
            if (e == cudaSuccess) e = cudaStreamSynchronize(s);
            if (e != cudaSuccess && rc == KB_OK) rc = cuda_fail(e, "result copy");
        }
        cudaFreeAsync(dY, s);
        cudaStreamSynchronize(s);
        return rc;
    } catch (...) {
        return fail(KB_ERR_CUDA, "unexpected exception");
    }
}

extern "C" int kb_workspace_bytes(kb_graph *g, kb_method method, kb_phi phi, const kb_params *params,
                                  int32_t M, int32_t m, uint64_t *bytes) {
    try {
        if (!bytes) return fail(KB_ERR_ARG, "bytes is NULL");
        if (!g) return fail(KB_ERR_ARG, "graph is NULL");
        if (M < 1 || M > g->dev.n) return fail(KB_ERR_ARG, "M out of range");
        // validate everything but the node list (a dummy non-null list of distinct nodes)
        std::vector<int32_t> dummy(static_cast<size_t>(M));
        for (int i = 0; i < M; ++i) dummy[i] = i;
        int s_int = 0;
        const float probe = 0.f;
        int rc = validate(g, method, phi, params, dummy.data(), M, m, &probe, &s_int);
        if (rc) return rc;
        // (the plan asks for the occupancy of kernels, which sets their attributes: on the graph's device)
        DeviceGuard dg;
        KB_CUDA_TRY(dg.set(g->device));
        auto quad = std::make_unique<QuadRule>();
        rc = quad_setup(g, method, phi, *params, *quad);
        if (rc) return rc;
        const Common c = solve_of(g, method, phi, *params, M, m, s_int, nullptr, *quad, true);
        switch (params->basis) {
            case KB_F64: *bytes = workspace_bytes_t<double>(c, method, M, m); break;
            case KB_BF16: *bytes = workspace_bytes_t<__nv_bfloat16>(c, method, M, m); break;
            default: *bytes = workspace_bytes_t<float>(c, method, M, m); break;
        }
        return KB_OK;
    } catch (...) {
        return fail(KB_ERR_CUDA, "unexpected exception");
    }
}

extern "C" int kb_exp_series_coeffs(double t, double lam, double tol, double *d, int32_t cap,
                                    int32_t *count) {
    if (!d || !count || !(lam > 0)) return fail(KB_ERR_ARG, "bad argument");
    const std::vector<double> v = exp_series_coeffs(t, lam, tol);
    *count = int32_t(v.size());
    for (int i = 0; i < int(v.size()) && i < cap; ++i) d[i] = v[i];
    return int(v.size()) <= cap ? KB_OK : fail(KB_ERR_ARG, "cap too small");
}

extern "C" int kb_cheb_lobatto_coeffs(kb_phi phi, const kb_params *params, int32_t m, double lam,
                                      int32_t sqrt_phi, double *c) {
    if (!params || !c || m < 1 || !(lam > 0)) return fail(KB_ERR_ARG, "bad argument");
    const std::vector<double> v = lobatto_coeffs(phi, *params, m, lam, sqrt_phi != 0);
    for (int k = 0; k <= m; ++k) c[k] = v[k];
    return KB_OK;
}
