// The projected problem U = phi(H_m) F_1 of the classical block Lanczos method
// (the projected step of Algorithm 1), in FP64 on the device.
//
// H_m is block tridiagonal: diagonal blocks H_kk (symmetric) and sub-diagonal blocks
// H_{k+1,k} = R (upper triangular), super-diagonal blocks R^T.  Its spectrum lies in
// [0, Lambda] (interlacing, proof of Theorem 3.1), so:
//   * exp:    U = sum_j d_j T_j(I - 2 H/Lambda) F_1 with the Chebyshev coefficients d_j
//             of e^{-t lambda} on [0, Lambda] (computed on the host from modified Bessel
//             functions), by the three-term recurrence on the block vectors V_j.  V_j is
//             supported on block rows 0..j, so iteration j touches only j+2 block rows.
//   * spline: for integer s, s solves with the SPD block tridiagonal eps I + H_m through
//             its block Cholesky factorisation (block Thomas algorithm).  For non-integer s
//             the fractional factor (eps I + H_m)^{-alpha} F_1 is the quadrature sum
//             sum_k W_k (sigma_k I + H_m)^{-1} F_1 over real shifts sigma_k > eps
//             (quadrature.cu), one block Cholesky factorisation and solve per node, the nodes
//             in parallel (one CTA each), followed by floor(s) solves with eps I + H_m.
// Both give the same U as the spectral evaluation assumed in Section 7, up to FP64
// rounding (the Chebyshev series is truncated below 1e-17 relative).
#include "kb_internal.cuh"
#include "kb_kernels.cuh"
#include "smallmat.cuh"

namespace kb {
namespace {

constexpr int TC = 4;    // output columns per CTA (many small CTAs: the FP64 work spreads over all SMs)

// U = 0, only when the solve has steps: the stopping rule's later checks run with no steps
// and must leave the buffer of the check that stopped the process as it is.
__global__ void k_zero_if_active(double *U, int64_t count, const Ctrl *ctrl) {
    if (ctrl->steps <= 0) return;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < count;
         i += int64_t(gridDim.x) * blockDim.x)
        U[i] = 0.0;
}
int zero_if_active(double *U, int64_t count, const Ctrl *ctrl, cudaStream_t s) {
    const int grid = int(std::max<int64_t>(1, std::min<int64_t>((count + 255) / 256, 4 * int64_t(num_sms()))));
    k_zero_if_active<<<grid, 256, 0, s>>>(U, count, ctrl);
    return 0;
}

__global__ void k_cheb_bt_seed(double *V0, double *U, int M, double d0, const Ctrl *ctrl) {
    const int i = threadIdx.x + blockIdx.x * blockDim.x;
    if (ctrl->steps > 0 && i < M) {
        V0[int64_t(i) * M + i] = 1.0;
        U[int64_t(i) * M + i] = d0;
    }
}

// V_{j+1} = beta (V_j - g H V_j) - gamma V_{j-1};  U += d_{j+1} V_{j+1}
__global__ void __launch_bounds__(256)
k_cheb_bt_iter(const double *__restrict__ Hd, const double *__restrict__ Hs,
               const double *__restrict__ Vp, const double *__restrict__ Vc, double *__restrict__ Vn,
               double *__restrict__ U, int M, double beta, double gamma, double dnext, double g,
               const Ctrl *ctrl) {
    const int r = blockIdx.x;
    const int steps = ctrl->steps;
    if (r >= steps) return;
    const int c0 = blockIdx.y * TC;
    extern __shared__ double sv[];   // [3][M][TC]
    double *s0 = sv, *s1 = sv + M * TC, *s2 = sv + 2 * M * TC;
    const int64_t MM = int64_t(M) * M;
    for (int idx = threadIdx.x; idx < M * TC; idx += blockDim.x) {
        const int k = idx / TC, cc = idx % TC, c = c0 + cc;
        double a = 0.0, b = 0.0, d = 0.0;
        if (c < M) {
            if (r > 0) a = Vc[(r - 1) * MM + int64_t(k) * M + c];
            b = Vc[r * MM + int64_t(k) * M + c];
            if (r + 1 < steps) d = Vc[(r + 1) * MM + int64_t(k) * M + c];
        }
        s0[idx] = a; s1[idx] = b; s2[idx] = d;
    }
    __syncthreads();
    const double *hd = Hd + r * MM;
    const double *hl = (r > 0) ? Hs + (r - 1) * MM : nullptr;   // H_{r, r-1} = R_{r-1} (upper)
    const double *hu = (r + 1 < steps) ? Hs + r * MM : nullptr; // H_{r, r+1} = R_r^T
    for (int idx = threadIdx.x; idx < M * TC; idx += blockDim.x) {
        const int i = idx / TC, cc = idx % TC, c = c0 + cc;
        if (c >= M) continue;
        double hv = 0.0;
        for (int k = 0; k < M; ++k) hv = fma(hd[i * M + k], s1[k * TC + cc], hv);
        if (hl)
            for (int k = i; k < M; ++k) hv = fma(hl[i * M + k], s0[k * TC + cc], hv);
        if (hu)
            for (int k = 0; k <= i; ++k) hv = fma(hu[k * M + i], s2[k * TC + cc], hv);
        const double av = s1[i * TC + cc] - g * hv;
        const int64_t o = r * MM + int64_t(i) * M + c;
        const double vn = beta * av - gamma * Vp[o];
        Vn[o] = vn;
        U[o] += dnext * vn;
    }
}

// ---------------------------------------------------------------- double-float recurrence
// The same recurrence with V held as unevaluated float pairs (hi + lo, about 48 significant
// bits) on the FP32 pipe, which this part runs at 64 times its FP64 rate.  The entries of H
// are FP32 values (the blocks are recorded as the FP32 recurrence subtracts them), so H is one
// float per entry.  The products are compensated dot products (Ogita, Rump and Oishi's
// Dot2): each h v term is split exactly by an FMA (TwoProd), the running sum by Knuth's
// TwoSum, and the rounding errors are summed beside it; the result is exact to about 2^-48
// relative, far below the 1e-14 the projected solve needs after thousands of terms.  U is
// accumulated in FP64.
struct dfl {
    float h, l;
};
__device__ __forceinline__ dfl dfl_fast(float s, float e) {   // |s| >= |e|
    const float h = s + e;
    return dfl{h, e - (h - s)};
}
// sum += a * b, exact products and sums tracked in (s, err)
__device__ __forceinline__ void dot2_step(float &s, float &err, dfl a, dfl b) {
    const float p = a.h * b.h;
    float pe = fmaf(a.h, b.h, -p);
    pe = fmaf(a.h, b.l, pe);
    pe = fmaf(a.l, b.h, pe);
    const float t = s + p;
    const float bb = t - s;
    err += ((s - (t - bb)) + (p - bb)) + pe;
    s = t;
}
// the same with a single float a
__device__ __forceinline__ void dot2_step(float &s, float &err, float a, dfl b) {
    const float p = a * b.h;
    const float pe = fmaf(a, b.l, fmaf(a, b.h, -p));
    const float t = s + p;
    const float bb = t - s;
    err += ((s - (t - bb)) + (p - bb)) + pe;
    s = t;
}
__host__ __device__ __forceinline__ dfl dfl_from(double v) {
    const float h = float(v);
    return dfl{h, float(v - double(h))};
}
__device__ __forceinline__ double dfl_val(dfl a) { return double(a.h) + double(a.l); }

// The float form of H, every block so that the recurrence reads it along rows of 2 floats: rows
// of ld = M rounded up to even, zeros in the padding.  Hdf: H_rr (symmetric); Hsf: R_r =
// H_{r+1,r} (upper triangular); Hst: R_r^T.  Once per projected solve.
__global__ void __launch_bounds__(256)
k_split_df(const double *__restrict__ Hd, const double *__restrict__ Hs, float *__restrict__ Hdf,
           float *__restrict__ Hsf, float *__restrict__ Hst, int M, int ld, const Ctrl *ctrl) {
    const int r = blockIdx.x;
    if (r >= ctrl->steps) return;
    const int64_t MM = int64_t(M) * M, LL = int64_t(M) * ld;
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int i = (threadIdx.x >> 5) + blockIdx.y * nw; i < M; i += nw * gridDim.y)
        for (int j = lane; j < ld; j += 32) {
            const bool in = j < M;
            Hdf[r * LL + i * ld + j] = in ? float(Hd[r * MM + i * M + j]) : 0.f;
            if (r + 1 < ctrl->steps) {
                Hsf[r * LL + i * ld + j] = in && j >= i ? float(Hs[r * MM + i * M + j]) : 0.f;
                Hst[r * LL + i * ld + j] = in && j <= i ? float(Hs[r * MM + j * M + i]) : 0.f;
            }
        }
}

__global__ void k_cheb_bt_seed_df(dfl *V0, double *U, int M, double d0, const Ctrl *ctrl) {
    const int i = threadIdx.x + blockIdx.x * blockDim.x;
    if (ctrl->steps > 0 && i < M) {
        V0[int64_t(i) * M + i] = dfl{1.f, 0.f};
        U[int64_t(i) * M + i] = d0;
    }
}

// V_{j+1} = beta (V_j - g H V_j) - gamma V_{j-1};  U += d_{j+1} V_{j+1}, in double-float.
// A CTA forms 8 columns of one block row.  The three blocks of H and the V columns of the three
// block rows that enter are copied to shared memory at once (cp.async; H_rr is symmetric,
// R_{r-1} comes transposed and R_r^T is read as R_r, so all are read along the output rows), and
// a thread owns 2 rows x 2 columns: two shared loads per 4 compensated terms of 11 operations,
// instead of one strided 8-byte global load and one shared load per term.  Bound by the
// FP32 pipe and the latency of a launch.  Per term, launch list: M = 64 with 30 blocks
// 30.3 -> 16.7 us, M = 40 with 20 blocks 16.9 -> 12.2 us.
constexpr int CBW = 8;
__global__ void __launch_bounds__(256)
k_cheb_bt_iter_df(const float *__restrict__ Hd, const float *__restrict__ Hs, const float *__restrict__ Hst,
                  const dfl *__restrict__ Vp, const dfl *__restrict__ Vc, dfl *__restrict__ Vn,
                  double *__restrict__ U, int M, int ld, float beta, float gamma, double dnext, dfl g,
                  const Ctrl *ctrl) {
    const int r = blockIdx.x;
    const int steps = ctrl->steps;
    if (r >= steps) return;
    const int c0 = blockIdx.y * CBW;
    extern __shared__ __align__(16) unsigned char svraw[];   // V [3][M][CBW] pairs, H [3][M][ld]
    dfl *s1 = reinterpret_cast<dfl *>(svraw), *s0 = s1 + M * CBW, *s2 = s0 + M * CBW;
    float *h1 = reinterpret_cast<float *>(s2 + M * CBW), *h0 = h1 + M * ld, *h2 = h0 + M * ld;
    const int64_t MM = int64_t(M) * M, LL = int64_t(M) * ld;
    auto copy8 = [](void *dst, const void *src) {
        const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
    };
    for (int i = threadIdx.x * 2; i < M * ld; i += blockDim.x * 2) {
        copy8(h1 + i, Hd + r * LL + i);
        if (r > 0) copy8(h0 + i, Hst + (r - 1) * LL + i);
        if (r + 1 < steps) copy8(h2 + i, Hs + r * LL + i);
    }
    for (int idx = threadIdx.x; idx < M * CBW; idx += blockDim.x) {
        const int k = idx / CBW, c = c0 + idx % CBW;
        const int64_t o = r * MM + int64_t(k) * M + c;
        if (c < M) {
            copy8(s1 + idx, Vc + o);
            if (r > 0) copy8(s0 + idx, Vc + o - MM);
            if (r + 1 < steps) copy8(s2 + idx, Vc + o + MM);
        } else {
            s1[idx] = s0[idx] = s2[idx] = dfl{0.f, 0.f};
        }
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    const int i0 = (threadIdx.x / 4) * 2, cc = (threadIdx.x % 4) * 2;
    if (i0 >= M || c0 + cc >= M) return;
    float s[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, err[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
    // rows k0 .. k1 - 1 of a block stored along the output rows, times V
    auto acc = [&](const float *H, const dfl *v, int k0, int k1) {
#pragma unroll 4
        for (int k = k0; k < k1; ++k) {
            const float2 h = *reinterpret_cast<const float2 *>(H + k * ld + i0);
            const float4 t = *reinterpret_cast<const float4 *>(v + k * CBW + cc);
            const dfl va{t.x, t.y}, vb{t.z, t.w};
            dot2_step(s[0][0], err[0][0], h.x, va);
            dot2_step(s[0][1], err[0][1], h.x, vb);
            dot2_step(s[1][0], err[1][0], h.y, va);
            dot2_step(s[1][1], err[1][1], h.y, vb);
        }
    };
    acc(h1, s1, 0, M);
    if (r > 0) acc(h0, s0, i0, M);                           // R_{r-1}: k >= i
    if (r + 1 < steps) acc(h2, s2, 0, min(i0 + 2, M));       // R_r^T: k <= i
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int i = i0 + a, c = c0 + cc + b;
            if (i >= M || c >= M) continue;
            // av = V_j - g (H V_j): one more compensated step with the pair -g
            const dfl hv = dfl_fast(s[a][b], err[a][b]);
            const dfl v1 = s1[i * CBW + cc + b];
            float s2v = v1.h, e2 = v1.l;
            dot2_step(s2v, e2, dfl{-g.h, -g.l}, hv);
            // vn = beta av - gamma V_{j-1} (beta in {1, 2}, gamma in {0, 1}: exact scalings)
            const int64_t o = r * MM + int64_t(i) * M + c;
            const dfl vp = Vp[o];
            float s3 = beta * s2v, e3 = beta * e2;
            dot2_step(s3, e3, -gamma, vp);
            const dfl vn = dfl_fast(s3, e3);
            Vn[o] = vn;
            U[o] += dnext * dfl_val(vn);
        }
}

// The whole series (terms j0 .. j0 + cc.n of it) in one cooperative launch: a CTA keeps up to NI
// items (8 columns of one block row), its U and V_{j-1} entries in registers and, with one item,
// the three blocks of H in shared memory for all terms; a term reads the neighbours' V from
// L2, and a grid barrier separates the terms.  A launch per term costs more than its
// arithmetic, above all with several solves in flight.  Row r of V_j is zero for r > j and never
// read.  V_j lives in slot j % 3.  Measured, a whole series, launch list:
// 65 terms, M = 64, 30 blocks 1085 -> 925 us; 48 terms, M = 40, 20 blocks 585 -> 447 us; the four
// concurrent requests of the serving mix on a hub graph (5300 terms) 41.0 -> 33.7 ms.
template <int NI>
__global__ void __launch_bounds__(256)
k_cheb_bt_all(const float *__restrict__ Hd, const float *__restrict__ Hs, const float *__restrict__ Hst, dfl *V0,
              dfl *V1, dfl *V2, double *__restrict__ U, int M, int ld, ChebCoef cc, int j0, dfl g,
              const Ctrl *ctrl, int32_t *sync, Ctrl *proc, int spins) {
    const int steps = ctrl->steps;
    if (steps <= 0) return;
    extern __shared__ __align__(16) unsigned char svraw[];   // V [3][M][CBW] pairs, H [3][M][ld]
    dfl *s1 = reinterpret_cast<dfl *>(svraw), *s0 = s1 + M * CBW, *s2 = s0 + M * CBW;
    float *h1 = reinterpret_cast<float *>(s2 + M * CBW), *h0 = h1 + M * ld, *h2 = h0 + M * ld;
    const int64_t MM = int64_t(M) * M, LL = int64_t(M) * ld;
    const int slabs = (M + CBW - 1) / CBW, items = steps * slabs;
    const int i0 = int(threadIdx.x / 4) * 2, cc2 = int(threadIdx.x % 4) * 2;
    auto slot = [&](int j) { return j % 3 == 0 ? V0 : j % 3 == 1 ? V1 : V2; };
    dfl vp[NI][2][2];      // V_{j-2} at this thread's entries
    double u[NI][2][2];
#pragma unroll
    for (int n = 0; n < NI; ++n) {
        const int id = blockIdx.x + n * gridDim.x, r = id % steps, c0 = id / steps * CBW;
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const int i = i0 + a, c = c0 + cc2 + b;
                vp[n][a][b] = dfl{0.f, 0.f};
                u[n][a][b] = 0.0;
                if (id >= items || i >= M || c >= M) continue;
                const int64_t o = r * MM + int64_t(i) * M + c;
                if (j0 == 0) {
                    // V_0 = F_1
                    const float e = r == 0 && i == c ? 1.f : 0.f;
                    if (r == 0) V0[o] = dfl{e, 0.f};
                    u[n][a][b] = cc.d[0] * double(e);
                } else {
                    u[n][a][b] = U[o];
                    if (r <= j0 - 2) vp[n][a][b] = slot(j0 - 2)[o];
                }
            }
    }
    int target = 0;
    bool good = true;
    if (j0 == 0) good = grid_barrier(sync, sync + 1, target += gridDim.x, spins);
    auto copy8 = [](void *dst, const void *src) {
        const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
    };
    for (int q = j0 == 0 ? 1 : 0; good && q < cc.n; ++q) {
        const int j = j0 + q;
        const dfl *Vc = slot(j - 1);
        dfl *Vn = slot(j);
        const float beta = j == 1 ? 1.f : 2.f, gamma = j == 1 ? 0.f : 1.f;
#pragma unroll
        for (int n = 0; n < NI; ++n) {
            const int id = blockIdx.x + n * gridDim.x, r = id % steps, c0 = id / steps * CBW;
            if (id >= items || r > j) continue;   // (uniform; V_j is zero there)
            if (NI > 1 || q == (j0 == 0 ? 1 : 0) || r == j) {
                // H of this item (with one item: once, when its row is first reached)
                for (int i = threadIdx.x * 2; i < M * ld; i += blockDim.x * 2) {
                    copy8(h1 + i, Hd + r * LL + i);
                    if (r > 0) copy8(h0 + i, Hst + (r - 1) * LL + i);
                    if (r + 1 < steps) copy8(h2 + i, Hs + r * LL + i);
                }
            }
            // (V through L2: its slots are rewritten by other SMs)
            for (int idx = threadIdx.x; idx < M * CBW; idx += blockDim.x) {
                const int k = idx / CBW, c = c0 + idx % CBW;
                const int64_t o = r * MM + int64_t(k) * M + c;
                float2 a{0.f, 0.f}, b{0.f, 0.f}, d{0.f, 0.f};
                if (c < M) {
                    if (r > 0) a = __ldcg(reinterpret_cast<const float2 *>(Vc + o - MM));
                    if (r <= j - 1) b = __ldcg(reinterpret_cast<const float2 *>(Vc + o));
                    if (r + 1 <= j - 1 && r + 1 < steps) d = __ldcg(reinterpret_cast<const float2 *>(Vc + o + MM));
                }
                s0[idx] = dfl{a.x, a.y};
                s1[idx] = dfl{b.x, b.y};
                s2[idx] = dfl{d.x, d.y};
            }
            asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
            __syncthreads();
            if (i0 < M && c0 + cc2 < M) {
                float s[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, err[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
                auto acc = [&](const float *H, const dfl *v, int k0, int k1) {
#pragma unroll 4
                    for (int k = k0; k < k1; ++k) {
                        const float2 h = *reinterpret_cast<const float2 *>(H + k * ld + i0);
                        const float4 t = *reinterpret_cast<const float4 *>(v + k * CBW + cc2);
                        const dfl va{t.x, t.y}, vb{t.z, t.w};
                        dot2_step(s[0][0], err[0][0], h.x, va);
                        dot2_step(s[0][1], err[0][1], h.x, vb);
                        dot2_step(s[1][0], err[1][0], h.y, va);
                        dot2_step(s[1][1], err[1][1], h.y, vb);
                    }
                };
                if (r <= j - 1) acc(h1, s1, 0, M);
                if (r > 0) acc(h0, s0, i0, M);                                             // R_{r-1}: k >= i
                if (r + 1 <= j - 1 && r + 1 < steps) acc(h2, s2, 0, min(i0 + 2, M));       // R_r^T: k <= i
#pragma unroll
                for (int a = 0; a < 2; ++a)
#pragma unroll
                    for (int b = 0; b < 2; ++b) {
                        const int i = i0 + a, c = c0 + cc2 + b;
                        if (i >= M || c >= M) continue;
                        const dfl hv = dfl_fast(s[a][b], err[a][b]);
                        const dfl v1 = s1[i * CBW + cc2 + b];
                        float s2v = v1.h, e2 = v1.l;
                        dot2_step(s2v, e2, dfl{-g.h, -g.l}, hv);
                        float s3 = beta * s2v, e3 = beta * e2;
                        dot2_step(s3, e3, -gamma, vp[n][a][b]);
                        const dfl vn = dfl_fast(s3, e3);
                        Vn[r * MM + int64_t(i) * M + c] = vn;
                        vp[n][a][b] = v1;
                        u[n][a][b] += cc.d[q] * dfl_val(vn);
                    }
            }
            __syncthreads();
        }
        if (q + 1 < cc.n) good = grid_barrier(sync, sync + 1, target += gridDim.x, spins);
    }
    // a barrier ran out: U is not to be used, and the process ends
    if (!good && proc && threadIdx.x == 0) {
        proc->status = KB_ERR_CUDA;
        proc->steps = steps;
        proc->stop = 1;
    }
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
#pragma unroll
    for (int n = 0; n < NI; ++n) {
        const int id = blockIdx.x + n * gridDim.x, r = id % steps, c0 = id / steps * CBW;
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const int i = i0 + a, c = c0 + cc2 + b;
                if (id < items && i < M && c < M) U[r * MM + int64_t(i) * M + c] = good ? u[n][a][b] : nan;
            }
    }
}

// ---------------------------------------------------------------- block Cholesky (spline)
// One CTA; all scratch in global memory (L1/L2 resident for the sizes used).
__device__ void chol_lower_inplace(double *A, int M) {
    // A = L L^T, lower L overwrites A (upper part left as is); the trailing update runs rows
    // by warp and columns by lane (no index division, no idle half)
    __shared__ double piv, rpiv;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int j = 0; j < M; ++j) {
        if (threadIdx.x == 0) {
            double d = A[j * M + j];
            piv = sqrt(fmax(d, 1e-300));
            rpiv = 1.0 / piv;
            A[j * M + j] = piv;
        }
        __syncthreads();
        for (int i = j + 1 + threadIdx.x; i < M; i += blockDim.x) A[i * M + j] *= rpiv;
        __syncthreads();
        for (int a = j + 1 + warp; a < M; a += nw) {
            const double laj = A[a * M + j];
            for (int b = j + 1 + lane; b <= a; b += 32) A[a * M + b] -= laj * A[b * M + j];
        }
        __syncthreads();
    }
}

// Spline kernel, s_int times U <- (eps I + H)^{-1} U through the block Cholesky factorisation
// eps I + H = L L^T (L block lower bidiagonal: R_r^T on the diagonal, Ls_r below it).  All in
// FP64, whose rate on this part is two FMAs per clock and SM, so everything but the Cholesky
// of one diagonal block is spread over many SMs, and the triangular solves are turned into
// products with the inverses Ri_r = R_r^{-1}, whose terms are independent:
//   k_bt_ls      Ls_{r-1} = H_{r,r-1} Ri_{r-1}
//   k_bt_schur   D_r = eps I + H_rr - Ls_{r-1} Ls_{r-1}^T, and K_{r-1} = Ls_{r-1} Ri_{r-1}^T
//   k_bt_dchol   D_r = R_r^T R_r, Ri_r and its transpose (one CTA)
//   k_bt_gt      G_r^T = Ls_{r-1}^T Ri_r for all new blocks
//   k_bt_subst   Y_r = Ri_r^T rhs_r - G_r Y_{r-1} upwards, U_r = Ri_r Y_r - K_r^T U_{r+1}
//                downwards, one CTA per column of U
// The leading blocks of eps I + H_k do not change as k grows, nor do their Y_r for the first
// solve: a stopping-rule check extends what the check before it left (blocks r0 and up).
// Each launch does nothing when its block lies past the process's steps, or once a check has
// stopped the process.  Measured (four concurrent requests, RGG of 55392 rows, M = 64 and less,
// (0.1 I + L)^{-1}, up to 100 steps, checks at 8 to 96): sums of the launch list 239 -> 62 ms
// (every check factored all blocks and solved triangular systems with one warp per column),
// the requests 156 -> 81 ms; with the blocks factored beside the Lanczos steps, as krylov.cu has
// it, and the steps' other changes 62 ms.
struct BtArgs {
    const double *Hd, *Hs;
    double *Ri, *RiT, *Y, *GT, *K, *Ls;   // Ls: two blocks, by the parity of r
    int M;
};
__device__ __forceinline__ bool bt_skip(const Ctrl *fc, int r) { return r >= fc->steps || fc->from_check >= 0; }

// sum of four interleaved partial sums of a(k) b(k), k0 <= k < k1
template <typename FA, typename FB>
__device__ __forceinline__ double dot4(int k0, int k1, const FA &a, const FB &b) {
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    int k = k0;
    for (; k + 3 < k1; k += 4)
#pragma unroll
        for (int u = 0; u < 4; ++u) s[u] = fma(a(k + u), b(k + u), s[u]);
    for (; k < k1; ++k) s[0] = fma(a(k), b(k), s[0]);
    return (s[0] + s[1]) + (s[2] + s[3]);
}

// row i = blockIdx.x of Ls_{r-1} (both factors upper triangular)
__global__ void __launch_bounds__(128) k_bt_ls(BtArgs a, int r, const Ctrl *fc) {
    pdl_wait();
    if (bt_skip(fc, r)) return;
    pdl_trigger();
    const int M = a.M, i = blockIdx.x;
    const int64_t MM = int64_t(M) * M;
    const double *h = a.Hs + (r - 1) * MM + int64_t(i) * M, *Ri = a.Ri + (r - 1) * MM;
    double *out = a.Ls + ((r - 1) & 1) * MM + int64_t(i) * M;
    for (int j = threadIdx.x; j < M; j += blockDim.x)
        out[j] = j < i ? 0.0 : dot4(i, j + 1, [&](int k) { return h[k]; }, [&](int k) { return Ri[int64_t(k) * M + j]; });
}

// row i: of D_r (blockIdx.y = 0, into Ri_r, lower triangle transposed to the upper one) and of
// K_{r-1} (blockIdx.y = 1)
__global__ void __launch_bounds__(128) k_bt_schur(BtArgs a, int r, double eps, const Ctrl *fc) {
    pdl_wait();
    if (bt_skip(fc, r)) return;
    pdl_trigger();
    const int M = a.M, i = blockIdx.x;
    const int64_t MM = int64_t(M) * M;
    const double *L = a.Ls + ((r - 1) & 1) * MM;
    if (blockIdx.y == 0) {
        for (int j = threadIdx.x; j < M; j += blockDim.x) {
            if (j < i) continue;
            double v = a.Hd[r * MM + int64_t(i) * M + j] + (i == j ? eps : 0.0);
            if (r > 0)   // (rows of an upper triangular matrix: k >= j)
                v -= dot4(j, M, [&](int k) { return L[int64_t(i) * M + k]; }, [&](int k) { return L[int64_t(j) * M + k]; });
            a.Ri[r * MM + int64_t(i) * M + j] = v;
        }
    } else {
        const double *RiT = a.RiT + (r - 1) * MM;
        for (int j = threadIdx.x; j < M; j += blockDim.x)
            a.K[(r - 1) * MM + int64_t(i) * M + j] =
                dot4(max(i, j), M, [&](int k) { return L[int64_t(i) * M + k]; },
                     [&](int k) { return RiT[int64_t(k) * M + j]; });
    }
}

__global__ void __launch_bounds__(512) k_bt_dchol(BtArgs a, int r, const Ctrl *fc) {
    pdl_wait();
    if (bt_skip(fc, r)) return;
    extern __shared__ __align__(16) double bsm[];
    const int M = a.M, lda = (M + 1) / 2 * 2;
    double *A = bsm, *scr = A + lda * lda, *tmp = scr + sm::NB * sm::NB;
    const int64_t o = r * int64_t(M) * M;
    sm::each(M, M, [&](int i, int j) { A[i * lda + j] = j >= i ? __ldcg(a.Ri + o + i * M + j) : 0.0; });
    __syncthreads();
    const bool ok = sm::chol_blocked<double>(A, nullptr, lda, M, 0.0, scr);
    if (ok) {
        sm::each(M, M, [&](int i, int j) {
            if (j < i) A[i * lda + j] = 0.0;
        });
        __syncthreads();
        sm::tri_inv_diag<double>(A, lda, M);
        sm::tri_inv_merge<double>(A, lda, M, tmp);
    }
    pdl_trigger();
    // a block that is not positive definite (lost orthogonality) shows as NaN
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    sm::each(M, M, [&](int i, int j) {
        a.Ri[o + i * M + j] = ok ? A[i * lda + j] : nan;
        a.RiT[o + i * M + j] = ok ? A[j * lda + i] : nan;
    });
}

// row i = blockIdx.x of G_r^T (Ri_r upper triangular, Ls_{r-1} upper triangular)
__global__ void __launch_bounds__(128) k_bt_gt(BtArgs a, int r, const Ctrl *fc) {
    pdl_wait();
    if (bt_skip(fc, r)) return;
    pdl_trigger();
    const int M = a.M, i = blockIdx.x;
    const int64_t MM = int64_t(M) * M;
    const double *L = a.Ls + ((r - 1) & 1) * MM, *Ri = a.Ri + r * MM;
    for (int j = threadIdx.x; j < M; j += blockDim.x)
        a.GT[r * MM + int64_t(i) * M + j] =
            dot4(0, min(i, j) + 1, [&](int k) { return L[int64_t(k) * M + i]; }, [&](int k) { return Ri[int64_t(k) * M + j]; });
}

// One column c = blockIdx.x of U per CTA.  A product with an M x M matrix stored by the input
// index (rows contiguous in the output index) gives each thread one output row and a part of
// the inputs; the parts are added in shared memory.  y0: first block whose Y of the first
// solve is not known yet.
constexpr int BTS_THREADS = 256;
__global__ void __launch_bounds__(BTS_THREADS)
k_bt_subst(BtArgs a, int s_int, int y0, double *__restrict__ U, const Ctrl *ctrl, int rhs_in_u) {
    const int steps = ctrl->steps, M = a.M, c = blockIdx.x;
    if (steps <= 0) return;
    __shared__ double v[2][128], w[2][128], part[BTS_THREADS];
    const int64_t MM = int64_t(M) * M;
    int Mp = 32;
    while (Mp < M) Mp *= 2;
    const int row = threadIdx.x % Mp, ks = threadIdx.x / Mp, nks = BTS_THREADS / Mp;
    // part of sum_k A[k][row] x_k over this thread's inputs
    auto mv = [&](const double *A, const double *x) -> double {
        if (row >= M) return 0.0;
        double s0 = 0.0, s1 = 0.0;
        int k = ks;
        for (; k + nks < M; k += 2 * nks) {
            s0 = fma(A[int64_t(k) * M + row], x[k], s0);
            s1 = fma(A[int64_t(k + nks) * M + row], x[k + nks], s1);
        }
        if (k < M) s0 = fma(A[int64_t(k) * M + row], x[k], s0);
        return s0 + s1;
    };
    auto total = [&](double p) -> double {   // valid for ks == 0
        part[threadIdx.x] = p;
        __syncthreads();
        double t = 0.0;
        if (ks == 0)
            for (int q = 0; q < nks; ++q) t += part[q * Mp + row];
        return t;
    };
    for (int rep = 0; rep < s_int; ++rep) {
        // upwards: Y_r = Ri_r^T rhs_r - G_r Y_{r-1}
        const bool unit = rep == 0 && !rhs_in_u;     // rhs = F_1
        const int r0 = unit ? y0 : 0;
        if (r0 > 0 && threadIdx.x < M) v[(r0 - 1) & 1][threadIdx.x] = a.Y[(r0 - 1) * MM + int64_t(c) * M + threadIdx.x];
        for (int r = r0; r < steps; ++r) {
            double p = 0.0;
            if (!unit) {
                if (threadIdx.x < M) w[r & 1][threadIdx.x] = U[r * MM + int64_t(threadIdx.x) * M + c];
                __syncthreads();
                p = mv(a.Ri + r * MM, w[r & 1]);
            } else if (r == 0 && ks == 0 && row < M) {
                p = a.Ri[int64_t(c) * M + row];
            }
            __syncthreads();
            if (r > 0) p -= mv(a.GT + r * MM, v[(r - 1) & 1]);
            const double t = total(p);
            if (ks == 0 && row < M) {
                v[r & 1][row] = t;
                a.Y[r * MM + int64_t(c) * M + row] = t;
            }
            __syncthreads();
        }
        // downwards: U_r = Ri_r Y_r - K_r^T U_{r+1}
        for (int r = steps - 1; r >= 0; --r) {
            if (threadIdx.x < M) w[r & 1][threadIdx.x] = a.Y[r * MM + int64_t(c) * M + threadIdx.x];
            __syncthreads();
            double p = mv(a.RiT + r * MM, w[r & 1]);
            if (r + 1 < steps) p -= mv(a.K + r * MM, v[(r + 1) & 1]);
            const double t = total(p);
            if (ks == 0 && row < M) {
                v[r & 1][row] = t;
                U[r * MM + int64_t(row) * M + c] = t;
            }
            __syncthreads();
        }
    }
}

// ---------------------------------------------------------------- quadrature nodes (spline)
// One CTA per quadrature node: Y = (sigma I + H)^{-1} F_1 through the block Cholesky
// factorisation sigma I + H = L L^T (L block lower bidiagonal: diagonal blocks Ld_r lower
// triangular, sub-diagonal blocks Ls_r = L_{r+1,r}), forward and backward block substitution.
// The triangular solves give each thread one row (Ls) or one right-hand-side column (Y), so
// they need no barrier inside a block.  Per-node scratch (bt_quad_node_doubles): Ld, Ls, Y
// (mcap blocks of M x M each) and the reciprocal diagonals of the Ld blocks (mcap x M).
constexpr int QN_THREADS = 128;

__global__ void __launch_bounds__(QN_THREADS)
k_bt_shift_solve(const double *__restrict__ Hd, const double *__restrict__ Hs, int M, int mcap,
                 QuadRule q, int node0, double *scratch, const Ctrl *ctrl) {
    const int node = node0 + int(blockIdx.x);
    if (node >= q.n) return;
    const int steps = ctrl->steps;
    const double sigma = q.shift[node];
    const int64_t MM = int64_t(M) * M;
    double *Ld = scratch + int64_t(blockIdx.x) * int64_t(bt_quad_node_doubles(M, mcap));
    double *Ls = Ld + int64_t(mcap) * MM;
    double *Y = Ls + int64_t(mcap) * MM;
    double *rd = Y + int64_t(mcap) * MM;
    const int tid = threadIdx.x;
    for (int r = 0; r < steps; ++r) {
        // D_r = sigma I + H_rr - Ls_{r-1} Ls_{r-1}^T (lower triangle), then D_r = Ld_r Ld_r^T
        double *D = Ld + r * MM;
        const double *P = r > 0 ? Ls + (r - 1) * MM : nullptr;
        for (int idx = tid; idx < M * M; idx += blockDim.x) {
            const int i = idx / M, j = idx % M;
            double v = 0.0;
            if (j <= i) {
                v = Hd[r * MM + idx] + (i == j ? sigma : 0.0);
                if (P)
                    for (int k = 0; k < M; ++k) v = fma(-P[i * M + k], P[j * M + k], v);
            }
            D[idx] = v;
        }
        __syncthreads();
        chol_lower_inplace(D, M);
        for (int i = tid; i < M; i += blockDim.x) rd[r * M + i] = 1.0 / D[i * M + i];
        __syncthreads();
        if (r + 1 < steps) {
            // Ls_r = H_{r+1,r} D_r^{-T}: row i solves D_r x = (row i of H_{r+1,r})^T
            const double *Hsub = Hs + r * MM;
            double *Pn = Ls + r * MM;
            for (int i = tid; i < M; i += blockDim.x)
                for (int j = 0; j < M; ++j) {
                    double v = Hsub[i * M + j];
                    for (int k = 0; k < j; ++k) v = fma(-D[j * M + k], Pn[i * M + k], v);
                    Pn[i * M + j] = v * rd[r * M + j];
                }
            __syncthreads();
        }
    }
    // forward: Y_0 = D_0^{-1} I, Y_r = D_r^{-1} (-Ls_{r-1} Y_{r-1}); one column per thread
    for (int r = 0; r < steps; ++r) {
        const double *D = Ld + r * MM;
        const double *P = r > 0 ? Ls + (r - 1) * MM : nullptr;
        const double *Yp = r > 0 ? Y + (r - 1) * MM : nullptr;
        double *Yr = Y + r * MM;
        for (int c = tid; c < M; c += blockDim.x)
            for (int i = 0; i < M; ++i) {
                double v = (r == 0 && i == c) ? 1.0 : 0.0;
                if (P)
                    for (int k = 0; k < M; ++k) v = fma(-P[i * M + k], Yp[k * M + c], v);
                for (int k = 0; k < i; ++k) v = fma(-D[i * M + k], Yr[k * M + c], v);
                Yr[i * M + c] = v * rd[r * M + i];
            }
        __syncthreads();
    }
    // backward: U_r = D_r^{-T} (Y_r - Ls_r^T U_{r+1}), in place in Y
    for (int r = steps - 1; r >= 0; --r) {
        const double *D = Ld + r * MM;
        const double *P = r + 1 < steps ? Ls + r * MM : nullptr;
        const double *Un = r + 1 < steps ? Y + (r + 1) * MM : nullptr;
        double *Yr = Y + r * MM;
        for (int c = tid; c < M; c += blockDim.x)
            for (int i = M - 1; i >= 0; --i) {
                double v = Yr[i * M + c];
                if (P)
                    for (int k = 0; k < M; ++k) v = fma(-P[k * M + i], Un[k * M + c], v);
                for (int k = i + 1; k < M; ++k) v = fma(-D[k * M + i], Yr[k * M + c], v);
                Yr[i * M + c] = v * rd[r * M + i];
            }
        __syncthreads();
    }
}

// U += sum_{j < nb} W_{node0+j} Y_j over the steps blocks, in a fixed order (deterministic).
__global__ void __launch_bounds__(256)
k_quad_accumulate(const double *__restrict__ scratch, int M, int mcap, int nb, QuadRule q, int node0,
                  double *U, const Ctrl *ctrl) {
    const int64_t cnt = int64_t(ctrl->steps) * M * M;
    const int64_t per = int64_t(bt_quad_node_doubles(M, mcap));
    const int64_t yoff = 2 * int64_t(mcap) * M * M;
    for (int64_t idx = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; idx < cnt;
         idx += int64_t(gridDim.x) * blockDim.x) {
        double acc = U[idx];
        for (int j = 0; j < nb; ++j) acc = fma(q.weight[node0 + j], scratch[j * per + yoff + idx], acc);
        U[idx] = acc;
    }
}

}  // namespace

int launch_cheb_bt(const double *Hd, const double *Hs, int M, int m, double lam,
                   const std::vector<double> &d, double *V0, double *V1, double *V2, double *U,
                   const Ctrl *ctrl, cudaStream_t s, double *Hdf, int32_t *sync, int kmax, Ctrl *proc,
                   int spins) {
    if (kmax <= 0 || kmax > m) kmax = m;
    const size_t bytes = sizeof(double) * size_t(m) * M * M;
    prof_begin(KernelClass::PROJECTED, s);
    if (Hdf) {
        // double-float recurrence: H as floats once, V_j as float pairs in the V buffers
        const int ld = (M + 1) / 2 * 2;
        float *hd = reinterpret_cast<float *>(Hdf), *hs = hd + size_t(m) * M * ld, *ht = hs + size_t(m) * M * ld;
        k_split_df<<<dim3(m, 2), 256, 0, s>>>(Hd, Hs, hd, hs, ht, M, ld, ctrl);
        const size_t smem = sizeof(dfl) * 3 * M * CBW + sizeof(float) * 3 * M * ld;
        const int threads = std::max(32, ((M + 1) / 2 * 4 + 31) / 32 * 32);
        const dfl g = dfl_from(2.0 / lam);
        // all terms in one cooperative launch while a CTA has at most four items (the steps known to
        // the host bound the block rows)
        const int items = kmax * ((M + CBW - 1) / CBW);
        constexpr int SMEM_MAX = int(sizeof(dfl) * 3 * 128 * CBW + sizeof(float) * 3 * 128 * 128);
        static const cudaError_t attrs[] = {
            cudaFuncSetAttribute(k_cheb_bt_all<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX),
            cudaFuncSetAttribute(k_cheb_bt_all<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX),
            cudaFuncSetAttribute(k_cheb_bt_all<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX),
            cudaFuncSetAttribute(k_cheb_bt_iter_df, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX)};
        (void)attrs;
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_cheb_bt_all<4>, threads, smem);
        const int cap = per_sm * num_sms();
        if (sync && cap > 0 && items <= 4 * cap && d.size() >= 2) {
            zero_if_active(U, int64_t(m) * M * M, ctrl, s);
            const int ni = items <= cap ? 1 : items <= 2 * cap ? 2 : 4;
            const int grid = (items + ni - 1) / ni;
            dfl *v[3] = {reinterpret_cast<dfl *>(V0), reinterpret_cast<dfl *>(V1), reinterpret_cast<dfl *>(V2)};
            int launches = 2;
            for (size_t j0 = 0; j0 < d.size(); j0 += ChebCoef::CAP) {
                ChebCoef cc{};
                cc.n = int(std::min<size_t>(ChebCoef::CAP, d.size() - j0));
                for (int q = 0; q < cc.n; ++q) cc.d[q] = d[j0 + q];
                KB_CUDA_TRY(cudaMemsetAsync(sync, 0, 2 * sizeof(int32_t), s));
                cudaLaunchConfig_t cfg{};
                cudaLaunchAttribute at[1];
                at[0].id = cudaLaunchAttributeCooperative;
                at[0].val.cooperative = 1;
                cfg.gridDim = unsigned(grid);
                cfg.blockDim = unsigned(threads);
                cfg.dynamicSmemBytes = smem;
                cfg.stream = s;
                cfg.attrs = at;
                cfg.numAttrs = 1;
                auto kern = ni == 1 ? k_cheb_bt_all<1> : ni == 2 ? k_cheb_bt_all<2> : k_cheb_bt_all<4>;
                KB_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, (const float *)hd, (const float *)hs, (const float *)ht, v[0],
                                               v[1], v[2], U, M, ld, cc, int(j0), g, ctrl, sync, proc, spins));
                ++launches;
            }
            KB_CUDA_TRY(cudaGetLastError());
            prof_end(KernelClass::PROJECTED, s, 0, 0, launches);
            return 0;
        }
        KB_CUDA_TRY(cudaMemsetAsync(V0, 0, bytes, s));
        KB_CUDA_TRY(cudaMemsetAsync(V1, 0, bytes, s));
        KB_CUDA_TRY(cudaMemsetAsync(V2, 0, bytes, s));
        zero_if_active(U, int64_t(m) * M * M, ctrl, s);
        dfl *pp = reinterpret_cast<dfl *>(V2), *pc = reinterpret_cast<dfl *>(V0), *pn = reinterpret_cast<dfl *>(V1);
        k_cheb_bt_seed_df<<<(M + 127) / 128, 128, 0, s>>>(pc, U, M, d[0], ctrl);
        for (size_t j = 0; j + 1 < d.size(); ++j) {
            const int nrb = std::min<int>(int(j) + 2, m);
            dim3 grid(nrb, (M + CBW - 1) / CBW);
            const float beta = j == 0 ? 1.f : 2.f, gamma = j == 0 ? 0.f : 1.f;
            k_cheb_bt_iter_df<<<grid, threads, smem, s>>>(hd, hs, ht, pp, pc, pn, U, M, ld, beta, gamma, d[j + 1], g,
                                                          ctrl);
            dfl *t = pp; pp = pc; pc = pn; pn = t;
        }
        KB_CUDA_TRY(cudaGetLastError());
        prof_end(KernelClass::PROJECTED, s, 0, 0, int(d.size()) + 2);
        return 0;
    }
    KB_CUDA_TRY(cudaMemsetAsync(V0, 0, bytes, s));
    KB_CUDA_TRY(cudaMemsetAsync(V1, 0, bytes, s));
    KB_CUDA_TRY(cudaMemsetAsync(V2, 0, bytes, s));
    zero_if_active(U, int64_t(m) * M * M, ctrl, s);
    k_cheb_bt_seed<<<(M + 127) / 128, 128, 0, s>>>(V0, U, M, d[0], ctrl);
    const size_t smem = sizeof(double) * 3 * M * TC;
    // function-local static: initialised once, thread-safe (several serving workers)
    static const cudaError_t attr = cudaFuncSetAttribute(
        k_cheb_bt_iter, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sizeof(double) * 3 * 128 * TC));
    (void)attr;
    double *pp = V2, *pc = V0, *pn = V1;
    const double g = 2.0 / lam;
    for (size_t j = 0; j + 1 < d.size(); ++j) {
        const int nrb = std::min<int>(int(j) + 2, m);
        dim3 grid(nrb, (M + TC - 1) / TC);
        const double beta = j == 0 ? 1.0 : 2.0, gamma = j == 0 ? 0.0 : 1.0;
        k_cheb_bt_iter<<<grid, 256, smem, s>>>(Hd, Hs, pp, pc, pn, U, M, beta, gamma, d[j + 1], g, ctrl);
        double *t = pp; pp = pc; pc = pn; pn = t;
    }
    KB_CUDA_TRY(cudaGetLastError());
    prof_end(KernelClass::PROJECTED, s, 0, 0, int(d.size()));
    return 0;
}

// Factors blocks r0 .. kmax - 1 (the ones before are known); returns the launch count.
static int bt_factor(const BtArgs &a, int r0, int kmax, double eps, const Ctrl *fc, cudaStream_t s) {
    const int M = a.M, lda = (M + 1) / 2 * 2;
    const size_t smem = sizeof(double) * (size_t(lda) * lda + sm::NB * sm::NB + sm::tri_tmp_elems(M));
    static const cudaError_t attr = cudaFuncSetAttribute(
        k_bt_dchol, cudaFuncAttributeMaxDynamicSharedMemorySize,
        int(sizeof(double) * (128 * 128 + sm::NB * sm::NB + sm::tri_tmp_elems(128))));
    (void)attr;
    int launches = 0;
    for (int r = r0; r < kmax; ++r) {
        // (a failed launch shows in the caller's cudaGetLastError)
        if (r > 0) (void)launch_dep(k_bt_ls, dim3(M), 128, 0, s, 0, a, r, fc);
        (void)launch_dep(k_bt_schur, dim3(M, r > 0 ? 2 : 1), 128, 0, s, 0, a, r, eps, fc);
        (void)launch_dep(k_bt_dchol, dim3(1), 512, smem, s, 0, a, r, fc);
        if (r > 0) (void)launch_dep(k_bt_gt, dim3(M), 128, 0, s, 0, a, r, fc);
        launches += r > 0 ? 4 : 2;
    }
    return launches;
}

int launch_bt_factor(const double *Hd, const double *Hs, int M, double eps, const SplineBufs &b, const Ctrl *fc,
                     cudaStream_t s, int r0, int kmax) {
    const BtArgs a{Hd, Hs, b.Ri, b.RiT, b.Y, b.GT, b.K, b.Ls, M};
    prof_begin(KernelClass::PROJECTED, s);
    const int launches = bt_factor(a, r0, kmax, eps, fc, s);
    KB_CUDA_TRY(cudaGetLastError());
    prof_end(KernelClass::PROJECTED, s, 0, 0, launches);
    return 0;
}

int launch_bt_spline(const double *Hd, const double *Hs, int M, int m, double eps, int s_int,
                     const SplineBufs &b, double *U, const Ctrl *fc, const Ctrl *ctrl, cudaStream_t s,
                     const QuadRule *q, double *qscr, int qbatch, int r0, int y0, int kmax) {
    if (kmax <= 0 || kmax > m) kmax = m;
    const BtArgs a{Hd, Hs, b.Ri, b.RiT, b.Y, b.GT, b.K, b.Ls, M};
    prof_begin(KernelClass::PROJECTED, s);
    int launches = 1;   // zero_if_active
    // (blocks past the steps stay zero: the bound check reads all m of them)
    zero_if_active(U, int64_t(m) * M * M, ctrl, s);
    const bool frac = q && q->n > 0;
    if (frac) {
        if (!qscr || qbatch < 1) return fail(KB_ERR_ARG, "spline quadrature without scratch");
        const int acc_grid = int(std::min<int64_t>((int64_t(m) * M * M + 255) / 256, 4 * int64_t(num_sms())));
        for (int j0 = 0; j0 < q->n; j0 += qbatch) {
            const int nb = std::min(qbatch, q->n - j0);
            k_bt_shift_solve<<<nb, QN_THREADS, 0, s>>>(Hd, Hs, M, m, *q, j0, qscr, ctrl);
            k_quad_accumulate<<<std::max(acc_grid, 1), 256, 0, s>>>(qscr, M, m, nb, *q, j0, U, ctrl);
            launches += 2;
        }
    }
    if (s_int > 0) {
        launches += bt_factor(a, r0, kmax, eps, fc, s) + 1;
        k_bt_subst<<<M, BTS_THREADS, 0, s>>>(a, s_int, y0, U, ctrl, frac ? 1 : 0);
    }
    KB_CUDA_TRY(cudaGetLastError());
    prof_end(KernelClass::PROJECTED, s, 0, 0, launches);
    return 0;
}

}  // namespace kb
