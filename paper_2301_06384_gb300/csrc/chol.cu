// Small dense kernel of the classical block Lanczos step (Algorithm 1).
//
//  * k_chol  reduced QR of the new block by CholeskyQR: Cholesky factor (FP32 first, FP64
//            fallback), its inverse and the FP64 factor consistent with the applied inverse;
//            the second pass forms H_{k+1,k} = R2 R1 and the transposed block used by the next
//            three-term step (H_{k-1,k} = H_{k,k-1}^T).  Invariant subspaces stop the
//            process, rank-deficient blocks report a breakdown (the paper assumes full rank).
#include "kb_internal.cuh"
#include "kb_kernels.cuh"
#include "smallmat.cuh"

namespace kb {

// Reduced QR of the new block by CholeskyQR (Algorithm 1), pass 1 or 2 of CholeskyQR2.
// Outputs: Rinv (W x W, basis precision) applied by the row-block kernels; pass 1 records
// R1 = the FP64 inverse of the applied inverse; pass 2 records H_{k+1,k} = R2 R1 (rounded to
// the basis precision) and B = H^T.
//
// Pass 1 of the FP32 path (G = X^T X, any conditioning) factors G in FP32: it only has to
// bring X close to orthonormal, the second pass corrects what is left, and R1 is the inverse
// of the applied FP32 inverse S whatever R it came from.  M <= 64: with S R = I - E,
// S^{-1} = R (I - E)^{-1} = R + R E + R E^2 + O(E^3), E (of the order of the FP32 rounding)
// from a residual in pairs of floats, the corrections in FP32 (relative error of R1 1e-14 to
// 4e-14, below the FP32 rounding of H by six orders).  M > 64: S is inverted in FP64 (2e-16 to
// 7e-16; the corrected form reaches 1e-13 there).  A pivot below 1e-5 of the largest diagonal
// entry, or max |E_ij| >= 1e-3, is not trusted in FP32: the factorisation is then done in FP64
// (which alone decides a breakdown) and S is inverted in FP64.
// Pass 2 of the FP32 path (G = I + E, ||E|| of the order of the FP32 rounding of pass 1): to
// first order R2 = I + Phi(E) with Phi = strict upper part plus half the diagonal,
// R2^{-1} = I - Phi(E) (the orthogonality of Q = X1 (I - Phi(E)) is then I + O(||E||^2)); the
// applied inverse I - F has the inverse I + F + F^2 + O(F^3), so H = R1 + F R1 + F (F R1), the
// corrections formed in FP32.  When max |E_ij| >= 1e-4, and always in the FP64 mode, pass 2
// takes the general path.
//
// Bound: latency of one CTA (smallmat.cuh).  Per launch, FP32, pass 1 and
// pass 2 (us, launch list): 31 / 15 at M = 40, 17 / 9 at M = 16; with one barrier per column
// and 4 x 4 tiles on few threads 69 / 19 and 43 / 11.  FP64, M = 33: 58 / 49, before 112 / 90.  (Pivot
// reciprocals rounded to nearest add 1 us to pass 1 at M = 16, 3 us at M = 64.)
constexpr int CHOL_THREADS = 512;
constexpr int CORRECTED_MAX = 64;   // widest block whose R1 is the corrected FP32 factor

struct CholLayout {
    // byte offsets of the dynamic shared memory: three FP32 matrices (general FP32 path), or one
    // FP64 matrix and a second region (FP64 factorisation and FP64 mode)
    size_t mat32, dbl, second, scr, total;
    int lda;
};
template <typename T>
__host__ __device__ inline CholLayout chol_layout(int M) {
    CholLayout l;
    l.lda = (M + 1) / 2 * 2;
    const size_t e = size_t(l.lda) * ((M + 1) / 2 * 2);
    l.mat32 = e * sizeof(float);
    l.dbl = 0;
    l.second = e * sizeof(double);
    // second: the FP64 inverse and its scratch (T = double); the FP32 inverse and its scratch,
    // then the scratch of the FP64 inversion of that (FP32 path)
    const size_t tmp = size_t(sm::tri_tmp_elems(M)) * sizeof(T);
    const size_t sec = e * sizeof(T) + tmp;   // (>= 2 tmp)
    const size_t a = 3 * l.mat32 + size_t(sm::tri_tmp_elems(M)) * sizeof(float), b = l.second + sec;
    l.scr = ((sizeof(T) == 4 && a > b ? a : b) + 15) & ~size_t(15);
    l.total = l.scr + sm::NB * sm::NB * sizeof(double);
    return l;
}

template <typename T>
__global__ void __launch_bounds__(CHOL_THREADS) k_chol(const double *G, int M, int W, int pass, int step,
                                              double inv_thresh2, double piv_rel2, double *R1,
                                              T *Rinv, double *Hs, T *Bout, Ctrl *ctrl) {
    pdl_wait();
    if (ctrl->stop) return;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int bad, small;
    __shared__ double maxdiag;
    __shared__ unsigned int emax_bits;
    __shared__ double s_diag[128];
    const CholLayout L = chol_layout<T>(M);
    const int lda = L.lda;
    float *F0 = reinterpret_cast<float *>(smem);                     // FP32 path: G, then R
    float *F1 = reinterpret_cast<float *>(smem + L.mat32);           // S
    float *F2 = reinterpret_cast<float *>(smem + 2 * L.mat32);       // E
    float *Ft = reinterpret_cast<float *>(smem + 3 * L.mat32);       // merge scratch
    double *A = reinterpret_cast<double *>(smem);                    // FP64 factorisation
    double *scr = reinterpret_cast<double *>(smem + L.scr);
    constexpr bool FP32 = sizeof(T) == 4;
    auto none = [](int, int) { return 0; };
    const bool try_small = pass == 2 && FP32;
    // pass 1 in FP32: S is inverted in FP64 (its copy in the second region is at F2)
    bool inverted = FP32 && pass == 1 && M > CORRECTED_MAX;
    if (threadIdx.x == 0) {
        emax_bits = 0u;
        bad = 0;
    }
    __syncthreads();
    // FP32 path: pass 1 keeps G in FP32, pass 2 keeps E = G - I; FP64 mode: G
    unsigned my_e = 0u;   // bits of max |E_ij| (the order of non-negative floats; a NaN stays)
    sm::load_square(G, W, M, [&](int i, int j, double g) {
        if (i == j) s_diag[i] = g;
        if (FP32) {
            const float e = try_small ? float(i == j ? g - 1.0 : g) : float(g);
            F0[i * lda + j] = e;
            my_e = max(my_e, __float_as_uint(fabsf(e)));
        } else {
            A[i * lda + j] = g;
        }
    });
    if (try_small) {
        const unsigned b = __reduce_max_sync(0xffffffffu, my_e);
        if ((threadIdx.x & 31) == 0) atomicMax(&emax_bits, b);
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        // trace and largest diagonal entry
        double tr = 0.0, mx = 0.0;
        for (int i = threadIdx.x; i < M; i += 32) {
            tr += s_diag[i];
            mx = fmax(mx, fabs(s_diag[i]));
        }
        for (int off = 16; off > 0; off >>= 1) {
            tr += __shfl_xor_sync(0xffffffffu, tr, off);
            mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, off));
        }
        if (threadIdx.x == 0) {
            maxdiag = mx;
            small = (try_small && __uint_as_float(emax_bits) < 1e-4f) ? 1 : 0;
            emax_bits = 0u;
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
    if constexpr (FP32) {
        if (small) {
            // ---- pass 2, first order: S = I - Phi(E) applied; F = I - S exactly.  E is in F0,
            // R1 goes to F1, F to F2, then C = F R1 over E.
            sm::each(W, W, [&](int i, int j) {
                float v = 0.f;
                if (i < M && j < M && j >= i) {
                    const float e = F0[i * lda + j];
                    v = i == j ? 1.f - 0.5f * e : -e;
                }
                Rinv[i * W + j] = v;
                if (i < M && j < M) F2[i * lda + j] = j >= i ? (i == j ? 1.f : 0.f) - v : 0.f;
                // entries outside H's upper triangle are zero
                if (!(i < M && j < M && j >= i)) {
                    if (i < M && j < M) Hs[i * M + j] = 0.0;
                    Bout[j * W + i] = 0.f;
                }
            });
            sm::load_square(R1, M, M, [&](int i, int j, double v) { F1[i * lda + j] = j >= i ? float(v) : 0.f; });
            __syncthreads();
            sm::each(M, M, [&](int i, int j) {
                if (j < i) F0[i * lda + j] = 0.f;
            });
            sm::tri_mm(F2, F1, lda, M, none, [&](int i, int j, float c, int) { F0[i * lda + j] = c; });
            __syncthreads();
            pdl_trigger();   // (not earlier: the next kernel's CTAs would hold their SMs meanwhile)
            // H = (I + F + F^2) R1 = R1 + (C + F C), the corrections of relative size ||E||
            sm::tri_mm(F2, F0, lda, M, [&](int i, int j) { return __ldcg(R1 + i * M + j); },
                       [&](int i, int j, float c2, double r1) {
                const double h = r1 + double(F0[i * lda + j] + c2);
                const float ht = float(h);
                Hs[i * M + j] = double(ht);
                Bout[j * W + i] = ht;
            });
            return;
        }
        if (pass == 1) {
            // ---- FP32 factor, its inverse and the FP64 inverse of that
            sm::each(M, M, [&](int i, int j) { F1[i * lda + j] = 0.f; });
            __syncthreads();
            if (sm::chol_blocked<float>(F0, F1, lda, M, 1e-5f * float(maxdiag), reinterpret_cast<float *>(scr))) {
                // S starts as the inverted diagonal blocks and R's entries above them
                sm::each(M, M, [&](int i, int j) {
                    if (j < i) F0[i * lda + j] = 0.f;
                    else if (i / sm::NB != j / sm::NB) F1[i * lda + j] = F0[i * lda + j];
                });
                __syncthreads();
                sm::tri_inv_merge<float>(F1, lda, M, Ft);
                sm::each(W, W, [&](int i, int j) {
                    const bool in = i < M && j < M;
                    const float v = in && j >= i ? F1[i * lda + j] : 0.f;
                    Rinv[i * W + j] = v;
                    if (in && (inverted || j < i)) F2[i * lda + j] = v;   // (S, or E's zeros below the diagonal)
                });
                if (!inverted) {
                    unsigned my = 0u;
                    sm::tri_residual(F1, F0, lda, M, [&](int i, int j, float e) {
                        F2[i * lda + j] = e;
                        my = max(my, __float_as_uint(fabsf(e)));
                    });
                    atomicMax(&emax_bits, my);
                    __syncthreads();
                    if (__uint_as_float(emax_bits) < 1e-3f) {
                        // C1 = R E over S (zeros below the diagonal), then R1 = R + (C1 + C1 E)
                        sm::tri_mm(F0, F2, lda, M, none, [&](int i, int j, float c, int) { F1[i * lda + j] = c; });
                        __syncthreads();
                        pdl_trigger();
                        sm::tri_mm(F1, F2, lda, M, none, [&](int i, int j, float c2, int) {
                            R1[i * M + j] = double(F0[i * lda + j]) + double(F1[i * lda + j] + c2);
                        });
                        sm::each(M, M, [&](int i, int j) {
                            if (j < i) R1[i * M + j] = 0.0;
                        });
                        return;
                    }
                }
            } else {
                inverted = false;
            }
            __syncthreads();
        }
        if (!inverted) {
            // ---- FP64 factorisation (from G again)
            sm::load_square(G, W, M, [&](int i, int j, double g) { A[i * lda + j] = g; });
            __syncthreads();
        }
    }
    T *B = reinterpret_cast<T *>(smem + L.second);   // the applied inverse
    T *Bt = B + size_t(lda) * ((M + 1) / 2 * 2);     // scratch of its merge levels
    bool ok;
    if constexpr (FP32) {
        ok = inverted || sm::chol_blocked<double>(A, nullptr, lda, M, piv_rel2 * maxdiag, scr);
    } else {
        sm::each(M, M, [&](int i, int j) { B[i * lda + j] = 0.0; });
        __syncthreads();
        ok = sm::chol_blocked<double>(A, B, lda, M, piv_rel2 * maxdiag, scr);
    }
    if (!ok) {
        if (threadIdx.x == 0) {
            ctrl->status = KB_ERR_BREAKDOWN;
            ctrl->stop = 1;
            ctrl->steps = step;
            ctrl->breakdown_step = step;
        }
        return;
    }
    if constexpr (FP32) {
        // S = the FP32 inverse of the rounded factor; A = the FP64 inverse of S
        if (!inverted) {
            sm::each(M, M, [&](int i, int j) { B[i * lda + j] = j >= i ? float(A[i * lda + j]) : 0.f; });
            __syncthreads();
            sm::tri_inv_diag<float>(B, lda, M);
            sm::tri_inv_merge<float>(B, lda, M, Bt);
            sm::each(W, W, [&](int i, int j) {
                Rinv[i * W + j] = i < M && j < M && j >= i ? B[i * lda + j] : 0.f;
            });
        }
        sm::each(M, M, [&](int i, int j) { A[i * lda + j] = j >= i ? double(B[i * lda + j]) : 0.0; });
        __syncthreads();
        sm::tri_inv_diag<double>(A, lda, M);
        sm::tri_inv_merge<double>(A, lda, M, reinterpret_cast<double *>(smem + L.second));
    } else {
        sm::each(M, M, [&](int i, int j) {
            if (j < i) A[i * lda + j] = 0.0;
            else if (i / sm::NB != j / sm::NB) B[i * lda + j] = A[i * lda + j];
        });
        __syncthreads();
        sm::tri_inv_merge<T>(B, lda, M, Bt);
        sm::each(W, W, [&](int i, int j) { Rinv[i * W + j] = (i < M && j < M && j >= i) ? B[i * lda + j] : T(0); });
    }
    pdl_trigger();
    // A: the upper triangular R whose inverse is applied (FP64)
    if (pass == 1) {
        sm::each(M, M, [&](int i, int j) { R1[i * M + j] = j >= i ? A[i * lda + j] : 0.0; });
    } else {
        // H_{k+1,k} = R2 R1 (upper triangular); B = H^T for the next three-term step.  H is
        // recorded rounded to the basis precision, i.e. exactly as the next step subtracts it.
        sm::each(W, W, [&](int i, int j) {
            if (i < M && j < M && j >= i) return;
            if (i < M && j < M) Hs[i * M + j] = 0.0;
            Bout[j * W + i] = T(0);
        });
        __syncthreads();
        // R1 over the second region where it fits beside A (FP64 mode; FP32 up to M = 8, whose second
        // region is sized for floats), else over the product's own loads from global memory
        double *R = reinterpret_cast<double *>(smem + L.second);
        if (L.second + size_t(lda) * ((M + 1) / 2 * 2) * sizeof(double) <= L.scr) {
            sm::load_square(R1, M, M, [&](int i, int j, double v) { R[i * lda + j] = j >= i ? v : 0.0; });
            __syncthreads();
            sm::tri_mm<double>(A, R, lda, M, none, [&](int i, int j, double h, int) {
                const T ht = T(h);
                Hs[i * M + j] = double(ht);
                Bout[j * W + i] = ht;
            });
        } else {
            sm::tri_tiles<1, true>(M, [&](int i, int j) {
                double h = 0.0;
#pragma unroll 8
                for (int k = i; k <= j; ++k) h = fma(A[i * lda + k], __ldcg(R1 + k * M + j), h);
                const T ht = T(h);
                Hs[i * M + j] = double(ht);
                Bout[j * W + i] = ht;
            });
        }
    }
}

// ---------------------------------------------------------------- launchers
template <typename T>
int launch_chol(const double *G, int M, int W, int pass, int step, double inv_thresh2,
                double piv_rel2, double *R1, T *Rinv, double *Hs, T *Bout, Ctrl *ctrl,
                cudaStream_t s) {
    const size_t smem = chol_layout<T>(M).total;
    // FP64 blocks are at most 64 wide; function-local static: set once, thread-safe
    static const cudaError_t attr = cudaFuncSetAttribute(
        k_chol<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(chol_layout<T>(sizeof(T) == 8 ? 64 : 128).total));
    (void)attr;
    prof_begin(KernelClass::SMALL, s);
    KB_CUDA_TRY(launch_dep(k_chol<T>, dim3(1), CHOL_THREADS, smem, s, 0, G, M, W, pass, step, inv_thresh2, piv_rel2, R1,
                           Rinv, Hs, Bout, ctrl));
    prof_end(KernelClass::SMALL, s, 0, 0);
    return 0;
}

#define KB_INST(T)                                                                              \
    template int launch_chol<T>(const double *, int, int, int, int, double, double, double *,   \
                                T *, double *, T *, Ctrl *, cudaStream_t);
KB_INST(float)
KB_INST(double)
#undef KB_INST

}  // namespace kb
