// Dispatch of the tall-skinny block kernels (rowblock.cuh) and the reduction of their Gram
// partials.
#include "rowblock.cuh"

#include <cstdlib>

namespace kb {
namespace rb {
// instantiated in rowblock_f32.cu, rowblock_f32_wide.cu, rowblock_f64.cu and rowblock_bf16.cu
#define KB_RB_EXT(T, W) extern template int launch_w<T, W>(int, const RowArgs<T> &, cudaStream_t, int *);
KB_RB_EXT(float, 16) KB_RB_EXT(float, 32) KB_RB_EXT(float, 64) KB_RB_EXT(float, 128)
KB_RB_EXT(double, 16) KB_RB_EXT(double, 32) KB_RB_EXT(double, 64)
KB_RB_EXT(__nv_bfloat16, 16) KB_RB_EXT(__nv_bfloat16, 32) KB_RB_EXT(__nv_bfloat16, 64) KB_RB_EXT(__nv_bfloat16, 128)
#undef KB_RB_EXT
// rowblock_ordered.cu
extern template int launch_ordered<16>(int, const RowArgs<float> &, cudaStream_t, int *);
extern template int launch_ordered<32>(int, const RowArgs<float> &, cudaStream_t, int *);
extern template int launch_ordered<64>(int, const RowArgs<float> &, cudaStream_t, int *);
extern template int launch_ordered<128>(int, const RowArgs<float> &, cudaStream_t, int *);
}  // namespace rb

namespace {

// ---------------------------------------------------------------- deterministic reduction
// The diagonal block H_kk = (G + G^T) / 2 of Algorithm 1, formed by the reduction's last CTA: Hd (M x
// M) and C (W x W, the small matrix of the update), rounded to the basis precision, exactly as
// the update subtracts it.  cnt: a counter that wraps to zero by itself.
template <typename P>
struct HkkOut {
    double *Hd = nullptr;
    P *C = nullptr;
    unsigned *cnt = nullptr;
    int M = 0, W = 0;
};

// out[e] = sum of the partials' entries e.  32 entries per CTA, its warps over the partials with
// RU loads in flight per lane (each into its own accumulator, merged in a fixed order), then a
// fixed-order combination of the warps' sums by warp 0.  FP32 partials are summed in
// double-float on the FP32 pipe.
template <typename P>
__global__ void __launch_bounds__(1024) k_reduce(const P *__restrict__ parts, int nparts, int len,
                                                  double *__restrict__ out, const Ctrl *ctrl,
                                                  P *__restrict__ out_p, const int32_t *skip, HkkOut<P> h) {
    pdl_wait();
    if ((ctrl && ctrl->stop) || (skip && *skip)) return;
    __shared__ double s[32][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int e = blockIdx.x * 32 + lane;
    if constexpr (std::is_same<P, float>::value) {
        // (two accumulators, each its own partials in rising order: the order of these sums is part
        // of the ordered form's fixed rounding)
        DF a0{0.f, 0.f}, a1{0.f, 0.f};
        if (e < len) {
            int p = warp;
            for (; p + 7 * nw < nparts; p += 8 * nw) {
                float v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = parts[int64_t(p + u * nw) * len + e];
#pragma unroll
                for (int u = 0; u < 8; u += 2) {
                    df_add(a0, v[u]);
                    df_add(a1, v[u + 1]);
                }
            }
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = p + u * nw < nparts ? parts[int64_t(p + u * nw) * len + e] : 0.f;
            // the last pair is taken together only when both exist; an odd one goes to a0
#pragma unroll
            for (int u = 0; u < 8; u += 2)
                if (p + u * nw < nparts) {
                    df_add(a0, v[u]);
                    if (p + (u + 1) * nw < nparts) df_add(a1, v[u + 1]);
                }
        }
        df_merge(a0, a1);
        reinterpret_cast<DF *>(&s[warp][0])[lane] = a0;
        __syncthreads();
        if (warp == 0 && e < len) {
            DF t = reinterpret_cast<const DF *>(&s[0][0])[lane];
            for (int w = 1; w < nw; ++w) df_merge(t, reinterpret_cast<const DF *>(&s[w][0])[lane]);
            const double v = df_value(t);
            out[e] = v;
            if (out_p) out_p[e] = P(v);
        }
    } else {
        double acc = 0.0;
        if (e < len)
            for (int p = warp; p < nparts; p += nw) acc += double(parts[int64_t(p) * len + e]);
        s[warp][lane] = acc;
        __syncthreads();
        if (warp == 0 && e < len) {
            double t = 0.0;
            for (int w = 0; w < nw; ++w) t += s[w][lane];
            out[e] = t;
            if (out_p) out_p[e] = P(t);
        }
    }
    pdl_trigger();
    if (h.cnt) {
        __shared__ unsigned last;
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) last = atomicInc(h.cnt, gridDim.x - 1);
        __syncthreads();
        if (last != gridDim.x - 1) return;
        __threadfence();
        for (int i = warp; i < h.W; i += nw)
            for (int j = lane; j < h.W; j += 32) {
                double v = 0.0;
                if (i < h.M && j < h.M) v = 0.5 * (__ldcg(out + i * h.W + j) + __ldcg(out + j * h.W + i));
                const P vt = P(v);
                if (i < h.M && j < h.M) h.Hd[i * h.M + j] = double(vt);
                h.C[i * h.W + j] = vt;
            }
    }
}

}  // namespace

// The tensor-core kernels are used when the environment variable KB_TENSOR_CORES is "1" at
// the start of a solve (RowArgs::tc).  They are not the default: with the frontier
// restriction most launches of a solve cover few tiles, and one 192 KB CTA per SM keeps other
// streams' kernels off the SM (measured slower in the multi-stream throughput run).
bool rowblock_tc_enabled() {
    const char *e = std::getenv("KB_TENSOR_CORES");
    return e && e[0] == '1';
}

template <typename T>
static int launch_simt(int mode, int W, const RowArgs<T> &a, cudaStream_t s, int *grid_out) {
    if constexpr (std::is_same<T, float>::value) {
        if (a.ordered && mode != RB_MUL && mode != RB_ASM) {
            switch (W) {
                case 16: return rb::launch_ordered<16>(mode, a, s, grid_out);
                case 32: return rb::launch_ordered<32>(mode, a, s, grid_out);
                case 64: return rb::launch_ordered<64>(mode, a, s, grid_out);
                default: return rb::launch_ordered<128>(mode, a, s, grid_out);
            }
        }
    }
    switch (W) {
        case 16: return rb::launch_w<T, 16>(mode, a, s, grid_out);
        case 32: return rb::launch_w<T, 32>(mode, a, s, grid_out);
        case 64: return rb::launch_w<T, 64>(mode, a, s, grid_out);
        case 128:
            if constexpr (sizeof(typename Cmp<T>::type) == 4) return rb::launch_w<T, 128>(mode, a, s, grid_out);
    }
    return fail(KB_ERR_ARG, "unsupported block width");
}

template <typename T>
int launch_rowblock(int mode, int W, const RowArgs<T> &a, cudaStream_t s, int *grid_out,
                    int64_t M_alg) {
    if (sizeof(typename Cmp<T>::type) == 8 && W > 64) return fail(KB_ERR_UNSUPPORTED, "FP64 blocks wider than 64");
    const int cls = mode == RB_ASM ? KernelClass::ASSEMBLE : KernelClass::ROWBLOCK;
    RowArgs<T> aa = a;
    aa.M = int(M_alg);
    aa.prof = prof_begin(cls, s);
    int rc = 0;
    bool tc = false;
    // (launches under a device skip flag take the SIMT kernels, which read the flag)
    if constexpr (std::is_same<T, float>::value)
        tc = a.tc && !a.skip && rowblock_tc_supported(mode, W);
    if (tc) {
        // FP32 blocks of width 64: tensor-core kernel (rowblock_tc.cu)
        if constexpr (std::is_same<T, float>::value) rc = launch_rowblock_tc(mode, aa, s, aa.max_grid, grid_out);
    } else {
        rc = launch_simt<T>(mode, W, aa, s, grid_out);
    }
    if (rc) return rc;
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return cuda_fail(err, tc ? "k_rowblock_tc launch" : "k_rowblock launch");
    const double blk = double(a.n) * double(M_alg) * sizeof(T);
    const double row = double(M_alg) * sizeof(T);             // bytes of one block row
    const double fr = 2.0 * double(M_alg) * double(M_alg);    // flops of one row times M x M
    double bytes = 0, flops = 0, per_row = 0, per_unit = 0, frow = 0, fixed = 0;
    const double mm = double(a.n) * fr;
    // algorithmic flops count the structure of the small matrices: a product with a
    // triangular factor (H_{k-1,k}, R^{-1}) is half of a general one, a Gram X^T X is
    // symmetric (half); the kernels compute little more (the blocks that meet the half, M rounded up to 4)
    switch (mode) {
        case RB_PROJ: bytes = 2 * blk; flops = mm; per_row = 2 * row; frow = fr; break;
        case RB_UPD:
            bytes = (a.qa ? 4 : 3) * blk; flops = (a.qa ? 2.0 : 1.5) * mm;
            per_row = (a.qa ? 4 : 3) * row; frow = (a.qa ? 2.0 : 1.5) * fr; break;
        case RB_MULGRAM: bytes = 2 * blk; flops = mm; per_row = 2 * row; frow = fr; break;
        case RB_MUL: bytes = 2 * blk; flops = 0.5 * mm; per_row = 2 * row; frow = 0.5 * fr; break;
        case RB_ASM:
            // block rows read (counted per tile and block) + the FP32 output written in full
            bytes = (a.nblk + 1) * blk; flops = a.nblk * mm;
            per_unit = row; fixed = double(a.n) * double(M_alg) * 4.0; break;
        case RB_ASMSUB:
            bytes = (a.nblk + 2) * blk; flops = a.nblk * mm + mm;
            per_row = 2 * row; per_unit = row; frow = fr; break;
    }
    prof_end(cls, s, bytes, flops, 1, per_row, per_unit, frow, fixed);
    return 0;
}

template <typename T>
int rowblock_max_grid(int W, int M, int64_t n, bool ordered, bool tc) {
    int most = 0;
    for (const int mode : {RB_PROJ, RB_UPD, RB_MULGRAM, RB_ASMSUB}) {
        RowArgs<T> a;
        a.n = n;
        a.M = M;
        a.ordered = ordered ? 1 : 0;
        a.plan = 1;
        int grid = 0;
        if (launch_simt<T>(mode, W, a, nullptr, &grid) == 0) most = std::max(most, grid);
    }
    if constexpr (std::is_same<T, float>::value) {
        if (tc && rowblock_tc_supported(RB_PROJ, W)) most = std::max(most, rowblock_tc_max_grid());
    }
    return most;
}

template <typename P>
static int reduce_impl(const P *parts, int nparts, int len, double *out, cudaStream_t s, const Ctrl *ctrl, P *out_p,
                       const int32_t *skip, const HkkOut<P> &h) {
    prof_begin(KernelClass::REDUCE, s);
    const cudaError_t err = launch_dep(k_reduce<P>, dim3((len + 31) / 32), 1024, 0, s, 0, parts, nparts, len, out, ctrl,
                                       out_p, skip, h);
    if (err != cudaSuccess) return cuda_fail(err, "k_reduce launch");
    prof_end(KernelClass::REDUCE, s, double(nparts) * len * sizeof(P), 0);
    return 0;
}

template <typename P>
int launch_reduce(const P *parts, int nparts, int len, double *out, cudaStream_t s,
                  const Ctrl *ctrl, P *out_p, const int32_t *skip) {
    return reduce_impl<P>(parts, nparts, len, out, s, ctrl, out_p, skip, HkkOut<P>{});
}

template <typename P>
int launch_reduce_hkk(const P *parts, int nparts, int M, int W, double *G, double *Hd, P *C, unsigned *cnt,
                      const Ctrl *ctrl, cudaStream_t s) {
    HkkOut<P> h;
    h.Hd = Hd;
    h.C = C;
    h.cnt = cnt;
    h.M = M;
    h.W = W;
    return reduce_impl<P>(parts, nparts, W * W, G, s, ctrl, nullptr, nullptr, h);
}

template int launch_reduce_hkk<float>(const float *, int, int, int, double *, double *, float *, unsigned *,
                                      const Ctrl *, cudaStream_t);
template int launch_reduce_hkk<double>(const double *, int, int, int, double *, double *, double *, unsigned *,
                                       const Ctrl *, cudaStream_t);
template int launch_rowblock<float>(int, int, const RowArgs<float> &, cudaStream_t, int *, int64_t);
template int launch_rowblock<double>(int, int, const RowArgs<double> &, cudaStream_t, int *, int64_t);
template int rowblock_max_grid<float>(int, int, int64_t, bool, bool);
template int rowblock_max_grid<double>(int, int, int64_t, bool, bool);
template int launch_rowblock<__nv_bfloat16>(int, int, const RowArgs<__nv_bfloat16> &, cudaStream_t, int *, int64_t);
template int rowblock_max_grid<__nv_bfloat16>(int, int, int64_t, bool, bool);
template int launch_reduce<float>(const float *, int, int, double *, cudaStream_t, const Ctrl *, float *,
                                  const int32_t *);
template int launch_reduce<double>(const double *, int, int, double *, cudaStream_t, const Ctrl *, double *,
                                   const int32_t *);

}  // namespace kb
