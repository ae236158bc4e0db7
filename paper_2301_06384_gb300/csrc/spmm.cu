// Block SpMM with the Laplacian: out = epilogue(L x), x an n x W row-major block.
//
// This is the "MV" of Table 1 (Section 7), the operation the paper names the most
// expensive for large graphs; every method performs m of them per solve.
//
// Schedule (GB300).  A row of x is W elements; W/8 lanes cover it with two 16-byte vectors
// each (float4, or 2 x double2), so a warp takes 32/(W/8) rows at once, one lane group per
// row: a warp's unit of work, all in one 32-row frontier tile.  Warps walk their units
// independently (no barrier, no shared staging) over the active-tile list, or over all rows
// without one.  Row pointers come one unit ahead; the lanes of a group load a chunk of the
// row's neighbour indices with one coalesced load and pass them round by shuffles; U rows are
// gathered with independent 16-byte loads before they are used.  Rows beyond the frontier
// inside an active tile are written as zeros without their gathers.  Bound by the latency
// and the L2 bandwidth of the gathers.  Against CTA tiles with row pointers and indices staged
// in shared memory (three barriers per tile) and 32-row units that left half of the warps idle
// at W = 32: RGG of 2e4 rows, M = 37, 30 products 447 -> 345 us.
//
// Long rows (hubs).  A lane group's row is a serial chain of one gather latency per U neighbours,
// and its warp waits for it.  Rows above long_row_degree are therefore listed at graph creation and
// taken first, a CTA each: its 256 / LPR lane groups share the row's neighbours, and the partial
// sums meet by shuffles and in shared memory in a fixed order.  Preferential attachment (5 edges a
// node, 4e5 rows, rows up to some 3000 long), 10 products, ms: M = 16 7.1 -> 1.0, M = 64 12.7 -> 2.5,
// with column dots 10.9 -> 4.3; the tiles with staged indices took 6.4, 9.0 and 12.0.  A star of
// 3e4 rows, M = 16: 40 -> 0.5.  A warp per long row was slower (M = 64 7.9, with dots 11.4).
//
// The Laplacian is applied in difference form (L x)_i = sum_j w_ij (x_i - x_j) + r_i x_i,
// which gives L 1 = 0 exactly for D - A and drops the diagonal load for standard
// Laplacians.  Epilogue coefficients arrive in FP64; in the FP32 path each is split into
// a float pair (hi + lo) so that c * (L x) carries only the rounding of the final sum.
#include <algorithm>
#include <type_traits>

#include "kb_internal.cuh"

namespace kb {
namespace {

// Raw: the values as loaded.  Gathers stay in that form until they are used: BF16 rows widened at
// once take twice the registers, and a load's conversion waits for it before the next is issued (RGG
// of 3e5 rows, M = 128, 20 products 2.78 -> 1.39 ms; random graph of mean degree 100, 5e4 rows, M = 64, 10
// products 1.26 -> 0.81 ms).
template <typename T> struct V4;
template <> struct V4<float> {
    float v[4];
    using Raw = V4;
    __device__ __forceinline__ static Raw load_raw(const float *p) { return load(p); }
    __device__ __forceinline__ static V4 widen(const Raw &r) { return r; }
    __device__ __forceinline__ static V4 load(const float *p) {
        float4 t = __ldg(reinterpret_cast<const float4 *>(p));
        return V4{{t.x, t.y, t.z, t.w}};
    }
    __device__ __forceinline__ void store(float *p) const {
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    }
};
template <> struct V4<__nv_bfloat16> {
    // four BF16 values (8 bytes) widened to FP32
    float v[4];
    using Raw = uint2;
    __device__ __forceinline__ static Raw load_raw(const __nv_bfloat16 *p) {
        return __ldg(reinterpret_cast<const uint2 *>(p));
    }
    __device__ __forceinline__ static V4 load(const __nv_bfloat16 *p) { return widen(load_raw(p)); }
    __device__ __forceinline__ static V4 widen(const Raw &raw) {
        const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw.x));
        const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw.y));
        return V4{{a.x, a.y, b.x, b.y}};
    }
    __device__ __forceinline__ void store(__nv_bfloat16 *p) const {
        const __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]);
        const __nv_bfloat162 b = __floats2bfloat162_rn(v[2], v[3]);
        uint2 raw;
        raw.x = *reinterpret_cast<const unsigned int *>(&a);
        raw.y = *reinterpret_cast<const unsigned int *>(&b);
        *reinterpret_cast<uint2 *>(p) = raw;
    }
};
template <> struct V4<double> {
    double v[4];
    using Raw = V4;
    __device__ __forceinline__ static Raw load_raw(const double *p) { return load(p); }
    __device__ __forceinline__ static V4 widen(const Raw &r) { return r; }
    __device__ __forceinline__ static V4 load(const double *p) {
        double2 a = __ldg(reinterpret_cast<const double2 *>(p));
        double2 b = __ldg(reinterpret_cast<const double2 *>(p + 2));
        return V4{{a.x, a.y, b.x, b.y}};
    }
    __device__ __forceinline__ void store(double *p) const {
        reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
        reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
    }
};

constexpr int SPMM_THREADS = 256;
constexpr int WARPS = SPMM_THREADS / 32;
constexpr int VPL = 2;          // 16-byte vectors per lane (8 elements of a row)
constexpr int U = 4;            // neighbour rows gathered per lane before use

template <int W>
struct SpmmGeo {
    static constexpr int LPR = W / (4 * VPL);   // lanes per row
    static constexpr int RPW = 32 / LPR;        // rows of a warp's unit of work
    static constexpr int UPT = ACT_ROWS / RPW;  // units of a 32-row tile
};

// Packed FP32 pairs (Blackwell add/sub/fma.rn.f32x2): each lane of the pair is rounded as
// the scalar instruction would round it, so the packed neighbour loop gives bit-identical
// sums with half the floating-point instructions.
using f2 = unsigned long long;
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
    f2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f2 f2_pack(float lo, float hi) {
    f2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ void f2_unpack(f2 v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
// 16 bytes of a read-only FP32 row as two packed pairs
__device__ __forceinline__ void ldg_f2x2(const float *p, f2 &a, f2 &b) {
    asm("ld.global.nc.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p));
}

// Four consecutive coefficients from shared memory in one 16-byte (FP32) or two 16-byte
// (FP64) loads; c is a multiple of 4 and the arrays are 16-byte aligned.
template <typename C>
__device__ __forceinline__ void lds4(const C *p, C (&v)[4]) {
    if constexpr (sizeof(C) == 4) {
        const float4 t = *reinterpret_cast<const float4 *>(p);
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else {
        const double2 a = reinterpret_cast<const double2 *>(p)[0];
        const double2 b = reinterpret_cast<const double2 *>(p)[1];
        v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    }
}

// Resident CTAs per SM the register budget is sized for.  Measured, RGG of 10^6 rows, M = 64,
// 30 products (ms), four / three / five CTAs: without column dots 1.58 / 1.66 / 1.87; with
// them (8 more accumulators) 3.62 / 3.45.  Two or eight gathers in flight instead of U = 4:
// 1.74 / 1.78 and 4.10 / 3.89.
template <typename T, bool DOT>
struct SpmmOcc {
    static constexpr int value = sizeof(typename Cmp<T>::type) == 8 ? 3 : (DOT ? 3 : 4);
};

// WGT: the graph stores edge weights (false: unit weights, w_ij = 1).  LONG: the graph has long
// rows (a variant of its own: graphs without them keep the registers of the loop over units).
template <typename T, int W, bool DOT, bool WGT, bool LONG>
__global__ void __launch_bounds__(SPMM_THREADS, (SpmmOcc<T, DOT>::value))
k_spmm(GraphDev g, const T *__restrict__ x, LinEpi<T> e, int64_t ldo, int mo, int mcols) {
    using G = SpmmGeo<W>;
    using C = typename Cmp<T>::type;   // arithmetic type
    constexpr int LPR = G::LPR, RPW = G::RPW, UPT = G::UPT;
    constexpr int CPL = LPR >= 8 ? 1 : 8 / LPR;   // neighbour indices a lane loads at once
    constexpr int CHUNK = LPR * CPL;
    pdl_wait();
    if (e.ctrl && e.ctrl->stop) return;
    __shared__ __align__(16) C s_coef[5][W];       // c1 hi, c1 lo, c0, c2 hi, c2 lo
    __shared__ C s_sc[2];                          // s3, wE in the arithmetic type
    __shared__ double s_dot[DOT ? WARPS : 1][W];
    __shared__ C s_part[LONG ? WARPS : 1][LONG ? W : 1];   // sums of a long row, by warp
    if (threadIdx.x == 0) {
        s_sc[0] = C(e.s3);
        s_sc[1] = C(e.wE);
    }
    for (int c = threadIdx.x; c < W; c += blockDim.x) {
        const double d1 = e.a1 ? e.a1[c] : e.s1;
        const double d2 = e.a2 ? e.a2[c] : e.s2;
        const C h1 = C(d1), h2 = C(d2);
        s_coef[0][c] = h1;
        s_coef[1][c] = C(d1 - double(h1));
        s_coef[2][c] = C(e.a0 ? e.a0[c] : e.s0);
        s_coef[3][c] = h2;
        s_coef[4][c] = C(d2 - double(h2));
    }
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int grp = lane / LPR;
    // columns of this lane: 4 consecutive columns in each of VPL slices of 4 * LPR columns,
    // so that one 16-byte load instruction of a lane group reads one contiguous 4 * LPR
    // column span (whole 32-byte sectors) of the gathered row
    const int sub = lane % LPR;
#define KB_COL(v) (((v) * LPR + sub) * 4)
    // columns past the block's M hold zeros in every operand: neither gathered nor read
    bool cin[VPL];
#pragma unroll
    for (int v = 0; v < VPL; ++v) cin[v] = KB_COL(v) < mcols;
    C dot[VPL][4];
#pragma unroll
    for (int v = 0; v < VPL; ++v)
#pragma unroll
        for (int q = 0; q < 4; ++q) dot[v][q] = C(0);
    unsigned my_rows = 0, my_nnz = 0;
    // a unit of work is RPW rows of a 32-row tile, one warp's; tiles past `active` (beyond the
    // frontier limit) are only written, with zeros, where the launch asks for it
    const int64_t nt = (g.n + ACT_ROWS - 1) / ACT_ROWS;
    const int64_t active = e.tgen ? int64_t(*e.acount) : nt;
    const int64_t nunits = (e.tgen && !e.zero_inactive ? active : nt) * UPT;
    const int64_t step = int64_t(gridDim.x) * WARPS;
    __syncthreads();
    // row, its reach flag and its neighbour range for unit `w` (w < nunits)
    auto row_of = [&](int64_t w) -> int64_t {
        const int64_t t = w / UPT;
        return (e.tgen ? int64_t(__ldg(e.alist + t)) : t) * ACT_ROWS + (w % UPT) * RPW + grp;
    };
    // The rows come one unit ahead (list entry, hop distance, row pointers), so that a unit's
    // chain of dependent loads is only neighbour indices -> gathered rows.
    int64_t row = -1;
    int beg = 0, end = 0;
    bool act = false;
    auto fetch = [&](int64_t w, int64_t &r, int &b, int &en, bool &on) {
        r = -1;
        b = en = 0;
        on = false;
        if (w >= nunits) return;
        r = row_of(w);
        if (r >= g.n) {
            r = -1;
            return;
        }
        on = w / UPT < active && (!e.tgen || int(__ldg(e.gen + r)) <= e.limit);
        b = __ldg(g.rowptr + r);
        en = __ldg(g.rowptr + r + 1);
        if (LONG && on && en - b > g.long_row) {
            r = -1;   // (done by a CTA)
            on = false;
        }
    };
    const int64_t w0 = int64_t(blockIdx.x) * WARPS + warp;
    fetch(w0, row, beg, end, act);
    int64_t lnext = blockIdx.x;   // (of the long rows; uniform in the CTA)
    for (int64_t w = w0; w < nunits || (LONG && lnext < g.nlong); w += step) {
        int64_t nrow;
        int nbeg, nend;
        bool nact;
        V4<T> xi[VPL];
        typename V4<T>::Raw xr[VPL];   // (as loaded)
        C acc[VPL][4];
        if (LONG && lnext < g.nlong) {
            // a long row, by all lane groups of the CTA: each takes U neighbours in turn; the unit waits
            nrow = row;
            nbeg = beg;
            nend = end;
            nact = act;
            w -= step;
            row = __ldg(g.longs + lnext);
            lnext += gridDim.x;
            act = !e.tgen || int(__ldg(e.gen + row)) <= e.limit;   // (else its unit writes the zeros)
            const int lbeg = __ldg(g.rowptr + row), deg = act ? __ldg(g.rowptr + row + 1) - lbeg : 0;
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
                xr[v] = act && cin[v] ? V4<T>::load_raw(x + row * W + KB_COL(v)) : typename V4<T>::Raw{};
                xi[v] = V4<T>::widen(xr[v]);
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[v][q] = C(0);
            }
            for (int p0 = (warp * RPW + grp) * U; p0 < deg; p0 += WARPS * RPW * U) {
                typename V4<T>::Raw xj[U][VPL];
                C wv[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const bool in = p0 + u < deg;
                    const int j = in ? __ldg(g.col + lbeg + p0 + u) : 0;
                    wv[u] = WGT && in ? C(__ldg(g.w + lbeg + p0 + u)) : C(1);
#pragma unroll
                    for (int v = 0; v < VPL; ++v)
                        xj[u][v] = in && cin[v] ? V4<T>::load_raw(x + int64_t(j) * W + KB_COL(v)) : xr[v];
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int v = 0; v < VPL; ++v) {
                        const V4<T> xw = V4<T>::widen(xj[u][v]);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const C d = xi[v].v[q] - xw.v[q];
                            acc[v][q] = WGT ? fma(wv[u], d, acc[v][q]) : acc[v][q] + d;
                        }
                    }
            }
            __syncthreads();   // (the sums of the row before are read)
#pragma unroll
            for (int v = 0; v < VPL; ++v)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
#pragma unroll
                    for (int off = LPR; off < 32; off <<= 1) acc[v][q] += __shfl_xor_sync(0xffffffffu, acc[v][q], off);
                    if (grp == 0) s_part[warp][KB_COL(v) + q] = acc[v][q];
                }
            __syncthreads();
            // the first group finishes the row
            if (warp != 0 || grp != 0 || !act) {
                row = -1;
            } else {
#pragma unroll
                for (int v = 0; v < VPL; ++v)
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        for (int w2 = 1; w2 < WARPS; ++w2) acc[v][q] += s_part[w2][KB_COL(v) + q];
                if (sub == 0) {
                    ++my_rows;
                    my_nnz += unsigned(deg);
                }
            }
        } else {
            fetch(w + step, nrow, nbeg, nend, nact);
            const int deg = act ? end - beg : 0;
            if (sub == 0 && act) {
                ++my_rows;
                my_nnz += unsigned(deg);
            }
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
                xr[v] = act && cin[v] ? V4<T>::load_raw(x + row * W + KB_COL(v)) : typename V4<T>::Raw{};
                xi[v] = V4<T>::widen(xr[v]);
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[v][q] = C(0);
            }
            // neighbours: the lanes of a group load the indices (and weights) of a chunk of 8 or
            // LPR; the group then takes them in order by shuffles.  The loop runs to the longest row of the
            // warp; slots past a row's end contribute x_i - x_i, an exact zero.
            const int maxdeg = __reduce_max_sync(0xffffffffu, deg);
            for (int p0 = 0; p0 < maxdeg; p0 += CHUNK) {
                int mj[CPL];
                float mw[CPL];
#pragma unroll
                for (int q = 0; q < CPL; ++q) {
                    const int p = p0 + q * LPR + sub;
                    mj[q] = p < deg ? __ldg(g.col + beg + p) : 0;
                    if (WGT) mw[q] = p < deg ? __ldg(g.w + beg + p) : 0.f;
                }
#pragma unroll
                for (int u0 = 0; u0 < CHUNK; u0 += U) {
                    if (p0 + u0 >= maxdeg) break;
                    if constexpr (std::is_same<T, float>::value) {
                        f2 xj[U][VPL][2], xi2[VPL][2];
                        f2 wv[U];
#pragma unroll
                        for (int v = 0; v < VPL; ++v) {
                            xi2[v][0] = f2_pack(xi[v].v[0], xi[v].v[1]);
                            xi2[v][1] = f2_pack(xi[v].v[2], xi[v].v[3]);
                        }
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            const int j = __shfl_sync(0xffffffffu, mj[(u0 + u) / LPR], (u0 + u) % LPR, LPR);
                            if (WGT) {
                                const float wj = __shfl_sync(0xffffffffu, mw[(u0 + u) / LPR], (u0 + u) % LPR, LPR);
                                wv[u] = f2_pack(wj, wj);
                            }
                            const bool in = p0 + u0 + u < deg;
                            const float *xr = reinterpret_cast<const float *>(x) + int64_t(j) * W;
#pragma unroll
                            for (int v = 0; v < VPL; ++v) {
                                xj[u][v][0] = xi2[v][0];
                                xj[u][v][1] = xi2[v][1];
                                if (in && cin[v]) ldg_f2x2(xr + KB_COL(v), xj[u][v][0], xj[u][v][1]);
                            }
                        }
#pragma unroll
                        for (int v = 0; v < VPL; ++v) {
                            f2 a0 = f2_pack(acc[v][0], acc[v][1]), a1 = f2_pack(acc[v][2], acc[v][3]);
#pragma unroll
                            for (int u = 0; u < U; ++u) {
                                const f2 d0 = f2_sub(xi2[v][0], xj[u][v][0]), d1 = f2_sub(xi2[v][1], xj[u][v][1]);
                                a0 = WGT ? f2_fma(wv[u], d0, a0) : f2_add(a0, d0);
                                a1 = WGT ? f2_fma(wv[u], d1, a1) : f2_add(a1, d1);
                            }
                            f2_unpack(a0, acc[v][0], acc[v][1]);
                            f2_unpack(a1, acc[v][2], acc[v][3]);
                        }
                    } else {
                        typename V4<T>::Raw xj[U][VPL];
                        C wv[U];
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            const int j = __shfl_sync(0xffffffffu, mj[(u0 + u) / LPR], (u0 + u) % LPR, LPR);
                            wv[u] = WGT ? C(__shfl_sync(0xffffffffu, mw[(u0 + u) / LPR], (u0 + u) % LPR, LPR)) : C(1);
                            const bool in = p0 + u0 + u < deg;
#pragma unroll
                            for (int v = 0; v < VPL; ++v)
                                xj[u][v] = in && cin[v] ? V4<T>::load_raw(x + int64_t(j) * W + KB_COL(v)) : xr[v];
                        }
#pragma unroll
                        for (int u = 0; u < U; ++u)
#pragma unroll
                            for (int v = 0; v < VPL; ++v) {
                                const V4<T> xw = V4<T>::widen(xj[u][v]);
#pragma unroll
                                for (int q = 0; q < 4; ++q) {
                                    const C d = xi[v].v[q] - xw.v[q];
                                    acc[v][q] = WGT ? fma(wv[u], d, acc[v][q]) : acc[v][q] + d;
                                }
                            }
                    }
                }
            }
        }
        if (row >= 0) {
            const C r = g.rdiag && act ? C(__ldg(g.rdiag + row)) : C(0);
            const int mk = e.marker && act ? __ldg(e.marker + row) : -1;
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
                const int c = KB_COL(v);
                C o[4] = {0, 0, 0, 0};
                if (act && cin[v]) {
                    C k1h[4], k1l[4], k0[4];
                    lds4(&s_coef[0][c], k1h);
                    lds4(&s_coef[1][c], k1l);
                    lds4(&s_coef[2][c], k0);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const C a = fma(r, xi[v].v[q], acc[v][q]);
                        o[q] = fma(k1h[q], a, fma(k1l[q], a, k0[q] * xi[v].v[q]));
                    }
                    if (e.y) {
                        const V4<T> yi = V4<T>::load(e.y + row * W + c);
                        C k2h[4], k2l[4];
                        lds4(&s_coef[3][c], k2h);
                        lds4(&s_coef[4][c], k2l);
#pragma unroll
                        for (int q = 0; q < 4; ++q) o[q] = fma(k2h[q], yi.v[q], fma(k2l[q], yi.v[q], o[q]));
                    }
                    if (e.z) {
                        const V4<T> zi = V4<T>::load(e.z + row * W + c);
#pragma unroll
                        for (int q = 0; q < 4; ++q) o[q] = fma(s_sc[0], zi.v[q], o[q]);
                    }
                    // (constant indices: a computed index would put o in local memory)
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (mk == c + q) o[q] += s_sc[1];
                }
                if (!e.yout) {
                    // narrowed blocks: the dot below is that of the stored values
                    if constexpr (!std::is_same<T, C>::value) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) o[q] = C(T(o[q]));
                    }
                    V4<T> ov;
#pragma unroll
                    for (int q = 0; q < 4; ++q) ov.v[q] = o[q];
                    ov.store(e.out + row * W + c);
                } else {
                    float *y = e.yout + row * ldo + c;
                    if (c + 3 < mo && ((ldo & 3) == 0) && (reinterpret_cast<uintptr_t>(y) & 15) == 0) {
                        *reinterpret_cast<float4 *>(y) = make_float4(float(o[0]), float(o[1]), float(o[2]), float(o[3]));
                    } else {
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            if (c + q < mo) y[q] = float(o[q]);
                    }
                }
                if (DOT) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) dot[v][q] = fma(xi[v].v[q], o[q], dot[v][q]);
                }
            }
        }
        row = nrow;
        beg = nbeg;
        end = nend;
        act = nact;
    }
    pdl_trigger();
    if (e.prof.rows && my_rows) {
        atomicAdd(e.prof.rows, (unsigned long long)my_rows);
        atomicAdd(e.prof.nnz, (unsigned long long)my_nnz);
    }
    if constexpr (DOT && std::is_same<C, float>::value) {
        // double-float combination on the FP32 pipe; partials written as DF pairs
        DF *sd = reinterpret_cast<DF *>(&s_dot[0][0]);
#pragma unroll
        for (int v = 0; v < VPL; ++v)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                DF d{dot[v][q], 0.f};
#pragma unroll
                for (int off = LPR; off < 32; off <<= 1) {
                    const DF o{__shfl_xor_sync(0xffffffffu, d.hi, off), __shfl_xor_sync(0xffffffffu, d.lo, off)};
                    df_merge(d, o);
                }
                if (grp == 0) sd[warp * W + KB_COL(v) + q] = d;
            }
        __syncthreads();
        DF *out = reinterpret_cast<DF *>(e.dot_partials);
        for (int c = threadIdx.x; c < W; c += blockDim.x) {
            DF s = sd[c];
            for (int w2 = 1; w2 < WARPS; ++w2) df_merge(s, sd[w2 * W + c]);
            out[int64_t(blockIdx.x) * W + c] = s;
        }
    } else if constexpr (DOT) {
#pragma unroll
        for (int v = 0; v < VPL; ++v)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                double dd = double(dot[v][q]);
#pragma unroll
                for (int off = LPR; off < 32; off <<= 1) dd += __shfl_xor_sync(0xffffffffu, dd, off);
                if (grp == 0) s_dot[warp][KB_COL(v) + q] = dd;
            }
        __syncthreads();
        for (int c = threadIdx.x; c < W; c += blockDim.x) {
            double s = 0.0;
            for (int w2 = 0; w2 < WARPS; ++w2) s += s_dot[w2][c];
            e.dot_partials[int64_t(blockIdx.x) * W + c] = s;
        }
    }
}

#undef KB_COL

template <typename T, int W, bool DOT, bool LONG>
int occupancy_spmm() {
    // the weighted and unweighted kernels share the launch bounds
    // function-local static: computed once, thread-safe (several serving workers)
    static const int per_sm = [] {
        int v = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_spmm<T, W, DOT, true, LONG>, SPMM_THREADS, 0);
        return v < 1 ? 1 : v;
    }();
    return per_sm;
}

template <typename T, int W, bool DOT, bool LONG>
int launch_wd(const GraphDev &g, const T *x, const LinEpi<T> &e, int64_t ldo, int mo, int mcols,
              cudaStream_t s, int *grid_out) {
    const int64_t units = (g.n + SpmmGeo<W>::RPW - 1) / SpmmGeo<W>::RPW;
    int grid = int(std::min<int64_t>((units + WARPS - 1) / WARPS, int64_t(num_sms()) * occupancy_spmm<T, W, DOT, LONG>()));
    if (grid < 1) grid = 1;
    if (grid_out) *grid_out = grid;
    const cudaError_t err =
        launch_dep(g.w ? k_spmm<T, W, DOT, true, LONG> : k_spmm<T, W, DOT, false, LONG>, dim3(grid), SPMM_THREADS, 0, s, 0,
                   g, x, e, ldo, mo, mcols);
    return err == cudaSuccess ? 0 : cuda_fail(err, "k_spmm launch");
}

template <typename T, int W>
int launch_w(const GraphDev &g, const T *x, const LinEpi<T> &e, int64_t ldo, int mo, int mcols,
             cudaStream_t s, int *grid_out) {
    if (g.nlong && !e.one_group)
        return e.dot_partials ? launch_wd<T, W, true, true>(g, x, e, ldo, mo, mcols, s, grid_out)
                              : launch_wd<T, W, false, true>(g, x, e, ldo, mo, mcols, s, grid_out);
    return e.dot_partials ? launch_wd<T, W, true, false>(g, x, e, ldo, mo, mcols, s, grid_out)
                          : launch_wd<T, W, false, false>(g, x, e, ldo, mo, mcols, s, grid_out);
}

// CTAs per SM of the kernels that write dot partials
template <typename T, int W>
int max_occupancy() {
    return std::max(occupancy_spmm<T, W, true, false>(), occupancy_spmm<T, W, true, true>());
}

}  // namespace

// The line between the two.  A CTA spends about as long on any long row of less than some 500
// entries, so they have to be few: at most one row in 64, and longer than four mean rows (with every
// row of mean degree 100 taken by a CTA, 5e4 rows, M = 24: 1.70 ms for 10 products, 0.63 by units; one
// row in 20 of 105 entries, 4e5 rows, column dots, M = 24: 2.54 and 2.30).  Between 64 and 256 as the
// smallest length, preferential attachment of 4e5 rows, M = 64: 2.52 at 64, 2.65 at 128, 3.03 at 256;
// at 32 2.77.
int32_t long_row_degree(const int32_t *rowptr, int64_t n, std::vector<int32_t> *rows) {
    int64_t t = std::max<int64_t>(64, 4 * int64_t(rowptr[n]) / n);
    rows->clear();
    for (int64_t i = 0; i < n; ++i)
        if (rowptr[i + 1] - rowptr[i] > t) rows->push_back(int32_t(i));
    while (int64_t(rows->size()) > std::max<int64_t>(1, n / 64)) {
        t *= 2;
        rows->erase(std::remove_if(rows->begin(), rows->end(), [&](int32_t i) { return rowptr[i + 1] - rowptr[i] <= t; }),
                    rows->end());
    }
    return int32_t(std::min<int64_t>(t, INT32_MAX));
}

template <typename T>
int launch_spmm(const GraphDev &g, int W, const T *x, const LinEpi<T> &e, cudaStream_t s,
                int *grid_out, int64_t M_alg, int n_dense_in, int64_t ldo, int mo) {
    if (ldo <= 0) { ldo = W; mo = W; }
    LinEpi<T> ee = e;
    ee.prof = prof_begin(KernelClass::SPMM, s);
    const int mcols = int(M_alg);
    int rc = 0;
    switch (W) {
        case 16: rc = launch_w<T, 16>(g, x, ee, ldo, mo, mcols, s, grid_out); break;
        case 32: rc = launch_w<T, 32>(g, x, ee, ldo, mo, mcols, s, grid_out); break;
        case 64: rc = launch_w<T, 64>(g, x, ee, ldo, mo, mcols, s, grid_out); break;
        case 128: rc = launch_w<T, 128>(g, x, ee, ldo, mo, mcols, s, grid_out); break;
        default: return fail(KB_ERR_ARG, "unsupported block width");
    }
    if (rc) return rc;
    // algorithmic bytes: CSR (+weights, +diagonal excess) once, the gathered block once,
    // the other dense inputs once each, the output once; flops 3 per nonzero per column
    double csr = 4.0 * double(g.n + 1) + 4.0 * double(g.nnz) + (g.w ? 4.0 * double(g.nnz) : 0.0) +
                 (g.rdiag ? 4.0 * double(g.n) : 0.0);
    double blk = double(g.n) * double(M_alg) * double(sizeof(T));
    // per processed row: its row pointer (+ diagonal excess), the gathered block counted
    // once, the other dense inputs and the output; per stored nonzero: index (+ weight)
    const double per_row = 4.0 + (g.rdiag ? 4.0 : 0.0) +
                           double(M_alg) * double(sizeof(T)) * (2 + n_dense_in);
    const double per_nnz = 4.0 + (g.w ? 4.0 : 0.0);
    const double flops_per_row = 3.0 * double(M_alg) * double(g.nnz) / double(g.n);
    prof_end(KernelClass::SPMM, s, csr + blk * (2 + n_dense_in), 3.0 * double(g.nnz) * double(M_alg),
             1, per_row, per_nnz, flops_per_row, 4.0);
    return 0;
}

template <typename T>
int spmm_max_grid(int W) {
    // dot partials are written only by the DOT variant; its grid bounds the buffer
    switch (W) {
        case 16: return num_sms() * max_occupancy<T, 16>();
        case 32: return num_sms() * max_occupancy<T, 32>();
        case 64: return num_sms() * max_occupancy<T, 64>();
        default: return num_sms() * max_occupancy<T, 128>();
    }
}

template int launch_spmm<float>(const GraphDev &, int, const float *, const LinEpi<float> &,
                                cudaStream_t, int *, int64_t, int, int64_t, int);
template int launch_spmm<double>(const GraphDev &, int, const double *, const LinEpi<double> &,
                                 cudaStream_t, int *, int64_t, int, int64_t, int);
template int launch_spmm<__nv_bfloat16>(const GraphDev &, int, const __nv_bfloat16 *,
                                        const LinEpi<__nv_bfloat16> &, cudaStream_t, int *, int64_t,
                                        int, int64_t, int);
template int spmm_max_grid<float>(int);
template int spmm_max_grid<double>(int);
template int spmm_max_grid<__nv_bfloat16>(int);

}  // namespace kb
