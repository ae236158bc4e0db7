// Tall-skinny block kernels of the classical block Lanczos step (Algorithm 1: diagonal
// block, three-term update, reduced QR) and of its final assembly: products of n x W blocks
// with W x W matrices and Gram matrices A^T B of n x W blocks.  Included by one translation
// unit per stored type.
//
// Rows.  The unit of rows is the 32-row frontier tile.  A CTA works on virtual tiles of TR
// rows, TR / 32 consecutive entries of the active-tile list (or consecutive tiles of the
// matrix without one), so every row of a virtual tile is an active one wherever it lies.  An
// operand block that is zero in a sub-tile (its hop distance exceeds the block's reach) is
// filled with zeros on the way to shared memory and never read from HBM.
//
// Columns.  Everything is sized by M rounded up to 4 and not by the width W of the layout:
// CG = ceil(M / 4) column groups of 4, RG row groups of RPT rows, CG * RG <= 256 threads.
// FP64 solves (bound by the FP64 pipe) and ragged widths do no arithmetic on padding.
//
// Product.  The operand's columns come in chunks of 64 bytes per row, with the matching rows
// of the small matrix, through a ring of cp.async stages that runs on across virtual tiles:
// one barrier per chunk, and loads of the next chunks are in flight during the arithmetic,
// the epilogue and the Gram sums.  A thread owns RPT rows x 4 columns.  Chunks that meet the
// zero half of a triangular factor are skipped by warps, and the warps' columns are permuted
// so that the skips fall evenly on the SM's four schedulers.
//
// Gram.  The 8 x 4 (8 x 8 at W = 128) blocks of G are spread over the threads, as many row
// groups as fit in 256 threads; X^T X takes only the blocks meeting the upper triangle.
// FP32 sums have two levels (at most about 64 rows, then across tiles); the row groups are
// combined in a fixed order at the end, one partial G per CTA, summed by k_reduce.
//
// Ordered form (ORD; FP32 solves with full reorthogonalisation).  Full reorthogonalisation is
// asked for where the result is sensitive to the rounding of the basis: with the spline kernel
// on hub graphs (BA, 5e5 rows, (0.1 I + L)^{-2}) another order of the Gram sums, no less
// accurate, moves single entries of Y by 10^-3 to 10^-2 of their root mean square.  Such
// solves keep one order of every FP32 sum: the rows of a tile of 4096 / W one after the other
// (one row group), a CTA's tiles by rising index from the step's list in index order, a fixed
// number of CTAs per SM.  (Products have no freedom: a chain over k per entry.)
//
// Bound, W >= 64: latency between a stage's arrival, its shared loads and the FMAs that depend on
// them at 16 warps per SM (M = 64: FMA pipe 47 to 58 % busy, no pipe saturated); 8 x 4 register tiles take 12 16-byte
// loads of 4 wavefronts per 128 FMAs.  HBM below; the FP64 pipe in FP64.
//
// CTAs per SM, from the shared memory that the geometry takes: two of 256 threads at M = 37..64 and 121..128, one
// at M = 33..36 (tiles of 224 rows) and 65..120 (two to five Gram row groups beside the tile); whole cbl
// solves there, RGG of 3e5 rows, 12 steps, before -> now: M = 33 3.46 -> 1.87 ms, 72 11.2 -> 5.1, 112 17.1 -> 10.2.
//
// Measured (launch list, mean us of a solve's launches; before: synchronous staging, 4 x 4
// tiles, all W columns, full Grams):                          PROJ     UPD  MULGRAM     MUL
//   RGG 10^6 rows, M = 64, 30 steps, before                   68.3   170.9    100.0    56.3
//                                    now                      38.0    90.6     53.5    32.9
//   128^3 grid, M = 32, 40 steps,    before                  242.8   451.8    291.6   155.8
//                                    now                      65.4   137.2     79.1    53.1
//   BA 5e5 rows, M = 128, ordered,   before                  280.8  1675.7    962.6   665.5
//                                    now, whole solve 243 -> 172 ms
//   RGG 10^5 rows, M = 33, FP64,     before                  477.6  1193.7    743.4   305.1
//                                    now                     104.3   234.1    136.7    67.4
// With scalar FMAs, list lookups and 64-bit addresses per copy, and the first level of the Gram
// sums held across the products, UPD at M = 64 took 113.4.
#pragma once
#include <algorithm>
#include <atomic>
#include <climits>
#include <type_traits>

#include "kb_internal.cuh"

namespace kb {
namespace rb {

constexpr int NST = 3;   // cp.async stages

template <typename C>
__device__ __forceinline__ void ld4(const C *p, C (&v)[4]) {
    if constexpr (sizeof(C) == 4) {
        const float4 t = *reinterpret_cast<const float4 *>(p);
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else {
        const double2 a = reinterpret_cast<const double2 *>(p)[0];
        const double2 b = reinterpret_cast<const double2 *>(p)[1];
        v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    }
}
// N consecutive elements (N = 1, 2 or a multiple of 4)
template <typename C, int N>
__device__ __forceinline__ void ldn(const C *p, C (&v)[N]) {
    if constexpr (N % 4 == 0) {
#pragma unroll
        for (int u = 0; u < N; u += 4) {
            C t[4];
            ld4<C>(p + u, t);
#pragma unroll
            for (int w = 0; w < 4; ++w) v[u + w] = t[w];
        }
    } else {
#pragma unroll
        for (int u = 0; u < N; ++u) v[u] = p[u];
    }
}
template <typename C>
__device__ __forceinline__ void st4(C *p, const C (&v)[4]) {
    if constexpr (sizeof(C) == 4) {
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
        reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
        reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
    }
}
// Global block access: load 4 stored elements widened to the compute type, store narrowed.
template <typename T>
__device__ __forceinline__ void ldg4(const T *p, typename Cmp<T>::type (&v)[4]) {
    if constexpr (std::is_same<T, __nv_bfloat16>::value) {
        const uint2 raw = *reinterpret_cast<const uint2 *>(p);
        const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw.x));
        const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw.y));
        v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    } else {
        ld4<T>(p, v);
    }
}
template <typename T>
__device__ __forceinline__ void stg4(T *p, const typename Cmp<T>::type (&v)[4]) {
    if constexpr (std::is_same<T, __nv_bfloat16>::value) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]);
        const __nv_bfloat162 b = __floats2bfloat162_rn(v[2], v[3]);
        uint2 raw;
        raw.x = *reinterpret_cast<const unsigned int *>(&a);
        raw.y = *reinterpret_cast<const unsigned int *>(&b);
        *reinterpret_cast<uint2 *>(p) = raw;
    } else {
        st4<T>(p, v);
    }
}
// Packed FP32 pairs (fma.rn.f32x2): each lane rounds as the scalar instruction would, at half
// the issue slots; these kernels are bound by those (65 % of them busy with scalar FMAs).
using f2 = unsigned long long;
__device__ __forceinline__ f2 f2_pack(float lo, float hi) {
    f2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
// c[i] += a b[i] over N (even) consecutive entries
template <typename C, int N>
__device__ __forceinline__ void fma_row(C (&c)[N], C a, const C (&b)[N]) {
    if constexpr (sizeof(C) == 4 && N % 2 == 0) {
        const f2 aa = f2_pack(a, a);
#pragma unroll
        for (int i = 0; i < N; i += 2) {
            const f2 t = f2_fma(aa, f2_pack(b[i], b[i + 1]), f2_pack(c[i], c[i + 1]));
            asm("mov.b64 {%0, %1}, %2;" : "=f"(c[i]), "=f"(c[i + 1]) : "l"(t));
        }
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) c[i] = fma(a, b[i], c[i]);
    }
}
// 16 bytes global -> shared, asynchronous; zeros when !in (the address is then not read)
__device__ __forceinline__ void cp16(void *dst, const void *src, bool in) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <typename T, int W, bool ORD = false>
struct Geo {
    using C = typename Cmp<T>::type;
    static constexpr int VEC = 16 / int(sizeof(C));
    static constexpr int KC = 64 / int(sizeof(C));        // columns of a product chunk (64 bytes)
    // row strides shifted by 16 bytes: eight consecutive rows hit all 32 banks
    static constexpr int LDA = KC + VEC;
    static constexpr int LDO = W + VEC;
    static constexpr bool TWO = sizeof(C) == 4;           // two-level Gram sums
    static constexpr bool G2S = W == 128;                 // second level in shared memory
    static constexpr int BI = ORD ? W / 16 : 8, BJ = ORD ? W / 16 : G2S ? 8 : 4;   // Gram block of a thread
    static constexpr int TO = 4096 / W;                   // ORD: rows of a tile
    static constexpr int SO = W == 128 ? 2 : 1;           // ORD: such tiles of a virtual tile
    static constexpr int CTAS = W >= 128 ? 2 : W >= 32 ? 4 : 3;   // ORD: CTAs per SM
    static constexpr int PR = 2048 / W;                   // rows of a PROJ chunk
};

// Runtime geometry of a launch, the same on host and device.
struct RowGeo {
    int Mk, CG, RG, TR;      // columns in use (multiple of 4), column groups, row groups, rows
    int NI, NJ, NB, NGR;     // Gram blocks along i and j, their number, row groups of the Gram
};
template <typename T, int W, int MODE, int RPT, bool ORD, int NT>
__host__ __device__ inline RowGeo row_geo(int M) {
    using G = Geo<T, W, ORD>;
    RowGeo r;
    r.Mk = (M + 3) / 4 * 4;
    r.CG = r.Mk / 4;
    const int cap = NT == 128 ? 128 : 256;   // rows: bounds the shared memory of narrow blocks
    int tr = (NT / r.CG) * RPT;
    tr = (tr < cap ? tr : cap) / 32 * 32;
    r.TR = tr < 32 ? 32 : tr;
    if (ORD) r.TR = G::TO * G::SO;
    r.RG = r.TR / RPT;
    r.NI = (M + G::BI - 1) / G::BI;
    r.NJ = (M + G::BJ - 1) / G::BJ;
    if (MODE == RB_PROJ) r.NB = r.NI * r.NJ;
    else if (G::BJ == G::BI) r.NB = r.NI * (r.NI + 1) / 2;
    else {
        // blocks (bi, bj) with bj >= 2 bi
        r.NB = 0;
        for (int b = 0; b < r.NI; ++b) r.NB += r.NJ - 2 * b;
    }
    r.NGR = NT / r.NB;
    if (ORD || r.NGR < 1) r.NGR = 1;
    return r;
}
template <typename T, int W, int MODE>
__host__ __device__ inline size_t stage_elems(const RowGeo &r) {
    using G = Geo<T, W>;
    if (MODE == RB_PROJ) return size_t(2) * G::PR * W;
    return size_t(r.TR) * G::LDA + size_t(G::KC) * W;
}
template <typename T, int W, int MODE, bool ORD>
inline size_t smem_bytes(const RowGeo &r) {
    using G = Geo<T, W, ORD>;
    using C = typename G::C;
    const bool gram = MODE == RB_PROJ || MODE == RB_UPD || MODE == RB_MULGRAM || MODE == RB_ASMSUB;
    size_t e = NST * stage_elems<T, W, MODE>(r);
    if (MODE != RB_PROJ) e += size_t(r.TR) * G::LDO;
    // final combination of the Gram row groups (reuses the stages and the output tile) and,
    // at W = 128, the second-level sums
    const size_t comb = gram ? size_t(r.NGR) * r.NB * G::BI * G::BJ : 0;
    if (gram && G::G2S) e += comb;
    else e = std::max(e, comb);
    return e * sizeof(C);
}

template <typename T, int W, int MODE, int RPT, bool ORD, int NT>
__global__ void __launch_bounds__(NT, sizeof(typename Cmp<T>::type) == 8 ? 1 : 512 / NT)
k_rowblock(RowArgs<T> a) {
    using G = Geo<T, W, ORD>;
    using C = typename G::C;
    constexpr bool PROD = MODE != RB_PROJ;
    constexpr bool GRAM = MODE == RB_PROJ || MODE == RB_UPD || MODE == RB_MULGRAM || MODE == RB_ASMSUB;
    constexpr bool SUBX = MODE == RB_UPD || MODE == RB_ASMSUB;     // out = X - product
    constexpr bool MULTI = MODE == RB_ASM || MODE == RB_ASMSUB;    // product over basis blocks
    constexpr bool ASYNC_X = SUBX && std::is_same<T, typename G::C>::value;   // X comes by cp.async
    constexpr int BI = G::BI, BJ = G::BJ, KC = G::KC, LDA = G::LDA, LDO = G::LDO, VEC = G::VEC;
    pdl_wait();
    if (MODE != RB_ASM && a.ctrl && a.ctrl->stop) return;
    if (a.skip && *a.skip) return;

    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *sm = reinterpret_cast<C *>(smem_raw);
    const RowGeo q = row_geo<T, W, MODE, RPT, ORD, NT>(a.M);
    const int SE = int(stage_elems<T, W, MODE>(q));
    C *sO = sm + NST * SE;                                          // [TR][LDO]
    C *sG = PROD ? sO + q.TR * LDO : sO;                            // [NGR * NB][BI * BJ] (W = 128)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t nt = (a.n + ACT_ROWS - 1) / ACT_ROWS;             // frontier tiles of the matrix
    // (ASM writes all of y; a launch that adds to it only the tiles that its block reaches)
    const int64_t cnt = a.alist && (MODE != RB_ASM || a.accumulate) ? int64_t(*a.acount) : nt;
    auto tile_at = [&](int64_t i) -> int64_t {
        return i >= cnt ? -1 : (a.alist ? int64_t(__ldg(a.alist + i)) : i);
    };

    // Ordered form: positions of the step's list (or tiles of TO rows without one); a tile of
    // several listed frontier tiles is taken at the first of them.
    constexpr int AO = ORD ? G::TO / ACT_ROWS : 1;
    const int64_t olen = ORD ? (a.alist ? int64_t(*a.acount) : (a.n + G::TO - 1) / G::TO) : 0;
    auto otile = [&](int64_t i) -> int64_t {
        return i >= olen ? -1 : (a.alist ? int64_t(__ldg(a.alist + i)) / AO : i);
    };
    auto onorm = [&](int64_t i) -> int64_t {
        if (AO > 1 && a.alist)
            while (i < olen && i > 0 && otile(i - 1) == otile(i)) i += gridDim.x;
        return i;
    };

    // ---- Gram state
    const bool glive = GRAM && tid < q.NB * q.NGR;
    int gi0 = 0, gj0 = 0, grp = 0;
    C g1[GRAM ? BI : 1][GRAM ? BJ : 1], g2[(GRAM && !G::G2S) ? BI : 1][(GRAM && !G::G2S) ? BJ : 1];
    C *gown = nullptr;
    int grows = 0;    // rows since the last flush of the first level
    if constexpr (GRAM) {
        if (glive) {
            grp = tid / q.NB;
            int b = tid % q.NB, bi = 0;
            if (MODE == RB_PROJ) {
                bi = b / q.NJ;
                b = b % q.NJ;
            } else {
                constexpr int S = BI / BJ;   // first block column of row bi is S * bi
                while (b >= q.NJ - S * bi) {
                    b -= q.NJ - S * bi;
                    ++bi;
                }
                b += S * bi;
            }
            gi0 = bi * BI;
            gj0 = b * BJ;
        }
        if constexpr (G::G2S) {
            gown = sG + tid;   // entry e of this thread at stride NB * NGR
            if (glive)
                for (int e = 0; e < BI * BJ; ++e) gown[e * q.NB * q.NGR] = C(0);
        }
#pragma unroll
        for (int i = 0; i < BI; ++i)
#pragma unroll
            for (int j = 0; j < BJ; ++j) {
                g1[i][j] = 0;
                if constexpr (!G::G2S) g2[i][j] = 0;
            }
    }
    auto flush = [&]() {
        if constexpr (GRAM) {
#pragma unroll
            for (int i = 0; i < BI; ++i)
#pragma unroll
                for (int j = 0; j < BJ; ++j) {
                    if constexpr (G::G2S) {
                        if (glive) gown[(i * BJ + j) * q.NB * q.NGR] += g1[i][j];
                    } else {
                        g2[i][j] += g1[i][j];
                    }
                    g1[i][j] = 0;
                }
            grows = 0;
        }
    };
    // G += left^T right over R rows (this thread's block and row group)
    auto gram_rows = [&](const C *left, const C *right, int ld, int R) {
        if constexpr (GRAM) {
            if (glive) {
#pragma unroll 2
                for (int r = grp; r < R; r += q.NGR) {
                    C av[BI], bv[BJ];
                    ldn<C, BI>(left + r * ld + gi0, av);
                    ldn<C, BJ>(right + r * ld + gj0, bv);
#pragma unroll
                    for (int i = 0; i < BI; ++i) {
                        if constexpr (G::TWO) fma_row<C, BJ>(g1[i], av[i], bv);
                        else fma_row<C, BJ>(g2[i], av[i], bv);
                    }
                }
            }
            if constexpr (G::TWO && !ORD) {
                // (a product's tile ends the first level, which then takes no registers beside the
                // product's)
                grows += R / q.NGR;
                if (PROD || grows >= 32) flush();
            }
        }
    };
    unsigned long long my_rows = 0, my_units = 0;

    if constexpr (!PROD) {
        // ---------------------------------------------------------------- PROJ: G = Qa^T X
        constexpr int PR = G::PR;
        constexpr int EPC = PR >= ACT_ROWS ? PR / ACT_ROWS : 1;    // list entries of a chunk
        constexpr int CPE = PR < ACT_ROWS ? ACT_ROWS / PR : 1;     // chunks of a list entry
        const int64_t nch = PR >= ACT_ROWS ? (cnt + EPC - 1) / EPC : cnt * CPE;
        auto issue = [&](int64_t ch, int st) {
            if (ch < nch) {
                C *dx = sm + st * SE, *dq = dx + PR * W;
                constexpr int EPV = std::is_same<T, C>::value ? VEC : 4;   // elements of a copy
                for (int i = tid; i < PR * W / EPV; i += NT) {
                    const int r = i / (W / EPV), c = (i % (W / EPV)) * EPV;
                    if (c >= q.Mk) continue;   // (columns past M are not read by the sums)
                    const int64_t t = PR >= ACT_ROWS ? tile_at(ch * EPC + r / ACT_ROWS) : tile_at(ch / CPE);
                    const int64_t row = t * ACT_ROWS + (PR >= ACT_ROWS ? r % ACT_ROWS : int(ch % CPE) * PR + r);
                    const bool in = t >= 0 && row < a.n;
                    const int64_t off = in ? row * W + c : 0;
                    if constexpr (std::is_same<T, C>::value) {
                        cp16(dx + r * W + c, a.x + off, in);
                        cp16(dq + r * W + c, a.qa + off, in);
                    } else {
                        C v[4] = {0, 0, 0, 0}, w[4] = {0, 0, 0, 0};
                        if (in) {
                            ldg4<T>(a.x + off, v);
                            ldg4<T>(a.qa + off, w);
                        }
                        st4<C>(dx + r * W + c, v);
                        st4<C>(dq + r * W + c, w);
                    }
                }
            }
            cp_commit();
        };
        // columns Mk .. roundup(M, 8) are read by the blocks at the edge: zero them once
        for (int i = tid; i < NST * 2 * PR * (W - q.Mk); i += NT) {
            const int c = q.Mk + i % (W - q.Mk), r = i / (W - q.Mk);
            sm[r * W + c] = C(0);
        }
        int st = 0;
        if constexpr (ORD) {
            // the two chunks of each tile, one flush per tile
            int64_t pvt = onorm(blockIdx.x);
            int ph = 0;
            auto issue_o = [&](int s) {
                if (pvt < olen) {
                    C *dx = sm + s * SE, *dq = dx + PR * W;
                    const int64_t r0 = otile(pvt) * G::TO + ph * PR;
                    for (int i = tid; i < PR * W / VEC; i += NT) {
                        const int r = i / (W / VEC), c = (i % (W / VEC)) * VEC;
                        if (c >= q.Mk) continue;
                        const bool in = r0 + r < a.n;
                        const int64_t off = in ? (r0 + r) * W + c : 0;
                        cp16(dx + r * W + c, a.x + off, in);
                        cp16(dq + r * W + c, a.qa + off, in);
                    }
                    ph ^= 1;
                    if (ph == 0) pvt = onorm(pvt + gridDim.x);
                }
                cp_commit();
            };
            for (int s = 0; s < NST - 1; ++s) issue_o(s);
            for (int64_t vt = onorm(blockIdx.x); vt < olen; vt = onorm(vt + gridDim.x)) {
                for (int h = 0; h < G::TO / PR; ++h) {
                    cp_wait<NST - 2>();
                    __syncthreads();
                    issue_o(st == 0 ? NST - 1 : st - 1);
                    const C *dx = sm + st * SE;
                    gram_rows(dx + PR * W, dx, W, PR);
                    st = st + 1 == NST ? 0 : st + 1;
                }
                flush();
                if (tid == 0) {
                    my_rows += G::TO;
                    my_units += G::TO;
                }
            }
        }
        int64_t ch = ORD ? nch : blockIdx.x;
        int64_t pf = ch;
        if (!ORD)
            for (int s = 0; s < NST - 1; ++s, pf += gridDim.x) issue(pf, s);
        for (; ch < nch; ch += gridDim.x, pf += gridDim.x) {
            cp_wait<NST - 2>();
            __syncthreads();
            issue(pf, st == 0 ? NST - 1 : st - 1);
            const C *dx = sm + st * SE;
            gram_rows(dx + PR * W, dx, W, PR);
            st = st + 1 == NST ? 0 : st + 1;
            if (tid == 0) {
                my_rows += PR;
                my_units += PR;
            }
        }
        cp_wait<0>();
        __syncthreads();
    } else {
        // ---------------------------------------------------------------- products
        // permuted warps: with eight the columns of warps w and w + 4 (one scheduler) are w and
        // 7 - w; with four the columns go round from CTA to CTA
        const int pt = (NT == 128 ? (warp + int(blockIdx.x)) % 4 : warp < 4 ? warp : 11 - warp) * 32 + lane;
        const bool live = pt < q.CG * q.RG;
        const int cg = live ? pt / q.RG : 0, rg = live ? pt % q.RG : 0;
        const int col4 = cg * 4;
        int cmin = live ? col4 : W, cmax = live ? col4 + 3 : -1;
        for (int o = 16; o > 0; o >>= 1) {
            cmin = min(cmin, __shfl_xor_sync(0xffffffffu, cmin, o));
            cmax = max(cmax, __shfl_xor_sync(0xffffffffu, cmax, o));
        }
        const int nsub = q.TR / ACT_ROWS;
        const int n32 = int(a.n);
        const int64_t nvt = ORD ? olen : (cnt + nsub - 1) / nsub;
        const int64_t vt0 = ORD ? onorm(blockIdx.x) : int64_t(blockIdx.x);
        auto vt_next = [&](int64_t vt) -> int64_t {
            return ORD ? onorm(vt + int64_t(gridDim.x) * G::SO) : vt + gridDim.x;
        };
        // 32-row tile `u` of a virtual tile, -1 past the end
        auto vt_tile = [&](int64_t vt, int u) -> int64_t {
            if constexpr (ORD) {
                const int64_t t = otile(vt + int64_t(u / AO) * gridDim.x);
                const int64_t f = t * AO + u % AO;
                return t < 0 || f >= nt ? -1 : f;
            } else {
                return tile_at(vt * nsub + u);
            }
        };
        int nkb = 1;
        if (MODE == RB_UPD) nkb = a.qa ? 2 : 1;
        if (MODE == RB_ASM) nkb = a.ctrl ? min(a.ctrl->steps, a.nblk) : a.nblk;
        if (MODE == RB_ASMSUB) nkb = a.nblk;
        // first K block that is not zero in a virtual tile; nkb: the whole product is zero there
        auto first_kb = [&](int64_t vt) -> int {
            if (!MULTI || !a.tgen) return 0;
            int m = INT_MAX;
            for (int u = 0; u < nsub; ++u) {
                const int64_t t = vt_tile(vt, u);
                if (t >= 0) m = min(m, __ldg(a.tgen + t));
            }
            return min(max(m - a.kbase, 0), nkb);
        };
        // chunk cursor of the loads
        int64_t pvt = vt0;
        int pkb = 0, pk0 = 0;
        auto skip_empty = [&]() {
            while (pvt < nvt) {
                pkb = first_kb(pvt);
                if (pkb < nkb) break;
                pvt = vt_next(pvt);
            }
            pk0 = 0;
        };
        skip_empty();
        // The rows this thread copies of a virtual tile, and their tiles' distances, looked up once per
        // tile: a copy then costs one address.
        constexpr int EPV = std::is_same<T, C>::value ? VEC : 4;
        constexpr int VPR = KC / EPV;                                        // copies per row
        constexpr int NA = ((NT == 128 ? 128 : 256) * VPR + NT - 1) / NT;    // copies per thread, at most
        static_assert(NT % VPR == 0, "a thread's copies share their column");
        int prow[NA], pdist[NA];
        int64_t plook = -1;                                                  // the tile looked up
        const int pc = (tid % VPR) * EPV;
        auto look_up = [&]() {
            plook = pvt;
#pragma unroll
            for (int j = 0; j < NA; ++j) {
                const int r = tid / VPR + j * (NT / VPR);
                prow[j] = -1;
                pdist[j] = 0;
                if (r < q.TR) {
                    const int64_t t = vt_tile(pvt, r / ACT_ROWS);
                    const int64_t row = t * ACT_ROWS + r % ACT_ROWS;
                    if (t >= 0 && row < a.n) {
                        prow[j] = int(row);
                        if (a.tgen) pdist[j] = __ldg(a.tgen + t);
                    }
                }
            }
        };
        auto issue = [&](int st) {
            if (pvt < nvt) {
                if (plook != pvt) look_up();
                const T *src;
                const C *cmat;
                int lim;
                if (MODE == RB_UPD) {
                    const bool first = a.qa && pkb == 0;
                    src = first ? a.qa : a.qb;
                    cmat = first ? a.ca : a.cb;
                    lim = first ? a.lim_a : a.lim_b;
                } else if (MULTI) {
                    src = a.basis + int64_t(pkb) * a.block_stride;
                    cmat = a.ca + int64_t(pkb) * W * W;
                    lim = a.kbase + pkb;
                } else {
                    src = a.x;
                    cmat = a.ca;
                    lim = INT_MAX;
                }
                C *dA = sm + st * SE, *dC = dA + q.TR * LDA;
                if (pk0 + pc < q.Mk) {
#pragma unroll
                    for (int j = 0; j < NA; ++j) {
                        const int r = tid / VPR + j * (NT / VPR);
                        if (r >= q.TR) break;
                        const bool in = prow[j] >= 0 && pdist[j] <= lim;
                        const T *from = src + (in ? int64_t(prow[j]) * W + pk0 + pc : 0);
                        if constexpr (std::is_same<T, C>::value) {
                            cp16(dA + r * LDA + pc, from, in);
                        } else {
                            C v[4] = {0, 0, 0, 0};
                            if (in) ldg4<T>(from, v);
                            st4<C>(dA + r * LDA + pc, v);
                        }
                    }
                }
                const int crows = min(KC, q.Mk - pk0);
                for (int i = tid; i < crows * W / VEC; i += NT)
                    cp16(dC + i * VEC, cmat + pk0 * W + i * VEC, true);
                pk0 += KC;
                if (pk0 >= q.Mk) {
                    pk0 = 0;
                    if (++pkb >= nkb) {
                        pvt = vt_next(pvt);
                        skip_empty();
                    }
                }
            }
            cp_commit();
        };
        // the columns past Mk of the output tile stay zero
        for (int i = tid; i < q.TR * (LDO - q.Mk); i += NT)
            sO[(i / (LDO - q.Mk)) * LDO + q.Mk + i % (LDO - q.Mk)] = C(0);
        for (int s = 0; s < NST - 1; ++s) issue(s);
        // X of a virtual tile to the output tile, asynchronously, once the previous tile is done
        // with that; its copies belong to the next chunk's group
        auto load_x = [&](const int *rows) {
            for (int i = tid; i < q.TR * (W / VEC); i += NT) {
                const int r = i / (W / VEC), c = (i % (W / VEC)) * VEC;
                if (c >= q.Mk) continue;
                const int b = rows[r / ACT_ROWS], row = b + r % ACT_ROWS;
                const bool in = b >= 0 && row < n32;
                cp16(sO + r * LDO + c, a.x + (in ? int64_t(row) * W + c : 0), in);
            }
        };
        // the current tile's 32-row tiles (first row, -1: none), by parity of the tile: written
        // before the tile's first barrier, read after it
        __shared__ int s_row[2][8];
        int par = 0;
        int st = 0;
        for (int64_t vt = vt0; vt < nvt; vt = vt_next(vt), par ^= 1) {
            const int kb0 = first_kb(vt);
            if (tid < nsub) s_row[par][tid] = int(max(int64_t(-1), vt_tile(vt, tid) * ACT_ROWS));
            if (tid == 0) {
                const int64_t rows = ORD ? q.TR : min(int64_t(q.TR), (cnt - vt * nsub) * ACT_ROWS);
                my_rows += rows;
                my_units += (unsigned long long)(rows) * (nkb - kb0);
            }
            C acc[RPT][4];
#pragma unroll
            for (int r = 0; r < RPT; ++r)
#pragma unroll
                for (int u = 0; u < 4; ++u) acc[r][u] = 0;
            if (MODE == RB_ASM && a.accumulate && live) {
                // continue the accumulation of the earlier blocks from y (FP32, as stored)
#pragma unroll
                for (int r = 0; r < RPT; ++r) {
                    const int lr = rg + q.RG * r;
                    const int64_t t = vt_tile(vt, lr / ACT_ROWS);
                    const int64_t row = t * ACT_ROWS + lr % ACT_ROWS;
                    if (t >= 0 && row < a.n)
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (col4 + u < a.mo) acc[r][u] = C(a.y[row * a.ldy + col4 + u]);
                }
            }
            for (int kb = kb0; kb < nkb; ++kb)
                for (int k0 = 0; k0 < q.Mk; k0 += KC) {
                    cp_wait<NST - 2>();
                    __syncthreads();
                    if constexpr (ASYNC_X) {
                        if (kb == kb0 && k0 == 0) load_x(s_row[par]);
                    }
                    issue(st == 0 ? NST - 1 : st - 1);
                    const C *pA = sm + st * SE + rg * LDA;
                    const C *pC = sm + st * SE + q.TR * LDA + col4;
                    st = st + 1 == NST ? 0 : st + 1;
                    // R^{-1} (MUL, MULGRAM) is upper triangular: rows k > c add nothing to
                    // column c.  H_{k-1,k} (UPD with tri_a, first K block) is lower triangular:
                    // rows k < c add nothing.
                    int ks = 0, ke = min(KC, q.Mk - k0);
                    if (MODE == RB_MUL || MODE == RB_MULGRAM) ke = min(ke, cmax + 1 - k0);
                    if (MODE == RB_UPD && a.qa && a.tri_a && kb == 0) ks = max(0, cmin - k0);
                    if (cmax < 0) ke = 0;
                    auto step = [&](int k) {
                        C av[RPT][4], cv[4][4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) ld4<C>(pC + (k + j) * W, cv[j]);
#pragma unroll
                        for (int r = 0; r < RPT; ++r) ld4<C>(pA + q.RG * r * LDA + k, av[r]);
#pragma unroll
                        for (int j = 0; j < 4; ++j)
#pragma unroll
                            for (int r = 0; r < RPT; ++r) fma_row<C, 4>(acc[r], av[r][j], cv[j]);
                    };
                    if (ks == 0 && ke == KC) {
#pragma unroll
                        for (int k = 0; k < KC; k += 4) step(k);
                    } else {
#pragma unroll 1
                        for (int k = ks; k < ke; k += 4) step(k);
                    }
                }
            // The register tile goes to shared memory (UPD subtracts it from X on the way).
            // With an empty K loop no barrier has separated this from the previous tile.
            if (kb0 >= nkb) __syncthreads();
            if constexpr (ASYNC_X) {
                // (kb0 < nkb: UPD has a block always, ASMSUB the block of the seeds or a nearer one;
                // otherwise X is loaded here)
                if (kb0 >= nkb) {
                    load_x(s_row[par]);
                    cp_commit();
                }
                // the chunks after the one X came with may be too few to have waited for it
                if ((nkb - kb0) * ((q.Mk + KC - 1) / KC) < NST) cp_wait<0>();
                // other threads' copies
                __syncthreads();
            }
            if (live) {
#pragma unroll
                for (int r = 0; r < RPT; ++r) {
                    const int lr = rg + q.RG * r;
                    C o[4];
                    if (SUBX) {
                        C xv[4] = {0, 0, 0, 0};
                        if constexpr (std::is_same<T, C>::value) {
                            ld4<C>(sO + lr * LDO + col4, xv);
                        } else {
                            const int b = s_row[par][lr / ACT_ROWS], row = b + lr % ACT_ROWS;
                            if (b >= 0 && row < n32) ldg4<T>(a.x + int64_t(row) * W + col4, xv);
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u) o[u] = xv[u] - acc[r][u];
                    } else {
#pragma unroll
                        for (int u = 0; u < 4; ++u) o[u] = acc[r][u];
                    }
                    // narrow stored blocks now, so the Gram below is that of the stored values
                    if constexpr (!std::is_same<T, C>::value && MODE != RB_ASM) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) o[u] = C(T(o[u]));
                    }
                    st4<C>(sO + lr * LDO + col4, o);
                }
            }
            __syncthreads();
            // whole rows to HBM
            constexpr int CPR = W / 4;
            for (int i = tid; i < q.TR * CPR; i += NT) {
                const int r = i / CPR, c = (i % CPR) * 4;
                const int b = s_row[par][r / ACT_ROWS], rl = b + r % ACT_ROWS;
                if (b < 0 || rl >= n32) continue;
                const int64_t row = rl;
                C o[4];
                ld4<C>(sO + r * LDO + c, o);
                if (MODE == RB_ASM) {
                    float *y = a.y + row * a.ldy + c;
                    if (c + 3 < a.mo && (a.ldy & 3) == 0 && (reinterpret_cast<uintptr_t>(y) & 15) == 0) {
                        *reinterpret_cast<float4 *>(y) = make_float4(float(o[0]), float(o[1]), float(o[2]), float(o[3]));
                    } else {
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (c + u < a.mo) y[u] = float(o[u]);
                    }
                } else {
                    stg4<T>(a.out + row * W + c, o);
                }
            }
            if constexpr (ORD) {
#pragma unroll
                for (int u = 0; u < G::SO; ++u) {
                    gram_rows(sO + u * G::TO * LDO, sO + u * G::TO * LDO, LDO, G::TO);
                    flush();
                }
            } else {
                gram_rows(sO, sO, LDO, q.TR);
            }
        }
        cp_wait<0>();
        __syncthreads();
    }
    pdl_trigger();
    if (tid == 0 && a.prof.rows) {
        atomicAdd(a.prof.rows, my_rows);
        atomicAdd(a.prof.nnz, my_units);
    }
    if constexpr (GRAM) {
        // combine the row groups in a fixed order and write this CTA's W x W partial
        if constexpr (G::TWO && !ORD) flush();
        C *comb = G::G2S ? sG : sm;
        const int nth = q.NB * q.NGR;
        if constexpr (!G::G2S) {
            if (glive)
#pragma unroll
                for (int i = 0; i < BI; ++i)
#pragma unroll
                    for (int j = 0; j < BJ; ++j) comb[(i * BJ + j) * nth + tid] = g2[i][j];
        }
        __syncthreads();
        C *p = a.partials + int64_t(blockIdx.x) * W * W;
        for (int e = tid; e < W * W; e += NT) {
            int i = e / W, j = e % W;
            C v = 0;
            if (i < a.M && j < a.M) {
                constexpr int S = BI / BJ;
                if (MODE != RB_PROJ && j / BJ < S * (i / BI)) {   // below: the transposed entry
                    const int t = i;
                    i = j;
                    j = t;
                }
                const int bi = i / BI, bj = j / BJ;
                const int b = MODE == RB_PROJ ? bi * q.NJ + bj : bi * q.NJ - S * (bi * (bi - 1) / 2) + bj - S * bi;
                const C *src = comb + ((i % BI) * BJ + j % BJ) * nth + b;
                for (int w = 0; w < q.NGR; ++w) v += src[w * q.NB];
            }
            p[e] = v;
        }
    }
}

constexpr int RB_MAX_CTAS = 5;   // per SM

// Resident CTAs per SM of an instance with the shared memory that blocks of M columns take.  The
// runtime is asked once (several microseconds, and a solve needs it for every launch and for its plan);
// devices are taken to be alike, as in num_sms().  The attribute is raised once per instance to the
// most any block can take.
template <typename T, int W, int MODE, int RPT, bool ORD, int NT>
int occupancy(int M, size_t smem) {
    static std::atomic<int> known[W + 1];   // (zero: not asked yet)
    if (const int v = known[M].load(std::memory_order_relaxed)) return v;
    static const cudaError_t attr = cudaFuncSetAttribute(
        k_rowblock<T, W, MODE, RPT, ORD, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
    (void)attr;
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_rowblock<T, W, MODE, RPT, ORD, NT>, NT, smem);
    const int v = std::max(1, std::min(per_sm, RB_MAX_CTAS));
    if (per_sm > 0) known[M].store(v, std::memory_order_relaxed);
    return v;
}

template <typename T, int W, int MODE, int RPT, bool ORD, int NT>
int launch_r(const RowArgs<T> &a, cudaStream_t s, int *grid_out) {
    using G = Geo<T, W, ORD>;
    const RowGeo q = row_geo<T, W, MODE, RPT, ORD, NT>(a.M);
    const size_t smem = smem_bytes<T, W, MODE, ORD>(q);
    const int64_t unit = ORD ? G::TO : MODE == RB_PROJ ? G::PR : q.TR;
    const int64_t nvt = (a.n + unit - 1) / unit;
    const int per_sm = occupancy<T, W, MODE, RPT, ORD, NT>(a.M, smem);
    int grid = int(std::min<int64_t>(nvt, int64_t(num_sms()) * (ORD ? G::CTAS : per_sm)));
    if (MODE == RB_PROJ || MODE == RB_UPD || MODE == RB_MULGRAM || MODE == RB_ASMSUB) grid = std::min(grid, a.max_grid);
    if (grid < 1) grid = 1;
    if (grid_out) *grid_out = grid;
    if (a.plan) return 0;
    const cudaError_t e = launch_dep(k_rowblock<T, W, MODE, RPT, ORD, NT>, dim3(grid), NT, smem, s, 0, a);
    return e == cudaSuccess ? 0 : cuda_fail(e, "k_rowblock launch");
}

// Rows per thread.  FP32: 8 (12 shared loads per 128 FMAs instead of 8 per 64), 4 at W = 16
// where 8 would need more rows than a tile holds; 2 (4 at W = 128: a tile has at least 32
// rows) when the matrix has too few rows for one tile per SM, so that a small graph still
// spreads over the chip.  FP64: 4.
template <typename T, int W, int MODE>
int launch_mode(const RowArgs<T> &a, cudaStream_t s, int *grid_out) {
    constexpr int R = sizeof(typename Cmp<T>::type) == 8 || W == 16 ? 4 : 8;
    // Threads: CTAs of 256, two per SM where they fit, or four of 128 for the narrow blocks, whose tiles are
    // short of arithmetic between their barriers (128^3 grid, M = 32, 40 steps: 24.8 / 24.0 ms;
    // RGG of 10^6 rows, M = 64, where the taller tile shares the small matrix: 13.2 / 13.6 ms).
    constexpr int NT = sizeof(typename Cmp<T>::type) == 8 || MODE == RB_PROJ || W >= 64 ? 256 : 128;
    if constexpr (MODE != RB_PROJ) {
        const RowGeo q = row_geo<T, W, MODE, R, false, 256>(a.M);
        if (a.n < int64_t(q.TR) * num_sms()) return launch_r<T, W, MODE, W == 128 ? 4 : 2, false, 256>(a, s, grid_out);
    }
    return launch_r<T, W, MODE, R, false, NT>(a, s, grid_out);
}

template <typename T, int W>
int launch_w(int mode, const RowArgs<T> &a, cudaStream_t s, int *grid_out) {
    switch (mode) {
        case RB_PROJ: return launch_mode<T, W, RB_PROJ>(a, s, grid_out);
        case RB_UPD: return launch_mode<T, W, RB_UPD>(a, s, grid_out);
        case RB_MULGRAM: return launch_mode<T, W, RB_MULGRAM>(a, s, grid_out);
        case RB_MUL: return launch_mode<T, W, RB_MUL>(a, s, grid_out);
        case RB_ASM: return launch_mode<T, W, RB_ASM>(a, s, grid_out);
        case RB_ASMSUB: return launch_mode<T, W, RB_ASMSUB>(a, s, grid_out);
    }
    return fail(KB_ERR_ARG, "bad row-block mode");
}

// Ordered form: the modes with a Gram.
template <int W>
int launch_ordered(int mode, const RowArgs<float> &a, cudaStream_t s, int *grid_out) {
    constexpr int R = W == 128 ? 8 : 4;
    switch (mode) {
        case RB_PROJ: return launch_r<float, W, RB_PROJ, R, true, 256>(a, s, grid_out);
        case RB_UPD: return launch_r<float, W, RB_UPD, R, true, 256>(a, s, grid_out);
        case RB_MULGRAM: return launch_r<float, W, RB_MULGRAM, R, true, 256>(a, s, grid_out);
        case RB_ASMSUB: return launch_r<float, W, RB_ASMSUB, R, true, 256>(a, s, grid_out);
    }
    return fail(KB_ERR_ARG, "bad ordered row-block mode");
}

}  // namespace rb
}  // namespace kb
