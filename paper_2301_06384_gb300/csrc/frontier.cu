// Frontier restriction: hop distances from the node set, the 32-row tiles in order of their
// distance, and the zeros that the restricted kernels rely on.
//
// All of it is known before the first step.  One cooperative kernel runs the whole
// breadth-first search with a barrier between the levels, instead of two launches per step. A
// second one makes the tile lists of all steps at once, one CTA each.  A third writes the zeros
// that blocks need just beyond their reach, instead of clearing all of them.
//
// Measured, whole solves before -> after (per-step list and expansion launches, all blocks
// cleared in full): RGG of 10^6 rows, M = 64, 30 steps: gbl 4.82 -> 3.45 ms, cheb 2.16 -> 1.58
// ms; 128^3 grid, sbl, M = 128, 20 steps 14.7 -> 12.9 ms (22.5 GB of zeros not written).
#include "kb_internal.cuh"
#include "kb_kernels.cuh"

namespace kb {
namespace {

constexpr int BFS_THREADS = 512;
constexpr int BFS_ROWS = 8;    // queue rows a warp expands together
constexpr int BFS_U = 4;       // edges per lane in flight
// Breadth-first search from the nodes up to `levels` hops in one cooperative launch.  The queue
// holds the reached rows level after level; a row is claimed by an atomicOr on its bit of vis,
// whose 32-bit words are the 32-row tiles, so the claim that finds the word empty has found a
// new tile and its distance.  A warp takes 8 queue rows and spreads all their edges over its
// lanes (hubs are no serial loop of one thread).  qlev[k], tcnt[k]: rows and tiles first
// reached at level k.  Bound by latency: about five dependent L2 accesses and the barrier per
// level.
__global__ void __launch_bounds__(BFS_THREADS)
k_bfs(GraphDev g, NodeChunk seeds, int levels, uint8_t *gen, int32_t *tgen, uint32_t *vis, int32_t *queue,
      int32_t *qlev, int32_t *tcnt, int32_t *bar, int32_t *err, int spins) {
    const int lane = threadIdx.x & 31;
    const int gw = (int(blockIdx.x) * BFS_THREADS + int(threadIdx.x)) >> 5;
    const int nw = int(gridDim.x) * (BFS_THREADS / 32);
    int target = 0;
    if (blockIdx.x == 0 && threadIdx.x < seeds.cnt) {
        const int v = seeds.idx[threadIdx.x];
        const uint32_t old = atomicOr(vis + (v >> 5), 1u << (v & 31));
        gen[v] = 0;
        queue[threadIdx.x] = v;
        if (old == 0u) {
            tgen[v >> 5] = 0;
            atomicAdd(tcnt, 1);
        }
    }
    if (!grid_barrier(bar, err, target += gridDim.x, spins)) return;
    int start = 0, end = seeds.cnt;
    for (int k = 1; k <= levels && start < end; ++k) {
        for (int64_t base = start + int64_t(gw) * BFS_ROWS; base < end; base += int64_t(nw) * BFS_ROWS) {
            int beg = 0, deg = 0;
            if (lane < BFS_ROWS && base + lane < end) {
                const int i = __ldcg(queue + base + lane);
                beg = __ldg(g.rowptr + i);
                deg = __ldg(g.rowptr + i + 1) - beg;
            }
            int incl = deg;   // inclusive scan over the rows
#pragma unroll
            for (int o = 1; o < BFS_ROWS; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += u;
            }
            const int total = __shfl_sync(0xffffffffu, incl, BFS_ROWS - 1);
            const int shift = beg - (incl - deg);   // edge e of this row is col[shift + e]
            for (int e0 = 0; e0 < total; e0 += 32 * BFS_U) {
                int j[BFS_U];
#pragma unroll
                for (int u = 0; u < BFS_U; ++u) {
                    const int e = e0 + u * 32 + lane;
                    int r = 0;   // the row of edge e: number of inclusive sums <= e
#pragma unroll
                    for (int o = BFS_ROWS / 2; o > 0; o >>= 1)
                        if (__shfl_sync(0xffffffffu, incl, r + o - 1) <= e) r += o;
                    const int sh = __shfl_sync(0xffffffffu, shift, r);
                    j[u] = e < total ? __ldg(g.col + sh + e) : -1;
                }
                bool fresh[BFS_U];
#pragma unroll
                for (int u = 0; u < BFS_U; ++u)
                    fresh[u] = j[u] >= 0 && !((__ldcg(vis + (j[u] >> 5)) >> (j[u] & 31)) & 1u);
                int total_new = 0, tiles_new = 0;
                unsigned mask[BFS_U];
#pragma unroll
                for (int u = 0; u < BFS_U; ++u) {
                    bool tile = false;
                    if (fresh[u]) {
                        const uint32_t bit = 1u << (j[u] & 31);
                        const uint32_t old = atomicOr(vis + (j[u] >> 5), bit);
                        fresh[u] = !(old & bit);
                        tile = old == 0u;
                    }
                    if (tile) tgen[j[u] >> 5] = k;
                    mask[u] = __ballot_sync(0xffffffffu, fresh[u]);
                    total_new += __popc(mask[u]);
                    tiles_new += __popc(__ballot_sync(0xffffffffu, tile));
                }
                if (total_new == 0) continue;
                int pos = 0;
                if (lane == 0) {
                    pos = end + atomicAdd(qlev + k, total_new);
                    if (tiles_new) atomicAdd(tcnt + k, tiles_new);
                }
                pos = __shfl_sync(0xffffffffu, pos, 0);
#pragma unroll
                for (int u = 0; u < BFS_U; ++u) {
                    if (fresh[u]) {
                        queue[pos + __popc(mask[u] & ((1u << lane) - 1u))] = j[u];
                        gen[j[u]] = uint8_t(k);
                    }
                    pos += __popc(mask[u]);
                }
            }
        }
        if (!grid_barrier(bar, err, target += gridDim.x, spins)) return;
        start = end;
        end += __ldcg(qlev + k);
    }
}

// Compaction of the 32-row tiles whose distance satisfies in(tgen) into list[first ..], in index
// order, by one CTA of 1024 threads; returns their number.  Each warp owns a contiguous range
// of 32-tile groups and reads them coalesced, eight groups in flight; a ballot gives the group's
// members, kept in shared memory for the second pass (up to LIST_MASKS groups; beyond that the
// array is read again), and a block-wide exclusive scan of the warps' counts their offsets.
constexpr int LIST_MASKS = 8192;
template <typename P>
__device__ int compact_tiles(const int32_t *tgen, int64_t nact, const P &in, int first, int32_t *list) {
    __shared__ int wsum[33];
    __shared__ unsigned s_mask[LIST_MASKS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int64_t ngrp = (nact + 31) / 32;
    const bool cached = ngrp <= LIST_MASKS;
    const int64_t gper = (ngrp + nw - 1) / nw;
    const int64_t g0 = int64_t(warp) * gper;
    const int64_t g1 = g0 + gper < ngrp ? g0 + gper : ngrp;
    auto masks = [&](int64_t g, unsigned (&mk)[8]) {
        int32_t v[8];
        bool on[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int64_t a = (g + u) * 32 + lane;
            on[u] = g + u < g1 && a < nact;
            v[u] = on[u] ? __ldg(tgen + a) : 0;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) mk[u] = __ballot_sync(0xffffffffu, on[u] && in(v[u]));
    };
    int c = 0;
    for (int64_t g = g0; g < g1; g += 8) {
        unsigned mk[8];
        masks(g, mk);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (cached && lane == 0 && g + u < g1) s_mask[g + u] = mk[u];
            c += __popc(mk[u]);
        }
    }
    if (lane == 0) wsum[warp] = c;
    __syncthreads();
    if (warp == 0) {
        const int own = lane < nw ? wsum[lane] : 0;
        int incl = own;
        for (int off = 1; off < 32; off <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += u;
        }
        wsum[lane] = incl - own;               // exclusive offset of warp `lane`
        if (lane == 31) wsum[32] = incl;
    }
    __syncthreads();
    int pos = first + wsum[warp];
    const unsigned below = (1u << lane) - 1u;
    for (int64_t g = g0; g < g1; g += 8) {
        unsigned mk[8];
        if (cached) {
#pragma unroll
            for (int u = 0; u < 8; ++u) mk[u] = g + u < g1 ? s_mask[g + u] : 0u;
        } else {
            masks(g, mk);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if ((mk[u] >> lane) & 1u) list[pos + __popc(mk[u] & below)] = int32_t((g + u) * 32 + lane);
            pos += __popc(mk[u]);
        }
    }
    return wsum[32];
}

// The lists, one CTA each, all at once.  blockIdx.y = 0: the tiles at distance b = blockIdx.x (b =
// levels + 1: all that were not reached) into alist[acount[b - 1] ..], so alist holds all tiles by
// rising distance.  blockIdx.y = 1: the tiles within b hops in index order into lists[b]: in that
// order neighbouring rows are at work at the same time, and their gathers meet in L2 (RGG of
// 10^6 rows, M = 64, SpMM mean per launch 36.2 -> 34.5 us, with column dots 50.8 -> 46.7 us).
__global__ void __launch_bounds__(1024) k_tile_sort(int32_t *tgen, uint8_t *gen, int64_t n, int64_t nact, int levels,
                                                    const int32_t *__restrict__ tcnt, const int32_t *err,
                                                    int32_t *__restrict__ acount, int32_t *__restrict__ alist,
                                                    int32_t *__restrict__ lists) {
    __shared__ int s_before, s_own;
    const int b = blockIdx.x;
    if (*err) {
        // the search gave up: every row counts as reached at once
        const int64_t stride = int64_t(gridDim.x) * blockDim.x, i0 = int64_t(b) * blockDim.x + threadIdx.x;
        if (blockIdx.y == 0) {
            for (int64_t i = i0; i < n; i += stride) gen[i] = 0;
            for (int64_t i = i0; i < nact; i += stride) {
                tgen[i] = 0;
                alist[i] = int32_t(i);
            }
            if (b <= levels && threadIdx.x == 0) acount[b] = int32_t(nact);
        } else if (b <= levels) {
            for (int64_t i = threadIdx.x; i < nact; i += blockDim.x) lists[b * nact + i] = int32_t(i);
        }
        return;
    }
    if (blockIdx.y == 1) {
        if (b <= levels) compact_tiles(tgen, nact, [&](int v) { return v <= b; }, 0, lists + b * nact);
        return;
    }
    // tiles nearer than b, by warp 0
    if (threadIdx.x < 32) {
        int t = 0;
        for (int k = threadIdx.x; k < b; k += 32) t += tcnt[k];
        t = __reduce_add_sync(0xffffffffu, t);
        if (threadIdx.x == 0) {
            s_before = t;
            s_own = b <= levels ? tcnt[b] : int(nact - t);
            if (b <= levels) acount[b] = t + s_own;
        }
    }
    __syncthreads();
    if (s_own == 0) return;
    compact_tiles(tgen, nact, [&](int v) { return b <= levels ? v == b : v > levels; }, s_before, alist);
}

// Zeros on the listed tiles.  ring: block b of the stored basis is written on the tiles within
// b hops and read within b + 2 (by the next product's gathers), so a tile at distance d gets
// zeros in blocks d - 1 and d - 2, and in block 0 when d = 0 (before its unit entries are set).
// !ring: all nblk blocks on every listed tile (blocks that rotate through few buffers).
// Bytes: 2 (ring) or nblk tiles' rows per active tile, not nblk whole blocks.
__global__ void __launch_bounds__(256)
k_zero_tiles(unsigned char *blocks, int64_t block_bytes, int nblk, int row_bytes, int64_t n, int ring,
             const int32_t *__restrict__ tgen, const int32_t *__restrict__ alist, const int32_t *acount) {
    const int per = ring ? 2 : nblk;
    const int64_t total = int64_t(*acount) * per;
    for (int64_t it = blockIdx.x; it < total; it += gridDim.x) {
        const int tile = __ldg(alist + it / per);
        int b = int(it % per);
        if (ring) {
            const int d = __ldg(tgen + tile);
            b = d == 0 ? (b == 0 ? 0 : -1) : d - 1 - b;
            if (b < 0 || b >= nblk) continue;
        }
        const int64_t rows = n - int64_t(tile) * ACT_ROWS < ACT_ROWS ? n - int64_t(tile) * ACT_ROWS : ACT_ROWS;
        uint4 *p = reinterpret_cast<uint4 *>(blocks + b * block_bytes + int64_t(tile) * ACT_ROWS * row_bytes);
        for (int i = threadIdx.x; i < int(rows * row_bytes / 16); i += 256) p[i] = make_uint4(0, 0, 0, 0);
    }
}

}  // namespace

// qlev, tcnt (with the barrier behind them) and vis; the queue
constexpr size_t LV = FRONTIER_MAX_HOPS + 6;
static size_t zeroed_bytes(int64_t n) { return sizeof(int32_t) * 2 * LV + sizeof(uint32_t) * size_t((n + ACT_ROWS - 1) / ACT_ROWS); }
static size_t queue_offset(int64_t n) { return (zeroed_bytes(n) + 255) & ~size_t(255); }
size_t frontier_search_bytes(int64_t n) { return queue_offset(n) + sizeof(int32_t) * size_t(n); }

void plan_frontier(FrontierBufs &f, int64_t n, int levels, unsigned char *base, size_t *bytes, unsigned char *search) {
    f.levels = levels;
    f.nt = (n + ACT_ROWS - 1) / ACT_ROWS;
    const size_t nt = size_t((n + ACT_ROWS - 1) / ACT_ROWS);
    size_t off = 0;
    auto take = [&](size_t b) {
        unsigned char *p = base ? base + off : nullptr;
        off += (b + 255) & ~size_t(255);
        return p;
    };
    f.zeroed = search;
    f.zero_bytes = zeroed_bytes(n);
    f.qlev = reinterpret_cast<int32_t *>(f.zeroed);
    f.tcnt = f.qlev + LV;
    f.sync = f.tcnt + LV - 2;
    f.vis = reinterpret_cast<uint32_t *>(f.tcnt + LV);
    f.queue = reinterpret_cast<int32_t *>(search ? search + queue_offset(n) : nullptr);
    f.acount = reinterpret_cast<int32_t *>(take(sizeof(int32_t) * LV));
    f.gen = take(size_t(n));
    f.tgen = reinterpret_cast<int32_t *>(take(sizeof(int32_t) * nt));
    f.alist = reinterpret_cast<int32_t *>(take(sizeof(int32_t) * nt));
    f.lists = reinterpret_cast<int32_t *>(take(sizeof(int32_t) * nt * size_t(levels + 1)));
    *bytes = off;
}

int launch_frontier(const GraphDev &g, FrontierBufs &f, const int32_t *nodes, int M, cudaStream_t s, int spins) {
    const int levels = f.levels;
    const int64_t nt = (g.n + ACT_ROWS - 1) / ACT_ROWS;
    NodeChunk ch;
    if (M > NodeChunk::CAP || levels > FRONTIER_MAX_HOPS + 2) return fail(KB_ERR_ARG, "frontier too large");
    ch.cnt = M;
    ch.col0 = 0;
    for (int j = 0; j < M; ++j) ch.idx[j] = nodes[j];
    prof_begin(KernelClass::OTHER, s);
    KB_CUDA_TRY(cudaMemsetAsync(f.zeroed, 0, f.zero_bytes, s));
    KB_CUDA_TRY(cudaMemsetAsync(f.gen, 0xFF, size_t(g.n), s));
    KB_CUDA_TRY(cudaMemsetAsync(f.tgen, 0x7F, sizeof(int32_t) * size_t(nt), s));
    // one CTA per SM; a small graph has no use for all of them
    const unsigned grid = unsigned(std::max<int64_t>(1, std::min<int64_t>(num_sms(), (g.n + 2047) / 2048)));
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.gridDim = grid;
    cfg.blockDim = BFS_THREADS;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    KB_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_bfs, g, ch, levels, f.gen, f.tgen, f.vis, f.queue, f.qlev, f.tcnt,
                                   f.sync, f.sync + 1, spins));
    k_tile_sort<<<dim3(levels + 2, 2), 1024, 0, s>>>(f.tgen, f.gen, g.n, nt, levels, f.tcnt, f.sync + 1, f.acount,
                                                     f.alist, f.lists);
    KB_CUDA_TRY(cudaGetLastError());
    prof_end(KernelClass::OTHER, s, double(g.n) + 4.0 * double(nt), 0, 2);
    return 0;
}

int launch_zero_tiles(void *blocks, int64_t block_bytes, int nblk, int row_bytes, int64_t n, bool ring,
                      const FrontierBufs &f, cudaStream_t s) {
    const int64_t nt = (n + ACT_ROWS - 1) / ACT_ROWS;
    const int grid = int(std::max<int64_t>(1, std::min<int64_t>(nt * (ring ? 2 : nblk), int64_t(num_sms()) * 8)));
    k_zero_tiles<<<grid, 256, 0, s>>>(static_cast<unsigned char *>(blocks), block_bytes, nblk, row_bytes, n,
                                      ring ? 1 : 0, f.tgen, f.alist, f.acount + f.levels);
    count_launches(1);
    KB_CUDA_TRY(cudaGetLastError());
    return 0;
}

}  // namespace kb
