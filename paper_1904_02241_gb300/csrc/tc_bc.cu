// Betweenness centrality (the traversal benchmark of Sec. 3.3 and Sec. 4).
//
// Forward sweep: the shortest-path calculation of Alg. 3 (depth delta and shortest-path count
// sigma from one source), level by level, in the direction each level is cheaper in (Sec. 3.3's
// push-pull-push pattern: the first and last levels have small frontiers, the middle ones large):
//  * push: the frontier (the vertices of depth L, kept as a list) scatters over its out-edges;
//    an unreached target takes depth L+1 by compare-and-swap and every parent adds its sigma
//    with an FP64 atomic.  sigma counts paths, so every partial sum is an integer below 2^53
//    and exact: the result does not depend on the order of the additions.
//  * pull: every unreached vertex adds sigma over its in-neighbours of depth L (G^T), with no
//    atomics; a thread walks a short in-row, a warp a long one (in-degree >= 32, Sec. 3.2's
//    binning).  A vertex reads depth[u] of in-neighbours that other threads may set to L+1 in
//    the same launch; the old value (-1) and the new one both differ from L, so the read is
//    unaffected, and sigma[u] is read only for vertices of depth L, which no one writes now.
// Both directions append the vertices they reach to the next frontier list.
//
// Backward sweep: the dependency back-propagation of the BC the paper cites, over the level
// lists from the deepest, pulled over the out-edges of G: for a vertex v of depth L,
//   dep[v] = sum over out-neighbours w of depth L+1 of sigma[v] / sigma[w] * (1 + dep[w])
//          = sigma[v] * sum over those w of coef[w],   coef[w] = (1 + dep[w]) / sigma[w],
// so each vertex divides once (when its dependency is known) and each edge only adds; FP64
// division is slow on this GPU.  A lane group, a warp or a CTA per vertex: each lane adds its strided
// share of the row in order, then a fixed tree adds the lane sums; every vertex other than the source
// adds dep[v] to its score.  Operations are rounded one by one (no fused multiply-add).  A
// vertex's dependency reads only final values of the next level, so the order of a level's list
// (which the forward sweep fills as vertices are reached) does not change any result.
//
// sigma, the coefficients and the scores are FP64.  The coefficients are kept in two arrays by the parity
// of the vertex's depth, zero in the other one, so that an edge of the backward sweep reads one value
// and no depth: a vertex of depth L that reads the array of parity L+1 meets nonzero values at depth
// L+1 only (no out-edge spans two levels, and shallower levels have no coefficients yet), and adding
// the zeros of the others changes no sum.
#include <vector>

#include "tc_common_dev.cuh"
#include "tc_walk.cuh"

namespace tc {

constexpr int BC_THREADS = 256;
constexpr int BC_WARPS = BC_THREADS / 32;
constexpr int BC_LONG = 32;  // rows with at least this many edges get a warp in pull levels

struct BcPair {  // one array per parity of the depth
    double *even, *odd;
    __host__ __device__ __forceinline__ double *at(int32_t L) const { return (L & 1) ? odd : even; }
};

// This lane's share of a row: x of the columns first, first + step, ... below e, added in order; with
// `depth`, of those of depth L only.  The whole warp calls it (a lane without a row passes an empty one).
// Two things bound a row.  One load at a time, it is a chain of dependent round trips, and a level waits
// for its longest one (a hub's share of its CTA), so up to U loads of each kind are in flight.  And an
// FP64 addition takes its SM some 16 cycles per warp however few lanes need it, so a lane skips to its
// next nonzero value and the warp adds as often as its fullest lane needs (tested on the bits: comparing
// doubles is FP64 work too).
constexpr unsigned FULL_WARP = 0xffffffffu;
__device__ __forceinline__ bool bc_any(double x) { return __any_sync(FULL_WARP, __double_as_longlong(x) != 0ll); }

template <int U>
__device__ __forceinline__ double bc_row_sum(const int32_t *__restrict__ colidx, int32_t first, int32_t e, int32_t step,
                                             const double *x, const int32_t *depth = nullptr, int32_t L = 0) {
    double t = 0.0;
    for (int64_t i = first; __any_sync(FULL_WARP, i < e); i += (int64_t)U * step) {
        int32_t c[U];
        double y[U];
#pragma unroll
        for (int k = 0; k < U; ++k) c[k] = i + (int64_t)k * step < e ? __ldg(colidx + i + (int64_t)k * step) : -1;
        if (depth) {
            int32_t d[U];
#pragma unroll
            for (int k = 0; k < U; ++k) d[k] = c[k] >= 0 ? depth[c[k]] : -1;
#pragma unroll
            for (int k = 0; k < U; ++k)
                if (d[k] != L) c[k] = -1;
        }
#pragma unroll
        for (int k = 0; k < U; ++k) y[k] = c[k] >= 0 ? x[c[k]] : 0.0;
        unsigned m = 0;  // this lane's nonzero values, added lowest first
#pragma unroll
        for (int k = 0; k < U; ++k) m |= __double_as_longlong(y[k]) != 0ll ? 1u << k : 0u;
        while (__any_sync(FULL_WARP, m != 0u)) {
            double z = 0.0;
#pragma unroll
            for (int k = U - 1; k >= 0; --k)
                if ((m >> k) & 1u) z = y[k];
            m &= m - 1u;
            t = __dadd_rn(t, z);
        }
    }
    return t;
}

// The lanes' shares in a fixed tree over groups of G lanes; every lane of the group gets the sum.
template <int G>
__device__ __forceinline__ double bc_group_sum(double t) {
    if (bc_any(t)) {
#pragma unroll
        for (int q = G / 2; q > 0; q >>= 1) t = __dadd_rn(t, __shfl_xor_sync(FULL_WARP, t, q));
    }
    return t;
}

__global__ void k_bc_init(int32_t V, int32_t source, int32_t *depth, double *sigma, int32_t *order) {
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < V; v += (int64_t)gridDim.x * blockDim.x) {
        depth[v] = v == source ? 0 : -1;
        sigma[v] = v == source ? 1.0 : 0.0;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) order[0] = source;  // level 0
}

__global__ void k_bc_zero(int32_t V, double *score) {
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < V; v += (int64_t)gridDim.x * blockDim.x)
        score[v] = 0.0;
}

// out-degree of every frontier vertex (for the push level's edge prefix)
__global__ void k_bc_front_deg(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ front, int64_t nf,
                               int32_t *deg) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nf; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t u = front[i];
        deg[i] = __ldg(rowptr + u + 1) - __ldg(rowptr + u);
    }
}

// push level L, edge-balanced: thread t takes edges t, t + stride, ... of the frontier's
// concatenated out-rows (pre = exclusive prefix of their lengths, total = the sum) and finds its
// row by binary search, so a hub's row spreads over the whole grid.  The first edge to reach w
// claims it with a CAS on depth; every edge into a vertex of depth L+1 adds sigma[u] (integers
// below 2^53: exact in any order).  The next frontier and its out-edge count (the direction rule's
// m_f) go through the warps' queues.
__global__ void __launch_bounds__(BC_THREADS) k_bc_push_edges(const int32_t *__restrict__ rowptr,
                                                              const int32_t *__restrict__ colidx,
                                                              const int32_t *__restrict__ front, int64_t nf,
                                                              const int64_t *__restrict__ pre, int64_t total,
                                                              int32_t L, int32_t *depth, double *sigma, int32_t *next,
                                                              unsigned long long *count) {
    __shared__ int32_t wq_buf[BC_WARPS * WQ_ENTRIES];
    WarpQueue wq(wq_buf);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    // warp-uniform loop: the queue's ballots see the whole warp
    for (int64_t base = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); base < total; base += stride) {
        const int64_t e = base + (threadIdx.x & 31);
        bool claimed = false;
        int32_t w = 0, deg = 0;
        if (e < total) {
            int64_t lo = 0, hi = nf;  // last i with pre[i] <= e
            while (hi - lo > 1) {
                const int64_t mid = (lo + hi) >> 1;
                if (__ldg(pre + mid) <= e) lo = mid; else hi = mid;
            }
            const int32_t u = __ldg(front + lo);
            w = __ldg(colidx + __ldg(rowptr + u) + (e - __ldg(pre + lo)));
            int32_t dw = *(volatile int32_t *)(depth + w);
            if (dw == -1) {
                dw = atomicCAS(depth + w, -1, L + 1);
                if (dw == -1) {  // this edge reached w first
                    dw = L + 1;
                    claimed = true;
                    deg = __ldg(rowptr + w + 1) - __ldg(rowptr + w);
                }
            }
            if (dw == L + 1) atomicAdd(sigma + w, sigma[u]);
        }
        wq.push(claimed, w, deg, next, count);
    }
    wq.finish(next, count, count + 1);
}

// pull level L.  The first nhubs CTAs take a hub row each (more than hub_degree in-edges); in the
// others a warp takes 32 consecutive vertices: a lane sums a short in-row of an unreached one, the
// warp the rows of BC_LONG or more in-edges.  The sums are integers: exact in any order.  One
// launch instead of one per class: rows of the classes share the reads of depth and the row
// offsets, and hubs spread over a CTA instead of one warp.
__global__ void __launch_bounds__(BC_THREADS) k_bc_pull(const int32_t *__restrict__ in_rowptr,
                                                        const int32_t *__restrict__ in_colidx,
                                                        const int32_t *__restrict__ out_rowptr, int32_t V,
                                                        const int32_t *__restrict__ hubs, int32_t nhubs,
                                                        int32_t hub_degree, int32_t L, int32_t *depth, double *sigma,
                                                        int32_t *next, unsigned long long *count) {
    __shared__ int32_t wq_buf[BC_WARPS * WQ_ENTRIES];
    __shared__ double red[32];
    WarpQueue wq(wq_buf);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if ((int32_t)blockIdx.x < nhubs) {
        const int32_t v = hubs[blockIdx.x];
        const bool open = depth[v] == -1;  // the same for the whole CTA: only this CTA sets it
        double acc = 0.0;
        if (open) acc = bc_row_sum<8>(in_colidx, in_rowptr[v] + threadIdx.x, in_rowptr[v + 1], BC_THREADS, sigma, depth, L);
        acc = block_sum<double>(acc, red);  // every thread has read depth[v] by now
        const bool hit = open && acc != 0.0 && threadIdx.x == 0;  // sigma of a reached vertex is at least 1
        if (hit) {
            depth[v] = L + 1;
            sigma[v] = acc;
        }
        wq.push(hit, v, hit ? out_rowptr[v + 1] - out_rowptr[v] : 0, next, count);
    } else {
        const int64_t nw = (int64_t)(gridDim.x - nhubs) * BC_WARPS;
        for (int64_t grp = (int64_t)(blockIdx.x - nhubs) * BC_WARPS + warp; grp * 32 < V; grp += nw) {
            const int64_t v = grp * 32 + lane;
            int32_t s = 0, e = 0;
            if (v < V && depth[v] == -1) {
                s = in_rowptr[v];
                e = in_rowptr[v + 1];
                if (e - s > hub_degree) e = s;  // its own CTA
            }
            double acc = bc_row_sum<4>(in_colidx, s, e - s < BC_LONG ? e : s, 1, sigma, depth, L);
            unsigned long_rows = __ballot_sync(0xffffffffu, e - s >= BC_LONG);
            while (long_rows) {
                const int l = __ffs(long_rows) - 1;
                long_rows &= long_rows - 1;
                const int32_t ls = __shfl_sync(0xffffffffu, s, l), le = __shfl_sync(0xffffffffu, e, l);
                const double w = bc_group_sum<32>(bc_row_sum<8>(in_colidx, ls + lane, le, 32, sigma, depth, L));
                if (lane == l) acc = w;
            }
            const bool hit = __double_as_longlong(acc) != 0ll;
            if (hit) {
                depth[v] = L + 1;
                sigma[v] = acc;
            }
            wq.push(hit, (int32_t)v, hit ? __ldg(out_rowptr + v + 1) - __ldg(out_rowptr + v) : 0, next, count);
        }
    }
    wq.finish(next, count, count + 1);
}

// Blocked pull level (TOCAB, Sec. 3.3 with sigma sums as the "next" values): local row r of a
// pull partition (block b's in-edges of destination id_map[r]) gets the sum of sigma over its
// sources of depth L, 0 when it has none or its destination is already reached.  A lane takes a
// row below 32 edges, a warp a longer one.  The sums are integers: exact in any order.
__global__ void __launch_bounds__(BC_THREADS) k_bc_block_level(const int32_t *__restrict__ rowptr,
                                                               const int32_t *__restrict__ colidx,
                                                               const int32_t *__restrict__ id_map, int64_t R,
                                                               int32_t L, const int32_t *__restrict__ depth,
                                                               const double *__restrict__ sigma,
                                                               double *__restrict__ partial) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * BC_WARPS;
    for (int64_t grp = (blockIdx.x * (int64_t)BC_THREADS + threadIdx.x) >> 5; grp * 32 < R; grp += nw) {
        const int64_t r = grp * 32 + lane;
        int32_t s = 0, e = 0;
        if (r < R && depth[__ldg(id_map + r)] == -1) {
            s = __ldg(rowptr + r);
            e = __ldg(rowptr + r + 1);
        }
        double acc = bc_row_sum<4>(colidx, s, e - s < BC_LONG ? e : s, 1, sigma, depth, L);
        unsigned long_rows = __ballot_sync(0xffffffffu, e - s >= BC_LONG);
        while (long_rows) {
            const int l = __ffs(long_rows) - 1;
            long_rows &= long_rows - 1;
            const int32_t ls = __shfl_sync(0xffffffffu, s, l), le = __shfl_sync(0xffffffffu, e, l);
            const double w = bc_group_sum<32>(bc_row_sum<8>(colidx, ls + lane, le, 32, sigma, depth, L));
            if (lane == l) acc = w;
        }
        if (r < R) partial[r] = acc;
    }
}

// The blocked level's merge (Fig. 5): CTA j adds the partial sums of vertices [j k, (j+1) k) over
// the blocks in order, then every unreached vertex with a nonzero sum takes depth L+1 and that
// sigma and joins the next frontier.
__global__ void __launch_bounds__(BC_THREADS) k_bc_block_merge(const double *__restrict__ partial,
                                                               const int32_t *__restrict__ id_map,
                                                               const int32_t *__restrict__ merge_off, int32_t B,
                                                               int32_t nranges, int32_t k, int32_t V, int32_t L,
                                                               const int32_t *__restrict__ out_rowptr,
                                                               int32_t *depth, double *sigma, int32_t *next,
                                                               unsigned long long *count) {
    extern __shared__ double bacc[];  // [k]
    __shared__ int32_t wq_buf[BC_WARPS * WQ_ENTRIES];
    WarpQueue wq(wq_buf);
    for (int32_t j = blockIdx.x; j < nranges; j += gridDim.x) {
        const int32_t vbase = j * k;
        for (int32_t t = threadIdx.x; t < k; t += BC_THREADS) bacc[t] = 0.0;
        __syncthreads();
        for (int32_t b = 0; b < B; ++b) {
            const int32_t *o = merge_off + (int64_t)b * (nranges + 1) + j;
            const int32_t r0 = __ldg(o), r1 = __ldg(o + 1);
            for (int32_t r = r0 + threadIdx.x; r < r1; r += BC_THREADS) {
                const double x = partial[r];
                if (x != 0.0) bacc[__ldg(id_map + r) - vbase] = __dadd_rn(bacc[__ldg(id_map + r) - vbase], x);
            }
            __syncthreads();
        }
        for (int32_t t0 = 0; t0 < k && vbase + t0 < V; t0 += BC_THREADS) {  // the same steps for the whole CTA
            const int32_t t = t0 + (int32_t)threadIdx.x;
            const int32_t v = vbase + t;
            const bool in = t < k && v < V;
            const double x = in ? bacc[t] : 0.0;
            const bool hit = x != 0.0 && depth[v] == -1;
            if (hit) {
                depth[v] = L + 1;
                sigma[v] = x;
            }
            wq.push(hit, v, hit ? __ldg(out_rowptr + v + 1) - __ldg(out_rowptr + v) : 0, next, count);
        }
        __syncthreads();
    }
    wq.finish(next, count, count + 1);
}

// dependency of v from t = the sum over its children of (1 + dep[w]) / sigma[w]: dep[v] =
// sigma[v] t goes to the score, and (1 + dep[v]) / sigma[v] to coef[v] for v's parents
__device__ __forceinline__ void bc_dep_update(int32_t v, double t, int32_t source, const double *__restrict__ sigma,
                                              double *coef, double *score) {
    const double sv = sigma[v];
    const double d = __dmul_rn(sv, t);
    coef[v] = __ddiv_rn(__dadd_rn(1.0, d), sv);  // for the parents of v, one level up
    if (v != source) score[v] = __dadd_rn(score[v], d);
}

// Dependencies of the vertices of depth L (those of depth L+1 are final), by out-degree class:
// above the hub degree a CTA each (the first nhubs CTAs, one per hub of the graph's list; hubs at
// other depths leave at once), up to BC_SMALL a group of 8 lanes (four vertices per warp), between
// them the warp that met the vertex.  Each class adds in a fixed order, so scores repeat bit for bit.
// One launch per level instead of one per class, which read the level's list twice and cost three
// launches on the small levels (4 sources on a symmetrised R-MAT 18: 1,077 us of 2,096 in 75 launches).
// Bound by FP64 instructions where rows have many children, else by the longest row a warp meets.  With
// batched loads, skipped zeros, 32 divisions at a time and one vertex per warp step on all but the largest
// levels: 4 sources on a symmetrised R-MAT 18 1,702 to 1,422 us (the sweep's largest level 103 to 53 us).
constexpr int32_t BC_SMALL = 64;

__global__ void __launch_bounds__(BC_THREADS) k_bc_backward(const int32_t *__restrict__ rowptr,
                                                            const int32_t *__restrict__ colidx,
                                                            const int32_t *__restrict__ level_list, int64_t n,
                                                            const int32_t *__restrict__ hubs, int32_t nhubs, int32_t L,
                                                            int32_t source, int32_t small_max, int32_t hub_degree, int32_t per,
                                                            const int32_t *__restrict__ depth,
                                                            const double *__restrict__ sigma,
                                                            const double *coef_next, double *coef,
                                                            double *score) {
    __shared__ double red[32];
    if ((int32_t)blockIdx.x < nhubs) {
        const int32_t v = hubs[blockIdx.x];
        if (depth[v] != L) return;  // the same for the whole CTA
        double t = bc_row_sum<8>(colidx, rowptr[v] + threadIdx.x, rowptr[v + 1], BC_THREADS, coef_next);
        t = block_sum<double>(t, red);
        if (threadIdx.x == 0) bc_dep_update(v, t, source, sigma, coef, score);
        return;
    }
    // the vertices' sums wait here until 32 of them take their divisions together: one update per four
    // vertices kept the FP64 unit busy with four lanes of a warp
    __shared__ double wait_t[BC_WARPS][32];
    __shared__ int32_t wait_v[BC_WARPS][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane & 7;
    int nwait = 0;  // warp-uniform, at most 28 before a step
    // `per` vertices at a time (4 or 1), neighbours in the list to different CTAs: a level's long rows
    // stand close together in it, and are walked one after the other by the warp that meets them
    const int64_t ctas = gridDim.x - nhubs, step = ctas * BC_WARPS * per;
    // warp-uniform loop: the votes and shuffles below see the whole warp
    for (int64_t base = ((int64_t)warp * ctas + (blockIdx.x - nhubs)) * per; base < n; base += step) {
        const int64_t k = base + (lane >> 3);
        int32_t v = -1, s = 0, e = 0;
        if ((lane >> 3) < per && k < n) {
            v = level_list[k];
            s = rowptr[v];
            e = rowptr[v + 1];
        }
        const bool small = e - s <= small_max;
        double t = bc_group_sum<8>(bc_row_sum<4>(colidx, lane_first(s, e, sub), small ? e : s, 8, coef_next));
        unsigned wm = __ballot_sync(FULL_WARP, sub == 0 && !small && e - s <= hub_degree);
        while (wm) {
            const int l = __ffs(wm) - 1;
            wm &= wm - 1;
            const int32_t ls = __shfl_sync(FULL_WARP, s, l), le = __shfl_sync(FULL_WARP, e, l);
            const double x = bc_group_sum<32>(bc_row_sum<8>(colidx, ls + lane, le, 32, coef_next));
            if (lane == l) t = x;
        }
        const bool done = sub == 0 && v >= 0 && e - s <= hub_degree;
        const unsigned m = __ballot_sync(FULL_WARP, done);
        if (done) {
            const int at = nwait + __popc(m & ((1u << lane) - 1u));
            wait_t[warp][at] = t;
            wait_v[warp][at] = v;
        }
        nwait += __popc(m);
        if (nwait > 28) {
            __syncwarp();
            if (lane < nwait) bc_dep_update(wait_v[warp][lane], wait_t[warp][lane], source, sigma, coef, score);
            __syncwarp();
            nwait = 0;
        }
    }
    __syncwarp();
    if (lane < nwait) bc_dep_update(wait_v[warp][lane], wait_t[warp][lane], source, sigma, coef, score);
}

// A level runs in the push direction while its frontier's out-edges are fewer than
// 1 / BC_PUSH_RATIO of the out-edges of the vertices not yet reached (Beamer's rule).  The
// direction changes only the time: depths and the integer sigma sums are the same either way.
constexpr int64_t BC_PUSH_RATIO = 14;

struct BcScratch {
    DevBuf depth, sigma, coef, score, order, counter, bpartial;
    DevBuf fdeg, fpre, fws;  // push levels: frontier out-degrees, their prefix, scan scratch
    std::vector<int64_t> off;  // level L of `order` is [off[L], off[L+1])
    int grid = 1;
    // the odd levels' coefficients take the place of the push levels' prefix, which the backward sweep
    // does not need
    BcPair coefs() const { return BcPair{coef.as<double>(), fpre.as<double>()}; }
    int setup(const tc_graph *g, bool need_score, cudaStream_t s, const tc_part *part = nullptr) {
        if (part) {
            TC_TRY(bpartial.alloc((size_t)(part->R > 0 ? part->R : 1) * 8));
            TC_CUDA(cudaFuncSetAttribute(k_bc_block_merge, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)((size_t)part->k * 8)));
        }
        const int32_t V = g->V;
        DeviceCaps caps;
        TC_TRY(device_caps(&caps));
        grid = caps.sms * 8;
        TC_TRY(depth.alloc((size_t)V * 4));
        TC_TRY(sigma.alloc((size_t)V * 8));
        TC_TRY(coef.alloc((size_t)V * 8));
        TC_TRY(order.alloc((size_t)V * 4));
        if (need_score) TC_TRY(score.alloc((size_t)V * 8));
        TC_TRY(counter.alloc(16));
        TC_TRY(fdeg.alloc((size_t)V * 4 + 16));
        TC_TRY(fpre.alloc((size_t)V * 8 + 16));
        TC_TRY(fws.alloc((size_t)(scan_ws_elems(V) + 16) * 8));
        return TC_OK;
    }
};

// Forward sweep from `source`: depth/sigma, and w.order holding the reached vertices level by
// level.  *max_depth = the deepest level (levels 0 .. *max_depth).  *pushed counts push levels.
static int bc_forward_impl(const tc_graph *g, const tc_part *part, int32_t source, BcScratch &w, cudaStream_t s,
                           int32_t *max_depth, int32_t *pushed) {
    const int32_t V = g->V;
    int32_t *depth = w.depth.as<int32_t>(), *order = w.order.as<int32_t>();
    double *sigma = w.sigma.as<double>();
    unsigned long long *cnt = w.counter.as<unsigned long long>();  // found vertices, their out-edges
    const int32_t *orp = g->out_rowptr.as<int32_t>();
    k_bc_init<<<w.grid, BC_THREADS, 0, s>>>(V, source, depth, sigma, order);
    TC_LAUNCH_CHECK();
    w.off.assign(1, 0);
    w.off.push_back(1);
    // out-edges of the frontier (m_f) and of the vertices not yet reached (m_u)
    int32_t sdeg[2] = {0, 0};
    TC_CUDA(cudaMemcpyAsync(sdeg, orp + source, 8, cudaMemcpyDeviceToHost, s));
    TC_CUDA(cudaStreamSynchronize(s));
    int64_t m_f = sdeg[1] - sdeg[0], m_u = g->E - m_f;
    int32_t L = 0, np = 0;
    for (;; ++L) {
        const int64_t f0 = w.off[(size_t)L], nf = w.off[(size_t)L + 1] - f0;
        const int64_t reached = w.off[(size_t)L + 1];
        TC_CUDA(cudaMemsetAsync(cnt, 0, 16, s));
        int32_t *next = order + reached;
        if (m_f * BC_PUSH_RATIO < m_u) {  // push, edge-balanced over the frontier's out-rows
            if (m_f > 0) {
                k_bc_front_deg<<<w.grid, BC_THREADS, 0, s>>>(orp, order + f0, nf, w.fdeg.as<int32_t>());
                TC_LAUNCH_CHECK();
                TC_TRY(scan_i32_to_i64_ws(w.fdeg.as<int32_t>(), nf, w.fpre.as<int64_t>(), w.fws.as<int64_t>(), s));
                const int64_t want = (m_f + BC_THREADS - 1) / BC_THREADS;
                const int grid = (int)(want < w.grid ? want : w.grid);
                k_bc_push_edges<<<grid, BC_THREADS, 0, s>>>(orp, g->out_colidx.as<int32_t>(), order + f0, nf,
                                                            w.fpre.as<int64_t>(), m_f, L, depth, sigma, next, cnt);
                TC_LAUNCH_CHECK();
            }
            ++np;
        } else if (part) {  // blocked pull level (TOCAB) and its merge
            if (part->R > 0) {
                k_bc_block_level<<<w.grid, BC_THREADS, 0, s>>>(part->rowptr.as<int32_t>(), part->colidx.as<int32_t>(),
                                                               part->id_map.as<int32_t>(), part->R, L, depth, sigma,
                                                               w.bpartial.as<double>());
                TC_LAUNCH_CHECK();
            }
            const size_t smem = (size_t)part->k * 8;
            const int mgrid = part->nranges < w.grid ? (part->nranges > 0 ? part->nranges : 1) : w.grid;
            k_bc_block_merge<<<mgrid, BC_THREADS, smem, s>>>(w.bpartial.as<double>(), part->id_map.as<int32_t>(),
                                                             part->merge_off.as<int32_t>(), part->B, part->nranges,
                                                             part->k, V, L, orp, depth, sigma, next, cnt);
            TC_LAUNCH_CHECK();
        } else {
            k_bc_pull<<<w.grid + g->num_in_hubs, BC_THREADS, 0, s>>>(
                g->in_rowptr.as<int32_t>(), g->in_colidx.as<int32_t>(), orp, V, g->in_hubs.as<int32_t>(),
                g->num_in_hubs, g->hub_degree, L, depth, sigma, next, cnt);
            TC_LAUNCH_CHECK();
        }
        unsigned long long hc[2] = {0, 0};
        TC_CUDA(cudaMemcpyAsync(hc, cnt, 16, cudaMemcpyDeviceToHost, s));
        TC_CUDA(cudaStreamSynchronize(s));
        const unsigned long long found = hc[0];
        if (found == 0) break;
        w.off.push_back(reached + (int64_t)found);
        m_f = (int64_t)hc[1];
        m_u -= m_f;
    }
    *max_depth = L;
    if (pushed) *pushed = np;
    return TC_OK;
}

}  // namespace tc

extern "C" int tc_bc_forward(const tc_graph *g, int32_t source, int out_mem, int32_t *depth_out, double *sigma_out,
                             void *stream) {
    using namespace tc;
    if (!g || !depth_out || !sigma_out) return fail(TC_ERR_INVALID_ARG, "tc_bc_forward: null graph or output");
    if (source < 0 || source >= g->V) return fail(TC_ERR_INVALID_ARG, "tc_bc_forward: source outside [0, V)");
    if (out_mem != TC_MEM_HOST && out_mem != TC_MEM_DEVICE) return fail(TC_ERR_INVALID_ARG, "tc_bc_forward: bad out_mem");
    cudaStream_t s = (cudaStream_t)stream;
    const int32_t V = g->V;
    BcScratch w;
    TC_TRY(w.setup(g, false, s));
    int32_t maxd = 0;
    TC_TRY(bc_forward_impl(g, nullptr, source, w, s, &maxd, nullptr));
    const cudaMemcpyKind kind = out_mem == TC_MEM_DEVICE ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    TC_CUDA(cudaMemcpyAsync(depth_out, w.depth.p, (size_t)V * 4, kind, s));
    TC_CUDA(cudaMemcpyAsync(sigma_out, w.sigma.p, (size_t)V * 8, kind, s));
    TC_CUDA(cudaStreamSynchronize(s));
    return TC_OK;
}

namespace tc {
static int bc_impl(const tc_graph *g, const tc_part *part, const int32_t *sources, int32_t num_sources, int out_mem,
                   double *scores_out, void *stream);
}  // namespace tc

extern "C" int tc_bc(const tc_graph *g, const int32_t *sources, int32_t num_sources, int out_mem, double *scores_out,
                     void *stream) {
    return tc::bc_impl(g, nullptr, sources, num_sources, out_mem, scores_out, stream);
}

extern "C" int tc_bc_tocab(const tc_graph *g, const tc_part *part, const int32_t *sources, int32_t num_sources,
                           int out_mem, double *scores_out, void *stream) {
    using namespace tc;
    if (!part) return fail(TC_ERR_INVALID_ARG, "tc_bc_tocab: null partition");
    if (part->g != g || part->dir != TC_PULL)
        return fail(TC_ERR_INVALID_ARG, "tc_bc_tocab: the partition must be a TC_PULL partition of this graph");
    if (part->order != TC_ORDER_NATURAL)
        return fail(TC_ERR_UNSUPPORTED, "tc_bc_tocab: renumbered (TC_ORDER_OUTDEGREE) partitions are not supported");
    if ((size_t)part->k * 8 > 200 * 1024)
        return fail(TC_ERR_UNSUPPORTED, "tc_bc_tocab: merge_range above 25,600");
    return bc_impl(g, part, sources, num_sources, out_mem, scores_out, stream);
}

namespace tc {
static int bc_impl(const tc_graph *g, const tc_part *part, const int32_t *sources, int32_t num_sources, int out_mem,
                   double *scores_out, void *stream) {
    if (!g || !scores_out || (num_sources > 0 && !sources))
        return fail(TC_ERR_INVALID_ARG, "tc_bc: null graph, sources or output");
    if (num_sources < 0) return fail(TC_ERR_INVALID_ARG, "tc_bc: num_sources < 0");
    if (out_mem != TC_MEM_HOST && out_mem != TC_MEM_DEVICE) return fail(TC_ERR_INVALID_ARG, "tc_bc: bad out_mem");
    for (int32_t k = 0; k < num_sources; ++k)
        if (sources[k] < 0 || sources[k] >= g->V) return fail(TC_ERR_INVALID_ARG, "tc_bc: a source is outside [0, V)");
    cudaStream_t s = (cudaStream_t)stream;
    const int32_t V = g->V;
    if (V == 0) return TC_OK;
    BcScratch w;
    const bool dev_out = out_mem == TC_MEM_DEVICE;
    TC_TRY(w.setup(g, !dev_out, s, part));
    double *score = dev_out ? scores_out : w.score.as<double>();
    k_bc_zero<<<w.grid, BC_THREADS, 0, s>>>(V, score);
    TC_LAUNCH_CHECK();
    const BcPair coef = w.coefs();
    const int32_t small_max = BC_SMALL < g->hub_degree ? BC_SMALL : g->hub_degree;
    for (int32_t k = 0; k < num_sources; ++k) {
        int32_t maxd = 0;
        TC_TRY(bc_forward_impl(g, part, sources[k], w, s, &maxd, nullptr));
        TC_CUDA(cudaMemsetAsync(coef.even, 0, (size_t)V * 8, s));
        TC_CUDA(cudaMemsetAsync(coef.odd, 0, (size_t)V * 8, s));
        for (int32_t L = maxd; L >= 0; --L) {
            const int64_t a = w.off[(size_t)L], n = w.off[(size_t)L + 1] - a;
            // one vertex per warp step up to four steps of the whole grid, else four (4 sources on symmetrised
            // R-MAT 18 / R-MAT 21 / uniform 524,288: 1,356 / 3,799 / 2,103 us; always one 1,455 / 4,636 / 2,533,
            // always four 1,403 / 3,793 / 2,046)
            const int32_t per = n <= 4 * (int64_t)w.grid * BC_WARPS ? 1 : 4;
            const int grid = (int)(n < w.grid ? n : w.grid);
            k_bc_backward<<<grid + g->num_out_hubs, BC_THREADS, 0, s>>>(
                g->out_rowptr.as<int32_t>(), g->out_colidx.as<int32_t>(), w.order.as<int32_t>() + a, n,
                g->out_hubs.as<int32_t>(), g->num_out_hubs, L, sources[k], small_max, g->hub_degree, per,
                w.depth.as<int32_t>(), w.sigma.as<double>(), coef.at(L + 1), coef.at(L), score);
            TC_LAUNCH_CHECK();
        }
    }
    if (!dev_out) TC_CUDA(cudaMemcpyAsync(scores_out, score, (size_t)V * 8, cudaMemcpyDeviceToHost, s));
    TC_CUDA(cudaStreamSynchronize(s));
    return TC_OK;
}
}  // namespace tc
