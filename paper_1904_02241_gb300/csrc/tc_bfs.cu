// Topology-driven pull BFS with bitmap status arrays (Sec. 3.3, Fig. 1e/f).
//   unblocked level : warp per 32 vertices (one bitmap word); every unvisited vertex scans
//                     its in-edges with early exit until it finds a frontier source.
//   TOCAB level     : per block, a local "next" bit per local row (rows are scanned only
//                     over the block's sources), then a merge kernel ORs the local bits of
//                     all blocks per vertex range and writes levels, next and visited.
// Levels run TOCAB only when the frontier exceeds a fraction of V (Sec. 3.3).
#include "tc_common_dev.cuh"

namespace tc {

constexpr int BFS_THREADS = 256;
constexpr int BFS_WARPS = BFS_THREADS / 32;

// Where a scan looks a source up: the frontier bitmap, or a slice of it in shared memory that starts at
// source lo (a multiple of 32).
struct FrontBits {
    const uint32_t *__restrict__ front;
    __device__ __forceinline__ uint32_t word(int32_t u) const { return __ldg(front + (u >> 5)); }
};
struct SliceBits {
    const uint32_t *sl;
    int32_t lo;
    __device__ __forceinline__ uint32_t word(int32_t u) const { return sl[(u - lo) >> 5]; }
};

// Does one of the lane's edges [s, e) come from the frontier?  Early exit after 1, 4, 8, 12, ... edges: the
// loads of a step are in flight together (one by one, a row is a chain of two dependent round trips per
// edge), and the first edge alone, which is a hit for most rows when the frontier is large.
template <int N, class Bits>
__device__ __forceinline__ bool scan_step(const int32_t *__restrict__ colidx, int32_t i, int32_t e, Bits bits) {
    int32_t c[N];
    uint32_t hit = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) c[k] = k < e - i ? __ldg(colidx + i + k) : -1;
#pragma unroll
    for (int k = 0; k < N; ++k) hit |= (c[k] >= 0 ? bits.word(c[k]) : 0u) >> (c[k] & 31);
    return hit & 1u;
}
template <class Bits>
__device__ __forceinline__ bool scan_serial(const int32_t *__restrict__ colidx, int32_t s, int32_t e, Bits bits) {
    if (s >= e) return false;
    if (scan_step<1>(colidx, s, e, bits)) return true;
    if (e - s > 1 && scan_step<3>(colidx, s + 1, e, bits)) return true;
    for (int32_t left = e - s - 4; left > 0; left -= 4)
        if (scan_step<4>(colidx, e - left, e, bits)) return true;
    return false;
}

// Warp-cooperative scan of the rows flagged in `wm` (one at a time, early exit per chunk of 64 edges).
template <class Bits>
__device__ __forceinline__ bool scan_warp_rows(unsigned wm, int32_t s, int32_t e, const int32_t *__restrict__ colidx,
                                               Bits bits, bool found) {
    const int lane = threadIdx.x & 31;
    while (wm) {
        const int l = __ffs(wm) - 1;
        wm &= wm - 1;
        const int32_t ws = __shfl_sync(0xffffffffu, s, l), we = __shfl_sync(0xffffffffu, e, l);
        bool hit = false;
        for (int64_t base = ws; base < we; base += 64) {
            const int64_t i = base + lane;
            const int32_t c0 = i < we ? __ldg(colidx + i) : -1, c1 = i + 32 < we ? __ldg(colidx + i + 32) : -1;
            const uint32_t h0 = (c0 >= 0 ? bits.word(c0) : 0u) >> (c0 & 31);
            const uint32_t h1 = (c1 >= 0 ? bits.word(c1) : 0u) >> (c1 & 31);
            if (__any_sync(0xffffffffu, (h0 | h1) & 1u)) {
                hit = true;
                break;
            }
        }
        if (lane == l) found = hit;
    }
    return found;
}

// The rows of a warp's candidates, a lane each: short rows whole, the first SCAN_PROBE edges of a longer
// one; the longer rows without a hit there go to the whole warp one after the other, which is what a
// level waits for (the first pull level of a search on a symmetrised R-MAT 22: 93 us with every long row
// going there and one edge at a time, 49 us so).  Probes of 4 to 32 edges: all within 2%.
constexpr int SCAN_PROBE = 16;
template <class Bits>
__device__ __forceinline__ bool scan_rows(bool cand, int32_t s, int32_t e, const int32_t *__restrict__ colidx,
                                          Bits bits) {
    const bool is_long = e - s >= 32;
    const bool found = cand && scan_serial(colidx, s, is_long ? s + SCAN_PROBE : e, bits);
    return scan_warp_rows(__ballot_sync(0xffffffffu, cand && is_long && !found), is_long ? s + SCAN_PROBE : s, e, colidx,
                          bits, found);
}

__global__ void __launch_bounds__(BFS_THREADS) k_bfs_init(int32_t *level, uint32_t *visited, uint32_t *front,
                                                          int32_t V, int32_t nwords, int32_t source) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < V; i += (int64_t)gridDim.x * blockDim.x)
        level[i] = (i == source) ? 0 : -1;
    for (int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; w < nwords; w += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t bit = (w == (source >> 5)) ? (1u << (source & 31)) : 0u;
        visited[w] = bit;
        front[w] = bit;
    }
}

// Unblocked pull level.  next is written whole (one word per warp), visited updated,
// count accumulates the size of the new frontier.
__global__ void __launch_bounds__(BFS_THREADS, 8) k_bfs_pull_level(const int32_t *__restrict__ rowptr,
                                                                const int32_t *__restrict__ colidx, int32_t V,
                                                                int32_t nwords, const uint32_t *__restrict__ front,
                                                                uint32_t *__restrict__ next, uint32_t *visited,
                                                                int32_t *level, int32_t new_level,
                                                                unsigned long long *count,
                                                                const int32_t *__restrict__ out_rowptr) {
    __shared__ unsigned long long red[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long found_total = 0, deg_total = 0;
    const int64_t nw = (int64_t)gridDim.x * BFS_WARPS;
    for (int64_t w = (int64_t)blockIdx.x * BFS_WARPS + warp; w < nwords; w += nw) {
        const uint32_t vis = visited[w];
        const int64_t v = w * 32 + lane;
        const bool cand = v < V && !((vis >> lane) & 1u);
        uint32_t nb = 0;
        if (__any_sync(0xffffffffu, cand)) {
            int32_t s = 0, e = 0;
            if (cand) {
                s = __ldg(rowptr + v);
                e = __ldg(rowptr + v + 1);
            }
            const bool found = scan_rows(cand, s, e, colidx, FrontBits{front});
            nb = __ballot_sync(0xffffffffu, found);
            if (found) {
                level[v] = new_level;
                deg_total += (unsigned long long)(__ldg(out_rowptr + v + 1) - __ldg(out_rowptr + v));
            }
            if (lane == 0 && nb) visited[w] = vis | nb;
        }
        if (lane == 0) {
            next[w] = nb;
            found_total += __popc(nb);
        }
    }
    const unsigned long long t = block_sum<unsigned long long>(found_total, red);
    const unsigned long long dt = block_sum<unsigned long long>(deg_total, red);
    if (threadIdx.x == 0 && t) atomicAdd(count, t);
    if (threadIdx.x == 0 && dt) atomicAdd(count + 1, dt);
}

// TOCAB level, phase 1 (Alg. 4 form for traversal): local row r of the row space belongs to
// destination id_map[r]; bit r of rowbits = "some in-edge of r inside its block comes from
// the frontier", computed only for unvisited destinations.
__global__ void __launch_bounds__(BFS_THREADS, 8) k_bfs_block_level(const int32_t *__restrict__ rowptr,
                                                                 const int32_t *__restrict__ colidx,
                                                                 const int32_t *__restrict__ id_map, int64_t R,
                                                                 const uint32_t *__restrict__ front,
                                                                 const uint32_t *__restrict__ visited,
                                                                 uint32_t *__restrict__ rowbits) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t ngroups = (R + 31) >> 5;
    const int64_t nw = (int64_t)gridDim.x * BFS_WARPS;
    for (int64_t grp = (int64_t)blockIdx.x * BFS_WARPS + warp; grp < ngroups; grp += nw) {
        const int64_t r = grp * 32 + lane;
        bool cand = false;
        int32_t s = 0, e = 0;
        if (r < R) {
            const int32_t v = __ldg(id_map + r);
            cand = !((visited[v >> 5] >> (v & 31)) & 1u);
            if (cand) {
                s = __ldg(rowptr + r);
                e = __ldg(rowptr + r + 1);
            }
        }
        const bool found = scan_rows(cand, s, e, colidx, FrontBits{front});
        const uint32_t nb = __ballot_sync(0xffffffffu, found);
        if (lane == 0) rowbits[grp] = nb;
    }
}

// TOCAB level, phase 1, with the block's slice of the frontier bitmap in shared memory, for levels
// that still have most of the edges to scan.  CTAs draw chunks of BLK_CHUNK rows from a queue, in
// block order, and load a block's slice when they come to it; a block without a frontier vertex sets
// no bit and reads no edge.  Two ways through a group of 32 rows:
//   stream : the group's edges are read as one coalesced stream and every edge is tested; the row of
//            a hit comes from one ballot over the row offsets.  For small frontiers, where nearly every
//            edge is scanned anyway;
//   else   : a lane per row with early exit (scan_rows).  Streaming here too, with an edge's row from the
//            count of rows started up to it, was bound by its instructions: 385 against 363 us on the
//            level with the largest frontier with cold caches, and slower still with warm ones.
// Bound by reading the edges when it streams, by its instructions else (60% of issue slots); a lane per row
// waits for uncoalesced loads and random bitmap reads there.  Two searches on a symmetrised R-MAT of 5M
// vertices, 8 blocks, every level blocked: 5,781 us with k_bfs_block_level alone, then still an edge at a
// time (1,018 us for each of the first two levels), 2,770 us with this one in the levels above the line at its
// launch, 2,106 us with rows loaded a group ahead and scanned in steps and the merge as below.
constexpr int BLK_THREADS = 1024;
constexpr int BLK_CHUNK = 8192;  // rows: 8 groups per warp
constexpr size_t BLK_MAX_SMEM = 104 * 1024;  // slices of up to 851,968 sources: two CTAs per SM
// Below, a level has too few chunks to fill the chip and the slices' loads show.  Two searches on symmetrised
// graphs, 8 blocks, without and with this kernel: R-MAT of 1.8M edges 463 and 606 us, 7.6M 581 and 606, 15M 677
// and 702, 31M 1,172 and 939; uniform 8M 593 and 628, 17M 904 and 907, 34M 1,346 and 1,287.
constexpr int64_t BLK_MIN_EDGES = 1 << 24;

// Bit test of column c against the slice that starts at column lo (a multiple of 32).
__device__ __forceinline__ bool in_slice(const uint32_t *sl, int32_t c, int32_t lo) {
    const int32_t i = c - lo;
    return (sl[i >> 5] >> (i & 31)) & 1u;
}

__global__ void __launch_bounds__(BLK_THREADS, 2) k_bfs_block_smem(
    const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colidx, const int32_t *__restrict__ id_map,
    int64_t R, const int64_t *__restrict__ blk_rows, int32_t B, int32_t W, int32_t nwords,
    const uint32_t *__restrict__ front, const uint32_t *__restrict__ visited, uint32_t *__restrict__ rowbits,
    unsigned long long *queue, int stream) {
    extern __shared__ uint32_t sl[];  // W / 32 words: the slice of block `held`
    __shared__ long long s_chunk;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t held = -1;
    bool empty = false;  // the held slice has no frontier vertex (CTA-uniform)
    for (;;) {
        __syncthreads();  // the previous chunk is done with the slice and s_chunk
        if (threadIdx.x == 0) s_chunk = (long long)atomicAdd(queue, 1ull);
        __syncthreads();
        const int64_t c0 = s_chunk * BLK_CHUNK;
        if (c0 >= R) break;
        const int64_t c1 = c0 + BLK_CHUNK < R ? c0 + BLK_CHUNK : R;
        int32_t b = 0;  // the block of the chunk's first row: the last b with blk_rows[b] <= c0
        {
            int32_t hi = B - 1;
            while (b < hi) {
                const int32_t mid = (b + hi + 1) >> 1;
                if (__ldg(blk_rows + mid) <= c0) b = mid; else hi = mid - 1;
            }
        }
        const bool one = __ldg(blk_rows + b + 1) >= c1;  // the whole chunk lies in block b
        const int32_t lo = b * W;
        if (one && held != b) {
            const int32_t w0 = lo >> 5, n = min(W >> 5, nwords - w0);
            uint32_t any = 0;
            for (int32_t i = threadIdx.x; i < n; i += BLK_THREADS) {
                const uint32_t x = __ldg(front + w0 + i);
                sl[i] = x;
                any |= x;
            }
            empty = !__syncthreads_or(any != 0u);
            held = b;
        }
        // the next group's row offsets and vertices load while this one is scanned
        int32_t nv = -1, ns = INT32_MAX, ne = 0;
        auto rows_of = [&](int64_t r) {
            nv = -1;
            ns = INT32_MAX;
            ne = 0;
            if (r < c1) {
                nv = __ldg(id_map + r);
                ns = __ldg(rowptr + r);
                ne = __ldg(rowptr + r + 1);
            }
        };
        const bool skip = one && empty;
        if (!skip) rows_of(c0 + (int64_t)warp * 32 + lane);
        for (int64_t g0 = c0 + (int64_t)warp * 32; g0 < c1; g0 += BLK_THREADS) {
            uint32_t nb = 0;
            if (!skip) {
                const int32_t v = nv, s = ns;
                int32_t e = ne;
                rows_of(g0 + BLK_THREADS + lane);
                const bool cand = v >= 0 && !((__ldg(visited + (v >> 5)) >> (v & 31)) & 1u);
                const unsigned cm = __ballot_sync(0xffffffffu, cand);
                if (cm != 0u && one && stream) {
                    const int32_t t0 = __shfl_sync(0xffffffffu, s, 0);
                    const int32_t t1 = (int32_t)__reduce_max_sync(0xffffffffu, (unsigned)e);
                    unsigned rows = 0;  // rows with a hit (warp-uniform)
                    for (int64_t base = t0 & ~3; base < t1; base += 128) {
                        const int64_t i = base + 4 * lane;
                        unsigned h = 0;
                        if (i >= t0 && i + 3 < t1) {
                            const int4 c = __ldg(reinterpret_cast<const int4 *>(colidx + i));
                            h = (unsigned)in_slice(sl, c.x, lo) | ((unsigned)in_slice(sl, c.y, lo) << 1) |
                                ((unsigned)in_slice(sl, c.z, lo) << 2) | ((unsigned)in_slice(sl, c.w, lo) << 3);
                        } else {  // the ragged ends of the group's edges
                            for (int k = 0; k < 4; ++k)
                                if (i + k >= t0 && i + k < t1 && in_slice(sl, __ldg(colidx + i + k), lo)) h |= 1u << k;
                        }
                        unsigned m = __ballot_sync(0xffffffffu, h != 0u);
                        while (m) {
                            const int l = __ffs(m) - 1;
                            m &= m - 1;
                            unsigned hl = __shfl_sync(0xffffffffu, h, l);
                            while (hl) {
                                const int32_t at = (int32_t)base + 4 * l + __ffs(hl) - 1;
                                hl &= hl - 1;
                                // its row: the last one that starts at or before it
                                rows |= 1u << (__popc(__ballot_sync(0xffffffffu, s <= at)) - 1);
                            }
                        }
                    }
                    nb = rows & cm;
                } else if (cm != 0u) {
                    if (!cand) e = s;
                    const bool found = one ? scan_rows(cand, s, e, colidx, SliceBits{sl, lo})
                                           : scan_rows(cand, s, e, colidx, FrontBits{front});
                    nb = __ballot_sync(0xffffffffu, found);
                }
            }
            if (lane == 0) rowbits[g0 >> 5] = nb;
        }
    }
}

// TOCAB level, phase 2 (the reduction of the local next arrays, Sec. 3.3, in the merge
// kernel of Fig. 5): CTA j owns vertices [j*k, (j+1)*k); it ORs the local bits of every
// block's slice of that range, then writes next, visited and levels for the range.
__global__ void __launch_bounds__(BFS_THREADS) k_bfs_merge(const uint32_t *__restrict__ rowbits,
                                                           const int32_t *__restrict__ id_map,
                                                           const int32_t *__restrict__ merge_off, int32_t B,
                                                           int32_t nranges, int32_t k, int32_t V, int32_t nwords,
                                                           uint32_t *__restrict__ next, uint32_t *visited,
                                                           int32_t *level, int32_t new_level,
                                                           unsigned long long *count,
                                                           const int32_t *__restrict__ out_rowptr, int split) {
    extern __shared__ uint32_t hit[];  // k/32 words
    __shared__ unsigned long long red[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t j = blockIdx.x;
    const int32_t vbase = j * k;
    const int kw = k >> 5;
    for (int t = threadIdx.x; t < kw; t += BFS_THREADS) hit[t] = 0u;
    __syncthreads();
    // a warp per slice, or (`split`: few blocks, long slices) all warps along each; four rows of a lane in
    // flight.  8 blocks of a 5M-vertex R-MAT, a level that reaches most vertices: 87 us a warp per slice and a
    // row at a time, 50 us so
    const int32_t first = split ? warp * 128 : 0, step = split ? BFS_WARPS * 128 : 128;
    for (int32_t b = split ? 0 : warp; b < B; b += split ? 1 : BFS_WARPS) {
        const int32_t *o = merge_off + (int64_t)b * (nranges + 1) + j;
        const int32_t r0 = __ldg(o), r1 = __ldg(o + 1);
        for (int64_t r = (int64_t)r0 + first + lane; r < r1; r += step) {
            bool set[4];
            int32_t id[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int64_t q = r + 32 * k;
                set[k] = q < r1 && ((__ldg(rowbits + (q >> 5)) >> (q & 31)) & 1u);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) id[k] = set[k] ? __ldg(id_map + r + 32 * k) - vbase : 0;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (set[k]) atomicOr(&hit[id[k] >> 5], 1u << (id[k] & 31));
        }
    }
    __syncthreads();
    // a word per lane, then the warp takes its 32 words one by one with a vertex per lane: the level
    // stores and row offsets are coalesced and independent (a lane walking its own word's bits waited for
    // every vertex)
    unsigned long long found_total = 0, deg_total = 0;
    for (int t0 = warp * 32; t0 < kw; t0 += BFS_THREADS) {
        const int t = t0 + lane;
        const int64_t w = (int64_t)(vbase >> 5) + t;
        uint32_t nb = 0;
        if (t < kw && w < nwords) {
            const uint32_t vis = visited[w];
            nb = hit[t] & ~vis;
            next[w] = nb;
            if (nb) visited[w] = vis | nb;
        }
        found_total += __popc(nb);
        unsigned m = __ballot_sync(0xffffffffu, nb != 0u);
        while (m) {
            const int l = __ffs(m) - 1;
            m &= m - 1;
            const uint32_t x = __shfl_sync(0xffffffffu, nb, l);
            if ((x >> lane) & 1u) {
                const int64_t v = ((int64_t)(vbase >> 5) + t0 + l) * 32 + lane;
                level[v] = new_level;
                deg_total += (unsigned long long)(__ldg(out_rowptr + v + 1) - __ldg(out_rowptr + v));
            }
        }
    }
    const unsigned long long tot = block_sum<unsigned long long>(found_total, red);
    const unsigned long long dt = block_sum<unsigned long long>(deg_total, red);
    if (threadIdx.x == 0 && tot) atomicAdd(count, tot);
    if (threadIdx.x == 0 && dt) atomicAdd(count + 1, dt);
}

// Push (top-down, data-driven) levels for small frontiers (Sec. 3.3: the push phases of the
// push-pull-push schedule, Alg. 3 without sigma): every frontier vertex in the queue scans its
// out-edges; an unvisited neighbour is claimed with an atomic OR on the visited bitmap, gets
// its level, joins the next bitmap and is appended to the next queue (through its warp's queue).
// Edge-balanced push level: the out-degrees of the queue are scanned (pre[q+1]); thread t takes
// edges t, t + stride, ... of the frontier's concatenated out-rows, finds its row by binary
// search in pre, and claims the neighbour as above.  Hubs spread over the whole grid.
__global__ void k_push_degrees(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ queue, int32_t qn,
                               int32_t *deg) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < qn; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t u = queue[i];
        deg[i] = __ldg(rowptr + u + 1) - __ldg(rowptr + u);
    }
}

__global__ void __launch_bounds__(BFS_THREADS) k_bfs_push_edges(const int32_t *__restrict__ rowptr,
                                                                const int32_t *__restrict__ colidx,
                                                                const int32_t *__restrict__ queue, int32_t qn,
                                                                const int64_t *__restrict__ pre, int64_t total,
                                                                uint32_t *visited, uint32_t *next, int32_t *level,
                                                                int32_t new_level, int32_t *next_queue,
                                                                unsigned long long *count) {
    __shared__ int32_t wq_buf[BFS_WARPS * WQ_ENTRIES];
    WarpQueue wq(wq_buf);
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < total; base += stride) {
        const int64_t e = base + lane;
        bool claimed = false;
        int32_t v = 0;
        if (e < total) {
            int32_t lo = 0, hi = qn;  // last i with pre[i] <= e
            while (hi - lo > 1) {
                const int32_t mid = (lo + hi) >> 1;
                if (__ldg(pre + mid) <= e) lo = mid; else hi = mid;
            }
            const int32_t u = __ldg(queue + lo);
            v = __ldg(colidx + __ldg(rowptr + u) + (e - __ldg(pre + lo)));
            const uint32_t bit = 1u << (v & 31);
            if (!(visited[v >> 5] & bit)) {
                const uint32_t old = atomicOr(visited + (v >> 5), bit);
                claimed = !(old & bit);
            }
        }
        int32_t dg = 0;
        if (claimed) {
            level[v] = new_level;
            atomicOr(next + (v >> 5), 1u << (v & 31));
            dg = __ldg(rowptr + v + 1) - __ldg(rowptr + v);
        }
        wq.push(claimed, v, dg, next_queue, count);
    }
    wq.finish(next_queue, count, count + 1);
}

// ---- cluster-resident push levels ------------------------------------------------------------
// Consecutive push levels with small frontiers run inside ONE launch of a thread-block cluster: a
// level costs a few dependent memory round trips instead of a host round trip and five launches.
// The grid is exactly one cluster, so every CTA is co-scheduled by construction.
//
// Such a level is bound by its chain of dependent round trips, so the chain is kept to two of them
// (an out-row's neighbours, then the claims), plus one exchange through distributed shared memory:
//   * a CTA expands the vertices it claimed itself, whose out-edge ranges it kept in shared memory;
//   * a neighbour's row offsets are loaded beside the atomic OR on visited that claims it, not after;
//   * up to RES_DEG out-edges per vertex a thread walks its own vertex, all its loads in flight; only
//     batches with longer rows scan the degrees and deal the edges out one per thread;
//   * a level ends when every CTA's counts (claimed vertices, their out-edges) have arrived in this
//     CTA's mailbox: one asynchronous remote store per pair, completing on the receiver's mbarrier
//     (bounded wait).  Nothing else crosses CTAs, so the levels and queues written to global memory
//     are not waited for; only a level that deals the frontier out anew (one CTA holds more than
//     RES_THREADS out-edges and more than twice the mean) or the end of the launch uses the cluster
//     barrier with its release of global writes.  Two mailboxes alternate: a CTA sends level l + 1's
//     counts after it has read level l's, so a slot is free before it is written again.
// The counts tell every thread the same, and it takes the decision that the host would: stop when
// the frontier is empty, when direction optimisation switches to pull (14 m_f > m_u), or when the
// next level has more than `cap` vertices or out-edges.  At the end the claimed vertices are copied,
// in CTA order, into the host's queue for the next level.  What other CTAs wrote during the launch is
// read with L2 loads (ld.global.cg), never through L1.
// Measured on a 2048^2 grid with 5% of its edges removed (some 3,000 levels): 24.2 ms with the frontier kept in
// global queues and the cluster barrier at every level, 12.7 ms so.
constexpr int RES_THREADS = 1024;
constexpr int RES_WARPS = RES_THREADS / 32;
constexpr int RES_MAX_CTAS = 16;
constexpr int RES_DEG = 4;      // out-edges of a vertex walked by its own thread: 2 / 4 / 8 on that grid 9.8 /
                                // 10.6 / 10.9 ms back to back
constexpr int RES_KEEP = 2048;  // claimed vertices per CTA and level whose ranges stay in shared memory (512: the same)

struct ResOut {  // written by CTA 0, thread 0 when the launch ends
    unsigned long long front;  // frontier size of level `lvl`
    double m_f, m_u;           // its out-edges, and those of the unvisited vertices
    int32_t lvl;               // the next level to expand
    int32_t levels;            // levels expanded by the launch
    int32_t timeout;           // nonzero: a wait for the counts gave up
};

__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The address of this CTA's shared-memory word in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t remote_smem(const void *p, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr(p)), "r"(rank));
    return r;
}
// Asynchronous 8-byte store to a CTA of the cluster; its bytes complete on that CTA's mbarrier.
__device__ __forceinline__ void remote_store_async(uint32_t dst, unsigned long long x, uint32_t mbar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(dst), "l"(x),
                 "r"(mbar)
                 : "memory");
}
// mbar_wait with cluster-scope acquire (the awaited bytes come from other CTAs).
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t *bar, uint32_t parity) {
    const long long t0 = clock64();
    for (;;) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(smem_addr(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
        if (clock64() - t0 > (1LL << 31)) return false;
    }
}

// Exclusive prefix sum over the CTA (RES_THREADS threads); *total gets the sum.  All threads call it.
__device__ __forceinline__ int32_t res_block_scan(int32_t x, int32_t *wsum /* [RES_WARPS + 1] */, int32_t *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t inc = x;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += y;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const int32_t w = wsum[lane];
        int32_t wi = w;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, wi, d);
            if (lane >= d) wi += y;
        }
        wsum[lane] = wi - w;  // exclusive over warps
        if (lane == 31) wsum[RES_WARPS] = wi;
    }
    __syncthreads();
    *total = wsum[RES_WARPS];
    return wsum[warp] + inc - x;
}

// What a CTA's threads append to: its segments of one level.
struct ResSeg {
    int32_t *v;         // [cap] claimed vertices (global)
    int2 *r;            // [cap] their out-edge ranges from RES_KEEP on (global)
    int2 *keep;         // [RES_KEEP] the first ones' ranges (shared)
    unsigned *cnt;      // claimed vertices, their out-edges (shared)
    int32_t cap;
};

// The whole warp appends the lanes' claims: bit k of `claimed` = vertex v[k] with range r[k].
template <int K>
__device__ __forceinline__ void res_append(const ResSeg &q, unsigned claimed, const int32_t *v, const int2 *r) {
    if (!__any_sync(0xffffffffu, claimed != 0u)) return;
    const int lane = threadIdx.x & 31;
    const unsigned c = (unsigned)__popc(claimed);
    unsigned dg = 0;
#pragma unroll
    for (int k = 0; k < K; ++k)
        if ((claimed >> k) & 1u) dg += (unsigned)(r[k].y - r[k].x);
    unsigned inc = c;
    if (K == 1) {
        const unsigned m = __ballot_sync(0xffffffffu, claimed != 0u);
        inc = (unsigned)__popc(m & ((2u << lane) - 1u));
    } else {
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, inc, d);
            if (lane >= d) inc += y;
        }
    }
    dg = __reduce_add_sync(0xffffffffu, dg);
    unsigned base = 0;
    if (lane == 31) {
        base = atomicAdd(q.cnt, inc);
        atomicAdd(q.cnt + 1, dg);
    }
    unsigned p = __shfl_sync(0xffffffffu, base, 31) + inc - c;
#pragma unroll
    for (int k = 0; k < K; ++k)
        if ((claimed >> k) & 1u) {
            if (p < (unsigned)q.cap) {  // always: a CTA claims at most the level's edges
                q.v[p] = v[k];
                if (p < (unsigned)RES_KEEP) q.keep[p] = r[k];
                else q.r[p] = r[k];
            }
            ++p;
        }
}

// Claims v for level new_level; its out-edge range is loaded beside the claim.
__device__ __forceinline__ bool res_claim(const int32_t *__restrict__ rowptr, uint32_t *visited, int32_t *level,
                                          int32_t v, int32_t new_level, int2 *range) {
    const uint32_t bit = 1u << (v & 31);
    const uint32_t old = atomicOr(visited + (v >> 5), bit);
    range->x = __ldg(rowptr + v);
    range->y = __ldg(rowptr + v + 1);
    if (old & bit) return false;
    level[v] = new_level;
    return true;
}

// seg_v / seg_r: [2 parities][C CTAs][cap] vertex IDs and out-edge ranges of the claimed vertices.
__global__ void __launch_bounds__(RES_THREADS, 1) k_bfs_push_resident(
    const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colidx, uint32_t *visited, int32_t *level,
    int32_t *q0, int32_t *q1, int32_t *seg_v, int2 *seg_r, int64_t *trace, int32_t lvl0, int32_t n0, int64_t mu0,
    int32_t cap, int32_t max_levels, ResOut *out) {
    __shared__ int32_t sh_start[RES_THREADS], sh_off[RES_THREADS];
    __shared__ int2 keep[2][RES_KEEP];
    __shared__ int32_t wsum[RES_WARPS + 1];
    __shared__ unsigned s_cnt[2][2];                         // this CTA's claims by level parity: vertices, out-edges
    __shared__ unsigned long long s_mail[2][RES_MAX_CTAS];   // every CTA's counts by level parity
    __shared__ __align__(8) uint64_t s_bar[2];
    __shared__ int32_t s_pre[RES_MAX_CTAS + 1];              // prefix of the segment counts
    __shared__ int s_failed;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t C = (int32_t)gridDim.x, c = (int32_t)blockIdx.x;
    if (tid < 4) s_cnt[tid >> 1][tid & 1] = 0u;
    if (tid == 0) {
        mbar_init(&s_bar[0], 1);
        mbar_init(&s_bar[1], 1);
        s_failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    cluster_barrier();  // every CTA's mailboxes exist
    int32_t lvl = lvl0, levels = 0, n = n0, mine = 0;
    int64_t mf = 0, mu = mu0;
    enum { QUEUE, OWN, DEALT } from = QUEUE;  // the frontier: the host's queue, this CTA's claims, or all CTAs' segments
    bool failed = false;
    for (;;) {
        const int par = lvl & 1;  // this level's claims: counters, mailbox and segments of parity par
        if (tid == 0) {
            s_cnt[par ^ 1][0] = s_cnt[par ^ 1][1] = 0u;  // the next level's: sent before the last wait
            mbar_expect_tx(&s_bar[par], (uint32_t)C * 8u);
        }
        const int32_t *hq = (lvl & 1) ? q1 : q0;
        const int2 *in_r = seg_r + (size_t)(par ^ 1) * C * cap;
        ResSeg out_q;
        out_q.v = seg_v + ((size_t)par * C + c) * cap;
        out_q.r = seg_r + ((size_t)par * C + c) * cap;
        out_q.keep = keep[par];
        out_q.cnt = s_cnt[par];
        out_q.cap = cap;
        const int32_t lo = from == OWN ? 0 : (int32_t)((int64_t)n * c / C);
        const int32_t hi = from == OWN ? mine : (int32_t)((int64_t)n * (c + 1) / C);
        for (int32_t b0 = lo; b0 < hi; b0 += RES_THREADS) {
            const int32_t i = b0 + tid;
            int32_t s = 0, e = 0;
            if (i < hi) {
                if (from == QUEUE) {
                    const int32_t u = __ldcg(hq + i);
                    s = __ldg(rowptr + u);
                    e = __ldg(rowptr + u + 1);
                } else {
                    int2 r;
                    if (from == OWN) {
                        r = i < RES_KEEP ? keep[par ^ 1][i] : __ldcg(in_r + (size_t)c * cap + i);
                    } else {  // entry i of the concatenated segments
                        int32_t a = 0;
                        while (a + 1 < C && s_pre[a + 1] <= i) ++a;
                        r = __ldcg(in_r + (size_t)a * cap + (i - s_pre[a]));
                    }
                    s = r.x;
                    e = r.y;
                }
            }
            if (!__syncthreads_or(e - s > RES_DEG)) {  // short rows: a thread walks its own vertex
                int32_t v[RES_DEG];
                int2 r[RES_DEG];
                unsigned claimed = 0;
#pragma unroll
                for (int k = 0; k < RES_DEG; ++k) v[k] = s + k < e ? __ldg(colidx + s + k) : -1;
#pragma unroll
                for (int k = 0; k < RES_DEG; ++k) {
                    r[k] = make_int2(0, 0);
                    if (v[k] >= 0 && res_claim(rowptr, visited, level, v[k], lvl + 1, &r[k])) claimed |= 1u << k;
                }
                res_append<RES_DEG>(out_q, claimed, v, r);
                continue;
            }
            int32_t total;
            const int32_t off = res_block_scan(e - s, wsum, &total);
            sh_start[tid] = s;
            sh_off[tid] = off;
            __syncthreads();
            const int32_t nb = min(RES_THREADS, hi - b0);
            for (int32_t base = warp * 32; base < total; base += RES_THREADS) {
                const int32_t k = base + lane;
                unsigned claimed = 0;
                int32_t v = 0;
                int2 r = make_int2(0, 0);
                if (k < total) {  // the last vertex of the batch whose edges start at or before k
                    int32_t a = 0, z = nb - 1;
                    while (a < z) {
                        const int32_t mid = (a + z + 1) >> 1;
                        if (sh_off[mid] <= k) a = mid; else z = mid - 1;
                    }
                    v = __ldg(colidx + sh_start[a] + (k - sh_off[a]));
                    claimed = res_claim(rowptr, visited, level, v, lvl + 1, &r) ? 1u : 0u;
                }
                res_append<1>(out_q, claimed, &v, &r);
            }
            __syncthreads();  // the batch's offsets are read before the next batch overwrites them
        }
        ++levels;
        __syncthreads();  // the CTA's claims are counted
        if (tid < C)
            remote_store_async(remote_smem(&s_mail[par][c], (uint32_t)tid),
                               ((unsigned long long)s_cnt[par][0] << 32) | s_cnt[par][1],
                               remote_smem(&s_bar[par], (uint32_t)tid));
        // level lvl0 + i completes phase i / 2 of its barrier; the CTA agrees on whether it did
        failed = __syncthreads_or(!mbar_wait_cluster(&s_bar[par], (uint32_t)(((levels - 1) >> 1) & 1)));
        if (failed) break;
        const unsigned long long mail = lane < C ? s_mail[par][lane] : 0ull;
        const unsigned cn = (unsigned)(mail >> 32), ce = (unsigned)mail;
        n = (int32_t)__reduce_add_sync(0xffffffffu, cn);
        mf = (int64_t)__reduce_add_sync(0xffffffffu, ce);  // at most the graph's edges, below 2^31
        const unsigned most = __reduce_max_sync(0xffffffffu, ce);
        mine = (int32_t)__shfl_sync(0xffffffffu, cn, c);
        mu -= mf;
        ++lvl;
        if (c == 0 && tid == 0 && lvl < TC_BFS_TRACE) trace[lvl] = n;
        // 14 mf > mu is the host's mf > mu / 14 for integers
        const bool stop = n == 0 || 14 * mf > mu || n > cap || mf > (int64_t)cap || levels >= max_levels;
        from = OWN;
        const bool deal = !stop && most > (unsigned)RES_THREADS && (int64_t)most * C > 2 * mf;
        if (stop || deal) {  // rare
            if (warp == 0) {
                unsigned inc = cn;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const unsigned y = __shfl_up_sync(0xffffffffu, inc, d);
                    if (lane >= d) inc += y;
                }
                if (lane < C) s_pre[lane + 1] = (int32_t)inc;
                if (lane == 0) s_pre[0] = 0;
            }
            __syncthreads();
        }
        if (deal) {
            int2 *seg = seg_r + ((size_t)par * C + c) * cap;
            for (int32_t i = tid; i < mine && i < RES_KEEP; i += RES_THREADS) seg[i] = keep[par][i];
            cluster_barrier();
            from = DEALT;
        }
        if (stop) break;
    }
    // the frontier of level lvl into the host's queue for it, segments in CTA order
    if (!failed) {
        const int32_t *src = seg_v + ((size_t)((lvl - 1) & 1) * C + c) * cap;
        int32_t *dst = ((lvl & 1) ? q1 : q0) + s_pre[c];
        const int32_t cnt = s_pre[c + 1] - s_pre[c];
        for (int32_t i = tid; i < cnt; i += RES_THREADS) dst[i] = __ldcg(src + i);
    }
    if (failed && tid == 0)
        asm volatile("st.shared::cluster.u32 [%0], 1;" ::"r"(remote_smem(&s_failed, 0u)) : "memory");
    // No CTA leaves while another may still store into its shared memory.  Twice: a CTA whose wait gave up
    // may meet the others' barrier of a dealt level here, and they send it one more message after that.
    cluster_barrier();
    if (c == 0 && tid == 0) {
        out->timeout = s_failed;
        out->front = (unsigned long long)n;
        out->m_f = (double)mf;
        out->m_u = (double)mu;
        out->lvl = lvl;
        out->levels = levels;
    }
    cluster_barrier();
}

// front = the bits of the queue's vertices (the frontier bitmap after resident push levels).
__global__ void k_queue_bits(const int32_t *__restrict__ queue, int64_t qn, uint32_t *front) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < qn; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t v = queue[i];
        atomicOr(front + (v >> 5), 1u << (v & 31));
    }
}

// Cluster size for the resident push levels: 16 CTAs when the device schedules such a cluster
// of RES_THREADS-thread CTAs, else 8, else 0 (resident levels off).
static int res_cluster_size(cudaStream_t s) {
    static int chosen = -1;
    if (chosen >= 0) return chosen;
    chosen = 0;
    for (int C : {16, 8}) {
        if (C > 8 && cudaFuncSetAttribute(k_bfs_push_resident, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
                         cudaSuccess) {
            cudaGetLastError();
            continue;
        }
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(C);
        cfg.blockDim = dim3(RES_THREADS);
        cfg.stream = s;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = C;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int nclusters = 0;
        if (cudaOccupancyMaxActiveClusters(&nclusters, k_bfs_push_resident, &cfg) == cudaSuccess && nclusters >= 1) {
            chosen = C;
            break;
        }
        cudaGetLastError();
    }
    return chosen;
}

// Queue of the vertices set in a bitmap (for a push level after a pull level), in any order, through the
// warps' queues: one launch instead of a popcount, a scan and a write (five launches, 17 us).
__global__ void __launch_bounds__(BFS_THREADS) k_bitmap_queue(const uint32_t *__restrict__ bits, int32_t nwords,
                                                              int32_t *queue, unsigned long long *count) {
    __shared__ int32_t wq_buf[BFS_WARPS * WQ_ENTRIES];
    WarpQueue wq(wq_buf);
    const int lane = threadIdx.x & 31;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t w0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); w0 < nwords; w0 += step) {
        const uint32_t mine = w0 + lane < nwords ? __ldg(bits + w0 + lane) : 0u;
        unsigned m = __ballot_sync(0xffffffffu, mine != 0u);
        while (m) {
            const int l = __ffs(m) - 1;
            m &= m - 1;
            const uint32_t w = __shfl_sync(0xffffffffu, mine, l);
            wq.push((w >> lane) & 1u, (int32_t)((w0 + l) * 32 + lane), 0, queue, count);
        }
    }
    wq.finish(queue, count, count);  // no weights: nothing is added to the second word
}

// edges_reached = sum of out-degrees of vertices with level >= 0; reached = their count.
__global__ void __launch_bounds__(BFS_THREADS) k_bfs_stats(const int32_t *level, const int32_t *out_rowptr, int32_t V,
                                                           unsigned long long *out) {
    __shared__ unsigned long long red[32];
    unsigned long long n = 0, m = 0;
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < V; v += (int64_t)gridDim.x * blockDim.x) {
        if (level[v] >= 0) {
            ++n;
            m += (unsigned long long)(out_rowptr[v + 1] - out_rowptr[v]);
        }
    }
    n = block_sum<unsigned long long>(n, red);
    m = block_sum<unsigned long long>(m, red);
    if (threadIdx.x == 0) {
        atomicAdd(out, n);
        atomicAdd(out + 1, m);
    }
}

__global__ void k_set_int(int32_t *p, int32_t v) { *p = v; }

static int bfs_impl(const tc_graph *cg, const tc_part *part, int32_t source, const tc_bfs_params *bp,
                    int32_t *levels_out, tc_bfs_stats *stats, cudaStream_t s) {
    tc_graph *g = const_cast<tc_graph *>(cg);
    const int32_t V = g->V;
    const int32_t nwords = (V + 31) / 32;
    DeviceCaps caps;
    TC_TRY(device_caps(&caps));
    TC_TRY(g->ws_bits.alloc((size_t)nwords * 4 * 3 + 64));
    uint32_t *visited = g->ws_bits.as<uint32_t>();
    uint32_t *bufs[2] = {visited + nwords, visited + 2 * nwords};
    unsigned long long *cnt = reinterpret_cast<unsigned long long *>(visited + 3 * nwords + (nwords & 1));
    int32_t *level = levels_out;
    if (bp->out_mem == TC_MEM_HOST) {
        TC_TRY(g->ws_misc.alloc((size_t)V * 4 + 256));
        level = g->ws_misc.as<int32_t>();
    }
    const int grid = caps.sms * 8;
    float ms_total = 0;
    cudaEvent_t ev[2] = {nullptr, nullptr};
    if (bp->profile) {
        TC_CUDA(cudaEventCreate(&ev[0]));
        TC_CUDA(cudaEventCreate(&ev[1]));
        TC_CUDA(cudaEventRecord(ev[0], s));
    }
    k_bfs_init<<<grid, BFS_THREADS, 0, s>>>(level, visited, bufs[0], V, nwords, source);
    TC_LAUNCH_CHECK();
    const bool can_push = bp->push_threshold > 0.0f;
    // push-level buffers live with the graph (no allocation, and so no synchronisation, per call)
    DevBuf &queues = g->ws_queue, &qcnt = g->ws_qcnt, &qpos = g->ws_qpos;
    int32_t *q[2] = {nullptr, nullptr};
    const int64_t cap = (int64_t)(V > nwords ? V : nwords) + 16;
    if (can_push) {
        TC_TRY(queues.alloc((size_t)2 * V * 4 + 64));
        TC_TRY(qcnt.alloc((size_t)cap * 4));
        TC_TRY(qpos.alloc((size_t)cap * 8));
        TC_TRY(g->ws_scan.alloc((size_t)(scan_ws_elems(cap) + 16) * 8));
        q[0] = queues.as<int32_t>();
        q[1] = q[0] + V;
        k_set_int<<<1, 1, 0, s>>>(q[0], source);
        TC_LAUNCH_CHECK();
    }
    bool have_queue = can_push;  // the queue q[lvl & 1] holds the current frontier
    unsigned long long front_count = 1;
    if (!g->h_counts) TC_CUDA(cudaMallocHost(&g->h_counts, 64));
    unsigned long long *h_cnt = g->h_counts;
    // resident push levels: one cluster runs consecutive push levels whose frontier has at most
    // res_cap vertices and out-edges (queue segments of res_cap entries per CTA and parity)
    const int32_t res_cap = bp->resident_edges < 0 ? TC_BFS_RESIDENT_DEFAULT : bp->resident_edges;
    const int res_C = (can_push && res_cap > 0) ? res_cluster_size(s) : 0;
    int32_t *res_v = nullptr;  // [2][res_C][res_cap] queue segments
    int2 *res_r = nullptr;     // their out-edge ranges
    int64_t *res_trace = nullptr;
    ResOut *res_out = nullptr;
    if (res_C > 0) {
        const size_t nseg = (size_t)2 * res_C * res_cap;
        TC_TRY(g->ws_res.alloc(nseg * 12 + 64 + TC_BFS_TRACE * 8 + 64));
        res_r = g->ws_res.as<int2>();
        res_v = reinterpret_cast<int32_t *>(res_r + nseg);
        res_out = reinterpret_cast<ResOut *>(reinterpret_cast<unsigned char *>(res_v + nseg) + 64 -
                                             (reinterpret_cast<uintptr_t>(res_v + nseg) & 63));
        res_trace = reinterpret_cast<int64_t *>(reinterpret_cast<unsigned char *>(res_out) + 64);
    }
    bool bits_valid = true;  // bufs[lvl & 1] holds the frontier (not after resident push levels)
    int resident_levels = 0;
    // direction switching (Beamer et al.): edges out of the frontier (m_f) against edges out of
    // unvisited vertices (m_u); push -> pull when m_f > m_u / 14, pull -> push when the
    // frontier holds fewer than push_threshold * V vertices
    int32_t *sdeg = reinterpret_cast<int32_t *>(h_cnt);
    TC_CUDA(cudaMemcpyAsync(sdeg, g->out_rowptr.as<int32_t>() + source, 8, cudaMemcpyDeviceToHost, s));
    TC_CUDA(cudaStreamSynchronize(s));
    double m_f = (double)(sdeg[1] - sdeg[0]);
    double m_u = (double)g->E - m_f;
    bool pushing = can_push;
    int lvl = 0, tocab_levels = 0, push_levels = 0;
    int st = TC_OK;
    cudaEvent_t lev[2] = {nullptr, nullptr};
    if (bp->profile && stats) {
        TC_CUDA(cudaEventCreate(&lev[0]));
        TC_CUDA(cudaEventCreate(&lev[1]));
    }
    const int merge_split = part && part->R > (int64_t)part->B * part->nranges * 512 ? 1 : 0;
    const size_t merge_smem = part ? (size_t)(part->k / 32) * 4 : 0;
    // blocked levels with the slice in shared memory: two CTAs per SM
    int blk_grid = 0;
    const size_t blk_smem = part ? (size_t)(part->W / 32) * 4 : 0;
    if (part && g->E >= BLK_MIN_EDGES && bp->tocab_threshold >= 0.0f && part->R > 0 && part->W % 32 == 0 && blk_smem <= BLK_MAX_SMEM) {
        TC_CUDA(cudaFuncSetAttribute(k_bfs_block_smem, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BLK_MAX_SMEM));
        const int64_t chunks = (part->R + BLK_CHUNK - 1) / BLK_CHUNK;
        blk_grid = (int)(chunks < 2 * caps.sms ? chunks : 2 * caps.sms);
    }
    while (front_count > 0) {
        uint32_t *front = bufs[lvl & 1], *next = bufs[(lvl + 1) & 1];
        // the level's counts and the blocked level's chunk queue
        if (cudaMemsetAsync(cnt, 0, 24, s) != cudaSuccess) { st = fail(TC_ERR_CUDA, "memset failed"); break; }
        if (can_push) {
            if (pushing && m_f > m_u / 14.0) pushing = false;
            else if (!pushing && (double)front_count < (double)bp->push_threshold * (double)V) pushing = true;
        }
        const bool use_push = can_push && pushing;
        const bool use_tocab = !use_push && part && bp->tocab_threshold >= 0.0f &&
                               (double)front_count > (double)bp->tocab_threshold * (double)V;
        if (stats && lvl < TC_BFS_TRACE) {
            stats->level_kind[lvl] = use_push ? 2 : (use_tocab ? 1 : 0);
            stats->level_frontier[lvl] = (int64_t)front_count;
        }
        if (lev[0]) cudaEventRecord(lev[0], s);
        if (use_push && res_C > 0 && have_queue && (int64_t)front_count <= res_cap && m_f <= (double)res_cap) {
            // consecutive push levels in one cluster launch; the host reads where they stopped
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(res_C);
            cfg.blockDim = dim3(RES_THREADS);
            cfg.stream = s;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = res_C;
            at[0].val.clusterDim.y = 1;
            at[0].val.clusterDim.z = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            cudaError_t e = cudaLaunchKernelEx(&cfg, k_bfs_push_resident, (const int32_t *)g->out_rowptr.as<int32_t>(),
                                               (const int32_t *)g->out_colidx.as<int32_t>(), visited, level, q[0],
                                               q[1], res_v, res_r, res_trace, (int32_t)lvl, (int32_t)front_count,
                                               (int64_t)m_u, res_cap, (int32_t)(V + 1), res_out);
            if (lev[1] && e == cudaSuccess) e = cudaEventRecord(lev[1], s);
            if (e == cudaSuccess) e = cudaMemcpyAsync(h_cnt + 2, res_out, sizeof(ResOut), cudaMemcpyDeviceToHost, s);
            if (e == cudaSuccess) e = cudaStreamSynchronize(s);
            if (e != cudaSuccess) { st = fail(TC_ERR_CUDA, "bfs resident levels from %d: %s", lvl, cudaGetErrorString(e)); break; }
            ResOut ro;
            memcpy(&ro, h_cnt + 2, sizeof(ro));
            if (ro.timeout) { st = fail(TC_ERR_TIMEOUT, "bfs resident levels from %d: a bounded device wait gave up", lvl); break; }
            if (ro.levels < 1 || ro.lvl != lvl + ro.levels) { st = fail(TC_ERR_CUDA, "bfs resident levels: bad exit state"); break; }
            if (stats) {
                float seg_ms = 0.0f;
                if (lev[1]) cudaEventElapsedTime(&seg_ms, lev[0], lev[1]);
                const int hi = ro.lvl < TC_BFS_TRACE ? ro.lvl : TC_BFS_TRACE;
                if (lvl + 1 < hi) {
                    e = cudaMemcpy(stats->level_frontier + lvl + 1, res_trace + lvl + 1, (size_t)(hi - lvl - 1) * 8,
                                   cudaMemcpyDeviceToHost);
                    if (e != cudaSuccess) { st = fail(TC_ERR_CUDA, "bfs trace copy: %s", cudaGetErrorString(e)); break; }
                }
                for (int l = lvl; l < hi; ++l) {
                    stats->level_kind[l] = 3;
                    stats->level_ms[l] = seg_ms / (float)ro.levels;
                }
            }
            push_levels += ro.levels;
            resident_levels += ro.levels;
            front_count = ro.front;
            m_f = ro.m_f;
            m_u = ro.m_u;
            lvl = ro.lvl;
            have_queue = true;
            bits_valid = false;
            continue;
        }
        if (!use_push && !bits_valid) {  // pull levels read the frontier bitmap: rebuild it from the queue
            if (cudaMemsetAsync(front, 0, (size_t)nwords * 4, s) != cudaSuccess) { st = fail(TC_ERR_CUDA, "memset failed"); break; }
            k_queue_bits<<<grid, BFS_THREADS, 0, s>>>(q[lvl & 1], (int64_t)front_count, front);
            if (cudaGetLastError() != cudaSuccess) { st = fail(TC_ERR_CUDA, "launch failed"); break; }
        }
        bits_valid = true;
        push_levels += use_push ? 1 : 0;
        if (use_push) {
            if (!have_queue) {  // frontier came from a pull level: bitmap -> queue
                k_bitmap_queue<<<grid, BFS_THREADS, 0, s>>>(front, nwords, q[lvl & 1], cnt + 2);
                if (cudaGetLastError() != cudaSuccess) { st = fail(TC_ERR_CUDA, "launch failed"); break; }
            }
            if (cudaMemsetAsync(next, 0, (size_t)nwords * 4, s) != cudaSuccess) { st = fail(TC_ERR_CUDA, "memset failed"); break; }
            // out-degree prefix of the queue: frontier edges m_f are already known on the host
            const int32_t qn = (int32_t)front_count;
            k_push_degrees<<<grid, BFS_THREADS, 0, s>>>(g->out_rowptr.as<int32_t>(), q[lvl & 1], qn,
                                                        qcnt.as<int32_t>());
            if (cudaGetLastError() != cudaSuccess) { st = fail(TC_ERR_CUDA, "launch failed"); break; }
            st = scan_i32_to_i64_ws(qcnt.as<int32_t>(), qn, qpos.as<int64_t>(), g->ws_scan.as<int64_t>(), s);
            if (st != TC_OK) break;
            const int64_t total = (int64_t)(m_f + 0.5);
            if (total > 0)
                k_bfs_push_edges<<<grid, BFS_THREADS, 0, s>>>(g->out_rowptr.as<int32_t>(), g->out_colidx.as<int32_t>(),
                                                              q[lvl & 1], qn, qpos.as<int64_t>(), total, visited, next,
                                                              level, lvl + 1, q[(lvl + 1) & 1], cnt);
            have_queue = true;
        } else if (use_tocab) {
            // most edges still to scan: the bitmap slice in shared memory, streamed while the frontier is
            // small (an edge hits with a chance of about m_f / E, so early exit saves little below 1/32).
            // Two searches on a symmetrised R-MAT of 5M vertices, 8 blocks: a line at 1/2 to 1/64 of the
            // edges to scan 2,291 to 2,327 us, at all of them (never) 4,158, none (always) 2,505; streaming
            // below 1/4 to 1/16 of the edges 2,590, 1/32 2,324, 1/64 and 1/128 2,190, always 2,426, never 2,589
            if (blk_grid > 0 && m_u * 4.0 > (double)g->E)
                k_bfs_block_smem<<<blk_grid, BLK_THREADS, blk_smem, s>>>(
                    part->rowptr.as<int32_t>(), part->colidx.as<int32_t>(), part->id_map.as<int32_t>(), part->R,
                    part->blk_rows_dev.as<int64_t>(), part->B, part->W, nwords, front, visited,
                    part->rowbits.as<uint32_t>(), cnt + 2, m_f * 32.0 < (double)g->E ? 1 : 0);
            else
                k_bfs_block_level<<<grid, BFS_THREADS, 0, s>>>(part->rowptr.as<int32_t>(), part->colidx.as<int32_t>(),
                                                               part->id_map.as<int32_t>(), part->R, front, visited,
                                                               part->rowbits.as<uint32_t>());
            k_bfs_merge<<<part->nranges, BFS_THREADS, merge_smem, s>>>(part->rowbits.as<uint32_t>(),
                                                                       part->id_map.as<int32_t>(),
                                                                       part->merge_off.as<int32_t>(), part->B,
                                                                       part->nranges, part->k, V, nwords, next,
                                                                       visited, level, lvl + 1, cnt,
                                                                       g->out_rowptr.as<int32_t>(), merge_split);
            ++tocab_levels;
            have_queue = false;
        } else {
            k_bfs_pull_level<<<grid, BFS_THREADS, 0, s>>>(g->in_rowptr.as<int32_t>(), g->in_colidx.as<int32_t>(), V,
                                                          nwords, front, next, visited, level, lvl + 1, cnt,
                                                          g->out_rowptr.as<int32_t>());
            have_queue = false;
        }
        if (lev[1]) cudaEventRecord(lev[1], s);
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(h_cnt, cnt, 16, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) { st = fail(TC_ERR_CUDA, "bfs level %d: %s", lvl, cudaGetErrorString(e)); break; }
        front_count = h_cnt[0];
        m_f = (double)h_cnt[1];
        m_u -= m_f;
        if (lev[1] && lvl < TC_BFS_TRACE) cudaEventElapsedTime(&stats->level_ms[lvl], lev[0], lev[1]);
        ++lvl;
    }
    if (lev[0]) {
        cudaEventDestroy(lev[0]);
        cudaEventDestroy(lev[1]);
    }
    TC_TRY(st);
    if (bp->profile) {
        TC_CUDA(cudaEventRecord(ev[1], s));
        TC_CUDA(cudaEventSynchronize(ev[1]));
        TC_CUDA(cudaEventElapsedTime(&ms_total, ev[0], ev[1]));
        cudaEventDestroy(ev[0]);
        cudaEventDestroy(ev[1]);
    }
    if (stats) {
        TC_CUDA(cudaMemsetAsync(cnt, 0, 16, s));
        k_bfs_stats<<<grid, BFS_THREADS, 0, s>>>(level, g->out_rowptr.as<int32_t>(), V, cnt);
        TC_LAUNCH_CHECK();
        unsigned long long hs[2];
        TC_CUDA(cudaMemcpyAsync(hs, cnt, 16, cudaMemcpyDeviceToHost, s));
        TC_CUDA(cudaStreamSynchronize(s));
        stats->levels = lvl;
        stats->tocab_levels = tocab_levels;
        stats->push_levels = push_levels;
        stats->resident_levels = resident_levels;
        stats->reached = (int64_t)hs[0];
        stats->edges_reached = (int64_t)hs[1];
        stats->ms_total = ms_total;
    }
    if (bp->out_mem == TC_MEM_HOST) {
        TC_CUDA(cudaMemcpyAsync(levels_out, level, (size_t)V * 4, cudaMemcpyDeviceToHost, s));
        TC_CUDA(cudaStreamSynchronize(s));
    }
    return TC_OK;
}

}  // namespace tc

extern "C" int tc_bfs_pull(const tc_graph *g, const tc_part *part, int32_t source, const tc_bfs_params *params,
                           int32_t *levels_out, tc_bfs_stats *stats, void *stream) {
    using namespace tc;
    if (!g || !params || !levels_out) return fail(TC_ERR_INVALID_ARG, "tc_bfs_pull: null graph, params or output");
    if (source < 0 || source >= g->V) return fail(TC_ERR_INVALID_ARG, "tc_bfs_pull: source outside [0, V)");
    if (params->out_mem != TC_MEM_HOST && params->out_mem != TC_MEM_DEVICE)
        return fail(TC_ERR_INVALID_ARG, "tc_bfs_pull: bad out_mem");
    if (part && (part->g != g || part->dir != TC_PULL))
        return fail(TC_ERR_INVALID_ARG, "tc_bfs_pull: partition must be a TC_PULL partition of this graph");
    if (params->resident_edges > TC_BFS_RESIDENT_MAX)
        return fail(TC_ERR_INVALID_ARG, "tc_bfs_pull: resident_edges above %d", TC_BFS_RESIDENT_MAX);
    if (part && part->order != TC_ORDER_NATURAL)
        return fail(TC_ERR_UNSUPPORTED, "tc_bfs_pull: renumbered (TC_ORDER_OUTDEGREE) partitions are not supported");
    if (stats) memset(stats, 0, sizeof(*stats));
    return bfs_impl(g, part, source, params, levels_out, stats, (cudaStream_t)stream);
}
