// Staged push scatter: Alg. 5 with each block's destination range held in shared memory.
//
// A TC_PUSH partition cuts the destinations into ranges of W vertices (Sec. 3.1, Fig. 3 with
// the roles of rows and columns swapped); the paper keeps a block's range of `sums` resident in
// L2 and adds every edge's contribution there with a global atomic.  When the range fits in
// shared memory (W * 8 bytes), a CTA instead adds a slice of the block's edges into a shared
// copy of the range and then adds each nonzero sum of the copy to global memory once: the
// per-edge reductions become shared-memory atomics, and the global ones drop from one per edge
// to at most one per destination per CTA.
//
// Fixed-point sums go further: whatever the partition's block width, the library cuts the edges into
// destination ranges that fit shared memory and fuses the scatter with the rank update (k_push_cut).
//
// Sums are 64-bit fixed-point integers (exact in any order, so the ranks repeat bit for bit) or,
// in the paper's form, FP32 (order-dependent rounding).
#include <algorithm>
#include <vector>

#include "tc_common_dev.cuh"
#include "tc_walk.cuh"

namespace tc {

constexpr int PS_THREADS = 1024;

// Widest destination range whose 8-byte sums fit one CTA's shared memory (a multiple of 32).
int32_t push_smem_width(int max_smem_optin) {
    int64_t W = ((int64_t)max_smem_optin - 1024) / 8;
    W = W / 32 * 32;
    return W > 0 ? (int32_t)W : 0;
}

// Adds x to the 64-bit sum lo + 2^32 hi: the low half's carry comes from the value its atomic returns.
// A 64-bit shared atomic is a compare-and-swap loop on this GPU; the contributions' high half is mostly
// zero, which leaves one native 32-bit add per edge.
__device__ __forceinline__ void ps_add64(uint32_t *lo, uint32_t *hi, unsigned long long x) {
    const uint32_t xl = (uint32_t)x;
    uint32_t xh = (uint32_t)(x >> 32);
    const uint32_t old = atomicAdd(lo, xl);
    xh += (uint32_t)(old + xl < old);
    if (xh) atomicAdd(hi, xh);
}

// One CTA per tile (block b, edges [e0, e1)): shared sums of the block's range, then one global
// addition per nonzero entry.  scalef: the fixed-point scale (FIXED only).
template <bool FIXED>
__global__ void __launch_bounds__(PS_THREADS, 1) k_push_smem(const int4 *__restrict__ tiles,
                                                             const int32_t *__restrict__ esrc,
                                                             const int32_t *__restrict__ dst, int32_t W, int32_t V,
                                                             const float *__restrict__ contrib, void *sums,
                                                             const float *fx_scale) {
    extern __shared__ __align__(16) unsigned char psm[];
    uint32_t *acc_lo = reinterpret_cast<uint32_t *>(psm);  // FIXED: [W] low halves, [W] high halves
    uint32_t *acc_hi = acc_lo + W;
    float *acc32 = reinterpret_cast<float *>(psm);
    const int4 t = tiles[blockIdx.x];
    const int64_t lo = (int64_t)t.x * W;
    const int32_t w = (int32_t)(((int64_t)V - lo) < W ? ((int64_t)V - lo) : W);
    const int64_t e0 = ((int64_t)t.z << 31) | (uint32_t)t.y;  // 62-bit edge bounds split in two ints
    const int64_t e1 = e0 + (uint32_t)t.w;
    const float scalef = FIXED ? *fx_scale * 0x1p-6f : 1.0f;  // |sum| < 2^55
    for (int32_t v = threadIdx.x; v < w; v += PS_THREADS) {
        acc_lo[v] = 0u;  // the bits of 0.0f too
        if (FIXED) acc_hi[v] = 0u;
    }
    __syncthreads();
    int64_t i = e0 + threadIdx.x;
    for (; i + 3 * PS_THREADS < e1; i += 4 * PS_THREADS) {  // four edges in flight per thread
        int32_t sv[4], dv[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            sv[k] = __ldg(esrc + i + k * PS_THREADS);
            dv[k] = (int32_t)(__ldg(dst + i + k * PS_THREADS) - lo);
        }
        float cv[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) cv[k] = __ldg(contrib + sv[k]);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (cv[k] == 0.0f) continue;
            if (FIXED) ps_add64(acc_lo + dv[k], acc_hi + dv[k], fx_round64(cv[k] * scalef));
            else atomicAdd(acc32 + dv[k], cv[k]);
        }
    }
    for (; i < e1; i += PS_THREADS) {
        const float c = __ldg(contrib + __ldg(esrc + i));
        if (c == 0.0f) continue;
        const int32_t d = (int32_t)(__ldg(dst + i) - lo);
        if (FIXED) ps_add64(acc_lo + d, acc_hi + d, fx_round64(c * scalef));
        else atomicAdd(acc32 + d, c);
    }
    __syncthreads();
    for (int32_t v = threadIdx.x; v < w; v += PS_THREADS) {
        if (FIXED) {
            const unsigned long long x = ((unsigned long long)acc_hi[v] << 32) | acc_lo[v];
            if (x) atomicAdd(static_cast<unsigned long long *>(sums) + lo + v, x);
        } else {
            const float x = acc32[v];
            if (x != 0.0f) atomicAdd(static_cast<float *>(sums) + lo + v, x);
        }
    }
}

// Tiles of the staged push: block b's edges cut into n_b = max(1, round(E_b / T)) equal slices,
// T = E / (three waves of one CTA per SM); the largest blocks' tiles first.
int build_push_tiles(tc_part *p, int sms, cudaStream_t s) {
    p->nptiles = 0;
    if (p->E == 0) return TC_OK;
    TC_CUDA(cudaStreamSynchronize(s));  // the host copies of the block bounds
    const int64_t T = p->E / (3LL * sms) > 0 ? p->E / (3LL * sms) : 1;
    std::vector<int4> h;
    std::vector<int64_t> cost;
    for (int32_t b = 0; b < p->B; ++b) {
        const int64_t eb = p->h_blk_edges[b + 1] - p->h_blk_edges[b];
        if (eb == 0) continue;
        int64_t n = (eb + T / 2) / T;
        if (n < 1) n = 1;
        for (int64_t k = 0; k < n; ++k) {
            const int64_t a = p->h_blk_edges[b] + eb * k / n, z = p->h_blk_edges[b] + eb * (k + 1) / n;
            if (z - a > INT32_MAX) return fail(TC_ERR_UNSUPPORTED, "build_push_tiles: a tile over 2^31 edges");
            h.push_back(make_int4(b, (int32_t)(a & 0x7fffffff), (int32_t)(a >> 31), (int32_t)(z - a)));
            cost.push_back(z - a);
        }
    }
    std::vector<int32_t> order(h.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = (int32_t)i;
    std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) { return cost[x] > cost[y]; });
    std::vector<int4> hs(h.size());
    for (size_t i = 0; i < order.size(); ++i) hs[i] = h[(size_t)order[i]];
    TC_TRY(p->ptiles.alloc(hs.size() * sizeof(int4)));
    TC_CUDA(cudaMemcpyAsync(p->ptiles.p, hs.data(), hs.size() * sizeof(int4), cudaMemcpyHostToDevice, s));
    TC_CUDA(cudaStreamSynchronize(s));  // hs is freed at return
    p->nptiles = (int32_t)hs.size();
    return TC_OK;
}

int launch_push_smem(const tc_part *p, const float *contrib, void *sums, const float *fx_scale, bool fixed,
                     cudaStream_t s) {
    if (p->nptiles == 0) return TC_OK;
    const size_t smem = (size_t)p->W * (fixed ? 8 : 4);
    const void *k = fixed ? (const void *)k_push_smem<true> : (const void *)k_push_smem<false>;
    TC_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (fixed)
        k_push_smem<true><<<p->nptiles, PS_THREADS, smem, s>>>(p->ptiles.as<int4>(), p->esrc.as<int32_t>(),
                                                               p->colidx.as<int32_t>(), p->W, p->V, contrib, sums,
                                                               fx_scale);
    else
        k_push_smem<false><<<p->nptiles, PS_THREADS, smem, s>>>(p->ptiles.as<int4>(), p->esrc.as<int32_t>(),
                                                                p->colidx.as<int32_t>(), p->W, p->V, contrib, sums,
                                                                fx_scale);
    TC_LAUNCH_CHECK();
    return TC_OK;
}

// ---------------------------------------------------------------------------------------------
// Push iteration by destination ranges, scatter and update in one kernel.
// ---------------------------------------------------------------------------------------------
// For fixed-point sums the library cuts the edges of a push partition once more, into ranges of cut_W
// destinations whose sums fit a share of shared memory, whatever the partition's own block width is
// (sums are exact integers, so the order of the edges does not show).  Edges keep their source order
// inside a range, so neighbouring lanes mostly read the same or nearby contributions.
//
// A CTA scatters one tile (a range's edges, or a slice of them) into shared sums.  A range with one tile
// is finished there: its ranks, next contributions and dangling mass come straight from shared memory.
// The tiles of a range with more edges add their sums to `sums` in global memory, and the last one to
// arrive finishes the range (and zeroes its sums again).
//
// What bounds it: the L1 requests for the contributions of distinct sources (some 15 lines per 32 edges
// at R-MAT skew; L1 68%, L2 59% busy), next to one shared atomic per edge.  Wider ranges mean fewer distinct
// sources, but the lines of requests in flight need L1 too, so two CTAs of 1024 threads share an SM with at
// most CUT_WIDTH * 8 bytes each.  Lanes take consecutive edges: four per lane as one wide load spread a
// warp's sources over four times the lines (204 against 184 us per iteration).
// 20 iterations on R-MAT 22: 11,790 us by global 64-bit atomics and a separate update; 7,850 us with one
// wide range per SM, 3,980 us with ranges of 7,168, 3,670 us so.  6.9M-vertex R-MAT: 22.5 to 6.8 ms; R-MAT
// 16: 487 to 360 us; 3M uniform: 7.4 to 2.9 ms.
constexpr int CUT_WIDTH = 11264;

__device__ __forceinline__ int32_t ld_stream(const int32_t *p) {  // read once: not kept in L1
    int32_t r;
    asm("ld.global.nc.L1::no_allocate.s32 %0, [%1];" : "=r"(r) : "l"(p));
    return r;
}
__device__ __forceinline__ uint32_t ld_stream(const uint16_t *p) {
    uint16_t r;
    asm("ld.global.nc.L1::no_allocate.u16 %0, [%1];" : "=h"(r) : "l"(p));
    return r;
}

// The fixed-point total of a vertex as FP32 (|tot| < 2^55), without FP64.
__device__ __forceinline__ float cut_float(unsigned long long u) {
    const long long tot = (long long)u;
    return fmaf((float)(int32_t)(tot >> 24), 16777216.0f, (float)(uint32_t)(tot & 0xFFFFFFll));
}

__global__ void __launch_bounds__(PS_THREADS, 2) k_push_cut(const int4 *__restrict__ tiles,
                                                            const int32_t *__restrict__ src,
                                                            const uint16_t *__restrict__ dst, PushCutArgs a) {
    extern __shared__ __align__(16) unsigned char psm[];
    uint32_t *acc_lo = reinterpret_cast<uint32_t *>(psm);
    uint32_t *acc_hi = acc_lo + a.W;
    __shared__ bool s_last;
    const int4 t = tiles[blockIdx.x];  // (range, first edge, end edge, tiles of the range)
    const int32_t lo = t.x * a.W;
    const int32_t w = a.V - lo < a.W ? a.V - lo : a.W;
    for (int32_t v = threadIdx.x; v < w; v += PS_THREADS) {
        acc_lo[v] = 0u;
        acc_hi[v] = 0u;
    }
    const float scalef = *a.fx_scale * 0x1p-6f;  // |sum| < 2^55
    __syncthreads();
    // a lane's edges are 32 apart: consecutive edges, whose sources are close, share a load
    walk_batched<4, PS_THREADS>(
        (uint32_t)t.y + threadIdx.x, (uint32_t)t.z,
        [&](uint32_t i) {
            int32_t sv[4];
            uint32_t dv[4];
            float cv[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                sv[k] = ld_stream(src + i + k * PS_THREADS);
                dv[k] = ld_stream(dst + i + k * PS_THREADS);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) cv[k] = __ldg(a.contrib + sv[k]);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (cv[k] != 0.0f) ps_add64(acc_lo + dv[k], acc_hi + dv[k], fx_round64(cv[k] * scalef));
        },
        [&](uint32_t i) {
            const uint32_t d = ld_stream(dst + i);
            const float c = __ldg(a.contrib + ld_stream(src + i));
            if (c != 0.0f) ps_add64(acc_lo + d, acc_hi + d, fx_round64(c * scalef));
        });
    __syncthreads();
    const bool shared_range = t.w > 1;
    if (shared_range) {
        for (int32_t v = threadIdx.x; v < w; v += PS_THREADS) {
            const unsigned long long x = ((unsigned long long)acc_hi[v] << 32) | acc_lo[v];
            if (x) atomicAdd(a.sums + lo + v, x);
        }
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) s_last = atomicAdd(a.range_count + t.x, 1) == t.w - 1;
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        if (threadIdx.x == 0) a.range_count[t.x] = 0;
    }
    const float spread = a.drop ? 0.0f : *a.S_cur;
    const float inv_scalef = 1.0f / scalef;  // a power of two
    DanglingSum dangling;
    for (int32_t v = threadIdx.x; v < w; v += PS_THREADS) {
        unsigned long long x;
        if (shared_range) {
            x = __ldcg(a.sums + lo + v);
            a.sums[lo + v] = 0ull;
        } else {
            x = ((unsigned long long)acc_hi[v] << 32) | acc_lo[v];
        }
        const float r = a.base + a.damping * (cut_float(x) * inv_scalef + spread);
        if (a.rank_out) a.rank_out[lo + v] = r;
        const float inv = __ldg(a.inv_outdeg + lo + v);
        a.contrib_next[lo + v] = r * inv;
        if (inv == 0.0f) dangling.add(r, scalef, inv_scalef);
    }
    dangling.finish(t.x, a.B, a.dslot, a.drest, a.counter, scalef, a.D_next, a.spread);
}

// First edge of every range (keys ascending by range, n of them), b in [0, B].
__global__ void k_cut_bounds(const int32_t *__restrict__ key, int64_t n, int32_t W, int32_t B, int64_t *out) {
    for (int32_t b = blockIdx.x * blockDim.x + threadIdx.x; b <= B; b += gridDim.x * blockDim.x) {
        int64_t lo = 0, hi = n;
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if ((int64_t)key[mid] < (int64_t)b * W) lo = mid + 1; else hi = mid;
        }
        out[b] = lo;
    }
}

__global__ void k_cut_offsets(const int32_t *__restrict__ key, int64_t n, DivBy W, int32_t Wi, uint16_t *out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t d = key[i];
        out[i] = (uint16_t)(d - div_apply(d, W) * Wi);
    }
}

static int build_push_cut(tc_part *p, cudaStream_t s) {
    DeviceCaps caps;
    TC_TRY(device_caps(&caps));
    const int64_t E = p->E, V = p->V;
    // two CTAs per SM, as few whole waves of equal ranges as CUT_WIDTH allows, with a sixteenth of the
    // slots left for the ranges cut into slices
    const int64_t slots = 2LL * caps.sms * 15 / 16;
    const int64_t m = (V + slots * CUT_WIDTH - 1) / (slots * CUT_WIDTH);
    const int32_t W = (int32_t)(((V + slots * m - 1) / (slots * m) + 31) / 32 * 32);
    const int32_t B = (int32_t)((V + W - 1) / W);
    DevBuf keys, kt, vt, bounds;
    TC_TRY(p->cut_src.alloc((size_t)E * 4));
    TC_TRY(p->cut_dst.alloc((size_t)E * 2));
    TC_TRY(p->cut_count.alloc((size_t)B * 4));
    TC_TRY(keys.alloc((size_t)E * 4));
    TC_TRY(kt.alloc((size_t)E * 4));
    TC_TRY(vt.alloc((size_t)E * 4));
    TC_TRY(bounds.alloc(((size_t)B + 1) * 8));
    int bits = 1;
    while ((1LL << bits) < (int64_t)B) ++bits;
    TC_TRY(stable_bucket_sort(p->colidx.as<int32_t>(), p->esrc.as<int32_t>(), keys.as<int32_t>(),
                              p->cut_src.as<int32_t>(), kt.as<int32_t>(), vt.as<int32_t>(), E, W, bits, s));
    k_cut_bounds<<<(B + 256) / 256, 256, 0, s>>>(keys.as<int32_t>(), E, W, B, bounds.as<int64_t>());
    TC_LAUNCH_CHECK();
    k_cut_offsets<<<caps.sms * 8, 256, 0, s>>>(keys.as<int32_t>(), E, div_by(W), W, p->cut_dst.as<uint16_t>());
    TC_LAUNCH_CHECK();
    TC_CUDA(cudaMemsetAsync(p->cut_count.p, 0, (size_t)B * 4, s));
    std::vector<int64_t> eb((size_t)B + 1);
    TC_CUDA(cudaMemcpyAsync(eb.data(), bounds.p, ((size_t)B + 1) * 8, cudaMemcpyDeviceToHost, s));
    TC_CUDA(cudaStreamSynchronize(s));
    // a range of more than 3/2 of the mean edges is cut into equal slices of about the mean
    const int64_t T = E / B > 0 ? E / B : 1;
    std::vector<int4> h;
    for (int32_t b = 0; b < B; ++b) {
        const int64_t ne = eb[(size_t)b + 1] - eb[(size_t)b];
        const int64_t n = (ne + T / 2) / T > 1 ? (ne + T / 2) / T : 1;
        for (int64_t k = 0; k < n; ++k)
            h.push_back(make_int4(b, (int32_t)(eb[(size_t)b] + ne * k / n), (int32_t)(eb[(size_t)b] + ne * (k + 1) / n),
                                  (int32_t)n));
    }
    std::stable_sort(h.begin(), h.end(), [](const int4 &x, const int4 &y) { return x.z - x.y > y.z - y.y; });
    TC_TRY(p->cut_tiles.alloc(h.size() * sizeof(int4)));
    TC_CUDA(cudaMemcpyAsync(p->cut_tiles.p, h.data(), h.size() * sizeof(int4), cudaMemcpyHostToDevice, s));
    TC_CUDA(cudaStreamSynchronize(s));  // h is freed at return
    p->cut_W = W;
    p->cut_B = B;
    p->cut_ntiles = (int32_t)h.size();
    return TC_OK;
}

// The cut is built, and kept with the partition, by the call that brings the iterations asked of it to
// CUT_MIN_ITERS: building it takes as long as it saves in 2.2 to 2.8 iterations (16M to 110M edges; R-MAT 22
// 1,036 us, 578 against 184 us per iteration).  Small graphs pay some 125 us of launches and copies, saved in
// 24 iterations at 1M edges (21 against 16 us).  Not under a memory cap and not while the stream is
// captured, nor when its memory is not to be had: the scatter over the partition's own edges gives the same
// ranks bit for bit and needs none of it.
constexpr int64_t CUT_MIN_ITERS = 3;

int ensure_push_cut(tc_part *p, int32_t iters, cudaStream_t s) {
    if (p->cut_tried || p->E == 0 || p->smem_stage < 0) return TC_OK;
    p->push_iters += iters;
    if (iters == 0 || p->push_iters < CUT_MIN_ITERS || cache_get_limit()) return TC_OK;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return TC_OK;
    }
    p->cut_tried = true;
    const KeptError kept;
    const int st = build_push_cut(p, s);
    if (st == TC_OK) return TC_OK;
    cudaStreamSynchronize(s);
    for (DevBuf *d : {&p->cut_src, &p->cut_dst, &p->cut_count, &p->cut_tiles}) d->release();
    if (st != TC_ERR_OOM) return st;
    kept.restore();
    return TC_OK;
}

int launch_push_cut(const tc_part *p, PushCutArgs a, cudaStream_t s) {
    a.W = p->cut_W;
    a.B = p->cut_B;
    a.range_count = p->cut_count.as<int32_t>();
    const size_t smem = (size_t)a.W * 8;
    TC_CUDA(cudaFuncSetAttribute(k_push_cut, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_push_cut<<<p->cut_ntiles, PS_THREADS, smem, s>>>(p->cut_tiles.as<int4>(), p->cut_src.as<int32_t>(),
                                                       p->cut_dst.as<uint16_t>(), a);
    TC_LAUNCH_CHECK();
    return TC_OK;
}

}  // namespace tc
