// Device helpers shared by the iteration kernels: block reductions and the
// "last CTA finishes the reduction" pattern used for the dangling rank mass.
#pragma once
#include "tc_internal.cuh"

namespace tc {

// ---- PTX helpers: mbarrier and bulk asynchronous copies -------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait: gives up after ~2^31 cycles (about a second), records `code` in *err.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, int *err, int code) {
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (clock64() - t0 > (1LL << 31)) {
            atomicCAS(err, 0, code);
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

// Bulk store shared -> global (TMA unit), one per call, committed as its own group; both
// addresses 16-byte aligned and the size a multiple of 16.
__device__ __forceinline__ void bulk_store_s2g(void *gdst, const void *ssrc, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gdst), "r"(smem_addr(ssrc)),
                 "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// Waits until this thread's bulk stores have read their shared-memory sources.
__device__ __forceinline__ void bulk_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
// Waits until this thread's bulk stores are complete.
__device__ __forceinline__ void bulk_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// Orders this thread's generic-proxy shared-memory writes before later bulk-copy reads.
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Programmatic dependent launch: a kernel launched with the programmatic stream serialization
// attribute may start while the previous kernel in the stream finishes; pdl_wait() blocks until
// that kernel has completed and its writes are visible (a no-op without the attribute), and
// pdl_trigger() lets the next kernel start launching.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }


// Sum over the block in a fixed tree order (deterministic for a fixed launch shape).
// All threads must call it; the result is valid in every thread.
template <class T>
__device__ __forceinline__ T block_sum(T x, T *smem /* >= 32 entries */) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) x += __shfl_down_sync(0xffffffffu, x, d);
    __syncthreads();
    if (lane == 0) smem[warp] = x;
    __syncthreads();
    T t = 0;
    if (warp == 0) {
        t = lane < nw ? smem[lane] : T(0);
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) t += __shfl_down_sync(0xffffffffu, t, d);
        if (lane == 0) smem[0] = t;
    }
    __syncthreads();
    t = smem[0];
    __syncthreads();
    return t;
}

// D / V as the next kernel's threads use it, written beside D by the thread that writes D: this GPU has
// so little FP64 throughput that a division in every thread showed (20 pull iterations on R-MAT 16: 528
// to 501 us without it and without the FP64 steps that scaled the sums).
struct SpreadOut {
    float *out = nullptr;  // null: not wanted
    int32_t V = 1;
    __device__ __forceinline__ void write(double D) const {
        if (out) *out = (float)(D / (double)V);
    }
};

// Every CTA contributes `mine` (valid in thread 0); the last CTA to arrive sums all the
// contributions in CTA order and stores the total plus `extra` to *out, then re-arms the counter.
__device__ __forceinline__ void grid_sum_last_cta(double mine, double *part, unsigned *counter, double *out,
                                                  double extra = 0.0, SpreadOut spread = SpreadOut()) {
    __shared__ bool am_last;
    __shared__ double red[32];
    if (threadIdx.x == 0) {
        part[blockIdx.x] = mine;
        __threadfence();
        const unsigned ticket = atomicAdd(counter, 1u);
        am_last = (ticket == gridDim.x - 1);
    }
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    double t = 0.0;
    for (unsigned i = threadIdx.x; i < gridDim.x; i += blockDim.x) t += __ldcg(part + i);
    t = block_sum<double>(t, red);
    if (threadIdx.x == 0) {
        *out = t + extra;
        spread.write(t + extra);
        *counter = 0u;
    }
}

// Every CTA has written its share into slots of part[0, nslots) (any CTA any slot); the last
// CTA to arrive sums the slots in slot order (deterministic whichever CTA filled which slot),
// stores the total to *out and re-arms the counter and *queue (a work queue the CTAs drew from,
// idle by now: every CTA drew its last item before arriving).  All threads must call it.
__device__ __forceinline__ void grid_sum_slots_last_cta(const double *part, int32_t nslots, unsigned *counter,
                                                        unsigned *queue, double *out, double extra,
                                                        SpreadOut spread) {
    __shared__ bool am_last3;
    __shared__ double red3[32];
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned ticket = atomicAdd(counter, 1u);
        am_last3 = (ticket == gridDim.x - 1);
    }
    __syncthreads();
    if (!am_last3) return;
    __threadfence();
    double t = 0.0;
    for (int32_t i = threadIdx.x; i < nslots; i += blockDim.x) t += __ldcg(part + i);
    t = block_sum<double>(t, red3);
    if (threadIdx.x == 0) {
        *out = t + extra;
        spread.write(t + extra);
        *counter = 0u;
        *queue = 0u;
    }
}

// Two sums at once (a in x, b in y), same protocol as grid_sum_last_cta.
// Returns true in every thread of the last CTA (after the sums are written).
__device__ __forceinline__ bool grid_sum2_last_cta(double a, double b, double *part /* 2 per CTA */,
                                                   unsigned *counter, double *out_a, double *out_b) {
    __shared__ bool am_last2;
    __shared__ double red2[32];
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = a;
        part[2 * blockIdx.x + 1] = b;
        __threadfence();
        const unsigned ticket = atomicAdd(counter, 1u);
        am_last2 = (ticket == gridDim.x - 1);
    }
    __syncthreads();
    if (!am_last2) return false;
    __threadfence();
    double ta = 0.0, tb = 0.0;
    for (unsigned i = threadIdx.x; i < gridDim.x; i += blockDim.x) {
        ta += __ldcg(part + 2 * i);
        tb += __ldcg(part + 2 * i + 1);
    }
    ta = block_sum<double>(ta, red2);
    tb = block_sum<double>(tb, red2);
    if (threadIdx.x == 0) {
        *out_a = ta;
        *out_b = tb;
        *counter = 0u;
    }
    return true;
}

// round(y) as a 64-bit two's-complement integer for |y| < 2^62, from the FP32 bits (integer
// operations only: 64-bit float-to-integer conversions run on the FP64 unit).
__device__ __forceinline__ unsigned long long fx_round64(float y) {
    const uint32_t b = __float_as_uint(y);
    const uint32_t a = b & 0x7fffffffu;
    const int e = (int)(a >> 23);
    const unsigned long long m = (a & 0x7fffffu) | (e ? 0x800000u : 0u);
    const int sh = (e ? e : 1) - 150;  // |y| = m * 2^sh
    unsigned long long r;
    if (sh >= 0) r = m << sh;
    else if (sh <= -25) r = 0ull;
    else r = (m + (1ull << (-sh - 1))) >> (-sh);  // to nearest, ties away from zero
    return (b >> 31) ? (0ull - r) : r;
}

// The last CTA's part of DanglingSum, a call of its own: inlined, its FP64 arithmetic cost k_push_update the
// registers of three CTAs per SM (46 instead of 32 per thread; R-MAT 22, 130 to 144 us).
static __device__ __noinline__ void dangling_total(int32_t n, const unsigned long long *slot, const double *rest,
                                                   unsigned *counter, float scalef, double *D, SpreadOut spread) {
    __shared__ unsigned long long red5[32];
    __shared__ double redd5[32];
    __threadfence();
    unsigned long long t = 0;
    double z = 0.0;
    for (int32_t k = threadIdx.x; k < n; k += blockDim.x) {
        t += __ldcg(slot + k);
        const double x = __ldcg(rest + k);
        if (__double_as_longlong(x) != 0ll) z += x;  // (an FP64 addition is slow here)
    }
    t = block_sum<unsigned long long>(t, red5);
    if (__syncthreads_or(__double_as_longlong(z) != 0ll)) z = block_sum<double>(z, redd5);
    if (threadIdx.x == 0) {
        const double d = (double)(long long)t / (double)scalef + z;
        *D = d;
        spread.write(d);
        *counter = 0u;
    }
}

// The dangling mass of a push iteration in fixed point (`scalef` per unit).  A thread adds its vertices to
// a DanglingSum; all threads of the CTA call finish(i): the CTA's sum goes to slot[i] and rest[i], and the
// last of n arrivals adds the slots and writes D and D / V.  Integers: the same for any division of the
// vertices among CTAs.  What the fixed point does not hold is summed beside it in FP32, with the CTAs' sums
// in FP64: ranks that are not finite, and the fractions of ranks below 2^-32 of the caller's L1 mass (the
// ranks themselves below 2^-56 of it), which are all there is when the dangling vertices hold next to
// nothing of a large mass.
struct DanglingSum {
    unsigned long long t = 0;
    float odd = 0.0f;
    __device__ __forceinline__ void add(float r, float scalef, float inv_scalef) {
        const float y = r * scalef, a = fabsf(y);
        if (a >= 0x1p23f && a < 0x1p62f) {  // a whole number: no rounding
            const uint32_t b = __float_as_uint(y);
            const unsigned long long u = (unsigned long long)((b & 0x7fffffu) | 0x800000u) << (((b >> 23) & 0xffu) - 150u);
            t += (b >> 31) ? 0ull - u : u;
        } else if (a < 0x1p23f) {
            const int32_t u = __float2int_rn(y);
            t += (unsigned long long)(long long)u;
            odd += r - (float)u * inv_scalef;  // exact
        } else {
            odd += r;
        }
    }
    __device__ __forceinline__ void finish(int32_t i, int32_t n, unsigned long long *slot, double *rest,
                                           unsigned *counter, float scalef, double *D, SpreadOut spread) {
        __shared__ bool am_last4;
        __shared__ unsigned long long red4[32];
        __shared__ float redf4[32];
        t = block_sum<unsigned long long>(t, red4);
        if (__syncthreads_or(odd != 0.0f)) odd = block_sum<float>(odd, redf4);
        if (threadIdx.x == 0) {
            slot[i] = t;
            rest[i] = (double)odd;
            __threadfence();
            am_last4 = atomicAdd(counter, 1u) == (unsigned)n - 1u;
        }
        __syncthreads();
        if (am_last4) dangling_total(n, slot, rest, counter, scalef, D, spread);
    }
};

// Appends to a queue in global memory, staged per warp in shared memory: `count` moves by one atomic
// per 32 entries (and one per CTA at the end) instead of one per entry or per warp step.  An atomic
// per entry on one address bounded the traversal levels that had it (BC from 4 sources on a
// symmetrised R-MAT 18, with the classes of a level in one launch: 2,552 to 1,698 us).  The entries' weights (out-degrees) are summed
// per lane and leave as one atomic per CTA.  All threads of the CTA call finish() once.
constexpr int WQ_ENTRIES = 64;  // per warp: below 32 entries wait, at most 32 arrive at once
struct WarpQueue {
    int32_t *buf;                // this warp's WQ_ENTRIES words of shared memory
    int32_t n = 0;               // entries waiting (warp-uniform)
    unsigned long long w = 0;    // this lane's weights
    __device__ explicit WarpQueue(int32_t *smem) : buf(smem + (threadIdx.x >> 5) * WQ_ENTRIES) {}
    // The whole warp calls it; lanes with `has` append v.
    __device__ __forceinline__ void push(bool has, int32_t v, int32_t weight, int32_t *queue, unsigned long long *count) {
        const int lane = threadIdx.x & 31;
        const unsigned m = __ballot_sync(0xffffffffu, has);
        if (m == 0u) return;
        if (has) {
            buf[n + __popc(m & ((1u << lane) - 1u))] = v;
            w += (unsigned long long)weight;
        }
        n += __popc(m);
        if (n < 32) return;
        __syncwarp();
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(count, 32ull);
        base = __shfl_sync(0xffffffffu, base, 0);
        queue[base + lane] = buf[lane];
        const int32_t rest = lane < n - 32 ? buf[32 + lane] : 0;
        __syncwarp();
        if (lane < n - 32) buf[lane] = rest;
        n -= 32;
        __syncwarp();
    }
    // The waiting entries of all warps, and the CTA's weights (added to *weight_sum).
    __device__ __forceinline__ void finish(int32_t *queue, unsigned long long *count, unsigned long long *weight_sum) {
        __shared__ int32_t wq_n[32];
        __shared__ unsigned long long wq_red[32], wq_base;
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
        const unsigned long long sum = block_sum<unsigned long long>(w, wq_red);
        if (lane == 0) wq_n[warp] = n;
        __syncthreads();
        if (threadIdx.x == 0) {
            int32_t t = 0;
            for (int i = 0; i < nw; ++i) {
                const int32_t x = wq_n[i];
                wq_n[i] = t;
                t += x;
            }
            wq_base = t > 0 ? atomicAdd(count, (unsigned long long)t) : 0ull;
            if (sum) atomicAdd(weight_sum, sum);
        }
        __syncthreads();
        if (lane < n) queue[wq_base + wq_n[warp] + lane] = buf[lane];
    }
};

// What the push iteration by destination ranges works on (tc_push.cu); the launch fills W, B and
// range_count from the partition.
struct PushCutArgs {
    float base, damping;          // (1-d)/V and d
    int drop;                     // 1: dangling mass is not redistributed
    int32_t V, W, B;              // vertices, width and number of the ranges
    const float *S_cur;           // D / V of the contributions read
    double *D_next;               // dangling mass of the ranks written, with D / V in `spread`
    SpreadOut spread;
    const float *inv_outdeg;
    const float *contrib;
    float *contrib_next;
    float *rank_out;              // may be null
    const float *fx_scale;
    unsigned long long *sums;     // zero between launches; ranges of several tiles meet there
    int32_t *range_count;
    unsigned long long *dslot;    // [B]
    double *drest;                // [B]
    unsigned *counter;
};
int launch_push_cut(const tc_part *p, PushCutArgs a, cudaStream_t s);

}  // namespace tc
