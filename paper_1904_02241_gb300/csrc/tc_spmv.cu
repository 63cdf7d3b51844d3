// Sparse matrix-vector product y = A x (the SpMV benchmark of Sec. 4, the generalised form of
// the graph operators): A is the CSR loaded as a graph's out-edges (row i = output i), with one
// FP32 value per stored entry in the loaded order.  Rows are mapped the way Sec. 3.2 bins
// them: a group of L lanes per row (L a power of two picked from the mean row length, so a row
// of about 16 entries does not leave 28 of a warp's lanes idle), and a CTA per hub row (more
// than the graph's hub degree, 2048 by default).  Each lane strides its row's entries
// (coalesced column and value loads, random gathers of x) and a fixed shuffle / shared-memory
// tree adds the lane sums, so the result does not depend on timing.  FP32 throughout.
#include <vector>

#include "tc_internal.cuh"
#include "tc_walk.cuh"

namespace tc {

constexpr int SP_THREADS = 256;

template <int L>
__global__ void __launch_bounds__(SP_THREADS) k_spmv_rows(const int32_t *__restrict__ rowptr,
                                                          const int32_t *__restrict__ colidx,
                                                          const float *__restrict__ vals,
                                                          const float *__restrict__ x, float *__restrict__ y,
                                                          int32_t nrows, int32_t hub_degree) {
    constexpr int G = 32 / L;  // rows per warp step
    const int lane = threadIdx.x & 31, sub = lane % L, grp = lane / L;
    const int64_t nw = (int64_t)gridDim.x * (SP_THREADS / 32);
    // every lane runs the same number of steps, so the shuffles below see the whole warp
    for (int64_t base = ((blockIdx.x * (int64_t)SP_THREADS + threadIdx.x) >> 5) * G; base < nrows; base += nw * G) {
        const int64_t r = base + grp;
        int32_t s = 0, e = 0;
        bool mine = false;  // a row of this kernel (not past the end, not a hub row)
        if (r < nrows) {
            s = __ldg(rowptr + r);
            e = __ldg(rowptr + r + 1);
            mine = e - s <= hub_degree;
            if (!mine) e = s;  // k_spmv_hub
        }
        float acc = 0.0f;
        for (int32_t k = s + sub; k < e; k += L) acc = fmaf(__ldg(vals + k), __ldg(x + __ldg(colidx + k)), acc);
#pragma unroll
        for (int d = L / 2; d > 0; d >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, d);
        if (sub == 0 && mine) y[r] = acc;
    }
}

// a CTA per hub row
__global__ void __launch_bounds__(SP_THREADS) k_spmv_hub(const int32_t *__restrict__ rowptr,
                                                         const int32_t *__restrict__ colidx,
                                                         const float *__restrict__ vals, const float *__restrict__ x,
                                                         float *__restrict__ y, const int32_t *__restrict__ hubs) {
    __shared__ float part[SP_THREADS / 32];
    const int32_t r = hubs[blockIdx.x];
    const int32_t s = rowptr[r], e = rowptr[r + 1];
    float acc = 0.0f;
    for (int32_t k = s + threadIdx.x; k < e; k += SP_THREADS) acc = fmaf(__ldg(vals + k), __ldg(x + __ldg(colidx + k)), acc);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, d);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.0f;
        for (int w = 0; w < SP_THREADS / 32; ++w) t += part[w];
        y[r] = t;
    }
}

}  // namespace tc

extern "C" int tc_spmv(const tc_graph *g, const float *vals, const float *x, float *y, int mem, void *stream) {
    using namespace tc;
    if (!g || !x || !y || (g->E > 0 && !vals)) return fail(TC_ERR_INVALID_ARG, "tc_spmv: null matrix, values or vector");
    if (mem != TC_MEM_DEVICE && mem != TC_MEM_HOST) return fail(TC_ERR_INVALID_ARG, "tc_spmv: bad mem");
    if (mem != TC_MEM_DEVICE) return fail(TC_ERR_UNSUPPORTED, "tc_spmv: vals, x and y must be device pointers");
    const int32_t V = g->V;
    if (V == 0) return TC_OK;
    DeviceCaps caps;
    TC_TRY(device_caps(&caps));
    cudaStream_t s = (cudaStream_t)stream;
    // lanes per row: the power of two nearest half the mean row length, 4 to 32
    const double mean = (double)g->E / (double)V;
    int L = 4;
    while (L < 32 && 2.0 * L < mean) L *= 2;
    const int64_t want = ((int64_t)V * L + SP_THREADS - 1) / SP_THREADS;
    const int grid = (int)(want < (int64_t)caps.sms * 16 ? (want > 0 ? want : 1) : (int64_t)caps.sms * 16);
    const int32_t *rp = g->out_rowptr.as<int32_t>(), *ci = g->out_colidx.as<int32_t>();
    const int32_t hd = g->hub_degree;
    switch (L) {
        case 4: k_spmv_rows<4><<<grid, SP_THREADS, 0, s>>>(rp, ci, vals, x, y, V, hd); break;
        case 8: k_spmv_rows<8><<<grid, SP_THREADS, 0, s>>>(rp, ci, vals, x, y, V, hd); break;
        case 16: k_spmv_rows<16><<<grid, SP_THREADS, 0, s>>>(rp, ci, vals, x, y, V, hd); break;
        default: k_spmv_rows<32><<<grid, SP_THREADS, 0, s>>>(rp, ci, vals, x, y, V, hd); break;
    }
    TC_LAUNCH_CHECK();
    if (g->num_out_hubs > 0) {
        k_spmv_hub<<<g->num_out_hubs, SP_THREADS, 0, s>>>(rp, ci, vals, x, y, g->out_hubs.as<int32_t>());
        TC_LAUNCH_CHECK();
    }
    return TC_OK;
}

// ---------------------------------------------------------------------------------------------
// GC-pull SpMV (Sec. 4's SpMV with TOCAB, a value stream of 4 B per entry): a TC_PUSH partition
// of the matrix's CSR cuts its columns into ranges of W (so x[block] is the block's working set,
// Sec. 3.1 with the value read from x instead of the contributions); each (block, row) piece is a
// local row whose partial sum goes to partial[], and the merge of Fig. 5 adds a row's pieces in
// block order into y.  FP32; deterministic (a fixed order everywhere).
// ---------------------------------------------------------------------------------------------
namespace tc {

__global__ void k_iota(int64_t n, int32_t *out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (int32_t)i;
}

__global__ void k_gather_vals(const int32_t *__restrict__ perm, const float *__restrict__ vals, int64_t n,
                              float *__restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = vals[perm[i]];
}

// Local rows: a lane each below 32 entries (in order), a warp each from 32 (lane strides in
// order, then a fixed shuffle tree).
__global__ void __launch_bounds__(SP_THREADS) k_spmv_block_rows(const int32_t *__restrict__ rowptr,
                                                                const int32_t *__restrict__ colidx,
                                                                const float *__restrict__ pvals,
                                                                const float *__restrict__ x, int64_t R,
                                                                float *__restrict__ partial) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (SP_THREADS / 32);
    for (int64_t grp = (blockIdx.x * (int64_t)SP_THREADS + threadIdx.x) >> 5; grp * 32 < R; grp += nw) {
        const int64_t r = grp * 32 + lane;
        int32_t s = 0, e = 0;
        if (r < R) {
            s = __ldg(rowptr + r);
            e = __ldg(rowptr + r + 1);
        }
        float acc = 0.0f;
        if (e - s < 32)
            for (int32_t k = s; k < e; ++k) acc = fmaf(__ldg(pvals + k), __ldg(x + __ldg(colidx + k)), acc);
        unsigned long_rows = __ballot_sync(0xffffffffu, e - s >= 32);
        while (long_rows) {
            const int l = __ffs(long_rows) - 1;
            long_rows &= long_rows - 1;
            const int32_t ls = __shfl_sync(0xffffffffu, s, l), le = __shfl_sync(0xffffffffu, e, l);
            float w = 0.0f;
            for (int32_t k = ls + lane; k < le; k += 32) w = fmaf(__ldg(pvals + k), __ldg(x + __ldg(colidx + k)), w);
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) w += __shfl_xor_sync(0xffffffffu, w, d);
            if (lane == l) acc = w;
        }
        if (r < R) partial[r] = acc;
    }
}

// Fig. 5: CTA j owns rows [j k, (j+1) k); it adds block b's slice for b = 0, 1, ... in order (the
// rows of one slice are distinct, so its threads never collide), then writes y.
__global__ void __launch_bounds__(SP_THREADS) k_spmv_merge(const float *__restrict__ partial,
                                                           const int32_t *__restrict__ id_map,
                                                           const int32_t *__restrict__ merge_off, int32_t B,
                                                           int32_t nranges, int32_t k, int32_t V, float *y) {
    extern __shared__ float macc[];  // [k]
    for (int32_t j = blockIdx.x; j < nranges; j += gridDim.x) {
        const int32_t vbase = j * k;
        for (int32_t t = threadIdx.x; t < k; t += SP_THREADS) macc[t] = 0.0f;
        __syncthreads();
        for (int32_t b = 0; b < B; ++b) {
            const int32_t *o = merge_off + (int64_t)b * (nranges + 1) + j;
            const int32_t r0 = __ldg(o), r1 = __ldg(o + 1);
            for (int32_t r = r0 + threadIdx.x; r < r1; r += SP_THREADS) macc[__ldg(id_map + r) - vbase] += __ldg(partial + r);
            __syncthreads();
        }
        for (int32_t t = threadIdx.x; t < k && vbase + t < V; t += SP_THREADS) y[vbase + t] = macc[t];
        __syncthreads();
    }
}

// Staged GC-pull.  With blocks of x that only fit the L2, an entry costs a random L2 request, and those
// come at some 190 G/s whatever the order of the rows.  So from SPM_MIN_ENTRIES entries on (below, a product
// gains 8 to 20 of 36 to 50 us, and setting the values takes some 500 us longer), where it pays, the values get a finer cut of the matrix whose blocks of x
// fit one CTA's shared memory, in the staged form of the rank gather (tc_tile.cu) with a value per entry:
// the entries stream at 6 B each and x is read in shared memory.
// More pieces come with it, so their merge is a kernel of its own.  R-MAT 22, 8 blocks: 404 us the general
// way; 129 us for the staged gather and 95 us for the merge, whose 64-bit shared reads and writes at random
// rows bound it (bank conflicts).  R-MAT of 131,072 rows, 16 blocks: 57 to 32 us.
//
// CTA j owns rows [j k, (j+1) k).  The order is the same fixed one as k_spmv_merge's, block after block
// with a barrier, but a thread's entries (SPAN per block) of the next DEPTH blocks load while those of
// the DEPTH blocks before are added.
// There are several times the pieces of the loaded blocks, so the additions are compensated (the error of
// every one, by Knuth's TwoSum, is added up beside the sum): without it y was further from the exact
// product than with eight blocks (R-MAT 22: 1.7e-7 against 9.9e-8 in the 2-norm).
constexpr int SPM_THREADS = 512;
constexpr int64_t SPM_MIN_ENTRIES = 1 << 20;
// Pieces are walked with signed 32-bit positions (with unsigned ones the walk past SPAN took R-MAT 23 in 16
// blocks from 498 to 617 us), which a thread takes at most this far past the last piece.
constexpr int SPM_PAST = 6 * SPM_THREADS;
__device__ __forceinline__ void spm_add(float2 *acc, float v) {  // x: the sum, y: its error
    const float2 a = *acc;
    const float t = a.x + v;
    const float z = t - a.x;
    *acc = make_float2(t, a.y + ((a.x - (t - z)) + (v - z)));
}
template <int DEPTH, int SPAN>
__global__ void __launch_bounds__(SPM_THREADS, DEPTH * SPAN <= 4 ? 4 : 2) k_spmv_merge_staged(const float *__restrict__ partial,
                                                                   const uint16_t *__restrict__ id16,
                                                                   const int32_t *__restrict__ offT, int32_t B,
                                                                   int32_t k, int32_t V, const int *err, float *y) {
    extern __shared__ float2 sacc[];  // [k], then block b's rows of the range, [off[b], off[B + b])
    int32_t *off = reinterpret_cast<int32_t *>(sacc + k);
    const int32_t j = blockIdx.x;
    for (int32_t t = threadIdx.x; t < k; t += SPM_THREADS) sacc[t] = make_float2(0.0f, 0.0f);
    for (int32_t b = threadIdx.x; b < 2 * B; b += SPM_THREADS) off[b] = __ldg(offT + (int64_t)j * B + b);
    __syncthreads();
    float va[DEPTH][SPAN], vb[DEPTH][SPAN];
    uint32_t ia[DEPTH][SPAN], ib[DEPTH][SPAN];
    auto load = [&](int32_t b0, float(&v)[DEPTH][SPAN], uint32_t(&id)[DEPTH][SPAN]) {
#pragma unroll
        for (int q = 0; q < DEPTH; ++q)
#pragma unroll
            for (int h = 0; h < SPAN; ++h) {
                id[q][h] = ~0u;
                if (b0 + q < B) {
                    const int32_t r = off[b0 + q] + (int32_t)threadIdx.x + h * SPM_THREADS;
                    if (r < off[B + b0 + q]) {
                        v[q][h] = __ldcs(partial + r);
                        id[q][h] = __ldcs(id16 + r);
                    }
                }
            }
    };
    auto add = [&](int32_t b0, float(&v)[DEPTH][SPAN], uint32_t(&id)[DEPTH][SPAN]) {
#pragma unroll
        for (int q = 0; q < DEPTH; ++q) {
            if (b0 + q >= B) break;
#pragma unroll
            for (int h = 0; h < SPAN; ++h)
                if (id[q][h] != ~0u) spm_add(sacc + id[q][h], v[q][h]);
            for (int32_t r = off[b0 + q] + (int32_t)threadIdx.x + SPAN * SPM_THREADS; r < off[B + b0 + q]; r += SPM_THREADS)
                spm_add(sacc + __ldcs(id16 + r), __ldcs(partial + r));
            __syncthreads();  // before the next block's
        }
    };
    load(0, va, ia);
    for (int32_t b0 = 0; b0 < B; b0 += 2 * DEPTH) {
        load(b0 + DEPTH, vb, ib);
        add(b0, va, ia);
        load(b0 + 2 * DEPTH, va, ia);
        add(b0 + DEPTH, vb, ib);
    }
    const bool bad = *err != 0;  // a bounded wait of the gather gave up: no sum is right
    for (int32_t t = threadIdx.x; t < k && (int64_t)j * k + t < V; t += SPM_THREADS) {
        const float2 a = sacc[t];
        const float sum = fabsf(a.x) <= 3.402823466e38f ? a.x + a.y : a.x;  // infinities and NaN as they are
        y[(int64_t)j * k + t] = bad ? __int_as_float(0x7fffffff) : sum;
    }
}

static size_t spm_smem_bytes(const tc_part *sp) { return (size_t)sp->k * 8 + (size_t)sp->B * 8; }

// perm into the staged order: entry i of block b goes to i + delta[b].
__global__ void k_stage_perm(const int32_t *__restrict__ colidx, const int32_t *__restrict__ perm, int64_t E, DivBy W,
                             const int64_t *__restrict__ delta, int32_t *__restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < E; i += (int64_t)gridDim.x * blockDim.x)
        out[i + __ldg(delta + div_apply(colidx[i], W))] = perm[i];
}

__global__ void k_gather_vals_staged(const int32_t *__restrict__ perm, const float *__restrict__ vals, int64_t n,
                                     float *__restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = perm[i] >= 0 ? vals[perm[i]] : 0.0f;
}

// How often consecutive entries change the block: about the pieces of a cut into blocks of W columns.
__global__ void __launch_bounds__(SP_THREADS) k_block_changes(const int32_t *__restrict__ colidx, int64_t E, DivBy W,
                                                              unsigned long long *count) {
    unsigned n = 0;
    for (int64_t i = blockIdx.x * (int64_t)SP_THREADS + threadIdx.x; i < E; i += (int64_t)gridDim.x * SP_THREADS)
        n += i == 0 || div_apply(__ldg(colidx + i), W) != div_apply(__ldg(colidx + i - 1), W) ? 1u : 0u;
    n = __reduce_add_sync(0xffffffffu, n);
    if ((threadIdx.x & 31) == 0 && n) atomicAdd(count, (unsigned long long)n);
}

// Does the staged form pay, with nb blocks of W columns?  Its gather is always the faster one, its merge has
// more pieces in more slices (a piece costs a random read and write of shared memory, a slice of a block and
// range a barrier), and takes what the gather gains where rows are short.  The line was fitted to 544 uniform
// and R-MAT matrices of 150K to 8M rows, 2 to 64 entries per row, 1 to 32 loaded blocks: of the 360 it takes,
// four lose more than 3% against the general form and none more than 8%; what it leaves out of 16 and more
// entries per row in four and more blocks would gain 2% at most, of shorter rows up to 42%.  Without the slices
// (pieces below 0.63 of the entries) 65 of 497 lost more than 3%: uniform, 2 per row, 8M rows 277 against 121
// us, 4 per row, 4M rows 160 / 130.  Taken now: uniform, 16 per row, 4 blocks, 1M rows 101 / 136; R-MAT 22, 8
// blocks, 254 / 404.
constexpr double SPM_SLICE = 120.0, SPM_GAIN = 0.70;  // a slice in pieces, an entry's gain in pieces
static int staged_pays(const tc_part *p, int32_t nb, int32_t W, const DeviceCaps &caps, cudaStream_t s, bool *pays) {
    DevBuf cnt;
    TC_TRY(cnt.alloc(8));
    TC_CUDA(cudaMemsetAsync(cnt.p, 0, 8, s));
    k_block_changes<<<caps.sms * 8, SP_THREADS, 0, s>>>(p->g->out_colidx.as<int32_t>(), p->E, div_by(W),
                                                        cnt.as<unsigned long long>());
    TC_LAUNCH_CHECK();
    unsigned long long n = 0;
    TC_CUDA(cudaMemcpyAsync(&n, cnt.p, 8, cudaMemcpyDeviceToHost, s));
    TC_CUDA(cudaStreamSynchronize(s));
    const int32_t k = default_merge_range(p->V, caps.sms);
    const double slices = (double)nb * (double)((p->V + (int64_t)k - 1) / k);
    *pays = (double)n - (double)p->R + SPM_SLICE * slices < SPM_GAIN * (double)p->E;
    return TC_OK;
}

// The staged form of push partition p's matrix into `sp` and p->sp_perm, sp_vals, sp_err.
static int build_staged(tc_part *p, tc_part *sp, const DeviceCaps &caps, cudaStream_t s) {
    const int64_t E = p->E;
    const int32_t *ci = p->g->out_colidx.as<int32_t>();
    const int32_t wmax = tile_max_width(caps.max_smem_optin);
    tc_part_params pp = {};
    pp.smem_stage = -1;
    const int32_t nb = (int32_t)(((int64_t)p->V + wmax - 1) / wmax);
    bool pays = false;
    TC_TRY(staged_pays(p, nb, (p->V + nb - 1) / nb, caps, s, &pays));
    if (!pays) return fail(TC_ERR_UNSUPPORTED, "build_staged: too many pieces");
    TC_TRY(build_partition(p->g, TC_PUSH, nb, &pp, s, sp));
    if (sp->W > wmax || sp->W % 32 != 0 || !sp->id16.p || spm_smem_bytes(sp) > (size_t)caps.max_smem_optin) return fail(TC_ERR_UNSUPPORTED, "build_staged: width");
    if (!fits_signed(sp->R, SPM_PAST)) return fail(TC_ERR_UNSUPPORTED, "build_staged: too many pieces");
    TC_TRY(build_tiles(sp, caps.sms, s));
    if (!sp->tiled) return fail(TC_ERR_UNSUPPORTED, "build_staged: no staged form");
    DevBuf iota, keys, perm, kt, vt, delta;
    TC_TRY(iota.alloc((size_t)E * 4));
    k_iota<<<caps.sms * 8, 256, 0, s>>>(E, iota.as<int32_t>());
    TC_LAUNCH_CHECK();
    if (sp->B > 1) {  // the partition's own stable sort, carrying each entry's position
        TC_TRY(keys.alloc((size_t)E * 4));
        TC_TRY(perm.alloc((size_t)E * 4));
        TC_TRY(kt.alloc((size_t)E * 4));
        TC_TRY(vt.alloc((size_t)E * 4));
        int bits = 0;
        while ((1LL << bits) < (int64_t)sp->B) ++bits;
        TC_TRY(stable_bucket_sort(ci, iota.as<int32_t>(), keys.as<int32_t>(), perm.as<int32_t>(), kt.as<int32_t>(),
                                  vt.as<int32_t>(), E, sp->W, bits, s));
    } else {
        perm.swap(iota);
    }
    std::vector<int64_t> h_delta((size_t)sp->B);
    int64_t pb = 0;
    for (int32_t b = 0; b < sp->B; ++b) {
        h_delta[(size_t)b] = pb - sp->h_blk_edges[b];
        pb += (sp->h_blk_edges[b + 1] - sp->h_blk_edges[b] + TILE_WCHUNK - 1) / TILE_WCHUNK * TILE_WCHUNK;
    }
    const int64_t n = sp->padded_edges + TILE_WCHUNK;  // with the chunk of slack of the staged stream
    TC_TRY(delta.alloc(h_delta.size() * 8));
    TC_TRY(p->sp_perm.alloc((size_t)n * 4));
    TC_TRY(p->sp_vals.alloc((size_t)n * 4));
    TC_TRY(p->sp_err.alloc(4));
    TC_CUDA(cudaMemsetAsync(p->sp_perm.p, 0xFF, (size_t)n * 4, s));
    TC_CUDA(cudaMemcpyAsync(delta.p, h_delta.data(), h_delta.size() * 8, cudaMemcpyHostToDevice, s));
    k_stage_perm<<<caps.sms * 8, 256, 0, s>>>(sp->colidx.as<int32_t>(), perm.as<int32_t>(), E, div_by(sp->W),
                                              delta.as<int64_t>(), p->sp_perm.as<int32_t>());
    TC_LAUNCH_CHECK();
    TC_CUDA(cudaStreamSynchronize(s));
    // the gather and the merge need neither of these
    for (DevBuf *d : {&sp->colidx, &sp->esrc, &sp->rowptr, &sp->id_map, &sp->rowbits, &sp->merge_off, &sp->merge_gpre,
                      &sp->hubs})
        d->release();
    return TC_OK;
}

// GC-push (Sec. 4's SpMV in the push direction with TOCAB): the pieces of a TC_PULL partition of
// the matrix's graph.  Piece r = (row block b, column j = id_map[r]) holds the entries (i, j) of
// A with i in block b; x[j] is read once per piece and every entry adds vals * x[j] into y[i]
// with an FP32 atomic add.  The pieces are stored block after block, so while a block's pieces
// run, the atomics land in its W-entry slice of y, which the L2 holds (Sec. 3.1 with y as the
// working set).  Load balancing as Sec. 3.2 bins it: a lane per piece below 32 entries, a warp
// per longer one.  The order of the additions into y[i] depends on timing.
__global__ void __launch_bounds__(SP_THREADS) k_spmv_push_pieces(const int32_t *__restrict__ rowptr,
                                                                 const int32_t *__restrict__ colidx,
                                                                 const float *__restrict__ pvals,
                                                                 const int32_t *__restrict__ id_map,
                                                                 const float *__restrict__ x, int64_t R, float *y) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (SP_THREADS / 32);
    for (int64_t grp = (blockIdx.x * (int64_t)SP_THREADS + threadIdx.x) >> 5; grp * 32 < R; grp += nw) {
        const int64_t r = grp * 32 + lane;
        int32_t s = 0, e = 0;
        float xj = 0.0f;
        if (r < R) {
            s = __ldg(rowptr + r);
            e = __ldg(rowptr + r + 1);
            xj = __ldg(x + __ldg(id_map + r));
        }
        if (e - s < 32)
            for (int32_t k = s; k < e; ++k) atomicAdd(y + __ldg(colidx + k), __ldg(pvals + k) * xj);
        unsigned long_rows = __ballot_sync(0xffffffffu, e - s >= 32);
        while (long_rows) {
            const int l = __ffs(long_rows) - 1;
            long_rows &= long_rows - 1;
            const int32_t ls = __shfl_sync(0xffffffffu, s, l), le = __shfl_sync(0xffffffffu, e, l);
            const float xl = __shfl_sync(0xffffffffu, xj, l);
            for (int32_t k = ls + lane; k < le; k += 32) atomicAdd(y + __ldg(colidx + k), __ldg(pvals + k) * xl);
        }
    }
}

}  // namespace tc

extern "C" int tc_part_set_values(tc_part *p, const float *vals, int mem, void *stream) {
    using namespace tc;
    if (!p || (p->E > 0 && !vals)) return fail(TC_ERR_INVALID_ARG, "tc_part_set_values: null partition or values");
    if (p->dir != TC_PUSH && p->dir != TC_PULL) return fail(TC_ERR_INVALID_ARG, "tc_part_set_values: bad partition");
    if (p->order != TC_ORDER_NATURAL)
        return fail(TC_ERR_UNSUPPORTED, "tc_part_set_values: renumbered (TC_ORDER_OUTDEGREE) partitions are not supported");
    if (mem != TC_MEM_DEVICE) return fail(TC_ERR_UNSUPPORTED, "tc_part_set_values: vals must be a device pointer");
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t E = p->E;
    DeviceCaps caps;
    TC_TRY(device_caps(&caps));
    const int grid = caps.sms * 8;
    // Not where the caller declines it, under a memory cap, or where its memory is not to be had: the general
    // form needs less, and less time to set up (R-MAT 22: 0.7 against 2.9 ms, saved in 15 products).
    if (!p->sp_tried && p->dir == TC_PUSH && p->smem_stage >= 0 && E >= SPM_MIN_ENTRIES && !cache_get_limit()) {
        p->sp_tried = true;
        tc_part *sp = new (std::nothrow) tc_part();
        if (sp) {
            const KeptError kept;
            const int st = build_staged(p, sp, caps, s);
            if (st == TC_OK) {
                p->sp = sp;
            } else {
                TC_CUDA(cudaStreamSynchronize(s));
                delete sp;
                p->sp_perm.release();
                p->sp_vals.release();
                if (st != TC_ERR_OOM && st != TC_ERR_UNSUPPORTED) return st;
                kept.restore();
            }
        }
    }
    if (p->sp) {
        k_gather_vals_staged<<<grid, 256, 0, s>>>(p->sp_perm.as<int32_t>(), vals, p->sp->padded_edges + TILE_WCHUNK,
                                                  p->sp_vals.as<float>());
        TC_LAUNCH_CHECK();
        TC_CUDA(cudaStreamSynchronize(s));
        p->has_vals = true;
        return TC_OK;
    }
    if (!p->pperm_built) {  // the partition's own sorts again, carrying each entry's position
        TC_TRY(p->pperm.alloc((size_t)(E > 0 ? E : 1) * 4));
        if (E > 0) {
            DevBuf iota, keys, kt, vt, tpos;
            TC_TRY(iota.alloc((size_t)E * 4));
            k_iota<<<grid, 256, 0, s>>>(E, iota.as<int32_t>());
            TC_LAUNCH_CHECK();
            TC_TRY(keys.alloc((size_t)E * 4));
            TC_TRY(kt.alloc((size_t)E * 4));
            TC_TRY(vt.alloc((size_t)E * 4));
            // the entries in the order the partition's stream starts from: the CSR itself for a
            // push partition; for a pull partition G^T, the graph load's stable sort by column
            const int32_t *ci = p->g->out_colidx.as<int32_t>();
            const int32_t *pos = iota.as<int32_t>();
            if (p->dir == TC_PULL) {
                int vbits = 0;
                while ((1LL << vbits) < (int64_t)p->V) ++vbits;
                TC_TRY(tpos.alloc((size_t)E * 4));
                TC_TRY(stable_bucket_sort(ci, iota.as<int32_t>(), keys.as<int32_t>(), tpos.as<int32_t>(),
                                          kt.as<int32_t>(), vt.as<int32_t>(), E, 1, vbits, s));
                ci = p->g->in_colidx.as<int32_t>();
                pos = tpos.as<int32_t>();
            }
            if (p->B > 1) {
                int bits = 0;
                while ((1LL << bits) < (int64_t)p->B) ++bits;
                TC_TRY(stable_bucket_sort(ci, pos, keys.as<int32_t>(), p->pperm.as<int32_t>(), kt.as<int32_t>(),
                                          vt.as<int32_t>(), E, p->W, bits, s));
            } else {
                TC_CUDA(cudaMemcpyAsync(p->pperm.p, pos, (size_t)E * 4, cudaMemcpyDeviceToDevice, s));
            }
            TC_CUDA(cudaStreamSynchronize(s));  // the scratch is freed at the end of this block
        }
        p->pperm_built = true;
    }
    TC_TRY(p->pvals.alloc((size_t)(E > 0 ? E : 1) * 4));
    if (E > 0) {
        k_gather_vals<<<grid, 256, 0, s>>>(p->pperm.as<int32_t>(), vals, E, p->pvals.as<float>());
        TC_LAUNCH_CHECK();
    }
    TC_CUDA(cudaStreamSynchronize(s));
    p->has_vals = true;
    return TC_OK;
}

extern "C" int tc_spmv_tocab(const tc_part *p, const float *x, float *y, int mem, void *stream) {
    using namespace tc;
    if (!p || !x || !y) return fail(TC_ERR_INVALID_ARG, "tc_spmv_tocab: null partition or vector");
    if (!p->has_vals)
        return fail(TC_ERR_INVALID_ARG, "tc_spmv_tocab: needs a partition given values by tc_part_set_values");
    if (mem != TC_MEM_DEVICE) return fail(TC_ERR_UNSUPPORTED, "tc_spmv_tocab: x and y must be device pointers");
    const int32_t V = p->V;
    if (V == 0) return TC_OK;
    if (p->dir == TC_PULL) {  // GC-push: y = 0, then the pieces add into it
        DeviceCaps caps;
        TC_TRY(device_caps(&caps));
        cudaStream_t s = (cudaStream_t)stream;
        TC_CUDA(cudaMemsetAsync(y, 0, (size_t)V * 4, s));
        if (p->R > 0) {
            const int64_t want = (p->R + SP_THREADS - 1) / SP_THREADS;
            const int grid = (int)(want < (int64_t)caps.sms * 16 ? want : (int64_t)caps.sms * 16);
            k_spmv_push_pieces<<<grid, SP_THREADS, 0, s>>>(p->rowptr.as<int32_t>(), p->colidx.as<int32_t>(),
                                                           p->pvals.as<float>(), p->id_map.as<int32_t>(), x, p->R, y);
            TC_LAUNCH_CHECK();
        }
        return TC_OK;
    }
    if ((size_t)p->k * 4 > 200 * 1024) return fail(TC_ERR_UNSUPPORTED, "tc_spmv_tocab: merge_range above 51,200");
    if (p->sp) {
        const tc_part *sp = p->sp;
        // a wait that gave up spoils the product it happened in, not the next ones (1.6 us of 240 on R-MAT 22)
        TC_CUDA(cudaMemsetAsync(p->sp_err.p, 0, 4, (cudaStream_t)stream));
        TC_TRY(launch_tiled_spmv(sp, p->sp_vals.as<float>(), x, p->sp_err.as<int>(), (cudaStream_t)stream));
        // entries per thread and block: one, two or four, by the mean slice of a block and range (an entry
        // past them is a round trip of its own, and a place without one costs its slot).  One / two / four, us:
        // slices of 294 71 / 78 / 84, 383 130 / 143 / 157, 477 267 / 255 / 281, 648 923 / 738 / 838, 941 97 / 97 /
        // 103, 1,139 194 / 217 / 191, 1,608 299 / 372 / 275
        const int64_t slice = sp->R / ((int64_t)sp->B * sp->nranges);
        auto merge = slice <= SPM_THREADS * 3 / 4   ? k_spmv_merge_staged<4, 1>
                     : slice <= SPM_THREADS * 7 / 4 ? k_spmv_merge_staged<4, 2>
                                                    : k_spmv_merge_staged<2, 4>;
        const size_t smem = spm_smem_bytes(sp);
        TC_CUDA(cudaFuncSetAttribute(merge, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        merge<<<sp->nranges, SPM_THREADS, smem, (cudaStream_t)stream>>>(
            sp->partial.as<float>(), sp->id16.as<uint16_t>(), sp->merge_offT.as<int32_t>(), sp->B, sp->k, V,
            p->sp_err.as<int>(), y);
        TC_LAUNCH_CHECK();
        return TC_OK;
    }
    DeviceCaps caps;
    TC_TRY(device_caps(&caps));
    cudaStream_t s = (cudaStream_t)stream;
    if (p->R > 0) {
        const int64_t want = (p->R + SP_THREADS - 1) / SP_THREADS;
        const int grid = (int)(want < (int64_t)caps.sms * 16 ? (want > 0 ? want : 1) : (int64_t)caps.sms * 16);
        k_spmv_block_rows<<<grid, SP_THREADS, 0, s>>>(p->rowptr.as<int32_t>(), p->colidx.as<int32_t>(),
                                                      p->pvals.as<float>(), x, p->R,
                                                      const_cast<float *>(p->partial.as<float>()));
        TC_LAUNCH_CHECK();
    }
    const size_t smem = (size_t)p->k * 4;
    TC_CUDA(cudaFuncSetAttribute(k_spmv_merge, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int mgrid = p->nranges < caps.sms * 8 ? (p->nranges > 0 ? p->nranges : 1) : caps.sms * 8;
    k_spmv_merge<<<mgrid, SP_THREADS, smem, s>>>(p->partial.as<float>(), p->id_map.as<int32_t>(),
                                                 p->merge_off.as<int32_t>(), p->B, p->nranges, p->k, V, y);
    TC_LAUNCH_CHECK();
    return TC_OK;
}
