// Strided walks over edge positions.  A graph may have 2^31 - 2 edges, so a signed 32-bit position that
// steps past the end of the last edges wraps to a negative one, below the end again.  The walks' positions
// are unsigned: a thread's last step leaves them below 2^32 as long as the batch is below 2^31.  Compiles
// as plain C++ too, for the check of the positions on the host.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define TC_WALK __device__ __forceinline__
#else
#define TC_WALK inline
#endif

namespace tc {

// Whether signed 32-bit positions of n items do not wrap when they go up to `past` beyond the end.
constexpr bool fits_signed(int64_t n, int64_t past) { return n + past <= INT32_MAX; }

// The first position of lane `lane` in [s, e): s + lane, or e if that is past the end (rows shorter than
// the lanes that share them, where the sum could wrap).
TC_WALK int32_t lane_first(int32_t s, int32_t e, int32_t lane) { return lane < e - s ? s + lane : e; }

// one(i) for the positions i, i + STEP, ... below `end`.
template <int STEP, class One>
TC_WALK void walk(uint32_t i, uint32_t end, One one) {
    for (; i < end; i += STEP) one(i);
}

// batch(i) takes the positions i, i + STEP, ..., i + (N - 1) STEP, all below `end`; one(i) those left over.
template <int N, int STEP, class Batch, class One>
TC_WALK void walk_batched(uint32_t i, uint32_t end, Batch batch, One one) {
    for (; i + (N - 1) * STEP < end; i += N * STEP) batch(i);
    walk<STEP>(i, end, one);
}

}  // namespace tc
