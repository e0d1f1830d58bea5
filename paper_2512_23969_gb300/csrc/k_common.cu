// k_common.cu -- kernels shared by every parameter set: message offsets.
#include <cuda_runtime.h>
#include "hs_launch.h"

namespace hs {

// ------------------------------------------------------------- offsets
// offsets[i] = lens[0] + ... + lens[i-1], i = 0..count (one CTA of 1024): a
// coalesced row of 1024 lengths at a time, scanned by shuffles in the warps
// and once across them, the next row's loads in flight.  One CTA's latency
// bounds it; a chunk of consecutive lengths per thread (uncoalesced, two
// passes, ten barriers' scan) took 31 us for 16384 messages.
__global__ void __launch_bounds__(1024) offsets_kernel(const uint64_t* __restrict__ lens, uint32_t count,
                                                       uint64_t* __restrict__ off) {
    __shared__ uint64_t sums[2][32];
    const uint32_t t = threadIdx.x, lane = t & 31, warp = t >> 5;
    uint64_t before = 0, next = t < count ? lens[t] : 0;
    for (uint64_t base = 0; base < count; base += 1024) {
        const uint64_t i = base + t, v = next;
        next = i + 1024 < count ? lens[i + 1024] : 0;
        uint64_t x = v;                                  // inclusive scan in the warp
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, x, d);
            if (lane >= (uint32_t)d) x += y;
        }
        uint64_t* s = sums[(base >> 10) & 1];            // two rows apart, a barrier between: no third barrier
        if (lane == 31) s[warp] = x;
        __syncthreads();
        uint64_t w = s[lane];                            // every warp scans the 32 sums
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, w, d);
            if (lane >= (uint32_t)d) w += y;
        }
        const uint64_t head = __shfl_sync(0xFFFFFFFFu, w, warp ? warp - 1 : 0);
        if (i < count) off[i] = before + (warp ? head : 0) + x - v;
        before += __shfl_sync(0xFFFFFFFFu, w, 31);
    }
    if (t == 0) off[count] = before;
}

cudaError_t launch_offsets(const Batch& b, cudaStream_t s) {
    if (!needs_offsets(b)) return cudaSuccess;
    offsets_kernel<<<1, 1024, 0, s>>>(b.lens, b.count, b.offsets);
    return cudaGetLastError();
}

}  // namespace hs
