// Prefix sums of a few thousand counts in one launch.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace gts {

constexpr int64_t kScanBlockMax = 16384;

// out[i] = in[0] + .. + in[i - 1] for i <= n (out[n]: the total), n <=
// kScanBlockMax, one block of 1024 threads.  The device-wide scan of so few
// counts takes three launches (widening to 64 bits, tile states, scan) and an
// allocation: about 8 us more.
template <class T>
__global__ void __launch_bounds__(1024) k_scan_block(const T *__restrict__ in, int64_t n, int64_t *__restrict__ out) {
    __shared__ int64_t wtot[32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int per = (int)((n + 1023) / 1024);
    const int64_t a = (int64_t)t * per, b = a + per < n ? a + per : n;
    int64_t sum = 0;
    for (int64_t i = a; i < b; ++i) sum += (int64_t)in[i];
    int64_t incl = sum;
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) wtot[warp] = incl;
    __syncthreads();
    int64_t before = 0;
    for (int w = 0; w < warp; ++w) before += wtot[w];
    int64_t run = before + incl - sum;
    for (int64_t i = a; i < b; ++i) {
        out[i] = run;
        run += (int64_t)in[i];
    }
    if (t == 1023) out[n] = before + incl;
}

}  // namespace gts
