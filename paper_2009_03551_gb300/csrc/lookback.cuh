// Prefix sums across the CTAs of one launch: a CTA publishes its sum and adds up
// those of the CTAs before it, back to the nearest that knows its own prefix
// (decoupled look-back: Merrill and Garland, Single-pass Parallel Prefix Scan
// with Decoupled Look-back, 2016).  CTAs are numbered in the order in which they
// start, so that those a CTA waits for are running and publish before they
// wait themselves; the wait is bounded all the same.
#pragma once

#include <stdint.h>

namespace rdm {
namespace {

// A wait is bounded by the number of looks (~1 us each), not by the clock, which
// runs on while the whole context is descheduled.
constexpr int kLookPolls = 1 << 21;

// 64-bit words of state for `grid` CTAs, zeroed before the launch: the number of
// CTAs that have started, then per CTA 1 << 32 | sum or 2 << 32 | prefix + sum
inline int lookback_words(int grid) { return grid + 1; }

// this CTA's number (all threads; a barrier)
__device__ __forceinline__ int lookback_id(unsigned long long *look, int *sh) {
    if (threadIdx.x == 0) *sh = (int)atomicAdd(look, 1ull);
    __syncthreads();
    return *sh;
}

// sum over the CTAs numbered below `bid`, all lanes of one warp; `total`: this
// CTA's sum.  A wait that runs out sets *err and the missing sums count as 0, so
// that a place computed from them is too small but never outside the list
// (polls = 0, a test setting: every wait runs out).
__device__ __forceinline__ int lookback_sum(unsigned long long *look, int bid, int total, int *err, int polls) {
    const int lane = threadIdx.x & 31;
    volatile unsigned long long *st = look + 1;
    if (lane == 0) st[bid] = ((bid == 0 ? 2ull : 1ull) << 32) | (unsigned)total;
    if (bid == 0) return 0;
    int sum = 0;
    for (int j = bid - 1;; j -= 32) {
        unsigned long long v = 2ull << 32;
        if (j - lane >= 0) {
            v = 0ull;
            for (int n = 0; v == 0ull && n < polls; ++n) v = st[j - lane];
            if (v == 0ull) {
                atomicOr(err, 1);
                v = 2ull << 32;
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, (v >> 32) == 2ull);
        const int last = m ? __ffs(m) - 1 : 31;
        int x = lane <= last ? (int)(unsigned)v : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        sum += x;
        if (m) break;
    }
    if (lane == 0) st[bid] = (2ull << 32) | (unsigned)(sum + total);
    return sum;
}

}  // namespace
}  // namespace rdm
