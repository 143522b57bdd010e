// Greedy placement in waves, by one block (plan.cu, vrsp.cu).  Thread i stands for the i-th of W bins, which are kept as
// an array of keys (load << 10 | bin) in ascending order, all different, and for the i-th of the coming items.  Item i
// goes to key[i] as long as key[i] lies below every key put back by the items before it: nothing put back can then
// overtake it.  The longest such prefix is placed at once, one item per bin, and the keys put back are merged into the
// rest of the array.  Item for item this is the one-by-one rule (least load, lowest index).
//
// The chain of waves bounds it, about 800 clk plus 7 per item of a wave.  One warp with waves of at most 32 items took
// 3000 clk a wave: 16384 query-major tiles on 148 workers were 524 such waves and are 111 of these.
#pragma once
#include <stdint.h>

namespace libra {

constexpr int kWaveMaxBins = 1024;

struct WaveSmem {
    uint64_t key[2][kWaveMaxBins];   // the sorted array and its next version
    uint64_t put[kWaveMaxBins];      // keys put back, in item order
    uint64_t back[kWaveMaxBins];     // the same in ascending order
    uint64_t warp_min[32];
    int warp_fit[32];
};

// Items of the coming wave.  `key`: this thread's bin, `put`: what it would put back (~0: nothing, the bin is full);
// `live`: there are such a bin and such an item.  Ends with a barrier.
__device__ __forceinline__ int wave_take(WaveSmem& sm, uint64_t key, uint64_t put, bool live) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    uint64_t before = put;   // smallest key put back by this thread and those below it
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t other = __shfl_up_sync(0xffffffffu, before, o);
        if (lane >= o && other < before) before = other;
    }
    if (lane == 31) sm.warp_min[warp] = before;
    before = __shfl_up_sync(0xffffffffu, before, 1);
    if (lane == 0) before = ~0ull;
    __syncthreads();
    for (int w = 0; w < warp; ++w)
        if (sm.warp_min[w] < before) before = sm.warp_min[w];
    const unsigned fits = __ballot_sync(0xffffffffu, live && key < before);
    if (lane == 0) sm.warp_fit[warp] = ~fits == 0u ? 32 : __ffs(~fits) - 1;
    __syncthreads();
    int take = 0;
    for (int w = 0; w < n_warps; ++w) {
        const int f = sm.warp_fit[w];
        take += f;
        if (f < 32) break;
    }
    return take;
}

// Number of a[0 .. n) below k (a ascending).
__device__ __forceinline__ int count_below(const uint64_t* a, int n, uint64_t k) {
    int lo = 0;
    for (int step = n > 0 ? 1 << (31 - __clz(n)) : 0; step > 0; step >>= 1)
        if (lo + step <= n && a[lo + step - 1] < k) lo += step;
    return lo;
}

// The first `take` keys leave the array, the threads with `keeps` put theirs back.  Returns the number of keys now in
// sm.key[cur ^ 1].  Ends with a barrier.
__device__ __forceinline__ int wave_merge(WaveSmem& sm, int cur, int W, int take, uint64_t key, uint64_t put, bool keeps) {
    const int i = threadIdx.x;
    const uint64_t* rest = sm.key[cur] + take;
    uint64_t* nxt = sm.key[cur ^ 1];
    if (i < take) sm.put[i] = keeps ? put : ~0ull;
    const int nput = __syncthreads_count(keeps);
    if (keeps) {
        int rank = 0;
#pragma unroll 8
        for (int j = 0; j < take; ++j) rank += sm.put[j] < put ? 1 : 0;
        sm.back[rank] = put;
        nxt[rank + count_below(rest, W - take, put)] = put;
    }
    __syncthreads();
    if (i >= take && i < W) nxt[i - take + count_below(sm.back, nput, key)] = key;
    __syncthreads();
    return W - take + nput;
}

}  // namespace libra
