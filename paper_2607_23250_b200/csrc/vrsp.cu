// Variance-Reduced Sequence Placement (Algorithm 1) on the device.
//
// Packed sequences of one optimizer-step window are grouped into K = D / P pools of exactly P
// sequences so that the pools' summed attention work is even: sequences in decreasing work order
// (ties: lower index first) each go to the least-loaded pool that still has room (ties: lower pool
// index).  The paper runs this on a CPU core per step (48-106 us for D = 128-256); here it is three
// small kernels on the caller's stream so that a data path that already lives on the GPU does not
// have to come back to the host.  Integer only; results are bit-identical to the sequential rule.
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/libra.h"
#include "common.h"
#include "ptx.cuh"
#include "waves.cuh"

namespace libra {

// F_i = sum over the samples of sequence i of len^2 (the work proxy of Section 4.2).  One warp per sequence: a thread
// of its own per sequence walks its samples one L2 latency after the other.
__global__ void k_vrsp_work(const int32_t* __restrict__ sample_offsets, const int32_t* __restrict__ seq_first_sample,
                            int D, int64_t* __restrict__ work) {
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    grid_dep_wait();
    grid_dep_launch();
    if (i >= D) return;
    int64_t f = 0;
    const int end = seq_first_sample[i + 1];
    for (int j = seq_first_sample[i] + lane; j < end; j += 32) {
        const int64_t len = (int64_t)sample_offsets[j + 1] - sample_offsets[j];
        f += len * len;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
    if (lane == 0) work[i] = f;
}

// rank of sequence i in the order (work descending, index ascending); sixteen lanes per sequence share the comparisons,
// so that a window of a few hundred sequences fills more than a block or two.
__global__ void __launch_bounds__(256) k_vrsp_rank(const int64_t* __restrict__ work, int D, int32_t* __restrict__ sorted) {
    __shared__ int64_t sw[1024];
    grid_dep_wait();
    grid_dep_launch();
    const int i = blockIdx.x * 16 + (threadIdx.x >> 4), sub = threadIdx.x & 15;
    const int64_t wi = i < D ? work[i] : 0;
    int rank = 0;
    for (int base = 0; base < D; base += 1024) {
        const int lim = D - base < 1024 ? D - base : 1024;
        for (int o = threadIdx.x; o < lim; o += 256) sw[o] = work[base + o];
        __syncthreads();
        for (int k = sub; k < lim; k += 16) {
            const int64_t w = sw[k];
            rank += (w > wi) || (w == wi && base + k < i);
        }
        __syncthreads();
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
    if (i < D && sub == 0) sorted[rank] = i;
}

// Placement in waves by one block (waves.cuh): the bins are the pools with room; a full pool leaves the array.  Needs
// 0 <= work and loads below 2^53 (the caller checks).  1024 sequences into 128 pools, all three kernels: 29 us; 502 us
// with an arg-min over all pools per sequence, 75 us in waves of up to 32 by one warp.
__device__ void vrsp_place_waves(const int64_t* __restrict__ work, const int32_t* __restrict__ sorted, int D, int P, int K,
                                 int32_t* __restrict__ order, int32_t* __restrict__ pool_of_seq,
                                 int64_t* __restrict__ pool_load) {
    __shared__ WaveSmem sm;
    __shared__ int32_t cnt[kWaveMaxBins];
    constexpr int kBatch = 512;
    __shared__ int64_t wbuf[kBatch];
    __shared__ int32_t sbuf[kBatch];
    const int i = threadIdx.x, nthr = blockDim.x;
    if (i < K) { sm.key[0][i] = (uint64_t)i; cnt[i] = 0; }
    const int batch = 4 * nthr < kBatch ? 4 * nthr : kBatch;
    int64_t w_n[4];
    int32_t s_n[4];
    auto fetch = [&](int x0) {                   // this thread's sequences of the batch at position x0 of the order
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int x = x0 + i + k * nthr;
            const bool in = i + k * nthr < batch && x < D;
            s_n[k] = in ? sorted[x] : 0;
            w_n[k] = in ? work[s_n[k]] : 0;
        }
    };
    fetch(0);
    int W = K, cur = 0;                          // pools with room
    for (int x0 = 0; x0 < D; x0 += batch) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i + k * nthr < batch) { wbuf[i + k * nthr] = w_n[k]; sbuf[i + k * nthr] = s_n[k]; }
        __syncthreads();
        if (x0 + batch < D) fetch(x0 + batch);
        const int lim = D - x0 < batch ? D - x0 : batch;
        for (int b = 0; b < lim;) {
            const bool live = i < W && b + i < lim;
            const int64_t w = live ? wbuf[b + i] : 0;
            const uint64_t key = i < W ? sm.key[cur][i] : ~0ull;
            const int pool = (int)(key & 1023u);
            const int had = live ? cnt[pool] : 0;
            const bool full = had + 1 >= P;
            const uint64_t put = live && !full ? key + ((uint64_t)w << 10) : ~0ull;
            const int take = wave_take(sm, key, put, live);   // >= 1: the first key always fits
            const bool placed = i < take;
            if (placed) {
                const int32_t sq = sbuf[b + i];
                order[(int64_t)pool * P + had] = sq;   // pools are laid end to end in pool order
                pool_of_seq[sq] = pool;
                cnt[pool] = had + 1;
                if (full) pool_load[pool] = (int64_t)(key >> 10) + w;
            }
            W = wave_merge(sm, cur, W, take, key, put, placed && !full);
            cur ^= 1;
            b += take;
        }
    }
}

// Work that may add up beyond 53 bits, or negative work (which no sequence has): one sequence after the other, an
// arg-min over all pools each (0.45 us a sequence with 128 pools).  Pool k's load and fill count live in lane
// k % 32, register k / 32; a full pool's load is replaced by INT64_MAX in the comparison, which is
// what removing it from the algorithm's heap does.  Popping the heap's minimum (load, k) is the
// lexicographic arg-min taken here.
template <int PER>
__global__ void __launch_bounds__(1024) k_vrsp_place(const int64_t* __restrict__ work, const int32_t* __restrict__ sorted,
                                                   int D, int P, int K, int32_t* __restrict__ order,
                                                   int32_t* __restrict__ pool_of_seq, int64_t* __restrict__ pool_load) {
    const int lane = threadIdx.x;
    grid_dep_wait();
    {   // sorted descending: the first work bounds every load, the last one tells whether any is negative
        const int64_t most = work[sorted[0]], least = work[sorted[D - 1]];
        if (least >= 0 && most < (int64_t(1) << 52) / P) {
            vrsp_place_waves(work, sorted, D, P, K, order, pool_of_seq, pool_load);
            return;
        }
    }
    if (threadIdx.x >= 32) return;
    int64_t load[PER];
    int32_t cnt[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        load[i] = 0;
        cnt[i] = (lane + 32 * i < K) ? 0 : P;  // pools that do not exist count as full
    }
    for (int x0 = 0; x0 < D; x0 += 32) {
        const int xl = x0 + lane;
        int32_t s_l = 0;
        int64_t w_l = 0;
        if (xl < D) { s_l = sorted[xl]; w_l = work[s_l]; }
        const int lim = D - x0 < 32 ? D - x0 : 32;
        for (int i = 0; i < lim; ++i) {
            const int64_t w = __shfl_sync(0xffffffffu, w_l, i);
            const int32_t sq = __shfl_sync(0xffffffffu, s_l, i);
            int64_t best = INT64_MAX;
            int32_t bidx = INT32_MAX;
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                if (cnt[k] < P && (load[k] < best || bidx == INT32_MAX)) { best = load[k]; bidx = lane + 32 * k; }
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                const int64_t ob = __shfl_xor_sync(0xffffffffu, best, off);
                const int32_t oi = __shfl_xor_sync(0xffffffffu, bidx, off);
                // a lane without a candidate carries bidx = INT32_MAX and never wins
                if (oi != INT32_MAX && (bidx == INT32_MAX || ob < best || (ob == best && oi < bidx))) { best = ob; bidx = oi; }
            }
            if (bidx != INT32_MAX && (bidx & 31) == lane) {
#pragma unroll
                for (int k = 0; k < PER; ++k) {
                    if (k == (bidx >> 5)) {
                        order[(int64_t)bidx * P + cnt[k]] = sq;  // pools are concatenated in pool order
                        load[k] += w;
                        cnt[k] += 1;
                    }
                }
                pool_of_seq[sq] = bidx;
            }
        }
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int k = lane + 32 * i;
        if (k < K) pool_load[k] = load[i];
    }
}

}  // namespace libra

using namespace libra;

extern "C" int libra_vrsp_work(const int32_t* sample_offsets_dev, const int32_t* seq_first_sample_dev, int n_sequences,
                               int64_t* work_dev, void* stream) {
    if (!sample_offsets_dev || !seq_first_sample_dev || !work_dev || n_sequences <= 0) return LIBRA_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    count_launch(1);
    const cudaError_t e = launch_dependent(k_vrsp_work, (unsigned)((n_sequences + 7LL) / 8), 256u, 0, s, sample_offsets_dev, seq_first_sample_dev,
                                           n_sequences, work_dev);
    return e == cudaSuccess ? LIBRA_OK : LIBRA_ERR_CUDA;
}

extern "C" int libra_vrsp_place(const int64_t* work_dev, int n_sequences, int pool_size, int32_t* order_dev,
                                int32_t* pool_of_seq_dev, int64_t* pool_load_dev, int32_t* scratch_dev, void* stream) {
    if (!work_dev || !order_dev || !pool_of_seq_dev || !pool_load_dev || !scratch_dev) return LIBRA_ERR_INVALID_ARG;
    if (n_sequences <= 0 || pool_size <= 0 || n_sequences % pool_size != 0) return LIBRA_ERR_INVALID_ARG;
    const int D = n_sequences, P = pool_size, K = D / P;
    if (K > 1024 || D > (1 << 20)) return LIBRA_ERR_UNSUPPORTED;
    cudaStream_t s = (cudaStream_t)stream;
    const int threads = (K + 31) / 32 * 32;
    cudaError_t e = launch_dependent(k_vrsp_rank, (unsigned)((D + 15) / 16), 256u, 0, s, work_dev, D, scratch_dev);
    if (e == cudaSuccess) {
        auto place = K <= 32 ? k_vrsp_place<1> : (K <= 128 ? k_vrsp_place<4> : k_vrsp_place<32>);
        e = launch_dependent(place, 1u, (unsigned)threads, 0, s, work_dev, scratch_dev, D, P, K, order_dev, pool_of_seq_dev, pool_load_dev);
    }
    count_launch(2);
    return e == cudaSuccess ? LIBRA_OK : LIBRA_ERR_CUDA;
}
