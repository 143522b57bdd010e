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

namespace libra {

// F_i = sum over the samples of sequence i of len^2 (the work proxy of Section 4.2).  One warp per sequence: a thread
// of its own per sequence walks its samples one L2 latency after the other.
__global__ void k_vrsp_work(const int32_t* __restrict__ sample_offsets, const int32_t* __restrict__ seq_first_sample,
                            int D, int64_t* __restrict__ work) {
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
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

// Placement in waves by one warp.  The pools with room form one sorted array of keys (load << 10 | pool) in shared
// memory.  Sequence s of the coming batch goes to key[s] as long as key[s] lies below every key put back by the
// sequences before it: nothing put back can then be the minimum earlier.  The longest such prefix (at most 32) is
// placed at once, one sequence per pool; the keys put back by pools that still have room are ranked among themselves
// and merged with the rest of the array, every key finding its place by a binary search in the other sequence; a full
// pool leaves the array.  Sequence for sequence this is the one-by-one rule.  Needs 0 <= work and loads below 2^53
// (the caller checks).  The serial chain is what bounds it: 1024 sequences into 128 pools, all three kernels: 76 us,
// with an arg-min over all pools per sequence 502 us.
__device__ void vrsp_place_waves(const int64_t* __restrict__ work, const int32_t* __restrict__ sorted, int D, int P, int K,
                                 int32_t* __restrict__ order, int32_t* __restrict__ pool_of_seq,
                                 int64_t* __restrict__ pool_load, uint64_t* cur, uint64_t* nxt, int32_t* cnt) {
    __shared__ uint64_t put_raw[32], back[32];
    const int lane = threadIdx.x;
    for (int k = lane; k < K; k += 32) { cur[k] = (uint64_t)k; cnt[k] = 0; }
    __syncwarp();
    int W = K;                                   // pools with room
    int32_t s_l = lane < D ? sorted[lane] : 0;   // the coming 32 sequences, and the 32 after them
    int64_t w_l = lane < D ? work[s_l] : 0;
    for (int x0 = 0; x0 < D; x0 += 32) {
        const int lim = D - x0 < 32 ? D - x0 : 32;
        const int xn = x0 + 32 + lane;
        const int32_t s_n = xn < D ? sorted[xn] : 0;
        const int64_t w_n = xn < D ? work[s_n] : 0;
        for (int i = 0; i < lim;) {
            const int64_t w_s = __shfl_sync(0xffffffffu, w_l, (i + lane) & 31);
            const int32_t sq = __shfl_sync(0xffffffffu, s_l, (i + lane) & 31);
            const bool live = i + lane < lim && lane < W;
            const uint64_t mine = lane < W ? cur[lane] : ~0ull;
            const int pool = (int)(mine & 1023u);
            const int had = live ? cnt[pool] : 0;
            const bool full = had + 1 >= P;
            const uint64_t put = live && !full ? mine + ((uint64_t)w_s << 10) : ~0ull;
            uint64_t before = put;               // smallest key put back by the lanes below this one
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint64_t other = __shfl_up_sync(0xffffffffu, before, o);
                if (lane >= o && other < before) before = other;
            }
            before = __shfl_up_sync(0xffffffffu, before, 1);
            if (lane == 0) before = ~0ull;
            const unsigned fits = __ballot_sync(0xffffffffu, live && mine < before);
            const int take = (~fits == 0u) ? 32 : __ffs(~fits) - 1;   // >= 1: the first key always fits
            const bool placed = lane < take;
            if (placed) {
                order[(int64_t)pool * P + had] = sq;   // pools are laid end to end in pool order
                pool_of_seq[sq] = pool;
                cnt[pool] = had + 1;
                if (full) pool_load[pool] = (int64_t)(mine >> 10) + w_s;
            }
            const unsigned keep = __ballot_sync(0xffffffffu, placed && !full);
            const int nput = __popc(keep);
            if (placed && !full) put_raw[__popc(keep & ((1u << lane) - 1u))] = put;
            __syncwarp();
            if (lane < nput) {
                const uint64_t k = put_raw[lane];
                int rank = 0;
                for (int j = 0; j < nput; ++j) rank += put_raw[j] < k ? 1 : 0;   // all keys differ
                back[rank] = k;
            }
            __syncwarp();
            const int na = W - take;
            for (int idx = lane; idx < na; idx += 32) {
                const uint64_t k = cur[take + idx];
                int lo = 0, hi = nput;
                while (lo < hi) { const int mid = (lo + hi) >> 1; if (back[mid] < k) lo = mid + 1; else hi = mid; }
                nxt[idx + lo] = k;
            }
            if (lane < nput) {
                const uint64_t k = back[lane];
                int lo = 0, hi = na;
                while (lo < hi) { const int mid = (lo + hi) >> 1; if (cur[take + mid] < k) lo = mid + 1; else hi = mid; }
                nxt[lane + lo] = k;
            }
            __syncwarp();
            uint64_t* tmp = cur; cur = nxt; nxt = tmp;
            W = na + nput;
            i += take;
        }
        s_l = s_n;
        w_l = w_n;
    }
}

// Work that may add up beyond 53 bits, or negative work (which no sequence has): one sequence after the other, an
// arg-min over all pools each (0.45 us a sequence with 128 pools).  Pool k's load and fill count live in lane
// k % 32, register k / 32; a full pool's load is replaced by INT64_MAX in the comparison, which is
// what removing it from the algorithm's heap does.  Popping the heap's minimum (load, k) is the
// lexicographic arg-min taken here.
template <int PER>
__global__ void __launch_bounds__(32) k_vrsp_place(const int64_t* __restrict__ work, const int32_t* __restrict__ sorted,
                                                   int D, int P, int K, int32_t* __restrict__ order,
                                                   int32_t* __restrict__ pool_of_seq, int64_t* __restrict__ pool_load) {
    const int lane = threadIdx.x;
    {   // sorted descending: the first work bounds every load, the last one tells whether any is negative
        extern __shared__ __align__(16) uint64_t keys[];   // two key arrays and the fill counts, K entries each
        const int64_t most = work[sorted[0]], least = work[sorted[D - 1]];
        if (least >= 0 && most < (int64_t(1) << 52) / P) {
            vrsp_place_waves(work, sorted, D, P, K, order, pool_of_seq, pool_load, keys, keys + K,
                             reinterpret_cast<int32_t*>(keys + 2 * K));
            return;
        }
    }
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
    k_vrsp_work<<<(n_sequences + 7) / 8, 256, 0, s>>>(sample_offsets_dev, seq_first_sample_dev, n_sequences, work_dev);
    count_launch(1);
    return cudaGetLastError() == cudaSuccess ? LIBRA_OK : LIBRA_ERR_CUDA;
}

extern "C" int libra_vrsp_place(const int64_t* work_dev, int n_sequences, int pool_size, int32_t* order_dev,
                                int32_t* pool_of_seq_dev, int64_t* pool_load_dev, int32_t* scratch_dev, void* stream) {
    if (!work_dev || !order_dev || !pool_of_seq_dev || !pool_load_dev || !scratch_dev) return LIBRA_ERR_INVALID_ARG;
    if (n_sequences <= 0 || pool_size <= 0 || n_sequences % pool_size != 0) return LIBRA_ERR_INVALID_ARG;
    const int D = n_sequences, P = pool_size, K = D / P;
    if (K > 1024 || D > (1 << 20)) return LIBRA_ERR_UNSUPPORTED;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t smem = (size_t)K * (2 * sizeof(uint64_t) + sizeof(int32_t));   // at most 20 KB
    k_vrsp_rank<<<(D + 15) / 16, 256, 0, s>>>(work_dev, D, scratch_dev);
    if (K <= 32)
        k_vrsp_place<1><<<1, 32, smem, s>>>(work_dev, scratch_dev, D, P, K, order_dev, pool_of_seq_dev, pool_load_dev);
    else if (K <= 128)
        k_vrsp_place<4><<<1, 32, smem, s>>>(work_dev, scratch_dev, D, P, K, order_dev, pool_of_seq_dev, pool_load_dev);
    else
        k_vrsp_place<32><<<1, 32, smem, s>>>(work_dev, scratch_dev, D, P, K, order_dev, pool_of_seq_dev, pool_load_dev);
    count_launch(2);
    return cudaGetLastError() == cudaSuccess ? LIBRA_OK : LIBRA_ERR_CUDA;
}
