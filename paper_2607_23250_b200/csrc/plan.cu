// Device tile planner: SH-Tile construction (Section 4.3.1, Eq. 5), tile weights (Eq. 6) and
// heaviest-first placement (Algorithm 2 with a zero communication term) as CUDA kernels.
//
// Integer work only; every result must equal the step-by-step definition bit for bit.
#include <stdio.h>

#include <mutex>
#include <new>

#include "common.h"
#include "waves.cuh"

namespace libra {

std::atomic<int64_t> g_launches{0};

static std::atomic<int> g_cfg[kMaxDevices][kCfgSlots];
bool cfg_done(int slot) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return false;
    return g_cfg[dev][slot].load(std::memory_order_acquire) != 0;
}
void cfg_mark(int slot) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return;
    g_cfg[dev][slot].store(1, std::memory_order_release);
}
int check_plan_device(const libra_plan* plan) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return LIBRA_ERR_NO_DEVICE;
    return dev == plan->device ? LIBRA_OK : LIBRA_ERR_PLAN_MISMATCH;
}

namespace {
struct ScratchPools {
    std::mutex mu;
    cudaMemPool_t pool[kMaxDevices] = {};
    ~ScratchPools() {
        for (cudaMemPool_t q : pool)
            if (q) cudaMemPoolDestroy(q);
    }
};
}  // namespace

cudaError_t scratch_alloc(void** p, size_t bytes, cudaStream_t s) {
    static ScratchPools pools;
    int dev = 0;
    if (const cudaError_t e = cudaGetDevice(&dev); e != cudaSuccess) return e;
    cudaMemPool_t pool = nullptr;
    // A stream under capture takes the driver's default pool: the first call could not make one of our own there, and the
    // memory belongs to the graph anyway.
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (s)   // (the legacy stream cannot be captured)
        if (const cudaError_t e = cudaStreamIsCapturing(s, &capture); e != cudaSuccess) return e;
    if (capture == cudaStreamCaptureStatusNone && dev >= 0 && dev < kMaxDevices) {
        std::lock_guard<std::mutex> lock(pools.mu);
        if (!pools.pool[dev]) {
            cudaMemPoolProps props = {};
            props.allocType = cudaMemAllocationTypePinned;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = dev;
            cudaMemPool_t made;
            if (cudaMemPoolCreate(&made, &props) == cudaSuccess) {
                uint64_t keep = kPoolKeep;
                cudaMemPoolSetAttribute(made, cudaMemPoolAttrReleaseThreshold, &keep);
                pools.pool[dev] = made;
            } else {
                cudaGetLastError();   // no pool of our own: the driver's default one below
            }
        }
        pool = pools.pool[dev];
    }
    return pool ? cudaMallocFromPoolAsync(p, bytes, pool, s) : cudaMallocAsync(p, bytes, s);
}

// ---- kernels --------------------------------------------------------------------------------

// cu_seqlens checks (starts at 0, non-decreasing, ends at T) and, for every token, the bounds [start, end) of the sample
// that holds it.  The search keeps every index inside [0, n] whatever cu contains, and the bounds are clamped to
// start <= t < end <= T, so that a malformed cu_seqlens (flagged in *status) can never make a
// later kernel form an address outside its tensors.
__global__ void k_token_bounds(const int32_t* __restrict__ cu, int n, int64_t T, int32_t* __restrict__ tok_start,
                               int32_t* __restrict__ tok_end, int* status) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t <= n) {
        bool bad = false;
        if (t == 0 && cu[0] != 0) bad = true;
        if (t == n && cu[n] != T) bad = true;
        if (t < n && cu[t + 1] < cu[t]) bad = true;
        if (bad) atomicExch(status, LIBRA_ERR_BAD_SEQLENS);
    }
    if (t >= T) return;
    int lo = 0, hi = n;  // find the last j in [0, n) with cu[j] <= t
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (cu[mid] <= t) lo = mid; else hi = mid;
    }
    const int64_t a = cu[lo], e = cu[lo + 1];
    tok_start[t] = (int32_t)(a < 0 ? 0 : (a > t ? t : a));
    tok_end[t] = (int32_t)(e < t + 1 ? t + 1 : (e > T ? T : e));
}

// What the kernels below need of one direction; the directions of a plan share launches.
struct DirView {
    int64_t NB, NT;
    int tile, H, W, key_major, g, unit_cost;   // g: cost_block of LIBRA_WEIGHT_BLOCKS, 0 = pair counts
    int64_t* weight_blk;
    int32_t* blk_order;     // null: pair tiles (id = head * NB + block, placed in id order)
    int32_t* cta_of_tile;
    int32_t* pos;
    int32_t* cta_offsets;
    int32_t* cta_tiles;
    int32_t* cta_exec;
    int64_t* loads;
};
struct DirViews {
    DirView v[libra_plan::kDirs];
};

// Weight of block b (Eq. 6): a token at position p of a sample of length len contributes
// p + 1 pairs as a query (keys 0..p) and len - p pairs as a key (queries p..len-1).
// Block-count weight (LIBRA_WEIGHT_BLOCKS): the token axis is cut into chunks at multiples of g.  For a
// chunk of query rows [r0, r1] the visible keys span the chunks from the one holding the first key of r0's
// sample to the one holding r1 (row r0 sees a key in every chunk of that range, later rows see no chunk
// outside it); for a chunk of keys [c0, c1] the attending queries span the chunks from the one holding c0
// to the one holding the last token of c1's sample.
// One warp per block (a thread per block read its tokens one after the other: 20 us at 32768 tokens, 4 now).
__global__ void k_block_weights(const int32_t* __restrict__ tok_start, const int32_t* __restrict__ tok_end,
                                int64_t T, const DirViews views) {
    const DirView& d = views.v[blockIdx.y];
    const int64_t b = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (b >= d.NB) return;
    const int64_t t0 = b * d.tile;
    const int64_t t1 = (t0 + d.tile < T) ? t0 + d.tile : T;
    int64_t w = 0;
    if (d.g == 0) {
        for (int64_t t = t0 + lane; t < t1; t += 32)
            w += d.key_major ? (int64_t)tok_end[t] - t : t - (int64_t)tok_start[t] + 1;
    } else {
        for (int64_t c = t0 / d.g + lane; c * d.g < t1; c += 32) {
            const int64_t first = c * d.g > t0 ? c * d.g : t0;
            const int64_t last = ((c + 1) * d.g < t1 ? (c + 1) * d.g : t1) - 1;
            const int64_t n = d.key_major ? ((int64_t)tok_end[last] - 1) / d.g - first / d.g + 1
                                          : last / d.g - (int64_t)tok_start[first] / d.g + 1;
            w += 8 * n + d.unit_cost;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
    if (lane == 0) d.weight_blk[b] = w;
}

// Order of Algorithm 2: decreasing weight, then increasing id.  All H shards of a block weigh
// the same and their ids b*H+h are consecutive, so ordering the blocks orders the tiles.
// rank(b) = number of blocks that precede b; sixteen lanes share a block's comparisons.
__global__ void __launch_bounds__(256) k_rank_blocks(const DirViews views) {
    const DirView& d = views.v[blockIdx.y];
    __shared__ int64_t sw[1024];
    if (blockIdx.x * (int64_t)16 >= d.NB) return;
    const int64_t b = blockIdx.x * (int64_t)16 + (threadIdx.x >> 4);
    const int sub = threadIdx.x & 15;
    const int64_t wb = b < d.NB ? d.weight_blk[b] : 0;
    int rank = 0;
    for (int64_t base = 0; base < d.NB; base += 1024) {
        const int lim = (int)(d.NB - base < 1024 ? d.NB - base : 1024);
        for (int o = threadIdx.x; o < lim; o += 256) sw[o] = d.weight_blk[base + o];
        __syncthreads();
        for (int k = sub; k < lim; k += 16) {
            const int64_t w = sw[k];
            rank += (w > wb) || (w == wb && base + k < b);
        }
        __syncthreads();
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
    if (b < d.NB && sub == 0) d.blk_order[rank] = (int32_t)b;
}

// Placement (Algorithm 2's greedy rule: the next tile goes to the least-loaded worker, lowest index among equals) in
// waves, one block per direction (waves.cuh).  There are at most 1024 workers, so a key has 54 bits for the load: enough for
// pair counts by the host's bound on H T^2; block counts with a large unit cost can exceed them, which k_check_loads finds
// in the lists (they hold every tile once all the same, in no particular balance).  Tiles come in batches held in shared
// memory, the next batch in registers.  Both directions of 131072 tokens with 32 / 8 heads (16384 and 13464 tiles): 0.6 ms,
// by a warp per direction 1.4 ms; of two 65536-token samples (69632 pair tiles): 1.5 and 5.3 ms.
constexpr int kPlaceBatch = 512;

__global__ void __launch_bounds__(kWaveMaxBins) k_place(const DirViews views) {
    const DirView& jb = views.v[blockIdx.x];
    __shared__ WaveSmem sm;
    __shared__ int32_t cnt[kWaveMaxBins];        // tiles per worker so far
    __shared__ int64_t wbuf[kPlaceBatch];
    __shared__ int32_t tbuf[kPlaceBatch];
    __shared__ int32_t warp_sum[32];
    const int i = threadIdx.x, nthr = blockDim.x, lane = i & 31, warp = i >> 5;
    const int64_t NT = jb.NT, NB = jb.NB;
    const int H = jb.H, W = jb.W;
    if (i < W) sm.key[0][i] = (uint64_t)i;
    cnt[i] = 0;
    const int batch = 4 * nthr < kPlaceBatch ? 4 * nthr : kPlaceBatch;
    int64_t w_n[4];
    int32_t t_n[4];
    auto fetch = [&](int64_t x0) {               // this thread's tiles of the batch at position x0 of the order
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t x = x0 + i + (int64_t)k * nthr;
            w_n[k] = 0;
            t_n[k] = 0;
            if (i + k * nthr < batch && x < NT) {
                const int64_t blk = jb.blk_order ? jb.blk_order[x / H] : x % NB;
                w_n[k] = jb.weight_blk[blk];
                t_n[k] = jb.blk_order ? (int32_t)(blk * H + x % H) : (int32_t)x;   // pair tiles: in id order
            }
        }
    };
    fetch(0);
    int cur = 0;
    for (int64_t x0 = 0; x0 < NT; x0 += batch) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i + k * nthr < batch) { wbuf[i + k * nthr] = w_n[k] > 0 ? w_n[k] : 0; tbuf[i + k * nthr] = t_n[k]; }
        __syncthreads();
        fetch(x0 + batch);
        const int lim = (int)(NT - x0 < batch ? NT - x0 : batch);
        for (int b = 0; b < lim;) {
            const bool live = i < W && b + i < lim;
            const uint64_t key = i < W ? sm.key[cur][i] : ~0ull;
            const uint64_t put = live ? key + ((uint64_t)wbuf[b + i] << 10) : ~0ull;
            const int take = wave_take(sm, key, put, live);   // >= 1: the first key always fits
            if (i < take) {
                const int32_t t = tbuf[b + i];
                const int r = (int)(key & 1023u), had = cnt[r];
                jb.cta_of_tile[t] = r;
                jb.pos[t] = had;
                cnt[r] = had + 1;
            }
            wave_merge(sm, cur, W, take, key, put, i < take);
            cur ^= 1;
            b += take;
        }
    }
    __syncthreads();
    if (i < W) {
        const uint64_t k = sm.key[cur][i];
        jb.loads[k & 1023u] = (int64_t)(k >> 10);
    }
    int incl = i < W ? cnt[i] : 0;               // counts -> offsets
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += v; }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    for (int w = 0; w < warp; ++w) incl += warp_sum[w];
    if (i < W) jb.cta_offsets[i + 1] = incl;
    if (i == 0) jb.cta_offsets[0] = 0;
}

__global__ void k_scatter_lists(const DirViews views) {
    const DirView& d = views.v[blockIdx.y];
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= d.NT) return;
    d.cta_tiles[d.cta_offsets[d.cta_of_tile[t]] + d.pos[t]] = (int32_t)t;
}

// Execution order inside a worker's list.  The placement fixes WHICH tiles a worker runs; the order
// it runs them in is free.  Sorting every list by (head shard, block) makes all workers sweep
// the same head and neighbouring blocks at about the same time, so that the tiles several workers
// read (K/V in the forward and the dQ kernel, Q/dO in the dK/dV kernel) are more often found in L2.
// One thread block per worker, rank sort.  (Pair tiles are placed in id order: their lists are in execution order.)
__global__ void k_exec_order(const DirViews views) {
    const DirView& d = views.v[blockIdx.y];
    const int r = blockIdx.x;
    if (!d.blk_order || r >= d.W) return;
    const int beg = d.cta_offsets[r], n = d.cta_offsets[r + 1] - beg;
    if (n > 16384) {  // quadratic sort too slow: keep placement order
        for (int i = threadIdx.x; i < n; i += blockDim.x) d.cta_exec[beg + i] = d.cta_tiles[beg + i];
        return;
    }
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int32_t t = d.cta_tiles[beg + i];
        const int64_t key = (int64_t)(t % d.H) * d.NB + t / d.H;
        int rank = 0;
        for (int j = 0; j < n; ++j) {
            const int32_t u = d.cta_tiles[beg + j];
            rank += ((int64_t)(u % d.H) * d.NB + u / d.H) < key;
        }
        d.cta_exec[beg + rank] = t;
    }
}

// Did the workers' loads of a direction fit their keys?  (~0 stands for none.)  Launched only where block counts might add
// up that far.
__global__ void k_check_loads(const DirView d, int* __restrict__ status) {
    __shared__ unsigned long long load;
    const int beg = d.cta_offsets[blockIdx.x], end = d.cta_offsets[blockIdx.x + 1];
    if (threadIdx.x == 0) load = 0;
    __syncthreads();
    const unsigned long long full = (1ull << 54) - 1;
    unsigned long long sum = 0;                       // at most `full`, so that the total fits 64 bits
    for (int i = beg + threadIdx.x; i < end; i += blockDim.x) {
        const unsigned long long w = (unsigned long long)d.weight_blk[d.cta_tiles[i] / d.H];
        sum = w < full - sum ? sum + w : full;
    }
    atomicAdd(&load, sum);
    __syncthreads();
    if (threadIdx.x == 0 && load >= full) atomicCAS(status, LIBRA_OK, LIBRA_ERR_OVERFLOW);
}

// ---- pair tiles: key block x query chunk x head (the fused backward's units) ---------------------------------
// The score matrix in tile x tile cells: cell (i, j) is live when a query of row block i attends a key of key
// block j; for a key block the live cells are the row blocks j .. last(j), last(j) = the block of the last token
// of the sample that holds the key block's last key.  Pair-block (c, j) = key block j against the R = chunk / tile
// row blocks of query chunk c, present when one of them is live; numbered chunk by chunk, key blocks ascending.
// last(j) never decreases with j, so the key blocks of a chunk are the range first(c) .. min(NKB, (c+1) R) - 1.
// Key blocks of kt tokens against row blocks of rt tokens (kt a multiple of rt; the pair tiles proper have kt = rt).
__device__ __forceinline__ int64_t pair_last_row_block(const int32_t* tok_end, int64_t T, int kt, int rt, int64_t j) {
    const int64_t last_key = ((j + 1) * kt < T ? (j + 1) * kt : T) - 1;
    return ((int64_t)tok_end[last_key] - 1) / rt;
}
// Chunk sizes under consideration, for the tiles proper and the wide ones: one block each finds the key-block range of
// every query chunk, the exclusive prefix sum of the counts and their total (base[NC] and totals[block]); one more block
// for either finds the most live cells of a key block (totals[kPairCands + k]) and the sum over all of them
// (totals[kPairCands + 2 + k]).
struct PairTables { int dir = 0, kt = 0, R = 0; int32_t* first_j = nullptr; int32_t* count = nullptr; int64_t* base = nullptr; int64_t NC = 0; };
constexpr int kChunkSizes = 6, kPairCands = 3 * kChunkSizes, kPairTotals = kPairCands + 4;
struct PairCands { PairTables c[kPairCands]; int n = 0; int rt = 0; int kt[2] = {}; int n_longest = 0; };
__global__ void __launch_bounds__(1024) k_pair_chunks(const int32_t* __restrict__ tok_end, int64_t T, const __grid_constant__ PairCands cands,
                                                      int64_t* __restrict__ totals) {
    const int rt = cands.rt;
    if ((int)blockIdx.x >= cands.n) {
        __shared__ int longest;
        __shared__ unsigned long long cells;
        const int k = blockIdx.x - cands.n, kt = cands.kt[k];
        if (threadIdx.x == 0) { longest = 0; cells = 0; }
        __syncthreads();
        int most = 0;
        unsigned long long sum = 0;
        for (int64_t j = threadIdx.x; j * kt < T; j += 1024) {
            const int64_t n = pair_last_row_block(tok_end, T, kt, rt, j) - j * kt / rt + 1;
            most = n > most ? (int)n : most;
            sum += n;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if ((threadIdx.x & 31) == 0) atomicAdd(&cells, sum);   // (64 bits by every thread: 25 us)
        atomicMax(&longest, most);
        __syncthreads();
        if (threadIdx.x == 0) { totals[kPairCands + k] = longest; totals[kPairCands + 2 + k] = (int64_t)cells; }
        return;
    }
    const PairTables& t = cands.c[blockIdx.x];
    const int kt = t.kt, R = t.R;
    const int64_t NKB = (T + kt - 1) / kt, NC = t.NC;
    int32_t *first_j = t.first_j, *count = t.count;
    int64_t* base = t.base;
    __shared__ int64_t part[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t run = 0;
    for (int64_t c0 = 0; c0 < NC; c0 += 1024) {
        const int64_t c = c0 + threadIdx.x;
        int64_t n = 0;
        if (c < NC) {
            int64_t lo = 0, hi = NKB;   // first j with last(j) / R >= c
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if (pair_last_row_block(tok_end, T, kt, rt, mid) / R >= c) hi = mid; else lo = mid + 1;
            }
            const int64_t end = ((c + 1) * R * rt - 1) / kt;   // the key block of the chunk's last row
            const int64_t last = end < NKB - 1 ? end : NKB - 1;
            n = last >= lo ? last - lo + 1 : 0;
            first_j[c] = (int32_t)lo;
            count[c] = (int32_t)n;
        }
        int64_t incl = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int64_t v = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += v; }
        if (lane == 31) part[warp] = incl;
        __syncthreads();
        int64_t before = 0, all = 0;
        for (int w = 0; w < 32; ++w) { if (w < warp) before += part[w]; all += part[w]; }
        if (c < NC) base[c] = run + before + incl - n;
        run += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) { base[NC] = run; totals[blockIdx.x] = run; }
}
// Weight of pair-block (c, j): its live cells, min(last(j), c R + R - 1) - max(j, c R) + 1.
__global__ void k_pair_fill(const int32_t* __restrict__ tok_end, int64_t T, int kt, int rt, int R, int64_t NC,
                            const int32_t* __restrict__ first_j, const int32_t* __restrict__ count,
                            const int64_t* __restrict__ base, int32_t* __restrict__ u_blk,
                            int32_t* __restrict__ u_chunk, int64_t* __restrict__ weight_blk) {
    const int64_t c = blockIdx.x;
    if (c >= NC) return;
    for (int x = threadIdx.x; x < count[c]; x += blockDim.x) {
        const int64_t j = first_j[c] + x, u = base[c] + x;
        const int64_t last = pair_last_row_block(tok_end, T, kt, rt, j), first = j * kt / rt;
        const int64_t i0 = first > c * R ? first : c * R, i1 = last < c * R + R - 1 ? last : c * R + R - 1;
        u_blk[u] = (int32_t)j;
        u_chunk[u] = (int32_t)c;
        weight_blk[u] = i1 - i0 + 1;
    }
}

// Expanders used by libra_plan_export.
__global__ void k_expand_weight(const int64_t* __restrict__ weight_blk, int64_t NT, int H, int64_t NB_headmajor,
                                int64_t* __restrict__ out) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t < NT) out[t] = NB_headmajor ? weight_blk[t % NB_headmajor] : weight_blk[t / H];
}
__global__ void k_expand_order(const int32_t* __restrict__ blk_order, int64_t NT, int H, int32_t* __restrict__ out) {
    const int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (x < NT) out[x] = blk_order ? (int32_t)((int64_t)blk_order[x / H] * H + x % H) : (int32_t)x;
}

// ---- host ---------------------------------------------------------------------------------

static inline unsigned grid_for(int64_t n, int block) { return (unsigned)((n + block - 1) / block); }

// The plan's device memory: two stream-ordered blocks, carved into arrays.  (A cudaMalloc and a cudaFree per
// array cost 0.5 + 0.4 ms a plan, and now and then ten times that.)
static int plan_block(libra_plan* p, size_t bytes, uint8_t** out) {
    if (p->n_blocks == libra_plan::kMaxBlocks) return LIBRA_ERR_CUDA;
    // A stream-ordered allocation would become part of a graph that is being captured, and the plan's memory would only
    // exist while the graph runs.  A plain one outlives it where the capture's mode allows it, and fails elsewhere.
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    void* q = nullptr;
    cudaError_t e = p->stream ? cudaStreamIsCapturing(p->stream, &capture) : cudaSuccess;
    p->plain_memory = capture != cudaStreamCaptureStatusNone;
    if (e == cudaSuccess) e = p->plain_memory ? cudaMalloc(&q, bytes ? bytes : 1) : scratch_alloc(&q, bytes ? bytes : 1, p->stream);
    if (e != cudaSuccess) return LIBRA_ERR_CUDA;
    p->blocks[p->n_blocks++] = q;
    *out = reinterpret_cast<uint8_t*>(q);
    return LIBRA_OK;
}
struct Carver {
    uint8_t* at = nullptr;   // null: only sizes are added up
    size_t used = 0;
    template <typename X>
    void take(X** p, int64_t n) {
        if (at) *p = reinterpret_cast<X*>(at + used);
        used += (sizeof(X) * (size_t)(n ? n : 1) + 255) & ~size_t(255);
    }
};
// Arrays that start out as zeros (`zeros`), then the rest.
static void carve_dir(PlanDir& d, Carver& c, bool zeros, bool pairs) {
    if (zeros) {
        c.take(&d.d_busy, 2 * (d.W + 1));    // kernels on pairs of CTAs round the workers up to even
        c.take(&d.d_busy2, 2 * (d.W + 1));
        c.take(&d.d_tile_ns, d.NT);
        return;
    }
    c.take(&d.d_weight_blk, d.NB);
    if (!pairs) c.take(&d.d_blk_order, d.NB);
    c.take(&d.d_cta_of_tile, d.NT);
    c.take(&d.d_pos, d.NT);
    c.take(&d.d_cta_offsets, d.W + 1);
    c.take(&d.d_cta_tiles, d.NT);
    if (!pairs) c.take(&d.d_cta_exec, d.NT);
    c.take(&d.d_loads, d.W);
    if (pairs) {
        c.take(&d.d_u_blk, d.NB);
        c.take(&d.d_u_chunk, d.NB);
        d.d_cta_exec = d.d_cta_tiles;   // placed in id order: the lists already are in execution order
    }
}

// Sizes a direction's kernels and tables can take; NB is known.
static int check_dir(const libra_plan* p, PlanDir& d, bool pairs) {
    const int64_t T = p->T;
    if (d.NB * (int64_t)d.H >= (int64_t)INT32_MAX) return LIBRA_ERR_OVERFLOW;
    // a worker's load is at most the weight total <= H * T^2 / 2 + ...; the placement packs load * 1024 + index
    if ((long double)d.H * (long double)T * (long double)T >= 9.0e15L) return LIBRA_ERR_OVERFLOW;
    if (!pairs && d.NB > 65536) return LIBRA_ERR_UNSUPPORTED;  // the rank sort is quadratic in blocks
    if (d.W > kWaveMaxBins) return LIBRA_ERR_UNSUPPORTED;
    d.NT = d.NB * d.H;
    return LIBRA_OK;
}

static DirView view_of(const PlanDir& d, int key_major, const libra_plan_opts& o) {
    DirView v = {};
    v.NB = d.NB; v.NT = d.NT; v.tile = d.tile; v.H = d.H; v.W = d.W; v.key_major = key_major;
    v.g = o.weight_model == LIBRA_WEIGHT_BLOCKS ? (o.cost_block ? o.cost_block : 128) : 0;
    v.unit_cost = key_major ? o.unit_cost_kv : o.unit_cost_q;
    v.weight_blk = d.d_weight_blk; v.blk_order = d.d_blk_order; v.cta_of_tile = d.d_cta_of_tile; v.pos = d.d_pos;
    v.cta_offsets = d.d_cta_offsets; v.cta_tiles = d.d_cta_tiles; v.cta_exec = d.d_cta_exec; v.loads = d.d_loads;
    return v;
}

// ---- the pair-blocks of a plan: one table per chunk size under consideration; their totals are read back in one synchronous
// copy and decide the size.
static int64_t pair_chunks_of(int64_t T, int rt, int R) { return ((T + rt - 1) / rt + R - 1) / R; }
// Chunk sizes for direction k, the largest first: the one asked for, or halves down to a row block.
static void add_pair_cands(const libra_plan* p, PairCands& cands, int k, bool halves) {
    const PlanDir& d = p->dir[k];
    int R = d.chunk / cands.rt;
    for (int x = 0; x < (halves ? kChunkSizes : 1) && R > 0; ++x, R /= 2) {
        PairTables& t = cands.c[cands.n++];
        t.dir = k;
        t.kt = d.tile;
        t.R = R;
        t.NC = pair_chunks_of(p->T, cands.rt, R);
    }
}
// The chunk size of direction k.  In units of one cell of one query head (3.1 us), a worker's time over its mean is about
// the tiles it starts, 3 each (operands in, accumulators out), and up to the length of one tile, R cells of G heads: idle
// at the end.  Backward (us) with the best of 4096 ... 128 rows and with 4096: one sequence of 1500 tokens, 32 / 8 heads: 256, 97
// (133); 10007 tokens in samples of up to 400, 8 / 2 heads: 128, 86 (109); one of 4000, 8 / 2 heads: 512, 114 (289); 12000 tokens,
// 4 / 1 heads: 1024, 407 (426); 16000, 32 / 4 heads: 1024, 5190 (5230); 8 samples of 4096, 32 / 8 heads: 4096, 3320, with 128: 4350;
// one sample of 32768: 4096, 21.0 ms, 2048: 21.3, 128: 29.9.  On 13 further pools the choice was within 4 % of the best.
static const PairTables* choose_pair_chunk(const libra_plan* p, const PairCands& cands, const int64_t* totals, int k, double G) {
    const PairTables* best = nullptr;
    double least = 0;
    for (int x = 0; x < cands.n; ++x) {
        const PairTables& t = cands.c[x];
        if (t.dir != k || totals[x] > 262144) continue;
        const double longest = (double)totals[kPairCands + k - 2];
        const double cost = 3.0 * totals[x] * p->dir[k].H / p->dir[k].W + G * (t.R < longest ? t.R : longest);
        if (!best || cost < least) { best = &t; least = cost; }
    }
    return best;
}
// Whether the fused backward runs on pairs of CTAs with 256 keys a tile, from the live 128 x 128 cells and the 256 x 128 ones.
// A pair's cell costs it as much where only one of its key blocks sees the row block.  That is so at the diagonal, once a
// wide key block, and in the row blocks past the end of the lower key block's samples.  Backward on pairs over the same on single
// CTAs, fitted to 44 pools of 30000 to 131072 tokens (log-normal and equal samples of 300 to 5000, 148 workers): 0.96 + 0.12
// diagonal + 0.65 past ends, as shares of the live cells; to 44 of 8200 to 33000 on 16 workers 0.93 + 0.66 + 0.83.  The line lies
// between the two.  Some of the pools, single / pairs in us with 148 workers, 32 / 8 or 8 / 2 heads: 20 samples of the usual
// log-normal mix in 33000 tokens 6192 / 5732 at past ends + 0.4 diagonal = 0.009, 32 of 1024 1319 / 1263 (0.044), 43 of 3000 2764 /
// 2738 (0.050), log-normal of median 500 2760 / 2755 (0.059); and beyond the line 62 of 2100 2187 / 2223 (0.071), 119 of 1100
// 1489 / 1564 (0.121), 204 of 640 1051 / 1124 (0.233).
// An odd worker has no CTA to pair with, and with it goes the balance of longer lists: 4096 tokens, 8 / 2 heads, on 7, 9, 13, 37, 63 and
// 147 workers: single / pairs 0.92, 0.94, 0.95, 0.98, 1.01, 1.04; 16384 tokens on 9, 37, 147: 0.98, 1.05, 1.06.
// Of a pool with few tiles a worker the launch counts and the coarser tiles leave more of the last round idle, as far as the
// chunk was the planner's to choose: 1500 tokens, 8 / 2 heads, a chunk of one row block: 40.2 us on single CTAs and 42.8 on pairs; 1500,
// 32 / 8 heads, 2.3 tiles a worker: 91.7 and 100.0; 3000, 8 / 2 heads, 2.1: 91.0 and 102.8; 9 samples of 1024, 2.4: 115.6 and 109.0; 4096, 3.7:
// 115.1 and 110.8.
static bool fused_on_pairs(const libra_plan* p, int64_t cells, int64_t wide_cells, int64_t wide_tiles, int R, bool own_choice) {
    const int64_t wide_blocks = (p->T + 255) / 256;
    const double past_ends = (double)(2 * wide_cells - cells - wide_blocks) / cells, diagonal = (double)wide_blocks / cells;
    const double cost = 0.94 + past_ends + 0.4 * diagonal + (p->W % 2 ? 2.0 / p->W : 0.0);
    if (cost >= 1.0) return false;
    return !own_choice || (R > 1 && wide_tiles * p->dir[4].H >= 2.4 * p->dir[4].W);
}
static double heads_per_kv(const libra_plan* p) { return p->dir[0].H > p->dir[2].H ? (double)p->dir[0].H / p->dir[2].H : 1.0; }
// Counts, choice and, while every size has more than 262144 pair-blocks, twice the largest.  `pairs`: whether the fused kernel's
// wide tiles are under consideration, and whether they were taken.
static int count_pair_blocks(libra_plan* p, PairCands& cands, int64_t* d_totals, PairTables (&chosen)[libra_plan::kDirs], double G,
                             bool own_choice, bool& pairs) {
    const int dirs = cands.n_longest;
    for (;;) {
        int64_t totals[kPairTotals];
        k_pair_chunks<<<cands.n + dirs, 1024, 0, p->stream>>>(p->d_tok_end, p->T, cands, d_totals);
        count_launch();
        if (cudaMemcpyAsync(totals, d_totals, sizeof(totals), cudaMemcpyDeviceToHost, p->stream) != cudaSuccess ||
            cudaStreamSynchronize(p->stream) != cudaSuccess)
            return LIBRA_ERR_CUDA;
        bool all = true;
        for (int k = 2; k < 2 + dirs; ++k) {
            const PairTables* t = choose_pair_chunk(p, cands, totals, k, G);
            if (t) {
                p->dir[k].NB = totals[t - cands.c];
                p->dir[k].chunk = t->R * cands.rt;
                chosen[k] = *t;
                continue;
            }
            all = false;
            for (int x = 0; x < cands.n; ++x) {
                PairTables& c = cands.c[x];
                if (c.dir != k && !(k == 2 && c.dir == 4)) continue;
                if ((int64_t)c.R * 2 * cands.rt > (int64_t)1 << 30) return LIBRA_ERR_UNSUPPORTED;
                c.R *= 2;
                c.NC = pair_chunks_of(p->T, cands.rt, c.R);   // never more than the tables were carved for
            }
        }
        if (!all) continue;
        for (int x = 0; x < cands.n && pairs; ++x)   // the fused kernel's wide tiles have the chunks of the others
            if (cands.c[x].dir == 4 && cands.c[x].R == chosen[2].R) {
                p->dir[4].NB = totals[x];
                p->dir[4].chunk = p->dir[2].chunk;
                chosen[4] = cands.c[x];
            }
        if (pairs) pairs = fused_on_pairs(p, totals[kPairCands + 2], totals[kPairCands + 3], p->dir[4].NB, chosen[2].R, own_choice);
        return LIBRA_OK;
    }
}

// Placement and lists of n directions, side by side.
static void place_lists(const DirViews& views, int n, int max_w, int64_t max_nt, cudaStream_t s) {
    k_place<<<n, (max_w + 31) / 32 * 32, 0, s>>>(views);
    k_scatter_lists<<<dim3(grid_for(max_nt > 0 ? max_nt : 1, 256), n), 256, 0, s>>>(views);
    count_launch(2);
}

// Builds the directions asked for; p->dir[k].tile / H / W / chunk are set.
static int build_plan(libra_plan* p, const int32_t* cu, const libra_plan_opts& o, const bool (&want)[libra_plan::kDirs]) {
    constexpr int kDirs = libra_plan::kDirs;
    const int64_t T = p->T;
    cudaStream_t s = p->stream;
    const bool wide_pairs = want[3] && want[2];                   // the wide tiles are pair tiles
    const bool sorted[kDirs] = {want[0], want[1], false, want[3] && !want[2], false};   // sizes known, placed heaviest first
    bool pairs[kDirs] = {false, false, want[2], wide_pairs, want[4]};
    for (int k = 0; k < kDirs; ++k) {
        if (!sorted[k]) continue;
        p->dir[k].NB = (T + p->dir[k].tile - 1) / p->dir[k].tile;
        if (const int rc = check_dir(p, p->dir[k], false); rc != LIBRA_OK) return rc;
    }
    PairCands cands;
    PairTables chosen[kDirs];
    int64_t* d_totals = nullptr;
    if (want[2]) {
        if (p->dir[2].chunk % p->dir[2].tile) return LIBRA_ERR_INVALID_ARG;
        cands.rt = p->dir[2].tile;
        cands.n_longest = wide_pairs ? 2 : 1;
        for (int k = 2; k < kDirs; ++k) {
            if (!pairs[k]) continue;
            if (k < 4) cands.kt[k - 2] = p->dir[k].tile;
            add_pair_cands(p, cands, k, o.pair_chunk == 0);
        }
    }
    // ---- token bounds, the directions whose sizes are known, the pair tables; zeros first
    size_t zero_bytes = 0;
    auto carve = [&](Carver& c) {
        c.take(&p->d_status, 1);
        for (int k = 0; k < 4; ++k) c.take(&p->d_outcome[k], p->W + 1);
        for (int k = 0; k < kDirs; ++k)
            if (sorted[k]) carve_dir(p->dir[k], c, true, false);
        zero_bytes = c.used;
        c.take(&p->d_tok_start, T);
        c.take(&p->d_tok_end, T);
        for (int k = 0; k < kDirs; ++k)
            if (sorted[k]) carve_dir(p->dir[k], c, false, false);
        if (want[2]) {
            c.take(&d_totals, kPairTotals);
            for (int x = 0; x < cands.n; ++x) {
                PairTables& t = cands.c[x];
                c.take(&t.first_j, t.NC);
                c.take(&t.count, t.NC);
                c.take(&t.base, t.NC + 1);
            }
        }
    };
    Carver sizes, mem;
    carve(sizes);
    if (const int rc = plan_block(p, sizes.used, &mem.at); rc != LIBRA_OK) return rc;
    carve(mem);
    cudaMemsetAsync(mem.at, 0, zero_bytes, s);
    const int64_t span = T > p->n + 1 ? T : p->n + 1;
    k_token_bounds<<<grid_for(span, 256), 256, 0, s>>>(cu, p->n, T, p->d_tok_start, p->d_tok_end, p->d_status);
    count_launch();
    // ---- pair tiles: their number comes back, then their arrays
    if (want[2]) {
        if (const int rc = count_pair_blocks(p, cands, d_totals, chosen, heads_per_kv(p), o.pair_chunk == 0, pairs[4]); rc != LIBRA_OK)
            return rc;
        Carver ps, pm;
        size_t pair_zero = 0;
        for (int k = 2; k < kDirs; ++k) {
            if (!pairs[k]) continue;
            if (const int rc = check_dir(p, p->dir[k], true); rc != LIBRA_OK) return rc;
            p->dir[k].d_first_j = chosen[k].first_j;
            p->dir[k].d_base = chosen[k].base;
        }
        auto carve_pairs = [&](Carver& c) {
            for (int k = 2; k < kDirs; ++k)
                if (pairs[k]) carve_dir(p->dir[k], c, true, true);
            pair_zero = c.used;
            for (int k = 2; k < kDirs; ++k)
                if (pairs[k]) carve_dir(p->dir[k], c, false, true);
        };
        carve_pairs(ps);
        if (const int rc = plan_block(p, ps.used, &pm.at); rc != LIBRA_OK) return rc;
        carve_pairs(pm);
        cudaMemsetAsync(pm.at, 0, pair_zero, s);
        for (int k = 2; k < kDirs; ++k) {
            if (!pairs[k]) continue;
            PlanDir& d = p->dir[k];
            const PairTables& t = chosen[k];
            k_pair_fill<<<(unsigned)t.NC, 128, 0, s>>>(p->d_tok_end, T, t.kt, cands.rt, t.R, t.NC, t.first_j, t.count, t.base, d.d_u_blk,
                                                       d.d_u_chunk, d.d_weight_blk);
            count_launch();
        }
    }
    // ---- weights, order, placement and lists of all directions together
    DirViews views = {};
    int n = 0, max_w = 0;
    int64_t max_nb = 0, max_nt = 0;
    for (int k = 0; k < kDirs; ++k)
        if (sorted[k]) {
            views.v[n++] = view_of(p->dir[k], k != 0, o);
            max_nb = p->dir[k].NB > max_nb ? p->dir[k].NB : max_nb;
        }
    if (n > 0) {
        k_block_weights<<<dim3(grid_for(max_nb * 32, 256), n), 256, 0, s>>>(p->d_tok_start, p->d_tok_end, T, views);
        k_rank_blocks<<<dim3(grid_for(max_nb, 16), n), 256, 0, s>>>(views);
        count_launch(2);
    }
    const int n_sorted = n;
    // No kernel walks the lists of the 128-key pair tiles where the fused backward has its wide ones: they are made when they
    // are exported.
    const bool listed[kDirs] = {sorted[0], sorted[1], pairs[2] && !pairs[4], sorted[3] || pairs[3], pairs[4]};
    for (int k = 2; k < kDirs; ++k)
        if (listed[k] && !sorted[k]) views.v[n++] = view_of(p->dir[k], 1, o);
    if (n == 0) return LIBRA_OK;
    for (int k = 0; k < kDirs; ++k)
        if (listed[k]) {
            max_nt = p->dir[k].NT > max_nt ? p->dir[k].NT : max_nt;
            max_w = p->dir[k].W > max_w ? p->dir[k].W : max_w;
        }
    place_lists(views, n, max_w, max_nt, s);
    if (n_sorted > 0) {
        k_exec_order<<<dim3(max_w, n_sorted), 256, 0, s>>>(views);
        count_launch();
    }
    for (int k = 0; k < 2; ++k) {   // (not the internal direction, whose tiles are twice as heavy: only its balance would suffer)
        if (!want[k] || o.weight_model != LIBRA_WEIGHT_BLOCKS) continue;
        const DirView v = view_of(p->dir[k], k != 0, o);
        const double chunks = (double)((T + v.g - 1) / v.g);   // at most each of them against all
        if (v.H * chunks * (8 * chunks + v.unit_cost) < 0x1p53) continue;
        k_check_loads<<<v.W, 256, 0, s>>>(v, p->d_status);
        count_launch();
    }
    for (int k = 0; k < kDirs; ++k) p->dir[k].enabled = sorted[k] || pairs[k] ? 1 : 0;
    return cudaGetLastError() == cudaSuccess ? LIBRA_OK : LIBRA_ERR_CUDA;
}

}  // namespace libra

using namespace libra;

extern "C" int libra_plan_tiles(const int32_t* cu_seqlens_dev, int n_samples, int n_heads, int tile_q,
                                const libra_plan_opts* opts, void* stream, libra_plan_t** plan_out) {
    if (!cu_seqlens_dev || !plan_out || n_samples <= 0 || n_heads <= 0 || tile_q <= 0) return LIBRA_ERR_INVALID_ARG;
    *plan_out = nullptr;
    libra_plan_opts o = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    if (opts) o = *opts;
    if (o.n_workers < 0 || o.tile_kv < 0 || o.n_heads_kv < 0 || o.total_tokens < 0) return LIBRA_ERR_INVALID_ARG;
    if (o.directions & ~(LIBRA_DIR_Q | LIBRA_DIR_KV | LIBRA_DIR_PAIR)) return LIBRA_ERR_INVALID_ARG;
    if (o.pair_chunk < 0) return LIBRA_ERR_INVALID_ARG;
    if (o.weight_model != LIBRA_WEIGHT_PAIRS && o.weight_model != LIBRA_WEIGHT_BLOCKS) return LIBRA_ERR_INVALID_ARG;
    if (o.cost_block < 0 || o.unit_cost_q < 0 || o.unit_cost_kv < 0) return LIBRA_ERR_INVALID_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return LIBRA_ERR_NO_DEVICE;
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return LIBRA_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;
    int64_t T = o.total_tokens;
    if (T == 0) {
        int32_t last = 0;
        if (cudaMemcpyAsync(&last, cu_seqlens_dev + n_samples, sizeof(int32_t), cudaMemcpyDeviceToHost, s) !=
                cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            return LIBRA_ERR_CUDA;
        T = last;
    }
    if (T <= 0 || T >= (int64_t)INT32_MAX) return LIBRA_ERR_INVALID_ARG;

    libra_plan* p = new (std::nothrow) libra_plan();
    if (!p) return LIBRA_ERR_CUDA;
    p->T = T; p->n = n_samples; p->device = dev; p->sm_count = sms; p->stream = s;
    if (s) p->other_stream = 1;
    p->W = o.n_workers ? o.n_workers : sms;
    const int dirs = o.directions ? o.directions : (LIBRA_DIR_Q | LIBRA_DIR_KV);
    const int tile_kv = o.tile_kv ? o.tile_kv : 128;
    const bool keys = (dirs & (LIBRA_DIR_KV | LIBRA_DIR_PAIR)) != 0;
    const bool want[libra_plan::kDirs] = {(dirs & LIBRA_DIR_Q) != 0, (dirs & LIBRA_DIR_KV) != 0, (dirs & LIBRA_DIR_PAIR) != 0,
                                          keys && tile_kv == 128,
                                          (dirs & LIBRA_DIR_PAIR) != 0 && tile_kv == 128 && p->W >= 2};
    for (int k = 0; k < libra_plan::kDirs; ++k) {
        PlanDir& d = p->dir[k];
        d.tile = k == 0 ? tile_q : (k >= 3 ? 256 : tile_kv);
        d.H = k == 0 ? n_heads : (o.n_heads_kv ? o.n_heads_kv : n_heads);
        d.W = k == 3 ? (p->W + 1) / 2 : (k == 4 ? p->W / 2 : p->W);
        d.chunk = k >= 2 ? (o.pair_chunk ? o.pair_chunk : 4096) : 0;
        if (k == 3) {
            // The 256-wide kernels go through a tile's heads one after the other and their workers are out of step, so what
            // the workers of a query chunk read lies anywhere in its Q and dO of a kv head's group: 1 KB a row and head,
            // 134 MB at 4096 rows of 32 heads, more than L2 holds.  At most 16384 rows x heads keep it at 16 MB (dV + dK of
            // 32768 tokens, 32 query heads per kv head: 37.0 ms with 4096 rows a chunk, 33.9 with 512; 256 gained no more).
            const int64_t rows = (int64_t)16384 * d.H / n_heads / 128 * 128;
            const int64_t least = rows < 128 ? 128 : rows;
            if (d.chunk > least) d.chunk = (int)least;
        }
    }
    const int rc = build_plan(p, cu_seqlens_dev, o, want);
    if (rc != LIBRA_OK) {
        libra_plan_destroy(p);
        cudaGetLastError();   // not the next call's
        return rc;
    }
    *plan_out = p;
    return LIBRA_OK;
}

static PlanDir* dir_of(const libra_plan_t* plan, int direction) {
    if (!plan) return nullptr;
    if (direction == LIBRA_DIR_Q) return plan->dir[0].enabled ? const_cast<PlanDir*>(&plan->dir[0]) : nullptr;
    if (direction == LIBRA_DIR_KV) return plan->dir[1].enabled ? const_cast<PlanDir*>(&plan->dir[1]) : nullptr;
    if (direction == LIBRA_DIR_PAIR) return plan->dir[2].enabled ? const_cast<PlanDir*>(&plan->dir[2]) : nullptr;
    return nullptr;
}

extern "C" int libra_plan_info(const libra_plan_t* plan, int direction, int64_t* n_tiles, int* n_workers,
                               int64_t* n_blocks, int* tile, int* n_heads) {
    if (!plan) return LIBRA_ERR_INVALID_ARG;
    PlanDir* d = dir_of(plan, direction);
    if (!d) return LIBRA_ERR_PLAN_MISMATCH;
    if (n_tiles) *n_tiles = d->NT;
    if (n_workers) *n_workers = d->W;
    if (n_blocks) *n_blocks = d->NB;
    if (tile) *tile = d->tile;
    if (n_heads) *n_heads = d->H;
    return LIBRA_OK;
}

extern "C" int libra_plan_status(const libra_plan_t* plan) {
    if (!plan) return LIBRA_ERR_INVALID_ARG;
    int st = 0;
    if (cudaStreamSynchronize(plan->stream) != cudaSuccess) return LIBRA_ERR_CUDA;
    if (cudaMemcpy(&st, plan->d_status, sizeof(st), cudaMemcpyDeviceToHost) != cudaSuccess) return LIBRA_ERR_CUDA;
    return st;
}

extern "C" int libra_plan_export(const libra_plan_t* plan, int direction, int64_t* weight_host, int32_t* order_host,
                                 int32_t* cta_of_tile_host, int32_t* cta_offsets_host, int32_t* cta_tiles_host,
                                 int64_t* loads_host) {
    if (!plan) return LIBRA_ERR_INVALID_ARG;
    PlanDir* d = dir_of(plan, direction);
    if (!d) return LIBRA_ERR_PLAN_MISMATCH;
    cudaStream_t s = plan->stream;
    cudaError_t e = cudaSuccess;
    auto ok = [&](cudaError_t x) { if (e == cudaSuccess) e = x; };
    void* tmp = nullptr;
    if (weight_host || order_host) ok(cudaMalloc(&tmp, sizeof(int64_t) * (d->NT ? d->NT : 1)));
    if (e != cudaSuccess) return LIBRA_ERR_CUDA;
    // Pair tiles whose lists no kernel walks: made here, the same ones at every call.
    if (d == &plan->dir[2] && plan->dir[4].enabled && (cta_of_tile_host || cta_offsets_host || cta_tiles_host || loads_host)) {
        DirViews views = {};
        views.v[0] = view_of(*d, 1, libra_plan_opts{});
        place_lists(views, 1, d->W, d->NT, s);
        ok(cudaGetLastError());
    }
    if (weight_host) {
        k_expand_weight<<<grid_for(d->NT, 256), 256, 0, s>>>(d->d_weight_blk, d->NT, d->H, d->d_u_blk ? d->NB : 0,
                                                             (int64_t*)tmp);
        count_launch();
        ok(cudaMemcpyAsync(weight_host, tmp, sizeof(int64_t) * d->NT, cudaMemcpyDeviceToHost, s));
        ok(cudaStreamSynchronize(s));
    }
    if (order_host) {
        k_expand_order<<<grid_for(d->NT, 256), 256, 0, s>>>(d->d_u_blk ? nullptr : d->d_blk_order, d->NT, d->H,
                                                            (int32_t*)tmp);
        count_launch();
        ok(cudaMemcpyAsync(order_host, tmp, sizeof(int32_t) * d->NT, cudaMemcpyDeviceToHost, s));
        ok(cudaStreamSynchronize(s));
    }
    if (cta_of_tile_host)
        ok(cudaMemcpyAsync(cta_of_tile_host, d->d_cta_of_tile, sizeof(int32_t) * d->NT, cudaMemcpyDeviceToHost, s));
    if (cta_offsets_host)
        ok(cudaMemcpyAsync(cta_offsets_host, d->d_cta_offsets, sizeof(int32_t) * (d->W + 1), cudaMemcpyDeviceToHost, s));
    if (cta_tiles_host)
        ok(cudaMemcpyAsync(cta_tiles_host, d->d_cta_tiles, sizeof(int32_t) * d->NT, cudaMemcpyDeviceToHost, s));
    if (loads_host) ok(cudaMemcpyAsync(loads_host, d->d_loads, sizeof(int64_t) * d->W, cudaMemcpyDeviceToHost, s));
    ok(cudaStreamSynchronize(s));
    cudaFree(tmp);
    return e == cudaSuccess ? LIBRA_OK : LIBRA_ERR_CUDA;
}

extern "C" int libra_plan_export_pairs(const libra_plan_t* plan, int32_t* key_block_host, int32_t* query_chunk_host,
                                       int* chunk_tokens_host) {
    if (!plan) return LIBRA_ERR_INVALID_ARG;
    PlanDir* d = dir_of(plan, LIBRA_DIR_PAIR);
    if (!d) return LIBRA_ERR_PLAN_MISMATCH;
    cudaError_t e = cudaStreamSynchronize(plan->stream);
    if (e == cudaSuccess && key_block_host)
        e = cudaMemcpy(key_block_host, d->d_u_blk, sizeof(int32_t) * d->NB, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && query_chunk_host)
        e = cudaMemcpy(query_chunk_host, d->d_u_chunk, sizeof(int32_t) * d->NB, cudaMemcpyDeviceToHost);
    if (chunk_tokens_host) *chunk_tokens_host = d->chunk;
    return e == cudaSuccess ? LIBRA_OK : LIBRA_ERR_CUDA;
}

extern "C" int libra_plan_fused_ctas(const libra_plan_t* plan) {
    if (!plan) return LIBRA_ERR_INVALID_ARG;
    if (!plan->dir[2].enabled) return LIBRA_ERR_PLAN_MISMATCH;
    return plan->dir[4].enabled ? 2 : 1;
}

extern "C" int libra_plan_destroy(libra_plan_t* plan) {
    if (!plan) return LIBRA_OK;
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev != plan->device) cudaSetDevice(plan->device);
    // Used on the legacy stream only (which outlives every plan): its order keeps the memory until the last kernel that
    // reads it is done, and the caller's next launches need not wait for an idle GPU.
    if (plan->other_stream && plan->n_blocks > 0) cudaDeviceSynchronize();
    for (int k = 0; k < plan->n_blocks; ++k) {
        if (plan->plain_memory) cudaFree(plan->blocks[k]);
        else scratch_free(plan->blocks[k], nullptr);
    }
    if (dev != plan->device) cudaSetDevice(dev);
    for (int a = 0; a < libra_plan::kTimedKernels; ++a)
        for (int r = 0; r < libra_plan::kTimeRing; ++r)
            for (int b = 0; b < 2; ++b)
                if (plan->ev[a][r][b]) cudaEventDestroy(plan->ev[a][r][b]);
    delete plan;
    return LIBRA_OK;
}

extern "C" int libra_busy_times(const libra_plan_t* plan, int which, uint64_t* ns_host) {
    if (!plan || !ns_host) return LIBRA_ERR_INVALID_ARG;
    if ((which < LIBRA_KERNEL_FWD || which > LIBRA_KERNEL_BWD_DQ) && which != LIBRA_KERNEL_BWD_FUSED) return LIBRA_ERR_INVALID_ARG;
    // the forward and the dQ kernel walk the query-major lists, the dK/dV kernel the key-major ones, the fused
    // backward the pair tiles
    PlanDir* d = dir_of(plan, which == LIBRA_KERNEL_BWD_FUSED ? LIBRA_DIR_PAIR
                                                              : (which == LIBRA_KERNEL_BWD_DKDV ? LIBRA_DIR_KV : LIBRA_DIR_Q));
    if (!d) return LIBRA_ERR_PLAN_MISMATCH;
    if (cudaDeviceSynchronize() != cudaSuccess) return LIBRA_ERR_CUDA;
    const size_t most = (size_t)d->W + 1;
    uint64_t* tmp = new (std::nothrow) uint64_t[3 * most];   // the stamps, then one kernel's outcomes
    if (!tmp) return LIBRA_ERR_CUDA;
    int* outcome = reinterpret_cast<int*>(tmp + 2 * most);
    int st = 0;
    const uint64_t* src = which == LIBRA_KERNEL_BWD_DQ ? d->d_busy2 : d->d_busy;
    cudaError_t e = cudaMemcpy(tmp, src, sizeof(uint64_t) * 2 * d->W, cudaMemcpyDeviceToHost);
    const int mask = which == LIBRA_KERNEL_FWD ? 1 : plan->bwd_mask;
    for (int k = 0; k < 4 && e == cudaSuccess; ++k) {
        if (!((mask >> k) & 1)) continue;
        const int n = plan->n_outcome[k];   // words beyond are an earlier launch's
        e = cudaMemcpy(outcome, plan->d_outcome[k], sizeof(int) * n, cudaMemcpyDeviceToHost);
        for (int r = 0; r < n && e == cudaSuccess; ++r)
            if (outcome[r] != 0) st = outcome[r];
    }
    const int ran = plan->n_outcome[which == LIBRA_KERNEL_FWD ? 0 : (which == LIBRA_KERNEL_BWD_DQ ? 3 : 1)];
    for (int r = 0; r < d->W; ++r)
        ns_host[r] = r < ran && tmp[2 * r + 1] >= tmp[2 * r] ? tmp[2 * r + 1] - tmp[2 * r] : 0;
    delete[] tmp;
    if (e != cudaSuccess) return LIBRA_ERR_CUDA;
    return st;
}

extern "C" int libra_tile_times(const libra_plan_t* plan, int which, uint32_t* ns_host) {
    if (!plan || !ns_host) return LIBRA_ERR_INVALID_ARG;
    if (which != LIBRA_KERNEL_FWD && which != LIBRA_KERNEL_BWD_FUSED) return LIBRA_ERR_INVALID_ARG;
    PlanDir* d = dir_of(plan, which == LIBRA_KERNEL_BWD_FUSED ? LIBRA_DIR_PAIR : LIBRA_DIR_Q);
    if (!d) return LIBRA_ERR_PLAN_MISMATCH;
    if (cudaDeviceSynchronize() != cudaSuccess) return LIBRA_ERR_CUDA;
    return cudaMemcpy(ns_host, d->d_tile_ns, sizeof(uint32_t) * d->NT, cudaMemcpyDeviceToHost) == cudaSuccess
               ? LIBRA_OK : LIBRA_ERR_CUDA;
}

extern "C" int libra_plan_set_timing(libra_plan_t* plan, int enabled) {
    if (!plan) return LIBRA_ERR_INVALID_ARG;
    if (enabled) {
        for (int a = 0; a < libra_plan::kTimedKernels; ++a)
            for (int r = 0; r < libra_plan::kTimeRing; ++r)
                for (int b = 0; b < 2; ++b)
                    if (!plan->ev[a][r][b] && cudaEventCreate(&plan->ev[a][r][b]) != cudaSuccess) return LIBRA_ERR_CUDA;
        for (int a = 0; a < libra_plan::kTimedKernels; ++a) plan->ev_count[a] = 0;   // a fresh record
    }
    plan->timing = enabled ? 1 : 0;
    return LIBRA_OK;
}

extern "C" int libra_plan_set_wait_limit_ns(libra_plan_t* plan, uint64_t ns) {
    if (!plan || ns > 4000000000ull) return LIBRA_ERR_INVALID_ARG;
    plan->wait_limit_ns = ns ? (uint32_t)ns : 2000000000u;
    return LIBRA_OK;
}

extern "C" int libra_plan_inject_stall(libra_plan_t* plan, int enabled) {
    if (!plan) return LIBRA_ERR_INVALID_ARG;
    plan->inject_stall = enabled ? 1 : 0;
    return LIBRA_OK;
}

static int kernel_time(const libra_plan_t* plan, int a, int64_t launch, float* ms) {
    cudaEvent_t e0 = plan->ev[a][launch % libra_plan::kTimeRing][0], e1 = plan->ev[a][launch % libra_plan::kTimeRing][1];
    if (cudaEventSynchronize(e1) != cudaSuccess) return LIBRA_ERR_CUDA;
    return cudaEventElapsedTime(ms, e0, e1) == cudaSuccess ? LIBRA_OK : LIBRA_ERR_CUDA;
}

extern "C" int libra_kernel_time_ms(const libra_plan_t* plan, int which, float* ms_host) {
    if (!plan || !ms_host) return LIBRA_ERR_INVALID_ARG;
    const int a = which - 1;  // LIBRA_KERNEL_FWD / _BWD_DKDV / _BWD_DQ / _BWD_PREP
    if (a < 0 || a >= libra_plan::kTimedKernels) return LIBRA_ERR_INVALID_ARG;
    if (plan->ev_count[a] == 0) return LIBRA_ERR_PLAN_MISMATCH;
    return kernel_time(plan, a, plan->ev_count[a] - 1, ms_host);
}

extern "C" int libra_kernel_times_ms(const libra_plan_t* plan, int which, float* ms_host, int capacity, int* n_out) {
    if (!plan || !ms_host || !n_out || capacity < 0) return LIBRA_ERR_INVALID_ARG;
    const int a = which - 1;
    if (a < 0 || a >= libra_plan::kTimedKernels) return LIBRA_ERR_INVALID_ARG;
    int64_t n = plan->ev_count[a] < libra_plan::kTimeRing ? plan->ev_count[a] : libra_plan::kTimeRing;
    if (n > capacity) n = capacity;
    for (int64_t i = 0; i < n; ++i) {   // oldest first
        const int rc = kernel_time(plan, a, plan->ev_count[a] - n + i, ms_host + i);
        if (rc != LIBRA_OK) return rc;
    }
    *n_out = (int)n;
    return LIBRA_OK;
}

extern "C" int64_t libra_launch_count(void) { return g_launches.load(); }

extern "C" const char* libra_strerror(int code) {
    switch (code) {
        case LIBRA_OK: return "ok";
        case LIBRA_ERR_INVALID_ARG: return "invalid argument";
        case LIBRA_ERR_UNSUPPORTED: return "unsupported configuration";
        case LIBRA_ERR_PLAN_MISMATCH: return "plan does not match the call";
        case LIBRA_ERR_CUDA: return "CUDA call failed";
        case LIBRA_ERR_OVERFLOW: return "integer overflow in plan sizes";
        case LIBRA_ERR_TIMEOUT: return "a bounded device-side wait timed out";
        case LIBRA_ERR_BAD_SEQLENS: return "cu_seqlens is malformed";
        case LIBRA_ERR_NO_DEVICE: return "no usable CUDA device";
        case LIBRA_ERR_SCRATCH_TOO_SMALL: return "problem exceeds the library's built-in scratch (use libra_attn_pool_bwd with a caller workspace)";
        default: return "unknown error";
    }
}
