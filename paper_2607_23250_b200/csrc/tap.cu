// Communication-aware SH-Tile placement for a sequence pool spread over several workers
// (Section 4.3: tiles and KV groups, Algorithm 2, exchange planning), as device kernels.
//
// The pool holds P packed sequences; sequence s belongs to the CP workers s*CP .. s*CP+CP-1, worker c of
// the group holding the c-th run of ceil(L_s / CP) consecutive tokens (the paper leaves this split open).
// A block's KV groups are the samples with a token in it, which is a contiguous range of sample indices,
// so K(t) is kept as (first sample, last sample, head shard) instead of a list; samples of length zero
// inside the range weigh nothing and change no decision.
//
// Placement is sequential by nature (every choice depends on the loads and residency left by the previous
// ones), so the latency of one step bounds it.  Up to 128 workers whose tables fit shared memory: one block whose
// warps work on neighbouring steps (k_tap_place_team).  Otherwise: one CTA with a thread per worker, block-wide
// arg-min, tables in global memory.  1024 tiles on 16 workers with their schedule: 0.25 ms, with one warp for all of a
// step 0.65 ms, all in the second form 2.8 ms.
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/libra.h"
#include "common.h"
#include "ptx.cuh"

namespace libra {

struct TapGeom {
    const int32_t* cu;        // [n+1] sample offsets of the pool
    const int32_t* seq_off;   // [P+1] token offsets of the packed sequences
    const int32_t* blk_off;   // [P+1] first block of each sequence
    int n, P, CP, B, H, hq, hkv, d;
};
// The two tables of a pool of up to SEQS sequences, as a kernel argument: the first kernel of a call reads them there and
// leaves them in the call's scratch for the others.  (A copy from pageable memory instead took the host 10 us a call and
// the stream 3; and a graph that is captured around the call would read that memory at every replay.)  2 KB for the usual
// pools, 8 KB for as many sequences as there can be workers.
constexpr int kTapFewSeqs = 255, kTapMaxWorkers = 1024;
template <int SEQS>
struct TapTables {
    int32_t seq_off[SEQS + 1], blk_off[SEQS + 1];
};

__device__ __forceinline__ int tap_seq_of_token(const TapGeom& g, int64_t tok) {
    int s = 0;
    while (s + 1 < g.P && g.seq_off[s + 1] <= tok) ++s;
    return s;
}
__device__ __forceinline__ int tap_owner(const TapGeom& g, int s, int64_t tok) {
    const int64_t len = g.seq_off[s + 1] - g.seq_off[s];
    const int64_t run = (len + g.CP - 1) / g.CP;
    return s * g.CP + (int)((tok - g.seq_off[s]) / (run > 0 ? run : 1));
}
// Index of the sample that holds token tok (the last j with cu[j] <= tok; it is never empty), by a warp, 32 probes at a time.
__device__ __forceinline__ int tap_sample_of_token_warp(const TapGeom& g, int64_t tok) {
    const int lane = threadIdx.x & 31;
    int lo = 0, len = g.n;   // the sample is one of [lo, lo + len)
    while (len > 1) {
        const int step = (len + 31) / 32, at = lo + lane * step;
        const unsigned below = __ballot_sync(0xffffffffu, lane == 0 || (lane * step < len && g.cu[at] <= tok));
        const int skip = (31 - __clz(below)) * step;
        lo += skip;
        len = len - skip < step ? len - skip : step;
    }
    return lo;
}

// What the first kernel of a call writes: per block its work (Eq. 6 in closed form), Q-home, Q + output bytes, first and
// last sample; per sample the bytes of its K and V on one head shard and the worker that holds all of it (or -1).  The grid
// also clears up to three arrays of 64-bit words, the status and the volume total, which later kernels add to.
struct TapSetup {
    int64_t NB;
    int block_ctas;          // CTAs that go through blocks, a warp each; the rest through samples
    int32_t *seq_off, *blk_off;   // where the tables go
    int64_t* f_blk;
    int32_t* q_home;
    int64_t* v_qo;
    int32_t *j_first, *j_last;
    int64_t* v_smp;
    int32_t* res_smp;
    int64_t* clear[3];
    int64_t n_clear[3];
    int* status;
    int64_t* comm_total;
};
template <int SEQS>
__global__ void __launch_bounds__(128) k_tap_setup(TapGeom g, const TapSetup p, const __grid_constant__ TapTables<SEQS> tables) {
    grid_dep_wait();
    grid_dep_launch();
    if (blockIdx.x == 0)
        for (int q = threadIdx.x; q <= g.P; q += 128) { p.seq_off[q] = tables.seq_off[q]; p.blk_off[q] = tables.blk_off[q]; }
    g.seq_off = tables.seq_off;
    g.blk_off = tables.blk_off;
    const int64_t all = (int64_t)gridDim.x * 128, at = blockIdx.x * (int64_t)128 + threadIdx.x;
#pragma unroll
    for (int k = 0; k < 3; ++k)
        for (int64_t x = at; x < p.n_clear[k]; x += all) p.clear[k][x] = 0;
    if (at == 0 && p.status) *p.status = 0;
    if (at == 0 && p.comm_total) *p.comm_total = 0;
    if ((int)blockIdx.x < p.block_ctas) {
        const int64_t b = at >> 5;
        const int lane = threadIdx.x & 31;
        if (b >= p.NB) return;
        int s = 0;
        while (s + 1 < g.P && g.blk_off[s + 1] <= b) ++s;
        const int64_t q0 = g.seq_off[s] + (b - g.blk_off[s]) * g.B;
        const int64_t q1 = q0 + g.B < g.seq_off[s + 1] ? q0 + g.B : g.seq_off[s + 1];
        const int j0 = tap_sample_of_token_warp(g, q0), j1 = tap_sample_of_token_warp(g, q1 - 1);
        int64_t w = 0;
        for (int j = j0 + lane; j <= j1; j += 32) {
            const int64_t lo = q0 > g.cu[j] ? q0 : g.cu[j], hi = q1 < g.cu[j + 1] ? q1 : g.cu[j + 1];
            if (lo < hi) {
                const int64_t a = lo - g.cu[j], e = hi - g.cu[j];
                w += (e * (e + 1) - a * (a + 1)) / 2;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
        if (lane == 0) {
            if (p.f_blk) p.f_blk[b] = w;
            p.q_home[b] = tap_owner(g, s, q0);
            if (p.v_qo) p.v_qo[b] = 2 * ((q1 - q0) * (g.hq / g.H) * g.d * 2);
            p.j_first[b] = j0;
            p.j_last[b] = j1;
        }
        return;
    }
    const int64_t j = at - (int64_t)p.block_ctas * 128;
    if (j >= g.n) return;
    const int64_t a = g.cu[j], e = g.cu[j + 1];
    const int kvps = g.H <= g.hkv ? g.hkv / g.H : 1;
    if (p.v_smp) p.v_smp[j] = 2 * (e - a) * kvps * g.d * 2;
    int res = -1;
    if (e > a) {
        const int s = tap_seq_of_token(g, a);
        const int first = tap_owner(g, s, a), last = tap_owner(g, s, e - 1);
        res = first == last ? first : -1;
    }
    p.res_smp[j] = res;
}

// A block as the placement reads it.
struct __align__(16) TapRec {
    int64_t f, v_qo;
    int32_t q_home, j0, j1, blk;
};

// Blocks by (work descending, index ascending); sixteen lanes share a block's comparisons, so that a few hundred blocks
// fill more than one CTA (256 blocks: 9 us by a thread each, 4 so).
__global__ void __launch_bounds__(256) k_tap_rank(const int64_t* __restrict__ f_blk, int64_t NB, const int32_t* __restrict__ q_home,
                                                  const int64_t* __restrict__ v_qo, const int32_t* __restrict__ j_first,
                                                  const int32_t* __restrict__ j_last, int32_t* __restrict__ blk_order, TapRec* __restrict__ rec) {
    __shared__ int64_t sw[1024];
    const int64_t b = blockIdx.x * (int64_t)16 + (threadIdx.x >> 4);
    const int sub = threadIdx.x & 15;
    grid_dep_wait();
    grid_dep_launch();
    const int64_t wb = b < NB ? f_blk[b] : 0;
    int rank = 0;
    for (int64_t base = 0; base < NB; base += 1024) {
        const int lim = (int)(NB - base < 1024 ? NB - base : 1024);
        for (int o = threadIdx.x; o < lim; o += 256) sw[o] = f_blk[base + o];
        __syncthreads();
        for (int k = sub; k < lim; k += 16) {
            const int64_t w = sw[k];
            rank += (w > wb) || (w == wb && base + k < b);
        }
        __syncthreads();
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
    if (b < NB && sub == 0) {
        blk_order[rank] = (int32_t)b;
        rec[rank] = TapRec{wb, v_qo[b], q_home[b], j_first[b], j_last[b], (int32_t)b};
    }
}

struct TapKey {
    int64_t a, b;
    int32_t r;   // -1: no candidate
};
__device__ __forceinline__ bool tap_less(const TapKey& x, const TapKey& y) {
    if (y.r < 0) return x.r >= 0;
    if (x.r < 0) return false;
    if (x.a != y.a) return x.a < y.a;
    if (x.b != y.b) return x.b < y.b;
    return x.r < y.r;
}
__device__ __forceinline__ TapKey tap_shfl_xor(const TapKey& k, int off) {
    TapKey o;
    o.a = __shfl_xor_sync(0xffffffffu, k.a, off);
    o.b = __shfl_xor_sync(0xffffffffu, k.b, off);
    o.r = __shfl_xor_sync(0xffffffffu, k.r, off);
    return o;
}

// Algorithm 2.  blockDim.x = W rounded up to a warp; thread r is worker r.
__global__ void __launch_bounds__(1024) k_tap_place(
    const int64_t* __restrict__ f_blk, const int32_t* __restrict__ blk_order, const int32_t* __restrict__ q_home,
    const int64_t* __restrict__ v_qo, const int32_t* __restrict__ j_first, const int32_t* __restrict__ j_last,
    const int64_t* __restrict__ v_smp, const int32_t* __restrict__ res_smp, int64_t NB, int H, int W, int n,
    int tau_num, int tau_den, uint32_t* __restrict__ Cbits /*[W][words]*/, int words, int32_t* __restrict__ sigma,
    int64_t* __restrict__ loads, int64_t* __restrict__ comm_total, int* __restrict__ status) {
    __shared__ TapKey sk_f[32], sk_w[32];
    __shared__ int64_t s_sum[32];
    __shared__ int s_pick;
    __shared__ int64_t s_pick_delta;
    const int r = threadIdx.x, lane = r & 31, warp = r >> 5, nwarps = blockDim.x >> 5;
    const bool live = r < W;
    grid_dep_wait();
    // residency rows start with the groups the worker already holds in full
    if (live) {
        uint32_t* row = Cbits + (size_t)r * words;
        for (int w = 0; w < words; ++w) row[w] = 0;
        for (int j = 0; j < n; ++j)
            if (res_smp[j] == r)
                for (int h = 0; h < H; ++h) { const int g = j * H + h; row[g >> 5] |= 1u << (g & 31); }
    }
    // sum of f over all tiles
    int64_t part = 0;
    for (int64_t b = r; b < NB; b += blockDim.x) part += f_blk[b] * H;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
    if (lane == 0) s_sum[warp] = part;
    __syncthreads();
    int64_t sum_f = 0;
    for (int w = 0; w < nwarps; ++w) sum_f += s_sum[w];
    if (sum_f > (INT64_MAX / ((int64_t)(tau_den + tau_num) * 2)) / W) {  // the integer cap test would overflow
        if (r == 0) *status = LIBRA_ERR_OVERFLOW;   // the exchange kernels see the flag and add nothing
        for (int64_t t = r; t < NB * H; t += blockDim.x) sigma[t] = q_home[t / H];   // defined output: every tile stays home
        return;
    }
    const int64_t cap_rhs = (int64_t)(tau_den + tau_num) * sum_f;
    int64_t L = 0, comm = 0;
    uint32_t* my_row = Cbits + (size_t)(live ? r : 0) * words;
    const int64_t NT = NB * H;
    for (int64_t x = 0; x < NT; ++x) {
        const int32_t blk = blk_order[x / H];
        const int h = (int)(x % H);
        const int64_t f = f_blk[blk];
        const int j0 = j_first[blk], j1 = j_last[blk];
        TapKey kf, kw;
        kf.r = kw.r = -1; kf.a = kf.b = kw.a = kw.b = 0;
        int64_t delta = 0;
        if (live) {
            delta = r != q_home[blk] ? v_qo[blk] : 0;
            for (int j = j0; j <= j1; ++j) {
                const int g = j * H + h;
                if (!((my_row[g >> 5] >> (g & 31)) & 1u)) delta += v_smp[j];
            }
            if ((int64_t)tau_den * W * (L + f) <= cap_rhs) { kf.a = delta; kf.b = L; kf.r = r; }
            kw.a = L; kw.b = delta; kw.r = r;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const TapKey of = tap_shfl_xor(kf, off), ow = tap_shfl_xor(kw, off);
            if (tap_less(of, kf)) kf = of;
            if (tap_less(ow, kw)) kw = ow;
        }
        if (lane == 0) { sk_f[warp] = kf; sk_w[warp] = kw; }
        __syncthreads();
        if (r == 0) {
            TapKey bf = sk_f[0], bw = sk_w[0];
            for (int w = 1; w < nwarps; ++w) {
                if (tap_less(sk_f[w], bf)) bf = sk_f[w];
                if (tap_less(sk_w[w], bw)) bw = sk_w[w];
            }
            if (bf.r >= 0) { s_pick = bf.r; s_pick_delta = bf.a; }   // some worker stays under the soft cap
            else           { s_pick = bw.r; s_pick_delta = bw.b; }   // nobody does: least loaded
            sigma[(int64_t)blk * H + h] = s_pick;
        }
        __syncthreads();
        if (r == s_pick) {
            L += f;
            for (int j = j0; j <= j1; ++j) { const int g = j * H + h; my_row[g >> 5] |= 1u << (g & 31); }
        }
        if (r == 0) comm += s_pick_delta;
        // the next iteration's first barrier orders these reads of s_pick before its rewrite
    }
    if (live) loads[r] = L;
    if (r == 0) *comm_total = comm;
}

// Smallest x among the lanes with `in`; `in` is left set on the lanes that hold it.  Values are not negative.
__device__ __forceinline__ uint64_t tap_warp_min(uint64_t x, bool& in) {
    const uint32_t hi = __reduce_min_sync(0xffffffffu, in ? (uint32_t)(x >> 32) : 0xffffffffu);
    in = in && (uint32_t)(x >> 32) == hi;
    const uint32_t lo = __reduce_min_sync(0xffffffffu, in ? (uint32_t)x : 0xffffffffu);
    in = in && (uint32_t)x == lo;
    return (uint64_t)hi << 32 | lo;
}

// Algorithm 2 by one block (PER * 32 >= W); same choices as k_tap_place.  Up to kTapTeam shards of a block are a step, and
// three kinds of warps work on neighbouring steps, with a barrier between steps:
//   placing     one warp; lane l is the workers l, l + 32, ..., whose loads it keeps.  Step s.
//   walking     one per shard of a step: what every worker would have to fetch for its tile of step s + 1, once as things
//               stand without step s and once as if it were given step s's tile of the shard, so that the placing warp
//               only has to choose between the two.
//   recording   one per shard: enters step s - 1's pick into the residency, per shard and sample a bit for each worker.  A
//               walking warp may meet a word before or after that; it looks at the pick itself.
// What is serial is the placing warp's minimum and the load it changes, 290 clk a tile (1024 tiles, 4 shards, 16 workers: 1165 a
// step, of which the placing warp is busy 1100 and the others as long); one warp that did all of it took 1100 clk a tile.
// Its loop over the shards is unrolled: rolled up, with the next shard's volumes fetched ahead, it took 1.3 times as long.
// Volumes are multiples of 4 head_dim bytes and are kept in that unit, in 32 bits where a block's samples and its rows fit
// them together (Delta).
// Dynamic shared memory: sample volumes [n] (64 bits), then residency [H][n][PER].
constexpr int kTapTeam = 8;
constexpr int kTapThreads = 32 * (1 + 2 * kTapTeam);
constexpr size_t kTapTeamStatic = 2 * kTapTeam * 32 * 16 + 1024;   // shared memory beside the tables, a PER
constexpr size_t kTapTeamSmem = 227 * 1024 - 4 * kTapTeamStatic;
template <typename Delta> struct __align__(2 * sizeof(Delta)) TapDelta { Delta as_is, if_given; };

struct TapPlace {
    const TapRec* rec;        // the blocks in placement order
    const int64_t* v_smp;
    const int32_t* res_smp;
    int64_t NB, unit;         // unit: bytes a volume counts in
    int H, W, n, tau_num, tau_den, words;
    uint32_t* Cbits;          // [W][words]
    int32_t* sigma;
    int64_t* loads;
    int64_t* comm_total;
    int* status;
};

template <int PER, typename Mask, typename Delta>
__device__ __forceinline__ void tap_place_steps(const TapPlace& p, int64_t cap, const uint64_t* v_smp, Mask* held, void* deltas,
                                                int (*s_pick)[kTapTeam]) {
    using Two = TapDelta<Delta>;
    Two (*s_delta)[kTapTeam][32 * PER] = reinterpret_cast<Two (*)[kTapTeam][32 * PER]>(deltas);   // [2]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n = p.n, H = p.H, W = p.W;
    const int groups = (H + kTapTeam - 1) / kTapTeam;   // steps a block takes
    const int64_t NB = p.NB, steps = NB * groups;
    const TapRec* __restrict__ rec = p.rec;
    if (warp == 0) {
        int64_t L[PER];
        uint64_t comm = 0;
        int last[kTapTeam];   // picks of the step before
#pragma unroll
        for (int u = 0; u < PER; ++u) L[u] = 0;
#pragma unroll
        for (int k = 0; k < kTapTeam; ++k) last[k] = -1;
        int64_t f_in = rec[lane < NB ? lane : NB - 1].f, f_next = f_in;
        int64_t x = 0;
        int grp = 0;
        __syncthreads();
        for (int64_t st = 0; st < steps; ++st) {
            const int buf = (int)(st & 1), cnt = H - grp * kTapTeam < kTapTeam ? H - grp * kTapTeam : kTapTeam;
            constexpr bool kAhead = PER * sizeof(Delta) <= 8;   // all at once while registers last
            Two two[kTapTeam][PER];
#pragma unroll
            for (int k = 0; k < kTapTeam && kAhead; ++k)
#pragma unroll
                for (int u = 0; u < PER; ++u) two[k][u] = s_delta[buf][k][lane + 32 * u];
            if (grp == 0 && (x & 31) == 0) {   // the next batch of blocks lands while this one is placed
                if (x > 0) f_in = f_next;
                const int64_t xn = x + 32 + lane;
                f_next = rec[xn < NB ? xn : NB - 1].f;
            }
            const int64_t f = __shfl_sync(0xffffffffu, f_in, (int)(x & 31));
            const int64_t room = cap - f;
#pragma unroll
            for (int k = 0; k < kTapTeam; ++k) {
                if (k >= cnt) break;
                // the lane's best worker under the soft cap, by (delta, load, index)
                Delta d[PER], bd = 0;
                int64_t bl = 0;
                int br = -1;
#pragma unroll
                for (int u = 0; u < PER; ++u) {
                    const int r = lane + 32 * u;
                    if (!kAhead) two[k][u] = s_delta[buf][k][r];
                    d[u] = last[k] == r ? two[k][u].if_given : two[k][u].as_is;
                    if (r < W && L[u] <= room && (br < 0 || d[u] < bd || (d[u] == bd && L[u] < bl))) { bd = d[u]; bl = L[u]; br = r; }
                }
                bool in = br >= 0, some;
                int pick;
                Delta pick_delta;
                if (sizeof(Delta) == 4) {
                    pick_delta = (Delta)__reduce_min_sync(0xffffffffu, in ? (uint32_t)bd : 0xffffffffu);
                    some = (uint32_t)pick_delta != 0xffffffffu;
                    in = in && bd == pick_delta;
                } else {
                    some = __any_sync(0xffffffffu, in);
                    pick_delta = (Delta)tap_warp_min(bd, in);
                }
                if (some) {                                    // some worker stays under the soft cap
                    unsigned who = __ballot_sync(0xffffffffu, in);
                    if (who & (who - 1)) {
                        tap_warp_min((uint64_t)bl, in);
                        who = __ballot_sync(0xffffffffu, in);
                    }
                    if (PER == 1) pick = __ffs(who) - 1;
                    else pick = (int)__reduce_min_sync(0xffffffffu, in ? (uint32_t)br : 0xffffffffu);
                } else {                                       // nobody does: by (load, delta, index)
#pragma unroll
                    for (int u = 0; u < PER; ++u) {
                        const int r = lane + 32 * u;
                        if (r < W && (br < 0 || L[u] < bl || (L[u] == bl && d[u] < bd))) { bd = d[u]; bl = L[u]; br = r; }
                    }
                    in = br >= 0;
                    tap_warp_min((uint64_t)bl, in);
                    pick_delta = (Delta)tap_warp_min(bd, in);
                    pick = (int)__reduce_min_sync(0xffffffffu, in ? (uint32_t)br : 0xffffffffu);
                }
#pragma unroll
                for (int u = 0; u < PER; ++u)
                    if (pick == lane + 32 * u) L[u] += f;
                if (lane == 0) s_pick[buf][k] = pick;
                last[k] = groups == 1 ? pick : -1;   // with more than one step a block the next step has other shards
                comm += pick_delta;
            }
            if (++grp == groups) { grp = 0; ++x; }
            __syncthreads();
        }
#pragma unroll
        for (int u = 0; u < PER; ++u)
            if (lane + 32 * u < W) p.loads[lane + 32 * u] = L[u];
        if (lane == 0) *p.comm_total = (int64_t)(comm * (uint64_t)p.unit);
        __syncthreads();
        return;
    }
    const bool walks = warp <= kTapTeam;
    const int k = (warp - 1) % kTapTeam;
    // the blocks of steps s - 1, s and s + 1; h: the warp's shard, H or more: none
    int j0_a = 0, j1_a = -1, h_a = H, blk_a = 0, j0_b = 0, j1_b = -1, h_b = H, blk_b = 0;
    TapRec in = rec[lane < NB ? lane : NB - 1], next_in = in;
    in.v_qo /= p.unit;
    int64_t x = 0;             // the block of step s + 1
    int grp = 0;
    for (int64_t st = -1; st <= steps; ++st) {
        int j0 = 0, j1 = -1, h = H, blk = 0, home = 0;
        Delta vqo = 0;
        if (st + 1 < steps) {
            if (grp == 0 && (x & 31) == 0) {
                if (x > 0) { in = next_in; in.v_qo /= p.unit; }
                const int64_t xn = x + 32 + lane;
                next_in = rec[xn < NB ? xn : NB - 1];
            }
            const int src = (int)(x & 31);
            j0 = __shfl_sync(0xffffffffu, in.j0, src);
            j1 = __shfl_sync(0xffffffffu, in.j1, src);
            blk = __shfl_sync(0xffffffffu, in.blk, src);
            home = __shfl_sync(0xffffffffu, in.q_home, src);
            vqo = __shfl_sync(0xffffffffu, (Delta)in.v_qo, src);
            h = grp * kTapTeam + k;
            if (++grp == groups) { grp = 0; ++x; }
        }
        if (st >= 0) __syncthreads();   // step st - 1 is placed
        const int pick = h_a < H ? s_pick[(st + 1) & 1][k] : -1;
        if (walks) {
            if (h < H) {
                const Mask* row = held + (size_t)h * n * PER;
                const bool same = h == h_a;   // (else that pick was of another shard)
                Two d[PER];
#pragma unroll
                for (int u = 0; u < PER; ++u) d[u].as_is = d[u].if_given = lane + 32 * u != home ? vqo : 0;
#pragma unroll 4
                for (int j = j0; j <= j1; ++j) {
                    const Delta v = (Delta)v_smp[j];
                    const Delta v_other = j >= j0_b && j <= j1_b ? 0 : v;
                    const bool just = same && j >= j0_a && j <= j1_a;
#pragma unroll
                    for (int u = 0; u < PER; ++u) {
                        const bool has = (((uint32_t)row[j * PER + u] >> lane) & 1u) || (just && pick == lane + 32 * u);
                        d[u].as_is += has ? 0 : v;
                        d[u].if_given += has ? 0 : v_other;
                    }
                }
#pragma unroll
                for (int u = 0; u < PER; ++u) s_delta[(st + 1) & 1][k][lane + 32 * u] = d[u];
            }
        } else if (h_a < H) {
            Mask* row = held + (size_t)h_a * n * PER + (PER > 1 ? pick >> 5 : 0);
            for (int j = j0_a + lane; j <= j1_a; j += 32) row[j * PER] |= (Mask)(1u << (pick & 31));
            if (lane == 0) p.sigma[(int64_t)blk_a * H + h_a] = pick;
        }
        j0_a = j0_b; j1_a = j1_b; h_a = h_b; blk_a = blk_b;
        j0_b = j0; j1_b = j1; h_b = h; blk_b = blk;
    }
    __syncthreads();
}

template <int PER, typename Mask>
__global__ void __launch_bounds__(kTapThreads) k_tap_place_team(const TapPlace p) {
    static_assert(PER == 1 || sizeof(Mask) == 4, "a worker's bit is in word r / 32");
    extern __shared__ __align__(16) uint8_t tap_smem[];
    uint64_t* v_smp = reinterpret_cast<uint64_t*>(tap_smem);
    Mask* held = reinterpret_cast<Mask*>(v_smp + p.n);
    __shared__ TapDelta<uint64_t> s_delta[2][kTapTeam][32 * PER];
    __shared__ int s_pick[2][kTapTeam];
    __shared__ unsigned long long s_sum, s_vol;
    const int n = p.n, H = p.H, W = p.W;
    grid_dep_wait();
    if (threadIdx.x == 0) s_sum = s_vol = 0;
    __syncthreads();
    unsigned long long part = 0, vol = 0, most = 0;
    for (int j = threadIdx.x; j < n; j += kTapThreads) { v_smp[j] = (uint64_t)(p.v_smp[j] / p.unit); vol += v_smp[j]; }
    for (int j = threadIdx.x; j < n; j += kTapThreads) {   // the groups a worker holds in full
        const int r = p.res_smp[j];
        for (int h = 0; h < H; ++h)
#pragma unroll
            for (int u = 0; u < PER; ++u)
                held[((size_t)h * n + j) * PER + u] = r >= 0 && r < W && r >> 5 == u ? (Mask)(1u << (r & 31)) : (Mask)0;
    }
    for (int64_t b = threadIdx.x; b < p.NB; b += kTapThreads) {
        part += (unsigned long long)p.rec[b].f * H;
        const unsigned long long v = (unsigned long long)(p.rec[b].v_qo / p.unit);
        most = v > most ? v : most;
    }
    if (most >> 31) vol += 1ull << 32;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {   // (an atomic a thread took 10 us)
        part += __shfl_xor_sync(0xffffffffu, part, o);
        vol += __shfl_xor_sync(0xffffffffu, vol, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&s_sum, part);
        atomicAdd(&s_vol, vol);
    }
    __syncthreads();
    const int64_t sum_f = (int64_t)s_sum;
    if (sum_f > (INT64_MAX / ((int64_t)(p.tau_den + p.tau_num) * 2)) / W) {  // the integer cap test would overflow
        if (threadIdx.x == 0) *p.status = LIBRA_ERR_OVERFLOW;   // the exchange kernels see the flag and add nothing
        for (int64_t x = threadIdx.x; x < p.NB * H; x += kTapThreads) p.sigma[(int64_t)p.rec[x / H].blk * H + x % H] = p.rec[x / H].q_home;
        return;
    }
    // tau_den W (L + f) <= (tau_den + tau_num) sum f, as a bound on L + f
    const int64_t cap = (int64_t)(p.tau_den + p.tau_num) * sum_f / ((int64_t)p.tau_den * W);
    if (s_vol >> 31 == 0) tap_place_steps<PER, Mask, uint32_t>(p, cap, v_smp, held, s_delta, s_pick);
    else tap_place_steps<PER, Mask, uint64_t>(p, cap, v_smp, held, s_delta, s_pick);
    grid_dep_launch();   // (not before: the next kernel's blocks would sit on the other SMs all the while)
    for (int64_t i = threadIdx.x; i < (int64_t)W * p.words; i += kTapThreads) {   // as bit rows per worker
        const int r = (int)(i / p.words), g0 = (int)(i % p.words) * 32;
        uint32_t bits = 0;
        for (int b = 0; b < 32 && g0 + b < n * H; ++b) {
            const int j = (g0 + b) / H, h = (g0 + b) % H;
            bits |= ((uint32_t)held[((size_t)h * n + j) * PER + (r >> 5)] >> (r & 31) & 1u) << b;
        }
        p.Cbits[i] = bits;
    }
}

// Forward / backward send-byte matrices [src][dst]: a thread per tile (Q and output), then one per worker and KV group.
__global__ void k_tap_exchange(TapGeom g, int64_t NT, const int32_t* __restrict__ sigma, const int32_t* __restrict__ q_home,
                               const int64_t* __restrict__ v_qo, const uint32_t* __restrict__ Cbits, int words,
                               const int32_t* __restrict__ res_smp, int W, const int* __restrict__ status,
                               unsigned long long* __restrict__ fwd, unsigned long long* __restrict__ bwd) {
    grid_dep_wait();
    grid_dep_launch();
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (*status != 0) return;   // a placement that gave up left the bit rows unwritten
    if (t < NT) {
        const int q = q_home[t / g.H], r = sigma[t];
        if (q == r || r < 0 || r >= W || q < 0 || q >= W) return;
        const unsigned long long v = (unsigned long long)(v_qo[t / g.H] / 2);
        atomicAdd(&fwd[(size_t)q * W + r], v);   // Q out
        atomicAdd(&fwd[(size_t)r * W + q], v);   // output back
        atomicAdd(&bwd[(size_t)q * W + r], v);   // dO along the Q path
        atomicAdd(&bwd[(size_t)r * W + q], v);   // dQ along the output path
        return;
    }
    const int64_t idx = t - NT, NG = (int64_t)g.n * g.H;
    if (idx >= NG * W) return;
    const int r = (int)(idx / NG);
    const int grp = (int)(idx % NG), j = grp / g.H;
    if (!((Cbits[(size_t)r * words + (grp >> 5)] >> (grp & 31)) & 1u) || res_smp[j] == r) return;
    const int64_t a = g.cu[j], e = g.cu[j + 1];
    if (e <= a) return;
    const int kvps = g.H <= g.hkv ? g.hkv / g.H : 1;
    const int s = tap_seq_of_token(g, a);
    const int64_t len = g.seq_off[s + 1] - g.seq_off[s];
    const int64_t run = (len + g.CP - 1) / g.CP;
    for (int w = tap_owner(g, s, a); w <= tap_owner(g, s, e - 1); ++w) {   // the sample's token runs, owner by owner
        if (w == r) continue;
        const int64_t w0 = g.seq_off[s] + (int64_t)(w - s * g.CP) * run, w1 = w0 + run;
        const int64_t lo = a > w0 ? a : w0, hi = e < w1 ? e : w1;
        const unsigned long long bytes = (unsigned long long)((hi - lo) * 2 * kvps * g.d * 2);
        atomicAdd(&fwd[(size_t)w * W + r], bytes);
        atomicAdd(&bwd[(size_t)r * W + w], bytes);
    }
}


// ---- exchange schedule (Section 4.3.3): the transfer records implied by an assignment ----------------------
// Record = 6 x int32 (kind, src, dst, tok0, ntok, shard); kind 0: Q rows of a tile placed away from its Q-home
// (output back the same way, dO / dQ in the backward pass), kind 1: the K / V rows of a selected KV group held by
// another worker (dK / dV back the same way).  Order: kind 0 by tile id, then kind 1 by (dst, sample, shard, src).

// The KV groups some tile placed at r refers to, as bit rows [W][words].
__global__ void k_tap_mark(const int32_t* __restrict__ sigma, const int32_t* __restrict__ j_first,
                           const int32_t* __restrict__ j_last, int64_t NT, int H, int W, int words,
                           uint32_t* __restrict__ marks) {
    grid_dep_wait();
    grid_dep_launch();
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= NT) return;
    const int r = sigma[t], h = (int)(t % H);
    if (r < 0 || r >= W) return;
    for (int j = j_first[t / H]; j <= j_last[t / H]; ++j) {
        const int g = j * H + h;
        atomicOr(&marks[(size_t)r * words + (g >> 5)], 1u << (g & 31));
    }
}

// Records slot x of the enumeration produces: slot x < NT is tile x (0 or 1), slot NT + r * NG + g is group g
// at destination r (one per token run of the sample on another worker).
__device__ __forceinline__ int tap_slot_count(const TapGeom& g, int64_t x, int64_t NT, int64_t NG, int W,
                                              const int32_t* sigma, const int32_t* q_home, const uint32_t* marks,
                                              int words, const int32_t* res_smp) {
    if (x < NT) {
        const int r = sigma[x];
        return (r >= 0 && r < W && r != q_home[x / g.H]) ? 1 : 0;
    }
    const int64_t y = x - NT;
    const int r = (int)(y / NG);
    const int grp = (int)(y % NG), j = grp / g.H;
    if (!((marks[(size_t)r * words + (grp >> 5)] >> (grp & 31)) & 1u) || res_smp[j] == r) return 0;
    const int64_t a = g.cu[j], e = g.cu[j + 1];
    if (e <= a) return 0;
    const int s = tap_seq_of_token(g, a);
    int c = 0;
    for (int w = tap_owner(g, s, a); w <= tap_owner(g, s, e - 1); ++w) c += (w != r);
    return c;
}

constexpr int kTapSlots = 256;         // slots per CTA
constexpr int kTapInlineCtas = 2048;   // up to so many CTAs each adds up the totals of those before it; beyond, k_tap_sched_scan

// Inclusive prefix sum over the CTA's kTapSlots threads.
__device__ __forceinline__ int tap_scan(int c, int* part) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, c, o); if (lane >= o) c += v; }
    if (lane == 31) part[warp] = c;
    __syncthreads();
    for (int w = 0; w < warp; ++w) c += part[w];
    return c;
}

// Records ahead of each slot among its CTA's, and the CTA's total.
__global__ void __launch_bounds__(kTapSlots) k_tap_sched_count(TapGeom g, int64_t NT, int64_t NG, int W, const int32_t* __restrict__ sigma,
                                  const int32_t* __restrict__ q_home, const uint32_t* __restrict__ marks, int words,
                                  const int32_t* __restrict__ res_smp, int32_t* __restrict__ ahead /*[slots]*/, int64_t* __restrict__ total) {
    __shared__ int part[kTapSlots / 32];
    grid_dep_wait();
    grid_dep_launch();
    const int64_t x = blockIdx.x * (int64_t)kTapSlots + threadIdx.x;
    const int c = x < NT + NG * W ? tap_slot_count(g, x, NT, NG, W, sigma, q_home, marks, words, res_smp) : 0;
    const int incl = tap_scan(c, part);
    if (x < NT + NG * W) ahead[x] = incl - c;
    if (threadIdx.x == kTapSlots - 1) total[blockIdx.x] = incl;
}

// One block: exclusive prefix sum of n numbers in place, 4096 of them per pass, total to n_out.
__global__ void __launch_bounds__(1024) k_tap_sched_scan(int64_t n, int64_t* __restrict__ sums, int64_t* n_out) {
    __shared__ int64_t part[32];
    grid_dep_wait();
    grid_dep_launch();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t run = 0;
    for (int64_t base = 0; base < n; base += 4096) {
        const int64_t x0 = base + threadIdx.x * 4;
        int64_t c[4], sum = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) { c[k] = x0 + k < n ? sums[x0 + k] : 0; sum += c[k]; }
        int64_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int64_t v = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += v; }
        if (lane == 31) part[warp] = incl;
        __syncthreads();
        int64_t before = 0, all = 0;
        for (int w = 0; w < 32; ++w) { if (w < warp) before += part[w]; all += part[w]; }
        int64_t at = run + before + incl - sum;
#pragma unroll
        for (int k = 0; k < 4; ++k) { if (x0 + k < n) sums[x0 + k] = at; at += c[k]; }
        run += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) *n_out = run;
}

__global__ void __launch_bounds__(kTapSlots) k_tap_sched_fill(TapGeom g, int64_t NT, int64_t NG, int W, const int32_t* __restrict__ sigma,
                                 const int32_t* __restrict__ q_home, const uint32_t* __restrict__ marks, int words,
                                 const int32_t* __restrict__ res_smp, const int32_t* __restrict__ ahead, const int64_t* __restrict__ total,
                                 int scanned, int64_t* __restrict__ n_out, int64_t capacity, int32_t* __restrict__ rec) {
    __shared__ unsigned long long s_before;
    if (threadIdx.x == 0) s_before = 0;
    grid_dep_wait();
    grid_dep_launch();
    __syncthreads();
    if (scanned) {
        if (threadIdx.x == 0) s_before = (unsigned long long)total[blockIdx.x];
    } else {
        unsigned long long sum = 0;
        for (unsigned c = threadIdx.x; c < blockIdx.x; c += kTapSlots) sum += (unsigned long long)total[c];
        if (sum) atomicAdd(&s_before, sum);
    }
    __syncthreads();
    if (!scanned && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *n_out = (int64_t)s_before + total[blockIdx.x];
    const int64_t x = blockIdx.x * (int64_t)kTapSlots + threadIdx.x;
    if (x >= NT + NG * W) return;
    int64_t at = (int64_t)s_before + ahead[x];
    if (x < NT) {
        const int r = sigma[x];
        const int64_t b = x / g.H;
        if (!(r >= 0 && r < W && r != q_home[b]) || at >= capacity) return;
        int s = 0;
        while (s + 1 < g.P && g.blk_off[s + 1] <= b) ++s;
        const int64_t q0 = g.seq_off[s] + (b - g.blk_off[s]) * g.B;
        const int64_t q1 = q0 + g.B < g.seq_off[s + 1] ? q0 + g.B : g.seq_off[s + 1];
        int32_t* o = rec + at * 6;
        o[0] = 0; o[1] = q_home[b]; o[2] = r; o[3] = (int32_t)q0; o[4] = (int32_t)(q1 - q0); o[5] = (int32_t)(x % g.H);
        return;
    }
    const int64_t y = x - NT;
    const int r = (int)(y / NG);
    const int grp = (int)(y % NG), j = grp / g.H;
    if (!((marks[(size_t)r * words + (grp >> 5)] >> (grp & 31)) & 1u) || res_smp[j] == r) return;
    const int64_t a = g.cu[j], e = g.cu[j + 1];
    if (e <= a) return;
    const int s = tap_seq_of_token(g, a);
    const int64_t len = g.seq_off[s + 1] - g.seq_off[s];
    const int64_t run = (len + g.CP - 1) / g.CP;
    for (int w = tap_owner(g, s, a); w <= tap_owner(g, s, e - 1); ++w) {
        if (w == r) continue;
        if (at >= capacity) return;
        const int64_t w0 = g.seq_off[s] + (int64_t)(w - s * g.CP) * run, w1 = w0 + run;
        const int64_t lo = a > w0 ? a : w0, hi = e < w1 ? e : w1;
        int32_t* o = rec + at * 6;
        o[0] = 1; o[1] = w; o[2] = r; o[3] = (int32_t)lo; o[4] = (int32_t)(hi - lo); o[5] = grp % g.H;
        ++at;
    }
}

}  // namespace libra

using namespace libra;

extern "C" int64_t libra_tap_num_tiles(const int32_t* seq_offsets_host, int n_sequences, int block, int n_shards) {
    if (!seq_offsets_host || n_sequences <= 0 || block <= 0 || n_shards <= 0) return LIBRA_ERR_INVALID_ARG;
    int64_t nb = 0;
    for (int s = 0; s < n_sequences; ++s) {
        if (seq_offsets_host[s + 1] < seq_offsets_host[s]) return LIBRA_ERR_INVALID_ARG;
        nb += ((int64_t)seq_offsets_host[s + 1] - seq_offsets_host[s] + block - 1) / block;
    }
    return nb * n_shards;
}

// First kernel of a call.  The tables of the pool go with it as an argument and stay in `table` (2 (P + 1) words of scratch).
template <int SEQS>
static cudaError_t launch_setup_of(TapGeom& g, TapSetup p, const int32_t* seq_offsets_host, int32_t* table, cudaStream_t s) {
    TapTables<SEQS> tables;
    int64_t nb = 0;
    for (int q = 0; q <= g.P; ++q) {
        tables.seq_off[q] = seq_offsets_host[q];
        tables.blk_off[q] = (int32_t)nb;
        if (q < g.P) nb += ((int64_t)seq_offsets_host[q + 1] - seq_offsets_host[q] + g.B - 1) / g.B;
    }
    p.seq_off = table;
    p.blk_off = table + g.P + 1;
    g.seq_off = p.seq_off;
    g.blk_off = p.blk_off;
    p.block_ctas = (int)((p.NB + 3) / 4);
    const unsigned sample_ctas = (unsigned)(((int64_t)g.n + 127) / 128);
    count_launch();
    return launch_dependent(k_tap_setup<SEQS>, (unsigned)p.block_ctas + sample_ctas, 128u, 0, s, g, p, tables);
}
static int launch_setup(TapGeom& g, const TapSetup& p, const int32_t* seq_offsets_host, int32_t* table, cudaStream_t s) {
    const cudaError_t e = g.P <= kTapFewSeqs ? launch_setup_of<kTapFewSeqs>(g, p, seq_offsets_host, table, s)
                                             : launch_setup_of<kTapMaxWorkers>(g, p, seq_offsets_host, table, s);
    return e == cudaSuccess ? LIBRA_OK : LIBRA_ERR_CUDA;
}

extern "C" int libra_tap_plan(const int32_t* cu_seqlens_dev, int n_samples, const int32_t* seq_offsets_host,
                              int n_sequences, const libra_tap_opts* o, int32_t* sigma_dev, int64_t* loads_dev,
                              int64_t* fwd_bytes_dev, int64_t* bwd_bytes_dev, int64_t* comm_total_dev,
                              int* status_dev, void* stream) {
    if (!cu_seqlens_dev || !seq_offsets_host || !o || !sigma_dev || !loads_dev || !fwd_bytes_dev || !bwd_bytes_dev ||
        !comm_total_dev || !status_dev)
        return LIBRA_ERR_INVALID_ARG;
    if (n_samples <= 0 || n_sequences <= 0 || o->cp <= 0 || o->block <= 0 || o->n_shards <= 0 || o->hq <= 0 ||
        o->hkv <= 0 || o->head_dim <= 0 || o->tau_num < 0 || o->tau_den <= 0 || o->hq % o->n_shards != 0)
        return LIBRA_ERR_INVALID_ARG;
    if (!((o->n_shards <= o->hkv && o->hkv % o->n_shards == 0) || (o->n_shards > o->hkv && o->n_shards % o->hkv == 0)))
        return LIBRA_ERR_INVALID_ARG;
    if ((int64_t)n_sequences * o->cp > kTapMaxWorkers) return LIBRA_ERR_UNSUPPORTED;
    const int P = n_sequences, W = P * o->cp, H = o->n_shards;
    const int64_t NT = libra_tap_num_tiles(seq_offsets_host, P, o->block, H);
    if (NT <= 0) return LIBRA_ERR_INVALID_ARG;
    const int64_t NB = NT / H;
    if (NT >= INT32_MAX || NB > 65536) return LIBRA_ERR_UNSUPPORTED;  // the rank sort is quadratic in blocks
    {   // the work total (at most H * T (T + 1) / 2) must itself fit 64 bits before the device can test the cap
        const long double Tl = (long double)seq_offsets_host[P] - (long double)seq_offsets_host[0];
        if ((long double)H * Tl * (Tl + 1) / 2 > 4.0e18L) return LIBRA_ERR_OVERFLOW;
    }
    cudaStream_t s = (cudaStream_t)stream;
    const int words = (int)(((int64_t)n_samples * H + 31) / 32);

    uint8_t* scratch = nullptr;
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t at = off; off += (bytes + 255) & ~size_t(255); return at; };
    const size_t o_tab = take(sizeof(int32_t) * 2 * (P + 1));
    const size_t o_f = take(sizeof(int64_t) * NB), o_vqo = take(sizeof(int64_t) * NB);
    const size_t o_q = take(sizeof(int32_t) * NB), o_j0 = take(sizeof(int32_t) * NB), o_j1 = take(sizeof(int32_t) * NB);
    const size_t o_ord = take(sizeof(int32_t) * NB), o_rec = take(sizeof(TapRec) * NB);
    const size_t o_vs = take(sizeof(int64_t) * n_samples), o_rs = take(sizeof(int32_t) * n_samples);
    const size_t o_c = take(sizeof(uint32_t) * (size_t)words * W);
    if (scratch_alloc((void**)&scratch, off, s) != cudaSuccess) return LIBRA_ERR_CUDA;
    int64_t* f_blk = (int64_t*)(scratch + o_f);
    int64_t* v_qo = (int64_t*)(scratch + o_vqo);
    int32_t* q_home = (int32_t*)(scratch + o_q);
    int32_t* j0 = (int32_t*)(scratch + o_j0);
    int32_t* j1 = (int32_t*)(scratch + o_j1);
    int32_t* ord = (int32_t*)(scratch + o_ord);
    TapRec* rec = (TapRec*)(scratch + o_rec);
    int64_t* v_smp = (int64_t*)(scratch + o_vs);
    int32_t* res_smp = (int32_t*)(scratch + o_rs);
    uint32_t* cbits = (uint32_t*)(scratch + o_c);
    TapGeom g;
    g.cu = cu_seqlens_dev;
    g.n = n_samples; g.P = P; g.CP = o->cp; g.B = o->block; g.H = H; g.hq = o->hq; g.hkv = o->hkv; g.d = o->head_dim;
    // W * W byte matrices, loads, the volume total and the status start from zero
    const TapSetup setup = {NB, 0, nullptr, nullptr, f_blk, q_home, v_qo, j0, j1, v_smp, res_smp,
                            {fwd_bytes_dev, bwd_bytes_dev, loads_dev}, {(int64_t)W * W, (int64_t)W * W, W}, status_dev, comm_total_dev};
    int rc = launch_setup(g, setup, seq_offsets_host, (int32_t*)(scratch + o_tab), s);
    auto launched = [&](cudaError_t e) { if (e != cudaSuccess) rc = LIBRA_ERR_CUDA; };
    if (rc == LIBRA_OK) {
        launched(launch_dependent(k_tap_rank, (unsigned)((NB + 15) / 16), 256u, 0, s, f_blk, NB, q_home, v_qo, j0, j1, ord, rec));
        // By one block while its tables fit shared memory.  (Bytes for up to eight workers: as few bits a group as the
        // general kernel's bit rows, so that many shards of many samples fit as well.)
        const int per = W <= 32 ? 1 : (W <= 64 ? 2 : 4);
        const size_t smem = sizeof(int64_t) * n_samples + (W <= 8 ? sizeof(uint8_t) : sizeof(uint32_t)) * (size_t)per * H * n_samples;
        if (W <= 128 && smem <= kTapTeamSmem) {
            auto place = W <= 8 ? k_tap_place_team<1, uint8_t>
                                : (W <= 32 ? k_tap_place_team<1, uint32_t> : (W <= 64 ? k_tap_place_team<2, uint32_t> : k_tap_place_team<4, uint32_t>));
            if (smem > 48 * 1024 - kTapTeamStatic * per &&
                cudaFuncSetAttribute(place, cudaFuncAttributeMaxDynamicSharedMemorySize, kTapTeamSmem) != cudaSuccess)
                rc = LIBRA_ERR_CUDA;
            const TapPlace tp = {rec, v_smp, res_smp, NB, (int64_t)4 * o->head_dim, H, W, n_samples, o->tau_num, o->tau_den, words, cbits,
                                 sigma_dev, loads_dev, comm_total_dev, status_dev};
            launched(launch_dependent(place, 1u, kTapThreads, smem, s, tp));
        } else {
            launched(launch_dependent(k_tap_place, 1u, (unsigned)((W + 31) / 32 * 32), 0, s, f_blk, ord, q_home, v_qo, j0, j1, v_smp, res_smp,
                                      NB, H, W, n_samples, o->tau_num, o->tau_den, cbits, words, sigma_dev, loads_dev, comm_total_dev,
                                      status_dev));
        }
        const int64_t threads = NT + (int64_t)n_samples * H * W;
        launched(launch_dependent(k_tap_exchange, (unsigned)((threads + 255) / 256), 256u, 0, s, g, NT, sigma_dev, q_home, v_qo, cbits, words,
                                  res_smp, W, status_dev, (unsigned long long*)fwd_bytes_dev, (unsigned long long*)bwd_bytes_dev));
        count_launch(3);
    }
    scratch_free(scratch, s);
    return rc;
}

extern "C" int libra_tap_schedule(const int32_t* cu_seqlens_dev, int n_samples, const int32_t* seq_offsets_host,
                                  int n_sequences, const libra_tap_opts* o, const int32_t* sigma_dev,
                                  int32_t* records_dev, int64_t capacity, int64_t* n_records_dev, void* stream) {
    if (!cu_seqlens_dev || !seq_offsets_host || !o || !sigma_dev || !records_dev || !n_records_dev || capacity < 0)
        return LIBRA_ERR_INVALID_ARG;
    if (n_samples <= 0 || n_sequences <= 0 || o->cp <= 0 || o->block <= 0 || o->n_shards <= 0 || o->hq <= 0 ||
        o->hkv <= 0 || o->head_dim <= 0 || o->hq % o->n_shards != 0)
        return LIBRA_ERR_INVALID_ARG;
    if ((int64_t)n_sequences * o->cp > kTapMaxWorkers) return LIBRA_ERR_UNSUPPORTED;
    const int P = n_sequences, W = P * o->cp, H = o->n_shards;
    const int64_t NT = libra_tap_num_tiles(seq_offsets_host, P, o->block, H);
    if (NT <= 0) return LIBRA_ERR_INVALID_ARG;
    const int64_t NB = NT / H, NG = (int64_t)n_samples * H;
    if (NT >= INT32_MAX || NG * W >= INT32_MAX) return LIBRA_ERR_UNSUPPORTED;
    cudaStream_t s = (cudaStream_t)stream;
    const int words = (int)((NG + 31) / 32);
    const int64_t slots = NT + NG * W, ctas = (slots + kTapSlots - 1) / kTapSlots;
    uint8_t* scratch = nullptr;
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t at = off; off += (bytes + 255) & ~size_t(255); return at; };
    const size_t o_tab = take(sizeof(int32_t) * 2 * (P + 1));
    const size_t o_q = take(sizeof(int32_t) * NB), o_j0 = take(sizeof(int32_t) * NB), o_j1 = take(sizeof(int32_t) * NB);
    const size_t o_rs = take(sizeof(int32_t) * n_samples);
    const size_t o_m = take(sizeof(uint32_t) * ((size_t)words * W + 1));
    const size_t o_ahead = take(sizeof(int32_t) * (size_t)slots), o_total = take(sizeof(int64_t) * (size_t)ctas);
    if (scratch_alloc((void**)&scratch, off, s) != cudaSuccess) return LIBRA_ERR_CUDA;
    TapGeom g;
    g.cu = cu_seqlens_dev;
    g.n = n_samples; g.P = P; g.CP = o->cp; g.B = o->block; g.H = H; g.hq = o->hq; g.hkv = o->hkv; g.d = o->head_dim;
    int32_t* q_home = (int32_t*)(scratch + o_q);
    int32_t* j0 = (int32_t*)(scratch + o_j0);
    int32_t* j1 = (int32_t*)(scratch + o_j1);
    int32_t* res_smp = (int32_t*)(scratch + o_rs);
    uint32_t* marks = (uint32_t*)(scratch + o_m);
    int32_t* ahead = (int32_t*)(scratch + o_ahead);
    int64_t* total = (int64_t*)(scratch + o_total);
    // the marks start from zero (rows rounded up to whole 64-bit words)
    const TapSetup setup = {NB, 0, nullptr, nullptr, nullptr, q_home, nullptr, j0, j1, nullptr, res_smp,
                            {(int64_t*)marks, nullptr, nullptr}, {((int64_t)words * W + 1) / 2, 0, 0}, nullptr, nullptr};
    int rc = launch_setup(g, setup, seq_offsets_host, (int32_t*)(scratch + o_tab), s);
    auto launched = [&](cudaError_t e) { if (e != cudaSuccess) rc = LIBRA_ERR_CUDA; };
    if (rc == LIBRA_OK) {
        launched(launch_dependent(k_tap_mark, (unsigned)((NT + 255) / 256), 256u, 0, s, sigma_dev, j0, j1, NT, H, W, words, marks));
        launched(launch_dependent(k_tap_sched_count, (unsigned)ctas, kTapSlots, 0, s, g, NT, NG, W, sigma_dev, q_home, marks, words, res_smp,
                                  ahead, total));
        const bool scan = ctas > kTapInlineCtas;
        if (scan) launched(launch_dependent(k_tap_sched_scan, 1u, 1024u, 0, s, ctas, total, n_records_dev));
        launched(launch_dependent(k_tap_sched_fill, (unsigned)ctas, kTapSlots, 0, s, g, NT, NG, W, sigma_dev, q_home, marks, words, res_smp,
                                  ahead, total, scan ? 1 : 0, n_records_dev, capacity, records_dev));
        count_launch(scan ? 4 : 3);
    }
    scratch_free(scratch, s);
    return rc;
}
