// Forward pool attention for sm_100a: one persistent, warp-specialised kernel.
//
// Each CTA walks the query-major tile list the planner gave it.  A tile is 256 query rows
// (two 128-row sub-tiles, "slots") of one head shard; for every head of the shard the CTA
// streams the key/value blocks the rows can see, from the diagonal block down to the block that
// holds the start of the first row's sample.  Blocks are cut at multiples of 128 on the
// pool's token axis, so the diagonal block of a sub-tile is aligned with it and every other
// visible block is either dense or needs the per-row sample-start mask.
//
// Roles (384 threads): warps 0-3 and 4-7 are the softmax groups of slot 0 and 1 (one row per
// thread, S read from TMEM, P written back to TMEM as bf16 over S), warp 8 issues TMA loads,
// warp 9 issues tcgen05.mma, warps 10-11 only hand their registers to the softmax groups.
// TMEM: S0 | S1 | O0 | O1, 128 fp32 columns each.
// Pipeline per key block j:   PV0(j) S0(j-1) PV1(j) S1(j-1)   on the tensor pipe, while the
// softmax group of one slot works during the other slot's MMAs.  Slot 1 sees one block more than slot 0; walking
// the blocks downwards puts its solitary block at the start of a tile, where slot 0 is still storing its last O.
// P is handed over in two parts (keys 0-95, then 96-127), so that only a quarter of PV(j) is left to run when the
// last exponential is done (two 65536-token samples, Hq 32: 60.9 ms, with halves 62.6).
//
// What bounds it: per key block and slot a chain S -> maximum -> exponentials -> PV -> S of about 3100 clk for 2048 clk
// of MMA, and between tiles the drain and refill of that chain.  Masks as bit words and the O tile through a staging
// tile and a bulk tensor store took most off the latter (a masked block cost 1000-3400 clk more than a dense one, the
// row-per-thread stores 3500 clk per slot): 4096 tokens, 4 heads of 64: 39.0 -> 31.3 us; 10007 tokens in samples of up to
// 400, 8 heads of 128: 45.1 -> 32.3 us; 131072 tokens, 32 / 8 heads of 128: 6.63 -> 6.25 ms (945 -> 1000 TFLOP/s).
#include <math.h>

#include "common.h"
#include "ptx.cuh"

#ifndef LIBRA_FWD_REG_DEC
#define LIBRA_FWD_REG_DEC 56
#define LIBRA_FWD_REG_INC 216
#endif

namespace libra {

constexpr int kBM = 128;            // rows per slot
constexpr int kBN = 128;            // keys per block
constexpr int kFwdThreads = 384;  // warps 10-11 only donate registers
constexpr int kPFirst = 96;       // keys of P handed to the MMA role in the first part
constexpr float kRescaleThreshold = 8.0f;  // log2 units: O is rescaled only when the max grows by more
constexpr uint64_t kFwdDrainNs = 2000000;  // teardown after a give-up: budget for work already in flight to land

constexpr int kShareBlocks = 6;    // key blocks of a tile from which two CTAs share it; the hand-over costs two or three of them

template <int D>
struct FwdSmem {
    static constexpr int kHalfBytes = 128 * 128;              // 128 rows x 64 bf16 (one swizzle column)
    static constexpr int kTileBytes = kHalfBytes * (D / 64);  // one 128 x D operand tile
    static constexpr int kStages = (D == 128) ? 4 : 8;
    static constexpr int kQOff = 0;
    static constexpr int kRingOff = 2 * kTileBytes;
    static constexpr int kStageOff = kRingOff + kStages * kTileBytes;  // O staging: per softmax warp 32 rows x 64 bf16
    static constexpr int kBarOff = kStageOff + 8 * 4096;
    // barriers: full[kStages], empty[kStages], q_full, q_empty, s_full[2], p_ready[2], o_done[2], p_part[2], drain, spent,
    // partial
    static constexpr int kNumBars = 2 * kStages + 13;
    static constexpr int kMiscOff = kBarOff + kNumBars * 8;
    static constexpr int kBytes = kMiscOff + 16;
    static constexpr int kAlloc = kBytes + 1024;  // slack to align the base to 1024 B
};

struct FwdParams {
    float* lse;
    const int32_t* cta_offsets;
    const int32_t* cta_tiles;
    const int32_t* tok_start;
    int64_t T;
    int hq, hkv, H;
    float scale_log2;  // softmax scale * log2(e)
    int* outcome;      // [gridDim.x] 0 or what kept this CTA from doing its work
    const int* plan_status;  // the planner's verdict on cu_seqlens: non-zero = do not run
    uint32_t wait_limit_ns;  // budget of one device-side wait
    int inject_stall;        // test aid: the producer (PAIR: of rank 1) issues no loads, so the consumers' waits run out
    uint64_t* busy;    // [2 * gridDim.x]
    uint32_t* tile_ns; // [tiles] time spent on each tile (slot 0's first softmax thread), ns
};

// One tile of the CTA's list: id, first row, key blocks lo[g] .. hi[g] of slot g (lo > hi: the slot lies past T).
struct FwdTile {
    int t;
    int64_t q0;
    int lo[2], hi[2];
    // A tile that a pair of CTAs shares: `shared`, and part[g] when both have key blocks of slot g.
    bool shared, part[2];
    // Takes the CTA's part: rank 0 the upper half of the key blocks, rank 1 the lower; false when nothing is left for it.
    __device__ __forceinline__ bool take_half(uint32_t rank) {
        const int top = hi[1] >= 0 ? hi[1] : hi[0], n = top - lo[0] + 1;
        shared = n >= kShareBlocks;
        part[0] = part[1] = false;
        if (!shared) return rank == 0;
        const int mid = (lo[0] + top + 2) / 2;   // lo[0] < mid <= hi[0]
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            part[g] = lo[g] <= hi[g] && lo[g] < mid;
            if (rank == 0) lo[g] = part[g] ? mid : lo[g];
            else { hi[g] = part[g] ? mid - 1 : -1; lo[g] = part[g] ? lo[g] : 0; }   // slot 1's sample may start in the upper half
        }
        return true;
    }
};
// Walks the list.  Ids are fetched two tiles and sample starts one tile ahead: a chain of two dependent global
// loads between tiles would leave the tensor pipe idle for about 2000 clk.
struct FwdTiles {
    const FwdParams& p;
    int idx, end;
    int t1, t2, a1, b1;   // next tile: id, tok_start of the first row of each slot; id of the one after
    __device__ __forceinline__ FwdTiles(const FwdParams& p_, int begin, int end_) : p(p_), idx(begin), end(end_), a1(0), b1(0) {
        t1 = idx < end ? p.cta_tiles[idx] : -1;
        t2 = idx + 1 < end ? p.cta_tiles[idx + 1] : -1;
        fetch();
    }
    __device__ __forceinline__ void fetch() {
        if (t1 < 0) return;
        const int64_t q0 = (int64_t)(t1 / p.H) * (2 * kBM);
        a1 = p.tok_start[q0];
        b1 = q0 + kBM < p.T ? p.tok_start[q0 + kBM] : 0;
    }
    __device__ __forceinline__ bool next(FwdTile& x) {
        if (t1 < 0) return false;
        x.t = t1;
        x.q0 = (int64_t)(t1 / p.H) * (2 * kBM);
        x.hi[0] = (int)(x.q0 / kBN);
        x.lo[0] = a1 / kBN;
        const bool two = x.q0 + kBM < p.T;
        x.hi[1] = two ? x.hi[0] + 1 : -1;
        x.lo[1] = two ? b1 / kBN : 0;
        ++idx;
        t1 = t2;
        t2 = idx + 1 < end ? p.cta_tiles[idx + 1] : -1;
        fetch();
        return true;
    }
};

// What a thread of a shared tile does when its slot's MMAs are done.  take: 0 the other CTA has nothing of the slot; 1 it
// takes the other's partial output over into its own, in TMEM; 2 it gives its own away.  Returns false on a timeout.  (A
// function of its own: inlined, it cost the loop over key blocks 0.4 us each in spilled registers.)
template <int D>
__device__ __noinline__ bool exchange_partial(uint8_t* smem, uint64_t* bars, uint32_t tmem_base, int take, float& m_ref, float& l_sum) {
    using L = FwdSmem<D>;
    uint64_t* bar_spent = bars + 2 * L::kStages + 11;
    uint64_t* bar_partial = bar_spent + 1;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::kMiscOff + 4);
    const int warp = threadIdx.x >> 5, g = warp >> 2, row_in_tile = threadIdx.x & 127;
    const uint32_t peer = cluster_rank() ^ 1;
    const uint32_t t_o = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + 2 * kBN + g * D;
    float4* partial = reinterpret_cast<float4*>(smem + L::kRingOff) + row_in_tile;   // [D / 4][128]
    float* sums = reinterpret_cast<float*>(smem + L::kQOff) + row_in_tile;           // [2][128]
    // this CTA's ring and Q tiles are spent when the threads of both slots have arrived
    fence_cluster();
    mbar_arrive_cluster(map_to_rank(bar_spent, peer));
    if (take == 0) return true;
    if (take == 2) {
        if (!warp_wait(bar_spent, 0, abort_flag)) return false;
        fence_cluster();
        const uint32_t dst = map_to_rank(partial, peer), dst_s = map_to_rank(sums, peer);
#pragma unroll
        for (int c = 0; c < D; c += 32) {
            uint32_t o[32];
            tmem_ld32(t_o + c, o);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 32; i += 4) st_cluster4(dst + (c + i) * (kBM * 4), o + i);
        }
        st_cluster(dst_s, m_ref);
        st_cluster(dst_s + kBM * 4, l_sum);
        fence_cluster();
        mbar_arrive_cluster(map_to_rank(bar_partial, peer));
        return true;
    }
    if (!warp_wait(bar_partial, 0, abort_flag)) return false;
    fence_cluster();
    const float m1 = sums[0], l1 = sums[kBM], m = fmaxf(m_ref, m1);
    const float own = m > -INFINITY ? ex2_approx(m_ref - m) : 1.0f, other = m > -INFINITY ? ex2_approx(m1 - m) : 0.f;
    m_ref = m;
    l_sum = l_sum * own + l1 * other;
#pragma unroll
    for (int c = 0; c < D; c += 32) {
        uint32_t o[32];
        tmem_ld32(t_o + c, o);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
            const float4 v = partial[(c + i) / 4 * kBM];
            o[i] = __float_as_uint(__uint_as_float(o[i]) * own + v.x * other);
            o[i + 1] = __float_as_uint(__uint_as_float(o[i + 1]) * own + v.y * other);
            o[i + 2] = __float_as_uint(__uint_as_float(o[i + 2]) * own + v.z * other);
            o[i + 3] = __float_as_uint(__uint_as_float(o[i + 3]) * own + v.w * other);
        }
        tmem_st32(t_o + c, o);
    }
    tmem_st_wait();
    return true;
}

// PAIR: a cluster of two CTAs goes through the list of a worker of its own and shares its tiles by key blocks.  When there
// is no more than a tile for every two SMs, the longest tile is the launch: 16 of its key blocks take 26 us (4096 tokens, 4
// heads of 64), at the rate of one slot's chain for each, with 84 SMs idle.  Each rank takes
// the other's maxima, sums and output of the slot of its own number through distributed shared memory and combines: 28.4 ->
// 21.5 us there, one sample of 4096 tokens, 4 heads of 128: 55.3 -> 38.1.
template <int D, bool PAIR>
__global__ void __launch_bounds__(kFwdThreads, 1)
k_attn_fwd(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
           const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_out, const FwdParams p) {
    using L = FwdSmem<D>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::kBarOff);
    uint64_t* bar_full = bars;
    uint64_t* bar_empty = bars + L::kStages;
    uint64_t* bar_qfull = bars + 2 * L::kStages;
    uint64_t* bar_qempty = bar_qfull + 1;
    uint64_t* bar_sfull = bar_qfull + 2;   // [2]
    uint64_t* bar_pready = bar_qfull + 4;  // [2]
    uint64_t* bar_odone = bar_qfull + 6;   // [2]
    uint64_t* bar_ppart = bar_qfull + 8;   // [2] P of the first kPFirst keys is in TMEM
    uint64_t* bar_drain = bar_qfull + 10;  // teardown after a give-up: every MMA issued so far has completed
    uint64_t* bar_spent = bar_qfull + 11;    // PAIR: the other CTA's ring is spent, a partial output may go there
    uint64_t* bar_partial = bar_qfull + 12;  // PAIR: the other CTA's partial output is here
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::kMiscOff);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::kMiscOff + 4);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const uint32_t rank = PAIR ? cluster_rank() : 0;
    const int worker = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
    const int cta = PAIR ? worker + (int)(rank * (gridDim.x >> 1)) : worker;   // where the CTA reports

    if (threadIdx.x == 0) {
        mbar_init(bar_spent, 2 * kBM);
        mbar_init(bar_partial, kBM);
        for (int i = 0; i < L::kStages; ++i) { mbar_init(&bar_full[i], 1); mbar_init(&bar_empty[i], 1); }
        mbar_init(bar_qfull, 1);
        mbar_init(bar_qempty, 1);
        for (int g = 0; g < 2; ++g) {
            mbar_init(&bar_sfull[g], 1);
            mbar_init(&bar_pready[g], kBM);
            mbar_init(&bar_odone[g], 1);
            mbar_init(&bar_ppart[g], kBM);
        }
        mbar_init(bar_drain, 1);
        abort_flag[0] = 0;
        abort_flag[1] = (int)p.wait_limit_ns;
        fence_mbar_init();
    }
    if (warp == 8 && lane == 0) {
        prefetch_tmap(&tm_q);
        prefetch_tmap(&tm_k);
        prefetch_tmap(&tm_v);
        prefetch_tmap(&tm_out);
    }
    if (PAIR) cluster_arrive();
    grid_dep_wait();
    // A plan whose cu_seqlens failed the planner's check is never executed: report and leave.
    if (const int ps = *p.plan_status; ps != 0) {
        if (threadIdx.x == 0) { p.outcome[cta] = ps; p.busy[2 * cta] = p.busy[2 * cta + 1] = 0; }
        if (PAIR) cluster_wait();
        return;
    }
    if (threadIdx.x == 0) p.busy[2 * cta] = globaltimer_ns();
    if (warp == 9) {
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    if (PAIR) cluster_wait();   // the other CTA's barriers are initialised
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    const int tile_begin = p.cta_offsets[worker];
    const int tile_end = p.cta_offsets[worker + 1];
    const int heads_per_shard = p.hq / p.H;
    const int G = p.hq / p.hkv;

    // The softmax groups hold a whole 128-column row of S in registers; the producer / MMA
    // warpgroup needs few registers and hands the rest over.
    if (warp >= 10) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(LIBRA_FWD_REG_DEC));
    } else if (warp == 8) {
        // ---------------- TMA producer ----------------
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(LIBRA_FWD_REG_DEC));
        if (elect_one()) {  // one elected thread runs the whole role
            uint32_t ring = 0, qcnt = 0;
            bool ok = true;
            FwdTiles tiles(p, tile_begin, tile_end);
            FwdTile x;
            while (ok && !(p.inject_stall && (!PAIR || cluster_rank() == 1)) && tiles.next(x)) {
                if (PAIR && !x.take_half(cluster_rank())) continue;
                const bool act1 = x.hi[1] >= 0;
                const int top = act1 ? x.hi[1] : x.hi[0];
                for (int hh = 0; hh < heads_per_shard && ok; ++hh) {
                    const int h = (x.t % p.H) * heads_per_shard + hh;
                    const int kvh = h / G;
                    for (int j = top; j >= x.lo[0] && ok; --j) {
                        for (int kv = 0; kv < 2; ++kv) {  // K_j then V_j
                            const uint32_t st = ring % L::kStages;
                            ok = mbar_wait(&bar_empty[st], ((ring / L::kStages) & 1) ^ 1, abort_flag);
                            if (!ok) break;
                            mbar_arrive_expect_tx(&bar_full[st], L::kTileBytes);
                            for (int half = 0; half < D / 64; ++half)
                                tma_load_3d(smem + L::kRingOff + st * L::kTileBytes + half * L::kHalfBytes,
                                            kv == 0 ? &tm_k : &tm_v, &bar_full[st], half * 64, kvh, j * kBN);
                            ++ring;
                            if (j == top && kv == 0) {   // Q behind the first K: the wait for its tile holds nothing else up
                                ok = mbar_wait(bar_qempty, (qcnt & 1) ^ 1, abort_flag);
                                if (!ok) break;
                                mbar_arrive_expect_tx(bar_qfull, (act1 ? 2 : 1) * L::kTileBytes);
                                for (int g = 1; g >= 0; --g)
                                    for (int half = 0; half < D / 64; ++half)
                                        if (g == 0 || act1)
                                            tma_load_3d(smem + L::kQOff + g * L::kTileBytes + half * L::kHalfBytes, &tm_q,
                                                        bar_qfull, half * 64, h, (int)(x.q0 + g * kBM));
                                ++qcnt;
                            }
                        }
                    }
                }
            }
            if (!ok || abort_flag[0]) {
                // Give-up path: nothing new is issued; the copies already issued land before shared memory is released.
                if (qcnt > 0) mbar_wait_drain(bar_qfull, (qcnt - 1) & 1, kFwdDrainNs);
                for (uint32_t b = 1; b <= (uint32_t)L::kStages && b <= ring; ++b)
                    mbar_wait_drain(&bar_full[(ring - b) % L::kStages], ((ring - b) / L::kStages) & 1, kFwdDrainNs);
            }
        }
        __syncwarp();
    } else if (warp == 9) {
        // ---------------- MMA issuer ----------------
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(LIBRA_FWD_REG_DEC));
        if (elect_one()) {  // one elected thread runs the whole role
            constexpr uint32_t idesc_s = make_idesc(kBM, kBN, 0, 0);
            constexpr uint32_t idesc_pv = make_idesc(kBM, D, 0, 1);
            const uint32_t smem_base = smem_u32(smem);
            uint32_t ring = 0, qcnt = 0;
            uint32_t pcnt[2] = {0, 0};
            bool ok = true;
            // Base descriptors are built once; every MMA only adds a constant to them.
            const uint64_t desc_q = make_sdesc(smem_base + L::kQOff, 16, 1024);                  // K-major Q slot 0
            const uint64_t desc_k = make_sdesc(smem_base + L::kRingOff, 16, 1024);               // K-major ring stage 0
            const uint64_t desc_v = make_sdesc(smem_base + L::kRingOff, L::kHalfBytes, 1024);    // MN-major ring stage 0
            auto issue_s = [&](int g, uint32_t stage) {
                const uint64_t qa = sdesc_advance(desc_q, g * L::kTileBytes);
                const uint64_t ka = sdesc_advance(desc_k, stage * L::kTileBytes);
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk) {
                    const uint32_t off = (kk / 4) * L::kHalfBytes + (kk % 4) * 32;
                    mma_ss(tmem_base + g * kBN, sdesc_advance(qa, off), sdesc_advance(ka, off), idesc_s, kk > 0);
                }
                tc_commit(&bar_sfull[g]);
            };
            // O[g] (+)= P[g] V over the key steps [kk0, kk1) of 16 keys; the softmax group hands P over in two parts
            auto issue_pv = [&](int g, uint32_t stage, bool accumulate, int kk0, int kk1) {
                const uint64_t va = sdesc_advance(desc_v, stage * L::kTileBytes);
#pragma unroll
                for (int kk = kk0; kk < kk1; ++kk) {
                    mma_ts(tmem_base + 2 * kBN + g * D, tmem_base + g * kBN + kk * 8, sdesc_advance(va, kk * 2048), idesc_pv,
                           (accumulate || kk > 0) ? 1u : 0u);
                }
                if (kk1 == kBN / 16) tc_commit(&bar_odone[g]);
            };
            FwdTiles tiles(p, tile_begin, tile_end);
            FwdTile x;
            while (ok && tiles.next(x)) {
                if (PAIR && !x.take_half(cluster_rank())) continue;
                const bool act1 = x.hi[1] >= 0;
                const int top = act1 ? x.hi[1] : x.hi[0], lo = x.lo[0];
                for (int hh = 0; hh < heads_per_shard && ok; ++hh) {
                    // prologue: S of the top block (slot 1's diagonal block; slot 0's when the tile has no slot 1)
                    uint32_t st = ring % L::kStages;
                    ok = mbar_wait(&bar_full[st], (ring / L::kStages) & 1, abort_flag);
                    if (ok) ok = mbar_wait(bar_qfull, qcnt & 1, abort_flag);
                    if (!ok) break;
                    ++qcnt;
                    tc_fence_after();
                    issue_s(act1 ? 1 : 0, st);
                    if (PAIR && act1 && x.hi[0] == top) issue_s(0, st);   // the lower half of a shared tile
                    tc_commit(&bar_empty[st]);
                    if (lo == top) tc_commit(bar_qempty);  // no later MMA of this tile reads Q
                    ++ring;
                    for (int j = top; j >= lo && ok; --j) {
                        const uint32_t st_v = ring % L::kStages;
                        const uint32_t ph_v = (ring / L::kStages) & 1;
                        ++ring;
                        const bool more = j - 1 >= lo;
                        const uint32_t st_k = ring % L::kStages;
                        bool have_k = false, have_v = false;
#pragma unroll
                        for (int g = 0; g < 2; ++g) {
                            if (j >= x.lo[g] && j <= x.hi[g]) {
                                if (!have_v) { ok = mbar_wait(&bar_full[st_v], ph_v, abort_flag); have_v = true; }
                                if (ok) ok = mbar_wait(&bar_ppart[g], pcnt[g] & 1, abort_flag);   // P of the first kPFirst keys
                                if (!ok) break;
                                tc_fence_after();
                                issue_pv(g, st_v, j != x.hi[g], 0, kPFirst / 16);
                                ok = mbar_wait(&bar_pready[g], pcnt[g] & 1, abort_flag);  // the rest, while those MMAs run
                                if (!ok) break;
                                ++pcnt[g];
                                tc_fence_after();
                                issue_pv(g, st_v, j != x.hi[g], kPFirst / 16, kBN / 16);
                            }
                            if (more && j - 1 >= x.lo[g] && j - 1 <= x.hi[g]) {
                                if (!have_k) { ok = mbar_wait(&bar_full[st_k], (ring / L::kStages) & 1, abort_flag); have_k = true; }
                                if (!ok) break;
                                issue_s(g, st_k);
                            }
                        }
                        if (!ok) break;
                        tc_commit(&bar_empty[st_v]);
                        if (more) { tc_commit(&bar_empty[st_k]); ++ring; }
                        if (j - 1 == lo) tc_commit(bar_qempty);  // S(lo) was the last reader of Q: the next
                    }                                            // tile's Q load overlaps the last block
                }
            }
            if (!ok || abort_flag[0]) {   // give-up path: the MMAs already issued finish before TMEM is freed
                tc_commit(bar_drain);
                mbar_wait_drain(bar_drain, 0, kFwdDrainNs);
            }
        }
        __syncwarp();
    } else {
        // ---------------- softmax groups ----------------
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(LIBRA_FWD_REG_INC));
        const int g = warp >> 2;
        const int row_in_tile = (warp & 3) * 32 + lane;
        const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t t_s = tmem_base + lane_addr + g * kBN;
        const uint32_t t_o = tmem_base + lane_addr + 2 * kBN + g * D;
        uint8_t* stage = smem + L::kStageOff + warp * 4096;
        const uint64_t scale2 = f2_pack(p.scale_log2, p.scale_log2);
        uint32_t scnt = 0, ocnt = 0;
        bool ok = true;
        // O *= factor, once the PV of the previous block has landed in it
        auto rescale_o = [&](float factor) -> bool {
            if (!warp_wait(&bar_odone[g], (ocnt - 1) & 1, abort_flag)) return false;
            tc_fence_after();
#pragma unroll
            for (int c = 0; c < D; c += 32) {
                uint32_t orow[32];
                tmem_ld32(t_o + c, orow);
                tmem_ld_wait();
#pragma unroll
                for (int i = 0; i < 32; ++i) orow[i] = __float_as_uint(__uint_as_float(orow[i]) * factor);
                tmem_st32(t_o + c, orow);
            }
            tmem_st_wait();
            return true;
        };
        FwdTiles tiles(p, tile_begin, tile_end);
        FwdTile x;
        while (ok && tiles.next(x)) {
            if (PAIR && !x.take_half(cluster_rank())) continue;
            const int64_t qs = x.q0 + g * kBM;
            const int lo = x.lo[g], hi = x.hi[g];
            if (lo > hi) {  // slot past the end of the pool, or all in the other CTA
                if (PAIR && x.shared) mbar_arrive_cluster(map_to_rank(bar_spent, cluster_rank() ^ 1));
                continue;
            }
            const uint64_t tile_t0 = threadIdx.x == 0 ? globaltimer_ns() : 0;
            const int64_t row = qs + row_in_tile;
            const bool row_ok = row < p.T;
            const int kstart = row_ok ? p.tok_start[row] : 0;
            // last valid row of the slot decides which blocks need the sample-start mask
            const int64_t last_row = (qs + kBM <= p.T ? qs + kBM : p.T) - 1;
            const int max_kstart = p.tok_start[last_row];
            for (int hh = 0; hh < heads_per_shard && ok; ++hh) {
                const int h = (x.t % p.H) * heads_per_shard + hh;
                float m_ref = -INFINITY, l_sum = 0.f;
                for (int j = hi; j >= lo && ok; --j) {
                    ok = warp_wait(&bar_sfull[g], scnt & 1, abort_flag);
                    if (!ok) break;
                    ++scnt;
                    tc_fence_after();
                    uint32_t sr[kBN];
                    tmem_ld32(t_s, sr);
                    tmem_ld32(t_s + 32, sr + 32);
                    tmem_ld32(t_s + 64, sr + 64);
                    tmem_ld32(t_s + 96, sr + 96);
                    tmem_ld_wait();
                    const int k0 = j * kBN;
                    if (j == hi || k0 < max_kstart) {   // (rows past the pool: anything finite)
                        const int c_lo = row_ok ? kstart - k0 : 0;           // first visible column
                        const int c_hi = row_ok ? (int)(row - k0) : kBN;     // last visible column
#pragma unroll
                        for (int w = 0; w < kBN / 32; ++w) {
                            const uint32_t vis = range_bits(c_lo - 32 * w, c_hi - 32 * w);
#pragma unroll
                            for (int i = 0; i < 32; ++i) sr[32 * w + i] = (vis >> i) & 1u ? sr[32 * w + i] : 0xff800000u;  // -inf
                        }
                    }
                    float mx;
                    {   // eight independent chains keep the 3-input max off the latency-bound path
                        float pm[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) pm[u] = fmaxf(__uint_as_float(sr[2 * u]), __uint_as_float(sr[2 * u + 1]));
#pragma unroll
                        for (int i = 16; i < kBN; i += 16)
#pragma unroll
                            for (int u = 0; u < 8; ++u)
                                pm[u] = max3(pm[u], __uint_as_float(sr[i + 2 * u]), __uint_as_float(sr[i + 2 * u + 1]));
                        mx = fmaxf(max3(pm[0], pm[1], pm[2]), max3(pm[3], pm[4], pm[5]));
                        mx = max3(mx, pm[6], pm[7]);
                    }
                    mx *= p.scale_log2;  // scale > 0, so the max commutes with it
                    // lazy rescale: keep the old reference unless the max grew by > threshold
                    float factor = 1.0f;
                    if (mx > m_ref + kRescaleThreshold) {
                        factor = ex2_approx(m_ref - mx);   // m_ref = -inf gives 0
                        m_ref = mx;
                    }
                    if (j != hi && __any_sync(0xffffffffu, factor != 1.0f)) {
                        ok = rescale_o(factor);
                        if (!ok) break;
                    }
                    l_sum *= factor;
                    const float m_use = (m_ref == -INFINITY) ? 0.f : m_ref;
                    const uint64_t negm2 = f2_pack(-m_use, -m_use);
                    uint64_t psum2[4] = {f2_pack(0.f, 0.f), f2_pack(0.f, 0.f), f2_pack(0.f, 0.f), f2_pack(0.f, 0.f)};
#pragma unroll
                    for (int c = 0; c < kBN; c += 32) {
                        uint32_t pk[16];
#pragma unroll
                        for (int i = 0; i < 32; i += 2) {
                            float x0, x1;
                            f2_unpack(f2_fma(f2_pack(__uint_as_float(sr[c + i]), __uint_as_float(sr[c + i + 1])), scale2, negm2),
                                      x0, x1);
                            const float p0 = ex2_approx(x0), p1 = ex2_approx(x1);
                            psum2[(i >> 1) & 3] = f2_add(psum2[(i >> 1) & 3], f2_pack(p0, p1));
                            pk[i >> 1] = pack_bf16x2(p0, p1);
                        }
                        tmem_st16(t_s + (c >> 1), pk);
                        if (c == kPFirst - 32) {  // P of the first kPFirst keys is complete: its PV steps can start
                            tmem_st_wait();
                            tc_fence_before();
                            mbar_arrive(&bar_ppart[g]);
                        }
                    }
                    {
                        float a, b;
                        f2_unpack(f2_add(f2_add(psum2[0], psum2[1]), f2_add(psum2[2], psum2[3])), a, b);
                        l_sum += a + b;
                    }
                    tmem_st_wait();
                    tc_fence_before();
                    mbar_arrive(&bar_pready[g]);
                    ++ocnt;
                }
                if (!ok) break;
                // epilogue: wait for the last PV, normalise, store
                ok = warp_wait(&bar_odone[g], (ocnt - 1) & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                if (PAIR && x.shared) {
                    const int take = x.part[g] ? ((int)cluster_rank() == g ? 1 : 2) : 0;
                    float m = m_ref, l = l_sum;
                    ok = __all_sync(0xffffffffu, exchange_partial<D>(smem, bars, tmem_base, take, m, l));
                    m_ref = m;
                    l_sum = l;
                    if (!ok || take == 2) break;
                }
                const float inv_l = (l_sum > 0.f) ? 1.0f / l_sum : 0.f;
                // Through the warp's staging tile (32 rows x 128 bytes, 128-byte swizzle) and a bulk tensor store: one row
                // per thread stored straight from registers touches 32 cache lines per instruction.  Rows past the end
                // of the pool are dropped by the hardware.
#pragma unroll
                for (int c = 0; c < D; c += 64) {
                    uint32_t orow[64];
                    tmem_ld32(t_o + c, orow);
                    tmem_ld32(t_o + c + 32, orow + 32);
                    tmem_ld_wait();
                    if (lane == 0) tma_store_wait_read();   // the store that last used the tile has read it
                    __syncwarp();
#pragma unroll
                    for (int ch = 0; ch < 8; ++ch) {
                        uint4 v;
                        const uint32_t* o = orow + 8 * ch;
                        v.x = pack_bf16x2(__uint_as_float(o[0]) * inv_l, __uint_as_float(o[1]) * inv_l);
                        v.y = pack_bf16x2(__uint_as_float(o[2]) * inv_l, __uint_as_float(o[3]) * inv_l);
                        v.z = pack_bf16x2(__uint_as_float(o[4]) * inv_l, __uint_as_float(o[5]) * inv_l);
                        v.w = pack_bf16x2(__uint_as_float(o[6]) * inv_l, __uint_as_float(o[7]) * inv_l);
                        *reinterpret_cast<uint4*>(stage + lane * 128 + ((ch ^ (lane & 7)) << 4)) = v;
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        tma_store_3d(&tm_out, stage, c, h, (int)(qs + (warp & 3) * 32));
                        tma_store_commit();
                    }
                }
                if (row_ok) p.lse[(size_t)h * p.T + row] = (m_ref + log2f(l_sum)) * 0.6931471805599453f;
                // the next PV into this slot's O may only start after these reads: it is issued
                // after this group's next P arrival, which follows in program order
                tc_fence_before();
            }
            if (threadIdx.x == 0 && ok && (!PAIR || cluster_rank() == 0)) p.tile_ns[x.t] = (uint32_t)(globaltimer_ns() - tile_t0);
        }
        // every bulk store this warp issued has completed before the CTA leaves
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }

    // ---------------- teardown ----------------
    tc_fence_before();
    __syncthreads();
    if (PAIR) cluster_sync();   // nothing of the other CTA is on its way here any more
    if (warp == 9) tmem_dealloc(tmem_base, 512);
    if (threadIdx.x == 0) {
        p.outcome[cta] = *abort_flag ? LIBRA_ERR_TIMEOUT : LIBRA_OK;
        p.busy[2 * cta + 1] = globaltimer_ns();
    }
}

// ---- host ---------------------------------------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn get_encode() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(ptr);
    }
    return fn;
}

// bf16 tensor [T, H, d] viewed as (d, H, T); box = 64 x 1 x 128 rows, 128-byte swizzle, zero fill.
int make_thd_map(CUtensorMap* m, const void* base, int64_t T, int H, int d, int box_rows) {
    EncodeTiledFn enc = get_encode();
    if (!enc) return LIBRA_ERR_CUDA;
    cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)H, (cuuint64_t)T};
    cuuint64_t strides[2] = {(cuuint64_t)d * 2, (cuuint64_t)H * d * 2};
    cuuint32_t box[3] = {64, 1, (cuuint32_t)box_rows};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? LIBRA_OK : LIBRA_ERR_CUDA;
}

int make_f32_3d_map(CUtensorMap* m, const void* base, int64_t T, int H, int d, int box_cols, int box_rows) {
    EncodeTiledFn enc = get_encode();
    if (!enc) return LIBRA_ERR_CUDA;
    cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)H, (cuuint64_t)T};
    cuuint64_t strides[2] = {(cuuint64_t)d * 4, (cuuint64_t)H * d * 4};
    cuuint32_t box[3] = {(cuuint32_t)box_cols, 1, (cuuint32_t)box_rows};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(base), dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? LIBRA_OK : LIBRA_ERR_CUDA;
}

template <int D, bool PAIR>
static int launch_fwd(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tout,
                      const FwdParams& prm, int W, libra_plan_t* mp, cudaStream_t s) {
    using L = FwdSmem<D>;
    constexpr int kSlot = (D == 128 ? 0 : 1) + (PAIR ? 5 : 0);
    if (!cfg_done(kSlot)) {   // per device: the attribute belongs to the device's copy of the kernel
        if (cudaFuncSetAttribute(k_attn_fwd<D, PAIR>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::kAlloc) != cudaSuccess)
            return LIBRA_ERR_CUDA;
        if (!regs_pool_ok(k_attn_fwd<D, PAIR>, 256, LIBRA_FWD_REG_INC, 128, LIBRA_FWD_REG_DEC)) return LIBRA_ERR_UNSUPPORTED;
        cfg_mark(kSlot);
    }
    count_launch();
    mp->n_outcome[0] = PAIR ? W / 2 * 2 : W;
    const cudaError_t e = launch_dependent<PAIR ? 2 : 1>(k_attn_fwd<D, PAIR>, mp->n_outcome[0], kFwdThreads, L::kAlloc, s, tq, tk, tv,
                                                         tout, prm);
    return e == cudaSuccess ? LIBRA_OK : LIBRA_ERR_CUDA;
}

}  // namespace libra

using namespace libra;


extern "C" int libra_attn_pool_fwd(const void* q_dev, const void* k_dev, const void* v_dev,
                                   const int32_t* cu_seqlens_dev, const libra_plan_t* plan, void* out_dev,
                                   float* lse_dev, const libra_dims* dims, void* stream) {
    if (!q_dev || !k_dev || !v_dev || !cu_seqlens_dev || !plan || !out_dev || !lse_dev || !dims)
        return LIBRA_ERR_INVALID_ARG;
    if (dims->hq <= 0 || dims->hkv <= 0 || dims->hq % dims->hkv) return LIBRA_ERR_INVALID_ARG;
    if (dims->head_dim != 64 && dims->head_dim != 128 && dims->head_dim != 256) return LIBRA_ERR_UNSUPPORTED;
    const PlanDir& d = plan->dir[0];
    if (!d.enabled || plan->T != dims->total_tokens) return LIBRA_ERR_PLAN_MISMATCH;
    if (d.tile != 2 * kBM) return LIBRA_ERR_UNSUPPORTED;
    if (dims->hq % d.H) return LIBRA_ERR_INVALID_ARG;
    if (d.W > plan->sm_count) return LIBRA_ERR_UNSUPPORTED;  // one CTA per SM owns all 512 TMEM columns
    if (((uintptr_t)q_dev | (uintptr_t)k_dev | (uintptr_t)v_dev | (uintptr_t)out_dev) & 15) return LIBRA_ERR_INVALID_ARG;
    if (int rcd = check_plan_device(plan); rcd != LIBRA_OK) return rcd;

    const float scale = dims->softmax_scale > 0.f ? dims->softmax_scale : 1.0f / sqrtf((float)dims->head_dim);
    cudaStream_t s = (cudaStream_t)stream;
    libra_plan_t* mp = const_cast<libra_plan_t*>(plan);
    if (s) mp->other_stream = 1;
    if (dims->head_dim == 256) {
        time_begin(mp, 0, s);
        const int rc256 = launch_fwd_d256(q_dev, k_dev, v_dev, out_dev, lse_dev, plan, dims, scale, s);
        time_end(mp, 0, s);
        return rc256;
    }
    CUtensorMap tq, tk, tv, tout;
    int rc = make_thd_map(&tq, q_dev, plan->T, dims->hq, dims->head_dim, kBM);
    if (rc == LIBRA_OK) rc = make_thd_map(&tk, k_dev, plan->T, dims->hkv, dims->head_dim, kBN);
    if (rc == LIBRA_OK) rc = make_thd_map(&tv, v_dev, plan->T, dims->hkv, dims->head_dim, kBN);
    if (rc == LIBRA_OK) rc = make_thd_map(&tout, out_dev, plan->T, dims->hq, dims->head_dim, 32);
    if (rc != LIBRA_OK) return rc;

    FwdParams prm;
    prm.lse = lse_dev;
    prm.cta_offsets = d.d_cta_offsets;
    prm.cta_tiles = d.d_cta_exec;
    prm.tok_start = plan->d_tok_start;
    prm.T = plan->T;
    prm.hq = dims->hq;
    prm.hkv = dims->hkv;
    prm.H = d.H;
    prm.scale_log2 = scale * 1.4426950408889634f;
    prm.outcome = plan->d_outcome[0];
    prm.plan_status = plan->d_status;
    prm.wait_limit_ns = plan->wait_limit_ns;
    prm.inject_stall = plan->inject_stall;
    prm.busy = d.d_busy;
    prm.tile_ns = d.d_tile_ns;
    time_begin(mp, 0, s);
    // Two CTAs a tile when there are two for each (the first NT workers then have one tile each), a tile is one head (the
    // exchange goes through the spent ring) and samples, empty ones counted, average four key blocks (the longest, which
    // bounds the launch, is not known here): 4000 tokens, 4 heads of 128, in samples of up to 300 / 800 / 4000 tokens took
    // 12.0 / 18.0 / 55.3 us with one CTA a tile and 14.0 / 18.4 / 38.1 with two.
    const bool pair = d.NT <= d.W / 2 && d.H == dims->hq && plan->T >= 4 * kBN * (int64_t)plan->n;
    if (dims->head_dim == 128)
        rc = pair ? launch_fwd<128, true>(tq, tk, tv, tout, prm, d.W, mp, s) : launch_fwd<128, false>(tq, tk, tv, tout, prm, d.W, mp, s);
    else
        rc = pair ? launch_fwd<64, true>(tq, tk, tv, tout, prm, d.W, mp, s) : launch_fwd<64, false>(tq, tk, tv, tout, prm, d.W, mp, s);
    time_end(mp, 0, s);
    return rc;
}

