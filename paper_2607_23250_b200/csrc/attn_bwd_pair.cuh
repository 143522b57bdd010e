// Fused backward on pairs of CTAs (included by attn_bwd.cu): the five GEMMs of attn_bwd_fused.cuh for 256 keys, two
// neighbouring key blocks, with cta_group::2 MMAs.
//
// What bounds the kernel of one CTA is the bandwidth of shared memory: of a 128 x 128 cell its MMAs read 256 KB (S and dP
// 64 each, dQ 64, dV and dK 32), the copies of Q and dO write 64, dS^T 32, and dQ goes in and out of its staging tile,
// 128 KB: 480 KB, 3840 clk at 128 bytes a clk, for 2560 of MMA, and 5350 in all.  A pair halves every B operand and adds the
// two key blocks' dQ up before it leaves: 384 KB or 3072 clk a cell, 4140 in all, which is at neither limit, and half the
// reduce-adds in L2, which cost the most power.
//
// CTA c of a pair has key block 2 J + c in its TMEM lanes and owns K and V of it.  Of what the GEMMs multiply with it holds
//   Qr, dOr  rows 64 c .. 64 c + 63 of the query block, all columns    (B of S^T and dP^T, N = queries)
//   Qc, dOc  all rows, columns 64 c .. 64 c + 63                       (B of dK and dV, N = head-dim columns)
//   Kc       K of all 256 keys, columns 64 c .. 64 c + 63              (B of dQ)
//   dS       dS^T of all 256 keys, queries 64 c .. 64 c + 63           (A of dQ, M = 128 = 64 rows of either CTA)
// so half of each CTA's dS^T tile goes to the other, a bulk copy of 4 KB a warp between the two shared memories (stores into
// the other CTA's with a fence behind them held an iteration up by 5000 clk); a thread of the receiving CTA tells the
// leader.  dQ of M = 128 lies in TMEM as 64 rows x 128 columns on 128 lanes x 64 columns: lanes 64 .. 127 hold columns
// 64 .. 127 of the same rows.
// TMEM: X | P^T | dS^T | dK | dV = 128 + 64 + 64 + 128 + 128 columns; X holds S^T, then dP^T; dQ goes over dS^T, which dK has
// read (MMAs run in issue order).  P^T of the next iteration does not wait for dQ.
// MMA order per iteration: S(it+1), dV(it), dP(it+1), dK(it), dQ(it), all issued by the leader (even rank), whose barriers
// count the copies and the warps of both; commits arrive in both.
// Roles (640 threads): two exp groups, a dS group, a dQ group (TMEM -> staging -> bulk reduce-adds), the TMA thread, the
// MMA thread, the thread that waits for the other CTA's half of dS, and the one that watches the clock for all of them.
// The roles' code has to stay in the instruction caches: what is larger comes from caches that neighbouring SMs share, and
// then they hold one another up.  clk a cell with four pairs at work and with all 74, by size of the kernel: 82 KB 4400 and
// 7050; 67 KB 4290 and 5490; 60 KB with the MMA thread's loops rolled up 4790 and 5100; this, 57 KB, 4140 and 4260.  Hence one
// site for all loads, one warp that looks at the clock for all waits, and the exponentials of both halves in one loop.
// Fused kernel of 65536 / 16384 tokens in one sample, 32 / 8 heads: 92.5 -> 80.6, 5.94 -> 5.16 ms; 16 samples of 2048: 1.72 ->
// 1.57; 32 of 1024: 0.965 -> 0.940.
// A key block that sees nothing of a query block (the upper one at the diagonal, the lower one past the end of its
// samples) leaves its lanes out of dV and dK and its keys out of dQ, so that an infinity or NaN spreads no further than
// its 128 x 128 cell, as in the kernel of one CTA.
#pragma once

#include "drain.cuh"

namespace libra {

constexpr int kPairThreads = 640;
constexpr int kPrDqWarp = 12, kPrTmaWarp = 16, kPrMmaWarp = 17, kPrInWarp = 18, kPrWatchWarp = 19;
// setmaxnreg: 640 threads x 96 compiled registers = 256 x 104 + 128 x (120 + 80 + 72)
constexpr int kPrRegsExp = 104, kPrRegsDs = 120, kPrRegsDq = 80, kPrRegsOther = 72;

struct PairSmem {
    static constexpr int kTile = 32768;        // 128 x 128 bf16
    static constexpr int kHalf = 16384;        // 128 x 64
    static constexpr int kRowHalf = 8192;      // 64 x 64
    static constexpr int kKOff = 0;
    static constexpr int kVOff = kTile;
    static constexpr int kKcOff = 2 * kTile;
    static constexpr int kQrOff = 3 * kTile;   // two column halves of 64 rows
    static constexpr int kQcOff = kQrOff + kHalf;
    static constexpr int kDorOff = kQcOff + kHalf;
    static constexpr int kDocOff = kDorOff + kHalf;
    static constexpr int kDsOff = kDocOff + kHalf;
    static constexpr int kOutOff = kDsOff + kTile;         // dS^T of this CTA's keys and the other's queries
    static constexpr int kStageOff = kOutOff + kHalf;      // per dQ warp a tile of 32 rows x 32 floats, swizzled
    static constexpr int kLseOff = kStageOff + kHalf;      // two buffers of lse2[128], by the iteration's parity
    static constexpr int kDvecOff = kLseOff + 2 * 512;     // and of dvec[128]
    static constexpr int kBarOff = kDvecOff + 2 * 512;
    enum Bar {
        // leader: both CTAs' copies have landed.  Their order is that of the loads' kinds (PairLoad).
        kQrFull, kDocFull, kDorFull, kQcFull, kKvFull,
        // both: the MMAs that read them have run (S^T, dP^T: so they are in TMEM)
        kSFull, kDocEmpty, kDpFull, kQcEmpty, kKvEmpty,
        // each CTA's own copies
        kLseFull, kLseFull1, kDvecFull, kDvecFull1,
        kDqFull, kDkvFull,                             // both: dQ is in TMEM; a unit's dK and dV are
        // leader: dP^T, S^T read; P^T in TMEM; dS^T in TMEM and in the CTAs' own halves of dS; the other halves
        kXFree2, kXFree1, kPReady, kDsTmem, kDsSmem,
        kPHalf, kPLocal, kPRead, kZFree,               // own: P^T of 2 x 32 queries, all of it; read by the dS group; dQ read
        kDsIn,                                         // own: the other CTA's half of dS is here
        kDkvEmpty,                                     // both: dK and dV of a unit have left both CTAs
        kDrain,
        kNumBars
    };
    static constexpr int kMiscOff = kBarOff + kNumBars * 8;
    static constexpr int kBytes = kMiscOff + 16 + 2 * 5 * 4 + 4 * 4 + 16;
    static_assert(kBytes <= kSmemMax, "exceeds the shared memory of an sm_100 CTA");
};
enum PairLoad { kLoadQr, kLoadDoc, kLoadDor, kLoadQc, kLoadKv, kPairLoads };   // in the order of an iteration
__device__ constexpr uint32_t pair_load_bytes(int kind) { return kind == kLoadKv ? 3 * 32768 : 16384; }   // by either CTA

struct PairParams {
    const float* lse2;  // [Hq, Tpad]  LSE * log2(e)
    const float* dvec;  // [Hq, Tpad]  D_i
    const int32_t* cta_offsets;
    const int32_t* cta_tiles;
    const int32_t* u_blk;     // 256-key block of wide pair-block u
    const int32_t* u_chunk;   // query chunk of it
    const int32_t* tok_end;
    int64_t T, Tpad;
    int NU;                   // wide pair-blocks
    int hq, hkv, R;           // R = row blocks per query chunk
    float scale_log2;
    int* outcome;
    const int* plan_status;
    uint32_t wait_limit_ns;
    int inject_stall;         // test aid: the odd CTAs' producers issue no loads
    uint64_t* busy;
    // times by 128-key pair tiles, the halves of the wide ones (same chunks): tile h NU128 + base[c] + j - first_j[c]
    uint32_t* tile_ns;
    const int32_t* first_j;
    const int64_t* base;
    int64_t NU128;
};

// The row blocks [i0, i0 + n_blk) that a wide pair tile walks for every head of its group.
struct PairUnit {
    int kvh, c, j0, i0, n_blk;
    int last0;                // last row block that sees the lower key block
    bool two;                 // the upper key block exists
    // row blocks of it that see key block j0 + r
    __device__ __forceinline__ int seen(uint32_t r) const {
        const int end = i0 + n_blk;
        if (r == 0) return (last0 < end ? last0 + 1 : end) - i0;
        return two ? end - (i0 > j0 ? i0 : j0 + 1) : 0;
    }
    // bit r: row block i sees key block j0 + r
    __device__ __forceinline__ uint32_t see(int i) const { return (i <= last0 ? 1u : 0u) | (two && i > j0 ? 2u : 0u); }
};
__device__ __forceinline__ PairUnit pair_unit(const PairParams& p, int t) {
    PairUnit u;
    u.kvh = t / p.NU;
    const int pb = t - u.kvh * p.NU;
    u.j0 = 2 * p.u_blk[pb];
    u.c = p.u_chunk[pb];
    const int64_t k1 = (int64_t)(u.j0 + 1) * kBlk;
    u.last0 = last_q_block(p.tok_end, p.T, (int64_t)u.j0 * kBlk);
    u.two = k1 < p.T;
    const int last = u.two ? last_q_block(p.tok_end, p.T, k1) : u.last0;
    const int lo = u.c * p.R > u.j0 ? u.c * p.R : u.j0;
    const int hi = u.c * p.R + p.R - 1 < last ? u.c * p.R + p.R - 1 : last;
    u.i0 = lo;
    u.n_blk = hi - lo + 1;
    return u;
}

// Bulk copy from this CTA's shared memory into another's (cluster addresses), counted on a barrier there.
__device__ __forceinline__ void bulk_copy_to_cta(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "r"(smem_u32(src)), "r"(bytes), "r"(bar)
                 : "memory");
}
// An arrival that hands over what the whole warp has done (tensor memory, or reads of it).
__device__ __forceinline__ void warp_arrive(uint64_t* bar, int lane) {
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
}
__device__ __forceinline__ void warp_arrive_cluster(uint32_t bar, int lane) {
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive_cluster(bar);
}
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
k_attn_bwd_pair(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_do,
                const __grid_constant__ CUtensorMap tm_q64, const __grid_constant__ CUtensorMap tm_do64,
                const __grid_constant__ CUtensorMap tm_dqacc, const __grid_constant__ CUtensorMap tm_dkacc,
                const __grid_constant__ CUtensorMap tm_dvacc, const PairParams p) {
    using L = PairSmem;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::kBarOff);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::kMiscOff);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::kMiscOff + 4);
    volatile uint32_t* peer_gave_up = reinterpret_cast<volatile uint32_t*>(smem + L::kMiscOff + 12);
    volatile uint32_t* issued = peer_gave_up + 1;   // [2][kPairLoads] leader: loads of each kind that either CTA has issued
    volatile uint32_t* sent = issued + 2 * kPairLoads;   // [4] copies of dS that each dS warp of the other CTA has issued
    volatile uint32_t* taken = sent + 4;            // iterations whose copies have arrived; [1] whether the next was expected
    volatile uint32_t* progress = taken + 2;        // iterations begun and units finished by the first exp warp
    uint32_t* finished = const_cast<uint32_t*>(progress) + 1;   // warps whose role is over

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int worker = (int)(blockIdx.x >> 1);
    const int cta = worker + (int)(rank * (gridDim.x >> 1));   // where the CTA reports

    if ((smem_u32(smem) & 1023u) != 0) {   // (the same in both CTAs)
        if (threadIdx.x == 0) p.outcome[cta] = LIBRA_ERR_CUDA;
        return;
    }
    if (threadIdx.x == 0) {
#pragma unroll 1
        for (int b = 0; b < L::kNumBars; ++b) {
            int n = 1;
            if (b == L::kXFree1 || b == L::kPReady || b == L::kDkvEmpty) n = 16;
            if (b == L::kXFree2 || b == L::kDsTmem || b == L::kPHalf || b == L::kPLocal) n = 8;
            if (b == L::kPRead || b == L::kZFree) n = 4;
            if (b == L::kDsSmem) n = 2;
            mbar_init(&bars[b], n);
        }
        abort_flag[0] = 0;
        *peer_gave_up = 0;
        *progress = 0;
        *finished = 0;
        for (int k = 0; k < 2 * kPairLoads; ++k) issued[k] = 0;
        fence_mbar_init();
    }
    if (warp == kPrTmaWarp && lane == 0) {
        prefetch_tmap(&tm_q);
        prefetch_tmap(&tm_k);
        prefetch_tmap(&tm_v);
        prefetch_tmap(&tm_do);
        prefetch_tmap(&tm_q64);
        prefetch_tmap(&tm_do64);
        prefetch_tmap(&tm_dqacc);
        prefetch_tmap(&tm_dkacc);
        prefetch_tmap(&tm_dvacc);
    }
    grid_dep_wait();
    if (const int ps = *p.plan_status; ps != 0) {  // malformed cu_seqlens: report and leave
        if (threadIdx.x == 0) { p.outcome[cta] = ps; p.busy[2 * cta] = p.busy[2 * cta + 1] = 0; }
        return;
    }
    if (threadIdx.x == 0) p.busy[2 * cta] = globaltimer_ns();
    if (warp == kPrMmaWarp) {
        tmem_alloc_pair(tmem_slot, 512);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();      // both CTAs' barriers are initialised and their TMEM is allocated
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    constexpr uint32_t kColX = 0, kColP = 128, kColDS = 192, kColDQ = 192, kColDK = 256, kColDV = 384;

    const int unit_begin = p.cta_offsets[worker];
    const int unit_end = p.cta_offsets[worker + 1];
    const int G = p.hq / p.hkv;

    if (warp == kPrWatchWarp) {
        // ------- the clock of all waits: no iteration has begun and no unit's products have ended for the budget of one -------
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kPrRegsOther));
        if (elect_one()) watch_progress(progress, finished, kPairThreads / 32 - 1, p.wait_limit_ns, abort_flag);
        __syncwarp();
    } else if (warp == kPrInWarp) {
        // ---------------- the other CTA's half of dS: its copies count on a barrier here, the leader is told ----------------
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kPrRegsOther));
        if (elect_one()) {
            const uint32_t ds_smem = map_to_rank(&bars[L::kDsSmem], 0);
            uint32_t n = 0, armed = 0;
            bool ok = true;
            for (int idx = unit_begin; idx < unit_end && ok; ++idx) {
                const PairUnit u = pair_unit(p, p.cta_tiles[idx]);
                const int n_it = G * u.n_blk;
                for (int it = 0; it < n_it; ++it) {
                    mbar_arrive_expect_tx(&bars[L::kDsIn], L::kHalf);
                    armed = 1;
                    ok = watched_wait(&bars[L::kDsIn], n & 1, abort_flag);
                    if (!ok) break;
                    armed = 0;
                    ++n;
                    mbar_arrive_cluster(ds_smem);
                }
            }
            taken[0] = n;
            taken[1] = armed;
        }
        __syncwarp();
    } else if (warp == kPrTmaWarp) {
        // ---------------- TMA producer (each CTA loads its own parts; the leader's barriers count both) ----------------
        // Loads go out in the order in which the MMAs free their buffers: Qr(n) [S(n-1) has run], dOc(n-1) [dV(n-2)],
        // dOr(n) [dP(n-1)], Qc(n-1) [dK(n-2)].  The statistics have two buffers: lse2(n) may replace lse2(n-2) once dV(n-2) has
        // run, which P^T(n-2) of all exp warps preceded, and dvec(n) dvec(n-2) once dK(n-2) has, which followed dS^T(n-2).
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kPrRegsOther));
        if (elect_one()) {
            uint32_t n_lse = 0, n_dvec = 0, phase = 0;   // phase: bit per kind of load
            bool ok = true;
            int idx = p.inject_stall && rank == 1 ? unit_end : unit_begin;
            int prev_h = 0, prev_qb = -1;   // iteration n - 1
            uint32_t n = 0;
            PairUnit u = {};
            int h = 0, h_end = 0, i = 0;
            auto stat = [&](const float* src, int off, int bar, int qb) {
                mbar_arrive_expect_tx(&bars[bar + (n & 1)], 512);
                bulk_load_1d(smem + off + (n & 1) * 512, src + (size_t)h * p.Tpad + qb, 512, &bars[bar + (n & 1)]);
            };
            while (ok) {
                const bool unit = h == h_end, more = !unit || idx < unit_end;   // the last round only has loads of iteration n - 1
                if (unit && more) {
                    u = pair_unit(p, p.cta_tiles[idx++]);
                    h = u.kvh * G;
                    h_end = h + G;
                    i = 0;
                }
                const int qb = (u.i0 + i) * kBlk;
#pragma unroll 1
                for (int k = 0; k < kPairLoads; ++k) {
                    const bool rows = k == kLoadQr || k == kLoadDor, prev = k == kLoadDoc || k == kLoadQc;
                    if (prev ? prev_qb >= 0 : more && (rows || unit)) {   // (K and V behind the last loads of the unit before)
                        ok = watched_wait(&bars[L::kSFull + k], ((phase >> k) & 1) ^ 1, abort_flag);
                        if (!ok) break;
                        phase ^= 1u << k;
                        issued[rank * kPairLoads + k] = issued[rank * kPairLoads + k] + 1;
                        if (rank == 0) mbar_arrive_expect_tx(&bars[L::kQrFull + k], 2 * pair_load_bytes(k));
                        const uint32_t full = map_to_rank(&bars[L::kQrFull + k], 0);
                        if (k == kLoadKv) {
                            const int k0 = u.j0 * kBlk, k_own = k0 + (int)rank * kBlk;
#pragma unroll 1
                            for (int half = 0; half < 2; ++half) {
                                tma_load_3d_pair(smem + L::kKOff + half * L::kHalf, &tm_k, full, half * 64, u.kvh, k_own);
                                tma_load_3d_pair(smem + L::kVOff + half * L::kHalf, &tm_v, full, half * 64, u.kvh, k_own);
                                tma_load_3d_pair(smem + L::kKcOff + half * L::kHalf, &tm_k, full, 64 * (int)rank, u.kvh, k0 + half * kBlk);
                            }
                        } else {
                            const CUtensorMap* tm = k == kLoadQr ? &tm_q64 : (k == kLoadDor ? &tm_do64 : (k == kLoadQc ? &tm_q : &tm_do));
                            uint8_t* dst = smem + (k == kLoadQr ? L::kQrOff : (k == kLoadDor ? L::kDorOff : (k == kLoadQc ? L::kQcOff : L::kDocOff)));
                            tma_load_3d_pair(dst, tm, full, rows ? 0 : 64 * (int)rank, rows ? h : prev_h, rows ? qb + 64 * (int)rank : prev_qb);
                            if (rows) tma_load_3d_pair(dst + L::kRowHalf, tm, full, 64, h, qb + 64 * (int)rank);
                        }
                    }
                    if (more && k == kLoadDoc) { stat(p.lse2, L::kLseOff, L::kLseFull, qb); ++n_lse; }
                    if (more && k == kLoadQc) { stat(p.dvec, L::kDvecOff, L::kDvecFull, qb); ++n_dvec; }
                }
                if (!more) break;
                prev_h = h;
                prev_qb = qb;
                ++n;
                if (++i == u.n_blk) { i = 0; ++h; }
            }
            if (rank == 1)
                for (int k = 0; k < kPairLoads; ++k)
                    st_cluster(map_to_rank(const_cast<const uint32_t*>(issued) + kPairLoads + k, 0), issued[kPairLoads + k]);
            if (!ok || abort_flag[0]) {   // give-up path: this CTA's own copies (the others: see the teardown)
                for (uint32_t b = 1; b <= 2 && b <= n_lse; ++b)
                    mbar_wait_drain(&bars[L::kLseFull + ((n_lse - b) & 1)], ((n_lse - b) >> 1) & 1, kDrainNs);
                for (uint32_t b = 1; b <= 2 && b <= n_dvec; ++b)
                    mbar_wait_drain(&bars[L::kDvecFull + ((n_dvec - b) & 1)], ((n_dvec - b) >> 1) & 1, kDrainNs);
            }
        }
        __syncwarp();
    } else if (warp == kPrMmaWarp) {
        // ---------------- MMA issuer (the leader's, for both) ----------------
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kPrRegsOther));
        if (rank == 0 && elect_one()) {
            constexpr uint32_t idesc_x = make_idesc(256, 128, 0, 0);     // S^T, dP^T: both operands K-major
            constexpr uint32_t idesc_acc = make_idesc(256, 128, 0, 1);   // dV, dK: A from TMEM, B MN-major
            constexpr uint32_t idesc_dq = make_idesc(128, 128, 1, 1);    // dQ: A = dS^T read along queries, B = K, both MN-major
            const uint32_t sb = smem_u32(smem);
            const uint64_t kdesc0 = make_sdesc(sb, 16, 1024);            // K-major view of a tile at offset 0
            const uint64_t mdesc0 = make_sdesc(sb, L::kHalf, 1024);      // MN-major view (64 columns: one atom)
            uint32_t ucnt = 0, n = 0;
            bool ok = true;
            auto wait = [&](int bar, uint32_t parity) { ok = watched_wait(&bars[bar], parity & 1, abort_flag); return ok; };
            auto issue_x = [&](uint32_t a_off, uint32_t b_off) {
                const uint64_t da = sdesc_advance(kdesc0, a_off), db = sdesc_advance(kdesc0, b_off);
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)
                    mma_ss_pair(tmem_base + kColX, sdesc_advance(da, (kk / 4) * L::kHalf + (kk % 4) * 32),
                                sdesc_advance(db, (kk / 4) * L::kRowHalf + (kk % 4) * 32), idesc_x, kk > 0);
            };
            // acc[256 keys] (+)= A (TMEM) * B over the 128 queries, of the CTAs in `see`; those in `begun` add
            auto issue_acc = [&](uint32_t d_col, uint32_t a_col, uint32_t b_off, uint32_t see, uint32_t begun) {
                const uint64_t db = sdesc_advance(mdesc0, b_off);
                const uint32_t adds = see & begun;
                if (see == 3 && adds == 3) {
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)
                        mma_ts_pair(tmem_base + d_col, tmem_base + a_col + kk * 8, sdesc_advance(db, kk * 2048), idesc_acc, 1);
                    return;
                }
                int kk = 0;
                uint32_t add = adds;
                if (see == 3 && adds != 0) {   // a CTA's first product overwrites; these two did not begin with the same row block
                    mma_ts_pair_of(tmem_base + d_col, tmem_base + a_col, db, idesc_acc, 1, adds);
                    mma_ts_pair_of(tmem_base + d_col, tmem_base + a_col, db, idesc_acc, 0, 3 - adds);
                    kk = 1;
                    add = 1;
                }
#pragma unroll 1
                for (; kk < 8; ++kk) {
                    mma_ts_pair_of(tmem_base + d_col, tmem_base + a_col + kk * 8, sdesc_advance(db, kk * 2048), idesc_acc, add, see);
                    add = 1;
                }
            };
            for (int idx = unit_begin; idx < unit_end && ok; ++idx) {
                const PairUnit u = pair_unit(p, p.cta_tiles[idx]);
                const int n_it = G * u.n_blk;
                uint32_t begun = 0;              // bit per CTA: its rows of dV and dK have been written
                if (!wait(L::kKvFull, ucnt)) break;
                for (int it = -1, i = 0; it < n_it && ok; ++it) {   // n: iteration `it` of the unit, or the one ahead of it
                    const bool more = it + 1 < n_it;
                    const uint32_t nx = n + (it >= 0 ? 1 : 0), see = u.see(u.i0 + i);
                    if (more) {   // S(it+1), once dP(it) has been read out of X
                        if (!wait(L::kQrFull, nx) || (nx > 0 && !wait(L::kXFree2, nx - 1))) break;
                        tc_fence_after();
                        issue_x(L::kKOff, L::kQrOff);
                        tc_commit_pair(&bars[L::kSFull]);
                    }
                    if (it >= 0) {   // dV(it) += P^T dO
                        if (!wait(L::kDocFull, n) || !wait(L::kPReady, n)) break;
                        if (it == 0 && ucnt > 0 && !wait(L::kDkvEmpty, ucnt - 1)) break;
                        tc_fence_after();
                        issue_acc(kColDV, kColP, L::kDocOff, see, begun);
                        tc_commit_pair(&bars[L::kDocEmpty]);
                    }
                    if (more) {   // dP(it+1) over S(it+1), once the exp groups hold that
                        if (!wait(L::kDorFull, nx) || !wait(L::kXFree1, nx)) break;
                        tc_fence_after();
                        issue_x(L::kVOff, L::kDorOff);
                        tc_commit_pair(&bars[L::kDpFull]);
                    }
                    if (it < 0) continue;
                    // dK(it) += dS^T Q
                    if (!wait(L::kQcFull, n) || !wait(L::kDsTmem, n)) break;
                    tc_fence_after();
                    issue_acc(kColDK, kColDS, L::kQcOff, see, begun);
                    tc_commit_pair(&bars[L::kQcEmpty]);
                    begun |= see;
                    // dQ(it) = dS K over dS^T's columns, which dK(it) has read by then; the keys of the CTAs that see the rows
                    if (!wait(L::kDsSmem, n)) break;
                    tc_fence_after();
                    {
                        const uint64_t da = sdesc_advance(mdesc0, L::kDsOff), db = sdesc_advance(mdesc0, L::kKcOff);
                        if (see == 3) {
#pragma unroll
                            for (int kk = 0; kk < 16; ++kk)   // 16 keys per step
                                mma_ss_pair(tmem_base + kColDQ, sdesc_advance(da, kk * 2048), sdesc_advance(db, kk * 2048), idesc_dq, kk > 0);
                        } else {
                            const int k0 = see & 1 ? 0 : 8;
#pragma unroll 1
                            for (int kk = k0; kk < k0 + 8; ++kk)
                                mma_ss_pair(tmem_base + kColDQ, sdesc_advance(da, kk * 2048), sdesc_advance(db, kk * 2048), idesc_dq, kk > k0);
                        }
                    }
                    tc_commit_pair(&bars[L::kDqFull]);
                    if (!more) { tc_commit_pair(&bars[L::kKvEmpty]); tc_commit_pair(&bars[L::kDkvFull]); }   // the unit's last MMAs
                    if (++i == u.n_blk) i = 0;
                    ++n;
                }
                ++ucnt;
            }
            if (!ok || abort_flag[0]) {
                tc_commit_pair(&bars[L::kDrain]);
                mbar_wait_drain(&bars[L::kDrain], 0, kDrainNs);
            }
        }
        __syncwarp();
    } else if (warp >= kPrDqWarp) {
        // ---------------- dQ group ----------------
        // Warp w of it: query rows 64 rank + 32 (w & 1) .. and head-dim columns 64 (w >> 1) .. 64 (w >> 1) + 63.
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kPrRegsDq));
        const int w = warp & 3;
        const uint32_t t_dq = tmem_base + ((uint32_t)(w * 32) << 16) + kColDQ;
        uint8_t* stage = smem + L::kStageOff + w * 4096;
        uint32_t n = 0;
        bool ok = true;
        for (int idx = unit_begin; idx < unit_end && ok; ++idx) {
            const PairUnit u = pair_unit(p, p.cta_tiles[idx]);
            const int n_it = G * u.n_blk;
            for (int it = 0, i = 0, h = u.kvh * G; it < n_it; ++it, ++n) {
                const int row = (u.i0 + i) * kBlk + 64 * (int)rank + 32 * (w & 1), head = h;
                if (++i == u.n_blk) { i = 0; ++h; }
                ok = watched_warp_wait(&bars[L::kDqFull], n & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                uint32_t v[64];
                tmem_ld32(t_dq, v);
                tmem_ld32(t_dq + 32, v + 32);
                tmem_ld_wait();
                warp_arrive(&bars[L::kZFree], lane);
                fused_stage_dq(&tm_dqacc, stage, v, lane, 64 * (w >> 1), head, row);
                fused_stage_dq(&tm_dqacc, stage, v + 32, lane, 64 * (w >> 1) + 32, head, row);
            }
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    } else if (warp >= 8) {
        // ---------------- dS group ----------------
        // Thread r owns key row r: it turns dP^T and P^T (read back as bf16) into dS^T, which goes to TMEM (the A
        // operand of dK) and to the shared memory of both CTAs (the A operand of dQ: queries 0 .. 63 to the leader's).
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kPrRegsDs));
        const int r = (warp & 3) * 32 + lane;
        const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t t_x = tmem_base + lane_addr + kColX;
        const uint32_t t_p = tmem_base + lane_addr + kColP;
        const uint32_t t_ds = tmem_base + lane_addr + kColDS;
        uint8_t* ds_own = smem + L::kDsOff + rank * L::kHalf + r * 128;
        uint8_t* ds_out = smem + L::kOutOff + r * 128;
        uint8_t *row0 = rank == 0 ? ds_own : ds_out, *row1 = rank == 0 ? ds_out : ds_own;   // queries 0 .. 63, 64 .. 127
        const uint32_t out_dst = map_to_rank(smem + L::kDsOff + rank * L::kHalf + (warp & 3) * 4096, rank ^ 1),
                       ds_in = map_to_rank(&bars[L::kDsIn], rank ^ 1);
        const uint32_t xfree2 = map_to_rank(&bars[L::kXFree2], 0), ds_tmem = map_to_rank(&bars[L::kDsTmem], 0);
        uint32_t ucnt = 0, n = 0, n_sent = 0;
        bool ok = true;
        for (int idx = unit_begin; idx < unit_end && ok; ++idx) {
            const PairUnit u = pair_unit(p, p.cta_tiles[idx]);
            const int n_it = G * u.n_blk;
            for (int it = 0; it < n_it && ok; ++it, ++n) {
                const float* dvec = reinterpret_cast<const float*>(smem + L::kDvecOff + (n & 1) * 512);
                ok = watched_warp_wait(&bars[L::kDvecFull + (n & 1)], (n >> 1) & 1, abort_flag) && watched_warp_wait(&bars[L::kDpFull], n & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                uint32_t xs[64];   // (dP^T - D) as packed bf16 pairs
                {
                    const uint64_t neg1 = f2_pack(-1.f, -1.f);
#pragma unroll
                    for (int part = 0; part < 4; ++part) {   // 32 columns at a time keeps the live registers down
                        uint32_t dpv[32];
                        tmem_ld32(t_x + part * 32, dpv);
                        tmem_ld_wait();
                        if (part == 3) warp_arrive_cluster(xfree2, lane);   // dP^T(it) is in registers: S^T(it+1) may take the columns
#pragma unroll
                        for (int j = 0; j < 32; j += 4) {
                            const ulonglong2 d4 = *reinterpret_cast<const ulonglong2*>(dvec + part * 32 + j);
                            float a0, a1, b0, b1;
                            f2_unpack(f2_fma(d4.x, neg1, f2_pack(__uint_as_float(dpv[j]), __uint_as_float(dpv[j + 1]))), a0, a1);
                            f2_unpack(f2_fma(d4.y, neg1, f2_pack(__uint_as_float(dpv[j + 2]), __uint_as_float(dpv[j + 3]))), b0, b1);
                            xs[part * 16 + (j >> 1)] = pack_bf16x2(a0, a1);
                            xs[part * 16 + (j >> 1) + 1] = pack_bf16x2(b0, b1);
                        }
                    }
                }
                // dQ(it-1) has been read out of dS^T's columns (so its MMA, which read dS of both CTAs, has run); the last unit's
                // dK and dV have left both CTAs through the dS tiles
                if (n > 0) ok = watched_warp_wait(&bars[L::kZFree], (n - 1) & 1, abort_flag);
                if (ok && it == 0 && ucnt > 0) ok = watched_warp_wait(&bars[L::kDkvEmpty], (ucnt - 1) & 1, abort_flag);
                if (!ok) break;
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    ok = watched_warp_wait(&bars[half == 0 ? L::kPHalf : L::kPLocal], n & 1, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    uint32_t pa[16], pb[16];   // queries 32 half .. and 64 + 32 half ..
                    tmem_ld16(t_p + half * 16, pa);
                    tmem_ld16(t_p + 32 + half * 16, pb);
                    tmem_ld_wait();
                    if (half == 1) warp_arrive(&bars[L::kPRead], lane);
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        pa[j] = mul_bf16x2(pa[j], xs[half * 16 + j]);
                        pb[j] = mul_bf16x2(pb[j], xs[32 + half * 16 + j]);
                    }
                    tmem_st16(t_ds + half * 16, pa);
                    tmem_st16(t_ds + 32 + half * 16, pb);
                    // row 128 rank + r of the dS tiles, 16-byte chunks of 8 queries, 128-byte swizzle
#pragma unroll
                    for (int ch = 0; ch < 4; ++ch) {
                        const int at = ((half * 4 + ch) ^ (r & 7)) << 4;
                        *reinterpret_cast<uint4*>(row0 + at) = make_uint4(pa[4 * ch], pa[4 * ch + 1], pa[4 * ch + 2], pa[4 * ch + 3]);
                        *reinterpret_cast<uint4*>(row1 + at) = make_uint4(pb[4 * ch], pb[4 * ch + 1], pb[4 * ch + 2], pb[4 * ch + 3]);
                    }
                }
                if (!ok) break;
                fence_proxy_async_smem();     // the copy and the MMA read the tiles through the async proxy
                tmem_st_wait();
                __syncwarp();
                if (lane == 0) bulk_copy_to_cta(out_dst, smem + L::kOutOff + (warp & 3) * 4096, 4096, ds_in);
                warp_arrive_cluster(ds_tmem, lane);
                ++n_sent;
            }
            ++ucnt;
        }
        if (lane == 0) st_cluster(map_to_rank(const_cast<const uint32_t*>(sent) + (warp & 3), rank ^ 1), n_sent);
    } else {
        // ---------------- exp groups ----------------
        // Thread r of group grp owns key row r and the query columns [64 grp, 64 grp + 64) of S^T.
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kPrRegsExp));
        const int grp = warp >> 2;
        const int r = (warp & 3) * 32 + lane;
        const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t t_x = tmem_base + lane_addr + kColX;
        const uint32_t t_p = tmem_base + lane_addr + kColP;
        const int c0 = 64 * grp;
        const uint64_t neg_scale2 = f2_pack(-p.scale_log2, -p.scale_log2);
        const uint32_t xfree1 = map_to_rank(&bars[L::kXFree1], 0), pready = map_to_rank(&bars[L::kPReady], 0);
        uint8_t* stage = smem + L::kDsOff + warp * 4096;      // between units: this warp's staging tile for dK and dV
        uint32_t ucnt = 0, n = 0;
        bool ok = true;
        for (int idx = unit_begin; idx < unit_end && ok; ++idx) {
            const uint64_t tile_t0 = threadIdx.x == 0 ? globaltimer_ns() : 0;
            const PairUnit u = pair_unit(p, p.cta_tiles[idx]);
            const int n_it = G * u.n_blk;
            const int64_t k0 = (int64_t)(u.j0 + rank) * kBlk, key = k0 + r;
            const bool key_ok = key < p.T;
            const int kend = key_ok ? p.tok_end[key] : 0;
            const int min_kend = k0 < p.T ? p.tok_end[k0] : 0;
            const bool partial = k0 + kBlk > p.T;
            for (int it = 0, i = 0; it < n_it && ok; ++it, ++n) {
                const int qb = (u.i0 + i) * kBlk;
                if (++i == u.n_blk) i = 0;
                if (threadIdx.x == 0) *progress = n + ucnt + 1;
                const float* lse2 = reinterpret_cast<const float*>(smem + L::kLseOff + (n & 1) * 512) + c0;
                const bool need_mask = (qb <= k0) || (qb + kBlk - 1 >= min_kend) || partial;
                const int j_lo = (int)(key - qb) - c0;
                const int j_hi = kend - 1 - qb - c0;
                ok = watched_warp_wait(&bars[L::kLseFull + (n & 1)], (n >> 1) & 1, abort_flag) && watched_warp_wait(&bars[L::kSFull], n & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                uint32_t sv[32], sv2[32];   // S^T of the 32 queries at hand and of the other 32
                tmem_ld32(t_x + c0, sv);
                tmem_ld32(t_x + c0 + 32, sv2);
                tmem_ld_wait();
                warp_arrive_cluster(xfree1, lane);
                // (one copy of the code for both halves)
#pragma unroll 1
                for (int half = 0; half < 2; ++half) {
                    const float* l2 = lse2 + 32 * half;
                    float pf[32];
#pragma unroll
                    for (int j = 0; j < 32; j += 4) {
                        const ulonglong2 l4 = *reinterpret_cast<const ulonglong2*>(l2 + j);
                        float x0, x1, x2, x3;
                        f2_unpack(f2_fma(f2_pack(__uint_as_float(sv[j]), __uint_as_float(sv[j + 1])), neg_scale2, l4.x), x0, x1);
                        f2_unpack(f2_fma(f2_pack(__uint_as_float(sv[j + 2]), __uint_as_float(sv[j + 3])), neg_scale2, l4.y), x2, x3);
                        pf[j] = ex2_approx(-x0);
                        pf[j + 1] = ex2_approx(-x1);
                        pf[j + 2] = ex2_approx(-x2);
                        pf[j + 3] = ex2_approx(-x3);
                    }
                    if (need_mask) {   // a uniform branch: the exponentials above stay one straight run
                        const uint32_t vis = range_bits(j_lo - half * 32, j_hi - half * 32);
#pragma unroll
                        for (int j = 0; j < 32; ++j) pf[j] = (vis >> j) & 1u ? pf[j] : 0.f;
                    }
                    uint32_t pk[16];
#pragma unroll
                    for (int j = 0; j < 32; j += 2) pk[j >> 1] = pack_bf16x2(pf[j], pf[j + 1]);
#pragma unroll
                    for (int j = 0; j < 32; ++j) sv[j] = sv2[j];
                    if (half == 0 && n > 0) {   // P^T(it-1) has been read by the dS group and consumed by dV(it-1)
                        ok = watched_warp_wait(&bars[L::kPRead], (n - 1) & 1, abort_flag) && watched_warp_wait(&bars[L::kDocEmpty], (n - 1) & 1, abort_flag);
                        if (!ok) break;
                        tc_fence_after();
                    }
                    tmem_st16(t_p + c0 / 2 + half * 16, pk);
                    tmem_st_wait();
                    warp_arrive(&bars[L::kPHalf + half], lane);
                    if (half == 1 && lane == 0) mbar_arrive_cluster(pready);
                }
            }
            if (!ok) break;
            ++ucnt;
            // ---- unit epilogue: dK and dV of the CTA's key block are added to the fp32 accumulators, through the dS tile (dQ has
            // read it) and bulk reduce-adds of 32 key rows x 32 head-dim columns ----
            ok = watched_warp_wait(&bars[L::kDkvFull], (ucnt - 1) & 1, abort_flag);
            if (!ok) break;
            if (threadIdx.x == 0) *progress = n + ucnt;
            tc_fence_after();
            // of a query chunk's row blocks this CTA's keys may have seen none
            const int seen = u.seen(rank);
            if (seen > 0) {
#pragma unroll 1
                for (int c = 0; c < 4; ++c) {
                    uint32_t v[32];
                    const int col = c0 + (c & 1) * 32;
                    tmem_ld32(tmem_base + lane_addr + (c < 2 ? kColDK : kColDV) + col, v);
                    tmem_ld_wait();
                    fused_stage_dq(c < 2 ? &tm_dkacc : &tm_dvacc, stage, v, lane, col, u.kvh, (int)k0 + (warp & 3) * 32);
                }
                if (lane == 0) tma_store_wait_read();
            }
            tc_fence_before();
            __syncwarp();
            if (lane < 2) mbar_arrive_cluster(map_to_rank(&bars[L::kDkvEmpty], (uint32_t)lane));
            if (threadIdx.x == 0 && seen > 0)   // of the time of both halves the part in which this one had work
                p.tile_ns[u.kvh * p.NU128 + p.base[u.c] + u.j0 + rank - p.first_j[u.c]] = (uint32_t)((globaltimer_ns() - tile_t0) * seen / u.n_blk);
        }
        // every bulk reduce this warp issued has completed before the CTA leaves
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }

    // ---------------- teardown ----------------
    if (warp != kPrWatchWarp && lane == 0) atomicAdd(finished, 1u);
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && abort_flag[0]) st_cluster(map_to_rank(const_cast<const uint32_t*>(peer_gave_up), rank ^ 1), 1u);
    cluster_sync();      // no role of either CTA runs any more
    if (abort_flag[0] | (int)*peer_gave_up) {   // give-up path: the copies already issued land before the CTAs leave
        if (threadIdx.x == 0) {   // copies of dS of the iteration that was not taken any more: those not sent count as arrived
            uint32_t here = 0;
            for (int w = 0; w < 4; ++w) here += sent[w] > taken[0] ? 1 : 0;
            if (here > 0) {
                if (!taken[1]) mbar_arrive_expect_tx(&bars[L::kDsIn], L::kHalf);
                if (here < 4) mbar_complete_tx(&bars[L::kDsIn], (4 - here) * 4096);
                mbar_wait_drain(&bars[L::kDsIn], taken[0] & 1, kDrainNs);
            }
        }
        if (threadIdx.x == 0 && rank == 0) {
#pragma unroll 1
            for (int k = 0; k < kPairLoads; ++k)
                open_loads(issued[k], issued[kPairLoads + k], 1, [](uint32_t) { return 0u; },
                           [&](uint32_t, uint32_t parity, bool mine, bool peers) {
                               // a part that never was issued is counted as arrived, one that the leader had not got to is expected now
                               uint64_t* bar = &bars[L::kQrFull + k];
                               if (!mine) mbar_arrive_expect_tx(bar, pair_load_bytes(k));
                               if (!peers) mbar_complete_tx(bar, pair_load_bytes(k));
                               mbar_wait_drain(bar, parity, kDrainNs);
                           });
        }
        cluster_sync();  // the leader's wait is for the other CTA's copies, too
    }
    tc_fence_after();
    if (warp == kPrMmaWarp) tmem_dealloc_pair(tmem_base, 512);
    if (threadIdx.x == 0) {
        p.outcome[cta] = abort_flag[0] ? LIBRA_ERR_TIMEOUT : LIBRA_OK;
        p.busy[2 * cta + 1] = globaltimer_ns();
    }
}

}  // namespace libra
