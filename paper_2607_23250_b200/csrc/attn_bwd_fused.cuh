// Fused backward kernel (included by attn_bwd.cu): dQ, dK and dV of a pair tile in one pass, five GEMMs per
// 128 x 128 cell instead of the seven of the two-kernel form (S and dP are computed once).  On single CTAs: for pools of
// short samples and pools cut into single row blocks; the others run on pairs of CTAs (attn_bwd_pair.cuh).
//
// A unit is a pair tile: 128 keys of one kv head against the query row blocks of one query chunk, for every
// query head of the kv head's group.  K and V stay in shared memory, dK and dV accumulate in TMEM over the
// unit; every iteration (one query head, one 128-row query block) also yields that block's dQ contribution,
// which leaves through shared memory as a bulk tensor reduce-add into an fp32 accumulator in global memory.
// dK and dV of the unit are added to fp32 accumulators as well (a key block meets several query chunks); a
// last kernel scales and rounds the three accumulators to bf16.  The plan runs the pair tiles in id order
// (head, query chunk, key block) on all CTAs in step, so the accumulator rows and the Q / dO tiles of a query
// chunk are shared by the CTAs while they are in L2.
//
// Keys sit in TMEM lanes:
//   S^T  = K Q^T   (SS) -> X     P^T  = exp2(S^T c - LSE)      -> bf16, own TMEM columns    dV += P^T dO  (A in TMEM)
//   dP^T = V dO^T  (SS) -> X     dS^T = P^T o (dP^T - D)       -> bf16, own TMEM columns    dK += dS^T Q  (A in TMEM)
//                                                               and the same tile in shared memory:
//   dQ   = dS K    (SS, A = the shared-memory dS^T read along its contiguous query axis) -> Y
// TMEM: X | Y | dK | dV = 128 + 128 + 128 + 128 columns.  X holds S^T, then dP^T (fp32), and is free again as soon
// as it has been READ, so S^T(it+1) and dP^T(it+1) run ahead.  Y holds P^T and dS^T (bf16, 64 columns each) and,
// once dV(it) and dK(it) have consumed them, receives dQ(it) (fp32, 128 columns: the MMAs run in issue order, so
// the overwrite needs no extra barrier); P^T(it+1), already computed in registers, is written as soon as dQ(it) has
// been read out.
// Roles (640 threads): two exp groups (64 query columns of S^T each), a dS group, a dQ group, the TMA thread, the MMA thread, the thread that watches the
// clock for all of them; a warp only hands its registers over.  The exp groups moved dQ between their exponentials before
// (512 threads); with that, the waits' code in one place and one copy of the exponentials' the kernel is 50 KB instead of
// 63: backward of 10 samples of 1000 tokens, 8 / 2 heads, 137.0 -> 133.4 us, of one of 1500 42.8 -> 40.2.
#pragma once

namespace libra {

constexpr int kFusedThreads = 640;
constexpr int kFuDqWarp = 12, kFuTmaWarp = 16, kFuMmaWarp = 17, kFuWatchWarp = 19;   // (warp 18 only donates registers)
// setmaxnreg budgets: 640 threads x 96 compiled registers = 256 x 112 + 128 x (128 + 48 + 80)
constexpr int kFuRegsExp = 112, kFuRegsDs = 128, kFuRegsDq = 48, kFuRegsOther = 80;

struct FusedSmem {
    static constexpr int kTile = 32768;        // 128 x 128 bf16
    static constexpr int kHalf = 16384;
    static constexpr int kQStages = 2;         // Q(it) lives from S(it) to dK(it), which runs behind dP(it+1)
    static constexpr int kKOff = 0;
    static constexpr int kVOff = kTile;
    static constexpr int kQOff = 2 * kTile;
    static constexpr int kDoOff = kQOff + kQStages * kTile;
    static constexpr int kDsOff = kDoOff + kTile;          // dS^T tile (bf16, the operand layout of K / V tiles)
    static constexpr int kStageOff = kDsOff + kTile;       // dQ staging: tiles of 32 rows x 32 floats, swizzled
    static constexpr int kLseOff = kStageOff + 2 * kHalf;  // per Q stage: lse2[128]
    static constexpr int kDvecOff = kLseOff + kQStages * 512;   // two buffers: dvec(it+1) lands while dvec(it) is read
    static constexpr int kBarOff = kDvecOff + 2 * 512;
    // kv_full, kv_empty, q_full[2], q_empty[2], do_full, do_empty, s_full, x_free1, dp_full, x_free2, dq_full,
    // y_free[2], p_ready, ds_ready, dkv_full, dkv_empty, drain
    static constexpr int kNumBars = 2 + 2 * kQStages + 15;
    static constexpr int kMiscOff = kBarOff + kNumBars * 8;
    static constexpr int kBytes = kMiscOff + 24;
    static_assert(kBytes <= kSmemMax, "exceeds the shared memory of an sm_100 CTA");
};

struct FusedParams {
    const float* lse2;  // [Hq, Tpad]  LSE * log2(e)
    const float* dvec;  // [Hq, Tpad]  D_i
    const int32_t* cta_offsets;
    const int32_t* cta_tiles;
    const int32_t* u_blk;     // key block of pair-block u
    const int32_t* u_chunk;   // query chunk of pair-block u
    const int32_t* tok_end;
    int64_t T, Tpad, NU;
    int hq, hkv, R;           // R = row blocks per query chunk
    float scale_log2;
    int* outcome;
    const int* plan_status;
    uint32_t wait_limit_ns;
    int inject_stall;
    uint64_t* busy;
    uint32_t* tile_ns;        // [tiles] time spent on each pair tile (first exp thread), ns
};

// The row blocks [i0, i1] a pair tile walks for every head of its group.
struct FusedUnit {
    int kvh, i0, n_blk;
    int64_t k0;
};
__device__ __forceinline__ FusedUnit fused_unit(const FusedParams& p, int t) {
    FusedUnit u;
    const int pb = (int)(t % p.NU);
    u.kvh = (int)(t / p.NU);
    const int j = p.u_blk[pb], c = p.u_chunk[pb];
    u.k0 = (int64_t)j * kBlk;
    const int last = last_q_block(p.tok_end, p.T, u.k0);
    const int lo = c * p.R > j ? c * p.R : j;
    const int hi = c * p.R + p.R - 1 < last ? c * p.R + p.R - 1 : last;
    u.i0 = lo;
    u.n_blk = hi - lo + 1;
    return u;
}

// Bulk tensor reduce-add of a shared-memory tile into global memory (fp32 elements, given by the tensor map).
__device__ __forceinline__ void tma_reduce_add_3d(const CUtensorMap* m, const void* smem_src, int c0, int c1, int c2) {
    asm volatile("cp.reduce.async.bulk.tensor.3d.global.shared::cta.add.tile.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(
                     reinterpret_cast<uint64_t>(m)),
                 "r"(smem_u32(smem_src)), "r"(c0), "r"(c1), "r"(c2)
                 : "memory");
}

// Waits of kernels that have one warp look at the clock for all of them (a wait of mbar_wait's kind has that code at every
// place).  They end when the phase has completed or the CTA has given up.
__device__ __forceinline__ bool watched_wait(uint64_t* bar, uint32_t parity, volatile int* ctl) {
    while (!mbar_try_wait(bar, parity))
        if (ctl[0]) return false;
    return true;
}
__device__ __forceinline__ bool watched_warp_wait(uint64_t* bar, uint32_t parity, volatile int* ctl) {
    return __all_sync(0xffffffffu, watched_wait(bar, parity, ctl));
}
// That warp's thread: the CTA gives up when *progress has not moved for the budget of a wait.  Ends with the other warps.
__device__ __forceinline__ void watch_progress(const volatile uint32_t* progress, const volatile uint32_t* finished, uint32_t warps,
                                               uint32_t limit_ns, volatile int* ctl) {
    uint64_t t0 = globaltimer_ns();
    uint32_t seen = 0;
    while (*finished < warps && !ctl[0]) {
        asm volatile("nanosleep.u32 100;");
        const uint64_t t = globaltimer_ns();
        const uint32_t now = *progress;
        if (now != seen) {
            seen = now;
            t0 = t;
        } else if (t - t0 > (uint64_t)limit_ns) {
            ctl[0] = 1;
        }
    }
}
// 32 columns of a row per thread, through the warp's staging tile (32 rows of 128 bytes, 128-byte swizzle) into the fp32
// accumulator: one bulk tensor reduce-add of 32 head-dim columns (from column col0), rows row0 .. row0 + 31 of head h.
// The reduce that last used the tile must have finished reading it: all but the last PENDING of this thread's have.
template <int PENDING = 0>
__device__ __forceinline__ void fused_stage_dq(const CUtensorMap* tm, uint8_t* stage, const uint32_t* dq, int lane,
                                               int col0, int h, int row0) {
    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(PENDING) : "memory");
    __syncwarp();
#pragma unroll
    for (int ch = 0; ch < 8; ++ch) {
        const int at = lane * 128 + ((ch ^ (lane & 7)) << 4);
        *reinterpret_cast<uint4*>(stage + at) = make_uint4(dq[4 * ch], dq[4 * ch + 1], dq[4 * ch + 2], dq[4 * ch + 3]);
    }
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) {
        tma_reduce_add_3d(tm, stage, col0, h, row0);
        tma_store_commit();
    }
}

__global__ void __launch_bounds__(kFusedThreads, 1)
k_attn_bwd_fused(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                 const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_do,
                 const __grid_constant__ CUtensorMap tm_dqacc, const __grid_constant__ CUtensorMap tm_dkacc,
                 const __grid_constant__ CUtensorMap tm_dvacc, const FusedParams p) {
    using L = FusedSmem;
    constexpr int D = 128, QS = L::kQStages;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::kBarOff);
    uint64_t* bar_kvfull = bars + 0;
    uint64_t* bar_kvempty = bars + 1;
    uint64_t* bar_qfull = bars + 2;             // [QS]
    uint64_t* bar_qempty = bar_qfull + QS;      // [QS] dK(it) has run: Q stage free, TMEM dS^T columns free
    uint64_t* b2 = bar_qempty + QS;
    uint64_t* bar_dofull = b2 + 0;
    uint64_t* bar_doempty = b2 + 1;    // dV(it) has run: the dO tile is free
    uint64_t* bar_sfull = b2 + 2;
    uint64_t* bar_xfree1 = b2 + 3;     // S^T(it) has been read out of X: dP^T(it) may overwrite it
    uint64_t* bar_dpfull = b2 + 4;
    uint64_t* bar_xfree2 = b2 + 5;     // dP^T(it) has been read out: S^T(it+1) may overwrite it
    uint64_t* bar_dqfull = b2 + 6;     // dQ(it) is in Y (so dV(it), dK(it) and dQ(it) have all run)
    uint64_t* bar_yfree = b2 + 7;      // [2] dQ(it) has been read out of Y's first 64 columns: P^T(it+1) may be written; of the
                                       // other 64: dS^T(it+1) may (and dQ(it) has run, so that the shared-memory dS^T is spent)
    uint64_t* bar_pready = b2 + 9;
    uint64_t* bar_dsready = b2 + 10;   // dS^T(it) is in TMEM and in shared memory
    uint64_t* bar_dkvfull = b2 + 11;
    uint64_t* bar_dkvempty = b2 + 12;
    uint64_t* bar_drain = b2 + 13;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::kMiscOff);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::kMiscOff + 4);
    volatile uint32_t* progress = reinterpret_cast<volatile uint32_t*>(smem + L::kMiscOff + 12);   // iterations begun and units finished by the first exp warp
    uint32_t* finished = reinterpret_cast<uint32_t*>(smem + L::kMiscOff + 16);                     // warps whose role is over

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int cta = blockIdx.x;

    if ((smem_u32(smem) & 1023u) != 0) {
        if (threadIdx.x == 0) p.outcome[cta] = LIBRA_ERR_CUDA;
        return;
    }
    if (threadIdx.x == 0) {
        mbar_init(bar_kvfull, 1);
        mbar_init(bar_kvempty, 1);
        for (int s = 0; s < QS; ++s) { mbar_init(&bar_qfull[s], 1); mbar_init(&bar_qempty[s], 1); }
        mbar_init(bar_dofull, 1);
        mbar_init(bar_doempty, 1);
        mbar_init(bar_sfull, 1);
        mbar_init(bar_xfree1, 256);
        mbar_init(bar_dpfull, 1);
        mbar_init(bar_xfree2, 128);
        mbar_init(bar_dqfull, 1);
        mbar_init(&bar_yfree[0], 128);
        mbar_init(&bar_yfree[1], 128);
        mbar_init(bar_pready, 256);
        mbar_init(bar_dsready, 128);
        mbar_init(bar_dkvfull, 1);
        mbar_init(bar_dkvempty, 256);
        mbar_init(bar_drain, 1);
        abort_flag[0] = 0;
        *progress = 0;
        *finished = 0;
        fence_mbar_init();
    }
    if (warp == kFuTmaWarp && lane == 0) {
        prefetch_tmap(&tm_q);
        prefetch_tmap(&tm_k);
        prefetch_tmap(&tm_v);
        prefetch_tmap(&tm_do);
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
    if (warp == kFuMmaWarp) {
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    constexpr uint32_t kColX = 0, kColY = 128, kColP = 128, kColDS = 192, kColDK = 256, kColDV = 384;

    const int unit_begin = p.cta_offsets[cta];
    const int unit_end = p.cta_offsets[cta + 1];
    const int G = p.hq / p.hkv;

    if (warp > kFuMmaWarp) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kFuRegsOther));
        if (warp == kFuWatchWarp) {
            if (elect_one()) watch_progress(progress, finished, kFusedThreads / 32 - 1, p.wait_limit_ns, abort_flag);
            __syncwarp();
        }
    } else if (warp == kFuTmaWarp) {
        // ---------------- TMA producer ----------------
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kFuRegsOther));
        if (elect_one()) {
            uint32_t ucnt = 0, it_all = 0, n_do = 0;
            bool ok = true;
            for (int idx = unit_begin; idx < unit_end && ok && !p.inject_stall; ++idx) {
                const FusedUnit u = fused_unit(p, p.cta_tiles[idx]);
                ok = watched_wait(bar_kvempty, (ucnt & 1) ^ 1, abort_flag);
                if (!ok) break;
                mbar_arrive_expect_tx(bar_kvfull, 2 * L::kTile);
                for (int half = 0; half < 2; ++half) {
                    tma_load_3d(smem + L::kKOff + half * L::kHalf, &tm_k, bar_kvfull, half * 64, u.kvh, (int)u.k0);
                    tma_load_3d(smem + L::kVOff + half * L::kHalf, &tm_v, bar_kvfull, half * 64, u.kvh, (int)u.k0);
                }
                ++ucnt;
                const int n_it = G * u.n_blk;
                for (int it = 0, i = 0, h = u.kvh * G; it < n_it && ok; ++it, ++it_all) {
                    const int qb = (u.i0 + i) * kBlk;
                    const uint32_t qs = it_all % QS;
                    ok = watched_wait(&bar_qempty[qs], ((it_all / QS) & 1) ^ 1, abort_flag);
                    if (!ok) break;
                    mbar_arrive_expect_tx(&bar_qfull[qs], L::kTile + 512);
                    for (int half = 0; half < 2; ++half)
                        tma_load_3d(smem + L::kQOff + qs * L::kTile + half * L::kHalf, &tm_q, &bar_qfull[qs], half * 64, h, qb);
                    bulk_load_1d(smem + L::kLseOff + qs * 512, p.lse2 + (size_t)h * p.Tpad + qb, 512, &bar_qfull[qs]);
                    ok = watched_wait(bar_doempty, (it_all & 1) ^ 1, abort_flag);
                    if (!ok) { mbar_wait_drain(&bar_qfull[qs], (it_all / QS) & 1, kDrainNs); break; }
                    mbar_arrive_expect_tx(bar_dofull, L::kTile + 512);
                    ++n_do;
                    for (int half = 0; half < 2; ++half)
                        tma_load_3d(smem + L::kDoOff + half * L::kHalf, &tm_do, bar_dofull, half * 64, h, qb);
                    bulk_load_1d(smem + L::kDvecOff + (it_all & 1) * 512, p.dvec + (size_t)h * p.Tpad + qb, 512, bar_dofull);
                    if (++i == u.n_blk) { i = 0; ++h; }
                }
            }
            if (!ok || abort_flag[0]) {   // give-up path: the copies already issued land before shared memory is released
                if (ucnt > 0) mbar_wait_drain(bar_kvfull, (ucnt - 1) & 1, kDrainNs);
                for (uint32_t b = 1; b <= (uint32_t)QS && b <= it_all; ++b)
                    mbar_wait_drain(&bar_qfull[(it_all - b) % QS], ((it_all - b) / QS) & 1, kDrainNs);
                if (n_do > 0) mbar_wait_drain(bar_dofull, (n_do - 1) & 1, kDrainNs);
            }
        }
        __syncwarp();
    } else if (warp == kFuMmaWarp) {
        // ---------------- MMA issuer ----------------
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kFuRegsOther));
        if (elect_one()) {
            constexpr uint32_t idesc_s = make_idesc(128, 128, 0, 0);   // S^T, dP^T: both operands K-major
            constexpr uint32_t idesc_acc = make_idesc(128, D, 0, 1);   // dV, dK: A from TMEM, B MN-major
            constexpr uint32_t idesc_dq = make_idesc(128, D, 1, 1);    // dQ: A = dS^T read along queries, B = K, both MN-major
            const uint32_t sb = smem_u32(smem);
            uint32_t ucnt = 0, it_all = 0;
            bool ok = true;
            const uint64_t kdesc0 = make_sdesc(sb, 16, 1024);          // K-major view of a tile at offset 0
            const uint64_t mdesc0 = make_sdesc(sb, L::kHalf, 1024);    // MN-major view
            auto issue_kmajor = [&](uint32_t a_off, uint32_t b_off) {
                const uint64_t da = sdesc_advance(kdesc0, a_off), db = sdesc_advance(kdesc0, b_off);
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk) {
                    const uint32_t off = (kk / 4) * L::kHalf + (kk % 4) * 32;
                    mma_ss(tmem_base + kColX, sdesc_advance(da, off), sdesc_advance(db, off), idesc_s, kk > 0);
                }
            };
            auto issue_acc = [&](uint32_t d_col, uint32_t a_col, uint32_t b_off, bool accumulate) {
                const uint64_t db = sdesc_advance(mdesc0, b_off);
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)
                    mma_ts(tmem_base + d_col, tmem_base + a_col + kk * 8, sdesc_advance(db, kk * 2048), idesc_acc,
                           (accumulate || kk > 0) ? 1u : 0u);
            };
            for (int idx = unit_begin; idx < unit_end && ok; ++idx) {
                const FusedUnit u = fused_unit(p, p.cta_tiles[idx]);
                const int n_it = G * u.n_blk;
                ok = watched_wait(bar_kvfull, ucnt & 1, abort_flag);
                if (!ok) break;
                // S(0): X is free once dP of the previous unit's last iteration has been read
                ok = watched_wait(&bar_qfull[it_all % QS], (it_all / QS) & 1, abort_flag);
                if (ok && it_all > 0) ok = watched_wait(bar_xfree2, (it_all - 1) & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                issue_kmajor(L::kKOff, L::kQOff + (it_all % QS) * L::kTile);
                tc_commit(bar_sfull);
                for (int it = 0; it < n_it && ok; ++it, ++it_all) {
                    const uint32_t nx = it_all + 1;
                    const bool more = it + 1 < n_it;
                    // dP(it) over S(it), as soon as the exp groups hold S(it) in registers
                    ok = watched_wait(bar_dofull, it_all & 1, abort_flag);
                    if (ok) ok = watched_wait(bar_xfree1, it_all & 1, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    issue_kmajor(L::kVOff, L::kDoOff);
                    tc_commit(bar_dpfull);
                    // S(it+1) over dP(it), as soon as the dS group holds dP(it) in registers
                    if (more) {
                        ok = watched_wait(&bar_qfull[nx % QS], (nx / QS) & 1, abort_flag);
                        if (ok) ok = watched_wait(bar_xfree2, it_all & 1, abort_flag);
                        if (!ok) break;
                        tc_fence_after();
                        issue_kmajor(L::kKOff, L::kQOff + (nx % QS) * L::kTile);
                        tc_commit(bar_sfull);
                    }
                    // dV(it) += P^T dO
                    ok = watched_wait(bar_pready, it_all & 1, abort_flag);
                    if (ok && it == 0 && ucnt > 0) ok = watched_wait(bar_dkvempty, (ucnt - 1) & 1, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    issue_acc(kColDV, kColP, L::kDoOff, it > 0);
                    tc_commit(bar_doempty);
                    // dK(it) += dS^T Q from the TMEM copy of dS^T, then dQ(it) = dS K from the shared-memory copy,
                    // into Y over P^T and dS^T: dV(it) and dK(it) precede it in issue order
                    ok = watched_wait(bar_dsready, it_all & 1, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    issue_acc(kColDK, kColDS, L::kQOff + (it_all % QS) * L::kTile, it > 0);
                    tc_commit(&bar_qempty[it_all % QS]);
                    {
                        const uint64_t da = sdesc_advance(mdesc0, L::kDsOff), db = sdesc_advance(mdesc0, L::kKOff);
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk)   // 16 keys per step
                            mma_ss(tmem_base + kColY, sdesc_advance(da, kk * 2048), sdesc_advance(db, kk * 2048), idesc_dq, kk > 0);
                        tc_commit(bar_dqfull);
                        if (!more) { tc_commit(bar_kvempty); tc_commit(bar_dkvfull); }   // the unit's last MMAs
                    }
                }
                ++ucnt;
            }
            if (!ok || abort_flag[0]) {
                tc_commit(bar_drain);
                mbar_wait_drain(bar_drain, 0, kDrainNs);
            }
        }
        __syncwarp();
    } else if (warp >= 8 && warp < kFuDqWarp) {
        // ---------------- dS group ----------------
        // Thread r owns key row r: it turns dP^T and P^T (read back as bf16) into dS^T, which goes to TMEM (the A
        // operand of dK) and to shared memory (the A operand of dQ).
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kFuRegsDs));
        const int r = (warp & 3) * 32 + lane;
        const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t t_x = tmem_base + lane_addr + kColX;
        const uint32_t t_p = tmem_base + lane_addr + kColP;
        const uint32_t t_ds = tmem_base + lane_addr + kColDS;
        uint8_t* ds_row = smem + L::kDsOff + r * 128;
        uint32_t ucnt = 0, it_all = 0;
        bool ok = true;
        for (int idx = unit_begin; idx < unit_end && ok; ++idx) {
            const FusedUnit u = fused_unit(p, p.cta_tiles[idx]);
            const int n_it = G * u.n_blk;
            for (int it = 0; it < n_it && ok; ++it, ++it_all) {
                const float* dvec = reinterpret_cast<const float*>(smem + L::kDvecOff + (it_all & 1) * 512);
                ok = watched_warp_wait(bar_dofull, it_all & 1, abort_flag) && watched_warp_wait(bar_dpfull, it_all & 1, abort_flag);
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
                        if (part == 3) {
                            tc_fence_before();
                            mbar_arrive(bar_xfree2);   // dP^T(it) is in registers: S^T(it+1) may take the columns
                        }
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
                // dQ(it-1) has been read out of Y's dS^T columns, so both copies of dS^T(it-1) have been consumed; the last
                // unit's dK and dV have left through the shared-memory tile
                if (it_all > 0) ok = watched_warp_wait(&bar_yfree[1], (it_all - 1) & 1, abort_flag);
                if (ok && it == 0 && ucnt > 0) ok = watched_warp_wait(bar_dkvempty, (ucnt - 1) & 1, abort_flag);
                if (ok) ok = watched_warp_wait(bar_pready, it_all & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    uint32_t pa[16], pb[16];   // queries 32 half .. and 64 + 32 half ..
                    tmem_ld16(t_p + half * 16, pa);
                    tmem_ld16(t_p + 32 + half * 16, pb);
                    tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        pa[j] = mul_bf16x2(pa[j], xs[half * 16 + j]);
                        pb[j] = mul_bf16x2(pb[j], xs[32 + half * 16 + j]);
                    }
                    tmem_st16(t_ds + half * 16, pa);
                    tmem_st16(t_ds + 32 + half * 16, pb);
                    // the same values into the shared-memory tile: row r, 16-byte chunks of 8 queries, 128-byte swizzle;
                    // queries 0..63 in the first 16 KB half of the tile, 64..127 in the second
#pragma unroll
                    for (int ch = 0; ch < 4; ++ch) {
                        const int chunk_a = half * 4 + ch;            // queries 32 half + 8 ch ..
                        *reinterpret_cast<uint4*>(ds_row + ((chunk_a ^ (r & 7)) << 4)) =
                            make_uint4(pa[4 * ch], pa[4 * ch + 1], pa[4 * ch + 2], pa[4 * ch + 3]);
                        *reinterpret_cast<uint4*>(ds_row + L::kHalf + ((chunk_a ^ (r & 7)) << 4)) =
                            make_uint4(pb[4 * ch], pb[4 * ch + 1], pb[4 * ch + 2], pb[4 * ch + 3]);
                    }
                }
                tmem_st_wait();
                fence_proxy_async_smem();     // the MMA reads the shared-memory tile through the async proxy
                tc_fence_before();
                mbar_arrive(bar_dsready);
            }
            ++ucnt;
        }
    } else if (warp >= kFuDqWarp) {
        // ---------------- dQ group ----------------
        // Thread r owns query row r of dQ.  (The exp groups moved it between their exponentials before: with a group of its own
        // 3320 -> 3170 ns a cell and CTA on 8192 tokens, 8 / 2 heads.)
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kFuRegsDq));
        const uint32_t t_y = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + kColY;
        uint8_t* stage = smem + L::kStageOff + (warp & 3) * 8192;   // two tiles of 32 rows x 32 floats
        uint32_t it_all = 0;
        bool ok = true;
        for (int idx = unit_begin; idx < unit_end && ok; ++idx) {
            const FusedUnit u = fused_unit(p, p.cta_tiles[idx]);
            const int n_it = G * u.n_blk;
            for (int it = 0, i = 0, h = u.kvh * G; it < n_it; ++it, ++it_all) {
                const int row = (u.i0 + i) * kBlk + (warp & 3) * 32, head = h;
                if (++i == u.n_blk) { i = 0; ++h; }
                ok = watched_warp_wait(bar_dqfull, it_all & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
#pragma unroll 1
                for (int half = 0; half < 2; ++half) {
                    uint32_t v[32];
                    tmem_ld32(t_y + 64 * half, v);
                    tmem_ld_wait();
                    fused_stage_dq<1>(&tm_dqacc, stage, v, lane, 64 * half, head, row);
                    tmem_ld32(t_y + 64 * half + 32, v);
                    tmem_ld_wait();
                    tc_fence_before();
                    mbar_arrive(&bar_yfree[half]);
                    fused_stage_dq<1>(&tm_dqacc, stage + 4096, v, lane, 64 * half + 32, head, row);
                }
            }
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    } else {
        // ---------------- exp groups ----------------
        // Thread r of group grp owns key row r and the query columns [64 grp, 64 grp + 64) of S^T.
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kFuRegsExp));
        const int grp = warp >> 2;
        const int r = (warp & 3) * 32 + lane;
        const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t t_x = tmem_base + lane_addr + kColX;
        const uint32_t t_p = tmem_base + lane_addr + kColP;
        const int c0 = 64 * grp;
        const uint64_t neg_scale2 = f2_pack(-p.scale_log2, -p.scale_log2);
        uint8_t* stage = smem + L::kDsOff + warp * 4096;      // between units: this warp's staging tile for dK and dV
        uint32_t ucnt = 0, it_all = 0;
        bool ok = true;
        for (int idx = unit_begin; idx < unit_end && ok; ++idx) {
            const uint64_t tile_t0 = threadIdx.x == 0 ? globaltimer_ns() : 0;
            const FusedUnit u = fused_unit(p, p.cta_tiles[idx]);
            const int n_it = G * u.n_blk;
            const int64_t key = u.k0 + r;
            const bool key_ok = key < p.T;
            const int kend = key_ok ? p.tok_end[key] : 0;
            const int min_kend = p.tok_end[u.k0];
            const bool partial = u.k0 + kBlk > p.T;
            for (int it = 0, i = 0; it < n_it && ok; ++it, ++it_all) {
                const int qb = (u.i0 + i) * kBlk;
                if (++i == u.n_blk) i = 0;
                if (threadIdx.x == 0) *progress = it_all + ucnt + 1;
                const uint32_t qs = it_all % QS;
                const float* lse2 = reinterpret_cast<const float*>(smem + L::kLseOff + qs * 512) + c0;
                const bool need_mask = (qb == u.k0) || (qb + kBlk - 1 >= min_kend) || partial;
                const int j_lo = (int)(key - qb) - c0;
                const int j_hi = kend - 1 - qb - c0;
                ok = watched_warp_wait(&bar_qfull[qs], (it_all / QS) & 1, abort_flag) && watched_warp_wait(bar_sfull, it_all & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                uint32_t sv[32], sv2[32];   // S^T of the 32 queries at hand and of the other 32
                tmem_ld32(t_x + c0, sv);
                tmem_ld32(t_x + c0 + 32, sv2);
                tmem_ld_wait();
                tc_fence_before();
                mbar_arrive(bar_xfree1);
                // (one copy of the code for both halves)
#pragma unroll 1
                for (int half = 0; half < 2; ++half) {
                    const float* l2 = lse2 + 32 * half;
                    float pf[32];
#pragma unroll
                    for (int j = 0; j < 32; j += 4) {
                        const ulonglong2 l4 = *reinterpret_cast<const ulonglong2*>(l2 + j);
                        float x0, x1, x2, x3;   // LSE - S c
                        f2_unpack(f2_fma(f2_pack(__uint_as_float(sv[j]), __uint_as_float(sv[j + 1])), neg_scale2, l4.x), x0, x1);
                        f2_unpack(f2_fma(f2_pack(__uint_as_float(sv[j + 2]), __uint_as_float(sv[j + 3])), neg_scale2, l4.y), x2, x3);
                        pf[j] = ex2_approx(-x0);
                        pf[j + 1] = ex2_approx(-x1);
                        pf[j + 2] = ex2_approx(-x2);
                        pf[j + 3] = ex2_approx(-x3);
                    }
                    if (need_mask) {   // as bits: compares per element became branches (10007 tokens in samples of up to
                        // 400, 8 heads: this kernel 112.9 us with them, 102.6 without)
                        const uint32_t vis = range_bits(j_lo - half * 32, j_hi - half * 32);
#pragma unroll
                        for (int j = 0; j < 32; ++j) pf[j] = (vis >> j) & 1u ? pf[j] : 0.f;
                    }
                    uint32_t pk[16];
#pragma unroll
                    for (int j = 0; j < 32; j += 2) pk[j >> 1] = pack_bf16x2(pf[j], pf[j + 1]);
#pragma unroll
                    for (int j = 0; j < 32; ++j) sv[j] = sv2[j];
                    // dQ(it-1) has left Y's P^T columns (its MMA ran behind dV(it-1), so P^T(it-1) is spent)
                    if (half == 0 && it_all > 0) {
                        ok = watched_warp_wait(&bar_yfree[0], (it_all - 1) & 1, abort_flag);
                        if (!ok) break;
                        tc_fence_after();
                    }
                    tmem_st16(t_p + c0 / 2 + half * 16, pk);
                }
                if (!ok) break;
                tmem_st_wait();
                tc_fence_before();
                mbar_arrive(bar_pready);
            }
            if (!ok) break;
            ++ucnt;
            // ---- unit epilogue: dK and dV of the pair tile are added to the fp32 accumulators ----
            ok = watched_warp_wait(bar_dkvfull, (ucnt - 1) & 1, abort_flag);
            if (!ok) break;
            if (threadIdx.x == 0) *progress = it_all + ucnt;
            tc_fence_after();
            // through the shared-memory dS^T tile, which dQ has read, like dQ: bulk reduce-adds of 32 key rows x 32 head-dim
            // columns (rows past the end of the pool are dropped by the hardware)
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
                uint32_t v[32];
                const int col = c0 + (c & 1) * 32;
                tmem_ld32(tmem_base + lane_addr + (c < 2 ? kColDK : kColDV) + col, v);
                tmem_ld_wait();
                fused_stage_dq(c < 2 ? &tm_dkacc : &tm_dvacc, stage, v, lane, col, u.kvh, (int)u.k0 + (warp & 3) * 32);
            }
            if (lane == 0) tma_store_wait_read();
            __syncwarp();
            tc_fence_before();
            mbar_arrive(bar_dkvempty);
            if (threadIdx.x == 0) p.tile_ns[p.cta_tiles[idx]] = (uint32_t)(globaltimer_ns() - tile_t0);
        }
        // every bulk reduce this warp issued has completed before the CTA leaves
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }

    // ---------------- teardown ----------------
    if (warp != kFuWatchWarp && lane == 0) atomicAdd(finished, 1u);
    tc_fence_before();
    __syncthreads();
    if (warp == kFuMmaWarp) tmem_dealloc(tmem_base, 512);
    if (threadIdx.x == 0) {
        p.outcome[cta] = abort_flag[0] ? LIBRA_ERR_TIMEOUT : LIBRA_OK;
        p.busy[2 * cta + 1] = globaltimer_ns();
    }
}

// dq = scale * dq_acc, dk = scale * dk_acc, dv = dv_acc, rounded to bf16 (8 elements per thread), in one launch.
struct FinishArgs {
    const float* acc[3];
    void* out[3];
    int64_t n8[3];
    float mul[3];
};
__global__ void k_bwd_fused_finish(const FinishArgs f) {
    grid_dep_wait();
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    // (selected, not indexed: an index into the arguments would copy them to local memory, twice the time)
    const float* acc = f.acc[0];
    void* out = f.out[0];
    float mul = f.mul[0];
    int64_t n = f.n8[0];
    if (i >= n) { i -= n; acc = f.acc[1]; out = f.out[1]; mul = f.mul[1]; n = f.n8[1];
        if (i >= n) { i -= n; acc = f.acc[2]; out = f.out[2]; mul = f.mul[2]; n = f.n8[2]; }
    }
    if (i >= n) return;
    const float4 a = reinterpret_cast<const float4*>(acc)[2 * i], b = reinterpret_cast<const float4*>(acc)[2 * i + 1];
    uint4 w;
    w.x = pack_bf16x2(a.x * mul, a.y * mul);
    w.y = pack_bf16x2(a.z * mul, a.w * mul);
    w.z = pack_bf16x2(b.x * mul, b.y * mul);
    w.w = pack_bf16x2(b.z * mul, b.w * mul);
    reinterpret_cast<uint4*>(out)[i] = w;
}
static cudaError_t launch_finish(const FinishArgs& f, cudaStream_t s) {
    const int64_t n = f.n8[0] + f.n8[1] + f.n8[2];
    count_launch();
    return launch_dependent(k_bwd_fused_finish, (unsigned)((n + 255) / 256), 256u, 0, s, f);
}

}  // namespace libra
