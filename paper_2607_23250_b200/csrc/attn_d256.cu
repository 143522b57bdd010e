// Pool attention at head_dim 256 (the micro-benchmark head shape Hq 128 / Hkv 4 / d 256 of the paper's Table 1).
//
// A 128 x 256 bf16 operand tile is 64 KB and an accumulator of 128 rows x 256 head-dim columns takes half of
// TMEM, so the 128-wide kernels do not stretch to this width.  One kernel template covers the four passes; every
// pass keeps one side of the score matrix stationary (its operand tile(s) stay in shared memory, its
// accumulator in TMEM) and streams the other side in blocks of 64 rows:
//
//   FWD  queries stationary   S  = Q K^T          P = softmax (online, lazy rescale)      O  += P V
//   DV   keys stationary      S^T = K Q^T         P^T = exp2(S^T c - LSE)                 dV += P^T dO
//   DK   keys stationary      S^T, dP^T = V dO^T  dS^T = P^T o (dP^T - D)                 dK += dS^T Q
//   DQ   queries stationary   S, dP = dO V^T      dS = P o (dP - D)                       dQ += dS K
//
// dK and dV cannot share TMEM with S^T and dP^T at this width (2 x 256 accumulator columns), so the gradient takes
// three passes and recomputes S (eight GEMMs per cell for the five of the definition).
//
// Two CTAs work on 256 stationary rows (128 each) with cta_group::2 MMAs, so that each loads only half of every streamed
// tile: with 128 rows per CTA a pass read 64 KB from L2 for 128 x 64 x 512 MACs per GEMM pair, 5 to 7 TB/s, and each of its
// N = 64 MMAs took 48 cycles for the 32 of its products (forward / dV + dK / dQ of one 32768-token sequence at Hq 128, Hkv 4:
// 21.5 / 54.1 / 22.7 ms, now 14.3 / 33.9 / 20.7; the clock is at 1.35 GHz then, the power limit's).  Of a streamed tile that is the B operand of an X GEMM (N = its 64 rows) a CTA holds 32 rows;
// of one that the accumulating GEMM multiplies with (N = 256 head-dim columns) it holds 128 columns; the tile that is
// both (Q in DK, K in DQ) is loaded in both halves.  The leader (even rank) issues all MMAs; its barriers count the
// copies and the compute warps of both CTAs; commits arrive in both.  A block that no row of one of the two sees (past its
// diagonal, before its first sample) leaves that one's lanes out of the accumulating GEMM.
//
// TMEM: X1, X2, W (32 columns a block: the bf16 result of the element-wise step, A operand of the last GEMM) in 256
// columns, acc (256).  FWD, DV: X1 3 x 64 | W 2 x 32; X1 runs two blocks ahead.  DK, DQ: X1 2 x 64 | X2 2 x 64, one block
// ahead; W lies over the first half of each thread group's columns of X1, which that group has read by then.
// Roles (320 threads): warps 0-7 compute, warp 8 one TMA thread, warp 9 one MMA thread.  In the gradient passes two
// threads share a stationary row (32 of the block's 64 columns each; warps w and w + 4 reach the same TMEM lanes); the
// forward keeps one thread per row, because the running maximum and sum of a row live in its registers (warps 4-7 write
// the output tiles there).  Per streamed block: X1 (and X2) are issued, the compute warps turn them into W, the accumulating GEMM
// is issued; X1 and X2 of the next block are issued ahead, so they run under the element-wise step of the current one
// (a dV / dK / dQ block: 1650 / 2330 / 2400 cycles with only X1 ahead and one W, 1220 / 1920 / 2020 now; of MMAs 1024 /
// 1536 / 1536).
// Masks follow the sample bounds per element, in blocks that a bound crosses.
#include <math.h>

#include "common.h"
#include "drain.cuh"
#include "ptx.cuh"

namespace libra {
namespace d256 {

constexpr int kThreads = 320;
constexpr int kTmaWarp = 8, kMmaWarp = 9;
constexpr int kRows = 128;       // stationary rows per unit
constexpr int kBlk = 64;         // streamed rows per block
constexpr int kD = 256;
constexpr uint32_t kColAcc = 256;
constexpr uint64_t kDrainNs = 2000000;
constexpr int kSmemMax = 232448;
enum Mode { FWD = 0, DV = 1, DK = 2, DQ = 3 };   // (also the index of the pass's outcome words)

template <int MODE>
struct Cfg {
    static constexpr bool kKeyStationary = (MODE == DV || MODE == DK);
    static constexpr bool kHasX2 = (MODE == DK || MODE == DQ);
    static constexpr int kGroups = MODE == FWD ? 1 : 2;      // compute threads per stationary row
    static constexpr int kCols = 64 / kGroups;               // columns of a streamed block per compute thread
    static constexpr int kStationary = kHasX2 ? 2 : 1;       // resident 64 KB tiles per CTA
    static constexpr int kStreams = kHasX2 ? 3 : 2;          // streamed halves per block: X1's, [X2's,] the accumulating GEMM's
    static constexpr int kAcc = kStreams - 1;                // the last one
    // FWD holds the tiles of this unit and the next: its units are a few blocks of a short sample.  A DV tile has all the
    // heads of the group: three blocks in flight for that cost its launch 20 % (dV + dK 34.9 -> 37.7 ms).
    static constexpr int kStBufs = MODE == FWD ? 2 : 1;
    static constexpr int kStages = kHasX2 ? 2 : (MODE == FWD ? 3 : 4);   // blocks in flight
    static constexpr int kBig = 65536, kBigHalf = 16384;     // 128 x 256 bf16: four column halves of 128 rows x 128 B
    static constexpr int kHalfTile = 16384;                  // 32 x 256: four columns of 32 rows x 128 B, or 64 x 128: two of 64
    static constexpr int kRowHalf = 4096, kColHalf = 8192;   // one such column of 64 elements
    static constexpr int kStatBytes = MODE == DV ? 256 : (MODE == DK ? 512 : 0);   // per streamed block: lse2[64], dvec[64]
    static constexpr int kSaOff = 0;
    static constexpr int kSbOff = kBig;
    static constexpr int kRingOff = kStationary * kStBufs * kBig;
    static constexpr int kStatOff = kRingOff + kStreams * kStages * kHalfTile;
    static constexpr int kBarOff = kStatOff + kStages * 512;
    // FWD: 1 / row sum of the last three units' rows, in place of the statistics
    static_assert(kHasX2 || kStages * 512 >= 3 * kRows * 4, "row sums");
    // full, empty [kStreams][kStages], stat[kStages], acc_done, acc_free, drain, x1_full[3], x2_full[2], w_ready[2],
    // acc_step[2], st_full[2], st_empty[2], l_full[3]
    static constexpr int kNumBars = 2 * kStreams * kStages + kStages + 19;
    static constexpr int kMiscOff = kBarOff + kNumBars * 8;
    static constexpr int kBytes = kMiscOff + 32;
    static_assert(kBytes <= kSmemMax, "exceeds the shared memory of an sm_100 CTA");
    // TMEM columns of a block's X1, X2 and W (see above)
    static constexpr uint32_t kX1Bufs = kHasX2 ? 2 : 3;
    __device__ static constexpr uint32_t col_x1(uint32_t b) { return 64 * b; }
    __device__ static constexpr uint32_t col_x2(uint32_t b) { return 128 + 64 * b; }
    // W columns of the block's streamed rows 16 kk .. 16 kk + 15; b is the block's parity
    __device__ static constexpr uint32_t col_w(uint32_t b, uint32_t kk) {
        return kHasX2 ? col_x1(b) + (kk >> 1) * 32 + (kk & 1) * 8 : 192 + 32 * b + 8 * kk;
    }
    __host__ __device__ static constexpr int tile_off(int stream, uint32_t stage) {
        return kRingOff + (stream * kStages + (int)stage) * kHalfTile;
    }
};

struct Params {
    __nv_bfloat16* out;     // DV: dv, DK: dk [T, Hkv, 256]; DQ: dq [T, Hq, 256]
    float* lse;             // FWD: [Hq, T]
    const float* lse2;      // backward passes: [Hq, Tpad]  LSE * log2(e)
    const float* dvec;      // backward passes: [Hq, Tpad]  D_i
    const int32_t* cta_offsets;
    const int32_t* cta_tiles;
    const int32_t* tok_start;
    const int32_t* tok_end;
    int64_t T, Tpad;
    int hq, hkv, H;         // H: head shards of the query-major lists (FWD, DQ)
    int W;                  // FWD, DQ: workers of the lists; a pair of CTAs runs the lists of two
    // key-stationary passes over pair tiles (256 keys x query chunk x kv head) instead of key-major tiles: the
    // accumulator of a unit is added to acc32 [T, Hkv, 256] (fp32) and rounded by a later kernel
    float* acc32;           // null: key-major tiles, results stored as bf16 by the pass itself
    const int32_t* u_blk;   // [NU] key block of pair-block u
    const int32_t* u_chunk; // [NU] query chunk of pair-block u
    int64_t NU;
    int R;                  // 128-row blocks per query chunk
    float scale, scale_log2;
    int* outcome;
    int side_by_side;       // DK, DQ: start without waiting for the pass ahead
    const int* plan_status;
    uint32_t wait_limit_ns;
    int inject_stall;
    uint64_t* busy;
};

// Walks the units of a CTA pair in the order every role of both CTAs uses.
//   key-stationary passes: one unit per tile of the pair's list (256 keys x one kv head); its iterations are the query
//   heads of the group times the 64-row query blocks from the diagonal to the end of the last key's sample (of the chunk);
//   query-stationary passes: a query-major tile (256 rows x head shard) of the lists of two workers gives one unit per
//   head; its iterations are the 64-key blocks from the start of the first row's sample to the diagonal.
// r0 is the first of this CTA's 128 stationary rows.
template <int MODE>
struct Units {
    static constexpr bool kKeys = Cfg<MODE>::kKeyStationary;
    const Params& p;
    int idx, end, hh, hps, G;
    int64_t base, r0;       // first stationary row of the pair and of this CTA
    int h, kvh, b_lo, n_blk, n_it;
    int bound0, bound1;     // of each CTA's rows: start of the first one's sample (queries), end of the last one's (keys)
    __device__ Units(const Params& p_, int cta) : p(p_) {
        const int c = cta >> 1;
        if (kKeys) {
            idx = p.cta_offsets[c];
            end = p.cta_offsets[c + 1];
        } else {   // neighbouring lists are contiguous
            idx = p.cta_offsets[2 * c];
            end = p.cta_offsets[2 * c + 2 < p.W ? 2 * c + 2 : p.W];
        }
        G = p.hq / p.hkv;
        hps = kKeys ? 1 : p.hq / p.H;
        hh = hps - 1;
        --idx;
    }
    __device__ bool next(uint32_t rank) {
        if (++hh == hps) { hh = 0; if (++idx >= end) return false; }
        const int t = p.cta_tiles[idx];
        if constexpr (kKeys) {
            const int j = p.acc32 ? p.u_blk[(int)(t % p.NU)] : t / p.hkv;
            kvh = p.acc32 ? (int)(t / p.NU) : t % p.hkv;
            base = (int64_t)j * (2 * kRows);
            bound0 = p.tok_end[base + kRows - 1 < p.T ? base + kRows - 1 : p.T - 1];
            bound1 = p.tok_end[base + 2 * kRows - 1 < p.T ? base + 2 * kRows - 1 : p.T - 1];
            int last64 = (bound1 - 1) / kBlk;
            b_lo = (int)(base / kBlk);
            if (p.acc32) {   // pair tile: the query blocks of one chunk only
                const int c = p.u_chunk[(int)(t % p.NU)], lo64 = 2 * c * p.R, hi64 = 2 * (c * p.R + p.R) - 1;
                b_lo = lo64 > b_lo ? lo64 : b_lo;
                last64 = hi64 < last64 ? hi64 : last64;
            }
            n_blk = last64 - b_lo + 1;
            h = kvh * G;
            n_it = G * n_blk;
        } else {
            base = (int64_t)(t / p.H) * (2 * kRows);
            bound0 = p.tok_start[base];
            const int64_t last_row = base + 2 * kRows - 1 < p.T ? base + 2 * kRows - 1 : p.T - 1;
            h = (t % p.H) * hps + hh;
            kvh = h / G;
            b_lo = bound0 / kBlk;
            n_blk = (int)(last_row / kBlk) - b_lo + 1;
            n_it = n_blk;
        }
        r0 = base + rank * kRows;
        return true;
    }
    // Streamed blocks of a head that some row of CTA c sees: [lo, hi], of the unit's 0 .. n_blk - 1 (lo > hi: none).
    __device__ void seen_by(uint32_t c, int& lo, int& hi) const {
        const int64_t a = base + c * kRows, z = a + kRows - 1 < p.T ? a + kRows - 1 : p.T - 1;
        const int bound = c == 0 ? bound0 : (kKeys ? bound1 : (a < p.T ? p.tok_start[a] : 0));   // (most roles do without the last)
        lo = kKeys ? (int)(a / kBlk) : bound / kBlk;
        hi = kKeys ? (bound - 1) / kBlk : (int)(z / kBlk);
        lo = lo > b_lo ? lo - b_lo : 0;
        hi = a >= p.T ? -1 : (hi - b_lo < n_blk ? hi - b_lo : n_blk - 1);
    }
    // First row of the streamed block j of a head; the iterations of a unit take its heads in turn, blocks ascending.
    __device__ int stream_row(int j) const { return (b_lo + j) * kBlk; }
};

template <int MODE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
k_attn_d256(const __grid_constant__ CUtensorMap tm_sa, const __grid_constant__ CUtensorMap tm_sb,
            const __grid_constant__ CUtensorMap tm_t0, const __grid_constant__ CUtensorMap tm_t1,
            const __grid_constant__ CUtensorMap tm_t2, const Params p) {
    using L = Cfg<MODE>;
    constexpr int S = L::kStages, N = L::kStreams;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::kBarOff);
    uint64_t* bar_full = bars;                 // [N][S] leader: both CTAs' halves have landed
    uint64_t* bar_empty = bars + N * S;        // [N][S] the MMA that read it has run
    uint64_t* bar_stat = bars + 2 * N * S;     // [S] statistics of a streamed block (each CTA its own copy)
    uint64_t* b2 = bar_stat + S;
    uint64_t* bar_accdone = b2 + 0;
    uint64_t* bar_accfree = b2 + 1;            // leader
    uint64_t* bar_drain = b2 + 2;
    uint64_t* bar_x1full = b2 + 3;     // [3] one per X1 buffer, [2] per X2 buffer: committed one or two blocks ahead
    uint64_t* bar_x2full = b2 + 6;
    // by the block's parity (the compute warps may be a block ahead of the issuer, the issuer of the accumulating GEMM):
    uint64_t* bar_wready = b2 + 8;     // [2] leader: W is in both CTAs' TMEM
    uint64_t* bar_accstep = b2 + 10;   // [2] the accumulating GEMM has run: W may be rewritten, acc rescaled
    uint64_t* bar_stfull = b2 + 12;    // [2] leader
    uint64_t* bar_stempty = b2 + 14;   // [2] FWD: the output tile has left the buffer; else the unit's X MMAs have run
    uint64_t* bar_lfull = b2 + 16;     // [3] FWD: the row sums of a unit are there
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::kMiscOff);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::kMiscOff + 4);
    volatile uint32_t* peer_gave_up = reinterpret_cast<volatile uint32_t*>(smem + L::kMiscOff + 12);
    volatile uint32_t* issued = peer_gave_up + 1;   // [2][2] leader: units and streamed tiles whose loads either CTA has issued

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int cta = blockIdx.x;
    const uint32_t rank = cluster_rank();

    if ((smem_u32(smem) & 1023u) != 0) {   // (the same in both CTAs)
        if (threadIdx.x == 0) p.outcome[cta] = LIBRA_ERR_CUDA;
        grid_dep_wait();
        return;
    }
    // The dK and dQ passes need what the dV pass had waited for and nothing of the pass ahead: they take the SMs that
    // fall free and wait for the pass ahead before they end.
    if (MODE == FWD || MODE == DV || !p.side_by_side) grid_dep_wait();
    if (MODE == DV || MODE == DK) grid_dep_launch();
    if (const int ps = ld_acquire(p.plan_status); ps != 0) {  // malformed cu_seqlens: report and leave
        if (threadIdx.x == 0) { p.outcome[cta] = ps; p.busy[2 * cta] = p.busy[2 * cta + 1] = 0; }
        if (MODE == DK || MODE == DQ) grid_dep_wait();
        return;
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < N * S; ++s) { mbar_init(&bar_full[s], 1); mbar_init(&bar_empty[s], 1); }
        for (int s = 0; s < S; ++s) mbar_init(&bar_stat[s], 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&bar_stfull[b], 1);
            mbar_init(&bar_stempty[b], MODE == FWD ? 4 : 1);
        }
        for (int b = 0; b < 3; ++b) mbar_init(&bar_lfull[b], 128);
        for (int b = 0; b < 3; ++b) mbar_init(&bar_x1full[b], 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&bar_x2full[b], 1);
            mbar_init(&bar_wready[b], 2 * 4 * L::kGroups);    // a compute warp's lanes arrive as one
            mbar_init(&bar_accstep[b], 1);
        }
        mbar_init(bar_accdone, 1);
        mbar_init(bar_accfree, 2 * 4 * L::kGroups);
        mbar_init(bar_drain, 1);
        abort_flag[0] = 0;
        abort_flag[1] = (int)p.wait_limit_ns;
        *peer_gave_up = 0;
        fence_mbar_init();
        p.busy[2 * cta] = globaltimer_ns();
    }
    if (warp == kMmaWarp) {
        tmem_alloc_pair(tmem_slot, 512);
        tmem_relinquish_pair();
    }
    if (warp == kTmaWarp && lane == 0) {
        prefetch_tmap(&tm_sa);
        if (L::kStationary == 2) prefetch_tmap(&tm_sb);
        prefetch_tmap(&tm_t0);
        prefetch_tmap(&tm_t1);
        if (N == 3 || MODE == FWD) prefetch_tmap(&tm_t2);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();      // both CTAs' barriers are initialised and their TMEM is allocated
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == kTmaWarp) {
        // ---------------- TMA producer (each CTA loads its own halves; the leader's barriers count both) ----------------
        if (elect_one()) {
            Units<MODE> u(p, cta);
            uint32_t n = 0, uc = 0;          // n: iterations so far (over all units)
            uint32_t tiles = 0;
            bool ok = true;
            while (ok && !(p.inject_stall && rank == 1) && u.next(rank)) {
                const uint32_t sbuf = uc % L::kStBufs, a_off = L::kSaOff + sbuf * L::kBig;
                ok = mbar_wait(&bar_stempty[sbuf], ((uc / L::kStBufs) & 1) ^ 1, abort_flag);
                if (!ok) break;
                if (rank == 0) mbar_arrive_expect_tx(&bar_stfull[sbuf], 2 * L::kStationary * L::kBig);
                const uint32_t stfull0 = map_to_rank(&bar_stfull[sbuf], 0);
                const int st_head = L::kKeyStationary ? u.kvh : u.h;
                for (int half = 0; half < 4; ++half) {
                    tma_load_3d_pair(smem + a_off + half * L::kBigHalf, &tm_sa, stfull0, half * 64, st_head, (int)u.r0);
                    if (L::kStationary == 2)
                        tma_load_3d_pair(smem + L::kSbOff + half * L::kBigHalf, &tm_sb, stfull0, half * 64, st_head, (int)u.r0);
                }
                ++uc;
                int sh = L::kKeyStationary ? u.h : u.kvh, j = 0;
                for (int it = 0; it < u.n_it && ok; ++it, ++n) {
                    const int row = u.stream_row(j);
                    const uint32_t s = n % S, ph = (n / S) & 1;
                    for (int k = 0; k < N && ok; ++k) {
                        ok = mbar_wait(&bar_empty[k * S + s], ph ^ 1, abort_flag);
                        if (!ok) break;
                        if (rank == 0) mbar_arrive_expect_tx(&bar_full[k * S + s], 2 * L::kHalfTile);
                        const uint32_t full0 = map_to_rank(&bar_full[k * S + s], 0);
                        uint8_t* dst = smem + L::tile_off(k, s);
                        if (k == L::kAcc) {
                            for (int c = 0; c < 2; ++c)   // this CTA's 128 of the 256 columns
                                tma_load_3d_pair(dst + c * L::kColHalf, N == 3 ? &tm_t2 : &tm_t1, full0, 128 * (int)rank + 64 * c, sh, row);
                        } else {
                            for (int c = 0; c < 4; ++c)   // this CTA's 32 of the 64 rows
                                tma_load_3d_pair(dst + c * L::kRowHalf, k == 0 ? &tm_t0 : &tm_t1, full0, 64 * c, sh, row + 32 * (int)rank);
                        }
                        if (k == L::kAcc && L::kStatBytes > 0) {   // the slot's last reader was ahead of this stream's MMA
                            mbar_arrive_expect_tx(&bar_stat[s], L::kStatBytes);
                            bulk_load_1d(smem + L::kStatOff + s * 512, p.lse2 + (size_t)sh * p.Tpad + row, 256, &bar_stat[s]);
                            if (L::kStatBytes == 512)
                                bulk_load_1d(smem + L::kStatOff + s * 512 + 256, p.dvec + (size_t)sh * p.Tpad + row, 256, &bar_stat[s]);
                        }
                        ++tiles;
                    }
                    if (++j == u.n_blk) { j = 0; ++sh; }
                }
            }
            issued[2 * rank] = uc;
            issued[2 * rank + 1] = tiles;
            if (rank == 1) {
                const uint32_t there = map_to_rank(const_cast<const uint32_t*>(issued) + 2, 0);
                st_cluster(there, uc);
                st_cluster(there + 4, tiles);
            }
        }
        __syncwarp();
    } else if (warp == kMmaWarp) {
        // ---------------- MMA issuer (the leader's, for both) ----------------
        if (rank == 0 && elect_one()) {
            constexpr uint32_t idesc_x = make_idesc(2 * kRows, kBlk, 0, 0);    // X = stationary x streamed^T, both K-major
            constexpr uint32_t idesc_acc = make_idesc(2 * kRows, kD, 0, 1);    // acc += W (TMEM) x streamed tile, MN-major
            const uint32_t sb = smem_u32(smem);
            const uint64_t kdesc0 = make_sdesc(sb, 16, 1024);               // K-major view at offset 0
            const uint64_t mdesc0 = make_sdesc(sb, L::kColHalf, 1024);      // MN-major view of a 64-row tile
            auto issue_x = [&](uint32_t d_col, uint32_t a_off, uint32_t b_off) {
                const uint64_t da = sdesc_advance(kdesc0, a_off), db = sdesc_advance(kdesc0, b_off);
#pragma unroll
                for (int kk = 0; kk < kD / 16; ++kk)
                    mma_ss_pair(tmem_base + d_col, sdesc_advance(da, (kk / 4) * L::kBigHalf + (kk % 4) * 32),
                                sdesc_advance(db, (kk / 4) * L::kRowHalf + (kk % 4) * 32), idesc_x, kk > 0);
            };
            Units<MODE> u(p, cta);
            uint32_t uc = 0, itc = 0;
            uint32_t xi = 0, xb = 0;   // next block to multiply, its X1 buffer
            bool ok = true;
            // X1 (and X2) of the next block; its streamed halves are free again as soon as they have run
            uint32_t a_off = 0;                 // stationary tile of the unit
            auto do_x = [&](bool last) -> bool {
                const uint32_t s = xi % S, ph = (xi / S) & 1;
                if (!mbar_wait(&bar_full[s], ph, abort_flag)) return false;
                tc_fence_after();
                issue_x(L::col_x1(xb), a_off, L::tile_off(0, s));
                tc_commit_pair(&bar_x1full[xb]);
                tc_commit_pair(&bar_empty[s]);
                if (L::kHasX2) {
                    if (!mbar_wait(&bar_full[S + s], ph, abort_flag)) return false;
                    tc_fence_after();
                    issue_x(L::col_x2(xb), L::kSbOff, L::tile_off(1, s));
                    tc_commit_pair(&bar_x2full[xb]);
                    tc_commit_pair(&bar_empty[S + s]);
                }
                // (the unit's stationary tiles are not read again; FWD stages its output there)
                if (MODE != FWD && last) tc_commit_pair(&bar_stempty[0]);
                ++xi;
                if (++xb == L::kX1Bufs) xb = 0;
                return true;
            };
            constexpr int kAhead = (int)L::kX1Bufs - 1;
            while (ok && u.next(rank)) {
                const uint32_t sbuf = uc % L::kStBufs;
                a_off = L::kSaOff + sbuf * L::kBig;
                ok = mbar_wait(&bar_stfull[sbuf], (uc / L::kStBufs) & 1, abort_flag);
                for (int it = 0; it < kAhead && it < u.n_it && ok; ++it) ok = do_x(it == u.n_it - 1);
                if (!ok) break;
                // The accumulating GEMM leaves out a CTA none of whose rows see the block: W is zero there, but times an
                // infinity or a NaN of the block that is NaN.
                int lo0, hi0, lo1, hi1, j = 0;
                u.seen_by(0, lo0, hi0);
                u.seen_by(1, lo1, hi1);
                uint32_t begun = 0;              // bit per CTA: its rows of the unit's accumulator have been written
                for (int it = 0; it < u.n_it && ok; ++it, ++itc) {
                    const uint32_t s = itc % S, ph = (itc / S) & 1, b = itc & 1;
                    // The X GEMMs of a block ahead run under the element-wise step of this one.  Their buffers were read out
                    // before W of the previous block was ready, and its accumulating GEMM, which may read W there, is ahead
                    // of them in the pipe.
                    if (it + kAhead < u.n_it) ok = do_x(it + kAhead == u.n_it - 1);
                    const uint32_t see = (j >= lo0 && j <= hi0 ? 1u : 0u) | (j >= lo1 && j <= hi1 ? 2u : 0u);
                    const bool plain = see == 3 && (begun == 0 || begun == 3);
                    if (++j == u.n_blk) j = 0;
                    if (ok) ok = mbar_wait(&bar_full[L::kAcc * S + s], ph, abort_flag);
                    if (ok) ok = mbar_wait(&bar_wready[b], (itc >> 1) & 1, abort_flag);
                    if (ok && it == 0 && uc > 0) ok = mbar_wait(bar_accfree, (uc - 1) & 1, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    {
                        const uint64_t db = sdesc_advance(mdesc0, L::tile_off(L::kAcc, s));
                        const uint32_t t_w = tmem_base + L::col_w(b, 0), adds = see & begun;
                        if (plain) {
#pragma unroll
                            for (int kk = 0; kk < kBlk / 16; ++kk)
                                mma_ts_pair(tmem_base + kColAcc, tmem_base + L::col_w(b, kk), sdesc_advance(db, kk * 2048), idesc_acc,
                                            (begun || kk > 0) ? 1u : 0u);
                        } else if (see == 3) {   // a CTA's first product overwrites; these two did not begin with the same block
                            mma_ts_pair_of(tmem_base + kColAcc, t_w, db, idesc_acc, 1, adds);
                            mma_ts_pair_of(tmem_base + kColAcc, t_w, db, idesc_acc, 0, 3 - adds);
#pragma unroll
                            for (int kk = 1; kk < kBlk / 16; ++kk)
                                mma_ts_pair(tmem_base + kColAcc, tmem_base + L::col_w(b, kk), sdesc_advance(db, kk * 2048), idesc_acc, 1);
                        } else if (see) {
#pragma unroll
                            for (int kk = 0; kk < kBlk / 16; ++kk)
                                mma_ts_pair_of(tmem_base + kColAcc, tmem_base + L::col_w(b, kk), sdesc_advance(db, kk * 2048), idesc_acc,
                                               (adds || kk > 0) ? 1u : 0u, see);
                        }
                        begun |= see;
                    }
                    tc_commit_pair(&bar_accstep[b]);
                    tc_commit_pair(&bar_empty[L::kAcc * S + s]);
                    if (it == u.n_it - 1) tc_commit_pair(bar_accdone);
                }
                ++uc;
            }
            if (!ok || abort_flag[0]) {
                tc_commit_pair(bar_drain);
                mbar_wait_drain(bar_drain, 0, kDrainNs);
            }
        }
        __syncwarp();
    } else if (warp < 4 * L::kGroups) {
        // ---------------- compute warps: thread (r, grp) owns stationary row r (TMEM lane r) and the columns
        // [col0, col0 + kCols) of every streamed block ----------------
        constexpr int NC = L::kCols;
        const int grp = warp >> 2;
        const int col0 = grp * NC;
        const int r = (warp & 3) * 32 + lane;
        const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t t_base = tmem_base + lane_addr;
        const uint32_t t_acc = t_base + kColAcc + grp * (kD / L::kGroups);
        const uint32_t wready0 = map_to_rank(bar_wready, 0), accfree0 = map_to_rank(bar_accfree, 0);
        Units<MODE> u(p, cta);
        uint32_t uc = 0, itc = 0;
        uint32_t xb = 0, xph = 0;                    // X1 buffer of the block and its phase
        uint32_t lb = 0;                             // FWD: the unit's slot of row sums
        bool ok = true;
        while (ok && u.next(rank)) {
            const int64_t row = u.r0 + r;            // this thread's query row (FWD, DQ) or key (DV, DK)
            bool row_ok = row < p.T;
            // visible columns of streamed block starting at b0: [lo_abs - b0, hi_abs - b0]
            //   query-stationary: keys from the start of the row's sample to the row itself
            //   key-stationary:   queries from the key itself to the end of its sample
            int lo_abs, hi_abs;
            if (L::kKeyStationary) {
                lo_abs = (int)row;
                hi_abs = row_ok ? p.tok_end[row] - 1 : -1;
            } else {
                lo_abs = row_ok ? p.tok_start[row] : 0;
                hi_abs = row_ok ? (int)row : -1;
            }
            lo_abs -= col0;                          // counted from this thread's first column
            hi_abs -= col0;
            float m_ref = -INFINITY, l_sum = 0.f;    // FWD
            float lse2r = 0.f, dvecr = 0.f;          // DQ
            if (MODE == DQ) {
                if (row_ok) {                                 // (this CTA's rows may lie past the end of the pool)
                    lse2r = p.lse2[(size_t)u.h * p.Tpad + row];
                    dvecr = p.dvec[(size_t)u.h * p.Tpad + row];
                }
            }
            int j = 0;
            for (int it = 0; it < u.n_it && ok; ++it, ++itc) {
                const int b0 = u.stream_row(j);
                if (++j == u.n_blk) j = 0;
                // first and last visible of this thread's columns
                const int c_lo = lo_abs - b0, c_hi = hi_abs - b0;
                const uint32_t wb = itc & 1;
                const bool need_mask = __any_sync(0xffffffffu, c_lo > 0 || c_hi < NC - 1);   // most blocks are dense
                const uint32_t s1 = itc % S;
                const float* st = reinterpret_cast<const float*>(smem + L::kStatOff + s1 * 512) + col0;
                if (L::kStatBytes > 0) {   // the streamed rows' statistics
                    ok = warp_wait(&bar_stat[s1], (itc / S) & 1, abort_flag);
                    if (!ok) break;
                }
                ok = warp_wait(&bar_x1full[xb], xph, abort_flag);
                if (!ok) break;
                tc_fence_after();
                uint32_t sr[NC];
#pragma unroll
                for (int c = 0; c < NC; c += 32) tmem_ld32(t_base + L::col_x1(xb) + col0 + c, sr + c);
                tmem_ld_wait();
                if (++xb == L::kX1Bufs) { xb = 0; xph ^= 1; }
                uint32_t pk[NC / 2];
                if constexpr (MODE == FWD) {
                    if (need_mask) {
#pragma unroll
                        for (int w = 0; w < kBlk / 32; ++w) {
                            const uint32_t vis = range_bits(c_lo - 32 * w, c_hi - 32 * w);
#pragma unroll
                            for (int i = 0; i < 32; ++i) sr[32 * w + i] = (vis >> i) & 1u ? sr[32 * w + i] : 0xff800000u;  // -inf
                        }
                    }
                    float mx = -INFINITY;
                    {
                        float pm[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) pm[q] = fmaxf(__uint_as_float(sr[2 * q]), __uint_as_float(sr[2 * q + 1]));
#pragma unroll
                        for (int i = 16; i < kBlk; i += 16)
#pragma unroll
                            for (int q = 0; q < 8; ++q)
                                pm[q] = max3(pm[q], __uint_as_float(sr[i + 2 * q]), __uint_as_float(sr[i + 2 * q + 1]));
                        mx = fmaxf(max3(pm[0], pm[1], pm[2]), max3(pm[3], pm[4], pm[5]));
                        mx = max3(mx, pm[6], pm[7]);
                    }
                    mx *= p.scale_log2;
                    // lazy rescale: the reference only moves when the maximum grew by more than 2^8
                    float m_new = m_ref;
                    bool grow = false;
                    if (mx > m_ref + 8.0f || (m_ref == -INFINITY && mx > -INFINITY)) { m_new = mx; grow = true; }
                    const float factor = grow ? ex2_approx(m_ref - m_new) : 1.0f;
                    l_sum *= factor;
                    m_ref = m_new;
                    const float m_use = (m_ref == -INFINITY) ? 0.f : m_ref;
                    float ps0 = 0.f, ps1 = 0.f;
#pragma unroll
                    for (int i = 0; i < kBlk; i += 2) {
                        const float p0 = ex2_approx(fmaf(__uint_as_float(sr[i]), p.scale_log2, -m_use));
                        const float p1 = ex2_approx(fmaf(__uint_as_float(sr[i + 1]), p.scale_log2, -m_use));
                        ps0 += p0;
                        ps1 += p1;
                        pk[i >> 1] = pack_bf16x2(p0, p1);
                    }
                    if (it > 0 && __any_sync(0xffffffffu, grow)) {
                        // O is rescaled once the previous block's accumulation has landed
                        ok = warp_wait(&bar_accstep[wb ^ 1], ((itc - 1) >> 1) & 1, abort_flag);
                        if (!ok) break;
                        tc_fence_after();
#pragma unroll
                        for (int c = 0; c < kD; c += 32) {
                            uint32_t orow[32];
                            tmem_ld32(t_acc + c, orow);
                            tmem_ld_wait();
#pragma unroll
                            for (int i = 0; i < 32; ++i) orow[i] = __float_as_uint(__uint_as_float(orow[i]) * factor);
                            tmem_st32(t_acc + c, orow);
                        }
                    }
                    l_sum += ps0 + ps1;
                } else {
                    // P = exp2(S c - LSE) on the visible elements, 0 elsewhere
                    float pf[NC];
                    const uint64_t scale2 = f2_pack(p.scale_log2, p.scale_log2), neg1 = f2_pack(-1.f, -1.f);
                    const uint64_t nl2 = f2_pack(-lse2r, -lse2r);
#pragma unroll
                    for (int i = 0; i < NC; i += 4) {   // 16-byte broadcast loads of the streamed rows' LSE
                        uint64_t n01 = nl2, n23 = nl2;
                        if (L::kKeyStationary) {
                            const ulonglong2 l4 = *reinterpret_cast<const ulonglong2*>(st + i);
                            n01 = f2_mul(l4.x, neg1);
                            n23 = f2_mul(l4.y, neg1);
                        }
                        float x0, x1, x2, x3;
                        f2_unpack(f2_fma(f2_pack(__uint_as_float(sr[i]), __uint_as_float(sr[i + 1])), scale2, n01), x0, x1);
                        f2_unpack(f2_fma(f2_pack(__uint_as_float(sr[i + 2]), __uint_as_float(sr[i + 3])), scale2, n23), x2, x3);
                        pf[i] = ex2_approx(x0);
                        pf[i + 1] = ex2_approx(x1);
                        pf[i + 2] = ex2_approx(x2);
                        pf[i + 3] = ex2_approx(x3);
                    }
                    if (need_mask) {
                        static_assert(MODE == FWD || NC == 32, "one mask word per compute thread");
                        const uint32_t vis = range_bits(c_lo, c_hi);
#pragma unroll
                        for (int i = 0; i < NC; ++i) pf[i] = (vis >> i) & 1u ? pf[i] : 0.f;
                    }
                    if (MODE == DV) {
#pragma unroll
                        for (int i = 0; i < NC; i += 2) pk[i >> 1] = pack_bf16x2(pf[i], pf[i + 1]);
                    } else {
                        ok = warp_wait(&bar_x2full[wb], (itc >> 1) & 1, abort_flag);
                        if (!ok) break;
                        tc_fence_after();
                        uint32_t dp[NC];
#pragma unroll
                        for (int c = 0; c < NC; c += 32) tmem_ld32(t_base + L::col_x2(wb) + col0 + c, dp + c);
                        tmem_ld_wait();
                        const uint64_t nd2 = f2_pack(-dvecr, -dvecr);
#pragma unroll
                        for (int i = 0; i < NC; i += 4) {
                            uint64_t n01 = nd2, n23 = nd2;
                            if (L::kKeyStationary) {
                                const ulonglong2 d4 = *reinterpret_cast<const ulonglong2*>(st + 64 + i);
                                n01 = f2_mul(d4.x, neg1);
                                n23 = f2_mul(d4.y, neg1);
                            }
                            float y0, y1, y2, y3;
                            f2_unpack(f2_mul(f2_pack(pf[i], pf[i + 1]),
                                             f2_add(f2_pack(__uint_as_float(dp[i]), __uint_as_float(dp[i + 1])), n01)), y0, y1);
                            f2_unpack(f2_mul(f2_pack(pf[i + 2], pf[i + 3]),
                                             f2_add(f2_pack(__uint_as_float(dp[i + 2]), __uint_as_float(dp[i + 3])), n23)), y2, y3);
                            pk[i >> 1] = pack_bf16x2(y0, y1);
                            pk[(i >> 1) + 1] = pack_bf16x2(y2, y3);
                        }
                    }
                }
                // (the results exist before the wait: left to itself the compiler moves the exponentials behind it)
#pragma unroll
                for (int i = 0; i < NC / 2; ++i) asm volatile("" : "+r"(pk[i]));
                if (!L::kHasX2 && itc > 1) {   // the accumulating GEMM of two blocks ago has consumed W
                    ok = warp_wait(&bar_accstep[wb], ((itc >> 1) - 1) & 1, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                }
#pragma unroll
                for (int c = 0; c < NC / 2; c += 16) tmem_st16(t_base + L::col_w(wb, (uint32_t)(col0 + 2 * c) / 16), pk + c);
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(wready0 + 8 * wb);
            }
            if (!ok) break;
            if constexpr (MODE == FWD) {   // warps 4-7 take it from here
                reinterpret_cast<float*>(smem + L::kStatOff)[lb * kRows + r] = (l_sum > 0.f) ? 1.0f / l_sum : 0.f;
                mbar_arrive(&bar_lfull[lb]);
                if (++lb == 3) lb = 0;
                if (row_ok) p.lse[(size_t)u.h * p.T + row] = (m_ref + log2f(l_sum)) * 0.6931471805599453f;
                continue;
            }
            // ---- unit epilogue: the accumulator leaves TMEM ----
            ok = warp_wait(bar_accdone, uc & 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            float mul = 1.0f;
            if (MODE == DK || MODE == DQ) mul = p.scale;
            const int n_heads = L::kKeyStationary ? p.hkv : p.hq;
            const int head = L::kKeyStationary ? u.kvh : u.h;
            __nv_bfloat16* dst_row = p.out + ((size_t)row * n_heads + head) * kD + grp * (kD / L::kGroups);
            if (L::kKeyStationary && p.acc32) {      // of a query chunk's blocks this CTA's keys may have seen none
                int lo, hi;
                u.seen_by(rank, lo, hi);
                row_ok = row_ok && lo <= hi;
            }
            float* acc_row = L::kKeyStationary && p.acc32
                                 ? p.acc32 + ((size_t)row * n_heads + head) * kD + grp * (kD / L::kGroups) : nullptr;
#pragma unroll
            for (int c = 0; c < kD / L::kGroups; c += 32) {
                uint32_t v[32];
                tmem_ld32(t_acc + c, v);
                tmem_ld_wait();
                if (acc_row) {   // a key block meets several query chunks: its partial sums are added up in fp32
                    if (row_ok) {
#pragma unroll
                        for (int i = 0; i < 32; i += 4)
                            asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(acc_row + c + i),
                                         "f"(__uint_as_float(v[i])), "f"(__uint_as_float(v[i + 1])),
                                         "f"(__uint_as_float(v[i + 2])), "f"(__uint_as_float(v[i + 3]))
                                         : "memory");
                    }
                } else if (row_ok) {
                    uint4* dst = reinterpret_cast<uint4*>(dst_row + c);
#pragma unroll
                    for (int i = 0; i < 32; i += 8) {
                        uint4 w;
                        w.x = pack_bf16x2(__uint_as_float(v[i]) * mul, __uint_as_float(v[i + 1]) * mul);
                        w.y = pack_bf16x2(__uint_as_float(v[i + 2]) * mul, __uint_as_float(v[i + 3]) * mul);
                        w.z = pack_bf16x2(__uint_as_float(v[i + 4]) * mul, __uint_as_float(v[i + 5]) * mul);
                        w.w = pack_bf16x2(__uint_as_float(v[i + 6]) * mul, __uint_as_float(v[i + 7]) * mul);
                        dst[i >> 3] = w;
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(accfree0);
            ++uc;
        }
    } else if (MODE == FWD) {
        // ---------------- FWD, warps 4-7: the output tile, through the unit's own Q tile (its MMAs have run) and bulk tensor
        // stores, while warps 0-3 are at the next unit's first blocks.  Before there was a second Q tile, and with the rows
        // stored from registers by warps 0-3: 410 us for 5000 tokens in samples of up to 200 at 128 heads, 315 now. ----------------
        const int w = warp - 4;
        const uint32_t t_acc = tmem_base + ((uint32_t)(w * 32) << 16) + kColAcc;
        const uint32_t accfree0 = map_to_rank(bar_accfree, 0);
        Units<MODE> u(p, cta);
        uint32_t uc = 0, lb = 0, lph = 0;
        while (u.next(rank)) {
            if (!warp_wait(bar_accdone, uc & 1, abort_flag) || !warp_wait(&bar_lfull[lb], lph, abort_flag)) break;
            tc_fence_after();
            const float mul = reinterpret_cast<const float*>(smem + L::kStatOff)[lb * kRows + w * 32 + lane];
            if (++lb == 3) { lb = 0; lph ^= 1; }
            uint8_t* stage = smem + L::kSaOff + (uc & 1) * L::kBig + w * 4096;   // 32 rows x 128 bytes of each column half
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t v[64];
                tmem_ld32(t_acc + 64 * c, v);
                tmem_ld32(t_acc + 64 * c + 32, v + 32);
                tmem_ld_wait();
                if (c == 3) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(accfree0);
                }
#pragma unroll
                for (int ch = 0; ch < 8; ++ch) {
                    uint4 x;
                    const uint32_t* o = v + 8 * ch;
                    x.x = pack_bf16x2(__uint_as_float(o[0]) * mul, __uint_as_float(o[1]) * mul);
                    x.y = pack_bf16x2(__uint_as_float(o[2]) * mul, __uint_as_float(o[3]) * mul);
                    x.z = pack_bf16x2(__uint_as_float(o[4]) * mul, __uint_as_float(o[5]) * mul);
                    x.w = pack_bf16x2(__uint_as_float(o[6]) * mul, __uint_as_float(o[7]) * mul);
                    *reinterpret_cast<uint4*>(stage + c * L::kBigHalf + lane * 128 + ((ch ^ (lane & 7)) << 4)) = x;
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    tma_store_3d(&tm_t2, stage + c * L::kBigHalf, 64 * c, u.h, (int)u.r0 + 32 * w);
                    tma_store_commit();
                }
            }
            if (lane == 0) {
                tma_store_wait_read();
                mbar_arrive(&bar_stempty[uc & 1]);
            }
            ++uc;
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }

    // ---------------- teardown ----------------
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && abort_flag[0]) st_cluster(map_to_rank(const_cast<const uint32_t*>(peer_gave_up), rank ^ 1), 1u);
    cluster_sync();      // no role of either CTA runs any more
    if (abort_flag[0] | (int)*peer_gave_up) {   // give-up path: the copies already issued land before the CTAs leave
        if (threadIdx.x == 0) {
            if (rank == 0) {
                // a half that never was issued is counted as arrived, one that the leader had not got to is expected now
                auto land = [&](uint64_t* bar, uint32_t parity, bool mine, bool peers, uint32_t half) {
                    if (!mine) mbar_arrive_expect_tx(bar, half);
                    if (!peers) mbar_complete_tx(bar, half);
                    mbar_wait_drain(bar, parity, kDrainNs);
                };
                open_loads(issued[0], issued[2], L::kStBufs, [](uint32_t m) { return m % L::kStBufs; },
                           [&](uint32_t b, uint32_t parity, bool mine, bool peers) {
                               land(&bar_stfull[b], parity, mine, peers, L::kStationary * L::kBig);
                           });
                open_loads(issued[1], issued[3], N * S, [](uint32_t m) { return stream_barrier(m, N, S); },
                           [&](uint32_t b, uint32_t parity, bool mine, bool peers) {
                               land(&bar_full[b], parity, mine, peers, L::kHalfTile);
                           });
            }
            if (L::kStatBytes > 0)               // issued with the last of a block's tiles, counted by this CTA alone
                open_loads(issued[2 * rank + 1] / N, 0, S, [](uint32_t m) { return m % S; },
                           [&](uint32_t b, uint32_t parity, bool, bool) { mbar_wait_drain(&bar_stat[b], parity, kDrainNs); });
        }
        cluster_sync();  // the leader's wait is for the other CTA's copies, too
    }
    tc_fence_after();
    if (warp == kMmaWarp) tmem_dealloc_pair(tmem_base, 512);
    if (threadIdx.x == 0) {
        p.outcome[cta] = abort_flag[0] ? LIBRA_ERR_TIMEOUT : LIBRA_OK;
        p.busy[2 * cta + 1] = globaltimer_ns();
    }
    if (MODE == DK || MODE == DQ) grid_dep_wait();
}

template <int MODE>
static int launch(const CUtensorMap& sa, const CUtensorMap& sb, const CUtensorMap& t0, const CUtensorMap& t1, const CUtensorMap& t2,
                  const Params& prm, int W, libra_plan* mp, cudaStream_t s) {
    using L = Cfg<MODE>;
    if (!cfg_done(8 + MODE)) {   // per device
        if (cudaFuncSetAttribute(k_attn_d256<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::kBytes) != cudaSuccess)
            return LIBRA_ERR_CUDA;
        cfg_mark(8 + MODE);
    }
    count_launch();
    const unsigned grid = 2 * ((W + 1) / 2);   // a pair of CTAs for every two workers
    mp->n_outcome[MODE] = (int)grid;
    return launch_dependent(k_attn_d256<MODE>, grid, kThreads, L::kBytes, s, sa, sb, t0, t1, t2, prm) == cudaSuccess ? LIBRA_OK
                                                                                                                : LIBRA_ERR_CUDA;
}

}  // namespace d256

// Forward at head_dim 256 over the plan's query-major lists.
int launch_fwd_d256(const void* q, const void* k, const void* v, void* out, float* lse, const libra_plan* plan,
                    const libra_dims* dims, float scale, cudaStream_t s) {
    using namespace d256;
    const PlanDir& d = plan->dir[0];
    CUtensorMap tq, tk, tv, to;   // K by halves of a block's rows, V by halves of its columns, out by a warp's rows
    int rc = make_thd_map(&tq, q, plan->T, dims->hq, kD, kRows);
    if (rc == LIBRA_OK) rc = make_thd_map(&tk, k, plan->T, dims->hkv, kD, kBlk / 2);
    if (rc == LIBRA_OK) rc = make_thd_map(&tv, v, plan->T, dims->hkv, kD, kBlk);
    if (rc == LIBRA_OK) rc = make_thd_map(&to, out, plan->T, dims->hq, kD, 32);
    if (rc != LIBRA_OK) return rc;
    Params prm = {};
    prm.lse = lse;
    prm.cta_offsets = d.d_cta_offsets;
    prm.cta_tiles = d.d_cta_exec;
    prm.tok_start = plan->d_tok_start;
    prm.tok_end = plan->d_tok_end;
    prm.T = plan->T;
    prm.Tpad = (plan->T + 127) / 128 * 128;
    prm.hq = dims->hq; prm.hkv = dims->hkv; prm.H = d.H; prm.W = d.W;
    prm.scale = scale; prm.scale_log2 = scale * 1.4426950408889634f;
    prm.outcome = plan->d_outcome[0]; prm.plan_status = plan->d_status;
    prm.wait_limit_ns = plan->wait_limit_ns; prm.inject_stall = plan->inject_stall;
    prm.busy = d.d_busy;
    return launch<FWD>(tq, tq, tk, tv, to, prm, d.W, const_cast<libra_plan*>(plan), s);
}

// Backward at head_dim 256: the dV and dK passes over the key-major lists, the dQ pass over the query-major lists.
// lse2 / dvec are the row statistics [Hq, Tpad] the caller has computed on the same stream.
int launch_bwd_d256(const void* q, const void* k, const void* v, const void* dout, void* dq, void* dk, void* dv,
                    const float* lse2, const float* dvec, int64_t Tpad, float* dk_acc, float* dv_acc,
                    const libra_plan* plan, const libra_dims* dims, float scale, cudaStream_t s) {
    using namespace d256;
    const PlanDir& dq_dir = plan->dir[0];
    const bool pairs = dk_acc != nullptr;            // key-stationary passes over pair tiles, fp32 accumulators
    const PlanDir& kv_dir = plan->dir[3];            // 256 keys a tile, in pair tiles or key-major
    if (!kv_dir.enabled || (kv_dir.d_u_blk != nullptr) != pairs) return LIBRA_ERR_PLAN_MISMATCH;
    // whole 128-row tiles (stationary), halves of a streamed block's rows (32) and of its columns (64-row boxes)
    CUtensorMap q128, do128, k128, v128, q32, do32, k32, v32, q64, do64, k64;
    int rc = make_thd_map(&q128, q, plan->T, dims->hq, kD, kRows);
    if (rc == LIBRA_OK) rc = make_thd_map(&do128, dout, plan->T, dims->hq, kD, kRows);
    if (rc == LIBRA_OK) rc = make_thd_map(&k128, k, plan->T, dims->hkv, kD, kRows);
    if (rc == LIBRA_OK) rc = make_thd_map(&v128, v, plan->T, dims->hkv, kD, kRows);
    if (rc == LIBRA_OK) rc = make_thd_map(&q32, q, plan->T, dims->hq, kD, kBlk / 2);
    if (rc == LIBRA_OK) rc = make_thd_map(&do32, dout, plan->T, dims->hq, kD, kBlk / 2);
    if (rc == LIBRA_OK) rc = make_thd_map(&k32, k, plan->T, dims->hkv, kD, kBlk / 2);
    if (rc == LIBRA_OK) rc = make_thd_map(&v32, v, plan->T, dims->hkv, kD, kBlk / 2);
    if (rc == LIBRA_OK) rc = make_thd_map(&q64, q, plan->T, dims->hq, kD, kBlk);
    if (rc == LIBRA_OK) rc = make_thd_map(&do64, dout, plan->T, dims->hq, kD, kBlk);
    if (rc == LIBRA_OK) rc = make_thd_map(&k64, k, plan->T, dims->hkv, kD, kBlk);
    if (rc != LIBRA_OK) return rc;
    Params prm = {};
    prm.lse2 = lse2; prm.dvec = dvec;
    prm.tok_start = plan->d_tok_start;
    prm.tok_end = plan->d_tok_end;
    prm.T = plan->T;
    prm.Tpad = Tpad;
    prm.hq = dims->hq; prm.hkv = dims->hkv; prm.H = dq_dir.H; prm.W = dq_dir.W;
    prm.scale = scale; prm.scale_log2 = scale * 1.4426950408889634f;
    prm.outcome = plan->d_outcome[1]; prm.plan_status = plan->d_status;
    prm.wait_limit_ns = plan->wait_limit_ns; prm.inject_stall = plan->inject_stall;
    libra_plan* mp = const_cast<libra_plan*>(plan);
    // dV and dK: key-major lists
    prm.cta_offsets = kv_dir.d_cta_offsets; prm.cta_tiles = kv_dir.d_cta_exec; prm.busy = plan->dir[pairs ? 2 : 1].d_busy2;   // the dK pass runs beside the dV pass and is the one reported
    if (pairs) { prm.u_blk = kv_dir.d_u_blk; prm.u_chunk = kv_dir.d_u_chunk; prm.NU = kv_dir.NB; prm.R = kv_dir.chunk / kRows; }
    time_begin(mp, 1, s);
    prm.out = reinterpret_cast<__nv_bfloat16*>(dv);
    prm.acc32 = dv_acc;
    rc = launch<DV>(k128, k128, q32, do64, do64, prm, plan->W, mp, s);
    prm.out = reinterpret_cast<__nv_bfloat16*>(dk);
    prm.acc32 = dk_acc;
    prm.outcome = plan->d_outcome[2];
    prm.side_by_side = side_by_side(kv_dir.NT, kv_dir.W);
    prm.busy = plan->dir[pairs ? 2 : 1].d_busy;
    if (rc == LIBRA_OK) rc = launch<DK>(k128, v128, q32, do32, q64, prm, plan->W, mp, s);
    time_end(mp, 1, s);
    prm.acc32 = nullptr;
    if (rc != LIBRA_OK) return rc;
    // dQ: query-major lists
    prm.cta_offsets = dq_dir.d_cta_offsets; prm.cta_tiles = dq_dir.d_cta_exec; prm.busy = dq_dir.d_busy2;
    prm.out = reinterpret_cast<__nv_bfloat16*>(dq);
    prm.outcome = plan->d_outcome[3];
    if (dq_in_place(dq, q, dout, dims)) prm.side_by_side = 0;
    time_begin(mp, 2, s);
    rc = launch<DQ>(q128, do128, k32, v32, k64, prm, dq_dir.W, mp, s);
    time_end(mp, 2, s);
    return rc;
}

}  // namespace libra
