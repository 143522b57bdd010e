// Host-side structures shared by the library's translation units.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "../../include/libra.h"

namespace libra {

// One direction (query-major or key-major) of a plan.  All d_* pointers are device memory.
struct PlanDir {
    int enabled = 0;
    int tile = 0;        // tokens per block
    int H = 0;           // head shards
    int W = 0;           // workers (persistent CTAs)
    int64_t NB = 0;      // blocks
    int64_t NT = 0;      // tiles = NB * H
    int64_t* d_weight_blk = nullptr;   // [NB]  weight of block b (every shard of it)
    int32_t* d_blk_order = nullptr;    // [NB]  blocks by (weight desc, index asc)
    int32_t* d_cta_of_tile = nullptr;  // [NT]
    int32_t* d_pos = nullptr;          // [NT]  position of the tile in its worker's list
    int32_t* d_cta_offsets = nullptr;  // [W+1]
    int32_t* d_cta_tiles = nullptr;    // [NT]  per-worker lists in placement order (the plan proper)
    int32_t* d_cta_exec = nullptr;     // [NT]  the same lists, each re-ordered for execution (head-major)
    int64_t* d_loads = nullptr;        // [W]
    uint64_t* d_busy = nullptr;        // [2*W] (start, end) global-timer stamps of the last run
    uint64_t* d_busy2 = nullptr;       // [2*W] same, for the second kernel that walks this direction (dQ)
    uint32_t* d_tile_ns = nullptr;     // [NT] time the last run spent on each tile (forward / fused backward), ns
    // pair tiles only (key block x query chunk x head): the "blocks" above are pair-blocks
    int chunk = 0;                     // tokens per query chunk
    int32_t* d_u_blk = nullptr;        // [NB] key block of pair-block u
    int32_t* d_u_chunk = nullptr;      // [NB] query chunk of pair-block u
    int32_t* d_first_j = nullptr;      // [chunks] first key block of a query chunk
    int64_t* d_base = nullptr;         // [chunks + 1] its pair-block
};

}  // namespace libra

struct libra_plan {
    int64_t T = 0;
    int n = 0;
    int device = 0;
    int sm_count = 0;
    cudaStream_t stream = nullptr;
    static constexpr int kMaxBlocks = 2;
    void* blocks[kMaxBlocks] = {};   // the device memory all pointers below lead into
    int n_blocks = 0;
    bool plain_memory = false;       // built while its stream was being captured: the blocks are not stream-ordered
    int other_stream = 0;            // built or used on a stream other than the legacy one
    int32_t* d_tok_start = nullptr;  // [T] first token of the sample that holds token t
    int32_t* d_tok_end = nullptr;    // [T] one past the last token of that sample
    int* d_status = nullptr;         // the planner's verdict on cu_seqlens
    // Outcome of each CTA of the last launch of a kernel (0 or LIBRA_ERR_*), written by every CTA when it leaves, so
    // that nothing has to be cleared before a launch: forward; dK/dV, fused or dV pass; dK pass; dQ kernel or pass.
    int* d_outcome[4] = {};          // [W + 1] each: kernels on pairs of CTAs round the workers up to even
    int n_outcome[4] = {};           // CTAs of that launch: clusters leave the last workers out, pairs may add one
    int W = 0;                       // workers of every direction
    int bwd_mask = 0;                // which of d_outcome[1..3] the last backward wrote
    // 0 = query-major, 1 = key-major, 2 = pair tiles (key block x query chunk), 3 = the key-stationary tiles of kernels that
    // run on pairs of CTAs: as 2 when that is there, else as 1, with 256 keys a tile and a worker for every two; 4 = the pair
    // tiles of the fused kernel on pairs of CTAs, 256 keys a tile and the query chunks of 2
    static constexpr int kDirs = 5;
    libra::PlanDir dir[kDirs];
    uint32_t wait_limit_ns = 2000000000u;  // budget of one device-side wait (libra_plan_set_wait_limit_ns)
    int inject_stall = 0;            // test aid: the producer role issues no loads (libra_plan_inject_stall)
    int timing = 0;                  // record events around the main kernels
    // [kernel][slot][begin, end]: a ring of the most recent launches of each kernel (LIBRA_KERNEL_* - 1)
    static constexpr int kTimedKernels = 6, kTimeRing = 64;
    cudaEvent_t ev[kTimedKernels][kTimeRing][2] = {};
    int64_t ev_count[kTimedKernels] = {0, 0, 0, 0, 0, 0};   // launches recorded since timing was switched on
};

namespace libra {
// Per-device one-time kernel configuration (dynamic shared memory size, register-pool check).  The
// attributes are per device, so the flag is kept per device ordinal; `slot` is a small integer the
// caller picks per kernel family.  Returns true when this (device, slot) has been configured.
constexpr int kMaxDevices = 64;
constexpr int kCfgSlots = 16;
bool cfg_done(int slot);
void cfg_mark(int slot);
// LIBRA_ERR_PLAN_MISMATCH when the current device is not the one the plan was built on.
int check_plan_device(const libra_plan* plan);
// Kernel timing (libra_plan_set_timing): events on the launch stream around kernel k (LIBRA_KERNEL_* - 1).
inline void time_begin(libra_plan* p, int k, cudaStream_t s) {
    if (p->timing) cudaEventRecord(p->ev[k][p->ev_count[k] % libra_plan::kTimeRing][0], s);
}
inline void time_end(libra_plan* p, int k, cudaStream_t s) {
    if (p->timing) { cudaEventRecord(p->ev[k][p->ev_count[k] % libra_plan::kTimeRing][1], s); ++p->ev_count[k]; }
}
// Stream-ordered device scratch from a memory pool of the library's own (one per device, made on first use, destroyed
// with the library).  The driver's default pool hands everything back at every synchronisation, after which an
// allocation costs from a hundred microseconds to tens of milliseconds; this one keeps at most kPoolKeep bytes across
// synchronisations and gives back what is above that.
constexpr size_t kPoolKeep = size_t(32) << 20;
cudaError_t scratch_alloc(void** p, size_t bytes, cudaStream_t s);
inline void scratch_free(void* p, cudaStream_t s) { if (p) cudaFreeAsync(p, s); }
extern std::atomic<int64_t> g_launches;
inline void count_launch(int n = 1) { g_launches.fetch_add(n, std::memory_order_relaxed); }
}  // namespace libra

namespace libra {
// bf16 [T, H, d] tensor viewed as (d, H, T); TMA box = 64 columns x 1 head x box_rows tokens,
// 128-byte swizzle, out-of-range rows read as zero.  Defined in attn_fwd.cu.
int make_thd_map(CUtensorMap* m, const void* base, int64_t T, int H, int d, int box_rows);
// fp32 tensor [T, H, d] viewed as (d, H, T); box = box_cols x 1 x box_rows, 128-byte swizzle.
int make_f32_3d_map(CUtensorMap* m, const void* base, int64_t T, int H, int d, int box_cols, int box_rows);
// head_dim 256 (attn_d256.cu): the forward over the plan's query-major lists; the three gradient passes over
// its key-major (dV, dK) and query-major (dQ) lists, given the row statistics lse2 / dvec [Hq, Tpad].
int launch_fwd_d256(const void* q, const void* k, const void* v, void* out, float* lse, const libra_plan* plan,
                    const libra_dims* dims, float scale, cudaStream_t s);
// dk_acc / dv_acc: fp32 accumulators [T, Hkv, 256], zero on entry, when the dV and dK passes are to walk the plan's
// pair tiles (the caller rounds them afterwards); null: key-major tiles, dk / dv written directly.
int launch_bwd_d256(const void* q, const void* k, const void* v, const void* dout, void* dq, void* dk, void* dv,
                    const float* lse2, const float* dvec, int64_t Tpad, float* dk_acc, float* dv_acc,
                    const libra_plan* plan, const libra_dims* dims, float scale, cudaStream_t s);
}  // namespace libra

// Launch whose blocks may start before the kernel ahead of it on the stream is done (programmatic dependent launch):
// launch latency and prologues then overlap that kernel's last blocks.  Every kernel launched so executes
// grid_dep_wait() (ptx.cuh) before it touches anything another kernel writes, or, where it only needs what the kernel
// ahead had itself waited for, before it ends.  A step on 10007 tokens (forward, statistics, fused backward,
// conversion): 175 -> 153 us with the clearing of accumulators and status words moved into those kernels.
template <unsigned CLUSTER = 1, typename... KArgs, typename... Args>
static inline cudaError_t launch_dependent(void (*kernel)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t s,
                                           const Args&... args) {
    cudaLaunchAttribute attrs[2] = {};
    cudaLaunchAttribute& attr = attrs[0];
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    attrs[1].id = cudaLaunchAttributeClusterDimension;
    attrs[1].val.clusterDim.x = CLUSTER;
    attrs[1].val.clusterDim.y = attrs[1].val.clusterDim.z = 1;
    cfg.attrs = attrs;
    cfg.numAttrs = CLUSTER > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

// Whether two backward kernels over the same pool that do not depend on one another run side by side: while the first has
// few tiles for the SMs (`tiles` on `workers`) the second takes the idle ones; beyond that they only push one another's
// tiles out of L2.  Backward of one sample, one after the other and side by side: 4 / 4 heads of 64 on 4096 / 16384 / 65536
// tokens (0.9, 3.5 and 13.8 tiles per worker): 121 -> 74, 597 -> 570, 9060 -> 9155 us; 32 / 1 heads of 256 on 1500 / 65536
// tokens (0.1, 3.5): 1.42 -> 0.88, 246 -> 240 ms; 32 / 8 heads of 256 on 32768 (13.8): 60.2 -> 61.4 ms.
constexpr int64_t kOverlapTiles = 8;   // per worker
inline bool side_by_side(int64_t tiles, int workers) { return tiles <= kOverlapTiles * workers; }
// dq may be written over q or dout: a kernel that writes dq reads of either only the tile it is about to replace, once the
// kernels ahead, which read all of both, are done.  Such a call's dQ kernel waits for them.
inline bool dq_in_place(const void* dq, const void* q, const void* dout, const libra_dims* dims) {
    const uintptr_t n = (uintptr_t)dims->total_tokens * dims->hq * dims->head_dim * 2, a = (uintptr_t)dq;
    auto meets = [&](const void* p) { return a < (uintptr_t)p + n && (uintptr_t)p < a + n; };
    return meets(q) || meets(dout);
}

// setmaxnreg moves registers inside the pool the CTA got at launch (registers per thread as compiled x
// threads): what the shrinking warps release must cover what the growing warps ask for, or the last
// warpgroup to grow waits for ever.  Checked on the host against the compiled register count before the
// first launch, so that a build with other flags fails with an error instead.
template <typename Kernel>
static inline bool regs_pool_ok(Kernel k, int threads_grow, int regs_grow, int threads_shrink, int regs_shrink) {
    cudaFuncAttributes a;
    if (cudaFuncGetAttributes(&a, k) != cudaSuccess) return false;
    const long long released = (long long)(a.numRegs - regs_shrink) * threads_shrink;
    const long long wanted = (long long)(regs_grow - a.numRegs) * threads_grow;
    return a.numRegs >= regs_shrink && wanted <= released;
}
