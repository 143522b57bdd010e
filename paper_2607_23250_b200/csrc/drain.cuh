// Loads of a pair of CTAs that may still be in flight when one of them has given up (attn_d256.cu).
//
// Each CTA issues its own half of every load, the leader's barriers count both halves, and the two producers stop where
// their own waits ran out.  A load is numbered by its place in the order that both follow; a barrier's phase for load m is
// only begun when its phase before has completed (the slot has been consumed), so that of each barrier the latest load alone
// can be open, and only if it is among the last `slots` that either CTA has begun.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define LIBRA_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define LIBRA_HOST_DEVICE inline
#endif

namespace libra {

// Calls f(barrier, parity, by_leader, by_peer) for every such load of one kind: `n_leader` and `n_peer` loads have been issued
// by the two CTAs, load m goes to barrier `index(m)` of a ring of `slots` and is its (m / slots)-th phase.
template <typename Index, typename F>
LIBRA_HOST_DEVICE void open_loads(uint32_t n_leader, uint32_t n_peer, uint32_t slots, Index index, F f) {
    const uint32_t most = n_leader > n_peer ? n_leader : n_peer;
    for (uint32_t m = most > slots ? most - slots : 0; m < most; ++m) f(index(m), (m / slots) & 1, m < n_leader, m < n_peer);
}
// Streamed tiles come block by block, `streams` of them each, in a ring of `stages` blocks; barriers are [stream][stage].
LIBRA_HOST_DEVICE uint32_t stream_barrier(uint32_t m, uint32_t streams, uint32_t stages) {
    return m % streams * stages + m / streams % stages;
}

}  // namespace libra
