// lbm_rendezvous.h -- what a rendezvous of a block's warps came to, when each
// warp's wait for the others is bounded.  (Host and device code: tests run the
// rule on the CPU.)
#pragma once

#ifdef __CUDACC__
#define LBM_HOST_DEVICE __host__ __device__
#else
#define LBM_HOST_DEVICE
#endif

namespace lbm {

// A warp whose wait gives up has arrived all the same, so the others may still
// meet after it; what each saw of its own wait must not decide what it does
// next.  One word decides for all: 2 c while rendezvous c (0, 1, ...) is open,
// 2 c + 1 once a warp gave up first, 2 c + 2 once a warp met first (every warp
// has arrived by then, and the word is open for rendezvous c + 1).  cas(expected,
// desired): compare-and-swap on that word, returning its value before.
template <typename Cas>
LBM_HOST_DEVICE inline bool rendezvous_met(bool met, unsigned c, Cas cas) {
    const unsigned open = 2u * c, mine = open + (met ? 2u : 1u);
    const unsigned before = cas(open, mine);
    return (before == open ? mine : before) == open + 2u;
}

}  // namespace lbm
