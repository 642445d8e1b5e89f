// A warp's answer to a wait, as host code and device code take it (no CUDA headers, so
// that the rule can be run on the CPU with 32 threads for lanes).
#pragma once
#ifdef __CUDACC__
#define PTEBD_HD __host__ __device__ __forceinline__
#else
#define PTEBD_HD inline
#endif

namespace ptebd {

// Lanes may poll apart from each other and see a counter or a barrier at different times.
// `seen`: this lane's poll succeeded; wait(): its bounded wait; vote(x): whether x holds on
// every lane, executed by all of them.  Each lane votes the same number of times and gets
// the same answer whatever the lanes have seen: one that went on alone would meet the
// others' vote with the shuffles of the work that follows.
template <typename Vote, typename Wait> PTEBD_HD bool warp_ready(bool seen, Vote&& vote, Wait&& wait) {
    return vote(seen) || vote(seen || wait());
}

}  // namespace ptebd
