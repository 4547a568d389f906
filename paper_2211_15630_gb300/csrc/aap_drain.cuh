// aap_drain.cuh -- which phase of an mbarrier to wait for, so that a block of
// the surrogate's tensor-core kernels that gave up a wait frees its TMEM only
// after the last MMAs it issued.  Plain integer rules, compiled by the host
// compiler too (the tests check them against a model of the barrier).
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define AAP_HD __host__ __device__
#else
#define AAP_HD
#endif

namespace aaps {

// Parity to wait with for the n-th completion (n >= 1) of a barrier that has
// completed n - 1 or n times: a wait of the other parity returns at once.
AAP_HD constexpr uint32_t nth_parity(int n) { return (uint32_t)(n - 1) & 1u; }

// Commits on the barrier of run t (0 .. 2) of the fused network once layer l
// (1 .. 4) has been issued: one per layer; the last layer has two runs.
AAP_HD constexpr int net_commits(int l, int t) { return l == 4 && t == 2 ? 3 : l; }

}  // namespace aaps
