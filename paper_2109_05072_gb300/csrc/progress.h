// Progress counters of the persistent kernels.  Plain C++, also compiled by the host tests.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define CEEDGB_HD __host__ __device__
#else
#define CEEDGB_HD
#endif

namespace ceedgb {

// Whether a counter of finished work has reached its target.  The fused PCG iteration counts on from one
// iteration to the next, and a launch may run any number of them, so counter and target are
// taken modulo 2^32; they never lie 2^31 apart (both advance by one iteration's work between two grid barriers).
CEEDGB_HD inline bool progress_reached(uint32_t count, uint32_t target) { return (int32_t)(count - target) >= 0; }

// The counter's value once `per_iteration` pieces of work have been counted in each of it + 1 iterations.
CEEDGB_HD inline uint32_t progress_target(uint32_t per_iteration, uint32_t it) { return per_iteration * (it + 1u); }

}  // namespace ceedgb
