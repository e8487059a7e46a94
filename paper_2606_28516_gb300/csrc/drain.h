// How a 2-SM GEMM that gave up lets its copies land (plain C++: the CPU tests compile it too).
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define CM_HD __host__ __device__
#else
#define CM_HD
#endif

namespace cm {

// The full barrier of a stage's k-th use completes after the even CTA's arrival, which expects both CTAs'
// bytes, and those bytes. When the producers stopped after n_even and n_odd stages, a stage that only one of
// them reached lacks the other's part, which the drain supplies before it waits:
struct DrainStep {
    bool arrive;      // the even CTA never arrived: arrive, expecting the odd CTA's bytes
    bool complete;    // the odd CTA's boxes never come: count their bytes as landed
};
CM_HD inline DrainStep drain_step(uint32_t k, uint32_t n_even, uint32_t n_odd) {
    return DrainStep{k >= n_even && k < n_odd, k < n_even && k >= n_odd};
}

}  // namespace cm
