// bin_map.h -- histogram bins of escape steps without FP64 arithmetic (host + device).
#pragma once

#include <cstdint>

#if !defined(FPT_HD)
#if defined(__CUDACC__)
#define FPT_HD __host__ __device__
#else
#define FPT_HD
#endif
#endif

namespace fpt {

// Histogram bins of escape steps in integers.  With t(k) = (x(k) - lo) inv_w in exact arithmetic and
// in units of 2^-32 bins, t is t_first + (k - first) slope 2^-32 to within eps for the `span` steps
// from `first` on; eps also covers the rounding of the FP64 formula that defines the bin, and within
// the span t keeps eps from both ends of the histogram.  So a step whose t is further than eps from
// a whole bin has the formula's bin (the high word of t), steps below k_under / from k_over on are
// outside the histogram, and all others take the formula.  Where there is no such map (a falling or
// constant x, bins narrower than a step) every step does: k_under = 0, k_over = 2^64 - 1, span = 0.
struct BinMap {
    uint64_t k_under, k_over;
    uint64_t t_first, slope;     // 2^-32 and 2^-64 bins
    uint32_t first, span, eps;
};

// Bin of a step below 2^32 by the map; -2: left open.
FPT_HD inline int mapped_bin(const BinMap &m, uint32_t k) {
    const uint32_t j = k - m.first;   // wraps beyond the span below `first`
    const uint64_t t = static_cast<uint64_t>(j) * static_cast<uint32_t>(m.slope >> 32) +
                       (m.t_first + ((static_cast<uint64_t>(j) * static_cast<uint32_t>(m.slope)) >> 32));
    const uint32_t frac = static_cast<uint32_t>(t);
    return j < m.span && frac - m.eps <= ~(2u * m.eps) ? static_cast<int>(t >> 32) : -2;
}

}  // namespace fpt
