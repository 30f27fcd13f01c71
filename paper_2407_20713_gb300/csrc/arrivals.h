// arrivals.h -- meetings of blocks on one 32-bit arrival counter.
#pragma once

#ifdef __CUDACC__
#define SABR_HD __host__ __device__
#else
#define SABR_HD
#endif

namespace sabr {

// Whether `count` arrivals have reached `target`.  Both are running sums modulo
// 2^32 (a meeting's target is the one before plus the number of blocks, and a
// calibration of many levels passes 2^32); they are never more than two
// meetings apart, so the sign of their difference tells.
SABR_HD inline bool arrived(unsigned count, unsigned target) { return (int)(count - target) >= 0; }

}  // namespace sabr
