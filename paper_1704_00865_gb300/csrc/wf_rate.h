// wf_rate.h -- the test of the adaptive cooling rule (Sec. 3.3): over a
// checkpoint of R sweeps Delta d^T Delta d went by the factor q, and lambda is
// lowered if |1 - q^(1/R)| < ratio.  The controller compares q with bounds the
// host computes once, since a power in its one thread is a long dependent
// chain.  Near 1 the bounds are held as their distance from 1: as numbers
// close to 1 they would lose a ratio below 1.1e-16 (and with it a residual
// that no longer changes at all).  Free of CUDA calls, so that it can be
// checked on a host without a GPU.
#pragma once

#include <math.h>

#ifdef __CUDACC__
#define WF_RATE_FN __host__ __device__ inline
#else
#define WF_RATE_FN inline
#endif

namespace wf {

struct RateBounds {
  double lo;              // (1 - ratio)^R, 0 from ratio = 1 on
  double lo_dev, hi_dev;  // (1 -+ ratio)^R - 1
};

inline RateBounds rate_bounds(double ratio, int R) {
  RateBounds b;
  const double l = ratio < 1.0 ? R * log1p(-ratio) : -HUGE_VAL;
  b.lo = exp(l);
  b.lo_dev = expm1(l);
  b.hi_dev = expm1(R * log1p(ratio));
  return b;
}

// false for NaN and for an infinite q
WF_RATE_FN bool rate_below(const RateBounds& b, double q) {
  const double dev = q - 1.0;  // exact from q = 1/2 to 2
  return dev < b.hi_dev && (q >= 0.5 ? dev > b.lo_dev : q > b.lo);
}

}  // namespace wf
