// adam_bias.h -- Adam's bias corrections 1 - beta^t (host and device code).
#pragma once
#include <cmath>

#ifdef __CUDACC__
#define MPBP_HD __host__ __device__
#else
#define MPBP_HD
#endif

namespace mpbp {

// 1 - b^t for 0 <= b < 1: binary powers, each kept as an FP64 pair (hi + lo),
// so that the result is good to an ulp or two for every t >= 1; the loop is
// far shorter than the library's pow, whose latency one thread would put in
// front of the whole step (minibatch step 47 -> 26 us with the fusions of the
// Adam form of the object synthesis).  t comes from the caller's state in
// device memory, restored from a checkpoint as it stands, so every value has
// to end: the loop runs over the bits of the unsigned magnitude (64 at most),
// and a negative count answers 1 - 1 / b^|t|, as pow would.
MPBP_HD inline double one_minus_pow(double b, long long t) {
  struct Dd {
    double h, l;
  };
  auto mul = [](Dd x, Dd y) {
    const double p = x.h * y.h;
    const double e = fma(x.h, y.h, -p) + fma(x.h, y.l, x.l * y.h);
    const double h = p + e;
    return Dd{h, e - (h - p)};
  };
  Dd r{1.0, 0.0}, x{b, 0.0};
  for (unsigned long long n = t < 0 ? 0ull - (unsigned long long)t : (unsigned long long)t; n != 0;) {
    if (n & 1) r = mul(r, x);
    n >>= 1;
    if (n != 0) x = mul(x, x);
  }
  return t < 0 ? 1.0 - 1.0 / r.h : (1.0 - r.h) - r.l;
}

}  // namespace mpbp
