// The plane rotation of the implicit QL iteration on T_k (sweep.cu).
#pragma once
#include <cmath>
#include <cstring>

namespace hs {

// r = |(f, g)|, s = f / r, c = g / r (f = g = 0: all 0). One reciprocal root gives the
// three: 7 FP64 instructions, where a hypot and two divisions are about 35 at 64
// cycles each. Only while f^2 + g^2 is a normal number with room to spare (2^-960
// to 2^1000): beyond, the squares lose bits or overflow, and hypot has the word.
__host__ __device__ inline void ql_rotation(double f, double g, double& r, double& s, double& c) {
  const double rr = f * f + g * g;
#ifdef __CUDA_ARCH__
  const unsigned hi = (unsigned)__double2hiint(rr);
#else
  unsigned long long bits;
  std::memcpy(&bits, &rr, sizeof bits);
  const unsigned hi = (unsigned)(bits >> 32);
#endif
  if ((hi >> 20) - (1023u - 960u) <= 960u + 1000u) {
    const double ir = rsqrt(rr);
    r = rr * ir;
    s = f * ir;
    c = g * ir;
    return;
  }
  r = hypot(f, g);
  s = r == 0.0 ? 0.0 : f / r;
  c = r == 0.0 ? 0.0 : g / r;
}

}  // namespace hs
