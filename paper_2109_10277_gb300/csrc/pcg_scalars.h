// Step sizes of an iteration of the explicit B_perp solver's conjugate gradients from its node sums
// (no CUDA headers: a host compiler can check them).
#pragma once

#include <string.h>

#ifdef __CUDACC__
#define HQ_HD __host__ __device__ __forceinline__
#else
#define HQ_HD inline
#endif

namespace hq {

struct PcgScalars {
  double alpha, beta, pq;   // p = z + beta p', x += alpha p, and p.Ap
};

// Sign and exponent word of v, with the top of its fraction: ordered like |v| without the sign, and 2^20
// more for 2 |v|.
HQ_HD int high_word(double v) {
  long long b;
  memcpy(&b, &v, 8);
  return (int)(b >> 32);
}

// Sums r.z, z.Az and p'.Az of this iteration, (r.z)' and p'.Ap' of the last one (first: there is none).
// p.Ap = z.Az + 2 beta p'.Az + beta^2 p'.Ap'; p'.Ap' is the last iteration's own p.Ap, carried along, not
// summed again over the direction as it was stored, so that with a residual at the floor of its number type
// the terms cancel to something that is only rounding, of either sign.  Below 2^-bits of the terms the
// iteration starts over along z, whose z.Az is a sum of this iteration.  (Compared by exponents: the FP64
// pipe takes 0.2 us for the four operations otherwise, and the whole pass waits for them.)  A zero denominator
// gives a zero step; NaN goes through to the solution, where it is reported.
HQ_HD PcgScalars pcg_scalars(bool first, double rz, double zaz, double paz, double rz_prev, double pq_prev, int bits) {
  PcgScalars s{0.0, 0.0, zaz};
  if (!first && rz_prev != 0.0) {
    s.beta = rz / rz_prev;
    const double b2pq = s.beta * s.beta * pq_prev;
    s.pq += 2.0 * s.beta * paz + b2pq;
    const int q = high_word(s.pq), z = high_word(zaz), o = high_word(b2pq) & 0x7fffffff;
    const bool nan = (q & 0x7fffffff) > 0x7ff00000;
    if (z > 0 && !nan && (q < 0 || q <= (z > o ? z : o) - (bits << 20))) {
      s.beta = 0.0;
      s.pq = zaz;
    }
  }
  s.alpha = s.pq != 0.0 ? rz / s.pq : 0.0;
  return s;
}

}  // namespace hq
