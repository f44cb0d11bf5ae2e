// Step sizes of an iteration of the explicit B_perp solver's conjugate gradients from its node sums
// (no CUDA headers: a host compiler can check them).
#pragma once

#ifdef __CUDACC__
#define HQ_HD __host__ __device__ __forceinline__
#else
#define HQ_HD inline
#endif

namespace hq {

struct PcgScalars {
  double alpha, beta, pq;   // p = z + beta p', x += alpha p, and p.Ap
};

// Sums r.z, z.Az and p'.Az of this iteration, (r.z)' and p'.Ap' of the last one (first: there is none).
// p.Ap = z.Az + 2 beta p'.Az + beta^2 p'.Ap'; p'.Ap' is the last iteration's own p.Ap, carried along, not
// summed again over the direction as it was stored, so that with a residual at the floor of its number type
// the terms cancel to something that is only rounding, of either sign.  Below `noise` of the terms the
// iteration starts over along z, whose z.Az is a sum of this iteration.  A zero denominator gives a zero
// step; NaN goes through to the solution, where it is reported.
HQ_HD PcgScalars pcg_scalars(bool first, double rz, double zaz, double paz, double rz_prev, double pq_prev,
                             double noise) {
  PcgScalars s{0.0, 0.0, zaz};
  if (!first && rz_prev != 0.0) {
    s.beta = rz / rz_prev;
    const double b2pq = s.beta * s.beta * pq_prev;
    s.pq += 2.0 * s.beta * paz + b2pq;
    if (zaz > 0.0 && s.pq <= noise * (zaz + (b2pq < 0.0 ? -b2pq : b2pq))) {
      s.beta = 0.0;
      s.pq = zaz;
    }
  }
  s.alpha = s.pq != 0.0 ? rz / s.pq : 0.0;
  return s;
}

}  // namespace hq
