// Explicit B_perp field solver (Sec. 3.2, "explicit field solver": a Helmholtz-like equation
// instead of the predictor-corrector iterations).
//
// Reading (the paper cites the equation): differentiating the deposited plasma current
// J_perp = sum q w S u_perp / ((1 + Psi) A) along zeta with the particle equations of Sec. 3.2
// gives d(Jx)/d(zeta) = Tx - chi By and d(Jy)/d(zeta) = Ty + chi Bx, with chi the deposited
// susceptibility sum q^2 w S / (M (1 + Psi) A) (B taken at the node) and T the part without
// B_perp: force terms deposited from the gathered ExmBy, EypBx, Ez, Bz, convective terms as
// central differences of the deposited a g^2 u_a u_b, and the beams' central difference of
// their slice deposits.  Eq. bxby then reads
//   (L - chi) Bx = -dy Jz + Ty,   (L - chi) By = dx Jz - Tx,
// solved here by preconditioned conjugate gradients on (chi - L) B = -rhs, preconditioner
// (c - L)^{-1} with c = n0_scale (one shifted DST-I solve per iteration, on the tensor cores in
// FP32 mode), starting from the guess 2 B(i-1) - B(i-2), a fixed number of iterations.
//
// Kernels: the source pass over the plasma particles, and per-node PCG steps (the residual and
// direction vectors are V2 records (Bx, By); the dot products are FP64 sums per iteration and
// right-hand side, accumulated with one atomic per block).
#include <algorithm>
#include <type_traits>

#include "hq_internal.cuh"
#include "pcg_scalars.h"

namespace hq {

namespace {

constexpr int kThreads = 128;

// ---------------------------------------------------------------- source pass
// Per particle at its current (slice i) position: a = q w / A, g = 1 / (1 + Psi),
// Psi' = -(q/M)(g (ux ExmBy + uy EypBx) - Ez),
// Fx = a (g Gx - ux g^2 Psi'), Gx = -(q/M)(gamma g ExmBy + Bz g uy),
// Fy = a (g Gy - uy g^2 Psi'), Gy = -(q/M)(gamma g EypBx - Bz g ux),
// Jxx = a g^2 ux^2, Jxy = a g^2 ux uy, Jyy = a g^2 uy^2, deposited with the particle's shape.
// Written for electrons (q = -1, q/M = -1); a multi-species grid (MS) takes each particle's
// species constants.
template <int P, typename T, bool CACHE, bool MS>
__global__ void __launch_bounds__(kThreads) k_explicit_src(Plasma<T> pl, Geom gm, const T* __restrict__ gf,
                                                           V4<T>* xs4, T* xs1, SpeciesTab tab) {
  pdl_trigger();
  pdl_wait();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= pl.n || !pl.alive[p]) return;
  int sp = 0;
  if constexpr (MS) sp = species_of(tab, p);
  T wx[P + 1], wy[P + 1];
  int ix0, iy0;
  T opp;
  if constexpr (CACHE) {
    const int cell = pl.cell[p];
    ix0 = shape_weights<P, T>(cell & 0xFFFF, T(pl.fx[p]), wx);
    iy0 = shape_weights<P, T>(cell >> 16, T(pl.fy[p]), wy);
    opp = T(pl.opp[p]);
  } else {
    int jx, jy;
    double fx, fy;
    split_coord(pl.x[p], gm.xmin, gm.dx, jx, fx);
    split_coord(pl.y[p], gm.ymin, gm.dy, jy, fy);
    ix0 = shape_weights<P, T>(jx, T(fx), wx);
    iy0 = shape_weights<P, T>(jy, T(fy), wy);
    opp = T(1.0 + pl.psi[p]);
  }
  T E[4] = {T(0), T(0), T(0), T(0)};   // ExmBy, EypBx, Ez, Bz
#pragma unroll
  for (int b = 0; b <= P; ++b) {
    const int iy = iy0 + b;
    if (!in_interior(iy, gm.ny)) continue;
#pragma unroll
    for (int a = 0; a <= P; ++a) {
      const int ix = ix0 + a;
      if (!in_interior(ix, gm.nx)) continue;
      const T* q = gf + ((int64_t)iy * gm.nx + ix) * kGF;
      const T w = wx[a] * wy[b];
#pragma unroll
      for (int c = 0; c < 4; ++c) E[c] += w * q[c];
    }
  }
  const T ux = pl.ux[p], uy = pl.uy[p];
  const T g = T(1) / opp;
  const T gam = (T(1) + ux * ux + uy * uy + opp * opp) * T(0.5) * g;
  // electrons: q = -1, q/M = -1; other species: a = q w / A and the rates scaled by -q/M
  T a, dpsi, gx, gy;
  if constexpr (MS) {
    const T q = sizeof(T) == 8 ? T(tab.q[sp]) : T(tab.fq[sp]);
    const T mqm = sizeof(T) == 8 ? T(-tab.qm[sp]) : T(-tab.fqm[sp]);
    a = sizeof(T) == 8 ? T((tab.q[sp] * (double)pl.w[p]) / (gm.dx * gm.dy)) : q * pl.w[p] * gm.f_inv_area;
    dpsi = mqm * (g * (ux * E[0] + uy * E[1]) - E[2]);
    gx = mqm * (gam * g * E[0] + E[3] * g * uy);
    gy = mqm * (gam * g * E[1] - E[3] * g * ux);
  } else {
    a = sizeof(T) == 8 ? T((-1.0 * (double)pl.w[p]) / (gm.dx * gm.dy)) : -pl.w[p] * gm.f_inv_area;
    dpsi = g * (ux * E[0] + uy * E[1]) - E[2];
    gx = gam * g * E[0] + E[3] * g * uy;
    gy = gam * g * E[1] - E[3] * g * ux;
  }
  const T g2 = g * g;
  const T fx = a * (g * gx - ux * g2 * dpsi), fy = a * (g * gy - uy * g2 * dpsi);
  const T jxx = a * g2 * ux * ux, jxy = a * g2 * ux * uy, jyy = a * g2 * uy * uy;
#pragma unroll
  for (int b = 0; b <= P; ++b) {
    const int iy = iy0 + b;
    if (!in_interior(iy, gm.ny)) continue;
#pragma unroll
    for (int a_ = 0; a_ <= P; ++a_) {
      const int ix = ix0 + a_;
      if (!in_interior(ix, gm.nx)) continue;
      const T w = wx[a_] * wy[b];
      const int64_t node = (int64_t)iy * gm.nx + ix;
      V4<T>* q = xs4 + node;
      if constexpr (sizeof(T) == 4) {
        atomicAdd(reinterpret_cast<float4*>(q), make_float4(w * fx, w * fy, w * jxx, w * jyy));
      } else {
        dadd(&q->a, w * fx, gm);
        dadd(&q->b, w * fy, gm);
        dadd(&q->c, w * jxx, gm);
        dadd(&q->d, w * jyy, gm);
      }
      dadd(xs1 + node, w * jxy, gm);
    }
  }
}

// ---------------------------------------------------------------- PCG on (chi - L) B = -rhs
// chi v - L v from the node's value c and its four neighbours.
template <typename T>
__device__ __forceinline__ V2<T> stencil_A(const Geom& gm, T k, const V2<T>& c, const V2<T>& l, const V2<T>& r,
                                           const V2<T>& d, const V2<T>& u) {
  if constexpr (sizeof(T) == 8) {
    const double dx2 = gm.dx * gm.dx, dy2 = gm.dy * gm.dy;
    return V2<T>{k * c.a - ((r.a - 2.0 * c.a + l.a) / dx2 + (u.a - 2.0 * c.a + d.a) / dy2),
                 k * c.b - ((r.b - 2.0 * c.b + l.b) / dx2 + (u.b - 2.0 * c.b + d.b) / dy2)};
  } else {
    const float ix2 = gm.f_inv_dx * gm.f_inv_dx, iy2 = gm.f_inv_dy * gm.f_inv_dy;
    return V2<T>{k * c.a - ((r.a - 2.0f * c.a + l.a) * ix2 + (u.a - 2.0f * c.a + d.a) * iy2),
                 k * c.b - ((r.b - 2.0f * c.b + l.b) * ix2 + (u.b - 2.0f * c.b + d.b) * iy2)};
  }
}

// A v = chi v - L v at interior node (iy, ix), v(o) the vector at node o (wall nodes read 0; every PCG
// vector is 0 there).
template <typename T, typename F>
__device__ __forceinline__ V2<T> apply_A(F&& v, const T* __restrict__ chi, const Geom& gm, int iy, int ix, const V2<T>& c) {
  const int nx = gm.nx;
  const int64_t o = (int64_t)iy * nx + ix;
  const V2<T> z{T(0), T(0)}, l = v(o - 1), d = v(o - nx);
  const V2<T> r = ix + 1 < nx ? v(o + 1) : z, u = iy + 1 < gm.ny ? v(o + nx) : z;
  return stencil_A<T>(gm, chi[o], c, l, r, d, u);
}

// Block sums of N FP64 values, block of 256 threads: one atomic per block and value into out[i], or
// (part non-null: deterministic FP64 mode) the block's sums stored at part[N * block] for k_ordered_sum.
// The values change hands through shared memory, a warp per value: the FP64 pipe takes a warp
// instruction per 16 clocks of an SM, and N shuffle trees in each of the eight warps are 240 of them for
// N = 6, against 78.
constexpr int kSumThreads = 256;
template <int N>
__device__ __forceinline__ void block_sum(const double* v, double* const* out, double* part_out) {
  __shared__ double part[N][kSumThreads];
#pragma unroll
  for (int i = 0; i < N; ++i) part[i][threadIdx.x] = v[i];
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (w >= N) return;
  double t = 0.0;
  for (int k = lane; k < kSumThreads; k += 32) t += part[w][k];
  for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  if (lane) return;
  if (part_out) part_out[(int64_t)N * blockIdx.x + w] = t;
  else if (t != 0.0) atomicAdd(out[w >> 1] + (w & 1), t);
}

// Sum c = blockIdx.x of the nb blocks' partial sums part[N b + c] in a fixed order (256 threads: strided
// partial sums in increasing b, then a fixed tree): the deterministic mode's dot products.
struct PcgSums { double* out[3]; };   // r.z, z.Az, p.Az: a pair (the right-hand sides) each
__global__ void k_ordered_sum(const double* __restrict__ part, int nb, PcgSums sums) {
  __shared__ double red[256];
  double a = 0.0;
  const int c = blockIdx.x;
  for (int i = threadIdx.x; i < nb; i += 256) a += part[(int64_t)gridDim.x * i + c];
  red[threadIdx.x] = a;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) sums.out[c >> 1][c & 1] = red[0];
}

// Per-node right-hand side of the two Helmholtz-like equations and the initial residual
// r = -rhs - A x0 (x0 = the guess in bm), written to pcg_r and, through the grid's operand
// writer, as the preconditioner solve's sources.  Also resets the slice i-1 record (it receives
// the next slice's deposit), as the predictor-corrector's last source kernel does.
template <typename T> struct PcgInit {
  static constexpr int NR = 2;
  const V4<T>* cur;
  const T* chi;
  const V4<T>* xs4;
  const T* xs1;
  const V2<T>* bjp;
  const V2<T>* bjn;
  const V2<T>* x;
  V2<T>* r;
  V4<T>* prev;
  T* chi_prev;
  float* ps_prev;
  const T* rho_ion;
  Geom gm;
  __device__ void operator()(int iy, int ix, T* v) const {
    const int nx = gm.nx;
    const int64_t o = (int64_t)iy * nx + ix;
    v[0] = v[1] = T(0);
    if (ix > 0 && iy > 0) {
      auto jz = [&](int y, int x_) { return cur[(int64_t)y * nx + x_].d; };
      auto fxx = [&](int y, int x_) { return xs4[(int64_t)y * nx + x_].c; };
      auto fyy = [&](int y, int x_) { return xs4[(int64_t)y * nx + x_].d; };
      auto fxy = [&](int y, int x_) { return xs1[(int64_t)y * nx + x_]; };
      const T i2x = gsel<T>(gm.inv2dx, gm.f_inv2dx), i2y = gsel<T>(gm.inv2dy, gm.f_inv2dy);
      const T i2z = gsel<T>(gm.inv2dz, gm.f_inv2dz);
      const V4<T> s = xs4[o];
      const V2<T> bp = bjp[o], bn = bjn[o];
      const T tx = s.a + dxc(fxx, iy, ix, nx, i2x) + dyc(fxy, iy, ix, gm.ny, i2y) + (bp.a - bn.a) * i2z;
      const T ty = s.b + dxc(fxy, iy, ix, nx, i2x) + dyc(fyy, iy, ix, gm.ny, i2y) + (bp.b - bn.b) * i2z;
      const T rx = -dyc(jz, iy, ix, gm.ny, i2y) + ty;
      const T ry = dxc(jz, iy, ix, nx, i2x) - tx;
      const V2<T> ax = apply_A<T>([&](int64_t i) { return x[i]; }, chi, gm, iy, ix, x[o]);
      v[0] = -rx - ax.a;
      v[1] = -ry - ax.b;
    }
    r[o] = V2<T>{v[0], v[1]};
    prev[o] = V4<T>{rho_ion[o], T(0), T(0), T(0)};
    chi_prev[o] = T(0);
    if (ps_prev) ps_prev[o] = 0.0f;
  }
};

template <typename T, typename Sink>
__global__ void k_pcg_init(PcgInit<T> f, Sink sink) {
  pdl_trigger();
  pdl_wait();
  visit_nodes<2, T>(f.gm, sink, 2, f);
}

// An iteration takes two node passes, with one reduction between them.  z = P r = -(solved) (the shifted
// solve gives (L - c)^{-1} r); with the last direction p' the new one is p = z + beta p', beta =
// (r.z) / (r.z)', and p.Ap = z.Az + 2 beta p'.Az + beta^2 p'.Ap', so that r.z, z.Az and p'.Az are all
// that the node sums have to give: beta is not needed before they are complete.  Forming p first and
// p.Ap from it took four passes (r.z; p; p.Ap; x and r) with a full drain between each two; at 256^2,
// where a pass is launch and latency and not its bytes, a slice (six iterations) took 241 us with four
// launches, 240 with one cooperative launch and three grid barriers, and takes 219 with two.

// First pass: the three sums.  Iteration 0 also clears the consumed source records.
template <typename T>
__global__ void __launch_bounds__(kSumThreads) k_pcg_dots(const T* __restrict__ solved, const V2<T>* __restrict__ r,
                                                  const V2<T>* __restrict__ p_old, const T* __restrict__ chi, Geom gm,
                                                  PcgSums sums, double* part, V4<T>* xs4, T* xs1, V2<T>* bjp, V2<T>* bjn) {
  pdl_trigger();
  pdl_wait();
  const int nx = gm.nx;
  const int64_t nn = (int64_t)nx * gm.ny;
  double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  const auto z = [&](int64_t i) { return V2<T>{-solved[i], -solved[nn + i]}; };
  for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < nn; o += (int64_t)gridDim.x * blockDim.x) {
    const int iy = (int)(o / nx), ix = (int)(o - (int64_t)iy * nx);
    const V2<T> zo = z(o), q = r[o];
    v[0] += (double)q.a * (double)zo.a;
    v[1] += (double)q.b * (double)zo.b;
    if (ix > 0 && iy > 0) {
      const V2<T> az = apply_A<T>(z, chi, gm, iy, ix, zo);
      v[2] += (double)zo.a * (double)az.a;
      v[3] += (double)zo.b * (double)az.b;
      if (p_old) {
        const V2<T> pp = p_old[o];
        v[4] += (double)pp.a * (double)az.a;
        v[5] += (double)pp.b * (double)az.b;
      }
    }
    if (!p_old) {
      xs4[o] = V4<T>{T(0), T(0), T(0), T(0)};
      xs1[o] = T(0);
      bjp[o] = V2<T>{T(0), T(0)};
      bjn[o] = V2<T>{T(0), T(0)};
    }
  }
  block_sum<6>(v, sums.out, part);
}

// z + beta p rounded to T, beta in 64 bits.  FP32: beta = bh + bl, the product and the sum with their
// rounding errors (Dekker's and Knuth's error-free forms), since a node needs its neighbours' values
// too: ten of these per node in FP64 (two conversions, a product and a rounding each, 16 clocks a warp
// instruction), with shuffle trees in the sums, made a slice of 256^2 take 276 us instead of 219.
__device__ __forceinline__ double axpy_rn(double z, double b, double p) { return z + b * p; }
struct Beta32 { float h, l; };
__device__ __forceinline__ float axpy_rn(float z, const Beta32& b, float p) {
  const float m = __fmul_rn(b.h, p), e = __fmaf_rn(b.l, p, __fmaf_rn(b.h, p, -m));
  const float t = __fadd_rn(z, m), u = __fsub_rn(t, z);
  const float d = __fadd_rn(__fsub_rn(z, __fsub_rn(t, u)), __fsub_rn(m, u));
  return __fadd_rn(t, __fadd_rn(d, e));
}

// Second pass: p = z + beta p' (into the other buffer: the neighbours' p' are still read), x += alpha p,
// r -= alpha A p, alpha = (r.z) / (p.Ap) (a zero denominator gives a zero factor); the new r goes to the
// operand writer as the next preconditioner solve's sources.
template <typename T> struct PcgStep {
  static constexpr int NR = 2;
  const T* solved;
  const V2<T>* p_old;        // null: first iteration
  V2<T>* p;
  const T* chi;
  V2<T>* x;
  V2<T>* r;
  PcgSums sums;              // r.z, z.Az, p'.Az
  const double* rz_prev;     // (r.z)', p'.Ap'
  const double* pq_prev;
  double* pq;                // p.Ap, kept for the next iteration
  Geom gm;
  T al[2];
  std::conditional_t<sizeof(T) == 8, double, Beta32> be[2];
  // alpha and beta, by two threads of the block (two divisions each: FP64 work worth doing once)
  __device__ void scalars(bool keep) {
    __shared__ double ab[2][2];
    const int c = threadIdx.x;
    if (c < 2) {
      // (the terms' rounding grows with A's condition: a direction 2^-13 of them in FP32, 2^-40 in FP64, is lost)
      const PcgScalars t = pcg_scalars(!p_old, sums.out[0][c], sums.out[1][c], sums.out[2][c], p_old ? rz_prev[c] : 0.0,
                                       p_old ? pq_prev[c] : 0.0, sizeof(T) == 8 ? 40 : 13);
      ab[0][c] = t.alpha;
      ab[1][c] = t.beta;
      if (keep) pq[c] = t.pq;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      al[i] = T(ab[0][i]);
      const double b = ab[1][i];
      if constexpr (sizeof(T) == 8) be[i] = b;
      else be[i] = Beta32{(float)b, (float)(b - (double)(float)b)};
    }
  }
  __device__ void operator()(int iy, int ix, T* v) const {
    const int64_t o = (int64_t)iy * gm.nx + ix, nn = (int64_t)gm.nx * gm.ny;
    v[0] = v[1] = T(0);
    const auto dir = [&](int64_t i) {
      V2<T> q{-solved[i], -solved[nn + i]};
      if (p_old) {
        const V2<T> w = p_old[i];
        q = V2<T>{axpy_rn(q.a, be[0], w.a), axpy_rn(q.b, be[1], w.b)};
      }
      return q;
    };
    const V2<T> pp = dir(o);
    p[o] = pp;
    if (ix > 0 && iy > 0) {
      const V2<T> ap = apply_A<T>(dir, chi, gm, iy, ix, pp);
      const V2<T> xx = x[o], rr = r[o];
      x[o] = V2<T>{xx.a + al[0] * pp.a, xx.b + al[1] * pp.b};
      v[0] = rr.a - al[0] * ap.a;
      v[1] = rr.b - al[1] * ap.b;
      r[o] = V2<T>{v[0], v[1]};
    }
  }
};

template <typename T, typename Sink>
__global__ void k_pcg_step(PcgStep<T> f, Sink sink) {
  pdl_trigger();
  pdl_wait();
  f.scalars(blockIdx.x == 0 && blockIdx.y == 0);
  visit_nodes<2, T>(f.gm, sink, 2, f);
}

template <typename T> Plasma<T> plasma_of(const hq_grid_s* g);
template <> Plasma<double> plasma_of<double>(const hq_grid_s* g) { return g->p64; }
template <> Plasma<float> plasma_of<float>(const hq_grid_s* g) { return g->p32; }

inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

// pcg_s layout: [which][k][rhs], which 0: r.z, 1: p.Ap, 2: z.Az, 3: p'.Az
inline double* pcg_at(const hq_grid_s* g, int which, int k) { return g->pcg_s + ((size_t)which * kMaxPcg + k) * 2; }

template <typename T>
void launch_explicit_src(const hq_grid_s* g, cudaStream_t s) {
  const unsigned nb = blocks_for(g->np, kThreads);
  const T* gf = reinterpret_cast<const T*>(g->gf);
  V4<T>* xs4 = reinterpret_cast<V4<T>*>(g->xs4);
  T* xs1 = reinterpret_cast<T*>(g->xs1);
  constexpr bool C = sizeof(T) == 4;
  const SpeciesTab& t = g->sp;
#define HQ_XS(P)                                                                                          \
  (g->multi ? launch_pdl(k_explicit_src<P, T, C, true>, nb, kThreads, 0, s, plasma_of<T>(g), g->geom, gf, xs4, xs1, t) \
            : launch_pdl(k_explicit_src<P, T, C, false>, nb, kThreads, 0, s, plasma_of<T>(g), g->geom, gf, xs4, xs1, t))
  switch (g->d.shape_order) {
    case 0: HQ_XS(0); break;
    case 1: HQ_XS(1); break;
    case 2: HQ_XS(2); break;
    default: HQ_XS(3); break;
  }
#undef HQ_XS
}

template <typename T>
void launch_pcg_init(const hq_grid_s* g, int slice, const void* cur, const void* chi_cur, void* prev, void* chi_prev,
                     cudaStream_t s) {
  cudaMemsetAsync(g->pcg_s, 0, sizeof(double) * 4 * kMaxPcg * 2, s);
  PcgInit<T> f{reinterpret_cast<const V4<T>*>(cur), reinterpret_cast<const T*>(chi_cur),
               reinterpret_cast<const V4<T>*>(g->xs4), reinterpret_cast<const T*>(g->xs1),
               reinterpret_cast<const V2<T>*>(bjp_at(g, slice + 1)), reinterpret_cast<const V2<T>*>(g->bjn),
               reinterpret_cast<const V2<T>*>(g->bm), reinterpret_cast<V2<T>*>(g->pcg_r),
               reinterpret_cast<V4<T>*>(prev), reinterpret_cast<T*>(chi_prev), psrc_of(g, prev),
               reinterpret_cast<const T*>(g->rho_ion), g->geom};
  with_sink<T>(g, [&](auto sink) { launch_pdl(k_pcg_init<T, decltype(sink)>, src_grid(g), 128, 0, s, f, sink); });
}

template <typename T>
void launch_pcg_iter(const hq_grid_s* g, int slice, int k, const void* chi_cur, cudaStream_t s) {
  const T* solved = reinterpret_cast<const T*>(g->solved);
  const T* chi = reinterpret_cast<const T*>(chi_cur);
  V2<T>* r = reinterpret_cast<V2<T>*>(g->pcg_r);
  V2<T>* p = reinterpret_cast<V2<T>*>(g->pcg_p) + (k & 1) * (int64_t)g->nnode;   // the two directions, by parity
  const V2<T>* p_old = k > 0 ? reinterpret_cast<V2<T>*>(g->pcg_p) + (~k & 1) * (int64_t)g->nnode : nullptr;
  const PcgSums sums{{pcg_at(g, 0, k), pcg_at(g, 2, k), pcg_at(g, 3, k)}};
  double* part = g->pcg_part;   // deterministic mode: per-block partial sums
  const unsigned nb = pcg_blocks(g->nnode);
  launch_pdl(k_pcg_dots<T>, nb, kSumThreads, 0, s, solved, r, p_old, chi, g->geom, sums, part, reinterpret_cast<V4<T>*>(g->xs4),
             reinterpret_cast<T*>(g->xs1), reinterpret_cast<V2<T>*>(bjp_at(g, slice + 1)), reinterpret_cast<V2<T>*>(g->bjn));
  if (part) k_ordered_sum<<<6, 256, 0, s>>>(part, (int)nb, sums);
  PcgStep<T> f{solved, p_old, p, chi, reinterpret_cast<V2<T>*>(g->bm), r, sums, k > 0 ? pcg_at(g, 0, k - 1) : nullptr,
               k > 0 ? pcg_at(g, 1, k - 1) : nullptr, pcg_at(g, 1, k), g->geom, {}, {}};
  with_sink<T>(g, [&](auto sink) { launch_pdl(k_pcg_step<T, decltype(sink)>, src_grid(g), 128, 0, s, f, sink); });
}

template void launch_explicit_src<float>(const hq_grid_s*, cudaStream_t);
template void launch_explicit_src<double>(const hq_grid_s*, cudaStream_t);
template void launch_pcg_init<float>(const hq_grid_s*, int, const void*, const void*, void*, void*, cudaStream_t);
template void launch_pcg_init<double>(const hq_grid_s*, int, const void*, const void*, void*, void*, cudaStream_t);
template void launch_pcg_iter<float>(const hq_grid_s*, int, int, const void*, cudaStream_t);
template void launch_pcg_iter<double>(const hq_grid_s*, int, int, const void*, cudaStream_t);

}  // namespace hq
