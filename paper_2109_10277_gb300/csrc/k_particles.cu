// Plasma particle kernels: initialization, deposition (Sec. 3.2, "current
// deposition": order 0 longitudinally, orders 0-3 transversely, atomics to global
// memory), field gather and the fifth-order Adams-Bashforth push (Sec. 3.2,
// equations for d(x_perp)/d(zeta), d(u_perp)/d(zeta), d(Psi)/d(zeta)).
//
// Layout: structure of arrays, one thread per particle, consecutive threads take
// consecutive particles (coalesced streams).  Deposits go to a packed per-node
// (rho, Jx, Jy, Jz) record with one vector atomic per node in FP32 mode.
//
// FP32 mode keeps x, y and Psi as FP64 accumulators.  The final pass, which
// advances the state, derives each particle's cell index and fractional node
// coordinate (and 1 + Psi, formed in FP64 and rounded once) and caches them, so
// the n_pc trial passes of the predictor-corrector run without FP64 work.
#include "hq_internal.cuh"

namespace hq {

namespace {

// 128 threads per block: with one particle per thread, the finer blocks leave a shorter tail
// of partly filled waves (trial and final passes 2.4 % faster on the blowout512 sweep than 256)
constexpr int kThreads = 128;

__device__ __forceinline__ void atomic_add4(V4<float>* p, float a, float b, float c, float d, const Geom&) {
  atomicAdd(reinterpret_cast<float4*>(p), make_float4(a, b, c, d));
}
__device__ __forceinline__ void atomic_add4(V4<double>* p, double a, double b, double c, double d, const Geom& gm) {
  dadd(&p->a, a, gm);
  dadd(&p->b, b, gm);
  dadd(&p->c, c, gm);
  dadd(&p->d, d, gm);
}
__device__ __forceinline__ void atomic_add2(V2<float>* p, float a, float b, const Geom&) {
  atomicAdd(reinterpret_cast<float2*>(p), make_float2(a, b));
}
__device__ __forceinline__ void atomic_add2(V2<double>* p, double a, double b, const Geom& gm) {
  dadd(&p->a, a, gm);
  dadd(&p->b, b, gm);
}

// Six gathered fields: ExmBy, EypBx, Ez, Bx, By, Bz.
template <typename T> struct F6 { T v[6]; };

// The six fields of one node: ExmBy, EypBx, Ez, Bz from the gather record, Bx, By from the
// B_perp record; o = (ExmBy, EypBx, Ez, Bx, By, Bz).
__device__ __forceinline__ void load_node(const float* q, const float* b, float* o) {
  const float4 a = __ldg(reinterpret_cast<const float4*>(q));
  const float2 c = __ldg(reinterpret_cast<const float2*>(b));
  o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = c.x; o[4] = c.y; o[5] = a.w;
}
__device__ __forceinline__ void load_node(const double* q, const double* b, double* o) {
  const double2 a = __ldg(reinterpret_cast<const double2*>(q));
  const double2 a2 = __ldg(reinterpret_cast<const double2*>(q + 2));
  const double2 c = __ldg(reinterpret_cast<const double2*>(b));
  o[0] = a.x; o[1] = a.y; o[2] = a2.x; o[3] = c.x; o[4] = c.y; o[5] = a2.y;
}

// Interpolate the packed fields at a particle whose x/y stencils start at ix0/iy0.
template <int P, typename T>
__device__ __forceinline__ F6<T> gather6(const T* __restrict__ gf, const T* __restrict__ bm, int nx, int ny, int ix0,
                                         int iy0, const T* wx, const T* wy) {
  F6<T> F;
#pragma unroll
  for (int c = 0; c < 6; ++c) F.v[c] = T(0);
#pragma unroll
  for (int b = 0; b <= P; ++b) {
    const int iy = iy0 + b;
    if (!in_interior(iy, ny)) continue;
#pragma unroll
    for (int a = 0; a <= P; ++a) {
      const int ix = ix0 + a;
      if (!in_interior(ix, nx)) continue;
      T q[6];
      const int64_t node = (int64_t)iy * nx + ix;
      load_node(gf + node * kGF, bm + node * 2, q);
      const T wgt = wx[a] * wy[b];
#pragma unroll
      for (int c = 0; c < 6; ++c) F.v[c] += wgt * q[c];
    }
  }
  return F;
}

__device__ __forceinline__ V2<float> load_b(const float* b) {
  const float2 c = __ldg(reinterpret_cast<const float2*>(b));
  return V2<float>{c.x, c.y};
}
__device__ __forceinline__ V2<double> load_b(const double* b) {
  const double2 c = __ldg(reinterpret_cast<const double2*>(b));
  return V2<double>{c.x, c.y};
}

// Bx, By alone at the same stencil, accumulated node by node as gather6 does.  BATCH: a stencil
// inside the array (wall nodes hold zeros) is read without per-node checks, all loads first; not
// in the FP32 final pass, whose 48 registers it would spill (33 us with the checks, 41 without,
// at 262144 particles, quadratic shape).
template <int P, typename T, bool BATCH = true>
__device__ __forceinline__ V2<T> gather_bperp(const T* __restrict__ bm, int nx, int ny, int ix0, int iy0, const T* wx,
                                              const T* wy) {
  T bx = T(0), by = T(0);
  if (BATCH && ix0 >= 0 && iy0 >= 0 && ix0 + P < nx && iy0 + P < ny) {
    const T* r = bm + ((int64_t)iy0 * nx + ix0) * 2;
    V2<T> c[P + 1][P + 1];
#pragma unroll
    for (int b = 0; b <= P; ++b)
#pragma unroll
      for (int a = 0; a <= P; ++a) c[b][a] = load_b(r + ((int64_t)b * nx + a) * 2);
#pragma unroll
    for (int b = 0; b <= P; ++b)
#pragma unroll
      for (int a = 0; a <= P; ++a) {
        const T wgt = wx[a] * wy[b];
        bx += wgt * c[b][a].a;
        by += wgt * c[b][a].b;
      }
    return V2<T>{bx, by};
  }
#pragma unroll
  for (int b = 0; b <= P; ++b) {
    const int iy = iy0 + b;
    if (!in_interior(iy, ny)) continue;
#pragma unroll
    for (int a = 0; a <= P; ++a) {
      const int ix = ix0 + a;
      if (!in_interior(ix, nx)) continue;
      const V2<T> c = load_b(bm + ((int64_t)iy * nx + ix) * 2);
      const T wgt = wx[a] * wy[b];
      bx += wgt * c.a;
      by += wgt * c.b;
    }
  }
  return V2<T>{bx, by};
}

// ExmBy, EypBx, Ez, Bz alone (B_perp zero).
template <int P>
__device__ __forceinline__ F6<float> gather4(const float* __restrict__ gf, int nx, int ny, int ix0, int iy0, const float* wx,
                                             const float* wy) {
  F6<float> F;
#pragma unroll
  for (int c = 0; c < 6; ++c) F.v[c] = 0.0f;
#pragma unroll
  for (int b = 0; b <= P; ++b) {
    const int iy = iy0 + b;
    if (!in_interior(iy, ny)) continue;
#pragma unroll
    for (int a = 0; a <= P; ++a) {
      const int ix = ix0 + a;
      if (!in_interior(ix, nx)) continue;
      const float4 q = __ldg(reinterpret_cast<const float4*>(gf) + (int64_t)iy * nx + ix);
      const float w = wx[a] * wy[b];
      F.v[0] += w * q.x;
      F.v[1] += w * q.y;
      F.v[2] += w * q.z;
      F.v[5] += w * q.w;
    }
  }
  return F;
}

// zeta-derivatives of a plasma particle, Sec. 3.2; opp = 1 + Psi.  Written for an electron
// (q/M = -1); a multi-species grid (MS) scales the momentum and Psi rates by mqm = -q/M.
template <typename T, bool MS = false>
__device__ __forceinline__ void derivs(T ux, T uy, T opp, const F6<T>& F, T* f, T mqm = T(1)) {
  const T g = T(1) / opp;
  const T gam = (T(1) + ux * ux + uy * uy + opp * opp) * T(0.5) * g;
  const T exmby = F.v[0], eypbx = F.v[1], ez = F.v[2], bx = F.v[3], by = F.v[4], bz = F.v[5];
  f[0] = -ux * g;
  f[1] = -uy * g;
  f[2] = gam * g * exmby + by + bz * g * uy;      // -(q/M)[...] with q/M = -1
  f[3] = gam * g * eypbx - bx - bz * g * ux;
  f[4] = g * (ux * exmby + uy * eypbx) - ez;
  if constexpr (MS) {
    f[2] = mqm * f[2];
    f[3] = mqm * f[3];
    f[4] = mqm * f[4];
  }
}

// The rates that do not depend on B_perp (TrialCache::rate): f_ux = A + m By, f_uy = C - m Bx.
template <typename T, bool MS>
__device__ __forceinline__ V4<T> rates_without_b(T ux, T uy, T opp, const F6<T>& F, T mqm) {
  const T g = T(1) / opp;
  const T gam = (T(1) + ux * ux + uy * uy + opp * opp) * T(0.5) * g;
  V4<T> r{gam * g * F.v[0] + F.v[5] * g * uy, gam * g * F.v[1] - F.v[5] * g * ux,
          g * (ux * F.v[0] + uy * F.v[1]) - F.v[2], g};
  if constexpr (MS) {
    r.a *= mqm;
    r.b *= mqm;
    r.c *= mqm;
  }
  return r;
}

__device__ __forceinline__ int pack_node(int iy, int ix) { return (iy << 16) | (ix & 0xffff); }
__device__ __forceinline__ int node_x(int i) { return (int)(short)(i & 0xffff); }
__device__ __forceinline__ int node_y(int i) { return i >> 16; }

// A particle's species constants on a multi-species grid (MS), else the electron's: -q/M,
// q/M (the chi factor q^2/M over q) and q, in the kernel's type.
template <typename T> struct SpC {
  T mqm, qm, q;
};
template <typename T, bool MS>
__device__ __forceinline__ SpC<T> spc_of(const SpeciesTab& tab, int s) {
  if constexpr (MS) {
    if constexpr (sizeof(T) == 8) return SpC<T>{T(-tab.qm[s]), T(tab.qm[s]), T(tab.q[s])};
    else return SpC<T>{-tab.fqm[s], tab.fqm[s], tab.fq[s]};
  } else {
    return SpC<T>{T(1), T(-1), T(-1)};
  }
}

// AB5 combination sum_k beta_k f_{i-k} for component c; history slots hold f_{i-1..i-4}.
template <typename T>
__device__ __forceinline__ T ab5_comb(const T* __restrict__ hist, int64_t n, int64_t p, int slice,
                                      int c, T f0) {
  T acc = T(ab5(0)) * f0;
#pragma unroll
  for (int k = 1; k <= 4; ++k) {
    const int slot = ((slice - k) % kRing + kRing) % kRing;
    acc += T(ab5(k)) * hist[((int64_t)slot * 5 + c) * n + p];
  }
  return acc;
}

// u_z = (1 + u_perp^2 - (1 + psi)^2) / (2 (1 + psi)) (the quasi-static constant of motion
// gamma - u_z = 1 + psi).  FP64 evaluates it as written (the oracle's arithmetic); FP32 as
// (u_perp^2 - psi (2 + psi)) g / 2 with psi (2 + psi) from the FP64 psi, since in FP32 the
// written form subtracts numbers near 1 and loses the plasma's small u_z.
template <typename T>
__device__ __forceinline__ T uz_of(T ux, T uy, T opp, double psi, T g) {
  if constexpr (sizeof(T) == 8) return (T(1) + ux * ux + uy * uy - opp * opp) * T(0.5) * g;
  else return (ux * ux + uy * uy - T(psi * (2.0 + psi))) * T(0.5) * g;
}

template <int P, typename T>
__device__ __forceinline__ void deposit_full(V4<T>* dep, T* chi, const Geom& gm, int ix0, int iy0,
                                             const T* wx, const T* wy, T rho, T jx, T jy, T jz, T ch) {
  const int nx = gm.nx, ny = gm.ny;
#pragma unroll
  for (int b = 0; b <= P; ++b) {
    const int iy = iy0 + b;
    if (!in_interior(iy, ny)) continue;
#pragma unroll
    for (int a = 0; a <= P; ++a) {
      const int ix = ix0 + a;
      if (!in_interior(ix, nx)) continue;
      const T wgt = wx[a] * wy[b];
      const int64_t node = (int64_t)iy * nx + ix;
      atomic_add4(dep + node, wgt * rho, wgt * jx, wgt * jy, wgt * jz, gm);
      if (chi) dadd(chi + node, wgt * ch, gm);
    }
  }
}

template <int P, typename T>
__device__ __forceinline__ void deposit_perp(V2<T>* tj, const Geom& gm, int ix0, int iy0,
                                             const T* wx, const T* wy, T jx, T jy) {
  const int nx = gm.nx, ny = gm.ny;
  if (ix0 >= 1 && iy0 >= 1 && ix0 + P < nx && iy0 + P < ny) {   // no wall node in the stencil
    V2<T>* r = tj + (int64_t)iy0 * nx + ix0;
#pragma unroll
    for (int b = 0; b <= P; ++b)
#pragma unroll
      for (int a = 0; a <= P; ++a) {
        const T wgt = wx[a] * wy[b];
        atomic_add2(r + (int64_t)b * nx + a, wgt * jx, wgt * jy, gm);
      }
    return;
  }
#pragma unroll
  for (int b = 0; b <= P; ++b) {
    const int iy = iy0 + b;
    if (!in_interior(iy, ny)) continue;
#pragma unroll
    for (int a = 0; a <= P; ++a) {
      const int ix = ix0 + a;
      if (!in_interior(ix, nx)) continue;
      const T wgt = wx[a] * wy[b];
      atomic_add2(tj + (int64_t)iy * nx + ix, wgt * jx, wgt * jy, gm);
    }
  }
}

// Stencil of a position given in FP64 (exact division, as in the oracle).
template <int P, typename T>
__device__ __forceinline__ void stencil_f64(const Geom& gm, double x, double y, int& ix0, int& iy0, T* wx, T* wy) {
  int jx, jy;
  double fx, fy;
  split_coord(x, gm.xmin, gm.dx, jx, fx);
  split_coord(y, gm.ymin, gm.dy, jy, fy);
  ix0 = shape_weights<P, T>(jx, T(fx), wx);
  iy0 = shape_weights<P, T>(jy, T(fy), wy);
}

// q w / A (an electron: q = -1).  FP64 mode divides by A = dx dy as the oracle does; FP32
// mode multiplies by the precomputed 1/A.
template <typename T>
__device__ __forceinline__ T charge_density(T w, const Geom& gm, T q = T(-1)) {
  if constexpr (sizeof(T) == 8) return (q * w) / (gm.dx * gm.dy);
  else return q * w * gm.f_inv_area;
}

// Removal rule (a reading; the paper is silent): finite, inside the open box,
// 1 + Psi >= psi_guard.
__device__ __forceinline__ bool state_ok(const Geom& gm, double x, double y, double opp, double guard) {
  return isfinite(x) && isfinite(y) && isfinite(opp) && x > gm.xmin && x < gm.xmax && y > gm.ymin &&
         y < gm.ymax && opp >= guard;
}

// Plasma particles per cell per axis, with the FP32 and FP64 reciprocals.
struct PpcInfo {
  int px, py;
  int pow2;   // both powers of two: the sub-cell offsets are exact in FP32
  float finv_x, finv_y;
  double inv_x, inv_y;
  double cell_w;   // dx dy / particles per cell
};

// ---------------------------------------------------------------- init
// Placement of plasma particle p (Sec. 2: unperturbed plasma ahead of the beams): cell-row-major,
// ppc_x x ppc_y at sub-cell centres, at rest.  A multi-species grid (MS) places each species'
// block [off[s], off[s + 1]) with that species' particles per cell, profile and density.
template <typename T, bool MS>
__global__ void k_plasma_init(Plasma<T> pl, Geom gm, int ppx, int ppy, const double* prof, int npf,
                              double rmax, double n0s, SpeciesTab tab, PpcInfo pc) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= pl.n) return;
  int64_t lp = p;
  if constexpr (MS) {
    const int s = species_of(tab, p);
    lp = p - tab.off[s];
    ppx = tab.ppx[s];
    ppy = tab.ppy[s];
    prof = tab.prof[s];
    npf = tab.npf[s];
    rmax = tab.rmax[s];
    n0s = tab.n0[s];
    pc.pow2 = tab.pow2[s];
    pc.inv_x = tab.inv_px[s];
    pc.inv_y = tab.inv_py[s];
    pc.cell_w = gm.dx * gm.dy / (double)(ppx * ppy);
  }
  const unsigned ppc = (unsigned)(ppx * ppy), l32 = (unsigned)lp;   // (fewer than 2^31 particles)
  const unsigned c = l32 / ppc;
  const int sub = (int)(l32 - c * ppc);
  const int iy = (int)(c / (unsigned)gm.nx), ix = (int)(c - (unsigned)iy * (unsigned)gm.nx);
  const int sx = sub % ppx, sy = sub / ppx;
  // (particle counts that are powers of two: the reciprocal is exact, and the FP64 pipe, which bounds
  // this kernel, is spared two divisions of ~10 instructions each)
  const double ox = (double)sx + 0.5, oy = (double)sy + 0.5;
  const double x = gm.xmin + ((double)ix + (pc.pow2 ? ox * pc.inv_x : ox / ppx)) * gm.dx;
  const double y = gm.ymin + ((double)iy + (pc.pow2 ? oy * pc.inv_y : oy / ppy)) * gm.dy;
  double dens = 1.0;
  if (prof) {
    const double r = sqrt(x * x + y * y);
    double t = r / rmax * (npf - 1);
    t = fmin(fmax(t, 0.0), (double)(npf - 1));
    int k0 = (int)floor(t);
    k0 = k0 < 0 ? 0 : (k0 > npf - 2 ? npf - 2 : k0);
    const double fr = t - (double)k0;
    dens = prof[k0] * (1.0 - fr) + prof[k0 + 1] * fr;
  }
  pl.x[p] = x;
  pl.y[p] = y;
  pl.psi[p] = 0.0;
  pl.ux[p] = T(0);
  pl.uy[p] = T(0);
  pl.w[p] = T(n0s * dens * pc.cell_w);
  pl.alive[p] = 1;
  if (pl.origin) pl.origin[p] = (int32_t)p;
  for (int k = 0; k < kRing * 5; ++k) pl.hist[(int64_t)k * pl.n + p] = T(0);
  if (pl.hsum)
    for (int c = 0; c < 5; ++c) pl.hsum[(int64_t)c * pl.n + p] = 0.0f;
  if (pl.cell) {
    const double ux = (x - gm.xmin) * gm.inv_dx, uy = (y - gm.ymin) * gm.inv_dy;
    const double jx = floor(ux), jy = floor(uy);
    pl.cell[p] = ((int)jy << 16) | (int)jx;
    pl.fx[p] = (float)(ux - jx);
    pl.fy[p] = (float)(uy - jy);
    pl.opp[p] = 1.0f;
  }
}

// Deposit of the current plasma state (slice 0), or of the immobile background
// rho_ion = -(q w / A) deposited from the initial positions (ion_only; on a multi-species grid
// only the species with a neutralizing background).
template <int P, typename T, bool MS>
__global__ void k_deposit_initial(Plasma<T> pl, Geom gm, V4<T>* dep, T* chi, T* rho_ion, SpeciesTab tab) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= pl.n || !pl.alive[p]) return;
  int s = 0;
  if constexpr (MS) {
    s = species_of(tab, p);
    if (rho_ion && !tab.neutral[s]) return;
  }
  const SpC<T> sc = spc_of<T, MS>(tab, s);
  T wx[P + 1], wy[P + 1];
  int ix0, iy0;
  if constexpr (sizeof(T) == 4) {   // FP32: the cached cell coordinates (no FP64 work)
    const int cell = pl.cell[p];
    ix0 = shape_weights<P, T>(cell & 0xFFFF, pl.fx[p], wx);
    iy0 = shape_weights<P, T>(cell >> 16, pl.fy[p], wy);
  } else {
    stencil_f64<P, T>(gm, pl.x[p], pl.y[p], ix0, iy0, wx, wy);
  }
  const T qw = charge_density<T>(pl.w[p], gm, sc.q);
  if (rho_ion) {
#pragma unroll
    for (int b = 0; b <= P; ++b) {
      const int iy = iy0 + b;
      if (!in_interior(iy, gm.ny)) continue;
#pragma unroll
      for (int a = 0; a <= P; ++a) {
        const int ix = ix0 + a;
        if (!in_interior(ix, gm.nx)) continue;
        dadd(rho_ion + (int64_t)iy * gm.nx + ix, -(wx[a] * wy[b] * qw), gm);
      }
    }
    return;
  }
  const T ux = pl.ux[p], uy = pl.uy[p];
  const T opp = T(1.0 + pl.psi[p]);
  const T g = T(1) / opp;
  const T gam = (T(1) + ux * ux + uy * uy + opp * opp) * T(0.5) * g;
  const T uz = uz_of<T>(ux, uy, opp, pl.psi[p], g);
  deposit_full<P, T>(dep, chi, gm, ix0, iy0, wx, wy, qw * gam * g, qw * ux * g, qw * uy * g,
                     qw * uz * g, qw * sc.qm * g);
}

// FP32 multi-species grids: the initial charge of the species without a neutralizing
// background, sum q w S(x0) / A over their particles, accumulated in FP64 (c0 of the psi source).
template <int P>
__global__ void k_species_c0(Plasma<float> pl, Geom gm, double* out, SpeciesTab tab) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= pl.n) return;
  const int s = species_of(tab, p);
  if (tab.neutral[s]) return;
  double wx[P + 1], wy[P + 1];
  int ix0, iy0;
  stencil_f64<P, double>(gm, pl.x[p], pl.y[p], ix0, iy0, wx, wy);
  const double qw = tab.q[s] * (double)pl.w[p] * gm.inv_area;
#pragma unroll
  for (int b = 0; b <= P; ++b) {
    const int iy = iy0 + b;
    if (!in_interior(iy, gm.ny)) continue;
#pragma unroll
    for (int a = 0; a <= P; ++a) {
      const int ix = ix0 + a;
      if (in_interior(ix, gm.nx)) atomicAdd(out + (int64_t)iy * gm.nx + ix, wx[a] * wy[b] * qw);
    }
  }
}

// ---------------------------------------------------------------- trial pass (predictor-corrector)
// Gather with B^(m-1), AB5 trial step to slice i+1, deposit J_perp of the trial
// particles into tj (Sec. 3.2, predictor-corrector field solver).  A slice's first iteration
// (FM 1) also writes the trial cache that its later iterations (k_trial_lin) and the final pass
// read; FM 3 only writes it (k_trial_lin4 then serves every iteration); FM 0 (HQ_NO_F4CACHE=1)
// evaluates everything in every iteration.
template <int P, typename T, bool CACHE, bool MS, int FM>
__global__ void __launch_bounds__(kThreads) k_trial_pass(Plasma<T> pl, Geom gm, const T* __restrict__ gf, const T* __restrict__ bm,
                                                         V2<T>* tj, int slice, double guard, SpeciesTab tab) {
  pdl_trigger();
  pdl_wait();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= pl.n) return;
  if (!pl.alive[p]) {
    if constexpr (FM != 0) pl.tc.idx[p] = make_int2(0, kNoTrial);
    return;
  }
  const SpC<T> sc = spc_of<T, MS>(tab, MS ? species_of(tab, p) : 0);
  const int64_t n = pl.n;
  T wx[P + 1], wy[P + 1];
  T ex, ey;
  int ix0, iy0;
  T opp;
  int jx = 0, jy = 0;
  T fxr = T(0), fyr = T(0);
  if constexpr (CACHE) {
    const int cell = pl.cell[p];
    jx = cell & 0xFFFF;
    jy = cell >> 16;
    fxr = T(pl.fx[p]);
    fyr = T(pl.fy[p]);
    opp = T(pl.opp[p]);
  } else {
    double dx, dy;
    split_coord(pl.x[p], gm.xmin, gm.dx, jx, dx);
    split_coord(pl.y[p], gm.ymin, gm.dy, jy, dy);
    fxr = T(dx);
    fyr = T(dy);
    opp = T(1.0 + pl.psi[p]);
  }
  ix0 = shape_offset<P, T>(jx, fxr, ex);
  iy0 = shape_offset<P, T>(jy, fyr, ey);
  shape_from_offset<P, T>(ex, wx);
  shape_from_offset<P, T>(ey, wy);
  const T ux = pl.ux[p], uy = pl.uy[p];
  F6<T> F;
  if constexpr (FM == 3) F = gather4<P>(gf, gm.nx, gm.ny, ix0, iy0, wx, wy);
  else F = gather6<P, T>(gf, bm, gm.nx, gm.ny, ix0, iy0, wx, wy);
  const V4<T> r = rates_without_b<T, MS>(ux, uy, opp, F, sc.mqm);
  const T f[5] = {-ux * r.d, -uy * r.d, r.a, r.b, r.c};   // f[2], f[3] without B_perp
  const T dz = CACHE ? T(gm.f_dz) : T(gm.dzeta);
  // AB5 combination beta_0 f_i + sum_{k>=1} beta_k f_{i-k}; FP32 reads the precomputed history part
  auto comb = [&](int c) -> T {
    if constexpr (CACHE) return T(ab5(0)) * f[c] + T(pl.hsum[(int64_t)c * n + p]);
    else return ab5_comb<T>(pl.hist, n, p, slice, c, f[c]);
  };
  const T cx = comb(0);
  const T cy = comb(1);
  const T ax0 = ux - dz * comb(2);   // trial u_perp without B_perp
  const T ay0 = uy - dz * comb(3);
  const T cpsi = comb(4);
  T tex, tey;
  int tix0, tiy0;
  T topp;
  bool ok;
  double tx = 0.0, ty = 0.0, tpsi = 0.0;
  if constexpr (CACHE) {
    // trial step in cell-relative coordinates (FP32 only)
    T ux_ = fxr - T(gm.f_dz_inv_dx) * cx;
    T uy_ = fyr - T(gm.f_dz_inv_dy) * cy;
    const T flx = floor(ux_), fly = floor(uy_);
    const int tjx = jx + (int)flx, tjy = jy + (int)fly;
    ux_ -= flx;
    uy_ -= fly;
    topp = opp - dz * cpsi;
    const T ax = T(tjx) + ux_, ay = T(tjy) + uy_;
    ok = isfinite(ax) && isfinite(ay) && isfinite(topp) && ax > T(0) && ax < T(gm.nx) && ay > T(0) && ay < T(gm.ny) &&
         topp >= T(gm.f_guard);
    tix0 = shape_offset<P, T>(tjx, ux_, tex);
    tiy0 = shape_offset<P, T>(tjy, uy_, tey);
  } else {
    tx = pl.x[p] - (double)dz * (double)cx;
    ty = pl.y[p] - (double)dz * (double)cy;
    tpsi = pl.psi[p] - (double)dz * (double)cpsi;
    topp = T(1.0 + tpsi);
    ok = state_ok(gm, tx, ty, 1.0 + tpsi, guard);
    int tjx, tjy;
    double dx, dy;
    split_coord(tx, gm.xmin, gm.dx, tjx, dx);
    split_coord(ty, gm.ymin, gm.dy, tjy, dy);
    tix0 = shape_offset<P, T>(tjx, T(dx), tex);
    tiy0 = shape_offset<P, T>(tjy, T(dy), tey);
  }
  const T tg = T(1) / topp;
  const T qt = charge_density<T>(pl.w[p], gm, sc.q) * tg;
  const T k = qt * (sc.mqm * dz * T(ab5(0)));
  if constexpr (FM != 0) {
    const TrialCache<T>& tc = pl.tc;
    tc.idx[p] = make_int2(pack_node(iy0, ix0), ok ? pack_node(tiy0, tix0) : kNoTrial);
    tc.e[p] = V2<T>{ex, ey};
    tc.te[p] = V2<T>{tex, tey};
    tc.a[p] = V2<T>{qt * ax0, qt * ay0};
    tc.qt[p] = qt;
    if constexpr (sizeof(T) == 4) {
      tc.f4[p] = make_float4(F.v[0], F.v[1], F.v[2], F.v[5]);
    } else {
      tc.rate[p] = r;
      tc.tg[p] = tg;
      tc.tx[p] = tx;
      tc.ty[p] = ty;
      tc.tpsi[p] = tpsi;
    }
  }
  if constexpr (FM == 3) return;
  if (!ok) return;
  T twx[P + 1], twy[P + 1];
  shape_from_offset<P, T>(tex, twx);
  shape_from_offset<P, T>(tey, twy);
  deposit_perp<P, T>(tj, gm, tix0, tiy0, twx, twy, qt * ax0 - k * F.v[4], qt * ay0 + k * F.v[3]);
}

// The later iterations of a slice: what they share is in the trial cache, so an iteration reads
// 36 B per particle (FP32) instead of 65 B, gathers B_perp and deposits.  FP32 is bound by memory
// latency and the atomics (262144 particles, quadratic: 12.4 -> 9.3 us; 4.2e6, cubic: 161 -> 134 us),
// FP64 by its pipe (100 instead of 300 FP64 instructions: 133 -> 52 us).
template <int P, typename T, bool MS>
__global__ void __launch_bounds__(kThreads) k_trial_lin(TrialCache<T> tc, int64_t n, Geom gm, const T* __restrict__ bm, V2<T>* tj, SpeciesTab tab) {
  pdl_trigger();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  // FP32: the launch before is a solve, and no FP32 solve is launched early (none has the
  // programmatic-serialization attribute): it started after the trial pass that filled the cache
  // had ended, so the cache is read while that solve drains.  (The FP64 solve's launches overlap
  // their predecessors: wait first; an FP32 solve launched early would need that here too.)
  if constexpr (sizeof(T) == 8) pdl_wait();
  const bool in = p < n;
  const int2 idx = in ? tc.idx[p] : make_int2(0, kNoTrial);
  const bool ok = idx.y != kNoTrial;
  V2<T> e{}, te{}, a{};
  T k = T(0);
  if (ok) {
    e = tc.e[p];
    te = tc.te[p];
    a = tc.a[p];
    const SpC<T> sc = spc_of<T, MS>(tab, MS ? species_of(tab, p) : 0);
    k = tc.qt[p] * (sc.mqm * (sizeof(T) == 8 ? T(gm.dzeta) : T(gm.f_dz)) * T(ab5(0)));
  }
  T wx[P + 1], wy[P + 1];
  shape_from_offset<P, T>(e.a, wx);
  shape_from_offset<P, T>(e.b, wy);
  if constexpr (sizeof(T) == 4) pdl_wait();
  if (!ok) return;
  const V2<T> b = gather_bperp<P, T>(bm, gm.nx, gm.ny, node_x(idx.x), node_y(idx.x), wx, wy);
  T twx[P + 1], twy[P + 1];
  shape_from_offset<P, T>(te.a, twx);
  shape_from_offset<P, T>(te.b, twy);
  deposit_perp<P, T>(tj, gm, node_x(idx.y), node_y(idx.y), twx, twy, a.a - k * b.b, a.b + k * b.a);
}

// The same for four particles per cell (one thread per cell's four, consecutive in memory): their
// stencils lie within one window of (P + 2)^2 nodes unless the flow has torn them more than a cell
// apart, so the window's B_perp is read once and every window node takes one atomic, 25 instead of 64
// for the cubic shape.  What bounds the pass is the L2's atomics:
// 4.2e6 particles, cubic: 134 -> 67 us.
template <int P>
__device__ __forceinline__ void window_weights(float e, int off, float* w5) {
  float w[P + 1];
  shape_from_offset<P, float>(e, w);
#pragma unroll
  for (int a = 0; a <= P + 1; ++a) {
    const float w0 = a <= P ? w[a <= P ? a : 0] : 0.0f, w1 = a >= 1 ? w[a >= 1 ? a - 1 : 0] : 0.0f;
    w5[a] = off ? w1 : w0;
  }
}
template <int P>
__global__ void __launch_bounds__(kThreads) k_trial_lin4(TrialCache<float> tc, int64_t n4, Geom gm, const float* __restrict__ bm,
                                                         V2<float>* tj, int first) {
  constexpr int W = P + 2;
  pdl_trigger();
  if (first) pdl_wait();   // the cache is the launch before's
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= n4) return;
  int2 idx[4];
  float2 e[4], te[4], a[4];
  float k[4];
  {
    const int4* pi = reinterpret_cast<const int4*>(tc.idx) + 2 * g;
    const float4* pe = reinterpret_cast<const float4*>(tc.e) + 2 * g;
    const float4* pt = reinterpret_cast<const float4*>(tc.te) + 2 * g;
    const float4* pa = reinterpret_cast<const float4*>(tc.a) + 2 * g;
    const float4 q = reinterpret_cast<const float4*>(tc.qt)[g];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int4 i = pi[h];
      const float4 x = pe[h], y = pt[h], z = pa[h];
      idx[2 * h] = make_int2(i.x, i.y);
      idx[2 * h + 1] = make_int2(i.z, i.w);
      e[2 * h] = make_float2(x.x, x.y);
      e[2 * h + 1] = make_float2(x.z, x.w);
      te[2 * h] = make_float2(y.x, y.y);
      te[2 * h + 1] = make_float2(y.z, y.w);
      a[2 * h] = make_float2(z.x, z.y);
      a[2 * h + 1] = make_float2(z.z, z.w);
    }
    const float f = gm.f_dz * (float)ab5(0);
    k[0] = q.x * f;
    k[1] = q.y * f;
    k[2] = q.z * f;
    k[3] = q.w * f;
    // what a particle that does not deposit left in the cache need not be finite, and a zero weight or current
    // would not keep it out of the window's sums
#pragma unroll
    for (int p = 0; p < 4; ++p)
      if (idx[p].y == kNoTrial) {
        e[p] = te[p] = a[p] = make_float2(0.0f, 0.0f);
        k[p] = 0.0f;
      }
  }
  // windows at the particles and at the trial positions, over the particles that deposit
  int gx = 1 << 20, gy = 1 << 20, tx = 1 << 20, ty = 1 << 20, gx1 = -2, gy1 = -2, tx1 = -2, ty1 = -2;
#pragma unroll
  for (int p = 0; p < 4; ++p)
    if (idx[p].y != kNoTrial) {
      const int x = node_x(idx[p].x), y = node_y(idx[p].x), u = node_x(idx[p].y), v = node_y(idx[p].y);
      gx = min(gx, x); gx1 = max(gx1, x);
      gy = min(gy, y); gy1 = max(gy1, y);
      tx = min(tx, u); tx1 = max(tx1, u);
      ty = min(ty, v); ty1 = max(ty1, v);
    }
  if (gx1 == -2) return;
  const int nx = gm.nx, ny = gm.ny;
  const bool together = gx1 - gx <= 1 && gy1 - gy <= 1 && tx1 - tx <= 1 && ty1 - ty <= 1 && min(gx, tx) >= 1 &&
                        min(gy, ty) >= 1 && max(gx, tx) + W <= nx && max(gy, ty) + W <= ny;
  if (!first) pdl_wait();   // (the cache was filled before the solve in between, see k_trial_lin)
  if (!together) {
#pragma unroll 1
    for (int p = 0; p < 4; ++p) {
      const int64_t q = 4 * g + p;
      const int2 id = tc.idx[q];
      if (id.y == kNoTrial) continue;
      const V2<float> ee = tc.e[q], tt = tc.te[q], aa = tc.a[q];
      const float kk = tc.qt[q] * (gm.f_dz * (float)ab5(0));
      float wx[P + 1], wy[P + 1];
      shape_from_offset<P, float>(ee.a, wx);
      shape_from_offset<P, float>(ee.b, wy);
      const V2<float> b = gather_bperp<P, float>(bm, nx, ny, node_x(id.x), node_y(id.x), wx, wy);
      shape_from_offset<P, float>(tt.a, wx);
      shape_from_offset<P, float>(tt.b, wy);
      deposit_perp<P, float>(tj, gm, node_x(id.y), node_y(id.y), wx, wy, aa.a - kk * b.b, aa.b + kk * b.a);
    }
    return;
  }
  float wx[4][W], wy[4][W], jx[4], jy[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const bool ok = idx[p].y != kNoTrial;
    window_weights<P>(e[p].x, ok ? node_x(idx[p].x) - gx : 0, wx[p]);
    window_weights<P>(e[p].y, ok ? node_y(idx[p].x) - gy : 0, wy[p]);
    jx[p] = jy[p] = 0.0f;   // By, Bx at the particle, then J_perp
  }
  const float2* bw = reinterpret_cast<const float2*>(bm) + (int64_t)gy * nx + gx;
#pragma unroll
  for (int b = 0; b < W; ++b) {
    float2 c[W];
#pragma unroll
    for (int i = 0; i < W; ++i) c[i] = __ldg(bw + (int64_t)b * nx + i);
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      float sx = 0.0f, sy = 0.0f;
#pragma unroll
      for (int i = 0; i < W; ++i) {
        sx += wx[p][i] * c[i].x;
        sy += wx[p][i] * c[i].y;
      }
      jy[p] += wy[p][b] * sx;
      jx[p] += wy[p][b] * sy;
    }
  }
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const bool ok = idx[p].y != kNoTrial;
    window_weights<P>(te[p].x, ok ? node_x(idx[p].y) - tx : 0, wx[p]);
    window_weights<P>(te[p].y, ok ? node_y(idx[p].y) - ty : 0, wy[p]);
    jx[p] = ok ? a[p].x - k[p] * jx[p] : 0.0f;
    jy[p] = ok ? a[p].y + k[p] * jy[p] : 0.0f;
  }
  V2<float>* out = tj + (int64_t)ty * nx + tx;
#pragma unroll
  for (int b = 0; b < W; ++b)
#pragma unroll
    for (int i = 0; i < W; ++i) {
      float sx = 0.0f, sy = 0.0f;
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const float w = wx[p][i] * wy[p][b];
        sx += w * jx[p];
        sy += w * jy[p];
      }
      atomic_add2(out + (int64_t)b * nx + i, sx, sy, gm);
    }
}

// ---------------------------------------------------------------- FP32 psi source
// A plasma particle's share of the psi source rho - J_z (Eq. for psi) is q w S(x): rho_p - J_zp
// = q w (gamma - u_z) / (1 + psi) S with gamma - u_z = 1 + psi.  The FP32 path accumulates the
// source ion-subtracted, q w (S(x) - S(x0)) with x0 the particle's initial position (the ion
// it left behind), so the unit ion background never meets the small plasma response in an
// FP32 sum.  When both stencils share their base node the weight differences are formed as
// exact polynomial differences carrying the factor (x - x0); otherwise the two stencils are
// deposited with opposite signs.  Node coordinates u = (x - x_min) / dx enter split as cell +
// fraction; only the move u - u0 is formed from the FP64 fractions.

// Start (ion) node coordinate of plasma particle p, split as cell + fraction: u0 = cx + fx,
// v0 = cy + fy (the placement of k_plasma_init: 32-bit index arithmetic, the sub-cell offset
// (s + 1/2) / ppc).  With ppc a power of two the FP32 fraction is exact and the FP64 copy its
// widening (one conversion); otherwise the FP64 fraction is computed and rounded.  On this
// GPU every FP64 instruction issues on a slow pipe, so the split keeps them to a minimum.
struct Start {
  int cx, cy;
  float fx, fy;
  double dfx, dfy;
};
__device__ __forceinline__ Start start_coord(int64_t p, const Geom& gm, const PpcInfo& pc) {
  const int pi = (int)p;
  const int ppc = pc.px * pc.py;
  const int c = ppc == 1 ? pi : pi / ppc;
  const int sub = pi - c * ppc;
  Start s;
  s.cy = c / gm.nx;
  s.cx = c - s.cy * gm.nx;
  const int sy = pc.px == 1 ? sub : sub / pc.px, sx = sub - sy * pc.px;
  if (pc.pow2) {
    s.fx = ((float)sx + 0.5f) * pc.finv_x;
    s.fy = ((float)sy + 0.5f) * pc.finv_y;
    s.dfx = (double)s.fx;
    s.dfy = (double)s.fy;
  } else {
    s.dfx = ((double)sx + 0.5) * pc.inv_x;
    s.dfy = ((double)sy + 0.5) * pc.inv_y;
    s.fx = (float)s.dfx;
    s.fy = (float)s.dfy;
  }
  return s;
}

// u - u0 in FP32 for u = j + df (df the FP64 fraction) and the start j0 + df0: the FP64
// fraction difference is exact, so a small move keeps its full relative precision.
__device__ __forceinline__ float move_of(int j, double df, int j0, double df0) {
  return (float)(j - j0) + (float)(df - df0);
}

// Weights w at u = j + d, w0 at u0 = j0 + d0 (bases b, b0) and, when b == b0, dw = w - w0 from
// the polynomial differences (each proportional to dl = u - u0).
template <int P>
__device__ __forceinline__ void weight_diff(int j, float d, int j0, float d0, float dl, float* w, float* w0, float* dw,
                                            int& b, int& b0) {
  b = shape_weights<P, float>(j, d, w);
  b0 = shape_weights<P, float>(j0, d0, w0);
  if (b != b0) return;
  if constexpr (P == 0) {
    dw[0] = 0.0f;
  } else if constexpr (P == 1) {
    dw[0] = -dl;
    dw[1] = dl;
  } else if constexpr (P == 2) {
    // offsets from the shared nearest node: e - e0 = u - u0
    const float s = (d >= 0.5f ? d - 1.0f : d) + (d0 >= 0.5f ? d0 - 1.0f : d0);
    dw[0] = -0.5f * dl * (1.0f - s);
    dw[1] = -dl * s;
    dw[2] = 0.5f * dl * (1.0f + s);
  } else {
    const float s = d + d0, q = d * d + d * d0 + d0 * d0;
    const float a = (1.0f - d) * (1.0f - d) + (1.0f - d) * (1.0f - d0) + (1.0f - d0) * (1.0f - d0);
    const float k = dl * (1.0f / 6.0f);
    dw[0] = -k * a;
    dw[1] = k * (3.0f * q - 6.0f * s);
    dw[2] = k * (3.0f + 3.0f * s - 3.0f * q);
    dw[3] = k * q;
  }
}

template <int P>
__device__ __forceinline__ void add_stencil(float* ps, int nx, int ny, int bx, int by, const float* wx, const float* wy,
                                            float q) {
#pragma unroll
  for (int b = 0; b <= P; ++b) {
    const int iy = by + b;
    if (!in_interior(iy, ny)) continue;
#pragma unroll
    for (int a = 0; a <= P; ++a) {
      const int ix = bx + a;
      if (in_interior(ix, nx)) atomicAdd(ps + (int64_t)iy * nx + ix, q * wx[a] * wy[b]);
    }
  }
}

// Quadratic B-spline B2(t) (t = u - node) and B2(t0 + dl) - B2(t0) for an exact dl: within one
// polynomial piece the difference carries the factor dl; across a piece boundary tb it is split
// there, (B2(t) - B2(tb)) + (B2(tb) - B2(t0)), with t - tb = (t0 - tb) + dl.  t0 (a start offset
// on the half-cell lattice) and tb are exact in FP32, so every factor is formed without
// cancellation.
__device__ __forceinline__ int b2_piece(float t) {
  const float a = fabsf(t);
  return a < 0.5f ? 0 : (a < 1.5f ? (t > 0.0f ? 1 : -1) : (t > 0.0f ? 2 : -2));
}
__device__ __forceinline__ float b2_value(float t) {
  const float a = fabsf(t);
  return a < 0.5f ? 0.75f - t * t : (a < 1.5f ? 0.5f * (1.5f - a) * (1.5f - a) : 0.0f);
}
__device__ __forceinline__ float b2_within(float t, float t0, float dl, int pc) {
  if (pc == 0) return -dl * (t + t0);
  if (pc == 1 || pc == -1) return -0.5f * (pc > 0 ? dl : -dl) * (3.0f - fabsf(t) - fabsf(t0));
  return 0.0f;
}
__device__ __forceinline__ float b2_diff(float t0, float dl) {
  const float t = t0 + dl;
  const int p = b2_piece(t), p0 = b2_piece(t0);
  if (p == p0) return b2_within(t, t0, dl, p);
  const float tb = (float)(p < p0 ? p : p0) + 0.5f;   // adjacent pieces: boundary at lo + 1/2
  return b2_within(t, tb, (t0 - tb) + dl, p) + b2_within(tb, t0, tb - t0, p0);
}

// q w (S(u, v) - S(u0, v0)) into ps; the new position u = jx + fx (FP32 fraction fx, FP64 dfx),
// v = jy + fy, and the start s0.
template <int P>
__device__ __forceinline__ void deposit_psi_src(float* ps, const Geom& gm, int jx, float fx, double dfx, int jy, float fy,
                                                double dfy, const Start& s0, float qw) {
  const float dlx = move_of(jx, dfx, s0.cx, s0.dfx), dly = move_of(jy, dfy, s0.cy, s0.dfy);
  if constexpr (P == 2) {
    // quadratic: the cell-centred start sits on a piece boundary, so the two stencils' bases
    // differ by one for about half the particles; difference over the 4-node union support.
    // With |u - u0| < 1 each node's offset crosses at most one piece boundary (pieces are one
    // cell wide), which b2_diff handles; farther moves take the two-stencil path below.
    // Nearest-node bases: floor(u + 1/2) - 1 = j + [f >= 1/2] - 1.
    const int bx = jx + (fx >= 0.5f ? 1 : 0) - 1, bx0 = s0.cx + (s0.fx >= 0.5f ? 1 : 0) - 1;
    const int by = jy + (fy >= 0.5f ? 1 : 0) - 1, by0 = s0.cy + (s0.fy >= 0.5f ? 1 : 0) - 1;
    if (fabsf(dlx) < 1.0f && fabsf(dly) < 1.0f) {
      const int ux = bx < bx0 ? bx : bx0, uy = by < by0 ? by : by0;
      const float tx0 = (float)(s0.cx - ux) + s0.fx, ty0 = (float)(s0.cy - uy) + s0.fy;   // u0 - ux, v0 - uy
      float wy[4], w0x[4], dwx[4], dwy[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float sx0 = tx0 - (float)k, sy0 = ty0 - (float)k;
        w0x[k] = b2_value(sx0);
        wy[k] = b2_value(sy0 + dly);
        dwx[k] = b2_diff(sx0, dlx);
        dwy[k] = b2_diff(sy0, dly);
      }
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int iy = uy + b;
        if (!in_interior(iy, gm.ny)) continue;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const int ix = ux + a;
          const float val = dwx[a] * wy[b] + w0x[a] * dwy[b];
          if (val != 0.0f && in_interior(ix, gm.nx)) atomicAdd(ps + (int64_t)iy * gm.nx + ix, qw * val);
        }
      }
      return;
    }
  }
  float wx[P + 1], w0x[P + 1], dwx[P + 1], wy[P + 1], w0y[P + 1], dwy[P + 1];
  int bx, bx0, by, by0;
  weight_diff<P>(jx, fx, s0.cx, s0.fx, dlx, wx, w0x, dwx, bx, bx0);
  weight_diff<P>(jy, fy, s0.cy, s0.fy, dly, wy, w0y, dwy, by, by0);
  if (bx == bx0 && by == by0) {
    // S - S0 = (wx - w0x) wy + w0x (wy - w0y)
#pragma unroll
    for (int b = 0; b <= P; ++b) {
      const int iy = by + b;
      if (!in_interior(iy, gm.ny)) continue;
#pragma unroll
      for (int a = 0; a <= P; ++a) {
        const int ix = bx + a;
        if (in_interior(ix, gm.nx)) atomicAdd(ps + (int64_t)iy * gm.nx + ix, qw * (dwx[a] * wy[b] + w0x[a] * dwy[b]));
      }
    }
  } else {
    add_stencil<P>(ps, gm.nx, gm.ny, bx, by, wx, wy, qw);
    add_stencil<P>(ps, gm.nx, gm.ny, bx0, by0, w0x, w0y, -qw);
  }
}

// The ion left behind by a removed particle: -q w S(u0, v0).
template <int P>
__device__ __forceinline__ void deposit_ion_src(float* ps, const Geom& gm, const Start& s0, float qw) {
  float wx[P + 1], wy[P + 1];
  const int bx = shape_weights<P, float>(s0.cx, s0.fx, wx);
  const int by = shape_weights<P, float>(s0.cy, s0.fy, wy);
  add_stencil<P>(ps, gm.nx, gm.ny, bx, by, wx, wy, -qw);
}

// ---------------------------------------------------------------- final pass
// Gather with the converged fields of slice i, store f_i in the AB5 history,
// advance to slice i+1, apply the removal rule and deposit rho, J, chi there.
// Resident CTAs the FP32 final pass is compiled for: the pass is memory-latency bound, and a register
// budget keeps more warps resident than its unconstrained 62 (cubic: 70) registers allow.  Quadratic
// shape, 96 slices of 512^2: 21.85 ms at 48 registers (with 32 bytes of spills) and at 56 (without), 22.14
// at 64.  Linear, 262144 particles: 32.6 us at 48, 27.6 at 56.  Cubic: 64.
template <int P, typename T> constexpr int final_min_blocks() {
  return sizeof(T) == 4 ? 65536 / ((P == 3 ? 64 : P == 2 ? 48 : 56) * kThreads) : 1;
}

// FM 2 (FP32, after a predictor-corrector whose first iteration kept the slice's ExmBy, EypBx,
// Ez, Bz per particle in the trial cache): read those back and gather the converged Bx, By alone.
// QUAD: rho, J and chi are left to k_deposit4 (the five values per particle in the trial cache's f4 and qt,
// which this slice no longer needs).
template <int P, typename T, bool CACHE, bool MS, int FM, bool QUAD = false>
__global__ void __launch_bounds__(kThreads, final_min_blocks<P, T>()) k_final_pass(Plasma<T> pl, Geom gm, const T* __restrict__ gf, const T* __restrict__ bm,
                                                         V4<T>* dep, T* chi, float* ps, PpcInfo pc, int slice,
                                                         double guard, unsigned long long* removed, SpeciesTab tab) {
  pdl_trigger();
  pdl_wait();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= pl.n) return;
  int sp = 0;
  int64_t lp = pl.origin ? (int64_t)pl.origin[p] : p;   // index in the initial placement (of its species)
  if constexpr (MS) {
    sp = species_of(tab, p);
    lp = p - tab.off[sp];
    pc.px = tab.ppx[sp];
    pc.py = tab.ppy[sp];
    pc.pow2 = tab.pow2[sp];
    pc.inv_x = tab.inv_px[sp];
    pc.inv_y = tab.inv_py[sp];
    pc.finv_x = tab.finv_px[sp];
    pc.finv_y = tab.finv_py[sp];
  }
  const SpC<T> sc = spc_of<T, MS>(tab, sp);
  Start s0{};
  if (ps) s0 = start_coord(lp, gm, pc);
  if (!pl.alive[p]) {
    if constexpr (sizeof(T) == 4)
      if (ps) deposit_ion_src<P>(ps, gm, s0, charge_density<T>(pl.w[p], gm, sc.q));
    return;
  }
  const int64_t n = pl.n;
  T wx[P + 1], wy[P + 1];
  int ix0, iy0;
  T opp;
  if constexpr (CACHE) {
    const int cell = pl.cell[p];
    ix0 = shape_weights<P, T>(cell & 0xFFFF, T(pl.fx[p]), wx);
    iy0 = shape_weights<P, T>(cell >> 16, T(pl.fy[p]), wy);
    opp = T(pl.opp[p]);
  } else {
    stencil_f64<P, T>(gm, pl.x[p], pl.y[p], ix0, iy0, wx, wy);
    opp = T(1.0 + pl.psi[p]);
  }
  const T ux = pl.ux[p], uy = pl.uy[p];
  F6<T> F;
  if constexpr (CACHE && FM == 2) {
    const float4 c = pl.tc.f4[p];
    const V2<T> b = gather_bperp<P, T, false>(bm, gm.nx, gm.ny, ix0, iy0, wx, wy);
    F.v[0] = c.x; F.v[1] = c.y; F.v[2] = c.z; F.v[3] = b.a; F.v[4] = b.b; F.v[5] = c.w;
  } else {
    F = gather6<P, T>(gf, bm, gm.nx, gm.ny, ix0, iy0, wx, wy);
  }
  T f[5];
  derivs<T, MS>(ux, uy, opp, F, f, sc.mqm);
  T comb[5];
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    T h[kRing + 1];   // h[k] = f_{i-k}
#pragma unroll
    for (int k = 1; k <= kRing; ++k) h[k] = pl.hist[((int64_t)(((slice - k) % kRing + kRing) % kRing) * 5 + c) * n + p];
    T acc = T(ab5(0)) * f[c];
#pragma unroll
    for (int k = 1; k <= kRing; ++k) acc += T(ab5(k)) * h[k];
    comb[c] = acc;
    if constexpr (CACHE) {
      // history part of the next slice's step: beta_1 f_i + beta_2 f_{i-1} + ... + beta_4 f_{i-3}
      T hn = T(ab5(1)) * f[c];
#pragma unroll
      for (int k = 2; k <= kRing; ++k) hn += T(ab5(k)) * h[k - 1];
      pl.hsum[(int64_t)c * n + p] = float(hn);
    }
  }
  const int slot = slice % kRing;
#pragma unroll
  for (int c = 0; c < 5; ++c) pl.hist[((int64_t)slot * 5 + c) * n + p] = f[c];
  const double dz = gm.dzeta;
  const double nxp = pl.x[p] - dz * (double)comb[0];
  const double nyp = pl.y[p] - dz * (double)comb[1];
  const double npsi = pl.psi[p] - dz * (double)comb[4];
  const T nux = ux - gsel<T>(dz, gm.f_dz) * comb[2];
  const T nuy = uy - gsel<T>(dz, gm.f_dz) * comb[3];
  const double nopp = 1.0 + npsi;
  int jx = 0, jy = 0;           // FP32 path: cell, FP64 and FP32 fraction of the new position
  double dfx = 0.0, dfy = 0.0;
  float frx = 0.0f, fry = 0.0f;
  bool ok;
  if constexpr (CACHE) {
    // the removal rule on the cell and the FP32 fraction: the FP64 pipe bounds this pass with many
    // particles, and the rule's FP64 comparisons were a fifth of its work
    const double ux_ = (nxp - gm.xmin) * gm.inv_dx, uy_ = (nyp - gm.ymin) * gm.inv_dy;
    const double flx = floor(ux_), fly = floor(uy_);
    jx = (int)flx;
    jy = (int)fly;
    dfx = ux_ - flx;
    dfy = uy_ - fly;
    frx = (float)dfx;
    fry = (float)dfy;
    ok = isfinite(frx) && isfinite(fry) && jx >= 0 && jx < gm.nx && jy >= 0 && jy < gm.ny && (jx > 0 || frx > 0.0f) &&
         (jy > 0 || fry > 0.0f) && isfinite((float)nopp) && nopp >= guard;
  } else {
    ok = state_ok(gm, nxp, nyp, nopp, guard);
  }
  if (!ok) {
    pl.alive[p] = 0;
    atomicAdd(removed, 1ull);
    if constexpr (sizeof(T) == 4)
      if (ps) deposit_ion_src<P>(ps, gm, s0, charge_density<T>(pl.w[p], gm, sc.q));
    return;
  }
  pl.x[p] = nxp;
  pl.y[p] = nyp;
  pl.psi[p] = npsi;
  pl.ux[p] = nux;
  pl.uy[p] = nuy;
  T topp;
  if constexpr (CACHE) {
    pl.cell[p] = (jy << 16) | jx;
    pl.fx[p] = frx;
    pl.fy[p] = fry;
    topp = (float)nopp;
    pl.opp[p] = topp;
    ix0 = shape_weights<P, T>(jx, T(frx), wx);
    iy0 = shape_weights<P, T>(jy, T(fry), wy);
  } else {
    topp = T(nopp);
    stencil_f64<P, T>(gm, nxp, nyp, ix0, iy0, wx, wy);
  }
  const T qw = charge_density<T>(pl.w[p], gm, sc.q);
  const T g = T(1) / topp;
  const T gam = (T(1) + nux * nux + nuy * nuy + topp * topp) * T(0.5) * g;
  const T uz = uz_of<T>(nux, nuy, topp, npsi, g);
  if constexpr (QUAD) {
    pl.tc.f4[p] = make_float4(qw * gam * g, qw * nux * g, qw * nuy * g, qw * uz * g);
    pl.tc.qt[p] = qw * sc.qm * g;
  } else {
    deposit_full<P, T>(dep, chi, gm, ix0, iy0, wx, wy, qw * gam * g, qw * nux * g, qw * nuy * g,
                       qw * uz * g, qw * sc.qm * g);
  }
  if constexpr (CACHE)
    if (ps) deposit_psi_src<P>(ps, gm, jx, frx, dfx, jy, fry, dfy, s0, qw);
}

// FP64 after a predictor-corrector: the final step moves x, y and Psi exactly as the trial step
// does (only u_perp sees B_perp), so the new position, its stencil, 1 / (1 + Psi), the removal test
// and the rates without B_perp come from the trial cache; left are the gather of the converged
// B_perp, u_perp, the history and the deposit.  The pass is bound by the FP64 pipe: 145 instead of
// 350 FP64 instructions per particle (155 us -> 85 us at 262144 particles, quadratic shape).
template <int P, bool MS>
__global__ void __launch_bounds__(kThreads) k_final_cached(Plasma<double> pl, Geom gm, const double* __restrict__ bm,
                                                           V4<double>* dep, double* chi, int slice,
                                                           unsigned long long* removed, SpeciesTab tab) {
  pdl_trigger();
  pdl_wait();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, n = pl.n;
  if (p >= n || !pl.alive[p]) return;
  const TrialCache<double>& tc = pl.tc;
  const SpC<double> sc = spc_of<double, MS>(tab, MS ? species_of(tab, p) : 0);
  double wx[P + 1], wy[P + 1];
  const int2 idx = tc.idx[p];
  const V2<double> e = tc.e[p];
  shape_from_offset<P, double>(e.a, wx);
  shape_from_offset<P, double>(e.b, wy);
  const V2<double> b = gather_bperp<P, double>(bm, gm.nx, gm.ny, node_x(idx.x), node_y(idx.x), wx, wy);
  const V4<double> r = tc.rate[p];
  const double ux = pl.ux[p], uy = pl.uy[p];
  const double f[5] = {-ux * r.d, -uy * r.d, r.a + sc.mqm * b.b, r.b - sc.mqm * b.a, r.c};
  const double nux = ux - gm.dzeta * ab5_comb<double>(pl.hist, n, p, slice, 2, f[2]);
  const double nuy = uy - gm.dzeta * ab5_comb<double>(pl.hist, n, p, slice, 3, f[3]);
#pragma unroll
  for (int c = 0; c < 5; ++c) pl.hist[((int64_t)(slice % kRing) * 5 + c) * n + p] = f[c];
  if (idx.y == kNoTrial) {
    pl.alive[p] = 0;
    atomicAdd(removed, 1ull);
    return;
  }
  const double psi = tc.tpsi[p], opp = 1.0 + psi, g = tc.tg[p], qg = tc.qt[p];
  pl.x[p] = tc.tx[p];
  pl.y[p] = tc.ty[p];
  pl.psi[p] = psi;
  pl.ux[p] = nux;
  pl.uy[p] = nuy;
  const V2<double> te = tc.te[p];
  shape_from_offset<P, double>(te.a, wx);
  shape_from_offset<P, double>(te.b, wy);
  const double gam = (1.0 + nux * nux + nuy * nuy + opp * opp) * 0.5 * g;
  const double uz = uz_of<double>(nux, nuy, opp, psi, g);
  deposit_full<P, double>(dep, chi, gm, node_x(idx.y), node_y(idx.y), wx, wy, qg * gam, qg * nux, qg * nuy, qg * uz,
                          qg * sc.qm);
}

// Deposit of rho, J, chi for four particles per cell, one thread per cell's four (see k_trial_lin4): one
// atomic pair per node of the common window instead of one per particle and node (4.2e6 particles,
// cubic: final pass 497 us, with this kernel 348 + 93 us).
template <int P>
__global__ void __launch_bounds__(kThreads) k_deposit4(Plasma<float> pl, int64_t n4, Geom gm, V4<float>* dep, float* chi) {
  constexpr int W = P + 2;
  pdl_trigger();
  pdl_wait();
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= n4) return;
  const uchar4 al = reinterpret_cast<const uchar4*>(pl.alive)[g];
  const bool live[4] = {al.x != 0, al.y != 0, al.z != 0, al.w != 0};
  const int4 c4 = reinterpret_cast<const int4*>(pl.cell)[g];
  const float4 fx4 = reinterpret_cast<const float4*>(pl.fx)[g], fy4 = reinterpret_cast<const float4*>(pl.fy)[g];
  const float4 q4 = reinterpret_cast<const float4*>(pl.tc.qt)[g];
  const int cell[4] = {c4.x, c4.y, c4.z, c4.w};
  const float fx[4] = {fx4.x, fx4.y, fx4.z, fx4.w}, fy[4] = {fy4.x, fy4.y, fy4.z, fy4.w};
  float ch[4] = {q4.x, q4.y, q4.z, q4.w};
  float4 v[4];
  int ix[4], iy[4], gx = 1 << 20, gy = 1 << 20, gx1 = -2, gy1 = -2;
  float ex[4], ey[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    v[p] = pl.tc.f4[4 * g + p];
    ix[p] = shape_offset<P, float>(cell[p] & 0xFFFF, fx[p], ex[p]);
    iy[p] = shape_offset<P, float>(cell[p] >> 16, fy[p], ey[p]);
    if (live[p]) {
      gx = min(gx, ix[p]); gx1 = max(gx1, ix[p]);
      gy = min(gy, iy[p]); gy1 = max(gy1, iy[p]);
    } else {
      // a removed particle's values need not be finite (1 / (1 + Psi) of a step that landed on zero): a
      // zero weight would not keep them out of the window's sums
      v[p] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      ch[p] = ex[p] = ey[p] = 0.0f;
    }
  }
  if (gx1 == -2) return;
  const int nx = gm.nx, ny = gm.ny;
  if (gx1 - gx > 1 || gy1 - gy > 1 || gx < 1 || gy < 1 || gx + W > nx || gy + W > ny) {
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      if (!live[p]) continue;
      float wx[P + 1], wy[P + 1];
      shape_from_offset<P, float>(ex[p], wx);
      shape_from_offset<P, float>(ey[p], wy);
      deposit_full<P, float>(dep, chi, gm, ix[p], iy[p], wx, wy, v[p].x, v[p].y, v[p].z, v[p].w, ch[p]);
    }
    return;
  }
  float wx[4][W], wy[4][W];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    window_weights<P>(ex[p], live[p] ? ix[p] - gx : 0, wx[p]);
    window_weights<P>(ey[p], live[p] ? iy[p] - gy : 0, wy[p]);
  }
#pragma unroll
  for (int b = 0; b < W; ++b)
#pragma unroll
    for (int a = 0; a < W; ++a) {
      float r = 0.0f, jx = 0.0f, jy = 0.0f, jz = 0.0f, c = 0.0f;
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const float w = wx[p][a] * wy[p][b];
        r += w * v[p].x;
        jx += w * v[p].y;
        jy += w * v[p].z;
        jz += w * v[p].w;
        c += w * ch[p];
      }
      const int64_t node = (int64_t)(gy + b) * nx + gx + a;
      atomic_add4(dep + node, r, jx, jy, jz, gm);
      atomicAdd(chi + node, c);
    }
}

template <typename T> Plasma<T> plasma_of(const hq_grid_s* g);
template <> Plasma<double> plasma_of<double>(const hq_grid_s* g) { return g->p64; }
template <> Plasma<float> plasma_of<float>(const hq_grid_s* g) { return g->p32; }

inline unsigned blocks_for(int64_t n) { return (unsigned)((n + kThreads - 1) / kThreads); }

PpcInfo ppc_of(const hq_grid_s* g) {
  PpcInfo pc;
  pc.px = g->d.ppc_x;
  pc.py = g->d.ppc_y;
  pc.pow2 = (pc.px & (pc.px - 1)) == 0 && (pc.py & (pc.py - 1)) == 0;
  pc.inv_x = 1.0 / pc.px;
  pc.inv_y = 1.0 / pc.py;
  pc.finv_x = (float)pc.inv_x;
  pc.finv_y = (float)pc.inv_y;
  pc.cell_w = g->geom.dx * g->geom.dy / (double)(pc.px * pc.py);
  return pc;
}

// One thread per cell's four particles (k_trial_lin4, k_deposit4): 2 x 2 particles per cell of the default
// plasma in its initial order, and enough of them for a quarter of the threads to fill the GPU (trial
// pass, cubic: 65536 particles 10.8 us against 12.1 with quads, 262144: 19.1 and 15.9).
constexpr int64_t kQuadMin = 1 << 18;
bool quads(const hq_grid_s* g) {
  return !g->fp64 && !g->no_f4 && !g->multi && g->d.resort_every == 0 && g->d.ppc_x == 2 && g->d.ppc_y == 2 &&
         g->d.shape_order >= 1 && g->np >= kQuadMin;
}

}  // namespace

// Shape-order and species dispatch of the particle kernels: the default electron plasma runs
// the MS = false instances (electron constants folded in), multi-species grids MS = true.
#define HQ_PDISPATCH(ORDER, MULTI, CALL)                                                  \
  switch ((ORDER) * 2 + ((MULTI) ? 1 : 0)) {                                                \
    case 0: { constexpr int P = 0; constexpr bool M = false; CALL; } break;                 \
    case 1: { constexpr int P = 0; constexpr bool M = true; CALL; } break;                  \
    case 2: { constexpr int P = 1; constexpr bool M = false; CALL; } break;                 \
    case 3: { constexpr int P = 1; constexpr bool M = true; CALL; } break;                  \
    case 4: { constexpr int P = 2; constexpr bool M = false; CALL; } break;                 \
    case 5: { constexpr int P = 2; constexpr bool M = true; CALL; } break;                  \
    case 6: { constexpr int P = 3; constexpr bool M = false; CALL; } break;                 \
    default: { constexpr int P = 3; constexpr bool M = true; CALL; } break;                 \
  }

template <typename T>
void launch_plasma_init(const hq_grid_s* g, cudaStream_t s) {
  const double* prof = g->profile.empty() ? nullptr : g->d_profile;
  if (g->multi)
    k_plasma_init<T, true><<<blocks_for(g->np), kThreads, 0, s>>>(plasma_of<T>(g), g->geom, 1, 1, nullptr, 0, 0.0,
                                                                   0.0, g->sp, PpcInfo{});
  else
    k_plasma_init<T, false><<<blocks_for(g->np), kThreads, 0, s>>>(
        plasma_of<T>(g), g->geom, g->d.ppc_x, g->d.ppc_y, prof, (int)g->profile.size(), g->d.profile_rmax,
        g->d.n0_scale, g->sp, ppc_of(g));
}

template <typename T>
void launch_deposit_initial(const hq_grid_s* g, void* dep, void* chi, int ion_only, cudaStream_t s) {
  const unsigned nb = blocks_for(g->np);
  V4<T>* d = reinterpret_cast<V4<T>*>(dep);
  T* c = reinterpret_cast<T*>(chi);
  T* ion = ion_only ? reinterpret_cast<T*>(g->rho_ion) : nullptr;
  HQ_PDISPATCH(g->d.shape_order, g->multi,
               (k_deposit_initial<P, T, M><<<nb, kThreads, 0, s>>>(plasma_of<T>(g), g->geom, d, c, ion, g->sp)));
}

void launch_species_c0(const hq_grid_s* g, double* out, cudaStream_t s) {
  const unsigned nb = blocks_for(g->np);
  switch (g->d.shape_order) {
    case 0: k_species_c0<0><<<nb, kThreads, 0, s>>>(g->p32, g->geom, out, g->sp); break;
    case 1: k_species_c0<1><<<nb, kThreads, 0, s>>>(g->p32, g->geom, out, g->sp); break;
    case 2: k_species_c0<2><<<nb, kThreads, 0, s>>>(g->p32, g->geom, out, g->sp); break;
    default: k_species_c0<3><<<nb, kThreads, 0, s>>>(g->p32, g->geom, out, g->sp); break;
  }
}

// (quads, their order-3 final pass: two kernels in the slice's first trial pass and in the final pass)
bool quads_final(const hq_grid_s* g, bool f4) { return f4 && quads(g) && g->d.shape_order == 3; }
int trial_launches(const hq_grid_s* g, int iter) { return iter == 0 && quads(g) ? 2 : 1; }
int final_launches(const hq_grid_s* g, bool f4) { return quads_final(g, f4) ? 2 : 1; }

template <typename T>
void launch_trial_pass(const hq_grid_s* g, int slice, int iter, cudaStream_t s) {
  const unsigned nb = blocks_for(g->np);
  const T* gf = reinterpret_cast<const T*>(g->gf);
  const T* bm = reinterpret_cast<const T*>(g->bm);
  V2<T>* tj = reinterpret_cast<V2<T>*>(g->tj);
  constexpr bool C = sizeof(T) == 4;
  const double gd = g->d.psi_guard;
  const Plasma<T> pl = plasma_of<T>(g);
  if constexpr (C)
    if (quads(g)) {
      const unsigned n4 = blocks_for(g->np / 4);
      auto go = [&](auto* prep, auto* lin) {
        if (iter == 0) launch_pdl(prep, nb, kThreads, 0, s, pl, g->geom, gf, bm, tj, slice, gd, g->sp);
        launch_pdl(lin, n4, kThreads, 0, s, pl.tc, g->np / 4, g->geom, bm, tj, iter == 0 ? 1 : 0);
      };
      switch (g->d.shape_order) {
        case 1: go(&k_trial_pass<1, float, true, false, 3>, &k_trial_lin4<1>); break;
        case 2: go(&k_trial_pass<2, float, true, false, 3>, &k_trial_lin4<2>); break;
        default: go(&k_trial_pass<3, float, true, false, 3>, &k_trial_lin4<3>); break;
      }
      return;
    }
  if (!g->no_f4 && iter > 0) {
    HQ_PDISPATCH(g->d.shape_order, g->multi,
                 (launch_pdl(k_trial_lin<P, T, M>, nb, kThreads, 0, s, pl.tc, g->np, g->geom, bm, tj, g->sp)));
    return;
  }
  HQ_PDISPATCH(g->d.shape_order, g->multi,
               (g->no_f4 ? launch_pdl(k_trial_pass<P, T, C, M, 0>, nb, kThreads, 0, s, pl, g->geom, gf, bm, tj, slice,
                                      gd, g->sp)
                         : launch_pdl(k_trial_pass<P, T, C, M, 1>, nb, kThreads, 0, s, pl, g->geom, gf, bm, tj, slice,
                                      gd, g->sp)));
}

template <typename T>
void launch_final_pass(const hq_grid_s* g, int slice, void* dep, void* chi, bool f4, cudaStream_t s) {
  const unsigned nb = blocks_for(g->np);
  const T* gf = reinterpret_cast<const T*>(g->gf);
  const T* bm = reinterpret_cast<const T*>(g->bm);
  V4<T>* d = reinterpret_cast<V4<T>*>(dep);
  T* c = reinterpret_cast<T*>(chi);
  constexpr bool C = sizeof(T) == 4;
  const double gd = g->d.psi_guard;
  unsigned long long* rm = g->d_removed;
  float* ps = psrc_of(g, dep);
  const PpcInfo pc = ppc_of(g);
  if constexpr (C)
    if (quads_final(g, f4)) {   // (lower orders: 95 -> 107, 103 -> 116 us at 2^20 particles)
      const unsigned n4 = blocks_for(g->np / 4);
      auto go = [&](auto* fin, auto* dep4) {
        launch_pdl(fin, nb, kThreads, 0, s, g->p32, g->geom, gf, bm, d, c, ps, pc, slice, gd, rm, g->sp);
        launch_pdl(dep4, n4, kThreads, 0, s, g->p32, g->np / 4, g->geom, d, c);
      };
      go(&k_final_pass<3, float, true, false, 2, true>, &k_deposit4<3>);
      return;
    }
  if constexpr (!C)
    if (f4) {
      HQ_PDISPATCH(g->d.shape_order, g->multi,
                   (launch_pdl(k_final_cached<P, M>, nb, kThreads, 0, s, g->p64, g->geom, bm, d, c, slice, rm, g->sp)));
      return;
    }
  HQ_PDISPATCH(g->d.shape_order, g->multi,
               (f4 && C ? launch_pdl(k_final_pass<P, T, C, M, C ? 2 : 0>, nb, kThreads, 0, s, plasma_of<T>(g), g->geom,
                                     gf, bm, d, c, ps, pc, slice, gd, rm, g->sp)
                        : launch_pdl(k_final_pass<P, T, C, M, 0>, nb, kThreads, 0, s, plasma_of<T>(g), g->geom, gf, bm,
                                     d, c, ps, pc, slice, gd, rm, g->sp)));
}
#undef HQ_PDISPATCH

template void launch_plasma_init<float>(const hq_grid_s*, cudaStream_t);
template void launch_plasma_init<double>(const hq_grid_s*, cudaStream_t);
template void launch_deposit_initial<float>(const hq_grid_s*, void*, void*, int, cudaStream_t);
template void launch_deposit_initial<double>(const hq_grid_s*, void*, void*, int, cudaStream_t);
template void launch_trial_pass<float>(const hq_grid_s*, int, int, cudaStream_t);
template void launch_trial_pass<double>(const hq_grid_s*, int, int, cudaStream_t);
template void launch_final_pass<float>(const hq_grid_s*, int, void*, void*, bool, cudaStream_t);
template void launch_final_pass<double>(const hq_grid_s*, int, void*, void*, bool, cudaStream_t);

}  // namespace hq
