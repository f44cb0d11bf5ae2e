// FP64 DST-I for the plain-double path (Sec. 3.2, fast Poisson solver).
//
// A Dirichlet solve f = (2/nx)(2/ny) S_y [(S_y s S_x) / lambda] S_x takes three launches over
// rows: along x (rows stored transposed), along y twice with the 1/lambda factors between the
// two transforms (a row of one kx never leaves shared memory), and along x again.
//
// n a power of two (k_dst_rows): a transform of two real rows packed as one complex row z.
// With D^0 = z and, at level l (N = n / 2^{l+1}),
//   S_j = D^l_j + D^l_{2N-j} (j < N), S_N = D^l_N,   D^{l+1}_j = D^l_j - D^l_{2N-j},
// the odd multiples of 2^l come from the sums alone: X_{2^l (2m+1)} = sum_{j=1..N} S_j
// sin(pi j (2m+1) / (2N)), a DST-III of N points, which one complex FFT of N points gives:
//   u_0 = S_N, u_k = exp(i pi k / 2N) (S_{N-k} - i S_k) / 2,  T = FFT(u) (positive sign),
//   X_{2^l (2m+1)} = T_{m/2} (m even), -T_{N-(m+1)/2} (m odd).
// The FFTs of all levels (N/2 + N/4 + ... points, level N at [N, 2N) of one array) run side by
// side, two radix-2 steps per pass in registers, each butterfly as six fused multiply-adds.
//
// What bounds it: the FP64 pipe (2 fused multiply-adds per SM and clock on this GPU), so the
// operation count decides: 16e3 FP64 instructions per pair of rows at n = 512 against 45e3 for
// the radix-2 FFT over the odd extension of 2n points used before, whose 64 CTAs per pass also
// left most of the 152 SMs idle; one pair of rows per CTA (or one pair per right-hand side where
// the sources or the mixing are fused) spreads a pass over all of them.  512 x 512, two
// right-hand sides: 466 us before, 103 us now.  No prefix sums (the short DST-I via an n-point
// real FFT needs them), so the rounding error stays that of an FFT (1.7e-15 both).
//
// n <= 64 (dst_direct): the folded sums directly, one thread per output and row.  A 64 x 64 sweep
// of 64 slices: 25.9 ms before, 19.3 ms with the fast transform, 11.1 ms with the direct sums.
//
// Other n: k_dst_sums64, the sine sums over the folded pairs (x_j + x_{n-j} for odd k,
// x_j - x_{n-j} for even k: half the terms).  The FP32 path uses tensor cores instead.
#include <atomic>

#include "hq_internal.cuh"

namespace hq {

namespace {

// ---------------------------------------------------------------- rows of a power of two
struct RowsArgs {
  int n, logn, M;          // row length, its log2, rows per right-hand side
  const double* tab;       // cos(pi t / n), -sin(pi t / n) pairs, t < n; n <= kDirect: the sine table
  const double* scale;     // TWICE: [M][n] factors between the two transforms
};

// Where the levels' FFTs keep X_k (k in [1, n)), and whether with the opposite sign.
__device__ __forceinline__ int dst_slot(int n, int k, bool& neg) {
  const int l = __ffs(k) - 1, m = (k >> l) >> 1, N = n >> (l + 1);
  neg = (m & 1) != 0;
  return N + (neg ? N - ((m + 1) >> 1) : (m >> 1));
}

// A: the complex row z (index 0 ignored); on return B holds the FFTs of all levels (2 X_k at
// dst_slot).  n >= 128.  Called by the tp threads of one pair (tid < tp); synchronizes the block.
// An FP64 instruction costs a warp the same 64 clocks whatever number of its lanes take part, so
// the levels of 8 points and fewer (15 outputs, n = 512: a third of the folds) are summed
// directly, one lane per output and row.
__device__ __forceinline__ void dst_pair(double2* A, double2* B, const double2* tw, int n, int logn, int tid, int tp) {
  // folds: level sums into B (bit-reversed within the level), differences back into A
  for (int l = 0; (n >> (l + 1)) >= 16; ++l) {
    const int N = n >> (l + 1), lb = logn - 1 - l;
    for (int i = tid; 2 * i < N; i += tp) {
      const int k = i + 1;
      if (2 * k == N) {
        // k = 0 and k = N / 2 (2 u = sqrt(2) S there)
        const double2 z = A[N], z1 = A[k], z2 = A[k + N];
        const double q = 1.4142135623730950488;
        B[N] = make_double2(2.0 * z.x, 2.0 * z.y);
        B[N + 1] = make_double2(q * (z1.x + z2.x), q * (z1.y + z2.y));
        A[k] = make_double2(z1.x - z2.x, z1.y - z2.y);
        continue;
      }
      const double2 z1 = A[k], z2 = A[2 * N - k], z3 = A[N - k], z4 = A[N + k], w = tw[k << l];
      const double sx = z1.x + z2.x, sy = z1.y + z2.y, tx = z3.x + z4.x, ty = z3.y + z4.y;   // S_k, S_{N-k}
      const double vx = tx + sy, vy = ty - sx, qx = sx + ty, qy = sy - tx;
      const int rk = (int)(__brev((unsigned)k) >> (32 - lb)), rm = (int)(__brev((unsigned)(N - k)) >> (32 - lb));
      B[N + rk] = make_double2(w.x * vx - w.y * vy, w.x * vy + w.y * vx);
      B[N + rm] = make_double2(w.y * qx - w.x * qy, w.y * qy + w.x * qx);
      A[k] = make_double2(z1.x - z2.x, z1.y - z2.y);
      A[N - k] = make_double2(z3.x - z4.x, z3.y - z4.y);
    }
    __syncthreads();
  }
  // (a, b) <- (a + w b, a - w b)
  auto bf = [](double2& a, double2& b, double wx, double wy) {
    const double x = fma(-wy, b.y, fma(wx, b.x, a.x)), y = fma(wy, b.x, fma(wx, b.y, a.y));
    b = make_double2(fma(2.0, a.x, -x), fma(2.0, a.y, -y));
    a = make_double2(x, y);
  };
  // two radix-2 steps (half widths h and 2h) per pass; group t of level N = 4 << floor(log2 t)
  for (int s = 0; (1 << s) < (n >> 1); s += 2) {
    const int h = 1 << s;
    for (int t = tid; t < (n >> 2); t += tp) {
      if (t < 4) continue;
      const int hb = 31 - __clz(t), N = 4 << hb, b = t - (1 << hb);
      if (N >= 4 * h) {
        const int pos = b & (h - 1);
        double2* x = B + N + ((b >> s) << (s + 2)) + pos;
        double2 x0 = x[0], x1 = x[h], x2 = x[2 * h], x3 = x[3 * h];
        if (s == 0) {
          const double2 a = make_double2(x0.x + x1.x, x0.y + x1.y), c = make_double2(x0.x - x1.x, x0.y - x1.y);
          const double2 d = make_double2(x2.x + x3.x, x2.y + x3.y), e = make_double2(x2.x - x3.x, x2.y - x3.y);
          x0 = make_double2(a.x + d.x, a.y + d.y);
          x2 = make_double2(a.x - d.x, a.y - d.y);
          x1 = make_double2(c.x - e.y, c.y + e.x);
          x3 = make_double2(c.x + e.y, c.y - e.x);
        } else {
          const double2 w1 = tw[pos << (logn - s)], w2 = tw[pos << (logn - s - 1)];
          bf(x0, x1, w1.x, w1.y);
          bf(x2, x3, w1.x, w1.y);
          bf(x0, x2, w2.x, w2.y);
          bf(x1, x3, -w2.y, w2.x);   // w2 exp(i pi / 2)
        }
        x[0] = x0;
        x[h] = x1;
        x[2 * h] = x2;
        x[3 * h] = x3;
      } else if (N == 2 * h) {
        // the last step of a level with an odd number of steps: two butterflies
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int pos = b + q * (N >> 2);
          const double2 w = tw[pos << (logn - s)];
          double2 x0 = B[N + pos], x1 = B[N + pos + h];
          bf(x0, x1, w.x, w.y);
          B[N + pos] = x0;
          B[N + pos + h] = x1;
        }
      }
    }
    if (s == 0 && tid < 30) {
      // the remaining DST-I of 16 points: X_{k n / 16}, k = 1 .. 15, of row tid & 1
      const int k = 1 + (tid >> 1), st = n >> 4;
      const double* a = reinterpret_cast<const double*>(A) + (tid & 1);
      double v = 0.0;
#pragma unroll
      for (int j = 1; j < 16; ++j) {
        const int t = (j * k) & 31;
        const double sn = tw[(t & 15) * st].y;
        v = fma(a[2 * j], t & 16 ? -sn : sn, v);
      }
      bool neg;
      const int o = dst_slot(n, k * st, neg);
      reinterpret_cast<double*>(B + o)[tid & 1] = neg ? -2.0 * v : 2.0 * v;
    }
    __syncthreads();
  }
}

// n <= 64 (any n): the folded sine sums directly, one thread per output and row: the fast
// transform would leave most lanes of its one warp idle and runs 4 times as long.  On return
// B[k] = X_k.  T: tab (see k_dst_sums64) in shared memory; tp >= 2 n threads.
__device__ __forceinline__ void dst_direct(double2* A, double2* B, const double* T, int n, int tid, int tp) {
  const int H = n >> 1, He = (n - 1) >> 1;
  for (int j = 1 + tid; j <= He; j += tp) {
    const double2 a = A[j], b = A[n - j];
    A[j] = make_double2(a.x + b.x, a.y + b.y);
    A[n - j] = make_double2(a.x - b.x, a.y - b.y);
  }
  __syncthreads();
  const int row = tid >= n ? 1 : 0, i = tid - row * n;
  if (tid < 2 * n && i < H + He) {
    const bool odd = i < H;
    const double* t = odd ? T + i : T + H * H + (i - H);
    const double* a = reinterpret_cast<const double*>(odd ? A + 1 : A + n - 1) + row;
    const int st = odd ? 2 : -2, m = odd ? H : He;
    double v0 = 0.0, v1 = 0.0;
    int j = 0;
    for (; j + 1 < m; j += 2) {
      v0 = fma(a[j * st], t[j * H], v0);
      v1 = fma(a[(j + 1) * st], t[(j + 1) * H], v1);
    }
    if (j < m) v0 = fma(a[j * st], t[j * H], v0);
    reinterpret_cast<double*>(B + (odd ? 2 * i + 1 : 2 * (i - H) + 2))[row] = v0 + v1;
  }
  __syncthreads();
}

// The transform of both rows at k (k in [1, n)): X_k, or 2 X_k with the fast algorithm (the
// factor 2 of each transform is divided out in the scale table).
template <bool DIRECT> __device__ __forceinline__ double2 dst_out(const double2* B, int n, int k) {
  if constexpr (DIRECT) {
    return B[k];
  } else {
    bool neg;
    const double2 v = B[dst_slot(n, k, neg)];
    return neg ? make_double2(-v.x, -v.y) : v;
  }
}

// Loaders: fill the A arrays (apart by `ld` elements) of the block's P pairs, rows m0, m0 + 1 of
// right-hand sides r0 .. r0 + P - 1.
template <int P> struct LoadRows {   // in[(r M + m) n + j]; wall: row 0 reads zero
  const double* in;
  bool wall;
  __device__ void operator()(const RowsArgs& a, double2* A, int ld, int m0, int r0) const {
    const bool one = !(wall && m0 == 0), two = m0 + 1 < a.M;
#pragma unroll
    for (int r = 0; r < P; ++r) {
      const double* p = in + ((int64_t)(r0 + r) * a.M + m0) * a.n;
      for (int j = threadIdx.x; j < a.n; j += blockDim.x)
        A[r * ld + j] = make_double2(one ? p[j] : 0.0, two ? p[a.n + j] : 0.0);
    }
  }
};
template <typename F> struct LoadSource {   // per-node sources f(iy, ix, v) of F::NR right-hand sides
  F f;
  static constexpr int NR = F::NR;
  __device__ void operator()(const RowsArgs& a, double2* A, int ld, int m0, int) const {
    for (int t = threadIdx.x; t < 2 * a.n; t += blockDim.x) {
      const int q = t >= a.n ? 1 : 0, j = t - q * a.n;
      double v[NR];
#pragma unroll
      for (int r = 0; r < NR; ++r) v[r] = 0.0;
      if (m0 + q < a.M) f(m0 + q, j, v);
#pragma unroll
      for (int r = 0; r < NR; ++r) reinterpret_cast<double*>(A + r * ld + j)[q] = v[r];
    }
  }
};

// Storers: rows m0, m0 + 1 of right-hand side r, by the tp threads of its pair.
struct StoreT {   // out[(r n + k) M + m]
  double* out;
  template <bool DIRECT>
  __device__ void put(const RowsArgs& a, const double2* B, int m0, int r, int tid, int tp) const {
    double* p = out + (int64_t)r * a.n * a.M + m0;
    const bool even = (a.M & 1) == 0, two = m0 + 1 < a.M;
    for (int k = tid; k < a.n; k += tp) {
      const double2 v = k ? dst_out<DIRECT>(B, a.n, k) : make_double2(0.0, 0.0);
      if (even) {
        *reinterpret_cast<double2*>(p + (int64_t)k * a.M) = v;
      } else {
        p[(int64_t)k * a.M] = v.x;
        if (two) p[(int64_t)k * a.M + 1] = v.y;
      }
    }
  }
};
struct StoreN {   // out[(r M + m) n + k]; row and column 0 (the wall) are zero
  double* out;
  template <bool DIRECT>
  __device__ void put(const RowsArgs& a, const double2* B, int m0, int r, int tid, int tp) const {
    double* p = out + ((int64_t)r * a.M + m0) * a.n;
    const bool two = m0 + 1 < a.M;
    for (int k = tid; k < a.n; k += tp) {
      const double2 v = k ? dst_out<DIRECT>(B, a.n, k) : make_double2(0.0, 0.0);
      p[k] = m0 ? v.x : 0.0;
      if (two) p[a.n + k] = v.y;
    }
  }
};
// Predictor-corrector mixing B <- w B_solved + (1 - w) B of component r into bm, and the
// residual sums of the slice's last iteration (rsum non-null).
struct StoreMix {
  V2<double>* bm;
  double w;
  int* status;
  double* rsum;
  template <bool DIRECT>
  __device__ void put(const RowsArgs& a, const double2* B, int m0, int r, int tid, int tp) const {
    double d2 = 0.0, b2 = 0.0;
    const double w1 = 1.0 - w;
    bool bad = false;
    for (int k = tid; k < a.n; k += tp) {
      const double2 v = k ? dst_out<DIRECT>(B, a.n, k) : make_double2(0.0, 0.0);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        if (m0 + q >= a.M) break;
        const double s = q ? v.y : (m0 ? v.x : 0.0);   // row 0: the wall
        double* p = reinterpret_cast<double*>(bm + (int64_t)(m0 + q) * a.n + k) + r;
        const double old = *p, nb = w * s + w1 * old;
        bad |= (__double2hiint(s) & 0x7ff00000) == 0x7ff00000;   // not finite (off the FP64 pipe)
        *p = nb;
        if (rsum) {
          d2 += (nb - old) * (nb - old);
          b2 += nb * nb;
        }
      }
    }
    if (bad) atomicOr(status, DEV_NONFINITE);
    if (rsum) pc_residual_add(rsum, d2, b2);
  }
};

// blockIdx.x: pair of rows; the block transforms P pairs (P right-hand sides from
// blockIdx.y * P on), tp = blockDim.x / P threads each (a multiple of 32).
template <typename Load, typename Store, int P, bool TWICE, bool DIRECT>
__global__ void k_dst_rows(RowsArgs a, Load ld, Store st) {
  extern __shared__ double2 sm[];
  const int tp = blockDim.x / P, pr = threadIdx.x / tp, tid = threadIdx.x - pr * tp;
  double2* A = sm;                 // P arrays A, P arrays B, then the twiddles or sine table
  double2* B = A + P * a.n;
  double2* tw = B + P * a.n;
  double* T = reinterpret_cast<double*>(tw);
  if constexpr (DIRECT) {
    pdl_trigger();
    const int H = a.n >> 1;
    for (int t = threadIdx.x; t < 2 * H * H; t += blockDim.x) T[t] = a.tab[t];
  } else {
    for (int t = threadIdx.x; t < a.n; t += blockDim.x) {
      const double2 w = reinterpret_cast<const double2*>(a.tab)[t];
      tw[t] = make_double2(w.x, -w.y);
    }
  }
  pdl_wait();
  const int m0 = 2 * blockIdx.x, r0 = blockIdx.y * P;
  ld(a, A, a.n, m0, r0);
  __syncthreads();
  double2* Ap = A + pr * a.n;
  double2* Bp = B + pr * a.n;
  auto transform = [&]() {
    if constexpr (DIRECT) dst_direct(Ap, Bp, T, a.n, tid, tp);
    else dst_pair(Ap, Bp, tw, a.n, a.logn, tid, tp);
  };
  transform();
  if constexpr (TWICE) {
    const double* s0 = a.scale + (int64_t)m0 * a.n;
    const double* s1 = m0 + 1 < a.M ? s0 + a.n : s0;
    for (int k = 1 + tid; k < a.n; k += tp) {
      const double2 v = dst_out<DIRECT>(Bp, a.n, k);
      Ap[k] = make_double2(v.x * s0[k], v.y * s1[k]);
    }
    __syncthreads();
    transform();
  }
  // long rows trigger only now: the next launch's CTAs placed while these compute would crowd
  // some SMs (243 us instead of 114 us for a 512^2 solve of two right-hand sides)
  if constexpr (!DIRECT) pdl_trigger();
  st.template put<DIRECT>(a, Bp, m0, r0 + pr, tid, tp);
}

// ---------------------------------------------------------------- rows of any length
// out[k] = sum_j in[j] sin(pi j k / n), folded: tab[0][j-1][i] = sin(pi j (2i+1) / n) weighs
// x_j + x_{n-j} (x_{n/2} alone once), tab[1][j-1][i] = sin(pi j (2i+2) / n) weighs x_j - x_{n-j};
// j = 1..H, H = n/2.  A warp forms 32 outputs of one parity of one row, a lane each: the table's
// values are read along a row of it, those of the folded row from shared memory (one for all lanes).
//
// What bounds it: the FP64 pipe, which takes a warp's multiply-add in 16 clocks of an SM, so that a
// multiply-add's two operands come fast enough without being kept for a second row, and what counts
// is that the warps are spread evenly: tiles of 32 rows x 64 outputs (a block of 16 multiply-adds per
// thread from registers) left most SMs idle up to 200 cells and the last wave nearly empty beyond, 2 and
// 4 rows per warp are up to 1.7 and 2.5 times as slow as one and never more than 2 % faster.  Solves:
//                                          100^2, 1 rhs  16 x 400, 1  400^2, 2  409^2, 3  1000^2, 1
//   a thread per output, n terms                    54 us        134        2094      1439      10715
//   the tiles                                      176           424        1570      2419       6567
//   this kernel                                     23            36         536       826       3662
constexpr int kSumRows = 4, kSumChunk = 256;   // rows (warps) of a block, folded terms staged at a time
__global__ void __launch_bounds__(32 * kSumRows) k_dst_sums64(const double* __restrict__ in, double* __restrict__ out, int n,
                                                              int M, const double* __restrict__ tab,
                                                              const double* __restrict__ scale, int transposed) {
  __shared__ alignas(16) double xs[kSumRows][kSumChunk];
  pdl_wait();
  const int H = n / 2, nt = (H + 31) / 32, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int par = blockIdx.y / nt, i = (blockIdx.y - par * nt) * 32 + lane, m = blockIdx.x * kSumRows + w, r = blockIdx.z;
  if (m < M) {
    const double* src = in + ((int64_t)r * M + m) * n;
    const double* t = tab + (int64_t)par * H * H + (i < H ? i : H - 1);
    double* x = xs[w];
    double acc0 = 0.0, acc1 = 0.0;
    for (int j0 = 0; j0 < H; j0 += kSumChunk) {
      const int kc = H - j0 < kSumChunk ? H - j0 : kSumChunk;
      __syncwarp();
      for (int jj = lane; jj < kc; jj += 32) {
        const int j = j0 + jj + 1;
        const double a = src[j], b = src[n - j];
        x[jj] = 2 * j == n ? (par ? 0.0 : a) : (par ? a - b : a + b);
      }
      __syncwarp();
      int jj = 0;
#pragma unroll 1
      for (; jj + 8 <= kc; jj += 8, t += 8 * (int64_t)H) {
        double s[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) s[c] = t[(int64_t)c * H];
#pragma unroll
        for (int c = 0; c < 8; c += 2) {
          const double2 v = *reinterpret_cast<const double2*>(x + jj + c);
          acc0 = fma(v.x, s[c], acc0);
          acc1 = fma(v.y, s[c + 1], acc1);
        }
      }
      for (; jj < kc; ++jj, t += H) acc0 = fma(x[jj], t[0], acc0);
    }
    pdl_trigger();
    auto put = [&](int k, double v) {
      if (transposed) out[((int64_t)r * n + k) * M + m] = v;
      else out[((int64_t)r * M + m) * n + k] = v;
    };
    const int k = 2 * i + 1 + par;
    const double v = acc0 + acc1;
    if (k < n) put(k, scale ? v * scale[(int64_t)m * n + k] : v);
    if (blockIdx.y == 0 && lane == 0) put(0, 0.0);
  }
}

bool is_pow2(int n) { return n > 0 && (n & (n - 1)) == 0; }
int ilog2(int n) { int l = 0; while ((1 << l) < n) ++l; return l; }

// Rows of up to kDirect points: direct sums; longer ones of a power of two: the fast algorithm;
// both in k_dst_rows.  The rest: k_dst_sums64.
constexpr int kDirect = 64;
bool rows_direct(int n) { return n <= kDirect; }
bool rows_ok(int n) { return rows_direct(n) || is_pow2(n); }

constexpr size_t kSmemMax = 226 * 1024;   // (of 227 KB: the residual sums take 512 static bytes)
size_t rows_smem(int n, int P) {
  const size_t tab = rows_direct(n) ? sizeof(double) * 2 * (n / 2) * (n / 2) : sizeof(double2) * n;
  return sizeof(double2) * 2 * P * (size_t)n + tab;
}

// Whether the kernel of rows of length n lets the next launch in only when its blocks are about to store
// (k_dst_rows of more than kDirect points, k_dst_sums64) and not when they begin (direct sums): the blocks of a
// long pass that are let in then crowd the SMs that have room (two right-hand sides of 200 x 16: 25 -> 76 us,
// five of 37 x 128: 32 -> 115 us), so that within a solve one is launched plainly behind direct sums.
bool rows_late(int n) { return !rows_direct(n); }

template <int P, bool TWICE, bool DIRECT, typename Load, typename Store>
void rows_launch_d(const hq_grid_s* g, int n, int M, int R, const double* tab, const double* scale, const Load& ld,
                   const Store& st, bool late, cudaStream_t s) {
  auto kern = k_dst_rows<Load, Store, P, TWICE, DIRECT>;
  static std::atomic<unsigned long long> done{0};   // devices whose shared-memory limit is raised
  const unsigned long long bit = 1ull << (g->dev & 63);
  if (!(done.load() & bit)) {
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
    done.fetch_or(bit);
  }
  // threads per pair: one radix-4 group each per pass, or one output and row each
  const int tp = DIRECT ? (2 * n + 31) / 32 * 32 : (n / 4 > 256 ? 256 : n / 4);
  RowsArgs a{n, DIRECT ? 0 : ilog2(n), M, tab, scale};
  const dim3 grid((unsigned)((M + 1) / 2), (unsigned)(R / P));
  if (DIRECT || late) launch_pdl(kern, grid, dim3((unsigned)(tp * P)), rows_smem(n, P), s, a, ld, st);
  else kern<<<grid, tp * P, rows_smem(n, P), s>>>(a, ld, st);
}
template <int P, bool TWICE, typename Load, typename Store>
void rows_launch(const hq_grid_s* g, int n, int M, int R, const double* tw, const double* tab, const double* scale,
                 const Load& ld, const Store& st, bool late, cudaStream_t s) {
  if (rows_direct(n)) rows_launch_d<P, TWICE, true>(g, n, M, R, tab, scale, ld, st, late, s);
  else rows_launch_d<P, TWICE, false>(g, n, M, R, tw, scale, ld, st, late, s);
}

// One transform along rows of length n ([R][M][n]): transposed or in place order.  late: rows_late of the launch
// before in the solve.
void one_pass(const hq_grid_s* g, const double* in, double* out, int n, int M, int R, const double* tw, const double* tab,
              const double* scale, bool transposed, bool late, cudaStream_t s) {
  if (rows_ok(n)) {
    const LoadRows<1> ld{in, transposed};   // (the transposed pass reads the caller's sources)
    if (transposed) rows_launch<1, false>(g, n, M, R, tw, tab, nullptr, ld, StoreT{out}, late, s);
    else rows_launch<1, false>(g, n, M, R, tw, tab, nullptr, ld, StoreN{out}, late, s);
    return;
  }
  const dim3 grid((unsigned)((M + kSumRows - 1) / kSumRows), (unsigned)(2 * ((n / 2 + 31) / 32)), (unsigned)R);
  const int tr = transposed ? 1 : 0;
  if (late) launch_pdl(k_dst_sums64, grid, dim3(32 * kSumRows), (size_t)0, s, in, out, n, M, tab, scale, tr);
  else k_dst_sums64<<<grid, 32 * kSumRows, 0, s>>>(in, out, n, M, tab, scale, tr);
}

// Along y of b = [R][nx][ny], forward, scaled and backward; the result [R][ny][nx] is in the
// returned buffer (a or b).
const double* y_both(const hq_grid_s* g, double* a, double* b, int R, const double* scale, cudaStream_t s) {
  const int nx = g->nx, ny = g->ny;
  if (rows_ok(ny)) {
    rows_launch<1, true>(g, ny, nx, R, g->tw_y, g->sin_y, scale, LoadRows<1>{b, false}, StoreT{a}, rows_late(nx), s);
    return a;
  }
  one_pass(g, b, a, ny, nx, R, g->tw_y, g->sin_y, scale, false, rows_late(nx), s);
  one_pass(g, a, b, ny, nx, R, g->tw_y, g->sin_y, nullptr, true, true, s);
  return b;
}

}  // namespace

// Sine table of the folded sums (see k_dst_sums64): [2][n/2][n/2] values sin(pi j k / n).
std::vector<double> dst_f64_table(int n, double (*sin_jk)(int64_t, int64_t, int)) {
  const int H = n / 2;
  std::vector<double> t(2 * (size_t)H * H, 0.0);
  for (int par = 0; par < 2; ++par)
    for (int j = 1; j <= H; ++j)
      for (int i = 0; i < H; ++i) {
        const int k = 2 * i + 1 + par;
        if (k < n) t[((size_t)par * H + j - 1) * H + i] = sin_jk(j, k, n);
      }
  return t;
}

// Each transform by the fast algorithm yields twice the sine sums: what the scale table divides out.
double dst_f64_norm(int nx, int ny) {
  auto fast = [](int n) { return rows_ok(n) && !rows_direct(n); };
  return (fast(nx) ? 0.25 : 1.0) * (fast(ny) ? 0.25 : 1.0);
}
bool dst_f64_twiddles(int n) { return rows_ok(n) && !rows_direct(n); }

// The sources of nr right-hand sides can be formed by the first pass (and the B_perp mixing done
// by the last): rows along x of every right-hand side in one CTA of k_dst_rows.
bool dst_f64_fused(const hq_grid_s* g, int nr) { return rows_ok(g->nx) && rows_smem(g->nx, nr) <= kSmemMax; }

int dst_f64_launches(const hq_grid_s* g) { return rows_ok(g->ny) ? 3 : 4; }

// src [R][ny][nx] -> dst [R][ny][nx] (row and column 0 of src are not read into the transforms;
// those of dst are zero).  src null: the sources in g->f64_a.
void dst_solve_f64(hq_grid_s* g, int R, cudaStream_t s, const double* scale, const double* src, double* dst) {
  if (!scale) scale = g->f64_scale;
  if (!src) src = g->f64_a;
  if (!dst) dst = reinterpret_cast<double*>(g->solved);
  const int nx = g->nx, ny = g->ny;
  one_pass(g, src, g->f64_b, nx, ny, R, g->tw_x, g->sin_x, nullptr, true, rows_ok(nx), s);   // (s S_x)^T [R][nx][ny]
  const double* q = y_both(g, g->f64_a, g->f64_b, R, scale, s);                        // [R][ny][nx]
  one_pass(g, q, dst, nx, ny, R, g->tw_x, g->sin_x, nullptr, false, rows_late(ny), s);
}

// psi, Ez, Bz of the deposit record dep -> g->solved, sources formed by the first pass.
void dst_f64_main(hq_grid_s* g, const void* dep, cudaStream_t s) {
  using F = SrcMain<double>;
  rows_launch<3, false>(g, g->nx, g->ny, 3, g->tw_x, g->sin_x, nullptr, LoadSource<F>{src_main_of<double>(g, dep)}, StoreT{g->f64_b},
                        true, s);
  const double* q = y_both(g, g->f64_a, g->f64_b, 3, g->f64_scale, s);
  one_pass(g, q, reinterpret_cast<double*>(g->solved), g->nx, g->ny, 3, g->tw_x, g->sin_x, nullptr, false,
           rows_late(g->ny), s);
}

// One predictor-corrector iteration: B_perp sources (which clear the trial J_perp and, on the
// last iteration, reset the slice i-1 record), solve, mixing into bm.
void dst_f64_bmix(hq_grid_s* g, const void* cur, void* prev, void* chi_prev, int last, cudaStream_t s) {
  using F = SrcBperp<double>;
  rows_launch<2, false>(g, g->nx, g->ny, 2, g->tw_x, g->sin_x, nullptr,
                        LoadSource<F>{src_bperp_of<double>(g, cur, prev, chi_prev, last)}, StoreT{g->f64_b}, true, s);
  const double* q = y_both(g, g->f64_a, g->f64_b, 2, g->f64_scale, s);
  rows_launch<2, false>(g, g->nx, g->ny, 2, g->tw_x, g->sin_x, nullptr, LoadRows<2>{q, false},
                        StoreMix{reinterpret_cast<V2<double>*>(g->bm), g->d.pc_mix, g->d_status, g->pc_rsum},
                        rows_late(g->ny), s);
}

}  // namespace hq
