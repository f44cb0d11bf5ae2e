// DST-I as dense matrix products on the 5th-generation tensor cores (tcgen05),
// for the FP32 path of the fast Poisson solver (Sec. 3.2: "fast Poisson solvers
// based on a Discrete Sine Transform of the first type").
//
// A Dirichlet solve is f = (2/nx)(2/ny) S_y [ (S_y s S_x) / lambda ] S_x.  With
// every operand kept K-major, each of the four products is a "TN" GEMM
//   D[m][n] = sum_k A[m][k] S[n][k]          (S symmetric)
// whose epilogue stores D transposed, so that the next product again reads its
// operand K-major: two such products give S_y s S_x.  R right-hand sides are
// stacked along m (R * 128-padded rows), so one launch transforms them all.
//
// Precision ("bf16x3"): every FP32 operand a is carried as a_hi + a_lo with
// a_hi = bf16(a), a_lo = bf16(a - a_hi) (16 significant bits); a product uses
// a_hi b_hi + a_hi b_lo + a_lo b_hi, accumulated in FP32 in tensor memory.
// The epilogue of each product re-splits its FP32 result for the next one and
// fuses the 1/lambda scaling (second product) or the final FP32 store (fourth).
// Precision "TF32x3" (the fused streamed solve below, instantiated on FP32 words): a_hi =
// a rounded to TF32 (cvt.rna), a_lo = a - a_hi, tcgen05.mma kind::tf32 (K = 8 per
// instruction); the byte layout of every stage, box and swizzle is the bf16 one, a 128-byte
// K block holding 32 elements instead of 64.
//
// Per-product kernel (k_dst_gemm, one product per launch; the allocation-free entry point
// at the end of this file runs it), one 128 x 128 output tile per CTA, 4 warps:
//   warp 0 lane 0  TMA producer: 128B-swizzled 128x64 bf16 boxes of A_hi, A_lo,
//                  S_hi, S_lo per stage (64 KB), 3-stage mbarrier ring;
//   warp 1 lane 0  MMA issuer: 12 tcgen05.mma (M=128, N=128, K=16) per stage,
//                  tcgen05.commit releases the stage, a final commit signals
//                  the epilogue;
//   warps 0-3      epilogue: tcgen05.ld 32x32b (lane = row), transposed store.
// Every wait on an mbarrier is bounded; on expiry the kernel sets a status bit,
// still drains its MMAs, frees its tensor memory and returns.
#include "hq_internal.cuh"

#include <algorithm>
#include <cstdlib>

namespace hq {

struct TensorMaps {
  CUtensorMap a0_hi, a0_lo;   // op[0] as [kMaxRhs * nyp][nxp]
  CUtensorMap a1_hi, a1_lo;   // op[1] as [kMaxRhs * nxp][nyp]
  CUtensorMap sx_hi[2], sx_lo[2];   // [nxp][nxp], boxes of 128 ([0]) or 64 ([1]) rows (per-product path)
  CUtensorMap sy_hi[2], sy_lo[2];   // [nyp][nyp]
  // fused solve, per N-tile width ([0]: 64, [1]: 32): S_x [nxp][nxp], or the fold matrix
  // [nxp][nxp/2], in boxes of BN rows; the FP32 scale [nyp][nxp] in 128 (x) by BN (y) boxes
  CUtensorMap bx_hi[2], bx_lo[2];
  CUtensorMap fx_hi, fx_lo, fy_hi, fy_lo;   // the same matrices in 128-row boxes (wide solve)
  int wide_ctas;                            // its co-resident CTAs
  CUtensorMap by_hi[2], by_lo[2];
  CUtensorMap scale[2];
  CUtensorMap scale_h[2];     // the shifted (Helmholtz) spectral factors, same boxes (explicit solver)
  int ctas[2];                // co-resident CTAs of each width
  bool wide_only;             // HQ_SOLVE_BN=64: never use the 32-wide tiles
  // resident fold-matrix solve (square folded grids, n = 256 or 512) and cluster solve:
  // op[0] .. op[2] in BN-row boxes ([0]: 64, [1]: 32)
  bool rs;
  CUtensorMap rx_hi[3][2], rx_lo[3][2];   // [operand][width]
  int rs_ctas[2];
  // cluster solve: its mode (0, 1, 2; -1: not used for this grid), and for 32 and 64 data rows per CTA the
  // largest number of right-hand sides whose clusters are all resident at once
  int cl_mode;
  int cl_rhs[2];
  int cl_max;   // resident clusters of mode 1
  bool all_smem;   // a solve kernel of this grid does not exclude others by its registers (see alone_by_registers)
};

namespace {

// A K block is 128 bytes of every operand row (one 128B-swizzle atom row): BK = 64 bf16
// elements, or 32 TF32 elements held in FP32 words (the TF32x3 split); byte sizes below are
// the same for both.
constexpr int BM = 128, BK = 64;
constexpr int A_BYTES = BM * 128;                  // 16 KB per A box
template <typename E> constexpr int kb_elems() { return 128 / (int)sizeof(E); }
// Tile shape per N-tile width: 128 (3 stages of 64 KB) or 64 (4 stages of 48 KB).
template <int BN, typename E = __nv_bfloat16> struct Cfg {
  static constexpr int B_BYTES = BN * 128;
  static constexpr int STAGE_BYTES = 2 * A_BYTES + 2 * B_BYTES;   // A_hi, A_lo, B_hi, B_lo
  static constexpr int STAGES = BN == 128 ? 3 : 4;
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 /*align*/ + 256 /*barriers*/;
  static constexpr uint32_t TMEM_COLS = BN;
  // instruction descriptor (kind::f16 with A = B = BF16 (1), or kind::tf32 with A = B = TF32
  // (2)): D = F32, both K-major, M = BM, N = BN
  static constexpr uint32_t FMT = sizeof(E) == 4 ? 2u : 1u;
  static constexpr uint32_t IDESC =
      (1u << 4) | (FMT << 7) | (FMT << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
  // the same with N = 2 BN: B_hi and B_lo, adjacent in a stage, read as one operand
  static constexpr uint32_t IDESC2 =
      (1u << 4) | (FMT << 7) | (FMT << 10) | ((uint32_t)(BN >> 2) << 17) | ((uint32_t)(BM >> 4) << 24);
};

struct Epi {
  int mode;          // 0: split + transposed bf16 store; 1: scale, split, store; 2: FP32 transposed store
  int P1;            // rows per right-hand side (padded), i.e. m extent per rhs
  int P2;            // padded n extent
  __nv_bfloat16* out_hi;
  __nv_bfloat16* out_lo;
  const float* scale;   // [P2][P1]
  float* out_f32;       // [R][n_real][m_real]
  int m_real, n_real;
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred P1;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 P1, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, P1;\n\t}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait (about two seconds of SM clock); false and a status bit on expiry.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int* status) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > (4ll << 30)) {
      atomicOr(status, DEV_TIMEOUT);
      return false;
    }
  }
  return true;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y)
      : "memory");
}

__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// K-major operand tile, 128B swizzle: rows of 64 bf16 (128 B), 8-row atoms 1024 B apart.
__device__ __forceinline__ uint64_t desc_k_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);   // start address, 16 B units
  d |= (uint64_t)1 << 16;                      // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;            // stride byte offset: 8 rows x 128 B
  d |= (uint64_t)1 << 46;                      // descriptor version (sm_100 family)
  d |= (uint64_t)2 << 61;                      // layout: SWIZZLE_128B
  return d;
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(idesc), "r"(accum));
}
// TF32 operands (kind::tf32, K = 8 per instruction: 32 bytes of each row, as for bf16)
__device__ __forceinline__ void mma_tf32(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(idesc), "r"(accum));
}
template <typename E>
__device__ __forceinline__ void mma_op(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accum) {
  if constexpr (sizeof(E) == 4) mma_tf32(tmem_d, a, b, idesc, accum);
  else mma_bf16(tmem_d, a, b, idesc, accum);
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* v) {
  tmem_ld32_issue(taddr, v);
  tmem_ld_wait();
}
__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
}
// W (16 or 32) columns of a stacked accumulator: x[j] = D[c0 + j] + D[BN + c0 + j] of this
// thread's lane
template <int BN, int W>
__device__ __forceinline__ void tmem_ld_pair(uint32_t taddr, float* x) {
  uint32_t v[W], u[W];
  if constexpr (W == 32) {
    tmem_ld32_issue(taddr, v);
    tmem_ld32_issue(taddr + (uint32_t)BN, u);
  } else {
    static_assert(W == 16, "16 or 32 columns");
    tmem_ld16_issue(taddr, v);
    tmem_ld16_issue(taddr + (uint32_t)BN, u);
  }
  tmem_ld_wait();
#pragma unroll
  for (int j = 0; j < W; ++j) x[j] = __uint_as_float(v[j]) + __uint_as_float(u[j]);
}

template <int BN>
__global__ void __launch_bounds__(128, 1)
    k_dst_gemm(const __grid_constant__ CUtensorMap ta_hi, const __grid_constant__ CUtensorMap ta_lo,
               const __grid_constant__ CUtensorMap tb_hi, const __grid_constant__ CUtensorMap tb_lo, int K, Epi ep,
               int* status) {
  using C = Cfg<BN>;
  constexpr int STAGES = C::STAGES, STAGE_BYTES = C::STAGE_BYTES;
  constexpr uint32_t TMEM_COLS = C::TMEM_COLS;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* basep = smem_raw + (base - raw);
  uint64_t* bars = reinterpret_cast<uint64_t*>(basep + STAGES * STAGE_BYTES);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 1);
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + STAGES), done = smem_u32(bars + 2 * STAGES);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  const int nk = K / BK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // everything above overlaps the previous kernel (programmatic dependent launch)
  pdl_trigger();
  pdl_wait();

  if (warp == 0 && lane == 0) {
    // TMA producer
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % STAGES;
      if (kb >= STAGES && !mbar_wait(empty0 + 8 * s, ((kb / STAGES) - 1) & 1, status)) break;
      const uint32_t st = base + s * STAGE_BYTES;
      const uint32_t fb = full0 + 8 * s;
      mbar_expect_tx(fb, STAGE_BYTES);
      tma_load_2d(st, &ta_hi, kb * BK, m0, fb);
      tma_load_2d(st + A_BYTES, &ta_lo, kb * BK, m0, fb);
      tma_load_2d(st + 2 * A_BYTES, &tb_hi, kb * BK, n0, fb);
      tma_load_2d(st + 2 * A_BYTES + C::B_BYTES, &tb_lo, kb * BK, n0, fb);
    }
  } else if (warp == 1 && lane == 0) {
    // MMA issuer
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % STAGES;
      if (!mbar_wait(full0 + 8 * s, (kb / STAGES) & 1, status)) break;
      tc_fence_after();
      const uint32_t st = base + s * STAGE_BYTES;
      const uint64_t ah = desc_k_sw128(st), al = desc_k_sw128(st + A_BYTES);
      const uint64_t bh = desc_k_sw128(st + 2 * A_BYTES), bl = desc_k_sw128(st + 2 * A_BYTES + C::B_BYTES);
#pragma unroll
      for (int k = 0; k < BK / 16; ++k) {
        const uint64_t off = (uint64_t)((k * 32) >> 4);  // 16 bf16 = 32 B along K inside the swizzle row
        mma_bf16(tmem, ah + off, bh + off, C::IDESC, (kb | k) != 0 ? 1u : 0u);
        mma_bf16(tmem, ah + off, bl + off, C::IDESC, 1u);
        mma_bf16(tmem, al + off, bh + off, C::IDESC, 1u);
      }
      mma_commit(empty0 + 8 * s);
    }
    mma_commit(done);
  }
  __syncwarp();
  mbar_wait(done, 0, status);
  tc_fence_after();

  // ---------------------------------------------------------------- epilogue
  const int row = warp * 32 + lane;
  const int m = m0 + row;
  const int r = m / ep.P1, ml = m - r * ep.P1;
#pragma unroll 1
  for (int c0 = 0; c0 < BN; c0 += 32) {
    uint32_t v[32];
    tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
    if (ep.mode == 2) {
      if (ml < ep.m_real) {
        bool bad = false;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const int n = n0 + c0 + j;
          const float x = __uint_as_float(v[j]);
          bad |= !isfinite(x);
          if (n < ep.n_real) ep.out_f32[((int64_t)r * ep.n_real + n) * ep.m_real + ml] = x;
        }
        if (bad) atomicOr(status, DEV_NONFINITE);
      }
    } else {
      float sc[32];
      if (ep.mode == 1) {
#pragma unroll
        for (int j = 0; j < 32; ++j) sc[j] = __ldg(ep.scale + (int64_t)(n0 + c0 + j) * ep.P1 + ml);
      }
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        const int n = n0 + c0 + j;
        float x = __uint_as_float(v[j]);
        if (ep.mode == 1) x *= sc[j];
        const __nv_bfloat16 h = __float2bfloat16_rn(x);
        const __nv_bfloat16 l = __float2bfloat16_rn(x - __bfloat162float(h));
        const int64_t o = ((int64_t)r * ep.P2 + n) * ep.P1 + ml;
        ep.out_hi[o] = h;
        ep.out_lo[o] = l;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// ---------------------------------------------------------------- fused persistent solve
// A whole Dirichlet solve in one cooperative launch: the four products run as
// phases separated by grid-wide barriers, with tensor memory, mbarriers and the
// shared-memory ring set up once and the intermediates kept in L2.  Phase p
// contracts along x (p = 0, 2: operand op[0], matrix S_x) or along y (p = 1, 3:
// op[1], S_y); its epilogue writes the next phase's operand transposed.
//
// Folded order (fold_pair; n a multiple of 128): every operand row holds its n/2
// pair sums followed by its n/2 pair differences, the output columns are slots, and
// an N-tile of odd (even) slots contracts over the sums (differences) only, K = n/2,
// against the fold matrix.  Rows 2u, 2u+1 of a tile are a pair, i.e. adjacent TMEM
// lanes, so the epilogue folds the next operand with one warp shuffle.
//
// Tiles are 128 x BN (BN = 32 when every tile still gets its own CTA, else 64), one CTA
// of 256 threads per SM: warp 0 lane 0 issues the TMA loads (A_hi, A_lo, B_hi, B_lo of a
// 128-byte K block per stage, 4-stage ring), warp 1 lane 0 the MMAs (two per K step:
// A_hi x [B_hi; B_lo] with N = 2 BN, A_lo x B_hi with N = BN, into a 2 BN-column TMEM
// accumulator), and all 8 warps the epilogue, each warpgroup half of the columns.
constexpr int kSolveThreads = 256;

// No two CTAs of solve kernels may share an SM, of one launch or of launches on different streams: most
// of them allocate all of tensor memory and then wait for other CTAs, so that two launches could each
// hold what the other waits for.  Two CTAs that take more than half of its registers each never do, and
// the solve kernels take 127 to 168 registers in 256 to 384 threads.  Should a build give one of them less,
// the grids that use it request (nearly) all of the shared memory for their launches, which leaves no room
// for a CTA that has any.  (Shared memory above one half for all of them, without the look at the
// registers, made a 512^2 sweep with the explicit solver 1.2 % slower: the SMs' split between L1 and shared
// memory changes between the solves and the node kernels.)
constexpr bool alone_by_registers(int regs, int threads) { return 2 * regs * threads > 65536; }
constexpr int kSmemAll = 226 * 1024;
static_assert(kSmemAll + 2 * 1024 >= 228 * 1024, "1 KB for the system per CTA: room for another CTA would be left");

// The caller's sources [nr][ny][nx] (hq_poisson_solve); row and column 0 read zero.
struct SrcGiven {
  static constexpr int NR = kMaxRhs;
  static constexpr bool kEffects = false;
  const float* src;
  Geom gm;
  int nr;
  struct In {
    float v[kMaxRhs];
  };
  __device__ In load(int iy, int ix) const {
    In q;
    const int64_t nn = (int64_t)gm.nx * gm.ny, o = (int64_t)iy * gm.nx + ix;
#pragma unroll
    for (int r = 0; r < kMaxRhs; ++r) q.v[r] = (r < nr && ix > 0 && iy > 0) ? src[r * nn + o] : 0.0f;
    return q;
  }
  __device__ void eval(int, int, const In& q, float* v) const {
#pragma unroll
    for (int r = 0; r < kMaxRhs; ++r) v[r] = q.v[r];
  }
  __device__ void effects(int, int) const {}
};

struct SolveArgs {
  int R;                               // right-hand sides
  int nxp, nyp;                        // operand extents (= nx, ny when folded)
  int fold;
  void *op_hi[3], *op_lo[3];           // op[0]: [R][nyp][nxp], op[1]: [R][nxp][nyp] (bf16 or TF32 words)
  const float* scale;                  // [nyp][nxp]: (4/(nx ny)) / lambda, slot order when folded
  int final_mode;                      // 2: FP32 store into out [R][ny][nx]; 3: predictor-corrector mixing
  float* out;
  int nx, ny;
  float* bm;                           // mode 3: B <- w B_solved + (1 - w) B in bm[node * 2 + r]
  float w;
  double* rsum;                        // mode 3: sum (B_new - B_old)^2, sum B_new^2 added here (or null)
  unsigned long long* gbar;            // grid-barrier counter (zero at launch, reset by the last CTA);
                                       // resident solve: exit counter, then the dependency counters
  int* status;
  int barrier_skew;                    // added to the first barrier's target (fault injection; 0)
  // source phase ahead of the four products: 0 none (sources already in op[0]); 1 the psi,
  // Ez, Bz sources of a deposit record (sm); 2 the B_perp sources of the predictor-corrector (sb);
  // 3 R given fields (sc)
  int pre;
  SrcMain<float> sm;
  SrcBperp<float> sb;
  SrcGiven sc;
  // the reset of the slice i-1 record (SrcBperp::reset) by the warps that filled tensor memory, off
  // the source phase: the later iterations' sources (mode 2) do not read what it writes
  int reset_late;
};
// Nodes of the reset, by `count` threads, this one `me`.
__device__ __forceinline__ void reset_nodes(const SolveArgs& a, int me, int count) {
  const int nn = a.nx * a.ny;
  for (int o = me; o < nn; o += count) a.sb.reset(o);
}

// bf16 hi/lo split of 8 values packed for two 16-byte stores.
__device__ __forceinline__ void split8(const float* v, uint4& hi, uint4& lo) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const __nv_bfloat16 h0 = __float2bfloat16_rn(v[2 * k]), h1 = __float2bfloat16_rn(v[2 * k + 1]);
    const __nv_bfloat16 l0 = __float2bfloat16_rn(v[2 * k] - __bfloat162float(h0));
    const __nv_bfloat16 l1 = __float2bfloat16_rn(v[2 * k + 1] - __bfloat162float(h1));
    h[k] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
    l[k] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
  }
  hi = make_uint4(h[0], h[1], h[2], h[3]);
  lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// Eight consecutive operand elements, split.
__device__ __forceinline__ void put_run8(__nv_bfloat16* hi, __nv_bfloat16* lo, const float* v) {
  uint4 h, l;
  split8(v, h, l);
  *reinterpret_cast<uint4*>(hi) = h;
  *reinterpret_cast<uint4*>(lo) = l;
}
__device__ __forceinline__ void put_run8(float* hi, float* lo, const float* v) {
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    float h[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) h[k] = round_tf32(v[4 * q + k]);
    reinterpret_cast<float4*>(hi)[q] = make_float4(h[0], h[1], h[2], h[3]);
    reinterpret_cast<float4*>(lo)[q] = make_float4(v[4 * q] - h[0], v[4 * q + 1] - h[1], v[4 * q + 2] - h[2], v[4 * q + 3] - h[3]);
  }
}

__device__ __forceinline__ void main_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }   // warps 0-7

// Source phase: every thread of the launch takes (row, column) items of the operand writer
// in turn (consecutive threads along a row), KB items at a time: all their reads are issued
// before any write, then the sources are evaluated, split into op[0] and the functor's own
// writes (clearing the trial J_perp) follow.
template <typename Sink, typename F, int NR>
__device__ __forceinline__ void solve_sources(const Geom& gm, const Sink& sink, const F& f, int nr = NR) {
  constexpr int KB = 4;
  constexpr int NN = Sink::kFold ? 2 : 1;   // nodes per item
  const int w = visit_width<Sink>(gm);
  const int total = w * gm.ny;
  const int stride = gridDim.x * kSolveThreads;   // (the first 256 threads of every block)
  for (int t0 = blockIdx.x * kSolveThreads + threadIdx.x; t0 < total; t0 += KB * stride) {
    int iy[KB][NN], ix[KB][NN];
    typename F::In in[KB][NN];
#pragma unroll
    for (int k = 0; k < KB; ++k) {
      const int t = t0 + k * stride;
      const int row = t < total ? t / w : 0, tx = t < total ? t % w : 0;
      if constexpr (Sink::kFold) {
        iy[k][0] = iy[k][NN - 1] = fold_node(row, gm.ny);
        fold_pair(tx, gm.nx, ix[k][0], ix[k][NN - 1]);
      } else {
        iy[k][0] = row;
        ix[k][0] = tx;
      }
#pragma unroll
      for (int j = 0; j < NN; ++j) in[k][j] = t < total ? f.load(iy[k][j], ix[k][j]) : typename F::In{};
    }
#pragma unroll
    for (int k = 0; k < KB; ++k) {
      const int t = t0 + k * stride;
      if (t >= total) break;
      float v[NN][NR];
#pragma unroll
      for (int j = 0; j < NN; ++j) f.eval(iy[k][j], ix[k][j], in[k][j], v[j]);
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        if (r >= nr) break;
        if constexpr (Sink::kFold) sink.put_pair(r, t / w, t % w, v[0][r], v[NN - 1][r]);
        else sink.put(r, t / w, t % w, v[0][r]);
      }
      if constexpr (F::kEffects) {
#pragma unroll
        for (int j = 0; j < NN; ++j) f.effects(iy[k][j], ix[k][j]);
      }
    }
  }
}
// The sources a launch asks for.
template <typename E> __device__ __forceinline__ void solve_sources_all(const SolveArgs& a) {
  const Geom& gm = a.pre == 1 ? a.sm.gm : (a.pre == 2 ? a.sb.gm : a.sc.gm);
  E* hi = reinterpret_cast<E*>(a.op_hi[0]);
  E* lo = reinterpret_cast<E*>(a.op_lo[0]);
  if (a.fold) {
    const SinkFold<E> sink{hi, lo, a.nx, a.ny};
    if (a.pre == 1) solve_sources<SinkFold<E>, SrcMain<float>, 3>(gm, sink, a.sm);
    else if (a.pre == 2) solve_sources<SinkFold<E>, SrcBperp<float>, 2>(gm, sink, a.sb);
    else solve_sources<SinkFold<E>, SrcGiven, kMaxRhs>(gm, sink, a.sc, a.R);
  } else {
    const SinkSplit<E> sink{hi, lo, a.nxp, a.nyp};
    if (a.pre == 1) solve_sources<SinkSplit<E>, SrcMain<float>, 3>(gm, sink, a.sm);
    else if (a.pre == 2) solve_sources<SinkSplit<E>, SrcBperp<float>, 2>(gm, sink, a.sb);
    else solve_sources<SinkSplit<E>, SrcGiven, kMaxRhs>(gm, sink, a.sc, a.R);
  }
}

// Bounded mbarrier wait that also gives up once another thread of the CTA has.
__device__ __forceinline__ bool mbar_wait_a(uint32_t bar, uint32_t parity, int* status, volatile int* abort_f) {
  const long long t0 = clock64();
  uint32_t it = 0;
  while (!mbar_try_wait(bar, parity)) {
    if ((++it & 63u) == 0 && (*abort_f || clock64() - t0 > (4ll << 30))) {
      atomicOr(status, DEV_TIMEOUT);
      *abort_f = 1;
      return false;
    }
  }
  return true;
}

// Grid-wide barrier (all CTAs co-resident: cooperative launch).  The counter is zero at
// launch and only grows within it: barrier b completes at (b + 1) * gridDim.x arrivals; after
// the last barrier every CTA arrives once more and the last one resets the counter to zero,
// so a launch needs no host-side state (and can be replayed from a CUDA graph).  The proxy
// fences order the epilogue's generic stores before the other CTAs' TMA (async-proxy)
// loads of the next phase.  Bounded: on expiry, or once another CTA has reported a
// timeout, the CTA sets DEV_TIMEOUT and leaves.
__device__ __forceinline__ bool grid_barrier(unsigned long long* ctr, unsigned long long target, int* status,
                                             volatile int* abort_f) {
  asm volatile("fence.proxy.async.global;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0) {
    if (!*abort_f) {
      asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(ctr) : "memory");
      const long long t0 = clock64();
      uint32_t it = 0;
      while (true) {
        unsigned long long v;
        asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(ctr) : "memory");
        if (v >= target) break;
        if ((++it & 15u) == 0 &&
            ((*reinterpret_cast<volatile int*>(status) & DEV_TIMEOUT) || clock64() - t0 > (4ll << 30))) {
          atomicOr(status, DEV_TIMEOUT);
          *abort_f = 1;
          break;
        }
      }
    }
    asm volatile("fence.proxy.async.global;" ::: "memory");
  }
  __syncthreads();
  return !*abort_f;
}

// Dependency counters of the resident solve, one per 128-byte line, zero at launch and reset by
// the last CTA to leave.  A producer's arrival follows its stores, a proxy fence and a CTA barrier;
// the consumer's TMA-issuing thread waits.
__device__ __forceinline__ void dep_arrive(unsigned long long* c) {
  asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(c) : "memory");
}
__device__ __forceinline__ bool dep_wait(const unsigned long long* c, unsigned long long target, int* status,
                                         volatile int* abort_f) {
  const long long t0 = clock64();
  uint32_t it = 0;
  while (true) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(c) : "memory");
    if (v >= target) break;
    if ((++it & 15u) == 0 &&
        ((*reinterpret_cast<volatile int*>(status) & DEV_TIMEOUT) || clock64() - t0 > (4ll << 30))) {
      atomicOr(status, DEV_TIMEOUT);
      *abort_f = 1;
      return false;
    }
  }
  asm volatile("fence.proxy.async.global;" ::: "memory");
  return true;
}

// One lane of a converged warp, chosen without divergence the compiler cannot see through (its
// tensor-core instructions then take their descriptors from uniform registers).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred P1;\n\telect.sync _|P1, 0xffffffff;\n\tselp.b32 %0, 1, 0, P1;\n\t}\n" : "=r"(p));
  return p != 0;
}

// The streamed solve runs 256 threads per CTA (warps 0, 1: TMA producer, MMA issuer; all 8
// warps: epilogue) on N tiles 64 wide, or 32 wide when that still gives every tile its own
// CTA (twice the tiles, so more of the SMs take part in each product).

// Shared memory of the solve: the stage ring, the FP32 scale tile of phase 1
// ([BN n][128 rows]), then the barriers (full, empty, done, scale) and the TMEM slot.
template <int BN> struct SolveSmem {
  static constexpr int STAGES = Cfg<BN>::STAGES;
  static constexpr int RING = STAGES * Cfg<BN>::STAGE_BYTES;
  static constexpr int SCALE = RING;
  static constexpr int BARS = SCALE + BN * BM * 4;
  static constexpr int BYTES = BARS + 256 + 1024 /*alignment*/;
};

template <int BN, bool RES, typename E>
__global__ void __launch_bounds__(kSolveThreads, 1)
    k_dst_solve(const __grid_constant__ CUtensorMap a0h, const __grid_constant__ CUtensorMap a0l,
                const __grid_constant__ CUtensorMap a1h, const __grid_constant__ CUtensorMap a1l,
                const __grid_constant__ CUtensorMap bxh, const __grid_constant__ CUtensorMap bxl,
                const __grid_constant__ CUtensorMap byh, const __grid_constant__ CUtensorMap byl,
                const __grid_constant__ CUtensorMap scm, const SolveArgs a) {
  using C = Cfg<BN, E>;
  using L = SolveSmem<BN>;
  constexpr int STAGES = C::STAGES, STAGE_BYTES = C::STAGE_BYTES;
  constexpr int KE = kb_elems<E>();   // elements per K block
  extern __shared__ uint8_t smem_raw[];
  __shared__ int s_abort;
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* basep = smem_raw + (base - raw);
  uint64_t* bars = reinterpret_cast<uint64_t*>(basep + L::BARS);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 2);
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + STAGES), done = smem_u32(bars + 2 * STAGES);
  const uint32_t sbar = smem_u32(bars + 2 * STAGES + 1);
  const float* scale_s = reinterpret_cast<const float*>(basep + L::SCALE);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort_f = &s_abort;

  if (threadIdx.x == 0) {
    for (const CUtensorMap* m : {&a0h, &a0l, &a1h, &a1l, &bxh, &bxl, &byh, &byl, &scm})
      prefetch_map(m);
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(done, 1);
    mbar_init(sbar, 1);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"((uint32_t)(2 * BN))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // stage-ring, accumulator and scale-tile counters across tiles
  uint32_t kb_run = 0, tiles_run = 0, scales_run = 0;
  auto phase_geom = [&](int q, int& P1, int& P2, int& mt, int& tiles, int& nk) {
    const bool ax = (q & 1) == 0;
    P1 = ax ? a.nyp : a.nxp;
    P2 = ax ? a.nxp : a.nyp;
    mt = a.R * P1 / BM;
    tiles = mt * (P2 / BN);
    nk = (a.fold ? P2 / 2 : P2) / KE;
  };
  // both axes' geometry and this CTA's first tile, computed before the first phase (after a
  // grid barrier they would sit on the path to the phase's first TMA issue)
  int P1x, P2x, mtx, tilesx, nkx, P1y, P2y, mty, tilesy, nky;
  phase_geom(0, P1x, P2x, mtx, tilesx, nkx);
  phase_geom(1, P1y, P2y, mty, tilesy, nky);
  const int final_mode = a.final_mode;
  const int t0 = (int)blockIdx.x;
  const int m0x = (t0 % mtx) * BM, n0x = (t0 / mtx) * BN, rx = m0x / P1x;
  const int m0y = (t0 % mty) * BM, n0y = (t0 / mty) * BN, ry = m0y / P1y;
  // source phase (its writes reach the other CTAs' TMA loads through the barrier's proxy fences)
  const unsigned nb0 = a.pre ? 1u : 0u;   // barriers before phase 0
  bool go = true;
  if (a.pre) {
    solve_sources_all<E>(a);
    go = grid_barrier(a.gbar, (unsigned long long)gridDim.x + (unsigned)a.barrier_skew, a.status, abort_f);
  }
  for (int p = 0; p < 4 && go; ++p) {
    const bool along_x = (p & 1) == 0;
    // rows per rhs, output columns (= contraction extent), tiles, K blocks
    const int P1 = along_x ? P1x : P1y, P2 = along_x ? P2x : P2y, mt = along_x ? mtx : mty;
    const int tiles = along_x ? tilesx : tilesy, nk = along_x ? nkx : nky;
    const CUtensorMap* tah = along_x ? &a0h : &a1h;
    const CUtensorMap* tal = along_x ? &a0l : &a1l;
    const CUtensorMap* tbh = along_x ? &bxh : &byh;
    const CUtensorMap* tbl = along_x ? &bxl : &byl;
    const int mode = p == 3 ? final_mode : (p == 1 ? 1 : 0);
    if (p == 3) pdl_trigger();
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
      const bool first = tile == t0;
      const int m0 = first ? (along_x ? m0x : m0y) : (tile % mt) * BM;
      const int n0 = first ? (along_x ? n0x : n0y) : (tile / mt) * BN;
      const int r = first ? (along_x ? rx : ry) : m0 / P1, ml0 = m0 - r * P1;   // a tile lies within one rhs
      const int koff = (a.fold && n0 >= P2 / 2) ? P2 / 2 : 0;
      if (warp == 0 && lane == 0) {
        // TMA producer (and the scale tile of the spectral division)
        if (mode == 1) {
          mbar_expect_tx(sbar, BN * BM * 4);
          tma_load_2d(base + L::SCALE, &scm, ml0, n0, sbar);
        }
        for (int kb = 0; kb < nk; ++kb) {
          const uint32_t g = kb_run + kb;
          const int s = g % STAGES;
          const uint32_t st = base + s * STAGE_BYTES;
          const uint32_t fb = full0 + 8 * s;
          // a tile starts on a drained ring (every thread waited for the previous tile's last
          // MMA), so only a stage reused within the tile needs its release
          if (kb >= STAGES && !mbar_wait_a(empty0 + 8 * s, ((g / STAGES) - 1) & 1, a.status, abort_f)) break;
          mbar_expect_tx(fb, STAGE_BYTES);
          tma_load_2d(st, tah, koff + kb * KE, m0, fb);
          tma_load_2d(st + A_BYTES, tal, koff + kb * KE, m0, fb);
          tma_load_2d(st + 2 * A_BYTES, tbh, kb * KE, n0, fb);
          tma_load_2d(st + 2 * A_BYTES + C::B_BYTES, tbl, kb * KE, n0, fb);
        }
      } else if (warp == 1 && lane == 0) {
        // MMA issuer
        for (int kb = 0; kb < nk; ++kb) {
          const uint32_t g = kb_run + kb;
          const int s = g % STAGES;
          if (!mbar_wait_a(full0 + 8 * s, (g / STAGES) & 1, a.status, abort_f)) break;
          tc_fence_after();
          const uint32_t st = base + s * STAGE_BYTES;
          const uint64_t ah = desc_k_sw128(st), al = desc_k_sw128(st + A_BYTES);
          const uint64_t bh = desc_k_sw128(st + 2 * A_BYTES);
          // columns [0, BN): A_hi B_hi + A_lo B_hi; columns [BN, 2 BN): A_hi B_lo (one MMA
          // with N = 2 BN covers both A_hi products: the tensor core's cost here is per instruction);
          // four 32-byte K steps per block (K = 16 bf16 or 8 TF32 each)
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const uint64_t off = (uint64_t)((k * 32) >> 4);
            mma_op<E>(tmem, ah + off, bh + off, C::IDESC2, (kb | k) != 0 ? 1u : 0u);
            mma_op<E>(tmem, al + off, bh + off, C::IDESC, 1u);
          }
          mma_commit(empty0 + 8 * s);
        }
        mma_commit(done);
      }
      __syncwarp();
      mbar_wait_a(done, tiles_run & 1, a.status, abort_f);
      if (mode == 1) mbar_wait_a(sbar, scales_run & 1, a.status, abort_f);
      tc_fence_after();

      // ------------------------------------------------ epilogue: TMEM lane = tile row; the
      // two warpgroups take one half of the columns each (a warp reads the lanes of its
      // quarter of the tile, warp % 4)
      constexpr int CH = BN / 2;
      const int row = (warp & 3) * 32 + lane;
      const int ml = ml0 + row;
      const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16);
      const int c0 = (warp >> 2) * CH;
      if (mode <= 1) {
        // scale (phase 1), fold with the pair partner (one shuffle), split and store the next
        // operand transposed: folded, even rows hold pair sums (column u), odd rows pair
        // differences (column P1/2 + u)
        const bool odd = (ml & 1) != 0, wall = a.fold && (ml >> 1) == P1 / 4;
        const int fcol = a.fold ? (odd ? P1 / 2 + (ml >> 1) : (ml >> 1)) : ml;
        E* oh = reinterpret_cast<E*>(a.op_hi[along_x ? 1 : 0]);
        E* ol = reinterpret_cast<E*>(a.op_lo[along_x ? 1 : 0]);
        {
          float x[CH];
          tmem_ld_pair<BN, CH>(tl + (uint32_t)c0, x);
          if (mode == 1) {
#pragma unroll
            for (int j = 0; j < CH; ++j) x[j] *= scale_s[(c0 + j) * BM + row];
          }
          if (a.fold) {
            // all exchanges first, so that the warp's shuffles overlap
            float y[CH];
#pragma unroll
            for (int j = 0; j < CH; ++j) y[j] = __shfl_xor_sync(0xffffffffu, x[j], 1);
#pragma unroll
            for (int j = 0; j < CH; ++j) x[j] = odd ? (wall ? 0.0f : y[j] - x[j]) : (wall ? y[j] : x[j] + y[j]);
          }
#pragma unroll
          for (int j = 0; j < CH; ++j) put_split(oh, ol, ((int64_t)r * P2 + n0 + c0 + j) * P1 + fcol, x[j]);
        }
      } else {
        // node of this row (rows run along x in the last phase)
        const int xn = a.fold ? fold_node(ml, a.nx) : ml;
        float x[CH];
        tmem_ld_pair<BN, CH>(tl + (uint32_t)c0, x);
        float d2 = 0.0f, b2 = 0.0f;   // mode 3 with RES: this thread's share of the residual (FP32)
        if (xn < a.nx) {
          auto ynode = [&](int j) { return a.fold ? fold_node(n0 + c0 + j, a.ny) : n0 + c0 + j; };
          if (mode == 2) {
#pragma unroll
            for (int j = 0; j < CH; ++j) {
              const int yn = ynode(j);
              if (yn < a.ny) a.out[((int64_t)r * a.ny + yn) * a.nx + xn] = x[j];
            }
          } else {
            // predictor-corrector mixing into bm[r] (all loads first, then mix and store)
            float old[CH];
#pragma unroll
            for (int j = 0; j < CH; ++j) {
              const int yn = ynode(j);
              const int64_t node = (int64_t)yn * a.nx + xn;
              old[j] = yn < a.ny ? a.bm[node * 2 + r] : 0.0f;
            }
            bool bad = false;
#pragma unroll
            for (int j = 0; j < CH; ++j) {
              const int yn = ynode(j);
              if (yn >= a.ny) continue;
              bad |= !isfinite(x[j]);
              const int64_t node = (int64_t)yn * a.nx + xn;
              const float nb = a.w * x[j] + (1.0f - a.w) * old[j];
              a.bm[node * 2 + r] = nb;
              if constexpr (RES) {
                const float d = nb - old[j];
                d2 += d * d;
                b2 += nb * nb;
              }
            }
            if (bad) atomicOr(a.status, DEV_NONFINITE);
          }
        }
        if constexpr (RES)
          if (mode == 3) pc_residual_add(a.rsum, (double)d2, (double)b2);   // every lane (mode is uniform)
      }
      kb_run += nk;
      ++tiles_run;
      if (mode == 1) ++scales_run;
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
      if (*abort_f) break;
    }
    if (p < 3 && !grid_barrier(a.gbar,
                               (unsigned long long)(nb0 + p + 1) * gridDim.x +
                                   (nb0 == 0 && p == 0 ? (unsigned)a.barrier_skew : 0u),
                               a.status, abort_f))
      break;
  }
  // exit arrival: the last CTA through resets the counter for the next launch
  if (threadIdx.x == 0 && !*abort_f) {
    const unsigned long long seen = atomicAdd(a.gbar, 1ull);
    if (seen == (nb0 + 4ull) * gridDim.x - 1ull) atomicExch(a.gbar, 0ull);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)(2 * BN)) : "memory");
  }
}

// Threads of the resident and cluster solves: warps 0-7 as in the streamed solve, 8-11 fill tensor
// memory while the others form the sources.
constexpr int kClThreads = 384;
__device__ __forceinline__ void mma_bf16_ta(uint32_t tmem_d, uint32_t tmem_a, uint64_t b, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(tmem_d),
      "r"(tmem_a), "l"(b), "r"(idesc), "r"(accum));
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint4* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
      "r"(v[0].x), "r"(v[0].y), "r"(v[0].z), "r"(v[0].w), "r"(v[1].x), "r"(v[1].y), "r"(v[1].z), "r"(v[1].w), "r"(v[2].x),
      "r"(v[2].y), "r"(v[2].z), "r"(v[2].w), "r"(v[3].x), "r"(v[3].y), "r"(v[3].z), "r"(v[3].w), "r"(v[4].x), "r"(v[4].y),
      "r"(v[4].z), "r"(v[4].w), "r"(v[5].x), "r"(v[5].y), "r"(v[5].z), "r"(v[5].w), "r"(v[6].x), "r"(v[6].y), "r"(v[6].z),
      "r"(v[6].w), "r"(v[7].x), "r"(v[7].y), "r"(v[7].z), "r"(v[7].w)
      : "memory");
}

// pc_residual_add for the first 256 threads of a block.
__device__ __forceinline__ void residual_add_main(double* rs, double d2, double b2) {
  __shared__ double part[2][kSolveThreads / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    d2 += __shfl_down_sync(0xffffffffu, d2, o);
    b2 += __shfl_down_sync(0xffffffffu, b2, o);
  }
  if ((threadIdx.x & 31) == 0) {
    part[0][threadIdx.x >> 5] = d2;
    part[1][threadIdx.x >> 5] = b2;
  }
  main_sync();
  if (threadIdx.x < 2) {
    double s = 0.0;
    for (int k = 0; k < kSolveThreads / 32; ++k) s += part[threadIdx.x][k];
    if (s != 0.0) atomicAdd(rs + 2 * (int)(blockIdx.x % kResLanes) + threadIdx.x, s);
  }
  main_sync();
}

// A slice of the fold (or sine) matrix, 128 slots x K, into tensor memory as a tcgen05.mma A operand:
// lane = slot, a 32-bit column = two consecutive K elements, K / 2 hi columns then K / 2 lo columns.
// By one warp per quarter of the lanes (quarter = warp mod 4); f: hq_grid_s::fxt.
template <int K>
__device__ __forceinline__ void fill_tmem(const uint4* __restrict__ f, int block, uint32_t taddr, int quarter, int lane) {
  const uint4* p = f + (int64_t)block * (K / 4) * BM + quarter * 32 + lane;
  const uint32_t t = taddr + ((uint32_t)(quarter * 32) << 16);
#pragma unroll 2
  for (int g = 0; g < K / 32; ++g) {
    uint4 v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = __ldg(p + (g * 8 + k) * BM);
    tmem_st32(t + 32u * g, v);
  }
}

// ---------------------------------------------------------------- resident fold-matrix solve
// The same four products for a square folded grid (nx = ny = n, n = 256 or 512) with the
// operand roles swapped: each CTA owns one block of 128 output slots for the whole launch,
// so its 128 x n/2 slice of the fold matrix (bf16 hi + lo, 64 or 128 KB) is put into tensor
// memory once, while the source phase runs, and only the data operand (BN rows of
// the previous phase's output) is streamed per tile:
//   D[s][c] = sum_u F[s][u] X[c][koff + u]   (A = F in tensor memory, B = X streamed),
// with koff = 0 for the odd-index slots (pair sums) and n/2 for the even ones (differences).
// A from tensor memory: with A in shared memory a tcgen05.mma costs ~90 clocks here whatever its
// N (4 KB of A at 64 B per clock; 1.4 us per product at n = 512), with A in tensor memory ~50.
// TMEM lane = output slot s, column = data row c.  The fold of the next operand pairs
// adjacent columns of one thread (no shuffle), and each thread stores its row of the next
// operand as contiguous 16-byte runs.  The third product writes its rows in node order, so
// the last one's output columns are consecutive x nodes.
// Between the products a tile waits for its producers only instead of a barrier of the whole grid
// (dependency counters, rs_wait: the 16 tiles of the slot block that wrote its rows at n = 512; for the
// last product, whose rows are nodes and come from two or three slot blocks, all 64 of its right-hand
// side).
template <int BN> struct RsSmem {
  static constexpr int KB_MAX = 4;                          // folded K = n/2 <= 256
  static constexpr int STAGE = 2 * BN * BK * 2;             // X_hi + X_lo rows of one K block
  static constexpr int RING = 0;
  static constexpr int TILE = BM * (BN + 1) * 4;            // the mixing's staged tile
  static constexpr int BARS = KB_MAX * STAGE > TILE ? KB_MAX * STAGE : TILE;
  static constexpr int BYTES = BARS + 256 + 1024 /*alignment*/;
  static constexpr uint32_t TX = 128;                       // tensor-memory columns: accumulator (2 BN), F slice
};

// Epilogue of one thread's CH consecutive columns (data rows i0 .. i0 + CH - 1 of rhs r) of
// output slot s.  Modes 0/1 (1: times the 1/lambda factors sc) fold adjacent column pairs into
// the next operand's row (r, orow) (orow = s, or its node for the third product): pair sums at column v, differences at n/2 + v (the wall
// pair (0, n/2) keeps x_{n/2} as its sum and 0 as its difference).  Mode 2 stores the
// solution (rows in node order: columns are consecutive x nodes); mode 3 is rs_mix.
template <int CH>
__device__ __forceinline__ void rs_epilogue(const SolveArgs& a, int mode, int s, int orow, int r, int i0, float* x,
                                            const float* sc, __nv_bfloat16* oh, __nv_bfloat16* ol) {
  const int n = a.nx, H = n / 2;
  if (mode <= 1) {
    if (mode == 1) {
#pragma unroll
      for (int j = 0; j < CH; ++j) x[j] *= sc[j];
    }
    float sum[CH / 2], dif[CH / 2];
    const int v0 = i0 >> 1;
#pragma unroll
    for (int k = 0; k < CH / 2; ++k) {
      const bool wall = v0 + k == n / 4;
      sum[k] = wall ? x[2 * k + 1] : x[2 * k] + x[2 * k + 1];
      dif[k] = wall ? 0.0f : x[2 * k] - x[2 * k + 1];
    }
    const int64_t base = ((int64_t)r * n + orow) * n;
#pragma unroll
    for (int k = 0; k < CH / 2; k += 8) {
      uint4 h, l;
      split8(sum + k, h, l);
      *reinterpret_cast<uint4*>(oh + base + v0 + k) = h;
      *reinterpret_cast<uint4*>(ol + base + v0 + k) = l;
      split8(dif + k, h, l);
      *reinterpret_cast<uint4*>(oh + base + H + v0 + k) = h;
      *reinterpret_cast<uint4*>(ol + base + H + v0 + k) = l;
    }
  } else if (mode == 2) {
    const int yn = fold_node(s, n);
    float4* o = reinterpret_cast<float4*>(a.out + ((int64_t)r * a.ny + yn) * a.nx + i0);
#pragma unroll
    for (int q = 0; q < CH / 4; ++q) o[q] = make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
  }
}

// Source phase of the resident and cluster solves (square folded grid, n <= 512): a CTA takes
// kSrcRows consecutive slot rows at a time (all their reads issued first), its threads read and
// evaluate the sources at consecutive nodes of a row (coalesced), stage them in shared memory S
// ([rows][nr][n] floats), write the folded pairs (x_a + x_b, x_a - x_b) of eight consecutive folded
// columns each (16-byte stores), and the CTA reports the rows to the counter of their data tile.
constexpr int kSrcRows = 4;
template <int BN, typename F, int NR>
__device__ __forceinline__ void solve_sources_rows(const Geom& gm, const F& f, __nv_bfloat16* hi, __nv_bfloat16* lo,
                                                   float* S, int nr, unsigned long long* ctr) {
  constexpr int NPT = 2;   // nodes per thread per row (n <= 2 x 256)
  constexpr int RPP = kSrcRows;
  const int n = gm.nx, H = n / 2;
  for (int sy0 = RPP * blockIdx.x; sy0 < gm.ny; sy0 += RPP * gridDim.x) {
    typename F::In in[RPP][NPT];
    int iy[RPP];
#pragma unroll
    for (int q = 0; q < RPP; ++q) {
      iy[q] = fold_node(sy0 + q, gm.ny);
#pragma unroll
      for (int k = 0; k < NPT; ++k) {
        const int x = threadIdx.x + k * kSolveThreads;
        in[q][k] = x < n ? f.load(iy[q], x) : typename F::In{};
      }
    }
#pragma unroll
    for (int q = 0; q < RPP; ++q) {
#pragma unroll
      for (int k = 0; k < NPT; ++k) {
        const int x = threadIdx.x + k * kSolveThreads;
        if (x >= n) continue;
        float v[NR];
        f.eval(iy[q], x, in[q][k], v);
#pragma unroll
        for (int r = 0; r < NR; ++r)
          if (r < nr) S[(q * nr + r) * n + x] = v[r];
        if constexpr (F::kEffects) f.effects(iy[q], x);
      }
    }
    main_sync();
    const int groups = H / 8;   // of eight folded columns
    for (int t = threadIdx.x; t < RPP * nr * groups; t += kSolveThreads) {
      const int qr = t / groups, u0 = (t - qr * groups) * 8, q = qr / nr, r = qr - q * nr;
      const float* row = S + qr * n;
      float sum[8], dif[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        int xa, xb;
        fold_pair(u0 + k, n, xa, xb);
        const float va = row[xa], vb = row[xb];
        const bool wall = u0 + k == n / 4;
        sum[k] = wall ? vb : va + vb;
        dif[k] = wall ? 0.0f : va - vb;
      }
      const int64_t o = ((int64_t)r * gm.ny + sy0 + q) * n + u0;
      uint4 h, l;
      split8(sum, h, l);
      *reinterpret_cast<uint4*>(hi + o) = h;
      *reinterpret_cast<uint4*>(lo + o) = l;
      split8(dif, h, l);
      *reinterpret_cast<uint4*>(hi + o + H) = h;
      *reinterpret_cast<uint4*>(lo + o + H) = l;
    }
    asm volatile("fence.proxy.async;" ::: "memory");
    main_sync();
    if (threadIdx.x == 0) dep_arrive(ctr + 16 * (sy0 / BN));
  }
}
// The sources a launch asks for.  S: kSrcRows x R x n floats.
template <int BN>
__device__ __forceinline__ void solve_sources_any(const SolveArgs& a, float* S, unsigned long long* ctr) {
  __nv_bfloat16* hi = reinterpret_cast<__nv_bfloat16*>(a.op_hi[0]);
  __nv_bfloat16* lo = reinterpret_cast<__nv_bfloat16*>(a.op_lo[0]);
  if (a.pre == 1) solve_sources_rows<BN, SrcMain<float>, 3>(a.sm.gm, a.sm, hi, lo, S, 3, ctr);
  else if (a.pre == 2) solve_sources_rows<BN, SrcBperp<float>, 2>(a.sb.gm, a.sb, hi, lo, S, 2, ctr);
  else solve_sources_rows<BN, SrcGiven, kMaxRhs>(a.sc.gm, a.sc, hi, lo, S, a.R, ctr);
}

// Predictor-corrector mixing B <- w B_solved + (1 - w) B of one tile (128 slots of y x BN
// consecutive x nodes from xb, component r) staged in shared memory ([128][BN + 1]): element
// e = (row, j) is taken by thread e mod 256, so a warp covers consecutive x nodes of one row;
// up to sixteen elements' loads are issued before their stores.
template <int BN, bool RES>
__device__ __forceinline__ void rs_mix(const SolveArgs& a, const float* tile, int s0, int r, int xb) {
  constexpr int LD = BN + 1, NE = BM * BN, UN = NE / kSolveThreads < 16 ? NE / kSolveThreads : 16;
  const int n = a.nx;
  bool bad = false;
  float d2 = 0.0f, b2 = 0.0f;   // RES (the slice's last iteration): residual sums in FP32
  for (int e0 = threadIdx.x; e0 < NE; e0 += UN * kSolveThreads) {
    float v[UN], old[UN];
    int64_t at[UN];
#pragma unroll
    for (int k = 0; k < UN; ++k) {
      const int e = e0 + k * kSolveThreads;
      const int row = e / BN, j = e - row * BN;
      v[k] = e < NE ? tile[row * LD + j] : 0.0f;
      at[k] = e < NE ? ((int64_t)fold_node(s0 + row, n) * a.nx + xb + j) * 2 + r : -1;
      old[k] = e < NE ? a.bm[at[k]] : 0.0f;
    }
#pragma unroll
    for (int k = 0; k < UN; ++k) {
      if (at[k] < 0) continue;
      bad |= !isfinite(v[k]);
      const float nb = a.w * v[k] + (1.0f - a.w) * old[k];
      a.bm[at[k]] = nb;
      if constexpr (RES) {
        const float d = nb - old[k];
        d2 += d * d;
        b2 += nb * nb;
      }
    }
  }
  if (bad) atomicOr(a.status, DEV_NONFINITE);
  if constexpr (RES) residual_add_main(a.rsum, (double)d2, (double)b2);
}

template <int BN, int N, bool RES>
__global__ void __launch_bounds__(kClThreads, 1)
    k_dst_solve_rs(const uint4* __restrict__ fxt, const __grid_constant__ CUtensorMap x0h, const __grid_constant__ CUtensorMap x0l,
                   const __grid_constant__ CUtensorMap x1h, const __grid_constant__ CUtensorMap x1l,
                   const __grid_constant__ CUtensorMap x2h, const __grid_constant__ CUtensorMap x2l, const SolveArgs a) {
  using L = RsSmem<BN>;
  constexpr int STAGES = L::KB_MAX;
  constexpr int CH = BN / 2;
  extern __shared__ uint8_t smem_raw[];
  __shared__ int s_abort;
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* basep = smem_raw + (base - raw);
  uint64_t* bars = reinterpret_cast<uint64_t*>(basep + L::BARS);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 2);
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + STAGES), done = smem_u32(bars + 2 * STAGES);
  const uint32_t tbar = smem_u32(bars + 2 * STAGES + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort_f = &s_abort;
  constexpr int n = N, H = n / 2, nk = H / BK, MB = n / BM, K = H;
  const int mb = (int)blockIdx.x % MB, s0 = mb * BM;
  const int koff = s0 < H ? 0 : H;          // odd slots (first half) contract over the pair sums
  const int NT = a.R * n / BN;               // data-row tiles per product
  const int nt0 = (int)blockIdx.x / MB, ntstep = (int)gridDim.x / MB;
  const bool tiles = nt0 < NT;               // a CTA beyond the tiles only forms sources
  const int NTR = n / BN;                    // data-row tiles per right-hand side
  unsigned long long* ctr_src = a.gbar + 16; // [NTR]: source rows of a data tile formed
  unsigned long long* ctr_p = ctr_src + 16 * NTR;   // [rs_counters]: rows of a product's output written

  if (threadIdx.x == 0) {
    for (const CUtensorMap* m : {&x0h, &x0l, &x1h, &x1l, &x2h, &x2l}) prefetch_map(m);
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(done, 1);
    mbar_init(tbar, 128);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  if (warp >= 8) {
    // this CTA's fold-matrix slice (slots s0 .. s0 + 127), resident for the launch
    if (tiles) {
      fill_tmem<K>(fxt, mb, tmem + L::TX, warp & 3, lane);
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      tc_fence_before();
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tbar) : "memory");
    }
    if (a.reset_late) reset_nodes(a, (int)blockIdx.x * 128 + (int)threadIdx.x - 256, (int)gridDim.x * 128);
    return;
  }
  // (the stage ring is idle until the first product: it holds the staged sources)
  if (a.pre) solve_sources_any<BN>(a, reinterpret_cast<float*>(basep + L::RING), ctr_src);
  uint32_t kb_run = 0, tiles_run = 0;
  bool f_ready = false;
  for (int p = 0; p < 4; ++p) {
    // Operands 0 -> 1 -> 2 -> 0: product 2 may overwrite operand 0, because its wait (every data
    // tile of the right-hand side through product 1, each of which waited for a slot block of
    // product 0) implies that all of product 0's tiles, operand 0's readers, are done; the same
    // does not hold for operand 1 in products 1 and 2, hence the third buffer.
    const CUtensorMap* xh = p == 1 ? &x1h : (p == 2 ? &x2h : &x0h);
    const CUtensorMap* xl = p == 1 ? &x1l : (p == 2 ? &x2l : &x0l);
    const int mode = p == 3 ? a.final_mode : (p == 1 ? 1 : 0);
    if (p == 3) pdl_trigger();   // the next kernel may be scheduled (it waits for this grid's end)
    for (int nt = nt0; nt < NT; nt += ntstep) {
      const int c0 = nt * BN;
      if (warp == 0 && lane == 0) {
        // data-tile producer: the whole folded K of BN rows, one stage per 64-wide K block, once
        // the rows' producers have reported (the source rows of the tile, or the tiles of the product
        // before that wrote them: rs_wait)
        bool ok = true;
        const int r_ = c0 / n, row0 = c0 - r_ * n;
        if (p > 0) {
          const RsWait w = rs_wait(p, a.R, MB, NTR, r_, row0);
          ok = dep_wait(ctr_p + 16 * w.counter,
                        (unsigned long long)w.target + (p == 1 && !a.pre ? (unsigned)a.barrier_skew : 0u), a.status, abort_f);
        } else if (a.pre)
          ok = dep_wait(ctr_src + 16 * (row0 / BN), (unsigned long long)(BN / kSrcRows) + (unsigned)a.barrier_skew, a.status,
                        abort_f);
        for (int kb = 0; ok && kb < nk; ++kb) {
          const uint32_t g = kb_run + kb;
          const int s = g % STAGES;
          const uint32_t st = base + L::RING + s * L::STAGE;
          const uint32_t fb = full0 + 8 * s;
          if (g >= (uint32_t)STAGES && !mbar_wait_a(empty0 + 8 * s, ((g / STAGES) - 1) & 1, a.status, abort_f)) break;
          mbar_expect_tx(fb, L::STAGE);
          tma_load_2d(st, xh, koff + kb * BK, c0, fb);
          tma_load_2d(st + BN * BK * 2, xl, koff + kb * BK, c0, fb);
        }
      } else if (warp == 1) {
        // MMA issuer: A = fold-matrix slice (resident), B = [X_hi; X_lo] (N = 2 BN) and X_hi
        bool ok = __all_sync(0xffffffffu, f_ready || mbar_wait_a(tbar, 0, a.status, abort_f));
        f_ready = ok;
        for (int kb = 0; ok && kb < nk; ++kb) {
          const uint32_t g = kb_run + kb;
          const int s = g % STAGES;
          ok = mbar_wait_a(full0 + 8 * s, (g / STAGES) & 1, a.status, abort_f);
          if (!__all_sync(0xffffffffu, ok)) break;
          tc_fence_after();
          const uint32_t st = base + L::RING + s * L::STAGE;
          const uint32_t ta = tmem + L::TX + (uint32_t)(kb * 32);
          const uint64_t bh = desc_k_sw128(st);
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < BK / 16; ++k) {
              const uint64_t off = (uint64_t)((k * 32) >> 4);
              mma_bf16_ta(tmem, ta + 8u * k, bh + off, Cfg<BN>::IDESC2, (kb | k) != 0 ? 1u : 0u);
              mma_bf16_ta(tmem, ta + (uint32_t)(K / 2) + 8u * k, bh + off, Cfg<BN>::IDESC, 1u);
            }
            mma_commit(empty0 + 8 * s);
          }
          __syncwarp();
        }
        if (elect_one()) mma_commit(done);
      }
      __syncwarp();
      // epilogue: TMEM lane = slot s0 + row, the two warpgroups take one half of the columns each
      const int row = (warp & 3) * 32 + lane;
      const int s = s0 + row;
      const int half = warp >> 2;
      const int r = c0 / n;
      const int i0 = c0 - r * n + half * CH;
      float sc[CH];   // the 1/lambda factors of this thread's elements, read while the MMAs run
      if (mode == 1) {
        const float4* q = reinterpret_cast<const float4*>(a.scale + (int64_t)s * n + i0);
#pragma unroll
        for (int k = 0; k < CH / 4; ++k) {
          const float4 f = __ldg(q + k);
          sc[4 * k] = f.x;
          sc[4 * k + 1] = f.y;
          sc[4 * k + 2] = f.z;
          sc[4 * k + 3] = f.w;
        }
      }
      mbar_wait_a(done, tiles_run & 1, a.status, abort_f);
      tc_fence_after();
      {
        float x[CH];
        tmem_ld_pair<BN, CH>(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(half * CH), x);
        const int orow = rs_out_row(p, s, n);
        if (mode == 3) {
          // predictor-corrector mixing into bm[node][r]: the tile goes through shared memory (the
          // drained stage ring) so that a warp updates consecutive nodes of one row
          constexpr int LD = BN + 1;
          float* tile = reinterpret_cast<float*>(basep + L::RING);
#pragma unroll
          for (int j = 0; j < CH; ++j) tile[row * LD + half * CH + j] = x[j];
          main_sync();
          if (!*abort_f) rs_mix<BN, RES>(a, tile, s0, r, c0 - r * n);
        } else if (!*abort_f) {
          const int o = p == 2 ? 0 : p + 1;
          rs_epilogue<CH>(a, mode, s, orow, r, i0, x, sc, p < 3 ? reinterpret_cast<__nv_bfloat16*>(a.op_hi[o]) : nullptr,
                          p < 3 ? reinterpret_cast<__nv_bfloat16*>(a.op_lo[o]) : nullptr);
        }
      }
      kb_run += nk;
      ++tiles_run;
      if (p < 3) asm volatile("fence.proxy.async.global;" ::: "memory");
      tc_fence_before();
      main_sync();
      tc_fence_after();
      if (*abort_f) break;
      if (p < 3 && threadIdx.x == 0) dep_arrive(ctr_p + 16 * rs_arrival(p, a.R, MB, r, mb));
    }
    if (*abort_f) break;
  }
  // the slice's stores must have ended before the tensor memory is given back (a CTA that gave up
  // may not have waited for them): a bounded wait that ignores the abort flag
  if (warp == 0 && tiles) mbar_wait(tbar, 0, a.status);
  // exit arrival: the last CTA through resets the counters for the next launch
  if (threadIdx.x == 0 && !*abort_f) {
    const unsigned long long seen = atomicAdd(a.gbar, 1ull);
    if (seen == gridDim.x - 1ull) {
      for (int i = 0; i < NTR + rs_counters(a.R, MB); ++i) ctr_src[16 * i] = 0ull;
      atomicExch(a.gbar, 0ull);
    }
  }
  tc_fence_before();
  main_sync();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

// ---------------------------------------------------------------- cluster solve
// The same four products with the operand exchanged inside thread-block clusters where the
// dependencies allow it.  A phase of the resident solve above spends 1.0 us until its stores are
// visible, 1.4 us on the dependency counter and 0.6 us on the TMA load of the next operand, against
// 0.7 us of MMAs and 0.7 us of epilogue.  Here the CTAs that hold one block of 128 kx slots of one
// right-hand side for every y (product 0: 8 CTAs of 32 data rows at n = 256) form a cluster: product
// 1 (along y) contracts exactly what the cluster holds, so product 0's epilogue writes the next
// operand, folded, split and swizzled, straight into the peers' shared memory, and a hardware
// cluster barrier replaces store, counter and load.  Product 1 -> 2 exchanges between clusters
// through global memory and the counters; product 2 -> 3 is again within the cluster.
//
// A CTA's output slots change between the x products (the cluster's block b) and the y products
// (block j = rank / TPB), so it needs two slices of the fold matrix.  The x slice lives in tensor
// memory (filled by four extra warps while the others form the sources): a tcgen05.mma whose A comes
// from shared memory costs ~90 clocks here whatever its N (4 KB of A at 64 B per clock), one
// whose A comes from tensor memory ~half.  n = 256 keeps both slices there.
//
// MODE 0 (nx, ny <= 128, sine matrices padded to 128, not folded) and MODE 2 (128 x 128, folded): one
// cluster holds all right-hand sides, sources included, and nothing but the results touches global
// memory.
// MODE 1: square folded grids of 256.  (512: eight clusters of 16 CTAs do not fit the GPU at once, and
// with 8 CTAs of 64 rows the exchange, 64 KB per CTA, takes 4 us: slower than through L2.)
// BN = 32 data rows per CTA and two data buffers, or (LOCAL, five right-hand sides) 64 and one.
template <int BN, int MODE> struct Cl {
  static constexpr bool LOCAL = MODE != 1, FOLD = MODE != 0;
  // MODE 2's one slot block has odd and even slots: its data rows keep sums and differences side by
  // side (K = 128) against a fold matrix with zeros in the other half
  static constexpr int N = LOCAL ? 128 : 256, K = 128, NK = K / BK, MB = N / BM;
  static constexpr int TPB = BM / BN, CPR = N / BN;        // tiles per slot block, CTAs per right-hand side (and block)
  static constexpr bool DB = BN == 32;                      // two data buffers
  static constexpr int STAGE = 2 * BN * 128;                // hi and lo rows of one K block
  static constexpr int BUF = NK * STAGE;
  static constexpr int TILE = BM * (BN + 1) * 4;            // staged output tile
  static constexpr int DATA = 0;
  static constexpr int DATA_BYTES = (DB ? 2 : 1) * BUF > TILE ? (DB ? 2 : 1) * BUF : (TILE + 127) / 128 * 128;
  // LOCAL: staged sources, BN rows (shared by R CTAs, rounded up) of R x 128 floats over R CTAs
  // MODE 1: kSrcRows rows of R x 256 floats (apart from the data buffers: a peer may already exchange)
  static constexpr int SRC = DATA + DATA_BYTES, SRC_BYTES = LOCAL ? (BN + kMaxRhs - 1) * 512 : kSrcRows * kMaxRhs * 1024;
  static constexpr int BARS = SRC + SRC_BYTES;
  static constexpr int BYTES = BARS + 128 + 1024;
  static constexpr uint32_t TX = 128, TY = TX + K;          // tensor-memory columns: accumulator, x slice, y slice
  // cluster barriers of a launch (each thread arrives at and waits for every one): the start, the
  // end of each exchange, and where a peer's buffer has to be drained first
  static constexpr int barriers(int pre) { return 1 + (LOCAL ? (pre ? 1 : 0) + 3 + (DB ? 0 : 3) : 2 + (DB ? 1 : 2)); }
};

__device__ __forceinline__ void cl_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cl_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, const uint4& v) {
  asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
               : "memory");
}
// 8 consecutive columns (col a multiple of 8) of operand row `row` into the data buffer at `buf` of
// CTA `rank`: 128B-swizzled K blocks, hi rows then lo rows.
template <int BN> __device__ __forceinline__ void put_operand8(uint32_t buf, uint32_t rank, int row, int col, const float* v) {
  uint4 h, l;
  split8(v, h, l);
  const uint32_t o = (uint32_t)((col >> 6) * (2 * BN * 128) + row * 128 + ((((col & 63) >> 3) ^ (row & 7)) << 4));
  const uint32_t d = mapa(buf + o, rank);
  st_cluster(d, h);
  st_cluster(d + BN * 128, l);
}
// LOCAL source phase: the R CTAs of data tile q share its rows (row i of the tile by the CTA of
// right-hand side i mod R): threads read and evaluate consecutive nodes (all of a batch's reads first),
// stage them in shared memory S ([rows][R][128] floats) and store eight operand columns at a time into the
// CTA that multiplies them.
template <int BN, bool FOLD, typename F, int NR>
__device__ __forceinline__ void cl_sources(const Geom& gm, const F& f, float* S, int R, int r, int q, uint32_t buf) {
  constexpr int CPR = 128 / BN, KB = 8;
  const int rows = (BN - r + R - 1) / R, W = gm.nx, total = rows * W;
  for (int e0 = threadIdx.x; e0 < total; e0 += KB * kSolveThreads) {
    typename F::In in[KB];
    int iy[KB], at[KB];   // node row (-1: none), place in S
#pragma unroll
    for (int k = 0; k < KB; ++k) {
      const int e = e0 + k * kSolveThreads, i = e / W, x = e - i * W, y = q * BN + r + i * R;
      at[k] = i * R * 128 + x;
      iy[k] = e < total ? (FOLD ? fold_node(y, 128) : y) : -2;
      if (iy[k] >= gm.ny) iy[k] = -1;
      in[k] = iy[k] >= 0 ? f.load(iy[k], x) : typename F::In{};
    }
#pragma unroll
    for (int k = 0; k < KB; ++k) {
      if (iy[k] == -2) break;
      const int x = at[k] & 127;
      float v[NR];
#pragma unroll
      for (int i = 0; i < NR; ++i) v[i] = 0.0f;
      if (iy[k] >= 0) {
        f.eval(iy[k], x, in[k], v);
        if constexpr (F::kEffects) f.effects(iy[k], x);
      }
#pragma unroll
      for (int i = 0; i < NR; ++i)
        if (i < R) S[at[k] + i * 128] = v[i];
    }
  }
  main_sync();
  constexpr int G = FOLD ? 8 : 16;   // groups of eight folded columns or nodes
  for (int t = threadIdx.x; t < rows * R * G; t += kSolveThreads) {
    const int qr = t / G, c = (t - qr * G) * 8, i = qr / R, k = qr - i * R;
    const float* row = S + qr * 128;
    const uint32_t rank = (uint32_t)(k * CPR + q);
    if constexpr (FOLD) {
      float sum[8], dif[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        int xa, xb;
        fold_pair(c + u, 128, xa, xb);
        const float va = row[xa], vb = row[xb];
        const bool wall = c + u == 32;
        sum[u] = wall ? vb : va + vb;
        dif[u] = wall ? 0.0f : va - vb;
      }
      put_operand8<BN>(buf, rank, r + i * R, c, sum);
      put_operand8<BN>(buf, rank, r + i * R, 64 + c, dif);
    } else {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = c + u < W ? row[c + u] : 0.0f;
      put_operand8<BN>(buf, rank, r + i * R, c, v);
    }
  }
}

// Node of column c (0 .. 127) of slot block b in the last product: the block's first nodes of the
// pairs in order, then their partners in reverse, so that a tile's columns are (almost) ascending
// nodes; and its inverse, the column of slot s of the block.
__device__ __forceinline__ int cl_node(int b, int c, int n) { return fold_node(b * BM + (c < 64 ? 2 * c : 2 * (127 - c) + 1), n); }
__device__ __forceinline__ int cl_col(int s) { return (s & 1) ? 127 - (s >> 1) : (s >> 1); }

// The solve's result: the tile [128 y slots][BN x columns] staged in shared memory is stored (final
// mode 2) or mixed into bm (mode 3); consecutive threads take consecutive columns of a row.
template <int BN, int MODE, bool RES>
__device__ __forceinline__ void cl_out(const SolveArgs& a, const float* tile, int j, int b, int t, int r) {
  using C = Cl<BN, MODE>;
  constexpr int LD = BN + 1, NE = BM * BN, UN = 16;
  bool bad = false;
  float d2 = 0.0f, b2 = 0.0f;
  for (int e0 = threadIdx.x; e0 < NE; e0 += UN * kSolveThreads) {
    float v[UN], old[UN];
    int64_t at[UN];
#pragma unroll
    for (int k = 0; k < UN; ++k) {
      const int e = e0 + k * kSolveThreads, row = e / BN, c = e - row * BN;
      const int y = C::FOLD ? fold_node(j * BM + row, C::N) : row;
      const int x = C::FOLD ? cl_node(b, t * BN + c, C::N) : t * BN + c;
      v[k] = tile[row * LD + c];
      at[k] = (C::FOLD || (y < a.ny && x < a.nx)) ? (int64_t)y * a.nx + x : -1;
      if (a.final_mode == 3) old[k] = at[k] >= 0 ? a.bm[at[k] * 2 + r] : 0.0f;
    }
#pragma unroll
    for (int k = 0; k < UN; ++k) {
      if (at[k] < 0) continue;
      if (a.final_mode == 2) {
        a.out[(int64_t)r * a.ny * a.nx + at[k]] = v[k];
        continue;
      }
      bad |= !isfinite(v[k]);
      const float nb = a.w * v[k] + (1.0f - a.w) * old[k];
      a.bm[at[k] * 2 + r] = nb;
      if constexpr (RES) {
        const float d = nb - old[k];
        d2 += d * d;
        b2 += nb * nb;
      }
    }
  }
  if (bad) atomicOr(a.status, DEV_NONFINITE);
  if constexpr (RES) residual_add_main(a.rsum, (double)d2, (double)b2);
}

template <int BN, int MODE, bool RES>
__global__ void __launch_bounds__(kClThreads, 1)
    k_dst_solve_cl(const __grid_constant__ CUtensorMap x0h, const __grid_constant__ CUtensorMap x0l,
                   const __grid_constant__ CUtensorMap x1h, const __grid_constant__ CUtensorMap x1l,
                   const uint4* __restrict__ fxt, const uint4* __restrict__ fyt, const SolveArgs a) {
  using C = Cl<BN, MODE>;
  constexpr int N = C::N, K = C::K, NK = C::NK, MB = C::MB, TPB = C::TPB, CPR = C::CPR;
  constexpr int CH = BN / 2, H = N / 2;
  extern __shared__ uint8_t smem_raw[];
  __shared__ int s_abort;
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* basep = smem_raw + (base - raw);
  uint64_t* bars = reinterpret_cast<uint64_t*>(basep + C::BARS);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + NK + 2);
  const uint32_t full0 = smem_u32(bars), done = smem_u32(bars + NK), tbar = smem_u32(bars + NK + 1);
  const uint32_t buf0 = base + C::DATA, buf1 = C::DB ? buf0 + C::BUF : buf0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort_f = &s_abort;
  uint32_t rank, cluster_ctas;
  asm("mov.u32 %0, %cluster_ctarank;" : "=r"(rank));
  asm("mov.u32 %0, %cluster_nctaid.x;" : "=r"(cluster_ctas));
  if (cluster_ctas != (uint32_t)(C::LOCAL ? a.R * CPR : CPR)) {
    // not launched in the clusters the exchange addresses (a tool that drops the launch attribute):
    // report it instead of writing to peers that do not exist
    if (threadIdx.x == 0) atomicOr(a.status, DEV_TIMEOUT);
    return;
  }
  // right-hand side r, x slot block b, position q among the CTAs of (r, b), y slot block j, tile t
  const int q = (int)rank % CPR, j = q / TPB, t = q - j * TPB;
  const int cl = (int)blockIdx.x / CPR;   // MODE > 0: cluster index (clusters of CPR CTAs)
  const int r = C::LOCAL ? (int)rank / CPR : cl / MB, b = C::LOCAL ? 0 : cl % MB;
  const int koffb = !C::LOCAL && b >= MB / 2 ? H : 0;
  unsigned long long* ctr_src = a.gbar + 16;          // [CPR]
  unsigned long long* ctr_p = ctr_src + 16 * CPR;     // [R][MB]

  if (threadIdx.x == 0) {
    for (const CUtensorMap* m : {&x0h, &x0l, &x1h, &x1l}) prefetch_map(m);
    for (int k = 0; k < NK; ++k) mbar_init(full0 + 8 * k, 1);
    mbar_init(done, 1);
    mbar_init(tbar, 128);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  if (!C::LOCAL && cl >= a.R * MB) {
    // clusters beyond the products' only form sources (256^2, two right-hand sides: 32 CTAs multiply)
    if (warp < 8) {
      solve_sources_any<BN>(a, reinterpret_cast<float*>(basep + C::SRC), ctr_src);
      if (threadIdx.x == 0) {
        const unsigned long long seen = atomicAdd(a.gbar, 1ull);
        if (seen == gridDim.x - 1ull) {
          for (int i = 0; i < CPR + a.R * MB; ++i) ctr_src[16 * i] = 0ull;
          atomicExch(a.gbar, 0ull);
        }
      }
      main_sync();
      if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    } else if (a.reset_late) {
      const int first = a.R * MB * CPR;
      reset_nodes(a, ((int)blockIdx.x - first) * 128 + (int)threadIdx.x - 256, ((int)gridDim.x - first) * 128);
    }
    return;
  }
  cl_arrive();   // barrier 0: every CTA of the cluster runs

  if (warp >= 8) {
    // the x slice (block b) and the y slice (block j)
    fill_tmem<K>(fxt, b, tmem + C::TX, warp & 3, lane);
    fill_tmem<K>(fyt, j, tmem + C::TY, warp & 3, lane);
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    tc_fence_before();
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tbar) : "memory");
    cl_wait();
    for (int k = 1; k < C::barriers(a.pre); ++k) {
      cl_arrive();
      cl_wait();
    }
    return;
  }

  bool started = false;   // barrier 0 waited for
  if (a.pre) {
    if constexpr (C::LOCAL) {
      cl_wait();
      started = true;
      float* S = reinterpret_cast<float*>(basep + C::SRC);
      if (a.pre == 1) cl_sources<BN, C::FOLD, SrcMain<float>, 3>(a.sm.gm, a.sm, S, a.R, r, q, buf0);
      else if (a.pre == 2) cl_sources<BN, C::FOLD, SrcBperp<float>, 2>(a.sb.gm, a.sb, S, a.R, r, q, buf0);
      else cl_sources<BN, C::FOLD, SrcGiven, kMaxRhs>(a.sc.gm, a.sc, S, a.R, r, q, buf0);
      asm volatile("fence.proxy.async.shared::cluster;" ::: "memory");
      cl_arrive();
      cl_wait();
      asm volatile("fence.proxy.async.shared::cluster;" ::: "memory");
    } else {
      solve_sources_any<BN>(a, reinterpret_cast<float*>(basep + C::SRC), ctr_src);
    }
  }
  const int row = (warp & 3) * 32 + lane, half = warp >> 2;
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const bool along_x = (p & 1) == 0;
    const bool exchange = p < 3 && (C::LOCAL || p != 1);   // the next operand goes to the cluster's peers
    const uint32_t buf = along_x ? buf0 : buf1;
    const bool load = p == 0 ? (!C::LOCAL || !a.pre) : (p == 2 && !C::LOCAL);   // the operand comes by TMA
    if (p == 3) pdl_trigger();
    if (warp == 0 && lane == 0 && load) {
      bool ok = true;
      if (p == 0 && a.pre && !C::LOCAL)
        ok = dep_wait(ctr_src + 16 * q, (unsigned long long)(BN / kSrcRows) + (unsigned)a.barrier_skew, a.status, abort_f);
      if (p == 2)
        ok = dep_wait(ctr_p + 16 * (r * MB + j), (unsigned long long)CPR + (a.pre ? 0u : (unsigned)a.barrier_skew), a.status,
                      abort_f);
      const CUtensorMap* mh = p == 0 ? &x0h : &x1h;
      const CUtensorMap* ml = p == 0 ? &x0l : &x1l;
      for (int kb = 0; ok && kb < NK; ++kb) {
        const uint32_t fb = full0 + 8 * kb;
        mbar_expect_tx(fb, C::STAGE);
        tma_load_2d(buf + kb * C::STAGE, mh, koffb + kb * BK, r * N + q * BN, fb);
        tma_load_2d(buf + kb * C::STAGE + BN * 128, ml, koffb + kb * BK, r * N + q * BN, fb);
      }
    } else if (warp == 1) {
      bool ok = true;
      if (p == 0) ok = mbar_wait_a(tbar, 0, a.status, abort_f);
      ok = __all_sync(0xffffffffu, ok);
      for (int kb = 0; ok && kb < NK; ++kb) {
        if (load) ok = __all_sync(0xffffffffu, mbar_wait_a(full0 + 8 * kb, (uint32_t)(p >> 1), a.status, abort_f));
        if (!ok) break;
        tc_fence_after();
        const uint64_t bh = desc_k_sw128(buf + kb * C::STAGE);
        const uint32_t ta = tmem + (along_x ? C::TX : C::TY) + (uint32_t)(kb * 32);
        if (elect_one()) {
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) {
            const uint64_t off = (uint64_t)((k * 32) >> 4);
            const uint32_t on = (kb | k) != 0 ? 1u : 0u;
            if constexpr (C::LOCAL) {
              // F_hi X_hi + F_hi X_lo and, apart, F_lo X_hi: the streamed solve's order of additions
              // (the faster grouping below flips last bits of the splits)
              mma_bf16_ta(tmem, ta + 8u * k, bh + off, Cfg<BN>::IDESC, on);
              mma_bf16_ta(tmem, ta + 8u * k, bh + off + (uint64_t)((BN * 128) >> 4), Cfg<BN>::IDESC, 1u);
              mma_bf16_ta(tmem + BN, ta + (uint32_t)(K / 2) + 8u * k, bh + off, Cfg<BN>::IDESC, on);
            } else {
              mma_bf16_ta(tmem, ta + 8u * k, bh + off, Cfg<BN>::IDESC2, on);
              mma_bf16_ta(tmem, ta + (uint32_t)(K / 2) + 8u * k, bh + off, Cfg<BN>::IDESC, 1u);
            }
          }
        }
        __syncwarp();
      }
      if (elect_one()) mma_commit(done);
    }
    __syncwarp();
    // output slot of this thread's lane and its first data row
    const int s = (along_x ? b : j) * BM + row;
    const int i0 = (along_x ? q * BN : b * BM + t * BN) + half * CH;
    float sc[CH];
    if (p == 1) {
      const float4* f4 = reinterpret_cast<const float4*>(a.scale + (int64_t)s * N + i0);
#pragma unroll
      for (int k = 0; k < CH / 4; ++k) {
        const float4 f = __ldg(f4 + k);
        sc[4 * k] = f.x;
        sc[4 * k + 1] = f.y;
        sc[4 * k + 2] = f.z;
        sc[4 * k + 3] = f.w;
      }
    }
    mbar_wait_a(done, (uint32_t)(p & 1), a.status, abort_f);
    tc_fence_after();
    float x[CH];
    tmem_ld_pair<BN, CH>(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(half * CH), x);
    tc_fence_before();
    if (p == 3) {
      float* tile = reinterpret_cast<float*>(basep + C::DATA);
      constexpr int LD = BN + 1;
#pragma unroll
      for (int k = 0; k < CH; ++k) tile[row * LD + half * CH + k] = x[k];
      main_sync();
      if (!*abort_f) cl_out<BN, MODE, RES>(a, tile, j, b, t, r);
      break;
    }
    if (p == 1) {
#pragma unroll
      for (int k = 0; k < CH; ++k) x[k] *= sc[k];
    }
    if (exchange) {
      if (!started) {
        cl_wait();
        started = true;
      }
      // the peers' buffer must be drained of their MMAs: with one buffer those of this product, with
      // two those of product 1 (whose end this CTA announced below)
      if (!C::DB) {
        cl_arrive();
        cl_wait();
      } else if (!C::LOCAL && p == 2) {
        cl_wait();
      }
      const uint32_t dst = along_x ? buf1 : buf0;
      if constexpr (C::FOLD) {
        const int v0 = i0 >> 1, cs = row;
        const int col = p == 2 ? cl_col(cs) : cs, tt = col / BN, orow = col - tt * BN;
        float sum[CH / 2], dif[CH / 2];
#pragma unroll
        for (int k = 0; k < CH / 2; ++k) {
          const bool wall = v0 + k == N / 4;
          sum[k] = wall ? x[2 * k + 1] : x[2 * k] + x[2 * k + 1];
          dif[k] = wall ? 0.0f : x[2 * k] - x[2 * k + 1];
        }
#pragma unroll
        for (int c = 0; c < CH / 2; c += 8) {
          if constexpr (C::LOCAL) {
            put_operand8<BN>(dst, (uint32_t)(r * CPR + tt), orow, v0 + c, sum + c);
            put_operand8<BN>(dst, (uint32_t)(r * CPR + tt), orow, H + v0 + c, dif + c);
          } else {
            put_operand8<BN>(dst, (uint32_t)tt, orow, v0 + c, sum + c);
            put_operand8<BN>(dst, (uint32_t)(TPB + tt), orow, v0 + c, dif + c);
          }
        }
      } else {
        const int tt = row / BN;
#pragma unroll
        for (int c = 0; c < CH; c += 8) put_operand8<BN>(dst, (uint32_t)(r * CPR + tt), row - tt * BN, i0 + c, x + c);
      }
      asm volatile("fence.proxy.async.shared::cluster;" ::: "memory");
      cl_arrive();
      cl_wait();
      asm volatile("fence.proxy.async.shared::cluster;" ::: "memory");
      tc_fence_after();
    } else {
      // product 1 of several clusters: through global memory, counted per slot block of y
      if (C::DB) cl_arrive();   // this CTA's product 1 has read its buffer
      if (!*abort_f)
        rs_epilogue<CH>(a, 0, s, s, r, i0, x, sc, reinterpret_cast<__nv_bfloat16*>(a.op_hi[1]),
                        reinterpret_cast<__nv_bfloat16*>(a.op_lo[1]));
      asm volatile("fence.proxy.async.global;" ::: "memory");
      main_sync();
      tc_fence_after();
      if (threadIdx.x == 0 && !*abort_f) dep_arrive(ctr_p + 16 * (r * MB + j));
    }
  }
  if (!C::LOCAL && threadIdx.x == 0 && !*abort_f) {
    // the last CTA through resets the counters for the next launch
    const unsigned long long seen = atomicAdd(a.gbar, 1ull);
    if (seen == gridDim.x - 1ull) {
      for (int i = 0; i < CPR + a.R * MB; ++i) ctr_src[16 * i] = 0ull;
      atomicExch(a.gbar, 0ull);
    }
  }
  tc_fence_before();
  main_sync();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

// ---------------------------------------------------------------- wide solve
// The same four products for grids with more than three 128 x 64 tiles per SM (1536^2 with two
// right-hand sides): 128 x 128 tiles with the roles of the resident solve (A = 128 slots of the
// fold or sine matrix, B = [X_hi; X_lo] of 128 data rows, N = 256, then A_lo x X_hi with N = 128),
// both streamed.  Here the products themselves cost something (206 GFLOP at 2048^2, two right-hand
// sides: 109 us at the measured bf16 rate; a K step reads 20 KB of operands from shared memory, which
// bounds it at ~340 clocks against 192 of tensor-core work), so loads, MMAs and epilogues run in warps of their own: two
// accumulators in tensor memory let a tile's epilogue run beside the next one's MMAs, and only the
// TMA producer waits for the other CTAs between products.
// Warps 0-7: sources and epilogues; warp 8: TMA producer (3-stage ring of A_hi, A_lo, X_hi, X_lo K
// blocks, 64 KB); warp 9: MMA issuer.
constexpr int kWideThreads = 320;
template <typename E> struct Wide {
  static constexpr int BN = 128, STAGES = 3, STAGE_BYTES = 4 * A_BYTES;
  static constexpr int TILE = STAGES * STAGE_BYTES, LD = 65;   // the mixing's staged columns, 128 x 64
  static constexpr int BARS = TILE + BM * LD * 4;
  static constexpr int BYTES = BARS + 256 + 1024;
};

// 32 consecutive data columns i0 .. of slot s into the next operand's row: ns slots, nd data rows per
// right-hand side; folded, adjacent columns are a pair (see rs_epilogue).
template <typename E>
__device__ __forceinline__ void wide_store(E* oh, E* ol, int fold, int r, int orow, int i0, int ns, int nd, const float* x) {
  const int64_t base = ((int64_t)r * ns + orow) * nd;
  if (fold) {
    const int v0 = i0 >> 1, H = nd / 2;
    float sum[16], dif[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const bool wall = v0 + k == nd / 4;
      sum[k] = wall ? x[2 * k + 1] : x[2 * k] + x[2 * k + 1];
      dif[k] = wall ? 0.0f : x[2 * k] - x[2 * k + 1];
    }
#pragma unroll
    for (int k = 0; k < 16; k += 8) {
      put_run8(oh + base + v0 + k, ol + base + v0 + k, sum + k);
      put_run8(oh + base + H + v0 + k, ol + base + H + v0 + k, dif + k);
    }
  } else {
#pragma unroll
    for (int k = 0; k < 32; k += 8) put_run8(oh + base + i0 + k, ol + base + i0 + k, x + k);
  }
}

template <bool RES, typename E>
__global__ void __launch_bounds__(kWideThreads, 1)
    k_dst_solve_wide(const __grid_constant__ CUtensorMap fxh, const __grid_constant__ CUtensorMap fxl,
                     const __grid_constant__ CUtensorMap fyh, const __grid_constant__ CUtensorMap fyl,
                     const __grid_constant__ CUtensorMap x0h, const __grid_constant__ CUtensorMap x0l,
                     const __grid_constant__ CUtensorMap x1h, const __grid_constant__ CUtensorMap x1l, const SolveArgs a) {
  using W = Wide<E>;
  using C = Cfg<W::BN, E>;
  constexpr int BN = W::BN, STAGES = W::STAGES, KE = kb_elems<E>();
  extern __shared__ uint8_t smem_raw[];
  __shared__ int s_abort;
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* basep = smem_raw + (base - raw);
  uint64_t* bars = reinterpret_cast<uint64_t*>(basep + W::BARS);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 5);
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + STAGES), tfull0 = smem_u32(bars + 2 * STAGES),
                 tempty0 = smem_u32(bars + 2 * STAGES + 2), drain = smem_u32(bars + 2 * STAGES + 4);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort_f = &s_abort;
  if (threadIdx.x == 0) {
    for (const CUtensorMap* m : {&fxh, &fxl, &fyh, &fyl, &x0h, &x0l, &x1h, &x1l}) prefetch_map(m);
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(tfull0 + 8 * s, 1);
      mbar_init(tempty0 + 8 * s, kSolveThreads);
    }
    mbar_init(drain, 1);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const unsigned nb0 = a.pre ? 1u : 0u;   // barriers before the first product
  // product p: slots and data rows per right-hand side, tiles (slot block fastest), K blocks
  struct Geo {
    int ns, nd, mt, tiles, nk;
  };
  auto geo = [&](int p) {
    Geo g;
    const bool ax = (p & 1) == 0;
    g.ns = ax ? a.nxp : a.nyp;
    g.nd = ax ? a.nyp : a.nxp;
    g.mt = g.ns / BM;
    g.tiles = g.mt * (a.R * g.nd / BN);
    g.nk = (a.fold ? g.ns / 2 : g.ns) / KE;
    return g;
  };

  if (warp == 8) {
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int p = 0; p < 4 && ok; ++p) {
        const Geo g = geo(p);
        const CUtensorMap *fh = p & 1 ? &fyh : &fxh, *fl = p & 1 ? &fyl : &fxl, *xh = p & 1 ? &x1h : &x0h, *xl = p & 1 ? &x1l : &x0l;
        const unsigned nbar = nb0 + (unsigned)p;   // barriers to pass
        if (nbar > 0) ok = dep_wait(a.gbar, (unsigned long long)nbar * gridDim.x + (nbar == 1 ? (unsigned)a.barrier_skew : 0u),
                                    a.status, abort_f);
        for (int tile = blockIdx.x; ok && tile < g.tiles; tile += gridDim.x) {
          const int s0 = (tile % g.mt) * BM, c0 = (tile / g.mt) * BN;
          const int koff = (a.fold && s0 >= g.ns / 2) ? g.ns / 2 : 0;
          for (int kb = 0; kb < g.nk; ++kb, ++it) {
            const uint32_t s = it % STAGES, st = base + s * W::STAGE_BYTES, fb = full0 + 8 * s;
            if (it >= (uint32_t)STAGES && !mbar_wait_a(empty0 + 8 * s, ((it / STAGES) - 1) & 1, a.status, abort_f)) {
              ok = false;
              break;
            }
            mbar_expect_tx(fb, W::STAGE_BYTES);
            tma_load_2d(st, fh, kb * KE, s0, fb);
            tma_load_2d(st + A_BYTES, fl, kb * KE, s0, fb);
            tma_load_2d(st + 2 * A_BYTES, xh, koff + kb * KE, c0, fb);
            tma_load_2d(st + 3 * A_BYTES, xl, koff + kb * KE, c0, fb);
          }
        }
      }
      // every load has landed before the CTA may leave
      for (uint32_t k = it > (uint32_t)STAGES ? it - STAGES : 0; k < it; ++k)
        mbar_wait(full0 + 8 * (k % STAGES), (k / STAGES) & 1, a.status);
    }
  } else if (warp == 9) {
    uint32_t it = 0, t = 0;
    bool ok = true;
    for (int p = 0; p < 4 && ok; ++p) {
      const Geo g = geo(p);
      for (int tile = blockIdx.x; ok && tile < g.tiles; tile += gridDim.x, ++t) {
        const uint32_t acc = t & 1, d = tmem + acc * (2 * BN);
        if (t >= 2) ok = __all_sync(0xffffffffu, mbar_wait_a(tempty0 + 8 * acc, ((t >> 1) - 1) & 1, a.status, abort_f));
        tc_fence_after();
        for (int kb = 0; ok && kb < g.nk; ++kb, ++it) {
          const uint32_t s = it % STAGES;
          ok = __all_sync(0xffffffffu, mbar_wait_a(full0 + 8 * s, (it / STAGES) & 1, a.status, abort_f));
          if (!ok) break;
          tc_fence_after();
          const uint32_t st = base + s * W::STAGE_BYTES;
          const uint64_t ah = desc_k_sw128(st), al = desc_k_sw128(st + A_BYTES), bh = desc_k_sw128(st + 2 * A_BYTES);
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const uint64_t off = (uint64_t)((k * 32) >> 4);
              mma_op<E>(d, ah + off, bh + off, C::IDESC2, (kb | k) != 0 ? 1u : 0u);
              mma_op<E>(d, al + off, bh + off, C::IDESC, 1u);
            }
            mma_commit(empty0 + 8 * s);
          }
          __syncwarp();
        }
        if (elect_one()) mma_commit(tfull0 + 8 * acc);
        __syncwarp();
      }
    }
    if (elect_one()) mma_commit(drain);
    __syncwarp();
    mbar_wait(drain, 0, a.status);
  } else {
    if (a.pre) {
      solve_sources_all<E>(a);
      asm volatile("fence.proxy.async.global;" ::: "memory");
      main_sync();
      if (threadIdx.x == 0) dep_arrive(a.gbar);
    }
    float* tilebuf = reinterpret_cast<float*>(basep + W::TILE);
    const int row = (warp & 3) * 32 + lane, half = warp >> 2;
    const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    uint32_t t = 0;
    float d2 = 0.0f, b2 = 0.0f;
    bool bad = false;
    // (after an abort the phases run through on waits that fail at once: the named barriers stay
    // matched, nothing is reported or stored as a result)
    for (int p = 0; p < 4; ++p) {
      const Geo g = geo(p);
      const int mode = p == 3 ? a.final_mode : (p == 1 ? 1 : 0);
      if (p == 3) pdl_trigger();
      E* oh = reinterpret_cast<E*>(a.op_hi[(p + 1) & 1]);
      E* ol = reinterpret_cast<E*>(a.op_lo[(p + 1) & 1]);
      for (int tile = blockIdx.x; tile < g.tiles; tile += gridDim.x, ++t) {
        const int s0 = (tile % g.mt) * BM, c0 = (tile / g.mt) * BN, r = c0 / g.nd, i00 = c0 - r * g.nd;
        const uint32_t acc = t & 1;
        const int s = s0 + row;
        mbar_wait_a(tfull0 + 8 * acc, (t >> 1) & 1, a.status, abort_f);
        tc_fence_after();
#pragma unroll 1
        for (int q = 0; q < 2; ++q) {
          const int cc = half * 64 + q * 32, i0 = i00 + cc;
          float x[32];
          tmem_ld_pair<BN, 32>(tl + acc * (2 * BN) + (uint32_t)cc, x);
          if (q == 1) {
            // both chunks of this thread are out of the accumulator
            tc_fence_before();
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tempty0 + 8 * acc) : "memory");
          }
          if (mode <= 1) {
            if (mode == 1) {   // [nyp][nxp]: this slot's row of the factors
              const float4* sc = reinterpret_cast<const float4*>(a.scale + (int64_t)s * a.nxp + i0);
#pragma unroll
              for (int k = 0; k < 8; ++k) {
                const float4 f = __ldg(sc + k);
                x[4 * k] *= f.x;
                x[4 * k + 1] *= f.y;
                x[4 * k + 2] *= f.z;
                x[4 * k + 3] *= f.w;
              }
            }
            // the third product's rows in node order: the last one's columns are consecutive x nodes
            const int orow = p == 2 && a.fold ? fold_node(s, g.ns) : s;
            wide_store<E>(oh, ol, a.fold, r, orow, i0, g.ns, g.nd, x);
            continue;
          }
          // result: staged, so that consecutive threads take consecutive nodes of a row
#pragma unroll
          for (int k = 0; k < 32; ++k) tilebuf[row * W::LD + half * 32 + k] = x[k];
          main_sync();
          constexpr int UN = 16;
          for (int e0 = threadIdx.x; e0 < BM * 64; e0 += UN * kSolveThreads) {
            float v[UN], old[UN];
            int64_t at[UN];
#pragma unroll
            for (int k = 0; k < UN; ++k) {
              const int e = e0 + k * kSolveThreads, rr = e >> 6, jj = e & 63;
              const int y = a.fold ? fold_node(s0 + rr, a.ny) : s0 + rr, xx = i00 + (jj >> 5) * 64 + q * 32 + (jj & 31);
              v[k] = tilebuf[rr * W::LD + jj];
              at[k] = (y < a.ny && xx < a.nx && !*abort_f) ? (int64_t)y * a.nx + xx : -1;
              if (mode == 3) old[k] = at[k] >= 0 ? a.bm[at[k] * 2 + r] : 0.0f;
            }
#pragma unroll
            for (int k = 0; k < UN; ++k) {
              if (at[k] < 0) continue;
              if (mode == 2) {
                a.out[(int64_t)r * a.ny * a.nx + at[k]] = v[k];
                continue;
              }
              bad |= !isfinite(v[k]);
              const float nb = a.w * v[k] + (1.0f - a.w) * old[k];
              a.bm[at[k] * 2 + r] = nb;
              if constexpr (RES) {
                const float d = nb - old[k];
                d2 += d * d;
                b2 += nb * nb;
              }
            }
          }
          main_sync();
        }
      }
      if (p < 3) {
        asm volatile("fence.proxy.async.global;" ::: "memory");
        main_sync();
        if (threadIdx.x == 0 && !*abort_f) dep_arrive(a.gbar);
      }
    }
    if (bad) atomicOr(a.status, DEV_NONFINITE);
    if constexpr (RES) residual_add_main(a.rsum, (double)d2, (double)b2);
  }
  tc_fence_before();
  __syncthreads();
  // exit arrival: the last CTA through resets the counter for the next launch
  if (threadIdx.x == 0 && !*abort_f) {
    const unsigned long long seen = atomicAdd(a.gbar, 1ull);
    if (seen == (nb0 + 4ull) * gridDim.x - 1ull) atomicExch(a.gbar, 0ull);
  }
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                              const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                              CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// A split operand [rows][cols] in 128B-swizzled boxes of one K block (128 bytes) by box_rows:
// bf16 elements, or (tf32) FP32 words.
int make_map(EncodeFn enc, CUtensorMap* map, void* ptr, uint64_t rows, uint64_t cols, std::string& err,
             uint32_t box_rows = 128, bool tf32 = false) {
  const uint32_t es = tf32 ? 4 : 2;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * es};
  cuuint32_t box[2] = {128 / es, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult rc = enc(map, tf32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ptr, dims,
                    strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (rc != CUDA_SUCCESS) {
    err = "cuTensorMapEncodeTiled failed (" + std::to_string((int)rc) + ")";
    return 1;
  }
  return 0;
}

// Unswizzled map with an arbitrary box (the FP32 scale tile).
int make_map_plain(EncodeFn enc, CUtensorMap* map, CUtensorMapDataType dt, uint32_t esize, void* ptr, uint64_t rows,
                   uint64_t cols, uint32_t box_x, uint32_t box_y, std::string& err) {
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * esize};
  cuuint32_t box[2] = {box_x, box_y};
  cuuint32_t estr[2] = {1, 1};
  CUresult rc = enc(map, dt, 2, ptr, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (rc != CUDA_SUCCESS) {
    err = "cuTensorMapEncodeTiled failed (" + std::to_string((int)rc) + ")";
    return 1;
  }
  return 0;
}

// N-tile width: 64 when 128-wide tiles would leave most of the 152 SMs idle.
inline int pick_bn(int M, int N) { return (M / BM) * (N / 128) < 152 ? 64 : 128; }

void gemm(const CUtensorMap& ah, const CUtensorMap& al, const CUtensorMap* bh, const CUtensorMap* bl, int M, int N,
          int K, const Epi& ep, int* status, cudaStream_t s) {
  if (pick_bn(M, N) == 128) {
    dim3 grid((unsigned)(M / BM), (unsigned)(N / 128));
    launch_pdl(k_dst_gemm<128>, grid, dim3(128), (size_t)Cfg<128>::SMEM_BYTES, s, ah, al, bh[0], bl[0], K, ep, status);
  } else {
    dim3 grid((unsigned)(M / BM), (unsigned)(N / 64));
    launch_pdl(k_dst_gemm<64>, grid, dim3(128), (size_t)Cfg<64>::SMEM_BYTES, s, ah, al, bh[1], bl[1], K, ep, status);
  }
}

}  // namespace

bool dst_tc_resident(const hq_grid_s* g) {
  const char* nors = std::getenv("HQ_NO_RS");
  return !g->fp64 && !g->tf32 && g->fold && g->nx == g->ny && (g->nx == 256 || g->nx == 512) && !(nors && nors[0] == '1');
}

int dst_tc_cluster_mode(const hq_grid_s* g) {
  const char* nc = std::getenv("HQ_NO_CLUSTER");
  const char* nors = std::getenv("HQ_NO_RS");
  const char* bn = std::getenv("HQ_SOLVE_BN");
  if (g->fp64 || g->tf32 || (nc && nc[0] == '1') || (nors && nors[0] == '1') || (bn && std::atoi(bn) == 64)) return -1;
  if (g->nx <= 128 && g->ny <= 128) return g->fault_barrier ? -1 : (g->fold ? 2 : 0);   // (one cluster: no counter to fail)
  if (!g->fold || g->nx != g->ny) return -1;
  return g->nx == 256 ? 1 : -1;
}

namespace {
template <int BN, int N, bool RES> auto* rs_kernel() { return &k_dst_solve_rs<BN, N, RES>; }
template <int BN, int MODE, bool RES> auto* cl_kernel() { return &k_dst_solve_cl<BN, MODE, RES>; }

static_assert(SolveSmem<64>::BYTES <= kSmemAll && SolveSmem<32>::BYTES <= kSmemAll && Wide<float>::BYTES <= kSmemAll &&
                  RsSmem<64>::BYTES <= kSmemAll && Cl<64, 0>::BYTES <= kSmemAll && Cl<32, 1>::BYTES <= kSmemAll,
              "a solve kernel needs more than a launch can request");
template <typename K> bool by_registers(K kern, int threads) {
  cudaFuncAttributes fa;
  if (cudaFuncGetAttributes(&fa, kern) == cudaSuccess) return alone_by_registers(fa.numRegs, threads);
  cudaGetLastError();
  return false;
}

// Right-hand sides whose clusters fit the GPU at once (0: none).
template <int BN, int MODE, bool RES> int cl_capacity(bool& all_smem, int* most = nullptr) {
  using C = Cl<BN, MODE>;
  auto kern = cl_kernel<BN, MODE, RES>();
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemAll) != cudaSuccess ||
      cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  all_smem |= !by_registers(kern, kClThreads);
  int best = 0;
  for (int R = 1; R <= kMaxRhs; ++R) {
    const int cs = C::LOCAL ? R * C::CPR : C::CPR, need = C::LOCAL ? 1 : R * C::MB;
    if (cs > 16) break;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(cs * need));
    cfg.blockDim = dim3(kClThreads);
    cfg.dynamicSmemBytes = kSmemAll;   // (one CTA per SM, whatever it requests)
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cs;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
      cudaGetLastError();
      break;
    }
    if (most) *most = n;
    if (n < need) break;
    best = R;
  }
  return best;
}
}  // namespace

int dst_tc_init(hq_grid_s* g, std::string& err) {
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
      fn == nullptr || q != cudaDriverEntryPointSuccess) {
    err = "cuTensorMapEncodeTiled not available from the driver";
    return 1;
  }
  EncodeFn enc = reinterpret_cast<EncodeFn>(fn);
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, g->dev) != cudaSuccess) {
    err = "cannot read the SM count";
    return 1;
  }
  g->tmaps = new TensorMaps();
  TensorMaps& t = *g->tmaps;
  t.all_smem = false;
  auto size_solve = [&](auto kern, int& ctas, int threads = kSolveThreads) {
    int per_sm = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemAll) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, kSmemAll) != cudaSuccess || per_sm < 1) {
      err = "cannot size the cooperative DST solve";
      return false;
    }
    t.all_smem |= !by_registers(kern, threads);
    ctas = sms;   // one CTA per SM
    return true;
  };
  int spare = 0;   // the residual-accumulating instances (the last P-C iteration): same resources
  const bool tf = g->tf32 != 0;
  using B16 = __nv_bfloat16;
  if (tf ? !(size_solve(k_dst_solve<64, false, float>, t.ctas[0]) && size_solve(k_dst_solve<32, false, float>, t.ctas[1]) &&
             size_solve(k_dst_solve<64, true, float>, spare) && size_solve(k_dst_solve<32, true, float>, spare) &&
             size_solve(k_dst_solve_wide<false, float>, t.wide_ctas, kWideThreads) &&
             size_solve(k_dst_solve_wide<true, float>, spare, kWideThreads))
         : !(size_solve(k_dst_solve<64, false, B16>, t.ctas[0]) && size_solve(k_dst_solve<32, false, B16>, t.ctas[1]) &&
             size_solve(k_dst_solve<64, true, B16>, spare) && size_solve(k_dst_solve<32, true, B16>, spare) &&
             size_solve(k_dst_solve_wide<false, B16>, t.wide_ctas, kWideThreads) &&
             size_solve(k_dst_solve_wide<true, B16>, spare, kWideThreads)))
    return 1;
  const char* bn = std::getenv("HQ_SOLVE_BN");
  t.wide_only = bn != nullptr && std::atoi(bn) == 64;
  // (the resident fold matrix is bf16: as TF32 words, hi and lo, it would fill tensor memory at 512^2)
  t.rs = dst_tc_resident(g);
  auto size_rs = [&](auto* w0, auto* n0, auto* w1, auto* n1) {
    return size_solve(w0, t.rs_ctas[0], kClThreads) && size_solve(n0, t.rs_ctas[1], kClThreads) &&
           size_solve(w1, spare, kClThreads) && size_solve(n1, spare, kClThreads);
  };
  if (t.rs && !(g->nx == 512 ? size_rs(rs_kernel<64, 512, false>(), rs_kernel<32, 512, false>(), rs_kernel<64, 512, true>(),
                                       rs_kernel<32, 512, true>())
                             : size_rs(rs_kernel<64, 256, false>(), rs_kernel<32, 256, false>(), rs_kernel<64, 256, true>(),
                                       rs_kernel<32, 256, true>())))
    return 1;
  t.cl_mode = dst_tc_cluster_mode(g);
  t.cl_rhs[0] = t.cl_rhs[1] = t.cl_max = 0;
  if (t.cl_mode == 0) {
    t.cl_rhs[0] = std::min(cl_capacity<32, 0, false>(t.all_smem), cl_capacity<32, 0, true>(t.all_smem));
    t.cl_rhs[1] = cl_capacity<64, 0, false>(t.all_smem);
  } else if (t.cl_mode == 2) {
    t.cl_rhs[0] = std::min(cl_capacity<32, 2, false>(t.all_smem), cl_capacity<32, 2, true>(t.all_smem));
    t.cl_rhs[1] = cl_capacity<64, 2, false>(t.all_smem);
  } else if (t.cl_mode == 1) {
    t.cl_rhs[0] = std::min(cl_capacity<32, 1, false>(t.all_smem, &t.cl_max), cl_capacity<32, 1, true>(t.all_smem));
  }
  const uint64_t nxp = g->nxp, nyp = g->nyp;
  int bad = 0;
  bad |= make_map(enc, &t.a0_hi, g->op_hi[0], kMaxRhs * nyp, nxp, err, 128, tf);
  bad |= make_map(enc, &t.a0_lo, g->op_lo[0], kMaxRhs * nyp, nxp, err, 128, tf);
  bad |= make_map(enc, &t.a1_hi, g->op_hi[1], kMaxRhs * nxp, nyp, err, 128, tf);
  bad |= make_map(enc, &t.a1_lo, g->op_lo[1], kMaxRhs * nxp, nyp, err, 128, tf);
  // S_x, S_y (or the fold matrices, half as wide) as [rows][K]
  const uint64_t kx = g->fold ? nxp / 2 : nxp, ky = g->fold ? nyp / 2 : nyp;
  bad |= make_map(enc, &t.fx_hi, g->sx_hi, nxp, kx, err, 128, tf);
  bad |= make_map(enc, &t.fx_lo, g->sx_lo, nxp, kx, err, 128, tf);
  bad |= make_map(enc, &t.fy_hi, g->sy_hi, nyp, ky, err, 128, tf);
  bad |= make_map(enc, &t.fy_lo, g->sy_lo, nyp, ky, err, 128, tf);
  for (int i = 0; i < 2; ++i) {
    const uint32_t bn = i == 0 ? 64 : 32;
    bad |= make_map(enc, &t.bx_hi[i], g->sx_hi, nxp, kx, err, bn, tf);
    bad |= make_map(enc, &t.bx_lo[i], g->sx_lo, nxp, kx, err, bn, tf);
    bad |= make_map(enc, &t.by_hi[i], g->sy_hi, nyp, ky, err, bn, tf);
    bad |= make_map(enc, &t.by_lo[i], g->sy_lo, nyp, ky, err, bn, tf);
    bad |= make_map_plain(enc, &t.scale[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, g->f32_scale, nyp, nxp, BM, bn, err);
    if (g->scale_h)
      bad |= make_map_plain(enc, &t.scale_h[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, g->scale_h, nyp, nxp, BM, bn, err);
  }
  if (t.rs || t.cl_mode >= 0) {
    for (int o = 0; o < (t.rs ? 3 : 2); ++o)
      for (int i = 0; i < 2; ++i) {
        const uint32_t bn = i == 0 ? 64 : 32;
        bad |= make_map(enc, &t.rx_hi[o][i], g->op_hi[o], kMaxRhs * nyp, nxp, err, bn);
        bad |= make_map(enc, &t.rx_lo[o][i], g->op_lo[o], kMaxRhs * nyp, nxp, err, bn);
      }
  }
  return bad;
}

void dst_tc_free(hq_grid_s* g) {
  delete g->tmaps;
  g->tmaps = nullptr;
}

namespace {

// One cooperative launch of k_dst_solve: on the sources in op[0] (pre = 0), or forming them
// first from the deposit records (pre = 1: psi, Ez, Bz of dep_cur; pre = 2: B_perp).
void solve_fused(hq_grid_s* g, int R, int final_mode, int last, cudaStream_t s, int pre = 0,
                 const void* dep_cur = nullptr, void* dep_prev = nullptr, void* chi_prev = nullptr,
                 bool shifted = false, const float* src = nullptr, float* dst = nullptr) {
  const TensorMaps& t = *g->tmaps;
  SolveArgs a{};
  a.R = R;
  a.nxp = g->nxp;
  a.nyp = g->nyp;
  a.fold = g->fold;
  a.op_hi[0] = g->op_hi[0];
  a.op_lo[0] = g->op_lo[0];
  a.op_hi[1] = g->op_hi[1];
  a.op_lo[1] = g->op_lo[1];
  a.op_hi[2] = g->op_hi[2];
  a.op_lo[2] = g->op_lo[2];
  a.scale = reinterpret_cast<const float*>(shifted ? g->scale_h : g->f32_scale);
  a.final_mode = final_mode;
  a.out = dst ? dst : reinterpret_cast<float*>(g->solved);
  a.nx = g->nx;
  a.ny = g->ny;
  a.bm = reinterpret_cast<float*>(g->bm);
  a.w = (float)g->d.pc_mix;
  a.rsum = g->pc_rsum;
  a.gbar = g->d_gbar;
  a.status = g->d_status;
  a.barrier_skew = g->fault_barrier;
  a.pre = pre;
  if (pre == 1) a.sm = src_main_of<float>(g, dep_cur);
  if (pre == 2) a.sb = src_bperp_of<float>(g, dep_cur, dep_prev, chi_prev, last);
  if (pre == 3) a.sc = SrcGiven{src, g->geom, R};
  const auto smem_of = [&](int need) { return (size_t)(t.all_smem ? kSmemAll : need); };
  auto late_reset = [&]() {
    if (pre == 2 && a.sb.reset_prev && a.sb.mode == 2) {
      a.sb.reset_prev = 0;
      a.reset_late = 1;
    }
  };
  if (t.cl_mode >= 0 && (R <= t.cl_rhs[0] || (R <= t.cl_rhs[1] && !a.rsum))) {
    const bool local = t.cl_mode != 1;
    const int v = R <= t.cl_rhs[0] ? 1 : 0, BNv = v ? 32 : 64, N = local ? 128 : 256;
    const int cpr = N / BNv, cs = local ? R * cpr : cpr;
    cudaLaunchConfig_t cfg = {};
    // (mode 1 with sources: at least a CTA per kSrcRows source rows)
    const int ctas = local ? cs : std::max(R * (N / BM) * cpr, pre ? std::min(N / kSrcRows, t.cl_max * cs) : 0);
    cfg.gridDim = dim3((unsigned)ctas);
    if (t.cl_mode == 1 && ctas > R * (N / BM) * cpr) late_reset();
    cfg.blockDim = dim3(kClThreads);
    cfg.stream = s;
    // cooperative: clusters wait for each other (the single cluster of a local solve does not)
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cs;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeCooperative;
    at[1].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = local ? 1 : 2;
    auto go = [&](auto* kern, int smem) {
      cfg.dynamicSmemBytes = smem_of(smem);
      cudaLaunchKernelEx(&cfg, kern, t.rx_hi[0][v], t.rx_lo[0][v], t.rx_hi[1][v], t.rx_lo[1][v],
                         static_cast<const uint4*>(g->fxt), static_cast<const uint4*>(g->fyt), a);
    };
    const bool res = a.rsum != nullptr;   // (the B_perp solves, two right-hand sides)
    if (t.cl_mode == 0) {
      if (!v) go(cl_kernel<64, 0, false>(), Cl<64, 0>::BYTES);
      else if (res) go(cl_kernel<32, 0, true>(), Cl<32, 0>::BYTES);
      else go(cl_kernel<32, 0, false>(), Cl<32, 0>::BYTES);
    } else if (t.cl_mode == 2) {
      if (!v) go(cl_kernel<64, 2, false>(), Cl<64, 2>::BYTES);
      else if (res) go(cl_kernel<32, 2, true>(), Cl<32, 2>::BYTES);
      else go(cl_kernel<32, 2, false>(), Cl<32, 2>::BYTES);
    } else {
      if (res) go(cl_kernel<32, 1, true>(), Cl<32, 1>::BYTES);
      else go(cl_kernel<32, 1, false>(), Cl<32, 1>::BYTES);
    }
    return;
  }
  if (t.rs) {
    // resident fold-matrix solve: MB slot blocks x (R n / BN) data-row tiles per product; the
    // grid is a multiple of MB (a CTA keeps its slot block)
    const int n = g->nx, MB = n / BM;
    const int tiles32 = MB * (R * n / 32);
    const bool narrow = !t.wide_only && tiles32 <= t.rs_ctas[1];
    const int v = narrow ? 1 : 0;
    const int tiles_v = MB * (R * n / (narrow ? 32 : 64));
    cudaLaunchConfig_t cfg = {};
    // (at least a CTA per kSrcRows source rows: 256^2, two right-hand sides has 32 tiles)
    cfg.gridDim = dim3((unsigned)std::min(std::max(tiles_v, pre ? n / kSrcRows : 0), t.rs_ctas[v] / MB * MB));
    cfg.blockDim = dim3(kClThreads);
    cfg.dynamicSmemBytes = smem_of(narrow ? RsSmem<32>::BYTES : RsSmem<64>::BYTES);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    late_reset();
    auto pick = [&](auto* w0, auto* w1, auto* n0, auto* n1) { return a.rsum ? (narrow ? n1 : w1) : (narrow ? n0 : w0); };
    auto* kern = n == 512 ? pick(rs_kernel<64, 512, false>(), rs_kernel<64, 512, true>(), rs_kernel<32, 512, false>(),
                                 rs_kernel<32, 512, true>())
                          : pick(rs_kernel<64, 256, false>(), rs_kernel<64, 256, true>(), rs_kernel<32, 256, false>(),
                                 rs_kernel<32, 256, true>());
    cudaLaunchKernelEx(&cfg, kern, static_cast<const uint4*>(g->fxt), t.rx_hi[0][v], t.rx_lo[0][v], t.rx_hi[1][v], t.rx_lo[1][v],
                       t.rx_hi[2][v], t.rx_lo[2][v], a);
    return;
  }
  // tiles of one product (the larger of the x and y products) at N-tile width bn
  auto tiles = [&](int bn) {
    return std::max(R * (g->nyp / BM) * (g->nxp / bn), R * (g->nxp / BM) * (g->nyp / bn));
  };
  const bool halves = !g->fold || (g->nx % 256 == 0 && g->ny % 256 == 0);   // a slot block lies in one half
  if (halves && tiles(64) > 3 * t.ctas[0] && !t.wide_only) {
    // more than three 128 x 64 tiles per CTA: 128 x 128 tiles, pipelined.  2048^2, two right-hand sides:
    // 295 us with 128 x 64 tiles, 228 us here; 1536^2: 150 and 122; with fewer tiles the last, half
    // empty wave of large tiles costs more than the overlap gains (1024^2, three: 86 and 92).
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)std::min(t.wide_ctas, tiles(128)));
    cfg.blockDim = dim3(kWideThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    auto go = [&](auto* kern, int smem) {
      cfg.dynamicSmemBytes = smem_of(smem);
      cudaLaunchKernelEx(&cfg, kern, t.fx_hi, t.fx_lo, t.fy_hi, t.fy_lo, t.a0_hi, t.a0_lo, t.a1_hi, t.a1_lo, a);
    };
    using B16 = __nv_bfloat16;
    if (g->tf32) go(a.rsum ? &k_dst_solve_wide<true, float> : &k_dst_solve_wide<false, float>, Wide<float>::BYTES);
    else go(a.rsum ? &k_dst_solve_wide<true, B16> : &k_dst_solve_wide<false, B16>, Wide<B16>::BYTES);
    return;
  }
  const bool narrow = !t.wide_only && tiles(32) <= t.ctas[1];
  const int v = narrow ? 1 : 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)std::min(t.ctas[v], tiles(narrow ? 32 : 64)));
  cfg.blockDim = dim3(kSolveThreads);
  cfg.dynamicSmemBytes = smem_of(narrow ? SolveSmem<32>::BYTES : SolveSmem<64>::BYTES);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // a launch error is reported by the caller's launch check
  auto kern = g->tf32 ? (a.rsum ? (narrow ? k_dst_solve<32, true, float> : k_dst_solve<64, true, float>)
                                : (narrow ? k_dst_solve<32, false, float> : k_dst_solve<64, false, float>))
                      : (a.rsum ? (narrow ? k_dst_solve<32, true, __nv_bfloat16> : k_dst_solve<64, true, __nv_bfloat16>)
                                : (narrow ? k_dst_solve<32, false, __nv_bfloat16>
                                          : k_dst_solve<64, false, __nv_bfloat16>));
  cudaLaunchKernelEx(&cfg, kern, t.a0_hi, t.a0_lo, t.a1_hi, t.a1_lo, t.bx_hi[v], t.bx_lo[v], t.by_hi[v], t.by_lo[v],
                     shifted ? t.scale_h[v] : t.scale[v], a);
}

}  // namespace

// B_perp solve with the predictor-corrector mixing fused into the last product's epilogue:
// sources (split, 2 rhs) in op[0] -> bm <- w B + (1 - w) bm.
void dst_solve_tc_bmix(hq_grid_s* g, int last, cudaStream_t s) { solve_fused(g, 2, 3, last, s); }

// sources (split) in op[0] -> FP32 solution in g->solved [R][ny][nx]
void dst_solve_tc(hq_grid_s* g, int R, cudaStream_t s) { solve_fused(g, R, 2, 0, s); }
// src [R][ny][nx] -> dst (16-byte aligned), both the caller's: read by the source phase, written by
// the last product
void dst_solve_tc_given(hq_grid_s* g, int R, const float* src, float* dst, cudaStream_t s) {
  solve_fused(g, R, 2, 0, s, 3, nullptr, nullptr, nullptr, false, src, dst);
}
void dst_solve_tc_shifted(hq_grid_s* g, int R, cudaStream_t s) {
  solve_fused(g, R, 2, 0, s, 0, nullptr, nullptr, nullptr, true);
}

// The same with the source kernels folded into the launch as its first phase: psi, Ez, Bz of
// the deposit record dep -> g->solved; the B_perp sources of the predictor-corrector (which
// clear the trial J_perp and, on the last iteration, reset dep_prev) -> mixing into bm.
void dst_solve_tc_main(hq_grid_s* g, const void* dep, cudaStream_t s) { solve_fused(g, 3, 2, 0, s, 1, dep); }
void dst_solve_tc_bmix_src(hq_grid_s* g, const void* cur, void* prev, void* chi_prev, int last, cudaStream_t s) {
  solve_fused(g, 2, 3, last, s, 2, cur, prev, chi_prev);
}

}  // namespace hq

// ---------------------------------------------------------------- allocation-free variant
// hq_poisson_solve_static: the same tensor-core Dirichlet solve for callers that
// cannot allocate device memory (all scratch in one file-scope static array).
#include <map>
#include <mutex>

namespace hq {
void set_global_error(const std::string& msg);  // defined in hq_api.cu

namespace {

constexpr int kStaticMaxN = 512;   // nx, ny <= 512 (so the padded extents are <= 512)
constexpr int kStaticMaxRhs = 3;
constexpr size_t kStaticOpBytes = (size_t)kStaticMaxRhs * kStaticMaxN * kStaticMaxN * 2;  // one bf16 operand buffer
constexpr size_t kStaticSBytes = (size_t)kStaticMaxN * kStaticMaxN * 2;                    // one bf16 sine matrix
constexpr size_t kStaticScaleBytes = (size_t)kStaticMaxN * kStaticMaxN * 4;                // FP32 1/lambda table
// layout: status word (256 B) | op_hi0 op_lo0 op_hi1 op_lo1 | sx_hi sx_lo sy_hi sy_lo | scale  (9 MiB + 256 B)
constexpr size_t kStaticBytes = 256 + 4 * kStaticOpBytes + 4 * kStaticSBytes + kStaticScaleBytes;
static __device__ __align__(256) unsigned char g_static_scratch[kStaticBytes];

struct StaticDev {
  uint8_t* base = nullptr;   // device address of g_static_scratch on this device
  int nx = 0, ny = 0;        // geometry the tables in the array hold (nx = 0: unknown, rebuild)
  double dx = 0.0, dy = 0.0;
  TensorMaps maps;           // encoded for (map_nx, map_ny)
  int map_nx = 0, map_ny = 0;
};
std::mutex g_static_mu;
std::map<int, StaticDev> g_static_dev;

// S_x, S_y (bf16 hi/lo, zero-padded) and the scale (4/(nx ny))/lambda for one grid.
__global__ void k_static_tables(__nv_bfloat16* sxh, __nv_bfloat16* sxl, __nv_bfloat16* syh, __nv_bfloat16* syl,
                                float* scale, int nx, int ny, int nxp, int nyp, double dx, double dy) {
  const int64_t tot = (int64_t)kStaticMaxN * kStaticMaxN;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < tot; t += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(t / kStaticMaxN), c = (int)(t % kStaticMaxN);
    if (r < nxp && c < nxp) {
      const float v = (r < nx && c < nx) ? (float)sinpi((double)(((int64_t)r * c) % (2 * nx)) / nx) : 0.0f;
      const __nv_bfloat16 h = __float2bfloat16_rn(v);
      sxh[(int64_t)r * nxp + c] = h;
      sxl[(int64_t)r * nxp + c] = __float2bfloat16_rn(v - __bfloat162float(h));
    }
    if (r < nyp && c < nyp) {
      const float v = (r < ny && c < ny) ? (float)sinpi((double)(((int64_t)r * c) % (2 * ny)) / ny) : 0.0f;
      const __nv_bfloat16 h = __float2bfloat16_rn(v);
      syh[(int64_t)r * nyp + c] = h;
      syl[(int64_t)r * nyp + c] = __float2bfloat16_rn(v - __bfloat162float(h));
    }
    if (r < nyp && c < nxp) {
      float s = 0.0f;
      if (r >= 1 && r < ny && c >= 1 && c < nx) {
        const double sx = sinpi(c / (2.0 * nx)), sy = sinpi(r / (2.0 * ny));
        const double lam = -(4.0 / (dx * dx)) * sx * sx - (4.0 / (dy * dy)) * sy * sy;
        s = (float)((4.0 / ((double)nx * ny)) / lam);
      }
      scale[(int64_t)r * nxp + c] = s;
    }
  }
}

// Sources into the zero-padded split operand layout [R][nyp][nxp]; every padded entry
// is written, so nothing left over from an earlier call of another size survives.
__global__ void k_static_src(const float* __restrict__ src, __nv_bfloat16* hi, __nv_bfloat16* lo, int R, int nx, int ny,
                             int nxp, int nyp) {
  const int64_t tot = (int64_t)R * nyp * nxp;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < tot; t += (int64_t)gridDim.x * blockDim.x) {
    const int ix = (int)(t % nxp);
    const int64_t ry = t / nxp;
    const int iy = (int)(ry % nyp), r = (int)(ry / nyp);
    const float v = (ix >= 1 && ix < nx && iy >= 1 && iy < ny) ? src[((int64_t)r * ny + iy) * nx + ix] : 0.0f;
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    hi[t] = h;
    lo[t] = __float2bfloat16_rn(v - __bfloat162float(h));
  }
}

EncodeFn static_encoder(std::string& err) {
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
      fn == nullptr || q != cudaDriverEntryPointSuccess) {
    err = "cuTensorMapEncodeTiled not available from the driver";
    return nullptr;
  }
  return reinterpret_cast<EncodeFn>(fn);
}

hq_status static_fail(hq_status st, const std::string& msg) {
  set_global_error(msg);
  return st;
}

}  // namespace
}  // namespace hq

using namespace hq;

extern "C" hq_status hq_poisson_solve_static(const float* src, float* dst, int32_t nx, int32_t ny, double dx, double dy,
                                             int32_t nrhs, void* cuda_stream) {
  if (!src || !dst) return static_fail(HQ_ERR_ARG, "hq_poisson_solve_static: src and dst must not be NULL");
  if (nx < 8 || ny < 8 || nx > kStaticMaxN || ny > kStaticMaxN)
    return static_fail(HQ_ERR_ARG, "hq_poisson_solve_static: nx and ny must be in 8..512 (static scratch limit)");
  if (nrhs < 1 || nrhs > kStaticMaxRhs)
    return static_fail(HQ_ERR_ARG, "hq_poisson_solve_static: nrhs must be in 1..3 (static scratch limit)");
  if (!(dx > 0.0) || !(dy > 0.0) || !std::isfinite(dx) || !std::isfinite(dy))
    return static_fail(HQ_ERR_ARG, "hq_poisson_solve_static: dx and dy must be finite and positive");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
  int dev = 0, sdev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return static_fail(HQ_ERR_CUDA, "hq_poisson_solve_static: no CUDA device");
  if (cudaStreamGetDevice(s, &sdev) != cudaSuccess)
    return static_fail(HQ_ERR_ARG, "hq_poisson_solve_static: cuda_stream is not a valid stream");
  if (sdev != dev)
    return static_fail(HQ_ERR_ARG, "hq_poisson_solve_static: cuda_stream belongs to device " + std::to_string(sdev) +
                                        ", not the current device " + std::to_string(dev));
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cap) != cudaSuccess)
    return static_fail(HQ_ERR_CUDA, "hq_poisson_solve_static: cannot query the stream's capture state");
  const bool capturing = cap != cudaStreamCaptureStatusNone;
  std::lock_guard<std::mutex> lock(g_static_mu);
  StaticDev& sd = g_static_dev[dev];
  std::string err;
  if (!sd.base) {
    // once per device: resolve the static array's device address (the host-side symbol is
    // only a stand-in) and allow the GEMM's shared-memory footprint
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, dev) != cudaSuccess || prop.major != 10 || prop.minor != 3)
      return static_fail(HQ_ERR_UNSUPPORTED, "hq_poisson_solve_static: needs an sm_103a (GB300) device");
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess || !p)
      return static_fail(HQ_ERR_CUDA, std::string("cudaGetSymbolAddress(static scratch): ") + cudaGetErrorString(e));
    if (cudaFuncSetAttribute(k_dst_gemm<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<128>::SMEM_BYTES) !=
            cudaSuccess ||
        cudaFuncSetAttribute(k_dst_gemm<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<64>::SMEM_BYTES) !=
            cudaSuccess)
      return static_fail(HQ_ERR_CUDA, "hq_poisson_solve_static: cannot raise the GEMM shared-memory limit");
    sd.base = static_cast<uint8_t*>(p);
  }
  uint8_t* b = sd.base;
  int* status = reinterpret_cast<int*>(b);
  __nv_bfloat16* op_hi0 = reinterpret_cast<__nv_bfloat16*>(b + 256);
  __nv_bfloat16* op_lo0 = reinterpret_cast<__nv_bfloat16*>(b + 256 + kStaticOpBytes);
  __nv_bfloat16* op_hi1 = reinterpret_cast<__nv_bfloat16*>(b + 256 + 2 * kStaticOpBytes);
  __nv_bfloat16* op_lo1 = reinterpret_cast<__nv_bfloat16*>(b + 256 + 3 * kStaticOpBytes);
  uint8_t* sb = b + 256 + 4 * kStaticOpBytes;
  __nv_bfloat16* sxh = reinterpret_cast<__nv_bfloat16*>(sb);
  __nv_bfloat16* sxl = reinterpret_cast<__nv_bfloat16*>(sb + kStaticSBytes);
  __nv_bfloat16* syh = reinterpret_cast<__nv_bfloat16*>(sb + 2 * kStaticSBytes);
  __nv_bfloat16* syl = reinterpret_cast<__nv_bfloat16*>(sb + 3 * kStaticSBytes);
  float* scale = reinterpret_cast<float*>(sb + 4 * kStaticSBytes);
  const int nxp = (nx + 127) / 128 * 128, nyp = (ny + 127) / 128 * 128;
  if (sd.map_nx != nx || sd.map_ny != ny) {
    // new extents: re-encode the tensor maps over the new padded extents (host-side, no
    // allocation)
    EncodeFn enc = static_encoder(err);
    if (!enc) return static_fail(HQ_ERR_CUDA, err);
    TensorMaps& t = sd.maps;
    int bad = 0;
    bad |= make_map(enc, &t.a0_hi, op_hi0, (uint64_t)kStaticMaxRhs * nyp, nxp, err);
    bad |= make_map(enc, &t.a0_lo, op_lo0, (uint64_t)kStaticMaxRhs * nyp, nxp, err);
    bad |= make_map(enc, &t.a1_hi, op_hi1, (uint64_t)kStaticMaxRhs * nxp, nyp, err);
    bad |= make_map(enc, &t.a1_lo, op_lo1, (uint64_t)kStaticMaxRhs * nxp, nyp, err);
    for (int i = 0; i < 2; ++i) {
      const uint32_t rows = i == 0 ? 128 : 64;
      bad |= make_map(enc, &t.sx_hi[i], sxh, nxp, nxp, err, rows);
      bad |= make_map(enc, &t.sx_lo[i], sxl, nxp, nxp, err, rows);
      bad |= make_map(enc, &t.sy_hi[i], syh, nyp, nyp, err, rows);
      bad |= make_map(enc, &t.sy_lo[i], syl, nyp, nyp, err, rows);
    }
    if (bad) {
      sd.map_nx = sd.map_ny = 0;
      sd.nx = sd.ny = 0;
      return static_fail(HQ_ERR_CUDA, err);
    }
    sd.map_nx = nx;
    sd.map_ny = ny;
  }
  // The sine matrices and the 1/lambda table in the array are rebuilt for a new (nx, ny, dx,
  // dy), and by every call made while the stream is being captured: what such a call enqueues
  // runs later, so the array's contents can no longer be tracked here and the next call
  // rebuilds them too.
  if (capturing || sd.nx != nx || sd.ny != ny || sd.dx != dx || sd.dy != dy) {
    sd.nx = sd.ny = 0;
    k_static_tables<<<256, 256, 0, s>>>(sxh, sxl, syh, syl, scale, nx, ny, nxp, nyp, dx, dy);
    const cudaError_t te = cudaGetLastError();
    if (te != cudaSuccess)
      return static_fail(HQ_ERR_CUDA, std::string("hq_poisson_solve_static: table build: ") + cudaGetErrorString(te));
    if (!capturing) {
      sd.nx = nx;
      sd.ny = ny;
      sd.dx = dx;
      sd.dy = dy;
    }
  }
  const TensorMaps& t = sd.maps;
  // the status word at the start of the array is not cleared here: a timeout or a non-finite
  // result stays flagged until hq_sync(NULL, ...) reads and clears it
  k_static_src<<<256, 256, 0, s>>>(src, op_hi0, op_lo0, nrhs, nx, ny, nxp, nyp);
  Epi e{};
  e = Epi{0, nyp, nxp, op_hi1, op_lo1, nullptr, nullptr, 0, 0};
  gemm(t.a0_hi, t.a0_lo, t.sx_hi, t.sx_lo, nrhs * nyp, nxp, nxp, e, status, s);
  e = Epi{1, nxp, nyp, op_hi0, op_lo0, scale, nullptr, 0, 0};
  gemm(t.a1_hi, t.a1_lo, t.sy_hi, t.sy_lo, nrhs * nxp, nyp, nyp, e, status, s);
  e = Epi{0, nyp, nxp, op_hi1, op_lo1, nullptr, nullptr, 0, 0};
  gemm(t.a0_hi, t.a0_lo, t.sx_hi, t.sx_lo, nrhs * nyp, nxp, nxp, e, status, s);
  e = Epi{2, nxp, nyp, nullptr, nullptr, nullptr, dst, nx, ny};
  gemm(t.a1_hi, t.a1_lo, t.sy_hi, t.sy_lo, nrhs * nxp, nyp, nyp, e, status, s);
  const cudaError_t le = cudaGetLastError();
  if (le != cudaSuccess) return static_fail(HQ_ERR_CUDA, std::string("hq_poisson_solve_static: ") + cudaGetErrorString(le));
  return HQ_OK;
}

namespace hq {
// Status of the allocation-free solves on the current device (hq_sync(NULL, ...)): waits for
// the device, reads the status word at the start of the static array and clears it.  A device
// on which no such solve was set up reports HQ_OK.
hq_status static_sync() {
  if (cudaDeviceSynchronize() != cudaSuccess) {
    const cudaError_t e = cudaGetLastError();
    return static_fail(HQ_ERR_CUDA, std::string("hq_sync(NULL): ") + cudaGetErrorString(e));
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return static_fail(HQ_ERR_CUDA, "hq_sync(NULL): no CUDA device");
  uint8_t* base = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_static_mu);
    auto it = g_static_dev.find(dev);
    if (it != g_static_dev.end()) base = it->second.base;
  }
  if (!base) return HQ_OK;
  int status = 0;
  if (cudaMemcpy(&status, base, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
    return static_fail(HQ_ERR_CUDA, "hq_sync(NULL): status read failed");
  if (!status) return HQ_OK;
  if (cudaMemset(base, 0, sizeof(int)) != cudaSuccess) return static_fail(HQ_ERR_CUDA, "hq_sync(NULL): status reset failed");
  if (status & DEV_TIMEOUT)
    return static_fail(HQ_ERR_TIMEOUT, "hq_poisson_solve_static: a bounded device wait ran out");
  return static_fail(HQ_ERR_NUMERIC, "hq_poisson_solve_static: a non-finite value reached the solution");
}
}  // namespace hq
