// Row orders of the folded FP32 solve and which rows its products wait for: index arithmetic
// alone, so that a host compiler can check the kernels' dependencies (no CUDA headers).
#pragma once

#ifdef __CUDACC__
#define HQ_HD __host__ __device__ __forceinline__
#else
#define HQ_HD inline
#endif

namespace hq {

// Folded DST-I order (Sec. 3.2 solver).  With S_jk = sin(pi j k / n),
// S_{n-j,k} = -(-1)^k S_jk: odd k see only x_j + x_{n-j}, even k only x_j - x_{n-j},
// so after folding the node pairs (j, n-j) every output needs n/2 terms.  The folded
// solver keeps each grid index in "slot order", pair u on slots 2u, 2u+1: pairs
// 0 .. n/4-1 are (1, n-1), (3, n-3), ...; pair n/4 is (0, n/2); the rest (2, n-2),
// (4, n-4), ...  Slots 0 .. n/2-1 thus hold the odd indices.  n must be a multiple of 4.
HQ_HD void fold_pair(int u, int n, int& a, int& b) {
  if (u < n / 4) {
    a = 2 * u + 1;
    b = n - a;
  } else {
    a = 2 * (u - n / 4);
    b = a == 0 ? n / 2 : n - a;
  }
}
HQ_HD int fold_node(int s, int n) {
  int a, b;
  fold_pair(s >> 1, n, a, b);
  return (s & 1) ? b : a;
}

// The resident solve's products p = 0 .. 3 on n x n, R right-hand sides.  A tile of product p
// multiplies one block of 128 slots (blocks = n / 128) by the data rows of one of ntr tiles of a
// right-hand side.  Its output slot s is row rs_out_row of that right-hand side's next operand:
// slot order, but node order after product 2 (the last product's columns are consecutive x nodes).
HQ_HD int rs_out_row(int p, int s, int n) { return p == 2 ? fold_node(s, n) : s; }

// Counter (of rs_counters) that a tile of product p < 3 reports its stores to: one per slot block,
// and one for the whole right-hand side after product 2, since a run of consecutive nodes comes from
// two or three of its slot blocks.
HQ_HD int rs_arrival(int p, int R, int blocks, int r, int block) { return (p * R + r) * blocks + (p == 2 ? 0 : block); }
HQ_HD int rs_counters(int R, int blocks) { return 3 * R * blocks; }

// The counter and its value that say that all of product p - 1 that the data rows from row0 on (less
// than a tile) of right-hand side r hold has been stored, for a tile of product p > 0.
struct RsWait {
  int counter, target;
};
HQ_HD RsWait rs_wait(int p, int R, int blocks, int ntr, int r, int row0) {
  return {rs_arrival(p - 1, R, blocks, r, row0 / 128), p == 3 ? blocks * ntr : ntr};
}

}  // namespace hq
