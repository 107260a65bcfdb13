// Indices into a boundary's cotangent table (M entries, 1/2 cot(pi j / M)) for the
// sources of a 32-node tile of that boundary (pair_sums.cuh).  The kernels walk all 32
// lanes of a tile; a lane past its n nodes stands for its last one (its weight is zero),
// so that one wrap is enough for every M: the lanes alone reach past twice the table
// where M < 16.
#pragma once
#ifdef __CUDACC__
#define PSUM_HD __host__ __device__ __forceinline__
#else
#define PSUM_HD inline
#endif

// (i_l - i_m) mod M for lane p, first = (i_{l0} - i_m) mod M of the tile's first node
PSUM_HD int psum_index_up(int first, int p, int n, int M) {
  const int i = first + (p < n ? p : n - 1);
  return i >= M ? i - M : i;
}
// (i_m - i_l) mod M for lane p, first = (i_m - i_{l0}) mod M
PSUM_HD int psum_index_down(int first, int p, int n, int M) {
  const int i = first - (p < n ? p : n - 1);
  return i < 0 ? i + M : i;
}
