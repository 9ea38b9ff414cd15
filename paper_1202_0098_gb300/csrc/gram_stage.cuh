// Sizes and indexes of the staged S_r products of the short recurrences' FP32 form (gram_s in chains.cu). Plain
// integer arithmetic that also compiles without CUDA, so that every index can be checked on the host.
#pragma once

#ifndef __CUDACC__
#define __host__
#define __device__
#endif

namespace mka {

// Floats between the vectors of a chunk of rc rows: an odd number of 16-byte groups, so that eight vectors in a
// row start in different banks.
__host__ __device__ constexpr int chunk_stride(int rc) { return 4 * (rc | 1); }

// Floats of Gs and gv, 16-byte aligned.
__host__ __device__ constexpr int gs_floats(int p) { return (4 * p * (p + 1) + 8 * p + 3) / 4 * 4; }

// Shared vectors of m rows hold the seam's Gs, gv and (FP32) two chunks of at least four rows of the p vectors and
// of all nu.
__host__ __device__ constexpr bool chains_fit(int m, int p, int nu, bool pairs) {
  return pairs ? gs_floats(p) + 4 * p * chunk_stride(4) <= 12 * m && 4 * nu * chunk_stride(4) <= 12 * m
               : gs_floats(p) <= 16 * m;
}

// A chunk's vectors: W 0..n1, then S W n0..n1.
__host__ __device__ constexpr int chunk_vectors(int n0, int n1) { return n1 + (n1 - n0); }

// Rows of a chunk: two buffers of nvec vectors fit in `floats`.
__host__ __device__ constexpr int chunk_rows(int nvec, int floats) {
  int rc = 32;
  while (rc > 4 && 2 * nvec * chunk_stride(rc) > floats) rc -= 4;
  return rc;
}

// Vector i of lane row t (0..7) against the pair of vectors that ends with nb. Beyond nb the product is not used and
// the lane reads nb again: a chunk has no more than chunk_vectors() of them, which the next multiple of eight can
// exceed when one of the chains is short.
__host__ __device__ constexpr int lane_vector(int t, int i, int nb) { return t + 8 * i < nb ? t + 8 * i : nb; }

}  // namespace mka
