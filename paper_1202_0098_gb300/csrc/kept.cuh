// Products with the kept data of a column: C (and V_j) by column, the pattern rows of U (device code shared by the
// density, Green's function and force kernels).
#pragma once

#include <stdint.h>

#include "mka_internal.h"

namespace mka {

// Columns of atom t: NX vectors g_x = C diag(x) V_j for per-level weights x[NX][4][nu] in shared memory (used up), g
// [NX][4][nu]. Threads run over the atom's four columns first: these lie next to each other in the kept layout, so that
// a warp reads whole 32-byte sectors (8 rows of C), where a thread order with the level first read each four times.
// C is real: every element read serves all NX vectors. (32,768 columns of nu = 30: density 0.63 -> 0.25 ms, 8,192 columns:
// Green's function 193 -> 100 us.)
template <int NX>
__device__ __forceinline__ void column_weights(const double* __restrict__ cv, int64_t t, int nu, double* x, double* g) {
  const double* b = cv + (size_t)((4 * t) >> 5) * kept_block_doubles(nu) * 32 + ((4 * t) & 31);
  for (int i = threadIdx.x; i < 4 * nu; i += blockDim.x) {
    const int c = i & 3, a = i >> 2;
    const double v = b[(size_t)(nu * nu + a) * 32 + c];
#pragma unroll
    for (int q = 0; q < NX; ++q) x[(q * 4 + c) * nu + a] *= v;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 4 * nu; i += blockDim.x) {
    const int c = i & 3, n = i >> 2;
    const double* bn = b + (size_t)n * nu * 32 + c;
    double s[NX];
#pragma unroll
    for (int q = 0; q < NX; ++q) s[q] = 0.0;
#pragma unroll 6
    for (int a = 0; a < nu; ++a) {
      const double e = __ldcs(bn + (size_t)a * 32);
#pragma unroll
      for (int q = 0; q < NX; ++q) s[q] = fma(e, x[(q * 4 + c) * nu + a], s[q]);
    }
#pragma unroll
    for (int q = 0; q < NX; ++q) g[(q * 4 + c) * nu + n] = s[q];
  }
  __syncthreads();
}

// s[q] = u . g_q for one kept row u of U (nu entries) and the column's NX vectors, `step` apart. Rows of an even nu start
// on 16 bytes (pair: the caller has looked at the base too), and are read two entries at a time.
template <int NX>
__device__ __forceinline__ void row_products(const double* __restrict__ u, const double* g, int step, int nu, bool pair,
                                             double s[NX]) {
#pragma unroll
  for (int q = 0; q < NX; ++q) s[q] = 0.0;
  if (pair) {
#pragma unroll 5
    for (int n = 0; n < nu; n += 2) {
      const double2 v = __ldg(reinterpret_cast<const double2*>(u + n));
#pragma unroll
      for (int q = 0; q < NX; ++q) {
        const double2 w = *reinterpret_cast<const double2*>(g + q * step + n);
        s[q] = fma(v.x, w.x, s[q]);
        s[q] = fma(v.y, w.y, s[q]);
      }
    }
  } else {
#pragma unroll 5
    for (int n = 0; n < nu; ++n) {
      const double v = __ldg(u + n);
#pragma unroll
      for (int q = 0; q < NX; ++q) s[q] = fma(v, g[q * step + n], s[q]);
    }
  }
}

__device__ __forceinline__ bool rows_paired(const double* vp, int nu) {
  return (nu & 1) == 0 && (reinterpret_cast<uintptr_t>(vp) & 15) == 0;
}

}  // namespace mka
