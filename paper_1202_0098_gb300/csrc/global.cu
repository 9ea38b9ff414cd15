// Global (all-column) kernels: mu, the density matrix with the band
// energy, the subspace Green's function, and the global block-sparse product.
//
// mu (Sec. 2, after Eq. EQ-DM): the electron count 2 sum_j sum_alpha f w is evaluated by one launch per step of a
// bracketing root finder (mu_root.cuh: a few bisection steps, then the Illinois secant, 10 to 15 passes on metallic
// levels where halving alone took 46, which a gap still takes); the launch's blocks write fixed-order partial sums, and the last block to finish
// (ticket counter) adds them in a fixed tree and takes the step, so the result does not depend on timing.
// f(x) = (1 - tanh((x - mu) / (2 kT))) / 2; for |x - mu| / (2 kT) > 20 the FP64
// tanh is exactly +-1, so those terms take f = 0 or 1 without calling it.
//
// rho (Eq. EQ-DM), G (Eq. EQ-SOLUTION-SUB-GZ) and E (Eq. EQ-ENE) read the kept
// pattern rows of v_alpha (row block k of column j, [c][r][alpha]).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "kept.cuh"
#include "mka_internal.h"
#include "spmv_rule.cuh"
#include "widen.cuh"
#include "mu_root.cuh"

namespace mka {
namespace {

constexpr int kRedThreads = 256;
// Grid of the reductions: 4 CTAs per SM of the current device, at most kMaxRedBlocks (the size of
// the partial-sum buffers).
int red_blocks() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    sms = 152;
  return std::max(1, std::min(kMaxRedBlocks, 4 * sms));
}

__device__ __forceinline__ double fermi(double x, double mu, double kT) {
  const double y = (x - mu) / (2.0 * kT);
  if (y > 20.0) return 0.0;
  if (y < -20.0) return 1.0;
  return 0.5 * (1.0 - tanh(y));
}

__device__ __forceinline__ double block_sum(double v, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0;
  if (threadIdx.x == 0)
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += red[k];
  __syncthreads();
  return s;  // valid in thread 0
}

// min / max of eps over entries with w != 0 (fixed-order two-level reduction).
__global__ void eps_range_kernel(const double* eps, const double* w, int64_t n, double* partial,
                                 unsigned* ticket, RootState* S) {
  __shared__ double rmin[kRedThreads / 32], rmax[kRedThreads / 32];
  __shared__ bool last;
  double mn = INFINITY, mx = -INFINITY;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    if (w[i] != 0.0) {
      mn = fmin(mn, eps[i]);
      mx = fmax(mx, eps[i]);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  if ((threadIdx.x & 31) == 0) {
    rmin[threadIdx.x >> 5] = mn;
    rmax[threadIdx.x >> 5] = mx;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < kRedThreads / 32; ++k) {
      mn = fmin(mn, rmin[k]);
      mx = fmax(mx, rmax[k]);
    }
    mn = fmin(mn, rmin[0]);
    mx = fmax(mx, rmax[0]);
    partial[2 * blockIdx.x] = mn;
    partial[2 * blockIdx.x + 1] = mx;
    __threadfence();
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (last) {
    __threadfence();
    mn = INFINITY;
    mx = -INFINITY;
    for (unsigned k = threadIdx.x; k < gridDim.x; k += blockDim.x) {
      mn = fmin(mn, partial[2 * k]);
      mx = fmax(mx, partial[2 * k + 1]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
      mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if ((threadIdx.x & 31) == 0) {
      rmin[threadIdx.x >> 5] = mn;
      rmax[threadIdx.x >> 5] = mx;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int k = 0; k < kRedThreads / 32; ++k) {
        mn = fmin(mn, rmin[k]);
        mx = fmax(mx, rmax[k]);
      }
      S->lo = mn - 40.0 * S->kT;
      S->hi = mx + 40.0 * S->kT;
      S->x = S->hi;              // first point: every level occupied (N(lo) = 0 needs no pass)
      S->flo = -S->target;
      S->fhi = 0.0;
      S->side = 0.0;
      S->rf = 0.0;
      S->probed = 0.0;
      S->iters = 0;
      *ticket = 0;
    }
  }
}

// Lanes that share a column's levels: one where the columns fill the chip, up to 32 where they are few and a thread's
// serial levels are what a pass takes.
int lanes_per_column(int64_t n_cols) {
  int l = 1;
  while (l < 32 && n_cols * l * 2 <= 65536) l *= 2;
  return l;
}

// One step of the root finder: N(x) = 2 sum f(eps; x) w over the columns (`share` threads per column), then the bracket.
// Measured at 32,768 columns of nu = 30: 81 us a halving (46 of them) when threads ran over single levels and one
// thread added the blocks' sums; the whole search now takes 0.4 ms of a batch instead of 5.2. Whole columns a thread at 4
// columns of nu = 100: 681 us a search, 221 with the levels shared.
__global__ void __launch_bounds__(kRedThreads) mu_pass_kernel(const double* eps, const double* w, int64_t n_cols, int nu,
                                                              int share, double* partial, unsigned* ticket, RootState* S, int left) {
  __shared__ double red[kRedThreads / 32];
  __shared__ bool last;
  if (!(S->hi - S->lo > S->tol)) return;   // converged: every block leaves before touching the ticket
  const double x = S->x, rk = 0.5 / S->kT;
  double acc = 0.0;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n_cols * share; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = t / share;
    acc += column_count(eps + i * nu, w + i * nu, nu, x, rk, (int)(t % share), share);
  }
  const double s = block_sum(acc, red);
  if (threadIdx.x == 0) {
    partial[blockIdx.x] = s;
    __threadfence();
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (last) {
    __threadfence();
    double t = 0.0;
    for (unsigned k = threadIdx.x; k < gridDim.x; k += blockDim.x) t += partial[k];
    t = block_sum(t, red);
    if (threadIdx.x == 0) {
      root_step_lowest(S, 2.0 * t, left);
      *ticket = 0;
    }
  }
}

// Bracket state of a stream-ordered root search (no host round trip): target, kT, tolerance,
// ticket cleared; the range kernel then sets lo / hi.
__global__ void mu_init_kernel(RootState* S, unsigned* ticket, double target, double kT, double tol) {
  S->target = target;
  S->kT = kT;
  S->tol = tol;
  S->iters = 0;
  *ticket = 0;
}

__global__ void mu_finish_kernel(const RootState* S, double* mu_out) { *mu_out = 0.5 * (S->lo + S->hi); }

// rho / E: one CTA per selected atom, thread per (block k, c, r) of its row:
// rho_ij = sum_alpha f_alpha V_i alpha V_j alpha = U_i . g_j with g_j = C diag(f) V_j.
// Output layout: the batch's (blocks at blk_off[t], E of atom t at e_partial[t]) when out_base < 0;
// otherwise the system's pattern order from block out_base on (blocks at row_ptr[atom] - out_base,
// E at e_partial[atom - e_base]).
__global__ void __launch_bounds__(128) density_kernel(const double* vp, const double* cv, const double* eps, const int64_t* blk_off,
                               const int64_t* sel, const int32_t* row_ptr, const void* valH, int storage,
                               int nu, double mu_host, const double* mu_dev, double kT, double* rho,
                               double* e_partial, int64_t out_base = -1, int64_t e_base = 0) {
  __shared__ double red[kRedThreads / 32];
  extern __shared__ __align__(16) double sm[];     // g, f: 4 nu each
  double *g = sm, *f = sm + 4 * nu;
  const bool pair = rows_paired(vp, nu);
  const double mu = mu_dev ? *mu_dev : mu_host;
  const int64_t t = blockIdx.x;
  const int64_t atom = sel[t];
  const int nrow = row_ptr[atom + 1] - row_ptr[atom];
  const int64_t b0 = blk_off[t];
  const int64_t ob = out_base < 0 ? b0 : (int64_t)row_ptr[atom] - out_base;
  for (int i = threadIdx.x; i < 4 * nu; i += blockDim.x) {
    const int c = i / nu;
    f[i] = fermi(eps[(4 * t + c) * nu + i % nu], mu, kT);
  }
  __syncthreads();
  column_weights<1>(cv, t, nu, f, g);
  double e = 0.0;
  for (int i = threadIdx.x; i < nrow * 16; i += blockDim.x) {
    const int k = i >> 4, c = (i >> 2) & 3, r = i & 3;
    const double* u = vp + ((b0 + k) * 16 + c * 4 + r) * (int64_t)nu;
    double s;
    row_products<1>(u, g + c * nu, 0, nu, pair, &s);
    if (rho) rho[(ob + k) * 16 + c * 4 + r] = s;
    const int64_t gk = (int64_t)row_ptr[atom] + k;
    double h;
    if (storage == MKA_FP64) h = reinterpret_cast<const double*>(valH)[gk * 16 + c * 4 + r];
    else if (storage == MKA_MIXED_FP32) h = reinterpret_cast<const float*>(valH)[gk * 16 + c * 4 + r];
    else h = __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(valH)[gk * 16 + c * 4 + r]);
    e += s * h;
  }
  const double s = block_sum(e, red);
  if (threadIdx.x == 0) e_partial[out_base < 0 ? t : atom - e_base] = 2.0 * s;
}

// G_ij(z) = sum_alpha V_i alpha V_j alpha / (z - eps_alpha) = U_i . (C diag(1 / (z - eps)) V_j).
__global__ void __launch_bounds__(128) greens_kernel(const double* vp, const double* cv, const double* eps, const int64_t* blk_off,
                              const int64_t* sel, const int32_t* row_ptr, int nu, double zr, double zi, double* g) {
  extern __shared__ __align__(16) double sm[];     // g, x: real and imaginary parts, 4 nu each
  double *gv = sm, *xr = sm + 8 * nu, *xi = xr + 4 * nu;
  const bool pair = rows_paired(vp, nu);
  const int64_t t = blockIdx.x;
  const int64_t atom = sel[t];
  const int nrow = row_ptr[atom + 1] - row_ptr[atom];
  const int64_t b0 = blk_off[t];
  for (int i = threadIdx.x; i < 4 * nu; i += blockDim.x) {
    const int c = i / nu;
    const double dr = zr - eps[(4 * t + c) * nu + i % nu];
    const double den = dr * dr + zi * zi;   // 1 / (z - e) = (dr - i zi) / den
    xr[i] = dr / den;
    xi[i] = -zi / den;
  }
  __syncthreads();
  column_weights<2>(cv, t, nu, xr, gv);
  for (int i = threadIdx.x; i < nrow * 16; i += blockDim.x) {
    const int k = i >> 4, c = (i >> 2) & 3, r = i & 3;
    const double* u = vp + ((b0 + k) * 16 + c * 4 + r) * (int64_t)nu;
    double s[2];
    row_products<2>(u, gv + c * nu, 4 * nu, nu, pair, s);
    g[2 * ((b0 + k) * 16 + c * 4 + r)] = s[0];
    g[2 * ((b0 + k) * 16 + c * 4 + r) + 1] = s[1];
  }
}

// Fixed-order sum of n doubles by one CTA (strided per thread, then the fixed tree).
__global__ void sum_kernel(const double* x, int64_t n, double* out) {
  __shared__ double red[kRedThreads / 32];
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) s += x[i];
  s = block_sum(s, red);
  if (threadIdx.x == 0) *out = s;
}

// 2 sum f(eps; mu) w over the columns: per-block partial sums (fixed grid), added by sum_kernel.
__global__ void __launch_bounds__(kRedThreads) count_partial_kernel(const double* eps, const double* w, int64_t n_cols,
                                                                    int nu, int share, double mu_host,
                                                                    const double* mu_dev, double kT, double* partial) {
  __shared__ double red[kRedThreads / 32];
  const double mu = mu_dev ? *mu_dev : mu_host, rk = 0.5 / kT;
  double acc = 0.0;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n_cols * share; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = t / share;
    acc += column_count(eps + i * nu, w + i * nu, nu, mu, rk, (int)(t % share), share);
  }
  const double s = block_sum(acc, red);
  if (threadIdx.x == 0) partial[blockIdx.x] = 2.0 * s;
}

// ---- global BSR SpMV: four lanes per block row, one per output row of the 4x4 blocks ----
// Lane (a, i) computes y[4a + i][0..K) = sum over the row's blocks k of sum_jj val[k][i][jj] x[4 col[k] + jj][0..K).
// Each lane streams its row of every block (4 values: 8 bytes in BF16, 16 in FP32, 32 in FP64), so the four
// lanes of a block row read each block's values as one contiguous piece; the column index is read by all
// four (one request), and x through the read-only cache, one 16-byte vector per (block column, jj) row
// group. Blocks are taken four at a time with their loads issued before the arithmetic.
template <typename TV>
struct RowVals;
template <>
struct RowVals<__nv_bfloat16> {
  static __device__ __forceinline__ void load(const __nv_bfloat16* v, int64_t k, int i, float out[4]) {
    const uint2 a = __ldcs(reinterpret_cast<const uint2*>(v + k * 16 + i * 4));
    out[0] = __uint_as_float(a.x << 16);
    out[1] = __uint_as_float(a.x & 0xFFFF0000u);
    out[2] = __uint_as_float(a.y << 16);
    out[3] = __uint_as_float(a.y & 0xFFFF0000u);
  }
};
template <>
struct RowVals<float> {
  static __device__ __forceinline__ void load(const float* v, int64_t k, int i, float out[4]) {
    const float4 a = __ldcs(reinterpret_cast<const float4*>(v + k * 16 + i * 4));
    out[0] = a.x; out[1] = a.y; out[2] = a.z; out[3] = a.w;
  }
};
template <>
struct RowVals<double> {
  static __device__ __forceinline__ void load(const double* v, int64_t k, int i, double out[4]) {
    const double2 a = __ldcs(reinterpret_cast<const double2*>(v + k * 16 + i * 4));
    const double2 b = __ldcs(reinterpret_cast<const double2*>(v + k * 16 + i * 4) + 1);
    out[0] = a.x; out[1] = a.y; out[2] = b.x; out[3] = b.y;
  }
};

// x rows 4 cb .. 4 cb + 3, K values each: xv[jj][c].
template <typename TX, int K>
__device__ __forceinline__ void load_x(const TX* __restrict__ x, int64_t cb, TX xv[4][K]) {
  const TX* p = x + cb * 4 * K;
  if constexpr (sizeof(TX) == 4) {
    const float4* q = reinterpret_cast<const float4*>(p);
#pragma unroll
    for (int t = 0; t < K; ++t) {        // 4 K floats = K float4
      const float4 a = __ldg(q + t);
      const float f[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) xv[(4 * t + u) / K][(4 * t + u) % K] = f[u];
    }
  } else {
    const double2* q = reinterpret_cast<const double2*>(p);
#pragma unroll
    for (int t = 0; t < 2 * K; ++t) {    // 4 K doubles = 2 K double2
      const double2 a = __ldg(q + t);
      xv[(2 * t) / K][(2 * t) % K] = a.x;
      xv[(2 * t + 1) / K][(2 * t + 1) % K] = a.y;
    }
  }
}

constexpr int kSpmvThreads = 128;
// CTAs on an SM, which sets the registers: four atoms' values and x rows in flight at K = 1, more warps with two or one
// (FP32 values and x, 262,144 atoms: K = 1 at 5 / 8 CTAs 50 / 68 us, K = 4 79 / 70).
template <typename TX, int K>
constexpr int kSpmvBlocks = sizeof(TX) == 8 ? (K == 1 ? 4 : 5) : (K == 1 ? 5 : 8);

// A warp takes PER neighbouring atoms at a time: lane = (place, slot, row i), 8 / SLOTS places of 4 / K atoms each; the
// lane has row i of the blocks slot, slot + SLOTS, ... of its place's atoms, so that a load takes whole blocks that lie
// next to each other, and 4 / K atoms of K vectors are four sums a lane, which the slots halve among themselves. Warps
// walk over the system with the next atoms' columns and row pointers loaded ahead, so that only one latency is left
// between values and products.
// Memory bounds FP32 and BF16 values, the FP64 pipe bounds FP64 vectors (stored FP32 values are widened by integer
// operations: 275 -> 136 us at K = 1). A thread per row with its 13 blocks one after another: FP32, K = 1, 262,144 atoms
// 57 us against 45 here (36 is the floor); 512 atoms, FP64, K = 4, on 8 SMs, 22.5 against 6.1.
template <typename TV, typename TX, int K, int SLOTS>
__global__ void __launch_bounds__(kSpmvThreads, (kSpmvBlocks<TX, K>))
    spmv_kernel(const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col, const TV* __restrict__ val,
                const TX* __restrict__ x, TX* __restrict__ y, int64_t n_rows) {
  using TL = typename std::conditional<std::is_same<TV, double>::value, double, float>::type;
  constexpr int A = 4 / K, PER = A * (8 / SLOTS), R = 2;
  constexpr bool kAhead = sizeof(TX) == 4;
  const int lane = threadIdx.x & 31, i = lane & 3, slot = (lane >> 2) % SLOTS, place = lane / (4 * SLOTS);
  const int64_t nw = (int64_t)gridDim.x * (kSpmvThreads / 32);
  const int64_t groups = (n_rows + PER - 1) / PER;
  int64_t g = ((int64_t)blockIdx.x * kSpmvThreads + threadIdx.x) >> 5;
  if (g >= groups) return;
  auto pointer = [&](int64_t gg) {      // lane l: row pointer of the group's atom l (the end beyond the last)
    const int64_t a = gg * PER + (lane < PER ? lane : PER);
    return gg < groups ? __ldg(row_ptr + (a < n_rows ? a : n_rows)) : 0;
  };
  int k0[A], k1[A], cb[A][R];
  auto take = [&](int rp) {             // the lane's atoms of a group: bounds and first columns
#pragma unroll
    for (int u = 0; u < A; ++u) {
      k0[u] = __shfl_sync(0xffffffffu, rp, place * A + u) + slot;
      k1[u] = __shfl_sync(0xffffffffu, rp, place * A + u + 1);
#pragma unroll
      for (int h = 0; h < R; ++h) cb[u][h] = k0[u] + SLOTS * h < k1[u] ? __ldg(col + k0[u] + SLOTS * h) : -1;
    }
  };
  int rp = pointer(g), next = pointer(g + nw);
  take(rp);
  for (; g < groups; g += nw) {
    TX s[4] = {0, 0, 0, 0};
    for (bool first = true;; first = false) {
      TL v[A][R][4];
      int c[A][R];
      bool more = false;
#pragma unroll
      for (int u = 0; u < A; ++u) {
#pragma unroll
        for (int h = 0; h < R; ++h) {
          c[u][h] = cb[u][h];
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) v[u][h][jj] = 0;
          if (c[u][h] >= 0) RowVals<TV>::load(val, k0[u] + SLOTS * h, i, v[u][h]);
        }
        more = more || k0[u] + SLOTS * R < k1[u];
      }
      const bool again = __any_sync(0xffffffffu, more);
      if (again) {
#pragma unroll
        for (int u = 0; u < A; ++u) {
          k0[u] = min(k0[u] + SLOTS * R, k1[u]);
#pragma unroll
          for (int h = 0; h < R; ++h) cb[u][h] = k0[u] + SLOTS * h < k1[u] ? __ldg(col + k0[u] + SLOTS * h) : -1;
        }
      } else {
        take(next);
        next = pointer(g + 2 * nw);
      }
      TX xs[A][R][4][K];                // FP32: all x rows in flight too; FP64 has not the registers, nor the need
      if constexpr (kAhead) {
#pragma unroll
        for (int u = 0; u < A; ++u)
#pragma unroll
          for (int h = 0; h < R; ++h) {
#pragma unroll
            for (int e = 0; e < 4 * K; ++e) xs[u][h][e / K][e % K] = 0;
            if (c[u][h] >= 0) load_x<TX, K>(x, c[u][h], xs[u][h]);
          }
      }
#pragma unroll
      for (int u = 0; u < A; ++u)
#pragma unroll
        for (int h = 0; h < R; ++h) {
          TX (&xv)[4][K] = xs[u][h];
          if constexpr (!kAhead) {
            if (c[u][h] < 0) continue;
            load_x<TX, K>(x, c[u][h], xv);
          }
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) {
            TX w;
            if constexpr (sizeof(TX) > sizeof(TL)) w = widen(v[u][h][jj]);
            else w = (TX)v[u][h][jj];
#pragma unroll
            for (int q = 0; q < K; ++q) s[u * K + q] = fma(w, xv[jj][q], s[u * K + q]);
          }
        }
      if (!again) break;
    }
    TX t[2];
    if constexpr (SLOTS == 8) {
      const int hi = lane >> 4 & 1, lo = lane >> 3 & 1;
#pragma unroll
      for (int q = 0; q < 2; ++q) t[q] = (hi ? s[2 + q] : s[q]) + __shfl_xor_sync(0xffffffffu, hi ? s[q] : s[2 + q], 16);
      TX r = (lo ? t[1] : t[0]) + __shfl_xor_sync(0xffffffffu, lo ? t[0] : t[1], 8);
      r += __shfl_xor_sync(0xffffffffu, r, 4);
      const int e = 2 * hi + lo;                  // atom e / K of the group, vector e % K
      const int64_t a = g * PER + e / K;
      if ((slot & 1) == 0 && a < n_rows) y[(4 * a + i) * K + e % K] = r;
    } else {
      const int hi = lane >> 3 & 1, lo = lane >> 2 & 1;
#pragma unroll
      for (int q = 0; q < 2; ++q) t[q] = (hi ? s[2 + q] : s[q]) + __shfl_xor_sync(0xffffffffu, hi ? s[q] : s[2 + q], 8);
      const TX r = (lo ? t[1] : t[0]) + __shfl_xor_sync(0xffffffffu, lo ? t[0] : t[1], 4);
      const int e = 2 * hi + lo;
      const int64_t a = g * PER + place * A + e / K;
      if (a < n_rows) y[(4 * a + i) * K + e % K] = r;
    }
  }
}

// A thread per row, its blocks four at a time with their loads in flight: the form for short rows, where most slots
// of the kernel above would be idle, for many rows of FP64 values, and for BF16 values with one or two FP32 vectors on large
// systems, where a block is 32 bytes and a load by slots half as wide as the lanes could take (spmv_rule.cuh).
template <typename TV, typename TX, int K>
__global__ void __launch_bounds__(256) spmv_rows_kernel(const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                                                        const TV* __restrict__ val, const TX* __restrict__ x,
                                                        TX* __restrict__ y, int64_t n_rows) {
  using TL = typename std::conditional<std::is_same<TV, double>::value, double, float>::type;
  auto entry = [](TL v) {
    if constexpr (sizeof(TX) > sizeof(TL)) return widen(v);
    else return (TX)v;
  };
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < 4 * n_rows; g += stride) {
    const int64_t a = g >> 2;
    const int i = (int)(g & 3);
    const int k0 = __ldg(row_ptr + a), k1 = __ldg(row_ptr + a + 1);
    TX acc[K];
#pragma unroll
    for (int c = 0; c < K; ++c) acc[c] = 0;
    int k = k0;
    for (; k + 4 <= k1; k += 4) {
      int cb[4];
      TL v[4][4];
#pragma unroll
      for (int u = 0; u < 4; ++u) cb[u] = __ldg(col + k + u);
#pragma unroll
      for (int u = 0; u < 4; ++u) RowVals<TV>::load(val, k + u, i, v[u]);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        TX xv[4][K];
        load_x<TX, K>(x, cb[u], xv);
#pragma unroll
        for (int jj = 0; jj < 4; ++jj)
#pragma unroll
          for (int c = 0; c < K; ++c) acc[c] = fma(entry(v[u][jj]), xv[jj][c], acc[c]);
      }
    }
    for (; k < k1; ++k) {
      TL v[4];
      TX xv[4][K];
      RowVals<TV>::load(val, k, i, v);
      load_x<TX, K>(x, __ldg(col + k), xv);
#pragma unroll
      for (int jj = 0; jj < 4; ++jj)
#pragma unroll
        for (int c = 0; c < K; ++c) acc[c] = fma(entry(v[jj]), xv[jj][c], acc[c]);
    }
#pragma unroll
    for (int c = 0; c < K; ++c) y[g * K + c] = acc[c];
  }
}

template <typename TV, typename TX, int K, int SLOTS>
void spmv_launch(const mka_system* s, const TV* val, const TX* x, TX* y, int sms, cudaStream_t st) {
  const int64_t per = (int64_t)(4 / K) * (8 / SLOTS) * (kSpmvThreads / 32);
  const int64_t blocks = std::min<int64_t>((s->n_atoms + per - 1) / per, (int64_t)sms * kSpmvBlocks<TX, K>);
  spmv_kernel<TV, TX, K, SLOTS><<<(unsigned)std::max<int64_t>(1, blocks), kSpmvThreads, 0, st>>>(
      s->d_row_ptr, s->d_col, val, x, y, s->n_atoms);
}

template <typename TV, typename TX, int K>
mka_status spmv_dispatch_k(const mka_system* s, const TV* val, const TX* x, TX* y, cudaStream_t st) {
  int dev = 0, sms = 0;
  MKA_CUDA_TRY(cudaGetDevice(&dev));
  MKA_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // Four slots waste less on rows of 13 blocks and add less (FP64, K = 4, 262,144 atoms: 492 against 539 us); eight spread
  // a small system over more warps (512 atoms, K = 4: 8.8 against 10.9 us; 4,096 atoms, K = 1: 12.9 against 15). They meet at
  // about eight warps an SM.
  const bool wide = s->n_atoms * K < (int64_t)sms * 64;
  if (spmv_by_rows(s->storage == MKA_FP64 ? 0 : s->storage == MKA_MIXED_FP32 ? 1 : 2, sizeof(TX) == 8, K, s->n_atoms, s->nnzb,
                   wide)) {
    const int64_t blocks = std::min<int64_t>((4 * s->n_atoms + 255) / 256, (int64_t)sms * 8);
    spmv_rows_kernel<TV, TX, K><<<(unsigned)blocks, 256, 0, st>>>(s->d_row_ptr, s->d_col, val, x, y, s->n_atoms);
  } else if (wide) {
    spmv_launch<TV, TX, K, 8>(s, val, x, y, sms, st);
  } else {
    spmv_launch<TV, TX, K, 4>(s, val, x, y, sms, st);
  }
  count_launches();
  MKA_CUDA_TRY(cudaGetLastError());
  return MKA_OK;
}

template <typename TV, typename TX>
mka_status spmv_dispatch_x(const mka_system* s, const TV* val, const void* x, void* y, int k, cudaStream_t st) {
  const TX* xx = reinterpret_cast<const TX*>(x);
  TX* yy = reinterpret_cast<TX*>(y);
  if (k == 1) return spmv_dispatch_k<TV, TX, 1>(s, val, xx, yy, st);
  if (k == 2) return spmv_dispatch_k<TV, TX, 2>(s, val, xx, yy, st);
  return spmv_dispatch_k<TV, TX, 4>(s, val, xx, yy, st);
}

template <typename TV>
mka_status spmv_dispatch(const mka_system* s, const void* val, int x_dtype, const void* x, void* y, int k,
                         cudaStream_t st) {
  if (x_dtype == MKA_FP64) return spmv_dispatch_x<TV, double>(s, (const TV*)val, x, y, k, st);
  return spmv_dispatch_x<TV, float>(s, (const TV*)val, x, y, k, st);
}

// ---- density of states: D(E) = -(1/pi) Im sum_j (G(E + i eta) S)_jj = (eta/pi) sum w / ((E - eps)^2 + eta^2) ----
// Grid (level chunks, energies in groups of 32 per warp): a CTA stages its chunk's levels through shared memory 256 at
// a time; its 8 warps take 8 groups of 32 energies, or, with fewer groups than warps, share a group's levels among
// them (interleaved, added in warp order), so that 41 energies do not leave 7 of 8 lanes idle. A second kernel
// adds the chunk sums in a fixed order, a warp per energy. FP64 throughout; the divisions bound it. The chunk grows with
// the levels: 32,768 levels a chunk left 14,800 levels to one CTA (12.1 ms for 201 energies, 0.11 with the chip full).
constexpr int kDosThreads = 256, kDosWarps = kDosThreads / 32;

__global__ void __launch_bounds__(kDosThreads) dos_partial_kernel(const double* eps, const double* w, int64_t n,
                                                                  const double* energies, int n_e, double eta,
                                                                  int64_t chunk, int share, double* partial) {
  __shared__ double se[kDosThreads], sw[kDosThreads], part[kDosThreads];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t l0 = (int64_t)blockIdx.x * chunk, l1 = min(n, l0 + chunk);
  const int k = (blockIdx.y * (kDosWarps / share) + wid / share) * 32 + lane, i0 = wid % share;
  const double E = k < n_e ? energies[k] : 0.0;
  const double eta2 = eta * eta;
  double acc = 0.0;
  for (int64_t t0 = l0; t0 < l1; t0 += kDosThreads) {
    const int64_t t = t0 + threadIdx.x;
    se[threadIdx.x] = t < l1 ? eps[t] : 0.0;
    sw[threadIdx.x] = t < l1 ? w[t] : 0.0;
    __syncthreads();
    const int cnt = (int)(l1 - t0 < kDosThreads ? l1 - t0 : kDosThreads);
#pragma unroll 4
    for (int i = i0; i < cnt; i += share) {
      const double wi = sw[i], d = E - se[i];
      if (wi != 0.0) acc += wi / fma(d, d, eta2);
    }
    __syncthreads();
  }
  part[threadIdx.x] = acc;
  __syncthreads();
  if (i0 == 0 && k < n_e) {
    for (int s = 1; s < share; ++s) acc += part[threadIdx.x + 32 * s];
    partial[(int64_t)k * gridDim.x + blockIdx.x] = acc;
  }
}

__global__ void __launch_bounds__(256) dos_sum_kernel(const double* partial, int64_t n_chunks, int n_e, double scale,
                                                      double* out) {
  const int k = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (k >= n_e) return;
  double s = 0.0;
  for (int64_t c = lane; c < n_chunks; c += 32) s += partial[k * n_chunks + c];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) out[k] = scale * s;
}

// H's on-site blocks += shift[a] on the diagonal (one thread per atom): the diagonal block of row a found in
// its sorted columns, the stored value decoded, shifted and stored again in its format.
__global__ void onsite_shift_kernel(const int32_t* row_ptr, const int32_t* col, void* valH, int storage,
                                    const double* shift, int64_t n) {
  for (int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; a < n; a += (int64_t)gridDim.x * blockDim.x) {
    int lo = row_ptr[a], hi = row_ptr[a + 1] - 1, k = -1;
    while (lo <= hi) {
      const int mid = (lo + hi) >> 1;
      if (col[mid] == a) { k = mid; break; }
      if (col[mid] < a) lo = mid + 1; else hi = mid - 1;
    }
    if (k < 0) continue;
    for (int o = 0; o < 4; ++o) {
      const int64_t i = (int64_t)k * 16 + 5 * o;
      if (storage == MKA_FP64) reinterpret_cast<double*>(valH)[i] += shift[a];
      else if (storage == MKA_MIXED_FP32) reinterpret_cast<float*>(valH)[i] = (float)((double)reinterpret_cast<float*>(valH)[i] + shift[a]);
      else {
        __nv_bfloat16* v = reinterpret_cast<__nv_bfloat16*>(valH);
        v[i] = __double2bfloat16((double)__bfloat162float(v[i]) + shift[a]);
      }
    }
  }
}

}  // namespace

mka_status launch_onsite_shift(mka_system* sys, const double* shift_host, cudaStream_t st) {
  double* d = nullptr;
  MKA_CUDA_TRY(cudaMallocAsync(&d, sizeof(double) * sys->n_atoms, st));
  cudaError_t e = cudaMemcpyAsync(d, shift_host, sizeof(double) * sys->n_atoms, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) {
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((sys->n_atoms + 255) / 256, 4096));
    onsite_shift_kernel<<<(unsigned)blocks, 256, 0, st>>>(sys->d_row_ptr, sys->d_col, sys->d_valH, sys->storage, d,
                                                         sys->n_atoms);
    count_launches();
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFreeAsync(d, st);
  if (e != cudaSuccess) return cuda_fail(e, "mka_system_shift_onsite");
  return MKA_OK;
}

mka_status launch_dos(const double* eps, const double* w, int64_t n, const double* energies, int n_e, double eta,
                      cudaStream_t st, double* dos_host) {
  // 8 groups of 32 energies a CTA; with fewer the warps share a group. About four CTAs per SM, 64 to 32,768 levels each.
  const int groups = (n_e + 31) / 32, share = groups >= 8 ? 1 : groups >= 4 ? 2 : groups >= 2 ? 4 : 8;
  const int gy = (groups + kDosWarps / share - 1) / (kDosWarps / share);
  const int64_t fill = std::max(1, red_blocks() / gy);   // chunks; one more than fill the SMs evenly costs a fifth
  int64_t chunk = (n + fill - 1) / fill;
  chunk = std::min<int64_t>(32768, std::max<int64_t>(64, (chunk + 63) / 64 * 64));
  const int64_t n_chunks = std::max<int64_t>(1, (n + chunk - 1) / chunk);
  double* buf = nullptr;
  MKA_CUDA_TRY(cudaMallocAsync(&buf, sizeof(double) * ((size_t)n_chunks * n_e + 2 * (size_t)n_e), st));
  double* d_e = buf + (size_t)n_chunks * n_e;
  double* d_out = d_e + n_e;
  cudaError_t e = cudaMemcpyAsync(d_e, energies, sizeof(double) * n_e, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) {
    const dim3 grid((unsigned)n_chunks, (unsigned)gy);
    dos_partial_kernel<<<grid, kDosThreads, 0, st>>>(eps, w, n, d_e, n_e, eta, chunk, share, buf);
    dos_sum_kernel<<<(n_e + 7) / 8, 256, 0, st>>>(buf, n_chunks, n_e, eta / 3.14159265358979323846, d_out);
    count_launches(2);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(dos_host, d_out, sizeof(double) * n_e, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFreeAsync(buf, st);
  if (e != cudaSuccess) return cuda_fail(e, "mka_dos");
  return MKA_OK;
}

static int blocks_of(int64_t n) {
  return (int)std::min<int64_t>(red_blocks(), std::max<int64_t>(1, (n + kRedThreads - 1) / kRedThreads));
}

size_t mu_buffer_bytes() { return sizeof(RootState) + sizeof(double) * 2 * kMaxRedBlocks + 64; }

mka_status find_mu_enqueue(const double* eps, const double* w, int64_t n_cols, int nu, double n_electrons, double kT,
                           double tol, int passes, void* buf, double* mu_dev_out, cudaStream_t st) {
  RootState* S = reinterpret_cast<RootState*>(buf);
  double* partial = reinterpret_cast<double*>(S + 1);
  unsigned* ticket = reinterpret_cast<unsigned*>(partial + 2 * kMaxRedBlocks);
  mu_init_kernel<<<1, 1, 0, st>>>(S, ticket, n_electrons, kT, tol);
  eps_range_kernel<<<blocks_of(n_cols * nu), kRedThreads, 0, st>>>(eps, w, n_cols * nu, partial, ticket, S);
  const int share = lanes_per_column(n_cols);
  for (int i = 0; i < passes; ++i)
    mu_pass_kernel<<<blocks_of(n_cols * share), kRedThreads, 0, st>>>(eps, w, n_cols, nu, share, partial, ticket, S,
                                                                      passes - 1 - i);
  mu_finish_kernel<<<1, 1, 0, st>>>(S, mu_dev_out);
  count_launches(3 + passes);
  MKA_CUDA_TRY(cudaGetLastError());
  return MKA_OK;
}

mka_status density_enqueue(const mka_system* sys, const int64_t* sel, const int64_t* blk_off, const double* vp,
                           const double* cv, const double* eps, const double* w, int64_t n_sel, int nu,
                           const double* mu_dev, double kT, double* rho_out, double* tmp, cudaStream_t st) {
  density_kernel<<<(unsigned)n_sel, 128, sizeof(double) * 8 * nu, st>>>(vp, cv, eps, blk_off, sel, sys->d_row_ptr, sys->d_valH,
                                                  sys->storage, nu, 0.0, mu_dev, kT, rho_out, tmp);
  sum_kernel<<<1, kRedThreads, 0, st>>>(tmp, n_sel, tmp + n_sel);
  const int rb = red_blocks();
  count_partial_kernel<<<rb, kRedThreads, 0, st>>>(eps, w, 4 * n_sel, nu, lanes_per_column(4 * n_sel), 0.0, mu_dev, kT,
                                                    tmp + n_sel + 2);
  sum_kernel<<<1, kRedThreads, 0, st>>>(tmp + n_sel + 2, rb, tmp + n_sel + 1);
  count_launches(4);
  MKA_CUDA_TRY(cudaGetLastError());
  return MKA_OK;
}

mka_status density_global_enqueue(const mka_system* sys, const int64_t* sel, const int64_t* blk_off, const double* vp,
                                  const double* cv, const double* eps, int64_t n_sel, int nu, double mu, double kT,
                                  double* rho, int64_t out_base, double* e_atom, int64_t e_base, cudaStream_t st) {
  density_kernel<<<(unsigned)n_sel, 128, sizeof(double) * 8 * nu, st>>>(vp, cv, eps, blk_off, sel, sys->d_row_ptr, sys->d_valH, sys->storage,
                                                  nu, mu, nullptr, kT, rho, e_atom, out_base, e_base);
  count_launches();
  MKA_CUDA_TRY(cudaGetLastError());
  return MKA_OK;
}

mka_status launch_find_mu(mka_result* res, double n_electrons, double kT, double tol, double* mu_out) {
  cudaStream_t st = res->stream;
  const int64_t n = res->n_cols * res->nu;
  if (!res->d_mu_state) {
    MKA_CUDA_TRY(cudaMalloc(&res->d_mu_state, mu_buffer_bytes()));
    MKA_CUDA_TRY(cudaMemsetAsync(res->d_mu_state, 0, mu_buffer_bytes(), st));
  }
  RootState* S = reinterpret_cast<RootState*>(res->d_mu_state);
  double* partial = reinterpret_cast<double*>(S + 1);
  unsigned* ticket = reinterpret_cast<unsigned*>(partial + 2 * kMaxRedBlocks);
  mu_init_kernel<<<1, 1, 0, st>>>(S, ticket, n_electrons, kT, tol);
  eps_range_kernel<<<blocks_of(n), kRedThreads, 0, st>>>(res->d_eps, res->d_w, n, partial, ticket, S);
  count_launches(2);
  MKA_CUDA_TRY(cudaGetLastError());
  // sixteen passes usually end the search (those after convergence return at once); the bracket comes back and
  // more follow while it is wider than tol
  constexpr int kBatch = 16, kTotal = 13 * kBatch;
  const int share = lanes_per_column(res->n_cols);
  RootState h{};
  for (int done = 0; done < kTotal; done += kBatch) {
    for (int i = 0; i < kBatch; ++i)
      mu_pass_kernel<<<blocks_of(res->n_cols * share), kRedThreads, 0, st>>>(res->d_eps, res->d_w, res->n_cols, res->nu, share,
                                                                             partial, ticket, S, kTotal - 1 - done - i);
    count_launches(kBatch);
    MKA_CUDA_TRY(cudaGetLastError());
    MKA_CUDA_TRY(cudaMemcpyAsync(&h, S, sizeof(RootState), cudaMemcpyDeviceToHost, st));
    MKA_CUDA_TRY(cudaStreamSynchronize(st));
    if (!(h.hi > h.lo) && h.iters == 0) return fail(MKA_ERR_INVALID_ARG, "no level with nonzero weight");
    if (!(h.hi - h.lo > tol)) break;
  }
  *mu_out = 0.5 * (h.lo + h.hi);
  return MKA_OK;
}

mka_status launch_density(mka_system* sys, mka_result* res, double mu, double kT, double* rho_out, double* e_band,
                          double* n_elec) {
  cudaStream_t st = res->stream;
  double* tmp = nullptr;
  const int rb = red_blocks();
  MKA_CUDA_TRY(cudaMallocAsync(&tmp, sizeof(double) * (res->n_sel + 2 + rb), st));
  density_kernel<<<(unsigned)res->n_sel, 128, sizeof(double) * 8 * res->nu, st>>>(res->d_vp, res->d_cv, res->d_eps, res->d_blk_off,
                                                       res->d_sel, sys->d_row_ptr, sys->d_valH, sys->storage,
                                                       res->nu, mu, nullptr, kT, rho_out, tmp);
  sum_kernel<<<1, kRedThreads, 0, st>>>(tmp, res->n_sel, tmp + res->n_sel);
  count_partial_kernel<<<rb, kRedThreads, 0, st>>>(res->d_eps, res->d_w, res->n_cols, res->nu, lanes_per_column(res->n_cols), mu,
                                                   nullptr, kT, tmp + res->n_sel + 2);
  sum_kernel<<<1, kRedThreads, 0, st>>>(tmp + res->n_sel + 2, rb, tmp + res->n_sel + 1);
  count_launches(4);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess && (e_band || n_elec)) {
    double h[2];
    e = cudaMemcpyAsync(h, tmp + res->n_sel, sizeof(h), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess) {
      if (e_band) *e_band = h[0];
      if (n_elec) *n_elec = h[1];
    }
  }
  cudaFreeAsync(tmp, st);
  if (e != cudaSuccess) return cuda_fail(e, "density");
  return MKA_OK;
}

mka_status launch_greens(mka_system* sys, mka_result* res, double z_re, double z_im, double* g_out) {
  greens_kernel<<<(unsigned)res->n_sel, 128, sizeof(double) * 16 * res->nu, res->stream>>>(res->d_vp, res->d_cv, res->d_eps, res->d_blk_off,
                                                               res->d_sel, sys->d_row_ptr, res->nu, z_re, z_im, g_out);
  count_launches();
  MKA_CUDA_TRY(cudaGetLastError());
  return MKA_OK;
}

mka_status launch_spmv(const mka_system* s, int which, int x_dtype, const void* x, void* y, int k, cudaStream_t st) {
  const void* val = which == 0 ? s->d_valH : s->d_valS;
  switch (s->storage) {
    case MKA_FP64: return spmv_dispatch<double>(s, val, x_dtype, x, y, k, st);
    case MKA_MIXED_FP32: return spmv_dispatch<float>(s, val, x_dtype, x, y, k, st);
    default: return spmv_dispatch<__nv_bfloat16>(s, val, x_dtype, x, y, k, st);
  }
}

}  // namespace mka
