// What the two per-atom kernels share: kernel arguments, stored-value loads, cluster extraction and
// its local block pattern, cluster products, and CTA sums (columns.cu: the general basis; chains.cu:
// the short-recurrence basis).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "mka_internal.h"
#include "widen.cuh"

namespace mka {
namespace {

constexpr int kMaxWarps = 16;   // CTAs of up to 512 threads
constexpr int kMaxCl = MKA_MAX_CLUSTER_ATOMS;  // power of two (bitonic sort size bound)
static_assert((kMaxCl & (kMaxCl - 1)) == 0, "cluster cap must be a power of two");

__host__ __device__ constexpr size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

enum ColStatus { ST_OK = 0, ST_NOT_SPD = MKA_ERR_NOT_SPD, ST_NOCONV = MKA_ERR_NO_CONVERGENCE,
                 ST_BREAKDOWN = MKA_ERR_BREAKDOWN, ST_TOOLARGE = MKA_ERR_CLUSTER_TOO_LARGE };
enum Src { SRC_E = 0, SRC_H = 1, SRC_S = 2, SRC_R = 3 };   // SRC_R: a raw power H^k s_j (reading B)
enum Act { ACT_NONE = 0, ACT_LOAD_K = 1, ACT_LOAD_S = 2 };

// ---- value loads: one row (4 entries) of a 4x4 block, decoded ----------------
// FP32 and BF16 values are widened to FP64 off the FP64 pipe (CG of 1,500 columns' atoms: 24.0 -> 17.5 ms).
template <typename TV, typename T>
struct RowLoad;
template <typename T>
struct RowLoad<double, T> {
  static __device__ __forceinline__ void load(const double* v, int64_t blk, int i, T out[4]) {
    const double2* p = reinterpret_cast<const double2*>(v + blk * 16 + i * 4);
    double2 a = __ldg(p), b = __ldg(p + 1);
    out[0] = (T)a.x; out[1] = (T)a.y; out[2] = (T)b.x; out[3] = (T)b.y;
  }
};
template <typename T>
struct RowLoad<float, T> {
  static __device__ __forceinline__ void load(const float* v, int64_t blk, int i, T out[4]) {
    float4 a = __ldg(reinterpret_cast<const float4*>(v + blk * 16 + i * 4));
    out[0] = widen_to<T>(a.x); out[1] = widen_to<T>(a.y); out[2] = widen_to<T>(a.z); out[3] = widen_to<T>(a.w);
  }
};
template <typename T>
struct RowLoad<__nv_bfloat16, T> {
  static __device__ __forceinline__ void load(const __nv_bfloat16* v, int64_t blk, int i, T out[4]) {
    uint2 a = __ldg(reinterpret_cast<const uint2*>(v + blk * 16 + i * 4));
    out[0] = widen_to<T>(__uint_as_float(a.x << 16)); out[1] = widen_to<T>(__uint_as_float(a.x & 0xFFFF0000u));
    out[2] = widen_to<T>(__uint_as_float(a.y << 16)); out[3] = widen_to<T>(__uint_as_float(a.y & 0xFFFF0000u));
  }
};

// ---- kernel arguments ----------------------------------------------------------
template <typename TV>
struct Args {
  // system
  int64_t n_atoms;
  const int32_t* row_ptr;
  const int32_t* col;
  const TV* valH;
  const TV* valS;
  const double* pos;
  const float* posf;      // positions rounded to FP32, for the distance prefilter
  double box[3];
  double R2;
  float pre_lo, pre_hi;   // FP32 prefilter: inside below pre_lo * R^2, outside above pre_hi * R^2
  int ncell[3];
  double cell_len[3];
  const int32_t* cell_start;
  const int32_t* cell_atoms;
  // work
  const int64_t* sel;
  const int32_t* order;   // optional work order (selection indices), NULL = selection order
  int64_t n_sel;
  const int* n_dev;       // selection size on the device (NULL: n_sel)
  int* work_counter;
  int32_t* redo;          // short-recurrence kernel: atoms left to the general one, and their count
  int* redo_count;
  int* late_count;        // those of them that the kernel had worked on
  // method
  int p, q, nu;
  double cg_tol;
  int cg_maxit;
  double tau;
  // scratch
  char* scratch;
  size_t slot_bytes;
  int mcap;            // 4 x (largest cluster of the selection)
  int lnnz_cap;        // local-block capacity per cluster
  int clcap;           // cluster list capacity (power of two)
  // outputs
  double* eps;
  double* w;
  int32_t* nu_eff;
  int32_t* cg_iters;
  int32_t* status;
  int keep;
  double* vp;
  const int64_t* blk_off;
  // learned warm start: predicted s_j on the 17-atom patch, or NULL for x0 = 0
  const float* x0;          // [4 n_sel][68]
  const int32_t* patch;     // [n_sel][17] atom ids (-1: none)
  int32_t* fallback;        // [4 n_sel]: 1 where the prediction was no better than x0 = 0 (may be NULL)
  // CG-only mode: stop after the inner CG and write s_j on the patch (training targets)
  int cg_only;
  float* cg_target;         // [4 n_sel][68]
  // 1: the s_j chain continues from its raw vector (the literal direct sum K_p(H; e_j) + K_q(H; s_j))
  int mode_b;
  // s_j of an earlier solve of the same atoms as the CG start: its clusters' atom ids [n_sel][prev_cap]
  // (ascending, -1 beyond the count) and values [4 n_sel][4 prev_cap] (NULL: not used)
  const int32_t* prev_cl;
  const double* prev_s;
  int prev_cap;
  // keep this solve's s_j the same way (NULL: not kept), keep_cap atoms per cluster
  int32_t* keep_cl;
  double* keep_s;
  int keep_cap;
  double* red;              // reduced-problem buffer, lane-interleaved per 32 columns
  unsigned long long zero;  // two FP32 zeros the assembler cannot fold (packed products in chains.cu)
};

// ---- small CTA helpers -------------------------------------------------------------
template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sums a[0..3] over the CTA; the result lands in out[0..3] (shared) for every thread.
__device__ __forceinline__ void cta_sum4(double a[4], double* red, double* out) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int c = 0; c < 4; ++c) a[c] = warp_sum(a[c]);
  if (lane == 0) {
#pragma unroll
    for (int c = 0; c < 4; ++c) red[wid * 4 + c] = a[c];
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double s = 0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += red[k * 4 + threadIdx.x];
    out[threadIdx.x] = s;
  }
  __syncthreads();
}

// Binary search of atom id c in the sorted cluster list; -1 when absent.
__device__ __forceinline__ int find_local(const int* cl, int n, int c) {
  int lo = 0, hi = n - 1;
  while (lo <= hi) {
    int mid = (lo + hi) >> 1;
    int v = cl[mid];
    if (v == c) return mid;
    if (v < c) lo = mid + 1; else hi = mid - 1;
  }
  return -1;
}

__device__ __forceinline__ double min_image(double d, double L) { return d - L * rint(d / L); }

// Is atom b within R of the point (px, py, pz) (minimum image)? An FP32 test decides every
// candidate whose FP32 distance is clear of the boundary by more than its rounding error
// (relative margin max(1e-3, 1e-5 L / R) on R^2); the rest get the exact FP64 test.
__device__ __forceinline__ bool within_R(const double* pos, const float* posf, const double box[3], double R2,
                                         float pre_lo, float pre_hi, int b, double px, double py, double pz,
                                         float pxf, float pyf, float pzf) {
  const float Lx = (float)box[0], Ly = (float)box[1], Lz = (float)box[2];
  float fx = posf[3 * b] - pxf, fy = posf[3 * b + 1] - pyf, fz = posf[3 * b + 2] - pzf;
  fx -= Lx * rintf(fx / Lx);
  fy -= Ly * rintf(fy / Ly);
  fz -= Lz * rintf(fz / Lz);
  const float r2f = fx * fx + fy * fy + fz * fz;
  const float R2f = (float)R2;
  if (r2f < pre_lo * R2f) return true;
  if (r2f > pre_hi * R2f) return false;
  const double dx = pos[3 * b] - px - box[0] * rint((pos[3 * b] - px) / box[0]);
  const double dy = pos[3 * b + 1] - py - box[1] * rint((pos[3 * b + 1] - py) / box[1]);
  const double dz = pos[3 * b + 2] - pz - box[2] * rint((pos[3 * b + 2] - pz) / box[2]);
  const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
  return r2 <= R2;
}

__device__ __forceinline__ int cell_range(int c, int n, int out[3]) {
  if (n < 3) {
    for (int i = 0; i < n; ++i) out[i] = i;
    return n;
  }
  out[0] = (c + n - 1) % n;
  out[1] = c;
  out[2] = (c + 1) % n;
  return 3;
}

__device__ __forceinline__ int cell_coord(double x, double len, int n) {
  int v = (int)floor(x / len);
  return v < 0 ? 0 : (v >= n ? n - 1 : v);
}

// Atoms within R of atom a (minimum image) appended to cl via the shared counter;
// returns the count (which may exceed A.clcap: then nothing beyond A.clcap is stored).
template <typename TV>
__device__ int gather_cluster(const Args<TV>& A, int64_t a, int* cl, int* cnt) {
  if (threadIdx.x == 0) *cnt = 0;
  __syncthreads();
  const double px = A.pos[3 * a], py = A.pos[3 * a + 1], pz = A.pos[3 * a + 2];
  const float pxf = A.posf[3 * a], pyf = A.posf[3 * a + 1], pzf = A.posf[3 * a + 2];
  int rx[3], ry[3], rz[3];
  const int nx = cell_range(cell_coord(px, A.cell_len[0], A.ncell[0]), A.ncell[0], rx);
  const int ny = cell_range(cell_coord(py, A.cell_len[1], A.ncell[1]), A.ncell[1], ry);
  const int nz = cell_range(cell_coord(pz, A.cell_len[2], A.ncell[2]), A.ncell[2], rz);
  const int ncells = nx * ny * nz;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int ci = wid; ci < ncells; ci += (int)(blockDim.x >> 5)) {
    const int ix = ci / (ny * nz), iy = (ci / nz) % ny, iz = ci % nz;
    const int c = (rx[ix] * A.ncell[1] + ry[iy]) * A.ncell[2] + rz[iz];
    const int s0 = A.cell_start[c], s1 = A.cell_start[c + 1];
    for (int k = s0 + lane; k < s1; k += 32) {
      const int b = A.cell_atoms[k];
      if (within_R(A.pos, A.posf, A.box, A.R2, A.pre_lo, A.pre_hi, b, px, py, pz, pxf, pyf, pzf)) {
        const int idx = atomicAdd(cnt, 1);
        if (idx < A.clcap) cl[idx] = b;
      }
    }
  }
  __syncthreads();
  return *cnt;
}

// Ascending bitonic sort of cl[0..n) (n <= the list's power-of-two capacity), padding with INT_MAX.
__device__ void sort_cluster(int* cl, int n) {
  int N = 2;
  while (N < n) N <<= 1;
  for (int i = n + threadIdx.x; i < N; i += blockDim.x) cl[i] = 0x7fffffff;
  __syncthreads();
  for (int k = 2; k <= N; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const int ixj = i ^ j;
        if (ixj > i) {
          const int x = cl[i], y = cl[ixj];
          const bool up = (i & k) == 0;
          if ((x > y) == up) {
            cl[i] = y;
            cl[ixj] = x;
          }
        }
      }
      __syncthreads();
    }
  }
}

// 16-byte (float) / 2 x 16-byte (double) access to one [row][4] entry of a work vector.
__device__ __forceinline__ void ld4(const float* p, float v[4]) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}
__device__ __forceinline__ void ld4(const double* p, double v[4]) {
  const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void st4(float* p, float a0, float a1, float a2, float a3) {
  *reinterpret_cast<float4*>(p) = make_float4(a0, a1, a2, a3);
}
__device__ __forceinline__ void st4(double* p, double a0, double a1, double a2, double a3) {
  reinterpret_cast<double2*>(p)[0] = make_double2(a0, a1);
  reinterpret_cast<double2*>(p)[1] = make_double2(a2, a3);
}

// y = A x on the cluster for the columns in `mask` (bit c = column c), rows 4t + i;
// x, y are [m][4] in shared memory; other columns of y are left untouched.
template <typename TV, typename T>
__device__ __forceinline__ void spmm4(const TV* __restrict__ val, const int* lrow, const uint16_t* lcol,
                                      const int* rbase, const uint8_t* loff, int ncl, const T* __restrict__ x, T* __restrict__ y,
                                      int mask) {
  const int m = 4 * ncl;
  for (int r = threadIdx.x; r < m; r += blockDim.x) {
    const int t = r >> 2, i = r & 3;
    const int rb = rbase[t];
    T a0 = 0, a1 = 0, a2 = 0, a3 = 0;
    const int e1 = lrow[t + 1];
#pragma unroll 4
    for (int e = lrow[t]; e < e1; ++e) {
      T v[4];
      RowLoad<TV, T>::load(val, rb + loff[e], i, v);
      const T* xb = x + (size_t)lcol[e] * 16;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        T xk[4];
        ld4(xb + 4 * k, xk);
        a0 += v[k] * xk[0];
        a1 += v[k] * xk[1];
        a2 += v[k] * xk[2];
        a3 += v[k] * xk[3];
      }
    }
    if (mask == 15) {
      st4(y + 4 * r, a0, a1, a2, a3);
    } else {
      if (mask & 1) y[4 * r + 0] = a0;
      if (mask & 2) y[4 * r + 1] = a1;
      if (mask & 4) y[4 * r + 2] = a2;
      if (mask & 8) y[4 * r + 3] = a3;
    }
  }
  __syncthreads();
}

// r = e_j - A (hi + lo) for x given as an FP32 pair: the hi part with error-free products and
// compensated sums as in resid4_comp, the small lo part (|lo| <= ulp(hi) / 2) in plain FP32.
template <typename TV>
__device__ void resid4_comp2(const TV* __restrict__ val, const int* lrow, const uint16_t* lcol, const int* rbase, const uint8_t* loff,
                             int ncl, const float* __restrict__ xh, const float* __restrict__ xl, float* __restrict__ r,
                             int jrow0) {
  for (int row = threadIdx.x; row < 4 * ncl; row += blockDim.x) {
    const int t = row >> 2, i = row & 3;
    const int rb = rbase[t];
    float hi[4] = {0, 0, 0, 0}, lo[4] = {0, 0, 0, 0}, sl[4] = {0, 0, 0, 0};
    for (int e = lrow[t]; e < lrow[t + 1]; ++e) {
      float v[4];
      RowLoad<TV, float>::load(val, rb + loff[e], i, v);
      const float* xb = xh + (size_t)lcol[e] * 16;
      const float* xc = xl + (size_t)lcol[e] * 16;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        float xk[4], xs[4];
        ld4(xb + 4 * k, xk);
        ld4(xc + 4 * k, xs);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float p = __fmul_rn(v[k], xk[q]);
          const float pe = fmaf(v[k], xk[q], -p);
          const float s = __fadd_rn(hi[q], p);
          const float bb = __fsub_rn(s, hi[q]);
          const float err = __fadd_rn(__fsub_rn(hi[q], __fsub_rn(s, bb)), __fsub_rn(p, bb));
          hi[q] = s;
          lo[q] = __fadd_rn(lo[q], __fadd_rn(err, pe));
          sl[q] = fmaf(v[k], xs[q], sl[q]);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float e = (row == jrow0 + q) ? 1.0f : 0.0f;
      r[4 * row + q] = __fsub_rn(__fsub_rn(__fsub_rn(e, hi[q]), lo[q]), sl[q]);
    }
  }
  __syncthreads();
}
// Per-column dot products over the cluster rows: per-thread partial sums in T
// (a few terms each), combined across threads in FP64.
template <typename T>
__device__ __forceinline__ void dot4(const T* a, const T* b, int m, double* red, double* out) {
  T part[4] = {0, 0, 0, 0};
  for (int r = threadIdx.x; r < m; r += blockDim.x) {
#pragma unroll
    for (int c = 0; c < 4; ++c) part[c] += a[4 * r + c] * b[4 * r + c];
  }
  double acc[4] = {(double)part[0], (double)part[1], (double)part[2], (double)part[3]};
  cta_sum4(acc, red, out);
}

template <typename TV>
void fill_system_args(Args<TV>& A, const mka_system* s) {
  A.n_atoms = s->n_atoms;
  A.row_ptr = s->d_row_ptr;
  A.col = s->d_col;
  A.valH = reinterpret_cast<const TV*>(s->d_valH);
  A.valS = reinterpret_cast<const TV*>(s->d_valS);
  A.pos = s->d_pos;
  A.posf = s->d_posf;
  for (int d = 0; d < 3; ++d) {
    A.box[d] = s->box[d];
    A.ncell[d] = s->cells.n[d];
    A.cell_len[d] = s->cells.len[d];
  }
  A.R2 = s->R * s->R;
  const double lmax = std::max(s->box[0], std::max(s->box[1], s->box[2]));
  const double margin = std::max(1e-3, 1e-5 * lmax / s->R);
  A.pre_lo = (float)(1.0 - margin);
  A.pre_hi = (float)(1.0 + margin);
  A.cell_start = s->cells.start;
  A.cell_atoms = s->cells.atoms;
}

template <typename TV>
void fill_args(Args<TV>& A, const mka_system* sys, const AtomsConfig& cf, const AtomsLaunchArgs& a) {
  fill_system_args(A, sys);
  A.sel = a.sel;
  A.order = a.order;
  A.n_sel = a.n_sel;
  A.work_counter = a.counter;
  A.p = a.p;
  A.q = a.q;
  A.nu = a.p + a.q;
  A.cg_tol = a.cg_tol;
  A.cg_maxit = a.cg_maxit;
  A.tau = 1e-10;
  A.scratch = a.scratch;
  A.slot_bytes = cf.slot_bytes;
  A.mcap = cf.mcap;
  A.lnnz_cap = cf.lnnz_cap;
  A.clcap = cf.clcap;
  A.eps = a.eps;
  A.w = a.w;
  A.nu_eff = a.nu_eff;
  A.cg_iters = a.cg_iters;
  A.status = a.status;
  A.keep = a.keep;
  A.vp = a.vp;
  A.blk_off = a.blk_off;
  A.x0 = a.x0;
  A.patch = a.patch;
  A.fallback = a.fallback;
  A.cg_only = a.cg_only;
  A.cg_target = a.cg_target;
  A.mode_b = a.mode_b;
  A.prev_cl = a.prev_cl;
  A.prev_s = a.prev_s;
  A.prev_cap = a.prev_cap;
  A.keep_cl = a.keep_cl;
  A.keep_s = a.keep_s;
  A.keep_cap = a.keep_cap;
  A.red = a.red;
}

// Dispatch on (storage type, arithmetic, CTA size).
#define MKA_DISPATCH_T(CALL, TV, T, threads)        \
  ((threads) == 128 ? CALL(TV, T, 128) : (threads) == 512 ? CALL(TV, T, 512) : CALL(TV, T, 256))
#define MKA_DISPATCH(CALL, storage, mixed, threads)                                                        \
  ((storage) == MKA_FP64 ? ((mixed) ? MKA_DISPATCH_T(CALL, double, float, threads)                         \
                                    : MKA_DISPATCH_T(CALL, double, double, threads))                       \
   : (storage) == MKA_MIXED_FP32 ? ((mixed) ? MKA_DISPATCH_T(CALL, float, float, threads)                  \
                                            : MKA_DISPATCH_T(CALL, float, double, threads))                \
   : ((mixed) ? MKA_DISPATCH_T(CALL, __nv_bfloat16, float, threads)                                        \
              : MKA_DISPATCH_T(CALL, __nv_bfloat16, double, threads)))

}  // namespace
}  // namespace mka
