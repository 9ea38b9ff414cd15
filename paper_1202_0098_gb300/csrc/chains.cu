// The per-atom kernel in short recurrences: the basis of K_p(H; e_j) (+) K_q(H; s_j) (reading A of the
// seam) without Gram-Schmidt against the whole basis.
//
// Only the span and its two Gram matrices enter the reduced problem (columns.cu forms S_r explicitly
// for the same reason), so the basis need not be S-orthonormal. Here it is 2-orthonormal, where H is
// symmetric, and every vector comes from the last two:
//   first chain    q_1 = e_j,  beta_n q_{n+1} = H q_n - alpha_n q_n - beta_{n-1} q_{n-1}   (Lanczos), n <= p;
//   second chain   the span wanted is K_p + K_q((I - Pi) H; (I - Pi) s_j), Pi the S-orthogonal projector
//     onto K_p. Modulo K_p, (I - Pi) v = v - (...) and H leaves K_p only through q_p, so that
//       (I - Pi) H (I - Pi) v = H v - (z.v) beta_p q_{p+1}   mod K_p,   z = S Q (Q^T S Q)^{-1} e_p:
//     one dot product with a fixed vector replaces the projection. On the complement of K_p that operator
//     is symmetric plus the rank-one term, which gives, for v_k orthonormal to K_p and to each other,
//       eta_{k+1} v_{k+1} = H v_k - beta (q.v_k) a_k - beta (z.v_k) b_k - eta_k v_{k-1} - h_k v_k,
//       a_k = q_p + sum_{i<k} (z.v_i) v_i,   b_k = q_{p+1} - sum_{i<k} (q.v_i) v_i,   q = q_{p+1},
//     v_1 = s_j less its part in K_p (taken out as the q_n appear), normalised.
// The span relations hold to rounding whatever orthogonality is lost; the Gram matrices
// W^T H W and W^T S W are summed at the end from the stored W, H W, S W, so lost orthogonality costs no
// accuracy either, as long as W stays well conditioned. It is watched through q_1 = e_j: |(w_n)_j| is
// the overlap of w_n with q_1. An atom goes to the general kernel (its index into `redo`) when that
// exceeds 1e-3, when a vector keeps less than 1e-6 of its norm, when s_j keeps less than 1e-7 (unless all
// four columns keep less than 1e-12: then s_j is in K_p, as for S = I, and the first chain simply
// continues), when an inner CG failed, or when its cluster is small against the subspace (m < 6 nu:
// there the recurrences lose orthogonality within 30 to 40 steps).
//
// What it costs, per atom of four columns at m = 632, nu = 30: the general kernel streams U, S U and the low half of
// U from DRAM at every step (23 MB an atom); here a step touches a few vectors and the basis is read back once for
// the Gram matrices. Measured on 8,192 atoms of the sigma = 0.1 A diamond system in the mixed form on BF16 values:
// 62.3 -> 30.6 ms; 2,501 atoms at sigma = 0.15 A, R = 7 A, nu = 40, FP32 values: 69.4 -> 38.8 ms; 2,999 atoms of the
// fcc system in FP64: 46.8 -> 37.2 ms. The FP64 form is bound by the FP64 pipe (the products are 3/4 of it), the
// FP32 form by the products' FP32 pipe and shared-memory gathers (a third of the time), then by the latency of the
// reductions between steps.
//
// One thread owns a row of all four columns. In the FP32 form every recurrence runs in FP32 pairs (hi + lo), scalars,
// z and dot products included, since rounding at FP32 level would be amplified by the lost orthogonality and at the
// seam; S w and the Gram matrices take FP32 from the hi parts, as the general kernel does, and H_r comes from the
// recurrence coefficients. Sums across threads are FP64.
#include <cuda_bf16.h>
#include <cuda_pipeline.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "atoms.cuh"
#include "gram_stage.cuh"
#include "mka_internal.h"

namespace mka {
namespace {

// ---- one entry of a work vector: FP64, or an FP32 pair ------------------------------------------
struct Pair {
  float h, l;
};
template <typename T>
struct Entry {
  using type = double;
};
template <>
struct Entry<float> {
  using type = Pair;
};

__device__ __forceinline__ void set_zero(double& a) { a = 0.0; }
__device__ __forceinline__ void set_zero(float& a) { a = 0.0f; }
__device__ __forceinline__ void set_zero(Pair& a) { a.h = a.l = 0.0f; }
__device__ __forceinline__ double to_double(double a) { return a; }
__device__ __forceinline__ double to_double(float a) { return (double)a; }
__device__ __forceinline__ double to_double(Pair a) { return (double)a.h + (double)a.l; }
__device__ __forceinline__ void from_double(double x, double& a) { a = x; }
__device__ __forceinline__ void from_double(double x, Pair& a) {
  a.h = (float)x;
  a.l = (float)(x - (double)a.h);
}
__device__ __forceinline__ double head(double a) { return a; }
__device__ __forceinline__ float head(Pair a) { return a.h; }

// hi + lo with |lo| <= ulp(hi) / 2, for |e| <= |p|
__device__ __forceinline__ Pair renorm(float p, float e) {
  Pair r;
  r.h = __fadd_rn(p, e);
  r.l = __fsub_rn(e, __fsub_rn(r.h, p));
  return r;
}
// product of two pairs, unnormalised
__device__ __forceinline__ Pair pair_mul(Pair a, Pair x) {
  Pair r;
  r.h = __fmul_rn(a.h, x.h);
  r.l = fmaf(a.h, x.h, -r.h);
  r.l = fmaf(a.h, x.l, r.l);
  r.l = fmaf(a.l, x.h, r.l);
  return r;
}
// s + (p, e) with the rounding of s + p kept
__device__ __forceinline__ Pair pair_add(Pair s, float p, float e) {
  const float t = __fadd_rn(s.h, p), bb = __fsub_rn(t, s.h);
  const float err = __fadd_rn(__fsub_rn(s.h, __fsub_rn(t, bb)), __fsub_rn(p, bb));
  return Pair{t, __fadd_rn(s.l, __fadd_rn(err, e))};
}
// y <- y - a x
__device__ __forceinline__ void sub_mul(double& y, double a, double x) { y = fma(-a, x, y); }
__device__ __forceinline__ void sub_mul(Pair& y, Pair a, Pair x) {
  const Pair p = pair_mul(a, x);
  const Pair s = pair_add(y, -p.h, -p.l);
  y = renorm(s.h, s.l);
}
__device__ __forceinline__ double scaled(double y, double a) { return y * a; }
__device__ __forceinline__ Pair scaled(Pair y, Pair a) {
  const Pair p = pair_mul(y, a);
  return renorm(p.h, p.l);
}
// s <- s + x y
__device__ __forceinline__ void dot_acc(double& s, double x, double y) { s = fma(x, y, s); }
__device__ __forceinline__ void dot_acc(Pair& s, Pair x, Pair y) {
  const Pair p = pair_mul(x, y);
  s = pair_add(s, p.h, p.l);
}
// the same for a plain FP32 x
__device__ __forceinline__ void dot_acc(Pair& s, float x, Pair y) {
  const float p = __fmul_rn(x, y.h);
  s = pair_add(s, p, fmaf(x, y.l, fmaf(x, y.h, -p)));
}
// s <- s + x y for plain x, y (FP32: the product exact and the sum compensated into a pair, or plain)
__device__ __forceinline__ void mac(double& s, double x, double y) { s = fma(x, y, s); }
__device__ __forceinline__ void mac(float& s, float x, float y) { s = fmaf(x, y, s); }
__device__ __forceinline__ void mac(Pair& s, float x, float y) {
  const float p = __fmul_rn(x, y);
  s = pair_add(s, p, fmaf(x, y, -p));
}
__device__ __forceinline__ double shfl_x(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ float shfl_x(float v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ Pair shfl_x(Pair v, int o) { return Pair{shfl_x(v.h, o), shfl_x(v.l, o)}; }
__device__ __forceinline__ double add(double a, double b) { return a + b; }
__device__ __forceinline__ float add(float a, float b) { return a + b; }
__device__ __forceinline__ Pair add(Pair a, Pair b) { return pair_add(a, b.h, b.l); }

// Four columns' sums over the warp, halving the columns a lane carries in the first two steps (the sums of
// the butterfly over lanes 16, 8, 4, 2, 1, with 6 instead of 20 additions): lane l ends with the sum of
// column 2 (l >> 4) + (l >> 3 & 1).
template <typename N>
__device__ __forceinline__ N warp_sum_cols(N v[4]) {
  const int lane = threadIdx.x & 31;
  const bool b16 = lane & 16, b8 = lane & 8;
  N a0 = add(b16 ? v[2] : v[0], shfl_x(b16 ? v[0] : v[2], 16));
  N a1 = add(b16 ? v[3] : v[1], shfl_x(b16 ? v[1] : v[3], 16));
  N r = add(b8 ? a1 : a0, shfl_x(b8 ? a0 : a1, 8));
  r = add(r, shfl_x(r, 4));
  r = add(r, shfl_x(r, 2));
  r = add(r, shfl_x(r, 1));
  return r;
}

// The warps' sums of four columns (value k of K) into red[warp][k][column], FP64.
template <typename N>
__device__ __forceinline__ void warp_partial(N v[4], double* red, int k, int K) {
  const N r = warp_sum_cols(v);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if ((lane & 7) == 0) red[(wid * K + k) * 4 + (lane >> 3)] = to_double(r);
}

// Work vectors [m_cap][4] of entries: hi (and, for pairs, lo) arrays.
template <typename T>
struct Vec {
  T* h;
  T* l;   // FP32 pairs only
};
__device__ __forceinline__ void ldv(const Vec<double>& v, int r, double x[4]) { ld4(v.h + 4 * r, x); }
__device__ __forceinline__ void ldv(const Vec<float>& v, int r, Pair x[4]) {
  float h[4], l[4];
  ld4(v.h + 4 * r, h);
  ld4(v.l + 4 * r, l);
#pragma unroll
  for (int c = 0; c < 4; ++c) x[c] = Pair{h[c], l[c]};
}
__device__ __forceinline__ void stv(const Vec<double>& v, int r, const double x[4]) { st4(v.h + 4 * r, x[0], x[1], x[2], x[3]); }
__device__ __forceinline__ void stv(const Vec<float>& v, int r, const Pair x[4]) {
  st4(v.h + 4 * r, x[0].h, x[1].h, x[2].h, x[3].h);
  st4(v.l + 4 * r, x[0].l, x[1].l, x[2].l, x[3].l);
}

// One row (4 entries) of a stored block, undecoded: loads of the next block are in flight while the current one's
// products run.
template <typename TV>
struct RawRow;
template <>
struct RawRow<__nv_bfloat16> {
  uint2 a;
  __device__ __forceinline__ void load(const __nv_bfloat16* v, int64_t blk, int i) {
    a = __ldg(reinterpret_cast<const uint2*>(v + blk * 16 + i * 4));
  }
  template <typename T>
  __device__ __forceinline__ void get(T out[4]) const {
    out[0] = (T)__uint_as_float(a.x << 16); out[1] = (T)__uint_as_float(a.x & 0xFFFF0000u);
    out[2] = (T)__uint_as_float(a.y << 16); out[3] = (T)__uint_as_float(a.y & 0xFFFF0000u);
  }
};
template <>
struct RawRow<float> {
  float4 a;
  __device__ __forceinline__ void load(const float* v, int64_t blk, int i) {
    a = __ldg(reinterpret_cast<const float4*>(v + blk * 16 + i * 4));
  }
  template <typename T>
  __device__ __forceinline__ void get(T out[4]) const {
    out[0] = (T)a.x; out[1] = (T)a.y; out[2] = (T)a.z; out[3] = (T)a.w;
  }
};
template <>
struct RawRow<double> {
  double2 a, b;
  __device__ __forceinline__ void load(const double* v, int64_t blk, int i) {
    const double2* p = reinterpret_cast<const double2*>(v + blk * 16 + i * 4);
    a = __ldg(p);
    b = __ldg(p + 1);
  }
  template <typename T>
  __device__ __forceinline__ void get(T out[4]) const {
    out[0] = (T)a.x; out[1] = (T)a.y; out[2] = (T)b.x; out[3] = (T)b.y;
  }
};

// X is swizzled: row k of cluster atom a is its 4-entry chunk 4 a + (k ^ swz(a)), so that the rows k of different
// atoms, which the lanes of a warp gather together, spread over the banks (without it a quarter warp's two
// atoms met in the same banks half the time in FP32, always in FP64: 46 % of the shared-load wavefronts
// were conflicts).
template <typename T>
__device__ __forceinline__ int swz(int a) { return sizeof(T) == 4 ? a >> 1 & 3 : a & 3; }
template <typename T>
__device__ __forceinline__ int xrow(int r) { return r ^ swz<T>(r >> 2); }
// A local block: its column atom's offset in X with the swizzle (low 16 bits; row k of it at `offset ^ 4 k`), and
// its offset within the global row.
template <typename T>
__device__ __forceinline__ uint32_t block_entry(int lc, int off) {
  return (uint32_t)(16 * lc + 4 * swz<T>(lc)) | (uint32_t)off << 16;
}

// Row `i` of a cluster atom with blocks ent[e0..e1): h = (H x)_row and sw = (S x)_row for the four columns. FP64.
template <typename TV>
__device__ __forceinline__ void row_hs(const TV* __restrict__ valH, const TV* __restrict__ valS, int rb, int e0, int e1,
                                       const uint32_t* ent, int i, const Vec<double>& x, unsigned long long, double h[4],
                                       double sw[4]) {
#pragma unroll
  for (int c = 0; c < 4; ++c) h[c] = sw[c] = 0.0;
#pragma unroll 2
  for (int e = e0; e < e1; ++e) {
    const uint32_t en = ent[e];
    double vh[4], vs[4];
    RowLoad<TV, double>::load(valH, rb + (int)(en >> 16), i, vh);
    RowLoad<TV, double>::load(valS, rb + (int)(en >> 16), i, vs);
    const uint32_t xo = en & 0xFFFFu;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      double xk[4];
      ld4(x.h + (xo ^ 4 * k), xk);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        h[c] = fma(vh[k], xk[c], h[c]);
        sw[c] = fma(vs[k], xk[c], sw[c]);
      }
    }
  }
}

// Two FP32 lanes in one instruction (IEEE-rounded each): the FP32 pipe's rate is the same, the issue slots
// halve, which leaves room for the loads.
typedef unsigned long long f2;
__device__ __forceinline__ f2 pack2(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// ap = (S x)_row for the inner CG, in the arithmetic type, entry by entry in order.
template <typename TV>
__device__ __forceinline__ void row_s(const TV* __restrict__ valS, int rb, int e0, int e1, const uint32_t* ent, int i,
                                      const double* x, double ap[4]) {
#pragma unroll
  for (int c = 0; c < 4; ++c) ap[c] = 0.0;
#pragma unroll 4
  for (int e = e0; e < e1; ++e) {
    const uint32_t en = ent[e];
    double v[4];
    RowLoad<TV, double>::load(valS, rb + (int)(en >> 16), i, v);
    const uint32_t xo = en & 0xFFFFu;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      double xk[4];
      ld4(x + (xo ^ 4 * k), xk);
#pragma unroll
      for (int c = 0; c < 4; ++c) ap[c] = fma(v[k], xk[c], ap[c]);
    }
  }
}
template <typename TV>
__device__ __forceinline__ void row_s(const TV* __restrict__ valS, int rb, int e0, int e1, const uint32_t* ent, int i,
                                      const float* x, float ap[4]) {
  f2 a01 = 0, a23 = 0;
#pragma unroll 4
  for (int e = e0; e < e1; ++e) {
    const uint32_t en = ent[e];
    float v[4];
    RowLoad<TV, float>::load(valS, rb + (int)(en >> 16), i, v);
    const uint32_t xo = en & 0xFFFFu;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const ulonglong2 xk = *reinterpret_cast<const ulonglong2*>(x + (xo ^ 4 * k));
      const f2 v2 = pack2(v[k], v[k]);
      a01 = fma2(v2, xk.x, a01);
      a23 = fma2(v2, xk.y, a23);
    }
  }
  unpack2(a01, ap[0], ap[1]);
  unpack2(a23, ap[2], ap[3]);
}

// r = (e_j - S x)_row for an FP32 x with error-free products and compensated sums (column c's e_j is row c after
// row 0 of atom a: dj = row - 4 t0).
template <typename TV>
__device__ __forceinline__ void row_resid(const TV* __restrict__ valS, int rb, int e0, int e1, const uint32_t* ent,
                                          int i, const float* x, int dj, float r[4]) {
  Pair s[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) set_zero(s[c]);
  for (int e = e0; e < e1; ++e) {
    const uint32_t en = ent[e];
    float v[4];
    RowLoad<TV, float>::load(valS, rb + (int)(en >> 16), i, v);
    const uint32_t xo = en & 0xFFFFu;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float xk[4];
      ld4(x + (xo ^ 4 * k), xk);
#pragma unroll
      for (int c = 0; c < 4; ++c) mac(s[c], v[k], xk[c]);
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) r[c] = __fsub_rn(__fsub_rn(dj == c ? 1.0f : 0.0f, s[c].h), s[c].l);
}

// FP32 pairs: H x with error-free products and compensated sums on the hi part, the lo part's products
// rounded; S x in FP32 from the hi part. The exact product v x enters the error term as one fma:
// (p - bb) + (v x - p) = v x - bb, nine operations an entry, two columns to an instruction. The rounded product
// p is an fma with `zero`, a 0 the assembler cannot see: a packed multiplication and the addition after it are
// contracted into one fma despite their .rn (measured: row error 7e-8 instead of 1e-13), which is not the sum the
// error terms belong to.
template <typename TV>
__device__ __forceinline__ void row_hs(const TV* __restrict__ valH, const TV* __restrict__ valS, int rb, int e0, int e1,
                                       const uint32_t* ent, int i, const Vec<float>& x, f2 zero, Pair h[4], float sw[4]) {
  f2 hh[2] = {0, 0}, hl[2] = {0, 0}, ss[2] = {0, 0};
  uint32_t en = 0;
  RawRow<TV> rh, rs;
  if (e0 < e1) {
    en = ent[e0];
    rh.load(valH, rb + (int)(en >> 16), i);
    rs.load(valS, rb + (int)(en >> 16), i);
  }
  for (int e = e0; e < e1; ++e) {
    float vh[4], vs[4];
    rh.get(vh);
    rs.get(vs);
    const uint32_t xo = en & 0xFFFFu;
    if (e + 1 < e1) {
      en = ent[e + 1];
      rh.load(valH, rb + (int)(en >> 16), i);
      rs.load(valS, rb + (int)(en >> 16), i);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const ulonglong2 xh = *reinterpret_cast<const ulonglong2*>(x.h + (xo ^ 4 * k));
      const ulonglong2 xl = *reinterpret_cast<const ulonglong2*>(x.l + (xo ^ 4 * k));
      const f2 v2 = pack2(vh[k], vh[k]), s2 = pack2(vs[k], vs[k]);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const f2 xc = c ? xh.y : xh.x, lc = c ? xl.y : xl.x;
        const f2 p = fma2(v2, xc, zero);
        const f2 s = add2(hh[c], p);
        const f2 nb = sub2(hh[c], s);            // -bb
        const f2 d = sub2(hh[c], add2(s, nb));
        const f2 f = fma2(v2, xc, nb);
        hh[c] = s;
        hl[c] = fma2(v2, lc, add2(hl[c], add2(d, f)));
        ss[c] = fma2(s2, xc, ss[c]);
      }
    }
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    float p0, p1, l0, l1;
    unpack2(hh[c], p0, p1);
    unpack2(hl[c], l0, l1);
    h[2 * c] = renorm(p0, l0);
    h[2 * c + 1] = renorm(p1, l1);
    unpack2(ss[c], sw[2 * c], sw[2 * c + 1]);
  }
}

// Two values from a T array as a vector load.
__device__ __forceinline__ void ld2(const float* p, float v[2]) {
  const float2 a = *reinterpret_cast<const float2*>(p);
  v[0] = a.x;
  v[1] = a.y;
}
__device__ __forceinline__ void ld2(const double* p, double v[2]) {
  const double2 a = *reinterpret_cast<const double2*>(p);
  v[0] = a.x;
  v[1] = a.y;
}

// Gram matrices of the basis vectors nn in [n0, n1) against mm <= nn: H_r[mm][nn] = w_mm.(H w_nn) and
// S_r[nn][mm] = w_mm.(S w_nn) into the reduced-problem buffer (upper triangle of H_r, lower of S_r: what the
// reduced kernel reads), S_r also into Gs (packed lower triangle per column, shared) when given.
//
// gram: straight from the slot. FP64: both matrices (bound by the FP64 pipe). Pairs: H_r alone with compensated
// sums, taken when too much orthogonality was lost. A warp takes 2 x 2 (4 x 2) vectors at a time, its
// lanes 16 rows x 2 column pairs, and one halving tree over the lanes ends a tile's sums.
template <typename T>
__device__ __noinline__ void gram(const T* W, const T* HW, const T* SW, int m, int m4, int n0, int n1, int nu,
                                  double* red, int64_t col0, double* Gs, int gs_stride) {
  constexpr bool kBoth = sizeof(T) == 8;
  constexpr int TI = kBoth ? 2 : 4, NM = kBoth ? 2 : 1, NV = TI * 2 * NM * 2;
  static_assert(NV == 16, "the halving tree has four steps");
  using N = typename Entry<T>::type;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  const int cp = lane & 1, r0 = lane >> 1;
  const size_t vs = (size_t)m4;
  int tile = 0;
  for (int nn = n0; nn < n1; nn += 2) {
    const int nb = min(nn + 2, n1) - 1;
    for (int mm = 0; mm <= nb; mm += TI, ++tile) {
      if (tile % nwarp != wid) continue;
      N acc[NV];
#pragma unroll
      for (int k = 0; k < NV; ++k) set_zero(acc[k]);
      const T* w0 = W + 2 * cp;
      const T* h0 = HW + (size_t)nn * vs + 2 * cp;
      const T* s0 = SW + (size_t)nn * vs + 2 * cp;
      const size_t dn = (size_t)(nb - nn) * vs;
      for (int r = r0; r < m; r += 16) {
        T w[TI][2], hv[2][2], sv[2][2];
#pragma unroll
        for (int i = 0; i < TI; ++i) ld2(w0 + (size_t)min(mm + i, nb) * vs + 4 * r, w[i]);
        ld2(h0 + 4 * r, hv[0]);
        ld2(h0 + dn + 4 * r, hv[1]);
        if (kBoth) {
          ld2(s0 + 4 * r, sv[0]);
          ld2(s0 + dn + 4 * r, sv[1]);
        }
#pragma unroll
        for (int i = 0; i < TI; ++i)
#pragma unroll
          for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
              const int k = (i * 2 + j) * NM * 2 + c;
              mac(acc[k], w[i][c], hv[j][c]);
              if constexpr (kBoth) mac(acc[k + 2], w[i][c], sv[j][c]);
            }
      }
      int id = 0;
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const int o = 16 >> s, half = NV >> (s + 1);
        const bool up = lane & o;
#pragma unroll
        for (int k = 0; k < half; ++k) {
          const N send = up ? acc[k] : acc[k + half];
          acc[k] = add(up ? acc[k + half] : acc[k], shfl_x(send, o));
        }
        id += up ? half : 0;
      }
      const int c = 2 * cp + (id & 1), ij = id / (2 * NM), a = mm + ij / 2, b = nn + ij % 2;
      if (a > b || b > nb) continue;
      double* R = red + (size_t)(col0 >> 5) * red_block_doubles(nu) * 32 + ((col0 + c) & 31);
      const double v = to_double(acc[0]);
      if (kBoth && (id & 2)) {
        R[(size_t)(nu * nu + b * nu + a) * 32] = v;
        if (Gs) Gs[c * gs_stride + b * (b + 1) / 2 + a] = v;
      } else {
        R[(size_t)(a * nu + b) * 32] = v;
      }
    }
  }
}

// gram_s: S_r of the FP32 form. Read vector by vector from the slot it was bound by L2 (3.8 MB an atom at nu = 30);
// here chunks of rows of every vector pass through shared memory once (double buffered, cp.async), and a warp
// holds two vectors nn against all mm: lane (t, c) has mm = t, t + 8, ... of column c. Sums of eight rows are FP32,
// their sum a pair (FP32 sums of whole columns were the largest error of the levels' weights:
// 4.6e-7 against 1.5e-7).
template <int NA>
__device__ __noinline__ void gram_s(const float* W, const float* SW, int m, int m4, int n0, int n1, int nu, double* red,
                                    int64_t col0, double* Gs, int gs_stride, float* stage, int stage_floats) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  const int t = lane >> 2, c = lane & 3;
  const int nvec = chunk_vectors(n0, n1), rc = chunk_rows(nvec, stage_floats);
  const int vs = chunk_stride(rc), nchunk = (m + rc - 1) / rc, npair = (n1 - n0 + 1) / 2;
  auto fetch = [&](int k) {
    float* dst = stage + (k & 1) * nvec * vs;
    const int r0 = k * rc, rows = min(rc, m - r0);
    for (int i = threadIdx.x; i < nvec * rows; i += blockDim.x) {
      const int v = i / rows, r = i - v * rows;
      const float* src = (v < n1 ? W + (size_t)v * m4 : SW + (size_t)(v - n1 + n0) * m4) + 4 * (r0 + r);
      __pipeline_memcpy_async(dst + v * vs + 4 * r, src, 16);
    }
    __pipeline_commit();
  };
  for (int j0 = 0; j0 < npair; j0 += nwarp) {
    const int nn = n0 + 2 * (j0 + wid), nb = min(nn + 1, n1 - 1);
    const int cnt = nn < n1 ? nb / 8 + 1 : 0;
    int at[NA];
#pragma unroll
    for (int i = 0; i < NA; ++i) at[i] = lane_vector(t, i, nb) * vs;
    Pair tot[2][NA];
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      set_zero(tot[0][i]);
      set_zero(tot[1][i]);
    }
    fetch(0);
    for (int k = 0; k < nchunk; ++k) {
      if (k + 1 < nchunk) {
        fetch(k + 1);
        __pipeline_wait_prior(1);
      } else {
        __pipeline_wait_prior(0);
      }
      __syncthreads();
      if (cnt) {
        const float* w = stage + (k & 1) * nvec * vs + c;
        const float* s0 = w + (n1 + nn - n0) * vs;
        const float* s1 = w + (n1 + nb - n0) * vs;
        const int rows = min(rc, m - k * rc);
        for (int rb = 0; rb < rows; rb += 8) {
          float p0[NA], p1[NA];
#pragma unroll
          for (int i = 0; i < NA; ++i) p0[i] = p1[i] = 0.0f;
#pragma unroll 4
          for (int r = rb; r < min(rows, rb + 8); ++r) {
            const float a = s0[4 * r], b = s1[4 * r];
#pragma unroll
            for (int i = 0; i < NA; ++i)
              if (i < cnt) {
                const float x = w[at[i] + 4 * r];
                p0[i] = fmaf(x, a, p0[i]);
                p1[i] = fmaf(x, b, p1[i]);
              }
          }
#pragma unroll
          for (int i = 0; i < NA; ++i)
            if (i < cnt) {
              tot[0][i] = pair_add(tot[0][i], p0[i], 0.0f);
              tot[1][i] = pair_add(tot[1][i], p1[i], 0.0f);
            }
        }
      }
      __syncthreads();
    }
    double* R = red + (size_t)(col0 >> 5) * red_block_doubles(nu) * 32 + ((col0 + c) & 31);
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int i = 0; i < NA; ++i) {
        const int a = t + 8 * i, b = nn + j;
        if (b >= n1 || a > b) continue;
        const double v = to_double(tot[j][i]);
        R[(size_t)(nu * nu + b * nu + a) * 32] = v;
        if (Gs) Gs[c * gs_stride + b * (b + 1) / 2 + a] = v;
      }
  }
}

// z = S (Q g) of the pair form into ZV, by way of X (free at the seam; gv lies within it) and `spare`. Out of line, as
// gram and gram_s: once an atom, and the kernel is sensitive to its own code size.
template <typename TV>
__device__ __noinline__ void seam_z(const TV* __restrict__ valS, f2 zero, const float* W, int p, int m, int m4, const Pair* gv,
                                    const Vec<float>& X, float* spare, const Vec<float>& ZV, const int* rbase, const int* lrow,
                                    const uint32_t* ent) {
  const Vec<float> QG{ZV.h, spare};
  for (int r = threadIdx.x; r < m; r += blockDim.x) {
    Pair y[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) set_zero(y[c]);
    for (int k = 0; k < p; ++k) {
      float q[4];
      ld4(W + (size_t)k * m4 + 4 * r, q);
#pragma unroll
      for (int c = 0; c < 4; ++c) dot_acc(y[c], q[c], gv[c * p + k]);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) y[c] = renorm(y[c].h, y[c].l);
    stv(QG, r, y);
  }
  __syncthreads();                     // gv has been read
  for (int r = threadIdx.x; r < m; r += blockDim.x) {
    Pair y[4];
    ldv(QG, r, y);
    stv(X, xrow<float>(r), y);
  }
  __syncthreads();
  for (int r = threadIdx.x; r < m; r += blockDim.x) {
    Pair z[4];
    float sw[4];
    row_hs<TV>(valS, valS, rbase[r >> 2], lrow[r >> 2], lrow[(r >> 2) + 1], ent, r & 3, X, zero, z, sw);
    stv(ZV, r, z);
  }
}

struct ChainState {
  double rr[4], alpha[4], cg_stop[4];
  int it[4], cg_active[4], status[4], fell[4];
  double be[4], ga[4], s0[4];    // beta_{n-1}, alpha_n; ||s_j||^2, then beta_p
  // bad: the atom goes to the general kernel, found by the threads that own the scalars between two barriers, so that
  // it may be read after the second. over: the same, found by the rows' threads as they write a vector; read only
  // behind the barrier that ends a step.
  int t0, flag, bad, over, drop, careful;
};

// The second chain's scalars of column c from beta_p, q.v_k and z.v_k.
template <typename N>
__device__ __forceinline__ void chain_scalars(double beta, double qv, double zv, N* sc, int c) {
  from_double(beta * qv, sc[8 + c]);
  from_double(beta * zv, sc[12 + c]);
  from_double(qv, sc[16 + c]);
  from_double(-zv, sc[20 + c]);
}

constexpr double kOverlapMax = 1e-3;           // |w_n . e_j| beyond which an atom goes to the general kernel

// Beyond this the FP32 form takes H_r from a Gram matrix too, instead of from the recurrence coefficients (whose
// error is about ||H|| times the lost orthogonality, up to a few hundred times the overlap with q_1).
constexpr double kOverlapExact = 1e-10;

__device__ __forceinline__ void check_overlap(ChainState& st, double x) {
  if (!(fabs(x) <= kOverlapMax)) st.over = 1;
  if (!(fabs(x) <= kOverlapExact)) st.careful = 1;
}

// Resident CTAs per SM the register budget is cut for.
template <typename T, int NT>
constexpr int chains_min_blocks() { return sizeof(T) == 4 ? 1024 / NT : 768 / NT > 0 ? 768 / NT : 1; }

// Streamed work vectors of a slot.
__host__ __device__ constexpr int work_vectors(size_t elem) { return elem == 4 ? 11 : 10; }

template <typename TV, typename T, int NT>
__global__ void __launch_bounds__(NT, chains_min_blocks<T, NT>()) chains_kernel(const Args<TV> A) {
  using N = typename Entry<T>::type;
  constexpr bool kPair = sizeof(T) == 4;
  extern __shared__ __align__(64) unsigned char smem_raw[];
  __shared__ ChainState st;
  __shared__ double red[kMaxWarps * 12];
  __shared__ T scal[8];
  __shared__ N sc[24];                          // recurrence scalars as the columns' threads use them
  __shared__ int64_t cur_atom;
  __shared__ int cnt;

  const int nu = A.nu, m_cap = A.mcap;
  int* cl = reinterpret_cast<int*>(smem_raw);
  int* lrow = cl + A.clcap;
  int* rbase = lrow + A.mcap / 4 + 1;
  uint32_t* ent = reinterpret_cast<uint32_t*>(rbase + A.mcap / 4);
  size_t off = (size_t)(A.clcap + 2 * (A.mcap / 4) + 1 + A.lnnz_cap) * sizeof(int);
  off = (off + 63) & ~(size_t)63;
  const int m4 = m_cap * 4;
  T* X0 = reinterpret_cast<T*>(smem_raw + off);
  // at the seam, over X and Y: Q^T S Q packed, per column, and its inverse's last column
  const int gst = A.p * (A.p + 1) / 2;
  double* Gs = reinterpret_cast<double*>(X0);
  N* gv = reinterpret_cast<N*>(Gs + 4 * gst);

  // global slot: W, H W, S W [nu][m_cap][4]; streamed work vectors [m_cap][4]; s_j in FP64
  char* slot = A.scratch + (size_t)blockIdx.x * A.slot_bytes;
  T* W = reinterpret_cast<T*>(slot);
  T* HW = W + (size_t)nu * m4;
  T* SW = HW + (size_t)nu * m4;
  T* B = SW + (size_t)nu * m4;
  double* SJd = reinterpret_cast<double*>(slot + align_up(sizeof(T) * ((size_t)3 * nu + work_vectors(sizeof(T))) * m4, 256));
  double* tri = SJd + m4;                       // alpha, beta, q.v, z.v of every step, [4][nu][4]
  // shared vectors: X, gathered by the products (CG: p), and the work vector Y (CG: S p). Pairs: X's low half
  // holds s_j during CG; Y's low half (CG: r) is read row by row only and lives in the slot, which lets
  // four CTAs share an SM at the usual clusters
  const Vec<T> X{X0, kPair ? X0 + m4 : nullptr};
  const Vec<T> Y{X0 + (kPair ? 2 : 1) * m4, B + 8 * m4};
  const Vec<T> PV{B, B + m4};                   // q_{n-1} (pairs: only its low half; hi is W[n-1])
  const Vec<T> SV{B + 2 * m4, B + 3 * m4};      // s_j less its part in the first chain; then a_k
  const Vec<T> BV{B + 4 * m4, B + 5 * m4};      // b_k
  const Vec<T> QV{B + 6 * m4, B + 9 * m4};      // q_{p+1}
  const Vec<T> ZV{B + 7 * m4, B + 10 * m4};     // z
  T* SJ = kPair ? X.l : B + 8 * m4;             // CG: s_j
  auto sjrow = [](int r) { return kPair ? xrow<T>(r) : r; };
  T* R = kPair ? Y.l : B;                       // CG: the residual
  const int tid = threadIdx.x;

  for (;;) {
    if (tid == 0) cur_atom = atomicAdd(A.work_counter, 1);
    __syncthreads();
    if (cur_atom >= A.n_sel) break;
    const int64_t widx = A.order ? (int64_t)A.order[cur_atom] : cur_atom;
    const int64_t atom = A.sel[widx];

    // ---- 1. cluster and its local block pattern ------------------------------------------------
    const int ncl = gather_cluster(A, atom, cl, &cnt);
    const int m = 4 * ncl;
    bool general = ncl > A.clcap || m > m_cap;  // the general kernel reports clusters beyond the cap
    if (!A.cg_only) general = general || m < 6 * nu || !chains_fit(m, A.p, nu, kPair);
    if (!general) {
      sort_cluster(cl, ncl);
      for (int t = tid; t < ncl; t += NT) {
        const int b = cl[t];
        int c = 0;
        for (int k = A.row_ptr[b]; k < A.row_ptr[b + 1]; ++k) c += find_local(cl, ncl, A.col[k]) >= 0;
        lrow[t + 1] = c;
      }
      __syncthreads();
      if (tid == 0) {
        lrow[0] = 0;
        for (int t = 0; t < ncl; ++t) lrow[t + 1] += lrow[t];
        st.t0 = find_local(cl, ncl, (int)atom);
        st.flag = lrow[ncl] <= A.lnnz_cap;
        st.bad = 0;
        st.over = 0;
        st.drop = 0;
        st.careful = 0;
      }
      __syncthreads();
      general = !st.flag;
    }
    if (general) {
      if (tid == 0) {
        if (A.cg_only) {
          for (int c = 0; c < 4; ++c) {
            A.status[4 * widx + c] = ST_TOOLARGE;
            A.cg_iters[4 * widx + c] = 0;
          }
        } else {
          A.redo[atomicAdd(A.redo_count, 1)] = (int32_t)widx;
        }
      }
      __syncthreads();
      continue;
    }
    for (int t = tid; t < ncl; t += NT) {
      const int b = cl[t];
      const int k0 = A.row_ptr[b];
      int e = lrow[t];
      rbase[t] = k0;
      for (int k = k0; k < A.row_ptr[b + 1]; ++k) {
        const int lc = find_local(cl, ncl, A.col[k]);
        if (lc >= 0) {
          ent[e++] = block_entry<T>(lc, k - k0);   // rows hold at most 255 blocks (checked at setup)
        }
      }
    }
    const int t0 = st.t0, j0 = 4 * t0;
    if (A.keep_cl)
      for (int t = tid; t < A.keep_cap; t += NT) A.keep_cl[widx * A.keep_cap + t] = t < ncl ? cl[t] : -1;

    // ---- 2. inner CG: S s = e_j (the arithmetic of the general kernel, sum for sum) ---------------
    T* P = X.h;
    T* AP = Y.h;
    if (tid < 4) {
      st.rr[tid] = 1.0;
      st.it[tid] = 0;
      st.status[tid] = ST_OK;
      st.fell[tid] = 0;
    }
    if (A.x0 || A.prev_s) {
      for (int r = tid; r < m; r += NT) {
        st4(SJ + 4 * sjrow(r), 0, 0, 0, 0);
        st4(P + 4 * xrow<T>(r), 0, 0, 0, 0);
      }
      __syncthreads();
      if (A.prev_s) {
        const int32_t* pc = A.prev_cl + widx * A.prev_cap;
        int np = 0;
        while (np < A.prev_cap && pc[np] >= 0) ++np;
        for (int t = tid; t < ncl; t += NT) {
          const int f = find_local(pc, np, cl[t]);
          if (f < 0) continue;
          for (int c = 0; c < 4; ++c)
            for (int o = 0; o < 4; ++o) {
              const T v = (T)A.prev_s[(4 * widx + c) * (4 * (int64_t)A.prev_cap) + 4 * f + o];
              SJ[4 * sjrow(4 * t + o) + c] = v;
              P[4 * xrow<T>(4 * t + o) + c] = v;
            }
        }
      } else {
        for (int i = tid; i < 4 * 68; i += NT) {
          const int c = i / 68, rem = i % 68, k = rem >> 2, o = rem & 3;
          const int pa = A.patch[widx * 17 + k];
          const int lk = pa >= 0 ? find_local(cl, ncl, pa) : -1;
          if (lk < 0) continue;
          const T v = (T)A.x0[(4 * widx + c) * 68 + rem];
          SJ[4 * sjrow(4 * lk + o) + c] = v;
          P[4 * xrow<T>(4 * lk + o) + c] = v;
        }
      }
      __syncthreads();
      T part[4] = {0, 0, 0, 0};
      for (int r = tid; r < m; r += NT) {
        T ap[4];
        row_s<TV>(A.valS, rbase[r >> 2], lrow[r >> 2], lrow[(r >> 2) + 1], ent, r & 3, P, ap);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          ap[c] = ((r == j0 + c) ? (T)1 : (T)0) - ap[c];
          part[c] += ap[c] * ap[c];
        }
        st4(R + 4 * r, ap[0], ap[1], ap[2], ap[3]);
      }
      double acc[4] = {(double)part[0], (double)part[1], (double)part[2], (double)part[3]};
      warp_partial(acc, red, 0, 1);
      __syncthreads();
      if (tid < 4) {
        double s = 0;
        for (int k = 0; k < NT / 32; ++k) s += red[k * 4 + tid];
        if (!(s < 1.0)) st.fell[tid] = 1;   // no better than x0 = 0: start from zero
        else st.rr[tid] = s;
      }
      __syncthreads();
      for (int r = tid; r < m; r += NT)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (st.fell[c]) {
            SJ[4 * sjrow(r) + c] = 0;
            R[4 * r + c] = (r == j0 + c) ? (T)1 : (T)0;
          }
          P[4 * xrow<T>(r) + c] = R[4 * r + c];
        }
    } else {
      for (int r = tid; r < m; r += NT) {
        const T e0 = r == j0 ? (T)1 : (T)0, e1 = r == j0 + 1 ? (T)1 : (T)0;
        const T e2 = r == j0 + 2 ? (T)1 : (T)0, e3 = r == j0 + 3 ? (T)1 : (T)0;
        st4(SJ + 4 * sjrow(r), 0, 0, 0, 0);
        st4(P + 4 * xrow<T>(r), e0, e1, e2, e3);
        st4(R + 4 * r, e0, e1, e2, e3);
      }
    }
    __syncthreads();
    if (tid < 4) {
      st.cg_stop[tid] = A.cg_tol;
      st.cg_active[tid] = sqrt(st.rr[tid]) > A.cg_tol;
    }
    __syncthreads();
    constexpr int kPhases = kPair ? 2 : 1;
    for (int phase = 0; phase < kPhases; ++phase) {
      int maxit = A.cg_maxit;
      if constexpr (kPair) {
        if (phase == 1) {   // the true residual of x (as a pair), then CG on the correction with x in FP64
          maxit = 20;
          for (int r = tid; r < m; r += NT) {
            float s[4];
            ld4(SJ + 4 * sjrow(r), s);
            st4(SJd + 4 * r, (double)s[0], (double)s[1], (double)s[2], (double)s[3]);
          }
          __syncthreads();
          float part[4] = {0, 0, 0, 0};
          for (int r = tid; r < m; r += NT) {
            float x[4];
            row_resid<TV>(A.valS, rbase[r >> 2], lrow[r >> 2], lrow[(r >> 2) + 1], ent, r & 3, SJ, r - j0, x);
#pragma unroll
            for (int c = 0; c < 4; ++c) part[c] += x[c] * x[c];
            st4(R + 4 * r, x[0], x[1], x[2], x[3]);
            st4(P + 4 * xrow<T>(r), x[0], x[1], x[2], x[3]);
          }
          double acc[4] = {(double)part[0], (double)part[1], (double)part[2], (double)part[3]};
          warp_partial(acc, red, 0, 1);
          __syncthreads();
          if (tid < 4) {
            double s = 0;
            for (int k = 0; k < NT / 32; ++k) s += red[k * 4 + tid];
            st.rr[tid] = s;
            st.cg_stop[tid] = 1e-6 * sqrt(s);
            st.cg_active[tid] = (st.status[tid] == ST_OK) && s > 0.0;
          }
          __syncthreads();
        }
      }
      for (int it = 0; it < maxit; ++it) {
        const int cmask = st.cg_active[0] | (st.cg_active[1] << 1) | (st.cg_active[2] << 2) | (st.cg_active[3] << 3);
        if (!cmask) break;
        // S p and p.(S p) in one pass over the rows
        T part[4] = {0, 0, 0, 0};
        for (int r = tid; r < m; r += NT) {
          T ap[4], pr[4];
          row_s<TV>(A.valS, rbase[r >> 2], lrow[r >> 2], lrow[(r >> 2) + 1], ent, r & 3, P, ap);
          st4(AP + 4 * r, ap[0], ap[1], ap[2], ap[3]);
          ld4(P + 4 * xrow<T>(r), pr);
#pragma unroll
          for (int c = 0; c < 4; ++c) part[c] += pr[c] * ap[c];
        }
        double acc[4] = {(double)part[0], (double)part[1], (double)part[2], (double)part[3]};
        warp_partial(acc, red, 0, 1);
        __syncthreads();
        if (tid < 4) {
          double s = 0;
          for (int k = 0; k < NT / 32; ++k) s += red[k * 4 + tid];
          double a = 0.0;
          if (st.cg_active[tid]) {
            if (!(s > 0.0)) {
              st.status[tid] = ST_NOT_SPD;
              st.cg_active[tid] = 0;
            } else {
              a = st.rr[tid] / s;
            }
          }
          st.alpha[tid] = a;
          scal[tid] = (T)a;
        }
        __syncthreads();
        const bool on0 = st.cg_active[0], on1 = st.cg_active[1], on2 = st.cg_active[2], on3 = st.cg_active[3];
        const bool on[4] = {on0, on1, on2, on3};
#pragma unroll
        for (int c = 0; c < 4; ++c) part[c] = 0;
        for (int r = tid; r < m; r += NT) {
          T pr[4], ap[4], x[4];
          ld4(P + 4 * xrow<T>(r), pr);
          ld4(AP + 4 * r, ap);
          ld4(R + 4 * r, x);
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            if (on[c]) x[c] -= scal[c] * ap[c];
            part[c] += x[c] * x[c];
          }
          st4(R + 4 * r, x[0], x[1], x[2], x[3]);
          if (phase == 0) {
            ld4(SJ + 4 * sjrow(r), x);
#pragma unroll
            for (int c = 0; c < 4; ++c)
              if (on[c]) x[c] += scal[c] * pr[c];
            st4(SJ + 4 * sjrow(r), x[0], x[1], x[2], x[3]);
          } else {
            double xd[4];
            ld4(SJd + 4 * r, xd);
#pragma unroll
            for (int c = 0; c < 4; ++c)
              if (on[c]) xd[c] += st.alpha[c] * (double)pr[c];
            st4(SJd + 4 * r, xd[0], xd[1], xd[2], xd[3]);
          }
        }
        double acc2[4] = {(double)part[0], (double)part[1], (double)part[2], (double)part[3]};
        warp_partial(acc2, red, 0, 1);
        __syncthreads();
        if (tid < 4 && st.cg_active[tid]) {
          double s = 0;
          for (int k = 0; k < NT / 32; ++k) s += red[k * 4 + tid];
          scal[4 + tid] = (T)(s / st.rr[tid]);
          st.rr[tid] = s;
          st.it[tid] += 1;
          if (sqrt(s) <= st.cg_stop[tid]) st.cg_active[tid] = 0;
        }
        __syncthreads();
        for (int r = tid; r < m; r += NT) {
          T pr[4], x[4];
          ld4(P + 4 * xrow<T>(r), pr);
          ld4(R + 4 * r, x);
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if (st.cg_active[c]) pr[c] = x[c] + scal[4 + c] * pr[c];
          st4(P + 4 * xrow<T>(r), pr[0], pr[1], pr[2], pr[3]);
        }
        __syncthreads();
      }
      if (tid < 4) {   // still running after the main phase: not converged; the refinement cap is no failure
        if (phase == 0 && st.cg_active[tid] && st.status[tid] == ST_OK) st.status[tid] = ST_NOCONV;
        st.cg_active[tid] = 0;
      }
      __syncthreads();
    }
    if (A.fallback && tid < 4) A.fallback[4 * widx + tid] = st.fell[tid];
    if (A.keep_s)
      for (int i = tid; i < 16 * A.keep_cap; i += NT) {
        const int c = i / (4 * A.keep_cap), rem = i % (4 * A.keep_cap), t = rem >> 2, o = rem & 3;
        double v = 0.0;
        if (t < ncl) v = kPair ? SJd[4 * (4 * t + o) + c] : (double)SJ[4 * (4 * t + o) + c];
        A.keep_s[(4 * widx + c) * (4 * (int64_t)A.keep_cap) + rem] = v;
      }
    if (A.cg_only) {
      for (int i = tid; i < 4 * 68; i += NT) {
        const int c = i / 68, rem = i % 68, k = rem >> 2, o = rem & 3;
        const int pa = A.patch[widx * 17 + k];
        const int lk = pa >= 0 ? find_local(cl, ncl, pa) : -1;
        float v = 0.0f;
        if (lk >= 0) v = kPair ? (float)SJd[4 * (4 * lk + o) + c] : (float)SJ[4 * (4 * lk + o) + c];
        A.cg_target[(4 * widx + c) * 68 + rem] = v;
      }
      if (tid < 4) {
        A.status[4 * widx + tid] = st.status[tid];
        A.cg_iters[4 * widx + tid] = st.it[tid];
      }
      __syncthreads();
      continue;
    }
    if (tid == 0 && (st.status[0] | st.status[1] | st.status[2] | st.status[3])) st.bad = 1;

    // S_r of vectors [n0, n1) in the FP32 form; the chunks go behind Gs in the shared vectors
    auto gram_pairs = [&](int n0, int n1, double* G) {
      if constexpr (kPair) {
        const int used = G ? gs_floats(A.p) : 0;
        float* stage = reinterpret_cast<float*>(X0) + used;
        if (n1 <= 32) gram_s<4>(W, SW, m, m4, n0, n1, nu, A.red, 4 * widx, G, gst, stage, 3 * m4 - used);
        else gram_s<6>(W, SW, m, m4, n0, n1, nu, A.red, 4 * widx, G, gst, stage, 3 * m4 - used);
      }
    };
    // ---- 3. the chains ------------------------------------------------------------------------------
    // s_j as entries (pairs) in SV; q_1 = e_j into X and W[0]
    for (int r = tid; r < m; r += NT) {
      N s[4], x[4];
      if constexpr (kPair) {
        double d[4];
        ld4(SJd + 4 * r, d);
#pragma unroll
        for (int c = 0; c < 4; ++c) from_double(d[c], s[c]);
      } else {
        ld4(SJ + 4 * sjrow(r), s);
      }
      stv(SV, r, s);
#pragma unroll
      for (int c = 0; c < 4; ++c) from_double(r == j0 + c ? 1.0 : 0.0, x[c]);
      stv(X, xrow<T>(r), x);
      if constexpr (kPair) st4(W + 4 * r, x[0].h, x[1].h, x[2].h, x[3].h);
      else st4(W + 4 * r, x[0], x[1], x[2], x[3]);
    }
    if (tid < 4) {
      st.be[tid] = 0.0;
      from_double(0.0, sc[tid]);
    }
    __syncthreads();
    // scalars: sc[0..3] beta_{n-1} / eta_k; sc[4..7] alpha_n / h_k, then 1 / beta_n; sc[8..11] s_j.q_n in the
    // first chain; in the second sc[8..11] beta (q.v_k), sc[12..15] beta (z.v_k), sc[16..19] q.v_k, sc[20..23] -z.v_k
    const int q_dim = A.q;
    for (int n = 0; n < nu && !st.bad && !st.over; ++n) {
      const bool second = n >= A.p && !st.drop;
      const bool last = n == nu - 1;
      const bool with_s = n < A.p && q_dim > 0;
      N d0[4], d1[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        set_zero(d0[c]);
        set_zero(d1[c]);
      }
      for (int r = tid; r < m; r += NT) {
        const int t = r >> 2;
        N h[4];
        T sw[4];
        row_hs<TV>(A.valH, A.valS, rbase[t], lrow[t], lrow[t + 1], ent, r & 3, X, A.zero, h, sw);
        const size_t o = (size_t)n * m4 + 4 * r;
        st4(HW + o, head(h[0]), head(h[1]), head(h[2]), head(h[3]));
        st4(SW + o, sw[0], sw[1], sw[2], sw[3]);
        if (!(last && !kPair)) stv(Y, r, h);    // FP64: the last H_r entry comes from the Gram matrix alone
      }
      if (last && !kPair) break;
      // own rows: h less its parts along the vectors before the current one, and the dot products with that
      for (int r = tid; r < m; r += NT) {
        const size_t o = (size_t)n * m4 + 4 * r;
        N h[4], x[4], v[4];
        ldv(Y, r, h);
        ldv(X, xrow<T>(r), x);
        if (n > 0 && !(second && n == A.p)) {   // v_1 has no predecessor
          if constexpr (kPair) {
            float a[4], b[4];
            ld4(W + o - m4, a);
            ld4(PV.l + 4 * r, b);
#pragma unroll
            for (int c = 0; c < 4; ++c) v[c] = Pair{a[c], b[c]};
          } else {
            ld4(W + o - m4, v);
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) sub_mul(h[c], sc[c], v[c]);
        }
        if (second) {
          ldv(SV, r, v);                       // a_k
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            sub_mul(h[c], sc[8 + c], v[c]);
            sub_mul(v[c], sc[20 + c], x[c]);
          }
          stv(SV, r, v);
          ldv(BV, r, v);                       // b_k
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            sub_mul(h[c], sc[12 + c], v[c]);
            sub_mul(v[c], sc[16 + c], x[c]);
          }
          stv(BV, r, v);
        }
        if (with_s) {
          ldv(SV, r, v);
#pragma unroll
          for (int c = 0; c < 4; ++c) dot_acc(d1[c], x[c], v[c]);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) dot_acc(d0[c], x[c], h[c]);
        stv(Y, r, h);
      }
      warp_partial(d0, red, 0, 2);
      if (with_s) warp_partial(d1, red, 1, 2);
      __syncthreads();
      if (tid < 8) {
        double s = 0;
        for (int k = 0; k < NT / 32; ++k) s += red[k * 8 + tid];
        if (tid < 4) {
          st.ga[tid] = s;
          tri[n * 4 + tid] = s;
        }
        if (tid < 4 || with_s) from_double(s, sc[4 + tid]);   // alpha_n, and s_j.q_n
      }
      __syncthreads();
      if (last) break;
      // h less its part along the current vector; the norms (and, for the second chain, q.w and z.w)
      const bool seam = with_s && n == A.p - 1;
      N d2[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        set_zero(d0[c]);
        set_zero(d1[c]);
        set_zero(d2[c]);
      }
      for (int r = tid; r < m; r += NT) {
        N x[4], h[4], v[4];
        ldv(X, xrow<T>(r), x);
        ldv(Y, r, h);
#pragma unroll
        for (int c = 0; c < 4; ++c) sub_mul(h[c], sc[4 + c], x[c]);
        stv(Y, r, h);
#pragma unroll
        for (int c = 0; c < 4; ++c) dot_acc(d0[c], h[c], h[c]);
        if (second) {
          N z[4];
          ldv(QV, r, v);
          ldv(ZV, r, z);
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            dot_acc(d1[c], v[c], h[c]);
            dot_acc(d2[c], z[c], h[c]);
          }
        }
        if (with_s) {
          ldv(SV, r, v);
          if (n == 0)
#pragma unroll
            for (int c = 0; c < 4; ++c) dot_acc(d2[c], v[c], v[c]);
#pragma unroll
          for (int c = 0; c < 4; ++c) sub_mul(v[c], sc[8 + c], x[c]);
          stv(SV, r, v);
          if (seam)
#pragma unroll
            for (int c = 0; c < 4; ++c) dot_acc(d1[c], v[c], v[c]);
        }
      }
      warp_partial(d0, red, 0, 3);
      warp_partial(d1, red, 1, 3);
      warp_partial(d2, red, 2, 3);
      __syncthreads();
      if (tid < 4) {
        const int c = tid;
        double b2 = 0, x1 = 0, x2 = 0;
        for (int k = 0; k < NT / 32; ++k) {
          b2 += red[(k * 3 + 0) * 4 + c];
          x1 += red[(k * 3 + 1) * 4 + c];
          x2 += red[(k * 3 + 2) * 4 + c];
        }
        const double al = st.ga[c], bp = st.be[c];
        double all = al * al + bp * bp + b2;
        if (second) {
          const double u = to_double(sc[8 + c]), w = to_double(sc[12 + c]);
          all += u * u + w * w;
        }
        if (!(b2 > 1e-12 * all)) st.bad = 1;    // the chain closes (or is not a number): the general kernel
        const double beta = sqrt(b2), inv = 1.0 / beta;
        st.be[c] = beta;
        tri[(nu + n) * 4 + c] = beta;
        from_double(beta, sc[c]);
        from_double(inv, sc[4 + c]);
        if (second) {                            // q.v_{k+1}, z.v_{k+1}
          chain_scalars(st.s0[c], x1 * inv, x2 * inv, sc, c);
          tri[(2 * nu + n + 1) * 4 + c] = x1 * inv;
          tri[(3 * nu + n + 1) * 4 + c] = x2 * inv;
        }
        if (with_s && n == 0) st.s0[c] = x2;     // ||s_j||^2
        if (seam) {
          const double ratio = sqrt(fmax(x1, 0.0) / st.s0[c]);
          const bool gone = ratio <= 1e-12;
          if (!gone && !(ratio > 1e-7)) st.bad = 1;
          atomicAdd(&st.drop, gone ? 1 : 0);
          st.alpha[c] = 1.0 / sqrt(x1);
        }
      }
      __syncthreads();
      if (st.bad) break;
      if (seam) {
        const int drop = st.drop;                // columns whose s_j lies in K_p
        __syncthreads();
        if (drop != 0 && drop != 4) {
          if (tid == 0) st.bad = 1;
          break;
        }
        if (drop == 0) {
          // q_{p+1} -> b_1 and QV, q_p -> a_1 (its hi part is W[p-1]); s_j stays in Y for v_1
          for (int r = tid; r < m; r += NT) {
            N x[4], h[4], v[4];
            ldv(X, xrow<T>(r), x);
            ldv(Y, r, h);
            ldv(SV, r, v);
#pragma unroll
            for (int c = 0; c < 4; ++c) h[c] = scaled(h[c], sc[4 + c]);
            stv(BV, r, h);
            stv(QV, r, h);
            stv(SV, r, x);
            N iv;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              from_double(st.alpha[c], iv);
              v[c] = scaled(v[c], iv);
            }
            stv(PV, r, v);                       // v_1, until the shared vectors are free again
          }
          __syncthreads();
          if constexpr (kPair) gram_pairs(0, A.p, Gs);
          else gram<T>(W, HW, SW, m, m4, 0, A.p, nu, A.red, 4 * widx, Gs, gst);
          __syncthreads();
          // g = (Q^T S Q)^{-1} e_p by Cholesky, one warp per column: L^{-1} e_p has only its last entry
          if (tid < 128) {
            const int c = tid >> 5, lane = tid & 31, p = A.p;
            double* G = Gs + c * gst;
            bool ok = true;
            for (int k = 0; k < p; ++k) {
              const double akk = G[k * (k + 1) / 2 + k];
              ok = ok && akk > 0.0;
              const double rd = 1.0 / sqrt(akk);
              __syncwarp();
              for (int i = k + lane; i < p; i += 32) G[i * (i + 1) / 2 + k] *= rd;   // row k: L_kk
              __syncwarp();
              for (int i = k + 1 + lane; i < p; i += 32) {
                const double lik = G[i * (i + 1) / 2 + k];
                for (int jj = k + 1; jj <= i; ++jj) G[i * (i + 1) / 2 + jj] -= lik * G[jj * (jj + 1) / 2 + k];
              }
              __syncwarp();
            }
            if (!ok && lane == 0) st.bad = 1;
            if (lane == 0)                       // back substitution L^T g = e_p / L_pp; g over the diagonal
              for (int i = p - 1; i >= 0; --i) {
                double s = i == p - 1 ? 1.0 / G[i * (i + 1) / 2 + i] : 0.0;
                for (int k = i + 1; k < p; ++k) s -= G[k * (k + 1) / 2 + i] * G[k * (k + 1) / 2 + k];
                s /= G[i * (i + 1) / 2 + i];
                G[i * (i + 1) / 2 + i] = s;
                from_double(s, gv[c * p + i]);
              }
          }
          if (tid < 4) {                         // beta_p stays for the whole second chain
            st.s0[tid] = st.be[tid];
            st.be[tid] = 0.0;
          }
          __syncthreads();
          if (st.bad) break;
          // z = S (Q g), and q.v_1, z.v_1. FP64 adds up the g_n S q_n. The second chain's span leans on z, in one of 10^5
          // columns 300 times as much as in most, and with z from the FP32 S q_n rho of such columns was off by up to 9e-7
          // (most: 1e-8); so the pair form multiplies the pair Q g by S once more, with compensated sums, and keeps z as a
          // pair: 1.6e-7 at most over 4.5e5 atoms of three systems, for 2 % of the kernel's time.
          if constexpr (kPair) seam_z<TV>(A.valS, A.zero, W, A.p, m, m4, gv, X, Y.l, ZV, rbase, lrow, ent);
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            set_zero(d0[c]);
            set_zero(d1[c]);
          }
          for (int r = tid; r < m; r += NT) {
            N v[4];
            ldv(PV, r, v);
            N z[4];
            if constexpr (kPair) {
              ldv(ZV, r, z);
            } else {
#pragma unroll
              for (int c = 0; c < 4; ++c) set_zero(z[c]);
              for (int k = 0; k < A.p; ++k) {
                T s[4];
                ld4(SW + (size_t)k * m4 + 4 * r, s);
#pragma unroll
                for (int c = 0; c < 4; ++c) dot_acc(z[c], s[c], gv[c * A.p + k]);
              }
            }
            N q[4];
            ldv(QV, r, q);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              dot_acc(d0[c], q[c], v[c]);
              dot_acc(d1[c], z[c], v[c]);
            }
            if constexpr (!kPair) stv(ZV, r, z);
          }
          warp_partial(d0, red, 0, 2);
          warp_partial(d1, red, 1, 2);
          __syncthreads();
          if (tid < 4) {
            double x1 = 0, x2 = 0;
            for (int k = 0; k < NT / 32; ++k) {
              x1 += red[k * 8 + tid];
              x2 += red[k * 8 + 4 + tid];
            }
            chain_scalars(st.s0[tid], x1, x2, sc, tid);
            tri[(2 * nu + A.p) * 4 + tid] = x1;
            tri[(3 * nu + A.p) * 4 + tid] = x2;
          }
          for (int r = tid; r < m; r += NT) {    // v_1 into X and W[p]
            N v[4];
            ldv(PV, r, v);
            stv(X, xrow<T>(r), v);
            st4(W + (size_t)A.p * m4 + 4 * r, head(v[0]), head(v[1]), head(v[2]), head(v[3]));
#pragma unroll
            for (int c = 0; c < 4; ++c)
              if (r == j0 + c) check_overlap(st, to_double(v[c]));
          }
          __syncthreads();
          continue;
        }
      }
      // the next vector: h / beta
      for (int r = tid; r < m; r += NT) {
        N x[4], h[4];
        if constexpr (kPair) {                   // the current vector's low half, for the next step
          float l[4];
          ld4(X.l + 4 * xrow<T>(r), l);
          st4(PV.l + 4 * r, l[0], l[1], l[2], l[3]);
        }
        ldv(Y, r, h);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          x[c] = scaled(h[c], sc[4 + c]);
          if (r == j0 + c) check_overlap(st, to_double(x[c]));
        }
        stv(X, xrow<T>(r), x);
        st4(W + (size_t)(n + 1) * m4 + 4 * r, head(x[0]), head(x[1]), head(x[2]), head(x[3]));
      }
      __syncthreads();
    }
    __syncthreads();
    if (st.bad || st.over) {
      if (tid == 0) {
        A.redo[atomicAdd(A.redo_count, 1)] = (int32_t)widx;
        atomicAdd(A.late_count, 1);
      }
      __syncthreads();
      continue;
    }
    // ---- 4. Gram matrices, rows j, outputs ------------------------------------------------------------
    const int p1 = q_dim > 0 && !st.drop ? A.p : nu;     // the first chain's length
    const int n_done = p1 < nu ? p1 : 0;                 // the seam has taken the first chain's Gram matrix
    if constexpr (!kPair) {
      gram<T>(W, HW, SW, m, m4, n_done, nu, nu, A.red, 4 * widx, nullptr, 0);
    } else {
      gram_pairs(n_done, nu, nullptr);
      if (st.careful) {
        gram<T>(W, HW, SW, m, m4, 0, nu, nu, A.red, 4 * widx, nullptr, 0);
      } else {
        // H_r from the coefficients: tridiagonal in the first chain, H(q_p, v_k) = beta q.v_k, and
        // v_i.(H v_k) = beta (q.v_k)(z.v_i) + (the second chain's tridiagonal) for i <= k
        double* R0 = A.red + (size_t)((4 * widx) >> 5) * red_block_doubles(nu) * 32 + ((4 * widx) & 31);
        for (int t = tid; t < 4 * nu * nu; t += NT) {
          const int c = t & 3, a = (t >> 2) / nu, b = (t >> 2) % nu;
          if (a > b) continue;
          double v = a == b ? tri[4 * a + c] : a == b - 1 ? tri[(nu + a) * 4 + c] : 0.0;
          if (b >= p1) {
            const double bq = tri[(nu + p1 - 1) * 4 + c] * tri[(2 * nu + b) * 4 + c];
            v = a >= p1 ? v + bq * tri[(3 * nu + a) * 4 + c] : a == p1 - 1 ? bq : 0.0;
          }
          R0[(size_t)(a * nu + b) * 32 + c] = v;
        }
      }
    }
    {
      double* red0 = A.red + (size_t)((4 * widx) >> 5) * red_block_doubles(nu) * 32;
      for (int i = tid; i < 4 * 2 * nu; i += NT) {
        const int c = i & 3, k = i >> 2, n = k % nu;
        const T* src = (k < nu ? W : SW) + (size_t)n * m4 + 4 * (j0 + c) + c;
        red0[((size_t)2 * nu * nu + k) * 32 + ((4 * widx + c) & 31)] = (double)*src;
      }
    }
    if (tid < 4) {
      A.status[4 * widx + tid] = st.status[tid];
      A.nu_eff[4 * widx + tid] = nu;
      A.cg_iters[4 * widx + tid] = st.it[tid];
    }
    if (A.keep) {   // pattern rows of W (zero outside the cluster)
      const int nrow = A.row_ptr[atom + 1] - A.row_ptr[atom];
      double* vpa = A.vp + A.blk_off[widx] * 16 * (int64_t)nu;
      const int e0 = lrow[t0], ne = lrow[t0 + 1] - e0;
      if (ne < nrow) {
        for (int i = tid; i < nrow * 16 * nu; i += NT) vpa[i] = 0.0;
        __syncthreads();
      }
      for (int i = tid; i < 16 * ne * nu; i += NT) {
        const int n = i % nu, rem = i / nu, e = e0 + (rem >> 4), c = rem >> 2 & 3, r = rem & 3;
        const int k = (int)(ent[e] >> 16), lc = (int)(ent[e] & 0xFFFFu) >> 4;
        vpa[((int64_t)k * 16 + c * 4 + r) * nu + n] = (double)W[(size_t)n * m4 + 4 * (4 * lc + r) + c];
      }
    }
    __syncthreads();
  }
}

// counter: see kAtomsCounters.
__global__ void __launch_bounds__(256) judge_kernel(int* counter, int32_t* redo, const int32_t* order, int64_t n_first,
                                                    int64_t n_sel, bool mixed) {
  const int left = counter[1], late = counter[3];
  __syncthreads();
  if (chains_pay(mixed, late, n_first - (left - late))) {
    if (threadIdx.x == 0) counter[0] = (int)n_first;
    return;
  }
  for (int64_t i = n_first + threadIdx.x; i < n_sel; i += 256) redo[left + i - n_first] = order ? order[i] : (int32_t)i;
  if (threadIdx.x == 0) {
    counter[0] = (int)n_sel;
    counter[1] = (int)(left + n_sel - n_first);
  }
}

size_t chains_smem_bytes(int clcap, int lnnz_cap, int mcap, size_t elem) {
  const size_t off = (size_t)(clcap + 2 * (mcap / 4) + 1 + lnnz_cap) * sizeof(int);
  return align_up(off, 64) + (size_t)mcap * 4 * (elem == 4 ? 3 * sizeof(float) : 2 * sizeof(double));
}

size_t chains_slot_bytes(int nu, int mcap, size_t elem) {
  return align_up(elem * ((size_t)3 * nu + work_vectors(elem)) * mcap * 4, 256) +
         align_up(sizeof(double) * (4 * (size_t)mcap + 16 * (size_t)nu), 256);
}

template <typename TV, typename T, int NT>
mka_status chains_config_t(int nu, int ctas_per_sm, AtomsConfig* cf) {
  auto kern = chains_kernel<TV, T, NT>;
  const size_t smem = chains_smem_bytes(cf->clcap, cf->lnnz_cap, cf->mcap, sizeof(T));
  int dev = 0, sms = 0, per_sm = 0;
  size_t most = 0;
  mka_status s = allow_shared(reinterpret_cast<const void*>(kern), &most);
  if (s) return s;
  if (smem > most) return MKA_OK;              // the general kernel takes every atom
  MKA_CUDA_TRY(cudaGetDevice(&dev));
  MKA_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  MKA_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, smem));
  if (per_sm < 1) return MKA_OK;
  if (ctas_per_sm > 0) per_sm = std::min(per_sm, ctas_per_sm);
  cf->chains = 1;
  cf->chains_smem = smem;
  cf->chains_slot = chains_slot_bytes(nu, cf->mcap, sizeof(T));
  cf->chains_grid = sms * per_sm;
  cf->per_sm = per_sm;
  return MKA_OK;
}

template <typename TV, typename T, int NT>
mka_status chains_launch_t(const mka_system* sys, const AtomsConfig& cf, const AtomsLaunchArgs& a, cudaStream_t st) {
  Args<TV> A{};
  fill_args(A, sys, cf, a);
  A.slot_bytes = cf.chains_slot;
  A.redo = a.redo;
  A.redo_count = a.counter + 1;
  A.late_count = a.counter + 3;
  const int grid = (int)std::min<int64_t>(a.n_sel, cf.chains_grid);
  chains_kernel<TV, T, NT><<<(unsigned)grid, NT, cf.chains_smem, st>>>(A);
  count_launches();
  MKA_CUDA_TRY(cudaGetLastError());
  return MKA_OK;
}

}  // namespace

mka_status chains_config(const mka_system* sys, int nu, int arith, int ctas_per_sm, AtomsConfig* cf) {
  const bool mixed = arith != MKA_FP64;
#define MKA_CFG(TV, T, NT) chains_config_t<TV, T, NT>(nu, ctas_per_sm, cf)
  return MKA_DISPATCH(MKA_CFG, sys->storage, mixed, cf->threads);
#undef MKA_CFG
}

mka_status chains_judge(int arith, const AtomsLaunchArgs& a, int64_t n_first, cudaStream_t st) {
  judge_kernel<<<1, 256, 0, st>>>(a.counter, a.redo, a.order, n_first, a.n_sel, arith != MKA_FP64);
  count_launches();
  MKA_CUDA_TRY(cudaGetLastError());
  return MKA_OK;
}

mka_status chains_launch(const mka_system* sys, int arith, const AtomsConfig& cf, const AtomsLaunchArgs& a,
                         cudaStream_t st) {
  const bool mixed = arith != MKA_FP64;
#define MKA_LAUNCH(TV, T, NT) chains_launch_t<TV, T, NT>(sys, cf, a, st)
  return MKA_DISPATCH(MKA_LAUNCH, sys->storage, mixed, cf.threads);
#undef MKA_LAUNCH
}

}  // namespace mka
