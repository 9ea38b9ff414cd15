// Learned warm start for the inner CG (S s_j = e_j, Sec. 2): input features, the network's
// forward / backward / Adam kernels, and the C entry points.
//
// Features of atom a (one warp per atom): its 32 nearest neighbours within 3 A (minimum
// image, distance order, ties by atom id) as (d, l, m, n) with (l, m, n) the direction
// cosines of r_b - r_a, zeros beyond; the 17-atom output patch is a and its 16 nearest
// neighbours. A column's input row is those 128 numbers and a one-hot of its orbital (132).
//
// Network 132 -> 128 -> 128 -> 68 with SiLU after the hidden layers. Parameters are kept in
// FP32 (Adam master copy) and rounded to BF16 for every product; activations and sums are
// FP32. Loss: mean of (y - t)^2 over the batch and the 68 outputs. Weight gradients are
// batch reductions in a fixed order (row chunks of a size given by the batch, then the chunks in turn), so training is
// deterministic.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <cstring>
#include <random>
#include <vector>

#include "mka_internal.h"

namespace mka {
namespace {

constexpr int kIn = 132, kHid = 128, kOut = 68;
constexpr int kNeigh = 32, kPatch = 17;
constexpr int kFeatGather = 256;                   // candidates per atom kept for selection
constexpr int64_t kP = (int64_t)kHid * kIn + kHid + (int64_t)kHid * kHid + kHid + (int64_t)kOut * kHid + kOut;
constexpr int64_t oW1 = 0, ob1 = oW1 + kHid * kIn, oW2 = ob1 + kHid, ob2 = oW2 + kHid * kHid, oW3 = ob2 + kHid,
                  ob3 = oW3 + kOut * kHid;

__device__ __forceinline__ float bf(const __nv_bfloat16* p, int64_t i) { return __bfloat162float(p[i]); }
__device__ __forceinline__ float silu_f(float x) { return x / (1.0f + __expf(-x)); }
__device__ __forceinline__ float dsilu_f(float x) {
  const float s = 1.0f / (1.0f + __expf(-x));
  return s * (1.0f + x * (1.0f - s));
}

// ---- features --------------------------------------------------------------------------
struct FeatArgs {
  const double* pos;
  const float* posf;
  double box[3], inv_box[3];
  float pre_hi;     // FP32 prefilter: candidates beyond pre_hi * r_gather^2 are dropped unseen
  int ncell[3];
  double cell_len[3];
  const int32_t* cell_start;
  const int32_t* cell_atoms;
  const int64_t* sel;
  int64_t n_sel;
  double r_gather2;
  float* X;         // [4 n_sel][132]
  int32_t* patch;   // [n_sel][17] atom ids, -1 where fewer atoms were found
};

__device__ __forceinline__ int cell_coord_f(double x, double len, int n) {
  int v = (int)floor(x / len);
  return v < 0 ? 0 : (v >= n ? n - 1 : v);
}

__device__ __forceinline__ int cell_range_f(int c, int n, int out[3]) {
  if (n < 3) {
    for (int i = 0; i < n; ++i) out[i] = i;
    return n;
  }
  out[0] = (c + n - 1) % n;
  out[1] = c;
  out[2] = (c + 1) % n;
  return 3;
}

// Minimum-image displacement and distance in the operation order of a plain evaluation
// (d = b - a; d -= L k with k = rint(d / L); r^2 = (dx^2 + dy^2) + dz^2), without contraction,
// so that neighbour order and the 3 A cut agree with any IEEE evaluation of the same formula.
// k is taken as rint(d * (1/L)): it differs from rint(d / L) only when d / L is within an ulp of
// +-1/2, i.e. for atoms half a box away, far outside the gather radius.
__device__ __forceinline__ double mi_comp(double pb, double pa, double L, double invL) {
  const double d = __dsub_rn(pb, pa);
  return __dsub_rn(d, __dmul_rn(L, rint(d * invL)));
}

// One warp per atom; per warp kFeatGather (distance, id) candidate slots in shared memory.
__global__ void __launch_bounds__(256) features_kernel(FeatArgs A) {
  __shared__ unsigned long long rk[8][kFeatGather];   // bits of the distance
  __shared__ int idk[8][kFeatGather];
  __shared__ int cnt[8];
  __shared__ int near[8][kNeigh];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t warp = (int64_t)blockIdx.x * 8 + wid, nw = (int64_t)gridDim.x * 8;
  for (int64_t t = warp; t < A.n_sel; t += nw) {
    const int64_t a = A.sel[t];
    const double px = A.pos[3 * a], py = A.pos[3 * a + 1], pz = A.pos[3 * a + 2];
    const float pxf = A.posf[3 * a], pyf = A.posf[3 * a + 1], pzf = A.posf[3 * a + 2];
    const float Lf[3] = {(float)A.box[0], (float)A.box[1], (float)A.box[2]};
    const float iLf[3] = {(float)A.inv_box[0], (float)A.inv_box[1], (float)A.inv_box[2]};
    const float rg2f = (float)A.r_gather2;
    int rx[3], ry[3], rz[3];
    const int nx = cell_range_f(cell_coord_f(px, A.cell_len[0], A.ncell[0]), A.ncell[0], rx);
    const int ny = cell_range_f(cell_coord_f(py, A.cell_len[1], A.ncell[1]), A.ncell[1], ry);
    const int nz = cell_range_f(cell_coord_f(pz, A.cell_len[2], A.ncell[2]), A.ncell[2], rz);
    if (lane == 0) cnt[wid] = 0;
    __syncwarp();
    for (int ci = 0; ci < nx * ny * nz; ++ci) {
      const int ix = ci / (ny * nz), iy = (ci / nz) % ny, iz = ci % nz;
      const int c = (rx[ix] * A.ncell[1] + ry[iy]) * A.ncell[2] + rz[iz];
      for (int k = A.cell_start[c] + lane; k < A.cell_start[c + 1]; k += 32) {
        const int b = A.cell_atoms[k];
        if (b == a) continue;
        float fx = A.posf[3 * b] - pxf, fy = A.posf[3 * b + 1] - pyf, fz = A.posf[3 * b + 2] - pzf;
        fx -= Lf[0] * rintf(fx * iLf[0]);
        fy -= Lf[1] * rintf(fy * iLf[1]);
        fz -= Lf[2] * rintf(fz * iLf[2]);
        if (fx * fx + fy * fy + fz * fz > A.pre_hi * rg2f) continue;
        const double dx = mi_comp(A.pos[3 * b], px, A.box[0], A.inv_box[0]);
        const double dy = mi_comp(A.pos[3 * b + 1], py, A.box[1], A.inv_box[1]);
        const double dz = mi_comp(A.pos[3 * b + 2], pz, A.box[2], A.inv_box[2]);
        const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
        if (r2 <= A.r_gather2) {
          const int s = atomicAdd(&cnt[wid], 1);
          if (s < kFeatGather) {
            rk[wid][s] = (unsigned long long)__double_as_longlong(__dsqrt_rn(r2));
            idk[wid][s] = b;
          }
        }
      }
    }
    __syncwarp();
    const int n = min(cnt[wid], kFeatGather);
    // the 32 nearest by (distance, id): a candidate's place is the number of candidates before it, counted on the bits
    // of the distances, whose order as integers is their own (none is negative). Repeated minima took 32 rounds of FP64
    // compares and shuffles, 2.27 ms for 13,824 atoms.
    if (lane < kNeigh) near[wid][lane] = -1;
    __syncwarp();
    for (int s0 = lane; s0 < n; s0 += 32) {
      const unsigned long long r = rk[wid][s0];
      const int id = idk[wid][s0];
      int before = 0;
      for (int s = 0; s < n; ++s) {
        const unsigned long long rs = rk[wid][s];
        before += rs < r || (rs == r && idk[wid][s] < id);
      }
      if (before < kNeigh) near[wid][before] = s0;
    }
    __syncwarp();
    float geo[4] = {0, 0, 0, 0};   // lane k < 32 keeps neighbour k's (d, l, m, n)
    int my_id = -1;
    const int bi = near[wid][lane];
    if (bi >= 0) {
      const int bid = idk[wid][bi];
      const double best = __longlong_as_double((long long)rk[wid][bi]);
      my_id = bid;
      if (best <= 3.0) {
        const double dx = mi_comp(A.pos[3 * bid], px, A.box[0], A.inv_box[0]);
        const double dy = mi_comp(A.pos[3 * bid + 1], py, A.box[1], A.inv_box[1]);
        const double dz = mi_comp(A.pos[3 * bid + 2], pz, A.box[2], A.inv_box[2]);
        geo[0] = (float)best;
        geo[1] = (float)__ddiv_rn(dx, best);
        geo[2] = (float)__ddiv_rn(dy, best);
        geo[3] = (float)__ddiv_rn(dz, best);
      }
    }
    for (int o = 0; o < 4; ++o) {
      float* row = A.X + (4 * t + o) * (int64_t)kIn;
      for (int q = 0; q < 4; ++q) row[4 * lane + q] = geo[q];
      if (lane < 4) row[128 + lane] = (lane == o) ? 1.0f : 0.0f;
    }
    if (lane == 0) A.patch[t * kPatch] = (int32_t)a;
    if (lane < kPatch - 1) A.patch[t * kPatch + 1 + lane] = my_id;
    __syncwarp();
  }
}

// ---- network kernels --------------------------------------------------------------------
// The three layers are a chain for each row and the weights are small (85 KB in BF16), so one CTA takes kTile rows the
// whole way: the weights of all layers in shared memory once (word [k / 2][o]: the pair k, k + 1 of output o, read along
// o forward and along k backward without bank conflicts), activations [k][row] beside them, thread (o, half) on
// output o of four rows, sums over k in order. With GRAD also the loss of the tile and the chain back to the first
// layer's pre-activation; what the weight gradients need goes to memory. CTAs walk over tiles, two on an SM. A
// kernel per layer and direction (seven) was bound by launches and each by one CTA's latency; forward, loss and all
// gradients of 1,024 rows: 461 -> 40 us with the two kernels below.
constexpr int kTile = 8, kRowThreads = 256;
constexpr int kStride1 = kHid + 1, kStride3 = kOut + 1;   // odd: neighbouring k pairs in different banks
constexpr int kWords = (kIn / 2 + kHid / 2) * kStride1 + kHid / 2 * kStride3;
constexpr size_t kRowSmem = sizeof(float) * (kWords + kTile * (kIn + 4 * kHid + kOut));

struct RowArgs {
  const float* X;
  const float* T;
  int64_t B;
  const __nv_bfloat16* P;
  float* Y;                  // forward only
  float *H1, *H2, *dY, *dZ2, *dZ1;   // GRAD: [B][128 or 68]
  float* loss;               // GRAD: [tiles] sums of (y - t)^2 inv
  float inv;                 // 1 / (68 B)
};

__device__ __forceinline__ float pair_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float pair_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

__device__ __forceinline__ void fma4(float (&a)[4], const float* x, float w) {
  const float4 v = *reinterpret_cast<const float4*>(x);
  a[0] += v.x * w;
  a[1] += v.y * w;
  a[2] += v.z * w;
  a[3] += v.w * w;
}

// acc[r] = sum_k in[k][r] W[o][k]
template <int N, int S>
__device__ __forceinline__ void layer_forward(const uint32_t* w, const float* in, int o, float (&acc)[4]) {
  acc[0] = acc[1] = acc[2] = acc[3] = 0.0f;
#pragma unroll 8
  for (int k = 0; k < N / 2; ++k) {
    const uint32_t u = w[k * S + o];
    fma4(acc, in + 2 * k * kTile, pair_lo(u));
    fma4(acc, in + (2 * k + 1) * kTile, pair_hi(u));
  }
}

// acc[r] = sum_o d[o][r] W[o][k]
template <int O, int S>
__device__ __forceinline__ void layer_backward(const uint32_t* w, const float* d, int k, float (&acc)[4]) {
  acc[0] = acc[1] = acc[2] = acc[3] = 0.0f;
  const uint32_t* wk = w + (k >> 1) * S;
#pragma unroll 8
  for (int o = 0; o < O; ++o) {
    const uint32_t u = wk[o];
    fma4(acc, d + o * kTile, k & 1 ? pair_hi(u) : pair_lo(u));
  }
}

// W [O][N] in BF16 to words [N / 2][S]
template <int N, int O, int S>
__device__ __forceinline__ void stage_weights(const __nv_bfloat16* __restrict__ W, uint32_t* w) {
  const uint32_t* p = reinterpret_cast<const uint32_t*>(W);
#pragma unroll 8
  for (int e = threadIdx.x; e < N / 2 * O; e += kRowThreads) w[e % (N / 2) * S + e / (N / 2)] = __ldg(p + e);
}

template <bool GRAD>
__global__ void __launch_bounds__(kRowThreads, 2) mlp_rows_kernel(const RowArgs A) {
  extern __shared__ __align__(16) float fsm[];
  __shared__ float red[kRowThreads / 32];
  float* xs = fsm;                                // [132][kTile], then the layers likewise
  float *h1 = xs + kIn * kTile, *h2 = h1 + kHid * kTile, *z1 = h2 + kHid * kTile, *z2 = z1 + kHid * kTile;
  float* dy = z2 + kHid * kTile;
  uint32_t* w1 = reinterpret_cast<uint32_t*>(dy + kOut * kTile);
  uint32_t *w2 = w1 + kIn / 2 * kStride1, *w3 = w2 + kHid / 2 * kStride1;
  stage_weights<kIn, kHid, kStride1>(A.P + oW1, w1);
  stage_weights<kHid, kHid, kStride1>(A.P + oW2, w2);
  stage_weights<kHid, kOut, kStride3>(A.P + oW3, w3);
  const int o = threadIdx.x & (kHid - 1), q = threadIdx.x / kHid * 4;
  const float b1 = bf(A.P, ob1 + o), b2 = bf(A.P, ob2 + o), b3 = o < kOut ? bf(A.P, ob3 + o) : 0.0f;
  const int64_t tiles = (A.B + kTile - 1) / kTile;
  for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int64_t r0 = t * kTile;
    const int rows = (int)(A.B - r0 < kTile ? A.B - r0 : kTile);
    for (int e = threadIdx.x; e < kTile * kIn; e += kRowThreads) {
      const int r = e / kIn, k = e % kIn;
      xs[k * kTile + r] = r < rows ? A.X[r0 * kIn + e] : 0.0f;
    }
    __syncthreads();
    float acc[4];
    layer_forward<kIn, kStride1>(w1, xs + q, o, acc);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float z = acc[r] + b1, h = silu_f(z);
      h1[o * kTile + q + r] = h;
      if (GRAD) {
        z1[o * kTile + q + r] = z;
        if (q + r < rows) A.H1[(r0 + q + r) * kHid + o] = h;
      }
    }
    __syncthreads();
    layer_forward<kHid, kStride1>(w2, h1 + q, o, acc);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float z = acc[r] + b2, h = silu_f(z);
      h2[o * kTile + q + r] = h;
      if (GRAD) {
        z2[o * kTile + q + r] = z;
        if (q + r < rows) A.H2[(r0 + q + r) * kHid + o] = h;
      }
    }
    __syncthreads();
    float part = 0.0f;
    if (o < kOut) {
      layer_forward<kHid, kStride3>(w3, h2 + q, o, acc);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float y = acc[r] + b3;
        const int64_t at = (r0 + q + r) * kOut + o;
        if (!GRAD) {
          if (q + r < rows) A.Y[at] = y;
          continue;
        }
        float dv = 0.0f;
        if (q + r < rows) {
          const float d = y - A.T[at];
          dv = 2.0f * d * A.inv;
          part += d * d * A.inv;
          A.dY[at] = dv;
        }
        dy[o * kTile + q + r] = dv;
      }
    }
    if (GRAD) {
      for (int s = 16; s > 0; s >>= 1) part += __shfl_xor_sync(0xffffffffu, part, s);
      if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
      __syncthreads();
      if (threadIdx.x == 0) {
        float s = 0.0f;
        for (int k = 0; k < kRowThreads / 32; ++k) s += red[k];
        A.loss[t] = s;
      }
      layer_backward<kOut, kStride3>(w3, dy + q, o, acc);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float d = acc[r] * dsilu_f(z2[o * kTile + q + r]);
        z2[o * kTile + q + r] = d;                // its own entries: dZ2 in their place
        if (q + r < rows) A.dZ2[(r0 + q + r) * kHid + o] = d;
      }
      __syncthreads();
      layer_backward<kHid, kStride1>(w2, z2 + q, o, acc);
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (q + r < rows) A.dZ1[(r0 + q + r) * kHid + o] = acc[r] * dsilu_f(z1[o * kTile + q + r]);
    }
    __syncthreads();
  }
}

// Weight gradients G[o][i] = sum_b d_out[b][o] in[b][i] and bias gradients sum_b d_out[b][o] of all layers: a CTA takes
// a tile of one layer's matrix (ten tiles of at most 68 x 68, 4 x 4 sums a thread) and one chunk of rows, 32 rows at a
// time through shared memory; grad_sum_kernel adds the chunks in turn. Up to kMaxChunks chunks, so that the partial sums
// stay small beside the batch and a batch of 1,024 still has 320 CTAs; a thread per weight walked the whole
// batch, 1,024 dependent steps on 330 warps.
constexpr int kGradSide = 17, kGradThreads = 320, kGradRows = 32, kMaxChunks = 64;

struct GradArgs {
  const float *X, *H1, *H2, *dZ1, *dZ2, *dY;
  int64_t B, chunk_rows;
  float* part;               // [chunks][kP]
};

__host__ __device__ inline int64_t grad_chunk_rows(int64_t B) {
  const int64_t per = (int64_t)kGradRows * kMaxChunks;
  return (B + per - 1) / per * kGradRows;
}

__global__ void __launch_bounds__(kGradThreads) grad_part_kernel(const GradArgs A) {
  __shared__ __align__(16) float ds[kGradRows][4 * kGradSide], is[kGradRows][4 * kGradSide];
  const int tile = blockIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int layer = tile < 4 ? 0 : tile < 8 ? 1 : 2, sub = tile - 4 * layer;
  const float* dout = layer == 0 ? A.dZ1 : layer == 1 ? A.dZ2 : A.dY;
  const float* in = layer == 0 ? A.X : layer == 1 ? A.H1 : A.H2;
  const int O = layer == 2 ? kOut : kHid, N = layer == 0 ? kIn : kHid;
  const int ow = layer == 2 ? kOut : kHid / 2, iw = N / 2;          // the tile: 68 or 64 outputs, 66 or 64 inputs
  const int o0 = layer == 2 ? 0 : (sub >> 1) * ow, i0 = (layer == 2 ? sub : sub & 1) * iw;
  const int ty = threadIdx.x / kGradSide, tx = threadIdx.x % kGradSide;
  const bool on = ty < kGradSide;
  const int64_t b0 = (int64_t)blockIdx.y * A.chunk_rows, b1 = b0 + A.chunk_rows < A.B ? b0 + A.chunk_rows : A.B;
  float acc[4][4], bias[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    bias[a] = 0.0f;
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.0f;
  }
  for (int64_t b = b0; b < b1; b += kGradRows) {
    for (int r = wid; r < kGradRows; r += kGradThreads / 32) {
      const bool real = b + r < b1;
      for (int c = lane; c < 4 * kGradSide; c += 32) {
        ds[r][c] = real && c < ow ? __ldg(dout + (b + r) * O + o0 + c) : 0.0f;
        is[r][c] = real && c < iw ? __ldg(in + (b + r) * N + i0 + c) : 0.0f;
      }
    }
    __syncthreads();
    if (on) {
#pragma unroll 8
      for (int r = 0; r < kGradRows; ++r) {
        const float4 d = *reinterpret_cast<const float4*>(&ds[r][4 * ty]);
        const float4 x = *reinterpret_cast<const float4*>(&is[r][4 * tx]);
        const float dv[4] = {d.x, d.y, d.z, d.w}, xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          bias[a] += dv[a];
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[a][c] += dv[a] * xv[c];
        }
      }
    }
    __syncthreads();
  }
  if (!on) return;
  float* G = A.part + (int64_t)blockIdx.y * kP + (layer == 0 ? oW1 : layer == 1 ? oW2 : oW3);
  float* Gb = A.part + (int64_t)blockIdx.y * kP + (layer == 0 ? ob1 : layer == 1 ? ob2 : ob3);
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int o = 4 * ty + a;
    if (o >= ow) continue;
    if (i0 == 0 && tx == 0) Gb[o0 + o] = bias[a];
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (4 * tx + c < iw) G[(int64_t)(o0 + o) * N + i0 + 4 * tx + c] = acc[a][c];
  }
}

// g = the chunks' sums in turn; the last block: the loss from the tiles' (strided per thread, then a fixed tree).
__global__ void __launch_bounds__(256) grad_sum_kernel(const float* __restrict__ part, int chunks, float* __restrict__ g,
                                                       const float* __restrict__ tile_loss, int64_t tiles, float* loss) {
  if (blockIdx.x + 1 < gridDim.x) {
    const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (e >= kP) return;
    float s = 0.0f;
#pragma unroll 8
    for (int c = 0; c < chunks; ++c) s += part[c * kP + e];
    g[e] = s;
    return;
  }
  __shared__ float red[8];
  float s = 0.0f;
  for (int64_t t = threadIdx.x; t < tiles; t += 256) s += tile_loss[t];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    s = 0.0f;
    for (int k = 0; k < 8; ++k) s += red[k];
    *loss = s;
  }
}

__global__ void adam_kernel(float* theta, __nv_bfloat16* thetab, const float* g, float* m, float* v, int64_t n, float lr,
                            float b1, float b2, float c1, float c2, float eps) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float t = theta[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    theta[i] = t;
    thetab[i] = __float2bfloat16_rn(t);
  }
}

__global__ void to_bf16_kernel(const float* x, __nv_bfloat16* y, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = __float2bfloat16_rn(x[i]);
}

unsigned blocks_for(int64_t n, int per) { return (unsigned)std::max<int64_t>(1, (n + per - 1) / per); }

}  // namespace
}  // namespace mka

struct mka_mlp {
  const uint64_t serial = mka::next_serial();
  float* theta = nullptr;          // FP32 master
  __nv_bfloat16* thetab = nullptr; // BF16 copy used by every product
  float* m = nullptr;
  float* v = nullptr;
  float* g = nullptr;
  float* loss = nullptr;
  int64_t t = 0;                   // Adam steps taken
  int64_t cap = 0;                 // batch capacity of the work buffers
  float* work = nullptr;           // H1, H2, dZ1, dZ2, dY, the tiles' losses, the chunks' gradients
};

namespace mka {

namespace {

template <bool GRAD>
mka_status rows_enqueue(const RowArgs& A, cudaStream_t st) {
  int dev = 0, sms = 0;
  MKA_CUDA_TRY(cudaGetDevice(&dev));
  MKA_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  mka_status s = allow_shared(reinterpret_cast<const void*>(mlp_rows_kernel<GRAD>), nullptr);
  if (s) return s;
  const unsigned grid = (unsigned)std::min<int64_t>((A.B + kTile - 1) / kTile, (int64_t)sms * 2);
  mlp_rows_kernel<GRAD><<<grid, kRowThreads, kRowSmem, st>>>(A);
  count_launches();
  MKA_CUDA_TRY(cudaGetLastError());
  return MKA_OK;
}

}  // namespace

uint64_t mlp_serial(const mka_mlp* net) { return net->serial; }

mka_status mlp_forward_enqueue(const mka_mlp* net, const float* X, int64_t B, float* Y, cudaStream_t st) {
  RowArgs A{};
  A.X = X;
  A.B = B;
  A.P = net->thetab;
  A.Y = Y;
  return rows_enqueue<false>(A, st);
}

mka_status features_enqueue(const mka_system* sys, const int64_t* d_sel, int64_t n, float* X, int32_t* patch,
                            cudaStream_t st) {
  FeatArgs A{};
  A.pos = sys->d_pos;
  A.posf = sys->d_posf;
  const double lmax = std::max(sys->box[0], std::max(sys->box[1], sys->box[2]));
  A.pre_hi = (float)(1.0 + std::max(1e-3, 1e-5 * lmax / 5.5));
  for (int d = 0; d < 3; ++d) {
    A.box[d] = sys->box[d];
    A.inv_box[d] = 1.0 / sys->box[d];
    A.ncell[d] = sys->cells.n[d];
    A.cell_len[d] = sys->cells.len[d];
  }
  A.cell_start = sys->cells.start;
  A.cell_atoms = sys->cells.atoms;
  A.sel = d_sel;
  A.n_sel = n;
  const double rg = std::min(5.5, std::min(sys->cells.len[0], std::min(sys->cells.len[1], sys->cells.len[2])));
  A.r_gather2 = rg * rg;
  A.X = X;
  A.patch = patch;
  features_kernel<<<blocks_for(n, 8), 256, 0, st>>>(A);
  count_launches();
  MKA_CUDA_TRY(cudaGetLastError());
  return MKA_OK;
}

}  // namespace mka

using namespace mka;

namespace {
mka_status mlp_reserve(mka_mlp* net, int64_t B) {
  if (B <= net->cap) return MKA_OK;
  cudaFree(net->work);
  net->work = nullptr;
  net->cap = 0;
  const int64_t floats = B * (4 * kHid + kOut) + (B + kTile - 1) / kTile + std::min<int64_t>(kMaxChunks, blocks_for(B, kGradRows)) * kP;
  MKA_CUDA_TRY(cudaMalloc(&net->work, sizeof(float) * floats));
  net->cap = B;
  return MKA_OK;
}

// forward + loss + backward into net->g (uses the BF16 weights), loss into net->loss[0]
mka_status mlp_grad_enqueue(mka_mlp* net, const float* X, const float* T, int64_t B, cudaStream_t st) {
  mka_status s = mlp_reserve(net, B);
  if (s) return s;
  RowArgs A{};
  A.X = X;
  A.T = T;
  A.B = B;
  A.P = net->thetab;
  A.inv = 1.0f / (float)(B * kOut);
  A.H1 = net->work;
  A.H2 = A.H1 + B * kHid;
  A.dZ1 = A.H2 + B * kHid;
  A.dZ2 = A.dZ1 + B * kHid;
  A.dY = A.dZ2 + B * kHid;
  A.loss = A.dY + B * kOut;
  s = rows_enqueue<true>(A, st);
  if (s) return s;
  const int64_t tiles = (B + kTile - 1) / kTile, chunk_rows = grad_chunk_rows(B);
  const int chunks = (int)((B + chunk_rows - 1) / chunk_rows);
  const GradArgs W{X, A.H1, A.H2, A.dZ1, A.dZ2, A.dY, B, chunk_rows, A.loss + tiles};
  grad_part_kernel<<<dim3(10, (unsigned)chunks), kGradThreads, 0, st>>>(W);
  grad_sum_kernel<<<blocks_for(kP, 256) + 1, 256, 0, st>>>(W.part, chunks, net->g, A.loss, tiles, net->loss);
  count_launches(2);
  MKA_CUDA_TRY(cudaGetLastError());
  return MKA_OK;
}
}  // namespace

extern "C" {

int64_t mka_mlp_num_params(void) { return kP; }

void mka_mlp_destroy(mka_mlp* net) {
  if (!net) return;
  cudaFree(net->theta);
  cudaFree(net->thetab);
  cudaFree(net->m);
  cudaFree(net->v);
  cudaFree(net->g);
  cudaFree(net->loss);
  cudaFree(net->work);
  delete net;
}

mka_status mka_mlp_create(uint64_t seed, mka_mlp** out) {
  if (!out) return fail(MKA_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  mka_mlp* net = new mka_mlp();
  cudaError_t e = cudaSuccess;
#define ALLOC(p, bytes) \
  if (e == cudaSuccess) e = cudaMalloc(&(p), (bytes))
  ALLOC(net->theta, sizeof(float) * kP);
  ALLOC(net->thetab, sizeof(__nv_bfloat16) * kP);
  ALLOC(net->m, sizeof(float) * kP);
  ALLOC(net->v, sizeof(float) * kP);
  ALLOC(net->g, sizeof(float) * kP);
  ALLOC(net->loss, sizeof(float) * 80);
#undef ALLOC
  if (e != cudaSuccess) {
    mka_mlp_destroy(net);
    return cuda_fail(e, "mka_mlp_create");
  }
  // He-uniform initialisation (weights U(-sqrt(6/fan_in), +)), zero biases, from a seeded mt19937_64
  std::vector<float> h(kP, 0.0f);
  std::mt19937_64 rng(seed);
  const int fan[3] = {kIn, kHid, kHid}, outd[3] = {kHid, kHid, kOut};
  const int64_t off[3] = {oW1, oW2, oW3};
  for (int l = 0; l < 3; ++l) {
    const double lim = std::sqrt(6.0 / fan[l]);
    std::uniform_real_distribution<double> U(-lim, lim);
    for (int64_t i = 0; i < (int64_t)fan[l] * outd[l]; ++i) h[off[l] + i] = (float)U(rng);
  }
  e = cudaMemcpy(net->theta, h.data(), sizeof(float) * kP, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(net->m, 0, sizeof(float) * kP);
  if (e == cudaSuccess) e = cudaMemset(net->v, 0, sizeof(float) * kP);
  if (e != cudaSuccess) {
    mka_mlp_destroy(net);
    return cuda_fail(e, "mka_mlp_create");
  }
  to_bf16_kernel<<<blocks_for(kP, 256), 256>>>(net->theta, net->thetab, kP);
  count_launches();
  e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    mka_mlp_destroy(net);
    return cuda_fail(e, "mka_mlp_create");
  }
  *out = net;
  return MKA_OK;
}

mka_status mka_mlp_set_params(mka_mlp* net, const float* host) {
  if (!net || !host) return fail(MKA_ERR_INVALID_ARG, "network and parameters are required");
  MKA_CUDA_TRY(cudaMemcpy(net->theta, host, sizeof(float) * kP, cudaMemcpyHostToDevice));
  MKA_CUDA_TRY(cudaMemset(net->m, 0, sizeof(float) * kP));
  MKA_CUDA_TRY(cudaMemset(net->v, 0, sizeof(float) * kP));
  net->t = 0;
  to_bf16_kernel<<<blocks_for(kP, 256), 256>>>(net->theta, net->thetab, kP);
  count_launches();
  MKA_CUDA_TRY(cudaDeviceSynchronize());
  return MKA_OK;
}

mka_status mka_mlp_get_params(const mka_mlp* net, float* host, int bf16_rounded) {
  if (!net || !host) return fail(MKA_ERR_INVALID_ARG, "network and output are required");
  if (!bf16_rounded) {
    MKA_CUDA_TRY(cudaMemcpy(host, net->theta, sizeof(float) * kP, cudaMemcpyDeviceToHost));
    return MKA_OK;
  }
  std::vector<uint16_t> b(kP);
  MKA_CUDA_TRY(cudaMemcpy(b.data(), net->thetab, sizeof(uint16_t) * kP, cudaMemcpyDeviceToHost));
  for (int64_t i = 0; i < kP; ++i) {
    const uint32_t u = (uint32_t)b[i] << 16;
    std::memcpy(&host[i], &u, 4);
  }
  return MKA_OK;
}

mka_status mka_mlp_forward(mka_mlp* net, const float* X, float* Y, int64_t B, void* stream) {
  if (!net || !X || !Y || B < 1) return fail(MKA_ERR_INVALID_ARG, "network, X, Y and B >= 1 are required");
  return mlp_forward_enqueue(net, X, B, Y, (cudaStream_t)stream);
}

mka_status mka_mlp_gradients(mka_mlp* net, const float* X, const float* T, int64_t B, float* grad, float* loss,
                             void* stream) {
  if (!net || !X || !T || B < 1) return fail(MKA_ERR_INVALID_ARG, "network, X, T and B >= 1 are required");
  cudaStream_t st = (cudaStream_t)stream;
  mka_status s = mlp_grad_enqueue(net, X, T, B, st);
  if (s) return s;
  if (grad) MKA_CUDA_TRY(cudaMemcpyAsync(grad, net->g, sizeof(float) * kP, cudaMemcpyDeviceToDevice, st));
  if (loss) MKA_CUDA_TRY(cudaMemcpyAsync(loss, net->loss, sizeof(float), cudaMemcpyDeviceToDevice, st));
  return MKA_OK;
}

mka_status mka_mlp_train_step(mka_mlp* net, const float* X, const float* T, int64_t B, float lr, float* loss,
                              void* stream) {
  if (!net || !X || !T || B < 1 || !(lr > 0)) return fail(MKA_ERR_INVALID_ARG, "bad training arguments");
  cudaStream_t st = (cudaStream_t)stream;
  mka_status s = mlp_grad_enqueue(net, X, T, B, st);
  if (s) return s;
  net->t += 1;
  const double b1 = 0.9, b2 = 0.999;
  const float c1 = (float)(1.0 - std::pow(b1, (double)net->t)), c2 = (float)(1.0 - std::pow(b2, (double)net->t));
  adam_kernel<<<blocks_for(kP, 256), 256, 0, st>>>(net->theta, net->thetab, net->g, net->m, net->v, kP, lr, (float)b1,
                                                   (float)b2, c1, c2, 1e-8f);
  count_launches();
  MKA_CUDA_TRY(cudaGetLastError());
  if (loss) MKA_CUDA_TRY(cudaMemcpyAsync(loss, net->loss, sizeof(float), cudaMemcpyDeviceToDevice, st));
  return MKA_OK;
}

mka_status mka_warm_start_features(const mka_system* sys, const int64_t* atoms, int64_t n, float* X, int32_t* patch,
                                   void* stream) {
  if (!sys || !atoms || n < 1 || !X || !patch) return fail(MKA_ERR_INVALID_ARG, "bad feature arguments");
  for (int64_t t = 0; t < n; ++t)
    if (atoms[t] < 0 || atoms[t] >= sys->n_atoms) return fail(MKA_ERR_INVALID_ARG, "atom index out of range");
  cudaStream_t st = (cudaStream_t)stream;
  int64_t* d_sel = nullptr;
  MKA_CUDA_TRY(cudaMallocAsync(&d_sel, sizeof(int64_t) * n, st));
  MKA_CUDA_TRY(cudaMemcpyAsync(d_sel, atoms, sizeof(int64_t) * n, cudaMemcpyHostToDevice, st));
  mka_status s = features_enqueue(sys, d_sel, n, X, patch, st);
  cudaFreeAsync(d_sel, st);
  return s;
}

mka_status mka_system_set_warm_start(mka_system* sys, mka_mlp* net) {
  if (!sys) return fail(MKA_ERR_INVALID_ARG, "system is NULL");
  sys->warm = net;
  return MKA_OK;
}

}  // extern "C"
