// The per-atom solve with a CTA for each of the atom's four columns: FP64, for selections too small to fill the chip.
//
// The kernels that take an atom's four columns together read every block once for the four, which is the better way
// where there are atoms enough: at FP64 an SM works off two lanes a cycle, and one atom's products, orthogonalisation
// and projection are 36 ms of them at nu = 100 (640 rows) whatever the other 151 SMs do; 8.4 with a CTA a column (1.6
// against 4.8 at nu = 30). The columns of an atom are independent, so up to a CTA per SM their four parts run side by
// side. The steps are the general kernel's (columns.cu) for one column: CG for s_j, then one classical Gram-Schmidt pass
// with the Gram correction c - E c a vector, the previous vector's projection in the same sweep; the sums' order differs.
// A row is a thread's in all of them: 640 rows are five warps to a scheduler, enough to hide the FP64 pipe's latency.
#include "atoms.cuh"

namespace mka {
namespace {

constexpr int kThreads = 512, kWarps = kThreads / 32;

struct SingleState {
  double rr, alpha, beta, csum;
  int n, src, seam_done, active, status, it, proj, accept, act, next_s, t0, fits;
};

// f(sum of v over the CTA) by thread 0; its effects are seen by all threads afterwards.
template <typename F>
__device__ __forceinline__ void cta_total(double v, double* red, F f) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  v = warp_sum(v);
  if (lane == 0) red[wid] = v;
  __syncthreads();
  if (wid == 0) {
    double s = lane < kWarps ? red[lane] : 0.0;
#pragma unroll
    for (int o = kWarps / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) f(s);
  }
  __syncthreads();
}

// Sums of three values over the warp with 6 additions: a's in lane 0, b's in lane 8, c's in lane 16.
__device__ __forceinline__ double warp_sum3(double a, double b, double c) {
  const int lane = threadIdx.x & 31;
  const bool b16 = lane & 16, b8 = lane & 8;
  const double a0 = (b16 ? c : a) + __shfl_xor_sync(0xffffffffu, b16 ? a : c, 16);
  const double a1 = (b16 ? 0.0 : b) + __shfl_xor_sync(0xffffffffu, b16 ? b : 0.0, 16);
  double r = (b8 ? a1 : a0) + __shfl_xor_sync(0xffffffffu, b8 ? a0 : a1, 8);
  r += __shfl_xor_sync(0xffffffffu, r, 4);
  r += __shfl_xor_sync(0xffffffffu, r, 2);
  r += __shfl_xor_sync(0xffffffffu, r, 1);
  return r;
}

// (A x) of row i of the cluster atom with blocks [e0, e1)
template <typename TV>
__device__ __forceinline__ double row_product(const TV* __restrict__ val, int rb, int e0, int e1, const uint16_t* lcol,
                                              const uint8_t* loff, int i, const double* x) {
  double a = 0.0;
#pragma unroll 4
  for (int e = e0; e < e1; ++e) {
    double v[4], xk[4];
    RowLoad<TV, double>::load(val, rb + loff[e], i, v);
    ld4(x + 4 * lcol[e], xk);
#pragma unroll
    for (int k = 0; k < 4; ++k) a = fma(v[k], xk[k], a);
  }
  return a;
}

template <typename TV>
__global__ void __launch_bounds__(kThreads, 2) single_kernel(const Args<TV> A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ SingleState st;
  __shared__ double red[kWarps];
  __shared__ int cnt;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int nu = A.nu, mcap = A.mcap, c = blockIdx.x & 3;
  const int64_t widx = blockIdx.x >> 2, col = 4 * widx + c, atom = A.sel[widx];
  int* cl = reinterpret_cast<int*>(smem_raw);                            // clcap
  int* lrow = cl + A.clcap;                                               // clcap + 1
  int* rbase = lrow + A.clcap + 1;                                        // clcap
  uint16_t* lcol = reinterpret_cast<uint16_t*>(rbase + A.clcap);          // lnnz_cap
  uint8_t* loff = reinterpret_cast<uint8_t*>(lcol + A.lnnz_cap);          // lnnz_cap
  size_t off = (size_t)(3 * A.clcap + 1) * sizeof(int) + (size_t)A.lnnz_cap * (sizeof(uint16_t) + 1);
  off = (off + 15) & ~(size_t)15;
  double* L = reinterpret_cast<double*>(smem_raw + off);   // p, then l
  double *SL = L + mcap, *KV = SL + mcap;                  // S p, then S l and S u; r, then H l and H u
  double *coef = KV + mcap, *coefT = coef + nu;
  char* slot = A.scratch + (size_t)blockIdx.x * A.slot_bytes;
  double* U = reinterpret_cast<double*>(slot);             // [nu][mcap]
  double *SU = U + (size_t)nu * mcap, *SJ = SU + (size_t)nu * mcap;
  float* Es = reinterpret_cast<float*>(SJ + mcap);         // S_r - I, [nu][nu]
  const int nrow = A.row_ptr[atom + 1] - A.row_ptr[atom];
  double* vpa = A.keep ? A.vp + A.blk_off[widx] * 16 * (int64_t)nu : nullptr;
  if (A.keep)                                              // the column's pattern rows of U: zero outside the cluster
    for (int i = tid; i < nrow * 4 * nu; i += kThreads)
      vpa[((int64_t)(i / (4 * nu)) * 16 + 4 * c) * nu + i % (4 * nu)] = 0.0;

  // ---- cluster and its block pattern
  const int ncl = gather_cluster(A, atom, cl, &cnt);
  bool fits = ncl <= A.clcap && 4 * ncl <= mcap;
  if (fits) {
    sort_cluster(cl, ncl);
    for (int t = tid; t < ncl; t += kThreads) {
      const int b = cl[t];
      int k = 0;
      for (int e = A.row_ptr[b]; e < A.row_ptr[b + 1]; ++e) k += find_local(cl, ncl, A.col[e]) >= 0;
      lrow[t + 1] = k;
    }
    __syncthreads();
    if (tid == 0) {
      lrow[0] = 0;
      for (int t = 0; t < ncl; ++t) lrow[t + 1] += lrow[t];
      st.t0 = find_local(cl, ncl, (int)atom);
      st.fits = lrow[ncl] <= A.lnnz_cap;
    }
    __syncthreads();
    fits = st.fits;
  }
  if (!fits) {
    if (tid == 0) {
      A.status[col] = ST_TOOLARGE;
      A.nu_eff[col] = 0;
      A.cg_iters[col] = 0;
    }
    return;
  }
  for (int t = tid; t < ncl; t += kThreads) {
    const int b = cl[t], k0 = A.row_ptr[b];
    int e = lrow[t];
    rbase[t] = k0;
    for (int k = k0; k < A.row_ptr[b + 1]; ++k) {
      const int lc = find_local(cl, ncl, A.col[k]);
      if (lc >= 0) {
        lcol[e] = (uint16_t)lc;
        loff[e] = (uint8_t)(k - k0);
        ++e;
      }
    }
  }
  const int m = 4 * ncl, j = 4 * st.t0 + c;
  // ---- inner CG: S s = e_j
  for (int r = tid; r < m; r += kThreads) {
    L[r] = KV[r] = r == j ? 1.0 : 0.0;
    SJ[r] = 0.0;
  }
  if (tid == 0) {
    st.rr = 1.0;
    st.it = 0;
    st.status = ST_OK;
    st.active = 1.0 > A.cg_tol;
  }
  __syncthreads();
  for (int it = 0; it < A.cg_maxit && st.active; ++it) {
    double part = 0.0;
    for (int r = tid; r < m; r += kThreads) {
      const double s = row_product<TV>(A.valS, rbase[r >> 2], lrow[r >> 2], lrow[(r >> 2) + 1], lcol, loff, r & 3, L);
      SL[r] = s;
      part = fma(L[r], s, part);
    }
    cta_total(part, red, [&](double s) {
      if (s > 0.0) st.alpha = st.rr / s;
      else {
        st.status = ST_NOT_SPD;
        st.active = 0;
      }
    });
    if (!st.active) break;
    const double al = st.alpha;
    part = 0.0;
    for (int r = tid; r < m; r += kThreads) {
      const double v = fma(-al, SL[r], KV[r]);
      SJ[r] = fma(al, L[r], SJ[r]);
      KV[r] = v;
      part = fma(v, v, part);
    }
    cta_total(part, red, [&](double s) {
      st.beta = s / st.rr;
      st.rr = s;
      st.it += 1;
      if (sqrt(s) <= A.cg_tol) st.active = 0;
    });
    const double be = st.beta;
    if (st.active)
      for (int r = tid; r < m; r += kThreads) L[r] = fma(be, L[r], KV[r]);
    __syncthreads();
  }
  __syncthreads();     // every thread has seen st.active for the last time
  // ---- basis, with the projection accumulated on the way
  if (tid == 0) {
    if (st.active && st.status == ST_OK) st.status = ST_NOCONV;
    st.n = 0;
    st.src = SRC_E;
    st.seam_done = A.q == 0;
    st.active = st.status == ST_OK;
    st.proj = 0;
    st.csum = 0.0;
  }
  for (int r = tid; r < m; r += kThreads) L[r] = r == j ? 1.0 : 0.0;
  __syncthreads();
  double* Hr = A.red + (size_t)(col >> 5) * red_block_doubles(nu) * 32 + (col & 31);
  double* Sr = Hr + (size_t)nu * nu * 32;
  // coef = (S U)^T l, and column n - 1 of H_r, S_r and E from H u, S u of the last vector (a warp per vector)
  auto sweep = [&](int n, bool proj) {
    for (int mm = wid; mm < n; mm += kWarps) {
      const double *su = SU + (size_t)mm * mcap, *u = U + (size_t)mm * mcap;
      double pc = 0.0, ph = 0.0, ps = 0.0;
      if (proj) {
#pragma unroll 4
        for (int r = lane; r < m; r += 32) {
          const double uv = u[r];
          pc = fma(su[r], L[r], pc);
          ph = fma(uv, KV[r], ph);
          ps = fma(uv, SL[r], ps);
        }
      } else {
#pragma unroll 4
        for (int r = lane; r < m; r += 32) pc = fma(su[r], L[r], pc);
      }
      const double s = warp_sum3(pc, ph, ps);
      if (lane == 0) coef[mm] = s;
      if (proj && lane == 8) Hr[(size_t)(mm * nu + n - 1) * 32] = Hr[(size_t)((n - 1) * nu + mm) * 32] = s;
      if (proj && lane == 16) {
        Sr[(size_t)(mm * nu + n - 1) * 32] = Sr[(size_t)((n - 1) * nu + mm) * 32] = s;
        Es[mm * nu + n - 1] = Es[(n - 1) * nu + mm] = (float)(s - (mm == n - 1 ? 1.0 : 0.0));
      }
    }
    __syncthreads();
  };
  for (int guard = 0; guard < nu + 4 && st.active; ++guard) {
    const int n = st.n;
    if (n > 0) {
      sweep(n, st.proj);
      for (int mm = tid; mm < n; mm += kThreads) {
        double corr = 0.0;
        for (int k = 0; k < n; ++k) corr = fma(widen(Es[k * nu + mm]), coef[k], corr);
        coefT[mm] = coef[mm] - corr;
      }
      if (wid == kWarps - 1) {
        double s = 0.0;
        for (int k = lane; k < n; k += 32) s = fma(coef[k], coef[k], s);
        s = warp_sum(s);
        if (lane == 0) st.csum = s;
      }
      __syncthreads();
      for (int r = tid; r < m; r += kThreads) {
        double v = L[r], v1 = 0.0;
        int mm = 0;
#pragma unroll 4
        for (; mm + 1 < n; mm += 2) {
          v = fma(-coefT[mm], U[(size_t)mm * mcap + r], v);
          v1 = fma(-coefT[mm + 1], U[(size_t)(mm + 1) * mcap + r], v1);
        }
        if (mm < n) v = fma(-coefT[mm], U[(size_t)mm * mcap + r], v);
        L[r] = v + v1;
      }
      __syncthreads();
    }
    double part = 0.0;
    for (int r = tid; r < m; r += kThreads) {
      const int rb = rbase[r >> 2], e0 = lrow[r >> 2], e1 = lrow[(r >> 2) + 1];
      double h = 0.0, s = 0.0;
#pragma unroll 2
      for (int e = e0; e < e1; ++e) {
        double vh[4], vs[4], xk[4];
        RowLoad<TV, double>::load(A.valH, rb + loff[e], r & 3, vh);
        RowLoad<TV, double>::load(A.valS, rb + loff[e], r & 3, vs);
        ld4(L + 4 * lcol[e], xk);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          h = fma(vh[k], xk[k], h);
          s = fma(vs[k], xk[k], s);
        }
      }
      KV[r] = h;
      SL[r] = s;
      part = fma(L[r], s, part);
    }
    cta_total(part, red, [&](double s) {
      const double b2 = fmax(s, 0.0), beta = sqrt(b2);
      st.accept = st.next_s = 0;
      st.act = ACT_NONE;
      if (beta > A.tau * sqrt(b2 + st.csum)) {
        st.accept = 1;
        st.alpha = 1.0 / beta;
        st.n = n + 1;
        if (n + 1 >= nu) {
          st.active = 0;
        } else if (n + 1 == A.p && !st.seam_done) {
          st.next_s = 1;                // the vector after u_p is s_j
          st.seam_done = 1;
          st.src = SRC_S;
        } else {
          st.src = SRC_H;
        }
      } else if (st.src == SRC_S && n > 0) {
        st.act = ACT_LOAD_K;            // s_j already in the span: continue with H u_n
        st.src = SRC_H;
      } else if (!st.seam_done) {
        st.act = ACT_LOAD_S;            // first chain closed early: start the second chain
        st.src = SRC_S;
        st.seam_done = 1;
      } else {
        st.active = 0;                  // basis ends with nu_eff = n
      }
      st.proj = st.accept;
      st.csum = 0.0;
    });
    if (st.accept) {
      const double bi = st.alpha;
      const bool next_s = st.next_s;
      for (int r = tid; r < m; r += kThreads) {
        const double u = L[r] * bi, k = KV[r] * bi, su = SL[r] * bi;
        U[(size_t)n * mcap + r] = u;
        SU[(size_t)n * mcap + r] = su;
        KV[r] = k;
        SL[r] = su;
        L[r] = next_s ? SJ[r] : k;
      }
    } else if (st.act == ACT_LOAD_K) {
      for (int r = tid; r < m; r += kThreads) L[r] = U[(size_t)(n - 1) * mcap + r];
      __syncthreads();
      for (int r = tid; r < m; r += kThreads)
        KV[r] = row_product<TV>(A.valH, rbase[r >> 2], lrow[r >> 2], lrow[(r >> 2) + 1], lcol, loff, r & 3, L);
      __syncthreads();
      for (int r = tid; r < m; r += kThreads) L[r] = KV[r];
    } else if (st.act == ACT_LOAD_S) {
      for (int r = tid; r < m; r += kThreads) L[r] = SJ[r];
    }
    __syncthreads();
  }
  const int n = st.n;
  if (st.proj) sweep(n, true);          // the last vector's projection
  // ---- row j of U and S U, and the pattern rows
  double* rows = Hr + (size_t)2 * nu * nu * 32;
  for (int i = tid; i < 2 * nu; i += kThreads)
    if (i % nu < n) rows[(size_t)i * 32] = (i < nu ? U : SU)[(size_t)(i % nu) * mcap + j];
  if (tid == 0) {
    A.status[col] = st.status;
    A.nu_eff[col] = n;
    A.cg_iters[col] = st.it;
  }
  if (A.keep) {
    const int e0 = lrow[st.t0], ne = lrow[st.t0 + 1] - e0;
    for (int i = tid; i < 4 * ne * n; i += kThreads) {
      const int k = i % n, er = i / n, e = e0 + er / 4, r = er % 4;
      vpa[((int64_t)loff[e] * 16 + c * 4 + r) * nu + k] = U[(size_t)k * mcap + 4 * lcol[e] + r];
    }
  }
}

size_t single_smem(int nu, const AtomsConfig& cf) {
  return align_up((size_t)(3 * cf.clcap + 1) * sizeof(int) + (size_t)cf.lnnz_cap * (sizeof(uint16_t) + 1), 16) +
         sizeof(double) * (3 * (size_t)cf.mcap + 2 * (size_t)nu);
}

size_t single_slot(int nu, const AtomsConfig& cf) {
  return align_up(sizeof(double) * (2 * (size_t)nu + 1) * cf.mcap + sizeof(float) * (size_t)nu * nu, 16);
}

template <typename TV>
mka_status single_config_t(int nu, AtomsConfig* cf) {
  size_t most = 0;
  mka_status s = allow_shared(reinterpret_cast<const void*>(single_kernel<TV>), &most);
  if (s) return s;
  int dev = 0, sms = 0;
  MKA_CUDA_TRY(cudaGetDevice(&dev));
  MKA_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // four columns' slots lie in one atom's slot of the general kernel
  if (single_smem(nu, *cf) > most || 4 * single_slot(nu, *cf) > cf->slot_bytes) return MKA_OK;
  // Levels in ms, this kernel against the others: nu = 30 (short recurrences) 1 atom 2.8 / 5.9, 114 6.0 / 6.9, 152 7.4 / 7.1,
  // 300 13.9 / 12.1; nu = 100 (general kernel) 1 atom 20 / 42, 38 21 / 49, 228 85 / 99, 300 112 / 114.
  cf->single_max = std::min(cf->grid_max, cf->chains ? sms * 3 / 4 : sms * 3 / 2);
  return MKA_OK;
}

template <typename TV>
mka_status single_launch_t(const mka_system* sys, const AtomsConfig& cf, const AtomsLaunchArgs& a, cudaStream_t st) {
  Args<TV> A{};
  fill_args(A, sys, cf, a);
  A.slot_bytes = single_slot(A.nu, cf);
  single_kernel<TV><<<(unsigned)(4 * a.n_sel), kThreads, single_smem(A.nu, cf), st>>>(A);
  count_launches();
  MKA_CUDA_TRY(cudaGetLastError());
  return MKA_OK;
}

}  // namespace

mka_status single_config(const mka_system* sys, int nu, AtomsConfig* cf) {
  return sys->storage == MKA_FP64         ? single_config_t<double>(nu, cf)
         : sys->storage == MKA_MIXED_FP32 ? single_config_t<float>(nu, cf)
                                          : single_config_t<__nv_bfloat16>(nu, cf);
}

mka_status single_launch(const mka_system* sys, const AtomsConfig& cf, const AtomsLaunchArgs& a, cudaStream_t st) {
  return sys->storage == MKA_FP64         ? single_launch_t<double>(sys, cf, a, st)
         : sys->storage == MKA_MIXED_FP32 ? single_launch_t<float>(sys, cf, a, st)
                                          : single_launch_t<__nv_bfloat16>(sys, cf, a, st);
}

}  // namespace mka
