// Batched reduced problems of the multiple Arnoldi method on sm_103a.
//
// Every column j ends its basis with the nu x nu projected matrices H_r = U^T H U and
// S_r = U^T S U (formed explicitly, so that a basis that is only nearly S-orthonormal
// still gives the Galerkin pencil of its span) and solves the generalized eigenproblem
// H_r c = eps S_r c (Eq. EQ-SUB-EIG-VEC): Cholesky S_r = L L^T, A = L^{-1} H_r L^{-T} (lower
// triangle), Householder tridiagonalisation A = Q T Q^T, the eigenvalues of T by the
// implicit-shift QL method, the eigenvectors Z of T by inverse iteration (re-orthogonalised
// within clusters of close eigenvalues), C = L^{-T} Q Z with Q applied as its reflectors. The
// outputs of a column are its levels eps_alpha in ascending order, w_alpha = V_{j alpha} (S V)_{j alpha} with V = U C (Eq. EQ-DM's
// weights), and, when vectors are kept, C and the row V_j = (row j of U) C in the same order:
// rho_ij = sum_alpha f_alpha V_i alpha V_j alpha = U_i . (C diag(f) V_j) and G_ij(z) likewise,
// so the kept pattern rows of U never need turning into rows of V.
//
// These solves are short chains of dependent FP64 operations (square roots, divisions,
// the QL recurrence), and the FP64 pipe of an SM issues one warp instruction every 16
// cycles. One lane per column makes every FP64 instruction serve 32 columns: the lane
// runs the textbook sequential algorithm on its own column, its matrices held in a
// lane-interleaved global buffer (element e of the lane's block at e * 32 + lane) so that
// the warp's accesses to the same element coalesce, its vectors in local memory.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "mka_internal.h"
#include "reduced_rule.cuh"

namespace mka {
namespace {

enum : int { RS_OK = 0, RS_NOT_SPD = MKA_ERR_NOT_SPD, RS_BREAKDOWN = MKA_ERR_BREAKDOWN };
constexpr int kTinyNu = 32, kSmallNu = 64;

struct RedArgs {
  double* blk;               // [groups][red_block_doubles(nu)][32], in place
  int64_t n_cols;
  int nu;
  int32_t* status;           // in: status after the basis; out: final status
  int32_t* nu_eff;           // in: basis size; out: subspace dimension used (0 on failure)
  double* eps;               // [n_cols][nu]
  double* w;                 // [n_cols][nu]
  double* cv;                // kept C and V_j (NULL: not kept), lane-interleaved by column col0 + col
  int64_t col0;
};

// Element (i, j) of the lane's matrices: H_r, then X = L^{-1} H_r (upper triangle) and A (lower
// triangle), then Q's reflectors (below the diagonal) at (i nu + j); S_r / L at nu^2 + (i nu + j);
// row j of U and of S U; the eigenvectors Z of T, then C, at 2 nu^2 + 2 nu + (i nu + j).
struct Lane {
  double* b;
  int nu;
  __device__ double& H(int i, int j) const { return b[(size_t)(i * nu + j) * 32]; }
  __device__ double& S(int i, int j) const { return b[(size_t)(nu * nu + i * nu + j) * 32]; }
  __device__ double UJ(int n) const { return b[(size_t)(2 * nu * nu + n) * 32]; }
  __device__ double SUJ(int n) const { return b[(size_t)(2 * nu * nu + nu + n) * 32]; }
  __device__ double& Z(int i, int j) const { return b[(size_t)(2 * nu * nu + 2 * nu + i * nu + j) * 32]; }
};

// A lane's vector in shared memory, `step` entries apart.
struct Strided {
  double* p;
  int step;
  __device__ double& operator[](int k) const { return p[k * step]; }
};

// S_r = L L^T in the lower triangle of S (right-looking); rdiag[k] = 1 / L_kk.
__device__ bool lane_cholesky(const Lane& M, int n, double* rdiag) {
  for (int k = 0; k < n; ++k) {
    const double akk = M.S(k, k);
    if (!(akk > 0.0)) return false;
    const double lkk = sqrt(akk);
    const double rd = 1.0 / lkk;
    rdiag[k] = rd;
    M.S(k, k) = lkk;
    for (int i = k + 1; i < n; ++i) M.S(i, k) *= rd;
    for (int i = k + 1; i < n; ++i) {
      const double lik = M.S(i, k);
      for (int j = k + 1; j <= i; ++j) M.S(i, j) -= lik * M.S(j, k);
    }
  }
  return true;
}

// The lower triangle of A = L^{-1} H L^{-T} in place of H's, using the symmetry of H and A (n^3 / 2
// FMAs): first the upper triangle of X = L^{-1} H over H's (row j from the rows above it), then A =
// L^{-1} X^T column by column, the entries of column j above the diagonal taken from row j of A. `row`
// and `col` (n doubles each, lane-local) hold the row of L and the column of A an inner loop reuses.
__device__ void lane_congruence(const Lane& M, int n, const double* rdiag, double* row, double* col) {
  for (int j = 0; j < n; ++j) {        // X(j, i), i >= j
    for (int k = 0; k < j; ++k) row[k] = M.S(j, k);
    for (int i = j; i < n; ++i) {
      double v = M.H(j, i);
      for (int k = 0; k < j; ++k) v -= row[k] * M.H(k, i);
      M.H(j, i) = v * rdiag[j];
    }
  }
  for (int j = 0; j < n; ++j) {        // A(i, j), i >= j
    for (int k = 0; k < j; ++k) col[k] = M.H(j, k);
    for (int i = j; i < n; ++i) {
      double v = M.H(j, i);
      for (int k = 0; k < i; ++k) v -= M.S(i, k) * col[k];
      col[i] = v * rdiag[i];
    }
    for (int i = j; i < n; ++i) M.H(i, j) = col[i];
  }
}

// Householder reduction T = Q^T A Q of A given by its lower triangle: diagonal d, off-diagonal e
// (e[k] couples k, k+1; e[n-1] = 0). Q = H_0 H_1 ... H_{n-3} is kept as its reflectors
// H_k = I - tau[k] v_k v_k^T, v_k in column k below the diagonal (rows k+1..n-1). v (n doubles,
// lane-local) holds the current Householder vector.
__device__ void lane_tridiag(const Lane& M, int n, double* d, double* e, double* p, double* tau, double* v) {
  for (int k = 0; k + 2 < n; ++k) {
    double s2 = 0.0;
    for (int i = k + 1; i < n; ++i) {
      v[i] = M.H(i, k);
      s2 += v[i] * v[i];
    }
    const double x0 = v[k + 1];
    const double nrm = sqrt(s2);
    const double alpha = x0 >= 0.0 ? -nrm : nrm;
    const double v0 = x0 - alpha;
    const double vtv = s2 - x0 * x0 + v0 * v0;
    const double tk = vtv > 0.0 ? 2.0 / vtv : 0.0;          // H_k = I - tk v v^T
    v[k + 1] = v0;
    M.H(k + 1, k) = v0;                                       // v = A[k+1.., k]
    d[k] = M.H(k, k);
    e[k] = alpha;
    tau[k] = tk;
    double pv = 0.0;
    for (int i = k + 1; i < n; ++i) {                         // p = tk B v, B from its lower triangle
      double acc = 0.0;
      for (int j = k + 1; j <= i; ++j) acc += M.H(i, j) * v[j];
      for (int j = i + 1; j < n; ++j) acc += M.H(j, i) * v[j];
      p[i] = tk * acc;
      pv += p[i] * v[i];
    }
    const double kc = 0.5 * tk * pv;
    for (int i = k + 1; i < n; ++i) p[i] -= kc * v[i];        // w = p - kc v
    for (int i = k + 1; i < n; ++i) {                         // B -= v w^T + w v^T, lower triangle
      const double vi = v[i], wi = p[i];
      for (int j = k + 1; j <= i; ++j) M.H(i, j) -= vi * p[j] + wi * v[j];
    }
  }
  if (n >= 2) {
    d[n - 2] = M.H(n - 2, n - 2);
    e[n - 2] = M.H(n - 1, n - 2);
  }
  d[n - 1] = M.H(n - 1, n - 1);
  e[n - 1] = 0.0;
}

// Eigenvalues of the tridiagonal (d, e) by the implicit-shift QL method (Bowdler, Martin,
// Reinsch & Wilkinson, Numer. Math. 11, 1968), in place on d (e is destroyed); rotation
// lengths from rsqrt(f^2 + g^2). False when an eigenvalue needs more than 60 sweeps.
template <typename V>
__device__ bool lane_tql_values(int n, V d, V e) {
  for (int l = 0; l < n; ++l) {
    for (int iter = 0;; ++iter) {
      int m = l;
      for (; m < n - 1; ++m) {
        const double dd = fabs(d[m]) + fabs(d[m + 1]);
        if (fabs(e[m]) <= 2.2204460492503131e-16 * dd) break;
      }
      if (m == l) break;
      if (iter == 60) return false;
      double g = (d[l + 1] - d[l]) / (2.0 * e[l]);
      double r = sqrt(g * g + 1.0);
      g = d[m] - d[l] + e[l] / (g + (g >= 0.0 ? r : -r));
      double s = 1.0, c = 1.0, p = 0.0;
      bool early = false;
      for (int i = m - 1; i >= l; --i) {
        const double f = s * e[i], b = c * e[i];
        const double t = f * f + g * g;
        if (t == 0.0) {
          e[i + 1] = 0.0;
          d[i + 1] -= p;
          e[m] = 0.0;
          early = true;
          break;
        }
        const double rinv = rsqrt(t);
        e[i + 1] = t * rinv;
        s = f * rinv;
        c = g * rinv;
        g = d[i + 1] - p;
        r = (d[i] - g) * s + 2.0 * c * b;
        p = s * r;
        d[i + 1] = g + p;
        g = c * r - b;
      }
      if (!early) {
        d[l] -= p;
        e[l] = g;
        e[m] = 0.0;
      }
    }
  }
  return true;
}

// Ascending.
template <typename V>
__device__ void lane_sort(int n, V d) {
  for (int a = 1; a < n; ++a) {
    const double t = d[a];
    int b = a - 1;
    for (; b >= 0 && d[b] > t; --b) d[b + 1] = d[b];
    d[b + 1] = t;
  }
}

// Gaussian elimination with partial pivoting of the tridiagonal T - lam I (d, e): the multipliers and
// row interchanges in (mlt, swp), U as reciprocal pivots r0 and the two superdiagonals (u1, u2); a
// pivot that vanishes is replaced by `tiny`. One division per row.
template <typename V>
__device__ void lane_tri_factor(int n, V d, V e, double lam, double tiny, double* r0, double* u1, double* u2,
                                double* mlt, int* swp) {
  double a = d[0] - lam, bb = n > 1 ? e[0] : 0.0;   // the working row: a at column k, bb at k + 1
  for (int k = 0; k + 1 < n; ++k) {
    const double sub = e[k], dn = d[k + 1] - lam, sp = k + 2 < n ? e[k + 1] : 0.0;
    if (fabs(a) >= fabs(sub)) {
      const double ra = 1.0 / (a != 0.0 ? a : tiny);
      mlt[k] = sub * ra;
      swp[k] = 0;
      r0[k] = ra;
      u1[k] = bb;
      u2[k] = 0.0;
      a = dn - mlt[k] * bb;
      bb = sp;
    } else {                               // row k + 1 becomes the pivot row
      const double rs = 1.0 / sub;
      mlt[k] = a * rs;
      swp[k] = 1;
      r0[k] = rs;
      u1[k] = dn;
      u2[k] = sp;
      a = bb - mlt[k] * dn;
      bb = -mlt[k] * sp;
    }
  }
  r0[n - 1] = 1.0 / (a != 0.0 ? a : tiny);
}

// x <- (T - lam I)^{-1} x from the factors of lane_tri_factor: the row operations, then back substitution.
__device__ void lane_tri_apply(int n, const double* r0, const double* u1, const double* u2, const double* mlt,
                               const int* swp, double* x) {
  for (int k = 0; k + 1 < n; ++k) {
    if (swp[k]) {
      const double xk = x[k];
      x[k] = x[k + 1];
      x[k + 1] = xk - mlt[k] * x[k + 1];
    } else {
      x[k + 1] -= mlt[k] * x[k];
    }
  }
  x[n - 1] *= r0[n - 1];
  if (n >= 2) x[n - 2] = (x[n - 2] - u1[n - 2] * x[n - 1]) * r0[n - 2];
  for (int k = n - 3; k >= 0; --k) x[k] = (x[k] - u1[k] * x[k + 1] - u2[k] * x[k + 2]) * r0[k];
}

// The eigenvectors of the tridiagonal (d, e) for its eigenvalues lam[0..n) (ascending) by inverse
// iteration (Wilkinson; the scheme of LAPACK's dstein): from a fixed quasi-random start, two solves
// of (T - lam_a I) x = x with one factorisation, each followed by modified Gram-Schmidt against the vectors of the same
// cluster already found (eigenvalues closer than 1e-3 ||T||_1 to their neighbour) and
// normalisation; stored as the columns of Z.
__device__ void lane_tri_vectors(const Lane& M, int n, const double* d, const double* e, const double* lam,
                                 double* x, double* r0, double* u1, double* u2, double* mlt, int* swp) {
  double tn = 0.0;
  for (int k = 0; k < n; ++k)
    tn = fmax(tn, fabs(d[k]) + (k + 1 < n ? fabs(e[k]) : 0.0) + (k > 0 ? fabs(e[k - 1]) : 0.0));
  const double ortol = 1e-3 * tn, tiny = 2.2204460492503131e-16 * (tn > 0.0 ? tn : 1.0);
  int cs = 0;
  for (int a = 0; a < n; ++a) {
    if (a == 0 || lam[a] - lam[a - 1] > ortol) cs = a;
    for (int i = 0; i < n; ++i) {        // start: an additive-recurrence (golden ratio) sequence in [0.5, 1.5)
      const double t = 0.7548776662466927 * (i + 1) + 0.5698402909980532 * (a + 1);
      x[i] = 0.5 + (t - floor(t));
    }
    lane_tri_factor(n, d, e, lam[a], tiny, r0, u1, u2, mlt, swp);
    for (int it = 0; it < 2; ++it) {
      lane_tri_apply(n, r0, u1, u2, mlt, swp, x);
      for (int b = cs; b < a; ++b) {
        double dot = 0.0;
        for (int i = 0; i < n; ++i) dot += M.Z(i, b) * x[i];
        for (int i = 0; i < n; ++i) x[i] -= dot * M.Z(i, b);
      }
      double s2 = 0.0;
      for (int i = 0; i < n; ++i) s2 += x[i] * x[i];
      const double sc = s2 > 0.0 ? 1.0 / sqrt(s2) : 0.0;
      for (int i = 0; i < n; ++i) x[i] *= sc;
    }
    for (int i = 0; i < n; ++i) M.Z(i, a) = x[i];
  }
}

// C = L^{-T} Q Z in place of Z, four columns at a time: the reflectors of Q applied to the block
// (H_{n-3} first), then the back substitution with L^T.
template <int NUCAP>
__device__ void lane_back_transform(const Lane& M, int n, const double* rdiag, const double* tau,
                                    double (*x4)[NUCAP]) {
  for (int a0 = 0; a0 < n; a0 += 4) {
    const int na = min(4, n - a0);
    for (int r = 0; r < 4; ++r)
      for (int k = 0; k < n; ++k) x4[r][k] = r < na ? M.Z(k, a0 + r) : 0.0;
    for (int k = n - 3; k >= 0; --k) {   // x <- (I - tau_k v_k v_k^T) x
      const double tk = tau[k];
      if (tk == 0.0) continue;
      double dot[4] = {0.0, 0.0, 0.0, 0.0};
      for (int i = k + 1; i < n; ++i) {
        const double vi = M.H(i, k);
#pragma unroll
        for (int r = 0; r < 4; ++r) dot[r] += vi * x4[r][i];
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) dot[r] *= tk;
      for (int i = k + 1; i < n; ++i) {
        const double vi = M.H(i, k);
#pragma unroll
        for (int r = 0; r < 4; ++r) x4[r][i] -= dot[r] * vi;
      }
    }
    for (int i = n - 1; i >= 0; --i) {   // C = L^{-T} (Q Z)
      double s[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) s[r] = x4[r][i];
      for (int k = i + 1; k < n; ++k) {
        const double l = M.S(k, i);
#pragma unroll
        for (int r = 0; r < 4; ++r) s[r] -= l * x4[r][k];
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) x4[r][i] = s[r] * rdiag[i];
    }
    for (int r = 0; r < na; ++r)
      for (int i = 0; i < n; ++i) M.Z(i, a0 + r) = x4[r][i];
  }
}

// NUCAP bounds nu: the lane's vectors live in local memory sized NUCAP, so subspaces up to 32 and 64
// take the small instances and larger ones (up to MKA_MAX_NU) the large one.
template <int NUCAP>
__global__ void __launch_bounds__(128) reduced_kernel(const RedArgs A) {
  const int64_t col = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= A.n_cols) return;
  const int nu = A.nu;
  const Lane M{A.blk + (size_t)(col >> 5) * red_block_doubles(nu) * 32 + (col & 31), nu};
  double d[NUCAP], e[NUCAP], rdiag[NUCAP], p[NUCAP], tau[NUCAP], v[NUCAP];
  double x4[4][NUCAP];
  int rank[NUCAP];
  const int n = A.nu_eff[col];
  const int st_in = A.status[col];
  bool ok = st_in == RS_OK && n > 0 && n <= nu;
  if (ok) ok = lane_cholesky(M, n, rdiag);
  if (ok) {
    lane_congruence(M, n, rdiag, v, p);
    lane_tridiag(M, n, d, e, p, tau, v);
    for (int k = 0; k < n; ++k) {      // the eigenvalues from copies: T stays for the eigenvectors,
      p[k] = d[k];                     // tau for the back-transform
      v[k] = e[k];
    }
    ok = lane_tql_values(n, p, v);
  }
  if (ok) {
    lane_sort(n, p);
    lane_tri_vectors(M, n, d, e, p, v, x4[0], x4[1], x4[2], x4[3], rank);
    lane_back_transform<NUCAP>(M, n, rdiag, tau, x4);
    for (int a = 0; a < n; ++a) {
      d[a] = p[a];
      rank[a] = a;
    }
  }
  int stc = st_in;
  if (stc == RS_OK && n < nu) stc = RS_BREAKDOWN;
  if (!ok && st_in == RS_OK) stc = RS_NOT_SPD;
  A.status[col] = stc;
  A.nu_eff[col] = ok ? n : 0;
  double* epsc = A.eps + col * nu;
  double* wc = A.w + col * nu;
  for (int a = 0; a < nu; ++a) {
    epsc[a] = 0.0;
    wc[a] = 0.0;
  }
  if (ok)
    for (int a = 0; a < n; ++a) {      // w_alpha = V_{j alpha} (S V)_{j alpha}
      double vj = 0.0, svj = 0.0;
      for (int k = 0; k < n; ++k) {
        const double ck = M.Z(k, a);
        vj += M.UJ(k) * ck;
        svj += M.SUJ(k) * ck;
      }
      epsc[rank[a]] = d[a];
      wc[rank[a]] = vj * svj;
    }
  if (A.cv) {                           // C and V_j, columns ranked, zero beyond nu_eff
    const int64_t ca = A.col0 + col;
    double* out = A.cv + (size_t)(ca >> 5) * kept_block_doubles(nu) * 32 + (ca & 31);
    const int ne = ok ? n : 0;
    int* inv = reinterpret_cast<int*>(tau);   // tau is free after the solve: rank -> eigenvector
    for (int a = 0; a < ne; ++a) inv[rank[a]] = a;
    if (ok)
      for (int a = 0; a < ne; ++a) {      // V_j alpha = (row j of U) . c_alpha
        double v = 0.0;
        for (int k = 0; k < ne; ++k) v += M.UJ(k) * M.Z(k, a);
        e[a] = v;
      }
    for (int r = 0; r < nu; ++r)
      for (int a = 0; a < nu; ++a)
        out[(size_t)(r * nu + a) * 32] = (r < ne && a < ne) ? M.Z(r, inv[a]) : 0.0;
    for (int a = 0; a < nu; ++a) out[(size_t)(nu * nu + a) * 32] = a < ne ? e[inv[a]] : 0.0;
  }
}

// ---- teams: several lanes per column ---------------------------------------------------------------
// One lane per column needs 32 columns a warp, its matrices stream through L2 (22 KB a column and matrix), and a column
// is one long serial chain: 6.9 ms for a single column of nu = 30, 15.9 ms for 32,768 (a third of the FP64 pipe),
// 445 ms for 148 columns of nu = 100. Here TL lanes share a column and CPW = 32 / TL columns share a warp
// (rows, or eigenvectors, strided over the lanes, so that the shrinking triangles keep the lanes busy and the square
// roots and divisions still serve CPW columns), with L and the matrix packed in shared memory, element by element
// [CPW]. Three launches, because the eigenvalues want the one-lane form: team_tridiag_kernel (Cholesky,
// congruence, Householder), ql_kernel (QL values, a thread per column; bisect_kernel for few) and team_vectors_kernel (inverse iteration,
// back-transform, outputs). The algorithm is the lane kernel's step by step; the sums' order differs.
__device__ __forceinline__ int pk(int i, int j) { return i * (i + 1) / 2 + j; }

// Between the kernels a column's d, e, tau, 1 / L_kk and eigenvalues sit in its scratch (4 nu + nu doubles).
struct Scratch {
  double* z;
  int nu;
  __device__ double& d(int k) const { return z[(size_t)k * 32]; }
  __device__ double& e(int k) const { return z[(size_t)(nu + k) * 32]; }
  __device__ double& tau(int k) const { return z[(size_t)(2 * nu + k) * 32]; }
  __device__ double& rdiag(int k) const { return z[(size_t)(3 * nu + k) * 32]; }
  __device__ double& lam(int k) const { return z[(size_t)(4 * nu + k) * 32]; }
};
__device__ __forceinline__ Scratch scratch_of(const Lane& M) { return Scratch{&M.Z(0, 0), M.nu}; }

template <int CPW>
__device__ __forceinline__ double team_sum(double v) {
#pragma unroll
  for (int o = 16; o >= CPW; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Doubles of shared memory per column: two packed triangles and three vectors.
__host__ __device__ constexpr int team_doubles(int n) { return n * (n + 1) + 3 * n; }

// TL lanes a column; a team of more than a warp has a CTA to itself: above nu = 64, where few columns fit on an SM and a
// warp's FP64 instructions, one in 64 cycles, are what a column waits for (148 columns of nu = 100: 6.6 -> 3.2 ms).
template <int TL>
__device__ __forceinline__ void team_sync() {
  if constexpr (TL > 32) __syncthreads();
  else __syncwarp();
}

template <int TL, int NS>
__global__ void __launch_bounds__(TL > 32 ? TL : 32) team_tridiag_kernel(const RedArgs A) {
  constexpr int CPW = TL > 32 ? 1 : 32 / TL;
  extern __shared__ double sm[];
  __shared__ double share[1 + 2 * (TL > 32 ? TL / 32 : 1)];   // across a team's warps: a pivot, two sums
  const int lane = threadIdx.x, c = lane % CPW, l = lane / CPW, nu = A.nu;
  const int64_t col = (int64_t)blockIdx.x * CPW + c;
  const bool real = col < A.n_cols;
  const int wl = TL > 32 ? l & ~31 : 0, ww_ = TL > 32 ? 32 : TL;   // the lanes of this warp within the team
  // sum over the team; `at` keeps neighbouring sums apart
  auto sum = [&](double v, int at) {
    if constexpr (TL > 32) {
      v = team_sum<1>(v);
      if ((l & 31) == 0) share[1 + at * (TL / 32) + (l >> 5)] = v;
      __syncthreads();
      v = 0.0;
#pragma unroll
      for (int w = 0; w < TL / 32; ++w) v += share[1 + at * (TL / 32) + w];
      return v;
    } else {
      return team_sum<CPW>(v);
    }
  };
  const int64_t colr = real ? col : A.n_cols - 1;
  const Lane M{A.blk + (size_t)(colr >> 5) * red_block_doubles(nu) * 32 + (colr & 31), nu};
  const Scratch Z = scratch_of(M);
  const int st_in = A.status[colr], n_in = A.nu_eff[colr];
  const int n = real && st_in == RS_OK && n_in > 0 && n_in <= nu ? n_in : 0;
  const int nm = __reduce_max_sync(0xffffffffu, n);
  double* L = sm + c;                                     // packed lower triangles, [element][CPW]
  double* H = L + (size_t)nm * (nm + 1) / 2 * CPW;
  double* vv = H + (size_t)nm * (nm + 1) / 2 * CPW;
  double* ww = vv + (size_t)nm * CPW;
  double* rd = ww + (size_t)nm * CPW;
  // S_r and H_r (upper triangle stored), padded to nm with the identity and zeros
  for (int i = l; i < nm; i += TL)
    for (int j = 0; j <= i; ++j) {
      const bool in = i < n;
      L[pk(i, j) * CPW] = in ? M.S(i, j) : (i == j ? 1.0 : 0.0);
      H[pk(i, j) * CPW] = in ? M.H(j, i) : 0.0;
    }
  team_sync<TL>();
  // Cholesky, a column at a time from the ones before
  bool spd = true;
  for (int k = 0; k < nm; ++k) {
    double v[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const int i = l + TL * s;
      v[s] = i >= k && i < nm ? L[pk(i, k) * CPW] : 0.0;
    }
    for (int j = 0; j < k; ++j) {
      const double lk = L[pk(k, j) * CPW];
#pragma unroll
      for (int s = 0; s < NS; ++s)
        if (wl + ww_ + TL * s > k && wl + TL * s < nm) v[s] = fma(-(l + TL * s < nm ? L[pk(l + TL * s, j) * CPW] : 0.0), lk, v[s]);
    }
    double dk = 0.0;
#pragma unroll
    for (int s = 0; s < NS; ++s)
      if (s == k / TL) dk = v[s];
    if constexpr (TL > 32) {
      if (l == k % TL) share[0] = dk;
      __syncthreads();
      dk = share[0];
    } else {
      dk = __shfl_sync(0xffffffffu, dk, (k % TL) * CPW + c);
    }
    if (!(dk > 0.0)) {
      spd = false;
      dk = 1.0;
    }
    const double lkk = sqrt(dk), r = 1.0 / lkk;
    team_sync<TL>();
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const int i = l + TL * s;
      if (i > k && i < nm) L[pk(i, k) * CPW] = v[s] * r;
      if (i == k) {
        L[pk(k, k) * CPW] = lkk;
        rd[k * CPW] = r;
      }
    }
    team_sync<TL>();
  }
  // X = L^{-1} H, upper triangle: row i of the packed lower triangle is column i of X, a lane's own
  for (int j = 0; j < nm; ++j) {
    double v[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const int i = l + TL * s;
      v[s] = i >= j && i < nm ? H[pk(i, j) * CPW] : 0.0;
    }
    for (int k = 0; k < j; ++k) {
      const double lk = L[pk(j, k) * CPW];
#pragma unroll
      for (int s = 0; s < NS; ++s)
        if (wl + ww_ + TL * s > j && wl + TL * s < nm) v[s] = fma(-(l + TL * s < nm ? H[pk(l + TL * s, k) * CPW] : 0.0), lk, v[s]);
    }
    const double r = rd[j * CPW];
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const int i = l + TL * s;
      if (i >= j && i < nm) H[pk(i, j) * CPW] = v[s] * r;
    }
  }
  team_sync<TL>();
  // A = L^{-1} X^T, lower triangle, column by column: the known part A(j, k), k < j, then the substitution
  for (int j = 0; j < nm; ++j) {
    double v[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const int i = l + TL * s;
      v[s] = i >= j && i < nm ? H[pk(i, j) * CPW] : 0.0;
    }
    for (int k = 0; k < j; ++k) {
      const double a = H[pk(j, k) * CPW];
#pragma unroll
      for (int s = 0; s < NS; ++s)
        if (wl + ww_ + TL * s > j && wl + TL * s < nm) v[s] = fma(-(l + TL * s < nm ? L[pk(l + TL * s, k) * CPW] : 0.0), a, v[s]);
    }
    for (int k = j; k < nm; ++k) {
#pragma unroll
      for (int s = 0; s < NS; ++s)
        if (l + TL * s == k) H[pk(k, j) * CPW] = v[s] * rd[k * CPW];
      team_sync<TL>();
      const double a = H[pk(k, j) * CPW];
#pragma unroll
      for (int s = 0; s < NS; ++s)
        if (wl + ww_ + TL * s > k && wl + TL * s < nm)
          v[s] = fma(-(l + TL * s > k && l + TL * s < nm ? L[pk(l + TL * s, k) * CPW] : 0.0), a, v[s]);
    }
  }
  // Householder reduction on the lower triangle; reflectors stay below the diagonal
  for (int k = 0; k + 2 < nm; ++k) {
    const bool on = k + 2 < n;                               // a smaller column of the warp is done: no reflector
    double v[NS], s2 = 0.0;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const int i = l + TL * s;
      v[s] = on && i > k && i < nm ? H[pk(i, k) * CPW] : 0.0;
      s2 = fma(v[s], v[s], s2);
    }
    s2 = sum(s2, 0);
    const double x0 = on ? H[pk(k + 1, k) * CPW] : 0.0;
    const double nrm = sqrt(s2);
    const double alpha = x0 >= 0.0 ? -nrm : nrm;
    const double v0 = x0 - alpha;
    const double vtv = s2 - x0 * x0 + v0 * v0;
    const double tk = vtv > 0.0 ? 2.0 / vtv : 0.0;          // H_k = I - tk v v^T
    team_sync<TL>();
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const int i = l + TL * s;
      if (on && i == k + 1) {
        v[s] = v0;
        H[pk(k + 1, k) * CPW] = v0;
      }
      if (i < nm) vv[i * CPW] = v[s];
    }
    if (l == 0 && on) {
      Z.d(k) = H[pk(k, k) * CPW];
      Z.e(k) = alpha;
      Z.tau(k) = tk;
    }
    team_sync<TL>();
    double p[NS], pv = 0.0;
#pragma unroll
    for (int s = 0; s < NS; ++s) p[s] = 0.0;
    for (int j = k + 1; j < nm; ++j) {                       // p = tk B v from B's lower triangle
      const double vj = vv[j * CPW];
      const int jr = pk(j, 0);
#pragma unroll
      for (int s = 0; s < NS; ++s)
        if (wl + ww_ + TL * s > k + 1 && wl + TL * s < nm) {
          const int i = l + TL * s;
          const int o = j <= i ? pk(i, j) : jr + i;
          p[s] = fma(i > k && i < nm ? H[o * CPW] : 0.0, vj, p[s]);
        }
    }
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      p[s] *= tk;
      pv = fma(p[s], v[s], pv);
    }
    pv = sum(pv, 1);
    const double kc = 0.5 * tk * pv;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      p[s] = fma(-kc, v[s], p[s]);                           // w = p - kc v
      if (l + TL * s < nm) ww[(l + TL * s) * CPW] = p[s];
    }
    team_sync<TL>();
    for (int j = k + 1; j < nm; ++j) {                       // B -= v w^T + w v^T
      const double vj = vv[j * CPW], wj = ww[j * CPW];
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        const int i = l + TL * s;
        if (i >= j && i < nm) {
          double* b = H + pk(i, j) * CPW;
          *b = fma(-p[s], vj, fma(-v[s], wj, *b));
        }
      }
    }
    team_sync<TL>();
  }
  if (!real) return;
  if (l == 0) {
    if (n >= 2) {
      Z.d(n - 2) = H[pk(n - 2, n - 2) * CPW];
      Z.e(n - 2) = H[pk(n - 1, n - 2) * CPW];
    }
    if (n >= 1) {
      Z.d(n - 1) = H[pk(n - 1, n - 1) * CPW];
      Z.e(n - 1) = 0.0;
    }
    int stc = st_in;
    if (n > 0 && !spd) stc = RS_NOT_SPD;
    else if (stc == RS_OK && n == 0) stc = RS_NOT_SPD;
    else if (stc == RS_OK && n < nu) stc = RS_BREAKDOWN;
    A.status[col] = stc;
    A.nu_eff[col] = spd ? n : 0;
  }
  for (int i = l; i < n; i += TL) {
    for (int j = 0; j <= i; ++j) M.S(i, j) = L[pk(i, j) * CPW];
    for (int j = 0; j < i; ++j) M.H(i, j) = H[pk(i, j) * CPW];
    Z.rdiag(i) = rd[i * CPW];
  }
}

// The eigenvalues, a thread per column (its d and e in shared memory), ascending. (FP32 values refined by Rayleigh
// quotients were tried instead: 2.8 -> 0.3 ms here at 32,768 columns of nu = 30, but the iterations for close pairs,
// which some lane of a warp always has, cost 5 ms in the vectors.)
__global__ void __launch_bounds__(32) ql_kernel(const RedArgs A) {
  extern __shared__ double sm[];
  const int64_t col = (int64_t)blockIdx.x * 32 + threadIdx.x;
  if (col >= A.n_cols) return;
  const int nu = A.nu, n = A.nu_eff[col];
  if (n <= 0) return;
  const Lane M{A.blk + (size_t)(col >> 5) * red_block_doubles(nu) * 32 + (col & 31), nu};
  const Scratch Z = scratch_of(M);
  const Strided d{sm + threadIdx.x, 32}, e{sm + (size_t)nu * 32 + threadIdx.x, 32};
  for (int k = 0; k < n; ++k) {
    d[k] = Z.d(k);
    e[k] = Z.e(k);
  }
  if (!lane_tql_values(n, d, e)) {
    A.status[col] = RS_NOT_SPD;
    A.nu_eff[col] = 0;
    return;
  }
  lane_sort(n, d);
  for (int k = 0; k < n; ++k) Z.lam(k) = d[k];
}

// The eigenvalues of few columns, a thread per eigenvalue: bisection on the sign changes of the leading principal minors
// of T - x I (Givens), p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2}. T is scaled by a power of two to |T| <= 1, so they
// grow by at most 2.5 a row; a pair below 2^-333 is scaled up again, looked at every 8 rows; a zero counts as a distance
// of 2^-60, far below the rounding of d_i. QL is one serial chain a column and an FP64 instruction holds a warp's scheduler for 64 cycles: 1.3 ms
// at nu = 30 and 15 ms at nu = 100, whatever the number of columns; four FP64 operations a row and step make this
// the shorter way (0.33 ms for 4 columns at nu = 30, 1.2 ms for 148 at nu = 100) for few columns, and the longer one
// beyond (six times the operations).
__global__ void __launch_bounds__(32) bisect_kernel(const RedArgs A) {
  extern __shared__ double sm[];
  const int lane = threadIdx.x, nu = A.nu, groups = (nu + 31) / 32;
  const int64_t col = blockIdx.x / groups;
  const int a = (int)(blockIdx.x % groups) * 32 + lane, n = A.nu_eff[col];
  if (n <= 0) return;
  const Lane M{A.blk + (size_t)(col >> 5) * red_block_doubles(nu) * 32 + (col & 31), nu};
  const Scratch Z = scratch_of(M);
  double *d = sm, *e2 = sm + n;
  double lo = INFINITY, hi = -INFINITY, big = 0.0;
  bool finite = true;
  for (int k = lane; k < n; k += 32) {
    const double dk = Z.d(k), r = (k + 1 < n ? fabs(Z.e(k)) : 0.0) + (k > 0 ? fabs(Z.e(k - 1)) : 0.0);
    finite &= fabs(dk) + r < INFINITY;
    lo = fmin(lo, dk - r);
    hi = fmax(hi, dk + r);
    big = fmax(big, fabs(dk) + r);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    big = fmax(big, __shfl_xor_sync(0xffffffffu, big, o));
  }
  if (!__all_sync(0xffffffffu, finite)) {                   // as a QL that does not converge
    if (a == 0) {
      A.status[col] = RS_NOT_SPD;
      A.nu_eff[col] = 0;
    }
    return;
  }
  const int ex = big > 0.0 ? ilogb(big) + 1 : 0;
  for (int k = lane; k < n; k += 32) {
    const double ek = k + 1 < n ? ldexp(Z.e(k), -ex) : 0.0;
    d[k] = ldexp(Z.d(k), -ex);
    e2[k] = ek * ek;
  }
  __syncwarp();
  lo = ldexp(lo, -ex) - 1e-15;
  hi = ldexp(hi, -ex) + 1e-15;
  for (int it = 0; it < 64 && hi - lo > 1e-16; ++it) {
    const double x = 0.5 * (lo + hi);
    if (!(lo < x && x < hi)) break;
    double p0 = 1.0, p1 = d[0] - x;
    if (p1 == 0.0) p1 = 0x1p-60;
    int below = p1 < 0.0;
    for (int i0 = 1; i0 < n; i0 += 8) {
      if (max(__double2hiint(p0) & 0x7fffffff, __double2hiint(p1) & 0x7fffffff) < (1023 - 333) << 20) {
        p0 *= 0x1p333;
        p1 *= 0x1p333;
      }
      const int i1 = min(i0 + 8, n);
      for (int i = i0; i < i1; ++i) {
        double p = fma(d[i] - x, p1, -e2[i - 1] * p0);
        if (p == 0.0) p = p1 * 0x1p-60;
        below += (__double2hiint(p) ^ __double2hiint(p1)) < 0;
        p0 = p1;
        p1 = p;
      }
    }
    if (below > a) hi = x;
    else lo = x;
  }
  if (a < n) Z.lam(a) = ldexp(0.5 * (lo + hi), ex);
}

// Eigenvectors and outputs. A lane takes the eigenvectors l, l + TL, ...: two inverse iterations with one factorisation;
// the vectors of a cluster (neighbours closer than 1e-3 ||T||_1) are then made orthonormal in order by the whole team,
// iterated once more and made orthonormal again. Q and L^{-T} are applied to up to four vectors at a time, and the column's
// levels, weights, C and V_j written.
template <int TL, int NS>
__global__ void __launch_bounds__(32) team_vectors_kernel(const RedArgs A) {
  constexpr int CPW = 32 / TL, NUCAP = TL * NS, R = NS < 4 ? NS : 4;
  extern __shared__ double sm[];
  const int lane = threadIdx.x, c = lane % CPW, l = lane / CPW, nu = A.nu;
  const int64_t col = (int64_t)blockIdx.x * CPW + c;
  const bool real = col < A.n_cols;
  const int64_t colr = real ? col : A.n_cols - 1;
  const Lane M{A.blk + (size_t)(colr >> 5) * red_block_doubles(nu) * 32 + (colr & 31), nu};
  const Scratch Z = scratch_of(M);
  const int n = real ? A.nu_eff[colr] : 0;
  const int nm = __reduce_max_sync(0xffffffffu, n);
  double* L = sm + c;
  double* H = L + (size_t)nm * (nm + 1) / 2 * CPW;
  double* d = H + (size_t)nm * (nm + 1) / 2 * CPW;
  double* e = d + (size_t)nm * CPW;
  double* lam = e + (size_t)nm * CPW;
  double tn = 0.0;
  for (int i = l; i < n; i += TL) {
    for (int j = 0; j <= i; ++j) L[pk(i, j) * CPW] = M.S(i, j);
    for (int j = 0; j < i; ++j) H[pk(i, j) * CPW] = M.H(i, j);
    d[i * CPW] = Z.d(i);
    e[i * CPW] = Z.e(i);
    lam[i * CPW] = Z.lam(i);
    H[pk(i, i) * CPW] = i + 2 < n ? Z.tau(i) : 0.0;          // tau on the reflectors' free diagonal
  }
  double rdl[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) rdl[s] = l + TL * s < n ? Z.rdiag(l + TL * s) : 0.0;
  __syncwarp();                                              // the scratch is free: Z's columns go there
  for (int k = 0; k < n; ++k)
    tn = fmax(tn, fabs(d[k * CPW]) + fabs(e[k * CPW]) + (k > 0 ? fabs(e[(k - 1) * CPW]) : 0.0));
  const double ortol = 1e-3 * tn, tiny = 2.2204460492503131e-16 * (tn > 0.0 ? tn : 1.0);
  double x4[4][NUCAP], mlt[NUCAP];
  int swp[NUCAP];
  const Strided sd{d, CPW}, se{e, CPW};
  double* x = x4[0];
  for (int a = l; a < n; a += TL) {
    for (int i = 0; i < n; ++i) {
      const double t = 0.7548776662466927 * (i + 1) + 0.5698402909980532 * (a + 1);
      x[i] = 0.5 + (t - floor(t));
    }
    lane_tri_factor(n, sd, se, lam[a * CPW], tiny, x4[1], x4[2], x4[3], mlt, swp);
    for (int it = 0; it < 2; ++it) {
      lane_tri_apply(n, x4[1], x4[2], x4[3], mlt, swp, x);
      double s2 = 0.0;
      for (int i = 0; i < n; ++i) s2 += x[i] * x[i];
      const double sc = s2 > 0.0 ? 1.0 / sqrt(s2) : 0.0;
      for (int i = 0; i < n; ++i) x[i] *= sc;
    }
    for (int i = 0; i < n; ++i) M.Z(i, a) = x[i];
  }
  __syncwarp();
  for (int it = 0; it < 2; ++it) {
    // clusters: orthonormal in order by the whole team, one more iteration, and again
    if (it == 1) {
      for (int a = l; a < n; a += TL) {
        if (a == 0 || !(lam[a * CPW] - lam[(a - 1) * CPW] <= ortol)) continue;
        for (int i = 0; i < n; ++i) x[i] = M.Z(i, a);
        lane_tri_factor(n, sd, se, lam[a * CPW], tiny, x4[1], x4[2], x4[3], mlt, swp);
        lane_tri_apply(n, x4[1], x4[2], x4[3], mlt, swp, x);
        double s2 = 0.0;
        for (int i = 0; i < n; ++i) s2 += x[i] * x[i];
        const double sc = s2 > 0.0 ? 1.0 / sqrt(s2) : 0.0;
        for (int i = 0; i < n; ++i) x[i] *= sc;
        for (int i = 0; i < n; ++i) M.Z(i, a) = x[i];
      }
      __syncwarp();
    }
    int cs = 0;
    bool any = false;
    for (int a = 1; a < nm; ++a) {
      if (a < n && lam[a * CPW] - lam[(a - 1) * CPW] > ortol) cs = a;
      const int len = a < n ? a - cs : 0;
      const int most = __reduce_max_sync(0xffffffffu, len);
      if (most == 0) continue;
      any = true;
      for (int b = 0; b < most; ++b) {
        const bool on = b < len;
        double dot = 0.0;
        if (on)
          for (int i = l; i < n; i += TL) dot = fma(M.Z(i, cs + b), M.Z(i, a), dot);
        dot = team_sum<CPW>(dot);
        if (on)
          for (int i = l; i < n; i += TL) M.Z(i, a) = fma(-dot, M.Z(i, cs + b), M.Z(i, a));
      }
      double s2 = 0.0;
      if (len)
        for (int i = l; i < n; i += TL) s2 = fma(M.Z(i, a), M.Z(i, a), s2);
      s2 = team_sum<CPW>(s2);
      const double sc = s2 > 0.0 ? 1.0 / sqrt(s2) : 0.0;
      if (len)
        for (int i = l; i < n; i += TL) M.Z(i, a) *= sc;
      __syncwarp();
    }
    if (!any) break;
  }
  // 1 / L_kk over d, which the eigenvectors no longer need
#pragma unroll
  for (int s = 0; s < NS; ++s)
    if (l + TL * s < n) d[(l + TL * s) * CPW] = rdl[s];
  __syncwarp();
  if (!real) return;
  double* epsc = A.eps + col * nu;
  double* wc = A.w + col * nu;
  const int64_t ca = A.col0 + col;
  double* out = A.cv ? A.cv + (size_t)(ca >> 5) * kept_block_doubles(nu) * 32 + (ca & 31) : nullptr;
  for (int a0 = l; a0 < nu; a0 += R * TL) {
    const int na = a0 < n ? min(R, (n - a0 + TL - 1) / TL) : 0;
    for (int r = 0; r < na; ++r)
      for (int i = 0; i < n; ++i) x4[r][i] = M.Z(i, a0 + TL * r);
    for (int r = na; r < R; ++r)
      for (int i = 0; i < n; ++i) x4[r][i] = 0.0;
    if (na) {
      for (int k = n - 3; k >= 0; --k) {                     // x <- (I - tau_k v_k v_k^T) x
        const double tk = H[pk(k, k) * CPW];
        double dot[R];
#pragma unroll
        for (int r = 0; r < R; ++r) dot[r] = 0.0;
        for (int i = k + 1; i < n; ++i) {
          const double vi = H[pk(i, k) * CPW];
#pragma unroll
          for (int r = 0; r < R; ++r) dot[r] = fma(vi, x4[r][i], dot[r]);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) dot[r] *= tk;
        for (int i = k + 1; i < n; ++i) {
          const double vi = H[pk(i, k) * CPW];
#pragma unroll
          for (int r = 0; r < R; ++r) x4[r][i] = fma(-dot[r], vi, x4[r][i]);
        }
      }
      for (int i = n - 1; i >= 0; --i) {                     // C = L^{-T} (Q Z)
        double s[R];
#pragma unroll
        for (int r = 0; r < R; ++r) s[r] = x4[r][i];
        for (int k = i + 1; k < n; ++k) {
          const double lk = L[pk(k, i) * CPW];
#pragma unroll
          for (int r = 0; r < R; ++r) s[r] = fma(-lk, x4[r][k], s[r]);
        }
        const double ri = d[i * CPW];
#pragma unroll
        for (int r = 0; r < R; ++r) x4[r][i] = s[r] * ri;
      }
    }
    double vj[R], svj[R];
#pragma unroll
    for (int r = 0; r < R; ++r) vj[r] = svj[r] = 0.0;
    for (int k = 0; k < n; ++k) {
      const double u = M.UJ(k), su = M.SUJ(k);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        vj[r] = fma(u, x4[r][k], vj[r]);
        svj[r] = fma(su, x4[r][k], svj[r]);
      }
    }
    for (int r = 0; r < R; ++r) {
      const int a = a0 + TL * r;
      if (a >= nu) break;
      const bool in = r < na;
      epsc[a] = in ? lam[a * CPW] : 0.0;
      wc[a] = in ? vj[r] * svj[r] : 0.0;
      if (out) {
        for (int i = 0; i < nu; ++i) out[(size_t)(i * nu + a) * 32] = in && i < n ? x4[r][i] : 0.0;
        out[(size_t)(nu * nu + a) * 32] = in ? vj[r] : 0.0;
      }
    }
  }
}

// TL1 lanes a column in the first kernel, TL2 in the last; nu <= TL NS.
template <int TL1, int NS1, int TL2, int NS2>
mka_status team_launch(const RedArgs& A, ReducedForm form, cudaStream_t st) {
  constexpr int C1 = TL1 > 32 ? 1 : 32 / TL1, C2 = 32 / TL2;
  auto k1 = team_tridiag_kernel<TL1, NS1>;
  auto k2 = team_vectors_kernel<TL2, NS2>;
  mka_status s = allow_shared(reinterpret_cast<const void*>(k1), nullptr);
  if (!s) s = allow_shared(reinterpret_cast<const void*>(ql_kernel), nullptr);
  if (!s) s = allow_shared(reinterpret_cast<const void*>(bisect_kernel), nullptr);
  if (!s) s = allow_shared(reinterpret_cast<const void*>(k2), nullptr);
  if (s) return s;
  const size_t smem = sizeof(double) * team_doubles(A.nu);
  k1<<<(unsigned)((A.n_cols + C1 - 1) / C1), TL1 > 32 ? TL1 : 32, smem * C1, st>>>(A);
  if (form == RF_FEW)
    bisect_kernel<<<(unsigned)(A.n_cols * ((A.nu + 31) / 32)), 32, sizeof(double) * 2 * A.nu, st>>>(A);
  else
    ql_kernel<<<(unsigned)((A.n_cols + 31) / 32), 32, sizeof(double) * 2 * A.nu * 32, st>>>(A);
  k2<<<(unsigned)((A.n_cols + C2 - 1) / C2), 32, smem * C2, st>>>(A);
  count_launches(3);
  MKA_CUDA_TRY(cudaGetLastError());
  return MKA_OK;
}

}  // namespace

mka_status reduced_launch(double* blk, int64_t n_cols, int64_t pick_cols, int nu, int32_t* status, int32_t* nu_eff, double* eps,
                          double* w, double* cv, int64_t col0, cudaStream_t st) {
  if (n_cols <= 0) return MKA_OK;
  RedArgs A{};
  A.blk = blk;
  A.n_cols = n_cols;
  A.nu = nu;
  A.status = status;
  A.nu_eff = nu_eff;
  A.eps = eps;
  A.w = w;
  A.cv = cv;
  A.col0 = col0;
  const ReducedForm form = reduced_form(nu, pick_cols);
  if (form != RF_LANES) {
    if (nu > 64) return team_launch<128, 2, 32, 5>(A, form, st);
    if (nu > 32) return form == RF_FEW ? team_launch<32, 2, 32, 2>(A, form, st) : team_launch<16, 4, 32, 2>(A, form, st);
    return form == RF_FEW ? team_launch<32, 1, 32, 1>(A, form, st) : team_launch<8, 4, 16, 2>(A, form, st);
  }
  const int threads = 128;
  const unsigned blocks = (unsigned)((n_cols + threads - 1) / threads);
  if (nu <= kTinyNu) reduced_kernel<kTinyNu><<<blocks, threads, 0, st>>>(A);
  else if (nu <= kSmallNu) reduced_kernel<kSmallNu><<<blocks, threads, 0, st>>>(A);
  else reduced_kernel<MKA_MAX_NU><<<blocks, threads, 0, st>>>(A);
  count_launches();
  MKA_CUDA_TRY(cudaGetLastError());
  return MKA_OK;
}

}  // namespace mka
