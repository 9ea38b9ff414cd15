// The root finders for N(mu) = N_e of the per-batch and the whole-system chemical potential: a bracket [lo, hi] with
// f = N - N_e at its ends and the next point x.
#pragma once

namespace mka {
namespace {

// side: the end that moved last (-1 lo, +1 hi); rf: whether x came from the secant; probed: see root_step_lowest.
struct RootState {
  double lo, hi, target, kT, tol, last, iters, x, flo, fhi, side, rf, probed;
};
constexpr double kSecantKT = 16.0;   // bisection while the bracket is wider than this many kT

// The whole system's step with the count t at S->x: the bracket end on its side moves to x. The next point is the midpoint
// while the bracket is wider than 16 kT, then the secant through the ends (regula falsi, with the Illinois rule:
// after two moves of the same end by the secant, the other end's f is halved), the midpoint when the secant leaves
// the bracket; a point where the count equals N_e exactly closes the bracket on it. IEEE-rounded operations
// throughout (no contraction), so that a host driver doing the same arithmetic on the same counts takes the same
// points bit for bit.
__device__ inline void root_step(RootState* S, double t) {
  const double x = S->x, fx = __dsub_rn(t, S->target);
  S->last = t;
  S->iters += 1;
  if (fx == 0.0) {                     // x is a root to rounding: the bracket closes on it
    S->lo = x;
    S->hi = x;
    S->flo = 0.0;
    S->fhi = 0.0;
    return;
  }
  if (fx < 0.0) {
    S->lo = x;
    S->flo = fx;
    if (S->rf != 0.0 && S->side == -1.0) S->fhi = __dmul_rn(0.5, S->fhi);
    S->side = -1.0;
  } else {
    S->hi = x;
    S->fhi = fx;
    if (S->rf != 0.0 && S->side == 1.0) S->flo = __dmul_rn(0.5, S->flo);
    S->side = 1.0;
  }
  const double lo = S->lo, hi = S->hi, mid = __dmul_rn(0.5, __dadd_rn(lo, hi));
  double nx = mid, rf = 0.0;
  if (!(__dsub_rn(hi, lo) > __dmul_rn(kSecantKT, S->kT))) {
    const double sx = __ddiv_rn(__dsub_rn(__dmul_rn(lo, S->fhi), __dmul_rn(hi, S->flo)), __dsub_rn(S->fhi, S->flo));
    if (lo < sx && sx < hi) {
      nx = sx;
      rf = 1.0;
    }
  }
  S->x = nx;
  S->rf = rf;
}

// The batch's step: to the lowest mu with N >= N_e, the value halving alone converges to, which matters where the
// count stands still (gapped levels, full or empty bands). A count at or above N_e moves the upper end; one that is N_e
// exactly is followed, once, by the point 3/4 tol below it, which ends the search unless the count stands still there.
// The next point is the secant's as in root_step, or the midpoint; always the midpoint when fewer than `left` - 1
// halvings would be left for the bracket: `left` passes follow this one, and a search that enough halvings can end is
// ended by them. (Passes in numpy over levels of 1 to 400 columns, tol 1e-12: 8 to 31 where levels lie at mu, up to
// 62 where mu is the edge of a gap.)
__device__ inline void root_step_lowest(RootState* S, double t, int left) {
  const double x = S->x, fx = t - S->target;
  S->last = t;
  S->iters += 1;
  if (fx < 0.0) {
    S->lo = x;
    S->flo = fx;
    if (S->rf != 0.0 && S->side == -1.0) S->fhi *= 0.5;
    S->side = -1.0;
  } else {
    S->hi = x;
    S->fhi = fx;
    if (S->rf != 0.0 && S->side == 1.0) S->flo *= 0.5;
    S->side = 1.0;
  }
  const double lo = S->lo, hi = S->hi, flo = S->flo, fhi = S->fhi;
  double nx = 0.5 * (lo + hi), rf = 0.0;
  if (hi - lo <= ldexp(S->tol, left - 1)) {
    if (fx == 0.0 && S->probed == 0.0) {
      const double below = x - 0.75 * S->tol;
      S->probed = 1.0;
      if (lo < below && below < hi) nx = below;
    } else if (!(hi - lo > kSecantKT * S->kT) && flo < 0.0 && fhi > 0.0) {
      const double sx = (lo * fhi - hi * flo) / (fhi - flo);
      if (lo < sx && sx < hi) {
        nx = sx;
        rf = 1.0;
      }
    }
  }
  S->x = nx;
  S->rf = rf;
}

// f w summed over a column's levels part, part + step, ... (ascending; entries with w = 0 add nothing). With step = 1
// a thread takes a whole column: at a given level index the lanes of a warp hold levels of much the same energy, so that
// they agree on whether f is 1, 0 or needs the tanh, which only a quarter of the levels do. rk = 1 / (2 kT).
__device__ __forceinline__ double column_count(const double* __restrict__ eps, const double* __restrict__ w, int nu,
                                               double mu, double rk, int part = 0, int step = 1) {
  double c = 0.0;
#pragma unroll 4
  for (int a = part; a < nu; a += step) {
    const double wi = w[a], y = (eps[a] - mu) * rk;
    if (wi != 0.0 && !(y > 20.0)) c += (y < -20.0 ? 1.0 : 0.5 * (1.0 - tanh(y))) * wi;
  }
  return c;
}

}  // namespace
}  // namespace mka
