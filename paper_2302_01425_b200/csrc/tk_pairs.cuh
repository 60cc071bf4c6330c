// tk_pairs.cuh -- the pair steps of the alternating-projection solver path (Algorithm 1 and App. A.8) and the
// solver on consecutive ranks per thread.  What is iterated is described in tk_dykstra.cu.
#pragma once

#include "tk_common.cuh"

namespace tk {

namespace {

// One Dykstra step on a pair in the metric (ca, cb): a, b are the current iterate, delta the
// stored correction; on return a >= b holds and delta is the new correction.
__device__ __forceinline__ void dyk_pair(float& a, float& b, float& delta, float ca, float cb) {
  const float ta = a - cb * delta, tb = b + ca * delta;
  const float d = fmaxf(0.0f, (tb - ta) / (ca + cb));
  a = ta + cb * d;
  b = tb - ca * d;
  delta = d;
}

// Dual coordinate of the constraint between keys s1 >= s2 (weights w1, w2), neighbours' duals fixed.
__device__ __forceinline__ float bca_alpha(float s1, float s2, float w1, float w2, float a_prev,
                                           float a_next, const Math& M) {
  const float c1 = w1 + a_prev, c2 = w2 - a_next;
  // s1 >= s2, so the separate minimisers s_i - lam cbrt(c_i) are in order whenever c1 <= c2: most
  // pairs (equal weights, no active neighbour) end here without a cube root
  if (c1 <= c2) return 0.0f;
  const float v1 = s1 - M.lam * cbrtf(c1), v2 = s2 - M.lam * cbrtf(c2);
  if (v1 >= v2) return 0.0f;
  const float d = 0.5f * (s1 - s2), m = 0.5f * (s1 + s2);
  const float B = 0.5f * M.lam3 * (c1 + c2);
  const float d2 = d * d;
  const float R = sqrtf(0.25f * B * B + d2 * d2 * d2);
  const float big = -copysignf(cbrtf(0.5f * fabsf(B) + R), B);
  float t = (big != 0.0f) ? big - d2 / big : 0.0f;
  {   // one Newton step on the increasing cubic t^3 + 3 d^2 t + B
    const float f = fmaf(t * t + 3.0f * d2, t, B), fp = 3.0f * (t * t + d2);
    if (fp > 0.0f) t -= f / fp;
  }
  const float z = (s1 - (m + t)) * M.inv_lam;
  return fmaxf(0.0f, c1 - z * z * z);
}

// ---- the same coordinate step for any q and for phi even (App. A.8 leaves the two-variable problem to a
// root solver; the closed form above is the special case q = 4, phi = x).  rho is odd: sign(t) |t/lambda|^(q-1).
__device__ __forceinline__ float bca_rho(const Math& M, float t) {
  const float a = fabsf(t) * M.inv_lam;
  return copysignf(M.gen ? powf(a, M.qm1) : (M.q4 ? a * a * a : a), t);
}
__device__ __forceinline__ float bca_drho(const Math& M, float t) {
  const float a = fabsf(t) * M.inv_lam;
  return (M.gen ? M.qm1 * powf(a, M.qm1 - 1.0f) : (M.q4 ? 3.0f * a * a : 1.0f)) * M.inv_lam;
}
__device__ __forceinline__ float bca_rho_inv(const Math& M, float z) {
  const float a = fabsf(z);
  return copysignf(M.lam * (M.gen ? powf(a, 1.0f / M.qm1) : (M.q4 ? cbrtf(a) : a)), z);
}
// Root of an increasing function inside [lo, hi] (f(lo) <= 0 <= f(hi)): Newton, bisection when a step
// leaves the bracket.  fd(x, f, df) evaluates the function and its derivative.
template <class FD>
__device__ __forceinline__ float bca_root(float lo, float hi, float x, FD fd) {
#pragma unroll 1
  for (int it = 0; it < 60; ++it) {
    float f, df;
    fd(x, f, df);
    if (f > 0.0f) hi = x; else lo = x;
    float nx = df > 0.0f ? x - f / df : 0.5f * (lo + hi);
    if (!(nx > lo && nx < hi)) nx = 0.5f * (lo + hi);
    if (fabsf(nx - x) <= 1e-7f * fabsf(nx) + 1e-30f || !(hi > lo)) { x = nx; break; }
    x = nx;
  }
  return x;
}
// argmin_v r*(s - v) + w phi(v) + c v: -rho(s - v) + w phi'(v) + c = 0
__device__ __forceinline__ float bca_shifted(const Math& M, float s, float w, float c) {
  if (!M.mag || w == 0.0f) return s - bca_rho_inv(M, (M.mag ? 0.0f : w) + c);
  // phi even, w = 1: with t = s - v, rho(t) + t = s + c, t between 0 and s + c
  const float R = s + c;
  if (R == 0.0f) return s;
  const float lo = fminf(0.0f, R), hi = fmaxf(0.0f, R);
  const float t = bca_root(lo, hi, 0.5f * R, [&](float x, float& f, float& df) {
    f = bca_rho(M, x) + x - R; df = bca_drho(M, x) + 1.0f; });
  return s - t;
}
// the dual of the constraint between keys s1 >= s2, neighbours' duals fixed
__device__ __forceinline__ float bca_alpha_any(float s1, float s2, float w1, float w2, float a_prev, float a_next,
                                              const Math& M) {
  const float c1 = a_prev, c2 = -a_next;
  if (!M.mag && w1 + c1 <= w2 + c2) return 0.0f;           // separate minimisers in order (rho_inv is increasing)
  const float v1 = bca_shifted(M, s1, w1, c1), v2 = bca_shifted(M, s2, w2, c2);
  if (v1 >= v2) return 0.0f;
  const float ws = w1 + w2, cs = c1 + c2;
  const float g = bca_root(v1, v2, 0.5f * (v1 + v2), [&](float x, float& f, float& df) {
    f = -bca_rho(M, s1 - x) - bca_rho(M, s2 - x) + (M.mag ? ws * x : ws) + cs;
    df = bca_drho(M, s1 - x) + bca_drho(M, s2 - x) + (M.mag ? ws : 0.0f); });
  return fmaxf(0.0f, -bca_rho(M, s1 - g) + (M.mag ? w1 * g : w1) + a_prev);
}
// y_i = rho(s_i - v_i) at the primal iterate v_i = argmin h_i(v) + (alpha_{i-1} - alpha_i) v
__device__ __forceinline__ float bca_output(const Math& M, float s, float w, float a_im1, float a_i) {
  if (!M.mag) return w + a_im1 - a_i;
  const float v = fmaxf(bca_shifted(M, s, w, a_im1 - a_i), 0.0f);
  return bca_rho(M, s - v);
}

// The solver on E consecutive ranks per thread.  Exchange with the neighbouring threads goes
// through the two callables: next0(x) returns the NEXT thread's x, prev_last(x) the PREVIOUS thread's.
// On return y[i] = rho(s_i - v_i).
// MAG (phi even) is a template flag: for phi = x every metric weight is the constant 1, the pair
// projection loses its division and the weights their registers.
// key_again(i): the key s[i] once more, for the output map of the p = 2 iteration, which does not
// touch s between its first line and its last: a kernel short of registers reads it from memory there.
// TOL (run to a tolerance, tk_opts.tol > 0): the largest move of an entry of the iterate (p = 2) or of a
// dual (p = 4/3) in any projection of a sweep is taken over the row by row_max(x), which returns the same
// value to every thread of the row; the sweeps end when it is at most P.tol, or at the cap `sweeps`
// (returns false then: not converged).
template <int E, bool MAG, bool TOL, typename NextF, typename PrevF, typename SyncF, typename KeyF, typename MaxF>
__device__ __forceinline__ bool solve_pairs_m(const Problem& P, const Math& M, const float (&s)[E], int rank0,
                                            bool has_next, bool has_prev, NextF next_of, PrevF prev_of,
                                            SyncF sync, KeyF key_again, MaxF row_max, float (&y)[E]) {
  const int n = P.n, k = P.k;
  const int sweeps = P.sweeps > 0 ? P.sweeps : 100;
  bool met = !TOL;
  const float s_next = next_of(s[0]);                      // key of the next thread's first rank
  sync();
  const bool cross = has_next && (rank0 + E) < n;          // pair (rank0 + E - 1, rank0 + E) exists
  auto wgt = [&](int rk) -> float { return rk < k ? 1.0f : 0.0f; };
  if (!M.q4) {
    float v[E], c[E], pd[E / 2], qd[E / 2];
#pragma unroll
    for (int i = 0; i < E; ++i) {
      const float w = wgt(rank0 + i);
      c[i] = MAG ? 1.0f + M.lam * w : 1.0f;
      v[i] = MAG ? s[i] / c[i] : s[i] - M.lam * w;
    }
#pragma unroll
    for (int j = 0; j < E / 2; ++j) { pd[j] = 0.0f; qd[j] = 0.0f; }
    const float c_next = MAG ? 1.0f + M.lam * wgt(rank0 + E) : 1.0f;
#pragma unroll 1
    for (int it = 0; it < sweeps; ++it) {
      float chg = 0.0f;                                    // TOL: largest move of one of this thread's entries
#pragma unroll
      for (int j = 0; j < E / 2; ++j)
        if (rank0 + 2 * j + 1 < n) {
          const float o0 = v[2 * j], o1 = v[2 * j + 1];
          dyk_pair(v[2 * j], v[2 * j + 1], pd[j], c[2 * j], c[2 * j + 1]);
          if (TOL) chg = fmaxf(chg, fmaxf(fabsf(v[2 * j] - o0), fabsf(v[2 * j + 1] - o1)));
        }
      // C2: the pair that crosses to the next thread, then the thread-local ones
      float nb = next_of(v[0]);
      float mine = v[E - 1];
      if (cross) {
        const float o0 = mine, o1 = nb;
        dyk_pair(mine, nb, qd[E / 2 - 1], c[E - 1], c_next);
        if (TOL) chg = fmaxf(chg, fmaxf(fabsf(mine - o0), fabsf(nb - o1)));
      }
      v[E - 1] = mine;
#pragma unroll
      for (int j = 0; j < E / 2 - 1; ++j)
        if (rank0 + 2 * j + 2 < n) {
          const float o0 = v[2 * j + 1], o1 = v[2 * j + 2];
          dyk_pair(v[2 * j + 1], v[2 * j + 2], qd[j], c[2 * j + 1], c[2 * j + 2]);
          if (TOL) chg = fmaxf(chg, fmaxf(fabsf(v[2 * j + 1] - o0), fabsf(v[2 * j + 2] - o1)));
        }
      sync();
      const float back = prev_of(nb);                      // what the previous thread made of my first rank
      if (has_prev && rank0 < n) v[0] = back;
      sync();
      if (TOL && row_max(chg) <= P.tol) { met = true; break; }
    }
#pragma unroll
    for (int i = 0; i < E; ++i) {
      const float vi = MAG ? fmaxf(v[i], 0.0f) : v[i];
      y[i] = (key_again(i) - vi) * M.inv_lam;
    }
  } else {
    // alpha of constraint (rank0 + i, rank0 + i + 1): i even -> ao[i/2], i odd -> ae[i/2]
    float ao[E / 2], ae[E / 2];
#pragma unroll
    for (int j = 0; j < E / 2; ++j) { ao[j] = 0.0f; ae[j] = 0.0f; }
    float prev_e = 0.0f;                                   // previous thread's last even-family dual
#pragma unroll 1
    for (int it = 0; it < sweeps; ++it) {
      float chg = 0.0f;                                    // TOL: largest move of one of this thread's duals
#pragma unroll
      for (int j = 0; j < E / 2; ++j) {
        const int rk = rank0 + 2 * j;
        if (rk + 1 < n) {
          const float a_prev = (j == 0) ? prev_e : ae[j - 1];
          const float old = ao[j];
          ao[j] = bca_alpha(s[2 * j], s[2 * j + 1], wgt(rk), wgt(rk + 1), a_prev, ae[j], M);
          if (TOL) chg = fmaxf(chg, fabsf(ao[j] - old));
        }
      }
      const float next_o = next_of(ao[0]);
      sync();
#pragma unroll
      for (int j = 0; j < E / 2; ++j) {
        const int rk = rank0 + 2 * j + 1;
        const float old = ae[j];
        if (j < E / 2 - 1) {
          if (rk + 1 < n) ae[j] = bca_alpha(s[2 * j + 1], s[2 * j + 2], wgt(rk), wgt(rk + 1), ao[j], ao[j + 1], M);
        } else if (cross) {
          const float a_next = (rk + 2 < n) ? next_o : 0.0f;
          ae[j] = bca_alpha(s[E - 1], s_next, wgt(rk), wgt(rk + 1), ao[j], a_next, M);
        }
        if (TOL) chg = fmaxf(chg, fabsf(ae[j] - old));
      }
      const float pe = prev_of(ae[E / 2 - 1]);
      prev_e = has_prev ? pe : 0.0f;
      sync();
      if (TOL && row_max(chg) <= P.tol) { met = true; break; }
    }
#pragma unroll
    for (int i = 0; i < E; ++i) {
      const float a_i = (i & 1) ? ae[i / 2] : ao[i / 2];
      const float a_im1 = (i == 0) ? prev_e : ((i & 1) ? ao[i / 2] : ae[i / 2 - 1]);
      y[i] = wgt(rank0 + i) - a_i + a_im1;
    }
  }
  return met;
}

// returns false when a run to tolerance (TOL) stopped at the cap
template <int E, bool TOL, typename NextF, typename PrevF, typename SyncF, typename KeyF, typename MaxF>
__device__ __forceinline__ bool solve_pairs(const Problem& P, const Math& M, const float (&s)[E], int rank0,
                                            bool has_next, bool has_prev, NextF next_of, PrevF prev_of,
                                            SyncF sync, KeyF key_again, MaxF row_max, float (&y)[E]) {
  if (M.mag) return solve_pairs_m<E, true, TOL>(P, M, s, rank0, has_next, has_prev, next_of, prev_of, sync, key_again, row_max, y);
  return solve_pairs_m<E, false, TOL>(P, M, s, rank0, has_next, has_prev, next_of, prev_of, sync, key_again, row_max, y);
}

}  // namespace

}  // namespace tk
