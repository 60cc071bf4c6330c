// tk_cols.cu -- the operator along the slow axis of an [n, cols] matrix (column c is one problem), forward pass
// by the threshold form (tk_newton_core.cuh) and VJP from saved row state, straight from the matrix as it lies in
// memory: no transpose.
//
// A thread block takes kColC = 8 neighbouring columns.  Lane l of a warp works on column l % 8 and on every
// S-th row from its slice on (S = 4 slices per warp * warps): one warp load reads 4 rows x 32 contiguous bytes, whole
// sectors, and the column's keys stay in registers (E per lane) through the iteration.  The only exchange is
// the column's sums: two shuffles, then one shared-memory slot per warp and a block barrier when the column
// takes several warps.  Every lane of a column replays the same scalar step, so no result has to be sent back.
//
// Why 8 columns: a block iterates until its slowest column is done (more columns, more passes), fewer than 8 would
// split sectors between blocks.
//
// What bounds it: the forward pass issue slots (70 %; half of its instructions are the passes' scalar steps and sums, which
// every warp of a column repeats), the VJP DRAM latency at 40 % occupancy.  400 x 32768, p = 2: forward 93 us as
// transpose + row kernel + transpose, 55 here, the copy of theta included; VJP 74 -> 34 us (12 bytes per element
// each: 24 us at the copy bandwidth).  Columns above 2048 rows would leave one block of 16 warps with 64 rows per lane on an
// SM, whose barriers nothing hides: 2814 x 1445 ran 120 us like that against 85 through the transposes, which stay there.
#include <type_traits>

#include "tk_newton_core.cuh"

namespace tk {

float upper_normal_quantile(double tail);      // tk_newton.cu

namespace {

constexpr int kColC = 8;                       // columns per thread block
constexpr int kColSlices = 32 / kColC;         // row slices per warp
constexpr int kColMaxWarps = 16;

struct ColArgs {
  const float* theta; long long ld_theta;      // [n, cols]
  const float* gout; long long ld_gout;        // VJP
  float* out; long long ld_out;
  float* copy;                                 // contiguous [n, cols] copy of theta for a later VJP, or null
};

// One slot of a column's sums: 2 or 4 words, moved as a vector.
template <int NV> struct ColSlot;
template <> struct ColSlot<2> { using type = float2; };
template <> struct ColSlot<4> { using type = float4; };

// Sums of NV words over the lanes of a column (word 0 as an unsigned integer when COUNT); every lane of it gets
// the same totals.  red: this phase's buffer of kColMaxWarps * kColC slots; the caller alternates between two, so one
// barrier per sum is enough.
template <int NV, bool COUNT>
__device__ __forceinline__ void col_allsum(float (&v)[NV], float* red, int warps) {
  using Slot = typename ColSlot<NV>::type;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto add = [](float a, float b, bool count) -> float {
    return count ? __uint_as_float(__float_as_uint(a) + __float_as_uint(b)) : a + b;
  };
  auto slices = [&]() {
#pragma unroll
    for (int o = kColC; o < 32; o <<= 1) {
#pragma unroll
      for (int i = 0; i < NV; ++i) v[i] = add(v[i], __shfl_xor_sync(0xffffffffu, v[i], o), COUNT && i == 0);
    }
  };
  slices();
  if (warps > 1) {
    Slot* slots = reinterpret_cast<Slot*>(red) + lane % kColC;
    if (lane < kColC) {
      Slot m;
      float* mw = reinterpret_cast<float*>(&m);
#pragma unroll
      for (int i = 0; i < NV; ++i) mw[i] = v[i];
      slots[warp * kColC] = m;
    }
    __syncthreads();
    // the four lanes of a column share the warps' slots out; a butterfly gives every lane the same total
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = 0.0f;
#pragma unroll 1
    for (int w = lane / kColC; w < warps; w += kColSlices) {
      const Slot m = slots[w * kColC];
      const float* mw = reinterpret_cast<const float*>(&m);
#pragma unroll
      for (int i = 0; i < NV; ++i) v[i] = add(v[i], mw[i], COUNT && i == 0);
    }
    slices();
  }
}

// The rows of one lane: element i is row sl + i * S of the column, at byte `at(i)` of a matrix with leading dimension ld.
// Groups of 4 elements below `fast` lie inside the column for every lane of the block, the groups from there to
// `groups` hold its end.  Off: uint32_t for matrices below 4 GB (one add per address), else uint64_t.
template <class Off>
struct ColRows {
  int sl, S, n, groups, fast;
  __device__ __forceinline__ ColRows(int n_) : n(n_) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    S = (int)(blockDim.x >> 5) * kColSlices;
    sl = warp * kColSlices + lane / kColC;
    groups = ((n + S - 1) / S + 3) >> 2;
    fast = (n / S) >> 2;
  }
  // the same rows for a later phase, with S hidden from the compiler: otherwise it keeps the offsets and the end tests of
  // one phase in registers for the next (30 of them spilled over the iteration)
  __device__ __forceinline__ ColRows again() const {
    ColRows r = *this;
    asm volatile("" : "+r"(r.S));
    return r;
  }
  __device__ __forceinline__ int row(int i) const { return sl + i * S; }
  __device__ __forceinline__ bool in(int i) const { return row(i) < n; }
};

template <class Off>
struct ColMatrix {
  const char* base;            // the block's first column (the same for every thread)
  Off first, step, lane_off;   // bytes: row 0 of this lane's column, from one element of a lane to the next, its first row
  long long extent; int32_t* status;          // range-checked build
  __device__ __forceinline__ ColMatrix(const float* m, long long ld, long long col0, int c, const ColRows<Off>& R, long long cols, int32_t* st)
      : base(reinterpret_cast<const char*>(m + col0)), first((Off)c * 4), step((Off)R.S * (Off)ld * 4),
        lane_off((Off)c * 4 + (Off)R.sl * (Off)ld * 4), extent(((R.n - 1) * ld + cols - col0) * 4), status(st) {}
  // past the column's end: its first row.  AGAIN: read before, the read-only path may be taken
  template <bool FAST, bool AGAIN = false>
  __device__ __forceinline__ float load(int i, const ColRows<Off>& R) const {
    const Off o = FAST || R.in(i) ? lane_off + (Off)i * step : first;
    const float* at = reinterpret_cast<const float*>(base + o);
    return TK_IN_BOUNDS(o, 4, extent, status) ? (AGAIN ? __ldg(at) : *at) : 0.0f;
  }
  template <bool FAST>
  __device__ __forceinline__ void store(int i, const ColRows<Off>& R, bool col_ok, float v) const {
    const Off o = lane_off + (Off)i * step;
    if (col_ok && (FAST || R.in(i)) && TK_IN_BOUNDS(o, 4, extent, status)) *reinterpret_cast<float*>(const_cast<char*>(base) + o) = v;
  }
};

// body(i, std::true_type) for the elements of the groups inside the column, body(i, std::false_type) for those at its end
template <int E, class Off, class F>
__device__ __forceinline__ void col_each(const ColRows<Off>& R, F body) {
#pragma unroll
  for (int g = 0; g < E / 4; ++g) {
    if (g < R.fast) {
#pragma unroll
      for (int j = 0; j < 4; ++j) body(4 * g + j, std::true_type());
    } else if (g < R.groups) {
#pragma unroll
      for (int j = 0; j < 4; ++j) body(4 * g + j, std::false_type());
    }
  }
}

// Forward pass, E rows per lane at most.
template <int E, bool Q4, bool MAG, class Off>
__global__ void __maxnreg__(E <= 16 ? 64 : 80) tk_cols_fwd_kernel(const Problem P, const ColArgs A, const float zq) {
  constexpr int NV = Q4 ? 4 : 2;
  __shared__ float4 red_s[2][kColMaxWarps * kColC];
  auto red = [&](int ph) -> float* { return reinterpret_cast<float*>(red_s[ph & 1]); };
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const int n = P.n, k = P.k;
  const long long cols = P.rows, col0 = (long long)blockIdx.x * kColC;
  const bool col_ok = col0 + lane % kColC < cols;
  const int c = col_ok ? lane % kColC : (int)(cols - 1 - col0);   // a lane past the last column repeats it, stores nothing
  const long long col = col0 + c;
  const ColRows<Off> R(n);
  const ColMatrix<Off> X(A.theta, A.ld_theta, col0, c, R, cols, P.status);
  const float lam = P.lam, inv_lam = P.inv_lam, lam3 = P.lam3;
  float wid = P.lam;
  constexpr float kTolRel = Q4 ? 1e-7f : 3e-7f;
  int phase = 0;

  overlap_wait();
  float d[E];
  col_each<E>(R, [&](int i, auto fast) { d[i] = X.template load<decltype(fast)::value>(i, R); });
  if (A.copy) {
    const ColRows<Off> Rc = R.again();
    const ColMatrix<Off> C(A.copy, cols, col0, c, Rc, cols, P.status);
    col_each<E>(Rc, [&](int i, auto fast) { C.template store<decltype(fast)::value>(i, Rc, col_ok, d[i]); });
  }

  // ---- start: moments of the keys (about the first key; phi even: about 0, and the keys above 0 counted)
  NtRow T;
  nt_row_init(T, k);
  bool bad = false;
  const float x0 = MAG ? 0.0f : X.template load<false>(n, R);     // (an element past every end: the column's first row)
  float m[2] = {0.f, 0.f}, nnz[2] = {0.f, 0.f};
#pragma unroll
  for (int g = 0; g < E / 4; ++g) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = 4 * g + j;
      if (g >= R.groups) { d[i] = -INFINITY; continue; }
      if (MAG) d[i] = fabsf(d[i]);
      float dd = d[i] - x0;
      if (g >= R.fast && !R.in(i)) { dd = 0.0f; d[i] = -INFINITY; }
      m[0] += dd; m[1] = fmaf(dd, dd, m[1]);
      if (MAG) nnz[0] += d[i] > 0.0f ? 1.0f : 0.0f;
    }
  }
  col_allsum<2, false>(m, red(phase++), warps);
  if (MAG) col_allsum<2, false>(nnz, red(phase++), warps);
  if (!(m[1] < INFINITY)) {                    // overflow, an infinity or a NaN: look at the keys themselves
#pragma unroll
    for (int i = 0; i < E; ++i) bad |= (i >> 2) < R.groups && R.in(i) && !(fabsf(d[i]) < INFINITY);
  }
  {
    const float inv_n = 1.0f / (float)n;
    const float mean_d = m[0] * inv_n;
    if (!MAG) {
      if (k == n) {
        T.piv = -FLT_MAX; T.off = -wid; T.done = true; T.noblock = true;
      } else {
        const float sd = sqrtf(fmaxf(m[1] * inv_n - mean_d * mean_d, 0.0f));
        float tau0 = (x0 + mean_d) + zq * sd - (Q4 ? 0.75f : 0.5f) * lam;
        if (!(fabsf(tau0) < FLT_MAX)) tau0 = x0;
        T.piv = tau0;
      }
    } else {
      if (k == n || (int)nnz[0] < k) {
        T.piv = 0.0f; T.off = 0.0f; T.done = true; T.noblock = true;
      } else {
        const float t0 = zq * sqrtf(m[1] * inv_n);
        float tau0 = Q4 ? t0 - 0.75f * lam * cbrtf(t0) : t0 / (1.0f + 0.5f * lam);
        if (!(tau0 > 0.0f && tau0 < FLT_MAX)) tau0 = 0.5f * t0;
        if (!(tau0 > 0.0f && tau0 < FLT_MAX)) tau0 = 1.0f;
        T.piv = tau0;
        T.lo_a = 0.0f; T.lo_o = -tau0;
      }
    }
  }
  const bool early = T.done && T.noblock;
#pragma unroll
  for (int i = 0; i < E; ++i) d[i] -= T.piv;

  // ---- the iteration: every warp of the block holds the same T for its 8 columns
#pragma unroll 1
  for (int pass = 0; pass < kNtMaxPasses; ++pass) {
    if (__all_sync(0xffffffffu, T.done)) break;
    if (MAG) wid = nt_width<Q4, true>(T.piv + T.off, lam);
    const float tol = kTolRel * (MAG ? fminf(wid, fmaxf(T.piv + T.off, 0.0f)) : wid);
    float ct[2] = {0.f, 0.f}, cm[2] = {0.f, 0.f}, s1[2] = {0.f, 0.f}, s2[2] = {0.f, 0.f}, s3[2] = {0.f, 0.f};
    const float off = T.off;
#pragma unroll
    for (int g = 0; g < E / 4; ++g) {
      if (g < R.groups) {
#pragma unroll
        for (int j = 0; j < 4; ++j) nt_classify<Q4>(d[4 * g + j] - off, wid, ct[j & 1], cm[j & 1], s1[j & 1], s2[j & 1], s3[j & 1]);
      }
    }
    float v[NV];
    v[0] = __uint_as_float((uint32_t)(int)(ct[0] + ct[1]) | ((uint32_t)(int)(cm[0] + cm[1]) << 16));
    v[1] = s1[0] + s1[1];
    if (Q4) { v[NV > 2 ? 2 : 0] = s2[0] + s2[1]; v[NV > 3 ? 3 : 0] = s3[0] + s3[1]; }
    col_allsum<NV, true>(v, red(phase++), warps);
    if (!T.done) {
      const uint32_t packed = __float_as_uint(v[0]);
      nt_step<Q4, MAG>(T, (int)(packed & 0xffffu), (int)(packed >> 16), v[1], Q4 ? v[NV > 2 ? 2 : 0] : 0.0f,
                       Q4 ? v[NV > 3 ? 3 : 0] : 0.0f, k, lam, lam3, wid, tol);
      if (T.repiv) {
        const ColRows<Off> Rp = R.again();
        const ColMatrix<Off> Xp(A.theta, A.ld_theta, col0, c, Rp, cols, P.status);
#pragma unroll
        for (int g = 0; g < E / 4; ++g) {
          if (g < Rp.groups) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int i = 4 * g + j;
              const float xv = Xp.template load<false, true>(i, Rp);
              d[i] = Rp.in(i) ? (MAG ? fabsf(xv) : xv) - T.piv : -INFINITY;
            }
            asm volatile("" ::: "memory");     // loads of the next group stay behind: the registers are full here
          }
        }
      }
    }
  }
  int flags = 0;
  if (!T.done) { flags |= TK_FLAG_NOT_CONVERGED; T.a0 = k; T.b0 = k; }
  if (T.b0 <= T.a0) { T.a0 = k; T.b0 = k; }
  const bool block = T.b0 > T.a0;
  if (MAG) wid = nt_width<Q4, true>(T.piv + T.off, lam);

  // ---- row state (see tk_newton.cu: without a block any pivot between the (k+1)-th and the k-th key serves)
  float piv_state = T.piv, off_state = T.off;
  {
    const bool want_p = !block && !early;
    const bool safe = wid > 9.6e-7f * (fabsf(T.piv) + fabsf(T.off));
    const bool scan = want_p && !safe;
    if (__any_sync(0xffffffffu, scan)) {       // the same in every warp
      float cmin = INFINITY;
      const ColRows<Off> Rp = R.again();
      const ColMatrix<Off> Xp(A.theta, A.ld_theta, col0, c, Rp, cols, P.status);
#pragma unroll
      for (int g = 0; g < E / 4; ++g) {
        if (g < Rp.groups) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int i = 4 * g + j;
            const float xv = Xp.template load<false, true>(i, Rp);
            if (Rp.in(i) && d[i] - T.off >= wid) cmin = fminf(cmin, MAG ? fabsf(xv) : xv);
          }
          asm volatile("" ::: "memory");
        }
      }
#pragma unroll
      for (int o = kColC; o < 32; o <<= 1) cmin = fminf(cmin, __shfl_xor_sync(0xffffffffu, cmin, o));
      if (warps > 1) {
        float* rb = red(phase++);
        if (lane < kColC) rb[warp * kColC + lane] = cmin;
        __syncthreads();
        for (int w = 0; w < warps; ++w) cmin = fminf(cmin, rb[w * kColC + lane % kColC]);
      }
      if (scan) piv_state = cmin;
    }
    if (want_p && safe) piv_state = (T.piv + T.off) + 0.5f * wid;
    if (!block) off_state = 0.0f;
  }
  if (P.state_out && col_ok && threadIdx.x < kColC) {
    tk_rowstate st;
    st.pivot = piv_state; st.offset = off_state; st.a = T.a0; st.b = T.b0;
    P.state_out[col] = st;
  }
  if (P.status) {
    if (bad) flags |= TK_FLAG_NONFINITE;
    if (flags) atomicOr(P.status, flags);
  }
  if (P.out == nullptr) return;                // the row state alone was asked for (a VJP without one)

  // ---- dual map
  const ColRows<Off> Ro = R.again();
  const ColMatrix<Off> O(A.out, A.ld_out, col0, c, Ro, cols, P.status);
  const ColMatrix<Off> Xo(A.theta, A.ld_theta, col0, c, Ro, cols, P.status);
  if (!MAG) {
    const float shift = -T.off * inv_lam;
    const bool times_x = P.mode == TK_TOPK;
    col_each<E>(Ro, [&](int i, auto fast) {
      const float a = __saturatef(fmaf(d[i], inv_lam, shift));
      float y = Q4 ? a * a * a : a;
      if (times_x) y *= Xo.template load<decltype(fast)::value, true>(i, Ro);
      O.template store<decltype(fast)::value>(i, Ro, col_ok, y);
      if (times_x && (i & 3) == 3) asm volatile("" ::: "memory");
    });
  } else {
    Math M = make_math(P);
    M.q4 = Q4; M.mag = true; M.gen = false;
    const float off = T.off;
    col_each<E>(Ro, [&](int i, auto fast) {
      const float xv = Xo.template load<decltype(fast)::value, true>(i, Ro);
      const float t = d[i] - off;
      float v = 0.0f;
      if (t >= wid) v = M.vtop(fabsf(xv));
      else if (t > 0.0f) v = M.rho(t);
      O.template store<decltype(fast)::value>(i, Ro, col_ok, signbit(xv) ? -v : v);
      if ((i & 3) == 3) asm volatile("" ::: "memory");
    });
  }
}

// VJP from saved row state (the sums and formulas of tk_vjp_team.cu), theta and the cotangent in registers.  The mask
// keeps rho' in the place of theta once an element is classified; the other modes classify again.
template <int E, bool Q4, int MODE, class Off>
__global__ void __maxnreg__(E <= 16 ? (MODE == TK_MASK ? 56 : 64) : 112) tk_cols_vjp_kernel(const Problem P, const ColArgs A) {
  constexpr bool MAG = MODE == TK_TOPKMAG, TOPK = MODE == TK_TOPK, MASK = MODE == TK_MASK;
  __shared__ float4 red_s[2][kColMaxWarps * kColC];
  const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  const int n = P.n;
  const long long cols = P.rows, col0 = (long long)blockIdx.x * kColC;
  const bool col_ok = col0 + lane % kColC < cols;
  const int c = col_ok ? lane % kColC : (int)(cols - 1 - col0);
  const ColRows<Off> R(n);
  const ColMatrix<Off> X(A.theta, A.ld_theta, col0, c, R, cols, P.status);
  const ColMatrix<Off> GM(A.gout, A.ld_gout, col0, c, R, cols, P.status);
  overlap_wait();
  float x[E], g[E];
  col_each<E>(R, [&](int i, auto fast) {
    x[i] = X.template load<decltype(fast)::value>(i, R);
    g[i] = GM.template load<decltype(fast)::value>(i, R);
  });
  if (A.copy) {
    const ColRows<Off> Rc = R.again();
    const ColMatrix<Off> C(A.copy, cols, col0, c, Rc, cols, P.status);
    col_each<E>(Rc, [&](int i, auto fast) { C.template store<decltype(fast)::value>(i, Rc, col_ok, x[i]); });
  }
  const tk_rowstate st = P.state_in[col0 + c];
  const bool has_block = st.b > st.a;
  const float piv = st.pivot, off = st.offset;
  Math M = make_math(P);
  M.q4 = Q4; M.mag = MAG; M.gen = false;
  const float wid = has_block ? M.width(piv + off) : 0.0f;
  const float fm = (float)(P.k - st.a);        // members of the pooled block with w = 1
  auto key_t = [&](float xv) -> float { return ((MAG ? fabsf(xv) : xv) - piv) - off; };
  // rho' of an element of the pooled block, else 0.  (without a block the width is 0: nothing is strictly inside)
  auto drho = [&](float t) -> float { return t > 0.0f && !(t >= wid) ? M.drho(t) : 0.0f; };
  auto chi_of = [&](float xv) -> float { return MAG ? (signbit(xv) ? -1.0f : 1.0f) : (TOPK ? xv : 1.0f); };
  float ratio = 0.0f, delta = 0.0f;
  const bool any = __any_sync(0xffffffffu, has_block);            // the same in every warp: same columns
  if (any || MASK) {
    float AD[2] = {0.f, 0.f};
#pragma unroll
    for (int q = 0; q < E / 4; ++q) {
      if (q < R.groups) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int i = 4 * q + j;
          float dr = drho(key_t(x[i]));
          if (q >= R.fast && !R.in(i)) dr = 0.0f;
          AD[0] = fmaf(MASK ? dr : dr * chi_of(x[i]), g[i], AD[0]);
          AD[1] += dr;
          if (MASK) x[i] = dr;
        }
      }
    }
    if (any) {
      col_allsum<2, false>(AD, reinterpret_cast<float*>(red_s[0]), warps);
      float D = AD[1];
      if (MAG) D += fm;
      const bool ok = has_block && D > 0.0f;
      ratio = ok ? AD[0] / D : 0.0f;
      float A2[2] = {0.f, 0.f};
#pragma unroll
      for (int q = 0; q < E / 4; ++q) {
        if (q < R.groups) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int i = 4 * q + j;
            float dr = MASK ? x[i] : drho(key_t(x[i]));
            if (!MASK && q >= R.fast && !R.in(i)) dr = 0.0f;
            A2[0] = fmaf(dr, MASK ? g[i] - ratio : fmaf(chi_of(x[i]), g[i], -ratio), A2[0]);
          }
        }
      }
      col_allsum<2, false>(A2, reinterpret_cast<float*>(red_s[1]), warps);
      if (MAG) A2[0] -= fm * ratio;
      delta = ok ? A2[0] / D : 0.0f;
    }
  }
  const ColRows<Off> Ro = R.again();
  const ColMatrix<Off> O(A.out, A.ld_out, col0, c, Ro, cols, P.status);
  col_each<E>(Ro, [&](int i, auto fast) {
    float o;
    if (MASK) {
      o = x[i] * ((g[i] - ratio) - delta);
    } else {
      const float xv = x[i], t = key_t(xv), dr = drho(t);
      const bool top = has_block ? t >= wid : (MAG ? fabsf(xv) : xv) - piv >= 0.0f;
      float f = 0.0f;
      if (MAG) f = top ? g[i] * M.top_slope(fabsf(xv)) : 0.0f;
      if (TOPK) f = g[i] * (top ? 1.0f : ((has_block && t > 0.0f) ? M.rho(t) : 0.0f));
      o = fmaf((MAG && signbit(xv)) ? -dr : dr, fmaf(chi_of(xv), g[i], -ratio) - delta, f);
    }
    O.template store<decltype(fast)::value>(i, Ro, col_ok, o);
  });
}

// warps of a block whose lanes hold up to E rows each
inline int col_warps(int n, int E) { return (n + kColSlices * E - 1) / (kColSlices * E); }

template <int E, class Off>
cudaError_t cols_fwd(const Problem& P, const ColArgs& A, float zq, cudaStream_t stream) {
  const unsigned blocks = (unsigned)((P.rows + kColC - 1) / kColC);
  const int threads = 32 * col_warps(P.n, E);
  cudaError_t err;
  const bool mag = P.mode == TK_TOPKMAG;
  if (P.q4) {
    if (mag) err = launch_overlapped(tk_cols_fwd_kernel<E, true, true, Off>, blocks, threads, 0, stream, P, A, zq);
    else err = launch_overlapped(tk_cols_fwd_kernel<E, true, false, Off>, blocks, threads, 0, stream, P, A, zq);
  } else {
    if (mag) err = launch_overlapped(tk_cols_fwd_kernel<E, false, true, Off>, blocks, threads, 0, stream, P, A, zq);
    else err = launch_overlapped(tk_cols_fwd_kernel<E, false, false, Off>, blocks, threads, 0, stream, P, A, zq);
  }
  return err;
}

template <int E, class Off>
cudaError_t cols_vjp(const Problem& P, const ColArgs& A, cudaStream_t stream) {
  const unsigned blocks = (unsigned)((P.rows + kColC - 1) / kColC);
  const int threads = 32 * col_warps(P.n, E);
  cudaError_t err;
  if (P.q4) {
    if (P.mode == TK_MASK) err = launch_overlapped(tk_cols_vjp_kernel<E, true, TK_MASK, Off>, blocks, threads, 0, stream, P, A);
    else if (P.mode == TK_TOPK) err = launch_overlapped(tk_cols_vjp_kernel<E, true, TK_TOPK, Off>, blocks, threads, 0, stream, P, A);
    else err = launch_overlapped(tk_cols_vjp_kernel<E, true, TK_TOPKMAG, Off>, blocks, threads, 0, stream, P, A);
  } else {
    if (P.mode == TK_MASK) err = launch_overlapped(tk_cols_vjp_kernel<E, false, TK_MASK, Off>, blocks, threads, 0, stream, P, A);
    else if (P.mode == TK_TOPK) err = launch_overlapped(tk_cols_vjp_kernel<E, false, TK_TOPK, Off>, blocks, threads, 0, stream, P, A);
    else err = launch_overlapped(tk_cols_vjp_kernel<E, false, TK_TOPKMAG, Off>, blocks, threads, 0, stream, P, A);
  }
  return err;
}

// offsets inside a matrix fit 32 bits of bytes
inline bool col_small(int n, long long ld) { return (long long)n * ld < (1ll << 30); }

}  // namespace

// Longest column these kernels hold: 16 warps of 32 rows per lane.
int cols_direct_max_n() { return kColSlices * kColMaxWarps * 32; }

// Forward pass (p = 2 or 4/3, no permutation output) on column-strided data; P.rows = number of columns.  P.out may be null:
// the row state alone.
cudaError_t launch_cols_fwd(const Problem& P, long long ld_theta, long long ld_out, float* copy, cudaStream_t stream) {
  ColArgs A = {};
  A.theta = P.theta; A.ld_theta = ld_theta; A.out = P.out; A.ld_out = ld_out; A.copy = copy;
  const double tail = ((double)P.k - 0.5) / (double)P.n;
  const float zq = upper_normal_quantile(P.mode == TK_TOPKMAG ? 0.5 * tail : tail);
  const bool small = col_small(P.n, ld_theta) && col_small(P.n, ld_out);
  if (P.n <= kColSlices * 16) return small ? cols_fwd<16, uint32_t>(P, A, zq, stream) : cols_fwd<16, uint64_t>(P, A, zq, stream);
  return small ? cols_fwd<32, uint32_t>(P, A, zq, stream) : cols_fwd<32, uint64_t>(P, A, zq, stream);
}

// VJP from saved row state on column-strided data.
cudaError_t launch_cols_vjp(const Problem& P, long long ld_theta, long long ld_gout, long long ld_out, float* copy,
                            cudaStream_t stream) {
  ColArgs A = {};
  A.theta = P.theta; A.ld_theta = ld_theta; A.gout = P.gout; A.ld_gout = ld_gout; A.out = P.out; A.ld_out = ld_out;
  A.copy = copy;
  const bool small = col_small(P.n, ld_theta) && col_small(P.n, ld_gout) && col_small(P.n, ld_out);
  if (P.n <= kColSlices * kColMaxWarps * 16) return small ? cols_vjp<16, uint32_t>(P, A, stream) : cols_vjp<16, uint64_t>(P, A, stream);
  return small ? cols_vjp<32, uint32_t>(P, A, stream) : cols_vjp<32, uint64_t>(P, A, stream);
}

}  // namespace tk
