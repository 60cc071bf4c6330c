// tk_w.cu -- the relaxed operator for any sorted w (Sec. 3: LP forms of sort and rank over the
// permutahedron P(w); Sec. 4 with phi(x) = x):
//   y_R(x, w) = argmax_{y in P(w)} <x, y> - R(y) = grad R*(x - u*),  u* = v*_{sigma^-1},
//   v* = argmin_{v_1 >= .. >= v_n} sum_i r*(s_i - v_i) + w_i v_i                     (Prop. 5),
// and its VJP in x (Prop. 7).  With w = 1_k this is the relaxed top-k mask, which the other kernels
// solve through its single pooled block; a general w pools many blocks, so this one runs pool-
// adjacent-violators itself, by divide and conquer over the lanes of a row's team (E = 8 or 16
// consecutive ranks per lane):
//   1. the row's KEYS alone are sorted, descending (network in registers, shuffles, with several warps
//      per row the last stages through shared memory);
//   2. prefix sums of the sorted keys (about a pivot, in fp64) and of w make the value of ANY
//      candidate block [lo, hi) an O(1) computation: gamma = (sum s - lambda sum w) / N for p = 2,
//      the root of N g^3 - 3 S1 g^2 + 3 S2 g - S3 + lambda^3 sum w = 0 for p = 4/3 (App. A.6);
//   3. every lane runs sequential PAV on its E ranks (block heads: a bit mask in a register, block
//      values in shared memory), then neighbouring solutions are joined pairwise, log2(lanes) levels.
//      Joining two solved halves at rank m pools ONE block [a, b) around m or none: the left blocks
//      with a value below its own value gamma and the right blocks above it.  gamma is the root of a
//      decreasing function of one variable, found by the same iteration as the top-k threshold:
//      from a point tau, the set it selects and the exact value of that set, and when that does not
//      settle inside a bracket; it ends when a set reproduces itself.  Pooling a violating pair is
//      always part of the solution (App. B.2), so the result is the partition sequential PAV ends with;
//   4. y^s_i = rho(s_i - gamma_B(i)) is computed rank by rank; every element of the row then finds its
//      rank by binary search of its key and picks its result up.  The VJP sends the cotangent through
//      the same ranks: D_B = sum rho', A_B = sum rho' g^s come from prefix sums again.  Equal keys share
//      their result in the forward pass; in the VJP a warp hands out the ranks of a run of equal keys
//      in index order (the stable sort's order), chunk by chunk.
// A warp holds 32/G rows of up to E G elements (G = 1..32 lanes), or 2 / 4 warps one row.
//
// What bounds it: issue slots (67 % at n = 512, p = 2, with 27 % of the warps an SM can hold: the
// fp64 prefix sums and block values are 20 bytes of shared memory per element, 20 warps per SM) -- not
// memory (DRAM 4 %).  A warp spends a third of its time joining, a quarter in the serial PAV, a
// quarter in the sort and the rank search.  8192 x 512, w a ramp, p = 2, forward + VJP: 328 + 359 us
// when a block of 256 threads sorted (key, index) words through shared memory and merged all blocks
// of the row in rounds (barriers, and a merge of m ranks took m rounds in the worst case); 82 + 116 us now.
#include "tk_common.cuh"
#include "tk_key_sort.cuh"

namespace tk {

namespace {

constexpr int kWMaxN = 2048;
constexpr int kWFar = 1 << 20;   // a rank past every row

// slot of rank r in a per-rank array: one word of padding per lane (E ranks), so that the lanes of a warp walk
// their ranks without bank conflicts
template <int E>
__device__ __forceinline__ int wp(int r) { return r + r / E; }

// small non-negative integer -> double without the conversion unit (which takes a quarter of the rate of an add)
__device__ __forceinline__ double w_dbl(int i) {
  return __hiloint2double(0x43300000, i) - 4503599627370496.0;
}

// Root of f(g) = N g^3 + 3 M2 g + c (M2 >= 0: increasing), the block's cubic about its own mean: fp32
// Cardano (written without cancellation) as the start, Newton in fp64 from there.
__device__ __forceinline__ double w_cubic_root(double N, double M2, double c) {
  if (c == 0.0) return 0.0;
  const float inv_n = 1.0f / (float)N;
  const float p3 = (float)M2 * inv_n, q = (float)c * inv_n;             // h^3 + 3 p3 h + q = 0
  const float R = sqrtf(fmaf(0.25f * q, q, p3 * p3 * p3));
  const float A = cbrtf(0.5f * fabsf(q) + R);
  const float B = A > 0.0f ? p3 / A : 0.0f;
  const float den = A * A + p3 + B * B;
  double g = (den > 0.0f && isfinite(den)) ? (double)(-q / den) : 0.0;
  if (!(den > 1e-30f) || !isfinite(den)) g = c > 0.0 ? -cbrt(c / N) : cbrt(-c / N);   // outside fp32's range
#pragma unroll 1
  for (int it = 0; it < 60; ++it) {
    const double f = (N * g * g + 3.0 * M2) * g + c;
    const double fp = 3.0 * (N * g * g + M2);
    if (!(fp > 0.0)) break;
    const double st = f / fp;
    g -= st;
    if (!(fabs(st) > 1e-15 * fabs(g))) break;
    if (it > 2 && !(fabs(st) > 4e-15 * fabs(g))) break;
  }
  return g;
}

// Per-rank arrays of one row: block values at the heads; prefix sums about the pivot, inclusive, in the rank's slot
// within the lane's own E ranks, and in slot E of a lane (the padding word) what all lanes before it add up to.
struct WRow {
  double* val;
  const double* p1;               // p = 2: prefix of d - lambda w; p = 4/3: of d
  const double* p2;               // p = 4/3: of d^2, d^3, w
  const double* p3;
  const double* pw;
  const float* s;                 // p = 4/3: the sorted keys, and whether they lie far apart
  bool wide;
};

template <int E>
__device__ __forceinline__ double w_range(const double* p, int a, int b) {   // sum over the ranks [a, b)
  const int lb = (b - 1) / E, la = a / E;
  double v = p[wp<E>(b - 1)];
  if (la != lb) v += p[lb * (E + 1) + E] - p[la * (E + 1) + E];
  return (a & (E - 1)) ? v - p[wp<E>(a - 1)] : v;
}

template <int E, bool Q4>
__device__ __forceinline__ double w_block_value(const WRow& A, int a, int b, double lam3) {
  const double N = (double)(b - a);
  const double S1 = w_range<E>(A.p1, a, b);
  if (!Q4) return S1 / N;
  const double W = w_range<E>(A.pw, a, b), S2 = w_range<E>(A.p2, a, b), S3 = w_range<E>(A.p3, a, b);
  const double mu = S1 / N;
  double M2 = fmax(S2 - S1 * mu, 0.0), M3 = S3 - 3.0 * mu * S2 + 2.0 * mu * mu * S1;
  if (A.wide) {
    // The moments about the block's mean are differences of prefix sums about the row's pivot: noise, for keys close together
    // and far from it (entries masked with -1e9).  The block's own keys bound them: within a range of r, N r^2 / 4 and
    // N r^3 / (6 sqrt 3).  Without that the noise decides which blocks pool, and the joins take many more rounds.
    const double r = (double)A.s[wp<E>(a)] - (double)A.s[wp<E>(b - 1)], nr2 = N * r * r, top3 = 0.0963 * nr2 * r;
    M2 = fmin(M2, 0.25 * nr2);
    M3 = fmin(fmax(M3, -top3), top3);
  }
  // sum (g - d_i)^3 + lam^3 W = 0 with g = mu + h:  N h^3 + 3 M2 h - M3 + lam^3 W = 0
  return mu + w_cubic_root(N, M2, lam3 * W - M3);
}

template <int W>
__device__ __forceinline__ void w_sync() {
  if (W == 1) __syncwarp(); else __syncthreads();
}

// Shared memory of a team (one warp's rows, or the row of W warps; see the carving in the kernel), teams per thread
// block and the resident blocks that memory leaves room for.  E = 16: 20 warps per SM for p = 2, 8 for p = 4/3.  E = 8
// (launches short of warps): every team a block of its own, so that they spread over the SMs.
template <int E, int W, bool Q4>
struct WGeom {
  static constexpr int SLOTS = 32 * W * (E + 1);
  static constexpr int TEAM_BYTES = SLOTS * 8 * (Q4 ? 5 : 2) + SLOTS * 4 + (W > 1 ? 256 : 0);
  static constexpr int TEAMS = W == 1 && !Q4 && E == 16 ? 4 : 1;
  static constexpr int MIN_BLOCKS = (Q4 ? 8 : 20) / (TEAMS * W);
  static constexpr int THREADS = 32 * W * TEAMS;
};

template <int E, int G, int W, bool Q4, bool VJP>
__global__ void __launch_bounds__(WGeom<E, W, Q4>::THREADS, WGeom<E, W, Q4>::MIN_BLOCKS)
    tk_w_kernel(const Problem P, const float* w_all, const int w_shared) {
  static_assert(W == 1 || G == 32, "several warps per row: every lane of them belongs to the row");
  constexpr int T = G * W, R = W > 1 ? 1 : 32 / G;                // lanes per row, rows per team
  constexpr int N = T * E, NP = N + T;                            // padded row length, its slots
  constexpr int TL = 32 * W;                                      // lanes of a team
  constexpr int SLOTS = R * NP;
  constexpr int TEAMS = WGeom<E, W, Q4>::TEAMS, TEAM_BYTES = WGeom<E, W, Q4>::TEAM_BYTES;
  constexpr int LOG_N = (N == 8 ? 3 : N == 16 ? 4 : N == 32 ? 5 : N == 64 ? 6 : N == 128 ? 7 : N == 256 ? 8 : N == 512 ? 9 : N == 1024 ? 10 : 11);
  extern __shared__ __align__(16) unsigned char w_smem[];
  __shared__ double rcp[E + 1];                                   // 1 / i
  if (threadIdx.x <= E) rcp[threadIdx.x] = 1.0 / (double)max((int)threadIdx.x, 1);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int team = W == 1 ? warp : 0;
  const int tid = W == 1 ? lane : (int)threadIdx.x;               // lane of the team
  const int rl = W == 1 ? lane / G : 0, lig = W == 1 ? lane % G : tid;   // row within the team, lane within the row
  const int n = P.n;
  const long long row0 = ((long long)blockIdx.x * TEAMS + team) * R;
  if (row0 >= P.rows) return;                                     // the whole team
  const int rows_here = (int)(P.rows - row0 < (long long)R ? P.rows - row0 : (long long)R);
  const int total = rows_here * n;                                // elements of the team's rows, contiguous in memory
  const long long first = row0 * (long long)n;
  // (every index into theta, the cotangent and the outputs below lies in [first, first + total))
  if (!TK_IN_BOUNDS(first, total, P.rows * (long long)n, P.status)) return;
  const double lam = (double)P.lam, lam3 = lam * lam * lam;
  const float inv_lam = P.inv_lam;

  unsigned char* ptr = w_smem + (size_t)team * TEAM_BYTES;
  double* val = reinterpret_cast<double*>(ptr); ptr += SLOTS * 8;
  double* p1 = reinterpret_cast<double*>(ptr); ptr += SLOTS * 8;
  double* p2 = p1; double* p3 = p1; double* pw = p1;
  if (Q4) {
    p2 = reinterpret_cast<double*>(ptr); ptr += SLOTS * 8;
    p3 = reinterpret_cast<double*>(ptr); ptr += SLOTS * 8;
    pw = reinterpret_cast<double*>(ptr); ptr += SLOTS * 8;
  }
  float* s = reinterpret_cast<float*>(ptr); ptr += SLOTS * 4;     // w, then the sorted keys, then the cotangent by rank
  float* xs = reinterpret_cast<float*>(p1);                       // the rows as they are in memory, until the prefix sums
  double* redd = reinterpret_cast<double*>(ptr);                  // W > 1: exchange between the warps
  int* redi = reinterpret_cast<int*>(redd + 16);
  const int rbase = rl * NP;                                      // this lane's row in the per-rank arrays
  const int base = lig * E;                                       // its first rank
  const int sbase = rbase + lig * (E + 1);                        // and that rank's slot
  WRow A;
  A.val = val + rbase; A.p1 = p1 + rbase; A.p2 = p2 + rbase; A.p3 = p3 + rbase; A.pw = pw + rbase; A.s = s + rbase; A.wide = false;
  // row of element e of the team's rows: exact for e < 2^16 (n == 1 would overflow the multiplier)
  const uint32_t magic = n > 1 ? 0xffffffffu / (uint32_t)n + 1u : 0u;
  auto row_of = [&](int e) -> int { return R == 1 ? 0 : (n > 1 ? (int)__umulhi((uint32_t)e, magic) : e); };

  overlap_wait();
  // ---- theta as it lies in memory, w by rank (in the keys' array, which is free until the sort is done).  Every
  // load is unconditional (past the end the last element again), so the loads of a lane are all in flight at once
  int flags = 0;
  if (VJP && 32 * tid < total)                                    // the cotangent is wanted after the solve: into L2 by then
    asm volatile("prefetch.global.L2 [%0];" ::"l"(P.gout + first + 32 * tid));
  {
    float v[E];
    const float* src = P.theta + first;
#pragma unroll
    for (int it = 0; it < E; ++it) v[it] = src[min(tid + it * TL, total - 1)];
#pragma unroll
    for (int it = 0; it < E; ++it) {
      if (!(fabsf(v[it]) < INFINITY)) flags = TK_FLAG_NONFINITE;
      if (tid + it * TL < total) xs[tid + it * TL] = v[it];
    }
    if (w_shared) {
      for (int i = tid; i < n; i += TL) s[wp<E>(i)] = w_all[i];
    } else {
      src = w_all + first;
#pragma unroll
      for (int it = 0; it < E; ++it) v[it] = src[min(tid + it * TL, total - 1)];
#pragma unroll
      for (int it = 0; it < E; ++it) {
        const int e = tid + it * TL, r = row_of(e);
        if (e < total) s[r * NP + wp<E>(e - r * n)] = v[it];
      }
    }
  }
  w_sync<W>();

  // ---- 1. sort the keys.  Which lane takes which element is free: strided, rotated per lane (no bank conflicts)
  float r[E];
#pragma unroll
  for (int i = 0; i < E; ++i) {
    const int e = lig + T * ((i + lane) & (E - 1));
    const bool in = e < n;
    const float x = (in && rl < rows_here) ? xs[rl * n + e] : 0.0f;
    r[i] = in ? sort_key(x, false) : -INFINITY;                   // slots past the row sort last
  }
  group_sort_keys<G, E>(r, lig & 31, 0xffffffffu);
  if (W > 1) {
    // the last levels of the network across warps, through the block values' array (free until step 2)
    float* ex = reinterpret_cast<float*>(val);
#pragma unroll 1
    for (int size = 64; size <= T; size <<= 1) {
#pragma unroll 1
      for (int st = size - 1; st >= 32; st = st == size - 1 ? size >> 2 : st >> 1) {   // the mirror, then strides
        const bool mirror = st == size - 1;
        const bool keepmax = (tid & (mirror ? size >> 1 : st)) == 0;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < E; ++i) ex[i * T + tid] = r[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < E; ++i) {
          const float o = ex[(mirror ? E - 1 - i : i) * T + (tid ^ st)];
          r[i] = keepmax ? fmaxf(r[i], o) : fminf(r[i], o);
        }
      }
#pragma unroll 1
      for (int st = 16; st >= 1; st >>= 1) {
        const bool keepmax = (lane & st) == 0;
#pragma unroll
        for (int i = 0; i < E; ++i) {
          const float o = __shfl_xor_sync(0xffffffffu, r[i], st);
          r[i] = keepmax ? fmaxf(r[i], o) : fminf(r[i], o);
        }
      }
      lane_merge_f<E>(r);
    }
    __syncthreads();
  }
  w_sync<W>();                                                    // the rows have been taken out of p1

  // ---- 2. prefix sums about a pivot (a key near the middle), singleton values.  p = 4/3: the key of rank n / 2 itself.  The
  // first key of that rank's lane is up to 15 ranks away, in a row of a few keys the largest one; the third powers of keys
  // far below it cancel to noise, and one far key decides about all the others: (x, -1e9, -1e9) came out thousands off.
  // (p = 2 has no powers to lose: 3 % slower with it, 8192 x 512.)
  const int plane = (n / 2) / E;
  float pivf = r[0];
  if (Q4) {
#pragma unroll
    for (int i = 1; i < E; ++i)
      if (i == (n / 2) % E) pivf = r[i];
  }
  if (W > 1 && tid == plane) redd[0] = (double)pivf;
  pivf = __shfl_sync(0xffffffffu, pivf, W == 1 ? rl * G + plane : plane & 31);
  if (W > 1) {
    __syncthreads();
    pivf = (float)redd[0];
    __syncthreads();
  }
  const double piv = (double)pivf;
  const int cl = min(max(n - base, 0), E);                        // ranks of this lane that exist
  // the sum of `mine` over the row's lanes before this one, into the padding word of the lane's slots
  auto lanes_before = [&](double mine, double* p) {
    double inc = mine;
#pragma unroll
    for (int o = 1; o < G; o <<= 1) {
      const double up = __shfl_up_sync(0xffffffffu, inc, o, G);
      if ((lig & (G - 1)) >= o) inc += up;
    }
    double before = inc - mine;
    if (Q4) {                                                     // (that loses the sum of third powers before a lane of far keys)
      before = __shfl_up_sync(0xffffffffu, inc, 1, G);
      if ((lig & (G - 1)) == 0) before = 0.0;
    }
    if (W > 1) {
      if (lane == 31) redd[warp] = inc;
      __syncthreads();
#pragma unroll
      for (int wv = 0; wv < W - 1; ++wv) if (wv < warp) before += redd[wv];
      __syncthreads();
    }
    p[sbase + E] = before;
  };
  const float* wl = s + (w_shared ? 0 : rbase) + lig * (E + 1);
  {
    constexpr int NS = Q4 ? 4 : 1;
    double run[NS], reach = 0.0;                                  // p = 4/3: this lane's largest distance from the pivot
#pragma unroll
    for (int q = 0; q < NS; ++q) run[q] = 0.0;
#pragma unroll
    for (int i = 0; i < E; ++i) {
      if (i < cl) {
        const double d = (double)r[i] - piv, wi = (double)wl[i];
        const double h = Q4 ? d - lam * cbrt(wi) : d - lam * wi;  // p = 4/3: (g - d)^3 + lam^3 w = 0
        val[sbase + i] = h;
        if (!Q4) { run[0] += h; p1[sbase + i] = run[0]; }
        else {
          if (i == 0 || i == cl - 1) reach = fmax(reach, fabs(d));
          run[0] += d; run[NS > 1 ? 1 : 0] += d * d; run[NS > 2 ? 2 : 0] += d * d * d; run[NS > 3 ? 3 : 0] += wi;
          p1[sbase + i] = run[0]; p2[sbase + i] = run[NS > 1 ? 1 : 0];
          p3[sbase + i] = run[NS > 2 ? 2 : 0]; pw[sbase + i] = run[NS > 3 ? 3 : 0];
        }
      }
    }
    lanes_before(run[0], p1);
    if (Q4) {
      lanes_before(run[NS > 1 ? 1 : 0], p2); lanes_before(run[NS > 2 ? 2 : 0], p3); lanes_before(run[NS > 3 ? 3 : 0], pw);
      // (within 256 lambda of the pivot the moments' noise is below 1e-8 N lambda^3, and a row does without their bounds)
      const bool wide = !(reach <= 256.0 * lam);
      if (W > 1) A.wide = __syncthreads_or(wide) != 0;
      else A.wide = (__ballot_sync(0xffffffffu, wide) >> (rl * G) & (0xffffffffu >> (32 - G))) != 0u;
    }
  }
  w_sync<W>();                                                    // w has been read everywhere
#pragma unroll
  for (int i = 0; i < E; ++i) s[sbase + i] = r[i];

  // ---- 3a. sequential PAV on the lane's own ranks.  heads: bit i = rank base + i starts a block.
  // p = 2: the stack holds block sums, two values S / N are compared as S N' against S' N (no division in the
  // serial chain), and the heads' values are formed afterwards, all at once
  unsigned heads = 0;
  if (Q4) {
    if (cl > 0) {
      int top = 0, cs = 0, j = 1;                                 // last block on the stack; the one being formed is [cs, j)
      double vtop = 0.0, cv = val[sbase];
#pragma unroll 1
      for (;;) {
        if (heads && vtop < cv) {                                 // pool it with the block before
          cs = top;
          cv = w_block_value<E, Q4>(A, base + cs, base + j, lam3);
          heads ^= 1u << top;
          if (heads) { top = 31 - __clz((int)heads); vtop = val[sbase + top]; }
        } else {
          val[sbase + cs] = cv;
          heads |= 1u << cs;
          top = cs; vtop = cv;
          if (j >= cl) break;
          cs = j; cv = val[sbase + j]; ++j;
        }
      }
    }
  } else {
    // one step = one push or one merge, chosen by selects: the lanes stay together
    int top = -1, cs = 0, j = 1;
    double St = 0.0, S = val[sbase];
    bool run = cl > 0;
    while (__any_sync(0xffffffffu, run)) {
      const bool viol = heads != 0 && St * w_dbl(j - cs) < S * w_dbl(cs - top);
      const unsigned after = viol ? heads ^ (1u << top) : heads | (1u << cs);
      const int ntop = 31 - __clz((int)after);
      const double x = val[sbase + (viol ? max(ntop, 0) : min(j, E - 1))];
      if (run) {
        if (!viol) val[sbase + cs] = S;
        const double sum = S + St;
        St = viol ? x : S;
        S = viol ? sum : x;
        cs = viol ? top : j;
        run = viol || j < cl;
        j += viol ? 0 : 1;
        heads = after;
        top = ntop;
      }
    }
#pragma unroll
    for (int i = 0; i < E; ++i) {
      const unsigned rest = heads >> i >> 1;                      // heads behind this one
      const int len = rest ? __ffs((int)rest) : cl - i;
      if (heads >> i & 1u) {
        // S / len from 1 / len and one correction step
        const double c = rcp[len], v = val[sbase + i], q = v * c;
        val[sbase + i] = fma(fma(-q, w_dbl(len), v), c, q);
      }
    }
  }
  w_sync<W>();

  // ---- 3b. join neighbouring solutions
  int phase = 0;
  // smallest candidate of this lane's half and of the other half
  auto half_min = [&](int c, int half, int& other) -> int {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
      if (o < half) c = min(c, __shfl_xor_sync(0xffffffffu, c, o));
    if (half < 32) { other = __shfl_xor_sync(0xffffffffu, c, half); return c; }
    int* slot = redi + (phase & 1) * 4;
    ++phase;
    if (lane == 0) slot[warp] = c;
    __syncthreads();
    if (half == 32) { other = slot[warp ^ 1]; return slot[warp]; }
    other = min(slot[warp ^ 2], slot[warp ^ 3]);
    return min(slot[warp], slot[warp ^ 1]);
  };
  // this lane's candidate for the set that tau selects: left, its first block below tau; right, its first block
  // not above tau
  auto candidate = [&](bool left, double tau) -> int {
    unsigned mk = heads;
    int c = kWFar;
    if (left) {
      while (mk) {
        const int b = 31 - __clz((int)mk);
        if (!(val[sbase + b] < tau)) break;
        c = base + b; mk ^= 1u << b;
      }
    } else {
      while (mk) {
        const int b = __ffs((int)mk) - 1;
        if (!(val[sbase + b] > tau)) { c = base + b; break; }
        mk &= mk - 1;
      }
    }
    return c;
  };
#pragma unroll 1
  for (int half = 1; half < T; half <<= 1) {
    const bool left = (lig & half) == 0;
    const bool wide = W > 1 && half >= 32;                        // the halves are whole warps
    const int g0 = lig & ~(2 * half - 1);
    const int m = (g0 + half) * E, end = min(n, (g0 + 2 * half) * E);
    // last block of the left half, first of the right
    int c, o;
    if (left) c = heads ? -(base + 31 - __clz((int)heads)) : kWFar;
    else c = heads ? base + __ffs((int)heads) - 1 : kWFar;
    c = half_min(c, half, o);
    const int last = left ? -c : -o, frst = left ? o : c;
    double lo = 0.0, hi = 0.0;
    bool act = m < n && last >= 0 && frst < n;
    if (act) { lo = A.val[wp<E>(last)]; hi = A.val[wp<E>(frst)]; act = lo < hi; }
    if (!(wide ? __syncthreads_or(act) : __any_sync(0xffffffffu, act))) continue;
    // First guess: those two blocks alone (the end of the second as its lane knows it; any point starts the
    // iteration).  Then in turn the value of a set and the set that value selects, until a set comes back
    int pa = last, pb = min(frst + 1, end);
    if (!wide) {
      const unsigned rest = heads & (heads - 1);
      const int second = rest ? base + __ffs((int)rest) - 1 : min(base + E, n);
      pb = __shfl_sync(0xffffffffu, second, (lane & ~(2 * half - 1)) + ((act ? frst / E : 0) & (2 * half - 1)));
    }
    double tau = 0.0;
    int tries = 0;
#pragma unroll 1
    for (int it = 0; it < 200; ++it) {
      bool own = true, last_point = false;                        // own: tau is the value of [pa, pb)
      if (act) {
        const double nv = w_block_value<E, Q4>(A, pa, pb, lam3);
        if (tries < 8) tau = nv;
        else {
          // it has not settled: keep the root inside the bracket (lo, hi]
          own = false;
          if (tries > 8) {
            if (nv > tau) lo = tau; else hi = tau;
            own = nv > lo && nv <= hi;
          }
          const double mid = 0.5 * (lo + hi);
          last_point = !own && !(mid > lo && mid < hi);           // the bracket holds no point but hi
          tau = own ? nv : (last_point ? hi : mid);
        }
      }
      c = act ? candidate(left, tau) : kWFar;
      c = half_min(c, half, o);
      const int a = left ? c : o;
      int b = left ? o : c;
      if (b >= kWFar) b = end;
      if (act) {
        const bool none = a >= m || b <= m;                       // tau is not between the two halves' edges
        const bool done = last_point || (own && a == pa && b == pb);
        ++tries;
        if (none) {                                               // a first guess off the mark: to the bracket at once
          if (tries > 8) act = false;                             // (not finite: nothing to pool)
          tries = 8;
        } else if (!done) {
          pa = a; pb = b;
        } else {
          act = false;
          const double nv = last_point ? w_block_value<E, Q4>(A, a, b, lam3) : tau;
          if (left) {
            const int kk = a - base;                              // the block at a stays, those after it go
            if (kk < 0) heads = 0;
            else if (kk < E) { heads &= (2u << kk) - 1u; val[sbase + kk] = nv; }
          } else {
            const int kk = b - base;                              // the blocks before b go
            if (kk >= E) heads = 0;
            else if (kk > 0) heads &= ~((1u << kk) - 1u);
          }
        }
      }
      if (!(wide ? __syncthreads_or(act) : __any_sync(0xffffffffu, act))) break;
    }
    if (act) flags |= TK_FLAG_NOT_CONVERGED;                      // (the cap)
    if (wide) __syncthreads(); else __syncwarp();
  }

  // ---- 4. results by rank.  The head of the block that reaches into this lane's ranks from before
  int carry = heads ? base + 31 - __clz((int)heads) : -1;
#pragma unroll
  for (int o = 1; o < G; o <<= 1) {
    const int up = __shfl_up_sync(0xffffffffu, carry, o, G);
    if ((lig & (G - 1)) >= o) carry = max(carry, up);
  }
  {
    const int incl = carry;
    carry = __shfl_up_sync(0xffffffffu, carry, 1, G);
    if ((lig & (G - 1)) == 0) carry = -1;
    if (W > 1) {
      if (lane == 31) redi[warp] = incl;
      __syncthreads();
#pragma unroll
      for (int wv = 0; wv < W - 1; ++wv) if (wv < warp) carry = max(carry, redi[wv]);
      __syncthreads();
    }
  }
  double gam = carry >= 0 ? A.val[wp<E>(carry)] : 0.0;
#pragma unroll
  for (int i = 0; i < E; ++i) {                                   // r becomes (s - gamma) / lambda
    if (heads >> i & 1u) gam = val[sbase + i];
    r[i] = (float)(((double)r[i] - piv) - gam) * inv_lam;
  }

  // rank of a key: the number of larger keys of its row (the first of a run of equal ones)
  auto rank_of = [&](const float* sr, float key) -> int {
    int pos = 0;
#pragma unroll
    for (int st = 1 << (LOG_N - 1); st > 0; st >>= 1) {
      const int q = pos + st;
      if (sr[wp<E>(q - 1)] > key) pos = q;
    }
    return pos < n ? pos : n - 1;
  };
  if (!VJP) {
    float* ys = reinterpret_cast<float*>(p1);                     // the prefix sums have served
    w_sync<W>();
#pragma unroll
    for (int i = 0; i < E; ++i) ys[sbase + i] = Q4 ? r[i] * r[i] * r[i] : r[i];
    w_sync<W>();
#pragma unroll 4
    for (int it = 0; it < E; ++it) {                              // theta again (L1 / L2)
      const int e = tid + it * TL, ec = min(e, total - 1);
      const float x = __ldg(P.theta + first + ec);
      const int rr = row_of(ec);
      const float y = ys[rr * NP + wp<E>(rank_of(s + rr * NP, sort_key(x, false)))];
      if (e < total) P.out[first + e] = y;
    }
  } else {
    // ---- ranks of the team's elements, E per lane (theta again: L1 / L2)
    int rk[E];
    float gv[E];
    bool tie = false;
#pragma unroll
    for (int it = 0; it < E; ++it) gv[it] = __ldg(P.theta + first + min(tid + it * TL, total - 1));
#pragma unroll
    for (int it = 0; it < E; ++it) {
      const int rr = row_of(min(tid + it * TL, total - 1));
      const float* sr = s + rr * NP;
      const float key = sort_key(gv[it], false);
      const int rank = rank_of(sr, key);
      tie |= rank + 1 < n && sr[wp<E>(rank + 1)] == key;
      rk[it] = rr * NP + wp<E>(rank);
    }
#pragma unroll
    for (int it = 0; it < E; ++it) gv[it] = P.gout[first + min(tid + it * TL, total - 1)];
    tie = W > 1 ? __syncthreads_or(tie) != 0 : __any_sync(0xffffffffu, tie);
    if (tie) {
      // runs of equal keys: ranks in index order.  One warp walks the elements 32 at a time; cnt: how many of a
      // run have been placed; the slots found above go through the array `at`
      int* cnt = reinterpret_cast<int*>(p1);
      uint16_t* at = reinterpret_cast<uint16_t*>(val);            // the block values have served
      w_sync<W>();
#pragma unroll
      for (int it = 0; it < E; ++it) {
        const int e = tid + it * TL;
        if (e < total) at[e] = (uint16_t)rk[it];
      }
      for (int i = tid; i < SLOTS; i += TL) cnt[i] = 0;
      w_sync<W>();
      if (W == 1 || warp == 0) {
#pragma unroll 1
        for (int e0 = 0; e0 < total; e0 += 32) {
          const int e = e0 + lane;
          const int slot = e < total ? (int)at[e] : SLOTS + lane;
          const unsigned same = __match_any_sync(0xffffffffu, slot);
          const int before = __popc(same & ((1u << lane) - 1u));
          int placed = 0;
          if (e < total) placed = cnt[slot];
          __syncwarp();
          if (e < total) {
            if (before == 0) cnt[slot] = placed + __popc(same);
            const int rr = row_of(e);
            const int q = slot - rr * NP, rank = q - q / (E + 1);
            at[e] = (uint16_t)(rr * NP + wp<E>(min(rank + placed + before, n - 1)));
          }
          __syncwarp();
        }
      }
      w_sync<W>();
#pragma unroll
      for (int it = 0; it < E; ++it) {
        const int e = tid + it * TL;
        if (e < total) rk[it] = (int)at[e];
      }
    }
    w_sync<W>();                                                  // the keys, the prefix sums and the block values are free now
    float* gs = s;
#pragma unroll
    for (int it = 0; it < E; ++it) {
      const int e = tid + it * TL;
      if (e < total && TK_IN_BOUNDS(rk[it], 1, SLOTS, P.status)) gs[rk[it]] = gv[it];
    }
    w_sync<W>();
    // ---- sums of rho' and rho' g through each rank.  p = 2: rho' is the same everywhere, so its sum is the
    // block's length
    double t1 = 0.0, t2 = 0.0;
#pragma unroll
    for (int i = 0; i < E; ++i) {
      if (i < cl) {
        const double g = (double)gs[sbase + i];
        if (!Q4) t2 += g;
        else {
          const double dr = 3.0 * (double)r[i] * (double)r[i];
          t1 += dr;
          t2 += dr * g;
          p2[sbase + i] = t1;
        }
        p1[sbase + i] = t2;
      }
    }
    lanes_before(t2, p1);
    if (Q4) lanes_before(t1, p2);
    // ---- the first head after this lane's ranks: where its last block ends
    int next = heads ? base + __ffs((int)heads) - 1 : kWFar;
#pragma unroll
    for (int o = 1; o < G; o <<= 1) {
      const int dn = __shfl_down_sync(0xffffffffu, next, o, G);
      if ((lig & (G - 1)) + o < G) next = min(next, dn);
    }
    {
      const int incl = next;
      next = __shfl_down_sync(0xffffffffu, next, 1, G);
      if ((lig & (G - 1)) == G - 1) next = kWFar;
      if (W > 1) {
        if (lane == 0) redi[warp] = incl;
        __syncthreads();
#pragma unroll
        for (int wv = 1; wv < W; ++wv) if (wv > warp) next = min(next, redi[wv]);
      }
      if (next > n) next = n;
    }
    w_sync<W>();
    // ---- A_B / D_B of the blocks that start here, in the place of their values
#pragma unroll
    for (int i = 0; i < E; ++i) {
      if (heads >> i & 1u) {
        const unsigned after = heads >> i >> 1;
        const int lo = base + i, hi = after ? lo + __ffs((int)after) : next;
        double mean = (double)gs[sbase + i];      // a singleton's own mean is its g (two prefix sums would leave rounding noise)
        if (hi - lo > 1) {
          const double D = Q4 ? w_range<E>(A.p2, lo, hi) : w_dbl(hi - lo);
          mean = D > 0.0 ? w_range<E>(A.p1, lo, hi) / D : 0.0;
        }
        const float mh = (float)mean;             // as a sum of two floats: g - mean keeps its own relative accuracy
        reinterpret_cast<float2*>(val)[sbase + i] = make_float2(mh, (float)(mean - (double)mh));
      }
    }
    w_sync<W>();                                                  // the prefix sums are free again
    float2 mean = carry >= 0 ? reinterpret_cast<const float2*>(A.val)[wp<E>(carry)] : make_float2(0.0f, 0.0f);
#pragma unroll
    for (int i = 0; i < E; ++i) {
      if (heads >> i & 1u) mean = reinterpret_cast<const float2*>(val)[sbase + i];
      if (i < cl) {
        const float dr = Q4 ? 3.0f * r[i] * r[i] * inv_lam : inv_lam;
        gs[sbase + i] = dr * ((gs[sbase + i] - mean.x) - mean.y);
        // the cotangent pulled back to w, in w's own order: A_B / D_B for every rank of the block (a
        // singleton has y = w: its entry is g also where rho' vanishes)
        if (P.sorted_out && rl < rows_here) xs[rl * n + base + i] = mean.x;
      }
    }
    w_sync<W>();
#pragma unroll
    for (int it = 0; it < E; ++it) {
      const int e = tid + it * TL;
      if (e < total) {
        P.out[first + e] = gs[rk[it]];
        if (P.sorted_out) P.sorted_out[first + e] = xs[e];
      }
    }
  }
  if (flags && P.status) atomicOr(P.status, flags);
}

template <int E, int G, int W, bool Q4, bool VJP>
cudaError_t w_launch(const Problem& P, const float* w, int w_shared, cudaStream_t stream) {
  constexpr int smem = WGeom<E, W, Q4>::TEAM_BYTES * WGeom<E, W, Q4>::TEAMS;
  constexpr int rows_per_block = WGeom<E, W, Q4>::TEAMS * (W > 1 ? 1 : 32 / G);
  auto kern = tk_w_kernel<E, G, W, Q4, VJP>;
  if (smem > 48 * 1024) {
    static bool configured[64];
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= 64 || !configured[dev]) {
      err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      if (err != cudaSuccess) return err;
      if (dev >= 0 && dev < 64) configured[dev] = true;
    }
  }
  const unsigned blocks = (unsigned)((P.rows + rows_per_block - 1) / rows_per_block);
  return launch_overlapped(kern, blocks, WGeom<E, W, Q4>::THREADS, smem, stream, P, w, w_shared);
}

// Lanes and warps of a row of n elements with E ranks per lane.
template <int E, bool Q4, bool VJP>
cudaError_t w_launch_n(const Problem& P, const float* w, int w_shared, cudaStream_t stream) {
  const int n = P.n;
  if (n <= E) return w_launch<E, 1, 1, Q4, VJP>(P, w, w_shared, stream);
  if (n <= 2 * E) return w_launch<E, 2, 1, Q4, VJP>(P, w, w_shared, stream);
  if (n <= 4 * E) return w_launch<E, 4, 1, Q4, VJP>(P, w, w_shared, stream);
  if (n <= 8 * E) return w_launch<E, 8, 1, Q4, VJP>(P, w, w_shared, stream);
  if (n <= 16 * E) return w_launch<E, 16, 1, Q4, VJP>(P, w, w_shared, stream);
  if (n <= 32 * E) return w_launch<E, 32, 1, Q4, VJP>(P, w, w_shared, stream);
  if (n <= 64 * E) return w_launch<E, 32, 2, Q4, VJP>(P, w, w_shared, stream);
  return w_launch<E, 32, 4, Q4, VJP>(P, w, w_shared, stream);
}

}  // namespace

int w_max_n() { return kWMaxN; }

// Forward pass (P.what == W_FWD) or VJP (W_VJP, cotangent in P.gout; in theta, and in w when P.sorted_out
// is given) of the relaxed operator over P(w); w: device [w_rows * n], every row non-increasing; w_rows is 1 or P.rows.
cudaError_t launch_w(const Problem& P, const float* w, long long w_rows, cudaStream_t stream) {
  const int shared = w_rows == 1 ? 1 : 0;
  const bool vjp = P.what == W_VJP;
  // 16 ranks per lane take the fewest instructions per element, 8 the shorter serial chains and half the shared memory
  // per warp.  p = 4/3 (five fp64 arrays per rank, a cubic per pooled block in the serial chain) wants 8 at every number of
  // rows: 4194 x 250 forward + VJP 177 -> 132 us, 2097 x 1000 396 -> 304.  p = 2 wants 8 for rows of up to 8 (no padding:
  // 262144 x 8 67 -> 47 us) and while 16 would leave fewer than 8 warps per SM: 524 x 250 44 -> 35, 2097 x 250 (7 warps)
  // 51 -> 42, but 4194 x 250 (14 warps) 63 -> 68.
  if (P.q4) {
    if (P.n > 1024) return vjp ? w_launch<16, 32, 4, true, true>(P, w, shared, stream) : w_launch<16, 32, 4, true, false>(P, w, shared, stream);
    return vjp ? w_launch_n<8, true, true>(P, w, shared, stream) : w_launch_n<8, true, false>(P, w, shared, stream);
  }
  int lanes = 1;                               // of a row, with 16 ranks each
  while (16 * lanes < P.n) lanes <<= 1;
  const long long warps = (P.rows * lanes + 31) / 32;
  if (P.n <= 8 || (P.n <= 1024 && warps < (long long)sm_count() * 8))
    return vjp ? w_launch_n<8, false, true>(P, w, shared, stream) : w_launch_n<8, false, false>(P, w, shared, stream);
  return vjp ? w_launch_n<16, false, true>(P, w, shared, stream) : w_launch_n<16, false, false>(P, w, shared, stream);
}

}  // namespace tk
