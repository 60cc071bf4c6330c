// tk_sweeps.cu -- a fixed number of sweeps of the alternating projections (Algorithm 1, App. A.8; the iterations
// themselves are described in tk_dykstra.cu) on the ranks they can reach.
//
// Before the first sweep the iterate is in order everywhere but at the one pair of ranks (k - 1, k): the keys are
// sorted, and w = 1_k moves the first k of them by the same amount (phi = x) or factor (phi = x^2/2, p = 2).  A pair in
// order whose correction (dual) is 0 stays exactly as it is, and so do its neighbours' duals: a half-sweep changes
// only pairs next to a changed one.  After t sweeps nothing outside the ranks [k - 1 - 2t, k + 2t) has moved, and there
// y_i = rho(s_i - v_i) is w_i (phi = x) or follows from s_i alone.  So the sweeps need the order of at most 4t + 6 ranks,
// by one warp (or the row's lanes of one), and no block barrier in any sweep.
//
// Most of that reach is not used either: the changes stop at the edge of the pooled block.  The sweeps start on 2 ranks
// per lane around k and move to 4, 8, 16 when a correction within two ranks of the present edge (what one more
// sweep can cross) becomes non-zero; the iterate and the corrections pass through shared memory there.  The iterates are
// those of the sweeps over the whole row.
//
// The rest is the order: the row's keys are sorted and every element finds its place in the window by binary search
// (tk_rank.cuh).  Keys equal inside the window get their ranks in index order.
//
// What bounds it now is the sort and the search (issue slots); 32768 x 400, p = 2, ten sweeps: 424 us with 64-bit words
// through the network and all 512 padded ranks swept by 128 threads with barriers, 150 us here.
//
// p = 2: consecutive ranks per lane.  p = 4/3: the window's pairs are dealt to the lanes round-robin, so that the heavy
// pairs (cube roots) around rank k are shared by all lanes.
#include "tk_pairs.cuh"
#include "tk_rank.cuh"

namespace tk {

namespace {

constexpr int kSwMaxWindow = 512;               // 16 ranks per lane of one warp

// One row's window: the ranks [lo, hi), lo even; arrays by rank - lo (s: rk_slot of the rank).
struct SwWin {
  const float* s;          // sorted keys of the row
  float* v;                // p = 2: the iterate; at the end the results
  float* del;              // correction (p = 2) or dual (p = 4/3) of the constraint between a rank and the next
  int lo, hi, k;
};

// the part [lo, hi) of the window that `ranks` ranks around k cover
__device__ __forceinline__ void sw_part(const SwWin& Wn, int ranks, int& lo, int& hi) {
  lo = max(Wn.lo, min((Wn.k - ranks / 2) & ~1, (Wn.hi - ranks + 1) & ~1));
  hi = min(Wn.hi, lo + ranks);
}

// p = 2: EW consecutive ranks per lane over GG lanes, from sweep `it` until `sweeps` or until the changes come near the
// edge of the part; returns the sweeps done.
template <int EW, int GG, bool MAG>
__device__ __forceinline__ int sw_dykstra(const SwWin& Wn, float lam, int it, int sweeps, int l) {
  int lo, hi;
  sw_part(Wn, GG * EW, lo, hi);
  const bool low_open = lo > Wn.lo, high_open = hi < Wn.hi;
  const int b = lo + l * EW;                                      // this lane's first rank
  float v[EW], c[EW], pd[EW / 2], qd[EW / 2];
#pragma unroll
  for (int i = 0; i < EW; ++i) {
    const int j = min(b + i, hi - 1) - Wn.lo;
    v[i] = Wn.v[j];
    if (i & 1) qd[i / 2] = b + i < hi ? Wn.del[j] : 0.0f; else pd[i / 2] = b + i < hi ? Wn.del[j] : 0.0f;
    c[i] = MAG && b + i < Wn.k ? 1.0f + lam : 1.0f;
  }
  const float c_next = MAG && b + EW < Wn.k ? 1.0f + lam : 1.0f;
  const bool cross = l < GG - 1 && b + EW < hi;
#pragma unroll 1
  while (it < sweeps) {
    ++it;
#pragma unroll
    for (int j = 0; j < EW / 2; ++j)
      if (b + 2 * j + 1 < hi) dyk_pair(v[2 * j], v[2 * j + 1], pd[j], c[2 * j], c[2 * j + 1]);
    float nb = __shfl_down_sync(0xffffffffu, v[0], 1, GG);
    if (cross) dyk_pair(v[EW - 1], nb, qd[EW / 2 - 1], c[EW - 1], c_next);
#pragma unroll
    for (int j = 0; j < EW / 2 - 1; ++j)
      if (b + 2 * j + 2 < hi) dyk_pair(v[2 * j + 1], v[2 * j + 2], qd[j], c[2 * j + 1], c[2 * j + 2]);
    const float back = __shfl_up_sync(0xffffffffu, nb, 1, GG);    // what the previous lane made of this one's first rank
    if (l > 0 && b < hi) v[0] = back;
    if (EW < 16) {
      // corrections on the ranks one more sweep could carry across the edge
      bool near = low_open && l == 0 && (pd[0] != 0.0f || qd[0] != 0.0f);
      near |= high_open && l == GG - 1 && (pd[EW / 2 - 1] != 0.0f || (EW > 2 && qd[EW > 2 ? EW / 2 - 2 : 0] != 0.0f));
      if (EW == 2) near |= high_open && l == GG - 2 && qd[0] != 0.0f;
      if (__any_sync(0xffffffffu, near)) break;
    }
  }
#pragma unroll
  for (int i = 0; i < EW; ++i)
    if (b + i < hi) {
      Wn.v[b + i - Wn.lo] = v[i];
      Wn.del[b + i - Wn.lo] = (i & 1) ? qd[i / 2] : pd[i / 2];
    }
  __syncwarp();
  return it;
}

// p = 4/3, phi = x: H pairs per lane, round-robin over GG lanes (pair q = ranks lo + 2q, lo + 2q + 1 of the part)
template <int H, int GG, int G, int W>
__device__ __forceinline__ int sw_bca(const SwWin& Wn, const Math& M, int it, int sweeps, int l) {
  int lo, hi;
  sw_part(Wn, 2 * GG * H, lo, hi);
  const bool low_open = lo > Wn.lo, high_open = hi < Wn.hi;
  const int cnt = hi - lo;
  float* al = Wn.del + (lo - Wn.lo);
  auto wgt = [&](int j) -> float { return lo + j < Wn.k ? 1.0f : 0.0f; };
  float s_lo[H], s_hi[H], s_nx[H], ao[H], ae[H];
#pragma unroll
  for (int j = 0; j < H; ++j) {
    const int q = l + j * GG;
    s_lo[j] = Wn.s[rk_slot<G, W>(min(lo + 2 * q, hi - 1))];
    s_hi[j] = Wn.s[rk_slot<G, W>(min(lo + 2 * q + 1, hi - 1))];
    s_nx[j] = Wn.s[rk_slot<G, W>(min(lo + 2 * q + 2, hi - 1))];
    ao[j] = 2 * q < cnt ? al[2 * q] : 0.0f;
    ae[j] = 2 * q + 1 < cnt ? al[2 * q + 1] : 0.0f;
  }
#pragma unroll 1
  while (it < sweeps) {
    ++it;
    // odd family: constraint (2q, 2q + 1); neighbours: the even duals of pairs q - 1 and q
#pragma unroll
    for (int j = 0; j < H; ++j) {
      const int q = l + j * GG;
      const float below = __shfl_up_sync(0xffffffffu, ae[j], 1, GG);
      const float wrap = j > 0 ? __shfl_sync(0xffffffffu, ae[j > 0 ? j - 1 : 0], GG - 1, GG) : 0.0f;
      if (2 * q + 1 < cnt) ao[j] = bca_alpha(s_lo[j], s_hi[j], wgt(2 * q), wgt(2 * q + 1), l > 0 ? below : wrap, ae[j], M);
    }
    // even family: constraint (2q + 1, 2q + 2); neighbours: the odd duals of pairs q and q + 1
#pragma unroll
    for (int j = 0; j < H; ++j) {
      const int q = l + j * GG;
      const float above = __shfl_down_sync(0xffffffffu, ao[j], 1, GG);
      const float wrap = j < H - 1 ? __shfl_sync(0xffffffffu, ao[j < H - 1 ? j + 1 : j], 0, GG) : 0.0f;
      if (2 * q + 2 < cnt)
        ae[j] = bca_alpha(s_hi[j], s_nx[j], wgt(2 * q + 1), wgt(2 * q + 2), ao[j], 2 * q + 3 < cnt ? (l < GG - 1 ? above : wrap) : 0.0f, M);
    }
    if (H < 8) {
      bool near = low_open && l == 0 && (ao[0] != 0.0f || ae[0] != 0.0f);
      near |= high_open && l + (H - 1) * GG >= cnt / 2 - 2 && (ao[H - 1] != 0.0f || ae[H - 1] != 0.0f);
      if (__any_sync(0xffffffffu, near)) break;
    }
  }
#pragma unroll
  for (int j = 0; j < H; ++j) {
    const int q = l + j * GG;
    if (2 * q < cnt) al[2 * q] = ao[j];
    if (2 * q + 1 < cnt) al[2 * q + 1] = ae[j];
  }
  __syncwarp();
  return it;
}

// All sweeps of a row, and the results of its window into Wn.v.
template <int GG, int G, int W, bool Q4, bool MAG>
__device__ __forceinline__ void sw_solve(const SwWin& Wn, const Math& M, int sweeps, int l) {
  const int cnt = Wn.hi - Wn.lo;
  for (int j = l; j < cnt; j += GG) {
    const float sj = Wn.s[rk_slot<G, W>(Wn.lo + j)];
    const bool top = Wn.lo + j < Wn.k;
    if (!Q4) Wn.v[j] = MAG ? (top ? sj / (1.0f + M.lam) : sj) : (top ? sj - M.lam : sj);
    Wn.del[j] = 0.0f;
  }
  __syncwarp();
  int it = 0;
  if (Q4) {
    if (GG >= 16) it = sw_bca<1, GG, G, W>(Wn, M, it, sweeps, l);
    if (GG >= 4 && it < sweeps) it = sw_bca<2, GG, G, W>(Wn, M, it, sweeps, l);
    if (GG >= 16 && it < sweeps) it = sw_bca<4, GG, G, W>(Wn, M, it, sweeps, l);
    if (it < sweeps) sw_bca<8, GG, G, W>(Wn, M, it, sweeps, l);
  } else {
    if (GG >= 16) it = sw_dykstra<2, GG, MAG>(Wn, M.lam, it, sweeps, l);
    if (GG >= 4 && it < sweeps) it = sw_dykstra<4, GG, MAG>(Wn, M.lam, it, sweeps, l);
    if (GG >= 16 && it < sweeps) it = sw_dykstra<8, GG, MAG>(Wn, M.lam, it, sweeps, l);
    if (it < sweeps) sw_dykstra<16, GG, MAG>(Wn, M.lam, it, sweeps, l);
  }
  for (int j = l; j < cnt; j += GG) {
    if (Q4) Wn.v[j] = (Wn.lo + j < Wn.k ? 1.0f : 0.0f) - Wn.del[j] + (j > 0 ? Wn.del[j - 1] : 0.0f);
    else Wn.v[j] = (Wn.s[rk_slot<G, W>(Wn.lo + j)] - (MAG ? fmaxf(Wn.v[j], 0.0f) : Wn.v[j])) * M.inv_lam;
  }
  if (l == 0) { Wn.v[cnt] = 0.0f; Wn.v[cnt + 1] = 1.0f; }
}

// Words of shared memory of a team: the sorted keys, then (v, del) of the window(s), where rank_ties counts too.
template <int G, int W>
struct SwGeom {
  using Geom = RankGeom<G, W>;
  static constexpr int VN = (W == 1 ? Geom::N : kSwMaxWindow) + 2;            // entries of v and of del
  static constexpr int KEYS = Geom::R * Geom::NP;
  static constexpr int WORK = Geom::R * 2 * VN > KEYS ? Geom::R * 2 * VN : KEYS;
};

// [lo, hi): the window, lo even.
template <int G, int W, bool Q4, bool MAG>
__global__ void __launch_bounds__(RankGeom<G, W>::THREADS, (W == 1 ? 5 : (W >= 16 ? 1 : 20 / W)))
    tk_sweeps_kernel(const Problem P, const int lo, const int hi) {
  using Geom = RankGeom<G, W>;
  constexpr int E = kRkE, T = Geom::T, R = Geom::R, NP = Geom::NP;
  __shared__ float sm[Geom::TEAMS][SwGeom<G, W>::KEYS + SwGeom<G, W>::WORK];
  const int lane = threadIdx.x & 31;
  const int team = W == 1 ? threadIdx.x >> 5 : 0;
  const int tid = W == 1 ? lane : (int)threadIdx.x;
  const int rl = W == 1 ? lane / G : 0, lig = W == 1 ? lane % G : tid;
  const long long row0 = ((long long)blockIdx.x * Geom::TEAMS + team) * R;
  if (row0 >= P.rows) return;                                     // the whole team
  const long long row = row0 + rl;
  const bool live = row < P.rows;                                 // a row past the last one repeats it, stores nothing
  const long long first = (live ? row : P.rows - 1) * (long long)P.n;
  const int n = P.n, cnt = hi - lo;
  float* s = sm[team] + rl * NP;
  float* work = sm[team] + SwGeom<G, W>::KEYS;
  float* ys = work + rl * 2 * SwGeom<G, W>::VN;
  const float* x_row = P.theta + first;

  overlap_wait();
  float key[E], r[E];
  bool bad = false;
#pragma unroll
  for (int i = 0; i < E; ++i) key[i] = x_row[min(lig + T * i, n - 1)];
#pragma unroll
  for (int i = 0; i < E; ++i) bad |= !(fabsf(key[i]) < INFINITY);
#pragma unroll
  for (int i = 0; i < E; ++i) {
    if (MAG) key[i] = fabsf(key[i]);
    if (bad && key[i] != key[i]) key[i] = INFINITY;               // (max and min drop a NaN)
    r[i] = lig + T * i < n ? key[i] : -INFINITY;
  }
  rank_sort<G, W>(r, tid, sm[team]);
  bool tie = rank_store<G, W>(r, s, n, lig);

  // ---- every element's place in the window: 0 .. cnt - 1, cnt below it, cnt + 1 above it
  int at[E];
#pragma unroll
  for (int i = 0; i < E; ++i) at[i] = rank_find<G, W>(s, n, key[i]);
  tie = W > 1 ? __syncthreads_or(tie) != 0 : __any_sync(0xffffffffu, tie);
  if (tie) rank_ties<G, W>(at, s, n, lig, rl, tid, reinterpret_cast<int*>(work));
#pragma unroll
  for (int i = 0; i < E; ++i) {
    const int e = lig + T * i;
    if (P.perm_out && live && e < n) P.perm_out[first + at[i]] = e;
    at[i] = at[i] < lo ? cnt + 1 : (at[i] < hi ? at[i] - lo : cnt);
  }

  // ---- the sweeps: the row's lanes, or the first warp of its warps
  Math M = make_math_q24(P);
  M.q4 = Q4; M.mag = MAG;
  if (W == 1 || threadIdx.x < 32) {
    SwWin Wn;
    Wn.s = s; Wn.v = ys; Wn.del = ys + SwGeom<G, W>::VN; Wn.lo = lo; Wn.hi = hi; Wn.k = P.k;
    sw_solve<W == 1 ? G : 32, G, W, Q4, MAG>(Wn, M, P.sweeps > 0 ? P.sweeps : 100, W == 1 ? lig : lane);
  }
  rk_sync<W>();

#pragma unroll
  for (int i = 0; i < E; ++i) {
    const int e = lig + T * i;
    float y = ys[at[i]];
    const float x = (MAG || P.mode == TK_TOPK) ? __ldg(x_row + min(e, n - 1)) : 0.0f;
    if (MAG) {
      const float a = fabsf(x);
      if (at[i] == cnt + 1) y = (a - a / (1.0f + M.lam)) * M.inv_lam;   // above the window: the separate minimiser s / c
      if (signbit(x)) y = -y;
    }
    if (P.mode == TK_TOPK) y *= x;
    if (live && e < n) P.out[first + e] = y;
  }
  if (bad && P.status) atomicOr(P.status, TK_FLAG_NONFINITE);
}

template <int G, int W>
cudaError_t sw_launch(const Problem& P, int lo, int hi, cudaStream_t stream) {
  using Geom = RankGeom<G, W>;
  constexpr int rows_per_block = Geom::TEAMS * Geom::R;
  const unsigned blocks = (unsigned)((P.rows + rows_per_block - 1) / rows_per_block);
  if (P.q4) return launch_overlapped(tk_sweeps_kernel<G, W, true, false>, blocks, Geom::THREADS, 0, stream, P, lo, hi);
  if (P.mode == TK_TOPKMAG) return launch_overlapped(tk_sweeps_kernel<G, W, false, true>, blocks, Geom::THREADS, 0, stream, P, lo, hi);
  return launch_overlapped(tk_sweeps_kernel<G, W, false, false>, blocks, Geom::THREADS, 0, stream, P, lo, hi);
}

// the ranks that `sweeps` sweeps can change, first of a pair of C1 onwards
void sw_window(const Problem& P, int* lo, int* hi) {
  const long long t = P.sweeps > 0 ? P.sweeps : 100;
  const long long a = (long long)P.k - 2 * t - 2, b = (long long)P.k + 2 * t + 2;
  *lo = a > 0 ? (int)(a & ~1ll) : 0;
  *hi = b < P.n ? (int)b : P.n;
}

}  // namespace

// A fixed number of sweeps whose window one warp holds, closed-form pair steps, rows of up to 4096 elements -- and where
// the whole-row kernels, which give a row two to four times the lanes, are not faster: rows of up to 256 elements want
// warps enough to fill the SMs (p = 2, 10 sweeps: 4194 x 250 17 -> 16 us, 16777 x 250 54 -> 45, but 1048 x 250 7 -> 11;
// 41943 x 400 540 -> 200, 655 x 400 14 -> 13), and p = 4/3 keeps them for rows of up to 64 (104857 x 40, 100 sweeps: 1690
// us there, 1833 here; 41943 x 100: 1385 and 1468) and, with p = 2 above 512 elements, for a window of several pairs per lane
// on few rows (655 x 400, p = 4/3, 100 sweeps: 115 and 139, but 2621 x 400 337 and 184; 262 x 1000, p = 2: 22 and 25).
bool sweeps_window_serves(const Problem& P) {
  if (P.tol > 0.0f || P.qm1 > 0.0f || (P.q4 && P.mode == TK_TOPKMAG) || P.n > 4096) return false;
  int lo, hi;
  sw_window(P, &lo, &hi);
  if (hi - lo > kSwMaxWindow) return false;
  int lanes = 1;
  while (16 * lanes < P.n) lanes <<= 1;
  const double warps = (double)P.rows * lanes / 32.0 / sm_count();            // per SM
  const bool several = hi - lo > 64;
  if (P.q4 && (P.n <= 64 || (P.n <= 128 && several))) return false;
  if (P.n <= 64) return warps >= 16.0;
  if (P.n <= 256) return warps >= 8.0;
  if (P.n <= 512) return !(P.q4 && several && warps < 8.0);
  return !(P.n <= 1024 && several && warps < 4.0);
}

cudaError_t launch_sweeps(const Problem& P, cudaStream_t stream) {
  int lo, hi;
  sw_window(P, &lo, &hi);
  if (P.n <= 16) return sw_launch<1, 1>(P, lo, hi, stream);
  if (P.n <= 32) return sw_launch<2, 1>(P, lo, hi, stream);
  if (P.n <= 64) return sw_launch<4, 1>(P, lo, hi, stream);
  if (P.n <= 128) return sw_launch<8, 1>(P, lo, hi, stream);
  if (P.n <= 256) return sw_launch<16, 1>(P, lo, hi, stream);
  if (P.n <= 512) return sw_launch<32, 1>(P, lo, hi, stream);
  if (P.n <= 1024) return sw_launch<32, 2>(P, lo, hi, stream);
  if (P.n <= 2048) return sw_launch<32, 4>(P, lo, hi, stream);
  return sw_launch<32, 8>(P, lo, hi, stream);
}

}  // namespace tk
