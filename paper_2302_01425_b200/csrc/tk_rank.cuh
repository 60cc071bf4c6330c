// tk_rank.cuh -- sorting a row's KEYS and finding every element's rank in the sorted row, by a team of lanes: G
// lanes of a warp (32 / G rows per warp) or W whole warps, 16 keys per lane.
//
// The stable descending argsort without moving indices through a network: the 32-bit keys alone are sorted (a
// compare-exchange is one max and one min; with a packed 64-bit (key, index) word it is a 64-bit compare and four
// selects), the sorted row goes to shared memory, and an element's rank is the number of larger keys, found by binary
// search.  Elements with equal keys find the same number; where a row has any, the ranks of a run are handed out in
// index order (rank_ties), which is the stable order.
#pragma once

#include "tk_key_sort.cuh"

namespace tk {

constexpr int kRkE = 16;                        // keys per lane

template <int G, int W>
struct RankGeom {
  static constexpr int T = G * W, R = W > 1 ? 1 : 32 / G;         // lanes per row, rows per team
  static constexpr int N = T * kRkE;                              // padded row length
  static constexpr int NP = N + T;                                // slots of a row: one word of padding per 16
  static constexpr int TL = 32 * W, TEAMS = W == 1 ? 4 : 1, THREADS = TL * TEAMS;
};

__device__ __forceinline__ int rk_slot(int r) { return r + (r >> 4); }

template <int W>
__device__ __forceinline__ void rk_sync() {
  if (W == 1) __syncwarp(); else __syncthreads();
}

// Sorts the team's rows, descending: on return lane l of a row holds the ranks 16 l .. 16 l + 15.  ex: T * 16 words of
// shared memory for the exchanges between warps (W > 1; free again on return).
template <int G, int W>
__device__ __forceinline__ void rank_sort(float (&r)[kRkE], int tid, float* ex) {
  constexpr int E = kRkE, T = G * W;
  const int lane = tid & 31;
  group_sort_keys<G, E>(r, W == 1 ? lane % G : lane, 0xffffffffu);
  if (W > 1) {
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
}

// number of keys of the sorted row s (padded slots) larger than key, at most n - 1
template <int G, int W>
__device__ __forceinline__ int rank_find(const float* s, int n, float key) {
  int pos = 0;
#pragma unroll
  for (int st = RankGeom<G, W>::N >> 1; st > 0; st >>= 1) {
    const int q = pos + st;
    if (s[rk_slot(q - 1)] > key) pos = q;
  }
  return pos < n ? pos : n - 1;
}

// Ranks of equal keys in index order.  rk[i]: what rank_find returned for element lig + T i of this lane's row (its
// place in the run's order is added); s: the row's sorted keys.  work: max(R * NP, kRkList + 1) words of shared memory.
// All lanes of the team call it.  Up to kRkList elements with equals: listed, and each counts the earlier ones of its
// run.  More: the row is walked 32 elements at a time in index order (128 steps of about 600 cycles at n = 4096).
constexpr int kRkList = 64;

template <int G, int W>
__device__ __forceinline__ void rank_ties(int (&rk)[kRkE], const float* s, int n, int lig, int rl, int tid, int* work) {
  using Geom = RankGeom<G, W>;
  const int lane = tid & 31, warp = W == 1 ? 0 : tid >> 5;
  rk_sync<W>();
  if (tid == 0) work[kRkList] = 0;
  rk_sync<W>();
  uint32_t* list = reinterpret_cast<uint32_t*>(work);
  uint32_t tied = 0;                            // bit i: rk[i] is the first rank of a run of several
#pragma unroll
  for (int i = 0; i < kRkE; ++i) {
    const int e = lig + Geom::T * i;
    if (e < n && rk[i] + 1 < n && s[rk_slot(rk[i] + 1)] == s[rk_slot(rk[i])]) {
      tied |= 1u << i;
      const int at = atomicAdd(work + kRkList, 1);
      if (at < kRkList) list[at] = (uint32_t)(rl * Geom::NP + rk_slot(rk[i])) << 16 | (uint32_t)e;
    }
  }
  rk_sync<W>();
  const int listed = work[kRkList];
  if (listed <= kRkList) {
#pragma unroll
    for (int i = 0; i < kRkE; ++i) {
      if (tied >> i & 1u) {
        const uint32_t mine = (uint32_t)(rl * Geom::NP + rk_slot(rk[i])) << 16 | (uint32_t)(lig + Geom::T * i);
        int before = 0;
        for (int j = 0; j < listed; ++j) before += (list[j] ^ mine) < 0x10000u && list[j] < mine;
        rk[i] = min(rk[i] + before, n - 1);
      }
    }
    rk_sync<W>();
    return;
  }
  rk_sync<W>();
  int* cnt = work;                              // how many of a run have been placed
  for (int i = tid; i < Geom::R * Geom::NP; i += Geom::TL) cnt[i] = 0;
  rk_sync<W>();
#pragma unroll
  for (int i = 0; i < kRkE; ++i) {
#pragma unroll 1
    for (int w = 0; w < W; ++w) {
      if (w == warp) {
        const bool in = lig + Geom::T * i < n;
        const int slot = rl * Geom::NP + rk_slot(rk[i]);
        const unsigned same = __match_any_sync(0xffffffffu, in ? slot : -1 - lane);
        const int before = __popc(same & ((1u << lane) - 1u));
        int placed = 0;
        if (in) placed = cnt[slot];
        __syncwarp();
        if (in) {
          if (before == 0) cnt[slot] = placed + __popc(same);
          rk[i] = min(rk[i] + placed + before, n - 1);
        }
        __syncwarp();
      }
      if (W > 1) __syncthreads();
    }
  }
  rk_sync<W>();
}

}  // namespace tk
