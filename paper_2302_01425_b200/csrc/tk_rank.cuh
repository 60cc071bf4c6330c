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
  static constexpr int TS = T + 1;                                // stride between the ranks of a lane (see rk_slot)
  static constexpr int PAD = W > 1 ? 0 : (G + 32 - (kRkE * TS) % 32) % 32;   // rows of a warp start G banks apart
  static constexpr int NP = kRkE * TS + PAD;                      // slots of a row
  static constexpr int TL = 32 * W, TEAMS = W == 1 ? 4 : 1, THREADS = TL * TEAMS;
};

// Slot of a rank in the row's shared array: rank 16 l + i of lane l lies at i * TS + l.  The lanes store their ranks
// without bank conflicts, and both halves of the binary search (over the lanes' first keys, then inside one lane's 16) step
// through addresses with constant offsets: a load, a compare and a predicated add per step (with consecutive ranks and
// a padding word per 16 the address took as many instructions again: 32768 x 400, ten sweeps: 160 -> 148 us).
template <int G, int W>
__device__ __forceinline__ int rk_slot(int r) { return (r & (kRkE - 1)) * RankGeom<G, W>::TS + (r >> 4); }
template <int G, int W>
__device__ __forceinline__ int rk_rank(int slot) { return (slot % RankGeom<G, W>::TS) * kRkE + slot / RankGeom<G, W>::TS; }

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

// The sorted ranks into the row's shared array; returns whether two keys of the row (ranks below n) are equal.
template <int G, int W>
__device__ __forceinline__ bool rank_store(const float (&r)[kRkE], float* s, int n, int lig) {
  using Geom = RankGeom<G, W>;
  bool tie = false;
#pragma unroll
  for (int i = 0; i < kRkE; ++i) {
    s[i * Geom::TS + lig] = r[i];
    if (i > 0) tie |= lig * kRkE + i < n && r[i] == r[i - 1];
  }
  rk_sync<W>();
  if (lig > 0) tie |= lig * kRkE < n && s[(kRkE - 1) * Geom::TS + lig - 1] == r[0];
  return tie;
}

// number of keys of the sorted row s larger than key (at most n - 1)
template <int G, int W>
__device__ __forceinline__ int rank_find(const float* s, int n, float key) {
  using Geom = RankGeom<G, W>;
  int b = 0;                                    // last lane whose first key is larger
#pragma unroll
  for (int st = Geom::T >> 1; st > 0; st >>= 1)
    if (s[b + st] > key) b += st;
  const float* c = s + b;
  int j = 0, rank = b * kRkE;                   // j: in steps of TS
#pragma unroll
  for (int st = kRkE >> 1; st > 0; st >>= 1)
    if (c[j + (st - 1) * Geom::TS] > key) { j += st * Geom::TS; rank += st; }
  if (c[j] > key) ++rank;
  return min(rank, n - 1);
}

// Ranks of equal keys in index order.  rk[i]: what rank_find returned for element lig + T i of this lane's row (its
// place in the run's order is added); s: the row's sorted keys.  work: max(R * NP, kRkList + 1) words of shared memory.
// All lanes of the team call it.  Up to kRkList elements with equals: listed, and each counts the earlier ones of its
// run.  More: the row is walked in index order.
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
    if (e < n && rk[i] + 1 < n && s[rk_slot<G, W>(rk[i] + 1)] == s[rk_slot<G, W>(rk[i])]) {
      tied |= 1u << i;
      const int at = atomicAdd(work + kRkList, 1);
      if (at < kRkList) list[at] = (uint32_t)(rl * Geom::NP + rk_slot<G, W>(rk[i])) << 16 | (uint32_t)e;
    }
  }
  rk_sync<W>();
  const int listed = work[kRkList];
  if (listed <= kRkList) {
#pragma unroll
    for (int i = 0; i < kRkE; ++i) {
      if (tied >> i & 1u) {
        const uint32_t mine = (uint32_t)(rl * Geom::NP + rk_slot<G, W>(rk[i])) << 16 | (uint32_t)(lig + Geom::T * i);
        int before = 0;
        for (int j = 0; j < listed; ++j) before += (list[j] ^ mine) < 0x10000u && list[j] < mine;
        rk[i] = min(rk[i] + before, n - 1);
      }
    }
    rk_sync<W>();
    return;
  }
  // Elements in index order, 32 at a time: a step finds which of them are equal, reads how many of their run have been
  // placed, and adds its own.
  rk_sync<W>();
  uint16_t* cnt = reinterpret_cast<uint16_t*>(work);              // [R * N], by rank: how many of a run have been placed
  for (int i = tid; i < Geom::R * Geom::N / 2; i += Geom::TL) work[i] = 0;
  if constexpr (W == 1) {
    __syncwarp();
#pragma unroll
    for (int i = 0; i < kRkE; ++i) {
      const bool in = lig + Geom::T * i < n;
      const int slot = rl * Geom::N + rk[i];
      const unsigned same = __match_any_sync(0xffffffffu, in ? slot : -1 - lane);
      const int before = __popc(same & ((1u << lane) - 1u));
      int placed = 0;
      if (in) placed = cnt[slot];
      __syncwarp();
      if (in) {
        if (before == 0) cnt[slot] = (uint16_t)(placed + __popc(same));
        rk[i] = min(rk[i] + placed + before, n - 1);
      }
      __syncwarp();
    }
  } else {
    // Each warp takes 512 consecutive elements (through shared memory) and finds the equal ones of all its steps first; then
    // the warps take turns, and a turn is 16 times read, add, write.  (Us, a third of the entries masked, every step of all
    // warps in turn with a block barrier after it / here: argsort 524 x 4000 85 / 52, with a 64-bit network 47; permutation
    // and values 256 x 8192 204 / 121.  One warp per row has no barriers to save, and the extra passes cost it 17 %.)
    uint16_t* ranks = cnt + Geom::N;                              // [N], by element
#pragma unroll
    for (int i = 0; i < kRkE; ++i) ranks[lig + Geom::T * i] = (uint16_t)rk[i];
    __syncthreads();
    uint16_t* mine = ranks + warp * (32 * kRkE) + lane;
    const int left = n - warp * (32 * kRkE) - lane;               // this lane's elements of the warp's: 32 i < left
    int at[kRkE];                               // rank of the run | earlier ones among the 32 | the run's share of them
#pragma unroll
    for (int i = 0; i < kRkE; ++i) {
      const int r = mine[32 * i];
      const unsigned same = __match_any_sync(0xffffffffu, 32 * i < left ? r : -1 - lane);
      at[i] = r | __popc(same & ((1u << lane) - 1u)) << 16 | __popc(same) << 24;
    }
#pragma unroll 1
    for (int w = 0; w < W; ++w) {
      if (w == warp) {
#pragma unroll
        for (int i = 0; i < kRkE; ++i) {
          const int r = at[i] & 0xffff, before = at[i] >> 16 & 0xff;
          int placed = 0;
          if (32 * i < left) placed = cnt[r];
          __syncwarp();
          if (32 * i < left && before == 0) cnt[r] = (uint16_t)(placed + (at[i] >> 24));
          at[i] = min(r + placed + before, n - 1);
          __syncwarp();
        }
      }
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < kRkE; ++i) mine[32 * i] = (uint16_t)at[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kRkE; ++i) rk[i] = ranks[lig + Geom::T * i];
  }
  rk_sync<W>();
}

}  // namespace tk
