// tk_perm.cu -- the stable descending argsort of rows of up to 8192 elements (Sec. 3, argsort / sort) and, with it,
// the hard operators of Sec. 3 (ones at sigma_1 .. sigma_k; theta there): one kernel for tk_argsort, for the permutation
// of a forward pass and for the straight-through output.
//
// The keys alone are sorted and every element finds its rank by binary search (tk_rank.cuh).  The rank is the
// element's place in the permutation and, against k, its hard result: the permutation goes through shared memory to a
// coalesced store, the result is stored where the element was loaded.
//
// What bounds it: the ALU pipe (84 %), two thirds of it the network's max and min, one third the search.  2048 x 2048:
// argsort 78 us with 64-bit (key, index) words through the network, 47 here; hard forward with row state (threshold
// form beside it) 155 -> 63.
#include "tk_rank.cuh"

namespace tk {

namespace {

struct PermArgs {
  const float* theta;
  int32_t* perm;           // [rows * n]
  float* sorted;           // sorted keys, or null
  float* hard;             // hard operator, or null
  int32_t* status;
  long long rows;
  int n, k, mode;
};

template <int G, int W>
__global__ void __launch_bounds__(RankGeom<G, W>::THREADS, (W == 1 ? 6 : (W >= 16 ? 1 : 24 / W))) tk_perm_kernel(const PermArgs P) {
  using Geom = RankGeom<G, W>;
  constexpr int E = kRkE, T = Geom::T, R = Geom::R, NP = Geom::NP;
  constexpr int WORK = R * NP;                                    // the permutation of the team's rows; rank_ties before
  extern __shared__ float pm_smem[];
  const int lane = threadIdx.x & 31;
  const int team = W == 1 ? threadIdx.x >> 5 : 0;
  const int tid = W == 1 ? lane : (int)threadIdx.x;
  const int rl = W == 1 ? lane / G : 0, lig = W == 1 ? lane % G : tid;
  const long long row0 = ((long long)blockIdx.x * Geom::TEAMS + team) * R;
  if (row0 >= P.rows) return;                                     // the whole team
  const bool live = row0 + rl < P.rows;                           // a row past the last one repeats it, stores nothing
  const int n = P.n;
  const long long first = (live ? row0 + rl : P.rows - 1) * (long long)n;
  float* sm = pm_smem + team * (R * NP + WORK);
  float* s = sm + rl * NP;
  int* work = reinterpret_cast<int*>(sm + R * NP);
  const bool mag = P.mode == TK_TOPKMAG;

  overlap_wait();
  float x[E], r[E];
  bool bad = false;
#pragma unroll
  for (int i = 0; i < E; ++i) x[i] = P.theta[first + min(lig + T * i, n - 1)];
#pragma unroll
  for (int i = 0; i < E; ++i) bad |= !(fabsf(x[i]) < INFINITY);
  auto key_of = [&](float v) -> float {
    const float key = mag ? fabsf(v) : v;
    return bad && key != key ? INFINITY : key;                    // (max and min drop a NaN)
  };
#pragma unroll
  for (int i = 0; i < E; ++i) r[i] = lig + T * i < n ? key_of(x[i]) : -INFINITY;
  rank_sort<G, W>(r, tid, sm);
  bool tie = rank_store<G, W>(r, s, n, lig);

  int rk[E];
#pragma unroll
  for (int i = 0; i < E; ++i) {
    rk[i] = rank_find<G, W>(s, n, key_of(x[i]));
  }
  tie = W > 1 ? __syncthreads_or(tie) != 0 : __any_sync(0xffffffffu, tie);
  if (tie) rank_ties<G, W>(rk, s, n, lig, rl, tid, work);
  int* p = work + rl * NP;
#pragma unroll
  for (int i = 0; i < E; ++i) {
    const int e = lig + T * i;
    if (e < n) {
      p[rk[i]] = e;
      if (P.hard && live) P.hard[first + e] = rk[i] < P.k ? (P.mode == TK_MASK ? 1.0f : x[i]) : 0.0f;
    }
  }
  rk_sync<W>();
#pragma unroll
  for (int i = 0; i < E; ++i) {
    const int e = lig + T * i;
    if (live && e < n) {
      P.perm[first + e] = p[e];
      if (P.sorted) P.sorted[first + e] = s[rk_slot<G, W>(e)] + 0.0f;   // (-0 and +0 are the same key: +0)
    }
  }
  if (bad && P.status) atomicOr(P.status, TK_FLAG_NONFINITE);
}

template <int G, int W>
cudaError_t pm_launch(const PermArgs& P, cudaStream_t stream) {
  using Geom = RankGeom<G, W>;
  constexpr int rows_per_block = Geom::TEAMS * Geom::R;
  constexpr int smem = Geom::TEAMS * 2 * Geom::R * Geom::NP * (int)sizeof(float);
  if (smem > 48 * 1024) {
    static bool configured[64];
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= 64 || !configured[dev]) {
      err = cudaFuncSetAttribute(tk_perm_kernel<G, W>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      if (err != cudaSuccess) return err;
      if (dev >= 0 && dev < 64) configured[dev] = true;
    }
  }
  const unsigned blocks = (unsigned)((P.rows + rows_per_block - 1) / rows_per_block);
  return launch_overlapped(tk_perm_kernel<G, W>, blocks, Geom::THREADS, smem, stream, P);
}

}  // namespace

int perm_max_n() { return 8192; }

// perm[r, i] = index of the i-th largest key of row r, stable; optionally the keys in that order and the hard operator.
cudaError_t launch_perm(const float* theta, long long rows, int n, int k, int mode, int32_t* perm, float* sorted,
                        float* hard, int32_t* status, cudaStream_t stream) {
  PermArgs P = {theta, perm, sorted, hard, status, rows, n, k, mode};
  if (n <= 16) return pm_launch<1, 1>(P, stream);
  if (n <= 32) return pm_launch<2, 1>(P, stream);
  if (n <= 64) return pm_launch<4, 1>(P, stream);
  if (n <= 128) return pm_launch<8, 1>(P, stream);
  if (n <= 256) return pm_launch<16, 1>(P, stream);
  if (n <= 512) return pm_launch<32, 1>(P, stream);
  if (n <= 1024) return pm_launch<32, 2>(P, stream);
  if (n <= 2048) return pm_launch<32, 4>(P, stream);
  if (n <= 4096) return pm_launch<32, 8>(P, stream);
  return pm_launch<32, 16>(P, stream);
}

}  // namespace tk
