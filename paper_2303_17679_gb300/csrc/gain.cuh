// Gains of nodes from packed net records: shared by label propagation (lp.cu)
// and the gain table (gaintable.cu).
#pragma once

#include "common.cuh"

namespace hgk {

constexpr int SUB_G = 8;       // lanes per node of the lane-group class
constexpr int NG = 32 / SUB_G;

// For every incidence (u, e) a gain needs w(e), Lambda(e) and whether
// Phi(e, Pi[u]) = 1.  They live in one 16-byte record per net and half of the
// blocks (k <= 32: one half), so the gain gathers one sector per incidence
// instead of three:
//   rec[H e + h] = {w(e), ones(e), Lambda(e), 0} for the blocks 32 h ..
// with ones(e) = {i : Phi(e, i) = 1}.
struct NetRec {
  int32_t w;
  unsigned ones, lam;
};

__device__ __forceinline__ NetRec load_rec(const int4* rec, int64_t i) {
  const int4 r = __ldcg(rec + i);
  return NetRec{r.x, (unsigned)r.y, (unsigned)r.z};
}

// Both halves of a record (k > 32).
struct WideRec {
  int32_t w;
  unsigned long long ones, lam;
};

// One 32-byte load: a gather is bound by its requests, a line each.  The records
// start on a 32-byte boundary (BUF_ALIGN).
__device__ __forceinline__ WideRec load_wide(const int4* rec, int32_t e) {
  unsigned r[8];  // w, ones, lam, 0 of either half
  asm volatile("ld.global.cg.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7])
               : "l"(rec + 2 * (int64_t)e)
               : "memory");
  return WideRec{(int32_t)r[0], (unsigned long long)r[1] | (unsigned long long)r[5] << 32,
                 (unsigned long long)r[2] | (unsigned long long)r[6] << 32};
}

// Sum over the W lanes of the caller's group (W a power of two); the whole warp
// calls it.
template <int W, typename T>
__device__ __forceinline__ T group_sum(T x) {
#pragma unroll
  for (int d = W / 2; d > 0; d >>= 1) x += __shfl_xor_sync(FULL, x, d);
  return x;
}
// Halving exchange over the W lanes of a group: afterwards acc[0 .. max(K/W,1))
// of lane l holds the group's totals of blocks first_block + i, where
// first_block is returned (K < W: W/K neighbouring lanes hold the same block).
template <int W, int K>
__device__ __forceinline__ int reduce_scatter(int l, int32_t (&acc)[K]) {
  int block = 0;
#pragma unroll
  for (int d = W / 2, h = K / 2; d > 0; d >>= 1, h >>= 1) {
    if (h > 0) {
      const bool up = (l & d) != 0;
      if (up) block += h;
#pragma unroll
      for (int i = 0; i < h; ++i) {
        const int32_t give = up ? acc[i] : acc[i + h];
        const int32_t keep = up ? acc[i + h] : acc[i];
        acc[i] = keep + __shfl_xor_sync(FULL, give, d);
      }
    } else {
      acc[0] += __shfl_xor_sync(FULL, acc[0], d);
    }
  }
  return block;
}

// Lanes of a team of W: W / H lanes share the incidences, the upper lanes take
// the upper half of the blocks.
template <int W, int H>
struct TeamLane {
  static constexpr int SHARE = W / H;
  int i, half;
  __device__ __forceinline__ explicit TeamLane(int l) : i(l % SHARE), half(l / SHARE) {}
};

// With b(u) = w(nets where u is the only pin of its block) and W_I = w(I(u)),
// the gain of Sec. 6 is
//   g(u, t) = b(u) - W_I + w({e in I(u) : t in Lambda(e)}),
// evaluated for all t at once; `bw` sums b(u) - W_I.  Graph levels (Sec. 10,
// "The Gain Table"): g(u, t) = w(u, V_t) - w(u, V_Pi(u)), `bw` sums
// -w(u, V_Pi(u)).
// Every lane sums per block in K = 8, 16 or 32 registers (two instructions per
// block and incidence), and the lanes combine the sums with a halving exchange
// that leaves each lane the totals of its own blocks (14 shuffles for 16
// blocks over 8 lanes instead of 48).  For k > 32 the lanes are split into H = 2
// halves: each half walks the same incidences with its half of the records.
// (Shared-memory counters with one atomic per block of Lambda(e), which k > 16
// used before, serialise on coarse levels, whose nets touch the same blocks:
// 37 us per sub-round at k = 64 and 31M pins, 60 us with lane groups.)
// Every sum is over distinct nets with one sign (bw subtracts them, and in the k > 32
// form adds others), so it lies between -W and W, W the total net weight: hg_create
// refuses W >= 2^31, and contraction keeps or drops nets but never adds weight.  So
// 32 bits hold them on every level, the atomics of a split node included.
template <bool GRAPH, int K, int H>
struct Gain {
  int32_t acc[K];
  int32_t bw;
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int t = 0; t < K; ++t) acc[t] = 0;
    bw = 0;
  }
  // incidence with net record r, seen by the lanes of half `half`; `from` is
  // the node's block relative to the half (outside [0, 32): another half's)
  __device__ __forceinline__ void add(const NetRec& r, int from) {
    // u is not the only pin of its block in e
    if ((H == 1 || (unsigned)from < 32u) && !((r.ones >> from) & 1u)) bw -= r.w;
    add_targets(r);
  }
  __device__ __forceinline__ void add_targets(const NetRec& r) {
#pragma unroll
    for (int t = 0; t < K; ++t)
      if (r.lam & (1u << t)) acc[t] += r.w;
  }
  // graph: edge of weight w to a node of block tb (relative to the half)
  __device__ __forceinline__ void add_edge(int32_t w, int tb, int from) {
    if (tb == from && (H == 1 || (unsigned)tb < 32u)) bw -= w;
#pragma unroll
    for (int t = 0; t < K; ++t)
      if (tb == t) acc[t] += w;
  }
};

}  // namespace hgk
