// Deterministic clustering for coarsening (Sec. 4.1 rating function, cluster
// weight limit and contraction limit; Sec. 11 "Deterministic Clustering for
// Coarsening"): the state of a level and the lists its sub-rounds work on.  The
// sub-rounds run in cluster.cu, the rating walk is in rating.cuh.
//
// Per sub-round s (nodes hashed into S sub-rounds):
//   rating   every unclustered node u of s picks the admissible cluster C
//            maximising r(u, C) = sum over e in I(u), e meeting C, of
//            w(e) / (|e| - 1), in Q20 fixed point with each net term floored,
//            nets of more than T pins skipped, a net counted once per cluster,
//            ties to the smaller id.  Admissible: C != u, C not an unclustered
//            node of the same sub-round, cw[C] + c(u) <= c_max (state at the
//            start of the sub-round).  While rating, the weights of the moves
//            into every target are summed (the paper's fast path).
//   approval a target whose moves all fit under c_max accepts them all;
//            otherwise its movers are sorted by (c(u), u) and the longest
//            prefix that fits is accepted.
//
// Device state per level:
//   rinfo[q] = {cluster, weight word} for every pin position q:
//              the cluster word is the cluster of the pin for the pins of
//              rated nets (2 <= |e| <= T), with every repeat of a cluster
//              inside its net replaced by -1, so a net contributes once per
//              cluster without any per-visit check (-1 for the pins of unrated
//              nets too); the weight word is the cluster's weight, or
//              INT32_MAX when the cluster is an unclustered node of this
//              sub-round (never a candidate).  Both are brought up to date
//              before every sub-round by one pass over the rated nets.  A pin
//              visit of the rating is then one coalesced 8-byte load, with no
//              dependent gather.
//   cst[C]   = {cw[C], status[C]}: cluster weight and status (the node's
//              sub-round while it is unclustered, -1 once it heads a cluster);
//              {cluster, -2} for a node that joined a cluster.
//   imeta[j] = {first pin, pins to visit, Q20 term} of an incident net; a
//              node's records with pins to visit sit at [ioff[u], rend[u]), and
//              lnode[x] = {u, ioff[u], rend[u], c(u)} for every listed node:
//              a node's walk reads its own record, then one record per net.
// Nodes are bucketed per level by class and sub-round.  With W(u) = the pins
// u's rating visits (its ranges of its rated nets) and D = min(W(u), n) (a
// bound on its distinct candidates), a team accumulates u's ratings in a
// shared-memory hash table of 2 D slots (rate_class; the D bounds are the
// autotuner's cutoffs, defaults shown):
//   class 0  D <= 256: one warp, 512 slots;
//   class 1  D <= 1024: four warps, 2048 slots;
//   class 2  on levels whose n fits a shared table direct-indexed by cluster
//            id, W <= 32768: eight, sixteen or 32 warps with that table (as many
//            teams per block as tables fit); on other levels D <= 2048,
//            W <= 65536: eight warps, 4096 slots;
//   class 3  D <= 4096, W <= 65536 (other levels): sixteen warps (32 with
//            64-bit ratings), 8192 slots;
//   class 4  the rest, split over the grid: a table in global memory direct-
//            indexed by cluster id when n <= min(2 W, 65536), filled by items
//            of 32 incident nets spread over the grid (the table padded to a
//            multiple of 4 entries); else P = ceil(D / 13516) parts (64-bit
//            ratings: ceil(D / 9830); P <= 12), a block each, owning the
//            candidates of one hash part in a 22528-slot (16384) shared table
//            with a list of its inserted slots; else a global hash table filled
//            by items.  A second step takes the argmax per node (or the best of
//            the parts' bests).
// Class 4 keeps the heaviest nodes (coarse levels: hundreds of thousands of
// pin visits per node) from serialising a sub-round on one block.  Ratings
// are accumulated in 32-bit words when the level's largest possible rating
// fits, else in 64-bit words; a hash table keeps its cluster ids and its
// ratings in separate arrays (a 32-bit CAS claims a key, an atomic add sums
// into the value).
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "pintile.cuh"
#include "rating.cuh"

namespace hgk {

namespace {

// ------------------------------------------------------- node bucketing

// Team class of a node from W(u) and D = min(W(u), n):
//   0 warp (512 slots)                     D <= 256
//   1 four warps (2048 slots)              D <= 1024 (unless the level is dense)
//   2 block, direct-indexed                the level fits a dense shared table,
//                                          W <= 32768
//     eight warps, 4096-slot hash          D <= 2048, W <= 65536 (other levels)
//   3 sixteen warps, 8192-slot hash        D <= 4096, W <= 65536 (other levels)
//   4 split over the grid                  the rest
__device__ __forceinline__ int rate_class(int64_t W, int32_t records, int32_t n, bool dense_block,
                                          RateCuts cut) {
  const int64_t D = W < n ? W : n;  // bound on the distinct candidate clusters
  if (D <= cut.warp) return 0;
  if (dense_block && W <= DENSE_W && records <= TEAM_RECORDS) return 2;
  if (D <= cut.pair) return 1;
  if (!dense_block && W <= TEAM_W && records <= TEAM_RECORDS) {
    if (D <= cut.quad) return 2;
    if (D <= cut.block) return 3;
  }
  return 4;
}

// W(u) (pins its rating visits: the ranges of its rated nets, or its rated
// incident edges on graph levels) of every node, and the largest bound on a node's rating (sum of its net terms),
// which decides the value width.
// floor(w(e) * 2^20 / (|e| - 1)) for the rated nets (2 <= |e| <= T), else 0;
// at least 1 for a rated net since |e| - 1 < 2^20.
__global__ void k_net_terms(const int32_t* __restrict__ eoff, const int32_t* __restrict__ w,
                            int32_t m, int T, IncMeta* __restrict__ nmeta) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    IncMeta x;
    x.start = eoff[e];
    x.eff = eoff[e + 1] - x.start;
    x.r = (x.eff >= 2 && x.eff <= T)
              ? (((unsigned long long)w[e]) << 20) / (unsigned long long)(x.eff - 1)
              : 0ull;
    if (x.r == 0) x.eff = 0;
    nmeta[e] = x;
  }
}

// ------------------------------------------------ grouped pin order

// A pin visit is wasted when the pin's cluster can never take u: it lies in
// another community, or cw[C] + c(u) > c_max.  Cluster weights only grow
// within a level and cw[C] >= c(v) for every member v, so the pins v with
// c(v) + c(u) > c_max are known before the first sub-round.  On levels where
// such pins abound the pins of every rated net of at most GROUP_NET pins are
// therefore sorted by (community, weight bucket) once per level, and an
// incidence (u, e) walks only the pins of u's community whose bucket does not
// exceed that of c_max - c(u); the exact tests stay in the walk.  The range
// holds all members of every admissible cluster (each is in u's community
// and weighs at most c_max - c(u)), so the cluster's first position, the one
// that carries its word, lies in it.
// Coarse levels: most clusters are too heavy to pair up (of the 440M pin
// visits of a level of 1571 nodes and 5.07M pins, 407M failed the weight test
// and none passed).  With communities: 99 % of the visits of a 1.35M-pin
// input were pins of other communities.  Measured (GB300, with the records
// compacted by k_node_work): coarsening of a 4e6-node large-net input at
// k = 64, 215 -> 143 ms (its levels of 377k nodes and fewer 36.5 -> 23.9,
// 41.2 -> 13.6, 25.3 -> 10.6 ms); with communities on the 1.35M-pin input
// 34.2 -> 16.2 ms; the sort and the range searches take 0.18 and 0.15 ms
// on a level of 5M pins.
constexpr int GROUP_IDX_BITS = 10;
constexpr int GROUP_NET = 1 << GROUP_IDX_BITS;
constexpr int GROUP_W_BITS = 8;
constexpr uint32_t GROUP_W_MASK = (1u << GROUP_W_BITS) - 1;
constexpr uint32_t GROUP_COMM_MASK = (1u << (32 - GROUP_IDX_BITS - GROUP_W_BITS)) - 1;
constexpr int GROUP_WARPS = 8;
constexpr int GROUP_LANES = 8;  // nets of up to as many pins: a lane group each
// Levels without communities are grouped when at least GROUP_HEAVY_NUM /
// GROUP_HEAVY_DEN of their incidences belong to nodes of more than c_max / 2
// (two of these never share a cluster): below that the sort and the range
// searches cost more than the visits they save.
constexpr unsigned long long GROUP_HEAVY_NUM = 1, GROUP_HEAVY_DEN = 4;

// Monotone in c >= 1: exact below 16, then three mantissa bits (at most 231).
__device__ __forceinline__ uint32_t weight_bucket(int32_t c) {
  if (c < 16) return (uint32_t)c;
  const int e = 31 - __clz(c);
  return (uint32_t)(((e - 3) << 3) + (c >> (e - 3)));
}

// Group key of a pin: low bits of its community, then its weight bucket.
__device__ __forceinline__ uint32_t group_key(int32_t comm, int32_t c) {
  return (((uint32_t)comm & GROUP_COMM_MASK) << GROUP_W_BITS) | weight_bucket(c);
}

// Incidences of the nodes of more than c_max / 2.
__global__ void k_heavy_pins(const int32_t* __restrict__ c, const int32_t* __restrict__ ioff,
                             int32_t n, int32_t c_max, unsigned long long* __restrict__ heavy) {
  unsigned long long h = 0;
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x)
    if (2ll * c[u] > (long long)c_max) h += (unsigned long long)(ioff[u + 1] - ioff[u]);
  const unsigned long long v[1] = {h};
  block_add_counters(heavy, v);
}

__device__ __forceinline__ bool level_grouped(const unsigned long long* heavy, int64_t p,
                                              bool comm) {
  return comm || GROUP_HEAVY_DEN * *heavy >= GROUP_HEAVY_NUM * (unsigned long long)p;
}

// The lowest weight bucket goes to the net record's upper bits (terms stay
// below 2^51): a node whose bound lies below it has no candidate in the net.
constexpr int TERM_BITS = 56;
constexpr unsigned long long TERM_MASK = (1ull << TERM_BITS) - 1;

// Sorts the sz <= 32 R pins of one net by group key with the warp: a bitonic
// network over {key, index in the net} words held R per lane (in-thread swaps
// below R, lane shuffles above).  The order of equal keys does not matter.
template <int R>
__device__ __forceinline__ void group_sort(int32_t b, int32_t sz, const int32_t* __restrict__ pins,
                                           const int32_t* __restrict__ c,
                                           const int32_t* __restrict__ comm,
                                           int32_t* __restrict__ gpins,
                                           uint32_t* __restrict__ gkey,
                                           IncMeta* __restrict__ nmeta) {
  const int lane = lane_id();
  uint32_t v[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int32_t i = r * 32 + lane;
    v[r] = ~0u;
    if (i < sz) {
      const int32_t x = pins[b + i];
      v[r] = (group_key(comm ? comm[x] : 0, c[x]) << GROUP_IDX_BITS) | (uint32_t)i;
    }
  }
#pragma unroll 1
  for (int kk = 2; kk <= 32 * R; kk <<= 1) {
#pragma unroll 1
    for (int j = kk >> 1; j >= R; j >>= 1) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int i = lane * R + r;
        const uint32_t y = __shfl_xor_sync(FULL, v[r], j / R);
        const bool keep_min = ((i & kk) == 0) == ((i & j) == 0);
        v[r] = keep_min ? min(v[r], y) : max(v[r], y);
      }
    }
#pragma unroll
    for (int j = R / 2; j > 0; j >>= 1) {
      if (j >= kk) continue;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if ((r ^ j) > r) {
          const bool up = ((lane * R + r) & kk) == 0;
          const uint32_t lo = min(v[r], v[r ^ j]), hi = max(v[r], v[r ^ j]);
          v[r] = up ? lo : hi;
          v[r ^ j] = up ? hi : lo;
        }
      }
    }
  }
  uint32_t low = GROUP_W_MASK;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int32_t i = lane * R + r;
    if (i < sz) {
      low = min(low, (v[r] >> GROUP_IDX_BITS) & GROUP_W_MASK);
      const int32_t from = b + (int32_t)(v[r] & (GROUP_NET - 1));
      gpins[b + i] = pins[from];
      gkey[b + i] = v[r] >> GROUP_IDX_BITS;
    }
  }
  low = __reduce_min_sync(FULL, low);
  if (lane == 0) nmeta->r |= (unsigned long long)low << TERM_BITS;
}

// Eight lanes or a warp per net: gpins = the grouped pin order, gkey = group key per
// position.  Rated nets of more than GROUP_NET pins keep their order.  Of unrated
// nets nothing but the pins' communities is ever read: without communities they
// are left out (on large-net inputs they hold most pins, and one warp each copied
// them: 1.2 ms per level of 31M pins, 0.9 ms without; 0.37 ms with four small nets
// per warp, most of the 864,000 nets).
__global__ void __launch_bounds__(GROUP_WARPS * 32)
k_group_nets(const int32_t* __restrict__ eoff, const int32_t* __restrict__ pins, int32_t m, int T,
             const int32_t* __restrict__ c, const int32_t* __restrict__ comm, int64_t p,
             const unsigned long long* __restrict__ heavy, int32_t* __restrict__ gpins,
             uint32_t* __restrict__ gkey, IncMeta* __restrict__ nmeta) {
  if (!level_grouped(heavy, p, comm != nullptr)) return;
  constexpr int PER = 32 / GROUP_LANES;
  const int lane = lane_id(), sub = lane % GROUP_LANES, first = lane - sub;
  const int64_t stride = (int64_t)gridDim.x * GROUP_WARPS * PER;
  for (int64_t e0 = ((int64_t)blockIdx.x * GROUP_WARPS + warp_in_block()) * PER; e0 < m;
       e0 += stride) {
    const int64_t e = e0 + lane / GROUP_LANES;
    const int32_t b = e < m ? eoff[e] : 0, sz = e < m ? eoff[e + 1] - b : 0;
    const bool rated = sz >= 2 && sz <= T, small = rated && sz <= GROUP_LANES;
    uint32_t v = ~0u;
    int32_t x = 0;
    if (small && sub < sz) {
      x = pins[b + sub];
      v = (group_key(comm ? comm[x] : 0, c[x]) << GROUP_IDX_BITS) | (uint32_t)sub;
    }
    uint32_t low = v == ~0u ? GROUP_W_MASK : (v >> GROUP_IDX_BITS) & GROUP_W_MASK;
#pragma unroll
    for (int kk = 2; kk <= GROUP_LANES; kk <<= 1)
#pragma unroll
      for (int j = kk >> 1; j > 0; j >>= 1) {
        const uint32_t y = __shfl_xor_sync(FULL, v, j);
        const bool keep_min = ((sub & kk) == 0) == ((sub & j) == 0);
        v = keep_min ? min(v, y) : max(v, y);
      }
#pragma unroll
    for (int d = GROUP_LANES / 2; d > 0; d >>= 1) low = min(low, __shfl_xor_sync(FULL, low, d));
    x = __shfl_sync(FULL, x, first + (int)(v & (GROUP_LANES - 1)));
    if (small && sub < sz) {
      gpins[b + sub] = x;
      gkey[b + sub] = v >> GROUP_IDX_BITS;
      if (sub == 0) nmeta[e].r |= (unsigned long long)low << TERM_BITS;
    }
    for (unsigned rest = __ballot_sync(FULL, sub == 0 && sz > 0 && !small && (rated || comm)); rest;
         rest &= rest - 1) {
      const int l = __ffs(rest) - 1;
      const int32_t wb = __shfl_sync(FULL, b, l), wsz = __shfl_sync(FULL, sz, l);
      IncMeta* meta = nmeta + e0 + l / GROUP_LANES;
      if (wsz < 2 || wsz > T || wsz > GROUP_NET) {
        for (int32_t q = wb + lane; q < wb + wsz; q += 32) gpins[q] = pins[q];
      } else if (wsz <= 32) {
        group_sort<1>(wb, wsz, pins, c, comm, gpins, gkey, meta);
      } else if (wsz <= 128) {
        group_sort<4>(wb, wsz, pins, c, comm, gpins, gkey, meta);
      } else if (wsz <= 512) {
        group_sort<16>(wb, wsz, pins, c, comm, gpins, gkey, meta);
      } else {
        group_sort<32>(wb, wsz, pins, c, comm, gpins, gkey, meta);
      }
    }
  }
}

// First index of gkey[lo, hi) that is >= key (hi if none).
__device__ __forceinline__ int32_t group_lower(const uint32_t* __restrict__ gkey, int32_t lo,
                                               int32_t hi, uint32_t key) {
  while (lo < hi) {
    const int32_t mid = (lo + hi) >> 1;
    if (gkey[mid] < key) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// {u, ioff[u], rend[u], c(u)} of every listed node.
__global__ void k_list_nodes(const int32_t* __restrict__ list, int32_t cnt,
                             const int32_t* __restrict__ ioff, const int32_t* __restrict__ rend,
                             const int32_t* __restrict__ c, int4* __restrict__ lnode) {
  for (int32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < cnt; x += gridDim.x * blockDim.x) {
    const int32_t u = list[x];
    lnode[x] = make_int4(u, ioff[u], rend[u], c[u]);
  }
}

// The weight and records of every node.  A record is the net's {start, pins,
// term} (one 16-byte gather), on grouped levels cut to the range of u's possible
// candidates; the records that hold a visit are written to the front of the
// node's range (rend[u] = their end), so the walks never load the records of
// unrated nets or of nets without a candidate (on large-net inputs most
// incidences are of unrated nets; on grouped coarse levels a node of thousands of
// nets may have a handful left).  Visits bound the records a walk loads.
//
// Bound by the gathers of the net records and, on grouped levels, by the
// dependent steps of the range searches: eight lanes take a node, a warp one of
// more than WORK_SMALL nets, a block one of more than WORK_WIDE, and warps queue
// the records that need a search until every lane has one (an incidence in ten or
// fewer does on coarse levels).
constexpr int WORK_LANES = 8;
constexpr int32_t WORK_SMALL = 64, WORK_WIDE = 512;
constexpr int WORK_WARPS = 8;

struct NodeRange {     // of a node on a grouped level
  uint32_t base, top;  // community part of its group key, highest weight bucket
  uint32_t own;        // its own weight bucket
  int32_t left;        // weight left beside it
};

struct WorkArgs {
  const int32_t *ioff, *inets;
  const IncMeta* nmeta;
  int32_t n;
  int64_t p;
  bool graph;
  const int32_t *c, *comm;
  int32_t c_max;
  const uint32_t* gkey;
  IncMeta* imeta;
  int32_t *wof, *rend;
  unsigned long long* max_r;  // largest rating, incidences of heavy nodes, total W
  int32_t *big, *nbig;        // nodes of more than WORK_WIDE nets
};

__device__ __forceinline__ NodeRange node_range(const WorkArgs& A, int64_t u) {
  const int32_t cu = A.c[u];
  NodeRange r;
  r.left = A.c_max - cu;
  r.top = r.left > 0 ? weight_bucket(r.left) : 0u;
  r.own = weight_bucket(cu);
  r.base = group_key(A.comm ? A.comm[u] : 0, cu) & ~GROUP_W_MASK;
  return r;
}

// The record of net e, empty if the lowest bucket already says so.
__device__ __forceinline__ IncMeta net_record(const WorkArgs& A, bool grouped, int32_t e,
                                              const NodeRange& r) {
  IncMeta x = A.nmeta[e];
  if (grouped) {
    const uint32_t low = (uint32_t)(x.r >> TERM_BITS);
    x.r &= TERM_MASK;
    if (x.eff <= GROUP_NET && (r.left <= 0 || low > r.top)) x.eff = 0;
  }
  return x;
}

// The range of the node's possible candidates (grouped levels).
__device__ __forceinline__ void cut_record(const WorkArgs& A, IncMeta& x, const NodeRange& r) {
  if (x.eff == 0 || x.eff > GROUP_NET) return;
  const int32_t end = x.start + x.eff;
  if (A.comm) x.start = group_lower(A.gkey, x.start, end, r.base);
  x.eff = group_lower(A.gkey, x.start, end, r.base + r.top + 1) - x.start;
  // a range holding u alone has no candidate
  if (x.eff == 1 && r.own <= r.top) x.eff = 0;
}

// The records [beg, end) of one node by `warps` warps, this one number wv;
// *to (shared) counts the records written.
__device__ __forceinline__ void walk_node(const WorkArgs& A, bool grouped, int32_t beg,
                                          int32_t end, const NodeRange& r, int wv, int warps,
                                          IncMeta* queue, int32_t* to, long long& W,
                                          unsigned long long& R) {
  const int lane = lane_id();
  const unsigned below = (1u << lane) - 1u;
  int held = 0;
  auto emit = [&](const IncMeta& x) {
    const unsigned live = __ballot_sync(FULL, x.eff != 0);
    if (!live) return;
    int32_t at = 0;
    if (lane == 0) at = atomicAdd(to, __popc(live));
    at = beg + __shfl_sync(FULL, at, 0) + __popc(live & below);
    if (x.eff != 0) {
      W += A.graph ? 1 : x.eff;  // a graph visits the other endpoint only
      R += x.r;
      if (!A.graph) A.imeta[at] = x;
    }
  };
  auto drain = [&](int count) {
    IncMeta x{0, 0, 0};
    held -= count;
    if (lane < count) x = queue[held + lane];
    __syncwarp();
    cut_record(A, x, r);
    emit(x);
  };
  for (int32_t j0 = beg + wv * 64; j0 < end; j0 += warps * 64) {
    const int32_t ja = j0 + lane, jb = ja + 32;
    IncMeta x[2] = {{0, 0, 0}, {0, 0, 0}};
    const int32_t ea = ja < end ? A.inets[ja] : -1, eb = jb < end ? A.inets[jb] : -1;
    if (ea >= 0) x[0] = net_record(A, grouped, ea, r);
    if (eb >= 0) x[1] = net_record(A, grouped, eb, r);
#pragma unroll
    for (int y = 0; y < 2; ++y) {
      if (!grouped) {
        emit(x[y]);
        continue;
      }
      const unsigned live = __ballot_sync(FULL, x[y].eff != 0);
      if (x[y].eff != 0) queue[held + __popc(live & below)] = x[y];
      __syncwarp();
      held += __popc(live);
      if (held >= 32) drain(32);
    }
  }
  if (held > 0) drain(held);
}

__global__ void __launch_bounds__(WORK_WARPS * 32) k_node_work(WorkArgs A) {
  constexpr int PER = 32 / WORK_LANES;
  __shared__ IncMeta s_queue[WORK_WARPS][64];
  __shared__ int32_t s_to[WORK_WARPS];
  unsigned long long lr = 0, lw = 0;
  const bool grouped = !A.graph && level_grouped(A.max_r + 1, A.p, A.comm != nullptr);
  const int lane = lane_id(), sub = lane % WORK_LANES, first = lane - sub;
  const int wv = warp_in_block();
  const int64_t stride = (((int64_t)gridDim.x * blockDim.x) >> 5) * PER;
  for (int64_t u0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * PER; u0 < A.n;
       u0 += stride) {
    const int64_t u = u0 + lane / WORK_LANES;
    const bool on = u < A.n;
    const int32_t beg = on ? A.ioff[u] : 0, end = on ? A.ioff[u + 1] : 0;
    NodeRange r{0u, 0u, 0u, 0};
    if (grouped && on) r = node_range(A, u);
    long long W = 0;
    unsigned long long R = 0;
    int32_t out = beg;
    const bool wide = end - beg > WORK_SMALL, big = end - beg > WORK_WIDE;
    const int32_t stop = wide ? beg : end;
    for (int32_t j0 = beg; __any_sync(FULL, j0 < stop); j0 += WORK_LANES) {
      const int32_t j = j0 + sub;
      IncMeta x{0, 0, 0};
      if (j < stop) {
        x = net_record(A, grouped, A.inets[j], r);
        if (grouped) cut_record(A, x, r);
      }
      const unsigned live =
          (__ballot_sync(FULL, x.eff != 0) >> first) & ((1u << WORK_LANES) - 1u);
      if (x.eff != 0) {
        W += A.graph ? 1 : x.eff;
        R += x.r;
        if (!A.graph) A.imeta[out + __popc(live & ((1u << sub) - 1u))] = x;
      }
      out += __popc(live);
    }
    for (unsigned rest = __ballot_sync(FULL, sub == 0 && wide && !big); rest; rest &= rest - 1) {
      const int l = __ffs(rest) - 1;
      const int32_t wb = __shfl_sync(FULL, beg, l), we = __shfl_sync(FULL, end, l);
      NodeRange wr;
      wr.base = __shfl_sync(FULL, r.base, l);
      wr.top = __shfl_sync(FULL, r.top, l);
      wr.own = __shfl_sync(FULL, r.own, l);
      wr.left = __shfl_sync(FULL, r.left, l);
      long long WW = 0;
      unsigned long long RR = 0;
      if (lane == 0) s_to[wv] = 0;
      __syncwarp();
      walk_node(A, grouped, wb, we, wr, 0, 1, s_queue[wv], &s_to[wv], WW, RR);
      __syncwarp();
      if (first == l) out = wb + s_to[wv];
      __syncwarp();
      // one lane of the node's group takes the warp's sums
      WW = warp_sum(WW);
      RR = warp_sum(RR);
      if (lane == l) {
        W += WW;
        R += RR;
      }
    }
#pragma unroll
    for (int d = WORK_LANES / 2; d > 0; d >>= 1) {
      W += __shfl_xor_sync(FULL, W, d);
      R += __shfl_xor_sync(FULL, R, d);
    }
    if (sub == 0 && on) {
      if (big) {
        A.big[atomicAdd(A.nbig, 1)] = (int32_t)u;
      } else {
        lr = R > lr ? R : lr;
        lw += (unsigned long long)W;
        A.wof[u] = W > 0x7fffffff ? 0x7fffffff : (int32_t)W;
        A.rend[u] = A.graph ? end : out;
      }
    }
  }
  lr = warp_max(lr);
  if (lane == 0 && lr) atomicMax(A.max_r, lr);
  const unsigned long long wsum[1] = {lw};
  block_add_counters(A.max_r + 2, wsum);
}

__global__ void __launch_bounds__(WORK_WARPS * 32) k_node_work_big(WorkArgs A) {
  __shared__ IncMeta s_queue[WORK_WARPS][64];
  __shared__ int32_t s_to;
  __shared__ unsigned long long s_red[32];
  const bool grouped = !A.graph && level_grouped(A.max_r + 1, A.p, A.comm != nullptr);
  const int32_t count = *A.nbig;
  unsigned long long lr = 0, lw = 0;
  for (int32_t i = blockIdx.x; i < count; i += gridDim.x) {
    const int32_t u = A.big[i];
    const int32_t beg = A.ioff[u], end = A.ioff[u + 1];
    NodeRange r{0u, 0u, 0u, 0};
    if (grouped) r = node_range(A, u);
    if (threadIdx.x == 0) s_to = 0;
    __syncthreads();
    long long W = 0;
    unsigned long long R = 0;
    walk_node(A, grouped, beg, end, r, warp_in_block(), WORK_WARPS, s_queue[warp_in_block()],
              &s_to, W, R);
    const unsigned long long WS = block_sum((unsigned long long)W, s_red);
    __syncthreads();
    R = block_sum(R, s_red);
    __syncthreads();
    if (threadIdx.x == 0) {
      lr = R > lr ? R : lr;
      lw += WS;
      A.wof[u] = WS > 0x7fffffffull ? 0x7fffffff : (int32_t)WS;
      A.rend[u] = A.graph ? end : beg + s_to;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0 && lr) atomicMax(A.max_r, lr);
  if (threadIdx.x == 0 && lw) atomicAdd(A.max_r + 2, lw);
}

// key = class * S + sub-round of every node with W(u) > 0, and the counts
// (collected per block: the atomics of all nodes on a hundred counters took 0.24
// ms at 1e6 nodes, 0.012 now).
__global__ void k_node_classify(const int32_t* __restrict__ wof, const int32_t* __restrict__ ioff,
                                const int32_t* __restrict__ rend, int32_t n, uint64_t seed,
                                int level, int S, bool dense_block, RateCuts cut, int nkeys,
                                int32_t* __restrict__ key_of, int32_t* __restrict__ kcount) {
  extern __shared__ int32_t s_cnt[];
  for (int i = threadIdx.x; i < nkeys; i += blockDim.x) s_cnt[i] = 0;
  __syncthreads();
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x) {
    const int32_t W = wof[u];
    int32_t key = -1;
    if (W > 0) {
      key = rate_class(W, rend[u] - ioff[u], n, dense_block, cut) * S +
            subround_of_node_cluster(seed, level, (int)u, S);
      atomicAdd(&s_cnt[key], 1);
    }
    key_of[u] = key;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nkeys; i += blockDim.x)
    if (s_cnt[i]) atomicAdd(&kcount[i], s_cnt[i]);
}

// Nodes to their key's range of the list: a block claims its tile's slots of
// every key at once.
constexpr int SCATTER_PER = 4;  // nodes per thread and tile

__global__ void __launch_bounds__(256)
k_node_scatter(const int32_t* __restrict__ key_of, int32_t n, int nkeys,
               const int32_t* __restrict__ kcount, int32_t* __restrict__ kfill,
               int32_t* __restrict__ list) {
  extern __shared__ int32_t s_off[];  // first slot of every key, then the tile's counts
  int32_t* s_cnt = s_off + nkeys;
  if (warp_in_block() == 0) {
    int32_t carry = 0;
    for (int i0 = 0; i0 < nkeys; i0 += 32) {
      const int i = i0 + lane_id();
      const int32_t x = i < nkeys ? kcount[i] : 0;
      const int32_t incl = warp_inclusive_scan(x);
      if (i < nkeys) s_off[i] = carry + incl - x;
      carry += __shfl_sync(FULL, incl, 31);
    }
  }
  for (int64_t b = (int64_t)blockIdx.x * 256 * SCATTER_PER; b < n;
       b += (int64_t)gridDim.x * 256 * SCATTER_PER) {
    for (int i = threadIdx.x; i < nkeys; i += 256) s_cnt[i] = 0;
    __syncthreads();
    int32_t key[SCATTER_PER], slot[SCATTER_PER];
#pragma unroll
    for (int x = 0; x < SCATTER_PER; ++x) {
      const int64_t u = b + x * 256 + threadIdx.x;
      key[x] = u < n ? key_of[u] : -1;
      if (key[x] >= 0) slot[x] = atomicAdd(&s_cnt[key[x]], 1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nkeys; i += 256)
      if (s_cnt[i]) s_cnt[i] = s_off[i] + atomicAdd(&kfill[i], s_cnt[i]);
    __syncthreads();
#pragma unroll
    for (int x = 0; x < SCATTER_PER; ++x)
      if (key[x] >= 0) list[s_cnt[key[x]] + slot[x]] = (int32_t)(b + x * 256 + threadIdx.x);
    __syncthreads();
  }
}

// Work items and global table of every split node (D = min(W(u), n)):
//   direct-indexed global table (n entries) when n <= min(2 W(u), 65536), so
//   the table costs no more than the accumulation: groups of 32 nets over
//   the grid (items);
//   else P = ceil(D / part_d) shared-memory parts when P <= part_max (no
//   global table);
//   else a global hash table of a power of two >= 2 D + 2 slots, with items.
__global__ void k_split_sizes(const int4* __restrict__ lsplit, int32_t nsplit,
                              const int32_t* __restrict__ wof,
                              int32_t n, int32_t part_d, int32_t part_max,
                              int32_t* __restrict__ items,
                              int32_t* __restrict__ parts, int32_t* __restrict__ cap,
                              int8_t* __restrict__ dense) {
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nsplit; i += gridDim.x * blockDim.x) {
    const int4 nd = lsplit[i];
    const int32_t u = nd.x, deg = nd.z - nd.y;
    const bool d = n <= SPLIT_DENSE_MAX && (int64_t)n <= 2 * (int64_t)wof[u];
    const int32_t D = min(wof[u], n);
    const int32_t P = d ? 0 : (D + part_d - 1) / part_d;
    const bool part = !d && P <= part_max;
    items[i] = part ? 0 : (deg + 31) / 32;
    parts[i] = part ? P : 0;
    dense[i] = d ? 1 : 0;
    if (d) {
      cap[i] = (n + 3) & ~3;  // a multiple of 4: every table starts 16-byte aligned
    } else if (part) {
      cap[i] = 0;
    } else {
      const int64_t want = 2 * (int64_t)D + 2;
      int64_t c = 1;
      while (c < want) c <<= 1;
      cap[i] = (int32_t)c;
    }
  }
}

__global__ void k_split_items(const int32_t* __restrict__ item_off, int32_t nsplit,
                              int32_t* __restrict__ item_node) {
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nsplit; i += gridDim.x * blockDim.x)
    for (int32_t t = item_off[i]; t < item_off[i + 1]; ++t) item_node[t] = i;
}

__global__ void k_widen(const int32_t* __restrict__ in, int64_t* __restrict__ out, int32_t cnt) {
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += gridDim.x * blockDim.x)
    out[i] = in[i];
}

template <typename VT>
__global__ void k_init_table(int32_t* key, VT* val, size_t cnt) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt;
       i += (size_t)gridDim.x * blockDim.x) {
    key[i] = EMPTY_KEY;
    val[i] = 0;
  }
}

// ---------------------------------------------- cluster words at the start

// The rated nets by size class.
__global__ void k_net_lists(const int32_t* __restrict__ eoff, int32_t m, int T, NetLists N,
                            int32_t* __restrict__ count) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); b < m; b += stride) {
    const int64_t e = b + lane_id();
    int cls = -1;
    int2 net = make_int2(0, 0);
    if (e < m) {
      net.x = eoff[e];
      net.y = eoff[e + 1] - net.x;
      if (net.y >= 2 && net.y <= T) cls = net_size_class(net.y);
    }
    const int32_t slot = warp_claim_slot(count, cls, __ballot_sync(FULL, e < m));
    if (slot >= 0) N.list[cls][slot] = net;
  }
}

// rinfo at the start of a level, for sub-round 0: cluster word = the pin for
// the pins of rated nets, -1 for the others; weight word = the pin's weight,
// or INT32_MAX for a node of sub-round 0 (pin tiles).
__global__ void __launch_bounds__(PIN_TILE_THREADS)
k_rinfo_init(const int32_t* __restrict__ eoff, const int32_t* __restrict__ pins,
             const int32_t* __restrict__ tile_net, int32_t m, int64_t p, int T,
             const int2* __restrict__ cst, int2* __restrict__ rinfo) {
  __shared__ int32_t s_off[PIN_TILE + 3];
  const int64_t ntiles = num_pin_tiles(p);
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    PinTileView v = stage_pin_tile(eoff, tile_net, m, p, t, s_off);
    for (int64_t q = v.q0 + threadIdx.x; q < v.q1; q += blockDim.x) {
      const int32_t i = net_in_tile(s_off, v.count, q);
      const int32_t sz = s_off[i + 1] - s_off[i];
      int2 r = make_int2(-1, 0);
      if (sz >= 2 && sz <= T) {
        r.x = pins[q];
        const int2 cs = cst[r.x];
        r.y = cs.y == 0 ? 0x7fffffff : cs.x;
      }
      rinfo[q] = r;
    }
    __syncthreads();
  }
}

// pcomm[q] = comm[pins[q]] for every pin position.
__global__ void k_pin_comm(const int32_t* __restrict__ pins, int64_t p,
                           const int32_t* __restrict__ comm, int32_t* __restrict__ pcomm) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < p;
       q += (int64_t)gridDim.x * blockDim.x)
    pcomm[q] = comm[pins[q]];
}

__global__ void k_init_cluster(const int32_t* __restrict__ c, int32_t n, uint64_t seed, int level,
                               int S, int32_t* __restrict__ rep, int2* __restrict__ cst,
                               int32_t* __restrict__ slot_of) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x) {
    rep[u] = (int32_t)u;
    cst[u] = make_int2(c[u], subround_of_node_cluster(seed, level, (int)u, S));
    slot_of[u] = -1;
  }
}


// ---------------------------------------------------------- host side

// The clustering of a level with split nodes of at most part_max parts.  Returns
// false (and nothing of use) when a part's table was full.
bool cluster_with_parts(const Ctx& cx, Level& L, const CoarsenParams& P, int32_t part_max,
                        CoarsenCounters& cc, DBuf<int32_t>& cw_out) {
  const int32_t n = L.n;
  const int S = P.S;
  const int nkeys = S * NCLASS;
  L.rep.alloc(&cx.alloc, (size_t)n);
  cw_out.alloc(&cx.alloc, (size_t)n);
  DBuf<int2> cst;
  DBuf<int32_t> target, gw, gcnt, slot_of, slot_c, slot_off, slot_fill, mv, touched, glist, key_of,
      wof, kcount, kfill, list, words, clusters;
  DBuf<int2> rinfo;
  DBuf<unsigned long long> stats, max_r;
  const size_t ncap = (size_t)n + 1;
  cst.alloc(&cx.alloc, ncap);
  target.alloc(&cx.alloc, ncap);
  gw.alloc(&cx.alloc, ncap);
  gcnt.alloc(&cx.alloc, ncap);
  slot_of.alloc(&cx.alloc, ncap);
  slot_c.alloc(&cx.alloc, ncap);
  slot_off.alloc(&cx.alloc, ncap);
  slot_fill.alloc(&cx.alloc, ncap);
  mv.alloc(&cx.alloc, ncap);
  touched.alloc(&cx.alloc, ncap);
  glist.alloc(&cx.alloc, ncap);
  key_of.alloc(&cx.alloc, ncap);
  wof.alloc(&cx.alloc, ncap);
  list.alloc(&cx.alloc, ncap);
  kcount.alloc(&cx.alloc, (size_t)nkeys);
  kfill.alloc(&cx.alloc, (size_t)nkeys);
  words.alloc(&cx.alloc, (size_t)S * CW_WORDS);
  clusters.alloc(&cx.alloc, 1);
  max_r.alloc(&cx.alloc, 3);  // largest possible rating, incidences of heavy nodes, total W
  stats.alloc(&cx.alloc, (size_t)ST_TOTAL + 1);  // then the barrier's two words
  rinfo.alloc(&cx.alloc, L.graph ? 1 : (size_t)std::max<int64_t>(L.p, 1));
  HG_CUDA(cudaMemsetAsync(gw.p, 0, gw.bytes(), cx.stream));
  HG_CUDA(cudaMemsetAsync(gcnt.p, 0, gcnt.bytes(), cx.stream));
  HG_CUDA(cudaMemsetAsync(slot_fill.p, 0, slot_fill.bytes(), cx.stream));
  HG_CUDA(cudaMemsetAsync(kcount.p, 0, kcount.bytes(), cx.stream));
  HG_CUDA(cudaMemsetAsync(kfill.p, 0, kfill.bytes(), cx.stream));
  HG_CUDA(cudaMemsetAsync(words.p, 0, words.bytes(), cx.stream));
  HG_CUDA(cudaMemsetAsync(max_r.p, 0, max_r.bytes(), cx.stream));
  HG_CUDA(cudaMemsetAsync(stats.p, 0, stats.bytes(), cx.stream));
  HG_CUDA(cudaMemcpyAsync(clusters.p, &n, sizeof(int32_t), cudaMemcpyHostToDevice, cx.stream));
  // graph levels rate from the adjacency array: no pin records, no
  // (net, cluster) map
  const bool records = L.p > 0 && !L.graph;
  DBuf<int32_t> tiles;
  const int g_nodes = grid_for(n, 256, cx.num_sms, 4);
  k_init_cluster<<<g_nodes, 256, 0, cx.stream>>>(L.c.p, n, P.seed, P.level, S, L.rep.p, cst.p,
                                                 slot_of.p);
  check_launch("init_cluster");
  DBuf<IncMeta> nmeta;
  nmeta.alloc(&cx.alloc, (size_t)std::max<int32_t>(L.m, 1));
  if (L.m > 0) {
    k_net_terms<<<grid_for(L.m, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(L.eoff.p, L.w.p, L.m,
                                                                          P.T, nmeta.p);
    check_launch("net_terms");
  }
  // hypergraph levels: the grouped pin order (where it pays, decided on the
  // device) and the net records of every node
  DBuf<IncMeta> imeta;
  DBuf<int32_t> gpins, rend;
  DBuf<uint32_t> gkey;
  rend.alloc(&cx.alloc, ncap);
  if (records) {
    gpins.alloc(&cx.alloc, (size_t)L.p);
    gkey.alloc(&cx.alloc, (size_t)L.p);
    imeta.alloc(&cx.alloc, (size_t)L.p);
    k_heavy_pins<<<g_nodes, 256, 0, cx.stream>>>(L.c.p, L.ioff.p, n, P.c_max, max_r.p + 1);
    check_launch("heavy_pins");
    k_group_nets<<<grid_for(L.m, GROUP_WARPS * (32 / GROUP_LANES), cx.num_sms, 8),
                   GROUP_WARPS * 32, 0, cx.stream>>>(
        L.eoff.p, L.pins.p, L.m, P.T, L.c.p, L.comm.p, L.p, max_r.p + 1, gpins.p, gkey.p,
        nmeta.p);
    check_launch("group_nets");
    if (cx.launches) *cx.launches += 2;
  }
  DBuf<int32_t> big;  // nodes of more than WORK_WIDE nets, then their number
  const size_t nb = (size_t)(L.p / (WORK_WIDE + 1)) + 1;
  big.alloc(&cx.alloc, nb + 1);
  HG_CUDA(cudaMemsetAsync(big.p + nb, 0, sizeof(int32_t), cx.stream));
  const WorkArgs wa{L.ioff.p, L.inets.p, nmeta.p, n,      L.p,    L.graph, L.c.p, L.comm.p,
                    P.c_max,  gkey.p,    imeta.p, wof.p,  rend.p, max_r.p, big.p, big.p + nb};
  k_node_work<<<grid_for(n, WORK_WARPS * (32 / WORK_LANES), cx.num_sms, 8), WORK_WARPS * 32, 0,
                cx.stream>>>(wa);
  check_launch("node_work");
  if (L.p > WORK_WIDE) {
    k_node_work_big<<<grid_for((int64_t)nb, 1, cx.num_sms, 8), WORK_WARPS * 32, 0, cx.stream>>>(wa);
    check_launch("node_work_big");
    if (cx.launches) *cx.launches += 1;
  }
  unsigned long long hmax[3];
  read_back(cx, hmax, max_r.p, sizeof(hmax));
  const unsigned long long hmax_r = hmax[0];
  // the pins the rating works on
  const bool grouped =
      records && (L.comm.p || GROUP_HEAVY_DEN * hmax[1] >= GROUP_HEAVY_NUM * (unsigned long long)L.p);
  const int32_t* rpins = grouped ? gpins.p : L.pins.p;
  if (!grouped) gpins.release();
  gkey.release();
  nmeta.release();
  if (records) {
    tiles.alloc(&cx.alloc, (size_t)num_pin_tiles(L.p) + 1);
    build_tile_index(cx, L.eoff.p, L.m, L.p, tiles.p);
    k_rinfo_init<<<grid_for(num_pin_tiles(L.p), 1, cx.num_sms, 8), PIN_TILE_THREADS, 0,
                   cx.stream>>>(L.eoff.p, rpins, tiles.p, L.m, L.p, P.T, cst.p,
                                rinfo.p);
    check_launch("rinfo_init");
    if (cx.launches) *cx.launches += 1;
  }
  // 32-bit rating words when no node's total rating can reach 2^31; block
  // tables are direct-indexed when one value and one used-list entry per
  // node of the level fit the shared-memory budget
  const bool narrow = hmax_r < (1ull << 31);
  const size_t vbytes = narrow ? 4 : 8;
  const size_t dense_bytes = (((size_t)n + 3) & ~(size_t)3) * (vbytes + 4);
  const bool dense_block = (size_t)n * (vbytes + 4) <= DENSE_SMEM;
  k_node_classify<<<g_nodes, 256, nkeys * sizeof(int32_t), cx.stream>>>(
      wof.p, L.ioff.p, rend.p, n, P.seed, P.level, S, dense_block, P.cuts, nkeys, key_of.p,
      kcount.p);
  check_launch("node_classify");
  k_node_scatter<<<grid_for(n, 256 * SCATTER_PER, cx.num_sms, 4), 256,
                   2 * nkeys * sizeof(int32_t), cx.stream>>>(key_of.p, n, nkeys, kcount.p,
                                                            kfill.p, list.p);
  check_launch("node_scatter");
  if (cx.launches) *cx.launches += 5;

  std::vector<int32_t> hcount(nkeys);
  read_back(cx, hcount.data(), kcount.p, sizeof(int32_t) * nkeys);
  std::vector<int32_t> hoff(nkeys + 1, 0);
  for (int i = 0; i < nkeys; ++i) hoff[i + 1] = hoff[i] + hcount[i];
  // per listed node {u, ioff[u], rend[u], c(u)}, for the rating walks
  DBuf<int4> lnode;
  lnode.alloc(&cx.alloc, (size_t)std::max<int32_t>(hoff[nkeys], 1));
  if (hoff[nkeys] > 0) {
    k_list_nodes<<<grid_for(hoff[nkeys], 256, cx.num_sms, 8), 256, 0, cx.stream>>>(
        list.p, hoff[nkeys], L.ioff.p, rend.p, L.c.p, lnode.p);
    check_launch("list_nodes");
    if (cx.launches) *cx.launches += 1;
  }

  // ---- the sub-rounds' node ranges and the split plan: items, parts, table
  // offsets and footprint per sub-round
  std::vector<SubPlan> plan((size_t)S);
  const int32_t split_base = hoff[SPLIT_CLASS * S];
  const int32_t nsplit = hoff[NCLASS * S] - split_base;
  for (int s = 0; s < S; ++s) {
    SubPlan& sp = plan[s];
    sp = SubPlan{};
    for (int c = 0; c < NCLASS; ++c) {
      sp.lo[c] = hoff[c * S + s];
      sp.hi[c] = hoff[c * S + s + 1];
    }
  }
  DBuf<int32_t> item_node, item_off, part_node, part_off, tnused, res_c, tkey, tused;
  DBuf<int64_t> tab_off, tab_cap;
  DBuf<int8_t> tab_dense;
  DBuf<unsigned char> res_v, tval;
  bool any_parts = false;
  if (nsplit > 0) {
    DBuf<int32_t> items, parts, cap32;
    items.alloc(&cx.alloc, (size_t)nsplit + 1);
    parts.alloc(&cx.alloc, (size_t)nsplit + 1);
    cap32.alloc(&cx.alloc, (size_t)nsplit + 1);
    item_off.alloc(&cx.alloc, (size_t)nsplit + 1);
    part_off.alloc(&cx.alloc, (size_t)nsplit + 1);
    tab_off.alloc(&cx.alloc, (size_t)nsplit + 1);
    tab_cap.alloc(&cx.alloc, (size_t)nsplit + 1);
    tab_dense.alloc(&cx.alloc, (size_t)nsplit + 1);
    tnused.alloc(&cx.alloc, (size_t)nsplit + 1);
    HG_CUDA(cudaMemsetAsync(tnused.p, 0, tnused.bytes(), cx.stream));
    const int gs = grid_for(nsplit, 256, cx.num_sms, 4);
    k_split_sizes<<<gs, 256, 0, cx.stream>>>(
        lnode.p + split_base, nsplit, wof.p, n, narrow ? PartCfg<uint32_t>::D : PartCfg<unsigned long long>::D,
        part_max, items.p, parts.p, cap32.p, tab_dense.p);
    check_launch("split_sizes");
    scan_exclusive_i32(cx, items.p, item_off.p, nsplit, item_off.p + nsplit);
    scan_exclusive_i32(cx, parts.p, part_off.p, nsplit, part_off.p + nsplit);
    scan_exclusive_i32_to_i64(cx, cap32.p, tab_off.p, nsplit, tab_off.p + nsplit);
    k_widen<<<gs, 256, 0, cx.stream>>>(cap32.p, tab_cap.p, nsplit);
    check_launch("widen");
    std::vector<int32_t> hio((size_t)nsplit + 1), hso((size_t)nsplit + 1);
    std::vector<int64_t> hto((size_t)nsplit + 1);
    wait_stream(cx);
    HG_CUDA(cudaMemcpyAsync(hio.data(), item_off.p, sizeof(int32_t) * hio.size(),
                            cudaMemcpyDeviceToHost, cx.stream));
    HG_CUDA(cudaMemcpyAsync(hso.data(), part_off.p, sizeof(int32_t) * hso.size(),
                            cudaMemcpyDeviceToHost, cx.stream));
    HG_CUDA(cudaMemcpyAsync(hto.data(), tab_off.p, sizeof(int64_t) * hto.size(),
                            cudaMemcpyDeviceToHost, cx.stream));
    check_status(cx);
    int64_t tab_span = 0;  // largest table footprint of one sub-round
    for (int s = 0; s < S; ++s) {
      SubPlan& sp = plan[s];
      const int32_t lo = sp.lo[SPLIT_CLASS] - split_base, hi = sp.hi[SPLIT_CLASS] - split_base;
      sp.item_lo = hio[lo];
      sp.item_hi = hio[hi];
      sp.part_lo = hso[lo];
      sp.part_hi = hso[hi];
      sp.tab_lo = hto[lo];
      tab_span = std::max<int64_t>(tab_span, hto[hi] - hto[lo]);
      // tables to scan, or nodes of more than one part
      sp.argmax = sp.item_hi > sp.item_lo || sp.part_hi - sp.part_lo > hi - lo;
      any_parts |= sp.part_hi > sp.part_lo;
    }
    item_node.alloc(&cx.alloc, (size_t)std::max<int32_t>(hio[nsplit], 1));
    k_split_items<<<gs, 256, 0, cx.stream>>>(item_off.p, nsplit, item_node.p);
    check_launch("split_items");
    const size_t nparts = (size_t)std::max<int32_t>(hso[nsplit], 1);
    part_node.alloc(&cx.alloc, nparts);
    res_v.alloc(&cx.alloc, nparts * vbytes);
    res_c.alloc(&cx.alloc, nparts);
    k_split_items<<<gs, 256, 0, cx.stream>>>(part_off.p, nsplit, part_node.p);
    check_launch("split_parts");
    const size_t span = (size_t)std::max<int64_t>(tab_span, 1);
    tval.alloc(&cx.alloc, span * vbytes);
    tkey.alloc(&cx.alloc, span);
    tused.alloc(&cx.alloc, span);
    const int gi = grid_for((int64_t)span, 256, cx.num_sms, 8);
    if (narrow)
      k_init_table<uint32_t><<<gi, 256, 0, cx.stream>>>(
          tkey.p, reinterpret_cast<uint32_t*>(tval.p), span);
    else
      k_init_table<unsigned long long><<<gi, 256, 0, cx.stream>>>(
          tkey.p, reinterpret_cast<unsigned long long*>(tval.p), span);
    check_launch("init_table");
    if (cx.launches) *cx.launches += 11;
  }

  // hypergraph levels: rated nets by size class, and node bitmaps for nets
  // above BIG_NET pins when such nets are rated
  ClusterArgs A{};
  DBuf<int2> netlist;
  DBuf<int32_t> netcount;
  DBuf<unsigned> bitmaps;
  if (records) {
    int64_t cap[NSIZE], total = 0;
    const int64_t least[NSIZE] = {1, 5, 9, 17, 33, BIG_NET + 1};
    for (int c = 0; c < NSIZE; ++c) {
      cap[c] = std::min<int64_t>(L.m, L.p / least[c]);
      total += cap[c];
    }
    netlist.alloc(&cx.alloc, (size_t)std::max<int64_t>(total, 1));
    netcount.alloc(&cx.alloc, NSIZE);
    HG_CUDA(cudaMemsetAsync(netcount.p, 0, netcount.bytes(), cx.stream));
    int2* at = netlist.p;
    for (int c = 0; c < NSIZE; ++c) {
      A.nets.list[c] = at;
      at += cap[c];
    }
    A.nets.count = netcount.p;
    if (P.T > BIG_NET && cap[NSIZE - 1] > 0) {
      A.nets.words = (n + 31) / 32;
      A.nets.bitmap_blocks = (int)std::max<int64_t>(
          1, std::min<int64_t>({cap[NSIZE - 1], (int64_t)cx.num_sms,
                                (256ll << 20) / ((int64_t)A.nets.words * 4)}));
      bitmaps.alloc(&cx.alloc, (size_t)A.nets.words * A.nets.bitmap_blocks);
      HG_CUDA(cudaMemsetAsync(bitmaps.p, 0, bitmaps.bytes(), cx.stream));
      A.nets.bitmaps = bitmaps.p;
    }
    k_net_lists<<<grid_for(L.m, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(L.eoff.p, L.m, P.T,
                                                                          A.nets, netcount.p);
    check_launch("net_lists");
    if (cx.launches) *cx.launches += 1;
  }

  RateArgs& R = A.R;
  R.rinfo = rinfo.p;
  R.adj = L.adj.p;
  R.rep = L.rep.p;
  R.comm = L.comm.p;
  DBuf<int32_t> pcomm;
  if (L.comm.p && records) {
    pcomm.alloc(&cx.alloc, (size_t)L.p);
    k_pin_comm<<<grid_for(L.p, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(rpins, L.p, L.comm.p,
                                                                         pcomm.p);
    check_launch("pin_comm");
    if (cx.launches) *cx.launches += 1;
    R.pcomm = pcomm.p;
  }
  R.imeta = imeta.p;
  R.lnode = lnode.p;
  R.split_base = split_base;
  R.cst = cst.p;
  R.c_max = P.c_max;
  R.n = n;
  R.clusters = clusters.p;
  R.target = target.p;
  R.gw = gw.p;
  R.gcnt = gcnt.p;
  R.mv = mv.p;
  R.touched = touched.p;
  R.stats = stats.p;
  R.status_word = cx.d_status;
  R.item_node = item_node.p;
  R.item_off = item_off.p;
  R.part_node = part_node.p;
  R.part_off = part_off.p;
  R.tab_off = tab_off.p;
  R.tab_cap = tab_cap.p;
  R.tab_dense = tab_dense.p;
  R.tkey = tkey.p;
  R.tused = tused.p;
  R.tnused = tnused.p;
  R.tval = tval.p;
  R.res_v = res_v.p;
  R.res_c = res_c.p;
  // direct-indexed levels: as many teams per block as tables fit
  R.dense_tw = !dense_block ? 0 : 4 * dense_bytes <= DENSE_SMEM ? 8
                               : 2 * dense_bytes <= DENSE_SMEM  ? 16 : 32;
  DBuf<SubPlan> dplan;
  dplan.alloc(&cx.alloc, (size_t)S);
  HG_CUDA(cudaMemcpyAsync(dplan.p, plan.data(), sizeof(SubPlan) * (size_t)S,
                          cudaMemcpyHostToDevice, cx.stream));
  A.plan = dplan.p;
  A.S = S;
  A.records = records;
  A.timing = cx.timing || cx.kernel_timing;
  A.words = words.p;
  A.slot_of = slot_of.p;
  A.slot_c = slot_c.p;
  A.slot_off = slot_off.p;
  A.slot_fill = slot_fill.p;
  A.glist = glist.p;
  A.c = L.c.p;
  A.rinfo = rinfo.p;
  A.p = records ? L.p : 0;
  A.barrier = reinterpret_cast<unsigned*>(stats.p + ST_TOTAL);
  // shared memory: the team tables, the level's direct-indexed tables and the
  // parts' tables take turns
  size_t smem = narrow ? TEAM_SMEM<uint32_t> : TEAM_SMEM<unsigned long long>;
  if (dense_block) smem = std::max(smem, dense_bytes * (size_t)(RUN_WARPS / R.dense_tw));
  if (any_parts) smem = std::max(smem, narrow ? part_bytes<uint32_t>() : part_bytes<unsigned long long>());
  if (hoff[nkeys] > 0) {
    cc.rating_launches += 1;
    run_subrounds(cx, A, narrow, L.graph, smem, hoff[nkeys], hoff[nkeys] - hoff[S],
                  (int64_t)hmax[2]);
  }
  // cluster weights for the contraction (valid at representatives)
  HG_CUDA(cudaMemcpy2DAsync(cw_out.p, sizeof(int32_t), cst.p, sizeof(int2), sizeof(int32_t),
                            (size_t)n, cudaMemcpyDeviceToDevice, cx.stream));
  unsigned long long hs[ST_TOTAL];
  const int32_t status = read_status(cx, hs, stats.p, sizeof(hs));
  if (status == DEV_HASH_FULL && any_parts) {
    HG_CUDA(cudaMemsetAsync(cx.d_status, 0, sizeof(int32_t), cx.stream));
    return false;
  }
  throw_status(cx, status);
  for (int c = 0; c < NCLASS; ++c) {
    const unsigned long long* h = hs + c * ST_WORDS;
    cc.rating_pin_visits += (int64_t)h[ST_PINS];
    cc.rating_incidences += (int64_t)h[ST_INCID];
    cc.rating_nodes += (int64_t)h[ST_NODES];
    cc.class_visits[c] += (int64_t)h[ST_PINS];
    const double ms = h[ST_NS] * 1e-6;
    if (cx.kernel_timing) {
      cc.ms_rating_kernels += ms;
      cc.class_ms[c] += ms;
    }
    if (cx.timing) cc.ms_rating += ms;
  }
  if (cx.timing) {
    cc.ms_approve += hs[ST_NS_APPROVE] * 1e-6;
    cc.ms_refresh += hs[ST_NS_REFRESH] * 1e-6;
  }
  return true;
}

}  // namespace

// The parts of a node hold its candidates by a fixed hash of their ids, so ids
// chosen to meet in one part overfill its table, which then drops candidates and
// says so.  Such a level is clustered once more with tables in global memory
// instead, which have a slot for every candidate.
void cluster_level(const Ctx& cx, Level& L, const CoarsenParams& P, CoarsenCounters& cc,
                   DBuf<int32_t>& cw_out) {
  if (!cluster_with_parts(cx, L, P, PART_MAX, cc, cw_out))
    cluster_with_parts(cx, L, P, 0, cc, cw_out);
}

}  // namespace hgk
