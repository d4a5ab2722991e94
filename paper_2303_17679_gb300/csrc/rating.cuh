// The rating of the clustering (Sec. 4.1): constants of the node classes, hash
// tables in shared memory and the walk over a node's candidate visits, shared
// by the preparation (coarsen.cu) and the sub-round kernel (cluster.cu).
#pragma once

#include "common.cuh"

namespace hgk {

constexpr int NCLASS = 5;
constexpr int SPLIT_CLASS = NCLASS - 1;
constexpr int32_t D_WARP = 256;
constexpr int32_t D_PAIR = 1024;
constexpr int32_t D_QUAD = 2048;
constexpr int32_t D_BLOCK = 4096;
constexpr int32_t TEAM_W = 65536;        // largest W of a node rated by one eight-warp team
constexpr int32_t DENSE_W = 32768;       // largest W of a direct-indexed block node
constexpr int32_t TEAM_RECORDS = 4096;   // most records of a node rated by one team or block
constexpr int32_t SPLIT_DENSE_MAX = 65536;
// Part blocks: see PartCfg (table slots and distinct candidates per part).  A node of
// more parts uses a global hash table, whose random sectors cost about fifteen times
// a visit that is only read.  Level of 118,445 nodes with 400 nets of 5000 pins, nine
// parts per node: 240 ms with global tables (a limit of 8), 95 ms in parts.
constexpr int32_t PART_MAX = 12;
constexpr int32_t EMPTY_KEY = -1;

constexpr int RUN_THREADS = 1024;        // the sub-round kernel: one block per SM
constexpr int RUN_WARPS = RUN_THREADS / 32;
// shared memory of the team tables (every team class fills it with its teams):
// 32-bit ratings fit 32 warps' worth of teams, 64-bit ones nearly that
template <typename VT>
constexpr size_t TEAM_SMEM = sizeof(VT) == 4 ? 160 * 1024 : 220 * 1024;
// a level whose value and used-list entries per node fit this is direct-indexed
constexpr size_t DENSE_SMEM = 200 * 1024;

// counters of a sub-round: movers, targets, contested targets and their list
// cursor, then the next node of every class
enum { CW_MOVES = 0, CW_TOUCHED = 1, CW_SLOTS = 2, CW_CURSOR = 3, CW_TICKET = 4, CW_WORDS = 12 };
// work counters per class, then phase times (ns)
enum { ST_PINS = 0, ST_INCID = 1, ST_NODES = 2, ST_NS = 3, ST_WORDS = 4 };
enum { ST_NS_APPROVE = NCLASS * ST_WORDS, ST_NS_REFRESH, ST_TOTAL };

// Of an incidence (u, e): the first pin position to visit, the number of pins
// to visit (the net's size, or u's range in it on grouped levels, when it is
// rated, 2 <= |e| <= T, else 0) and the Q20 term of the net (0 when not rated).
struct __align__(16) IncMeta {
  int32_t start, eff;
  unsigned long long r;
};

// Nodes and split work of one sub-round: ranges of the class-ordered node list,
// of the split plan's items and parts, and the first entry of its tables.
struct SubPlan {
  int32_t lo[NCLASS], hi[NCLASS];
  int32_t item_lo, item_hi, part_lo, part_hi;
  int32_t argmax;  // some split node needs the argmax pass
  int32_t pad;
  int64_t tab_lo;
};

struct RateArgs {
  const int2* rinfo;  // {deduplicated cluster, weight or INT32_MAX} per pin position
  // graph levels: visits come from the adjacency array, the cluster of a
  // neighbour from rep and its weight and status from cst
  const int2* adj;
  int32_t* rep;
  // community-aware coarsening (Sec. 4): comm[v] per node, pcomm[q] =
  // comm[pins[q]] per pin position (hypergraph levels); both NULL when off.
  // A cluster's members share its community, so the pin's community is the
  // community of the pin's cluster.
  const int32_t* comm;
  const int32_t* pcomm;
  // hypergraph levels: the metadata of every node's nets with pins to visit,
  // from ioff[u] on, so a walk reads one record per such net
  const IncMeta* imeta;
  // {u, ioff[u], rend[u], c(u)} of every listed node; the split nodes start
  // at split_base
  const int4* lnode;
  int32_t split_base;
  int2* cst;  // {cw, status}
  int32_t c_max, n;
  int32_t* clusters;
  int32_t* target;
  int32_t* gw;
  int32_t* gcnt;
  int32_t* mv;
  int32_t* touched;
  unsigned long long* stats;
  int32_t* status_word;
  // split plan
  const int32_t *item_node, *item_off, *part_node, *part_off;
  const int64_t *tab_off, *tab_cap;
  const int8_t* tab_dense;
  int32_t *tkey, *tused, *tnused;
  void *tval, *res_v;
  int32_t* res_c;
  int dense_tw;  // warps per team of a direct-indexed level (0: hash tables)
};

__device__ __forceinline__ uint32_t slot_hash(int32_t C) { return (uint32_t)C * 0x9E3779B1u; }

// ---------------------------------------------------- shared hash tables

// add() results besides the slot index of a new insertion
constexpr int32_t ADD_EXISTING = -1;
constexpr int32_t ADD_FULL = -2;

// 32-bit ratings: a key array and a value array (32-bit each).  An insertion
// claims the key with a 32-bit CAS and every visit adds its term with a
// 32-bit atomic add; both commute, so the sums do not depend on the order.
struct PackedHash {
  uint32_t* val;
  int32_t* key;
  uint32_t mask;
  static constexpr size_t BYTES_PER_SLOT = 8;
  __device__ __forceinline__ void init(uint32_t i) {
    key[i] = EMPTY_KEY;
    val[i] = 0;
  }
  // the slot index when C was inserted by this call, else ADD_EXISTING / ADD_FULL
  __device__ __forceinline__ int32_t add(int32_t C, uint32_t r) {
    uint32_t h = slot_hash(C) & mask;
    for (uint32_t probe = 0; probe <= mask; ++probe) {
      int32_t k = key[h];
      bool fresh = false;
      if (k == EMPTY_KEY) {
        const int32_t old = atomicCAS(&key[h], EMPTY_KEY, C);
        fresh = old == EMPTY_KEY;
        k = fresh ? C : old;
      }
      if (k == C) {
        atomicAdd(&val[h], r);
        return fresh ? (int32_t)h : ADD_EXISTING;
      }
      h = (h + 1) & mask;
    }
    return ADD_FULL;
  }
  // cluster and rating of slot i (C = -1 when empty); the slot is cleared
  __device__ __forceinline__ void take(uint32_t i, int32_t& C, uint32_t& v) {
    C = key[i];
    v = val[i];
    key[i] = EMPTY_KEY;
    val[i] = 0;
  }
};

// 64-bit ratings: separate key and value arrays.
struct WideHash {
  int32_t* key;
  unsigned long long* val;
  uint32_t mask;
  static constexpr size_t BYTES_PER_SLOT = 12;
  __device__ __forceinline__ void init(uint32_t i) {
    key[i] = EMPTY_KEY;
    val[i] = 0;
  }
  __device__ __forceinline__ int32_t add(int32_t C, unsigned long long r) {
    uint32_t h = slot_hash(C) & mask;
    for (uint32_t probe = 0; probe <= mask; ++probe) {
      int32_t k = key[h];
      bool fresh = false;
      if (k == EMPTY_KEY) {
        const int32_t old = atomicCAS(&key[h], EMPTY_KEY, C);
        fresh = old == EMPTY_KEY;
        k = fresh ? C : old;
      }
      if (k == C) {
        atomicAdd(&val[h], r);
        return fresh ? (int32_t)h : ADD_EXISTING;
      }
      h = (h + 1) & mask;
    }
    return ADD_FULL;
  }
  __device__ __forceinline__ void take(uint32_t i, int32_t& C, unsigned long long& v) {
    C = key[i];
    v = val[i];
    key[i] = EMPTY_KEY;
    val[i] = 0;
  }
};

// 32-bit ratings in a table of any size (not a power of two): the first slot
// is the high half of hash * slots, probing wraps at the end.  Used by the
// part blocks, whose table takes the whole shared-memory budget.
struct ModHash {
  uint32_t* val;
  int32_t* key;
  uint32_t slots;
  static constexpr size_t BYTES_PER_SLOT = 8;
  __device__ __forceinline__ void init(uint32_t i) {
    key[i] = EMPTY_KEY;
    val[i] = 0;
  }
  __device__ __forceinline__ int32_t add(int32_t C, uint32_t r) {
    uint32_t h = (uint32_t)(((uint64_t)slot_hash(C) * slots) >> 32);
    for (uint32_t probe = 0; probe < slots; ++probe) {
      int32_t k = key[h];
      bool fresh = false;
      if (k == EMPTY_KEY) {
        const int32_t old = atomicCAS(&key[h], EMPTY_KEY, C);
        fresh = old == EMPTY_KEY;
        k = fresh ? C : old;
      }
      if (k == C) {
        atomicAdd(&val[h], r);
        return fresh ? (int32_t)h : ADD_EXISTING;
      }
      h = h + 1 == slots ? 0 : h + 1;
    }
    return ADD_FULL;
  }
  __device__ __forceinline__ void take(uint32_t i, int32_t& C, uint32_t& v) {
    C = key[i];
    v = val[i];
    key[i] = EMPTY_KEY;
    val[i] = 0;
  }
};

template <typename VT> struct HashOf;
template <> struct HashOf<uint32_t> { using type = PackedHash; };
template <> struct HashOf<unsigned long long> { using type = WideHash; };

template <typename H>
__device__ __forceinline__ H make_hash(unsigned char* base, uint32_t slots);
template <>
__device__ __forceinline__ PackedHash make_hash<PackedHash>(unsigned char* base, uint32_t slots) {
  uint32_t* val = reinterpret_cast<uint32_t*>(base);
  return PackedHash{val, reinterpret_cast<int32_t*>(val + slots), slots - 1};
}
template <>
__device__ __forceinline__ ModHash make_hash<ModHash>(unsigned char* base, uint32_t slots) {
  uint32_t* val = reinterpret_cast<uint32_t*>(base);
  return ModHash{val, reinterpret_cast<int32_t*>(val + slots), slots};
}
template <>
__device__ __forceinline__ WideHash make_hash<WideHash>(unsigned char* base, uint32_t slots) {
  unsigned long long* val = reinterpret_cast<unsigned long long*>(base);
  return WideHash{reinterpret_cast<int32_t*>(val + slots), val, slots - 1};
}

// ------------------------------------------------------- the rating walk

// Visits per lane kept in flight (ILP, a template parameter of the walks):
// the record loads of ILP visits are issued before any of them is used.  The
// team kernels, whose time goes to the per-node steps, walk two at a time;
// the direct-indexed blocks, part blocks and split items, which walk the
// long visit lists of heavy nodes, four.
constexpr int TEAM_ILP = 2;
constexpr int DENSE_ILP = 4;
constexpr int PART_ILP = 4;
constexpr int SPLIT_ILP = 4;

// Adapts a per-visit adder f(C, r) to the batch interface of rate_group.
template <typename VT, int ILP, typename F>
struct EachVisit {
  F f;
  __device__ __forceinline__ void operator()(const int32_t (&C)[ILP], const VT (&rr)[ILP],
                                             const bool (&ok)[ILP]) const {
#pragma unroll
    for (int k = 0; k < ILP; ++k)
      if (ok[k]) f(C[k], rr[k]);
  }
};
template <typename VT, int ILP, typename F>
__device__ __forceinline__ EachVisit<VT, ILP, F> each_visit(F f) {
  return EachVisit<VT, ILP, F>{f};
}

// {cluster, weight word} of a batch of visits (-1 = no visit): on
// hypergraph levels q is a pin position and the record is rinfo[q]; on graph
// levels q is the neighbour node, whose cluster is rep[q] (a net of two pins
// needs no deduplication: u is a singleton, so rep[q] != u) and whose weight
// word is the cluster's weight, or INT32_MAX for an unclustered node of this
// sub-round.
// cmu >= 0: u's community; a visit in another community is dropped.
template <bool GRAPH, int ILP>
__device__ __forceinline__ void resolve_batch(const RateArgs& A, int s, const int32_t (&q)[ILP],
                                              int2 (&ri)[ILP], int32_t cmu) {
  if constexpr (!GRAPH) {
#pragma unroll
    for (int k = 0; k < ILP; ++k) ri[k] = q[k] >= 0 ? A.rinfo[q[k]] : make_int2(-1, 0);
    if (cmu >= 0) {
#pragma unroll
      for (int k = 0; k < ILP; ++k)
        if (ri[k].x >= 0 && A.pcomm[q[k]] != cmu) ri[k].x = -1;
    }
  } else {
    int32_t C[ILP];
#pragma unroll
    for (int k = 0; k < ILP; ++k)
      C[k] = q[k] >= 0 && (cmu < 0 || A.comm[q[k]] == cmu) ? A.rep[q[k]] : -1;
#pragma unroll
    for (int k = 0; k < ILP; ++k) {
      const int2 cs = C[k] >= 0 ? A.cst[C[k]] : make_int2(0, 0);
      ri[k] = make_int2(C[k], cs.y == s ? 0x7fffffff : cs.x);
    }
  }
}

// Filters a batch of visits (-1 = no visit) and hands it to `add`:
// admissible C is not u, not an unclustered node of this sub-round (weight
// word INT32_MAX), and fits c_max.
template <bool GRAPH, typename VT, int ILP, typename Add>
__device__ __forceinline__ void visit_filtered(const RateArgs& A, int s, int32_t u, int32_t cu,
                                               int32_t cmu, const int32_t (&q)[ILP],
                                               const VT (&rr)[ILP], Add& add) {
  int2 ri[ILP];
  resolve_batch<GRAPH, ILP>(A, s, q, ri, cmu);
  int32_t C[ILP];
  bool ok[ILP];
#pragma unroll
  for (int k = 0; k < ILP; ++k) {
    C[k] = ri[k].x;
    ok[k] = C[k] >= 0 && C[k] != u && (long long)ri[k].y + cu <= (long long)A.c_max;
  }
  add(C, rr, ok);
}

// Graph levels: the visits of incidences [lo, hi) of u are the other
// endpoints of its edges, each with the edge's term w(e) * 2^20 (the Q20 term
// of a two-pin net); chunk c of 32 * ILP incidences goes to warp c mod
// TW of the team.  Returns the visits in warp 0 (0 in the other warps).
template <typename VT, int ILP, typename Visit>
__device__ __forceinline__ int32_t graph_walk(const RateArgs& A, int32_t lo, int32_t hi, int wt,
                                              int TW, Visit& visit_batch) {
  constexpr int32_t CH = 32 * ILP;
  const int lane = lane_id();
  for (int32_t c0 = lo + CH * wt; c0 < hi; c0 += CH * TW) {
    int32_t q[ILP];
    VT rr[ILP];
#pragma unroll
    for (int k = 0; k < ILP; ++k) {
      const int32_t j = c0 + 32 * k + lane;
      if (j < hi) {
        const int2 a = A.adj[j];
        q[k] = a.x;
        rr[k] = (VT)((unsigned long long)(uint32_t)a.y << 20);
      } else {
        q[k] = -1;
        rr[k] = (VT)0;
      }
    }
    visit_batch(q, rr);
  }
  return wt == 0 ? hi - lo : 0;
}

// Adds one group of (up to) 32 consecutive records of u (one per lane)
// through `add`: the lanes walk the group's visits flattened, 32 * ILP of
// them at a time.  A visit's record is the number of records that end at or
// before it: one ballot counts those that end before the 32 visits at hand,
// and the ends that fall among them are collected as bits of one word (a
// warp-wide OR), so a lane counts the bits up to its own position.  Bound by
// instruction issue and L2 latency: a binary search through five dependent
// shuffles per visit, and one pass of every warp of a team over each net of
// 32 pins or more, cost more instructions than the visits themselves (1e6
// Zipf coarsening 76.8 -> 70.6 ms without them).  Every record holds a visit (k_node_work), so the ends are
// distinct.
// A team of TW warps (a power of two) shares the group: the chunks of
// 32 * ILP visits are numbered on from `run` (the chunks the team has walked
// before, for this node) and warp wt takes those whose number is wt modulo
// TW, so the team stays balanced across groups; `run` is advanced past the
// group's chunks.  Returns the group's pin visits in warp 0 (0 in the other
// warps, so the team counts each visit once).
// Per lane: first pin to visit, pins to visit (0: no record) and Q20 term of
// one incident net.
template <typename VT>
struct NetMeta {
  int32_t start, eff;
  VT r;
};

// The record at j (-1: none).
template <typename VT>
__device__ __forceinline__ NetMeta<VT> inc_meta(const RateArgs& A, int32_t j) {
  NetMeta<VT> m{0, 0, (VT)0};
  if (j >= 0) {
    const IncMeta x = A.imeta[j];
    m.start = x.start;
    m.eff = x.eff;
    m.r = (VT)x.r;
  }
  return m;
}

template <typename VT, int ILP, typename Visit>
__device__ __forceinline__ int32_t walk_group(const NetMeta<VT>& m, int wt, int TW, int32_t& run,
                                              Visit& visit_batch) {
  constexpr int32_t CH = 32 * ILP;
  const int lane = lane_id();
  const int32_t eff = m.eff;
  const VT r = m.r;
  const int32_t incl = warp_inclusive_scan(eff);
  const int32_t Z = __shfl_sync(FULL, incl, 31);
  const int32_t off = m.start - (incl - eff);  // visit f of this record is at off + f
  const unsigned upto = (2u << lane) - 1u;     // bits 0 .. lane
  const int32_t first = (wt - run) & (TW - 1);
  run += (Z + CH - 1) / CH;
  for (int32_t f0 = CH * first; f0 < Z; f0 += CH * TW) {
    int32_t q[ILP];
    VT rr[ILP];
#pragma unroll
    for (int k = 0; k < ILP; ++k) {
      const int32_t F = f0 + 32 * k;
      const int32_t d = incl - F;
      const int before = __popc(__ballot_sync(FULL, d <= 0));
      const unsigned ends = __reduce_or_sync(FULL, eff > 0 && d > 0 && d < 32 ? 1u << d : 0u);
      const int j = min(before + __popc(ends & upto), 31);
      const int32_t off_j = __shfl_sync(FULL, off, j);
      rr[k] = __shfl_sync(FULL, r, j);
      q[k] = F + lane < Z ? off_j + F + lane : -1;
    }
    visit_batch(q, rr);
  }
  return wt == 0 ? Z : 0;
}

// How a team of TW warps walks a node's records: a node of at least
// OWN_GROUPS groups of 32 records per warp gives each warp its own groups (a
// warp then loads and scans only those); nodes of fewer records share every
// group chunk by chunk, which balances them whatever their net sizes.
constexpr int32_t OWN_GROUPS = 4;
struct TeamWalk {
  int32_t first, step;
  int wt, TW;
};
template <bool GRAPH>
__device__ __forceinline__ TeamWalk team_walk(int32_t beg, int32_t end, int wt, int TW) {
  if (TW > 1 && !GRAPH && end - beg >= OWN_GROUPS * 32 * TW)
    return TeamWalk{beg + 32 * wt, 32 * TW, 0, 1};
  return TeamWalk{beg, 32, wt, TW};
}

template <bool GRAPH, typename VT, int ILP, typename Visit>
__device__ __forceinline__ int32_t rate_group_raw(const RateArgs& A, int32_t g0, int32_t end,
                                                  int wt, int TW, int32_t& run, Visit& visit_batch) {
  if constexpr (GRAPH) {
    return graph_walk<VT, ILP>(A, g0, min(g0 + 32, end), wt, TW, visit_batch);
  } else {
    const int32_t j = g0 + lane_id();
    return walk_group<VT, ILP>(inc_meta<VT>(A, j < end ? j : -1), wt, TW, run, visit_batch);
  }
}

// The groups g0 = first, first + step, ... (< end) of I(u), walked as by
// rate_group_raw with the load of the next group's net metadata issued
// before the current group is walked (graph levels: one walk over all of it).
template <bool GRAPH, typename VT, int ILP, typename Visit>
__device__ __forceinline__ int64_t rate_groups_raw(const RateArgs& A, int32_t first, int32_t end,
                                                   int32_t step, int wt, int TW, int32_t& run,
                                                   Visit& visit_batch) {
  if (first >= end) return 0;
  if constexpr (GRAPH) {
    return graph_walk<VT, ILP>(A, first, end, wt, TW, visit_batch);
  } else {
    const int lane = lane_id();
    int64_t visits = 0;
    int32_t g = first;
    NetMeta<VT> m = inc_meta<VT>(A, g + lane < end ? g + lane : -1);
    while (g < end) {
      const int32_t gn = g + step;
      const NetMeta<VT> mn = inc_meta<VT>(A, gn + lane < end ? gn + lane : -1);
      visits += walk_group<VT, ILP>(m, wt, TW, run, visit_batch);
      m = mn;
      g = gn;
    }
    return visits;
  }
}

// rate_group_raw / rate_groups_raw with the admissibility filter of
// visit_filtered in front of `add`.
template <bool GRAPH, typename VT, int ILP, typename Add>
__device__ __forceinline__ int32_t rate_group(const RateArgs& A, int s, int32_t u, int32_t cu,
                                              int32_t g0, int32_t end, int wt, int TW,
                                              int32_t& run, Add add) {
  const int32_t cmu = A.comm ? A.comm[u] : -1;
  auto visit = [&](const int32_t(&q)[ILP], const VT(&rr)[ILP]) HG_INLINE {
    visit_filtered<GRAPH, VT, ILP>(A, s, u, cu, cmu, q, rr, add);
  };
  return rate_group_raw<GRAPH, VT, ILP>(A, g0, end, wt, TW, run, visit);
}

template <bool GRAPH, typename VT, int ILP, typename Add>
__device__ __forceinline__ int64_t rate_groups(const RateArgs& A, int s, int32_t u, int32_t cu,
                                               const TeamWalk& tw, int32_t end, Add add) {
  const int32_t cmu = A.comm ? A.comm[u] : -1;
  auto visit = [&](const int32_t(&q)[ILP], const VT(&rr)[ILP]) HG_INLINE {
    visit_filtered<GRAPH, VT, ILP>(A, s, u, cu, cmu, q, rr, add);
  };
  int32_t run = 0;
  return rate_groups_raw<GRAPH, VT, ILP>(A, tw.first, end, tw.step, tw.wt, tw.TW, run, visit);
}

template <typename VT>
__device__ __forceinline__ void better(VT& bv, int32_t& bc, VT v, int32_t C) {
  if (C >= 0 && (bc < 0 || v > bv || (v == bv && C < bc))) {
    bv = v;
    bc = C;
  }
}

template <typename VT>
__device__ __forceinline__ void warp_argmax(VT& best_v, int32_t& best_c) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    const VT ov = __shfl_xor_sync(FULL, best_v, d);
    const int32_t oc = __shfl_xor_sync(FULL, best_c, d);
    better(best_v, best_c, ov, oc);
  }
}

// Shared memory of one team: the hash slots, then a list of the slots the
// current node inserted (capacity slots / 2: a class's distinct bound).
template <typename H>
__host__ __device__ constexpr size_t team_bytes(uint32_t slots) {
  return (size_t)slots * H::BYTES_PER_SLOT + (size_t)(slots / 2) * sizeof(int32_t);
}

// Table of a part block: SLOTS shared slots holding at most D distinct
// candidates per part (60 % load), and a list of the inserted slots of
// capacity CAP (more insertions: the whole table is scanned).  32-bit
// ratings take the whole shared-memory budget (22,528 slots, so fewer nodes
// need more than one part and every part re-reads the node's visits);
// 64-bit ratings 16,384 slots.
template <typename VT> struct PartCfg {
  using Hash = WideHash;
  static constexpr uint32_t SLOTS = 16384, CAP = 2048;
  static constexpr int32_t D = 9830;
};
template <> struct PartCfg<uint32_t> {
  using Hash = ModHash;
  static constexpr uint32_t SLOTS = 22528, CAP = 10240;
  static constexpr int32_t D = 13516;
};
template <typename VT>
constexpr size_t part_bytes() {
  return (size_t)PartCfg<VT>::SLOTS * PartCfg<VT>::Hash::BYTES_PER_SLOT +
         (size_t)PartCfg<VT>::CAP * 4;
}

__device__ __forceinline__ int32_t part_of(int32_t C, int32_t P) {
  return (int32_t)(((uint64_t)((uint32_t)C * 0x85EBCA77u) * (uint32_t)P) >> 32);
}

// Rated nets by size, for the upkeep of the cluster words: nets of up to 4, 8,
// 16 and 32 pins (a group of that many lanes each), up to BIG_NET (a warp and
// its shared memory), larger ones (a block and a node bitmap).
constexpr int NSIZE = 6;
constexpr int BIG_NET = 1024;

__host__ __device__ inline int net_size_class(int32_t sz) {
  return sz <= 4 ? 0 : sz <= 8 ? 1 : sz <= 16 ? 2 : sz <= 32 ? 3 : sz <= BIG_NET ? 4 : 5;
}

struct NetLists {
  int2* list[NSIZE];     // {first pin position, pins} of every rated net of a class
  const int32_t* count;  // NSIZE
  unsigned* bitmaps;     // one of `words` words per block of the largest class
  int32_t words, bitmap_blocks;
};

// Everything the sub-round kernel of a level works on.
struct ClusterArgs {
  RateArgs R;
  const SubPlan* plan;
  int S;
  bool records;  // hypergraph level with pins
  bool cluster;  // barrier of one thread-block cluster, else of the whole grid
  bool timing;
  int32_t* words;
  // approval
  int32_t *slot_of, *slot_c, *slot_off, *slot_fill, *glist;
  const int32_t* c;
  // cluster words
  int2* rinfo;
  int64_t p;
  NetLists nets;
  unsigned* barrier;  // two words (grid_sync)
};

// Runs the S sub-rounds of a level (cluster.cu).  `listed` nodes, `heavy` of
// them above the warp class, with at most `total_visits` pin visits (for the
// launch geometry).
void run_subrounds(const Ctx& cx, ClusterArgs A, bool narrow, bool graph, size_t smem,
                   int64_t listed, int64_t heavy, int64_t total_visits);

}  // namespace hgk
