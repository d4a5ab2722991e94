// Deterministic label propagation (Sec. 11 "Deterministic Label Propagation
// Refinement" with the gain of Sec. 6): one persistent kernel per call.
//
// A pass is S sub-rounds; a sub-round is three phases, each over the whole
// grid and each ended by a barrier of all blocks:
//   best moves   every listed node picks its best positive-gain target (a11);
//   selection    per block pair the moves are ordered by (gain desc, id asc)
//                and the last feasible prefix pair is chosen (a12);
//   application  Phi, the net records and Pi of the chosen moves (a13; graph
//                levels have no pin counts: the selection writes Pi).
// What bounds it: a level runs 80 sub-rounds of three dependent steps
// whatever its size, and all but the largest levels do little work in each, so
// the time is the chain of L2 accesses and of the boundaries between steps.
// As launches of a captured graph a sub-round cost two parallel best-move
// kernels, a selection and an application (18 us at n = 10,000, k = 2; 24 us
// on coarse levels of 5M pins, k = 8), plus capture, graph update and a host
// wait per pass.  Blocks that stay resident pay a barrier instead: 0.35-0.4 us
// in one thread-block cluster of up to 16 blocks (small levels), 1.4 us over
// the whole chip (cooperative launch), and no host interaction at all.
// Measured (GB300, whole call, before -> after): n = 10,000, k = 2 1.45 ->
// 0.69 ms; n = 500,009 Zipf, k = 16 2.79 -> 1.82 ms; all levels of the 1e6 Zipf
// V-cycle, k = 8 24.4 -> 17.9 ms; of the 4e6 large-net V-cycle, k = 64 87 -> 44 ms.
//
// State that changes during the kernel (Pi, Phi, records, lists, counters) is
// read with ld.cg or atomics, never through L1; the structure (ioff, inets,
// adj, node weights) is constant and read through the read-only path.
#include <algorithm>
#include <climits>

#include "gain.cuh"
#include "gridsync.cuh"

namespace hgk {

namespace {

constexpr int LP_THREADS = 512;
constexpr int LP_WARPS = LP_THREADS / 32;
constexpr int MAX_SUBROUNDS = 256;
// incidences of one warp item of a node above the lane-group class
constexpr int32_t ITEM_INC_MIN = 128, ITEM_INC_MAX = 1024;
constexpr int MACC_STRIDE = HG_MAX_K + 4; // sums of a node split over several items: k blocks, bw
constexpr int RANK_MAX = 1024;            // directions of up to this many moves: rank sort
constexpr int MAX_PAIRS = HG_MAX_K * (HG_MAX_K - 1) / 2;

// ------------------------------------------------ packed net records (a11)

// Phi stays the authority over the net records (gain.cuh): the application
// changes a pin count with an atomic that returns the old count, and flips the
// record's bits for the transitions it caused (0 <-> 1 toggles Lambda and ones,
// 1 <-> 2 toggles ones); the flips commute, so the records equal their
// definition whatever the order of the moves.

// ------------------------------------------------------------- arguments

// Counters of one sub-round (two sets, used in turn).
enum SubroundWord { SW_OVERFLOW = 0, SW_ITEMS = 1, SW_WORDS = 4 };
// Results and totals of a call.
enum LpResultWord {
  LR_MOVES = 0, LR_MOVED_INCID = 1, LR_OBJECTIVE = 2, LR_PASSES = 3,
  LR_NS_GAIN = 4, LR_NS_SELECT = 5, LR_NS_APPLY = 6, LR_NS_OBJECTIVE = 7, LR_WORDS = 8
};

struct LpArgs {
  // structure of the level
  const int32_t *ioff, *inets, *c, *eoff, *pins, *w;
  const int2* adj;
  int32_t n, m;
  // partition state
  int32_t* part;
  int32_t* phi;
  int4* rec;
  long long* bw;           // block weights at the start of the call
  // parameters
  int k, S, level, max_passes, block_deg, item_inc;
  uint64_t seed;
  long long lmax;
  bool cluster;            // barrier of one thread-block cluster, else of the whole grid
  bool timing;             // accumulate phase times
  // lists: items of every (sub-round, class) of the pass
  int4* items;             // {node, first incidence, end, accumulator slot or -1}
  int32_t *cnt, *fill;     // 2 S each
  int32_t* mslots;         // accumulator slots given out in the pass
  int32_t *macc, *mtick;   // sums and finished incidences per slot
  // moves of a sub-round: keys of the first dcap moves of every direction,
  // the others in the overflow list
  unsigned long long* dkeys;
  int32_t dcap;
  int32_t* dcnt;           // 2 x k k
  unsigned long long* ovf_key;
  int32_t* ovf_dir;
  int32_t* words;          // 2 x SW_WORDS
  long long* dbw;          // 2 x k: block-weight changes of a sub-round
  int4* ap;                // {node, first incidence, end, from | to << 8 | first item << 16}
  // directions too long for shared memory
  int sel_cap;
  unsigned long long* gkeys;
  int32_t* gpre;
  unsigned* barrier;       // two words (grid_sync)
  unsigned long long* res;
  int32_t* status;
};

// Sort key: gain descending, node id ascending (gains are < 2^31).
__device__ __forceinline__ unsigned long long sel_key(int32_t g, int32_t u) {
  return ((unsigned long long)(uint32_t)(0x7fffffff - g) << 32) | (unsigned)u;
}

__device__ __forceinline__ bool lp_sync(const LpArgs& A, unsigned& gen) {
  return grid_sync(A.cluster, A.barrier, A.status, gen);
}

// ------------------------------------------------- sub-round lists

// Every node with incident nets is listed by key = 2 * sub-round + class:
// class 0 (at most block_deg incident nets) has one item per node, taken by a
// lane group; class 1 one item per item_inc incidences, taken by a warp.  The
// block counts (scatter == false) or writes (true) its tiles of nodes; slots
// within a tile come from shared counters, one global atomic per tile and key.
__device__ __forceinline__ void list_nodes(const LpArgs& A, int pass, bool scatter,
                                           const int32_t* s_off, int32_t* s_hist,
                                           int32_t* s_base) {
  const int keys = 2 * A.S;
  for (int i = threadIdx.x; i < keys; i += LP_THREADS) s_hist[i] = 0;
  __syncthreads();
  const int64_t stride = (int64_t)gridDim.x * LP_THREADS;
  for (int64_t u0 = (int64_t)blockIdx.x * LP_THREADS; u0 < A.n; u0 += stride) {
    const int64_t u = u0 + threadIdx.x;
    int key = -1, slot = 0;
    int32_t beg = 0, end = 0, items = 0;
    if (u < A.n) {
      beg = __ldg(A.ioff + u);
      end = __ldg(A.ioff + u + 1);
      if (end > beg) {
        const bool wide_node = end - beg > A.block_deg;
        items = wide_node ? (end - beg + A.item_inc - 1) / A.item_inc : 1;
        key = 2 * subround_of_node_lp(A.seed, A.level, pass, (int)u, A.S) + (wide_node ? 1 : 0);
        slot = atomicAdd(&s_hist[key], items);
      }
    }
    if (!scatter) continue;
    __syncthreads();
    for (int i = threadIdx.x; i < keys; i += LP_THREADS) {
      s_base[i] = s_hist[i] ? atomicAdd(&A.fill[i], s_hist[i]) : 0;
      s_hist[i] = 0;
    }
    __syncthreads();
    if (key >= 0) {
      int4* out = A.items + s_off[key] + s_base[key] + slot;
      if (items == 1) {
        out[0] = make_int4((int)u, beg, end, -1);
      } else {
        const int32_t ms = atomicAdd(A.mslots, 1);
        for (int32_t i = 0; i < items; ++i)
          out[i] = make_int4((int)u, beg + i * A.item_inc,
                             (int)min((int64_t)end, beg + (int64_t)(i + 1) * A.item_inc), ms);
      }
    }
    __syncthreads();
  }
  if (!scatter) {
    __syncthreads();
    for (int i = threadIdx.x; i < keys; i += LP_THREADS)
      if (s_hist[i]) atomicAdd(&A.cnt[i], s_hist[i]);
  }
}

// Exclusive prefix sums of the 2 S counts into s_off[0 .. 2 S] (warp 0).
__device__ __forceinline__ void list_offsets(const LpArgs& A, int32_t* s_off) {
  const int keys = 2 * A.S;
  if (warp_in_block() == 0) {
    int32_t carry = 0;
    for (int i0 = 0; i0 < keys; i0 += 32) {
      const int i = i0 + lane_id();
      const int32_t x = i < keys ? __ldcg(A.cnt + i) : 0;
      const int32_t incl = warp_inclusive_scan(x);
      if (i < keys) s_off[i] = carry + incl - x;
      carry += __shfl_sync(FULL, incl, 31);
    }
    if (lane_id() == 0) s_off[keys] = carry;
  }
  __syncthreads();
}

// ------------------------------------------------- best moves (a11)

// Best candidate so far as one comparable word: gain descending, block id
// ascending; 0 when no gain is positive.
__device__ __forceinline__ void consider(unsigned long long& best, int32_t g, int t, int from,
                                         int k) {
  if (g > 0 && t != from && t < k) {
    const unsigned long long x = ((unsigned long long)(uint32_t)g << 8) | (unsigned)(255 - t);
    if (x > best) best = x;
  }
}

__device__ __forceinline__ void emit_move(const LpArgs& A, int par, int32_t u, int from,
                                          unsigned long long best) {
  if (!best) return;
  const int t = 255 - (int)(best & 0xff);
  const unsigned long long key = sel_key((int32_t)(best >> 8), u);
  const int d = from * A.k + t;
  const int32_t pos = atomicAdd(&A.dcnt[par * A.k * A.k + d], 1);
  if (pos < A.dcap) {
    A.dkeys[(size_t)d * A.dcap + pos] = key;
  } else {
    const int32_t o = atomicAdd(&A.words[par * SW_WORDS + SW_OVERFLOW], 1);
    A.ovf_key[o] = key;
    A.ovf_dir[o] = d;
  }
}

// Maximum over the W lanes of the caller's group (W a power of two); the whole
// warp calls it.
template <int W>
__device__ __forceinline__ unsigned long long group_max(unsigned long long x) {
#pragma unroll
  for (int d = W / 2; d > 0; d >>= 1) {
    const unsigned long long y = __shfl_xor_sync(FULL, x, d);
    x = y > x ? y : x;
  }
  return x;
}

// Edges j and j + share of a node whose edges end at `end` ({-1, 0} past it).
__device__ __forceinline__ void edge_pair(const LpArgs& A, int32_t j, int32_t share, int32_t end,
                                          int2& a0, int2& a1) {
  a0 = j < end ? __ldg(A.adj + j) : make_int2(-1, 0);
  a1 = j + share < end ? __ldg(A.adj + j + share) : make_int2(-1, 0);
}

// Class-0 nodes by groups of SUB_G lanes, one node (or none: an empty item) per
// group: NG nodes' load chains per warp in flight (nodes of a few nets leave
// most lanes of a warp idle and cost it a full chain of dependent loads each).
// The groups stay in step: trip counts are the warp's largest and all shuffles
// name the whole warp, because groups that diverge run one after the other
// (16 us instead of 5 for the best moves of 488 nodes on 512 groups).
template <bool GRAPH, int K, int H>
__device__ __forceinline__ void gain_groups(const LpArgs& A, int par, const int4 it, int sub) {
  using L = TeamLane<SUB_G, H>;
  const L lane(sub);
  const int32_t u = it.x;
  const bool on = it.z > it.y;
  const int from = on ? __ldcg(A.part + u) : 0, from_h = from - 32 * lane.half;
  Gain<GRAPH, K, H> g;
  g.init();
  // two incidences per lane in flight, on graph levels the edges of the next
  // step loaded ahead
  const int32_t steps = __reduce_max_sync(FULL, it.z - it.y);
  int2 a0 = make_int2(-1, 0), a1 = a0;
  if (GRAPH) edge_pair(A, it.y + lane.i, L::SHARE, it.z, a0, a1);
  for (int32_t x = lane.i; x - lane.i < steps; x += 2 * L::SHARE) {
    const int32_t j0 = it.y + x, j1 = j0 + L::SHARE;
    const bool v0 = j0 < it.z, v1 = j1 < it.z;
    if (GRAPH) {
      const int t0 = v0 ? __ldcg(A.part + a0.x) : 0, t1 = v1 ? __ldcg(A.part + a1.x) : 0;
      const int32_t w0 = a0.y, w1 = a1.y;
      edge_pair(A, j1 + L::SHARE, L::SHARE, it.z, a0, a1);
      g.add_edge(w0, t0 - 32 * lane.half, from_h);
      g.add_edge(w1, t1 - 32 * lane.half, from_h);
    } else {
      const int32_t e0 = v0 ? __ldg(A.inets + j0) : 0, e1 = v1 ? __ldg(A.inets + j1) : 0;
      NetRec r0{0, 0, 0}, r1{0, 0, 0};
      if (v0) r0 = load_rec(A.rec, (int64_t)H * e0 + lane.half);
      if (v1) r1 = load_rec(A.rec, (int64_t)H * e1 + lane.half);
      g.add(r0, from_h);
      g.add(r1, from_h);
    }
  }
  const int32_t bw = group_sum<SUB_G>(g.bw);
  const int b0 = 32 * lane.half + reduce_scatter<L::SHARE, K>(lane.i, g.acc);
  constexpr int OWN = K / L::SHARE > 0 ? K / L::SHARE : 1;
  unsigned long long best = 0;
#pragma unroll
  for (int i = 0; i < OWN; ++i) consider(best, bw + g.acc[i], b0 + i, from, A.k);
  best = group_max<SUB_G>(best);
  if (sub == 0 && on) emit_move(A, par, u, from, best);
  __syncwarp();
}

// The sums of a class-1 item: the node's best move, or, for one of several items,
// into the node's accumulators; the item that finishes last takes the maximum
// and clears them for the next pass.
template <bool GRAPH, int K, int H>
__device__ __forceinline__ void finish_item(const LpArgs& A, int par, const int4 it, int from,
                                            Gain<GRAPH, K, H>& g) {
  using L = TeamLane<32, H>;
  const int lane = lane_id();
  const L tl(lane);
  const int32_t u = it.x, beg = it.y, end = it.z, slot = it.w;
  int32_t bw = group_sum<32>(g.bw);
  const int b0 = 32 * tl.half + reduce_scatter<L::SHARE, K>(tl.i, g.acc);
  constexpr int OWN = K / L::SHARE > 0 ? K / L::SHARE : 1;
  unsigned long long best = 0;
  if (slot < 0) {
#pragma unroll
    for (int i = 0; i < OWN; ++i) consider(best, bw + g.acc[i], b0 + i, from, A.k);
  } else {
    int32_t* macc = A.macc + (int64_t)slot * MACC_STRIDE;
    constexpr int SAME = L::SHARE / K > 1 ? L::SHARE / K : 1;  // lanes holding the same block
    if (tl.i % SAME == 0) {
#pragma unroll
      for (int i = 0; i < OWN; ++i)
        if (g.acc[i]) atomicAdd(&macc[b0 + i], g.acc[i]);
    }
    if (lane == 0 && bw) atomicAdd(&macc[HG_MAX_K], bw);
    __threadfence();
    __syncwarp();
    int last = 0;
    if (lane == 0) {
      const int32_t deg = __ldg(A.ioff + u + 1) - __ldg(A.ioff + u);
      last = atomicAdd(&A.mtick[slot], end - beg) + (end - beg) == deg;
    }
    if (!__shfl_sync(FULL, last, 0)) return;
    __threadfence();
    bw = __ldcg(macc + HG_MAX_K);
    for (int t = lane; t < A.k; t += 32) consider(best, bw + __ldcg(macc + t), t, from, A.k);
    __syncwarp();
    for (int t = lane; t < MACC_STRIDE; t += 32) macc[t] = 0;
    if (lane == 0) A.mtick[slot] = 0;
  }
  best = group_max<32>(best);
  if (lane == 0) emit_move(A, par, u, from, best);
}

// A class-1 item by a warp: four consecutive incidences per lane and step (one
// 16-byte load of their net ids).
template <bool GRAPH, int K, int H>
__device__ __forceinline__ void gain_item(const LpArgs& A, int par, const int4 it) {
  using L = TeamLane<32, H>;
  const int lane = lane_id();
  const L tl(lane);
  const int32_t beg = it.y, end = it.z;
  const int from = __ldcg(A.part + it.x), from_h = from - 32 * tl.half;
  Gain<GRAPH, K, H> g;
  g.init();
  if (GRAPH) {
    int2 a0, a1;
    edge_pair(A, beg + tl.i, L::SHARE, end, a0, a1);
    for (int32_t j = beg + tl.i; j < end; j += 2 * L::SHARE) {
      const int t0 = __ldcg(A.part + a0.x), t1 = a1.x >= 0 ? __ldcg(A.part + a1.x) : 0;
      const int32_t w0 = a0.y, w1 = a1.y;
      edge_pair(A, j + 2 * L::SHARE, L::SHARE, end, a0, a1);
      g.add_edge(w0, t0 - 32 * tl.half, from_h);
      g.add_edge(w1, t1 - 32 * tl.half, from_h);
    }
  } else {
    // chunks start at a multiple of 4; positions outside [beg, end) are skipped
    for (int32_t c0 = beg & ~3; c0 < end; c0 += 4 * L::SHARE) {
      const int32_t j0 = c0 + 4 * tl.i;
      int32_t e[4];
      if (j0 >= beg && j0 + 4 <= end) {
        const int4 v = __ldg(reinterpret_cast<const int4*>(A.inets + j0));
        e[0] = v.x;
        e[1] = v.y;
        e[2] = v.z;
        e[3] = v.w;
      } else {
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const int32_t j = j0 + x;
          e[x] = j >= beg && j < end ? __ldg(A.inets + j) : -1;
        }
      }
      NetRec r[4];
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        r[x] = NetRec{0, 0, 0};
        if (e[x] >= 0) r[x] = load_rec(A.rec, (int64_t)H * e[x] + tl.half);
      }
#pragma unroll
      for (int x = 0; x < 4; ++x) g.add(r[x], from_h);
    }
  }
  finish_item<GRAPH, K, H>(A, par, it, from, g);
}

// The same for k > 32 (records in two halves).  Most incidences of the nodes of
// this class are of nets that have pins in every block: those count the same for
// every target, so they go into bw, nets inside the node's own block into no
// target at all, and only the others (one in eight on the coarse levels of a
// large-net input) are queued and added block by block, 16 at a time, each by a
// lane of either half.  The gathers of the records bound it, at one request
// each: one lane reads both halves with one load.  Measured (GB300, sub-round of
// 16,400 nodes and 1.96M incidences, k = 64): best moves 40 -> 19 us (36 us with
// a load per half).
__device__ __forceinline__ void gain_item_wide(const LpArgs& A, int par, const int4 it,
                                               int4* queue) {
  const int lane = lane_id();
  const TeamLane<32, 2> tl(lane);
  const unsigned below = (1u << lane) - 1u;
  const int32_t beg = it.y, end = it.z;
  const int from = __ldcg(A.part + it.x);
  const unsigned long long own = 1ull << from, full = ~0ull >> (64 - A.k);
  Gain<false, 32, 2> g;
  g.init();
  int held = 0;
  auto drain = [&](int count) {
    held -= count;
    NetRec r{0, 0, 0};
    if (tl.i < count) {
      const int4 q = queue[held + tl.i];
      r.w = q.x;
      r.lam = (unsigned)(tl.half ? q.z : q.y);
    }
    g.add_targets(r);
    __syncwarp();
  };
  // two records in flight per lane, the net ids of the next two loaded ahead
  int32_t e[2];
  auto nets = [&](int32_t c0) {
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const int32_t j = c0 + 32 * x + lane;
      e[x] = j < end ? __ldg(A.inets + j) : -1;
    }
  };
  nets(beg);
  for (int32_t c0 = beg; c0 < end; c0 += 64) {
    WideRec r[2];
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      r[x] = WideRec{0, 0, 0};
      if (e[x] >= 0) r[x] = load_wide(A.rec, e[x]);
    }
    nets(c0 + 64);
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const bool all = r[x].lam == full;
      if (all) g.bw += r[x].w;
      if (!(r[x].ones & own)) g.bw -= r[x].w;
      const bool mid = !all && (r[x].lam & ~own) != 0;
      const unsigned live = __ballot_sync(FULL, mid);
      if (mid)
        queue[held + __popc(live & below)] = make_int4(
            r[x].w, (int32_t)(uint32_t)r[x].lam, (int32_t)(uint32_t)(r[x].lam >> 32), 0);
      __syncwarp();
      held += __popc(live);
      while (held >= 16) drain(16);
    }
  }
  if (held > 0) drain(held);
  finish_item<false, 32, 2>(A, par, it, from, g);
}

// Class-0 nodes for k > 32, before gain_groups (32-bit sums: gain.cuh): no gain of
// u exceeds
//   w(nets where u is the only pin of its block) - w(nets inside its block)
// (a net outside every other block counts against every target), so only the
// nodes where that is positive are kept, in the block's list.  Eight lanes per
// node and LP_BOUND nodes per group in flight; the sums for 64 targets, most of
// a node's work, are left to the nodes that remain (18 % of the nodes of the
// finest level of a 4e6-node large-net V-cycle, 4 % on its coarse levels).
// Measured (GB300, that finest level, 250,000 nodes and 2.4M incidences per
// sub-round): best moves 81 -> 46 us.  For k <= 32 the sums cost less than a
// second walk (63 to 99 % of the nodes of a 21,000-node V-cycle at k = 32 remain).
constexpr int LP_BOUND = 2;
constexpr int LP_KEPT = 2048;  // nodes kept by a block at a time
constexpr int LP_QUEUE = 48;   // records queued by a warp: 15 left over and 32 new ones

__device__ __forceinline__ void bound_groups(const LpArgs& A, const int4 (&it)[LP_BOUND], int sub,
                                             int4* kept, int* nkept) {
  unsigned long long own[LP_BOUND];
  int32_t bound[LP_BOUND];
  int32_t most = 0;
#pragma unroll
  for (int y = 0; y < LP_BOUND; ++y) {
    own[y] = it[y].z > it[y].y ? 1ull << __ldcg(A.part + it[y].x) : 0;
    bound[y] = 0;
    most = max(most, it[y].z - it[y].y);
  }
  most = __reduce_max_sync(FULL, most);
  for (int32_t x = sub; x - sub < most; x += 2 * SUB_G) {
    int32_t e[LP_BOUND][2];
#pragma unroll
    for (int y = 0; y < LP_BOUND; ++y)
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        const int32_t j = it[y].y + x + z * SUB_G;
        e[y][z] = j < it[y].z ? __ldg(A.inets + j) : -1;
      }
    WideRec r[LP_BOUND][2];
#pragma unroll
    for (int y = 0; y < LP_BOUND; ++y)
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        r[y][z] = WideRec{0, 0, 0};
        if (e[y][z] >= 0) r[y][z] = load_wide(A.rec, e[y][z]);
      }
#pragma unroll
    for (int y = 0; y < LP_BOUND; ++y)
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        if (r[y][z].ones & own[y]) bound[y] += r[y][z].w;
        if (r[y][z].lam == own[y]) bound[y] -= r[y][z].w;
      }
  }
#pragma unroll
  for (int y = 0; y < LP_BOUND; ++y) {
    const int32_t sum = group_sum<SUB_G>(bound[y]);
    if (sub == 0 && sum > 0) kept[atomicAdd(nkept, 1)] = it[y];
  }
}

// ------------------------------------------------- pair selection (a12)

// The pair with index `pair` in the order (0,1), (0,2), ..., (k-2,k-1).
__device__ __forceinline__ void decode_pair(int pair, int k, int& a, int& b) {
  const float q = (float)(2 * k - 1);
  a = (int)((q - sqrtf(q * q - 8.0f * (float)pair)) * 0.5f);
  auto start = [&](int x) { return x * (2 * k - 1 - x) / 2; };
  while (a > 0 && start(a) > pair) --a;
  while (start(a + 1) <= pair) ++a;
  b = a + 1 + pair - start(a);
}

// Work items of the application: one per 32 incident nets of a moved node
// (hubs would serialise the warp that selected them).  The node writes its
// items at `slot`.
__device__ __forceinline__ void write_items(const LpArgs& A, int32_t slot, int32_t u, int32_t beg,
                                            int32_t end, int from, int to) {
  for (int32_t j = beg, i = 0; j < end; j += 32, ++i)
    A.ap[slot + i] = make_int4(u, j, min(end, j + 32), from | (to << 8) | (i == 0 ? 1 << 16 : 0));
}

// Moves taken by the lanes of a warp: Pi of graph levels, application items
// of hypergraph levels, and the incidences moved.  All lanes call it.
template <bool GRAPH>
__device__ __forceinline__ void take_moves(const LpArgs& A, int par, bool on, int32_t u, int from,
                                           int to, int32_t& incid) {
  int32_t beg = 0, end = 0;
  if (on) {
    beg = __ldg(A.ioff + u);
    end = __ldg(A.ioff + u + 1);
    incid += end - beg;
  }
  if (GRAPH) {
    if (on) A.part[u] = to;
    return;
  }
  const int32_t items = (end - beg + 31) / 32;
  const int32_t incl = warp_inclusive_scan(items);
  int32_t base = 0;
  if (lane_id() == 31 && incl)
    base = atomicAdd(&A.words[par * SW_WORDS + SW_ITEMS], incl);
  base = __shfl_sync(FULL, base, 31);
  if (on) write_items(A, base + incl - items, u, beg, end, from, to);
}

__device__ __forceinline__ void count_moves(const LpArgs& A, int par, int a, int b, int32_t moves,
                                            int32_t incid, int32_t delta) {
  // delta = weight moved a -> b minus weight moved b -> a
  atomic_add_i64(&A.dbw[par * A.k + a], -(long long)delta);
  atomic_add_i64(&A.dbw[par * A.k + b], (long long)delta);
  atomicAdd(&A.res[LR_MOVES], (unsigned long long)moves);
  atomicAdd(&A.res[LR_MOVED_INCID], (unsigned long long)incid);
}

// Sorts one 64-bit key per lane ascending within the first P lanes.
__device__ __forceinline__ unsigned long long warp_sort(unsigned long long x, int P) {
  const int lane = lane_id();
  for (int kk = 2; kk <= P; kk <<= 1)
    for (int j = kk >> 1; j > 0; j >>= 1) {
      const unsigned long long y = __shfl_xor_sync(FULL, x, j);
      const bool keep_min = ((lane & kk) == 0) == ((lane & j) == 0);
      x = keep_min == (x < y) ? x : y;
    }
  return x;
}

// A pair whose two directions have at most 32 moves each, by one warp: keys
// sorted in registers, weight prefixes by warp scans.  With A[i] and B[j] the
// weights of the first i and j moves, the merge path takes A's step i before
// B's step j when A[i] <= B[j]; lane l evaluates the states after A's step l
// and after B's step l, and the last feasible state wins.  (Bound by the
// latency of about 150 dependent instructions; the block form below needs a
// barrier per sorting stage.)
template <bool GRAPH>
__device__ __forceinline__ void select_warp(const LpArgs& A, int par, int a, int b, int na, int nb,
                                            const long long* s_slack) {
  const int lane = lane_id();
  const unsigned long long* da = A.dkeys + (size_t)(a * A.k + b) * A.dcap;
  const unsigned long long* db = A.dkeys + (size_t)(b * A.k + a) * A.dcap;
  unsigned long long ka = lane < na ? __ldcg(da + lane) : ~0ull;
  unsigned long long kb = lane < nb ? __ldcg(db + lane) : ~0ull;
  const int big = max(na, nb);
  const int P = big <= 1 ? 1 : 2 << (31 - __clz(big - 1));
  ka = warp_sort(ka, P);
  kb = warp_sort(kb, P);
  const int32_t ua = (int32_t)(uint32_t)ka, ub = (int32_t)(uint32_t)kb;
  const int32_t ca = lane < na ? __ldg(A.c + ua) : 0, cb = lane < nb ? __ldg(A.c + ub) : 0;
  const int32_t ia = warp_inclusive_scan(ca), ib = warp_inclusive_scan(cb);
  const int32_t xa = ia - ca, xb = ib - cb;  // A[lane], B[lane]
  int nB = 0, nA = 0;  // B steps before A's step `lane`, A steps before B's step `lane`
#pragma unroll
  for (int st = 32; st > 0; st >>= 1) {
    const int32_t pb = __shfl_sync(FULL, xb, (nB + st - 1) & 31);
    const int32_t pa = __shfl_sync(FULL, xa, (nA + st - 1) & 31);
    if (nB + st <= nb && pb < xa) nB += st;
    if (nA + st <= na && pa <= xb) nA += st;
  }
  const int32_t bB = __shfl_sync(FULL, ib, (nB - 1) & 31), bA = __shfl_sync(FULL, ia, (nA - 1) & 31);
  const long long lo = -s_slack[a], hi = s_slack[b];
  const long long x1 = (long long)ia - (nB ? bB : 0), x2 = (long long)(nA ? bA : 0) - ib;
  unsigned v = 0;
  if (lane < na && lo <= x1 && x1 <= hi)
    v = ((unsigned)(lane + nB + 1) << 16) | ((unsigned)(lane + 1) << 8) | (unsigned)nB;
  if (lane < nb && lo <= x2 && x2 <= hi)
    v = max(v, ((unsigned)(lane + nA + 1) << 16) | ((unsigned)nA << 8) | (unsigned)(lane + 1));
  v = __reduce_max_sync(FULL, v);
  const int ta = (int)((v >> 8) & 0xff), tb = (int)(v & 0xff);
  if (ta + tb == 0) return;
  const int32_t wa = __shfl_sync(FULL, ia, (ta - 1) & 31), wb = __shfl_sync(FULL, ib, (tb - 1) & 31);
  int32_t incid = 0;
  if (ta) take_moves<GRAPH>(A, par, lane < ta, ua, a, b, incid);
  if (tb) take_moves<GRAPH>(A, par, lane < tb, ub, b, a, incid);
  incid = warp_sum(incid);
  if (lane == 0) count_moves(A, par, a, b, ta + tb, incid, (ta ? wa : 0) - (tb ? wb : 0));
}

// Shared memory of the selection: keys and weight prefixes of both
// directions (cap moves each; the upper half of the keys takes the ranked
// copy of up to RANK_MAX <= cap / 2 keys).
__host__ __device__ constexpr size_t select_bytes(int cap) {
  return (size_t)2 * cap * 8 + (size_t)2 * (cap + 1) * 4;
}

// Ranks of up to RANK_MAX distinct keys by counting the smaller ones: every
// thread compares one key with all others (broadcast reads, two keys per
// load), one barrier instead of one per stage of a sorting network.
__device__ __forceinline__ void rank_sort2(const unsigned long long* a, int na,
                                           unsigned long long* oa, const unsigned long long* b,
                                           int nb, unsigned long long* ob) {
  for (int x = threadIdx.x; x < na + nb; x += LP_THREADS) {
    const unsigned long long* in = x < na ? a : b;
    const int i = x < na ? x : x - na, cnt = x < na ? na : nb;
    const unsigned long long mine = in[i];
    int rank = 0, j = 0;
    for (; j + 2 <= cnt; j += 2) {
      const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(in + j);
      rank += (v.x < mine) + (v.y < mine);
    }
    if (j < cnt) rank += in[j] < mine;
    (x < na ? oa : ob)[rank] = mine;
  }
  __syncthreads();
}

// Bitonic sorts of the two directions of a pair (Pa and Pb powers of two) by
// the block, stage by stage together.
__device__ void bitonic_sort2(unsigned long long* a, int Pa, unsigned long long* b, int Pb,
                              unsigned* barrier) {
  const int P = Pa > Pb ? Pa : Pb;
  for (int kk = 2; kk <= P; kk <<= 1) {
    for (int j = kk >> 1; j > 0; j >>= 1) {
      for (int64_t y = threadIdx.x; y < (int64_t)Pa + Pb; y += LP_THREADS) {
        beat_along(barrier, y);
        unsigned long long* buf = y < Pa ? a : b;
        const int i = (int)(y < Pa ? y : y - Pa);
        const int n = y < Pa ? Pa : Pb;
        if (kk > n) continue;
        const int ixj = i ^ j;
        if (ixj > i) {
          const unsigned long long u = buf[i], v = buf[ixj];
          const bool up = (i & kk) == 0;
          if ((u > v) == up) {
            buf[i] = v;
            buf[ixj] = u;
          }
        }
      }
      __syncthreads();
    }
  }
}

// Weight prefixes of both directions from one block-wide scan over the
// concatenation of their sorted moves: A[x] = weight of the first x moves
// a -> b (x = 0..na), B[x] likewise for b -> a.  A node is in one direction at most,
// so all of them together weigh c(V) < 2^31 at most (hg_create) and 32 bits do;
// their differences against the slack are taken in 64.
__device__ void weight_prefix2(const unsigned long long* ka, int na, const unsigned long long* kb,
                               int nb, const int32_t* __restrict__ c, int32_t* A, int32_t* B,
                               unsigned* barrier) {
  __shared__ int32_t s_sum[LP_WARPS];
  __shared__ int32_t s_total_a;
  const int cnt = na + nb;
  int32_t carry = 0;
  if (threadIdx.x == 0) {
    A[0] = 0;
    B[0] = 0;
    s_total_a = 0;
  }
  __syncthreads();
  for (int base = 0; base < cnt; base += LP_THREADS) {
    const int x = base + threadIdx.x;
    beat_along(barrier, x);
    int32_t v = 0;
    if (x < na) v = __ldg(c + (int32_t)(uint32_t)ka[x]);
    else if (x < cnt) v = __ldg(c + (int32_t)(uint32_t)kb[x - na]);
    const int32_t y = warp_inclusive_scan(v);
    if (lane_id() == 31) s_sum[warp_in_block()] = y;
    __syncthreads();
    int32_t before = 0, total = 0;
#pragma unroll
    for (int i = 0; i < LP_WARPS; ++i) {
      if (i < warp_in_block()) before += s_sum[i];
      total += s_sum[i];
    }
    const int32_t incl = carry + before + y;
    carry += total;
    if (x < na) A[x + 1] = incl;
    if (x == na - 1) s_total_a = incl;
    __syncthreads();
    if (x >= na && x < cnt) B[x - na + 1] = incl - s_total_a;
  }
  __syncthreads();
}

// A pair with more moves, by the whole block.
template <bool GRAPH>
__device__ void select_block(const LpArgs& P, int par, int a, int b, int na, int nb,
                             const long long* s_slack, unsigned char* smem) {
  __shared__ int s_red[2];
  const int cap = P.sel_cap, k = P.k;
  const int dab = a * k + b, dba = b * k + a;
  unsigned long long* s_keys0 = reinterpret_cast<unsigned long long*>(smem);
  unsigned long long* s_keys1 = s_keys0 + cap;
  unsigned long long* s_out0 = s_keys0 + cap / 2;
  unsigned long long* s_out1 = s_keys1 + cap / 2;
  int32_t* s_pre0 = reinterpret_cast<int32_t*>(s_keys1 + cap);
  int32_t* s_pre1 = s_pre0 + cap + 1;
  auto pow2 = [](int x) {
    int p = 1;
    while (p < x) p <<= 1;
    return p;
  };
  const int Pa = pow2(na), Pb = pow2(nb);
  const int32_t* dcnt = P.dcnt + par * k * k;
  if (threadIdx.x < 2) s_red[threadIdx.x] = 0;
  __syncthreads();
  int oa = 0, ob = 0;
  if (Pa > cap || Pb > cap) {
    // a region of 2 * count keys at twice the direction's offset
    int sa = 0, sb = 0;
    for (int d = threadIdx.x; d < k * k; d += LP_THREADS) {
      const int cd = __ldcg(dcnt + d);
      if (d < dab) sa += cd;
      if (d < dba) sb += cd;
    }
    sa = warp_sum(sa);
    sb = warp_sum(sb);
    if (lane_id() == 0) {
      atomicAdd(&s_red[0], sa);
      atomicAdd(&s_red[1], sb);
    }
    __syncthreads();
    oa = s_red[0];
    ob = s_red[1];
    __syncthreads();
    if (threadIdx.x < 2) s_red[threadIdx.x] = 0;
    __syncthreads();
  }
  unsigned long long* ka = Pa <= cap ? s_keys0 : P.gkeys + 2 * (int64_t)oa;
  unsigned long long* kb = Pb <= cap ? s_keys1 : P.gkeys + 2 * (int64_t)ob;
  int32_t* A = na <= cap ? s_pre0 : P.gpre + (int64_t)oa + dab;
  int32_t* B = nb <= cap ? s_pre1 : P.gpre + (int64_t)ob + dba;
  // the directions' key lists, then their moves in the overflow list
  const unsigned long long* da = P.dkeys + (size_t)dab * P.dcap;
  const unsigned long long* db = P.dkeys + (size_t)dba * P.dcap;
  const int la = min(na, P.dcap), lb = min(nb, P.dcap);
  for (int i = threadIdx.x; i < la; i += LP_THREADS) ka[i] = __ldcg(da + i);
  for (int i = threadIdx.x; i < lb; i += LP_THREADS) kb[i] = __ldcg(db + i);
  if (na > la || nb > lb) {
    const int32_t no = __ldcg(P.words + par * SW_WORDS + SW_OVERFLOW);
    for (int32_t i = threadIdx.x; i < no; i += LP_THREADS) {
      beat_along(P.barrier, i);
      const int32_t d = __ldcg(P.ovf_dir + i);
      if (d == dab) ka[la + atomicAdd(&s_red[0], 1)] = __ldcg(P.ovf_key + i);
      else if (d == dba) kb[lb + atomicAdd(&s_red[1], 1)] = __ldcg(P.ovf_key + i);
    }
  }
  if (max(na, nb) <= RANK_MAX) {
    __syncthreads();
    rank_sort2(ka, na, s_out0, kb, nb, s_out1);
    ka = s_out0;
    kb = s_out1;
  } else {
    for (int i = na + threadIdx.x; i < Pa; i += LP_THREADS) ka[i] = ~0ull;
    for (int i = nb + threadIdx.x; i < Pb; i += LP_THREADS) kb[i] = ~0ull;
    __syncthreads();
    bitonic_sort2(ka, Pa, kb, Pb, P.barrier);
  }
  weight_prefix2(ka, na, kb, nb, P.c, A, B, P.barrier);
  if (threadIdx.x == 0) s_red[0] = 0;
  __syncthreads();
  // diagonal r: i(r) = number of A steps among the first r
  auto steps = [&](int r) {
    int lo = r - nb > 0 ? r - nb : 0, hi = r < na ? r : na;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (A[mid] <= B[r - 1 - mid]) lo = mid + 1;
      else hi = mid;
    }
    return lo;
  };
  const long long lo = -s_slack[a], hi = s_slack[b];
  int best = 0;
  for (int r = threadIdx.x; r <= na + nb; r += LP_THREADS) {
    beat_along(P.barrier, r);
    const int i = steps(r);
    const long long x = (long long)A[i] - B[r - i];
    if (lo <= x && x <= hi) best = r > best ? r : best;
  }
  best = warp_max(best);
  if (lane_id() == 0) atomicMax(&s_red[0], best);
  __syncthreads();
  const int r = s_red[0];
  const int ta = steps(r), tb = r - ta;
  int32_t incid = 0;
  for (int i0 = 32 * warp_in_block(); i0 < ta + tb; i0 += LP_THREADS) {
    const int i = i0 + lane_id();
    beat_along(P.barrier, i);
    const bool from_a = i < ta;
    int32_t u = 0;
    if (i < ta + tb) u = (int32_t)(uint32_t)(from_a ? ka[i] : kb[i - ta]);
    take_moves<GRAPH>(P, par, i < ta + tb, u, from_a ? a : b, from_a ? b : a, incid);
  }
  incid = warp_sum(incid);
  if (lane_id() == 0 && incid) atomicAdd(&P.res[LR_MOVED_INCID], (unsigned long long)incid);
  if (threadIdx.x == 0 && r > 0) count_moves(P, par, a, b, r, 0, A[ta] - B[tb]);
  __syncthreads();
}

// ------------------------------------------------------- apply (a13)

// One warp per work item: for its <= 32 nets e: Phi(e, s) -= 1,
// Phi(e, t) += 1, and the flips of the record's bits for the transitions
// (Algorithm 3's updates); the atomic xor flips commute, so the final masks
// equal {i : Phi(e, i) > 0} and {i : Phi(e, i) = 1} whatever the order of the
// moves.  The node's first item sets Pi[u] = t.
template <int H>
__device__ __forceinline__ void apply_item(const LpArgs& A, const int4 it) {
  const int s = it.w & 0xff, t = (it.w >> 8) & 0xff;
  const int32_t j = it.y + lane_id();
  if (j < it.z) {
    const int32_t e = __ldg(A.inets + j);
    const int32_t os = atomicSub(&A.phi[(int64_t)e * A.k + s], 1);  // s: os -> os - 1
    const int32_t ot = atomicAdd(&A.phi[(int64_t)e * A.k + t], 1);  // t: ot -> ot + 1
    const unsigned bs = 1u << (s & 31), bt = 1u << (t & 31);
    int4* rs = A.rec + (int64_t)H * e + (H == 1 ? 0 : s >> 5);
    int4* rt = A.rec + (int64_t)H * e + (H == 1 ? 0 : t >> 5);
    if (os == 1 || os == 2) atomicXor(reinterpret_cast<unsigned*>(&rs->y), bs);
    if (os == 1) atomicXor(reinterpret_cast<unsigned*>(&rs->z), bs);
    if (ot == 0 || ot == 1) atomicXor(reinterpret_cast<unsigned*>(&rt->y), bt);
    if (ot == 0) atomicXor(reinterpret_cast<unsigned*>(&rt->z), bt);
  }
  if ((it.w >> 16) && lane_id() == 0) A.part[it.x] = t;
}

// ------------------------------------------------------------ the kernel

template <bool GRAPH, int K, int H>
__global__ void __launch_bounds__(LP_THREADS, 2) k_lp_run(const __grid_constant__ LpArgs A) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int32_t s_off[2 * MAX_SUBROUNDS + 1];
  __shared__ int32_t s_hist[2 * MAX_SUBROUNDS], s_base[2 * MAX_SUBROUNDS];
  __shared__ long long s_bw[HG_MAX_K], s_slack[HG_MAX_K];
  __shared__ uint16_t s_big[MAX_PAIRS];
  __shared__ int s_nbig, s_kept;
  __shared__ int64_t s_obj[32];
  const int lane = lane_id(), wv = warp_in_block();
  // consecutive work items go to different blocks: few items spread over the chip
  const int gw = wv * gridDim.x + blockIdx.x, NW = gridDim.x * LP_WARPS;
  const int grp = lane / SUB_G, sub = lane % SUB_G;
  const int k = A.k, kk = k * k;
  for (int i = threadIdx.x; i < k; i += LP_THREADS) s_bw[i] = __ldcg(A.bw + i);
  __syncthreads();
  unsigned gen = 0;
  unsigned long long moves_before = 0;
  unsigned long long t_gain = 0, t_select = 0, t_apply = 0, t0 = 0;
  const bool clock = A.timing && blockIdx.x == 0 && threadIdx.x == 0;
  int par = 0, passes = 0;
  for (int pass = 0; pass < A.max_passes; ++pass) {
    if (clock) t0 = now_ns();
    list_nodes(A, pass, false, s_off, s_hist, s_base);
    if (!lp_sync(A, gen)) return;
    list_offsets(A, s_off);
    list_nodes(A, pass, true, s_off, s_hist, s_base);
    if (!lp_sync(A, gen)) return;
    for (int s = 0; s < A.S; ++s, par ^= 1) {
      // ---- best moves.  The other set of counters (last read before the
      // barrier that ended the previous sub-round) is cleared for the next
      // one; the block weights take the previous sub-round's changes.
      for (int i = threadIdx.x; i < k; i += LP_THREADS) {
        const long long w = s_bw[i] + __ldcg(A.dbw + (par ^ 1) * k + i);
        s_bw[i] = w;
        s_slack[i] = (A.lmax - w > 0 ? A.lmax - w : 0) / (k - 1);
      }
      if (threadIdx.x == 0) s_nbig = 0;
      for (int i = blockIdx.x * LP_THREADS + threadIdx.x; i < kk; i += gridDim.x * LP_THREADS)
        A.dcnt[(par ^ 1) * kk + i] = 0;
      if (blockIdx.x == 0 && threadIdx.x < SW_WORDS) A.words[(par ^ 1) * SW_WORDS + threadIdx.x] = 0;
      if constexpr (!GRAPH && H == 2) {
        int4* kept = reinterpret_cast<int4*>(smem);
        int4* queue = kept + LP_KEPT + wv * LP_QUEUE;
        for (int32_t i = s_off[2 * s + 1] + gw; i < s_off[2 * s + 2]; i += NW)
          gain_item_wide(A, par, __ldcg(A.items + i), queue);
        // in chunks of at most LP_KEPT nodes per block
        constexpr int ROUNDS = LP_KEPT / (LP_WARPS * NG);
        const int32_t hi = s_off[2 * s + 1];
        for (int64_t c0 = s_off[2 * s]; c0 < hi; c0 += (int64_t)ROUNDS * NG * NW) {
          __syncthreads();
          if (threadIdx.x == 0) s_kept = 0;
          __syncthreads();
          for (int r = 0; r < ROUNDS; r += LP_BOUND) {
            int64_t i = c0 + (int64_t)r * NG * NW + (NW - 1 - gw);
            if (i >= hi) break;  // uniform in the warp
            i += grp * NW;
            int4 it[LP_BOUND];
#pragma unroll
            for (int y = 0; y < LP_BOUND; ++y, i += (int64_t)NG * NW)
              it[y] = i < hi ? __ldcg(A.items + i) : make_int4(0, 0, 0, -1);
            bound_groups(A, it, sub, kept, &s_kept);
          }
          __syncthreads();
          for (int x = wv * NG; x < s_kept; x += LP_WARPS * NG)
            gain_groups<GRAPH, K, H>(
                A, par, x + grp < s_kept ? kept[x + grp] : make_int4(0, 0, 0, -1), sub);
        }
        __syncthreads();
      } else {
        for (int32_t i = s_off[2 * s + 1] + gw; i < s_off[2 * s + 2]; i += NW)
          gain_item<GRAPH, K, H>(A, par, __ldcg(A.items + i));
        for (int32_t i0 = s_off[2 * s] + (NW - 1 - gw); i0 < s_off[2 * s + 1]; i0 += NG * NW) {
          const int32_t i = i0 + grp * NW;
          gain_groups<GRAPH, K, H>(
              A, par, i < s_off[2 * s + 1] ? __ldcg(A.items + i) : make_int4(0, 0, 0, -1), sub);
        }
      }
      __syncwarp();
      if (!lp_sync(A, gen)) return;
      if (clock) {
        const unsigned long long t = now_ns();
        t_gain += t - t0;
        t0 = t;
      }
      // ---- selection: warp w takes the pairs w, w + NW, ... (a lane loads
      // the counts of each); pairs with a long direction are left to the block
      for (int i = blockIdx.x * LP_THREADS + threadIdx.x; i < k; i += gridDim.x * LP_THREADS)
        A.dbw[(par ^ 1) * k + i] = 0;
      if (s == 0) {  // the lists are built: clear their counters for the next pass
        for (int i = blockIdx.x * LP_THREADS + threadIdx.x; i < 2 * A.S;
             i += gridDim.x * LP_THREADS) {
          A.cnt[i] = 0;
          A.fill[i] = 0;
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) *A.mslots = 0;
      }
      const int npairs = k * (k - 1) / 2;
      for (int p0 = gw; p0 < npairs; p0 += 32 * NW) {
        const int pair = p0 + lane * NW;
        int a = 0, b = 0, na = 0, nb = 0;
        if (pair < npairs) {
          decode_pair(pair, k, a, b);
          na = __ldcg(A.dcnt + par * kk + a * k + b);
          nb = __ldcg(A.dcnt + par * kk + b * k + a);
        }
        const bool small = na <= 32 && nb <= 32 && na <= A.dcap && nb <= A.dcap;
        if (!small) s_big[atomicAdd(&s_nbig, 1)] = (uint16_t)pair;
        unsigned todo = __ballot_sync(FULL, small && na + nb > 0);
        while (todo) {
          const int l = __ffs(todo) - 1;
          todo &= todo - 1;
          select_warp<GRAPH>(A, par, __shfl_sync(FULL, a, l), __shfl_sync(FULL, b, l),
                             __shfl_sync(FULL, na, l), __shfl_sync(FULL, nb, l), s_slack);
        }
      }
      __syncthreads();
      for (int x = 0; x < s_nbig; ++x) {
        int a, b;
        decode_pair(s_big[x], k, a, b);
        const int na = __ldcg(A.dcnt + par * kk + a * k + b);
        const int nb = __ldcg(A.dcnt + par * kk + b * k + a);
        select_block<GRAPH>(A, par, a, b, na, nb, s_slack, smem);
      }
      if (!lp_sync(A, gen)) return;
      if (clock) {
        const unsigned long long t = now_ns();
        t_select += t - t0;
        t0 = t;
      }
      // ---- application
      if (!GRAPH) {
        const int32_t na = __ldcg(A.words + par * SW_WORDS + SW_ITEMS);
        for (int32_t i = gw; i < na; i += NW) apply_item<H>(A, __ldcg(A.ap + i));
        if (!lp_sync(A, gen)) return;
        if (clock) {
          const unsigned long long t = now_ns();
          t_apply += t - t0;
          t0 = t;
        }
      }
    }
    passes = pass + 1;
    const unsigned long long moves = __ldcg(A.res + LR_MOVES);
    if (moves == moves_before) break;
    moves_before = moves;
  }
  // ---- objective (a14)
  if (clock) t0 = now_ns();
  int64_t f = 0;
  const int64_t stride = (int64_t)gridDim.x * LP_THREADS;
  for (int64_t e = (int64_t)blockIdx.x * LP_THREADS + threadIdx.x; e < A.m; e += stride) {
    if (GRAPH) {
      const int32_t b = __ldg(A.eoff + e);
      if (__ldcg(A.part + __ldg(A.pins + b)) != __ldcg(A.part + __ldg(A.pins + b + 1)))
        f += __ldg(A.w + e);
    } else {
      const NetRec r = load_rec(A.rec, (int64_t)H * e);
      int l = __popc(r.lam);
      if (H == 2) l += __popc(load_rec(A.rec, (int64_t)H * e + 1).lam);
      if (l > 1) f += (int64_t)(l - 1) * r.w;
    }
  }
  f = block_sum(f, s_obj);
  if (threadIdx.x == 0 && f) atomicAdd(&A.res[LR_OBJECTIVE], (unsigned long long)f);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    A.res[LR_PASSES] = (unsigned long long)passes;
    A.res[LR_NS_GAIN] = t_gain;
    A.res[LR_NS_SELECT] = t_select;
    A.res[LR_NS_APPLY] = t_apply;
    if (clock) A.res[LR_NS_OBJECTIVE] = now_ns() - t0;
  }
}

using LpKernel = void (*)(LpArgs);

LpKernel lp_kernel(bool graph, int k) {
  if (graph) {
    if (k <= 8) return k_lp_run<true, 8, 1>;
    if (k <= 16) return k_lp_run<true, 16, 1>;
    if (k <= 32) return k_lp_run<true, 32, 1>;
    return k_lp_run<true, 32, 2>;
  }
  if (k <= 8) return k_lp_run<false, 8, 1>;
  if (k <= 16) return k_lp_run<false, 16, 1>;
  if (k <= 32) return k_lp_run<false, 32, 1>;
  return k_lp_run<false, 32, 2>;
}

// Moves per direction sorted in shared memory (more go through global
// memory): pairs hold fewer moves as k grows, and two blocks share an SM.
int sel_cap_for(int k) { return k <= 8 ? 4096 : 2048; }
static_assert((LP_KEPT + LP_WARPS * LP_QUEUE) * sizeof(int4) <= select_bytes(2048),
              "the lists of the best moves take the selection's buffers");
static_assert(2 * RANK_MAX <= 2048, "the ranked keys take the upper half of the key buffers");

size_t lp_smem_bytes(int k) { return select_bytes(sel_cap_for(k)); }

constexpr int CLUSTER_MAX = 16;

}  // namespace

LPResult lp_refine_level(const Ctx& cx, const Level& L, int level_index, int k, int eps_ppm,
                         int max_passes, int S, uint64_t seed, int64_t total_node_weight,
                         int lp_block_deg, int32_t* part, RefineCounters& rc) {
  LPResult res;
  PinState st;
  {
    EventTimer tm(cx, &rc.ms_phi);
    build_pin_state(cx, L, k, part, st, L.graph ? PinMasks::none : PinMasks::records);
  }
  const int64_t per_block = (total_node_weight + k - 1) / k;
  const int kk = k * k;
  const int32_t n = L.n;
  const int64_t nodes_sr = ((int64_t)n + S - 1) / S, inc_sr = (L.p + S - 1) / S;

  // keys kept per direction: four times the mean of an even spread
  int32_t dcap = 64;
  while (dcap < RANK_MAX && (int64_t)dcap * kk < 4 * nodes_sr) dcap <<= 1;
  if (k <= 16) dcap = RANK_MAX;

  // items of nodes above the lane-group class: about one per warp of the chip
  int32_t item_inc = ITEM_INC_MIN;
  while (item_inc < ITEM_INC_MAX && inc_sr > (int64_t)item_inc * cx.num_sms * 2 * LP_WARPS)
    item_inc <<= 1;

  const size_t ncap = (size_t)n + 1;
  const size_t nitems = ncap + (size_t)(L.p / item_inc) + 1;
  const size_t nmulti = (size_t)std::min<int64_t>(n, L.p / item_inc) + 1;
  const size_t acap = L.graph ? 1 : ncap + (size_t)(L.p / 32) + 1;
  DBuf<int4> items, ap;
  DBuf<unsigned long long> dkeys, ovf_key, gkeys;
  DBuf<int32_t> ovf_dir, gpre;
  items.alloc(&cx.alloc, nitems);
  ap.alloc(&cx.alloc, acap);
  dkeys.alloc(&cx.alloc, (size_t)kk * dcap);
  ovf_key.alloc(&cx.alloc, ncap);
  ovf_dir.alloc(&cx.alloc, ncap);
  gkeys.alloc(&cx.alloc, 2 * ncap + 2);
  gpre.alloc(&cx.alloc, ncap + (size_t)kk + 2);
  // everything that must start at zero, in one piece: 64-bit words first
  const size_t z64 = LR_WORDS + 2 * (size_t)k;
  const size_t z32 = 4 * (size_t)S + 2 * (size_t)kk + 2 * SW_WORDS + 4 +
                     nmulti * (MACC_STRIDE + 1);
  DBuf<unsigned long long> zero;
  zero.alloc(&cx.alloc, z64 + (z32 + 1) / 2);
  HG_CUDA(cudaMemsetAsync(zero.p, 0, zero.bytes(), cx.stream));
  int32_t* z = reinterpret_cast<int32_t*>(zero.p + z64);

  LpArgs A{};
  A.ioff = L.ioff.p;
  A.inets = L.inets.p;
  A.c = L.c.p;
  A.eoff = L.eoff.p;
  A.pins = L.pins.p;
  A.w = L.w.p;
  A.adj = L.adj.p;
  A.n = n;
  A.m = L.m;
  A.part = part;
  A.phi = st.phi.p;
  A.rec = st.rec.p;
  A.bw = st.bw.p;
  A.k = k;
  A.S = S;
  A.level = level_index;
  A.max_passes = max_passes;
  A.block_deg = lp_block_deg;
  A.item_inc = item_inc;
  A.seed = seed;
  A.lmax = (long long)(per_block * (1000000 + (int64_t)eps_ppm) / 1000000);
  A.timing = cx.timing || cx.kernel_timing;
  A.items = items.p;
  A.res = zero.p;
  A.dbw = reinterpret_cast<long long*>(zero.p + LR_WORDS);
  A.cnt = z;
  A.fill = A.cnt + 2 * S;
  A.dcnt = A.fill + 2 * S;
  A.words = A.dcnt + 2 * kk;
  A.mslots = A.words + 2 * SW_WORDS;
  A.barrier = reinterpret_cast<unsigned*>(A.mslots + 1);
  A.mtick = A.mslots + 4;
  A.macc = A.mtick + nmulti;
  A.dkeys = dkeys.p;
  A.dcap = dcap;
  A.ovf_key = ovf_key.p;
  A.ovf_dir = ovf_dir.p;
  A.ap = ap.p;
  A.sel_cap = sel_cap_for(k);
  A.gkeys = gkeys.p;
  A.gpre = gpre.p;
  A.status = cx.d_status;

  // Blocks.  Small levels run as one cluster (its barrier is three times faster
  // than the grid's): those with at most a lane group per node and two
  // incidences per thread in 16 blocks; with more (eight per thread) the cluster
  // takes 14 us for the best moves of 58,000 incidences, the grid 6.  Of the
  // cluster sizes the largest that has work for every block is best: a sub-round
  // of 92 nodes takes 7.5 us in one block, 6 us in 16.  Larger levels spread over
  // the chip, two blocks per SM when there is work for them.  A call that
  // shares the GPU with others (inflight.cuh) takes no more blocks than its work
  // fills, a lane group per node and eight incidences per thread,
  // and at most half the chip (see run_subrounds in cluster.cu).
  const LpKernel kernel = lp_kernel(L.graph, k);
  const size_t bytes = lp_smem_bytes(k);
  prepare_kernel(cx, kernel, bytes, true);
  const bool shared = cx.shares_gpu();
  auto blocks_for = [&](int64_t nodes, int64_t inc) {
    return std::max<int64_t>({nodes_sr / nodes + 1, inc_sr / inc + 1, (int64_t)k * (k - 1) / 256 + 1});
  };
  const int64_t need = blocks_for(LP_WARPS * NG, LP_THREADS * 8);
  int blocks = 1;
  A.cluster = (shared ? need : blocks_for(LP_WARPS * NG, LP_THREADS * 2)) <= CLUSTER_MAX;
  if (A.cluster) {
    const int64_t want = shared ? need : blocks_for(LP_WARPS * NG / 8, LP_THREADS / 4);
    while (blocks < want && blocks < CLUSTER_MAX) blocks <<= 1;
  } else {
    int per_sm = 0;
    HG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_sm, reinterpret_cast<const void*>(kernel), LP_THREADS, bytes));
    if (per_sm < 1) throw HgError(HG_ERR_CUDA, "label propagation does not fit an SM");
    const int64_t most = (int64_t)cx.num_sms * std::min(per_sm, shared ? 1 : 2);
    blocks = (int)(shared ? std::min(need, most) : need <= cx.num_sms ? cx.num_sms : most);
  }
  launch_persistent(cx, kernel, blocks, LP_THREADS, bytes, A.cluster, A);
  unsigned long long hres[LR_WORDS];
  read_back(cx, hres, A.res, sizeof(hres));
  res.passes = (int)hres[LR_PASSES];
  res.moves = (int64_t)hres[LR_MOVES];
  res.objective = (int64_t)hres[LR_OBJECTIVE];
  rc.lp_passes += res.passes;
  rc.lp_nodes += (int64_t)res.passes * n;
  rc.lp_incidences += (int64_t)res.passes * L.p;
  rc.lp_moved_incidences += (int64_t)hres[LR_MOVED_INCID];
  rc.lp_gain_launches += 1;
  const double g = hres[LR_NS_GAIN] * 1e-6, s = hres[LR_NS_SELECT] * 1e-6,
               a = hres[LR_NS_APPLY] * 1e-6;
  if (cx.timing) {
    rc.ms_gain += g;
    rc.ms_select += s;
    rc.ms_apply += a;
    rc.ms_objective += hres[LR_NS_OBJECTIVE] * 1e-6;
  }
  if (cx.kernel_timing) {
    rc.ms_gain_kernels += g;
    rc.ms_select_kernels += s;
    rc.ms_apply_kernels += a;
  }
  return res;
}

}  // namespace hgk
