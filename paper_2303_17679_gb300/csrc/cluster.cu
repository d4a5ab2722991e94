// The sub-rounds of the clustering of a level (Sec. 11 "Deterministic Clustering
// for Coarsening") as one persistent kernel: rating, approval and the upkeep of
// the cluster words, with a barrier of all blocks between the steps.
//
// What bounds it: the rating of heavy nodes on fine levels; on coarse and small
// levels the 16 sub-rounds of dependent steps.  As launches of a captured graph
// a sub-round took 8 to 15 of them (one per node class, four for the approval,
// three for the cluster words), each with its own tail and 2 us at least, and
// the capture, instantiation and launch of the graph 0.25 to 0.4 ms of host time
// per level.  Here a sub-round has three to six barriers (0.5 us in a cluster,
// 1.4 us over the chip), the classes follow one another without one (a block
// that runs out of heavy nodes goes on to lighter ones), nodes are handed out
// by tickets, and movers are published 32 at a time: three dependent atomics
// per mover cost a warp about 2 us per node.
// Measured (GB300, clustering and contraction of all levels, as graphs -> when
// this form and the passes over the nets came in -> now): 1e6 Zipf, k = 8 70.6 ->
// 52 -> 45.6 ms; 4e6 large nets, k = 64 142 -> 107 -> 85.5 ms; one level of
// 500,009 nodes 10.8 -> 7.2 -> 6.5 ms; of 1471 nodes 1.67 -> 1.2 -> 1.09 ms.
#include <algorithm>
#include <climits>
#include <type_traits>

#include "gridsync.cuh"
#include "rating.cuh"

namespace hgk {

namespace {

template <typename VT>
struct RunShared {
  VT rv[RUN_WARPS];
  int32_t rc[RUN_WARPS];
  int32_t nused[RUN_WARPS][2];
  int32_t tick[RUN_WARPS][2];
  unsigned long long stats[ST_TOTAL];
};

// Movers a warp has found and not yet published, one per lane.
struct Pending {
  int32_t u = 0, c = 0, w = 0;
  int n = 0;  // the same in every lane
};

// Publishes the warp's movers: one claim of the mover list, the targets' sums
// by independent atomics, one claim of the list of touched targets.
__device__ __forceinline__ void publish(const RateArgs& A, int32_t* words, Pending& P) {
  if (P.n == 0) return;
  const int lane = lane_id();
  const bool on = lane < P.n;
  int32_t base = 0;
  if (lane == 0) base = atomicAdd(&words[CW_MOVES], P.n);
  bool first = false;
  if (on) {
    A.target[P.u] = P.c;
    atomicAdd(&A.gw[P.c], P.w);
    first = atomicAdd(&A.gcnt[P.c], 1) == 0;
  }
  base = __shfl_sync(FULL, base, 0);
  if (on) A.mv[base + lane] = P.u;
  const unsigned fresh = __ballot_sync(FULL, first);
  if (fresh) {
    int32_t tb = 0;
    if (lane == 0) tb = atomicAdd(&words[CW_TOUCHED], __popc(fresh));
    tb = __shfl_sync(FULL, tb, 0);
    if (first) A.touched[tb + __popc(fresh & ((1u << lane) - 1u))] = P.c;
  }
  P.n = 0;
}

// u of weight w joins c if c >= 0 (u, w and c the same in all lanes).
__device__ __forceinline__ void push_move(const RateArgs& A, int32_t* words, Pending& P, int32_t u,
                                          int32_t w, int32_t c) {
  if (c < 0) return;
  if (lane_id() == P.n) {
    P.u = u;
    P.w = w;
    P.c = c;
  }
  if (++P.n == 32) publish(A, words, P);
}

// Synchronises the TW warps of team `team` (TW = 1: the warp, else a named
// barrier per team).
__device__ __forceinline__ void team_sync(int team, int TW) {
  if (TW == 1) __syncwarp();
  else asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "r"(TW * 32) : "memory");
}

// Hands out the nodes [0, count) of a class to the teams of all blocks: the
// first `chunk` nodes of a team are fixed, the next come from a ticket that is
// drawn while the current ones are rated.  body(i) rates node i.
template <typename F>
__device__ __forceinline__ void for_nodes(int32_t count, int chunk, int32_t* ticket, int team,
                                          int teams_per_block, int TW, int tid,
                                          int32_t (*s_tick)[2], F&& body) {
  const int32_t teams = teams_per_block * gridDim.x;
  int32_t cur = (team * gridDim.x + blockIdx.x) * chunk;
  for (int round = 0; cur < count; ++round) {
    int32_t next = 0;
    if (tid == 0) next = atomicAdd(ticket, chunk) + teams * chunk;
    const int32_t end = min(cur + chunk, count);
    for (int32_t i = cur; i < end; ++i) body(i);
    if (TW == 1) {
      cur = __shfl_sync(FULL, next, 0);
    } else {
      if (tid == 0) s_tick[team][round & 1] = next;
      team_sync(team, TW);
      cur = s_tick[team][round & 1];
    }
  }
}

// The best of a team's candidates (bv, bc per thread) in its first warp; the
// other warps go on to the next node (the words read here are not written
// again before that node's first barrier).
template <typename VT>
__device__ __forceinline__ void team_best(RunShared<VT>& sh, int team, int wt, int TW, VT& bv,
                                          int32_t& bc) {
  warp_argmax(bv, bc);
  if (TW == 1) {
    __syncwarp();
    return;
  }
  const int lane = lane_id();
  if (lane == 0) {
    sh.rv[team * TW + wt] = bv;
    sh.rc[team * TW + wt] = bc;
  }
  team_sync(team, TW);
  if (wt == 0) {
    bv = lane < TW ? sh.rv[team * TW + lane] : (VT)0;
    bc = lane < TW ? sh.rc[team * TW + lane] : -1;
    warp_argmax(bv, bc);
  }
}

// Teams of TW warps per block: as many as have warps and room for their tables.
template <typename VT, int TW>
constexpr int team_count(uint32_t slots) {
  const size_t fit = TEAM_SMEM<VT> / team_bytes<typename HashOf<VT>::type>(slots);
  return fit < (size_t)(RUN_WARPS / TW) ? (int)fit : RUN_WARPS / TW;
}

// Hash-table classes: teams of TW warps, each rating one node at a time with a
// table of SLOTS shared slots and a list of the slots the node inserted (warps
// beyond the last team sit the class out).
template <typename VT, bool GRAPH, int TW, uint32_t SLOTS>
__device__ void rate_teams(const RateArgs& A, int s, int32_t* words, int cls, const int4* lnode,
                           int32_t count, int chunk, unsigned char* smem, RunShared<VT>& sh,
                           Pending& pend) {
  using H = typename HashOf<VT>::type;
  __syncthreads();  // the tables of the class before are done with
  const int team = warp_in_block() / TW, wt = warp_in_block() % TW;
  const int tid = threadIdx.x % (TW * 32);
  unsigned char* base = smem + (size_t)team * team_bytes<H>(SLOTS);
  constexpr int TEAMS = team_count<VT, TW>(SLOTS);
  H tab = make_hash<H>(base, SLOTS);
  int32_t* used = reinterpret_cast<int32_t*>(base + (size_t)SLOTS * H::BYTES_PER_SLOT);
  if (team >= TEAMS) return;
  for (uint32_t i = tid; i < SLOTS; i += TW * 32) tab.init(i);
  if (tid == 0) sh.nused[team][0] = sh.nused[team][1] = 0;
  team_sync(team, TW);
  int64_t visits = 0, incid = 0, nodes = 0;
  int it = 0;
  for_nodes(count, chunk, &words[CW_TICKET + cls], team, TEAMS, TW, tid, sh.tick, [&](int32_t i) {
    const int4 nd = lnode[i];
    const int32_t u = nd.x, beg = nd.y, end = nd.z, cu = nd.w;
    if (A.cst[u].y < 0) return;  // joined a cluster in an earlier sub-round
    // the used-slot counter of this node; the other one is cleared for the
    // next node once every thread has read this one
    int32_t* nused = &sh.nused[team][it & 1];
    visits += rate_groups<GRAPH, VT, TEAM_ILP>(
        A, s, u, cu, team_walk<GRAPH>(beg, end, wt, TW), end,
        each_visit<VT, TEAM_ILP>([&](int32_t C, VT r) HG_INLINE {
          const int32_t sl = tab.add(C, r);
          if (sl >= 0) used[atomicAdd(nused, 1)] = sl;
          else if (sl == ADD_FULL) dev_fail(A.status_word, DEV_HASH_FULL);
        }));
    team_sync(team, TW);
    VT bv = 0;
    int32_t bc = -1;
    const int32_t nu = *nused;
    if (tid == 0) sh.nused[team][(it + 1) & 1] = 0;
    for (int32_t x = tid; x < nu; x += TW * 32) {
      int32_t C;
      VT v;
      tab.take((uint32_t)used[x], C, v);
      better(bv, bc, v, C);
    }
    team_best(sh, team, wt, TW, bv, bc);
    if (wt == 0) push_move(A, words, pend, u, cu, bc);
    incid += end - beg;
    ++nodes;
    ++it;
  });
  if (lane_id() == 0 && visits)
    atomicAdd(&sh.stats[cls * ST_WORDS + ST_PINS], (unsigned long long)visits);
  if (tid == 0 && nodes) {
    atomicAdd(&sh.stats[cls * ST_WORDS + ST_INCID], (unsigned long long)incid);
    atomicAdd(&sh.stats[cls * ST_WORDS + ST_NODES], (unsigned long long)nodes);
  }
}

// Class 2 of levels whose n fits a shared table: teams of TW warps, each with a
// table direct-indexed by cluster id (n values, then the list of touched ids).
template <typename VT, bool GRAPH>
__device__ void rate_dense(const RateArgs& A, int s, int32_t* words, int cls, const int4* lnode,
                           int32_t count, unsigned char* smem, RunShared<VT>& sh, Pending& pend) {
  __syncthreads();
  const int TW = A.dense_tw;
  const int team = warp_in_block() / TW, wt = warp_in_block() % TW;
  const int tid = threadIdx.x - team * TW * 32;
  // both arrays of a team padded to 16 bytes
  const uint32_t cap = ((uint32_t)A.n + 3u) & ~3u;
  VT* val = reinterpret_cast<VT*>(smem + (size_t)team * cap * (sizeof(VT) + 4));
  int32_t* used = reinterpret_cast<int32_t*>(val + cap);
  for (uint32_t i = tid; i < cap; i += TW * 32) val[i] = 0;
  if (tid == 0) sh.nused[team][0] = sh.nused[team][1] = 0;
  team_sync(team, TW);
  int64_t visits = 0, incid = 0, nodes = 0;
  int it = 0;
  for_nodes(count, 1, &words[CW_TICKET + cls], team, RUN_WARPS / TW, TW, tid, sh.tick,
            [&](int32_t i) {
    const int4 nd = lnode[i];
    const int32_t u = nd.x, beg = nd.y, end = nd.z, cu = nd.w;
    if (A.cst[u].y < 0) return;
    int32_t* nused = &sh.nused[team][it & 1];
    visits += rate_groups<GRAPH, VT, DENSE_ILP>(
        A, s, u, cu, team_walk<GRAPH>(beg, end, wt, TW), end,
        each_visit<VT, DENSE_ILP>([&](int32_t C, VT r) HG_INLINE {
          // every term is >= 1, so a zero before the add marks the first touch
          if (atomicAdd(&val[C], r) == (VT)0) used[atomicAdd(nused, 1)] = C;
        }));
    team_sync(team, TW);
    VT bv = 0;
    int32_t bc = -1;
    const int32_t nu = *nused;
    if (tid == 0) sh.nused[team][(it + 1) & 1] = 0;
    for (int32_t x = tid; x < nu; x += TW * 32) {
      const int32_t C = used[x];
      better(bv, bc, val[C], C);
      val[C] = 0;
    }
    team_best(sh, team, wt, TW, bv, bc);
    if (wt == 0) push_move(A, words, pend, u, cu, bc);
    incid += end - beg;
    ++nodes;
    ++it;
  });
  if (lane_id() == 0 && visits)
    atomicAdd(&sh.stats[cls * ST_WORDS + ST_PINS], (unsigned long long)visits);
  if (tid == 0 && nodes) {
    atomicAdd(&sh.stats[cls * ST_WORDS + ST_INCID], (unsigned long long)incid);
    atomicAdd(&sh.stats[cls * ST_WORDS + ST_NODES], (unsigned long long)nodes);
  }
}

// Split nodes with a table in global memory: one warp per item (a node and 32
// of its records); accumulates into the node's table at tab_off[i] - tab_lo
// (values; keys in hash mode; the list of used slots with its counter
// tnused[i]).
template <typename VT, bool GRAPH>
__device__ void rate_items(const RateArgs& A, int s, const SubPlan& P, RunShared<VT>& sh) {
  const int4* lsplit = A.lnode + A.split_base;
  VT* tval = static_cast<VT*>(A.tval);
  int64_t visits = 0, incid = 0;
  for (int32_t t = P.item_lo + warp_in_block() * gridDim.x + blockIdx.x; t < P.item_hi;
       t += gridDim.x * RUN_WARPS) {
    const int32_t i = A.item_node[t];
    const int4 nd = lsplit[i];
    const int32_t u = nd.x, beg = nd.y, end = nd.z, cu = nd.w;
    if (A.cst[u].y < 0) continue;
    const int32_t g0 = beg + 32 * (t - A.item_off[i]);
    const int64_t base = A.tab_off[i] - P.tab_lo;
    VT* val = tval + base;
    int32_t* used = A.tused + base;
    int32_t* nused = A.tnused + i;
    int32_t run = 0;
    if (A.tab_dense[i]) {
      // direct-indexed: a reduction without a returned value; the argmax
      // scans the whole table, which is no larger than twice the visits
      visits += rate_group<GRAPH, VT, SPLIT_ILP>(
          A, s, u, cu, g0, end, 0, 1, run,
          each_visit<VT, SPLIT_ILP>([&](int32_t C, VT r) HG_INLINE { atomicAdd(&val[C], r); }));
    } else {
      int32_t* key = A.tkey + base;
      const uint32_t mask = (uint32_t)A.tab_cap[i] - 1;
      visits += rate_group<GRAPH, VT, SPLIT_ILP>(
          A, s, u, cu, g0, end, 0, 1, run,
          [&](const int32_t(&C)[SPLIT_ILP], const VT(&rr)[SPLIT_ILP],
              const bool(&ok)[SPLIT_ILP]) HG_INLINE {
            // the first slot of every visit of the batch is loaded at once
            uint32_t h[SPLIT_ILP];
            int32_t k0[SPLIT_ILP];
#pragma unroll
            for (int k = 0; k < SPLIT_ILP; ++k) {
              h[k] = slot_hash(C[k]) & mask;
              k0[k] = ok[k] ? key[h[k]] : C[k];
            }
#pragma unroll
            for (int k = 0; k < SPLIT_ILP; ++k) {
              if (!ok[k]) continue;
              uint32_t hh = h[k];
              int32_t kk = k0[k];
              bool found = false;
              for (uint32_t probe = 0; probe <= mask; ++probe) {
                if (kk == C[k]) {
                  found = true;
                  break;
                }
                if (kk == EMPTY_KEY) {
                  const int32_t old = atomicCAS(&key[hh], EMPTY_KEY, C[k]);
                  if (old == EMPTY_KEY) used[atomicAdd(nused, 1)] = (int32_t)hh;
                  if (old == EMPTY_KEY || old == C[k]) {
                    found = true;
                    break;
                  }
                }
                hh = (hh + 1) & mask;
                kk = key[hh];
              }
              if (found) atomicAdd(&val[hh], rr[k]);
              else dev_fail(A.status_word, DEV_HASH_FULL);
            }
          });
    }
    incid += min(32, end - g0);
  }
  if (lane_id() == 0 && visits) {
    atomicAdd(&sh.stats[SPLIT_CLASS * ST_WORDS + ST_PINS], (unsigned long long)visits);
    atomicAdd(&sh.stats[SPLIT_CLASS * ST_WORDS + ST_INCID], (unsigned long long)incid);
  }
}

// Hashed split nodes whose distinct candidates need more than one shared
// table: the candidates are partitioned over P blocks by a hash of the
// cluster id (part_of).  Every block walks all of the node's visits (the pin
// clusters are read P times, from L2 at the levels where this happens) and
// accumulates the candidates of its part in a shared table (PartCfg);
// P = ceil(min(W, n) / PartCfg::D) makes every table 60 % full at most where the ids
// spread evenly over the parts; a part whose table is full all the same fails the
// run, which cluster_level repeats without parts.  A node of one part publishes its
// argmax directly; otherwise each part leaves its best (rating, cluster) for the per-node
// combine in rate_split_best.  All warps of the block walk the node's groups of
// 32 records, sharing the chunks in turn.
template <typename VT, bool GRAPH>
__device__ void rate_parts(const RateArgs& A, int s, int32_t* words, const SubPlan& P,
                           unsigned char* smem, RunShared<VT>& sh, Pending& pend) {
  using H = typename PartCfg<VT>::Hash;
  constexpr uint32_t SLOTS = PartCfg<VT>::SLOTS;
  constexpr uint32_t CAP = PartCfg<VT>::CAP;
  const int4* lsplit = A.lnode + A.split_base;
  VT* res_v = static_cast<VT*>(A.res_v);
  __syncthreads();
  H tab = make_hash<H>(smem, SLOTS);
  int32_t* used = reinterpret_cast<int32_t*>(smem + (size_t)SLOTS * H::BYTES_PER_SLOT);
  for (uint32_t x = threadIdx.x; x < SLOTS; x += RUN_THREADS) tab.init(x);
  if (threadIdx.x == 0) sh.nused[0][0] = sh.nused[0][1] = 0;
  __syncthreads();
  const int wv = warp_in_block();
  int64_t visits = 0, incid = 0, nodes = 0;
  int it = 0;
  for_nodes(P.part_hi - P.part_lo, 1, &words[CW_TICKET + SPLIT_CLASS], 0, 1, RUN_WARPS,
            (int)threadIdx.x, sh.tick, [&](int32_t x) {
    const int32_t t = P.part_lo + x;
    const int32_t i = A.part_node[t];
    const int4 nd = lsplit[i];
    const int32_t u = nd.x, beg = nd.y, end = nd.z, cu = nd.w;
    if (A.cst[u].y < 0) return;  // joined a cluster in an earlier sub-round
    const int32_t parts = A.part_off[i + 1] - A.part_off[i], k = t - A.part_off[i];
    // slots inserted for this part (listed while they fit the list); the
    // other counter is cleared for the next part once every thread has read
    // this one
    int32_t* nused = &sh.nused[0][it & 1];
    const int32_t cmu = A.comm ? A.comm[u] : -1;
    bool full = false;  // nothing more is added: every probe would walk the table
    auto visit = [&](const int32_t(&q)[PART_ILP], const VT(&rr)[PART_ILP]) HG_INLINE {
      if (full) return;
      int2 ri[PART_ILP];
      resolve_batch<GRAPH, PART_ILP>(A, s, q, ri, cmu);
#pragma unroll
      for (int j = 0; j < PART_ILP; ++j) {
        const int32_t Cj = ri[j].x;
        if (Cj < 0 || Cj == u || (parts != 1 && part_of(Cj, parts) != k) ||
            (long long)ri[j].y + cu > (long long)A.c_max)
          continue;
        const int32_t sl = tab.add(Cj, rr[j]);
        if (sl >= 0) {
          const int32_t y = atomicAdd(nused, 1);
          if (y < (int32_t)CAP) used[y] = sl;
        } else if (sl == ADD_FULL) {
          dev_fail(A.status_word, DEV_HASH_FULL);
          full = true;
        }
      }
    };
    int32_t run = 0;
    const TeamWalk tw = team_walk<GRAPH>(beg, end, wv, RUN_WARPS);
    const int64_t v = rate_groups_raw<GRAPH, VT, PART_ILP>(A, tw.first, end, tw.step, tw.wt, tw.TW,
                                                           run, visit);
    if (k == 0) visits += v;
    team_sync(0, RUN_WARPS);
    const int32_t nu = *nused;
    if (threadIdx.x == 0) sh.nused[0][(it + 1) & 1] = 0;
    VT bv = 0;
    int32_t bc = -1;
    if (nu <= (int32_t)CAP) {
      for (int32_t y = threadIdx.x; y < nu; y += RUN_THREADS) {
        int32_t C;
        VT val;
        tab.take((uint32_t)used[y], C, val);
        better(bv, bc, val, C);
      }
    } else {  // more insertions than the list holds: every slot
      for (uint32_t y = threadIdx.x; y < SLOTS; y += RUN_THREADS) {
        int32_t C;
        VT val;
        tab.take(y, C, val);
        better(bv, bc, val, C);
      }
    }
    team_best(sh, 0, wv, RUN_WARPS, bv, bc);
    if (wv == 0) {
      if (parts == 1) {
        push_move(A, words, pend, u, cu, bc);
        ++nodes;
      } else if (lane_id() == 0) {
        res_v[t] = bv;
        A.res_c[t] = bc;
      }
      if (k == 0) incid += end - beg;
    }
    ++it;
  });
  if (lane_id() == 0 && visits)
    atomicAdd(&sh.stats[SPLIT_CLASS * ST_WORDS + ST_PINS], (unsigned long long)visits);
  if (threadIdx.x == 0 && (incid || nodes)) {
    atomicAdd(&sh.stats[SPLIT_CLASS * ST_WORDS + ST_INCID], (unsigned long long)incid);
    atomicAdd(&sh.stats[SPLIT_CLASS * ST_WORDS + ST_NODES], (unsigned long long)nodes);
  }
}

// The argmax of the split nodes: nodes of several parts take the best of their
// parts' bests (a warp each; the parts hold disjoint candidates), nodes with a
// table in global memory a block each, clearing the table on the way for the
// next sub-round.
template <typename VT>
__device__ void rate_split_best(const RateArgs& A, int32_t* words, const SubPlan& P,
                                RunShared<VT>& sh, Pending& pend) {
  const int4* lsplit = A.lnode + A.split_base;
  const int32_t lo = P.lo[SPLIT_CLASS] - A.split_base, hi = P.hi[SPLIT_CLASS] - A.split_base;
  const VT* res_v = static_cast<const VT*>(A.res_v);
  VT* tval = static_cast<VT*>(A.tval);
  unsigned long long nodes = 0;
  for (int32_t i = lo + warp_in_block() * gridDim.x + blockIdx.x; i < hi;
       i += gridDim.x * RUN_WARPS) {
    const int4 nd = lsplit[i];
    const int32_t b = A.part_off[i], e = A.part_off[i + 1];
    if (e - b <= 1 || A.cst[nd.x].y < 0) continue;
    VT bv = 0;
    int32_t bc = -1;
    const int32_t t = b + lane_id();  // PART_MAX <= 32 parts
    if (t < e) better(bv, bc, res_v[t], A.res_c[t]);
    warp_argmax(bv, bc);
    push_move(A, words, pend, nd.x, nd.w, bc);
    ++nodes;
  }
  if (P.item_hi > P.item_lo) {
    for (int32_t i = lo + blockIdx.x; i < hi; i += gridDim.x) {
      const int4 nd = lsplit[i];
      if (A.part_off[i + 1] != A.part_off[i] || A.cst[nd.x].y < 0) continue;
      const int64_t base = A.tab_off[i] - P.tab_lo;
      VT bv = 0;
      int32_t bc = -1;
      if (A.tab_dense[i]) {
        // 16-byte loads over the whole table (every table offset and capacity
        // is a multiple of 4 entries); only vectors holding a rating are
        // cleared
        constexpr int PER = 16 / (int)sizeof(VT);
        using V = typename std::conditional<sizeof(VT) == 4, uint4, ulonglong2>::type;
        const int32_t nvec = (int32_t)A.tab_cap[i] / PER;
        V* tv = reinterpret_cast<V*>(tval + base);
        for (int32_t x = threadIdx.x; x < nvec; x += RUN_THREADS) {
          const V vv = tv[x];
          const VT* e = reinterpret_cast<const VT*>(&vv);
          bool any = false;
#pragma unroll
          for (int q = 0; q < PER; ++q) {
            if (e[q] == (VT)0) continue;
            any = true;
            better(bv, bc, e[q], x * PER + q);
          }
          if (any) tv[x] = V{};
        }
      } else {
        const int32_t nu = A.tnused[i];
        for (int32_t x = threadIdx.x; x < nu; x += RUN_THREADS) {
          const int32_t sl = A.tused[base + x];
          better(bv, bc, tval[base + sl], A.tkey[base + sl]);
          tval[base + sl] = 0;
          A.tkey[base + sl] = EMPTY_KEY;
        }
      }
      __syncthreads();  // every thread has read tnused[i] and the words of the last node
      team_best(sh, 0, warp_in_block(), RUN_WARPS, bv, bc);
      if (warp_in_block() == 0) {
        if (lane_id() == 0) A.tnused[i] = 0;
        push_move(A, words, pend, nd.x, nd.w, bc);
        ++nodes;
      }
    }
  }
  if (lane_id() == 0 && nodes) atomicAdd(&sh.stats[SPLIT_CLASS * ST_WORDS + ST_NODES], nodes);
}

// ------------------------------------------------------------- approval

// Every touched target C: when all its movers fit, its weight and status take
// them (the movers follow in approve_movers); else it gets a slot in the
// list of contested targets.
__device__ __forceinline__ void approve_targets(const ClusterArgs& A, int32_t* words, int* s_sum) {
  const RateArgs& R = A.R;
  if (threadIdx.x == 0) *s_sum = 0;
  __syncthreads();
  const int32_t nt = words[CW_TOUCHED];
  int32_t joined = 0;
  for (int32_t i = blockIdx.x * RUN_THREADS + threadIdx.x; i < nt; i += gridDim.x * RUN_THREADS) {
    const int32_t C = R.touched[i];
    const int32_t cw = R.cst[C].x, g = R.gw[C], cnt = R.gcnt[C];
    if ((long long)cw + g <= (long long)R.c_max) {
      R.cst[C] = make_int2(cw + g, -1);
      joined += cnt;
      R.gw[C] = 0;
      R.gcnt[C] = 0;
    } else {
      const int32_t sl = atomicAdd(&words[CW_SLOTS], 1);
      A.slot_c[sl] = C;
      A.slot_off[sl] = atomicAdd(&words[CW_CURSOR], cnt);
      A.slot_of[C] = sl;
    }
  }
  joined = warp_sum(joined);
  if (lane_id() == 0 && joined) atomicAdd(s_sum, joined);
  __syncthreads();
  if (threadIdx.x == 0 && *s_sum) atomicSub(R.clusters, *s_sum);
}

// cst[u] of a node that joined cluster C: {C, JOINED}.
constexpr int32_t JOINED = -2;

// Every mover: joins its target, or enters the contested target's list.
__device__ __forceinline__ void approve_movers(const ClusterArgs& A, int32_t* words) {
  const RateArgs& R = A.R;
  const int32_t nm = words[CW_MOVES];
  for (int32_t i = blockIdx.x * RUN_THREADS + threadIdx.x; i < nm; i += gridDim.x * RUN_THREADS) {
    const int32_t u = R.mv[i];
    const int32_t C = R.target[u];
    const int32_t sl = A.slot_of[C];
    if (sl < 0) {
      R.rep[u] = C;
      R.cst[u] = make_int2(C, JOINED);
    } else {
      A.glist[A.slot_off[sl] + atomicAdd(&A.slot_fill[sl], 1)] = u;
    }
  }
}

constexpr int GROUP_SMEM_CAP = 4096;

__device__ void group_bitonic(unsigned long long* buf, int P) {
  for (int kk = 2; kk <= P; kk <<= 1)
    for (int j = kk >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < P; i += RUN_THREADS) {
        const int ixj = i ^ j;
        if (ixj > i) {
          const unsigned long long a = buf[i], b = buf[ixj];
          if ((a > b) == ((i & kk) == 0)) {
            buf[i] = b;
            buf[ixj] = a;
          }
        }
      }
      __syncthreads();
    }
}

// One block per contested target C: order the movers by (c(u), u), accept
// the longest prefix with cw[C] + weight <= c_max.
__device__ void approve_contested(const ClusterArgs& A, int32_t* words, unsigned char* smem) {
  __shared__ long long s_red[32];
  __shared__ unsigned long long s_acc;
  const RateArgs& R = A.R;
  unsigned long long* s_keys = reinterpret_cast<unsigned long long*>(smem);
  const int32_t nslots = words[CW_SLOTS];
  __syncthreads();
  for (int32_t sl = blockIdx.x; sl < nslots; sl += gridDim.x) {
    const int32_t C = A.slot_c[sl];
    const int32_t cnt = R.gcnt[C];
    const int32_t off = A.slot_off[sl];
    const long long cap = (long long)R.c_max - R.cst[C].x;
    if (threadIdx.x == 0) beat(A.barrier);
    long long added = 0;
    int32_t acc = 0;
    if (cnt <= GROUP_SMEM_CAP) {
      int P = 1;
      while (P < cnt) P <<= 1;
      for (int i = threadIdx.x; i < P; i += RUN_THREADS) {
        if (i < cnt) {
          const int32_t u = A.glist[off + i];
          s_keys[i] = ((unsigned long long)(uint32_t)A.c[u] << 32) | (uint32_t)u;
        } else {
          s_keys[i] = ~0ull;
        }
      }
      if (threadIdx.x == 0) s_acc = 0;
      __syncthreads();
      group_bitonic(s_keys, P);
      // the accepted count is the number of positions whose inclusive weight
      // prefix is <= cap (weights are positive, so these form a prefix)
      long long carry = 0;
      for (int base = 0; base < cnt; base += RUN_THREADS) {
        const int i = base + threadIdx.x;
        const long long v = i < cnt ? (long long)(s_keys[i] >> 32) : 0;
        const long long x = warp_inclusive_scan(v);
        if (lane_id() == 31) s_red[warp_in_block()] = x;
        __syncthreads();
        if (warp_in_block() == 0) {
          long long y = s_red[lane_id()];
          y = warp_inclusive_scan(y);
          s_red[lane_id()] = y;
        }
        __syncthreads();
        const long long incl = carry + (warp_in_block() ? s_red[warp_in_block() - 1] : 0) + x;
        const long long chunk_total = s_red[RUN_WARPS - 1];
        if (i < cnt && incl <= cap) atomicAdd(&s_acc, 1ull);
        carry += chunk_total;
        __syncthreads();
      }
      acc = (int32_t)s_acc;
      for (int i = threadIdx.x; i < acc; i += RUN_THREADS) {
        const int32_t u = (int32_t)(s_keys[i] & 0xffffffffu);
        R.rep[u] = C;
        R.cst[u] = make_int2(C, JOINED);
        added += (long long)(s_keys[i] >> 32);
      }
    } else {
      // large group: binary search for the first excluded key x, the largest
      // x with (sum of c over keys < x) <= cap; all keys < x are accepted
      unsigned long long lo = 0, hi = (1ull << 63);
      while (hi - lo > 1) {
        const unsigned long long mid = lo + ((hi - lo) >> 1);
        long long f = 0;
        for (int i = threadIdx.x; i < cnt; i += RUN_THREADS) {
          const int32_t u = A.glist[off + i];
          const unsigned long long kk = ((unsigned long long)(uint32_t)A.c[u] << 32) | (uint32_t)u;
          if (kk < mid) f += A.c[u];
          beat_along(A.barrier, i);
        }
        f = block_sum(f, s_red);
        if (f <= cap) lo = mid; else hi = mid;
      }
      for (int i = threadIdx.x; i < cnt; i += RUN_THREADS) {
        const int32_t u = A.glist[off + i];
        const unsigned long long kk = ((unsigned long long)(uint32_t)A.c[u] << 32) | (uint32_t)u;
        if (kk < lo) {
          R.rep[u] = C;
          R.cst[u] = make_int2(C, JOINED);
          added += A.c[u];
          ++acc;
        }
      }
      acc = (int32_t)block_sum((long long)acc, s_red);
    }
    added = block_sum(added, s_red);
    if (threadIdx.x == 0) {
      R.cst[C].x += (int32_t)added;
      if (acc > 0) {
        R.cst[C].y = -1;
        atomicSub(R.clusters, acc);
      }
      A.slot_of[C] = -1;
      A.slot_fill[sl] = 0;
      R.gw[C] = 0;
      R.gcnt[C] = 0;
    }
    __syncthreads();
  }
}

// ------------------------------------------ cluster word maintenance

// Before sub-round s every record of a rated net is brought up to date in one
// pass over the nets: a node that joined since hands its word to its cluster,
// a cluster found twice in the net keeps one record (-1 in the others; any one
// will do: they say the same, and the ranges of grouped levels hold all
// members of an admissible cluster), and the weight word becomes the cluster's
// weight, or INT32_MAX for an unclustered node of sub-round s.  A record of -1
// stays -1.  Repeats can only appear through records that joined.
// Bound by L2: one 8-byte record and one 8-byte gather of {weight, status} or,
// for a node that joined, {cluster, JOINED} per pin.  (A hash map from (net,
// cluster) to the first position, updated at the incidences of the joined
// nodes, read two or three random DRAM sectors per incidence in tables of
// 48 bytes per pin: 180 us per sub-round on 5M pins with the weight pass, plus
// 0.4 ms per level to fill.)

// The record's new cluster and its {weight, status}; `joined` when the record
// changed hands.
__device__ __forceinline__ int32_t resolve_record(const int2* cst, int32_t X, int2& cs,
                                                  bool& joined) {
  cs = X >= 0 ? cst[X] : make_int2(0, 0);
  joined = X >= 0 && cs.y == JOINED;
  if (joined) {
    X = cs.x;
    cs = cst[X];
  }
  return X;
}

__device__ __forceinline__ int32_t weight_word(int2 cs, int s) {
  return cs.y == s ? 0x7fffffff : cs.x;
}

// Nets of at most G pins by groups of G lanes; NET_ILP nets per group in flight.
constexpr int NET_ILP = 2;

template <int G>
__device__ __forceinline__ void refresh_small(const ClusterArgs& A, const int2* list, int32_t count,
                                              int s) {
  constexpr int PER = 32 / G;
  const int lane = lane_id(), sub = lane % G, grp = lane / G;
  const int64_t stride = (int64_t)gridDim.x * RUN_WARPS * PER;
  for (int64_t i0 = (int64_t)(warp_in_block() * gridDim.x + blockIdx.x) * PER; i0 < count;
       i0 += NET_ILP * stride) {
    int2 net[NET_ILP], r[NET_ILP], cs[NET_ILP];
    int32_t X[NET_ILP];
    bool joined[NET_ILP];
#pragma unroll
    for (int k = 0; k < NET_ILP; ++k) {
      const int64_t i = i0 + k * stride + grp;
      net[k] = i < count && i0 + k * stride < count ? list[i] : make_int2(0, 0);
    }
#pragma unroll
    for (int k = 0; k < NET_ILP; ++k)
      r[k] = sub < net[k].y ? A.rinfo[net[k].x + sub] : make_int2(-1, 0);
#pragma unroll
    for (int k = 0; k < NET_ILP; ++k) X[k] = resolve_record(A.R.cst, r[k].x, cs[k], joined[k]);
#pragma unroll
    for (int k = 0; k < NET_ILP; ++k) {
      if (__ballot_sync(FULL, joined[k])) {
        // the lowest lane of a net that holds a cluster keeps it
        const unsigned long long key =
            X[k] >= 0 ? ((unsigned long long)grp << 32) | (unsigned)X[k]
                      : (1ull << 63) | (unsigned)lane;
        const unsigned peers = __match_any_sync(FULL, key);
        if (peers & ((1u << lane) - 1u)) X[k] = -1;
      }
      if (r[k].x >= 0) {
        const int32_t w = X[k] >= 0 ? weight_word(cs[k], s) : 0;
        if (X[k] != r[k].x || w != r[k].y) A.rinfo[net[k].x + sub] = make_int2(X[k], w);
      }
    }
  }
}

// Nets of 33 to BIG_NET pins, one warp each.  The clusters that records joined
// enter a hash set in the warp's shared memory (a cluster found there already
// is a repeat), then every other record looks its cluster up and takes it from
// the record that joined.  (Comparing each joined record with all others: 45 us
// per sub-round on 1.1M pins.)
constexpr int JOIN_SLOTS = 512;
struct JoinSet {
  int32_t x[BIG_NET];         // the net's clusters (-1: none)
  int32_t key[JOIN_SLOTS];    // cluster
  uint16_t pos[JOIN_SLOTS];   // position in the net of the record that joined
};

__device__ __forceinline__ void refresh_big(const ClusterArgs& A, const int2* list, int32_t count,
                                            int s, JoinSet* sets) {
  JoinSet& J = sets[warp_in_block()];
  const int lane = lane_id();
  for (int i = lane; i < JOIN_SLOTS; i += 32) J.key[i] = -1;
  __syncwarp();
  for (int32_t i = warp_in_block() * gridDim.x + blockIdx.x; i < count;
       i += gridDim.x * RUN_WARPS) {
    const int2 net = list[i];
    int joins = 0;
    for (int q0 = 0; q0 < net.y; q0 += 128) {
      int2 r[4], cs[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const int q = q0 + 32 * h + lane;
        r[h] = q < net.y ? A.rinfo[net.x + q] : make_int2(-1, 0);
      }
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const int q = q0 + 32 * h + lane;
        bool joined;
        int32_t X = resolve_record(A.R.cst, r[h].x, cs[h], joined);
        const unsigned who = __ballot_sync(FULL, joined);
        if (who && joins + __popc(who) <= JOIN_SLOTS / 2 && joined) {
          uint32_t slot = slot_hash(X) >> 23;  // 9 bits
          for (;;) {  // at most half full: ends at an empty slot
            const int32_t old = atomicCAS(&J.key[slot], -1, X);
            if (old == -1) J.pos[slot] = (uint16_t)q;
            if (old == X) X = -1;
            if (old == -1 || old == X || X < 0) break;
            slot = (slot + 1) & (JOIN_SLOTS - 1);
          }
        }
        joins += __popc(who);
        if (q < net.y) {
          // while looking up, records that joined are told apart by the mark
          J.x[q] = joined && X >= 0 ? X | (int32_t)0x80000000 : X;
          if (r[h].x >= 0) {
            const int32_t w = X >= 0 ? weight_word(cs[h], s) : 0;
            if (X != r[h].x || w != r[h].y) A.rinfo[net.x + q] = make_int2(X, w);
          }
        }
      }
    }
    if (joins == 0) continue;
    __syncwarp();
    if (joins <= JOIN_SLOTS / 2) {
      for (int q = lane; q < net.y; q += 32) {
        const int32_t X = J.x[q];
        if (X < 0) continue;  // no record, or one that joined
        uint32_t slot = slot_hash(X) >> 23;
        for (int32_t k = J.key[slot]; k != -1; k = J.key[slot]) {
          if (k == X) {
            A.rinfo[net.x + J.pos[slot]].x = -1;
            break;
          }
          slot = (slot + 1) & (JOIN_SLOTS - 1);
        }
      }
    } else {
      // more records joined than the set takes: each is compared with all
      // others (another that did not join, or an earlier one that did, keeps
      // the cluster)
      for (int pos = 0; pos < net.y; ++pos) {
        const int32_t mine = J.x[pos];
        if (mine >= -1) continue;
        bool held = false;
        for (int q = lane; q < net.y; q += 32) {
          const int32_t v = J.x[q];
          held |= v != -1 && ((v ^ mine) & 0x7fffffff) == 0 && (v >= 0 || q < pos);
        }
        if (__any_sync(FULL, held) && lane == 0) A.rinfo[net.x + pos].x = -1;
      }
    }
    __syncwarp();
    for (int x = lane; x < JOIN_SLOTS; x += 32) J.key[x] = -1;
    __syncwarp();
  }
}

// Larger nets, one block each: the clusters seen so far are marked in the
// block's bitmap of the level's nodes, those that did not join first.
__device__ void refresh_huge(const ClusterArgs& A, const int2* list, int32_t count, int s) {
  if ((int)blockIdx.x >= A.nets.bitmap_blocks) return;
  unsigned* bm = A.nets.bitmaps + (size_t)blockIdx.x * A.nets.words;
  const int32_t step = min((int32_t)gridDim.x, A.nets.bitmap_blocks);
  for (int32_t i = blockIdx.x; i < count; i += step) {
    const int2 net = list[i];
    if (threadIdx.x == 0) beat(A.barrier);
    for (int turn = 0; turn < 2; ++turn) {
      for (int32_t q = threadIdx.x; q < net.y; q += RUN_THREADS) {
        const int2 r = A.rinfo[net.x + q];
        if (r.x < 0) continue;
        int2 cs;
        bool joined;
        const int32_t X = resolve_record(A.R.cst, r.x, cs, joined);
        if (joined != (turn == 1)) continue;
        const unsigned bit = 1u << (X & 31);
        const bool held = (atomicOr(&bm[X >> 5], bit) & bit) != 0 && joined;
        const int32_t w = held ? 0 : weight_word(cs, s);
        if (joined || w != r.y) A.rinfo[net.x + q] = make_int2(held ? -1 - X - 1 : X, w);
      }
      __syncthreads();
    }
    // clear the bits; a record that lost its cluster still names it (-2 - X)
    for (int32_t q = threadIdx.x; q < net.y; q += RUN_THREADS) {
      const int32_t X = A.rinfo[net.x + q].x;
      if (X == -1) continue;
      const int32_t C = X >= 0 ? X : -2 - X;
      bm[C >> 5] = 0u;
      if (X < 0) A.rinfo[net.x + q].x = -1;
    }
    __syncthreads();
  }
}

__device__ __forceinline__ void refresh_records(const ClusterArgs& A, int s, unsigned char* smem) {
  const NetLists& N = A.nets;
  if (N.count[4] > 0) refresh_big(A, N.list[4], N.count[4], s, reinterpret_cast<JoinSet*>(smem));
  refresh_small<32>(A, N.list[3], N.count[3], s);
  refresh_small<16>(A, N.list[2], N.count[2], s);
  refresh_small<8>(A, N.list[1], N.count[1], s);
  refresh_small<4>(A, N.list[0], N.count[0], s);
  if (N.count[5] > 0) refresh_huge(A, N.list[5], N.count[5], s);
}

// ------------------------------------------------------------ the kernel

template <typename VT, bool GRAPH>
__global__ void __launch_bounds__(RUN_THREADS, 1)
k_cluster_run(const __grid_constant__ ClusterArgs A) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ RunShared<VT> sh;
  __shared__ int s_sum;
  __shared__ SubPlan P;
  const RateArgs& R = A.R;
  for (int i = threadIdx.x; i < ST_TOTAL; i += RUN_THREADS) sh.stats[i] = 0;
  unsigned gen = 0;
  const bool clock = A.timing && blockIdx.x == 0 && threadIdx.x == 0;
  unsigned long long t0 = 0;
  auto lap = [&](int word) {
    if (!clock) return;
    const unsigned long long t = now_ns();
    if (word >= 0) sh.stats[word] += t - t0;
    t0 = t;
  };
  auto sync = [&]() { return grid_sync(A.cluster, A.barrier, R.status_word, gen); };
  for (int s = 0; s < A.S; ++s) {
    // the contraction limit of a level (stopped sub-rounds stay stopped)
    if (5ll * (long long)*R.clusters <= 2ll * (long long)R.n) break;
    int32_t* words = A.words + (size_t)s * CW_WORDS;
    __syncthreads();
    if (threadIdx.x < sizeof(SubPlan) / 4)
      reinterpret_cast<int32_t*>(&P)[threadIdx.x] =
          reinterpret_cast<const int32_t*>(A.plan + s)[threadIdx.x];
    __syncthreads();
    lap(-1);
    // ---- rating, heaviest classes first
    Pending pend;
    if (P.part_hi > P.part_lo) rate_parts<VT, GRAPH>(R, s, words, P, smem, sh, pend);
    if (P.item_hi > P.item_lo) rate_items<VT, GRAPH>(R, s, P, sh);
    lap(SPLIT_CLASS * ST_WORDS + ST_NS);
    auto list = [&](int c) { return R.lnode + P.lo[c]; };
    auto size = [&](int c) { return P.hi[c] - P.lo[c]; };
    if (size(3) > 0)
      rate_teams<VT, GRAPH, sizeof(VT) == 4 ? 16 : 32, 2 * D_BLOCK>(R, s, words, 3, list(3), size(3), 1,
                                                                   smem, sh, pend);
    lap(3 * ST_WORDS + ST_NS);
    if (size(2) > 0) {
      if (R.dense_tw)
        rate_dense<VT, GRAPH>(R, s, words, 2, list(2), size(2), smem, sh, pend);
      else
        rate_teams<VT, GRAPH, 8, 2 * D_QUAD>(R, s, words, 2, list(2), size(2), 1, smem, sh, pend);
    }
    lap(2 * ST_WORDS + ST_NS);
    if (size(1) > 0)
      rate_teams<VT, GRAPH, 4, 2 * D_PAIR>(R, s, words, 1, list(1), size(1), 2, smem, sh, pend);
    lap(1 * ST_WORDS + ST_NS);
    if (size(0) > 0)
      rate_teams<VT, GRAPH, 1, 2 * D_WARP>(R, s, words, 0, list(0), size(0), 4, smem, sh, pend);
    __syncwarp();
    if (P.argmax) {
      publish(R, words, pend);
      if (!sync()) return;
      rate_split_best<VT>(R, words, P, sh, pend);
      __syncwarp();
    }
    publish(R, words, pend);
    if (!sync()) return;
    lap(0 * ST_WORDS + ST_NS);
    // ---- approval
    approve_targets(A, words, &s_sum);
    if (!sync()) return;
    approve_movers(A, words);
    if (!sync()) return;
    if (words[CW_SLOTS] > 0) {
      approve_contested(A, words, smem);
      if (!sync()) return;
    }
    lap(ST_NS_APPROVE);
    // ---- cluster words of the next sub-round
    if (!GRAPH && A.records && s + 1 < A.S) {
      refresh_records(A, s + 1, smem);
      if (!sync()) return;
      lap(ST_NS_REFRESH);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < ST_TOTAL; i += RUN_THREADS)
    if (sh.stats[i]) atomicAdd(&R.stats[i], sh.stats[i]);
}

template <typename VT, bool GRAPH>
void launch_run(const Ctx& cx, const ClusterArgs& A, int blocks, size_t smem) {
  prepare_kernel(cx, &k_cluster_run<VT, GRAPH>,
                 std::max({part_bytes<VT>(), TEAM_SMEM<VT>, DENSE_SMEM + 64,
                           sizeof(JoinSet) * RUN_WARPS}),
                 true);
  launch_persistent(cx, k_cluster_run<VT, GRAPH>, blocks, RUN_THREADS, smem, A.cluster, A);
}

constexpr int CLUSTER_MAX = 16;

}  // namespace

void run_subrounds(const Ctx& cx, ClusterArgs A, bool narrow, bool graph, size_t smem,
                   int64_t listed, int64_t heavy, int64_t total_visits) {
  // Blocks of a sub-round's work: one light node per warp, four heavy ones per
  // block, 256 visits per warp, 16 records per thread.  Up to 16 blocks run as
  // one cluster, above that one block per SM.  A call that shares the GPU with
  // others (inflight.cuh) takes a quarter of that and at most half the SMs, so that
  // several levels are resident at once.  Serving 200 requests per second of 1e4
  // to 2e6 pins on 16 streams: p50 / p99 664 / 1420 ms without the limit, 25 / 112
  // ms with it, 21 / 83 ms with a quarter of the SMs, which a large request on two
  // streams pays for; as separate launches 56 / 230 ms.  Eight host threads with
  // plain handles (20,000 nodes, k = 32): 224 -> 459 partitions per second with
  // the limit (319 as separate launches), one thread 113.
  const int64_t S = A.S, share = cx.shares_gpu() ? 4 : 1;
  const int64_t need =
      std::max<int64_t>({(listed - heavy) / (S * RUN_WARPS), heavy / (S * 4),
                         total_visits / (S * RUN_WARPS * 256), A.p / (RUN_THREADS * 16)}) /
          share + 1;
  if (A.records) smem = std::max(smem, sizeof(JoinSet) * RUN_WARPS);
  int blocks = share == 1 ? cx.num_sms
                          : (int)std::min<int64_t>(need, std::max(1, cx.num_sms / 2));
  if (need <= CLUSTER_MAX) {
    A.cluster = true;
    blocks = 1;
    while (blocks < need) blocks <<= 1;
  }
  if (graph && narrow) launch_run<uint32_t, true>(cx, A, blocks, smem);
  else if (graph) launch_run<unsigned long long, true>(cx, A, blocks, smem);
  else if (narrow) launch_run<uint32_t, false>(cx, A, blocks, smem);
  else launch_run<unsigned long long, false>(cx, A, blocks, smem);
}

}  // namespace hgk
