// Community detection before coarsening (Sec. 4 "Community-Aware Coarsening",
// Sec. 11 "Deterministic Louvain Method") on the device.
//
// The hypergraph becomes its bipartite graph: a vertex per node (0..n-1) and
// per net (n + e), an edge {v, n + e} for every pin with weight
// floor(w(e) * 2^20 / |e|), an integer reading of the fractional w(e) / |e|
// model.  Every sum below is an integer sum, so the cluster volumes that the
// paper aggregates in a fixed order are exact here whatever the order of the
// atomics, and every decision is bit-identical from run to run.
//
// The Louvain method, per level: clusters start as singletons; up to
// LV_ROUNDS rounds of S synchronous sub-rounds (vertex i is in sub-round
// mix64(seed ^ 2^62 ^ level<<32 ^ (round+1)<<48 ^ i) mod S); in a sub-round
// every listed vertex picks, from the state at the sub-round's start, the
// neighbouring cluster C maximising s(C) = 2W k_{i,C} - k_i vol(C) (128-bit
// integers, ties to the smaller id) and moves when s(C) exceeds its own
// cluster's s(A) = 2W k_{i,A} - k_i (vol(A) - k_i); all moves are applied
// (no weight limit), volumes updated with integer atomics.  A round moving
// fewer than 1 % of the vertices ends the level; a level without any move
// ends the detection.  Otherwise the clusters are aggregated (coarse vertex
// = rank of the cluster id; edges between clusters summed, edges inside a
// cluster added to its self-loop weight) and the next level starts.
//
// Layout per level: CSR with int64 offsets, int32 neighbours, int64 weights,
// int64 self-loop weights, degrees k and volumes.
//
// The rounds of a level run as one persistent kernel (blocks meet at grid_sync;
// two or three barriers per sub-round).  Per round the vertices are listed by
// (sub-round, class): vertices of at most 8 (32) edges are decided by a group of
// eight lanes (a warp) that holds one edge per lane and sums the edges of a
// cluster by exchanging them; up to LV_SMALL edges by one warp with a shared
// table of the neighbouring clusters, up to LV_BLOCK by the block with all the
// tables as one; up to LV_HUGE in parts by a hash of the cluster, a block each,
// whose bests are compared after one more barrier; larger vertices by chunks of
// their edges, a block each, which sum a chunk in shared memory and add it to the
// vertex's table in global memory, read in pieces after a barrier.  Aggregation
// adds the edges to global tables, one per coarse vertex.
// What bounds it: some 25 rounds of 16 dependent sub-rounds, each a chain of
// gathers; as four or five launches per sub-round, with a host wait and the
// copy of all table offsets per round, the detection on 250,007 nodes and
// 1.35M pins took 30.1 ms, now 14.2 ms.
#include <algorithm>

#include "gridsync.cuh"
#include "louvain.cuh"
#include "pintile.cuh"

namespace hgk {

namespace {

constexpr int LV_LEVELS = 32;
constexpr int LV_THREADS = 512;
constexpr int LV_WARPS = LV_THREADS / 32;
constexpr int LV_SLOTS = 2 * LV_SMALL;  // slots per warp (load <= 1/2)
constexpr int LV_BLOCK_SLOTS = LV_SLOTS * LV_WARPS;
constexpr int LV_CHUNK_SLOTS = 2 * LV_CHUNK;
static_assert(2 * LV_BLOCK <= LV_BLOCK_SLOTS && LV_CHUNK_SLOTS <= LV_BLOCK_SLOTS,
              "the block's table is at most half full");
constexpr int32_t LV_EMPTY = -1;

using i128 = __int128;

__device__ __forceinline__ int subround_louvain(uint64_t seed, int level, int round, int64_t i,
                                                int S) {
  const uint64_t x = seed ^ (1ull << 62) ^ ((uint64_t)(uint32_t)level << 32) ^
                     ((uint64_t)(uint32_t)(round + 1) << 48) ^ (uint64_t)(uint32_t)i;
  return subround_mod(mix64(x), S);
}

// ------------------------------------------------------------ level 0

// Bipartite CSR from the hypergraph: node v's edges are its incidences
// (positions ioff[v]..), net e's edges its pins (positions p + eoff[e]..).
__device__ __forceinline__ long long lv_net_weight(const int32_t* __restrict__ eoff,
                                                   const int32_t* __restrict__ w, int32_t e) {
  const int32_t size = eoff[e + 1] - eoff[e];
  return (long long)(((unsigned long long)w[e] << 20) / (unsigned long long)size);
}

// One thread per incidence j = (v, e).
__global__ void k_lv_node_edges(const int32_t* __restrict__ eoff, const int32_t* __restrict__ w,
                                const int32_t* __restrict__ inets, int32_t n, int64_t p,
                                int32_t* __restrict__ adj, long long* __restrict__ aw) {
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < p;
       j += (int64_t)gridDim.x * blockDim.x) {
    const int32_t e = inets[j];
    adj[j] = n + e;
    aw[j] = lv_net_weight(eoff, w, e);
  }
}

// One thread per pin; adj and aw start at the nets' edges.
__global__ void __launch_bounds__(PIN_TILE_THREADS)
k_lv_net_edges(const int32_t* __restrict__ eoff, const int32_t* __restrict__ pins,
               const int32_t* __restrict__ w, const int32_t* __restrict__ tile_net, int32_t m,
               int64_t p, int32_t* __restrict__ adj, long long* __restrict__ aw) {
  __shared__ int32_t s_off[PIN_TILE + 3];
  const int64_t ntiles = num_pin_tiles(p);
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const PinTileView v = stage_pin_tile(eoff, tile_net, m, p, t, s_off);
    for (int64_t q = v.q0 + threadIdx.x; q < v.q1; q += blockDim.x) {
      adj[q] = pins[q];
      aw[q] = lv_net_weight(eoff, w, v.e_lo + net_in_tile(s_off, v.count, q));
    }
    __syncthreads();
  }
}

__global__ void k_lv_offsets(const int32_t* __restrict__ ioff, const int32_t* __restrict__ eoff,
                             int32_t n, int32_t m, int64_t p, long long* __restrict__ off) {
  const int64_t V = (int64_t)n + m;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= V;
       i += (int64_t)gridDim.x * blockDim.x)
    off[i] = i <= n ? (long long)ioff[i] : (long long)(p + eoff[i - n]);
}

// What k_lv_degrees adds up: the degrees, the table slots that the class 5
// vertices of one sub-round take at most, and those slots per round and sub-round.
enum { LD_TOTAL = 0, LD_MOST = 1, LD_SLOTS = 2 };

// k_i = 2 self_i + sum of i's edge weights (a warp per vertex); W2 = sum k_i.
__global__ void k_lv_degrees(const long long* __restrict__ off, const long long* __restrict__ aw,
                             const long long* __restrict__ self, int64_t V, uint64_t seed,
                             int level, int S, int huge, long long* __restrict__ k,
                             unsigned long long* __restrict__ sums) {
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  long long acc = 0;
  for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < V; i += nw) {
    long long s = 0;
    for (long long q = off[i] + lane_id(); q < off[i + 1]; q += 32) s += aw[q];
    s = warp_sum(s);
    s += 2 * self[i];
    if (lane_id() == 0) k[i] = s;
    acc += s;
    const long long deg = off[i + 1] - off[i];
    if (deg > huge && lane_id() < LV_ROUNDS) {
      const int r = lane_id();
      const unsigned long long slots = lv_slots(deg);
      const unsigned long long before =
          atomicAdd(&sums[LD_SLOTS + r * S + subround_louvain(seed, level, r, i, S)], slots);
      atomicMax(&sums[LD_MOST], before + slots);
    }
  }
  if (lane_id() == 0 && acc) atomicAdd(&sums[LD_TOTAL], (unsigned long long)acc);
}

__global__ void k_lv_init(int64_t V, const long long* __restrict__ k, int32_t* __restrict__ cl,
                          long long* __restrict__ vol) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < V;
       i += (int64_t)gridDim.x * blockDim.x) {
    cl[i] = (int32_t)i;
    vol[i] = k[i];
  }
}

// ------------------------------------------------------------ tables

// Adds `val` to `key`'s entry of a global table (keys LV_EMPTY when free).
__device__ __forceinline__ bool table_add(int32_t* keys, long long* vals, uint32_t mask,
                                          int32_t key, long long val) {
  uint32_t h = ((uint32_t)key * 0x9E3779B1u) & mask;
  for (uint32_t probe = 0; probe <= mask; ++probe) {
    int32_t k = keys[h];
    if (k == LV_EMPTY) {
      const int32_t old = atomicCAS(&keys[h], LV_EMPTY, key);
      k = old == LV_EMPTY ? key : old;
    }
    if (k == key) {
      atomicAdd(reinterpret_cast<unsigned long long*>(&vals[h]), (unsigned long long)val);
      return true;
    }
    h = (h + 1) & mask;
  }
  return false;
}

// Candidate (score, cluster) comparison: larger score, ties to smaller id.
struct Cand {
  i128 s;
  int32_t c;
};

__device__ __forceinline__ void cand_better(Cand& a, const Cand& b) {
  if (b.c >= 0 && (a.c < 0 || b.s > a.s || (b.s == a.s && b.c < a.c))) a = b;
}

__device__ __forceinline__ Cand shfl_cand(const Cand& x, int d) {
  Cand y;
  const unsigned long long lo = (unsigned long long)x.s;
  const long long hi = (long long)(x.s >> 64);
  const unsigned long long ylo = __shfl_xor_sync(FULL, lo, d);
  const long long yhi = __shfl_xor_sync(FULL, hi, d);
  y.s = ((i128)yhi << 64) | (i128)ylo;
  y.c = __shfl_xor_sync(FULL, x.c, d);
  return y;
}

__device__ __forceinline__ void warp_best(Cand& x) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) cand_better(x, shfl_cand(x, d));
}

// ------------------------------------------------------------ local moving

enum { LV_MOVES = 0, LV_WORDS = 4 };           // per sub-round (two sets)
enum { LR_MOVED = 0, LR_ROUNDS = 1, LR_LV_WORDS = 2 };

// Best of one part of a vertex.
struct PartBest {
  unsigned long long lo;
  long long hi, kia;
  int32_t c, pad;
};

// A class 5 vertex of the round: its list entries and its table.
struct HugeVertex {
  int32_t i, entries;
  unsigned long long tab, slots;
};

struct LvArgs {
  const long long* off;
  const int32_t* adj;
  const long long* aw;
  const long long* k;
  int32_t* cl;
  long long* vol;
  long long W2;
  int64_t V;
  uint64_t seed;
  int level, S;
  int huge_deg;     // class 5 above this degree
  int2* list;       // {vertex, part} by (sub-round, class); class 5 {index in huge, chunk}
  int32_t *cnt, *fill;  // LV_CLASSES S each
  HugeVertex* huge;
  int32_t* nhuge;
  unsigned long long* tabfill;  // S: table slots given out
  int32_t* tkey;                // tables of the class 5 vertices of a sub-round
  long long* tval;
  int2* mv;         // {vertex, cluster}
  int32_t* words;
  PartBest* parts;
  unsigned long long* res;
  unsigned* barrier;  // two words (grid_sync)
  int32_t* status;
};

// Counts (scatter == false) or writes the list entries of the block's tiles of
// vertices; one global claim per tile and key.
__device__ __forceinline__ void lv_list(const LvArgs& A, int round, bool scatter,
                                        const int32_t* s_off, int32_t* s_hist, int32_t* s_base) {
  const int keys = LV_CLASSES * A.S;
  for (int i = threadIdx.x; i < keys; i += LV_THREADS) s_hist[i] = 0;
  __syncthreads();
  const int64_t stride = (int64_t)gridDim.x * LV_THREADS;
  for (int64_t i0 = (int64_t)blockIdx.x * LV_THREADS; i0 < A.V; i0 += stride) {
    const int64_t i = i0 + threadIdx.x;
    int key = -1, slot = 0, cls = 0;
    int32_t entries = 0;
    long long deg = 0;
    if (i < A.V) {
      deg = A.off[i + 1] - A.off[i];
      if (deg > 0) {  // a vertex without neighbours never moves
        cls = lv_class(deg, A.huge_deg, entries);
        key = subround_louvain(A.seed, A.level, round, i, A.S) * LV_CLASSES + cls;
        slot = atomicAdd(&s_hist[key], entries);
      }
    }
    if (!scatter) continue;
    __syncthreads();
    for (int x = threadIdx.x; x < keys; x += LV_THREADS) {
      s_base[x] = s_hist[x] ? atomicAdd(&A.fill[x], s_hist[x]) : 0;
      s_hist[x] = 0;
    }
    __syncthreads();
    if (key >= 0) {
      int2* out = A.list + s_off[key] + s_base[key] + slot;
      int32_t name = (int32_t)i;
      if (cls == 5) {
        name = atomicAdd(A.nhuge, 1);
        const unsigned long long slots = lv_slots(deg);
        A.huge[name] = HugeVertex{(int32_t)i, entries,
                                  atomicAdd(&A.tabfill[key / LV_CLASSES], slots), slots};
      }
      for (int32_t x = 0; x < entries; ++x) out[x] = make_int2(name, x);
    }
    __syncthreads();
  }
  if (!scatter) {
    __syncthreads();
    for (int x = threadIdx.x; x < keys; x += LV_THREADS)
      if (s_hist[x]) atomicAdd(&A.cnt[x], s_hist[x]);
  }
}

__device__ __forceinline__ void lv_offsets_of(const LvArgs& A, int32_t* s_off) {
  const int keys = LV_CLASSES * A.S;
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

// Vertex i moves to the best other candidate iff s(best) > s(own), kia = the
// weight of its edges into its own cluster.
__device__ __forceinline__ bool lv_moves(const LvArgs& A, int32_t i, long long kia,
                                         const Cand& best) {
  if (best.c < 0) return false;
  const long long ki = A.k[i];
  return best.s > (i128)A.W2 * kia - (i128)ki * (A.vol[A.cl[i]] - ki);
}

// Lanes with `moves` enter {i, c} in the move list (the whole warp calls it).
__device__ __forceinline__ void lv_emit(const LvArgs& A, int32_t* words, bool moves, int32_t i,
                                        int32_t c) {
  const unsigned who = __ballot_sync(FULL, moves);
  if (!who) return;
  int32_t slot = 0;
  if (lane_id() == 0) slot = atomicAdd(&words[LV_MOVES], __popc(who));
  slot = __shfl_sync(FULL, slot, 0) + __popc(who & ((1u << lane_id()) - 1u));
  if (moves) A.mv[slot] = make_int2(i, c);
}

// Classes 0 and 1: G lanes per vertex of at most G edges, one edge per lane.
// Every lane sums the edges of its own cluster (equal lanes hold equal
// candidates); the groups of a warp stay in step.
template <int G>
__device__ __forceinline__ void lv_lanes(const LvArgs& A, int32_t* words, int32_t lo, int32_t hi,
                                         int64_t gw, int64_t NW) {
  constexpr int PER = 32 / G;
  const int lane = lane_id(), sub = lane % G, grp = lane / G;
  for (int64_t x0 = lo + gw * PER; x0 < hi; x0 += NW * PER) {
    const int64_t x = x0 + grp;
    const bool on = x < hi;
    const int32_t i = on ? A.list[x].x : 0;
    const long long b = on ? A.off[i] : 0;
    const int d = on ? (int)(A.off[i + 1] - b) : 0;
    int32_t C = -1;
    long long w = 0;
    if (sub < d) {
      C = A.cl[A.adj[b + sub]];
      w = A.aw[b + sub];
    }
    const int32_t own = on ? A.cl[i] : -1;
    const long long ki = on ? A.k[i] : 0;
    const long long vol = C >= 0 ? A.vol[C] : 0;
    const int steps = (int)__reduce_max_sync(FULL, (unsigned)d);
    long long kic = 0;
    for (int t = 0; t < steps; ++t) {
      const int32_t Ct = __shfl_sync(FULL, C, grp * G + t);
      const long long wt = __shfl_sync(FULL, w, grp * G + t);
      if (Ct == C) kic += wt;
    }
    Cand best{0, -1};
    if (C >= 0 && C != own) best = Cand{(i128)A.W2 * kic - (i128)ki * vol, C};
    long long kia = C >= 0 && C == own ? kic : 0;  // the same in every lane of the own cluster
#pragma unroll
    for (int s = G / 2; s > 0; s >>= 1) {
      cand_better(best, shfl_cand(best, s));
      const long long o = __shfl_xor_sync(FULL, kia, s);
      kia = o > kia ? o : kia;
    }
    lv_emit(A, words, on && sub == 0 && lv_moves(A, i, kia, best), i, best.c);
  }
}

// The best other candidate and the own cluster's entry among slots first,
// first + step, ... of a table, which are cleared.  Four slots at a time: the
// volumes are gathers, whose latencies would follow one another (V-cycle with
// communities on 250,007 nodes and 1.35M pins: 38.1 -> 37.1 ms; eight at a time
// is slower again).
__device__ __forceinline__ void lv_take(const LvArgs& A, int32_t i, int32_t* keys,
                                        long long* vals, int slots, int first, int step,
                                        Cand& best, long long& kia) {
  constexpr int AT_ONCE = 4;
  const int32_t own = A.cl[i];
  const long long ki = A.k[i];
  best = Cand{0, -1};
  kia = 0;
  for (int s0 = first; s0 < slots; s0 += AT_ONCE * step) {
    int32_t C[AT_ONCE];
    long long kic[AT_ONCE], vol[AT_ONCE];
#pragma unroll
    for (int x = 0; x < AT_ONCE; ++x) {
      const int s = s0 + x * step;
      C[x] = s < slots ? keys[s] : LV_EMPTY;
    }
#pragma unroll
    for (int x = 0; x < AT_ONCE; ++x) {
      const int s = s0 + x * step;
      kic[x] = vol[x] = 0;
      if (C[x] == LV_EMPTY) continue;
      kic[x] = vals[s];
      vol[x] = A.vol[C[x]];
      keys[s] = LV_EMPTY;
      vals[s] = 0;
    }
#pragma unroll
    for (int x = 0; x < AT_ONCE; ++x) {
      if (C[x] == own) kia = kic[x];
      else if (C[x] != LV_EMPTY) cand_better(best, Cand{(i128)A.W2 * kic[x] - (i128)ki * vol[x], C[x]});
    }
  }
  warp_best(best);
  kia = warp_sum(kia);
}

// Part of a cluster among `parts` (its own hash: the table's picks the slot).
__device__ __forceinline__ int lv_part(int32_t C, int parts) {
  return (int)(((mix64((uint64_t)(uint32_t)C ^ 0xA5A5A5A500000000ull) >> 32) * (uint64_t)parts) >>
               32);
}

// The best of the block's candidates and the sum of its kia, in warp 0.
__device__ __forceinline__ void lv_block_best(Cand& best, long long& kia) {
  __shared__ unsigned long long s_lo[LV_WARPS];
  __shared__ long long s_hi[LV_WARPS], s_kia[LV_WARPS];
  __shared__ int32_t s_c[LV_WARPS];
  const int l = lane_id();
  if (l == 0) {
    s_lo[warp_in_block()] = (unsigned long long)best.s;
    s_hi[warp_in_block()] = (long long)(best.s >> 64);
    s_c[warp_in_block()] = best.c;
    s_kia[warp_in_block()] = kia;
  }
  __syncthreads();
  if (warp_in_block() == 0) {
    best = Cand{0, -1};
    kia = 0;
    if (l < LV_WARPS) {
      best = Cand{((i128)s_hi[l] << 64) | (i128)s_lo[l], s_c[l]};
      kia = s_kia[l];
    }
    warp_best(best);
    kia = warp_sum(kia);
  }
}

__device__ __forceinline__ void lv_write_part(const LvArgs& A, int32_t x, const Cand& best,
                                              long long kia) {
  A.parts[x] = PartBest{(unsigned long long)best.s, (long long)(best.s >> 64), kia, best.c, 0};
}

// Classes 3 and 4: the block rates the entry's vertex over all its edges,
// keeping the clusters of one part.
__device__ __forceinline__ void lv_block(const LvArgs& A, int32_t* words, int32_t x,
                                         int32_t* keys, long long* vals) {
  const int2 nd = A.list[x];
  const int32_t i = nd.x;
  const long long b = A.off[i], e = A.off[i + 1];
  int32_t parts;
  lv_class(e - b, A.huge_deg, parts);
  for (long long q = b + threadIdx.x; q < e; q += LV_THREADS) {
    const int32_t C = A.cl[A.adj[q]];
    if (parts > 1 && lv_part(C, parts) != nd.y) continue;
    if (!table_add(keys, vals, LV_BLOCK_SLOTS - 1, C, A.aw[q])) dev_fail(A.status, DEV_HASH_FULL);
  }
  __syncthreads();
  Cand best;
  long long kia;
  lv_take(A, i, keys, vals, LV_BLOCK_SLOTS, threadIdx.x, LV_THREADS, best, kia);
  lv_block_best(best, kia);
  if (warp_in_block() == 0) {
    if (parts == 1)
      lv_emit(A, words, lane_id() == 0 && lv_moves(A, i, kia, best), i, best.c);
    else if (lane_id() == 0)
      lv_write_part(A, x, best, kia);
  }
  __syncthreads();
}

// Class 5: the entry's chunk of edges, summed per cluster in the block's table,
// then added to the vertex's.  (Edge by edge, the atomics of a hub whose
// neighbours have joined few clusters would meet at those slots.)
__device__ __forceinline__ void lv_insert_chunk(const LvArgs& A, int32_t x, int32_t* keys,
                                                long long* vals) {
  const int2 nd = A.list[x];
  const HugeVertex h = A.huge[nd.x];
  const long long b = A.off[h.i] + (long long)nd.y * LV_CHUNK;
  const long long e = min(b + LV_CHUNK, A.off[h.i + 1]);
  for (long long q = b + threadIdx.x; q < e; q += LV_THREADS)
    if (!table_add(keys, vals, LV_CHUNK_SLOTS - 1, A.cl[A.adj[q]], A.aw[q]))
      dev_fail(A.status, DEV_HASH_FULL);
  __syncthreads();
  for (int s = threadIdx.x; s < LV_CHUNK_SLOTS; s += LV_THREADS) {
    const int32_t C = keys[s];
    if (C == LV_EMPTY) continue;
    if (!table_add(A.tkey + h.tab, A.tval + h.tab, (uint32_t)(h.slots - 1), C, vals[s]))
      dev_fail(A.status, DEV_HASH_FULL);
    keys[s] = LV_EMPTY;
    vals[s] = 0;
  }
  __syncthreads();
}

// Class 5, after a barrier: the best of the entry's piece of the table, which is
// cleared for the next sub-round.
__device__ __forceinline__ void lv_scan_piece(const LvArgs& A, int32_t x) {
  const int2 nd = A.list[x];
  const HugeVertex h = A.huge[nd.x];
  const unsigned long long lo = h.slots * (unsigned)nd.y / (unsigned)h.entries;
  const unsigned long long hi = h.slots * (unsigned)(nd.y + 1) / (unsigned)h.entries;
  const int32_t own = A.cl[h.i];
  const long long ki = A.k[h.i];
  Cand best{0, -1};
  long long kia = 0;
  for (unsigned long long s = h.tab + lo + threadIdx.x; s < h.tab + hi; s += LV_THREADS) {
    const int32_t C = __ldcg(A.tkey + s);
    if (C == LV_EMPTY) continue;
    const long long kic = __ldcg(A.tval + s);
    __stcg(A.tkey + s, LV_EMPTY);
    __stcg(A.tval + s, 0ll);
    if (C == own) kia = kic;
    else cand_better(best, Cand{(i128)A.W2 * kic - (i128)ki * A.vol[C], C});
  }
  warp_best(best);
  kia = warp_sum(kia);
  lv_block_best(best, kia);
  if (threadIdx.x == 0) lv_write_part(A, x, best, kia);
  __syncthreads();
}

// HUGE: the level has class 5 vertices.  Their code stays out of the kernel of the
// other levels, which its presence alone slows (V-cycle with communities on
// 250,007 nodes and 1.35M pins: 37.1 ms, 39.9 with one kernel for all levels).
template <bool HUGE>
__global__ void __launch_bounds__(LV_THREADS, 2) k_lv_run(const __grid_constant__ LvArgs A) {
  extern __shared__ __align__(16) unsigned char smem[];
  long long* vals = reinterpret_cast<long long*>(smem);
  int32_t* keys = reinterpret_cast<int32_t*>(vals + LV_BLOCK_SLOTS);
  int32_t* s_off = keys + LV_BLOCK_SLOTS;
  const int nkeys = LV_CLASSES * A.S;
  int32_t* s_hist = s_off + nkeys + 1;
  int32_t* s_base = s_hist + nkeys;
  const int lane = lane_id(), wv = warp_in_block();
  const int64_t gw = (int64_t)wv * gridDim.x + blockIdx.x, NW = (int64_t)gridDim.x * LV_WARPS;
  // the warps' tables are consecutive pieces of the block's
  int32_t* wkeys = keys + wv * LV_SLOTS;
  long long* wvals = vals + wv * LV_SLOTS;
  for (int x = threadIdx.x; x < LV_BLOCK_SLOTS; x += LV_THREADS) {
    keys[x] = LV_EMPTY;
    vals[x] = 0;
  }
  __syncthreads();
  unsigned gen = 0;
  auto sync = [&]() { return grid_sync(false, A.barrier, A.status, gen); };
  unsigned long long before = 0;
  int par = 0, rounds = 0;
  for (int round = 0; round < LV_ROUNDS; ++round) {
    lv_list(A, round, false, s_off, s_hist, s_base);
    if (!sync()) return;
    lv_offsets_of(A, s_off);
    lv_list(A, round, true, s_off, s_hist, s_base);
    if (!sync()) return;
    for (int s = 0; s < A.S; ++s, par ^= 1) {
      int32_t* words = A.words + par * LV_WORDS;
      if (blockIdx.x == 0 && threadIdx.x < LV_WORDS) A.words[(par ^ 1) * LV_WORDS + threadIdx.x] = 0;
      if (s == 0)  // the lists are built: clear their counters for the next round
        for (int x = blockIdx.x * LV_THREADS + threadIdx.x; x < nkeys; x += gridDim.x * LV_THREADS) {
          A.cnt[x] = 0;
          A.fill[x] = 0;
          if (x < A.S) A.tabfill[x] = 0;
          if (x == 0) *A.nhuge = 0;
        }
      const int32_t* at = s_off + LV_CLASSES * s;
      // ---- decisions from the state at the start of the sub-round
      if constexpr (HUGE)
        for (int32_t x = at[5] + (int32_t)blockIdx.x; x < at[6]; x += gridDim.x)
          lv_insert_chunk(A, x, keys, vals);
      // classes 4 and 3
      for (int32_t x = at[5] - 1 - (int32_t)blockIdx.x; x >= at[3]; x -= gridDim.x)
        lv_block(A, words, x, keys, vals);
      for (int64_t x = at[2] + gw; x < at[3]; x += NW) {
        const int32_t i = A.list[x].x;
        const long long b = A.off[i], e = A.off[i + 1];
        for (long long q = b + lane; q < e; q += 32)
          if (!table_add(wkeys, wvals, LV_SLOTS - 1, A.cl[A.adj[q]], A.aw[q]))
            dev_fail(A.status, DEV_HASH_FULL);
        __syncwarp();
        Cand best;
        long long kia;
        lv_take(A, i, wkeys, wvals, LV_SLOTS, lane, 32, best, kia);
        lv_emit(A, words, lane == 0 && lv_moves(A, i, kia, best), i, best.c);
        __syncwarp();
      }
      lv_lanes<LV_LANES>(A, words, at[1], at[2], gw, NW);
      lv_lanes<LV_GROUP>(A, words, at[0], at[1], NW - 1 - gw, NW);
      __syncwarp();
      if (!sync()) return;
      if constexpr (HUGE) {
        if (at[6] > at[5]) {
          for (int32_t x = at[5] + (int32_t)blockIdx.x; x < at[6]; x += gridDim.x)
            lv_scan_piece(A, x);
          if (!sync()) return;
        }
      }
      if (at[6] > at[4]) {
        for (int64_t x = at[4] + gw; x < at[6]; x += NW) {
          const int2 nd = A.list[x];
          if (nd.y != 0) continue;  // the first entry of a vertex combines
          int32_t i = nd.x, parts;
          if (!HUGE || x < at[5]) {
            lv_class(A.off[i + 1] - A.off[i], A.huge_deg, parts);
          } else {
            parts = A.huge[nd.x].entries;
            i = A.huge[nd.x].i;
          }
          Cand best{0, -1};
          long long kia = 0;
          for (int t = lane; t < parts; t += 32) {
            const PartBest pb = A.parts[x + t];
            cand_better(best, Cand{((i128)pb.hi << 64) | (i128)pb.lo, pb.c});
            kia += pb.kia;
          }
          warp_best(best);
          kia = warp_sum(kia);
          lv_emit(A, words, lane == 0 && lv_moves(A, i, kia, best), i, best.c);
        }
        if (!sync()) return;
      }
      // ---- moves: clusters and integer volumes
      const int32_t nm = __ldcg(words + LV_MOVES);
      for (int32_t x = blockIdx.x * LV_THREADS + threadIdx.x; x < nm; x += gridDim.x * LV_THREADS) {
        const int2 mv = A.mv[x];
        const long long ki = A.k[mv.x];
        atomic_add_i64(&A.vol[A.cl[mv.x]], -ki);
        atomic_add_i64(&A.vol[mv.y], ki);
        A.cl[mv.x] = mv.y;
      }
      if (blockIdx.x == 0 && threadIdx.x == 0 && nm)
        atomicAdd(&A.res[LR_MOVED], (unsigned long long)nm);
      if (!sync()) return;
    }
    rounds = round + 1;
    const unsigned long long moved = __ldcg(A.res + LR_MOVED);
    if (100 * (long long)(moved - before) < A.V) break;
    before = moved;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) A.res[LR_ROUNDS] = (unsigned long long)rounds;
}

using LvKernel = void (*)(LvArgs);

size_t lv_smem(int S) {
  return (size_t)LV_BLOCK_SLOTS * 12 + (3 * (size_t)LV_CLASSES * S + 1) * sizeof(int32_t);
}

// ------------------------------------------------------------ aggregation

__global__ void k_lv_used(const int32_t* __restrict__ cl, int64_t V, int32_t* __restrict__ flag) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < V;
       i += (int64_t)gridDim.x * blockDim.x)
    flag[cl[i]] = 1;
}

// cv[i] = coarse vertex of i; per coarse vertex the sum of its members' degrees
// in the edge lists (a bound on its coarse degree) and of their self-loop
// weights.
__global__ void k_lv_coarse_of(const int32_t* __restrict__ cl, const int32_t* __restrict__ cid,
                               int64_t V, const long long* __restrict__ off,
                               const long long* __restrict__ self, int32_t* __restrict__ cv,
                               long long* __restrict__ bound, long long* __restrict__ self2) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < V;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t c = cid[cl[i]];
    cv[i] = c;
    const long long d = off[i + 1] - off[i], sl = self[i];
    if (d) atomic_add_i64(&bound[c], d);
    if (sl) atomic_add_i64(&self2[c], sl);
  }
}

// Table sizes (powers of two >= 2 bound + 2) and the largest.
__global__ void k_lv_table_sizes(const long long* __restrict__ bound, int32_t V2,
                                 int64_t* __restrict__ tsz, unsigned long long* __restrict__ most) {
  unsigned long long mx = 0;
  for (int32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < V2; c += gridDim.x * blockDim.x) {
    long long s = 4;
    while (s < 2 * bound[c] + 2) s <<= 1;
    tsz[c] = s;
    mx = (unsigned long long)s > mx ? (unsigned long long)s : mx;
  }
  mx = warp_max(mx);
  if (lane_id() == 0 && mx) atomicMax(most, mx);
}

// The largest x in [lo, hi] with first[x] <= y (first non-decreasing).
template <typename I>
__device__ __forceinline__ I owner_in(const long long* first, I lo, I hi, long long y) {
  while (lo < hi) {
    const I mid = lo + (hi - lo + 1) / 2;
    if (first[mid] <= y) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Positions [t0, t1) of a tile and the range of owners that can hold them: two
// searches per block of LV_TILE positions instead of one per position (19
// dependent loads each).
constexpr int LV_TILE = 2048;
struct OwnerTile {
  long long t0, t1;
  int64_t lo, hi;
};
__device__ __forceinline__ OwnerTile owner_tile(const long long* first, int64_t owners,
                                                long long tile, long long total, int64_t* s_own) {
  OwnerTile o;
  o.t0 = tile * LV_TILE;
  o.t1 = o.t0 + LV_TILE < total ? o.t0 + LV_TILE : total;
  __syncthreads();
  if (threadIdx.x < 2)
    s_own[threadIdx.x] = owner_in<int64_t>(first, 0, owners - 1, threadIdx.x ? o.t1 - 1 : o.t0);
  __syncthreads();
  o.lo = s_own[0];
  o.hi = s_own[1];
  return o;
}

// One thread per edge: an edge to another coarse vertex is added to the coarse
// vertex's table, an edge inside it to its internal weight.
__global__ void k_lv_agg_insert(int64_t V, long long E, const int32_t* __restrict__ cv,
                                const long long* __restrict__ off, const int32_t* __restrict__ adj,
                                const long long* __restrict__ aw, const long long* __restrict__ toff,
                                int32_t* __restrict__ tkey, long long* __restrict__ tval,
                                long long* __restrict__ internal, int32_t* status) {
  __shared__ int64_t s_own[2];
  for (long long tile = blockIdx.x; tile * LV_TILE < E; tile += gridDim.x) {
    const OwnerTile o = owner_tile(off, V, tile, E, s_own);
    for (long long q = o.t0 + threadIdx.x; q < o.t1; q += blockDim.x) {
      const int64_t i = owner_in<int64_t>(off, o.lo, o.hi, q);
      const int32_t ci = cv[i], cj = cv[adj[q]];
      if (ci == cj) {
        atomic_add_i64(&internal[ci], aw[q]);
      } else {
        const long long tb = toff[ci];
        const uint32_t mask = (uint32_t)(toff[ci + 1] - tb) - 1;
        if (!table_add(tkey + tb, tval + tb, mask, cj, aw[q])) dev_fail(status, DEV_HASH_FULL);
      }
    }
  }
}

// Distinct neighbours of every coarse vertex: one thread per table slot over
// all tables (a hub's table is spread over the grid), lanes of a warp that
// count for the same coarse vertex share one atomic.
__global__ void k_lv_agg_count(const long long* __restrict__ toff, int32_t V2,
                               const int32_t* __restrict__ tkey, int32_t* __restrict__ deg2) {
  __shared__ int64_t s_own[2];
  const long long total = toff[V2];
  for (long long tile = blockIdx.x; tile * LV_TILE < total; tile += gridDim.x) {
    const OwnerTile o = owner_tile(toff, V2, tile, total, s_own);
    for (long long b = o.t0 + (threadIdx.x & ~31); b < o.t1; b += blockDim.x) {
      const long long s = b + lane_id();
      const bool used = s < o.t1 && tkey[s] != LV_EMPTY;
      const int32_t c = used ? (int32_t)owner_in<int64_t>(toff, o.lo, o.hi, s) : -1;
      warp_claim_slot(deg2, c, __ballot_sync(FULL, used));
    }
  }
}

// Writes the coarse edge lists (order inside a list unspecified), again one
// thread per table slot; positions come from a per-vertex cursor claimed
// once per warp and coarse vertex.
__global__ void k_lv_agg_write(const long long* __restrict__ toff, int32_t V2,
                               const int32_t* __restrict__ tkey, const long long* __restrict__ tval,
                               const long long* __restrict__ off2, int32_t* __restrict__ adj2,
                               long long* __restrict__ aw2, int32_t* __restrict__ fill) {
  __shared__ int64_t s_own[2];
  const long long total = toff[V2];
  for (long long tile = blockIdx.x; tile * LV_TILE < total; tile += gridDim.x) {
    const OwnerTile o = owner_tile(toff, V2, tile, total, s_own);
    for (long long b = o.t0 + (threadIdx.x & ~31); b < o.t1; b += blockDim.x) {
      const long long s = b + lane_id();
      const int32_t key = s < o.t1 ? tkey[s] : LV_EMPTY;
      const bool used = key != LV_EMPTY;
      const int32_t c = used ? (int32_t)owner_in<int64_t>(toff, o.lo, o.hi, s) : -1;
      const int32_t slot = warp_claim_slot(fill, c, __ballot_sync(FULL, used));
      if (used) {
        const long long pos = off2[c] + slot;
        adj2[pos] = key;
        aw2[pos] = tval[s];
      }
    }
  }
}

// Coarse self-loop weights: own self loops plus half the internal weight
// (every internal edge was seen from both of its ends).
__global__ void k_lv_self2(int32_t V2, const long long* __restrict__ internal,
                           long long* __restrict__ self2) {
  for (int32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < V2; c += gridDim.x * blockDim.x)
    self2[c] += internal[c] / 2;
}

__global__ void k_lv_vmap(int32_t* __restrict__ vmap, int32_t n, const int32_t* __restrict__ cv) {
  for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
    vmap[v] = cv[vmap[v]];
}

// Distinct community ids among the nodes.
__global__ void k_lv_mark(const int32_t* __restrict__ comm, int32_t n, int32_t* __restrict__ flag) {
  for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
    flag[comm[v]] = 1;
}

// ------------------------------------------------------------ host

struct LvGraph {
  int64_t V = 0, E = 0;
  int huge = LV_HUGE;  // class 5 above this degree
  int64_t slots = 0;   // of the class 5 tables of a sub-round
  DBuf<long long> off, aw, self, k;
  DBuf<int32_t> adj;
};

void lv_degrees(const Ctx& cx, LvGraph& g, uint64_t seed, int level, int S, long long* W2) {
  g.k.alloc(&cx.alloc, (size_t)std::max<int64_t>(g.V, 1));
  DBuf<unsigned long long> sums;
  sums.alloc(&cx.alloc, LD_SLOTS + (size_t)LV_ROUNDS * S);
  HG_CUDA(cudaMemsetAsync(sums.p, 0, sums.bytes(), cx.stream));
  k_lv_degrees<<<grid_for(g.V, 8, cx.num_sms, 16), 256, 0, cx.stream>>>(
      g.off.p, g.aw.p, g.self.p, g.V, seed, level, S, g.huge, g.k.p, sums.p);
  check_launch("lv_degrees");
  unsigned long long h[LD_SLOTS];
  read_back(cx, h, sums.p, sizeof(h));
  *W2 = (long long)h[LD_TOTAL];
  g.slots = (int64_t)h[LD_MOST];
}

// Aggregates the clustering cl of g into the next level's graph; cv[i] =
// coarse vertex of i.
void lv_aggregate(const Ctx& cx, const LvGraph& g, const int32_t* cl, LvGraph& out,
                  DBuf<int32_t>& cv) {
  const int64_t V = g.V;
  const int gV = grid_for(V, 256, cx.num_sms, 8);
  DBuf<int32_t> flag, cid;
  flag.alloc(&cx.alloc, (size_t)V + 1);
  cid.alloc(&cx.alloc, (size_t)V + 1);
  HG_CUDA(cudaMemsetAsync(flag.p, 0, flag.bytes(), cx.stream));
  k_lv_used<<<gV, 256, 0, cx.stream>>>(cl, V, flag.p);
  check_launch("lv_used");
  scan_exclusive_i32(cx, flag.p, cid.p, V, cid.p + V);
  const int32_t V2 = read_i32(cx, cid.p + V);
  cv.alloc(&cx.alloc, (size_t)V);
  DBuf<long long> bound, tsz, toff, internal;
  DBuf<unsigned long long> most;
  bound.alloc(&cx.alloc, (size_t)V2 + 1);
  tsz.alloc(&cx.alloc, (size_t)V2 + 1);
  toff.alloc(&cx.alloc, (size_t)V2 + 1);
  internal.alloc(&cx.alloc, (size_t)V2 + 1);
  most.alloc(&cx.alloc, 1);
  out.self.alloc(&cx.alloc, (size_t)V2 + 1);
  HG_CUDA(cudaMemsetAsync(bound.p, 0, bound.bytes(), cx.stream));
  HG_CUDA(cudaMemsetAsync(out.self.p, 0, out.self.bytes(), cx.stream));
  HG_CUDA(cudaMemsetAsync(internal.p, 0, internal.bytes(), cx.stream));
  HG_CUDA(cudaMemsetAsync(most.p, 0, most.bytes(), cx.stream));
  k_lv_coarse_of<<<gV, 256, 0, cx.stream>>>(cl, cid.p, V, g.off.p, g.self.p, cv.p, bound.p,
                                            out.self.p);
  check_launch("lv_coarse_of");
  k_lv_table_sizes<<<grid_for(V2, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(
      bound.p, V2, reinterpret_cast<int64_t*>(tsz.p), most.p);
  check_launch("lv_table_sizes");
  scan_exclusive_i64(cx, reinterpret_cast<const int64_t*>(tsz.p),
                     reinterpret_cast<int64_t*>(toff.p), V2,
                     reinterpret_cast<int64_t*>(toff.p) + V2);
  long long tslots = 0;
  unsigned long long hmost = 0;
  wait_stream(cx);
  HG_CUDA(cudaMemcpyAsync(&tslots, toff.p + V2, sizeof(tslots), cudaMemcpyDeviceToHost, cx.stream));
  HG_CUDA(cudaMemcpyAsync(&hmost, most.p, sizeof(hmost), cudaMemcpyDeviceToHost, cx.stream));
  check_status(cx);
  if (hmost > (1ull << 31)) throw HgError(HG_ERR_UNSUPPORTED, "coarse vertex degree too large");
  DBuf<int32_t> tkey;
  DBuf<long long> tval;
  tkey.alloc(&cx.alloc, (size_t)std::max<long long>(tslots, 1));
  tval.alloc(&cx.alloc, (size_t)std::max<long long>(tslots, 1));
  HG_CUDA(cudaMemsetAsync(tkey.p, 0xff, tkey.bytes(), cx.stream));
  HG_CUDA(cudaMemsetAsync(tval.p, 0, tval.bytes(), cx.stream));
  k_lv_agg_insert<<<grid_for(g.E, LV_TILE, cx.num_sms, 8), 256, 0, cx.stream>>>(
      V, g.E, cv.p, g.off.p, g.adj.p, g.aw.p, toff.p, tkey.p, tval.p, internal.p, cx.d_status);
  check_launch("lv_agg_insert");
  DBuf<int32_t> deg2, fill2;
  deg2.alloc(&cx.alloc, (size_t)V2 + 1);
  fill2.alloc(&cx.alloc, (size_t)V2 + 1);
  HG_CUDA(cudaMemsetAsync(fill2.p, 0, fill2.bytes(), cx.stream));
  HG_CUDA(cudaMemsetAsync(deg2.p, 0, deg2.bytes(), cx.stream));
  const int gT = grid_for(tslots, LV_TILE, cx.num_sms, 8);
  k_lv_agg_count<<<gT, 256, 0, cx.stream>>>(toff.p, V2, tkey.p, deg2.p);
  check_launch("lv_agg_count");
  out.V = V2;
  out.off.alloc(&cx.alloc, (size_t)V2 + 1);
  scan_exclusive_i32_to_i64(cx, deg2.p, reinterpret_cast<int64_t*>(out.off.p), V2,
                            reinterpret_cast<int64_t*>(out.off.p) + V2);
  out.E = read_i64(cx, reinterpret_cast<const int64_t*>(out.off.p) + V2);
  out.adj.alloc(&cx.alloc, (size_t)std::max<int64_t>(out.E, 1));
  out.aw.alloc(&cx.alloc, (size_t)std::max<int64_t>(out.E, 1));
  k_lv_agg_write<<<gT, 256, 0, cx.stream>>>(toff.p, V2, tkey.p, tval.p, out.off.p, out.adj.p,
                                          out.aw.p, fill2.p);
  check_launch("lv_agg_write");
  k_lv_self2<<<grid_for(V2, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(V2, internal.p, out.self.p);
  check_launch("lv_self2");
  if (cx.launches) *cx.launches += 14;
}

// One Louvain level on g (clusters start as singletons).  Returns the moves, or -1
// when the table of a part was full.
int64_t lv_local_moving(const Ctx& cx, const LvGraph& g, long long W2, int S, uint64_t seed,
                        int level, DBuf<int32_t>& cl, LouvainCounters& lc) {
  const int64_t V = g.V;
  DBuf<long long> vol;
  cl.alloc(&cx.alloc, (size_t)std::max<int64_t>(V, 1));
  vol.alloc(&cx.alloc, (size_t)std::max<int64_t>(V, 1));
  const int gV = grid_for(V, 256, cx.num_sms, 8);
  k_lv_init<<<gV, 256, 0, cx.stream>>>(V, g.k.p, cl.p, vol.p);
  check_launch("lv_init");
  const size_t nkeys = (size_t)LV_CLASSES * S;
  // a list entry per vertex, and one per further part or chunk of a large vertex
  const size_t entries = (size_t)V + (size_t)(g.E / std::min(LV_PART, LV_CHUNK)) + 1;
  DBuf<HugeVertex> huge;
  DBuf<int32_t> tkey;
  DBuf<long long> tval;
  huge.alloc(&cx.alloc, g.slots ? (size_t)(g.E / g.huge) + 1 : 0);
  tkey.alloc(&cx.alloc, (size_t)g.slots);
  tval.alloc(&cx.alloc, (size_t)g.slots);
  if (g.slots) {
    HG_CUDA(cudaMemsetAsync(tkey.p, 0xff, tkey.bytes(), cx.stream));
    HG_CUDA(cudaMemsetAsync(tval.p, 0, tval.bytes(), cx.stream));
  }
  DBuf<int2> list, mv;
  DBuf<PartBest> parts;
  DBuf<unsigned long long> zero;  // results, table slots given out, then 32-bit counters
  list.alloc(&cx.alloc, entries);
  mv.alloc(&cx.alloc, (size_t)V + 1);
  parts.alloc(&cx.alloc, entries);
  zero.alloc(&cx.alloc, LR_LV_WORDS + (size_t)S + nkeys + LV_WORDS + 2);
  HG_CUDA(cudaMemsetAsync(zero.p, 0, zero.bytes(), cx.stream));
  int32_t* z = reinterpret_cast<int32_t*>(zero.p + LR_LV_WORDS + S);
  LvArgs A{};
  A.off = g.off.p;
  A.adj = g.adj.p;
  A.aw = g.aw.p;
  A.k = g.k.p;
  A.cl = cl.p;
  A.vol = vol.p;
  A.W2 = W2;
  A.V = V;
  A.seed = seed;
  A.level = level;
  A.S = S;
  A.huge_deg = g.huge;
  A.list = list.p;
  A.cnt = z;
  A.fill = z + nkeys;
  A.words = z + 2 * nkeys;
  A.barrier = reinterpret_cast<unsigned*>(z + 2 * nkeys + 2 * LV_WORDS);
  A.nhuge = z + 2 * nkeys + 2 * LV_WORDS + 2;
  A.tabfill = zero.p + LR_LV_WORDS;
  A.huge = huge.p;
  A.tkey = tkey.p;
  A.tval = tval.p;
  A.mv = mv.p;
  A.parts = parts.p;
  A.res = zero.p;
  A.status = cx.d_status;
  const LvKernel kernel = g.slots ? k_lv_run<true> : k_lv_run<false>;
  const size_t smem = lv_smem(S);
  prepare_kernel(cx, kernel, lv_smem(256));
  int per_sm = 0;
  HG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, LV_THREADS, smem));
  if (per_sm < 1) throw HgError(HG_ERR_CUDA, "local moving does not fit an SM");
  // a block per 16 vertices or 256 edges of a sub-round (coarse levels: heavy
  // vertices take a block each); four times that, and at most half the chip, when
  // the call shares the GPU with others (inflight.cuh)
  const int64_t share = cx.shares_gpu() ? 4 : 1;
  const int64_t need =
      std::max<int64_t>(V / (S * 16 * share), g.E / (S * 256 * share)) + 1;
  const int blocks =
      (int)std::min<int64_t>(need, (int64_t)cx.num_sms * std::min(per_sm, share == 1 ? 2 : 1));
  launch_persistent(cx, kernel, blocks, LV_THREADS, smem, false, A);
  lc.launches += 1;
  unsigned long long hres[LR_LV_WORDS];
  const int32_t status = read_status(cx, hres, A.res, sizeof(hres));
  if (status == DEV_HASH_FULL && g.huge > LV_BLOCK) {
    HG_CUDA(cudaMemsetAsync(cx.d_status, 0, sizeof(int32_t), cx.stream));
    return -1;
  }
  throw_status(cx, status);
  lc.rounds += (int64_t)hres[LR_ROUNDS];
  return (int64_t)hres[LR_MOVED];
}

}  // namespace

int32_t detect_communities(const Ctx& cx, const Level& L, int S, uint64_t seed,
                           DBuf<int32_t>& comm, LouvainCounters& lc) {
  const int32_t n = L.n, m = L.m;
  const int64_t p = L.p;
  comm.alloc(&cx.alloc, (size_t)n);
  iota_i32(cx, comm.p, n);  // vmap: node -> vertex of the current level
  if (p == 0) return n;
  LvGraph g;
  g.V = (int64_t)n + m;
  g.E = 2 * p;
  g.off.alloc(&cx.alloc, (size_t)g.V + 1);
  g.adj.alloc(&cx.alloc, (size_t)g.E);
  g.aw.alloc(&cx.alloc, (size_t)g.E);
  g.self.alloc(&cx.alloc, (size_t)g.V);
  HG_CUDA(cudaMemsetAsync(g.self.p, 0, g.self.bytes(), cx.stream));
  k_lv_offsets<<<grid_for(g.V + 1, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(
      L.ioff.p, L.eoff.p, n, m, p, g.off.p);
  check_launch("lv_offsets");
  {
    DBuf<int32_t> tiles;
    tiles.alloc(&cx.alloc, (size_t)num_pin_tiles(p) + 1);
    build_tile_index(cx, L.eoff.p, L.m, p, tiles.p);
    k_lv_node_edges<<<grid_for(p, 256, cx.num_sms, 16), 256, 0, cx.stream>>>(
        L.eoff.p, L.w.p, L.inets.p, n, p, g.adj.p, g.aw.p);
    check_launch("lv_node_edges");
    k_lv_net_edges<<<grid_for(num_pin_tiles(p), 1, cx.num_sms, 8), PIN_TILE_THREADS, 0,
                     cx.stream>>>(L.eoff.p, L.pins.p, L.w.p, tiles.p, L.m, p, g.adj.p + p,
                                  g.aw.p + p);
    check_launch("lv_net_edges");
  }
  long long W2 = 0;
  lv_degrees(cx, g, seed, 0, S, &W2);
  for (int level = 0; level < LV_LEVELS; ++level) {
    DBuf<int32_t> cl;
    int64_t moves = lv_local_moving(cx, g, W2, S, seed, level, cl, lc);
    if (moves < 0) {  // once more with a table for every vertex above LV_BLOCK
      g.huge = LV_BLOCK;
      long long same = 0;
      lv_degrees(cx, g, seed, level, S, &same);
      moves = lv_local_moving(cx, g, W2, S, seed, level, cl, lc);
    }
    lc.moves += moves;
    if (moves == 0) break;
    lc.levels = level + 1;
    LvGraph next;
    DBuf<int32_t> cv;
    lv_aggregate(cx, g, cl.p, next, cv);
    k_lv_vmap<<<grid_for(n, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(comm.p, n, cv.p);
    check_launch("lv_vmap");
    const bool shrank = next.V < g.V;
    long long W2n = 0;
    lv_degrees(cx, next, seed, level + 1, S, &W2n);
    g = std::move(next);
    if (!shrank) break;
  }
  check_status(cx);
  // number of distinct communities among the nodes
  DBuf<int32_t> flag;
  flag.alloc(&cx.alloc, (size_t)g.V + 1);
  HG_CUDA(cudaMemsetAsync(flag.p, 0, flag.bytes(), cx.stream));
  k_lv_mark<<<grid_for(n, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(comm.p, n, flag.p);
  check_launch("lv_mark");
  scan_exclusive_i32(cx, flag.p, flag.p, g.V, flag.p + g.V);
  return read_i32(cx, flag.p + g.V);
}

}  // namespace hgk
