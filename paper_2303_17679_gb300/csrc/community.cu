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
// int64 self-loop weights, degrees k and volumes.  Per round the vertices
// are listed by (sub-round, class): vertices of at most 8 (32) edges are decided
// by a group of eight lanes (a warp) that holds one edge per lane and sums the
// edges of a cluster by exchanging them; up to LV_SMALL edges by one warp with
// a shared-memory table of the neighbouring clusters; the rest insert their
// edges into per-vertex tables in global memory with one thread per edge over
// the whole grid, then one block per vertex takes the best entry.  Aggregation
// uses the same global tables, one per coarse vertex.
// What bounds it: 16 dependent sub-rounds of gathers per round, some 25 rounds.
// Most vertices have a handful of edges (a table of 512 slots, cleared and
// scanned per vertex, cost more than they did), and the host reads only the
// class boundaries of a round (copying the table offsets of all vertices took
// over a millisecond per round).
#include <algorithm>
#include <mutex>

#include "common.cuh"

namespace hgk {

namespace {

constexpr int LV_ROUNDS = 5;
constexpr int LV_LEVELS = 32;
constexpr int LV_CLASSES = 4;
constexpr int LV_GROUP = 8;            // class 0: degree <= 8, eight lanes per vertex
constexpr int LV_LANES = 32;           // class 1: degree <= 32, a warp per vertex
constexpr int LV_SMALL = 256;          // class 2: degree <= 256, a warp and a shared table
constexpr int LV_SLOTS = 2 * LV_SMALL;  // shared slots per warp (load <= 1/2)
constexpr int LV_WARPS = 8;
constexpr int LV_ARGMAX_THREADS = 256;
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
// One thread per incidence j = (v, e), q = ipin[j] the pin position.
__global__ void k_lv_bipartite(const int32_t* __restrict__ eoff, const int32_t* __restrict__ pins,
                               const int32_t* __restrict__ w, const int32_t* __restrict__ inets,
                               const int32_t* __restrict__ ipin, int32_t n, int64_t p,
                               int32_t* __restrict__ adj, long long* __restrict__ aw) {
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < p;
       j += (int64_t)gridDim.x * blockDim.x) {
    const int32_t e = inets[j];
    const int32_t q = ipin[j];
    const int32_t size = eoff[e + 1] - eoff[e];
    const long long we = (long long)(((unsigned long long)w[e] << 20) / (unsigned long long)size);
    adj[j] = n + e;
    aw[j] = we;
    adj[p + q] = pins[q];
    aw[p + q] = we;
  }
}

__global__ void k_lv_offsets(const int32_t* __restrict__ ioff, const int32_t* __restrict__ eoff,
                             int32_t n, int32_t m, int64_t p, long long* __restrict__ off) {
  const int64_t V = (int64_t)n + m;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= V;
       i += (int64_t)gridDim.x * blockDim.x)
    off[i] = i <= n ? (long long)ioff[i] : (long long)(p + eoff[i - n]);
}

// k_i = 2 self_i + sum of i's edge weights (a warp per vertex); W2 = sum k_i.
__global__ void k_lv_degrees(const long long* __restrict__ off, const long long* __restrict__ aw,
                             const long long* __restrict__ self, int64_t V,
                             long long* __restrict__ k, unsigned long long* __restrict__ total) {
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  long long acc = 0;
  for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < V; i += nw) {
    long long s = 0;
    for (long long q = off[i] + lane_id(); q < off[i + 1]; q += 32) s += aw[q];
    s = warp_sum(s);
    s += 2 * self[i];
    if (lane_id() == 0) k[i] = s;
    acc += s;
  }
  if (lane_id() == 0 && acc) atomicAdd(total, (unsigned long long)acc);
}

__global__ void k_lv_init(int64_t V, const long long* __restrict__ k, int32_t* __restrict__ cl,
                          long long* __restrict__ vol) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < V;
       i += (int64_t)gridDim.x * blockDim.x) {
    cl[i] = (int32_t)i;
    vol[i] = k[i];
  }
}

// ------------------------------------------------------------ lists

// key = sub-round * LV_CLASSES + class of every vertex with at least one edge.
__device__ __forceinline__ int lv_key(const long long* off, uint64_t seed, int level, int round,
                                      int64_t i, int S) {
  const long long deg = off[i + 1] - off[i];
  if (deg == 0) return -1;  // no neighbouring cluster: never moves
  const int cls = deg <= LV_GROUP ? 0 : deg <= LV_LANES ? 1 : deg <= LV_SMALL ? 2 : 3;
  return subround_louvain(seed, level, round, i, S) * LV_CLASSES + cls;
}

__global__ void k_lv_count(const long long* __restrict__ off, int64_t V, uint64_t seed, int level,
                           int round, int S, int32_t* __restrict__ cnt) {
  extern __shared__ int32_t s_cnt[];
  for (int i = threadIdx.x; i < LV_CLASSES * S; i += blockDim.x) s_cnt[i] = 0;
  __syncthreads();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < V;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int key = lv_key(off, seed, level, round, i, S);
    if (key >= 0) atomicAdd(&s_cnt[key], 1);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < LV_CLASSES * S; i += blockDim.x)
    if (s_cnt[i]) atomicAdd(&cnt[i], s_cnt[i]);
}

// Scatters vertices by key; the list order inside a key is unspecified
// (every later step is a set operation or an integer sum).
__global__ void k_lv_scatter(const long long* __restrict__ off, int64_t V, uint64_t seed,
                             int level, int round, int S, const int32_t* __restrict__ koff,
                             int32_t* __restrict__ fill, int32_t* __restrict__ list) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); b < V; b += stride) {
    const int64_t i = b + lane_id();
    const bool valid = i < V;
    const int key = valid ? lv_key(off, seed, level, round, i, S) : -1;
    const int32_t slot = warp_claim_slot(fill, key, __ballot_sync(FULL, valid));
    if (slot >= 0) list[koff[key] + slot] = (int32_t)i;
  }
}

// Degrees and global table sizes (power of two >= 2 deg + 2) of the vertices
// that need a table along the list of *listed <= cap vertices (zeros after it
// and for the others).
__global__ void k_lv_list_sizes(const int32_t* __restrict__ list, const int32_t* __restrict__ listed,
                                int32_t cap, const long long* __restrict__ off,
                                int32_t* __restrict__ deg, int32_t* __restrict__ tsize) {
  const int32_t cnt = *listed;
  for (int32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < cap; x += gridDim.x * blockDim.x) {
    int32_t d = 0, t = 0;
    if (x < cnt) {
      const int32_t i = list[x];
      d = (int32_t)(off[i + 1] - off[i]);
      if (d > LV_SMALL) {
        // at most 2^30 slots: a larger vertex fills its table, which the
        // insertion reports as a full table
        int64_t c = 4;
        while (c < 2 * (int64_t)d + 2 && c < (1ll << 30)) c <<= 1;
        t = (int32_t)c;
      }
    }
    deg[x] = d;
    tsize[x] = t;
  }
}

// The class boundaries of a round and the table offsets there.
__global__ void k_lv_bounds(const int32_t* __restrict__ koff, int nkeys,
                            const long long* __restrict__ toff, long long* __restrict__ out) {
  for (int i = threadIdx.x; i <= nkeys; i += blockDim.x) {
    out[i] = koff[i];
    out[nkeys + 1 + i] = toff[koff[i]];
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

struct LvArgs {
  const long long* off;
  const int32_t* adj;
  const long long* aw;
  const long long* k;
  const int32_t* cl;
  const long long* vol;
  long long W2;
  const int32_t* list;
  int32_t* mv_v;
  int32_t* mv_to;
  int32_t* words;  // [0] moves of the sub-round
  int32_t* status;
};

// The move of vertex i from its own cluster's entry kia and the best other
// candidate: moves iff s(best) > s(own).
__device__ __forceinline__ void lv_emit(const LvArgs& A, int32_t i, long long kia, const Cand& best) {
  const int32_t own = A.cl[i];
  const long long ki = A.k[i];
  const i128 s_own = (i128)A.W2 * kia - (i128)ki * (A.vol[own] - ki);
  if (best.c >= 0 && best.s > s_own) {
    const int32_t slot = atomicAdd(&A.words[0], 1);
    A.mv_v[slot] = i;
    A.mv_to[slot] = best.c;
  }
}

// Classes 0 and 1: G lanes per vertex of at most G edges, one edge per lane.
// Every lane sums the edges of its own cluster (equal lanes hold equal
// candidates); the groups of a warp stay in step.
template <int G>
__global__ void __launch_bounds__(LV_WARPS * 32) k_lv_lanes(LvArgs A, int32_t lo, int32_t hi) {
  constexpr int PER = 32 / G;
  const int lane = lane_id(), sub = lane % G, grp = lane / G;
  const int32_t stride = gridDim.x * LV_WARPS * PER;
  for (int32_t x0 = lo + (blockIdx.x * LV_WARPS + warp_in_block()) * PER; x0 < hi; x0 += stride) {
    const int32_t x = x0 + grp;
    const bool on = x < hi;
    const int32_t i = on ? A.list[x] : 0;
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
    const int steps = __reduce_max_sync(FULL, (unsigned)d);
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
    bool moves = false;
    if (on && sub == 0 && best.c >= 0)
      moves = best.s > (i128)A.W2 * kia - (i128)ki * (A.vol[own] - ki);
    const unsigned who = __ballot_sync(FULL, moves);
    if (who) {
      int32_t slot = 0;
      if (lane == 0) slot = atomicAdd(&A.words[0], __popc(who));
      slot = __shfl_sync(FULL, slot, 0) + __popc(who & ((1u << lane) - 1u));
      if (moves) {
        A.mv_v[slot] = i;
        A.mv_to[slot] = best.c;
      }
    }
  }
}

// Class 2: one warp per vertex, shared table of LV_SLOTS entries.
__global__ void __launch_bounds__(LV_WARPS * 32) k_lv_small(LvArgs A, int32_t lo, int32_t hi) {
  __shared__ int32_t s_key[LV_WARPS][LV_SLOTS];
  __shared__ long long s_val[LV_WARPS][LV_SLOTS];
  const int wv = warp_in_block(), lane = lane_id();
  int32_t* keys = s_key[wv];
  long long* vals = s_val[wv];
  for (int x = lane; x < LV_SLOTS; x += 32) {
    keys[x] = LV_EMPTY;
    vals[x] = 0;
  }
  __syncwarp();
  for (int32_t x = lo + blockIdx.x * LV_WARPS + wv; x < hi; x += gridDim.x * LV_WARPS) {
    const int32_t i = A.list[x];
    const long long b = A.off[i], e = A.off[i + 1];
    for (long long q = b + lane; q < e; q += 32) {
      const int32_t C = A.cl[A.adj[q]];
      if (!table_add(keys, vals, LV_SLOTS - 1, C, A.aw[q])) dev_fail(A.status, DEV_HASH_FULL);
    }
    __syncwarp();
    const int32_t own = A.cl[i];
    const long long ki = A.k[i];
    Cand best{0, -1};
    long long kia = 0;
    for (int s = lane; s < LV_SLOTS; s += 32) {
      const int32_t C = keys[s];
      if (C == LV_EMPTY) continue;
      const long long kic = vals[s];
      keys[s] = LV_EMPTY;
      vals[s] = 0;
      if (C == own) {
        kia = kic;
        continue;
      }
      cand_better(best, Cand{(i128)A.W2 * kic - (i128)ki * A.vol[C], C});
    }
    warp_best(best);
    kia = warp_sum(kia);
    if (lane == 0) lv_emit(A, i, kia, best);
    __syncwarp();
  }
}

// Class 3, step 1: one thread per edge of the listed vertices [lo, hi):
// lpre = exclusive prefix of their degrees along the list, toff = offsets of
// their global tables (relative to tbase).
__global__ void k_lv_big_insert(LvArgs A, int32_t lo, int32_t hi, const long long* __restrict__ lpre,
                                const long long* __restrict__ toff, long long tbase,
                                const int32_t* __restrict__ tsize, int32_t* __restrict__ tkey,
                                long long* __restrict__ tval) {
  const long long base = lpre[lo], cnt = lpre[hi] - base;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < cnt;
       t += (long long)gridDim.x * blockDim.x) {
    const long long y = base + t;
    int32_t a = lo, b = hi - 1;  // largest x in [lo, hi) with lpre[x] <= y
    while (a < b) {
      const int32_t mid = (a + b + 1) >> 1;
      if (lpre[mid] <= y) a = mid;
      else b = mid - 1;
    }
    const int32_t i = A.list[a];
    const long long q = A.off[i] + (y - lpre[a]);
    const long long tb = toff[a] - tbase;
    if (!table_add(tkey + tb, tval + tb, (uint32_t)tsize[a] - 1, A.cl[A.adj[q]], A.aw[q]))
      dev_fail(A.status, DEV_HASH_FULL);
  }
}

// Class 3, step 2: one block per listed vertex, best entry of its table
// (cleared on the way for the next sub-round).
__global__ void __launch_bounds__(LV_ARGMAX_THREADS)
k_lv_big_argmax(LvArgs A, int32_t lo, int32_t hi, const long long* __restrict__ toff,
                long long tbase, const int32_t* __restrict__ tsize, int32_t* __restrict__ tkey,
                long long* __restrict__ tval) {
  __shared__ long long s_lo[32], s_hi[32], s_kia[32];
  __shared__ int32_t s_c[32];
  for (int32_t x = lo + blockIdx.x; x < hi; x += gridDim.x) {
    const int32_t i = A.list[x];
    const int32_t own = A.cl[i];
    const long long ki = A.k[i];
    const long long tb = toff[x] - tbase;
    Cand best{0, -1};
    long long kia = 0;
    for (int32_t s = threadIdx.x; s < tsize[x]; s += blockDim.x) {
      const int32_t C = tkey[tb + s];
      if (C == LV_EMPTY) continue;
      const long long kic = tval[tb + s];
      tkey[tb + s] = LV_EMPTY;
      tval[tb + s] = 0;
      if (C == own) {
        kia = kic;
        continue;
      }
      cand_better(best, Cand{(i128)A.W2 * kic - (i128)ki * A.vol[C], C});
    }
    warp_best(best);
    kia = warp_sum(kia);
    if (lane_id() == 0) {
      s_lo[warp_in_block()] = (long long)(unsigned long long)best.s;
      s_hi[warp_in_block()] = (long long)(best.s >> 64);
      s_c[warp_in_block()] = best.c;
      s_kia[warp_in_block()] = kia;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      Cand b{0, -1};
      long long ka = 0;
      for (int wv = 0; wv < (int)(blockDim.x >> 5); ++wv) {
        cand_better(b, Cand{((i128)s_hi[wv] << 64) | (i128)(unsigned long long)s_lo[wv], s_c[wv]});
        ka += s_kia[wv];
      }
      lv_emit(A, i, ka, b);
    }
    __syncthreads();
  }
}

// Applies the sub-round's moves: cluster and integer volume updates.
__global__ void k_lv_apply(const int32_t* __restrict__ mv_v, const int32_t* __restrict__ mv_to,
                           const int32_t* __restrict__ words, const long long* __restrict__ k,
                           int32_t* __restrict__ cl, long long* __restrict__ vol,
                           unsigned long long* __restrict__ moved) {
  const int32_t nm = words[0];
  for (int32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < nm; x += gridDim.x * blockDim.x) {
    const int32_t i = mv_v[x], to = mv_to[x];
    const long long ki = k[i];
    atomic_add_i64(&vol[cl[i]], -ki);
    atomic_add_i64(&vol[to], ki);
    cl[i] = to;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0 && nm) atomicAdd(moved, (unsigned long long)nm);
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
  DBuf<long long> off, aw, self, k;
  DBuf<int32_t> adj;
};

void lv_degrees(const Ctx& cx, LvGraph& g, long long* W2) {
  g.k.alloc(&cx.alloc, (size_t)std::max<int64_t>(g.V, 1));
  DBuf<unsigned long long> tot;
  tot.alloc(&cx.alloc, 1);
  HG_CUDA(cudaMemsetAsync(tot.p, 0, sizeof(unsigned long long), cx.stream));
  k_lv_degrees<<<grid_for(g.V, 8, cx.num_sms, 16), 256, 0, cx.stream>>>(g.off.p, g.aw.p, g.self.p,
                                                                      g.V, g.k.p, tot.p);
  check_launch("lv_degrees");
  *W2 = read_i64(cx, reinterpret_cast<const int64_t*>(tot.p));
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

// One Louvain level on g (clusters start as singletons).  Returns the moves.
int64_t lv_local_moving(const Ctx& cx, const LvGraph& g, long long W2, int S, uint64_t seed,
                        int level, DBuf<int32_t>& cl, LouvainCounters& lc) {
  const int64_t V = g.V;
  DBuf<long long> vol;
  cl.alloc(&cx.alloc, (size_t)std::max<int64_t>(V, 1));
  vol.alloc(&cx.alloc, (size_t)std::max<int64_t>(V, 1));
  const int gV = grid_for(V, 256, cx.num_sms, 8);
  k_lv_init<<<gV, 256, 0, cx.stream>>>(V, g.k.p, cl.p, vol.p);
  check_launch("lv_init");
  DBuf<int32_t> cnt, fill, koff, list, mv_v, mv_to, words, ldeg, tsize;
  DBuf<long long> lpre, toff;
  DBuf<unsigned long long> moved;
  const int nkeys = LV_CLASSES * S;
  cnt.alloc(&cx.alloc, (size_t)nkeys);
  fill.alloc(&cx.alloc, (size_t)nkeys);
  koff.alloc(&cx.alloc, (size_t)nkeys + 1);
  list.alloc(&cx.alloc, (size_t)V + 1);
  mv_v.alloc(&cx.alloc, (size_t)V + 1);
  mv_to.alloc(&cx.alloc, (size_t)V + 1);
  words.alloc(&cx.alloc, (size_t)S * 4);
  ldeg.alloc(&cx.alloc, (size_t)V + 1);
  tsize.alloc(&cx.alloc, (size_t)V + 1);
  lpre.alloc(&cx.alloc, (size_t)V + 1);
  toff.alloc(&cx.alloc, (size_t)V + 1);
  moved.alloc(&cx.alloc, 1);
  DBuf<long long> bounds;
  bounds.alloc(&cx.alloc, 2 * ((size_t)nkeys + 1));
  DBuf<int32_t> tkey;
  DBuf<long long> tval;
  size_t tcap = 0;
  LvArgs A;
  A.off = g.off.p;
  A.adj = g.adj.p;
  A.aw = g.aw.p;
  A.k = g.k.p;
  A.cl = cl.p;
  A.vol = vol.p;
  A.W2 = W2;
  A.list = list.p;
  A.mv_v = mv_v.p;
  A.mv_to = mv_to.p;
  A.status = cx.d_status;
  int64_t level_moves = 0;
  for (int round = 0; round < LV_ROUNDS; ++round) {
    HG_CUDA(cudaMemsetAsync(cnt.p, 0, cnt.bytes(), cx.stream));
    HG_CUDA(cudaMemsetAsync(fill.p, 0, fill.bytes(), cx.stream));
    HG_CUDA(cudaMemsetAsync(words.p, 0, words.bytes(), cx.stream));
    HG_CUDA(cudaMemsetAsync(moved.p, 0, moved.bytes(), cx.stream));
    k_lv_count<<<gV, 256, nkeys * sizeof(int32_t), cx.stream>>>(g.off.p, V, seed, level, round, S,
                                                                 cnt.p);
    check_launch("lv_count");
    scan_exclusive_i32(cx, cnt.p, koff.p, nkeys, koff.p + nkeys);
    k_lv_scatter<<<gV, 256, 0, cx.stream>>>(g.off.p, V, seed, level, round, S, koff.p, fill.p,
                                            list.p);
    check_launch("lv_scatter");
    // degrees and table sizes along the list, class-3 tables per sub-round
    k_lv_list_sizes<<<gV, 256, 0, cx.stream>>>(list.p, koff.p + nkeys, (int32_t)V, g.off.p, ldeg.p,
                                               tsize.p);
    check_launch("lv_list_sizes");
    scan_exclusive_i32_to_i64(cx, ldeg.p, reinterpret_cast<int64_t*>(lpre.p), V,
                              reinterpret_cast<int64_t*>(lpre.p) + V);
    scan_exclusive_i32_to_i64(cx, tsize.p, reinterpret_cast<int64_t*>(toff.p), V,
                              reinterpret_cast<int64_t*>(toff.p) + V);
    k_lv_bounds<<<1, 256, 0, cx.stream>>>(koff.p, nkeys, toff.p, bounds.p);
    check_launch("lv_bounds");
    std::vector<long long> hb(2 * ((size_t)nkeys + 1));
    wait_stream(cx);
    HG_CUDA(cudaMemcpyAsync(hb.data(), bounds.p, sizeof(long long) * hb.size(),
                            cudaMemcpyDeviceToHost, cx.stream));
    check_status(cx);
    const long long* hkoff = hb.data();
    const long long* htoff = hb.data() + nkeys + 1;
    size_t need = 1;
    for (int s = 0; s < S; ++s)
      need = std::max<size_t>(need, (size_t)(htoff[LV_CLASSES * s + 4] - htoff[LV_CLASSES * s + 3]));
    if (need > tcap) {
      tkey.alloc(&cx.alloc, need);
      tval.alloc(&cx.alloc, need);
      HG_CUDA(cudaMemsetAsync(tkey.p, 0xff, tkey.bytes(), cx.stream));
      HG_CUDA(cudaMemsetAsync(tval.p, 0, tval.bytes(), cx.stream));
      tcap = need;
    }
    for (int s = 0; s < S; ++s) {
      A.words = words.p + 4 * s;
      int32_t at[LV_CLASSES + 1];
      for (int c = 0; c <= LV_CLASSES; ++c) at[c] = (int32_t)hkoff[LV_CLASSES * s + c];
      if (at[1] > at[0]) {
        k_lv_lanes<LV_GROUP><<<grid_for(at[1] - at[0], LV_WARPS * (32 / LV_GROUP), cx.num_sms, 8),
                               LV_WARPS * 32, 0, cx.stream>>>(A, at[0], at[1]);
        check_launch("lv_lanes");
        lc.launches += 1;
      }
      if (at[2] > at[1]) {
        k_lv_lanes<LV_LANES><<<grid_for(at[2] - at[1], LV_WARPS, cx.num_sms, 8), LV_WARPS * 32, 0,
                               cx.stream>>>(A, at[1], at[2]);
        check_launch("lv_lanes");
        lc.launches += 1;
      }
      if (at[3] > at[2]) {
        k_lv_small<<<grid_for(at[3] - at[2], LV_WARPS, cx.num_sms, 8), LV_WARPS * 32, 0,
                     cx.stream>>>(A, at[2], at[3]);
        check_launch("lv_small");
        lc.launches += 1;
      }
      if (at[4] > at[3]) {
        const long long tbase = htoff[LV_CLASSES * s + 3];
        k_lv_big_insert<<<cx.num_sms * 8, 256, 0, cx.stream>>>(A, at[3], at[4], lpre.p, toff.p,
                                                               tbase, tsize.p, tkey.p, tval.p);
        check_launch("lv_big_insert");
        k_lv_big_argmax<<<grid_for(at[4] - at[3], 1, cx.num_sms, 8), LV_ARGMAX_THREADS, 0,
                          cx.stream>>>(A, at[3], at[4], toff.p, tbase, tsize.p, tkey.p, tval.p);
        check_launch("lv_big_argmax");
        lc.launches += 2;
      }
      k_lv_apply<<<grid_for((V + S - 1) / S, 256, cx.num_sms, 4), 256, 0, cx.stream>>>(
          mv_v.p, mv_to.p, A.words, g.k.p, cl.p, vol.p, moved.p);
      check_launch("lv_apply");
      lc.launches += 1;
    }
    const int64_t m = read_i64(cx, reinterpret_cast<const int64_t*>(moved.p));
    level_moves += m;
    lc.rounds += 1;
    if (100 * m < V) break;
  }
  return level_moves;
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
  k_lv_bipartite<<<grid_for(p, 256, cx.num_sms, 16), 256, 0, cx.stream>>>(
      L.eoff.p, L.pins.p, L.w.p, L.inets.p, L.ipin.p, n, p, g.adj.p, g.aw.p);
  check_launch("lv_bipartite");
  long long W2 = 0;
  lv_degrees(cx, g, &W2);
  for (int level = 0; level < LV_LEVELS; ++level) {
    DBuf<int32_t> cl;
    const int64_t moves = lv_local_moving(cx, g, W2, S, seed, level, cl, lc);
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
    lv_degrees(cx, next, &W2n);
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
