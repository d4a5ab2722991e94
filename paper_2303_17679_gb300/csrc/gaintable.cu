// Gain table of Sec. 6.2: benefit b(u) = w({e in I(u) : Phi(e, Pi[u]) = 1})
// and penalty p(u, V_i) = w({e in I(u) : Phi(e, V_i) = 0}), so that the gain
// of Sec. 6 is g_u(V_t) = b(u) - p(u, V_t).
//
// Both need of a net only which blocks hold a pin and which hold exactly one.
// These masks come from one pass over the pins, combined by
//   seen = s1 | s2, twice = t1 | t2 | (s1 & s2)
// over lanes, with no pin counts in memory (the m x k table of counts, cleared
// and filled by atomics, took half of a build).
// Build: the net records, then a lane group or warp per node sums w(e) per
// block in registers (gain.cuh): p(u, V_i) = w(I(u)) - sum_i.
// Moves: for every net of a moved node the masks before and after all moves
// give the change of the table,
//   p(v, V_i) += w(e) (-= w(e)) for every pin v when V_i lost its last (got its
//   first) pin of e, and
//   b(v) += w(e) (-= w(e)) for the unmoved pins v of V_i when V_i got down to
//   (rose above) one pin of e,
// which is what the update rules of Sec. 6.2 add up to in any order of the moves
// (its lemma); the benefits of the moved nodes are recomputed from the masks
// after the moves.
// Measured (GB300, n = m = 1e6 Zipf, k = 8, 100,000 moves): build, moves and the
// exact gains of the sequence (gainrecalc.cu) together 1.18 -> 0.64 ms.
//
// Graph levels (Sec. 10, "The Gain Table"): the table of a graph is
// w(u, V_i), the weight of u's edges into V_i; the benefit and penalties follow:
//   b(u) = w(I(u)) - w(u, V_Pi(u)),  p(u, V_Pi(u)) = 0,
//   p(u, V_i) = w(I(u)) - w(u, V_i) for i != Pi(u)
// (an edge has no pin in V_i exactly when neither endpoint is in V_i).
#include <algorithm>

#include "gain.cuh"

namespace hgk {

namespace {

constexpr int GT_WARPS = 8;
// nets and nodes of at most GT_SMALL pins (nets) are taken by a lane group, up
// to GT_BIG_NET pins by a warp, larger nets by blocks
constexpr int32_t GT_SMALL = SMALL_TOUCHED;
constexpr int32_t GT_BIG_NET = 4096;
constexpr int GT_BIG_THREADS = 256;

using Mask = unsigned long long;

// Blocks seen and seen more than once.
struct Seen {
  Mask s = 0, t = 0;
  __device__ __forceinline__ void add(int block) {
    const Mask x = 1ull << block;
    t |= s & x;
    s |= x;
  }
  __device__ __forceinline__ void join(Mask s2, Mask t2) {
    t |= t2 | (s & s2);
    s |= s2;
  }
  // over the W lanes of the caller's group; the whole warp calls it
  template <int W>
  __device__ __forceinline__ void combine() {
#pragma unroll
    for (int d = W / 2; d > 0; d >>= 1) {
      const Mask s2 = __shfl_xor_sync(FULL, s, d), t2 = __shfl_xor_sync(FULL, t, d);
      join(s2, t2);
    }
  }
  __device__ __forceinline__ Mask ones() const { return s & ~t; }
};

__device__ __forceinline__ void write_rec(int4* rec, int64_t e, int k, int32_t w, const Seen& x) {
  const int H = k > 32 ? 2 : 1;
  for (int h = 0; h < H; ++h)
    rec[H * e + h] = make_int4(w, (int32_t)(uint32_t)(x.ones() >> (32 * h)),
                               (int32_t)(uint32_t)(x.s >> (32 * h)), 0);
}

// Lists the chunks of GT_BIG_NET pins of a larger net, {net, first of its chunks}
// each (one thread).
__device__ __forceinline__ void list_chunks(int32_t e, int32_t sz, int2* chunks, int32_t* nchunks) {
  const int32_t count = (sz + GT_BIG_NET - 1) / GT_BIG_NET;
  const int32_t first = atomicAdd(nchunks, count);
  for (int32_t c = 0; c < count; ++c) chunks[first + c] = make_int2(e, first);
}

// At most that many chunks on a level of p pins.
size_t chunk_cap(int64_t p) { return 2 * (size_t)(p / GT_BIG_NET) + 1; }

// Records of the nets of up to GT_BIG_NET pins; the chunks of larger ones are
// listed.  The partition has been checked.
__global__ void __launch_bounds__(GT_WARPS * 32)
k_gt_records(const int32_t* __restrict__ eoff, const int32_t* __restrict__ pins,
             const int32_t* __restrict__ w, const int32_t* __restrict__ part, int32_t m, int k,
             int4* __restrict__ rec, int2* __restrict__ chunks, int32_t* __restrict__ nchunks) {
  const int lane = lane_id(), sub = lane % SUB_G;
  const int64_t stride = (int64_t)gridDim.x * GT_WARPS * NG;
  for (int64_t e0 = ((int64_t)blockIdx.x * GT_WARPS + warp_in_block()) * NG; e0 < m; e0 += stride) {
    const int64_t e = e0 + lane / SUB_G;
    const int32_t b = e < m ? eoff[e] : 0, sz = e < m ? eoff[e + 1] - b : 0;
    const int32_t mine = sz <= GT_SMALL ? sz : 0;
    const int steps = __reduce_max_sync(FULL, (unsigned)mine);
    Seen x;
    for (int q = sub; q - sub < steps; q += 2 * SUB_G) {
      const bool v0 = q < mine, v1 = q + SUB_G < mine;
      const int32_t u0 = v0 ? pins[b + q] : 0, u1 = v1 ? pins[b + q + SUB_G] : 0;
      const int32_t p0 = v0 ? part[u0] : 0, p1 = v1 ? part[u1] : 0;
      if (v0) x.add(p0);
      if (v1) x.add(p1);
    }
    x.combine<SUB_G>();
    if (sub == 0 && e < m && sz <= GT_SMALL) write_rec(rec, e, k, w[e], x);
    unsigned wide = __ballot_sync(FULL, sub == 0 && sz > GT_SMALL);
    while (wide) {
      const int l = __ffs(wide) - 1;
      wide &= wide - 1;
      const int64_t we = e0 + l / SUB_G;
      const int32_t wb = __shfl_sync(FULL, b, l), ws = __shfl_sync(FULL, sz, l);
      if (ws > GT_BIG_NET) {
        if (lane == 0) list_chunks((int32_t)we, ws, chunks, nchunks);
        continue;
      }
      Seen y;
      for (int q = lane; q < ws; q += 64) {
        const bool v1 = q + 32 < ws;
        const int32_t u0 = pins[wb + q], u1 = v1 ? pins[wb + q + 32] : 0;
        const int32_t p0 = part[u0], p1 = v1 ? part[u1] : 0;
        y.add(p0);
        if (v1) y.add(p1);
      }
      y.combine<32>();
      if (lane == 0) write_rec(rec, we, k, w[we], y);
    }
  }
}

// A block's Seen over all its threads, in every thread of warp 0.
__device__ __forceinline__ Seen block_seen(Seen x) {
  __shared__ Mask s_s[32], s_t[32];
  x.combine<32>();
  __syncthreads();
  if (lane_id() == 0) {
    s_s[warp_in_block()] = x.s;
    s_t[warp_in_block()] = x.t;
  }
  __syncthreads();
  Seen y;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) y.join(s_s[i], s_t[i]);
  return y;
}

// Records of the larger nets, a block per listed chunk (whole nets one after the
// other, their chunks over the grid, left two blocks at work on nets of two chunks:
// 54 ms for 5000 of them, 0.5 now), joined in three words per net at its first
// chunk: seen, seen twice and the chunks done.
__global__ void __launch_bounds__(GT_BIG_THREADS)
k_gt_records_big(const int32_t* __restrict__ eoff, const int32_t* __restrict__ pins,
                 const int32_t* __restrict__ w, const int32_t* __restrict__ part, int k,
                 int4* __restrict__ rec, const int2* __restrict__ chunks,
                 const int32_t* __restrict__ nchunks, Mask* __restrict__ words) {
  const int32_t cnt = *nchunks;
  for (int32_t c = blockIdx.x; c < cnt; c += gridDim.x) {
    const int2 it = chunks[c];
    const int32_t e = it.x, b = eoff[e], sz = eoff[e + 1] - b;
    const int32_t lo = (c - it.y) * GT_BIG_NET, hi = min(sz - lo, GT_BIG_NET) + lo;
    Seen x;
    for (int32_t q = lo + threadIdx.x; q < hi; q += GT_BIG_THREADS) x.add(part[pins[b + q]]);
    __syncwarp();
    x = block_seen(x);
    if (threadIdx.x == 0) {
      Mask* acc = words + 3 * (int64_t)it.y;
      const Mask before = atomicOr(&acc[0], x.s);
      atomicOr(&acc[1], x.t | (before & x.s));
      __threadfence();
      if (atomicAdd(&acc[2], 1ull) == (Mask)((sz + GT_BIG_NET - 1) / GT_BIG_NET - 1)) {
        __threadfence();
        Seen y;
        y.s = atomicOr(&acc[0], 0ull);
        y.t = atomicOr(&acc[1], 0ull);
        write_rec(rec, e, k, w[e], y);
      }
    }
  }
}

// Table rows of the nodes: a lane group per node of at most GT_SMALL incident
// nets, a warp for up to GT_HUB; items of GT_ITEM incident nets of larger nodes are
// listed for a warp each, which add to the row (ADD).  One warp for a node of 5M
// nets took 434 ms at k = 64, whatever the rest of the chip did, and four neighbours
// of 2000 nets in one warp 0.64 ms for a complete graph of 2000 nodes (0.07 now;
// limits of 256 and 1024 are no different).
constexpr int32_t GT_HUB = 512, GT_ITEM = 512;

template <bool GRAPH, int K, int H, int W, bool ADD = false>
__device__ __forceinline__ void gt_row(const int32_t* __restrict__ inets,
                                       const int2* __restrict__ adj, const int4* __restrict__ rec,
                                       const int32_t* __restrict__ part, bool on, int64_t u,
                                       int32_t beg, int32_t end, int l, int k,
                                       long long* __restrict__ b, long long* __restrict__ p) {
  using L = TeamLane<W, H>;
  const L lane(l);
  const int from = on ? part[u] : 0, from_h = from - 32 * lane.half;
  Gain<GRAPH, K, H> g;
  g.init();
  int32_t wsum = 0;  // of distinct nets: below 2^31, as the sums of gain.cuh
  const int32_t steps = __reduce_max_sync(FULL, end - beg);
  for (int32_t x = lane.i; x - lane.i < steps; x += 2 * L::SHARE) {
    const int32_t j0 = beg + x, j1 = j0 + L::SHARE;
    const bool v0 = j0 < end, v1 = j1 < end;
    if (GRAPH) {
      const int2 a0 = v0 ? adj[j0] : make_int2(-1, 0), a1 = v1 ? adj[j1] : make_int2(-1, 0);
      const int t0 = v0 ? part[a0.x] : 0, t1 = v1 ? part[a1.x] : 0;
      g.add_edge(a0.y, t0 - 32 * lane.half, from_h);
      g.add_edge(a1.y, t1 - 32 * lane.half, from_h);
      wsum += a0.y + a1.y;
    } else {
      const int32_t e0 = v0 ? inets[j0] : 0, e1 = v1 ? inets[j1] : 0;
      NetRec r0{0, 0, 0}, r1{0, 0, 0};
      if (v0) r0 = load_rec(rec, (int64_t)H * e0 + lane.half);
      if (v1) r1 = load_rec(rec, (int64_t)H * e1 + lane.half);
      g.add(r0, from_h);
      g.add(r1, from_h);
      wsum += r0.w + r1.w;
    }
  }
  wsum = group_sum<W>(lane.half == 0 ? wsum : 0);  // both halves saw every net
  const int32_t bw = group_sum<W>(g.bw);           // b(u) - w(I(u))
  const int b0 = 32 * lane.half + reduce_scatter<L::SHARE, K>(lane.i, g.acc);
  constexpr int OWN = K / L::SHARE > 0 ? K / L::SHARE : 1;
  constexpr int SAME = L::SHARE / K > 1 ? L::SHARE / K : 1;
  if (on) {
    if (l == 0) {
      if (ADD) atomic_add_i64(&b[u], wsum + bw);
      else b[u] = wsum + bw;
    }
    if (lane.i % SAME == 0) {
#pragma unroll
      for (int i = 0; i < OWN; ++i)
        if (b0 + i < k) {
          const int32_t x = GRAPH && b0 + i == from ? 0 : wsum - g.acc[i];
          if (!ADD) p[u * k + b0 + i] = x;
          else if (x) atomic_add_i64(&p[u * k + b0 + i], x);
        }
    }
  }
}

// The same on graph levels for k > 16 with counters in shared memory (`cnt`, k words
// that are zero before and after): an edge is one add there, in registers a comparison
// with every block (n = 500,003, 2M edges, k = 64: 0.22 ms, 0.13 here).
constexpr int GT_COUNTERS = HG_MAX_K + 8;  // of a lane group: 8 banks apart

template <int W, bool ADD = false>
__device__ __forceinline__ void gt_row_counted(const int2* __restrict__ adj,
                                               const int32_t* __restrict__ part, bool on,
                                               int64_t u, int32_t beg, int32_t end, int l, int k,
                                               long long* __restrict__ b,
                                               long long* __restrict__ p, int32_t* cnt) {
  const int from = on ? part[u] : 0;
  int32_t wsum = 0;
  for (int32_t j = beg + l; j < end; j += 2 * W) {
    const bool two = j + W < end;
    const int2 a0 = adj[j], a1 = two ? adj[j + W] : make_int2(-1, 0);
    const int t0 = part[a0.x], t1 = two ? part[a1.x] : 0;
    atomicAdd(&cnt[t0], a0.y);
    if (two) atomicAdd(&cnt[t1], a1.y);
    wsum += a0.y + a1.y;
  }
  __syncwarp();
  wsum = group_sum<W>(wsum);
  for (int t = l; on && t < k; t += W) {
    const int32_t x = t == from ? 0 : wsum - cnt[t];
    if (t == from) {
      if (ADD) atomic_add_i64(&b[u], wsum - cnt[t]);
      else b[u] = wsum - cnt[t];
    }
    if (!ADD) p[u * k + t] = x;
    else if (x) atomic_add_i64(&p[u * k + t], x);
    cnt[t] = 0;
  }
  __syncwarp();
}

template <bool GRAPH, int K, int H>
__global__ void __launch_bounds__(GT_WARPS * 32)
k_gt_build(const int32_t* __restrict__ ioff, const int32_t* __restrict__ inets,
           const int2* __restrict__ adj, const int4* __restrict__ rec,
           const int32_t* __restrict__ part, int32_t n, int k, long long* __restrict__ b,
           long long* __restrict__ p, int2* __restrict__ items, int32_t* __restrict__ nitems) {
  constexpr bool COUNTED = GRAPH && K == 32;
  __shared__ int32_t s_cnt[COUNTED ? GT_WARPS : 1][NG][GT_COUNTERS];
  const int lane = lane_id();
  if (COUNTED) {
    for (int i = lane; i < NG * GT_COUNTERS; i += 32) (&s_cnt[warp_in_block()][0][0])[i] = 0;
    __syncwarp();
  }
  const int64_t stride = (int64_t)gridDim.x * GT_WARPS * NG;
  for (int64_t u0 = ((int64_t)blockIdx.x * GT_WARPS + warp_in_block()) * NG; u0 < n; u0 += stride) {
    const int64_t u = u0 + lane / SUB_G;
    const int32_t beg = u < n ? ioff[u] : 0, end = u < n ? ioff[u + 1] : 0;
    if (!__any_sync(FULL, end > beg)) {  // nodes without nets: whole rows of zeros
      const int64_t stop = (u0 + NG < n ? u0 + NG : n) * k;
      for (int64_t x = u0 * k + lane; x < stop; x += 32) p[x] = 0;
      if (u < n && lane % SUB_G == 0) b[u] = 0;
      continue;
    }
    const bool small = end - beg <= GT_SMALL;
    if constexpr (COUNTED)
      gt_row_counted<SUB_G>(adj, part, u < n && small, u, beg, small ? end : beg, lane % SUB_G, k,
                            b, p, s_cnt[warp_in_block()][lane / SUB_G]);
    else
      gt_row<GRAPH, K, H, SUB_G>(inets, adj, rec, part, u < n && small, u, beg, small ? end : beg,
                                 lane % SUB_G, k, b, p);
    unsigned wide = __ballot_sync(FULL, lane % SUB_G == 0 && !small);
    while (wide) {
      const int l = __ffs(wide) - 1;
      wide &= wide - 1;
      const int64_t wu = u0 + l / SUB_G;
      const int32_t wb = __shfl_sync(FULL, beg, l), we = __shfl_sync(FULL, end, l);
      if (we - wb > GT_HUB) {
        const int32_t count = (we - wb + GT_ITEM - 1) / GT_ITEM;
        int32_t first = 0;
        if (lane == 0) {
          first = atomicAdd(nitems, count);
          b[wu] = 0;
        }
        first = __shfl_sync(FULL, first, 0);
        for (int32_t i = lane; i < count; i += 32) items[first + i] = make_int2((int)wu, i);
        for (int t = lane; t < k; t += 32) p[wu * k + t] = 0;
        continue;
      }
      if constexpr (COUNTED)
        gt_row_counted<32>(adj, part, true, wu, wb, we, lane, k, b, p, s_cnt[warp_in_block()][0]);
      else
        gt_row<GRAPH, K, H, 32>(inets, adj, rec, part, true, wu, wb, we, lane, k, b, p);
    }
  }
}

template <bool GRAPH, int K, int H>
__global__ void __launch_bounds__(GT_WARPS * 32)
k_gt_build_hubs(const int32_t* __restrict__ ioff, const int32_t* __restrict__ inets,
                const int2* __restrict__ adj, const int4* __restrict__ rec,
                const int32_t* __restrict__ part, int k, long long* __restrict__ b,
                long long* __restrict__ p, const int2* __restrict__ items,
                const int32_t* __restrict__ nitems) {
  constexpr bool COUNTED = GRAPH && K == 32;
  __shared__ int32_t s_cnt[COUNTED ? GT_WARPS : 1][GT_COUNTERS];
  if (COUNTED) {
    for (int i = lane_id(); i < GT_COUNTERS; i += 32) s_cnt[warp_in_block()][i] = 0;
    __syncwarp();
  }
  const int32_t cnt = *nitems;
  for (int32_t x = warp_in_block() * gridDim.x + blockIdx.x; x < cnt; x += gridDim.x * GT_WARPS) {
    const int2 it = items[x];
    const int32_t beg = ioff[it.x] + it.y * GT_ITEM;
    const int32_t end = beg + min(GT_ITEM, ioff[it.x + 1] - beg);
    if constexpr (COUNTED)
      gt_row_counted<32, true>(adj, part, true, it.x, beg, end, lane_id(), k, b, p,
                               s_cnt[warp_in_block()]);
    else
      gt_row<GRAPH, K, H, 32, true>(inets, adj, rec, part, true, it.x, beg, end, lane_id(), k, b,
                                    p);
  }
}

template <bool GRAPH, int K, int H>
void build_rows(const Ctx& cx, const Level& L, int k, const int4* rec, const int32_t* part,
                long long* b, long long* p) {
  DBuf<int2> items;
  DBuf<int32_t> nitems;
  const bool hubs = L.p > GT_HUB;
  if (hubs) {
    items.alloc(&cx.alloc, (size_t)(L.p / GT_ITEM + L.p / GT_HUB) + 1);
    nitems.alloc(&cx.alloc, 1);
    HG_CUDA(cudaMemsetAsync(nitems.p, 0, sizeof(int32_t), cx.stream));
  }
  k_gt_build<GRAPH, K, H><<<grid_for(L.n, GT_WARPS * NG, cx.num_sms, 8), GT_WARPS * 32, 0,
                            cx.stream>>>(L.ioff.p, L.inets.p, L.adj.p, rec, part, L.n, k, b, p,
                                         items.p, nitems.p);
  check_launch("gt_build");
  if (hubs) {
    k_gt_build_hubs<GRAPH, K, H><<<grid_for(L.p, GT_ITEM * GT_WARPS, cx.num_sms, 8),
                                   GT_WARPS * 32, 0, cx.stream>>>(
        L.ioff.p, L.inets.p, L.adj.p, rec, part, k, b, p, items.p, nitems.p);
    check_launch("gt_build_hubs");
  }
  if (cx.launches) *cx.launches += 1 + hubs;
}

using BuildRows = void (*)(const Ctx&, const Level&, int, const int4*, const int32_t*, long long*,
                           long long*);

BuildRows build_rows_for(bool graph, int k) {
  if (graph) {
    if (k <= 8) return build_rows<true, 8, 1>;
    if (k <= 16) return build_rows<true, 16, 1>;
    return build_rows<true, 32, 1>;
  }
  if (k <= 8) return build_rows<false, 8, 1>;
  if (k <= 16) return build_rows<false, 16, 1>;
  if (k <= 32) return build_rows<false, 32, 1>;
  return build_rows<false, 32, 2>;
}

// ------------------------------------------------------------ moves

// The table changes of one net held by W threads with positions `at` of it
// (its pins at `at`, at + W, ...): masks before and after, then the updates.
struct MoveArgs {
  const int32_t *eoff, *pins, *w, *targets;
  const int2* info;      // {move index or -1, block} of every node
  int k;
  Mask* ones;            // ones(e) after the moves, per net
  unsigned long long *b, *p;
};

__device__ __forceinline__ void see_pin(const MoveArgs& A, int32_t v, Seen& was, Seen& is) {
  const int2 nd = A.info[v];
  was.add(nd.y);
  is.add(nd.x >= 0 ? A.targets[nd.x] : nd.y);
}

__device__ __forceinline__ void update_pin(const MoveArgs& A, int32_t v, unsigned long long we,
                                           Mask lam, Mask lam_x, Mask ones, Mask ones_x) {
  while (lam_x) {
    const int i = __ffsll((long long)lam_x) - 1;
    lam_x &= lam_x - 1;
    atomicAdd(&A.p[(int64_t)v * A.k + i], (lam >> i) & 1 ? 0ull - we : we);
  }
  if (ones_x) {
    const int2 nd = A.info[v];
    if (nd.x < 0 && ((ones_x >> nd.y) & 1))
      atomicAdd(&A.b[v], (ones >> nd.y) & 1 ? we : 0ull - we);
  }
}

// Listed nets (touched_nets): a lane group for up to GT_SMALL pins, a warp for up to
// GT_BIG_NET; of the chunks of larger nets, a block each, the masks before and after
// the moves, joined in four words per net at its first chunk.
__global__ void __launch_bounds__(GT_WARPS * 32)
k_gt_move_nets(MoveArgs A, const int32_t* __restrict__ list, const int32_t* __restrict__ count,
               int32_t m, const int2* __restrict__ chunks, Mask* __restrict__ words) {
  const int lane = lane_id(), sub = lane % SUB_G;
  const int32_t nchunks = count[TN_CHUNKS], nwide = count[TN_WIDE], cnt = count[TN_SMALL];
  for (int32_t c = blockIdx.x; c < nchunks; c += gridDim.x) {
    const int2 it = chunks[c];
    const int32_t b = A.eoff[it.x], sz = A.eoff[it.x + 1] - b;
    const int32_t lo = (c - it.y) * GT_BIG_NET, hi = min(sz - lo, GT_BIG_NET) + lo;
    Seen was, is;
    for (int32_t q = lo + threadIdx.x; q < hi; q += GT_WARPS * 32)
      see_pin(A, A.pins[b + q], was, is);
    __syncwarp();
    was = block_seen(was);
    is = block_seen(is);
    if (threadIdx.x == 0) {
      Mask* acc = words + 4 * (int64_t)it.y;
      const Mask w0 = atomicOr(&acc[0], was.s), i0 = atomicOr(&acc[2], is.s);
      atomicOr(&acc[1], was.t | (w0 & was.s));
      atomicOr(&acc[3], is.t | (i0 & is.s));
    }
    __syncthreads();
  }
  for (int32_t x = warp_in_block() * gridDim.x + blockIdx.x; x < nwide;
       x += gridDim.x * GT_WARPS) {
    const int32_t e = list[m - 1 - x];
    const int32_t b = A.eoff[e], sz = A.eoff[e + 1] - b;
    Seen was, is;
    for (int q = lane; q < sz; q += 32) see_pin(A, A.pins[b + q], was, is);
    __syncwarp();
    was.combine<32>();
    is.combine<32>();
    if (lane == 0) A.ones[e] = is.ones();
    const Mask lam_x = was.s ^ is.s, ones_x = was.ones() ^ is.ones();
    if (lam_x | ones_x) {
      const unsigned long long we = (unsigned long long)(long long)A.w[e];
      for (int q = lane; q < sz; q += 32)
        update_pin(A, A.pins[b + q], we, is.s, lam_x, is.ones(), ones_x);
    }
    __syncwarp();
  }
  const int64_t stride = (int64_t)gridDim.x * GT_WARPS * NG;
  for (int64_t x0 = ((int64_t)blockIdx.x * GT_WARPS + warp_in_block()) * NG; x0 < cnt;
       x0 += stride) {
    const int64_t x = x0 + lane / SUB_G;
    const int32_t e = x < cnt ? list[x] : 0;
    const int32_t b = x < cnt ? A.eoff[e] : 0, sz = x < cnt ? A.eoff[e + 1] - b : 0;
    Seen was, is;
    for (int q = sub; q < sz; q += SUB_G) see_pin(A, A.pins[b + q], was, is);
    __syncwarp();
    was.combine<SUB_G>();
    is.combine<SUB_G>();
    if (sz > 0) {
      if (sub == 0) A.ones[e] = is.ones();
      const Mask lam_x = was.s ^ is.s, ones_x = was.ones() ^ is.ones();
      if (lam_x | ones_x) {
        const unsigned long long we = (unsigned long long)(long long)A.w[e];
        for (int q = sub; q < sz; q += SUB_G)
          update_pin(A, A.pins[b + q], we, is.s, lam_x, is.ones(), ones_x);
      }
    }
    __syncwarp();
  }
}

// The updates of the larger nets, a block per chunk.  (A block per net: 104 ms for a
// net of 20M pins, 1.3 now.)
__global__ void __launch_bounds__(GT_BIG_THREADS)
k_gt_move_chunks(MoveArgs A, const int2* __restrict__ chunks, const int32_t* __restrict__ count,
                 const Mask* __restrict__ words) {
  const int32_t cnt = count[TN_CHUNKS];
  for (int32_t c = blockIdx.x; c < cnt; c += gridDim.x) {
    const int2 it = chunks[c];
    const Mask* acc = words + 4 * (int64_t)it.y;
    Seen was, is;
    was.join(acc[0], acc[1]);
    is.join(acc[2], acc[3]);
    if (c == it.y && threadIdx.x == 0) A.ones[it.x] = is.ones();
    const Mask lam_x = was.s ^ is.s, ones_x = was.ones() ^ is.ones();
    if (!(lam_x | ones_x)) continue;
    const int32_t b = A.eoff[it.x], sz = A.eoff[it.x + 1] - b;
    const int32_t lo = (c - it.y) * GT_BIG_NET, hi = min(sz - lo, GT_BIG_NET) + lo;
    const unsigned long long we = (unsigned long long)(long long)A.w[it.x];
    for (int32_t q = lo + threadIdx.x; q < hi; q += GT_BIG_THREADS)
      update_pin(A, A.pins[b + q], we, is.s, lam_x, is.ones(), ones_x);
  }
}

// Pi and b of the moved nodes from the masks after the moves, a lane group per
// move.
__global__ void __launch_bounds__(GT_WARPS * 32)
k_gt_moved(const int32_t* __restrict__ nodes, const int32_t* __restrict__ targets, int32_t l,
           const int32_t* __restrict__ ioff, const int32_t* __restrict__ inets,
           const int32_t* __restrict__ w, const Mask* __restrict__ ones,
           int32_t* __restrict__ part, long long* __restrict__ b) {
  const int lane = lane_id(), sub = lane % SUB_G;
  const int64_t stride = (int64_t)gridDim.x * GT_WARPS * NG;
  for (int64_t i0 = ((int64_t)blockIdx.x * GT_WARPS + warp_in_block()) * NG; i0 < l; i0 += stride) {
    const int64_t i = i0 + lane / SUB_G;
    const int32_t u = i < l ? nodes[i] : 0, t = i < l ? targets[i] : 0;
    const int32_t beg = i < l ? ioff[u] : 0, end = i < l ? ioff[u + 1] : 0;
    long long bu = 0;
    for (int32_t j = beg + sub; j < end; j += SUB_G) {
      const int32_t e = inets[j];
      if ((ones[e] >> t) & 1) bu += w[e];
    }
    __syncwarp();
    bu = group_sum<SUB_G>(bu);
    if (sub == 0 && i < l) {
      b[u] = bu;
      part[u] = t;
    }
  }
}

}  // namespace

void gain_table_build(const Ctx& cx, const Level& L, int k, const int32_t* part, int64_t* b,
                      int64_t* p) {
  validate_partition(cx, part, L.n, k);
  DBuf<int4> rec;
  if (!L.graph && L.m > 0) {
    const size_t cap = chunk_cap(L.p);
    DBuf<int2> chunks;
    DBuf<Mask> words;  // three per net, then the number of chunks
    rec.alloc(&cx.alloc, (size_t)L.m * (k > 32 ? 2 : 1));
    chunks.alloc(&cx.alloc, cap);
    words.alloc(&cx.alloc, 3 * cap + 1);
    HG_CUDA(cudaMemsetAsync(words.p, 0, words.bytes(), cx.stream));
    int32_t* nchunks = reinterpret_cast<int32_t*>(words.p + 3 * cap);
    k_gt_records<<<grid_for(L.m, GT_WARPS * NG, cx.num_sms, 8), GT_WARPS * 32, 0, cx.stream>>>(
        L.eoff.p, L.pins.p, L.w.p, part, L.m, k, rec.p, chunks.p, nchunks);
    check_launch("gt_records");
    if (L.p > GT_BIG_NET) {
      k_gt_records_big<<<grid_for(L.p, GT_BIG_NET, cx.num_sms, 8), GT_BIG_THREADS, 0, cx.stream>>>(
          L.eoff.p, L.pins.p, L.w.p, part, k, rec.p, chunks.p, nchunks, words.p);
      check_launch("gt_records_big");
    }
    if (cx.launches) *cx.launches += 1 + (L.p > GT_BIG_NET);
  }
  build_rows_for(L.graph, k)(cx, L, k, rec.p, part, reinterpret_cast<long long*>(b),
                             reinterpret_cast<long long*>(p));
  check_status(cx);
}

void gain_table_move(const Ctx& cx, const Level& L, int k, int32_t* part, int32_t l,
                     const int32_t* nodes, const int32_t* targets, int64_t* b, int64_t* p) {
  if (l == 0) {
    validate_partition(cx, part, L.n, k);
    return;
  }
  check_partition(cx, part, L.n, k);
  DBuf<int2> info;
  TouchedNets t;
  index_moves(cx, L, k, part, l, nodes, targets, info);
  check_status(cx);  // nothing below runs on a bad partition or bad moves
  touched_nets(cx, L, l, nodes, GT_BIG_NET, t);
  DBuf<Mask> ones;
  ones.alloc(&cx.alloc, (size_t)std::max<int32_t>(L.m, 1));
  MoveArgs A;
  A.eoff = L.eoff.p;
  A.pins = L.pins.p;
  A.w = L.w.p;
  A.info = info.p;
  A.targets = targets;
  A.k = k;
  A.ones = ones.p;
  A.b = reinterpret_cast<unsigned long long*>(b);
  A.p = reinterpret_cast<unsigned long long*>(p);
  DBuf<Mask> words;
  words.alloc(&cx.alloc, 4 * chunk_cap(L.p));
  HG_CUDA(cudaMemsetAsync(words.p, 0, words.bytes(), cx.stream));
  k_gt_move_nets<<<cx.num_sms * 8, GT_WARPS * 32, 0, cx.stream>>>(A, t.list.p, t.count.p, L.m,
                                                                  t.chunks.p, words.p);
  check_launch("gt_move_nets");
  if (L.p > GT_BIG_NET) {
    k_gt_move_chunks<<<grid_for(L.p, GT_BIG_NET, cx.num_sms, 8), GT_BIG_THREADS, 0, cx.stream>>>(
        A, t.chunks.p, t.count.p, words.p);
    check_launch("gt_move_chunks");
  }
  k_gt_moved<<<grid_for(l, GT_WARPS * NG, cx.num_sms, 8), GT_WARPS * 32, 0, cx.stream>>>(
      nodes, targets, l, L.ioff.p, L.inets.p, L.w.p, ones.p, part, reinterpret_cast<long long*>(b));
  check_launch("gt_moved");
  if (cx.launches) *cx.launches += 2 + (L.p > GT_BIG_NET);
  check_status(cx);
}

}  // namespace hgk
