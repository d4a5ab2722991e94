// Hypergraph structure on the device: the pin-tile index, the incident-net
// lists I(u) (the second adjacency array of Sec. 4.2, "The Contraction
// Algorithm"), the single adjacency array of graph levels (Sec. 10, "Graph
// Data Structure"), and validation of caller-provided device arrays.
#include <algorithm>

#include "common.cuh"
#include "pintile.cuh"

namespace hgk {

namespace {

// tile_net[t] = net containing pin position t * PIN_TILE.
__global__ void k_tile_index(const int32_t* __restrict__ eoff, int32_t m, int64_t ntiles,
                             int32_t* __restrict__ tile_net) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t a = eoff[e], b = eoff[e + 1];
    if (b <= a) continue;
    for (int64_t t = (a + PIN_TILE - 1) / PIN_TILE; t * PIN_TILE < b && t < ntiles; ++t)
      tile_net[t] = (int32_t)e;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) tile_net[ntiles] = m > 0 ? m - 1 : 0;
}

__global__ void k_degrees(const int32_t* __restrict__ pins, int64_t p, int32_t* __restrict__ deg) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < p;
       q += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(&deg[pins[q]], 1);
}

// Levels of few nodes and many pins: every block counts the pins of its run of
// tiles (graph levels: edges) per node in shared memory, claims that many
// slots of every node with one atomic and hands them out by counters in shared
// memory.  The atomics of all pins on a few thousand addresses bound the other
// form: 245 + 255 us (degrees, scatter) at 1571 nodes and 5.07M pins, 9 + 50 us this
// way; taken when a block has at least four pins per node and half the SMs
// get a block.
constexpr int LOCAL_THREADS = 1024;
constexpr int32_t LOCAL_N = 32768;
constexpr int64_t LOCAL_PINS = 4;

int local_blocks(const Ctx& cx, int32_t n, int64_t p, int64_t units) {
  if (n > LOCAL_N) return 0;
  const int per_sm = n <= LOCAL_N / 2 ? 2 : 1;
  const int64_t b = std::min(
      std::min(p / (LOCAL_PINS * n), units), (int64_t)cx.num_sms * per_sm);
  return b >= cx.num_sms / 2 ? (int)b : 0;
}

__global__ void __launch_bounds__(LOCAL_THREADS)
k_degrees_local(const int32_t* __restrict__ pins, int64_t p, int32_t n, int32_t* __restrict__ deg) {
  extern __shared__ int32_t s_n[];
  for (int32_t u = threadIdx.x; u < n; u += LOCAL_THREADS) s_n[u] = 0;
  __syncthreads();
  for (int64_t q = (int64_t)blockIdx.x * LOCAL_THREADS + threadIdx.x; q < p;
       q += (int64_t)gridDim.x * LOCAL_THREADS)
    atomicAdd(&s_n[pins[q]], 1);
  __syncthreads();
  for (int32_t u = threadIdx.x; u < n; u += LOCAL_THREADS)
    if (s_n[u]) atomicAdd(&deg[u], s_n[u]);
}

// Counts -> first slots of the block.
__device__ __forceinline__ void claim_slots(int32_t* s_n, int32_t n, int32_t* cursor) {
  __syncthreads();
  for (int32_t u = threadIdx.x; u < n; u += LOCAL_THREADS)
    if (s_n[u]) s_n[u] = atomicAdd(&cursor[u], s_n[u]);
  __syncthreads();
}

__global__ void __launch_bounds__(LOCAL_THREADS)
k_scatter_incidence_local(const int32_t* __restrict__ eoff, const int32_t* __restrict__ pins,
                          const int32_t* __restrict__ tile_net, int32_t m, int64_t p, int32_t n,
                          int32_t* __restrict__ cursor, int32_t* __restrict__ inets) {
  extern __shared__ int32_t s_n[];
  __shared__ int32_t s_off[PIN_TILE + 3];
  const int64_t ntiles = num_pin_tiles(p);
  const int64_t t0 = ntiles * blockIdx.x / gridDim.x, t1 = ntiles * (blockIdx.x + 1) / gridDim.x;
  const int64_t q1 = t1 * PIN_TILE < p ? t1 * PIN_TILE : p;
  for (int32_t u = threadIdx.x; u < n; u += LOCAL_THREADS) s_n[u] = 0;
  __syncthreads();
  for (int64_t q = t0 * PIN_TILE + threadIdx.x; q < q1; q += LOCAL_THREADS)
    atomicAdd(&s_n[pins[q]], 1);
  claim_slots(s_n, n, cursor);
  for (int64_t t = t0; t < t1; ++t) {
    const PinTileView v = stage_pin_tile(eoff, tile_net, m, p, t, s_off);
    for (int64_t q = v.q0 + threadIdx.x; q < v.q1; q += LOCAL_THREADS) {
      const int32_t e = v.e_lo + net_in_tile(s_off, v.count, q);
      inets[atomicAdd(&s_n[pins[q]], 1)] = e;
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(LOCAL_THREADS)
k_scatter_edges_local(const int2* __restrict__ pins, const int32_t* __restrict__ w, int32_t m,
                      int32_t n, int32_t* __restrict__ cursor, int32_t* __restrict__ inets,
                      int2* __restrict__ adj) {
  extern __shared__ int32_t s_n[];
  const int64_t e0 = (int64_t)m * blockIdx.x / gridDim.x;
  const int64_t e1 = (int64_t)m * (blockIdx.x + 1) / gridDim.x;
  for (int32_t u = threadIdx.x; u < n; u += LOCAL_THREADS) s_n[u] = 0;
  __syncthreads();
  for (int64_t e = e0 + threadIdx.x; e < e1; e += LOCAL_THREADS) {
    const int2 v = pins[e];
    atomicAdd(&s_n[v.x], 1);
    atomicAdd(&s_n[v.y], 1);
  }
  claim_slots(s_n, n, cursor);
  for (int64_t e = e0 + threadIdx.x; e < e1; e += LOCAL_THREADS) {
    const int2 v = pins[e];
    const int32_t we = w[e];
    const int32_t a = atomicAdd(&s_n[v.x], 1), b = atomicAdd(&s_n[v.y], 1);
    inets[a] = (int32_t)e;
    adj[a] = make_int2(v.y, we);
    inets[b] = (int32_t)e;
    adj[b] = make_int2(v.x, we);
  }
}

// Before a launch of one of the local forms.
template <typename K>
void prepare_local(const Ctx& cx, K* kernel) {
  prepare_kernel(cx, kernel, LOCAL_N * sizeof(int32_t));
}

// Scatter every pin (e, v) into I(v) at a slot taken from v's cursor.
__global__ void __launch_bounds__(PIN_TILE_THREADS)
k_scatter_incidence(const int32_t* __restrict__ eoff, const int32_t* __restrict__ pins,
                    const int32_t* __restrict__ tile_net, int32_t m, int64_t p,
                    int32_t* __restrict__ cursor, int32_t* __restrict__ inets) {
  __shared__ int32_t s_off[PIN_TILE + 3];
  const int64_t ntiles = num_pin_tiles(p);
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    PinTileView v = stage_pin_tile(eoff, tile_net, m, p, t, s_off);
    for (int64_t q = v.q0 + threadIdx.x; q < v.q1; q += blockDim.x) {
      const int32_t e = v.e_lo + net_in_tile(s_off, v.count, q);
      inets[atomicAdd(&cursor[pins[q]], 1)] = e;
    }
    __syncthreads();
  }
}

// The same for a graph level (net e's pins at 2 e), with the adjacency array:
// adj[j] = {the other endpoint, w(e)} of incidence j = (u, e).
__global__ void k_scatter_edges(const int2* __restrict__ pins, const int32_t* __restrict__ w,
                                int32_t m, int32_t* __restrict__ cursor,
                                int32_t* __restrict__ inets, int2* __restrict__ adj) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int2 v = pins[e];
    const int32_t we = w[e];
    const int32_t a = atomicAdd(&cursor[v.x], 1), b = atomicAdd(&cursor[v.y], 1);
    inets[a] = (int32_t)e;
    adj[a] = make_int2(v.y, we);
    inets[b] = (int32_t)e;
    adj[b] = make_int2(v.x, we);
  }
}

__global__ void k_validate_nets(const int32_t* __restrict__ eoff, int32_t m,
                                const int32_t* __restrict__ w, int32_t* status,
                                unsigned long long* total_w) {
  int64_t local = 0;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    if (eoff[e + 1] <= eoff[e]) dev_fail(status, DEV_BAD_INPUT);
    const int32_t x = w ? w[e] : 1;
    if (x <= 0) dev_fail(status, DEV_BAD_INPUT);
    local += x;
  }
  local = warp_sum(local);
  if (lane_id() == 0 && local) atomicAdd(total_w, (unsigned long long)local);
}

__global__ void k_validate_pins(const int32_t* __restrict__ pins, int64_t p, int32_t n,
                                int32_t* status) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < p;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int32_t v = pins[q];
    if (v < 0 || v >= n) dev_fail(status, DEV_BAD_INPUT);
  }
}

__global__ void k_validate_nodes(const int32_t* __restrict__ c, int32_t n, int32_t* status,
                                 unsigned long long* total_c) {
  int64_t local = 0;
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x) {
    const int32_t x = c ? c[u] : 1;
    if (x <= 0) dev_fail(status, DEV_BAD_INPUT);
    local += x;
  }
  local = warp_sum(local);
  if (lane_id() == 0 && local) atomicAdd(total_c, (unsigned long long)local);
}

// No node twice in a net.  A warp takes up to 32 nets (fewer when there is a
// warp for each): those of at most DISTINCT_LANE pins a lane each, comparing all
// pairs in registers; those of at most 32 pins by the warp, every lane against half
// of the others.  (A warp per net with a match over its lanes was bound by the match,
// a step per distinct pin: 1.27 ms at 4e6 edges, 0.04 ms now.)  Larger nets are
// listed by size: up to DISTINCT_SMALL pins for k_distinct_mid (a warp and a hash set
// in shared memory each; by the warp that found them, neighbouring nets of 900 pins
// queued up: hg_create with 3000 of them 0.44 -> 0.73 ms), larger ones for
// k_distinct_big (a block that looks for them among all nets waits on two offsets per
// net: 5 of 6 ms at 2e6 nets).  Runs only on offsets and pins already checked, so
// every read stays in bounds.
constexpr int DISTINCT_WARPS = 4;
constexpr int DISTINCT_SMALL = 1024;
constexpr int DISTINCT_LANE = 8;
// largest total of the per-block node bitmaps of k_distinct_big_bitmap
constexpr int64_t DISTINCT_BITMAP_BYTES = 256ll << 20;
constexpr int DISTINCT_SET = 2 * DISTINCT_SMALL;

__device__ __forceinline__ bool set_insert_new(int32_t* set, uint32_t mask, int32_t v) {
  uint32_t h = ((uint32_t)v * 0x9E3779B1u) & mask;
  for (uint32_t probe = 0; probe <= mask; ++probe) {
    const int32_t old = atomicCAS(&set[h], -1, v);
    if (old == -1) return true;
    if (old == v) return false;
    h = (h + 1) & mask;
  }
  return false;  // full: cannot happen at load <= 1/2
}

// Removes v (probing past empty slots: other pins of the net are erased at
// the same time and leave holes in the probe chains).
__device__ __forceinline__ void set_erase(int32_t* set, uint32_t mask, int32_t v) {
  uint32_t h = ((uint32_t)v * 0x9E3779B1u) & mask;
  for (uint32_t probe = 0; probe <= mask; ++probe) {
    if (set[h] == v) {
      set[h] = -1;
      return;
    }
    h = (h + 1) & mask;
  }
}

// The lists of nets of more than 32 pins and their lengths.
struct DistinctLists {
  int32_t *mid, *big, *count;  // count[0]: mid, [1]: big
};

__global__ void __launch_bounds__(DISTINCT_WARPS * 32)
k_distinct_small(const int32_t* __restrict__ eoff, const int32_t* __restrict__ pins, int32_t m,
                 int per, DistinctLists D, int32_t* status) {
  const int wv = warp_in_block(), lane = lane_id();
  const int64_t stride = (int64_t)gridDim.x * DISTINCT_WARPS * per;
  for (int64_t e0 = ((int64_t)blockIdx.x * DISTINCT_WARPS + wv) * per; e0 < m; e0 += stride) {
    const int64_t e = e0 + lane;
    const bool on = lane < per && e < m;
    const int32_t b = on ? eoff[e] : 0, sz = on ? eoff[e + 1] - b : 0;
    bool dup = false;
    if (sz > DISTINCT_SMALL) D.big[atomicAdd(&D.count[1], 1)] = (int32_t)e;
    if (sz <= DISTINCT_LANE) {
      int32_t v[DISTINCT_LANE];
#pragma unroll
      for (int i = 0; i < DISTINCT_LANE; ++i) v[i] = i < sz ? pins[b + i] : -1 - i;
#pragma unroll
      for (int i = 1; i < DISTINCT_LANE; ++i)
#pragma unroll
        for (int j = 0; j < i; ++j) dup |= v[i] == v[j];
    }
    __syncwarp();
    const bool mid = sz > 32 && sz <= DISTINCT_SMALL;
    const unsigned mids = __ballot_sync(FULL, mid);
    if (mids) {
      int32_t at = 0;
      if (lane == 0) at = atomicAdd(&D.count[0], __popc(mids));
      at = __shfl_sync(FULL, at, 0) + __popc(mids & ((1u << lane) - 1u));
      if (mid) D.mid[at] = (int32_t)e;
    }
    unsigned todo = __ballot_sync(FULL, sz > DISTINCT_LANE && sz <= 32);
    while (todo) {
      const int l = __ffs(todo) - 1;
      todo &= todo - 1;
      const int32_t wb = __shfl_sync(FULL, b, l), wsz = __shfl_sync(FULL, sz, l);
      const int32_t v = lane < wsz ? pins[wb + lane] : -1 - lane;
#pragma unroll
      for (int d = 1; d <= 16; ++d) dup |= __shfl_sync(FULL, v, (lane + d) & 31) == v;
    }
    if (__any_sync(FULL, dup) && lane == 0) dev_fail(status, DEV_BAD_INPUT);
  }
}

__global__ void __launch_bounds__(DISTINCT_WARPS * 32)
k_distinct_mid(const int32_t* __restrict__ eoff, const int32_t* __restrict__ pins,
               DistinctLists D, int32_t* status) {
  __shared__ int32_t s_set[DISTINCT_WARPS][DISTINCT_SET];
  const int wv = warp_in_block(), lane = lane_id();
  int32_t* set = s_set[wv];
  const int32_t cnt = D.count[0];
  int32_t x = wv * gridDim.x + blockIdx.x;
  if (x >= cnt) return;
  for (int i = lane; i < DISTINCT_SET; i += 32) set[i] = -1;
  __syncwarp();
  for (; x < cnt; x += gridDim.x * DISTINCT_WARPS) {
    const int32_t e = D.mid[x], b = eoff[e], sz = eoff[e + 1] - b;
    bool dup = false;
    for (int32_t q = lane; q < sz; q += 32)
      dup |= !set_insert_new(set, DISTINCT_SET - 1, pins[b + q]);
    __syncwarp();
    for (int32_t q = lane; q < sz; q += 32) set_erase(set, DISTINCT_SET - 1, pins[b + q]);
    __syncwarp();
    if (__any_sync(FULL, dup) && lane == 0) dev_fail(status, DEV_BAD_INPUT);
  }
}

// Nets above DISTINCT_SMALL pins: one block per net with a hash set of `cap`
// slots (a power of two >= twice the largest net) in this block's region of
// `scratch` (all slots -1 on entry, restored before the block moves on).
__global__ void k_distinct_big(const int32_t* __restrict__ eoff, const int32_t* __restrict__ pins,
                               const int32_t* __restrict__ big, const int32_t* __restrict__ nbig,
                               int32_t* __restrict__ scratch, uint32_t cap, int32_t* status) {
  int32_t* set = scratch + (size_t)blockIdx.x * cap;
  __shared__ int s_dup;
  const int32_t cnt = *nbig;
  for (int32_t x = blockIdx.x; x < cnt; x += gridDim.x) {
    const int32_t e = big[x];
    const int32_t b = eoff[e], sz = eoff[e + 1] - b;
    if (threadIdx.x == 0) s_dup = 0;
    __syncthreads();
    bool dup = false;
    for (int32_t q = threadIdx.x; q < sz; q += blockDim.x) dup |= !set_insert_new(set, cap - 1, pins[b + q]);
    if (dup) s_dup = 1;
    __syncthreads();
    for (int32_t q = threadIdx.x; q < sz; q += blockDim.x) set_erase(set, cap - 1, pins[b + q]);
    if (threadIdx.x == 0 && s_dup) dev_fail(status, DEV_BAD_INPUT);
    __syncthreads();
  }
}

// The same check with a bitmap of the n nodes per block (n bits), when the
// bitmaps of all blocks are small: one atomicOr per pin finds a repeat and one
// atomicAnd per pin clears the net's bits again, with no probing.
__global__ void k_distinct_big_bitmap(const int32_t* __restrict__ eoff,
                                      const int32_t* __restrict__ pins,
                                      const int32_t* __restrict__ big,
                                      const int32_t* __restrict__ nbig,
                                      uint32_t* __restrict__ scratch, int64_t words,
                                      int32_t* status) {
  uint32_t* set = scratch + (size_t)blockIdx.x * (size_t)words;
  __shared__ int s_dup;
  const int32_t cnt = *nbig;
  for (int32_t x = blockIdx.x; x < cnt; x += gridDim.x) {
    const int32_t e = big[x];
    const int32_t b = eoff[e], sz = eoff[e + 1] - b;
    if (threadIdx.x == 0) s_dup = 0;
    __syncthreads();
    bool dup = false;
    for (int32_t q = threadIdx.x; q < sz; q += blockDim.x) {
      const int32_t v = pins[b + q];
      const uint32_t bit = 1u << (v & 31);
      dup |= (atomicOr(&set[v >> 5], bit) & bit) != 0;
    }
    if (dup) s_dup = 1;
    __syncthreads();
    for (int32_t q = threadIdx.x; q < sz; q += blockDim.x) {
      const int32_t v = pins[b + q];
      atomicAnd(&set[v >> 5], ~(1u << (v & 31)));
    }
    if (threadIdx.x == 0 && s_dup) dev_fail(status, DEV_BAD_INPUT);
    __syncthreads();
  }
}

__global__ void k_max_net_size(const int32_t* __restrict__ eoff, int32_t m, int32_t* out) {
  int32_t mx = 0;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x)
    mx = max(mx, eoff[e + 1] - eoff[e]);
  mx = warp_max(mx);
  if (lane_id() == 0 && mx) atomicMax(out, mx);
}

__global__ void k_net_size_range(const int32_t* __restrict__ eoff, int32_t m,
                                 int32_t* __restrict__ out) {
  int32_t lo = 0x7fffffff, hi = 0;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int32_t sz = eoff[e + 1] - eoff[e];
    lo = min(lo, sz);
    hi = max(hi, sz);
  }
  lo = warp_min(lo);
  hi = warp_max(hi);
  if (lane_id() == 0) {
    atomicMin(&out[0], lo);
    atomicMax(&out[1], hi);
  }
}

}  // namespace

bool level_is_graph(const Ctx& cx, const Level& L) {
  if (L.m <= 0) return false;
  DBuf<int32_t> range;
  range.alloc(&cx.alloc, 2);
  const int32_t init[2] = {0x7fffffff, 0};
  HG_CUDA(cudaMemcpyAsync(range.p, init, sizeof(init), cudaMemcpyHostToDevice, cx.stream));
  k_net_size_range<<<grid_for(L.m, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(L.eoff.p, L.m,
                                                                            range.p);
  check_launch("net_size_range");
  if (cx.launches) *cx.launches += 1;
  int32_t h[2];
  read_back(cx, h, range.p, sizeof(h));
  return h[0] == 2 && h[1] == 2;
}

void build_tile_index(const Ctx& cx, const int32_t* eoff, int32_t m, int64_t p, int32_t* tile_net) {
  const int64_t ntiles = num_pin_tiles(p);
  k_tile_index<<<grid_for(m > 0 ? m : 1, 256, cx.num_sms, 16), 256, 0, cx.stream>>>(eoff, m, ntiles,
                                                                                  tile_net);
  check_launch("tile_index");
  if (cx.launches) *cx.launches += 1;
}

void build_incidence(const Ctx& cx, Level& L) {
  L.ioff.alloc(&cx.alloc, (size_t)L.n + 1);
  L.inets.alloc(&cx.alloc, (size_t)(L.p > 0 ? L.p : 1));
  if (L.graph) L.adj.alloc(&cx.alloc, (size_t)(L.p > 0 ? L.p : 1));
  HG_CUDA(cudaMemsetAsync(L.ioff.p, 0, sizeof(int32_t) * ((size_t)L.n + 1), cx.stream));
  const int local = L.p > 0 ? local_blocks(cx, L.n, L.p, num_pin_tiles(L.p)) : 0;
  const size_t smem = (size_t)L.n * sizeof(int32_t);
  if (local) {
    prepare_local(cx, k_degrees_local);
    k_degrees_local<<<local, LOCAL_THREADS, smem, cx.stream>>>(L.pins.p, L.p, L.n, L.ioff.p);
    check_launch("degrees_local");
  } else if (L.p > 0) {
    k_degrees<<<grid_for(L.p, 256, cx.num_sms, 16), 256, 0, cx.stream>>>(L.pins.p, L.p, L.ioff.p);
    check_launch("degrees");
  }
  scan_exclusive_i32(cx, L.ioff.p, L.ioff.p, L.n, L.ioff.p + L.n);
  if (L.p > 0) {
    DBuf<int32_t> cursor, tiles;
    cursor.alloc(&cx.alloc, (size_t)L.n);
    HG_CUDA(cudaMemcpyAsync(cursor.p, L.ioff.p, sizeof(int32_t) * (size_t)L.n,
                            cudaMemcpyDeviceToDevice, cx.stream));
    if (L.graph) {
      const int2* edges = reinterpret_cast<const int2*>(L.pins.p);
      if (local) {
        prepare_local(cx, k_scatter_edges_local);
        k_scatter_edges_local<<<local, LOCAL_THREADS, smem, cx.stream>>>(
            edges, L.w.p, L.m, L.n, cursor.p, L.inets.p, L.adj.p);
      } else {
        k_scatter_edges<<<grid_for(L.m, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(
            edges, L.w.p, L.m, cursor.p, L.inets.p, L.adj.p);
      }
    } else {
      tiles.alloc(&cx.alloc, (size_t)num_pin_tiles(L.p) + 1);
      build_tile_index(cx, L.eoff.p, L.m, L.p, tiles.p);
      if (local) {
        prepare_local(cx, k_scatter_incidence_local);
        k_scatter_incidence_local<<<local, LOCAL_THREADS, smem, cx.stream>>>(
            L.eoff.p, L.pins.p, tiles.p, L.m, L.p, L.n, cursor.p, L.inets.p);
      } else {
        k_scatter_incidence<<<grid_for(num_pin_tiles(L.p), 1, cx.num_sms, 8), PIN_TILE_THREADS, 0,
                              cx.stream>>>(L.eoff.p, L.pins.p, tiles.p, L.m, L.p, cursor.p,
                                           L.inets.p);
      }
    }
    check_launch("scatter_incidence");
    if (cx.launches) *cx.launches += 2;
  }
  if (cx.launches) *cx.launches += 1;
}

namespace {

// No node twice in a net (offsets and pin ranges already valid).
bool distinct_pins(const Ctx& cx, const Level& L) {
  if (L.m <= 0) return true;
  DBuf<int32_t> mx;
  mx.alloc(&cx.alloc, 1);
  HG_CUDA(cudaMemsetAsync(mx.p, 0, sizeof(int32_t), cx.stream));
  k_max_net_size<<<grid_for(L.m, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(L.eoff.p, L.m, mx.p);
  check_launch("max_net_size");
  DBuf<int32_t> lists;  // nets of 33 pins and more, of more than DISTINCT_SMALL, lengths
  const size_t nmid = (size_t)(L.p / 33) + 1, nb = (size_t)(L.p / (DISTINCT_SMALL + 1)) + 1;
  lists.alloc(&cx.alloc, nmid + nb + 2);
  const DistinctLists D{lists.p, lists.p + nmid, lists.p + nmid + nb};
  const int32_t *big = D.big, *nbig = D.count + 1;
  HG_CUDA(cudaMemsetAsync(D.count, 0, 2 * sizeof(int32_t), cx.stream));
  const int64_t warps = (int64_t)cx.num_sms * 6 * DISTINCT_WARPS;
  const int per = (int)std::min<int64_t>(32, (L.m + warps - 1) / warps);
  k_distinct_small<<<grid_for(L.m, DISTINCT_WARPS * per, cx.num_sms, 6), DISTINCT_WARPS * 32, 0,
                     cx.stream>>>(L.eoff.p, L.pins.p, L.m, per, D, cx.d_status);
  check_launch("distinct_small");
  k_distinct_mid<<<grid_for(L.p, 33 * DISTINCT_WARPS, cx.num_sms, 6), DISTINCT_WARPS * 32, 0,
                   cx.stream>>>(L.eoff.p, L.pins.p, D, cx.d_status);
  check_launch("distinct_mid");
  const int32_t biggest = read_i32(cx, mx.p);
  const int64_t words = ((int64_t)L.n + 31) / 32;
  if (biggest > DISTINCT_SMALL && (int64_t)cx.num_sms * words * 4 <= DISTINCT_BITMAP_BYTES) {
    const int blocks = cx.num_sms;
    DBuf<uint32_t> scratch;
    scratch.alloc(&cx.alloc, (size_t)blocks * (size_t)words);
    HG_CUDA(cudaMemsetAsync(scratch.p, 0, scratch.bytes(), cx.stream));
    k_distinct_big_bitmap<<<blocks, 1024, 0, cx.stream>>>(L.eoff.p, L.pins.p, big, nbig,
                                                          scratch.p, words, cx.d_status);
    check_launch("distinct_big_bitmap");
  } else if (biggest > DISTINCT_SMALL) {
    uint32_t cap = 1;
    while (cap < 2u * (uint32_t)biggest) cap <<= 1;
    const int blocks = cx.num_sms;
    DBuf<int32_t> scratch;
    scratch.alloc(&cx.alloc, (size_t)blocks * cap);
    HG_CUDA(cudaMemsetAsync(scratch.p, 0xff, scratch.bytes(), cx.stream));
    k_distinct_big<<<blocks, 1024, 0, cx.stream>>>(L.eoff.p, L.pins.p, big, nbig, scratch.p,
                                                   cap, cx.d_status);
    check_launch("distinct_big");
  }
  if (read_status(cx, nullptr, nullptr, 0) != DEV_OK) {
    int32_t zero = 0;
    HG_CUDA(cudaMemcpy(cx.d_status, &zero, sizeof(zero), cudaMemcpyHostToDevice));
    return false;
  }
  return true;
}

}  // namespace

bool validate_pins_device(const Ctx& cx, const Level& L) {
  if (L.p > 0) {
    k_validate_pins<<<grid_for(L.p, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(L.pins.p, L.p, L.n,
                                                                             cx.d_status);
    check_launch("validate_pins");
    if (read_status(cx, nullptr, nullptr, 0) != DEV_OK) {
      int32_t zero = 0;
      HG_CUDA(cudaMemcpy(cx.d_status, &zero, sizeof(zero), cudaMemcpyHostToDevice));
      return false;
    }
  }
  return distinct_pins(cx, L);
}

bool validate_level_device(const Ctx& cx, const Level& L, int64_t* total_node_w,
                           int64_t* total_net_w) {
  DBuf<unsigned long long> sums;
  sums.alloc(&cx.alloc, 2);
  HG_CUDA(cudaMemsetAsync(sums.p, 0, 2 * sizeof(unsigned long long), cx.stream));
  if (L.m > 0) {
    k_validate_nets<<<grid_for(L.m, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(
        L.eoff.p, L.m, L.w.p, cx.d_status, sums.p + 1);
    check_launch("validate_nets");
  }
  if (L.p > 0) {
    k_validate_pins<<<grid_for(L.p, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(L.pins.p, L.p, L.n,
                                                                             cx.d_status);
    check_launch("validate_pins");
  }
  k_validate_nodes<<<grid_for(L.n, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(L.c.p, L.n,
                                                                           cx.d_status, sums.p);
  check_launch("validate_nodes");
  unsigned long long h[2] = {0, 0};
  if (read_status(cx, h, sums.p, sizeof(h)) != DEV_OK) {
    int32_t zero = 0;
    HG_CUDA(cudaMemcpy(cx.d_status, &zero, sizeof(zero), cudaMemcpyHostToDevice));
    return false;
  }
  // offsets and pins are sound: no node twice in a net
  if (!distinct_pins(cx, L)) return false;
  *total_node_w = (int64_t)h[0];
  *total_net_w = (int64_t)h[1];
  return true;
}

}  // namespace hgk
