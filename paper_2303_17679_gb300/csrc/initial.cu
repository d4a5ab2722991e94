// Seeded initial partition (Sec. 5 is replaced by one deterministic rule): nodes
// in order of (mix64(seed ^ 2^63 ^ u), u), each to the lightest block so far, ties
// to the smaller block id.
//
// The order: mix64 is a bijection, so the keys are distinct and spread evenly;
// nodes are scattered into about n / 8 buckets by their keys' top bits and ranked
// within their bucket by counting.  The assignment is sequential by definition:
// one warp holds the block weights, one block per lane and register, and a step
// is one warp-wide minimum over {weight, block} words (about 26 ns, the latency of
// the chain minimum - compare - add).  On the host the same took a copy each way, a
// sort and a scan of k weights per node: 26 ms at n = 262,725, k = 64 (device:
// 7.2 ms), 0.33 ms at n = 4445, k = 32 (0.16 ms).
#include <algorithm>

#include "common.cuh"

namespace hgk {

namespace {

__device__ __forceinline__ uint64_t order_key(uint64_t seed, int32_t u) {
  return mix64(seed ^ (1ull << 63) ^ (uint64_t)(uint32_t)u);
}

// Nodes per bucket, and the largest node weight.
__global__ void k_init_count(const int32_t* __restrict__ c, int32_t n, uint64_t seed, int shift,
                             int32_t* __restrict__ cnt, int32_t* __restrict__ max_c) {
  int32_t mx = 0;
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x) {
    atomicAdd(&cnt[order_key(seed, (int32_t)u) >> shift], 1);
    mx = max(mx, c[u]);
  }
  mx = warp_max(mx);
  if (lane_id() == 0 && mx) atomicMax(max_c, mx);
}

__global__ void k_init_scatter(int32_t n, uint64_t seed, int shift,
                               const int32_t* __restrict__ off, int32_t* __restrict__ fill,
                               int32_t* __restrict__ nodes) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t b = order_key(seed, (int32_t)u) >> shift;
    nodes[off[b] + atomicAdd(&fill[b], 1)] = (int32_t)u;
  }
}

// {u, c(u)} in the order of the keys.
__global__ void k_init_rank(const int32_t* __restrict__ nodes, int32_t n, uint64_t seed, int shift,
                            const int32_t* __restrict__ off, const int32_t* __restrict__ c,
                            int2* __restrict__ order) {
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
       x += (int64_t)gridDim.x * blockDim.x) {
    const int32_t u = nodes[x];
    const uint64_t key = order_key(seed, u);
    const uint64_t b = key >> shift;
    const int32_t lo = off[b], hi = off[b + 1];
    int32_t rank = 0;
    for (int32_t y = lo; y < hi; ++y) rank += order_key(seed, nodes[y]) < key;
    order[lo + rank] = make_int2(u, c[u]);
  }
}

// Weights up to this fit the packed words: a batch of 32 nodes starts with block
// weights at most max_c above the lightest (each block was the lightest when it
// got its last node), so they stay below 33 * 2^20 < 2^26.
constexpr int32_t PACK_MAX_C = 1 << 20;

// The assignment by one warp, 32 nodes at a time: lane l holds the weights of
// blocks l and l + 32, relative to the lightest at the start of the batch.
__device__ __forceinline__ void assign_in_order(const int2* __restrict__ order, int32_t n, int k,
                                                bool packed, int32_t* __restrict__ part) {
  const int lane = lane_id();
  // weight << 6 | block, or the weight alone; all ones for no block.  Unpacked, a
  // block's weight is at most c(V) < 2^31 (hg_create).
  unsigned w0 = lane < k ? (packed ? (unsigned)lane : 0u) : ~0u;
  unsigned w1 = lane + 32 < k ? (packed ? (unsigned)lane + 32u : 0u) : ~0u;
  int2 next = lane < n ? order[lane] : make_int2(0, 0);
  for (int64_t i0 = 0; i0 < n; i0 += 32) {
    const int2 nd = next;
    next = i0 + 32 + lane < n ? order[i0 + 32 + lane] : make_int2(0, 0);
    const int count = n - i0 < 32 ? (int)(n - i0) : 32;
    int mine = 0;
    if (packed) {
      const unsigned base = __reduce_min_sync(FULL, min(w0, w1)) & ~63u;
      if (lane < k) w0 -= base;
      if (lane + 32 < k) w1 -= base;
      for (int i = 0; i < count; ++i) {
        const unsigned add = (unsigned)__shfl_sync(FULL, nd.y, i) << 6;
        const int b = (int)(__reduce_min_sync(FULL, min(w0, w1)) & 63u);
        if (lane == b) w0 += add;
        if (lane + 32 == b) w1 += add;
        if (lane == i) mine = b;
      }
    } else {
      for (int i = 0; i < count; ++i) {
        const unsigned add = (unsigned)__shfl_sync(FULL, nd.y, i);
        const unsigned m = __reduce_min_sync(FULL, min(w0, w1));
        const unsigned lower = __ballot_sync(FULL, w0 == m && lane < k);
        const unsigned upper = __ballot_sync(FULL, w1 == m && lane + 32 < k);
        const int b = lower ? __ffs(lower) - 1 : 31 + __ffs(upper);
        if (lane == b) w0 += add;
        if (lane + 32 == b) w1 += add;
        if (lane == i) mine = b;
      }
    }
    if (i0 + lane < n) part[nd.x] = mine;
  }
}

__global__ void __launch_bounds__(32)
k_init_assign(const int2* __restrict__ order, int32_t n, int k, const int32_t* __restrict__ max_c,
              int32_t* __restrict__ part) {
  assign_in_order(order, n, k, *max_c <= PACK_MAX_C, part);
}

// Levels of at most INIT_SMALL nodes: the same in one launch, buckets and order in
// shared memory (n = 746, k = 8: 100 us as separate launches, 50 us).
constexpr int INIT_THREADS = 1024;
constexpr int INIT_PER = 8;
constexpr int INIT_SMALL = INIT_THREADS * INIT_PER;
constexpr int INIT_BITS = 10;  // a bucket per thread
constexpr size_t INIT_SMEM = (size_t)INIT_SMALL * (sizeof(int2) + sizeof(int32_t));

__global__ void __launch_bounds__(INIT_THREADS)
k_init_small(const int32_t* __restrict__ c, int32_t n, uint64_t seed, int k,
             int32_t* __restrict__ part) {
  static_assert((1 << INIT_BITS) == INIT_THREADS, "a bucket per thread");
  extern __shared__ int2 s_order[];
  int32_t* s_nodes = reinterpret_cast<int32_t*>(s_order + INIT_SMALL);
  __shared__ int32_t s_cnt[INIT_THREADS + 1];
  __shared__ int32_t s_wsum[32];
  __shared__ int32_t s_max;
  const int t = threadIdx.x;
  constexpr int shift = 64 - INIT_BITS;
  s_cnt[t] = 0;
  if (t == 0) {
    s_cnt[INIT_THREADS] = n;
    s_max = 0;
  }
  __syncthreads();
  int32_t slot[INIT_PER];
  int32_t mx = 0;
#pragma unroll
  for (int r = 0; r < INIT_PER; ++r) {
    const int32_t u = r * INIT_THREADS + t;
    if (u < n) {
      slot[r] = atomicAdd(&s_cnt[order_key(seed, u) >> shift], 1);
      mx = max(mx, c[u]);
    }
  }
  mx = warp_max(mx);
  if (lane_id() == 0 && mx) atomicMax(&s_max, mx);
  __syncthreads();
  const int32_t mine = s_cnt[t];
  const int32_t incl = warp_inclusive_scan(mine);
  if (lane_id() == 31) s_wsum[warp_in_block()] = incl;
  __syncthreads();
  int32_t before = 0;
  for (int w = 0; w < warp_in_block(); ++w) before += s_wsum[w];
  s_cnt[t] = before + incl - mine;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < INIT_PER; ++r) {
    const int32_t u = r * INIT_THREADS + t;
    if (u < n) s_nodes[s_cnt[order_key(seed, u) >> shift] + slot[r]] = u;
  }
  __syncthreads();
  for (int32_t x = t; x < n; x += INIT_THREADS) {
    const int32_t u = s_nodes[x];
    const uint64_t key = order_key(seed, u);
    const int32_t lo = s_cnt[key >> shift], hi = s_cnt[(key >> shift) + 1];
    int32_t rank = 0;
    for (int32_t y = lo; y < hi; ++y) rank += order_key(seed, s_nodes[y]) < key;
    s_order[lo + rank] = make_int2(u, c[u]);
  }
  __syncthreads();
  if (t < 32) assign_in_order(s_order, n, k, s_max <= PACK_MAX_C, part);
}

}  // namespace

void initial_partition(const Ctx& cx, const Level& L, int k, uint64_t seed, int32_t* part) {
  const int32_t n = L.n;
  if (n <= 0) return;
  if (n <= INIT_SMALL) {
    prepare_kernel(cx, k_init_small, INIT_SMEM);
    k_init_small<<<1, INIT_THREADS, INIT_SMEM, cx.stream>>>(L.c.p, n, seed, k, part);
    check_launch("init_small");
    if (cx.launches) *cx.launches += 1;
    return;
  }
  int bits = 0;  // about 8 nodes per bucket
  while (bits < 27 && (8ll << bits) < n) ++bits;
  const int64_t buckets = 1ll << bits;
  const int shift = 64 - bits;
  DBuf<int32_t> cnt, fill, nodes, max_c;
  DBuf<int2> order;
  cnt.alloc(&cx.alloc, (size_t)buckets + 1);
  fill.alloc(&cx.alloc, (size_t)buckets);
  nodes.alloc(&cx.alloc, (size_t)n);
  order.alloc(&cx.alloc, (size_t)n);
  max_c.alloc(&cx.alloc, 1);
  HG_CUDA(cudaMemsetAsync(cnt.p, 0, cnt.bytes(), cx.stream));
  HG_CUDA(cudaMemsetAsync(fill.p, 0, fill.bytes(), cx.stream));
  HG_CUDA(cudaMemsetAsync(max_c.p, 0, max_c.bytes(), cx.stream));
  const int g = grid_for(n, 256, cx.num_sms, 8);
  k_init_count<<<g, 256, 0, cx.stream>>>(L.c.p, n, seed, shift, cnt.p, max_c.p);
  check_launch("init_count");
  scan_exclusive_i32(cx, cnt.p, cnt.p, buckets, cnt.p + buckets);
  k_init_scatter<<<g, 256, 0, cx.stream>>>(n, seed, shift, cnt.p, fill.p, nodes.p);
  check_launch("init_scatter");
  k_init_rank<<<g, 256, 0, cx.stream>>>(nodes.p, n, seed, shift, cnt.p, L.c.p, order.p);
  check_launch("init_rank");
  k_init_assign<<<1, 32, 0, cx.stream>>>(order.p, n, k, max_c.p, part);
  check_launch("init_assign");
  if (cx.launches) *cx.launches += 4;
}

}  // namespace hgk
