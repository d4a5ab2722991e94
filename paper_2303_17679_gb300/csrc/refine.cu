// Projection (Algorithm 1), pin counts and connectivity sets (Sec. 2, Sec. 6.1
// data layout) and the connectivity objective (Sec. 2) on the device.  Label
// propagation is in lp.cu.
//
// Layout: Phi is a dense m x k int32 table (row = net), Lambda one 64-bit
// mask per net (k <= 64), block weights int64[k].
#include <algorithm>

#include "common.cuh"

namespace hgk {

namespace {

// ------------------------------------------------------------ projection

__global__ void k_project(const int32_t* __restrict__ map, const int32_t* __restrict__ coarse_part,
                          int32_t n, int32_t* __restrict__ fine_part) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x)
    fine_part[u] = coarse_part[map[u]];
}

// ------------------------------------------------------ pin counts (a10)

// Phi, and Lambda or the packed records (gain.cuh), of every net: a net's pins
// are counted per block in shared memory by eight lanes (up to COUNT_SMALL
// pins) or a warp (up to COUNT_WARP), which then write the net's row of Phi and its
// masks once.  Larger nets: by chunks over the grid, added to the row (as one block's,
// a net of 20M pins took 24 ms, 1.2 now); on levels of at most COUNT_LEVEL pins by
// the block, after its other nets (the launch for the chunks costs 7 of 700 us of
// label propagation at n = 10,000).  Bound by the row writes on levels of small nets (m
// k words), by the pins' block ids on the others.  (A thread per pin that found
// equal (net, block) pairs by a match over the warp and added them with atomics to
// a cleared table, and a second pass for the records, took 0.53 + 0.23 ms per
// level of 35e6 pins at k = 64; 0.27 ms now.)
constexpr int COUNT_WARPS = 8, COUNT_LANES = 8;
constexpr int COUNT_NETS = 32 / COUNT_LANES;
constexpr int32_t COUNT_SMALL = 64, COUNT_WARP = 2048;
constexpr int COUNT_STRIDE = HG_MAX_K + 1;  // a warp's sets start in different banks
constexpr int32_t COUNT_CHUNK = 4096;
constexpr int64_t COUNT_LEVEL = 1 << 17;
constexpr int COUNT_BIG = 64;               // nets a block keeps for later

struct CountArgs {
  const int32_t *eoff, *pins, *part, *w;
  int32_t m;
  int k;
  int32_t* phi;             // when asked for
  unsigned long long* lam;  // or
  int4* rec;
  // chunks of the nets above COUNT_WARP: {net, its first chunk}, their number, and
  // the chunks done per net (at its first chunk); NULL on small levels
  int2* chunks;
  int32_t *nchunks, *done;
};

// Writes the row of net e from `sets` sets of counters `stride` apart and clears
// them; the lanes l = 0 .. W-1 of the caller share the blocks.  The masks of
// their blocks are returned.
template <int W, bool PHI>
__device__ __forceinline__ void write_row(const CountArgs& A, int32_t e, int32_t* cnt, int sets,
                                          int l, unsigned long long& ones,
                                          unsigned long long& lam) {
  ones = lam = 0;
  for (int t = l; t < A.k; t += W) {
    int32_t c = 0;
    for (int x = 0; x < sets; ++x) {
      c += cnt[x * COUNT_STRIDE + t];
      cnt[x * COUNT_STRIDE + t] = 0;
    }
    if (PHI) A.phi[(int64_t)e * A.k + t] = c;
    if (c == 1) ones |= 1ull << t;
    if (c > 0) lam |= 1ull << t;
  }
}

__device__ __forceinline__ void write_masks(const CountArgs& A, int32_t e, unsigned long long ones,
                                            unsigned long long lam) {
  if (A.lam) A.lam[e] = lam;
  if (!A.rec) return;
  const int32_t w = A.w[e];
  const int H = A.k > 32 ? 2 : 1;
  for (int h = 0; h < H; ++h)
    A.rec[(int64_t)H * e + h] = make_int4(w, (int32_t)(uint32_t)(ones >> (32 * h)),
                                          (int32_t)(uint32_t)(lam >> (32 * h)), 0);
}

template <int W>
__device__ __forceinline__ unsigned long long or_lanes(unsigned long long x) {
#pragma unroll
  for (int d = W / 2; d > 0; d >>= 1) x |= __shfl_xor_sync(FULL, x, d);
  return x;
}

// Counts the pins [b, b + sz), this thread number i of `threads`, four at a time.
__device__ __forceinline__ void count_pins(const CountArgs& A, int32_t b, int32_t sz, int i,
                                           int threads, int32_t* cnt) {
  for (int32_t q0 = i; q0 < sz; q0 += 4 * threads) {
    int32_t v[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int64_t q = (int64_t)q0 + x * threads;
      v[x] = q < sz ? A.pins[b + q] : -1;
    }
#pragma unroll
    for (int x = 0; x < 4; ++x)
      if (v[x] >= 0) v[x] = A.part[v[x]];
#pragma unroll
    for (int x = 0; x < 4; ++x)
      if (v[x] >= 0) atomicAdd(&cnt[v[x]], 1);
  }
}

// PHI: the counts themselves, else only Lambda.
template <bool PHI>
__global__ void __launch_bounds__(COUNT_WARPS * 32, 8) k_pin_counts(CountArgs A) {
  __shared__ int32_t s_cnt[COUNT_WARPS * COUNT_NETS * COUNT_STRIDE];
  __shared__ int32_t s_big[COUNT_BIG];
  __shared__ int s_nbig;
  __shared__ unsigned long long s_ones, s_lam;
  const int lane = lane_id(), sub = lane % COUNT_LANES, grp = lane / COUNT_LANES;
  int32_t* sets = s_cnt + warp_in_block() * COUNT_NETS * COUNT_STRIDE;
  int32_t* mine = sets + grp * COUNT_STRIDE;
  for (int i = threadIdx.x; i < COUNT_WARPS * COUNT_NETS * COUNT_STRIDE; i += blockDim.x)
    s_cnt[i] = 0;
  if (threadIdx.x == 0) s_nbig = 0;
  __syncthreads();
  auto by_warp = [&](int32_t e, int32_t b, int32_t sz) {
    count_pins(A, b, sz, lane, 32, mine);
    __syncwarp();
    unsigned long long ones, lam;
    write_row<32, PHI>(A, e, sets, COUNT_NETS, lane, ones, lam);
    ones = or_lanes<32>(ones);
    lam = or_lanes<32>(lam);
    if (lane == 0) write_masks(A, e, ones, lam);
    __syncwarp();
  };
  const int64_t stride = (int64_t)gridDim.x * COUNT_WARPS * COUNT_NETS;
  for (int64_t e0 = ((int64_t)blockIdx.x * COUNT_WARPS + warp_in_block()) * COUNT_NETS; e0 < A.m;
       e0 += stride) {
    const int64_t e = e0 + grp;
    const bool on = e < A.m;
    const int32_t b = on ? A.eoff[e] : 0, sz = on ? A.eoff[e + 1] - b : 0;
    if (sz <= COUNT_SMALL) count_pins(A, b, sz, sub, COUNT_LANES, mine);
    __syncwarp();
    unsigned long long ones = 0, lam = 0;
    if (on && sz <= COUNT_SMALL) write_row<COUNT_LANES, PHI>(A, (int32_t)e, mine, 1, sub, ones, lam);
    __syncwarp();
    ones = or_lanes<COUNT_LANES>(ones);
    lam = or_lanes<COUNT_LANES>(lam);
    if (on && sub == 0 && sz <= COUNT_SMALL) write_masks(A, (int32_t)e, ones, lam);
    for (unsigned rest = __ballot_sync(FULL, sub == 0 && sz > COUNT_SMALL); rest;
         rest &= rest - 1) {
      const int l = __ffs(rest) - 1;
      const int32_t we = (int32_t)(e0 + l / COUNT_LANES);
      const int32_t wb = __shfl_sync(FULL, b, l), wsz = __shfl_sync(FULL, sz, l);
      if (wsz > COUNT_WARP && A.chunks) {
        const int32_t count = (wsz + COUNT_CHUNK - 1) / COUNT_CHUNK;
        int32_t first = 0;
        if (lane == 0) first = atomicAdd(A.nchunks, count);
        first = __shfl_sync(FULL, first, 0);
        for (int32_t c = lane; c < count; c += 32) A.chunks[first + c] = make_int2(we, first);
        if (PHI)
          for (int t = lane; t < A.k; t += 32) A.phi[(int64_t)we * A.k + t] = 0;
        else if (lane == 0)
          A.lam[we] = 0;
        continue;
      }
      int slot = COUNT_BIG;
      if (wsz > COUNT_WARP) {
        if (lane == 0) slot = atomicAdd(&s_nbig, 1);
        slot = __shfl_sync(FULL, slot, 0);
        if (slot < COUNT_BIG && lane == 0) s_big[slot] = we;
      }
      if (slot >= COUNT_BIG) by_warp(we, wb, wsz);
    }
  }
  __syncthreads();
  const int big = min(s_nbig, COUNT_BIG);
  for (int x = 0; x < big; ++x) {
    const int32_t e = s_big[x], b = A.eoff[e], sz = A.eoff[e + 1] - b;
    count_pins(A, b, sz, threadIdx.x, COUNT_WARPS * 32, mine);
    if (threadIdx.x == 0) s_ones = s_lam = 0;
    __syncthreads();
    unsigned long long ones, lam;
    write_row<COUNT_WARPS * 32, PHI>(A, e, s_cnt, COUNT_WARPS * COUNT_NETS, threadIdx.x, ones, lam);
    if (ones) atomicOr(&s_ones, ones);
    if (lam) atomicOr(&s_lam, lam);
    __syncthreads();
    if (threadIdx.x == 0) write_masks(A, e, s_ones, s_lam);
    __syncthreads();
  }
}

// The chunks listed by k_pin_counts: a block counts one in shared memory and adds it
// to the net's row; the last chunk of a net writes its masks.
template <bool PHI>
__global__ void __launch_bounds__(COUNT_WARPS * 32) k_pin_counts_huge(CountArgs A) {
  __shared__ int32_t s_cnt[COUNT_WARPS * COUNT_STRIDE];
  __shared__ unsigned long long s_ones, s_lam;
  __shared__ int s_last;
  for (int i = threadIdx.x; i < COUNT_WARPS * COUNT_STRIDE; i += blockDim.x) s_cnt[i] = 0;
  __syncthreads();
  int32_t* mine = s_cnt + warp_in_block() * COUNT_STRIDE;
  const int32_t n = *A.nchunks;
  const int t = threadIdx.x;
  for (int32_t x = blockIdx.x; x < n; x += gridDim.x) {
    const int2 it = A.chunks[x];
    const int32_t e = it.x, b = A.eoff[e], sz = A.eoff[e + 1] - b;
    const int32_t at = (x - it.y) * COUNT_CHUNK, left = min(COUNT_CHUNK, sz - at);
    count_pins(A, b + at, left, t, COUNT_WARPS * 32, mine);
    if (t == 0) s_ones = s_lam = 0;
    __syncthreads();
    int32_t c = 0;
    if (t < A.k)
      for (int w = 0; w < COUNT_WARPS; ++w) {
        c += s_cnt[w * COUNT_STRIDE + t];
        s_cnt[w * COUNT_STRIDE + t] = 0;
      }
    if (!PHI) {
      if (c) atomicOr(&A.lam[e], 1ull << t);
      __syncthreads();
      continue;
    }
    if (c) atomicAdd(&A.phi[(int64_t)e * A.k + t], c);
    __threadfence();
    __syncthreads();
    if (t == 0) s_last = atomicAdd(&A.done[it.y], 1) == (sz + COUNT_CHUNK - 1) / COUNT_CHUNK - 1;
    __syncthreads();
    if (s_last) {
      __threadfence();
      if (t < A.k) {
        const int32_t all = __ldcg(&A.phi[(int64_t)e * A.k + t]);
        if (all == 1) atomicOr(&s_ones, 1ull << t);
        if (all > 0) atomicOr(&s_lam, 1ull << t);
      }
      __syncthreads();
      if (t == 0) write_masks(A, e, s_ones, s_lam);
    }
    __syncthreads();
  }
}

__global__ void k_block_weights(const int32_t* __restrict__ part, const int32_t* __restrict__ c,
                                int32_t n, int k, long long* __restrict__ bw) {
  __shared__ long long s_bw[HG_MAX_K];
  for (int i = threadIdx.x; i < k; i += blockDim.x) s_bw[i] = 0;
  __syncthreads();
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x)
    atomic_add_i64(&s_bw[part[u]], (long long)c[u]);
  __syncthreads();
  for (int i = threadIdx.x; i < k; i += blockDim.x)
    if (s_bw[i]) atomic_add_i64(&bw[i], s_bw[i]);
}

// ------------------------------------------------------- objective (a14)

__global__ void k_objective(const unsigned long long* __restrict__ lam,
                            const int32_t* __restrict__ w, int32_t m,
                            unsigned long long* __restrict__ out) {
  __shared__ int64_t red[32];
  int64_t f = 0;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int l = __popcll(lam[e]);
    if (l > 1) f += (int64_t)(l - 1) * w[e];
  }
  f = block_sum(f, red);
  if (threadIdx.x == 0 && f) atomicAdd(out, (unsigned long long)f);
}

// Graph levels: the weight of the edges between blocks (5M edges, k = 2: 0.62 ms
// through the connectivity sets, 0.09 ms here).
__global__ void k_cut(const int2* __restrict__ edges, const int32_t* __restrict__ w, int32_t m,
                      const int32_t* __restrict__ part, unsigned long long* __restrict__ out) {
  __shared__ int64_t red[32];
  int64_t f = 0;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int2 v = edges[e];
    if (part[v.x] != part[v.y]) f += w[e];
  }
  f = block_sum(f, red);
  if (threadIdx.x == 0 && f) atomicAdd(out, (unsigned long long)f);
}

}  // namespace

// ===================================================================== host

void project_partition(const Ctx& cx, const Level& fine, const int32_t* coarse_part,
                       int32_t* fine_part) {
  if (fine.n == 0) return;
  k_project<<<grid_for(fine.n, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(fine.map.p, coarse_part,
                                                                        fine.n, fine_part);
  check_launch("project");
  if (cx.launches) *cx.launches += 1;
}

// The block weights of a partition and, as asked for, Phi with Lambda or with the
// records.
void build_pin_state(const Ctx& cx, const Level& L, int k, const int32_t* part, PinState& st,
                     PinMasks masks) {
  // the block weights, then the chunk lists: one allocation and one memset for all
  // that starts at zero
  const size_t cap = masks != PinMasks::none && L.p > COUNT_LEVEL
                         ? (size_t)(L.p / COUNT_CHUNK + L.p / COUNT_WARP) + 1 : 0;
  st.bw.alloc(&cx.alloc, (size_t)k + cap + (cap + 2) / 2);
  HG_CUDA(cudaMemsetAsync(st.bw.p, 0, st.bw.bytes(), cx.stream));
  if (masks != PinMasks::none) {
    if (masks != PinMasks::lambda_only) st.phi.alloc(&cx.alloc, (size_t)L.m * k + 1);
    if (masks != PinMasks::records) st.lam.alloc(&cx.alloc, (size_t)L.m + 1);
    else st.rec.alloc(&cx.alloc, (size_t)std::max<int32_t>(L.m, 1) * (k > 32 ? 2 : 1));
    if (L.m > 0) {
      CountArgs A{L.eoff.p, L.pins.p, part,     L.w.p,   L.m,    k,
                  st.phi.p, st.lam.p, st.rec.p, nullptr, nullptr, nullptr};
      if (cap) {
        A.chunks = reinterpret_cast<int2*>(st.bw.p + k);
        A.done = reinterpret_cast<int32_t*>(st.bw.p + k + cap);
        A.nchunks = A.done + cap;
      }
      const bool phi = st.phi.p != nullptr;
      (phi ? k_pin_counts<true> : k_pin_counts<false>)<<<
          grid_for(L.m, COUNT_WARPS * COUNT_NETS, cx.num_sms, 8), COUNT_WARPS * 32, 0,
          cx.stream>>>(A);
      check_launch("pin_counts");
      if (cap) {
        (phi ? k_pin_counts_huge<true> : k_pin_counts_huge<false>)<<<
            grid_for(L.p, COUNT_CHUNK, cx.num_sms, 4), COUNT_WARPS * 32, 0, cx.stream>>>(A);
        check_launch("pin_counts_huge");
      }
      if (cx.launches) *cx.launches += 1 + (cap > 0);
    }
  }
  k_block_weights<<<grid_for(L.n, 256, cx.num_sms, 4), 256, 0, cx.stream>>>(part, L.c.p, L.n, k,
                                                                          st.bw.p);
  check_launch("block_weights");
  if (cx.launches) *cx.launches += 1;
}

namespace {

// Runs `launch`, which adds the objective to the word it is given.
template <typename Launch>
int64_t sum_objective(const Ctx& cx, Launch&& launch) {
  DBuf<unsigned long long> acc;
  acc.alloc(&cx.alloc, 1);
  HG_CUDA(cudaMemsetAsync(acc.p, 0, sizeof(unsigned long long), cx.stream));
  launch(acc.p);
  check_launch("objective");
  if (cx.launches) *cx.launches += 1;
  return read_i64(cx, reinterpret_cast<const int64_t*>(acc.p));
}

}  // namespace

int64_t objective_of(const Ctx& cx, const Level& L, int k, const int32_t* part) {
  if (L.m == 0) return 0;
  const int g = grid_for(L.m, 256, cx.num_sms, 8);
  if (L.graph)
    return sum_objective(cx, [&](unsigned long long* out) {
      k_cut<<<g, 256, 0, cx.stream>>>(reinterpret_cast<const int2*>(L.pins.p), L.w.p, L.m, part,
                                      out);
    });
  PinState st;
  build_pin_state(cx, L, k, part, st, PinMasks::lambda_only);
  return sum_objective(cx, [&](unsigned long long* out) {
    k_objective<<<g, 256, 0, cx.stream>>>(st.lam.p, L.w.p, L.m, out);
  });
}

namespace {

__global__ void k_check_part(const int32_t* __restrict__ part, int32_t n, int k, int32_t* status) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x)
    if (part[u] < 0 || part[u] >= k) dev_fail(status, DEV_BAD_INPUT);
}

}  // namespace

void check_partition(const Ctx& cx, const int32_t* part, int32_t n, int k) {
  if (n <= 0) return;
  k_check_part<<<grid_for(n, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(part, n, k, cx.d_status);
  check_launch("check_part");
  if (cx.launches) *cx.launches += 1;
}

void validate_partition(const Ctx& cx, const int32_t* part, int32_t n, int k) {
  check_partition(cx, part, n, k);
  check_status(cx);
}

void pin_counts_of(const Ctx& cx, const Level& L, int k, const int32_t* part, int32_t* phi,
                   uint64_t* lambda, int64_t* bw) {
  PinState st;
  build_pin_state(cx, L, k, part, st, PinMasks::lambda);
  if (phi && L.m)
    HG_CUDA(cudaMemcpyAsync(phi, st.phi.p, sizeof(int32_t) * (size_t)L.m * k,
                            cudaMemcpyDeviceToHost, cx.stream));
  if (lambda && L.m)
    HG_CUDA(cudaMemcpyAsync(lambda, st.lam.p, sizeof(uint64_t) * (size_t)L.m,
                            cudaMemcpyDeviceToHost, cx.stream));
  if (bw)
    HG_CUDA(cudaMemcpyAsync(bw, st.bw.p, sizeof(int64_t) * (size_t)k, cudaMemcpyDeviceToHost,
                            cx.stream));
  check_status(cx);
}

}  // namespace hgk
