// Exact gains of a move sequence M = <m_1, ..., m_l>, m_i = (u_i, Pi[u_i], t_i)
// with every node moved at most once (Sec. 6.3, "The Parallel Gain
// Recalculation Algorithm", Algorithm 4): g_i is the objective decrease that
// m_i causes when the moves are performed in sequence order.  Per net e that
// contains a moved pin, with first_in[b] = smallest index of a move into
// block b among the pins of e, last_out[b] = largest index of a move out of
// b, and non_moved[b] = pins of e in b that do not move:
//   m_i = (u, s, t) gains w(e) when last_out[s] = i, i < first_in[s] and
//   non_moved[s] = 0 (u is the last pin to leave s and nothing entered s
//   before), and loses w(e) when first_in[t] = i, i > last_out[t] and
//   non_moved[t] = 0 (u is the first pin to enter t after t was emptied).
// Only the nets of moved nodes are visited, each once.
#include <algorithm>

#include "common.cuh"

namespace hgk {

namespace {

constexpr int GR_WARPS = 8;
constexpr int GR_LANES = 8;   // lanes per move or per net of at most GR_SMALL pins
constexpr int32_t GR_SMALL = SMALL_TOUCHED, GR_BIG = 32768;

// info[v] = {index of v's move or -1, Pi[v]}: a pin costs one 8-byte gather.
__global__ void k_gr_info(const int32_t* __restrict__ part, int32_t n, int2* __restrict__ info) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x)
    info[v] = make_int2(-1, part[v]);
}

// A node moved twice, a node out of range, or a target outside [0, k) or equal
// to the node's block is bad input.
__global__ void k_gr_index(const int32_t* __restrict__ nodes, const int32_t* __restrict__ targets,
                           int32_t l, int32_t n, int k, int2* __restrict__ info, int32_t* status) {
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < l; i += gridDim.x * blockDim.x) {
    const int32_t u = nodes[i], t = targets[i];
    if (u < 0 || u >= n || t < 0 || t >= k || info[u].y < 0 || info[u].y >= k || t == info[u].y) {
      dev_fail(status, DEV_BAD_INPUT);
      continue;
    }
    if (atomicCAS(&info[u].x, -1, i) != -1) dev_fail(status, DEV_BAD_INPUT);
  }
}

// One bit per net of a moved node, eight lanes per move.
__global__ void __launch_bounds__(GR_WARPS * 32)
k_gr_mark(const int32_t* __restrict__ nodes, int32_t l, int32_t n,
          const int32_t* __restrict__ ioff, const int32_t* __restrict__ inets,
          unsigned* __restrict__ mark) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x / GR_LANES;
  for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / GR_LANES; i < l;
       i += stride) {
    const int32_t u = nodes[i];
    if (u < 0 || u >= n) continue;  // reported by k_gr_index
    for (int32_t j = ioff[u] + (int32_t)(threadIdx.x % GR_LANES); j < ioff[u + 1]; j += GR_LANES) {
      const int32_t e = inets[j];
      atomicOr(&mark[e >> 5], 1u << (e & 31));
    }
  }
}

// The marked nets by size: those of at most GR_SMALL pins from the front of the list,
// in ascending order within a warp's 1024, the others from its end (in one list
// neighbouring big nets fell to the lane groups of one warp: 5000 nets of 5000 pins
// 0.9 -> 1.4 ms), and with chunk > 0 the chunks of the nets above it in a list of
// their own, {net, first of its chunks}.  One claim per warp and list (an append per
// net or per lane group is a same-address atomic each).
__global__ void k_gr_list(const unsigned* __restrict__ mark, int32_t words,
                          const int32_t* __restrict__ eoff, int32_t m, int32_t chunk,
                          int32_t* __restrict__ list, int32_t* __restrict__ count,
                          int2* __restrict__ chunks) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < words;
       i0 += stride) {
    const int64_t i = i0 + lane_id();
    const int32_t e0 = (int32_t)(32 * i);
    unsigned small = 0, wide = 0;
    for (unsigned x = i < words ? mark[i] : 0u; x; x &= x - 1) {
      const int bit = __ffs(x) - 1;
      const int32_t sz = eoff[e0 + bit + 1] - eoff[e0 + bit];
      if (sz <= GR_SMALL) {
        small |= 1u << bit;
      } else if (chunk == 0 || sz <= chunk) {
        wide |= 1u << bit;
      } else {
        const int32_t n = (sz + chunk - 1) / chunk, first = atomicAdd(&count[TN_CHUNKS], n);
        for (int32_t c = 0; c < n; ++c) chunks[first + c] = make_int2(e0 + bit, first);
      }
    }
    __syncwarp();
    const int32_t ns = __popc(small), nw = __popc(wide);
    const int32_t is = warp_inclusive_scan(ns), iw = warp_inclusive_scan(nw);
    int32_t bs = 0, bw = 0;
    if (lane_id() == 31 && is) bs = atomicAdd(&count[TN_SMALL], is);
    if (lane_id() == 31 && iw) bw = atomicAdd(&count[TN_WIDE], iw);
    int32_t at = __shfl_sync(FULL, bs, 31) + is - ns;
    for (; small; small &= small - 1) list[at++] = e0 + __ffs(small) - 1;
    at = m - 1 - (__shfl_sync(FULL, bw, 31) + iw - nw);
    for (; wide; wide &= wide - 1) list[at--] = e0 + __ffs(wide) - 1;
  }
}

// The per-block arrays of one net: smallest index of a move into a block,
// largest of a move out of it, pins that do not move.
struct NetBlocks {
  int32_t first_in[HG_MAX_K], last_out[HG_MAX_K], non_moved[HG_MAX_K];
  __device__ __forceinline__ void clear(int b) {
    first_in[b] = INT32_MAX;
    last_out[b] = -1;
    non_moved[b] = 0;
  }
};

// The two loops of Algorithm 4 over pins [b, end) by W threads (`at` of them; more
// than a warp: the block), with the net's arrays clear on entry and cleared again.
template <int W>
__device__ __forceinline__ void net_sync() {
  if (W <= 32) __syncwarp();
  else __syncthreads();
}

template <int W>
__device__ __forceinline__ void gr_net(const int32_t* __restrict__ pins,
                                       const int2* __restrict__ info,
                                       const int32_t* __restrict__ targets, int k, int32_t b,
                                       int32_t end, long long we, int at, NetBlocks& N,
                                       unsigned long long* __restrict__ gains, int32_t* status) {
  // the first two pins of a thread stay in registers for the second loop
  int2 keep[2] = {make_int2(-1, 0), make_int2(-1, 0)};
#pragma unroll
  for (int x = 0; x < 2; ++x)
    if (b + at + x * W < end) keep[x] = info[pins[b + at + x * W]];
  auto enter = [&](const int2& nd) {
    const int32_t i = nd.x, s = nd.y;
    if (s < 0 || s >= k) {  // a block id out of range: bad input, never indexed
      dev_fail(status, DEV_BAD_INPUT);
    } else if (i >= 0) {
      atomicMax(&N.last_out[s], i);
      atomicMin(&N.first_in[targets[i]], i);
    } else {
      atomicAdd(&N.non_moved[s], 1);
    }
  };
#pragma unroll
  for (int x = 0; x < 2; ++x)
    if (b + at + x * W < end) enter(keep[x]);
  for (int32_t q = b + at + 2 * W; q < end; q += W) enter(info[pins[q]]);
  net_sync<W>();
  auto leave = [&](const int2& nd) {
    const int32_t i = nd.x;
    if (i < 0) return;
    const int s = nd.y, t = targets[i];  // both checked by k_gr_index
    long long d = 0;
    if (N.last_out[s] == i && i < N.first_in[s] && N.non_moved[s] == 0) d += we;
    if (N.first_in[t] == i && i > N.last_out[t] && N.non_moved[t] == 0) d -= we;
    if (d) atomicAdd(&gains[i], (unsigned long long)d);
  };
#pragma unroll
  for (int x = 0; x < 2; ++x) leave(keep[x]);
  for (int32_t q = b + at + 2 * W; q < end; q += W) leave(info[pins[q]]);
  net_sync<W>();
  for (int x = at; x < k; x += W) N.clear(x);
  net_sync<W>();
}

// Listed nets: eight lanes per net of at most GR_SMALL pins (most nets have a
// handful; a warp per net left its lanes idle), a warp for the others, a block for
// those above GR_BIG (listed with their first chunk; a net of 1M pins: 40 ms by a
// warp).
__global__ void __launch_bounds__(GR_WARPS * 32)
k_gr_net(const int32_t* __restrict__ list, const int32_t* __restrict__ count, int32_t m,
         const int32_t* __restrict__ eoff, const int32_t* __restrict__ pins,
         const int32_t* __restrict__ w, const int2* __restrict__ info,
         const int32_t* __restrict__ targets, int k, const int2* __restrict__ chunks,
         unsigned long long* __restrict__ gains, int32_t* status) {
  constexpr int PER = 32 / GR_LANES;
  __shared__ NetBlocks s_blocks[GR_WARPS][PER];
  const int wv = warp_in_block(), lane = lane_id(), sub = lane % GR_LANES, grp = lane / GR_LANES;
  for (int x = sub; x < HG_MAX_K; x += GR_LANES) s_blocks[wv][grp].clear(x);
  __syncthreads();
  const int32_t nchunks = count[TN_CHUNKS], nwide = count[TN_WIDE], cnt = count[TN_SMALL];
  for (int32_t c = blockIdx.x; c < nchunks; c += gridDim.x) {
    const int2 it = chunks[c];
    if (it.y == c)
      gr_net<GR_WARPS * 32>(pins, info, targets, k, eoff[it.x], eoff[it.x + 1], w[it.x],
                            (int)threadIdx.x, s_blocks[0][0], gains, status);
  }
  for (int32_t x = wv * gridDim.x + blockIdx.x; x < nwide; x += gridDim.x * GR_WARPS) {
    const int32_t e = list[m - 1 - x];
    gr_net<32>(pins, info, targets, k, eoff[e], eoff[e + 1], w[e], lane, s_blocks[wv][0], gains,
               status);
  }
  const int64_t stride = (int64_t)gridDim.x * GR_WARPS * PER;
  for (int64_t x0 = ((int64_t)blockIdx.x * GR_WARPS + wv) * PER; x0 < cnt; x0 += stride) {
    const int64_t x = x0 + grp;
    const int32_t e = x < cnt ? list[x] : 0;
    const int32_t b = x < cnt ? eoff[e] : 0, end = x < cnt ? eoff[e + 1] : 0;
    gr_net<GR_LANES>(pins, info, targets, k, b, end, end > b ? w[e] : 0, sub, s_blocks[wv][grp],
                     gains, status);
  }
}

}  // namespace

void index_moves(const Ctx& cx, const Level& L, int k, const int32_t* part, int32_t l,
                 const int32_t* nodes, const int32_t* targets, DBuf<int2>& info) {
  info.alloc(&cx.alloc, (size_t)L.n);
  k_gr_info<<<grid_for(L.n, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(part, L.n, info.p);
  check_launch("gr_info");
  k_gr_index<<<grid_for(l, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(nodes, targets, l, L.n, k,
                                                                     info.p, cx.d_status);
  check_launch("gr_index");
  if (cx.launches) *cx.launches += 2;
}

void touched_nets(const Ctx& cx, const Level& L, int32_t l, const int32_t* nodes, int32_t chunk,
                  TouchedNets& t) {
  DBuf<unsigned> mark;
  const int32_t words = (int32_t)((L.m + 31ll) / 32);
  mark.alloc(&cx.alloc, (size_t)words + 1);
  t.list.alloc(&cx.alloc, (size_t)std::max<int32_t>(L.m, 1));
  t.count.alloc(&cx.alloc, TN_WORDS);
  if (chunk > 0) t.chunks.alloc(&cx.alloc, 2 * (size_t)(L.p / chunk) + 1);
  HG_CUDA(cudaMemsetAsync(mark.p, 0, mark.bytes(), cx.stream));
  HG_CUDA(cudaMemsetAsync(t.count.p, 0, t.count.bytes(), cx.stream));
  k_gr_mark<<<grid_for(l, GR_WARPS * (32 / GR_LANES), cx.num_sms, 8), GR_WARPS * 32, 0,
              cx.stream>>>(nodes, l, L.n, L.ioff.p, L.inets.p, mark.p);
  check_launch("gr_mark");
  k_gr_list<<<grid_for(words, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(
      mark.p, words, L.eoff.p, L.m, chunk, t.list.p, t.count.p, t.chunks.p);
  check_launch("gr_list");
  if (cx.launches) *cx.launches += 2;
}

void recalculate_gains(const Ctx& cx, const Level& L, int k, const int32_t* part, int32_t l,
                       const int32_t* nodes, const int32_t* targets, int64_t* gains) {
  if (l == 0) return;
  HG_CUDA(cudaMemsetAsync(gains, 0, sizeof(int64_t) * (size_t)l, cx.stream));
  DBuf<int2> info;
  TouchedNets t;
  index_moves(cx, L, k, part, l, nodes, targets, info);
  touched_nets(cx, L, l, nodes, GR_BIG, t);
  k_gr_net<<<cx.num_sms * 8, GR_WARPS * 32, 0, cx.stream>>>(
      t.list.p, t.count.p, L.m, L.eoff.p, L.pins.p, L.w.p, info.p, targets, k,
      t.chunks.p, reinterpret_cast<unsigned long long*>(gains), cx.d_status);
  check_launch("gr_net");
  if (cx.launches) *cx.launches += 1;
  check_status(cx);
}

}  // namespace hgk
