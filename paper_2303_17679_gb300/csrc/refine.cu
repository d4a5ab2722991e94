// Projection (Algorithm 1), pin counts and connectivity sets (Sec. 2, Sec. 6.1
// data layout) and the connectivity objective (Sec. 2) on the device.  Label
// propagation is in lp.cu.
//
// Layout: Phi is a dense m x k int32 table (row = net), Lambda one 64-bit
// mask per net (k <= 64), block weights int64[k].
#include "common.cuh"
#include "pintile.cuh"

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

// Phi(e, V_i) += 1 and Lambda(e) |= bit(i) for every pin; lanes that hold the
// same (net, block) combine their increments first.
__global__ void __launch_bounds__(PIN_TILE_THREADS)
k_pin_counts(const int32_t* __restrict__ eoff, const int32_t* __restrict__ pins,
             const int32_t* __restrict__ tile_net, int32_t m, int64_t p,
             const int32_t* __restrict__ part, int k, int32_t* __restrict__ phi,
             unsigned long long* __restrict__ lam) {
  __shared__ int32_t s_off[PIN_TILE + 3];
  const int64_t ntiles = num_pin_tiles(p);
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    PinTileView v = stage_pin_tile(eoff, tile_net, m, p, t, s_off);
    for (int64_t base = v.q0; base < v.q1; base += blockDim.x) {
      const int64_t q = base + threadIdx.x;
      const bool valid = q < v.q1;
      int64_t key = -1 - (int64_t)threadIdx.x;  // unique for idle lanes
      int32_t e = 0, b = 0;
      if (valid) {
        e = v.e_lo + net_in_tile(s_off, v.count, q);
        b = part[pins[q]];
        key = (int64_t)e * k + b;
      }
      const unsigned peers = __match_any_sync(FULL, (unsigned long long)key);
      const int leader = __ffs(peers) - 1;
      if (valid && lane_id() == leader) {
        atomicAdd(&phi[(int64_t)e * k + b], __popc(peers));
        atomicOr(&lam[e], 1ull << b);
      }
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

// Phi, Lambda (unless counts == false: graph levels in label propagation)
// and the block weights of a partition.
void build_pin_state(const Ctx& cx, const Level& L, int k, const int32_t* part, PinState& st,
                     bool counts) {
  st.bw.alloc(&cx.alloc, (size_t)k);
  HG_CUDA(cudaMemsetAsync(st.bw.p, 0, st.bw.bytes(), cx.stream));
  if (counts) {
    st.phi.alloc(&cx.alloc, (size_t)L.m * k + 1);
    st.lam.alloc(&cx.alloc, (size_t)L.m + 1);
    HG_CUDA(cudaMemsetAsync(st.phi.p, 0, st.phi.bytes(), cx.stream));
    HG_CUDA(cudaMemsetAsync(st.lam.p, 0, st.lam.bytes(), cx.stream));
  }
  if (counts && L.p > 0) {
    st.tiles.alloc(&cx.alloc, (size_t)num_pin_tiles(L.p) + 1);
    build_tile_index(cx, L.eoff.p, L.m, L.p, st.tiles.p);
    k_pin_counts<<<grid_for(num_pin_tiles(L.p), 1, cx.num_sms, 8), PIN_TILE_THREADS, 0,
                   cx.stream>>>(L.eoff.p, L.pins.p, st.tiles.p, L.m, L.p, part, k, st.phi.p,
                                st.lam.p);
    check_launch("pin_counts");
  }
  k_block_weights<<<grid_for(L.n, 256, cx.num_sms, 4), 256, 0, cx.stream>>>(part, L.c.p, L.n, k,
                                                                          st.bw.p);
  check_launch("block_weights");
  if (cx.launches) *cx.launches += 3;
}

namespace {

int64_t objective_from_lambda(const Ctx& cx, const Level& L, const unsigned long long* lam) {
  DBuf<unsigned long long> acc;
  acc.alloc(&cx.alloc, 1);
  HG_CUDA(cudaMemsetAsync(acc.p, 0, sizeof(unsigned long long), cx.stream));
  if (L.m > 0) {
    k_objective<<<grid_for(L.m, 256, cx.num_sms, 4), 256, 0, cx.stream>>>(lam, L.w.p, L.m, acc.p);
    check_launch("objective");
    if (cx.launches) *cx.launches += 1;
  }
  return read_i64(cx, reinterpret_cast<const int64_t*>(acc.p));
}

}  // namespace

int64_t objective_of(const Ctx& cx, const Level& L, int k, const int32_t* part) {
  PinState st;
  build_pin_state(cx, L, k, part, st, true);
  return objective_from_lambda(cx, L, st.lam.p);
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
  build_pin_state(cx, L, k, part, st, true);
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
