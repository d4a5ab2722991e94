// hg_objective_noalloc: the connectivity objective (for every net, its
// weight times the number of blocks it touches minus one, summed) and the
// block weights of a partition of a caller-held device CSR, with no handle
// and no device allocation.  The paper has no counterpart; this is a library
// convenience for callers that must not allocate.
//
// All scratch lives in one file-scope device array.  Host code looks its
// address up with cudaGetSymbolAddress on every call (cheap, allocates
// nothing, and stays right if the module is loaded again, for example after
// cudaDeviceReset or under another context):
//   [0, NA_BLOCKS)            objective partial of every block (written by
//                             its block before it is read; no initial value)
//   [NA_BW, NA_BW + 64)       block-weight accumulators      - must be zero
//   NA_TICKET                 count of finished blocks       - must be zero
//   NA_STATUS                 bad-input flag                 - must be zero
//   [NA_RES, NA_RES + 66)     result record: status, objective, 64 weights;
//                             status 0 = unwritten, 1 = good, 2 = bad input
// Before every launch the host clears the zero words and the result's status
// (one cudaMemsetAsync, which allocates nothing), so a launch that did not
// finish is reported instead of leaving an earlier call's result to be read.
// What bounds it: at n = m = 10,000 the chain memset, kernel, copy; the kernel is
// a few dependent loads per net, so eight lanes take a net (most have a handful
// of pins) and the last block sums the partials with all its threads (one
// thread alone read up to 1,024 of them): 66.9 -> 42.4 us per call with the second
// memset gone.
#include <algorithm>

#include "common.cuh"

namespace {

constexpr int NA_BLOCKS = 1024;  // grid cap = objective partial slots
constexpr int NA_THREADS = 256;
constexpr int NA_BW = NA_BLOCKS;
constexpr int NA_TICKET = NA_BW + HG_MAX_K;
constexpr int NA_STATUS = NA_TICKET + 1;
constexpr int NA_RES = NA_STATUS + 1;  // status, objective, weights[64]
constexpr int NA_WORDS = NA_RES + 2 + HG_MAX_K;

static __device__ __align__(256) unsigned long long g_noalloc_scratch[NA_WORDS];

// Eight lanes per net: lambda(e) = popcount of the OR of the blocks of its pins
// (the lanes of a warp stay in step; a warp takes its longest net's trips).  A net of
// many pins is walked by the whole warp; neighbouring nets belong to different warps,
// since big nets often follow one another (30 nets of 60,000 pins: 2.7 ms with four
// neighbours per warp);
// one thread per node for the block weights.  Offsets outside [0, p], pins
// outside [0, n) and block ids outside [0, k) set the status word and are
// skipped, so no access leaves the caller's arrays.  The last block to finish
// sums the partials and publishes the result record.
constexpr int NA_LANES = 8;

__global__ void __launch_bounds__(NA_THREADS)
k_objective_noalloc(const int32_t* __restrict__ eoff, const int32_t* __restrict__ pins,
                    const int32_t* __restrict__ w, const int32_t* __restrict__ c, int32_t n,
                    int32_t m, int64_t p, int32_t k, const int32_t* __restrict__ part,
                    unsigned long long* __restrict__ S) {
  __shared__ unsigned long long s_bw[HG_MAX_K];
  __shared__ unsigned long long s_warp[NA_THREADS / 32];
  __shared__ bool s_last;
  const int lane = threadIdx.x & 31, wv = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < HG_MAX_K; i += blockDim.x) s_bw[i] = 0;
  __syncthreads();

  bool bad = false;
  unsigned long long obj = 0;
  const int sub = lane % NA_LANES;
  const int64_t warps = (int64_t)gridDim.x * (NA_THREADS / 32);
  for (int64_t e0 = (int64_t)blockIdx.x * (NA_THREADS / 32) + wv; e0 < m;
       e0 += warps * (32 / NA_LANES)) {
    const int64_t e = e0 + warps * (lane / NA_LANES);
    int64_t b = 0, t = 0;
    if (e < m) {
      b = eoff[e];
      t = eoff[e + 1];
      if (b < 0 || t < b || t > p) {
        bad = true;
        b = t = 0;
      }
    }
    unsigned long long mask = 0;
    // a net of many pins is walked by the whole warp
    unsigned wide = __ballot_sync(0xffffffffu, t - b > 16 * NA_LANES && sub == 0);
    const bool mine = t - b <= 16 * NA_LANES;
    for (int64_t q = b + sub; mine && q < t; q += NA_LANES) {
      const int32_t v = pins[q];
      if (v < 0 || v >= n) { bad = true; continue; }
      const int32_t blk = part[v];
      if (blk < 0 || blk >= k) { bad = true; continue; }
      mask |= 1ull << blk;
    }
    __syncwarp();
    while (wide) {
      const int l = __ffs(wide) - 1;
      wide &= wide - 1;
      const int64_t wb = __shfl_sync(0xffffffffu, b, l), wt = __shfl_sync(0xffffffffu, t, l);
      unsigned long long x = 0;
      for (int64_t q = wb + lane; q < wt; q += 32) {
        const int32_t v = pins[q];
        if (v < 0 || v >= n) { bad = true; continue; }
        const int32_t blk = part[v];
        if (blk < 0 || blk >= k) { bad = true; continue; }
        x |= 1ull << blk;
      }
      __syncwarp();
      for (int o = 16; o > 0; o >>= 1) x |= __shfl_xor_sync(0xffffffffu, x, o);
      if (lane == l) mask = x;
    }
    for (int o = NA_LANES / 2; o > 0; o >>= 1) mask |= __shfl_xor_sync(0xffffffffu, mask, o);
    const int lam = __popcll(mask);
    if (sub == 0 && lam > 1)
      obj += (unsigned long long)(lam - 1) * (unsigned long long)(w ? w[e] : 1);
  }
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x) {
    const int32_t blk = part[u];
    if (blk < 0 || blk >= k) { bad = true; continue; }
    atomicAdd(&s_bw[blk], (unsigned long long)(c ? c[u] : 1));
  }

  for (int o = 16; o > 0; o >>= 1) obj += __shfl_xor_sync(0xffffffffu, obj, o);
  if (lane == 0) s_warp[wv] = obj;
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(&S[NA_STATUS], 1ull);
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long sum = 0;
    for (int i = 0; i < NA_THREADS / 32; ++i) sum += s_warp[i];
    S[blockIdx.x] = sum;
  }
  for (int i = threadIdx.x; i < k; i += blockDim.x)
    if (s_bw[i]) atomicAdd(&S[NA_BW + i], s_bw[i]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0)
    s_last = atomicAdd(&S[NA_TICKET], 1ull) == (unsigned long long)gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;

  // last block: every other block's writes are visible after the fence
  __threadfence();
  unsigned long long sum = 0;
  for (unsigned i = threadIdx.x; i < gridDim.x; i += blockDim.x) sum += __ldcg(&S[i]);
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) s_warp[wv] = sum;
  for (int i = threadIdx.x; i < k; i += blockDim.x) S[NA_RES + 2 + i] = __ldcg(&S[NA_BW + i]);
  __syncthreads();
  if (threadIdx.x == 0) {
    sum = 0;
    for (int i = 0; i < NA_THREADS / 32; ++i) sum += s_warp[i];
    S[NA_RES + 1] = sum;
    S[NA_RES] = __ldcg(&S[NA_STATUS]) ? 2ull : 1ull;
  }
}

int cuda_fail(cudaError_t e) {
  return e == cudaErrorMemoryAllocation ? HG_ERR_OOM : HG_ERR_CUDA;
}

}  // namespace

extern "C" int hg_objective_noalloc(int32_t n, int32_t m, int64_t p, const int32_t* net_offsets,
                                    const int32_t* pins, const int32_t* net_weights,
                                    const int32_t* node_weights, int32_t k, const int32_t* part,
                                    void* cuda_stream, int64_t* out_objective,
                                    int64_t* out_block_weights) {
  if (n < 1 || m < 0 || p < 0 || p > INT32_MAX || out_objective == nullptr) return HG_ERR_INVALID;
  if (k < 1) return HG_ERR_INVALID;
  if (k > HG_MAX_K) return HG_ERR_UNSUPPORTED;  // 64 block-weight slots in the scratch
  if (net_offsets == nullptr || part == nullptr || (p > 0 && pins == nullptr))
    return HG_ERR_INVALID;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e);
  // the scratch address in the current context (the first call on a device
  // loads the module, so it should come before any stream capture)
  void* addr = nullptr;
  e = cudaGetSymbolAddress(&addr, g_noalloc_scratch);
  if (e != cudaSuccess) return cuda_fail(e);
  unsigned long long* S = static_cast<unsigned long long*>(addr);
  int sms = 0;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return cuda_fail(e);
  const cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const int64_t work = std::max<int64_t>((int64_t)m * NA_LANES, n);
  int64_t blocks = (work + NA_THREADS - 1) / NA_THREADS;
  blocks = std::min<int64_t>(blocks, std::min<int64_t>(NA_BLOCKS, (int64_t)sms * 8));
  blocks = std::max<int64_t>(blocks, 1);
  // zero words and the result's status cleared
  e = cudaMemsetAsync(S + NA_BW, 0, sizeof(unsigned long long) * (HG_MAX_K + 3), st);
  if (e != cudaSuccess) return cuda_fail(e);
  k_objective_noalloc<<<(unsigned)blocks, NA_THREADS, 0, st>>>(net_offsets, pins, net_weights,
                                                               node_weights, n, m, p, k, part, S);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e);
  unsigned long long res[2 + HG_MAX_K];
  e = cudaMemcpyAsync(res, S + NA_RES, sizeof(res[0]) * (2 + (size_t)k), cudaMemcpyDeviceToHost, st);
  if (e != cudaSuccess) return cuda_fail(e);
  e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail(e);
  if (res[0] == 0) return HG_ERR_CUDA;
  if (res[0] != 1) return HG_ERR_INVALID;
  *out_objective = (int64_t)res[1];
  if (out_block_weights)
    for (int i = 0; i < k; ++i) out_block_weights[i] = (int64_t)res[2 + i];
  return HG_OK;
}
