// Barrier of all blocks of a persistent kernel.
#pragma once

#include "common.cuh"

namespace hgk {

// Polls of a grid barrier without progress of the blocks it waits for (some ten
// seconds).
constexpr int SPIN_LIMIT = 1 << 24;

// The polls a wait may still spend: `limit` since the progress word last changed.
// The word counts units of work done by blocks that others may wait for long (a
// sort of millions of moves, a group of as many movers), so such a wait lasts as
// long as they work, and ends when nothing moves.
struct WaitBudget {
  int limit, polls = 0;
  unsigned seen = 0;
  __host__ __device__ explicit WaitBudget(int l) : limit(l) {}
  template <typename Progress>
  __host__ __device__ bool again(Progress&& progress) {
    if (++polls < limit) return true;
    const unsigned now = progress();
    if (now == seen) return false;
    seen = now;
    polls = 0;
    return true;
  }
};

// One thread of a block reports that the block got on with a long phase.
__device__ __forceinline__ void beat(unsigned* barrier) {
  asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(barrier + 1) : "memory");
}

// The same from a loop of a block over i = threadIdx.x, + blockDim.x, ... (a power
// of two): every 131072 entries, a few hundred microseconds of dependent accesses.
__device__ __forceinline__ void beat_along(unsigned* barrier, int64_t i) {
  if (i > 0 && (i & 0x1ffff) == 0) beat(barrier);  // thread 0's entries
}

// cluster: the blocks are one thread-block cluster (hardware barrier, 0.35 to
// 0.5 us, which waits until they arrive); else they were launched cooperatively
// and count arrivals in barrier[0], with the progress word in barrier[1] (both
// zero at the launch; 1.4 us over 152 blocks).  `gen` counts the barriers passed.
// Returns false when a grid barrier gave up: the status word is set and every
// thread of the block returns from the kernel.  The
// release and acquire of the barrier itself order everything the block has
// written and read; a fence of the device in front of them cost 4 ms of the 52 ms
// coarsening of 1e6 Zipf nodes.
__device__ __forceinline__ bool grid_sync(bool cluster, unsigned* barrier, int32_t* status,
                                          unsigned& gen, int limit = SPIN_LIMIT) {
  if (cluster) {
    // not the .aligned form: callers come from loops that lanes leave at
    // different times, and nothing makes the compiler rejoin them first
    asm volatile(
        "barrier.cluster.arrive.release;\n"
        "barrier.cluster.wait.acquire;" ::: "memory");
    return true;
  }
  ++gen;
  __syncthreads();
  bool ok = true;
  if (threadIdx.x == 0) {
    const unsigned target = gen * gridDim.x;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(barrier) : "memory");
    WaitBudget budget(limit);
    auto progress = [&]() {
      unsigned p;
      asm volatile("ld.relaxed.gpu.u32 %0, [%1];" : "=r"(p) : "l"(barrier + 1) : "memory");
      return p;
    };
    unsigned v;
    do {
      asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(v) : "l"(barrier) : "memory");
    } while ((int)(v - target) < 0 && budget.again(progress));
    ok = (int)(v - target) >= 0;
    if (!ok) dev_fail(status, DEV_TIMEOUT);
  }
  return __syncthreads_and(ok) != 0;
}

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// Launches a kernel of `blocks` blocks that meets at grid_sync: one cluster
// when cluster is set (1, 2, 4, 8 or 16 blocks), else cooperatively.
template <typename K, typename... Args>
void launch_persistent(const Ctx& cx, K kernel, int blocks, int threads, size_t smem, bool cluster,
                       Args... args) {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = cx.stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cluster) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)blocks;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
  } else {
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
  }
  HG_CUDA(cudaLaunchKernelEx(&cfg, kernel, args...));
  if (cx.launches) *cx.launches += 1;
}

}  // namespace hgk
