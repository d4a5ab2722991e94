// Contraction of a clustering (Sec. 4.2 "The Contraction Algorithm"):
//   a5  representatives -> consecutive coarse ids by a prefix sum over
//       representative flags (rank of the representative's id); coarse node
//       weight = cluster weight;
//   a6  every pin replaced by its coarse node, each net's pins sorted and
//       deduplicated, single-pin nets dropped;
//   a7  identical nets found by fingerprint (a 64-bit sum of hashed pins plus
//       the size) in a hash table keyed by the fingerprint, the smallest net
//       id of each fingerprint group as candidate representative, and an
//       exact pin-by-pin comparison; nets that differ from their group's
//       candidate go through further rounds among themselves; weights of
//       identical nets are summed at the representative (smallest id);
//   a8  kept nets compacted in order of their representative's id by prefix
//       sums over a keep flag and the kept sizes, then the incidence lists.
#include <algorithm>
#include <climits>

#include "common.cuh"

namespace hgk {

namespace {

// Net size classes of the remap: a thread, a warp, a block, a block per net.  A
// block per net of 33..1024 pins spends its time at the barriers of its sort and
// two block-wide sums; a warp needs none.  Where the coarse nodes fit a bitmap in
// shared memory, marking them replaces the O(log^2) steps of the sort and the
// cleared bitmap in global memory.  Measured (GB300, with compaction and the
// comparison of identical nets by eight lanes per net): coarsening of a 4e6-node
// large-net input, k = 64: 104.9 -> 95.8 ms; of 1e6 Zipf nodes, k = 8: 56 -> 52.5 ms.
constexpr int SMALL_NET = 32;
constexpr int WARP_NET = 1024;
constexpr int MID_NET = 4096;
constexpr int NCLS = 4;
constexpr int WARP_NETS = 8;        // warps per block of the warp class
constexpr int MID_THREADS = 256;
constexpr int BIG_THREADS = 512;
// Coarse nodes up to which a net's pins are marked in a shared bitmap instead
// of being sorted: a warp's bitmap of 2 KB, a block's of 64 KB.
constexpr int32_t WARP_BITMAP_N = 16384;
constexpr int32_t BLOCK_BITMAP_N = 1 << 19;
constexpr unsigned long long EMPTY_FP = ~0ull;

__global__ void k_rep_flags(const int32_t* __restrict__ rep, int32_t n, int32_t* __restrict__ flag) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x)
    flag[u] = rep[u] == (int32_t)u ? 1 : 0;
}

__global__ void k_map(const int32_t* __restrict__ rep, const int32_t* __restrict__ cid,
                      const int32_t* __restrict__ cw, int32_t n, int32_t* __restrict__ map,
                      int32_t* __restrict__ c2) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x) {
    const int32_t r = rep[u];
    map[u] = cid[r];
    if (r == (int32_t)u) c2[cid[u]] = cw[u];
  }
}

__global__ void k_classify_nets(const int32_t* __restrict__ eoff, int32_t m,
                                int32_t* __restrict__ lists, int32_t* __restrict__ counts) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); b < m; b += stride) {
    const int64_t e = b + lane_id();
    const bool valid = e < m;
    int cls = -1;
    if (valid) {
      const int32_t sz = eoff[e + 1] - eoff[e];
      cls = sz <= SMALL_NET ? 0 : sz <= WARP_NET ? 1 : sz <= MID_NET ? 2 : 3;
    }
    const int32_t slot = warp_claim_slot(counts, cls, __ballot_sync(FULL, valid));
    if (valid) lists[(int64_t)cls * m + slot] = (int32_t)e;
  }
}

__device__ __forceinline__ unsigned long long fingerprint_finish(unsigned long long sum, int32_t size,
                                                                 int bits) {
  unsigned long long f = sum + mix64((unsigned long long)(uint32_t)size ^ 0x5bd1e995ull);
  if (bits > 0 && bits < 64) f &= (1ull << bits) - 1;
  if (f == EMPTY_FP) f = EMPTY_FP - 1;
  return f;
}

// Nets of <= 32 pins: one thread per net, insertion sort in registers.
__global__ void k_remap_small(const int32_t* __restrict__ list, int32_t count,
                              const int32_t* __restrict__ eoff, const int32_t* __restrict__ pins,
                              const int32_t* __restrict__ map, int fp_bits,
                              int32_t* __restrict__ tpins, int32_t* __restrict__ tsize,
                              unsigned long long* __restrict__ fp) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t e = list[i];
    const int32_t b = eoff[e], sz = eoff[e + 1] - b;
    int32_t v[SMALL_NET];
    for (int q = 0; q < sz; ++q) {
      const int32_t x = map[pins[b + q]];
      int r = q;
      while (r > 0 && v[r - 1] > x) {
        v[r] = v[r - 1];
        --r;
      }
      v[r] = x;
    }
    int32_t out = 0;
    unsigned long long sum = 0;
    for (int q = 0; q < sz; ++q) {
      if (q == 0 || v[q] != v[q - 1]) {
        tpins[b + out] = v[q];
        sum += mix64((unsigned long long)(uint32_t)v[q]);
        ++out;
      }
    }
    tsize[e] = out;
    fp[e] = fingerprint_finish(sum, out, fp_bits);
  }
}

// Nets of 33..1024 pins on levels of few coarse nodes: one warp per net marks
// the coarse nodes in a bitmap in shared memory and writes the set bits in
// ascending order (each lane a run of words).
__global__ void __launch_bounds__(WARP_NETS * 32)
k_remap_warp_bitmap(const int32_t* __restrict__ list, int32_t count,
                    const int32_t* __restrict__ eoff, const int32_t* __restrict__ pins,
                    const int32_t* __restrict__ map, int32_t words, int fp_bits,
                    int32_t* __restrict__ tpins, int32_t* __restrict__ tsize,
                    unsigned long long* __restrict__ fp) {
  // one pad word per 32, so that the lanes' runs start in different banks
  constexpr int CAP = WARP_BITMAP_N / 32;
  __shared__ unsigned s_bits[WARP_NETS][CAP + CAP / 32 + 1];
  unsigned* bits = s_bits[warp_in_block()];
  const int lane = lane_id();
  const int per = (words + 31) / 32;  // words per lane
  auto at = [](int w) { return w + (w >> 5); };
  for (int w = lane; w < words; w += 32) bits[at(w)] = 0u;
  __syncwarp();
  for (int32_t i = blockIdx.x * WARP_NETS + warp_in_block(); i < count;
       i += gridDim.x * WARP_NETS) {
    const int32_t e = list[i];
    const int32_t b = eoff[e], sz = eoff[e + 1] - b;
    for (int q = lane; q < sz; q += 64) {
      const bool two = q + 32 < sz;
      const int32_t p0 = pins[b + q], p1 = two ? pins[b + q + 32] : p0;
      const int32_t v0 = map[p0], v1 = map[p1];
      atomicOr(&bits[at(v0 >> 5)], 1u << (v0 & 31));
      if (two) atomicOr(&bits[at(v1 >> 5)], 1u << (v1 & 31));
    }
    __syncwarp();
    int c = 0;
    for (int x = 0; x < per; ++x) {
      const int w = lane * per + x;
      if (w < words) c += __popc(bits[at(w)]);
    }
    const int incl = warp_inclusive_scan(c);
    int32_t pos = b + incl - c;
    unsigned long long sum = 0;
    for (int x = 0; x < per; ++x) {
      const int w = lane * per + x;
      if (w >= words) break;
      unsigned rest = bits[at(w)];
      bits[at(w)] = 0u;
      while (rest) {
        const int32_t v = (w << 5) + __ffs(rest) - 1;
        rest &= rest - 1;
        tpins[pos++] = v;
        sum += mix64((unsigned long long)(uint32_t)v);
      }
    }
    sum = warp_sum(sum);
    if (lane == 31) {
      tsize[e] = incl;
      fp[e] = fingerprint_finish(sum, incl, fp_bits);
    }
    __syncwarp();
  }
}

// One net of at most 32 R pins by the warp: a bitonic sort with R keys per lane
// in registers (in-thread swaps below R, lane shuffles above), then the first
// key of every run is kept.
template <int R>
__device__ __forceinline__ void remap_sort(int32_t e, int32_t b, int32_t sz,
                                           const int32_t* __restrict__ pins,
                                           const int32_t* __restrict__ map, int fp_bits,
                                           int32_t* __restrict__ tpins,
                                           int32_t* __restrict__ tsize,
                                           unsigned long long* __restrict__ fp) {
  const int lane = lane_id();
  int32_t v[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int32_t i = r * 32 + lane;  // any arrangement sorts
    v[r] = i < sz ? map[pins[b + i]] : INT_MAX;
  }
#pragma unroll 1
  for (int kk = 2; kk <= 32 * R; kk <<= 1) {
#pragma unroll 1
    for (int j = kk >> 1; j >= R; j >>= 1) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int i = lane * R + r;
        const int32_t y = __shfl_xor_sync(FULL, v[r], j / R);
        const bool keep_min = ((i & kk) == 0) == ((i & j) == 0);
        v[r] = keep_min ? min(v[r], y) : max(v[r], y);
      }
    }
#pragma unroll
    for (int j = R / 2; j > 0; j >>= 1) {
      if (j >= kk) continue;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if ((r ^ j) > r) {
          const bool up = ((lane * R + r) & kk) == 0;
          const int32_t lo = min(v[r], v[r ^ j]), hi = max(v[r], v[r ^ j]);
          v[r] = up ? lo : hi;
          v[r ^ j] = up ? hi : lo;
        }
      }
    }
  }
  // lane l holds keys l R .. l R + R - 1 of the sorted net
  const int32_t before = __shfl_up_sync(FULL, v[R - 1], 1);
  int c = 0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int32_t prev = r == 0 ? (lane == 0 ? -1 : before) : v[r - 1];
    c += v[r] != INT_MAX && v[r] != prev;
  }
  const int incl = warp_inclusive_scan(c);
  int32_t pos = b + incl - c;
  unsigned long long sum = 0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int32_t prev = r == 0 ? (lane == 0 ? -1 : before) : v[r - 1];
    if (v[r] != INT_MAX && v[r] != prev) {
      tpins[pos++] = v[r];
      sum += mix64((unsigned long long)(uint32_t)v[r]);
    }
  }
  sum = warp_sum(sum);
  if (lane == 31) {
    tsize[e] = incl;
    fp[e] = fingerprint_finish(sum, incl, fp_bits);
  }
}

// Nets of 33..1024 pins on the other levels, one warp per net.
__global__ void __launch_bounds__(WARP_NETS * 32)
k_remap_warp_sort(const int32_t* __restrict__ list, int32_t count,
                  const int32_t* __restrict__ eoff, const int32_t* __restrict__ pins,
                  const int32_t* __restrict__ map, int fp_bits, int32_t* __restrict__ tpins,
                  int32_t* __restrict__ tsize, unsigned long long* __restrict__ fp) {
  for (int32_t i = blockIdx.x * WARP_NETS + warp_in_block(); i < count;
       i += gridDim.x * WARP_NETS) {
    const int32_t e = list[i];
    const int32_t b = eoff[e], sz = eoff[e + 1] - b;
    if (sz <= 128) remap_sort<4>(e, b, sz, pins, map, fp_bits, tpins, tsize, fp);
    else if (sz <= 512) remap_sort<16>(e, b, sz, pins, map, fp_bits, tpins, tsize, fp);
    else remap_sort<32>(e, b, sz, pins, map, fp_bits, tpins, tsize, fp);
  }
}

// Nets of more than 1024 pins on levels whose coarse nodes fit a bitmap in
// shared memory: one block per net, every thread a run of words, one block-wide
// scan per net.
__global__ void __launch_bounds__(BIG_THREADS)
k_remap_block_bitmap(const int32_t* __restrict__ list, int32_t count,
                     const int32_t* __restrict__ eoff, const int32_t* __restrict__ pins,
                     const int32_t* __restrict__ map, int32_t words, int fp_bits,
                     int32_t* __restrict__ tpins, int32_t* __restrict__ tsize,
                     unsigned long long* __restrict__ fp) {
  extern __shared__ unsigned bits[];  // one pad word per 32
  __shared__ int32_t s_wsum[BIG_THREADS / 32];
  __shared__ unsigned long long s_red[32];
  const int per = (words + BIG_THREADS - 1) / BIG_THREADS;
  auto at = [](int w) { return w + (w >> 5); };
  for (int w = threadIdx.x; w < words; w += BIG_THREADS) bits[at(w)] = 0u;
  __syncthreads();
  for (int32_t i = blockIdx.x; i < count; i += gridDim.x) {
    const int32_t e = list[i];
    const int32_t b = eoff[e], sz = eoff[e + 1] - b;
    for (int32_t q0 = threadIdx.x; q0 < sz; q0 += 4 * BIG_THREADS) {
      int32_t v[4];
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int64_t q = (int64_t)q0 + x * BIG_THREADS;
        v[x] = q < sz ? pins[b + q] : -1;
      }
#pragma unroll
      for (int x = 0; x < 4; ++x)
        if (v[x] >= 0) v[x] = map[v[x]];
#pragma unroll
      for (int x = 0; x < 4; ++x)
        if (v[x] >= 0) atomicOr(&bits[at(v[x] >> 5)], 1u << (v[x] & 31));
    }
    __syncthreads();
    int c = 0;
    for (int x = 0; x < per; ++x) {
      const int w = threadIdx.x * per + x;
      if (w < words) c += __popc(bits[at(w)]);
    }
    const int incl = warp_inclusive_scan(c);
    if (lane_id() == 31) s_wsum[warp_in_block()] = incl;
    __syncthreads();
    int32_t before = 0, total = 0;
#pragma unroll
    for (int x = 0; x < BIG_THREADS / 32; ++x) {
      if (x < warp_in_block()) before += s_wsum[x];
      total += s_wsum[x];
    }
    int32_t pos = b + before + incl - c;
    unsigned long long sum = 0;
    for (int x = 0; x < per; ++x) {
      const int w = threadIdx.x * per + x;
      if (w >= words) break;
      unsigned rest = bits[at(w)];
      bits[at(w)] = 0u;
      while (rest) {
        const int32_t v = (w << 5) + __ffs(rest) - 1;
        rest &= rest - 1;
        tpins[pos++] = v;
        sum += mix64((unsigned long long)(uint32_t)v);
      }
    }
    sum = block_sum(sum, s_red);  // ends with the bitmap clear and a barrier passed
    if (threadIdx.x == 0) {
      tsize[e] = total;
      fp[e] = fingerprint_finish(sum, total, fp_bits);
    }
  }
}

// Nets of 1025..4096 pins on the other levels: one block per net, bitonic sort with the keys in
// registers (shared memory only for the exchanges between warps).
__global__ void __launch_bounds__(MID_THREADS, 1024 / MID_THREADS)
k_remap_mid(const int32_t* __restrict__ list, int32_t count, const int32_t* __restrict__ eoff,
            const int32_t* __restrict__ pins, const int32_t* __restrict__ map, int fp_bits,
            int32_t* __restrict__ tpins, int32_t* __restrict__ tsize,
            unsigned long long* __restrict__ fp) {
  __shared__ int32_t s[MID_NET];
  __shared__ int32_t s_wsum[MID_THREADS / 32];
  __shared__ unsigned long long s_red[32];
  constexpr int PER = MID_NET / MID_THREADS;  // 16 consecutive items per thread
  for (int32_t i = blockIdx.x; i < count; i += gridDim.x) {
    const int32_t e = list[i];
    const int32_t b = eoff[e], sz = eoff[e + 1] - b;
    int P = 64;
    while (P < sz) P <<= 1;
    // bitonic sort with the keys in registers: thread t holds items
    // [t*PER, t*PER+PER); distances below PER are swaps inside a thread,
    // below 32*PER lane shuffles, the rest exchanges through s (warps that
    // hold only padding sit the network out)
    const int t = threadIdx.x;
    const bool warp_live = warp_in_block() * 32 * PER < P;
    int32_t v[PER];
#pragma unroll
    for (int r = 0; r < PER; ++r) {
      const int q = t * PER + r;
      v[r] = q < sz ? map[pins[b + q]] : INT_MAX;
    }
    for (int kk = 2; kk <= P; kk <<= 1) {
      for (int j = kk >> 1; j >= PER; j >>= 1) {
        if (j >= 32 * PER) {
          __syncthreads();
#pragma unroll
          for (int r = 0; r < PER; ++r) s[t * PER + r] = v[r];
          __syncthreads();
#pragma unroll
          for (int r = 0; r < PER; ++r) {
            const int q = t * PER + r;
            if (q >= P) continue;
            const int32_t y = s[q ^ j];
            const bool up = (q & kk) == 0, lower = (q & j) == 0;
            const int32_t lo = min(v[r], y), hi = max(v[r], y);
            v[r] = lower == up ? lo : hi;
          }
        } else if (warp_live) {
          const int lj = j / PER;  // partner lane distance
#pragma unroll
          for (int r = 0; r < PER; ++r) {
            const int q = t * PER + r;
            const int32_t y = __shfl_xor_sync(FULL, v[r], lj);
            const bool up = (q & kk) == 0, lower = (q & j) == 0;
            const int32_t lo = min(v[r], y), hi = max(v[r], y);
            v[r] = lower == up ? lo : hi;
          }
        }
      }
      if (warp_live) {
#pragma unroll
        for (int jj = PER / 2; jj > 0; jj >>= 1) {
          if (jj >= kk) continue;
#pragma unroll
          for (int r = 0; r < PER; ++r) {
            const int l = r ^ jj;
            if (l > r) {
              const bool up = ((t * PER + r) & kk) == 0;
              const int32_t lo = min(v[r], v[l]), hi = max(v[r], v[l]);
              v[r] = up ? lo : hi;
              v[l] = up ? hi : lo;
            }
          }
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < PER; ++r) s[t * PER + r] = v[r];
    __syncthreads();
    // keep the first of every run: thread t owns items [t*PER, t*PER+PER)
    int32_t local = 0;
    bool keep[PER];
    int32_t vals[PER];
#pragma unroll
    for (int r = 0; r < PER; ++r) {
      const int q = threadIdx.x * PER + r;
      vals[r] = q < P ? s[q] : INT_MAX;
      keep[r] = q < sz && (q == 0 || s[q] != s[q - 1]);
      local += keep[r];
    }
    int32_t x = warp_inclusive_scan(local);
    if (lane_id() == 31) s_wsum[warp_in_block()] = x;
    __syncthreads();
    int32_t before = 0;
    for (int wv = 0; wv < warp_in_block(); ++wv) before += s_wsum[wv];
    int32_t total = 0;
    for (int wv = 0; wv < MID_THREADS / 32; ++wv) total += s_wsum[wv];
    int32_t pos = before + x - local;
    unsigned long long sum = 0;
#pragma unroll
    for (int r = 0; r < PER; ++r)
      if (keep[r]) {
        tpins[b + pos++] = vals[r];
        sum += mix64((unsigned long long)(uint32_t)vals[r]);
      }
    sum = block_sum(sum, s_red);
    if (threadIdx.x == 0) {
      tsize[e] = total;
      fp[e] = fingerprint_finish(sum, total, fp_bits);
    }
    __syncthreads();
  }
}

// Nets of more than 4096 pins: one block per net marks its coarse nodes in a
// bitmap (one bitmap per block, words = ceil(n2 / 32)) and writes the set
// bits in ascending order.
__global__ void __launch_bounds__(BIG_THREADS)
k_remap_big(const int32_t* __restrict__ list, int32_t count, const int32_t* __restrict__ eoff,
            const int32_t* __restrict__ pins, const int32_t* __restrict__ map, int32_t words,
            unsigned* __restrict__ bitmaps, int fp_bits, int32_t* __restrict__ tpins,
            int32_t* __restrict__ tsize, unsigned long long* __restrict__ fp) {
  __shared__ int32_t s_wsum[32];
  __shared__ unsigned long long s_red[32];
  __shared__ int32_t s_carry;
  unsigned* bm = bitmaps + (size_t)blockIdx.x * words;
  for (int32_t i = blockIdx.x; i < count; i += gridDim.x) {
    const int32_t e = list[i];
    const int32_t b = eoff[e], sz = eoff[e + 1] - b;
    for (int32_t q = threadIdx.x; q < words; q += blockDim.x) bm[q] = 0u;
    __syncthreads();
    for (int32_t q = threadIdx.x; q < sz; q += blockDim.x) {
      const int32_t v = map[pins[b + q]];
      atomicOr(&bm[v >> 5], 1u << (v & 31));
    }
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    unsigned long long sum = 0;
    for (int32_t base = 0; base < words; base += blockDim.x) {
      const int32_t q = base + threadIdx.x;
      const unsigned word = q < words ? bm[q] : 0u;
      const int32_t c = __popc(word);
      int32_t x = warp_inclusive_scan(c);
      if (lane_id() == 31) s_wsum[warp_in_block()] = x;
      __syncthreads();
      int32_t before = s_carry;
      for (int wv = 0; wv < warp_in_block(); ++wv) before += s_wsum[wv];
      int32_t pos = before + x - c;
      unsigned rest = word;
      while (rest) {
        const int bit = __ffs(rest) - 1;
        rest &= rest - 1;
        const int32_t v = (q << 5) + bit;
        tpins[b + pos++] = v;
        sum += mix64((unsigned long long)(uint32_t)v);
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        int32_t t = 0;
        for (int wv = 0; wv < (int)(blockDim.x >> 5); ++wv) t += s_wsum[wv];
        s_carry += t;
      }
      __syncthreads();
    }
    sum = block_sum(sum, s_red);
    if (threadIdx.x == 0) {
      tsize[e] = s_carry;
      fp[e] = fingerprint_finish(sum, s_carry, fp_bits);
    }
    __syncthreads();
  }
}

// --------------------------------------------------- identical nets (a7)

__global__ void k_candidates(const int32_t* __restrict__ tsize, int32_t m,
                             int32_t* __restrict__ list, int32_t* __restrict__ count) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x)
    if (tsize[e] >= 2) list[atomicAdd(count, 1)] = (int32_t)e;
}

__global__ void k_ident_insert(const int32_t* __restrict__ list, const int32_t* __restrict__ count,
                               const unsigned long long* __restrict__ fp, unsigned long long* tkey,
                               int32_t* tmin, uint64_t mask, int32_t* __restrict__ slot_of_net,
                               int32_t* status) {
  const int32_t cnt = *count;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t e = list[i];
    const unsigned long long f = fp[e];
    uint64_t h = mix64(f) & mask;
    int32_t slot = -1;
    for (uint64_t probe = 0; probe <= mask; ++probe) {
      const unsigned long long k = tkey[h];
      if (k == f) { slot = (int32_t)h; break; }
      if (k == EMPTY_FP) {
        const unsigned long long old = atomicCAS(&tkey[h], EMPTY_FP, f);
        if (old == EMPTY_FP || old == f) { slot = (int32_t)h; break; }
      }
      h = (h + 1) & mask;
    }
    if (slot < 0) {
      dev_fail(status, DEV_HASH_FULL);
      continue;
    }
    atomicMin(&tmin[slot], e);
    slot_of_net[e] = slot;
  }
}

// Eight lanes per candidate net: compare with its group's smallest id (nets of
// many pins by the whole warp).
constexpr int CMP_LANES = 8;
constexpr int32_t CMP_SMALL = 128;

__global__ void k_ident_compare(const int32_t* __restrict__ list, const int32_t* __restrict__ count,
                                const int32_t* __restrict__ eoff, const int32_t* __restrict__ tpins,
                                const int32_t* __restrict__ tsize,
                                const int32_t* __restrict__ slot_of_net,
                                const int32_t* __restrict__ tmin, int32_t* __restrict__ repnet,
                                int32_t* __restrict__ failed, int32_t* __restrict__ nfailed) {
  constexpr int PER = 32 / CMP_LANES;
  const int32_t cnt = *count;
  const int lane = lane_id(), sub = lane % CMP_LANES, grp = lane / CMP_LANES;
  const unsigned mine = ((1u << CMP_LANES) - 1u) << (grp * CMP_LANES);
  const int64_t stride = (((int64_t)gridDim.x * blockDim.x) >> 5) * PER;
  for (int64_t i0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * PER; i0 < cnt;
       i0 += stride) {
    const int64_t i = i0 + grp;
    const bool on = i < cnt;
    const int32_t e = on ? list[i] : 0;
    const int32_t r = on ? tmin[slot_of_net[e]] : 0;
    const int32_t sz = on ? tsize[e] : 0;
    bool same = true;
    const bool check = on && r != e;
    if (check) same = tsize[r] == sz;
    const int32_t ea = on ? eoff[e] : 0, eb = on ? eoff[r] : 0;
    const bool walk = check && same;
    for (int32_t q = sub; walk && sz <= CMP_SMALL && q < sz; q += CMP_LANES)
      if (tpins[ea + q] != tpins[eb + q]) same = false;
    __syncwarp();
    unsigned wide = __ballot_sync(FULL, walk && sz > CMP_SMALL && sub == 0);
    while (wide) {
      const int l = __ffs(wide) - 1;
      wide &= wide - 1;
      const int32_t wa = __shfl_sync(FULL, ea, l), wb = __shfl_sync(FULL, eb, l);
      const int32_t ws = __shfl_sync(FULL, sz, l);
      bool eq = true;
      for (int32_t q = lane; q < ws; q += 32) eq &= tpins[wa + q] == tpins[wb + q];
      eq = __all_sync(FULL, eq);
      if (lane / CMP_LANES == l / CMP_LANES) same = eq;
    }
    same = (__ballot_sync(FULL, same) & mine) == mine;
    if (sub == 0 && on) {
      if (same) repnet[e] = r;
      else failed[atomicAdd(nfailed, 1)] = e;
    }
  }
}

__global__ void k_net_weights(const int32_t* __restrict__ tsize, const int32_t* __restrict__ repnet,
                              const int32_t* __restrict__ w, int32_t m, int32_t* __restrict__ wsum,
                              int32_t* __restrict__ keep, int32_t* __restrict__ ksize) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    const bool valid = tsize[e] >= 2;
    const bool k = valid && repnet[e] == (int32_t)e;
    if (valid) atomicAdd(&wsum[repnet[e]], w[e]);
    keep[e] = k ? 1 : 0;
    ksize[e] = k ? tsize[e] : 0;
  }
}

// Eight lanes per kept net write its coarse offset, weight and pins (nets of
// many pins by the whole warp, four pins per lane in flight).
constexpr int CP_LANES = 8;
constexpr int32_t CP_SMALL = 64;

__global__ void k_compact(const int32_t* __restrict__ keep, const int32_t* __restrict__ newid,
                          const int32_t* __restrict__ poff, const int32_t* __restrict__ eoff,
                          const int32_t* __restrict__ tpins, const int32_t* __restrict__ tsize,
                          const int32_t* __restrict__ wsum, int32_t m, int32_t* __restrict__ eoff2,
                          int32_t* __restrict__ pins2, int32_t* __restrict__ w2) {
  constexpr int PER = 32 / CP_LANES;
  const int lane = lane_id(), sub = lane % CP_LANES;
  const int64_t stride = (((int64_t)gridDim.x * blockDim.x) >> 5) * PER;
  for (int64_t e0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * PER; e0 < m;
       e0 += stride) {
    const int64_t e = e0 + lane / CP_LANES;
    const bool on = e < m && keep[e];
    const int32_t dst = on ? poff[e] : 0, src = on ? eoff[e] : 0, sz = on ? tsize[e] : 0;
    if (on && sub == 0) {
      const int32_t id = newid[e];
      eoff2[id] = dst;
      w2[id] = wsum[e];
    }
    for (int32_t q = sub; sz <= CP_SMALL && q < sz; q += CP_LANES) pins2[dst + q] = tpins[src + q];
    __syncwarp();
    unsigned wide = __ballot_sync(FULL, sub == 0 && sz > CP_SMALL);
    while (wide) {
      const int l = __ffs(wide) - 1;
      wide &= wide - 1;
      const int32_t wd = __shfl_sync(FULL, dst, l), ws = __shfl_sync(FULL, src, l);
      const int32_t wz = __shfl_sync(FULL, sz, l);
      for (int32_t q0 = lane; q0 < wz; q0 += 128) {
        int32_t v[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) v[x] = q0 + 32 * x < wz ? tpins[ws + q0 + 32 * x] : 0;
#pragma unroll
        for (int x = 0; x < 4; ++x)
          if (q0 + 32 * x < wz) pins2[wd + q0 + 32 * x] = v[x];
      }
    }
  }
}

// ------------------------------------------------------------ graph levels

// A net of two pins is its pair of coarse nodes: the pair itself, {smaller,
// larger} in 64 bits, is the hash-table key, so equal keys are identical nets
// and the weights are summed at the key.  Three passes over the edges (insert,
// flag, write) instead of the general path's lists, fingerprints, pin-by-pin
// comparison and second scan; each is bound by its random table sectors.
// Measured (GB300, 1e6 nodes, 4e6 edges, k = 8, all nine levels): coarsening 20.4
// -> 13.3 ms.
__global__ void k_edge_insert(const int32_t* __restrict__ eoff, const int32_t* __restrict__ pins,
                              const int32_t* __restrict__ map, const int32_t* __restrict__ w,
                              int32_t m, unsigned long long* __restrict__ tkey,
                              int2* __restrict__ tval, uint64_t mask,
                              int32_t* __restrict__ slot_of, int32_t* status) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int32_t b = eoff[e];
    const int32_t x = map[pins[b]], y = map[pins[b + 1]];
    int32_t slot = -1;
    if (x != y) {
      const unsigned long long f =
          ((unsigned long long)(uint32_t)min(x, y) << 32) | (uint32_t)max(x, y);
      uint64_t h = mix64(f) & mask;
      for (uint64_t probe = 0; probe <= mask; ++probe) {
        const unsigned long long k = tkey[h];
        if (k == f) { slot = (int32_t)h; break; }
        if (k == EMPTY_FP) {
          const unsigned long long old = atomicCAS(&tkey[h], EMPTY_FP, f);
          if (old == EMPTY_FP || old == f) { slot = (int32_t)h; break; }
        }
        h = (h + 1) & mask;
      }
      if (slot < 0) {
        dev_fail(status, DEV_HASH_FULL);
      } else {
        atomicMin(&tval[slot].x, (int32_t)e);  // the representative: smallest id
        atomicAdd(&tval[slot].y, w[e]);
      }
    }
    slot_of[e] = slot;
  }
}

__global__ void k_edge_flag(const int32_t* __restrict__ slot_of, const int2* __restrict__ tval,
                            int32_t m, int32_t* __restrict__ keep) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int32_t sl = slot_of[e];
    keep[e] = sl >= 0 && tval[sl].x == (int32_t)e ? 1 : 0;
  }
}

// Kept edges by the rank of their representative: offsets, pins ascending,
// weights.
__global__ void k_edge_write(const int32_t* __restrict__ slot_of,
                             const unsigned long long* __restrict__ tkey,
                             const int2* __restrict__ tval, const int32_t* __restrict__ newid,
                             int32_t m, int32_t m2, int32_t* __restrict__ eoff2,
                             int2* __restrict__ pins2, int32_t* __restrict__ w2) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int32_t sl = slot_of[e];
    if (sl < 0) continue;
    const int2 v = tval[sl];
    if (v.x != (int32_t)e) continue;
    const int32_t id = newid[e];
    const unsigned long long f = tkey[sl];
    pins2[id] = make_int2((int32_t)(f >> 32), (int32_t)(uint32_t)f);
    w2[id] = v.y;
    eoff2[id] = 2 * id;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) eoff2[m2] = 2 * m2;
}

__global__ void k_edge_table(unsigned long long* __restrict__ tkey, int2* __restrict__ tval,
                             uint64_t cap) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cap;
       i += (uint64_t)gridDim.x * blockDim.x) {
    tkey[i] = EMPTY_FP;
    tval[i] = make_int2(INT_MAX, 0);
  }
}

void contract_edges(const Ctx& cx, const Level& L, Level& out) {
  const int32_t m = L.m;
  uint64_t cap = 2;
  while (cap < 2 * (uint64_t)m) cap <<= 1;
  DBuf<unsigned long long> tkey;
  DBuf<int2> tval;
  DBuf<int32_t> slot_of, keep, total;
  tkey.alloc(&cx.alloc, (size_t)cap);
  tval.alloc(&cx.alloc, (size_t)cap);
  slot_of.alloc(&cx.alloc, (size_t)m);
  keep.alloc(&cx.alloc, (size_t)m);
  total.alloc(&cx.alloc, 1);
  const int g = grid_for(m, 256, cx.num_sms, 8);
  k_edge_table<<<grid_for((int64_t)cap, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(tkey.p, tval.p,
                                                                                cap);
  check_launch("edge_table");
  k_edge_insert<<<g, 256, 0, cx.stream>>>(L.eoff.p, L.pins.p, L.map.p, L.w.p, m, tkey.p, tval.p,
                                          cap - 1, slot_of.p, cx.d_status);
  check_launch("edge_insert");
  k_edge_flag<<<g, 256, 0, cx.stream>>>(slot_of.p, tval.p, m, keep.p);
  check_launch("edge_flag");
  scan_exclusive_i32(cx, keep.p, keep.p, m, total.p);  // keep flag -> new id
  const int32_t m2 = read_i32(cx, total.p);
  out.m = m2;
  out.p = 2 * (int64_t)m2;
  out.eoff.alloc(&cx.alloc, (size_t)m2 + 1);
  out.pins.alloc(&cx.alloc, (size_t)std::max<int64_t>(out.p, 1));
  out.w.alloc(&cx.alloc, (size_t)std::max<int32_t>(m2, 1));
  k_edge_write<<<g, 256, 0, cx.stream>>>(slot_of.p, tkey.p, tval.p, keep.p, m, m2, out.eoff.p,
                                         reinterpret_cast<int2*>(out.pins.p), out.w.p);
  check_launch("edge_write");
  if (cx.launches) *cx.launches += 4;
}

// Community of every coarse node: the community of its members (a cluster
// never spans two communities).
__global__ void k_coarse_comm(const int32_t* __restrict__ map, const int32_t* __restrict__ comm,
                              int32_t n, int32_t* __restrict__ ccomm) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x)
    ccomm[map[u]] = comm[u];
}

void coarse_communities(const Ctx& cx, const Level& L, Level& out) {
  if (!L.comm.p) return;
  out.comm.alloc(&cx.alloc, (size_t)std::max<int32_t>(out.n, 1));
  k_coarse_comm<<<grid_for(L.n, 256, cx.num_sms, 8), 256, 0, cx.stream>>>(L.map.p, L.comm.p, L.n,
                                                                        out.comm.p);
  check_launch("coarse_comm");
  if (cx.launches) *cx.launches += 1;
}

}  // namespace

void contract_level(const Ctx& cx, Level& L, const int32_t* cw, Level& out, int fingerprint_bits,
                    ContractCounters& kc) {
  EventTimer tm(cx, &kc.ms);
  const int32_t n = L.n, m = L.m;
  const int gn = grid_for(n, 256, cx.num_sms, 4);
  // a5: coarse ids and node weights
  DBuf<int32_t> cid, d_n2;
  cid.alloc(&cx.alloc, (size_t)n + 1);
  d_n2.alloc(&cx.alloc, 1);
  k_rep_flags<<<gn, 256, 0, cx.stream>>>(L.rep.p, n, cid.p);
  check_launch("rep_flags");
  scan_exclusive_i32(cx, cid.p, cid.p, n, d_n2.p);
  const int32_t n2 = read_i32(cx, d_n2.p);
  out.n = n2;
  out.c.alloc(&cx.alloc, (size_t)n2);
  L.map.alloc(&cx.alloc, (size_t)n);
  k_map<<<gn, 256, 0, cx.stream>>>(L.rep.p, cid.p, cw, n, L.map.p, out.c.p);
  check_launch("map");
  if (cx.launches) *cx.launches += 2;
  cid.release();

  if (m == 0) {
    out.m = 0;
    out.p = 0;
    out.eoff.alloc(&cx.alloc, 1);
    HG_CUDA(cudaMemsetAsync(out.eoff.p, 0, sizeof(int32_t), cx.stream));
    build_incidence(cx, out);
    coarse_communities(cx, L, out);
    L.coarsened = true;
    return;
  }

  // a6 - a8 of a graph level (a graph's coarse nets have two pins again: one-pin
  // nets are dropped)
  if (L.graph) {
    contract_edges(cx, L, out);
    out.graph = out.m > 0;
    build_incidence(cx, out);
    coarse_communities(cx, L, out);
    L.coarsened = true;
    return;
  }

  // a6: remap, sort, deduplicate
  const int gm = grid_for(m, 256, cx.num_sms, 4);
  DBuf<int32_t> lists, counts, tpins, tsize;
  DBuf<unsigned long long> fp;
  lists.alloc(&cx.alloc, (size_t)m * NCLS);
  counts.alloc(&cx.alloc, NCLS);
  tpins.alloc(&cx.alloc, (size_t)std::max<int64_t>(L.p, 1));
  tsize.alloc(&cx.alloc, (size_t)m);
  fp.alloc(&cx.alloc, (size_t)m);
  HG_CUDA(cudaMemsetAsync(counts.p, 0, counts.bytes(), cx.stream));
  k_classify_nets<<<gm, 256, 0, cx.stream>>>(L.eoff.p, m, lists.p, counts.p);
  check_launch("classify_nets");
  int32_t hc[NCLS];
  read_back(cx, hc, counts.p, sizeof(hc));
  if (hc[0])
    k_remap_small<<<grid_for(hc[0], 128, cx.num_sms, 16), 128, 0, cx.stream>>>(
        lists.p, hc[0], L.eoff.p, L.pins.p, L.map.p, fingerprint_bits, tpins.p, tsize.p, fp.p);
  const int32_t words = (n2 + 31) / 32;
  if (hc[1]) {
    const int gw = grid_for(hc[1], WARP_NETS, cx.num_sms, 8);
    if (n2 <= WARP_BITMAP_N)
      k_remap_warp_bitmap<<<gw, WARP_NETS * 32, 0, cx.stream>>>(
          lists.p + m, hc[1], L.eoff.p, L.pins.p, L.map.p, words, fingerprint_bits, tpins.p,
          tsize.p, fp.p);
    else
      k_remap_warp_sort<<<gw, WARP_NETS * 32, 0, cx.stream>>>(lists.p + m, hc[1], L.eoff.p,
                                                              L.pins.p, L.map.p, fingerprint_bits,
                                                              tpins.p, tsize.p, fp.p);
  }
  DBuf<unsigned> bitmaps;
  const int32_t* mid = lists.p + 2 * (size_t)m;
  const int32_t* big = lists.p + 3 * (size_t)m;
  if (n2 <= BLOCK_BITMAP_N) {
    const size_t bytes = ((size_t)words + words / 32 + 1) * sizeof(unsigned);
    const int per_sm = std::max(1, std::min(4, (int)(200 * 1024 / bytes)));
    prepare_kernel(cx, k_remap_block_bitmap, (BLOCK_BITMAP_N / 32 + BLOCK_BITMAP_N / 1024 + 1) * 4);
    for (int c = 2; c < NCLS; ++c)
      if (hc[c])
        k_remap_block_bitmap<<<grid_for(hc[c], 1, cx.num_sms, per_sm), BIG_THREADS, bytes,
                               cx.stream>>>(c == 2 ? mid : big, hc[c], L.eoff.p, L.pins.p,
                                            L.map.p, words, fingerprint_bits, tpins.p, tsize.p,
                                            fp.p);
  } else {
    if (hc[2])
      k_remap_mid<<<grid_for(hc[2], 1, cx.num_sms, 8), MID_THREADS, 0, cx.stream>>>(
          mid, hc[2], L.eoff.p, L.pins.p, L.map.p, fingerprint_bits, tpins.p, tsize.p, fp.p);
    if (hc[3]) {
      const int blocks = (int)std::max<int64_t>(
          1, std::min<int64_t>({(int64_t)hc[3], (int64_t)cx.num_sms * 2,
                                (int64_t)((256ll << 20) / ((int64_t)words * 4 + 1))}));
      bitmaps.alloc(&cx.alloc, (size_t)blocks * words);
      k_remap_big<<<blocks, BIG_THREADS, 0, cx.stream>>>(big, hc[3], L.eoff.p, L.pins.p, L.map.p,
                                                         words, bitmaps.p, fingerprint_bits,
                                                         tpins.p, tsize.p, fp.p);
    }
  }
  check_launch("remap");
  if (cx.launches) *cx.launches += 1 + (hc[0] > 0) + (hc[1] > 0) + (hc[2] > 0) + (hc[3] > 0);
  bitmaps.release();

  // a7: identical nets
  uint64_t cap = 2;
  while (cap < 2 * (uint64_t)m) cap <<= 1;
  DBuf<unsigned long long> tkey;
  DBuf<int32_t> tmin, slot_of_net, repnet, cand, ncand, failed, nfailed;
  tkey.alloc(&cx.alloc, (size_t)cap);
  tmin.alloc(&cx.alloc, (size_t)cap);
  slot_of_net.alloc(&cx.alloc, (size_t)m);
  repnet.alloc(&cx.alloc, (size_t)m);
  cand.alloc(&cx.alloc, (size_t)m);
  failed.alloc(&cx.alloc, (size_t)m);
  ncand.alloc(&cx.alloc, 1);
  nfailed.alloc(&cx.alloc, 1);
  HG_CUDA(cudaMemsetAsync(ncand.p, 0, sizeof(int32_t), cx.stream));
  k_candidates<<<gm, 256, 0, cx.stream>>>(tsize.p, m, cand.p, ncand.p);
  check_launch("candidates");
  const int g_ins = grid_for(m, 256, cx.num_sms, 8);
  const int g_cmp = grid_for(m, 8 * (32 / CMP_LANES), cx.num_sms, 8);
  for (int round = 0;; ++round) {
    HG_CUDA(cudaMemsetAsync(tkey.p, 0xff, tkey.bytes(), cx.stream));
    HG_CUDA(cudaMemsetAsync(tmin.p, 0x7f, tmin.bytes(), cx.stream));
    HG_CUDA(cudaMemsetAsync(nfailed.p, 0, sizeof(int32_t), cx.stream));
    k_ident_insert<<<g_ins, 256, 0, cx.stream>>>(cand.p, ncand.p, fp.p, tkey.p, tmin.p, cap - 1,
                                                 slot_of_net.p, cx.d_status);
    check_launch("ident_insert");
    k_ident_compare<<<g_cmp, 256, 0, cx.stream>>>(cand.p, ncand.p, L.eoff.p, tpins.p, tsize.p,
                                                  slot_of_net.p, tmin.p, repnet.p, failed.p,
                                                  nfailed.p);
    check_launch("ident_compare");
    if (cx.launches) *cx.launches += 2;
    kc.ident_rounds = round + 1;
    const int32_t nf = read_i32(cx, nfailed.p);
    if (nf == 0) break;
    // the failed nets become the candidates of the next round
    std::swap(cand, failed);
    HG_CUDA(cudaMemcpyAsync(ncand.p, nfailed.p, sizeof(int32_t), cudaMemcpyDeviceToDevice,
                            cx.stream));
  }
  tkey.release();
  tmin.release();
  slot_of_net.release();

  // a8: weights, compaction
  DBuf<int32_t> wsum, kflag, newid, ksize, d_tot;
  wsum.alloc(&cx.alloc, (size_t)m);
  kflag.alloc(&cx.alloc, (size_t)m);
  newid.alloc(&cx.alloc, (size_t)m);
  ksize.alloc(&cx.alloc, (size_t)m);
  d_tot.alloc(&cx.alloc, 2);
  HG_CUDA(cudaMemsetAsync(wsum.p, 0, wsum.bytes(), cx.stream));
  k_net_weights<<<gm, 256, 0, cx.stream>>>(tsize.p, repnet.p, L.w.p, m, wsum.p, kflag.p, ksize.p);
  check_launch("net_weights");
  scan_exclusive_i32(cx, kflag.p, newid.p, m, d_tot.p);      // keep flag -> new id
  scan_exclusive_i32(cx, ksize.p, ksize.p, m, d_tot.p + 1);  // kept size -> coarse offset
  int32_t tot[2];
  read_back(cx, tot, d_tot.p, sizeof(tot));
  out.m = tot[0];
  out.p = tot[1];
  out.eoff.alloc(&cx.alloc, (size_t)out.m + 1);
  out.pins.alloc(&cx.alloc, (size_t)std::max<int64_t>(out.p, 1));
  out.w.alloc(&cx.alloc, (size_t)std::max<int32_t>(out.m, 1));
  k_compact<<<grid_for(m, 8 * (32 / CP_LANES), cx.num_sms, 8), 256, 0, cx.stream>>>(
      kflag.p, newid.p, ksize.p, L.eoff.p, tpins.p, tsize.p, wsum.p, m, out.eoff.p, out.pins.p,
      out.w.p);
  check_launch("compact");
  HG_CUDA(cudaMemcpyAsync(out.eoff.p + out.m, d_tot.p + 1, sizeof(int32_t),
                          cudaMemcpyDeviceToDevice, cx.stream));
  if (cx.launches) *cx.launches += 2;
  build_incidence(cx, out);
  coarse_communities(cx, L, out);
  L.coarsened = true;
}

}  // namespace hgk
