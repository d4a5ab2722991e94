// How the local moving of the Louvain method (community.cu) takes a vertex.
#pragma once

#include <stdint.h>

namespace hgk {

constexpr int LV_ROUNDS = 5;
constexpr int LV_CLASSES = 6;
constexpr int LV_GROUP = 8;       // class 0: degree <= 8, eight lanes per vertex
constexpr int LV_LANES = 32;      // class 1: degree <= 32, a warp per vertex
constexpr int LV_SMALL = 256;     // class 2: degree <= 256, a warp and a shared table
constexpr int LV_BLOCK = 4096;    // class 3: degree <= 4096, a block
constexpr int LV_HUGE = 32768;    // class 4: degree <= 32768, a block per part
constexpr int LV_PART = 2048;     //          of the neighbouring clusters
constexpr int LV_CHUNK = 1024;    // class 5: a block per chunk of the edges

// Class and list entries of a vertex of degree deg > 0.  The parts of a class 4
// vertex each walk all of its edges, sixteen times its degree at most; above that
// an edge is read once and its weight added to a table in global memory, at the
// price of the table's passes and a barrier.  Detection on 200,000 nodes with 60
// nets of 20,000, 30,000, 40,000 and 60,000 pins: in parts at any size 22.0, 21.5,
// 22.9 and 26.7 ms, with this limit 22.3, 19.3, 16.0 and 17.8 ms; one net of 1e6
// pins 55.8 -> 18.4 ms.  (Half the limit: 4 nets of 30,000 pins 5 % slower, 60 nets
// of 20,000 pins 5 % faster.)
// (The parts hold clusters by a hash of their ids; `huge` = LV_BLOCK leaves class 4
// out for ids that meet in one part.)
__host__ __device__ inline int lv_class(long long deg, int huge, int32_t& entries) {
  entries = 1;
  if (deg <= LV_GROUP) return 0;
  if (deg <= LV_LANES) return 1;
  if (deg <= LV_SMALL) return 2;
  if (deg <= LV_BLOCK) return 3;
  if (deg <= huge) {
    entries = (int32_t)((deg + LV_PART - 1) / LV_PART);
    return 4;
  }
  entries = (int32_t)((deg + LV_CHUNK - 1) / LV_CHUNK);
  return 5;
}

// Slots of a class 5 vertex's table: a power of two above twice its neighbours.
__host__ __device__ inline unsigned long long lv_slots(long long deg) {
  unsigned long long s = 4;
  while (s < 2ull * (unsigned long long)deg + 2) s <<= 1;
  return s;
}

}  // namespace hgk
