// Shared by the two partitioning passes (k_scatter.cu, k_partition.cu).
#pragma once

#include "xtn_common.cuh"

namespace xtn {

constexpr int PART_MAX_BITS = 13;  // partitions, at most 2^13

// s_cnt[0 .. 256 per) becomes its exclusive prefix sums, *s_total the sum
// (whole block; ends with a barrier).  Thread t < 256 takes `per` bins from
// t per on, four at a time where there are as many (one 16-byte access for
// four bins, which spares the bank conflicts of a stride).
__device__ __forceinline__ void scan_bins(uint32_t* s_cnt, uint32_t per, uint32_t* s_wsum,
                                          uint32_t* s_total) {
  const uint32_t warp = threadIdx.x >> 5, lane = lane_id();
  uint4* v4 = reinterpret_cast<uint4*>(s_cnt) + threadIdx.x * (per >> 2);
  uint32_t* v1 = s_cnt + threadIdx.x * per;
  uint32_t sum = 0, inc = 0;
  if (threadIdx.x < 256) {
    if (per >= 4) {
      for (uint32_t k = 0; k < per >> 2; ++k) {
        const uint4 c = v4[k];
        sum += c.x + c.y + c.z + c.w;
      }
    } else {
      for (uint32_t k = 0; k < per; ++k) sum += v1[k];
    }
    inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(FULL_MASK, inc, o);
      if (lane >= (uint32_t)o) inc += t;
    }
    if (lane == 31) s_wsum[warp] = inc;
  }
  __syncthreads();
  if (threadIdx.x < 256) {
    uint32_t at = inc - sum;
    for (uint32_t w = 0; w < warp; ++w) at += s_wsum[w];
    if (per >= 4) {
      for (uint32_t k = 0; k < per >> 2; ++k) {
        const uint4 c = v4[k];
        uint4 o;
        o.x = at;
        o.y = o.x + c.x;
        o.z = o.y + c.y;
        o.w = o.z + c.z;
        at = o.w + c.w;
        v4[k] = o;
      }
    } else {
      for (uint32_t k = 0; k < per; ++k) {
        const uint32_t c = v1[k];
        v1[k] = at;
        at += c;
      }
    }
    if (threadIdx.x == 255) *s_total = at;
  }
  __syncthreads();
}

// Room for a tile's records in every partition, after scan_bins: s_pos[b] +
// (the record's place in the tile) is its output index modulo 2^32, the
// partitions being `region` words long.  Neighbouring lanes
// reserve in neighbouring partitions, so that a warp's 32 atomics are one
// request to one L2 line (spread over the lanes by a stride they were the
// bottleneck: 430 us of a 1.27 ms pass).
template <int THREADS>
__device__ __forceinline__ void reserve_room(const uint32_t* s_cnt, uint32_t* s_pos, uint32_t P,
                                             uint32_t held, uint32_t region,
                                             uint32_t* __restrict__ part_count,
                                             uint32_t* s_over) {
  for (uint32_t b = threadIdx.x; b < P; b += THREADS) {
    const uint32_t at = s_cnt[b];
    const uint32_t c = (b + 1 < P ? s_cnt[b + 1] : held) - at;
    const uint32_t room = c ? atomicAdd(&part_count[b], c) : 0u;
    s_pos[b] = b * region + room - at;  // modulo 2^32
    if (room + c > region) *s_over = 1;
  }
}

}  // namespace xtn
