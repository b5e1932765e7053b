// Fingerprint partitions of the variant records (the coarse half of Appendix
// A, XTNeighbor step 4).
//
// Grouping needs equal fingerprints together, not a total order, and the
// fingerprints are uniform but for repeats.  So one pass takes every record
// to the partition named by its top pbits bits: 2^pbits regions of `region`
// records, a few standard deviations larger than the mean, filled through one
// counter per partition.  Against stable radix passes there is no digit count
// beforehand and no look-back: a tile reserves its room in every partition
// with atomics.  Records past a region's end go to a spill buffer, and the
// filter then hands the whole partition to the exact global grouping, so
// skewed inputs (one sequence many times) stay correct.
//
// What bounds a pass into thousands of partitions is the number of write
// requests: the memory system takes about 45 G lines/s, whatever part of a
// 128-byte line they hold (104.8 M records written in runs of 44: 148 us, of
// 11: 463 us, of 5: 725 us; every line reaches DRAM once all the same, as a
// region's open end stays in L2).  So a tile is as large as shared memory
// allows, and the partitions as few as the filter can take.
//
// A block loops over tiles: count the tile's records into shared-memory
// bins, scan the bins, reserve, place the records in shared memory in
// partition order, write the runs.  The next tile's loads are issued before
// the write-out, into the registers that the placing has freed.
#include <algorithm>
#include <cmath>

#include "partition.cuh"
#include "per_device.h"
#include "xtn_common.cuh"
#include "xtn_kernels.h"

namespace xtn {

namespace {

constexpr int PT_THREADS = 512;
constexpr int SPLIT_COARSE_BITS = 9;  // partitions of the first of two levels
constexpr int SPLIT_MAX_BITS = 8;     // and of each of those

// A tile's records, then the bins' counters and output offsets.
template <int ITEMS>
constexpr size_t partition_smem_bytes(int pbits) {
  return (size_t)PT_THREADS * ITEMS * 8 + ((size_t)8 << pbits);
}

template <int ITEMS, int MIN_BLOCKS>
__global__ void __launch_bounds__(PT_THREADS, MIN_BLOCKS)
    k_partition(const uint64_t* __restrict__ in, int64_t n_cap,
                const uint64_t* __restrict__ n_dev, int pbits, uint64_t* __restrict__ out,
                uint32_t region, uint32_t* __restrict__ part_count, uint64_t* __restrict__ spill,
                uint64_t spill_cap, unsigned long long* __restrict__ n_spill,
                uint32_t* __restrict__ err) {
  constexpr int TILE = PT_THREADS * ITEMS;
  constexpr int BATCH = ITEMS / 2;
  extern __shared__ __align__(16) unsigned char pt_smem[];
  uint64_t* s_stage = reinterpret_cast<uint64_t*>(pt_smem);
  const uint32_t P = 1u << pbits;
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(s_stage + TILE);
  uint32_t* s_pos = s_cnt + P;
  __shared__ uint32_t s_wsum[8];
  __shared__ uint32_t s_held, s_over, s_shift;
  const uint32_t warp = threadIdx.x >> 5, lane = lane_id();
  const int64_t n = n_dev ? min((int64_t)*n_dev, n_cap) : n_cap;
  const uint32_t shift = 32u - (uint32_t)pbits;
  const bool wide = ((uint64_t)region << pbits) >> 32 != 0;  // past 32-bit indices
  for (uint32_t k = threadIdx.x; k < P; k += PT_THREADS) s_cnt[k] = 0;
  if (threadIdx.x == 0) {
    s_over = 0;  // a region has run over
    s_shift = shift;
  }
  uint64_t rec[ITEMS];
  const uint32_t first = warp * 32 * ITEMS + lane;  // of this thread in a tile
  const int64_t n_tiles = (n + TILE - 1) / TILE;
  auto load = [&](int64_t t) {
    const uint64_t* src = in + t * TILE + first;
    if ((t + 1) * TILE <= n) {
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) rec[i] = __ldcs(src + i * 32);
    } else {
      const int64_t held = n - t * TILE;  // none or less for the tile after the last
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) rec[i] = first + i * 32 < held ? __ldcs(src + i * 32) : 0ull;
    }
  };
  load(blockIdx.x);
  __syncthreads();
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const uint32_t held = (uint32_t)min((int64_t)TILE, n - tile * TILE);
    const bool full = held == (uint32_t)TILE;
    auto bin_of = [&](uint64_t r, uint32_t sh) { return (uint32_t)(r >> 32) >> sh; };
    // 1. count
#pragma unroll
    for (int i = 0; i < ITEMS; ++i)
      if (full || first + i * 32 < held) atomicAdd(&s_cnt[bin_of(rec[i], shift)], 1u);
    __syncthreads();
    // 2. exclusive scan of the bins, then room in every partition
    scan_bins(s_cnt, P >> 8, s_wsum, &s_held);
    reserve_room<PT_THREADS>(s_cnt, s_pos, P, held, region, part_count, &s_over);
    __syncthreads();
    // 3. place in partition order: BATCH places are asked for before the
    // first is used, or each would wait for its own shared-memory round trip.
    // The shift is read back from shared memory so that the bins are computed
    // again: kept from step 1 they would cost a register per record.
    const uint32_t shift3 = s_shift;
#pragma unroll
    for (int i0 = 0; i0 < ITEMS; i0 += BATCH) {
      uint32_t at[BATCH];
#pragma unroll
      for (int x = 0; x < BATCH; ++x) {
        const int i = i0 + x;
        at[x] = TILE;
        if (full || first + i * 32 < held) at[x] = atomicAdd(&s_cnt[bin_of(rec[i], shift3)], 1u);
      }
#pragma unroll
      for (int x = 0; x < BATCH; ++x)
        if (at[x] < (uint32_t)TILE) s_stage[at[x]] = rec[i0 + x];
    }
    __syncthreads();
    // 4. write the runs out, the next tile's loads under way
    const bool over = s_over || wide;
    load(tile + gridDim.x);
    for (uint32_t k = threadIdx.x; k < P / 4; k += PT_THREADS)
      reinterpret_cast<uint4*>(s_cnt)[k] = make_uint4(0u, 0u, 0u, 0u);
    if (!over) {
#pragma unroll 4
      for (uint32_t j = threadIdx.x; j < held; j += PT_THREADS) {
        const uint64_t v = s_stage[j];
        out[s_pos[bin_of(v, shift)] + j] = v;
      }
    } else {
      for (uint32_t j = threadIdx.x; j < held; j += PT_THREADS) {
        const uint64_t v = s_stage[j];
        const uint32_t b = bin_of(v, shift);
        const uint32_t at = s_pos[b] + j - b * region;
        if (at < region) {
          out[(uint64_t)b * region + at] = v;
        } else {  // past the region's end
          const uint64_t o = atomicAdd(n_spill, 1ull);
          if (o < spill_cap) spill[o] = v;
          else atomicOr(err, DERR_RANGE);
        }
      }
    }
    __syncthreads();  // the stage and the bins are reused
  }
}

template <int ITEMS, int MIN_BLOCKS>
void partition_launch(const uint64_t* in, int64_t n, const uint64_t* n_dev, const Partitions& p,
                      int max_bits, int sms, uint32_t* err, cudaStream_t s) {
  auto f = k_partition<ITEMS, MIN_BLOCKS>;
  static PerDevice shared;
  shared([&] {
    return allow_shared((const void*)f, (int)partition_smem_bytes<ITEMS>(max_bits));
  });
  const int64_t tiles = (n + PT_THREADS * ITEMS - 1) / (PT_THREADS * ITEMS);
  f<<<(uint32_t)std::min<int64_t>(tiles, (int64_t)sms * MIN_BLOCKS), PT_THREADS,
      partition_smem_bytes<ITEMS>(p.pbits), s>>>(
      in, n, n_dev, p.pbits, p.rec, p.region, p.count, p.spill, p.spill_cap,
      reinterpret_cast<unsigned long long*>(p.n_spill), err);
}

// The second level: every coarse partition once more by the `sub` bits below
// its own, in tiles of one partition each, with k_partition's steps.  With 2^5
// to 2^8 bins a tile's runs are 36 to 290 records long, against five at the
// end of one level: 3.97 G records (36M sequences, d = 2) 15.4 ms, 4.1 TB/s
// (with 22 records a thread, which spill registers, 18.3; 16 15.6).
template <int ITEMS, int MIN_BLOCKS>
__global__ void __launch_bounds__(PT_THREADS, MIN_BLOCKS)
    k_split(const uint64_t* __restrict__ in, const uint32_t* __restrict__ count, uint32_t region,
            int pbits, int sub, uint64_t* __restrict__ out, uint32_t fine_region,
            uint32_t* __restrict__ fine_count, uint64_t* __restrict__ spill, uint64_t spill_cap,
            unsigned long long* __restrict__ n_spill, uint32_t* __restrict__ err) {
  constexpr uint32_t TILE = PT_THREADS * ITEMS;
  constexpr int BATCH = ITEMS / 2;
  extern __shared__ __align__(16) unsigned char pt_smem[];
  uint64_t* s_stage = reinterpret_cast<uint64_t*>(pt_smem);
  __shared__ __align__(16) uint32_t s_cnt[1 << SPLIT_MAX_BITS];
  __shared__ uint32_t s_pos[1 << SPLIT_MAX_BITS];
  __shared__ uint32_t s_wsum[8];
  __shared__ uint32_t s_held, s_over;
  __shared__ unsigned long long s_base;
  static_assert((1 << SPLIT_MAX_BITS) == 256, "one bin a thread in scan_bins");
  const uint32_t warp = threadIdx.x >> 5, lane = lane_id();
  const uint32_t F = 1u << sub;
  const uint32_t per = (region + TILE - 1) / TILE;  // tiles of a partition
  const uint32_t n_tiles = per << pbits;
  const bool wide = ((uint64_t)fine_region << (pbits + sub)) >> 32 != 0;  // past 32-bit indices
  if (threadIdx.x < 256) s_cnt[threadIdx.x] = 0;
  if (threadIdx.x == 0) s_over = 0;  // a region has run over
  uint64_t rec[ITEMS];
  const uint32_t first = warp * 32 * ITEMS + lane;  // of this thread in a tile
  // tile -> its partition, its records and whether the partition ran over
  auto locate = [&](uint32_t tile, uint32_t& part, uint32_t& at, bool& ran_over) -> uint32_t {
    part = tile / per;
    at = (tile - part * per) * TILE;
    ran_over = false;
    if (tile >= n_tiles) return 0u;
    const uint32_t m = count[part];
    ran_over = m > region;
    const uint32_t have = min(m, region);
    return have > at ? min(have - at, TILE) : 0u;
  };
  auto load = [&](uint32_t part, uint32_t at, uint32_t held) {
    const uint64_t* src = in + (uint64_t)part * region + at + first;
    if (held == TILE) {
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) rec[i] = __ldcs(src + i * 32);
    } else {
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) rec[i] = first + i * 32 < held ? __ldcs(src + i * 32) : 0ull;
    }
  };
  auto bin_of = [&](uint64_t r) { return (uint32_t)(r >> 32) << pbits >> (32 - sub); };
  uint32_t part, next_part, next_at;
  bool ran_over, next_over;
  uint32_t held = locate(blockIdx.x, part, next_at, ran_over);
  load(part, next_at, held);
  __syncthreads();
  for (uint32_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const uint32_t f0 = part << sub;  // its first fine partition
    const bool full = held == TILE;
    const uint32_t next = locate(tile + gridDim.x, next_part, next_at, next_over);
    if (ran_over) {  // uniform: the region's records to the global grouping
      if (threadIdx.x == 0 && held) s_base = atomicAdd(n_spill, (unsigned long long)held);
      __syncthreads();
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) {
        const uint32_t k = first + i * 32;
        if (k < held) {
          if (s_base + k < spill_cap) spill[s_base + k] = rec[i];
          else atomicOr(err, DERR_RANGE);
        }
      }
      load(next_part, next_at, next);
    } else if (held) {
      // 1. count
#pragma unroll
      for (int i = 0; i < ITEMS; ++i)
        if (full || first + i * 32 < held) atomicAdd(&s_cnt[bin_of(rec[i])], 1u);
      __syncthreads();
      // 2. exclusive scan of the bins, then room in every fine partition
      scan_bins(s_cnt, 1, s_wsum, &s_held);
      if (threadIdx.x < F) {
        const uint32_t b = threadIdx.x, at = s_cnt[b];
        const uint32_t c = (b + 1 < F ? s_cnt[b + 1] : held) - at;
        const uint32_t room = c ? atomicAdd(&fine_count[f0 + b], c) : 0u;
        s_pos[b] = (f0 + b) * fine_region + room - at;  // modulo 2^32
        if (room + c > fine_region) s_over = 1;
      }
      __syncthreads();
      // 3. place in partition order
#pragma unroll
      for (int i0 = 0; i0 < ITEMS; i0 += BATCH) {
        uint32_t at[BATCH];
#pragma unroll
        for (int x = 0; x < BATCH; ++x) {
          const int i = i0 + x;
          at[x] = TILE;
          if (full || first + i * 32 < held) at[x] = atomicAdd(&s_cnt[bin_of(rec[i])], 1u);
        }
#pragma unroll
        for (int x = 0; x < BATCH; ++x)
          if (at[x] < TILE) s_stage[at[x]] = rec[i0 + x];
      }
      __syncthreads();
      // 4. write the runs out, the next tile's loads under way
      const bool over = s_over || wide;
      load(next_part, next_at, next);
      if (threadIdx.x < 256) s_cnt[threadIdx.x] = 0;
      if (!over) {
#pragma unroll 4
        for (uint32_t j = threadIdx.x; j < held; j += PT_THREADS) {
          const uint64_t v = s_stage[j];
          out[s_pos[bin_of(v)] + j] = v;
        }
      } else {
        for (uint32_t j = threadIdx.x; j < held; j += PT_THREADS) {
          const uint64_t v = s_stage[j];
          const uint32_t b = bin_of(v), f = f0 + b;
          const uint32_t at = s_pos[b] + j - f * fine_region;
          if (at < fine_region) {
            out[(uint64_t)f * fine_region + at] = v;
          } else {  // past the region's end
            const uint64_t o = atomicAdd(n_spill, 1ull);
            if (o < spill_cap) spill[o] = v;
            else atomicOr(err, DERR_RANGE);
          }
        }
      }
    } else {
      load(next_part, next_at, next);
    }
    __syncthreads();  // the stage and the bins are reused
    part = next_part;
    ran_over = next_over;
    held = next;
  }
}

// Records of a region for `mean` expected ones.
uint32_t region_of(double mean) {
  return ((uint32_t)(mean + 8.0 * std::sqrt(mean)) + 128u + 15u) & ~15u;
}

}  // namespace

// 2^11 partitions where that leaves 20,000 to 80,000 records in one on
// average (times 2^(fx - 1)), more or fewer else: the filter's bitmaps take
// 50,000 well, but half as many partitions save the expansion more than the
// fuller bitmaps cost the filter (157 M records in 2^11 instead of 2^12: 1.28
// + 0.47 against 1.53 + 0.49 ms), and smaller ones let the last blocks of
// small inputs end together.  No more than 2^13 partitions, what a tile's
// counters leave room for, and no fewer than 2^8, so that every SM has some.
// More records than 2^13 such partitions take go through two levels, 2^9 and up
// to 2^8 each: fuller bitmaps keep more and more lone records, and a list is
// read once for every 5,600 of them.  Whole searches at d = 2, one level against
// two: 0.55 G records 8.8 and 9.2 ms, 0.77 G 13.2 and 11.9, 0.99 G 17.7 and
// 15.7 (0.9 more with 2^11 in the first level); 2.0 G 32 with two and 96 with
// one whose bitmap had a bit less to go by, 4.0 G 66 and 734.
PartitionShape choose_partitions(uint64_t n_rec, int fx) {
  PartitionShape g;
  const uint64_t most = (uint64_t)40000 << fx, least = (uint64_t)10000 << fx;
  int b = 11;
  while (b > 8 && (n_rec >> b) < least) --b;
  while (b < PART_MAX_BITS && (n_rec >> b) > most) ++b;
  g.pbits = b;
  if ((n_rec >> b) > most) {
    // split again before the filter
    int t = b;
    while (t < SPLIT_COARSE_BITS + SPLIT_MAX_BITS && (n_rec >> t) > most) ++t;
    b = SPLIT_COARSE_BITS;
    g.sub = t - b;
    g.fine_region = region_of(std::ldexp((double)n_rec, -t));
  }
  g.pbits = b;
  g.region = region_of(std::ldexp((double)n_rec, -b));
  return g;
}

void launch_split(const Partitions& p, uint64_t n_rec, int sms, uint32_t* err, cudaStream_t s) {
  constexpr int ITEMS = 18, MIN_BLOCKS = 2;
  constexpr int smem = PT_THREADS * ITEMS * 8;
  auto f = k_split<ITEMS, MIN_BLOCKS>;
  static PerDevice shared;
  shared([&] { return allow_shared((const void*)f, smem); });
  const Partitions q = p.fine();
  prof_begin(s, "k_split", (double)n_rec * 16.0);
  f<<<(uint32_t)sms * MIN_BLOCKS, PT_THREADS, smem, s>>>(
      p.rec, p.count, p.region, p.pbits, p.sub, q.rec, q.region, q.count, p.spill, p.spill_cap,
      reinterpret_cast<unsigned long long*>(p.n_spill), err);
  prof_end(s);
}

void launch_partition(const uint64_t* in, int64_t n, const uint64_t* n_dev, const Partitions& p,
                      int sms, uint32_t* err, cudaStream_t s) {
  if (n <= 0) return;
  prof_begin(s, "k_onesweep_records", (double)n * 16.0);
  // two blocks per SM as long as the counters leave room for two tiles
  if (p.pbits <= 11) partition_launch<22, 2>(in, n, n_dev, p, 11, sms, err, s);
  else if (p.pbits == 12) partition_launch<18, 2>(in, n, n_dev, p, 12, sms, err, s);
  else partition_launch<22, 1>(in, n, n_dev, p, PART_MAX_BITS, sms, err, s);
  prof_end(s);
}

}  // namespace xtn
