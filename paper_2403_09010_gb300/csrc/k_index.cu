// The query index out of fingerprint partitions (Sec. 2.2: the hash map as a
// record array ordered by fingerprint, Appendix A, SymDel step 1).
//
// The expansion leaves the records in partitions of their top fingerprint
// bits (k_scatter.cu, k_partition.cu); k_index_build turns each into its
// stretch of the index.  A block counts its partition's records by directory
// entry in shared memory; the prefix sums are the directory's entries; then,
// as many entries at a time as fit, the records are placed in shared memory
// and leave in one coalesced run.  A range of up to INDEX_SCAN records stays
// in the order it came in, since a lookup compares all of it; longer ones are
// sorted for its binary search.
//
// Each record is read twice (the second time out of L2) and written once,
// against two radix passes, a sort of every bucket in shared memory, a copy
// and a pass for the directory: 36 M records (300,000 sequences, d = 2)
// 305 + 535 + 85 + 119 us, now 208 (and 91 more for the expansion, into
// partitions).  Each phase waits on shared memory with one block an SM; twice
// as many partitions for blocks of half the size take 170 us here but 36 more
// in the expansion, and records kept in registers between the two readings
// 20 more.
#include <algorithm>
#include <cmath>

#include "partition.cuh"
#include "per_device.h"
#include "xtn_common.cuh"
#include "xtn_kernels.h"

namespace xtn {

namespace {

constexpr int IX_THREADS = 1024;
constexpr uint32_t IX_STAGE = 19456;              // records placed at once
constexpr uint32_t IX_BINS = 1u << INDEX_SUB_BITS;  // directory entries of a partition, at most
constexpr uint32_t IX_LIST = IX_STAGE / (INDEX_SCAN + 1) + 1;
constexpr uint32_t IX_WARP_SORT = 1024;           // longer ranges take the whole block

struct IndexSmem {
  uint64_t stage[IX_STAGE];
  uint32_t bin[IX_BINS];  // 16-byte aligned
  uint32_t wsum[IX_THREADS / 32];
  uint32_t total, base, b1, o1, heads, n_list;
  uint16_t list[IX_LIST];
};

// a[0, n) in ascending order by `threads` threads (t = 0 .. threads - 1) that
// sync() together: the bitonic network whose first step of each merge mirrors,
// so that every exchange puts the smaller word first and words past n, were
// they there, would never move.
template <class Sync>
__device__ __forceinline__ void sort_range(uint64_t* a, uint32_t n, uint32_t t, uint32_t threads,
                                           Sync sync) {
  uint32_t N = 2;
  while (N < n) N <<= 1;
  auto order = [&](uint32_t x, uint32_t y) {
    if (y < n && a[x] > a[y]) {
      const uint64_t w = a[x];
      a[x] = a[y];
      a[y] = w;
    }
  };
  for (uint32_t size = 2; size <= N; size <<= 1) {
    const uint32_t half = size >> 1;
    for (uint32_t k = t; k < N / 2; k += threads) {
      const uint32_t b = (k & ~(half - 1u)) << 1, o = k & (half - 1u);
      order(b + o, b + size - 1u - o);
    }
    sync();
    for (uint32_t step = half >> 1; step > 0; step >>= 1) {
      for (uint32_t k = t; k < N / 2; k += threads) {
        const uint32_t x = ((k & ~(step - 1u)) << 1) | (k & (step - 1u));
        order(x, x + step);
      }
      sync();
    }
  }
}

__global__ void __launch_bounds__(IX_THREADS, 1)
    k_index_build(const uint64_t* __restrict__ parts, const uint32_t* __restrict__ count,
                  uint32_t region, int pbits, int dir_bits, int gshift,
                  uint64_t* __restrict__ rec, uint64_t n_rec, uint32_t* __restrict__ dir,
                  uint32_t sample, unsigned long long* __restrict__ n_groups,
                  uint32_t* __restrict__ err) {
  extern __shared__ __align__(16) unsigned char index_smem[];
  IndexSmem& S = *reinterpret_cast<IndexSmem*>(index_smem);
  const uint32_t p = blockIdx.x, lane = lane_id(), warp = threadIdx.x >> 5;
  const uint32_t m = min(count[p], region);
  const uint64_t* in = parts + (uint64_t)p * region;
  const int sub = dir_bits - pbits;  // 0 .. INDEX_SUB_BITS
  const uint32_t nb = 1u << sub, bmask = nb - 1u;
  const int bshift = 64 - dir_bits;
  const bool counts = p % sample == 0;  // its distinct keys, for all `sample` of them
  // this partition's place: the records of those before it; and whether any
  // ran over, as the caller then sorts globally
  uint32_t before = 0;
  bool ran_over = false;
  for (uint32_t q = threadIdx.x; q < gridDim.x; q += IX_THREADS) {
    const uint32_t c = count[q];
    if (q < p) before += min(c, region);
    ran_over |= c > region;
  }
  before = __reduce_add_sync(FULL_MASK, before);
  if (threadIdx.x == 0) S.base = S.heads = 0;
  for (uint32_t b = threadIdx.x; b < max(nb, 256u); b += IX_THREADS) S.bin[b] = 0;
  if (__syncthreads_or(ran_over)) return;
  if (lane == 0 && before) atomicAdd(&S.base, before);
  auto each = [&](auto f) {  // the partition's records, four loads in flight
    for (uint32_t k0 = threadIdx.x; k0 < m; k0 += 4 * IX_THREADS) {
      uint64_t r[4];
#pragma unroll
      for (int x = 0; x < 4; ++x) r[x] = k0 + x * IX_THREADS < m ? in[k0 + x * IX_THREADS] : 0ull;
#pragma unroll
      for (int x = 0; x < 4; ++x)
        if (k0 + x * IX_THREADS < m) f(r[x], (uint32_t)(r[x] >> bshift) & bmask);
    }
  };
  each([&](uint64_t, uint32_t b) { atomicAdd(&S.bin[b], 1u); });
  __syncthreads();
  scan_bins(S.bin, max(nb / 256u, 1u), S.wsum, &S.total);
  const uint32_t base = S.base;
  if (base + (uint64_t)m > n_rec) {  // uniform: the partitions hold more than was counted
    if (threadIdx.x == 0) atomicOr(err, DERR_RANGE);
    return;
  }
  for (uint32_t b = threadIdx.x; b < nb; b += IX_THREADS)
    dir[((uint64_t)p << sub) + b] = base + S.bin[b];
  if (p + 1 == gridDim.x && threadIdx.x == 0) dir[1ull << dir_bits] = base + m;

  uint32_t heads = 0;
  uint32_t b0 = 0, o0 = 0;  // entries before b0, their records, are done
  while (o0 < m) {
    if (threadIdx.x == 0) {  // as many entries as the stage holds
      uint32_t lo = b0, hi = nb;
      while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if ((mid < nb ? S.bin[mid] : m) - o0 <= IX_STAGE) lo = mid; else hi = mid - 1;
      }
      S.b1 = lo;
      S.o1 = lo < nb ? S.bin[lo] : m;
      S.n_list = 0;
    }
    __syncthreads();
    const uint32_t b1 = S.b1, o1 = S.o1;
    if (b1 == b0) {  // uniform: one entry beyond the stage; the caller sorts globally
      if (threadIdx.x == 0) atomicOr(err, DERR_CAPACITY);
      return;
    }
    each([&](uint64_t r, uint32_t b) {
      if (b >= b0 && b < b1) S.stage[atomicAdd(&S.bin[b], 1u) - o0] = r;
    });
    __syncthreads();
    // each entry's counter has moved to its end
    auto begin = [&](uint32_t b) { return b == b0 ? 0u : S.bin[b - 1] - o0; };
    for (uint32_t b = b0 + threadIdx.x; b < b1; b += IX_THREADS)
      if (S.bin[b] - o0 - begin(b) > (uint32_t)INDEX_SCAN)
        S.list[atomicAdd(&S.n_list, 1u)] = (uint16_t)b;  // at most IX_STAGE / (INDEX_SCAN + 1)
    __syncthreads();
    const uint32_t n_list = S.n_list;
    bool block = false;  // a range for the whole block is left
    for (uint32_t k = warp; k < n_list; k += IX_THREADS / 32) {
      const uint32_t b = S.list[k], s = begin(b), n = S.bin[b] - o0 - s;
      if (n <= IX_WARP_SORT)
        sort_range(S.stage + s, n, lane, 32, [] { __syncwarp(); });
      else
        block = true;
    }
    if (__syncthreads_or(block)) {
      for (uint32_t k = 0; k < n_list; ++k) {
        const uint32_t b = S.list[k], s = begin(b), n = S.bin[b] - o0 - s;
        if (n <= IX_WARP_SORT) continue;
        sort_range(S.stage + s, n, threadIdx.x, IX_THREADS, [] { __syncthreads(); });
      }
    }
    for (uint32_t k = threadIdx.x; k < o1 - o0; k += IX_THREADS) {
      const uint64_t r = S.stage[k], g = r >> gshift;
      rec[(uint64_t)base + o0 + k] = r;
      if (!counts) continue;
      // the first of its group key?  One look back where the range is sorted,
      // a few over what stands before it else
      const uint32_t b = (uint32_t)(r >> bshift) & bmask, s = begin(b);
      uint32_t y = S.bin[b] - o0 - s > (uint32_t)INDEX_SCAN && k > s ? k - 1 : s;
      while (y < k && (S.stage[y] >> gshift) != g) ++y;
      heads += y == k;
    }
    b0 = b1;
    o0 = o1;
    __syncthreads();  // the stage and the list are reused
  }
  heads = __reduce_add_sync(FULL_MASK, heads);
  if (lane == 0 && heads) atomicAdd(&S.heads, heads);
  __syncthreads();
  if (threadIdx.x == 0 && S.heads) atomicAdd(n_groups, (unsigned long long)S.heads * sample);
}

}  // namespace

// 2^8 to 2^11 partitions of up to 17,000 records or so (one fill of the
// stage) and as many directory entries as the counters hold; past those the
// index is sorted globally.  Regions half as large again as the mean: copies
// of one sequence all fall into one partition.  Where one overflows all the
// same, the blocks leave and the caller sorts: 300,000 sequences and 15,000
// copies of one, d = 2, 1.97 ms, as long as sorting at once; 1M and 60,000,
// d = 1, 1.46 (1.52).
bool choose_index_partitions(uint64_t n_rec, int dir_bits, PartitionShape* g) {
  int b = 8;
  while (b < 11 && (n_rec >> b) > 17000) ++b;
  if (dir_bits < b || dir_bits - b > INDEX_SUB_BITS || (n_rec >> b) > 1u << 16) return false;
  g->pbits = b;
  g->region = ((uint32_t)(1.5 * (double)n_rec / (double)(1u << b)) + 1024u + 15u) & ~15u;
  return true;
}

void launch_index_build(const Partitions& p, uint64_t n_rec, int dir_bits, int gshift,
                        uint64_t* rec, uint32_t* dir, uint64_t* n_groups, uint32_t* err,
                        cudaStream_t s) {
  static PerDevice shared;
  shared([] { return allow_shared((const void*)k_index_build, (int)sizeof(IndexSmem), false); });
  prof_begin(s, "k_index_build", (double)n_rec * 24.0 + 4.0 * (double)(1ull << dir_bits));
  k_index_build<<<1u << p.pbits, IX_THREADS, sizeof(IndexSmem), s>>>(
      p.rec, p.count, p.region, p.pbits, dir_bits, gshift, rec, n_rec, dir,
      n_rec < 1u << 20 ? 1u : 16u, reinterpret_cast<unsigned long long*>(n_groups), err);
  prof_end(s);
}

}  // namespace xtn
