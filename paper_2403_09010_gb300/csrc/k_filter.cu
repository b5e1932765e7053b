// Grouping of variant records by their full group key, with the candidate
// pairs written at once (Appendix A, XTNeighbor steps 4-5), one fingerprint
// partition (k_partition.cu) at a time.
//
// Nearly every variant record shares its group key with no other record
// (about 95% of the 1M workload's records are alone), so the exact grouping
// only needs the few that do.
//   k_bucket_filter : one block per partition
//     1. marks the top SEEN key bits below the partition's in one bitmap
//        and, where a record met a set bit there, the top AGAIN of them in
//        another;
//     2. reads its partition again (from L2) and lists the records marked in
//        the second bitmap -- all members of groups of two or more, plus the
//        few lone records that another key's bits kept.
//     The bitmaps hold about 20 bits per record in the block's shared
//     memory, so one block covers tens of thousands of records and a second
//     partitioning pass is only needed past 655 M of them.
//   k_group_kept    : one block per list chains its records by a hash of
//     their key and lets each one walk the rest of its chain, writing a
//     candidate word (min id << id_bits | max id) for every record there with
//     the same key.  A longer list is taken in parts of its key space.
// The grouping is latency-bound (dependent shared-memory operations between
// barriers) while the filter streams, so each has blocks of its own size;
// in one kernel the long phases of few large blocks could not overlap.  The
// key compared is every fingerprint bit the record holds above its id, so
// unequal variants hardly ever make a candidate.
#include <algorithm>

#include "per_device.h"
#include "xtn_common.cuh"
#include "xtn_kernels.h"

namespace xtn {

namespace {

template <int SEEN, int AGAIN>
struct FilterSmem {
  uint32_t seen[(1 << SEEN) / 32];
  uint32_t again[(1 << AGAIN) / 32];
  uint32_t n_kept;
  unsigned long long base;
};

// LOW: the bits reach below the high word (shift < 32).
template <int THREADS, int SEEN, int AGAIN, int MIN_BLOCKS, bool LOW>
__global__ void __launch_bounds__(THREADS, MIN_BLOCKS)
    k_bucket_filter(const uint64_t* __restrict__ rec, const uint32_t* __restrict__ count,
                    uint32_t region, int shift, uint64_t* __restrict__ kept,
                    uint32_t* __restrict__ kept_count, uint64_t* __restrict__ spill, uint64_t spill_cap,
                    unsigned long long* __restrict__ n_spill, uint32_t* __restrict__ err) {
  using SM = FilterSmem<SEEN, AGAIN>;
  constexpr int U = 4;  // record pairs a thread holds of one chunk
  constexpr uint32_t CHUNK = U * THREADS;
  extern __shared__ __align__(16) unsigned char bf_smem[];
  SM& S = *reinterpret_cast<SM*>(bf_smem);
  const uint32_t m = count[blockIdx.x];
  const uint64_t* __restrict__ in = rec + (uint64_t)blockIdx.x * region;
  if (m < 2) return;  // its list count is zero
  if (m > region) {   // overflowed: all of it to the global grouping
    if (threadIdx.x == 0) S.base = atomicAdd(n_spill, (unsigned long long)region);
    __syncthreads();
    for (uint32_t k = threadIdx.x; k < region; k += THREADS) {
      if (S.base + k < spill_cap) spill[S.base + k] = in[k];
      else atomicOr(err, DERR_RANGE);
    }
    return;
  }
  for (int k = threadIdx.x; k < ((1 << SEEN) + (1 << AGAIN)) / 128; k += THREADS)
    reinterpret_cast<uint4*>(S.seen)[k] = make_uint4(0u, 0u, 0u, 0u);
  if (threadIdx.x == 0) S.n_kept = 0;
  __syncthreads();
  // Bit h of `seen`: the SEEN record bits below the partition's, from `shift`
  // up (id bits are left out: then fewer, above them)
  constexpr uint32_t HMASK = (1u << SEEN) - 1u;
  constexpr int DROP = SEEN - AGAIN;  // `again` tells the bits above the lowest DROP apart
  // The records two by two (regions start on 16-byte boundaries), in chunks
  // of U pairs a thread; the next chunk's loads are under way while one is
  // worked on.  Pair i of the partition holds records 2i and 2i + 1.
  const uint32_t pairs = (m + 1) / 2;
  const ulonglong2* __restrict__ in2 = reinterpret_cast<const ulonglong2*>(in) + threadIdx.x;
  ulonglong2 v[U], next[U];
  auto load = [&](ulonglong2* x, uint32_t i0) {
    if (i0 + CHUNK <= pairs) {
#pragma unroll
      for (int u = 0; u < U; ++u) x[u] = in2[i0 + u * THREADS];
    } else {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        x[u] = make_ulonglong2(0ull, 0ull);
        if (i0 + u * THREADS + threadIdx.x < pairs) x[u] = in2[i0 + u * THREADS];
      }
    }
  };
  auto rec_of = [&](int u) { return u & 1 ? v[u / 2].y : v[u / 2].x; };
  auto bits_of = [&](int u) {
    const uint64_t r = rec_of(u);
    return LOW ? __funnelshift_r((uint32_t)r, (uint32_t)(r >> 32), shift)
               : (uint32_t)(r >> 32) >> (shift - 32);
  };
  // the records of this thread's chunk at i0 that exist, a bit each
  auto there = [&](uint32_t i0) {
    uint32_t mask = (1u << (2 * U)) - 1u;
    if (2 * (i0 + CHUNK) > m) {
#pragma unroll
      for (int u = 0; u < 2 * U; ++u)
        if (2 * (i0 + (u / 2) * THREADS + threadIdx.x) + (u & 1) >= m) mask &= ~(1u << u);
    }
    return mask;
  };
  // 1. mark: all of a chunk's bits are set before the first answer is used
  load(v, 0);
  for (uint32_t i0 = 0; i0 < pairs; i0 += CHUNK) {
    load(next, i0 + CHUNK < pairs ? i0 + CHUNK : 0u);  // after the last, the first again
    const uint32_t mask = there(i0);
    uint32_t old[2 * U];
#pragma unroll
    for (int u = 0; u < 2 * U; ++u) {
      const uint32_t h = bits_of(u);
      old[u] = 0;
      if (mask >> u & 1u)
        old[u] = atomicOr(&S.seen[(h & HMASK) >> 5], 1u << (h & 31u)) >> (h & 31u);
    }
#pragma unroll
    for (int u = 0; u < 2 * U; ++u) {
      const uint32_t h = bits_of(u);
      if (old[u] & 1u) atomicOr(&S.again[(h & HMASK) >> (5 + DROP)], 1u << ((h >> DROP) & 31u));
    }
#pragma unroll
    for (int u = 0; u < U; ++u) v[u] = next[u];
  }
  __syncthreads();
  // 2. the kept records to the partition's list
  uint64_t* __restrict__ out = kept + (uint64_t)blockIdx.x * region;
  const uint32_t lane = lane_id();
  for (uint32_t i0 = 0; i0 < pairs; i0 += CHUNK) {
    load(next, i0 + CHUNK);
    uint32_t mask = 0;
#pragma unroll
    for (int u = 0; u < 2 * U; ++u) {
      const uint32_t h = bits_of(u);
      mask |= ((S.again[(h & HMASK) >> (5 + DROP)] >> ((h >> DROP) & 31u)) & 1u) << u;
    }
    mask &= there(i0);
    const uint32_t c = (uint32_t)__popc(mask);
    uint32_t at = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(FULL_MASK, at, o);
      if (lane >= (uint32_t)o) at += t;
    }
    uint32_t base = 0;
    if (lane == 31) base = atomicAdd(&S.n_kept, at);
    at += __shfl_sync(FULL_MASK, base, 31) - c;  // < region: the list holds a whole partition
#pragma unroll
    for (int u = 0; u < 2 * U; ++u)
      if (mask >> u & 1u) out[at++] = rec_of(u);
#pragma unroll
    for (int u = 0; u < U; ++u) v[u] = next[u];
  }
  __syncthreads();
  if (threadIdx.x == 0) kept_count[blockIdx.x] = S.n_kept;
}

constexpr int GK_THREADS = 512;
constexpr int GK_WARPS = GK_THREADS / 32;
constexpr int GK_LIST = 6144;       // records a block groups at once
constexpr uint32_t GK_FILL = 5632;  // records a part is sized for
constexpr int GK_HBITS = 12;        // log2 of the slots, at most
constexpr uint32_t GK_STASH = 256;  // candidate words a warp collects
constexpr int GK_LOADS = 8;         // loads a thread has under way
constexpr uint32_t GK_NIL = 0xffffu;
static_assert(GK_LIST < (int)GK_NIL, "16-bit links");

struct GroupSmem {
  uint32_t head[1 << GK_HBITS];  // first record of the slot's chain
  uint64_t list[GK_LIST];
  uint64_t stash[GK_WARPS][GK_STASH];
  uint16_t next[GK_LIST];
  uint32_t n_list;
  bool full;  // a warp has found the candidates past their buffer
};

// skip: key bits that all records of a list share (the partition's).
// count_all: the candidates are counted to the end, past cand_cap too; else a
// warp whose words no longer fit stops and its block leaves, as the caller
// starts over (100,000 sequences ten times each, d = 2: 472 M candidates of
// which 52 M fit, 1.0 ms instead of 14.6; 160,000 of six residues, d = 1, where
// every block is resident at once, 0.05 instead of 0.55).  The exit costs the
// kernel 170 instead of 164 us for 1M sequences, d = 2.
__global__ void __launch_bounds__(GK_THREADS, 2)
    k_group_kept(const uint64_t* __restrict__ kept, const uint32_t* __restrict__ kept_count,
                 uint32_t region, int skip, uint64_t* __restrict__ spill, uint64_t spill_cap,
                 unsigned long long* __restrict__ n_spill, uint64_t* __restrict__ cand,
                 uint64_t cand_cap, unsigned long long* __restrict__ cand_count, bool count_all,
                 int id_bits, uint32_t* __restrict__ err) {
  constexpr int THREADS = GK_THREADS;
  extern __shared__ __align__(16) unsigned char gk_smem[];
  GroupSmem& S = *reinterpret_cast<GroupSmem*>(gk_smem);
  const uint32_t lane = lane_id();
  const uint64_t idmask = (1ull << id_bits) - 1ull;
  if (threadIdx.x == 0) S.full = false;
  const uint32_t m = kept_count[blockIdx.x];
  if (m < 2) return;
  const uint64_t* __restrict__ in = kept + (uint64_t)blockIdx.x * region;
  int pb = 0;  // log2 of the parts
  while (pb < 16 && ((uint64_t)GK_FILL << pb) < m) ++pb;
  int hb = 9;  // slots: twice the records of a part
  while (hb < GK_HBITS && (1u << hb) < 2 * (m >> pb)) ++hb;
  // candidate words collect per warp: one reservation per flush
  uint64_t* stash = S.stash[threadIdx.x >> 5];
  uint32_t held = 0;
  auto flush = [&]() -> bool {  // false: none of the words fitted, and need not be counted
    __syncwarp();  // every lane's words are visible
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(cand_count, (unsigned long long)held);
    base = __shfl_sync(FULL_MASK, base, 0);
    for (uint32_t k = lane; k < held; k += 32) {
      if (base + k < cand_cap) cand[base + k] = stash[k];
      else atomicOr(err, DERR_CAPACITY);
    }
    __syncwarp();  // the stash is refilled next
    held = 0;
    return count_all || base < cand_cap;
  };
  for (uint32_t part = 0; part < (1u << pb); ++part) {
    // the part by the key bits below the shared ones
    auto in_part = [&](uint64_t r) { return r << skip >> 1 >> (63 - pb) == part; };
    for (int k = threadIdx.x; k < (1 << hb) / 4; k += THREADS)
      reinterpret_cast<uint4*>(S.head)[k] = make_uint4(GK_NIL, GK_NIL, GK_NIL, GK_NIL);
    if (threadIdx.x == 0) S.n_list = 0;
    __syncthreads();
    // 1. list the part's records, each put at the head of its slot's chain
    for (uint32_t k0 = 0; k0 < m; k0 += GK_LOADS * THREADS) {
      uint64_t r[GK_LOADS];
      uint32_t mask = 0;
#pragma unroll
      for (int u = 0; u < GK_LOADS; ++u) {
        const uint32_t k = k0 + u * THREADS + threadIdx.x;
        r[u] = 0;
        if (k < m) {
          r[u] = in[k];
          mask |= 1u << u;
        }
      }
      uint32_t at[GK_LOADS];
      if (pb == 0) {  // the whole list, in place
#pragma unroll
        for (int u = 0; u < GK_LOADS; ++u) at[u] = k0 + u * THREADS + threadIdx.x;
        if (threadIdx.x == 0) S.n_list = m;
      } else {
#pragma unroll
        for (int u = 0; u < GK_LOADS; ++u)
          if (!in_part(r[u])) mask &= ~(1u << u);
        const uint32_t c = (uint32_t)__popc(mask);
        uint32_t a = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t t = __shfl_up_sync(FULL_MASK, a, o);
          if (lane >= (uint32_t)o) a += t;
        }
        uint32_t base = 0;
        if (lane == 31) base = atomicAdd(&S.n_list, a);
        a += __shfl_sync(FULL_MASK, base, 31) - c;
#pragma unroll
        for (int u = 0; u < GK_LOADS; ++u) at[u] = a + (uint32_t)__popc(mask & ((1u << u) - 1u));
      }
#pragma unroll
      for (int u = 0; u < GK_LOADS; ++u) {
        if ((mask >> u & 1u) && at[u] < (uint32_t)GK_LIST) {
          S.list[at[u]] = r[u];
          const uint32_t h = (uint32_t)((r[u] >> id_bits) * 0x9E3779B97F4A7C15ull >> (64 - hb));
          S.next[at[u]] = (uint16_t)atomicExch(&S.head[h], at[u]);
        }
      }
    }
    __syncthreads();
    const uint32_t n = S.n_list;
    if (n > (uint32_t)GK_LIST) {  // a key repeated very often: to the global grouping
      for (uint32_t k = threadIdx.x; k < m; k += THREADS) {
        const uint64_t r = in[k];
        if (in_part(r)) {
          const uint64_t at = atomicAdd(n_spill, 1ull);
          if (at < spill_cap) spill[at] = r;
          else atomicOr(err, DERR_RANGE);
        }
      }
      __syncthreads();
      continue;
    }
    // 2. every record pairs with those behind it in its chain that share its
    // key (step by step, the warp's lanes together)
    for (uint32_t j0 = threadIdx.x & ~31u; j0 < n; j0 += THREADS) {
      const uint32_t j = j0 + lane;
      uint64_t r = 0;
      uint32_t k = GK_NIL;
      if (j < n) {
        r = S.list[j];
        k = S.next[j];
      }
      while (__any_sync(FULL_MASK, k != GK_NIL)) {  // ends: a chain has no loops
        uint64_t w = 0;
        bool same = false;
        if (k != GK_NIL) {
          const uint64_t q = S.list[k];
          same = ((r ^ q) & ~idmask) == 0;
          const uint64_t a = r & idmask, b = q & idmask;
          w = ((a < b ? a : b) << id_bits) | (a < b ? b : a);
          k = S.next[k];
        }
        const uint32_t bal = __ballot_sync(FULL_MASK, same);
        if (bal) {
          if (same) stash[held + __popc(bal & ((1u << lane) - 1u))] = w;
          held += (uint32_t)__popc(bal);
          if (held > GK_STASH - 32 && !flush()) {  // this warp is done
            if (lane == 0) S.full = true;
            goto part_done;
          }
        }
      }
    }
  part_done:
    __syncthreads();  // the next part reuses the tables
    if (S.full) return;
  }
  if (held) flush();
}

template <int THREADS, int SEEN, int AGAIN, int MIN_BLOCKS, bool LOW>
void filter_launch(const Partitions& p, int shift, uint32_t* err, cudaStream_t s) {
  using SM = FilterSmem<SEEN, AGAIN>;
  auto f = k_bucket_filter<THREADS, SEEN, AGAIN, MIN_BLOCKS, LOW>;
  static PerDevice shared;
  shared([&] { return allow_shared((const void*)f, (int)sizeof(SM)); });
  f<<<1u << p.pbits, THREADS, sizeof(SM), s>>>(
      p.rec, p.count, p.region, shift, p.kept, p.kept_count(), p.spill, p.spill_cap,
      reinterpret_cast<unsigned long long*>(p.n_spill), err);
}

template <int THREADS, int SEEN, int AGAIN, int MIN_BLOCKS>
void filter_launch(const Partitions& p, int id_bits, uint32_t* err, cudaStream_t s) {
  const int shift = std::max(64 - p.pbits - SEEN, id_bits);
  if (shift < 32) filter_launch<THREADS, SEEN, AGAIN, MIN_BLOCKS, true>(p, shift, err, s);
  else filter_launch<THREADS, SEEN, AGAIN, MIN_BLOCKS, false>(p, shift, err, s);
}

}  // namespace

void launch_group_filter(const Partitions& q, uint64_t n_rec, uint64_t* cand, uint64_t cand_cap,
                         uint64_t* cand_count, bool count_all, int id_bits, int sms,
                         uint32_t* err, cudaStream_t s) {
  if (q.sub) launch_split(q, n_rec, sms, err, s);
  const Partitions p = q.sub ? q.fine() : q;
  // the bitmaps hold about 20 bits per record of the expected partition
  const uint64_t mean = n_rec >> p.pbits;
  prof_begin(s, "k_bucket_filter", (double)n_rec * 8.0);
  if (mean <= 6500) filter_launch<256, 17, 15, 4>(p, id_bits, err, s);
  else if (mean <= 26500) filter_launch<512, 19, 17, 2>(p, id_bits, err, s);
  else filter_launch<1024, 20, 18, 1>(p, id_bits, err, s);
  prof_end(s);
  static PerDevice shared;
  shared([] { return allow_shared((const void*)k_group_kept, (int)sizeof(GroupSmem)); });
  prof_begin(s, "k_group_kept", 0.0);
  k_group_kept<<<1u << p.pbits, GK_THREADS, sizeof(GroupSmem), s>>>(
      p.kept, p.kept_count(), p.region, p.pbits, p.spill, p.spill_cap,
      reinterpret_cast<unsigned long long*>(p.n_spill), cand, cand_cap,
      reinterpret_cast<unsigned long long*>(cand_count), count_all, id_bits, err);
  prof_end(s);
}

}  // namespace xtn
