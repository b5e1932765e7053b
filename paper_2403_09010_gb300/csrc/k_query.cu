// Query-vs-reference lookup against a resident, sorted variant index: the
// SymDel step "reuse x to look up the hash map" (Appendix A, SymDel steps 2-3)
// with the hash map realised as the sorted record array of Sec. 2.2.
//
//   k_build_dir    : dir[t] = first index record whose top `dir_bits`
//                    fingerprint bits are >= t, so a lookup starts from a
//                    range of ~n_rec / 2^dir_bits records (a few, with the
//                    directory sized at about one entry per 4 records)
//                    instead of all.
//   k_query_candidates : the queries' variants (expand.cuh), a lane each: the
//                    variant's directory range is read and compared, and the
//                    references of equal fingerprint go out at once as
//                    candidate words (q << ref_bits) | r, collected per warp.
//                    Bound by the memory system's rate of random requests
//                    (about 30 G lines/s for reads of this kind, whatever
//                    their locality): a lookup is one line of the directory
//                    and 1.3 of the records, so 1.1 M of them (10,000 queries,
//                    d = 2, a 10M index) take 85 us alone, 120 here.  Lookup,
//                    count scan and emission as kernels of their own took
//                    128 + 19 + 16 us, through 20 bytes written and read a
//                    variant; 40 queries 17 + 8 + 11 us instead of 10.
//   k_query_spread : groups too large for one lane, a warp per 1,024 records.
#include <algorithm>

#include "expand.cuh"
#include "per_device.h"
#include "xtn_common.cuh"
#include "xtn_kernels.h"

namespace xtn {

// One thread per sorted position p in [0, n_rec]: the directory entries t
// in (top(rec[p-1]), top(rec[p])] all start at p (top(rec[-1]) = -1,
// top(rec[n_rec]) = 2^dir_bits), so every entry is written exactly once in
// one coalesced pass over the records.
// The same pass counts the groups (positions whose group key, the bits from
// gshift up, differs from the previous record's) into *n_groups.
__global__ void k_build_dir(const uint64_t* __restrict__ rec, uint64_t n_rec, int dir_bits,
                            int gshift, uint32_t* __restrict__ dir,
                            unsigned long long* __restrict__ n_groups) {
  const int64_t n_dir = 1ll << dir_bits;
  uint32_t heads = 0;
  for (uint64_t p = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; p <= n_rec;
       p += (uint64_t)gridDim.x * blockDim.x) {
    const int64_t prev = p == 0 ? -1 : (int64_t)(rec[p - 1] >> (64 - dir_bits));
    const int64_t cur = p == n_rec ? n_dir : (int64_t)(rec[p] >> (64 - dir_bits));
    for (int64_t t = prev + 1; t <= cur && t <= n_dir; ++t) dir[t] = (uint32_t)p;
    if (p < n_rec && (p == 0 || (rec[p] >> gshift) != (rec[p - 1] >> gshift))) ++heads;
  }
  heads = (uint32_t)__reduce_add_sync(FULL_MASK, heads);
  if (lane_id() == 0 && heads) atomicAdd(n_groups, (unsigned long long)heads);
}

void launch_build_dir(const uint64_t* rec, uint64_t n_rec, int dir_bits, int gshift,
                      uint32_t* dir, uint64_t* n_groups, cudaStream_t s) {
  const uint64_t n_dir = (1ull << dir_bits) + 1;
  prof_begin(s, "k_build_dir", (double)n_rec * 8.0 + (double)n_dir * 4.0);
  const uint32_t blocks = (uint32_t)std::min<uint64_t>((n_rec + 256) / 256, 152ull * 32);
  k_build_dir<<<blocks, 256, 0, s>>>(rec, n_rec, dir_bits, gshift, dir,
                                     reinterpret_cast<unsigned long long*>(n_groups));
  prof_end(s);
}

constexpr int QC_THREADS = 256;
constexpr int QC_WARPS = QC_THREADS / 32;
constexpr int QC_BLOCKS = 4;           // of an SM
constexpr uint32_t QC_FLUSH = 96;      // words a warp collects before a flush
constexpr uint32_t QC_DIRECT = 256;    // records of a group a warp emits by itself
constexpr uint32_t QC_CHUNK = 1024;    // and of larger ones, per entry of the list

template <int KIND>
struct QuerySmem {
  using K = VK<KIND>;
  uint64_t terms[QC_WARPS][K::PACK][K::STRIDE];
  uint64_t stash[QC_WARPS][QC_FLUSH + 32];
  uint64_t pow[N_POWERS<KIND>];
  VarMeta meta[QC_WARPS][K::PACK];
  uint16_t extra[QC_WARPS][K::PACK][K::EXTRA + 1];
  uint16_t comb[K::COMBS + 1];
};

// Group of key g in the index: number of its records, the first at `at`; the
// records are at + (the set bits of `mask`), or in a row where it is 0.
__device__ __forceinline__ uint32_t index_group(const uint64_t* __restrict__ rec, uint64_t n_rec,
                                                const uint32_t* __restrict__ dir, uint64_t top,
                                                int gshift, uint64_t g, uint32_t* err,
                                                uint32_t& at, uint32_t& mask) {
  uint64_t lo = __ldg(dir + top), hi = __ldg(dir + top + 1);
  if (hi > n_rec || lo > hi) {
    atomicOr(err, DERR_RANGE);
    return 0u;
  }
  if (hi - lo > (uint64_t)INDEX_SCAN) {
    uint64_t e = hi;  // lower bound
    while (lo < e) {
      const uint64_t mid = (lo + e) >> 1;
      if ((__ldg(rec + mid) >> gshift) < g) lo = mid + 1; else e = mid;
    }
    uint64_t c = lo;  // upper bound
    e = hi;
    while (c < e) {
      const uint64_t mid = (c + e) >> 1;
      if ((__ldg(rec + mid) >> gshift) <= g) c = mid + 1; else e = mid;
    }
    at = (uint32_t)lo;
    return (uint32_t)(c - lo);
  }
  for (uint64_t p = lo; p < hi; p += 4) {  // four at a time: one round trip, not four
    uint64_t r[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) r[k] = p + k < hi ? __ldg(rec + p + k) >> gshift : 0ull;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (p + k < hi && r[k] == g) mask |= 1u << (uint32_t)(p + k - lo);  // hi - lo <= 32
  }
  at = (uint32_t)lo;
  return (uint32_t)__popc(mask);
}

// A warp takes `pack` consecutive queries (or a share of them, `parts` warps
// the same ones): few queries would otherwise leave most of the chip idle
// and give a lane many lookups in turn.
template <int KIND>
__global__ void __launch_bounds__(QC_THREADS, QC_BLOCKS)
    k_query_candidates(ExpandSource src, int64_t n_q, int d, const uint64_t* __restrict__ rec,
                       uint64_t n_rec, const uint32_t* __restrict__ dir, int dir_bits, int gshift,
                       uint32_t ref_bits, int pack, int parts, uint64_t* __restrict__ cand,
                       uint64_t cand_cap, unsigned long long* __restrict__ n_cand,
                       QueryChunk* __restrict__ list, uint64_t list_cap,
                       unsigned long long* __restrict__ n_list,
                       unsigned long long* __restrict__ n_variants, uint32_t* __restrict__ err) {
  using K = VK<KIND>;
  extern __shared__ __align__(16) unsigned char query_smem[];
  QuerySmem<KIND>& S = *reinterpret_cast<QuerySmem<KIND>*>(query_smem);
  load_powers<KIND>(S.pow);
  load_combs<KIND>(S.comb);
  __syncthreads();
  const uint32_t warp = threadIdx.x >> 5, lane = lane_id();
  const uint64_t idmask = (1ull << ref_bits) - 1ull;
  uint64_t* stash = S.stash[warp];
  uint32_t held = 0;  // words in the stash, the same in every lane
  auto flush = [&] {
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(n_cand, (unsigned long long)held);
    base = __shfl_sync(FULL_MASK, base, 0);
    __syncwarp();  // every lane's words are visible
    for (uint32_t k = lane; k < held; k += 32)
      if (base + k < cand_cap) cand[base + k] = stash[k];  // past it: counted, the caller reruns
    __syncwarp();
    held = 0;
  };
  const int q = (int)lane / K::LANES;
  VarMeta* meta = S.meta[warp];
  uint64_t variants = 0;
  const int64_t units = (n_q + pack - 1) / pack * parts;
  const int64_t n_warps = (int64_t)gridDim.x * QC_WARPS;
  for (int64_t u = (int64_t)blockIdx.x * QC_WARPS + warp; u < units; u += n_warps) {
    const int64_t s0 = u / parts * pack;
    const uint32_t part = (uint32_t)(u % parts);
    const int64_t my = s0 + q;
    const bool have = q < pack && my < n_q;
    VarMeta m;
    uint64_t* terms = S.terms[warp][q];
    const uint32_t total =
        prepare_variants<KIND>(terms, S.extra[warp][q], S.pow, src, my, have, d, 0ull, lane, m,
                               [&](uint32_t a, uint64_t h) { terms[a] = h; });
    uint32_t end = total;
#pragma unroll
    for (int o = K::LANES; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(FULL_MASK, end, o);
      if (lane >= (uint32_t)o) end += t;
    }
    const uint32_t T = __shfl_sync(FULL_MASK, end, 31);
    if (part == 0) variants += T;
    if (lane % K::LANES == 0) {
      m.end = (int32_t)end;
      m.adj += (int32_t)(end - total);
      meta[q] = m;
    }
    __syncwarp();  // terms and meta, written above, are read by every lane
    const VarMeta* at = meta;
    VarMeta cur = meta[0];
    uint32_t id = (uint32_t)s0;
    const uint64_t* tab = S.terms[warp][0];
    const uint16_t* extra = S.extra[warp][0];
    for (uint32_t t0 = part * 32; t0 < T; t0 += 32u * (uint32_t)parts) {
      const uint32_t t = t0 + lane;
      uint32_t first = 0, count = 0, mask = 0;
      if (t < T) {
        while ((int32_t)t >= cur.end) {  // ends: t < T, the last query's end
          cur = *++at;
          ++id;
          tab += K::STRIDE;
          extra += K::EXTRA + 1;
        }
        const uint64_t h = mix64(variant_sum<KIND>(
            tab, extra, S.comb, (uint32_t)((int32_t)t - cur.adj), cur.c, cur.aux));
        count = index_group(rec, n_rec, dir, h >> (64 - dir_bits), gshift, h >> gshift, err,
                            first, mask);
        if (count > QC_DIRECT) {
          const uint32_t chunks = (count + QC_CHUNK - 1) / QC_CHUNK;
          const uint64_t base = atomicAdd(n_cand, (unsigned long long)count);
          const uint64_t slot = atomicAdd(n_list, (unsigned long long)chunks);
          for (uint32_t k = 0; k < chunks; ++k) {
            const uint32_t o = k * QC_CHUNK;
            if (slot + k < list_cap)
              list[slot + k] = QueryChunk{base + o, first + o, min(QC_CHUNK, count - o), id, 0u};
          }
          count = 0;
        }
      }
      // the round's records, 32 at a time whosever they are: a lane finds the
      // lane that a record belongs to among the counts' prefix sums
      uint32_t ends = count;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(FULL_MASK, ends, o);
        if (lane >= (uint32_t)o) ends += x;
      }
      const uint32_t words = __shfl_sync(FULL_MASK, ends, 31);
      for (uint32_t k0 = 0; k0 < words; k0 += 32) {
        const uint32_t k = k0 + lane;
        int owner = 0;  // lanes whose words all come before k
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
          if (__shfl_sync(FULL_MASK, ends, owner + o - 1) <= k) owner += o;
        owner = min(owner, 31);
        const uint32_t nth = k - __shfl_sync(FULL_MASK, ends - count, owner);
        uint32_t bits = __shfl_sync(FULL_MASK, mask, owner);
        uint32_t p = __shfl_sync(FULL_MASK, first, owner);
        if (bits == 0) {
          p += nth;
        } else if (k < words) {
          for (uint32_t x = 0; x < nth; ++x) bits &= bits - 1u;
          p += (uint32_t)__ffs((int)bits) - 1u;
        }
        const uint32_t whose = __shfl_sync(FULL_MASK, id, owner);
        if (k < words)
          stash[held + lane] = ((uint64_t)whose << ref_bits) | (__ldg(rec + p) & idmask);
        held += min(32u, words - k0);
        if (held >= QC_FLUSH) flush();  // at most QC_FLUSH + 31 words
      }
    }
    __syncwarp();  // the next queries reuse terms and meta
  }
  if (held) flush();
  if (lane == 0 && variants) atomicAdd(n_variants, (unsigned long long)variants);
}

template <int KIND>
static void query_launch(const ExpandSource& src, int64_t n_q, int d, const uint64_t* rec,
                         uint64_t n_rec, const uint32_t* dir, int dir_bits, int gshift,
                         uint32_t ref_bits, uint64_t* cand, uint64_t cand_cap, uint64_t* n_cand,
                         QueryChunk* list, uint64_t list_cap, uint64_t* n_list,
                         uint64_t* n_variants, int sms, uint32_t* err, cudaStream_t s) {
  using ull = unsigned long long;
  auto f = k_query_candidates<KIND>;
  static PerDevice shared;
  shared([&] { return allow_shared((const void*)f, (int)sizeof(QuerySmem<KIND>), false); });
  // `pack` as large as leaves a resident warp four units of work: one query a
  // unit for 10,000 (132 us with two), 30,000 of a 36M-record index 125 us
  // against 147 with six
  const int64_t warps = (int64_t)sms * QC_BLOCKS * QC_WARPS;  // resident at once
  const int pack =
      (int)std::min<int64_t>(VK<KIND>::PACK, std::max<int64_t>(1, n_q / (4 * warps)));
  const int64_t groups = (n_q + pack - 1) / pack;
  const int parts = (int)std::min<int64_t>(8, std::max<int64_t>(1, warps / groups));
  const uint32_t blocks =
      (uint32_t)std::min<int64_t>((groups * parts + QC_WARPS - 1) / QC_WARPS, sms * QC_BLOCKS);
  f<<<blocks, QC_THREADS, sizeof(QuerySmem<KIND>), s>>>(
      src, n_q, d, rec, n_rec, dir, dir_bits, gshift, ref_bits, pack, parts, cand, cand_cap,
      reinterpret_cast<ull*>(n_cand), list, list_cap, reinterpret_cast<ull*>(n_list),
      reinterpret_cast<ull*>(n_variants), err);
}

void launch_query_candidates(const ExpandSource& src, int64_t n_q, int d, const uint64_t* rec,
                             uint64_t n_rec, const uint32_t* dir, int dir_bits, int gshift,
                             uint32_t ref_bits, uint64_t* cand, uint64_t cand_cap,
                             uint64_t* n_cand, QueryChunk* list, uint64_t list_cap,
                             uint64_t* n_list, uint64_t* n_variants, int sms, uint32_t* err,
                             cudaStream_t s) {
  if (n_q <= 0) return;
  prof_begin(s, "k_query_candidates", (double)n_q * 32.0);
  auto f = d <= 1 ? query_launch<VK_D1> : d == 2 ? query_launch<VK_D2> : query_launch<VK_D3>;
  f(src, n_q, d, rec, n_rec, dir, dir_bits, gshift, ref_bits, cand, cand_cap, n_cand, list,
    list_cap, n_list, n_variants, sms, err, s);
  prof_end(s);
}

__global__ void __launch_bounds__(256)
    k_query_spread(const uint64_t* __restrict__ rec, uint64_t n_rec, uint32_t ref_bits,
                   const QueryChunk* __restrict__ list, uint64_t n_list,
                   uint64_t* __restrict__ cand, uint64_t cand_cap, uint32_t* __restrict__ err) {
  const uint64_t idmask = (1ull << ref_bits) - 1ull;
  const uint64_t stride = (uint64_t)gridDim.x * 8;
  for (uint64_t e = (uint64_t)blockIdx.x * 8 + (threadIdx.x >> 5); e < n_list; e += stride) {
    const QueryChunk c = list[e];
    if ((uint64_t)c.first + c.count > n_rec || c.base + c.count > cand_cap) {
      if (lane_id() == 0) atomicOr(err, DERR_RANGE);
      continue;
    }
    for (uint32_t k = lane_id(); k < c.count; k += 32)
      cand[c.base + k] = ((uint64_t)c.q << ref_bits) | (rec[c.first + k] & idmask);
  }
}

void launch_query_spread(const uint64_t* rec, uint64_t n_rec, uint32_t ref_bits,
                         const QueryChunk* list, uint64_t n_list, uint64_t* cand,
                         uint64_t cand_cap, int sms, uint32_t* err, cudaStream_t s) {
  if (n_list == 0) return;
  const int blocks = (int)std::min<uint64_t>((n_list + 7) / 8, (uint64_t)sms * 8);
  prof_begin(s, "k_query_spread", (double)n_list * QC_CHUNK * 16.0);
  k_query_spread<<<blocks, 256, 0, s>>>(rec, n_rec, ref_bits, list, n_list, cand, cand_cap, err);
  prof_end(s);
}

}  // namespace xtn
