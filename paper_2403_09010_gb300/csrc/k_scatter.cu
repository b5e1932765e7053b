// Expansion straight into fingerprint partitions (Appendix A, XTNeighbor
// steps 2-4: the expansion and the coarse half of the grouping in one pass).
//
// A block works in steps.  In each, every warp generates up to 32 * ITEMS
// consecutive records of its share into registers, counting them into
// shared-memory bins; the bins are scanned and room is reserved in every
// partition at once; the records are placed in shared memory in partition
// order over the dead terms; and leave in runs of one partition each
// (k_partition.cu describes the partitions and what the runs cost).  Against
// an expansion in sequence order and a pass over its records this saves
// writing and reading them once (16 of 24 bytes per record).
#include <algorithm>
#include <type_traits>

#include "expand.cuh"
#include "partition.cuh"
#include "per_device.h"
#include "xtn_common.cuh"
#include "xtn_kernels.h"

namespace xtn {

namespace {

// One block per SM, as many records as its registers hold.  With at most one
// deletion a record needs no terms in shared memory and fewer registers, and
// the records of two batches of sequences fill a warp's slots.
template <int KIND>
struct SC {
  static constexpr int THREADS = VK<KIND>::D == 1 ? 640 : 768;
  static constexpr int WARPS = THREADS / 32;
  static constexpr int ITEMS = VK<KIND>::D == 1 ? 32 : 22;
  static constexpr int BATCH = ITEMS / 2;
  static constexpr int SLOTS = 32 * ITEMS;     // records of a warp in one step
  static constexpr int TILE = WARPS * SLOTS;   // of a block
};

template <int KIND>
struct ScatterTerms {
  using K = VK<KIND>;
  uint64_t terms[SC<KIND>::WARPS][K::PACK][K::STRIDE];
  VarMeta meta[SC<KIND>::WARPS][K::PACK];
  uint16_t extra[SC<KIND>::WARPS][K::PACK][K::EXTRA + 1];
};

template <int KIND>
struct ScatterSmem {
  using K = VK<KIND>;
  union {
    typename std::conditional<K::D == 1, uint64_t, ScatterTerms<KIND>>::type t;
    uint64_t stage[SC<KIND>::TILE];
  };
  uint64_t pow[N_POWERS<KIND>];
  uint32_t wsum[8];
  uint32_t held;    // records of the step
  uint32_t pshift;  // 32 - pbits
  uint32_t over;  // a partition's region has run over
  uint16_t comb[K::COMBS + 1];
  // then, 16-byte aligned: the bins' counters and output offsets, 2^pbits each
};

template <int KIND>
constexpr size_t scatter_smem_bytes(int pbits) {
  return ((sizeof(ScatterSmem<KIND>) + 15) & ~(size_t)15) + ((size_t)8 << pbits);
}

// Sequence holding record r: the largest s with rec_off[s] <= r (whole warp).
__device__ __forceinline__ int64_t sequence_of(const uint64_t* __restrict__ rec_off, int64_t n,
                                               uint64_t r, uint32_t lane) {
  int64_t lo = 0, hi = n;  // rec_off[lo] <= r
  while (hi - lo > 1) {
    const int64_t step = (hi - lo + 31) / 32;
    const int64_t at = lo + (int64_t)lane * step;
    const uint32_t b = __ballot_sync(FULL_MASK, at < hi && (lane == 0 || rec_off[at] <= r));
    const int last = 31 - __clz((int)b);  // lane 0 always holds
    lo += last * step;
    hi = min(hi, lo + step);
  }
  return lo;
}

template <int KIND>
__global__ void __launch_bounds__(SC<KIND>::THREADS, 1)
    k_expand_scatter(ExpandSource src, const uint64_t* __restrict__ rec_off, int64_t n, int d,
                     const uint32_t* __restrict__ seq_rep, uint32_t id_bits, uint64_t n_cap,
                     int pbits, uint64_t* __restrict__ out, uint32_t region,
                     uint32_t* __restrict__ part_count, uint64_t* __restrict__ spill,
                     uint64_t spill_cap, unsigned long long* __restrict__ n_spill,
                     uint32_t* __restrict__ err) {
  using K = VK<KIND>;
  using C = SC<KIND>;
  extern __shared__ __align__(16) unsigned char scatter_smem[];
  ScatterSmem<KIND>& S = *reinterpret_cast<ScatterSmem<KIND>*>(scatter_smem);
  uint32_t* s_cnt =
      reinterpret_cast<uint32_t*>(scatter_smem + ((sizeof(ScatterSmem<KIND>) + 15) & ~(size_t)15));
  const uint32_t P = 1u << pbits;
  uint32_t* s_pos = s_cnt + P;
  const uint32_t warp = threadIdx.x >> 5, lane = lane_id();
  for (uint32_t k = threadIdx.x; k < P; k += C::THREADS) s_cnt[k] = 0;
  load_powers<KIND>(S.pow);
  load_combs<KIND>(S.comb);
  // this warp's share of the records: [r, r1)
  const uint64_t total = min(rec_off[n], n_cap);
  const uint64_t warps = (uint64_t)gridDim.x * C::WARPS;
  const uint64_t share = ((total + warps - 1) / warps + 31) & ~31ull;
  const uint64_t wid = (uint64_t)blockIdx.x * C::WARPS + warp;
  uint64_t r = min(wid * share, total);
  const uint64_t r1 = min(r + share, total);
  int64_t s = 0;
  uint32_t skip = 0;  // records of sequence s before r
  if (r < r1) {
    s = sequence_of(rec_off, n, r, lane);
    skip = (uint32_t)min(r - rec_off[s], (uint64_t)0x7fffffff);
  }
  const uint32_t q = lane / K::LANES;
  const uint32_t pshift = 32u - (uint32_t)pbits;
  const uint32_t idmask = (uint32_t)((1ull << id_bits) - 1ull);  // id_bits <= 32
  const bool wide = ((uint64_t)region << pbits) >> 32 != 0;  // words past 32-bit indices
  auto record = [&](uint64_t sum, uint32_t id) -> uint64_t {
    const uint64_t h = mix64(sum);
    return (h & 0xffffffff00000000ull) | (((uint32_t)h & ~idmask) | id);
  };
  if (threadIdx.x == 0) {
    S.over = 0;
    S.pshift = pshift;
  }

  while (__syncthreads_or(r < r1)) {
    // 1. generate: the warp's next T records
    uint32_t T = 0;
    const uint32_t id0 = (uint32_t)s;
    for (int batch = 0; batch < (K::D == 1 ? 2 : 1); ++batch) {
      if (r >= r1 || T >= (uint32_t)C::SLOTS) break;
      const int64_t my = s + q;
      const bool have = my < n;
      const uint64_t salt = have && seq_rep ? rep_salt(seq_rep[my]) : 0ull;
      VarMeta m;
      uint32_t cnt;
      if constexpr (K::D >= 2) {
        cnt = prepare_variants<KIND>(S.t.terms[warp][q], S.t.extra[warp][q], S.pow, src, my, have,
                                     d, salt, lane, m, [](uint32_t, uint64_t) {});
      } else {
        cnt = have ? canonical_total(src.eqprev[my], src.lens[my], d) : 0u;
        if (K::PAIRED && have) cnt += canonical_total(src.eq_b[my], src.lens_b[my], d) - 1u;
      }
      bool ok = !have || rec_off[my + 1] - rec_off[my] == cnt;
      uint32_t end = cnt;
#pragma unroll
      for (int o = K::LANES; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(FULL_MASK, end, o);
        if (lane >= (uint32_t)o) end += t;
      }
      ok = ok && (q > 0 || skip < cnt);
      if (!__all_sync(FULL_MASK, ok)) {  // record offsets that are not these sequences'
        if (lane == 0) atomicOr(err, DERR_RANGE);
        r = r1;
        break;
      }
      const uint32_t all = __shfl_sync(FULL_MASK, end, 31) - skip;
      const uint32_t N = (uint32_t)min(min((uint64_t)all, (uint64_t)(C::SLOTS - T)), r1 - r);
      if constexpr (K::D >= 2) {
        if (lane % K::LANES == 0) {
          m.end = (int32_t)(end - skip);
          m.adj += (int32_t)(end - cnt) - (int32_t)skip;
          S.t.meta[warp][q] = m;
        }
        __syncwarp();
      } else {
        // at most one deletion: the sums are the variants, written where
        // they stand in the warp's stream
        uint64_t* mine = S.stage + warp * C::SLOTS + T;
        // (with none at all only the last of them, put at index R, counts)
        uint32_t R = 0;
        if (d <= 0 && have) {
          R = canonical_total(src.eqprev[my], src.lens[my], 1) - 1u;
          if (K::PAIRED) R += canonical_total(src.eq_b[my], src.lens_b[my], 1) - 1u;
        }
        const int32_t adj = (int32_t)(end - cnt) - (int32_t)skip - (int32_t)R;
        prepare_variants<KIND>(nullptr, nullptr, S.pow, src, my, have, d, salt, lane, m,
                               [&](uint32_t a, uint64_t sum) {
                                 const int32_t t = adj + (int32_t)a;
                                 if (t >= 0 && (uint32_t)t < N && (d > 0 || a == R)) {
                                   const uint64_t v = record(sum, (uint32_t)my);
                                   mine[t] = v;
                                   atomicAdd(&s_cnt[(uint32_t)(v >> 32) >> pshift], 1u);
                                 }
                               });
      }
      // where the next records start
      const uint32_t done =
          __ballot_sync(FULL_MASK, lane % K::LANES == 0 && have && end - skip <= N);
      const uint32_t k = (uint32_t)__popc(done);  // sequences finished (a prefix)
      const uint32_t end_prev = __shfl_sync(FULL_MASK, end, (int)(k ? (k - 1) * K::LANES : 0));
      skip = k ? N + skip - end_prev : skip + N;
      s += k;
      r += N;
      T += N;
    }
    uint64_t rec[C::ITEMS];
    if constexpr (K::D >= 2) {
      const VarMeta* meta = S.t.meta[warp];
      const uint64_t* tab = S.t.terms[warp][0];
      const uint16_t* extra = S.t.extra[warp][0];
      VarMeta cur = meta[0];
      uint32_t id = id0;
#pragma unroll
      for (int i = 0; i < C::ITEMS; ++i) {
        const uint32_t t = i * 32 + lane;
        rec[i] = 0;  // (a value in every case, or the compiler carries the last step's along)
        if (t < T) {
          while ((int32_t)t >= cur.end) {  // ends: t < T <= the last sequence's end
            cur = *++meta;
            tab += K::STRIDE;
            extra += K::EXTRA + 1;
            ++id;
          }
          rec[i] = record(variant_sum<KIND>(tab, extra, S.comb, (uint32_t)((int32_t)t - cur.adj),
                                            cur.c, cur.aux),
                          id);
          atomicAdd(&s_cnt[(uint32_t)(rec[i] >> 32) >> pshift], 1u);
        }
      }
    }
    __syncthreads();  // the bins are complete, the terms dead
    if constexpr (K::D == 1) {
#pragma unroll
      for (int i = 0; i < C::ITEMS; ++i) {
        const uint32_t t = i * 32 + lane;
        rec[i] = t < T ? S.stage[warp * C::SLOTS + t] : 0ull;
      }
    }
    // 2. exclusive scan of the bins, then room in every partition
    scan_bins(s_cnt, P >> 8, S.wsum, &S.held);
    reserve_room<C::THREADS>(s_cnt, s_pos, P, S.held, region, part_count, &S.over);
    __syncthreads();
    // 3. place in partition order: C::BATCH places are asked for before the
    // first is used, or each would wait for its own shared-memory round trip.
    // The shift is read back from shared memory so that the bins are computed
    // again: kept from step 1 they would cost a register per record.
    const uint32_t pshift3 = S.pshift;
#pragma unroll
    for (int i0 = 0; i0 < C::ITEMS; i0 += C::BATCH) {
      uint32_t at[C::BATCH];
#pragma unroll
      for (int x = 0; x < C::BATCH; ++x) {
        const int i = i0 + x;
        at[x] = C::TILE;
        if ((uint32_t)(i * 32) + lane < T)
          at[x] = atomicAdd(&s_cnt[(uint32_t)(rec[i] >> 32) >> pshift3], 1u);
      }
#pragma unroll
      for (int x = 0; x < C::BATCH; ++x)
        if (at[x] < (uint32_t)C::TILE) S.stage[at[x]] = rec[i0 + x];
    }
    __syncthreads();
    // 4. write the runs out
    const uint32_t held = S.held;
    const bool over = S.over || wide;
    for (uint32_t k = threadIdx.x; k < P / 4; k += C::THREADS)
      reinterpret_cast<uint4*>(s_cnt)[k] = make_uint4(0u, 0u, 0u, 0u);
    if (!over) {
#pragma unroll 4
      for (uint32_t j = threadIdx.x; j < held; j += C::THREADS) {
        const uint64_t v = S.stage[j];
        out[s_pos[(uint32_t)(v >> 32) >> pshift] + j] = v;
      }
    } else {
      for (uint32_t j = threadIdx.x; j < held; j += C::THREADS) {
        const uint64_t v = S.stage[j];
        const uint32_t b = (uint32_t)(v >> 32) >> pshift;
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
  }
}

template <int KIND>
void scatter_launch(const ExpandSource& src, const uint64_t* rec_off, int64_t n, int d,
                    const uint32_t* seq_rep, uint32_t id_bits, uint64_t n_rec, int pbits,
                    uint64_t* out, uint32_t region, uint32_t* count, uint64_t* spill,
                    uint64_t spill_cap, uint64_t* n_spill, int sms, uint32_t* err,
                    cudaStream_t s) {
  auto f = k_expand_scatter<KIND>;
  static PerDevice shared;
  shared([&] {
    return allow_shared((const void*)f, (int)scatter_smem_bytes<KIND>(PART_MAX_BITS));
  });
  // small inputs: fewer records a warp, so that every SM has some
  using C = SC<KIND>;
  const uint64_t blocks =
      std::min<uint64_t>((n_rec + C::WARPS * 128 - 1) / (C::WARPS * 128), (uint64_t)sms);
  f<<<(uint32_t)blocks, C::THREADS, scatter_smem_bytes<KIND>(pbits), s>>>(
      src, rec_off, n, d, seq_rep, id_bits, n_rec, pbits, out, region, count, spill, spill_cap,
      reinterpret_cast<unsigned long long*>(n_spill), err);
}

}  // namespace

void launch_expand_scatter(const ExpandSource& src, const uint64_t* rec_off, int64_t n, int d,
                           const uint32_t* seq_rep, uint32_t id_bits, uint64_t n_rec,
                           const Partitions& p, int sms, uint32_t* err, cudaStream_t s) {
  if (n <= 0 || n_rec == 0) return;
  const bool paired = src.keys_b != nullptr;
  prof_begin(s, paired ? "k_expand_paired" : "k_expand",
             (double)n_rec * 8.0 + (double)n * (paired ? 58.0 : 29.0));
  auto go = [&](auto kind) {
    scatter_launch<decltype(kind)::value>(src, rec_off, n, d, seq_rep, id_bits, n_rec,
                                          p.pbits, p.rec, p.region, p.count,
                                          p.spill, p.spill_cap, p.n_spill, sms, err, s);
  };
  if (paired) {
    if (d <= 1) go(std::integral_constant<int, VK_PAIRED_D1>{});
    else go(std::integral_constant<int, VK_PAIRED_D2>{});
  } else if (d <= 1) {
    go(std::integral_constant<int, VK_D1>{});
  } else if (d == 2) {
    go(std::integral_constant<int, VK_D2>{});
  } else {
    go(std::integral_constant<int, VK_D3>{});
  }
  prof_end(s);
}

}  // namespace xtn
