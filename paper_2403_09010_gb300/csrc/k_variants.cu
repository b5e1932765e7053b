// Encoding and deletion-variant expansion (Appendix A, XTNeighbor steps 1-3;
// the `expand` primitive of Sec. 2.2: each input chunk writes a disjoint
// output chunk whose size is known ahead of time).
//
//   k_encode : ASCII sequence -> 128-bit key of 5-bit residue codes
//              (Appendix "Compression of TCR sequences"), its length, the
//              mask of positions equal to their left neighbour, the bit
//              planes of its codes (for the distance, k_verify.cu), and its
//              number of canonical deletion subsets (expand.cuh).
//   k_expand : the records  fingerprint[63:b] | id[b-1:0]  of every canonical
//              deletion variant, at rec_off (see expand.cuh).  The kernel also
//              accumulates the digit histograms of the radix passes that will
//              sort the records (all of them, or only the first when each
//              sort pass counts the next).
#include <algorithm>
#include <type_traits>

#include "expand.cuh"
#include "per_device.h"
#include "xtn_common.cuh"
#include "xtn_kernels.h"

namespace xtn {

// 'A'..'Z' -> residue code (alphabetical order of the 20 one-letter codes),
// 0 for letters outside the alphabet (B J O U X Z) and for anything else.
// Computed once a block for the encoder's table in shared memory (lanes of a
// warp read different letters, which a constant-memory table would serve one
// at a time).
constexpr uint32_t NOT_RESIDUE = (1u << 1) | (1u << 9) | (1u << 14) | (1u << 20) | (1u << 23) |
                                 (1u << 25);  // B J O U X Z
__device__ __forceinline__ uint32_t letter_code(uint32_t ch) {
  const uint32_t x = ch - (uint32_t)'A';
  if (x >= 26u || ((NOT_RESIDUE >> x) & 1u)) return 0u;
  return x + 1u - (uint32_t)__popc(NOT_RESIDUE & ((1u << x) - 1u));
}

constexpr int ENCODE_WARPS = 8;
constexpr int ENCODE_SPAN = 32 * XTN_MAX_LEN;       // letters of a warp's sequences, at most
constexpr int ENCODE_WORDS = ENCODE_SPAN / 4 + 10;  // and the words a lane reads past its own

// One warp per 32 consecutive sequences: their letters form one contiguous
// byte span, copied to shared memory four at a time; each lane then takes its
// own sequence as unaligned words, letter by letter through a 256-byte table
// (letters lie in different banks).  Six residues at a time are spread to
// five fields, one per code bit (one multiply and a mask each), which become
// the bit planes the distance needs; the equal-neighbour mask and the check
// for bad letters come from the planes.  About 250 instructions a sequence,
// against 500 for a loop over its letters and a match-vector kernel behind it
// (46 + 31 us for 1M sequences; 353 + 237 us for 10M).  Offsets are validated
// per lane first; a warp with an invalid offset reads each valid lane's
// letters directly instead.
//
// SCAN: the variant counts are not written but summed up to record offsets
// (single pass with decoupled look-back over the blocks), the total also to
// *total_out.  ROUNDS times 256 sequences a block, so that long inputs have
// fewer blocks to look back over: 1M sequences 53, 42, 39 and 44 us with 1, 2,
// 4 and 8 rounds, 10M 423, 283, 229 and 234 us (a scan kernel behind this one:
// 49 and 316 us for the two).
template <bool SCAN, int ROUNDS>
__global__ void __launch_bounds__(ENCODE_WARPS * 32, 8)
    k_encode(const uint8_t* __restrict__ seqs, const int64_t* __restrict__ off, int64_t n, int d,
             Key128* __restrict__ keys, uint8_t* __restrict__ lens,
             uint32_t* __restrict__ eqprev_out, uint32_t* __restrict__ vcount,
             uint64_t* __restrict__ rec_off, uint64_t* __restrict__ status,
             uint32_t* __restrict__ ctr, uint64_t* __restrict__ total_out,
             PlaneRow* __restrict__ rows, uint32_t* __restrict__ err) {
  __shared__ uint32_t s_words[ENCODE_WARPS][ENCODE_WORDS];
  __shared__ uint8_t s_code[256];
  __shared__ uint32_t s_sum[ENCODE_WARPS * ROUNDS];  // of each 32 sequences, then of all before
  __shared__ uint32_t s_before[SCAN ? ENCODE_WARPS * 32 * ROUNDS : 1];  // within its 32
  __shared__ uint64_t s_prefix;
  __shared__ uint32_t s_tile;
  static_assert(ENCODE_WARPS * 32 == 256, "one table entry per thread");
  static_assert(ENCODE_WARPS * ROUNDS <= 32, "one warp scans the sums");
  s_code[threadIdx.x] = (uint8_t)letter_code(threadIdx.x);
  const uint32_t warp = threadIdx.x >> 5, lane = lane_id();
  uint32_t tile = blockIdx.x;
  if (SCAN) tile = tile_id(ctr, &s_tile);  // in start order, for the look-back
  __syncthreads();
  const int64_t total = off[n];
#pragma unroll 1  // 32 registers, eight blocks an SM
  for (int round = 0; round < ROUNDS; ++round) {
    const int64_t s0 = (((int64_t)tile * ROUNDS + round) * ENCODE_WARPS + warp) * 32;
    const int64_t i = s0 + lane;
    const bool in = i < n;
    const int64_t a = in ? off[i] : 0, b = in ? off[i + 1] : 0;
    bool ok = in && a >= 0 && b >= a && b <= total;
    if (in && !ok) atomicOr(err, DERR_RANGE);
    if (i == 0 && a != 0) atomicOr(err, DERR_RANGE);  // offsets start at 0
    if (ok && b - a > XTN_MAX_LEN) {
      atomicOr(err, DERR_TOO_LONG);
      ok = false;
    }
    const bool all_ok = __all_sync(FULL_MASK, ok || !in);
    const int last = (int)max((int64_t)0, min((int64_t)31, n - s0 - 1));
    const int64_t A = __shfl_sync(FULL_MASK, a, 0), Bend = __shfl_sync(FULL_MASK, b, last);
    const uint32_t L = ok ? (uint32_t)(b - a) : 0u;
    uint32_t w[7];  // the sequence's letters, zeros behind them
    if (all_ok && Bend - A <= ENCODE_SPAN) {
      // byte k of the span sits at byte head + k of s_words, so that whole
      // words of the input land on whole words here
      __syncwarp();  // the round before is done with the words
      const uint8_t* src = seqs + A;
      const uint32_t head = (uint32_t)(reinterpret_cast<uintptr_t>(src) & 3u);
      const uint32_t bytes = head + (uint32_t)(Bend - A);
      uint8_t* dst = reinterpret_cast<uint8_t*>(s_words[warp]);
      const uint32_t w0 = head ? 1u : 0u, w1 = bytes / 4;  // whole words [w0, w1)
      const uint32_t* src4 = reinterpret_cast<const uint32_t*>(src - head);
      for (uint32_t k = w0 + lane; k < w1; k += 32) s_words[warp][k] = src4[k];
      if (head && lane >= head && lane < 4 && lane < bytes) dst[lane] = src[lane - head];
      const uint32_t tail = max(w0, w1) * 4 + lane;
      if (lane < 4 && tail < bytes) dst[tail] = src[tail - head];
      __syncwarp();
      const uint32_t o = head + (uint32_t)(a - A);
      const uint32_t sh = 8u * (o & 3u);
      const uint32_t* mine = s_words[warp] + (ok ? o / 4 : 0u);
      uint32_t lo = mine[0];
#pragma unroll
      for (int t = 0; t < 7; ++t) {
        const uint32_t hi = mine[t + 1];
        w[t] = __funnelshift_r(lo, hi, sh);
        lo = hi;
      }
    } else {
#pragma unroll
      for (int t = 0; t < 7; ++t) w[t] = 0;
#pragma unroll
      for (int p = 0; p < XTN_MAX_LEN; ++p)
        if ((uint32_t)p < L) w[p / 4] |= (uint32_t)seqs[a + p] << (8 * (p % 4));
    }
#pragma unroll
    for (int t = 0; t < 7; ++t) {  // clear what lies past the end
      const int left = (int)L - 4 * t;
      w[t] = left >= 4 ? w[t] : left > 0 ? w[t] & (0xffffffffu >> (32 - 8 * left)) : 0u;
    }
    Key128 key{0ull, 0ull};
    uint32_t plane[5] = {0u, 0u, 0u, 0u, 0u};
    const uint32_t longest = __reduce_max_sync(FULL_MASK, L);
#pragma unroll
    for (int g = 0; g < 5; ++g) {
      if ((uint32_t)(6 * g) >= longest) break;  // warp-uniform
      uint32_t acc = 0;  // five fields of six bits, the code's bits 0 .. 4
#pragma unroll
      for (int x = 0; x < 6; ++x) {
        const int p = 6 * g + x;
        acc >>= 1;
        if (p < XTN_MAX_LEN) {
          const uint32_t c = s_code[(w[p / 4] >> (8 * (p % 4))) & 255u];
          acc |= (c * 0x02108420u) & 0x20820820u;  // bit b of c to bit 6 b + 5
          if (5 * p < 64) key.lo |= (uint64_t)c << (5 * p < 64 ? 5 * p : 0);
          if (5 * p > 59)
            key.hi |= 5 * p < 64 ? (uint64_t)c >> (64 - 5 * p) : (uint64_t)c << (5 * p - 64);
        }
      }
#pragma unroll
      for (int k = 0; k < 5; ++k) plane[k] |= ((acc >> (6 * k)) & 63u) << (6 * g);
    }
    const uint32_t all = L ? 0xffffffffu >> (32 - L) : 0u;
    if ((plane[0] | plane[1] | plane[2] | plane[3] | plane[4]) != all)
      atomicOr(err, DERR_BAD_RESIDUE);  // a letter without a code
    uint32_t differs = 1u;  // from the left neighbour
#pragma unroll
    for (int k = 0; k < 5; ++k) differs |= plane[k] ^ (plane[k] << 1);
    const uint32_t eqprev = ~differs & all;
    const uint32_t count = in ? canonical_total(eqprev, L, d) : 0u;
    if (in) {
      keys[i] = key;
      lens[i] = (uint8_t)L;
      eqprev_out[i] = eqprev;
      if (!SCAN && vcount) vcount[i] = count;
      if (rows)
        store_row(rows + i, PlaneRow{make_uint4(plane[0], plane[1], plane[2], plane[3]),
                                     make_uint4(plane[4], L, 0u, 0u)});
    }
    if (SCAN) {
      uint32_t inc = count;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(FULL_MASK, inc, o);
        if (lane >= (uint32_t)o) inc += t;
      }
      s_before[round * ENCODE_WARPS * 32 + threadIdx.x] = inc - count;
      if (lane == 31) s_sum[round * ENCODE_WARPS + warp] = inc;
    }
  }
  if (!SCAN) return;
  __syncthreads();
  if (warp == 0) {
    const uint32_t v = lane < ENCODE_WARPS * ROUNDS ? s_sum[lane] : 0u;
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(FULL_MASK, inc, o);
      if (lane >= (uint32_t)o) inc += t;
    }
    if (lane < ENCODE_WARPS * ROUNDS) s_sum[lane] = inc - v;
    const uint32_t all = __shfl_sync(FULL_MASK, inc, 31);
    const uint64_t pre = warp_lookback(status, tile, all, err);
    if (lane == 0) {
      s_prefix = pre;
      if (((int64_t)tile + 1) * ROUNDS * ENCODE_WARPS * 32 >= n) {
        rec_off[n] = pre + all;
        *total_out = pre + all;
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int round = 0; round < ROUNDS; ++round) {
    const int64_t i = (((int64_t)tile * ROUNDS + round) * ENCODE_WARPS + warp) * 32 + lane;
    if (i < n) rec_off[i] = s_prefix + s_sum[round * ENCODE_WARPS + warp] +
                             s_before[round * ENCODE_WARPS * 32 + threadIdx.x];
  }
}

constexpr int EXPAND_THREADS = 256;

// One count per radix pass for record `rec` (8-bit digits from bit `lo`; the
// last digit keeps only `last_mask`).
// H: HIST_NONE, HIST_HIGH (lo >= 32 and every counted digit lies in the high
// word: 32-bit shifts) or HIST_ANY.
enum { HIST_NONE = 0, HIST_HIGH, HIST_ANY };
template <int H>
__device__ __forceinline__ void count_digits(uint32_t* s_hist, uint64_t rec, int lo, int passes,
                                             uint32_t last_mask) {
  if constexpr (H == HIST_NONE) return;
  if constexpr (H == HIST_HIGH) {
    const uint32_t r = (uint32_t)(rec >> 32) >> (lo - 32);
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      if (p < passes) {
        const uint32_t m = p == passes - 1 ? last_mask : 0xffu;
        atomicAdd(&s_hist[p * RADIX + ((r >> (8 * p)) & m)], 1u);
      }
    }
    return;
  }
  const uint64_t r = rec >> lo;
#pragma unroll
  for (int p = 0; p < MAX_PASSES; ++p) {
    if (p < passes) {
      const uint32_t m = p == passes - 1 ? last_mask : 0xffu;
      atomicAdd(&s_hist[p * RADIX + ((uint32_t)(r >> (8 * p)) & m)], 1u);
    }
  }
}

static_assert((1 << MAX_BIN_BITS) <= MAX_PASSES * RADIX, "bins share the digit histogram");

// Appended records (SEL_APPEND) collect per warp in shared memory and go out
// STAGE_FLUSH or more at a time: a warp reserves output space once per
// batch, not once per round (rounds keep a record in nearly every warp
// whatever the share of bins selected, and every reservation is an atomic
// on one counter), and the stores are contiguous runs.
constexpr uint32_t STAGE_FLUSH = 128;
constexpr uint32_t STAGE_CAP = STAGE_FLUSH + 32;
struct WarpStage {
  uint64_t* buf;  // STAGE_CAP words of this warp
  uint32_t n;     // staged records (the same in every lane)
};

__device__ __forceinline__ void flush_stage(WarpStage& st, uint64_t* __restrict__ out,
                                            uint64_t n_rec, const BinSel& sel, uint32_t lane,
                                            uint32_t* __restrict__ err) {
  if (st.n == 0) return;
  unsigned long long base = 0;
  if (lane == 0) base = atomicAdd(sel.append, (unsigned long long)st.n);
  base = __shfl_sync(FULL_MASK, base, 0);
  __syncwarp();  // every lane's staged records are visible
  for (uint32_t k = lane; k < st.n; k += 32) {
    const uint64_t slot = base + k;
    if (slot < n_rec)
      out[slot] = st.buf[k];
    else
      atomicOr(err, DERR_RANGE);
  }
  __syncwarp();  // read before the stage fills again
  st.n = 0;
}

// Where a finished record goes (all lanes of the warp call this together;
// `valid` says whether this lane holds a record):
//   SEL_ALL    out[pos], its digits counted for the sort
//   SEL_COUNT  only its fingerprint bin counted (s_hist holds the bins)
//   SEL_APPEND staged for appending when its bin lies in [sel.lo, sel.hi);
//              its digits counted
template <int SEL, int H>
__device__ __forceinline__ void place_record(uint64_t rec, bool valid, uint64_t pos,
                                             uint64_t* __restrict__ out, uint64_t n_rec,
                                             uint32_t* s_hist, int hist_lo, int hist_passes,
                                             uint32_t last_mask, const BinSel& sel, uint32_t lane,
                                             WarpStage& st, uint32_t* __restrict__ err) {
  if constexpr (SEL == SEL_ALL) {
    if (valid) {
      out[pos] = rec;
      count_digits<H>(s_hist, rec, hist_lo, hist_passes, last_mask);
    }
  } else {
    const uint32_t bin = (uint32_t)(rec >> sel.shift) & sel.mask;
    if constexpr (SEL == SEL_COUNT) {
      if (valid) atomicAdd(&s_hist[bin], 1u);
    } else {
      const bool keep = valid && bin >= sel.lo && bin < sel.hi;
      const uint32_t bal = __ballot_sync(FULL_MASK, keep);
      if (keep) {
        st.buf[st.n + __popc(bal & ((1u << lane) - 1u))] = rec;  // st.n + 32 <= STAGE_CAP
        count_digits<H>(s_hist, rec, hist_lo, hist_passes, last_mask);
      }
      st.n += __popc(bal);
      if (st.n >= STAGE_FLUSH) flush_stage(st, out, n_rec, sel, lane, err);
    }
  }
}

// Clears n 16-byte words for a later kernel (the record sort's look-back
// status), grid-stride: the expansion is bound by instruction issue, so these
// stores cost it almost nothing and spare the sort a memset or the clearing.
__device__ __forceinline__ void zero_fill(uint4* __restrict__ p, uint64_t n) {
  for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (uint64_t)gridDim.x * blockDim.x)
    p[k] = make_uint4(0u, 0u, 0u, 0u);
}

// The expansion into records at rec_off (SEL_ALL), or of selected bins.  A
// warp takes PACK consecutive sequences: its lanes prepare their terms
// (expand.cuh), then the warp walks the batch's records as one stream, lane
// by lane, each lane moving to the next sequence when its position passes
// the current one's end.  Every lane computes a record in every round and
// the batch's records are contiguous in the output, so stores coalesce.
constexpr int EXPAND_WARPS = EXPAND_THREADS / 32;

template <int KIND, int SEL, int H>
struct ExpandSmem {
  using K = VK<KIND>;
  uint64_t terms[EXPAND_WARPS][K::PACK][K::STRIDE];
  uint64_t stage[SEL == SEL_APPEND ? EXPAND_WARPS : 1][SEL == SEL_APPEND ? STAGE_CAP : 1];
  uint64_t pow[N_POWERS<KIND>];
  VarMeta meta[EXPAND_WARPS][K::PACK];
  uint32_t hist[H != HIST_NONE || SEL == SEL_COUNT ? MAX_PASSES * RADIX : 1];
  uint16_t extra[EXPAND_WARPS][K::PACK][K::EXTRA + 1];
  uint16_t comb[K::COMBS + 1];
};

template <int KIND, int SEL, int H>
__global__ void __launch_bounds__(EXPAND_THREADS, 4)
    k_expand(ExpandSource src, const uint64_t* __restrict__ rec_off, int64_t n, int d,
             const uint32_t* __restrict__ seq_rep, uint32_t id_bits, uint64_t* __restrict__ out,
             uint64_t n_rec, uint32_t* __restrict__ hist, int hist_lo, int hist_passes,
             int hist_hi, BinSel sel, uint32_t* __restrict__ err, uint4* __restrict__ zero,
             uint64_t n_zero) {
  using K = VK<KIND>;
  extern __shared__ __align__(16) unsigned char expand_smem[];
  ExpandSmem<KIND, SEL, H>& S = *reinterpret_cast<ExpandSmem<KIND, SEL, H>*>(expand_smem);
  zero_fill(zero, n_zero);
  const uint32_t warp = threadIdx.x >> 5, lane = lane_id();
  WarpStage st{S.stage[SEL == SEL_APPEND ? warp : 0], 0u};
  const int n_hist = SEL == SEL_COUNT ? (int)sel.mask + 1 : H ? hist_passes * RADIX : 0;
  for (int k = threadIdx.x; k < n_hist; k += blockDim.x) S.hist[k] = 0;
  load_powers<KIND>(S.pow);
  load_combs<KIND>(S.comb);
  __syncthreads();
  const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const uint32_t idmask = (uint32_t)((1ull << id_bits) - 1ull);  // id_bits <= 32
  const int last_bits = hist_hi - hist_lo - 8 * (hist_passes - 1);
  const uint32_t last_mask = (1u << last_bits) - 1u;
  const int q = (int)lane / K::LANES;  // this lane's sequence in the batch
  VarMeta* meta = S.meta[warp];
  for (int64_t s0 = warp0 * K::PACK; s0 < n; s0 += n_warps * K::PACK) {
    const int64_t my = s0 + q;
    const bool have = my < n;
    const uint64_t salt = have && seq_rep ? rep_salt(seq_rep[my]) : 0ull;
    VarMeta m;
    uint64_t* terms = S.terms[warp][q];
    uint32_t total =
        prepare_variants<KIND>(terms, S.extra[warp][q], S.pow, src, my, have, d, salt, lane, m,
                               [&](uint32_t a, uint64_t h) { terms[a] = h; });
    const uint64_t base = have ? rec_off[my] : 0ull;
    if (have) {
      const uint64_t cnt = rec_off[my + 1] - base;
      if (total != cnt || (SEL == SEL_ALL && base + cnt > n_rec)) {
        atomicOr(err, DERR_RANGE);
        total = 0;
      }
    }
    // where each sequence of the batch ends in the stream
    uint32_t end = total;
#pragma unroll
    for (int o = K::LANES; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(FULL_MASK, end, o);
      if (lane >= (uint32_t)o) end += t;
    }
    const uint32_t T = __shfl_sync(FULL_MASK, end, 31);
    const uint64_t base0 = __shfl_sync(FULL_MASK, base, 0);
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
    for (uint32_t t0 = 0; t0 < T; t0 += 32) {
      const uint32_t t = t0 + lane;
      uint64_t rec = 0;
      if (t < T) {
        while ((int32_t)t >= cur.end) {  // ends: t < T, the last sequence's end
          cur = *++at;
          ++id;
          tab += K::STRIDE;
          extra += K::EXTRA + 1;
        }
        const uint64_t h = mix64(variant_sum<KIND>(
            tab, extra, S.comb, (uint32_t)((int32_t)t - cur.adj), cur.c, cur.aux));
        rec = (h & 0xffffffff00000000ull) | (((uint32_t)h & ~idmask) | id);
      }
      place_record<SEL, H>(rec, t < T, base0 + t, out, n_rec, S.hist, hist_lo, hist_passes,
                             last_mask, sel, lane, st, err);
    }
    __syncwarp();  // the next batch overwrites the tables
  }
  if constexpr (SEL == SEL_APPEND) flush_stage(st, out, n_rec, sel, lane, err);
  __syncthreads();
  uint32_t* dst = SEL == SEL_COUNT ? sel.bin_count : hist;
  for (int k = threadIdx.x; k < n_hist; k += blockDim.x)
    if (S.hist[k]) atomicAdd(&dst[k], S.hist[k]);
}

// seq_rep[i] = repertoire of sequence i: the last r with rep_off[r] <= i.
__global__ void k_seq_rep(const int64_t* __restrict__ rep_off, int64_t n_rep,
                          uint32_t* __restrict__ seq_rep, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int64_t lo = 0, hi = n_rep;
  while (hi - lo > 1) {
    const int64_t mid = (lo + hi) >> 1;
    if (rep_off[mid] <= i) lo = mid; else hi = mid;
  }
  seq_rep[i] = (uint32_t)lo;
}

void launch_seq_rep(const int64_t* rep_off, int64_t n_rep, uint32_t* seq_rep, int64_t n,
                    cudaStream_t s) {
  if (n <= 0) return;
  prof_begin(s, "k_seq_rep", (double)n * 4.0);
  k_seq_rep<<<div_up_u32(n, 256), 256, 0, s>>>(rep_off, n_rep, seq_rep, n);
  prof_end(s);
}

void launch_encode(const uint8_t* seqs, const int64_t* off, int64_t n, int d, Key128* keys,
                   uint8_t* lens, uint32_t* eqprev, uint32_t* vcount, PlaneRow* rows,
                   uint32_t* err, cudaStream_t s) {
  if (n <= 0) return;
  prof_begin(s, "k_encode", (double)n * (16 + 16 + 1 + 4 + 4 + 8 + (rows ? 32 : 0)));
  k_encode<false, 1><<<div_up_u32(n, ENCODE_WARPS * 32), ENCODE_WARPS * 32, 0, s>>>(
      seqs, off, n, d, keys, lens, eqprev, vcount, nullptr, nullptr, nullptr, nullptr, rows, err);
  prof_end(s);
}

// Above this many sequences (two blocks an SM with four rounds each) a block
// takes four rounds of them; below, more blocks are worth more.
constexpr int64_t ENCODE_LONG = 1 << 18;

size_t encode_status_bytes(int64_t n) {
  const int64_t per = ENCODE_WARPS * 32 * (n > ENCODE_LONG ? 4 : 1);
  return (size_t)((n + per - 1) / per) * 8 + 16;
}

void launch_encode_scan(const uint8_t* seqs, const int64_t* off, int64_t n, int d, Key128* keys,
                        uint8_t* lens, uint32_t* eqprev, uint64_t* rec_off, uint64_t* total,
                        uint64_t* status, PlaneRow* rows, uint32_t* err, cudaStream_t s) {
  if (n <= 0) return;
  const size_t st = encode_status_bytes(n);
  uint32_t* ctr = reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(status) + st - 16);
  prof_begin(s, "k_encode", (double)n * (16 + 16 + 1 + 4 + 8 + 8 + (rows ? 32 : 0)));
  auto f = n > ENCODE_LONG ? k_encode<true, 4> : k_encode<true, 1>;
  f<<<(uint32_t)((st - 16) / 8), ENCODE_WARPS * 32, 0, s>>>(seqs, off, n, d, keys, lens, eqprev,
                                                            nullptr, rec_off, status, ctr, total,
                                                            rows, err);
  prof_end(s);
}

template <int KIND, int SEL, int H>
static void expand_launch(const ExpandSource& src, const uint64_t* rec_off, int64_t n, int d,
                          const uint32_t* seq_rep, uint32_t id_bits, uint64_t* out, uint64_t n_rec,
                          uint32_t* hist, int hist_lo, int hist_hi, const BinSel& sel, int sms,
                          uint32_t* err, cudaStream_t s, uint4* zero, uint64_t n_zero) {
  auto f = k_expand<KIND, SEL, H>;
  constexpr int smem = (int)sizeof(ExpandSmem<KIND, SEL, H>);
  static PerDevice shared;
  shared([&] { return allow_shared((const void*)f, smem); });
  const int per_block = EXPAND_WARPS * VK<KIND>::PACK;
  const int64_t blocks = std::min<int64_t>((n + per_block - 1) / per_block, (int64_t)sms * 8);
  f<<<(uint32_t)blocks, EXPAND_THREADS, smem, s>>>(src, rec_off, n, d, seq_rep, id_bits, out,
                                                   n_rec, hist, hist_lo, (hist_hi - hist_lo + 7) / 8,
                                                   hist_hi, sel, err, zero, n_zero);
}

void launch_expand(const ExpandSource& src, const uint64_t* rec_off, int64_t n, int d,
                   const uint32_t* seq_rep, uint32_t id_bits, uint64_t* out, uint64_t n_rec,
                   uint32_t* hist, int hist_lo, int hist_hi, int sms, uint32_t* err,
                   cudaStream_t s, const BinSel* sel, void* zero, size_t zero_bytes) {
  uint4* z = static_cast<uint4*>(zero);
  const uint64_t nz = z ? zero_bytes / 16 : 0;
  if (n <= 0) return;
  const BinSel none{};
  const bool paired = src.keys_b != nullptr;
  const bool high = hist_lo >= 32 && hist_hi <= 64;
  auto go = [&](auto kind) {
    constexpr int KIND = decltype(kind)::value;
    auto f = !hist  ? expand_launch<KIND, SEL_ALL, HIST_NONE>
             : high ? expand_launch<KIND, SEL_ALL, HIST_HIGH>
                    : expand_launch<KIND, SEL_ALL, HIST_ANY>;
    if constexpr (!VK<KIND>::PAIRED)
      if (sel)
        f = !sel->append ? expand_launch<KIND, SEL_COUNT, HIST_NONE>
            : hist       ? expand_launch<KIND, SEL_APPEND, HIST_ANY>
                         : expand_launch<KIND, SEL_APPEND, HIST_NONE>;
    f(src, rec_off, n, d, seq_rep, id_bits, out, n_rec, hist, hist_lo, hist_hi, sel ? *sel : none,
      sms, err, s, z, nz);
  };
  const char* name = paired ? "k_expand_paired"
                     : !sel ? "k_expand" : sel->append ? "k_expand_bins" : "k_expand_count";
  prof_begin(s, name, (sel && !sel->append ? 0.0 : (double)n_rec * 8.0) +
                          (double)n * (paired ? 58.0 : 29.0));
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
