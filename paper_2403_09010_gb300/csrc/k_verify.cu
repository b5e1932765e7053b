// Exact verification and duplicate removal (Appendix A, XTNeighbor steps 6-7:
// `map` + `if` with the edit distance, `sort` + `unique`), and the TCRdist
// post-filter (Results, "SymDel lookup can be combined with more advanced
// similarity metrics").
//
// The paper removes duplicate pairs first and verifies after; here every
// candidate is verified first and only the survivors are sorted: the
// duplicates of Fig. 1C are cheap to verify but costly to sort, and the
// output is the same set either way.
//
//   k_verify_candidates : per candidate (i, j): drop i == j (one sequence
//                         sharing a variant with itself through repeated
//                         residues) and pairs from different repertoires
//                         (from the same one when searching between them),
//                         reject |len_i - len_j| > d, compute the edit
//                         distance up to d, keep it if <= d.  Survivors
//                         are appended with one atomic per warp; their radix
//                         histograms are accumulated on the way.
//   k_unique_finalize   : over the sorted survivors, drop a word equal to its
//                         predecessor (the duplicates of Fig. 1C) and write
//                         {i, j, dist} rows in order (single-pass compaction
//                         with decoupled look-back).
//
// Edit distance: only distances up to d <= 3 matter, so instead of a table
// (or a bit-vector recurrence over every residue of the text) each edit count
// e = 0 .. d gets the furthest position reached on every diagonal with e edits
// (Ukkonen 1985; Landau & Vishkin 1989).  With the sequences as bit planes
// (PlaneRow) the differing positions of a diagonal are one 32-bit word, and
// sliding along equal residues is one count of trailing zeros.  About 110
// instructions a pair at d = 2, two row loads and no per-sequence tables,
// against 450, 16 gathered words and a table of 80 bytes per sequence for the
// bit-vector form (146 us for the 1M workload's 4.3 M candidates).
#include <algorithm>

#include "per_device.h"
#include "xtn_common.cuh"
#include "xtn_kernels.h"

namespace xtn {

constexpr int VER_THREADS = 256;
constexpr int VER_ITEMS = 8;
constexpr int VER_TILE = VER_THREADS * VER_ITEMS;
static_assert(VER_TILE == VERIFY_TILE, "status sizing in xtn_kernels.h assumes this tile");

struct Planes {
  uint32_t p[5];
  uint32_t n;  // length
};

__device__ __forceinline__ Planes load_planes(const PlaneRow* __restrict__ rows, uint64_t i) {
  const PlaneRow r = load_row(rows + i);
  return Planes{{r.a.x, r.a.y, r.a.z, r.a.w, r.b.x}, r.b.y};
}

// Diagonal k = (position in y) - (position in x), -3 <= k <= 3: bit p set
// where x[p] and y[p + k] differ, and past the diagonal's end, min(m, n - k).
__device__ __forceinline__ uint32_t diagonal(const Planes& x, const Planes& y, int k) {
  uint32_t diff = 0;
#pragma unroll
  for (int b = 0; b < 5; ++b) diff |= x.p[b] ^ ((y.p[b] << 3) >> (3 + k));
  const int end = max(0, min((int)x.n, (int)y.n - k));  // <= 25
  return diff | (0xffffffffu << end);
}

// The position reached from p on a diagonal without further edits.
__device__ __forceinline__ int slide(uint32_t diff, int p) {
  return p + __ffs((int)(diff >> p)) - 1;  // p <= end: a bit is left
}

// Levenshtein distance of x and y if it is at most D, else D + 1.
template <int D>
__device__ __forceinline__ uint32_t bounded_distance(const Planes& x, const Planes& y) {
  const int m = (int)x.n, n = (int)y.n, t = n - m;
  if (t > D || -t > D) return (uint32_t)D + 1u;
  // f[D + k]: furthest position in x on diagonal k with the edits so far
  constexpr int NONE = -64;
  const uint32_t diff0 = diagonal(x, y, 0);
  int f[2 * D + 1];
#pragma unroll
  for (int k = 0; k < 2 * D + 1; ++k) f[k] = NONE;
  f[D] = slide(diff0, 0);
  if (t == 0 && f[D] >= m) return 0u;
  // from diagonal k's neighbours: a substitution; a residue of x left out
  // (from k + 1); one of y (from k - 1)
  auto start = [&](int k) {
    int p = f[D + k] + 1;
    if (k < D) p = max(p, f[D + k + 1 <= 2 * D ? D + k + 1 : 0] + 1);
    if (k > -D) p = max(p, f[D + k - 1 >= 0 ? D + k - 1 : 0]);
    return min(p, min(m, n - k));
  };
  // a diagonal that no path has reached yet, or of no length, gives NONE
  auto run = [&](int k, int p) {
    return p >= 0 && p + k >= 0 ? slide(k == 0 ? diff0 : diagonal(x, y, k), p) : NONE;
  };
#pragma unroll
  for (int e = 1; e < D; ++e) {
    int g[2 * D + 1];
#pragma unroll
    for (int k = -D; k <= D; ++k) g[D + k] = k < -e || k > e ? NONE : run(k, start(k));
    int last = NONE;
#pragma unroll
    for (int k = -D; k <= D; ++k) {
      f[D + k] = g[D + k];
      if (k == t) last = g[D + k];
    }
    if (last >= m) return (uint32_t)e;
  }
  if (D > 0) {  // the last edit matters on the final diagonal only
    int p = NONE;
#pragma unroll
    for (int k = -D; k <= D; ++k)
      if (k == t) p = start(k);
    if (run(t, p) >= m) return (uint32_t)D;
  }
  return (uint32_t)D + 1u;
}

__device__ __forceinline__ uint32_t bounded_distance(const Planes& x, const Planes& y, int d) {
  switch (d) {  // uniform
    case 0: return bounded_distance<0>(x, y);
    case 1: return bounded_distance<1>(x, y);
    case 2: return bounded_distance<2>(x, y);
    default: return bounded_distance<3>(x, y);
  }
}

// Distance of candidate (i, j) for the last step, if it is at most d (else
// anything above d): metric 0 = Levenshtein, 1 = Hamming (equal lengths
// only), 2 = the sum of both chains' edit distances (paired receptors).
__device__ __forceinline__ uint32_t cand_distance(int metric, int d, const PairSide& si,
                                                  const PairSide& sj, uint64_t i, uint64_t j) {
  const Planes x = load_planes(si.rows, i), y = load_planes(sj.rows, j);
  if (metric == 1) {
    if (x.n != y.n) return (uint32_t)d + 1u;
    uint32_t diff = 0;
#pragma unroll
    for (int b = 0; b < 5; ++b) diff |= x.p[b] ^ y.p[b];
    return (uint32_t)__popc(diff);
  }
  uint32_t dist = bounded_distance(x, y, d);
  if (metric == 2 && dist <= (uint32_t)d)
    dist += bounded_distance(load_planes(si.rows_b, i), load_planes(sj.rows_b, j), d);
  return dist;
}

template <int THREADS>
__device__ __forceinline__ uint32_t block_excl_scan_u32(uint32_t v, uint32_t* s_w, uint32_t& excl) {
  const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
  uint32_t inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(FULL_MASK, inc, o);
    if (lane >= (uint32_t)o) inc += t;
  }
  if (lane == 31) s_w[warp] = inc;
  __syncthreads();
  uint32_t off = 0, total = 0;
#pragma unroll
  for (int w = 0; w < THREADS / 32; ++w) {
    if (w < (int)warp) off += s_w[w];
    total += s_w[w];
  }
  excl = off + inc - v;
  __syncthreads();
  return total;
}

// Whether candidate word w is a row, and its distance.
__device__ __forceinline__ bool verified(uint64_t w, uint32_t j_bits, const PairSide& si,
                                         const PairSide& sj, const uint32_t* __restrict__ seq_rep,
                                         int self_mode, int d, int metric,
                                         uint32_t* __restrict__ err, uint32_t& dist) {
  const uint64_t i = w >> j_bits, j = w & ((1ull << j_bits) - 1ull);
  if (i >= si.n || j >= sj.n) {
    atomicOr(err, DERR_RANGE);
    return false;
  }
  if (self_mode && i == j) return false;
  if (seq_rep && (seq_rep[i] == seq_rep[j]) != (self_mode != 2)) return false;
  dist = cand_distance(metric, d, si, sj, i, j);
  return dist <= (uint32_t)d;
}

constexpr uint32_t VER_STASH = 256;  // survivor words a warp collects before a flush

__global__ void __launch_bounds__(256)
    k_verify_candidates(const uint64_t* __restrict__ cand, uint64_t n_cap,
                        const uint64_t* __restrict__ n_dev, uint32_t j_bits, PairSide si,
                        PairSide sj, const uint32_t* __restrict__ seq_rep, int self_mode, int d,
                        int metric, uint64_t* __restrict__ surv, uint64_t surv_cap,
                        unsigned long long* __restrict__ n_surv, uint32_t* __restrict__ hist,
                        int hist_lo, int hist_hi, uint32_t* __restrict__ err) {
  __shared__ uint32_t s_hist[MAX_PASSES * RADIX];
  // survivors collect per warp and go out VER_STASH - 31 or more at a time:
  // one reservation on the shared counter per flush, not per 32 candidates
  __shared__ uint64_t s_stash[256 / 32][VER_STASH];
  const int passes = (hist_hi - hist_lo + 7) / 8;
  for (int k = threadIdx.x; k < passes * RADIX; k += blockDim.x) s_hist[k] = 0;
  __syncthreads();
  const uint64_t n = n_dev ? min(*n_dev, n_cap) : n_cap;
  const uint32_t lane = lane_id();
  uint64_t* stash = s_stash[threadIdx.x >> 5];
  uint32_t held = 0;  // words in this warp's stash
  auto flush = [&]() {
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(n_surv, (unsigned long long)held);
    base = __shfl_sync(FULL_MASK, base, 0);
    for (uint32_t k = lane; k < held; k += 32) {
      if (base + k < surv_cap) surv[base + k] = stash[k];
      else atomicOr(err, DERR_RANGE);
    }
    __syncwarp();  // the stash is refilled next
    held = 0;
  };
  const uint32_t lt_mask = (1u << lane) - 1u;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t t0 = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); t0 < n;
       t0 += stride) {
    const uint64_t t = t0 + lane;
    bool ok = false;
    uint64_t w = 0;
    if (t < n) {
      w = cand[t];
      uint32_t dist = 0;
      ok = verified(w, j_bits, si, sj, seq_rep, self_mode, d, metric, err, dist);
      // the distance rides above the pair bits, for the dedup to write it
      if (ok && hist_hi + 8 <= 64) w |= (uint64_t)dist << hist_hi;
    }
    const uint32_t bal = __ballot_sync(FULL_MASK, ok);
    if (ok) {
      stash[held + __popc(bal & lt_mask)] = w;
      for (int p = 0; p < passes; ++p) {
        const int sh = hist_lo + 8 * p;
        const int bits = min(8, hist_hi - sh);
        atomicAdd(&s_hist[p * RADIX + (uint32_t)((w >> sh) & ((1u << bits) - 1u))], 1u);
      }
    }
    held += (uint32_t)__popc(bal);
    __syncwarp();
    if (held > VER_STASH - 32) flush();  // warp-uniform
  }
  if (held) flush();
  __syncthreads();
  for (int k = threadIdx.x; k < passes * RADIX; k += blockDim.x)
    if (s_hist[k]) atomicAdd(&hist[k], s_hist[k]);
}

void launch_verify_candidates(const uint64_t* cand, uint64_t n, const uint64_t* n_dev,
                              uint32_t j_bits, const PairSide& si, const PairSide& sj,
                              const uint32_t* seq_rep, int self_mode, int d, int metric,
                              uint64_t* surv, uint64_t surv_cap, uint64_t* n_surv, uint32_t* hist,
                              int hist_lo, int hist_hi, int sms, uint32_t* err, cudaStream_t s) {
  if (n == 0) return;
  const int blocks = (int)std::min<uint64_t>((n + 255) / 256, (uint64_t)sms * 8);
  prof_begin(s, "k_verify_candidates", (double)n * (8.0 + 2 * 32.0));
  k_verify_candidates<<<blocks, 256, 0, s>>>(
      cand, n, n_dev, j_bits, si, sj, seq_rep, self_mode, d, metric, surv, surv_cap,
      reinterpret_cast<unsigned long long*>(n_surv), hist, hist_lo, hist_hi, err);
  prof_end(s);
}

__global__ void __launch_bounds__(VER_THREADS)
    k_unique_finalize(const uint64_t* __restrict__ pairs, int64_t n_cap,
                      const uint64_t* __restrict__ n_dev, uint32_t j_bits, PairSide si,
                      PairSide sj, int d, int metric, xtn_triple* __restrict__ out, int64_t cap,
                      uint64_t* __restrict__ status, uint32_t* __restrict__ ctr,
                      uint32_t* __restrict__ err, uint64_t* __restrict__ total_out,
                      int dist_shift) {
  __shared__ uint32_t s_tile;
  __shared__ uint32_t s_w[VER_THREADS / 32];
  __shared__ uint64_t s_prefix;
  const int64_t n = n_dev ? min((int64_t)*n_dev, n_cap) : n_cap;
  const uint32_t warp = threadIdx.x >> 5, lane = lane_id();
  const uint32_t lt_mask = (1u << lane) - 1u;
  const uint64_t jmask = (1ull << j_bits) - 1ull;
  // persistent: every block takes tiles in start order until the input runs out
  for (;;) {
  const uint32_t tile = tile_id(ctr, &s_tile);
  const int64_t tbase = (int64_t)tile * VER_TILE;
  if (tbase >= n) break;
  // warp w covers positions [wbase, wbase + 32 * ITEMS), lane l position
  // wbase + it * 32 + l of round it: reads coalesce and the rounds follow
  // position order, so ballots compact each round in order
  const int64_t wbase = tbase + (int64_t)warp * 32 * VER_ITEMS;
  uint32_t keep = 0, wtotal = 0;
  uint32_t rank[VER_ITEMS], dist[VER_ITEMS];
  uint64_t word[VER_ITEMS];
#pragma unroll
  for (int it = 0; it < VER_ITEMS; ++it) {
    const int64_t p = wbase + it * 32 + lane;
    bool ok = false;
    dist[it] = 0;
    word[it] = 0;
    if (p < n) {
      const uint64_t w = pairs[p];
      const uint64_t prev = p > 0 ? pairs[p - 1] : ~w;
      // with dist_shift the verified distance sits above the pair bits (the
      // same pair always carries the same distance, so equal pairs are equal
      // words); else it is computed again
      const uint64_t pw = dist_shift ? (w & ((1ull << dist_shift) - 1ull)) : w;
      const uint64_t i = pw >> j_bits, j = pw & jmask;
      ok = w != prev;
      if (i >= si.n || j >= sj.n) {
        atomicOr(err, DERR_RANGE);
        ok = false;
      }
      if (ok)
        dist[it] = dist_shift ? (uint32_t)((w >> dist_shift) & 0xffu)
                              : cand_distance(metric, d, si, sj, i, j);
      word[it] = pw;
    }
    const uint32_t bal = __ballot_sync(FULL_MASK, ok);
    rank[it] = wtotal + __popc(bal & lt_mask);
    wtotal += __popc(bal);
    keep |= (uint32_t)ok << it;
  }
  if (lane == 0) s_w[warp] = wtotal;
  __syncthreads();
  uint32_t woff = 0, total = 0;
#pragma unroll
  for (int w = 0; w < VER_THREADS / 32; ++w) {
    if (w < (int)warp) woff += s_w[w];
    total += s_w[w];
  }
  if (warp == 0) {
    const uint64_t pre = warp_lookback(status, tile, total, err);
    if (lane == 0) {
      s_prefix = pre;
      if (tbase + VER_TILE >= n) *total_out = pre + total;
    }
  }
  __syncthreads();
  const int64_t o0 = (int64_t)(s_prefix + woff);
#pragma unroll
  for (int it = 0; it < VER_ITEMS; ++it) {
    if (keep >> it & 1u) {
      const int64_t o = o0 + rank[it];
      if (o < cap) {
        xtn_triple t;
        t.i = (uint32_t)(word[it] >> j_bits);
        t.j = (uint32_t)(word[it] & jmask);
        t.dist = dist[it];
        out[o] = t;
      }
    }
  }
  __syncthreads();  // s_prefix, s_w and s_tile are reused by the next tile
  }
}

size_t verify_status_bytes(int64_t n) { return verify_status_bytes_for(n); }

void launch_unique_finalize(const uint64_t* pairs, int64_t n, const uint64_t* n_dev,
                            uint32_t j_bits, const PairSide& si, const PairSide& sj, int d,
                            int metric, xtn_triple* out, int64_t cap, uint64_t* status,
                            uint32_t* err, uint64_t* total, cudaStream_t s, int dist_shift,
                            bool status_zeroed) {
  if (n <= 0) return;
  const size_t st = verify_status_bytes(n);
  uint32_t* ctr = reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(status) + st - 16);
  if (!status_zeroed) cudaMemsetAsync(status, 0, st, s);
  prof_begin(s, "k_unique_finalize", (double)n * 8.0);
  k_unique_finalize<<<std::min<uint32_t>(div_up_u32(n, VER_TILE), 152 * 8), VER_THREADS, 0, s>>>(
      pairs, n, n_dev, j_bits, si, sj, d, metric, out, cap, status, ctr, err, total, dist_shift);
  prof_end(s);
}

// ----------------------------------------------------------- small results ---
// Drop duplicates (a hash table in shared memory), verify, sort and write rows
// in one block of one launch: for a few thousand candidates the general path
// (ten launches and clears) is all latency.  Duplicates go first because most
// candidates are some: a pair has one candidate per variant it shares.  The
// sort is bitonic with a thread's words in registers: exchanges across less
// than a warp are shuffles, and only those across warps go through shared
// memory, with a barrier each (15 of 55 steps for 1,024 words, 25 of 78 for
// 4,096).  10,000 sequences, d = 1: 18 us instead of about 70 for verify,
// sort passes and dedup; with every candidate verified and sorted it took 61.
// The limit is the table: 4,096 words in half of 64 KB.
constexpr int SR_THREADS = 1024;

// Sorts the block's SR_THREADS * K words, thread t holding words t + k *
// SR_THREADS; s_w: two buffers of SR_THREADS words for the exchanges.
template <int K>
__device__ __forceinline__ void block_sort(uint64_t (&r)[K], uint64_t* s_w) {
  const uint32_t t = threadIdx.x;
  uint32_t flip = 0;
  for (uint32_t size = 2; size <= (uint32_t)(SR_THREADS * K); size <<= 1) {
    for (uint32_t step = size >> 1; step > 0; step >>= 1) {
      if (step >= SR_THREADS) {  // between the thread's own words
        const int ks = (int)(step / SR_THREADS);
#pragma unroll
        for (int x = 0; x < K; ++x) {
#pragma unroll
          for (int y = x + 1; y < K; ++y) {
            if (y != (x ^ ks)) continue;
            const bool up = ((x * SR_THREADS + t) & size) == 0;
            const uint64_t lo = min(r[x], r[y]), hi = max(r[x], r[y]);
            r[x] = up ? lo : hi;
            r[y] = up ? hi : lo;
          }
        }
        continue;
      }
#pragma unroll
      for (int k = 0; k < K; ++k) {
        uint64_t o;
        if (step < 32) {
          o = __shfl_xor_sync(FULL_MASK, r[k], step);
        } else {
          // two buffers in turn: a barrier between a word's write and its
          // read also lies between that read and the buffer's next write
          uint64_t* buf = s_w + (flip & 1u) * SR_THREADS;
          ++flip;
          buf[t] = r[k];
          __syncthreads();
          o = buf[t ^ step];
        }
        const bool up = ((k * SR_THREADS + t) & size) == 0, low = (t & step) == 0;
        r[k] = up == low ? min(r[k], o) : max(r[k], o);
      }
    }
  }
}

// Words s_w[0, m) in order, as rows.
template <int K>
__device__ __forceinline__ void sorted_rows(const uint64_t* s_w, uint64_t* s_buf, uint32_t m,
                                            uint32_t j_bits, xtn_triple* __restrict__ rows,
                                            int64_t row_cap) {
  uint64_t r[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const uint32_t x = threadIdx.x + k * SR_THREADS;
    r[k] = x < m ? s_w[x] : ~0ull;
  }
  block_sort<K>(r, s_buf);
  const uint64_t jmask = (1ull << j_bits) - 1ull;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const uint32_t x = threadIdx.x + k * SR_THREADS;
    if (x < m && (int64_t)x < row_cap) {
      xtn_triple t;
      t.i = (uint32_t)(r[k] >> 2 >> j_bits);
      t.j = (uint32_t)(r[k] >> 2 & jmask);
      t.dist = (uint32_t)(r[k] & 3u);
      rows[x] = t;
    }
  }
}

__device__ __forceinline__ void sorted_rows(const uint64_t* s_w, uint64_t* s_buf, uint32_t m,
                                            uint32_t j_bits, xtn_triple* __restrict__ rows,
                                            int64_t row_cap) {
  if (m <= SR_THREADS)
    sorted_rows<1>(s_w, s_buf, m, j_bits, rows, row_cap);
  else if (m <= 2 * SR_THREADS)
    sorted_rows<2>(s_w, s_buf, m, j_bits, rows, row_cap);
  else
    sorted_rows<4>(s_w, s_buf, m, j_bits, rows, row_cap);
}

// Shared memory, in words: the hash table (later the sort's exchange
// buffers), the rows' words.
constexpr uint32_t SR_SLOTS = 2 * (uint32_t)SMALL_PAIRS;  // at most half full
constexpr size_t SR_SMEM = (SR_SLOTS + SMALL_PAIRS) * 8;

// Puts w in the table; whether it was not there.  Fewer than SR_SLOTS words
// ever go in, so the search ends.
__device__ __forceinline__ bool first_of(uint64_t* s_slot, uint64_t w) {
  uint32_t h = (uint32_t)((w * HASH_B) >> 32) % SR_SLOTS;
  for (;;) {
    const uint64_t old = atomicCAS(reinterpret_cast<unsigned long long*>(s_slot + h), ~0ull,
                                   (unsigned long long)w);
    if (old == w) return false;
    if (old == ~0ull) return true;
    h = (h + 1) % SR_SLOTS;
  }
}

__global__ void __launch_bounds__(SR_THREADS)
    k_small_rows(const uint64_t* __restrict__ cand, uint32_t n, uint32_t j_bits, PairSide si,
                 PairSide sj, const uint32_t* __restrict__ seq_rep, int self_mode, int d,
                 int metric, xtn_triple* __restrict__ rows, int64_t row_cap,
                 uint64_t* __restrict__ n_rows, uint32_t* __restrict__ err) {
  static_assert(SMALL_PAIRS == 4 * SR_THREADS, "up to four words a thread");
  extern __shared__ uint64_t s_slot[];
  uint64_t* s_w = s_slot + SR_SLOTS;  // pair << 2 | distance (at most 3)
  __shared__ uint32_t s_n;
  if (threadIdx.x == 0) s_n = 0;
  for (uint32_t k = threadIdx.x; k < SR_SLOTS; k += SR_THREADS) s_slot[k] = ~0ull;
  __syncthreads();
  for (uint32_t t0 = threadIdx.x & ~31u; t0 < n; t0 += SR_THREADS) {
    const uint32_t t = t0 + lane_id();
    uint64_t w = 0;
    uint32_t dist = 0;
    bool ok = false;
    if (t < n) {
      w = cand[t];  // not ~0: two bits are free above the pair
      ok = first_of(s_slot, w) &&
           verified(w, j_bits, si, sj, seq_rep, self_mode, d, metric, err, dist);
    }
    const uint32_t bal = __ballot_sync(FULL_MASK, ok);
    uint32_t at = 0;
    if (lane_id() == 0 && bal) at = atomicAdd(&s_n, (uint32_t)__popc(bal));
    at = __shfl_sync(FULL_MASK, at, 0) + __popc(bal & ((1u << lane_id()) - 1u));
    if (ok) s_w[at] = w << 2 | dist;  // at < n <= SMALL_PAIRS
  }
  __syncthreads();
  const uint32_t m = s_n;
  if (threadIdx.x == 0) *n_rows = m;
  sorted_rows(s_w, s_slot, m, j_bits, rows, row_cap);
}

void launch_small_rows(const uint64_t* cand, uint64_t n, uint32_t j_bits, const PairSide& si,
                       const PairSide& sj, const uint32_t* seq_rep, int self_mode, int d,
                       int metric, xtn_triple* rows, int64_t row_cap, uint64_t* n_rows,
                       uint32_t* err, cudaStream_t s) {
  static PerDevice shared;
  shared([] { return allow_shared((const void*)k_small_rows, (int)SR_SMEM, false); });
  prof_begin(s, "k_small_rows", (double)n * (8.0 + 2 * 32.0));
  k_small_rows<<<1, SR_THREADS, SR_SMEM, s>>>(cand, (uint32_t)n, j_bits, si, sj, seq_rep,
                                              self_mode, d, metric, rows, row_cap, n_rows, err);
  prof_end(s);
}

// -------------------------------------------------------- medium results ---
// The verified words lie grouped by their top 8 pair bits (one pass of the
// pair sort); a block takes a group of them, strips its duplicates, sorts the
// rest and writes the rows behind those of the groups before it.  Up to a
// million words or two the pair sort's further passes and the dedup are
// mostly latency, about 10 us a launch whatever the size.  Sort and dedup
// before, and now: 10,000 queries (230,000 candidates) 63 + 14 and 12 + 21
// us, 200,000 sequences (720,000) 68 + 14 and 12 + 29, overlap of 500,000
// (1.9 M) 94 + 14 and 14 + 27.  A group of more than 2,048 rows (300,000 to
// 500,000 sequences of one repertoire) takes the sort of four words a thread:
// 78 to 98 + 14 to 22 and 13 to 16 + 82 to 86.  A group with more distinct
// words than a block holds sets DERR_CAPACITY (the caller sorts).
__global__ void __launch_bounds__(SR_THREADS)
    k_bucket_rows(const uint64_t* __restrict__ words, const uint64_t* __restrict__ n_words,
                  const uint64_t* __restrict__ starts, uint32_t pair_bits, uint32_t j_bits,
                  xtn_triple* __restrict__ rows, int64_t row_cap, uint64_t* __restrict__ status,
                  uint32_t* __restrict__ ctr, uint64_t* __restrict__ n_rows,
                  uint32_t* __restrict__ err) {
  extern __shared__ uint64_t s_slot[];
  uint64_t* s_w = s_slot + SR_SLOTS;
  __shared__ uint32_t s_n, s_tile;
  __shared__ uint64_t s_prefix;
  if (threadIdx.x == 0) s_n = 0;
  for (uint32_t k = threadIdx.x; k < SR_SLOTS; k += SR_THREADS) s_slot[k] = ~0ull;
  const uint32_t b = tile_id(ctr, &s_tile);  // a barrier: the table is clear
  const uint64_t all = *n_words;
  const uint64_t p = min(starts[b], all), q = b + 1 < RADIX ? min(starts[b + 1], all) : all;
  const uint64_t pair_mask = (1ull << pair_bits) - 1ull;
  for (uint64_t t0 = p + (threadIdx.x & ~31u); t0 < q; t0 += SR_THREADS) {
    // one lane reads the counter that other warps add to: a warp whose lanes
    // read different values would part here, before the ballot of all 32
    uint32_t listed = 0;
    if (lane_id() == 0) listed = *(volatile uint32_t*)&s_n;
    if (__shfl_sync(FULL_MASK, listed, 0) > SMALL_PAIRS) break;  // at most 1,024 more go in
    const uint64_t t = t0 + lane_id();
    uint64_t w = 0;
    bool first = false;
    if (t < q) {
      w = words[t];
      w = (w & pair_mask) << 2 | (w >> pair_bits & 3u);
      first = first_of(s_slot, w);
    }
    const uint32_t bal = __ballot_sync(FULL_MASK, first);
    uint32_t at = 0;
    if (lane_id() == 0 && bal) at = atomicAdd(&s_n, (uint32_t)__popc(bal));
    at = __shfl_sync(FULL_MASK, at, 0) + __popc(bal & ((1u << lane_id()) - 1u));
    if (first && at < SMALL_PAIRS) s_w[at] = w;
  }
  __syncthreads();
  const uint32_t m = min(s_n, (uint32_t)SMALL_PAIRS);
  if (threadIdx.x == 0 && s_n > SMALL_PAIRS) atomicOr(err, DERR_CAPACITY);
  if (threadIdx.x < 32) {
    const uint64_t pre = warp_lookback(status, b, m, err);
    if (threadIdx.x == 0) {
      s_prefix = pre;
      if (b + 1 == RADIX) *n_rows = pre + m;
    }
  }
  __syncthreads();
  const int64_t pre = (int64_t)s_prefix;
  sorted_rows(s_w, s_slot, m, j_bits, rows + pre, row_cap - pre);
}

size_t bucket_rows_status_bytes() { return RADIX * 8 + 16; }

void launch_bucket_rows(const uint64_t* words, uint64_t n_max, const uint64_t* n_words,
                        const uint64_t* starts, uint32_t pair_bits, uint32_t j_bits,
                        xtn_triple* rows, int64_t row_cap, uint64_t* status, uint64_t* n_rows, uint32_t* err, cudaStream_t s) {
  static PerDevice shared;
  shared([] { return allow_shared((const void*)k_bucket_rows, (int)SR_SMEM, false); });
  prof_begin(s, "k_unique_finalize", (double)n_max * 8.0);
  k_bucket_rows<<<RADIX, SR_THREADS, SR_SMEM, s>>>(words, n_words, starts, pair_bits, j_bits, rows,
                                                   row_cap, status,
                                                   reinterpret_cast<uint32_t*>(status + RADIX),
                                                   n_rows, err);
  prof_end(s);
}

// ------------------------------------------------------------- TCRdist ---
// BLOSUM62 (Henikoff & Henikoff 1992), rows and columns in residue-code order
// A C D E F G H I K L M N P Q R S T V W Y.
__constant__ int8_t c_blosum62[20][20] = {
    /*A*/ {4, 0, -2, -1, -2, 0, -2, -1, -1, -1, -1, -2, -1, -1, -1, 1, 0, 0, -3, -2},
    /*C*/ {0, 9, -3, -4, -2, -3, -3, -1, -3, -1, -1, -3, -3, -3, -3, -1, -1, -1, -2, -2},
    /*D*/ {-2, -3, 6, 2, -3, -1, -1, -3, -1, -4, -3, 1, -1, 0, -2, 0, -1, -3, -4, -3},
    /*E*/ {-1, -4, 2, 5, -3, -2, 0, -3, 1, -3, -2, 0, -1, 2, 0, 0, -1, -2, -3, -2},
    /*F*/ {-2, -2, -3, -3, 6, -3, -1, 0, -3, 0, 0, -3, -4, -3, -3, -2, -2, -1, 1, 3},
    /*G*/ {0, -3, -1, -2, -3, 6, -2, -4, -2, -4, -3, 0, -2, -2, -2, 0, -2, -3, -2, -3},
    /*H*/ {-2, -3, -1, 0, -1, -2, 8, -3, -1, -3, -2, 1, -2, 0, 0, -1, -2, -3, -2, 2},
    /*I*/ {-1, -1, -3, -3, 0, -4, -3, 4, -3, 2, 1, -3, -3, -3, -3, -2, -1, 3, -3, -1},
    /*K*/ {-1, -3, -1, 1, -3, -2, -1, -3, 5, -2, -1, 0, -1, 1, 2, 0, -1, -2, -3, -2},
    /*L*/ {-1, -1, -4, -3, 0, -4, -3, 2, -2, 4, 2, -3, -3, -2, -2, -2, -1, 1, -2, -1},
    /*M*/ {-1, -1, -3, -2, 0, -3, -2, 1, -1, 2, 5, -2, -2, 0, -1, -1, -1, 1, -1, -1},
    /*N*/ {-2, -3, 1, 0, -3, 0, 1, -3, 0, -3, -2, 6, -2, 0, 0, 1, 0, -3, -4, -2},
    /*P*/ {-1, -3, -1, -1, -4, -2, -2, -3, -1, -3, -2, -2, 7, -1, -2, -1, -1, -2, -4, -3},
    /*Q*/ {-1, -3, 0, 2, -3, -2, 0, -3, 1, -2, 0, 0, -1, 5, 1, 0, -1, -2, -2, -1},
    /*R*/ {-1, -3, -2, 0, -3, -2, 0, -3, 2, -2, -1, 0, -2, 1, 5, -1, -1, -3, -3, -2},
    /*S*/ {1, -1, 0, 0, -2, 0, -1, -2, 0, -2, -1, 1, -1, 0, -1, 4, 1, -2, -3, -2},
    /*T*/ {0, -1, -1, -1, -2, -2, -2, -1, -1, -1, -1, 0, -1, -1, -1, 1, 5, 0, -2, -2},
    /*V*/ {0, -1, -3, -2, -1, -3, -3, 3, -2, 1, 1, -3, -2, -2, -3, -2, 0, 4, -3, -1},
    /*W*/ {-3, -2, -4, -3, 1, -2, -2, -3, -3, -2, -1, -4, -4, -2, -3, -3, -2, -3, 11, 2},
    /*Y*/ {-2, -2, -3, -2, 3, -3, 2, -1, -2, -1, -1, -2, -3, -1, -2, -2, -2, -1, 2, 7},
};

// TCRdist-style CDR3 score: gaps after the first floor(m/2) residues of the
// shorter sequence, mismatch cost min(4, 4 - BLOSUM62), gap cost 4, weight 3.
// cost: the mismatch costs by residue codes, 32 bytes a row.
__device__ __forceinline__ int tcrdist_score(const uint8_t* cost, const Key128& a, int la,
                                             const Key128& b, int lb) {
  const bool a_short = la <= lb;
  const Key128 s = a_short ? a : b;
  const Key128 l = a_short ? b : a;
  const int m = a_short ? la : lb;
  const int g = (a_short ? lb : la) - m;
  int sum = 4 * g;
  // the halves before and behind the gaps, residue by residue off the keys
  auto half = [&](Key128 x, Key128 y, int count) {
    for (int k = 0; k < count; ++k) {
      sum += cost[((uint32_t)x.lo & 31u) << 5 | ((uint32_t)y.lo & 31u)];
      x.lo = (x.lo >> 5) | (x.hi << 59);
      x.hi >>= 5;
      y.lo = (y.lo >> 5) | (y.hi << 59);
      y.hi >>= 5;
    }
  };
  const int p = m / 2;
  half(s, l, p);
  half(shr128(s, 5 * p), shr128(l, 5 * (p + g)), m - p);
  return 3 * sum;
}

// ITEMS rows a thread, in the order of the input.  `out` is left alone when
// the encoder has found a bad letter, length or offset.
template <int ITEMS>
__global__ void __launch_bounds__(VER_THREADS)
    k_tcrdist_filter(const xtn_triple* __restrict__ in, int64_t n, const Key128* __restrict__ keys,
                     const uint8_t* __restrict__ lens, int64_t n_seq, int max_score,
                     xtn_triple* __restrict__ out, uint64_t* __restrict__ status,
                     uint32_t* __restrict__ ctr, uint32_t* __restrict__ err,
                     uint64_t* __restrict__ total_out) {
  constexpr int TILE = VER_THREADS * ITEMS;
  __shared__ uint8_t s_cost[32 * 32];
  __shared__ uint32_t s_tile;
  __shared__ uint32_t s_w[VER_THREADS / 32];
  __shared__ uint64_t s_prefix;
  // codes 0 (a letter outside the alphabet: the call reports it) and past 20
  // cost like a gap
  for (int k = threadIdx.x; k < 32 * 32; k += VER_THREADS) {
    const int x = k >> 5, y = k & 31;
    s_cost[k] = x == y ? 0
                : x >= 1 && x <= 20 && y >= 1 && y <= 20
                    ? (uint8_t)min(4, 4 - (int)c_blosum62[x - 1][y - 1])
                    : 4;
  }
  // (a row out of range, which other blocks may report by now, spoils `out` anyway)
  const bool failed = *(volatile uint32_t*)err != 0;
  const uint32_t tile = tile_id(ctr, &s_tile);  // a barrier: the costs are complete
  const int64_t tbase = (int64_t)tile * TILE;
  const int64_t base = tbase + (int64_t)threadIdx.x * ITEMS;
  uint32_t keep = 0, cnt = 0;
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const int64_t p = base + it;
    if (p < n) {
      const xtn_triple t = in[p];
      bool ok = false;
      if (t.i < n_seq && t.j < n_seq) {
        ok = tcrdist_score(s_cost, keys[t.i], lens[t.i], keys[t.j], lens[t.j]) <= max_score;
      } else {
        atomicOr(err, DERR_RANGE);
      }
      keep |= (uint32_t)ok << it;
      cnt += ok;
    }
  }
  uint32_t excl;
  const uint32_t total = block_excl_scan_u32<VER_THREADS>(cnt, s_w, excl);
  if (threadIdx.x < 32) {
    const uint64_t pre = warp_lookback(status, tile, total, err);
    if (threadIdx.x == 0) {
      s_prefix = pre;
      if (tbase + TILE >= n) *total_out = pre + total;
    }
  }
  __syncthreads();
  int64_t o = (int64_t)(s_prefix + excl);
#pragma unroll
  for (int it = 0; it < ITEMS; ++it)
    if (keep >> it & 1u) {
      if (o < n && !failed) out[o] = in[base + it];
      ++o;
    }
}

void launch_tcrdist_filter(const xtn_triple* in, int64_t n, const Key128* keys,
                           const uint8_t* lens, int64_t n_seq, int max_score, xtn_triple* out,
                           uint64_t* status, uint32_t* err, uint64_t* total, cudaStream_t s) {
  if (n <= 0) return;
  const size_t st = verify_status_bytes(n);
  uint32_t* ctr = reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(status) + st - 16);
  // one row a thread while the blocks fit the chip at once: 11,700 rows on 6
  // blocks took 37 us, most of it the serial walk of eight rows; past it
  // eight rows amortise the look-back
  const bool few = n <= FEW_ROWS;
  static_assert(VER_TILE == VERIFY_TILE && VER_THREADS == VERIFY_TILE / 8,
                "the status is sized for both");
  cudaMemsetAsync(status, 0, st, s);
  prof_begin(s, "k_tcrdist_filter", (double)n * (12.0 * 2 + 2 * 17.0));
  if (few)
    k_tcrdist_filter<1><<<div_up_u32(n, VER_THREADS), VER_THREADS, 0, s>>>(
        in, n, keys, lens, n_seq, max_score, out, status, ctr, err, total);
  else
    k_tcrdist_filter<VER_ITEMS><<<div_up_u32(n, VER_TILE), VER_THREADS, 0, s>>>(
        in, n, keys, lens, n_seq, max_score, out, status, ctr, err, total);
  prof_end(s);
}

}  // namespace xtn
