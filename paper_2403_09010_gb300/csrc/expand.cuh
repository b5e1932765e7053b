// Canonical deletion variants as sums of per-position terms.
//
// With the prefix sums P of the polynomial fingerprint (xtn_common.cuh) and
// Q = B^-1 P, R = B^-2 P, S = B^-3 P, the fingerprint of a sequence without
// positions p1 < p2 < p3 splits into one term per deleted position:
//   H = (P[p1] - Q[p1+1]) + (Q[p2] - R[p2+1]) + (R[p3] - S[p3+1]) + S[L]
//     =        Y[p1]      +        M[p2]      +        Z[p3]
// (S[L] is added to every Y; for at most two deletions R[L] is, and Z falls
// away).  A missing deletion sits at the end of the sequence, which gives
// the sentinel terms M[L] = Q[L] - R[L] and Z[L] = R[L] - S[L].  So a warp
// prepares the terms of a few sequences once (about ten instructions per
// record at d = 2) and a record then costs two or three shared-memory loads
// and one or two 64-bit additions, where evaluating the polynomial took two
// 64-bit multiplies and five loads.
//
// The terms are kept by run of equal residues: every position of a run has
// the same M and the same Z (Q grows by what R loses), as deleting any of
// its residues gives one string.  A variant is therefore a choice of runs,
// repeated at most as often as the run is long, in ascending order, the
// sentinel (run index R, "no deletion") filling up to d:
//   d = 2: v < C(R+1, 2)  : runs a < b <= R in colex order, Y[a] + M[b]
//          then           : (R, R), and (a, a) for each run of two or more
//   d = 3: v < C(R+1, 3)  : runs a < b < c <= R, Y[a] + M[b] + Z[c]
//          then           : (a, R, R) for a <= R; (a, a, a) for each run of
//                           three or more; (k, k, o) in ascending order for
//                           each run k of two or more and each o != k, o <= R
//   d = 1: one run (R of them), none -- their sums stored outright.
// The first kind comes from one table of combinations, the second from a
// short list of the sequence's own ("extra"), both as the same packed run
// indices.  Exactly the distinct variant strings are numbered
// (canonical_total), so no lane computes a variant that is thrown away.
// Paired receptors are the joined string alpha + token + beta with the runs
// of both chains.
#pragma once

#include <type_traits>

#include "xtn_common.cuh"
#include "xtn_kernels.h"

namespace xtn {

enum { VK_D1 = 0, VK_D2, VK_D3, VK_PAIRED_D1, VK_PAIRED_D2 };

constexpr uint32_t TOKEN_CODE = 21;  // between two chains; outside the residue codes 1..20

// PACK: sequences a warp prepares at once; LANES lanes share one sequence's
// PER-position chunks.
template <int KIND>
struct VK {
  static constexpr bool PAIRED = KIND >= VK_PAIRED_D1;
  static constexpr int D = KIND == VK_D3 ? 3 : (KIND == VK_D2 || KIND == VK_PAIRED_D2) ? 2 : 1;
  static constexpr int POS = PAIRED ? 2 * XTN_MAX_LEN + 1 : XTN_MAX_LEN;
  static constexpr int RUNS = PAIRED ? 2 * XTN_MAX_LEN : XTN_MAX_LEN;
  static constexpr int DBL = PAIRED ? 2 * (XTN_MAX_LEN / 2) : XTN_MAX_LEN / 2;
  static constexpr int PACK = KIND == VK_D1 ? 32 : (KIND == VK_D2 || KIND == VK_PAIRED_D1) ? 8 : 4;
  static constexpr int LANES = 32 / PACK;
  static constexpr int PER = (POS + LANES - 1) / LANES;
  // one sequence's terms (64-bit words), an odd number to spread the banks
  static constexpr int Y = 0;
  static constexpr int M = D >= 2 ? RUNS + 1 : 0;
  static constexpr int Z = D == 3 ? M + RUNS + 1 : M;
  static constexpr int STRIDE = (Z + RUNS + 1) | 1;
  // its extra run choices: d = 2 (R, R) and the long runs; d = 3 the first
  // two lists, then the long runs' indices for the third
  static constexpr int EXTRA = D == 1 ? 0 : D == 2 ? 1 + DBL : RUNS + 1 + RUNS / 3 + DBL;
  // table of combinations over RUNS + 1 run indices
  static constexpr int COMBS = D == 3   ? (RUNS + 1) * RUNS * (RUNS - 1) / 6
                               : D == 2 ? (RUNS + 1) * RUNS / 2
                                        : 0;
};

// Canonical deletion subsets of at most d <= 3 positions (the variants
// prepare_variants numbers) of a sequence of length L; eq: positions equal to
// their left neighbour.
__device__ __forceinline__ uint32_t canonical_total(uint32_t eq, uint32_t L, int d) {
  const uint32_t runs = ~eq & (L ? 0xffffffffu >> (32 - L) : 0u);
  const uint32_t dbl = runs & (eq >> 1);
  const uint32_t R = (uint32_t)__popc(runs), nD = (uint32_t)__popc(dbl);
  uint32_t total = 1u;
  if (d >= 1) total += R;
  if (d >= 2) total += R * (R - 1) / 2 + nD;
  if (d >= 3 && R)
    total += R * (R - 1) * (R - 2) / 6 + nD * (R - 1) + (uint32_t)__popc(dbl & (eq >> 2));
  return total;
}

// Colex tables, made at compile time: t -> a | b << 8 (pairs), or
// a | b << 5 | c << 10 (triples).
template <int N, int K>
struct CombTable {
  static constexpr int SIZE = K == 2 ? N * (N - 1) / 2 : N * (N - 1) * (N - 2) / 6;
  uint16_t v[SIZE];
  constexpr CombTable() : v() {
    int t = 0;
    if (K == 2) {
      for (int b = 1; b < N; ++b)
        for (int a = 0; a < b; ++a) v[t++] = (uint16_t)(a | b << 8);
    } else {
      for (int c = 2; c < N; ++c)
        for (int b = 1; b < c; ++b)
          for (int a = 0; a < b; ++a) v[t++] = (uint16_t)(a | b << 5 | c << 10);
    }
  }
};
static __device__ constexpr CombTable<2 * XTN_MAX_LEN + 1, 2> d_pairs;  // its first words serve any N
static __device__ constexpr CombTable<XTN_MAX_LEN + 1, 3> d_triples;

template <int KIND>
__device__ __forceinline__ void load_combs(uint16_t* s_comb) {
  if constexpr (VK<KIND>::D == 3)
    for (int t = threadIdx.x; t < VK<KIND>::COMBS; t += blockDim.x) s_comb[t] = d_triples.v[t];
  else if constexpr (VK<KIND>::D == 2)
    for (int t = threadIdx.x; t < VK<KIND>::COMBS; t += blockDim.x) s_comb[t] = d_pairs.v[t];
}

// s_pow[k + 3] = B^k for k = -3 .. (B^-1 is an exact inverse), as far as the
// lanes' chunks reach; none for VK_D1, whose powers are constants.
template <int KIND>
constexpr int N_POWERS = KIND == VK_D1 ? 1 : VK<KIND>::PER * VK<KIND>::LANES + 4;
template <int KIND>
__device__ __forceinline__ void load_powers(uint64_t* s_pow) {
  if constexpr (KIND == VK_D1) return;
  for (int k = threadIdx.x; k < N_POWERS<KIND>; k += blockDim.x) {
    uint64_t p = HASH_BINV3;
    for (int e = 0; e < k; ++e) p *= HASH_B;
    s_pow[k] = p;
  }
}

// B^k, a constant where k is one.
__host__ __device__ constexpr uint64_t power_of_b(int k) {
  uint64_t p = 1;
  for (int e = 0; e < k; ++e) p *= HASH_B;
  return p;
}

// The sequences a kernel expands: one chain, or two with `b` fields set.
struct ExpandSource {
  const Key128* keys = nullptr;
  const uint8_t* lens = nullptr;
  const uint32_t* eqprev = nullptr;
  const Key128* keys_b = nullptr;
  const uint8_t* lens_b = nullptr;
  const uint32_t* eq_b = nullptr;
};

// Where a sequence's variants sit in the warp's stream of records: variant
// v = t - adj for stream positions t < end; c: variants that come from the
// combination table (d >= 2); aux: R | (extra choices outright) << 8 (d = 3).
struct __align__(16) VarMeta {
  int32_t end, adj;
  uint32_t c, aux;
};

__device__ __forceinline__ Key128 shl128(const Key128& k, uint32_t s) {
  if (s >= 128) return Key128{0ull, 0ull};
  if (s >= 64) return Key128{0ull, k.lo << (s - 64)};
  if (s == 0) return k;
  return Key128{k.lo << s, (k.hi << s) | (k.lo >> (64 - s))};
}

template <int W>
__device__ __forceinline__ uint64_t group_incl_scan_u64(uint64_t v, uint32_t sub) {
#pragma unroll
  for (int o = 1; o < W; o <<= 1) {
    const uint64_t t = __shfl_up_sync(FULL_MASK, v, o, W);
    if (sub >= (uint32_t)o) v += t;
  }
  return v;
}

// Whole warp: the LANES lanes of this lane's group compute the terms of
// sequence `i` (nothing when !have) and return its number of variants with
// at most d deletions and the fields of its VarMeta but `end` (adj relative
// to the sequence's first variant).  d >= 2: the terms go to `tab` and
// `extra`, and the caller orders those writes (__syncwarp) before they are
// read.  d <= 1: put(a, h) takes the sum of deleting run a, put(R, h) that of
// no deletion.  Codes past the end are zero, so the loops have no bounds.
template <int KIND, class Put>
__device__ __forceinline__ uint32_t prepare_variants(uint64_t* __restrict__ tab,
                                                     uint16_t* __restrict__ extra,
                                                     const uint64_t* __restrict__ s_pow,
                                                     const ExpandSource& src, int64_t i, bool have,
                                                     int d, uint64_t salt, uint32_t lane,
                                                     VarMeta& m, Put put) {
  using K = VK<KIND>;
  const uint32_t sub = lane % K::LANES;
  const int p0 = (int)sub * K::PER;
  // window of residue codes from p0, length, run starts
  Key128 k{0ull, 0ull};
  uint32_t L = 0;
  using Mask = typename std::conditional<K::PAIRED, uint64_t, uint32_t>::type;
  Mask runs = 0, dbl = 0, tri = 0;
  if (have) {
    auto starts = [](uint32_t len, uint32_t eq) {
      return ~eq & (len ? 0xffffffffu >> (32 - len) : 0u);
    };
    const uint32_t La = min((uint32_t)src.lens[i], (uint32_t)XTN_MAX_LEN);
    const uint32_t ea = src.eqprev[i];
    const uint32_t ra = starts(La, ea);
    k = shr128(src.keys[i], 5 * p0);
    if constexpr (K::PAIRED) {
      const uint32_t Lb = min((uint32_t)src.lens_b[i], (uint32_t)XTN_MAX_LEN);
      const uint32_t eb = src.eq_b[i];
      const uint32_t rb = starts(Lb, eb);
      const Key128 kb = src.keys_b[i];
      const Key128 tok{(uint64_t)TOKEN_CODE, 0ull};
      const Key128 t = (uint32_t)p0 <= La ? shl128(tok, 5 * (La - p0)) : Key128{0ull, 0ull};
      const Key128 b = (uint32_t)p0 > La ? shr128(kb, 5 * (p0 - La - 1))
                                         : shl128(kb, 5 * (La + 1 - p0));
      k.lo |= t.lo | b.lo;
      k.hi |= t.hi | b.hi;
      L = La + 1 + Lb;
      runs = (Mask)ra | ((Mask)rb << (La + 1));
      dbl = (Mask)(ra & (ea >> 1)) | ((Mask)(rb & (eb >> 1)) << (La + 1));
    } else {
      L = La;
      runs = ra;
      dbl = ra & (ea >> 1);
      if (K::D == 3) tri = dbl & (ea >> 2);
    }
  }
  auto popc = [](Mask x) -> uint32_t {
    return K::PAIRED ? (uint32_t)__popcll((uint64_t)x) : (uint32_t)__popc((uint32_t)x);
  };
  const uint32_t R = popc(runs), nD = popc(dbl), nT = popc(tri);
  const Mask before = ((Mask)1 << p0) - 1;  // p0 < the mask's width
  uint32_t a = popc(runs & before);
  const uint32_t my_runs = (uint32_t)(runs >> p0);  // PER <= 25 bits of interest
  auto code = [&](int q) -> uint32_t {              // q: a position of the chunk
    const int b = 5 * q;
    if (b + 5 <= 64) return (uint32_t)(k.lo >> b) & 31u;
    if (b >= 64) return (uint32_t)(k.hi >> (b - 64)) & 31u;
    return (uint32_t)((k.lo >> b) | (k.hi << (64 - b))) & 31u;
  };
  if constexpr (KIND == VK_D1) {
    // a lane has its sequence to itself: from one deleted position to the next
    // the sum changes by (c[p] - c[p+1]) B^p, and with the loops unrolled the
    // powers and the codes' shifts are constants: k_expand of 10M sequences
    // 1,000 us, 1,250 with prefix sums by a loop over the longest length
    const uint32_t longest = __reduce_max_sync(FULL_MASK, L);
    uint64_t y = 0;  // the sum without position 0
#pragma unroll
    for (int q = 1; q < XTN_MAX_LEN; ++q) {
      if ((uint32_t)q >= longest) break;  // uniform
      y += (uint64_t)code(q) * power_of_b(q - 1);
    }
    const uint64_t none = y * HASH_B + code(0) + salt;
    y += salt;
#pragma unroll
    for (int q = 0; q < XTN_MAX_LEN; ++q) {
      if ((uint32_t)q >= longest) break;
      if (my_runs >> q & 1u) put(a++, y);
      y += (uint64_t)((int64_t)code(q) - (int64_t)code(q + 1)) * power_of_b(q);
    }
    m.c = m.aux = 0;
    m.adj = d <= 0 ? -(int32_t)R : 0;  // only "none", numbered behind the runs
    if (!have) return 0u;
    put(R, none);
    return d <= 0 ? 1u : R + 1u;
  }
  constexpr int UNROLL = K::PER > 13 ? 5 : K::PER;
  // prefix sums at the chunk's start and at the end
  uint64_t sum = 0;
#pragma unroll UNROLL
  for (int q = 0; q < K::PER; ++q) sum += (uint64_t)code(q) * s_pow[p0 + q + 3];
  const uint64_t incl = group_incl_scan_u64<K::LANES>(sum, sub);
  const uint64_t PL = K::LANES > 1 ? __shfl_sync(FULL_MASK, incl, K::LANES - 1, K::LANES) : incl;
  const uint64_t QL = PL * HASH_BINV, RL = PL * HASH_BINV2;
  const uint64_t SL = K::D == 3 ? PL * HASH_BINV3 : 0ull;
  // what every Y carries
  const uint64_t C = (K::D == 1 ? QL : K::D == 2 ? RL : SL) + salt;
  uint64_t w1 = s_pow[p0 + 1], w2 = s_pow[p0 + 2];  // B^(p-2), B^(p-1)
  // the terms at p: Y - C = P[p] - Q[p+1], M = B^-1 (Y - C), Z = B^-1 M; one
  // position on, Y changes by (c[p] - c[p+1]) B^p, M by B^-1 of that, Z by B^-2
  // (1M sequences, d = 2: k_expand 633 us, 650 with P, Q, R carried along)
  const uint64_t P = incl - sum;
  const uint64_t y0 = P - P * HASH_BINV - (uint64_t)code(0) * w2;
  uint64_t y = y0 + C, mm = K::D >= 2 ? y0 * HASH_BINV : 0ull;
  uint64_t z = K::D == 3 ? mm * HASH_BINV : 0ull;
#pragma unroll UNROLL
  for (int q = 0; q < K::PER; ++q) {
    const uint64_t w3 = s_pow[p0 + q + 3];
    if ((my_runs >> q) & 1u) {
      if constexpr (K::D == 1) {
        put(a, y);
      } else {
        tab[K::Y + a] = y;
        tab[K::M + a] = mm;
        if constexpr (K::D == 3) {
          tab[K::Z + a] = z;
          extra[a] = (uint16_t)(a | R << 5 | R << 10);
        }
      }
      ++a;
    }
    const uint64_t step = (uint64_t)((int64_t)code(q) - (int64_t)code(q + 1));
    y += step * w3;
    if (K::D >= 2) mm += step * w2;
    if (K::D == 3) z += step * w1;
    w1 = w2;
    w2 = w3;
  }
  if constexpr (K::D >= 2) {  // the few long runs that start in this chunk
    for (Mask g = (dbl >> p0) & (((Mask)1 << K::PER) - 1); g; g &= g - 1) {
      const int p = p0 + (K::PAIRED ? __ffsll((long long)g) : __ffs((int)g)) - 1;
      const Mask below = ((Mask)1 << p) - 1;
      const uint32_t run = popc(runs & below);
      if constexpr (K::D == 2) {
        extra[1 + popc(dbl & below)] = (uint16_t)(run * 0x101u);
      } else {
        extra[R + 1 + nT + popc(dbl & below)] = (uint16_t)run;
        if ((tri >> p) & 1u) extra[R + 1 + popc(tri & below)] = (uint16_t)(run * 0x421u);
      }
    }
  }
  if (sub == 0 && have) {  // the sentinel
    if constexpr (K::D == 1) {
      put(R, PL + salt);
    } else {
      tab[K::Y + R] = PL - QL + C;
      tab[K::M + R] = QL - RL;
      if (K::D == 3) tab[K::Z + R] = RL - SL;
      extra[K::D == 2 ? 0 : R] = (uint16_t)(K::D == 2 ? R * 0x101u : R * 0x421u);
    }
  }
  m.c = 0;
  m.aux = 0;
  m.adj = 0;
  if (!have) return 0u;
  if constexpr (K::D == 1) {
    if (d <= 0) {  // only "none", numbered behind the runs
      m.adj = -(int32_t)R;
      return 1u;
    }
    return R + 1u;
  } else if constexpr (K::D == 2) {
    m.c = R * (R + 1) / 2;
    return m.c + 1u + nD;
  } else {
    const uint32_t e = 1u + R + nT;
    m.c = R ? (R + 1) * R * (R - 1) / 6 : 0u;
    m.aux = R | (e << 8);
    return m.c + e + nD * R;
  }
}

// Fingerprint before mixing of variant v of the sequence with terms `tab`.
template <int KIND>
__device__ __forceinline__ uint64_t variant_sum(const uint64_t* __restrict__ tab,
                                                const uint16_t* __restrict__ extra,
                                                const uint16_t* __restrict__ s_comb, uint32_t v,
                                                uint32_t c, uint32_t aux) {
  using K = VK<KIND>;
  if constexpr (K::D == 1) {
    return tab[K::Y + v];
  } else if constexpr (K::D == 2) {
    const uint32_t pr = *(v < c ? s_comb + v : extra + (v - c));
    return tab[K::Y + (pr & 255u)] + tab[K::M + (pr >> 8)];
  } else {
    uint32_t x;
    if (v < c) {
      x = s_comb[v];
    } else {
      const uint32_t R = aux & 255u, e = aux >> 8;
      uint32_t u = v - c;
      if (u < e) {
        x = extra[u];
      } else {
        u -= e;
        const uint32_t q = u / R;
        const uint32_t k = extra[e + q];
        uint32_t o = u - q * R;
        x = o < k ? (o | k << 5 | k << 10) : (k | k << 5 | (o + 1) << 10);
      }
    }
    return tab[K::Y + (x & 31u)] + tab[K::M + ((x >> 5) & 31u)] + tab[K::Z + (x >> 10)];
  }
}

}  // namespace xtn
