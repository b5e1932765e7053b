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
// Only run starts are deleted first (a run of equal residues gives one
// string whichever of its residues goes), so the terms are kept by run
// index, and the canonical subsets are numbered so that one table of
// combinations serves all of them, the sentinel being run index R:
//   d = 2: v < C(R+1, 2)  : runs a < b <= R in colex order, Y[a] + M[b]
//          then           : none; the first two residues of each long run
//   d = 3: v < C(R+1, 3)  : runs a < b < c <= R, Y[a] + M[b] + Z[c]
//          then           : none; one run; the first two residues of a long
//                           run; the first three of a run of three or more
//          then           : the first two of a long run k and another run o
//   d = 1: one run (R of them), none -- stored outright.
// Exactly the distinct variant strings are numbered (canonical_total), so no
// lane computes a variant that is thrown away.  Paired receptors are the
// joined string alpha + token + beta with the runs of both chains.
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
  // one sequence's terms (64-bit words)
  static constexpr int Y = 0;
  static constexpr int M = D >= 2 ? RUNS : 0;
  static constexpr int Z = M + (D >= 2 ? RUNS + 1 : 0);
  static constexpr int ZERO = Z + (D == 3 ? RUNS + 1 : 0);
  static constexpr int E = ZERO + (D >= 2 ? 1 : 0);
  static constexpr int N_E = D == 1 ? RUNS + 1 : D == 2 ? 1 + DBL : 1 + RUNS + DBL + RUNS / 3;
  static constexpr int DL = E + N_E;
  static constexpr int DR = DL + (D == 3 ? DBL : 0);
  static constexpr int DRUN = DR + (D == 3 ? DBL : 0);
  static constexpr int STRIDE = (DRUN + (D == 3 ? DBL : 0)) | 1;  // odd: spreads the banks
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

// s_pow[k + 3] = B^k for k = -3 .. POS (B^-1 is an exact inverse).
template <int KIND>
__device__ __forceinline__ void load_powers(uint64_t* s_pow) {
  for (int k = threadIdx.x; k < VK<KIND>::POS + 4; k += blockDim.x) {
    uint64_t p = HASH_BINV3;
    for (int e = 0; e < k; ++e) p *= HASH_B;
    s_pow[k] = p;
  }
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
// combination table (d >= 2); aux: R | (words in E) << 8 (d = 3).
struct __align__(16) VarMeta {
  int32_t end, adj;
  uint32_t c, aux;
};

__device__ __forceinline__ Key128 shr128(const Key128& k, uint32_t s) {
  if (s >= 128) return Key128{0ull, 0ull};
  if (s >= 64) return Key128{k.hi >> (s - 64), 0ull};
  if (s == 0) return k;
  return Key128{(k.lo >> s) | (k.hi << (64 - s)), k.hi >> s};
}
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

// Whole warp: the LANES lanes of this lane's group write the terms of
// sequence `i` (nothing when !have) to `tab` and return its number of
// variants with at most d deletions and the fields of its VarMeta but `end`
// (adj relative to the sequence's first variant).  The caller orders the
// writes (__syncwarp) before they are read.
template <int KIND>
__device__ __forceinline__ uint32_t prepare_variants(uint64_t* __restrict__ tab,
                                                     const uint64_t* __restrict__ s_pow,
                                                     const ExpandSource& src, int64_t i, bool have,
                                                     int d, uint64_t salt, uint32_t lane,
                                                     VarMeta& m) {
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
  // prefix sums at the chunk's start and at the end
  const uint32_t pe = min((uint32_t)(p0 + K::PER), L);
  uint64_t sum = 0;
  {
    Key128 w = k;
    for (uint32_t p = p0; p < pe; ++p) {
      sum += (uint64_t)((uint32_t)w.lo & 31u) * s_pow[p + 3];
      w.lo = (w.lo >> 5) | (w.hi << 59);
      w.hi >>= 5;
    }
  }
  const uint64_t incl = group_incl_scan_u64<K::LANES>(sum, sub);
  const uint64_t PL = K::LANES > 1 ? __shfl_sync(FULL_MASK, incl, K::LANES - 1, K::LANES) : incl;
  const uint64_t QL = PL * HASH_BINV, RL = PL * HASH_BINV2;
  const uint64_t SL = K::D == 3 ? PL * HASH_BINV3 : 0ull;
  uint64_t P = incl - sum, Q = P * HASH_BINV, Rr = K::D >= 2 ? P * HASH_BINV2 : 0ull;
  uint64_t S = K::D == 3 ? P * HASH_BINV3 : 0ull;
  // what every Y carries
  const uint64_t C = (K::D == 1 ? QL : K::D == 2 ? RL : SL) + salt;
  for (uint32_t p = p0; p < pe; ++p) {
    const uint64_t s0 = (uint32_t)k.lo & 31u;
    const uint64_t Pn = P + s0 * s_pow[p + 3];
    const uint64_t Qn = Q + s0 * s_pow[p + 2];
    const uint64_t Rn = K::D >= 2 ? Rr + s0 * s_pow[p + 1] : 0ull;
    const uint64_t Sn = K::D == 3 ? S + s0 * s_pow[p] : 0ull;
    if ((runs >> p) & 1u) {
      const Mask below = ((Mask)1 << p) - 1;
      const uint32_t a = popc(runs & below);
      const uint64_t y = P - Qn + C;
      if constexpr (K::D == 1) {
        tab[K::E + a] = y;
      } else {
        const uint64_t m = Q - Rn;
        tab[K::Y + a] = y;
        tab[K::M + a] = m;
        if (K::D == 3) {
          tab[K::Z + a] = Rr - Sn;
          tab[K::E + 1 + a] = y - SL + QL;  // this run alone
        }
        if ((dbl >> p) & 1u) {
          const uint32_t kd = popc(dbl & below);
          // the run's next residue is the same code: terms at p + 1 (and p + 2)
          const uint64_t m1 = Qn - (Rn + s0 * s_pow[p + 2]);
          if constexpr (K::D == 2) {
            tab[K::E + 1 + kd] = y + m1;
          } else {
            const uint64_t R2 = Rn + s0 * s_pow[p + 2], S2 = Sn + s0 * s_pow[p + 1];
            tab[K::E + 1 + R + kd] = y + m1 + (RL - SL);
            tab[K::DL + kd] = m + (Rn - S2);
            tab[K::DR + kd] = y + m1;
            tab[K::DRUN + kd] = a;
            if ((tri >> p) & 1u)
              tab[K::E + 1 + R + nD + popc(tri & below)] = y + m1 + (R2 - (S2 + s0 * s_pow[p + 2]));
          }
        }
      }
    }
    P = Pn;
    Q = Qn;
    Rr = Rn;
    S = Sn;
    k.lo = (k.lo >> 5) | (k.hi << 59);
    k.hi >>= 5;
  }
  if (sub == 0 && have) {
    if constexpr (K::D == 1) {
      tab[K::E + R] = PL + salt;
    } else {
      tab[K::ZERO] = 0ull;
      tab[K::E] = PL + salt;
      if (K::D == 2) tab[K::M + R] = QL - RL;
      if (K::D == 3) tab[K::Z + R] = RL - SL;
    }
  }
  m.c = 0;
  m.aux = 0;
  m.adj = 0;
  if (!have) return 0u;
  if constexpr (K::D == 1) {
    if (d <= 0) {  // only "none", stored behind the runs
      m.adj = -(int32_t)R;
      return 1u;
    }
    return R + 1u;
  } else if constexpr (K::D == 2) {
    m.c = R * (R + 1) / 2;
    return m.c + 1u + nD;
  } else {
    const uint32_t e = 1u + R + nD + nT;
    m.c = R ? (R + 1) * R * (R - 1) / 6 : 0u;
    m.aux = R | (e << 8);
    return m.c + e + (R ? nD * (R - 1) : 0u);
  }
}

// Fingerprint before mixing of variant v of the sequence with terms `tab`.
template <int KIND>
__device__ __forceinline__ uint64_t variant_sum(const uint64_t* __restrict__ tab,
                                                const uint16_t* __restrict__ s_comb, uint32_t v,
                                                uint32_t c, uint32_t aux) {
  using K = VK<KIND>;
  if constexpr (K::D == 1) {
    return tab[K::E + v];
  } else if constexpr (K::D == 2) {
    const bool in = v < c;
    const uint32_t pr = s_comb[in ? v : 0u];
    const uint32_t a = in ? (pr & 255u) + K::Y : v - c + K::E;
    const uint32_t b = in ? (pr >> 8) + K::M : (uint32_t)K::ZERO;
    return tab[a] + tab[b];
  } else {
    const bool in = v < c;
    const uint32_t pr = s_comb[in ? v : 0u];
    uint32_t a = (pr & 31u) + K::Y, b = ((pr >> 5) & 31u) + K::M, z = (pr >> 10) + K::Z;
    if (!in) {
      const uint32_t R = aux & 255u, e = aux >> 8;
      uint32_t u = v - c;
      z = K::ZERO;
      if (u < e) {
        a = K::E + u;
        b = K::ZERO;
      } else {
        u -= e;
        const uint32_t k = u / (R - 1), o = u - k * (R - 1);
        if (o < (uint32_t)tab[K::DRUN + k]) {
          a = K::Y + o;
          b = K::DL + k;
        } else {
          a = K::DR + k;
          b = K::Z + o + 1;
        }
      }
    }
    return tab[a] + tab[b] + tab[z];
  }
}

}  // namespace xtn
