// Paired chains (Discussion: the CDR3s of both chains joined by a
// non-deletable token).  A receptor is the string alpha + token + beta; its
// deletion variants delete up to d residues of either chain and never the
// token, and two receptors' distance is the edit distance of those strings
// with the token never deleted, inserted or substituted -- the two tokens
// always face each other, so the distance is Lev(alpha_i, alpha_j) +
// Lev(beta_i, beta_j) (computed in k_verify.cu, metric 2).
//
//   k_paired_counts : canonical variants per receptor (d <= 2): the token
//                     separates the chains, so the runs of equal residues
//                     are those of alpha plus those of beta, and the count
//                     is 1 + R + C(R, 2) + nD over both chains together.
// The expansion itself is k_expand's (expand.cuh, VK_PAIRED_*): the joined
// residue codes, token code 21 included, are fingerprinted as one string, so
// equal receptor variants meet in one group.
#include "xtn_common.cuh"
#include "xtn_kernels.h"

namespace xtn {

namespace {

__device__ __forceinline__ uint32_t runs_of(uint32_t L, uint32_t eq) {
  const uint32_t all = L ? (0xffffffffu >> (32 - L)) : 0u;
  return ~eq & all;
}

// Canonical variants with at most d <= 2 deletions of a receptor.
__device__ __forceinline__ uint32_t paired_count(uint32_t La, uint32_t eqa, uint32_t Lb,
                                                 uint32_t eqb, int d) {
  const uint32_t ra = runs_of(La, eqa), rb = runs_of(Lb, eqb);
  const uint32_t R = (uint32_t)(__popc(ra) + __popc(rb));
  const uint32_t nD = (uint32_t)(__popc(ra & (eqa >> 1)) + __popc(rb & (eqb >> 1)));
  if (d <= 0) return 1u;
  if (d == 1) return 1u + R;
  return 1u + R + R * (R - 1) / 2 + nD;
}

__global__ void k_paired_counts(const uint8_t* __restrict__ lens_a,
                                const uint32_t* __restrict__ eq_a,
                                const uint8_t* __restrict__ lens_b,
                                const uint32_t* __restrict__ eq_b, int64_t n, int d,
                                uint32_t* __restrict__ vcount) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  vcount[i] = paired_count(min((uint32_t)lens_a[i], (uint32_t)XTN_MAX_LEN), eq_a[i],
                           min((uint32_t)lens_b[i], (uint32_t)XTN_MAX_LEN), eq_b[i], d);
}

}  // namespace

void launch_paired_counts(const uint8_t* lens_a, const uint32_t* eq_a, const uint8_t* lens_b,
                          const uint32_t* eq_b, int64_t n, int d, uint32_t* vcount,
                          cudaStream_t s) {
  if (n <= 0) return;
  prof_begin(s, "k_paired_counts", (double)n * 14.0);
  k_paired_counts<<<div_up_u32(n, 256), 256, 0, s>>>(lens_a, eq_a, lens_b, eq_b, n, d, vcount);
  prof_end(s);
}

}  // namespace xtn
