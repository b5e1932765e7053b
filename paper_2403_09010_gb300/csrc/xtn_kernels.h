// Host-side launchers of the sm_103a kernels (one translation unit each) and
// the constants they share.  All launches are asynchronous on stream `s`.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <stdint.h>

#include "xtn.h"

namespace xtn {

struct Key128;
struct PlaneRow;

constexpr int RADIX = 256;       // 8-bit digits
constexpr int MAX_PASSES = 8;    // 64-bit keys

// api.cu: tuning knobs
std::atomic<int>& cfg_records();
std::atomic<int>& cfg_pairs();

// k_variants.cu ------------------------------------------------------------
void launch_encode(const uint8_t* seqs, const int64_t* off, int64_t n, int d, Key128* keys,
                   uint8_t* lens, uint32_t* eqprev, uint32_t* vcount, PlaneRow* rows,
                   uint32_t* err, cudaStream_t s);  // vcount and rows may be null
// The same with the counts summed up: rec_off[0, n], the total also to
// *total.  status: encode_status_bytes(n), zeroed.
size_t encode_status_bytes(int64_t n);
void launch_encode_scan(const uint8_t* seqs, const int64_t* off, int64_t n, int d, Key128* keys,
                        uint8_t* lens, uint32_t* eqprev, uint64_t* rec_off, uint64_t* total,
                        uint64_t* status, PlaneRow* rows, uint32_t* err, cudaStream_t s);
// Record selection by fingerprint bin, bin = (record >> shift) & mask, for
// searches that take the records in several passes.  With `append` null the
// expand kernel only counts records per bin into bin_count[0 .. mask] (mask
// < 2048) and writes nothing; otherwise it appends the records whose bin lies
// in [lo, hi) to out[0, n_rec), counting them in *append.
enum { SEL_ALL = 0, SEL_COUNT = 1, SEL_APPEND = 2 };
struct BinSel {
  uint32_t shift = 0, mask = 0;
  uint32_t lo = 0, hi = 0;
  uint32_t* bin_count = nullptr;
  unsigned long long* append = nullptr;
};
constexpr int MAX_BIN_BITS = 11;

// The sequences (or paired receptors, when src.keys_b is set: d <= 2, no bin
// selection) expanded into records.  sel null: every record of sequence i
// goes to out[rec_off[i] ...].
// hist: when not null, the digit counts of the sort passes over bits
// [hist_lo, hist_hi) are added there.
// zero: when not null, zero_bytes (a multiple of 16, 16-byte aligned) are
// cleared there as well (the record sort's look-back status).
struct ExpandSource;
void launch_expand(const ExpandSource& src, const uint64_t* rec_off, int64_t n, int d,
                   const uint32_t* seq_rep, uint32_t id_bits, uint64_t* out, uint64_t n_rec,
                   uint32_t* hist, int hist_lo, int hist_hi, int sms, uint32_t* err,
                   cudaStream_t s, const BinSel* sel = nullptr, void* zero = nullptr,
                   size_t zero_bytes = 0);
void launch_seq_rep(const int64_t* rep_off, int64_t n_rep, uint32_t* seq_rep, int64_t n,
                    cudaStream_t s);

// k_radix.cu ---------------------------------------------------------------
int onesweep_tile(int cfg);
int onesweep_configs();
size_t radix_status_bytes(int64_t n, int cfg);
void launch_histogram(const uint64_t* keys, int64_t n, const uint64_t* n_dev, int lo, int hi,
                      uint32_t* hist, int sms, cudaStream_t s);
// A configuration outside the tunable ones: one resident grid that loops over
// the tiles of the (device-side) key count.
constexpr int ONESWEEP_LOOP = 120;
// Clears the status area (radix_status_bytes(n, ONESWEEP_LOOP)) as far as a
// sort of *n_dev keys with that configuration reads it.
void launch_clear_status(uint64_t* status, int64_t n, const uint64_t* n_dev, int sms,
                         cudaStream_t s);
// Sorts a[0:n) on bits [lo, hi) using b as the second buffer; `hist` holds the
// digit histograms of every pass.  *sorted receives a or b.
// hist_in_passes: `hist` holds only pass 0's digit counts; every pass counts
// the next pass's digits itself (zeroed hist rows 1.. expected).
// n_dev: when not null the key count is read on the device (n is then a
// capacity that sizes the grid and the look-back status).
// bucket_start: when not null (2^(hi-lo) entries, all bits set on entry), the
// last pass leaves in bucket_start[b] the first sorted position whose bits
// [lo, hi) equal b; buckets without records keep all bits set.
// first_cfg: configuration of the first pass (>= 0), e.g. the unstable one;
// LSD order needs only the later passes to be stable.  Ignored when its tile
// differs from cfg's.
// status_zeroed: the whole status area (radix_status_bytes) is zero on entry,
// so the first two passes need no clearing.
cudaError_t radix_sort_passes(uint64_t* a, uint64_t* b, int64_t n, int lo, int hi, uint32_t* hist,
                              uint64_t* digit_base, uint64_t* status, int cfg, uint32_t* err,
                              uint64_t** sorted, const char* tag, cudaStream_t s,
                              bool hist_in_passes = false, const uint64_t* n_dev = nullptr,
                              uint64_t* bucket_start = nullptr, int first_cfg = -1,
                              bool status_zeroed = false);
// Unstable configuration with the same tile as cfg, for a sort's first pass.
int onesweep_unstable_config(int cfg);

// k_bucket.cu --------------------------------------------------------------
// Positions per flag tile of the group-bound kernels (head/tail counts are
// kept per tile of this many sorted records).
constexpr int GROUP_FLAG_TILE = 32768;
// Split of the hs group-key bits: the top G are sorted by global radix
// passes (bucket = those bits), the low L = hs - G in shared memory, 2^kbits
// buckets per block.  G depends only on (n_rec, hs); kbits also on the
// shared-memory step (hash grouping or sort).
struct GroupingShape {
  int G = 0, L = 0, kbits = 0;
};
GroupingShape choose_grouping(uint64_t n_rec, int hs, bool hash);
int bucket_capacity(bool hash);
// A holds n records sorted on their top G group-key bits (bits [lo + L, 64)),
// bucket_start as left by radix_sort_passes (unused when G == 0).  Writes the
// records to Y (A is scratch afterwards): with `hash`, every group's records
// contiguous in arbitrary order; without, sorted on all group-key bits.
// With `flags` (zeroed, group_flag_words(n)) and `tile_counts` (zeroed, one
// per GROUP_FLAG_TILE positions) also the head/tail flags k_group_write
// reads.  cap: records per shared-memory segment (0 = the full capacity).
// With `cand` (hash only): buckets that fit a segment write no records and no
// flags but append their candidate pair words (min id << id_bits | max id)
// to cand[0, cand_cap), counting them in cand_count[0] (DERR_CAPACITY past
// the capacity); larger buckets go the flag route as before and add their
// record count to cand_count[1].
void launch_bucket(bool hash, uint64_t* A, uint64_t* Y, int64_t n, const uint64_t* n_dev,
                   const uint64_t* bucket_start, const GroupingShape& g, int lo, int cap,
                   uint64_t* flags, uint64_t* tile_counts, uint64_t* cand, uint64_t cand_cap,
                   uint64_t* cand_count, int id_bits, uint32_t* err, cudaStream_t s);
// k_partition.cu, k_scatter.cu ----------------------------------------------
// Partitions of the variant records by their top pbits fingerprint bits:
// partition p fills rec[p * region ...] and counts its records in count[p]
// (which may pass `region`; the records past it go to spill).  The filter
// keeps a list per partition in `kept`, laid out alike.
// sub: when not 0, each partition is split once more, by the sub bits below,
// before the filter (launch_group_filter): into `kept`, fine_region words
// each, and the filter's lists then lie in `rec`.
struct PartitionShape {
  int pbits = 0;
  uint32_t region = 0;
  int sub = 0;
  uint32_t fine_region = 0;
  uint64_t words() const {
    const uint64_t a = (uint64_t)region << pbits, b = (uint64_t)fine_region << (pbits + sub);
    return a > b ? a : b;
  }
  uint64_t counts() const {
    return ((uint64_t)2 << (pbits + sub)) + (sub ? (uint64_t)1 << pbits : 0);
  }
};
// fx: the size of the partitions (see XTN_TUNE_FILTER_SEGMENT).
PartitionShape choose_partitions(uint64_t n_rec, int fx);
struct Partitions : PartitionShape {
  uint64_t* rec = nullptr;      // words()
  uint64_t* kept = nullptr;     // words()
  uint32_t* count = nullptr;    // counts() zeroed words: (the coarse partitions',) the
                                // partitions', then the lists'
  uint64_t* spill = nullptr;    // spill_cap words
  uint64_t spill_cap = 0;
  uint64_t* n_spill = nullptr;  // zeroed by the caller
  uint32_t* kept_count() const { return count + ((uint64_t)1 << pbits); }
  // the partitions after the split (sub != 0)
  Partitions fine() const {
    Partitions f = *this;
    f.pbits = pbits + sub;
    f.region = fine_region;
    f.sub = 0;
    f.fine_region = 0;
    f.rec = kept;
    f.kept = rec;
    f.count = count + ((uint64_t)1 << pbits);
    return f;
  }
};
// The records of every canonical variant, expanded straight into their
// partitions; rec_off as launch_expand takes it, its last entry the record
// count (at most n_rec, a capacity that sizes the grid).
void launch_expand_scatter(const ExpandSource& src, const uint64_t* rec_off, int64_t n, int d,
                           const uint32_t* seq_rep, uint32_t id_bits, uint64_t n_rec,
                           const Partitions& p, int sms, uint32_t* err, cudaStream_t s);
// The same for records already expanded to in[0, n) (n_dev: when not null the
// count is read on the device and n is a capacity).
void launch_partition(const uint64_t* in, int64_t n, const uint64_t* n_dev, const Partitions& p,
                      int sms, uint32_t* err, cudaStream_t s);
// The split of coarse partitions (p.sub != 0) into p.fine(); a partition that
// ran over goes to the spill whole.
void launch_split(const Partitions& p, uint64_t n_rec, int sms, uint32_t* err, cudaStream_t s);

// k_filter.cu --------------------------------------------------------------
// Appends the candidate words (min id << id_bits | max id) of every pair of
// records with equal group keys to cand[0, cand_cap), counting them in
// *cand_count (DERR_CAPACITY past the capacity, and without count_all perhaps
// not all of them counted then).  What a block cannot group
// on its own -- a partition or list that overflowed, a single key too
// frequent for its table -- is appended to p.spill (counted in *p.n_spill)
// for a global sort of those few.  n_rec: the expected records.
void launch_group_filter(const Partitions& p, uint64_t n_rec, uint64_t* cand, uint64_t cand_cap,
                         uint64_t* cand_count, bool count_all, int id_bits, int sms,
                         uint32_t* err, cudaStream_t s);
// k_pairs.cu ---------------------------------------------------------------
size_t scan_status_bytes(int64_t n);
size_t group_status_bytes(int64_t n);
void launch_scan_counts(const uint32_t* counts, int64_t n, uint64_t* out, uint64_t* status,
                        uint32_t* err, cudaStream_t s);
void launch_scan_group_pairs(const uint32_t* S, const uint32_t* E, int64_t n_groups,
                             const uint64_t* n_groups_dev, uint64_t* out, uint64_t* status,
                             uint32_t* err, cudaStream_t s);
size_t group_flag_words(int64_t n);
// Group bounds = flags (k_group_flags, or k_bucket_sort) + finish (tile
// prefix, k_group_write, group count).  `status` holds group_status_bytes(n).
uint64_t* group_tile_counts(uint64_t* status, int64_t n);
void launch_group_flags(const uint64_t* keys, int64_t n, const uint64_t* n_dev, int gshift,
                        uint64_t* flags, uint64_t* status, cudaStream_t s);
void launch_group_finish(const uint64_t* flags, int64_t n, const uint64_t* n_dev, uint32_t* S,
                         uint32_t* E, uint64_t cap, uint64_t* status, uint32_t* err,
                         uint64_t* n_groups, cudaStream_t s);
// Candidate words of the groups [S, E] into out[base + t], t < pairs of the
// groups, base = *out_base (0 when null); *n_pairs_out = base + pairs.
void launch_emit_pairs(const uint64_t* keys, uint64_t n_keys, const uint32_t* S,
                       const uint64_t* pair_off, int64_t n_groups, const uint64_t* n_groups_dev,
                       uint64_t pair_cap, uint32_t id_bits, uint64_t* out,
                       const uint64_t* out_base, uint64_t* n_pairs_out, int sms, uint32_t* err,
                       cudaStream_t s);

// k_verify.cu --------------------------------------------------------------
// Rows per tile of the dedup and TCRdist kernels, and the look-back status
// those kernels need for n rows (one word per tile plus a tile counter).  Up
// to FEW_ROWS the TCRdist kernel takes tiles of an eighth.
constexpr int VERIFY_TILE = 2048;
constexpr int64_t FEW_ROWS = 1 << 18;
constexpr size_t verify_status_bytes_for(int64_t n) {
  const int64_t few = n < FEW_ROWS ? n : FEW_ROWS;
  constexpr int64_t eighth = VERIFY_TILE / 8;
  const int64_t a = (n + VERIFY_TILE - 1) / VERIFY_TILE, b = (few + eighth - 1) / eighth;
  return (size_t)(a > b ? a : b) * 8 + 16;
}
// The sequences one side of the pairs indexes: their bit planes, and for
// paired receptors (metric 2) those of their second chains.
struct PairSide {
  const PlaneRow* rows = nullptr;
  const PlaneRow* rows_b = nullptr;
  uint64_t n = 0;
};
// metric: 0 = Levenshtein, 1 = Hamming (pairs of equal length only), 2 =
// paired chains (Levenshtein of the first chains plus that of the second).
// Verify counts the survivors' digits over bits [hist_lo, hist_hi) and writes
// a survivor's distance into bits [hist_hi, hist_hi + 8) of its word when they
// exist (hist_hi + 8 <= 64); the dedup then reads it there (dist_shift = hist_hi) instead of computing
// it again (dist_shift = 0).
// self_mode: 0 = query vs reference, 1 = self-search (pairs within a
// repertoire when seq_rep is given), 2 = self-search keeping only pairs
// between different repertoires.
size_t verify_status_bytes(int64_t n);
void launch_verify_candidates(const uint64_t* cand, uint64_t n, const uint64_t* n_dev,
                              uint32_t j_bits, const PairSide& si, const PairSide& sj,
                              const uint32_t* seq_rep, int self_mode, int d, int metric,
                              uint64_t* surv, uint64_t surv_cap, uint64_t* n_surv, uint32_t* hist,
                              int hist_lo, int hist_hi, int sms, uint32_t* err, cudaStream_t s);
void launch_unique_finalize(const uint64_t* pairs, int64_t n, const uint64_t* n_dev,
                            uint32_t j_bits, const PairSide& si, const PairSide& sj, int d,
                            int metric, xtn_triple* out, int64_t cap, uint64_t* status,
                            uint32_t* err, uint64_t* total, cudaStream_t s, int dist_shift,
                            bool status_zeroed = false);
// The same for words (with their distances) grouped by their top 8 pair bits,
// the groups beginning at starts[0, 256): duplicates out, sort and rows.
// status: bucket_rows_status_bytes(), cleared.  DERR_CAPACITY: a group has
// more than SMALL_PAIRS distinct words.
size_t bucket_rows_status_bytes();
void launch_bucket_rows(const uint64_t* words, uint64_t n_max, const uint64_t* n_words,
                        const uint64_t* starts, uint32_t pair_bits, uint32_t j_bits,
                        xtn_triple* rows, int64_t row_cap, uint64_t* status, uint64_t* n_rows, uint32_t* err, cudaStream_t s);
// The whole last step for at most SMALL_PAIRS candidates in one block: their
// distances, the sort, the duplicates out, the rows (*n_rows of them).
constexpr uint64_t SMALL_PAIRS = 4096;
void launch_small_rows(const uint64_t* cand, uint64_t n, uint32_t j_bits, const PairSide& si,
                       const PairSide& sj, const uint32_t* seq_rep, int self_mode, int d,
                       int metric, xtn_triple* rows, int64_t row_cap, uint64_t* n_rows,
                       uint32_t* err, cudaStream_t s);
void launch_tcrdist_filter(const xtn_triple* in, int64_t n, const Key128* keys,
                           const uint8_t* lens, int64_t n_seq, int max_score, xtn_triple* out,
                           uint64_t* status, uint32_t* err, uint64_t* total, cudaStream_t s);

// k_paired.cu --------------------------------------------------------------
// Canonical deletion variants (d <= 2) per receptor alpha + token + beta, the
// token never deleted.
void launch_paired_counts(const uint8_t* lens_a, const uint32_t* eq_a, const uint8_t* lens_b,
                          const uint32_t* eq_b, int64_t n, int d, uint32_t* vcount,
                          cudaStream_t s);

// k_query.cu ---------------------------------------------------------------
// Directory of the sorted index (entry t = first record whose top dir_bits
// bits are >= t) and, added into *n_groups, the number of distinct group keys
// (bits from gshift up).
void launch_build_dir(const uint64_t* rec, uint64_t n_rec, int dir_bits, int gshift,
                      uint32_t* dir, uint64_t* n_groups, cudaStream_t s);
// A directory range of at most this many records is compared whole by a
// lookup, so its records stand in any order; longer ones are sorted.
constexpr int INDEX_SCAN = 32;
// k_index.cu: the index out of partitions of the records.  False where its
// sizes do not take it (the records are then sorted, and launch_build_dir
// reads the directory off them).
constexpr int INDEX_SUB_BITS = 14;
bool choose_index_partitions(uint64_t n_rec, int dir_bits, PartitionShape* g);
// rec[0, n_rec), dir[0, 2^dir_bits]; *n_groups += the distinct group keys
// (bits from gshift up; of a million records or more 16 times those of every
// 16th partition, since counting all took 100 of 300 us and the number only
// feeds an estimate).  DERR_CAPACITY: one directory range is too long.
void launch_index_build(const Partitions& p, uint64_t n_rec, int dir_bits, int gshift,
                        uint64_t* rec, uint32_t* dir, uint64_t* n_groups, uint32_t* err,
                        cudaStream_t s);

// Records [first, first + count) of the index, candidates of query q, to
// cand[base ...]: a part of a group too large for one lane.
struct QueryChunk {
  uint64_t base;
  uint32_t first, count, q, unused;
};
// Candidate words of the queries: cand[0, *n_cand) but for the large groups,
// whose places are reserved and which `list` names (launch_query_spread
// writes them).  *n_cand above cand_cap or *n_list above list_cap: nothing is
// written past either, and the counts say what a rerun needs.  *n_variants
// receives the queries' variants.  The three counts begin at zero.
void launch_query_candidates(const ExpandSource& src, int64_t n_q, int d, const uint64_t* rec,
                             uint64_t n_rec, const uint32_t* dir, int dir_bits, int gshift,
                             uint32_t ref_bits, uint64_t* cand, uint64_t cand_cap,
                             uint64_t* n_cand, QueryChunk* list, uint64_t list_cap,
                             uint64_t* n_list, uint64_t* n_variants, int sms, uint32_t* err,
                             cudaStream_t s);
void launch_query_spread(const uint64_t* rec, uint64_t n_rec, uint32_t ref_bits,
                         const QueryChunk* list, uint64_t n_list, uint64_t* cand,
                         uint64_t cand_cap, int sms, uint32_t* err, cudaStream_t s);

}  // namespace xtn
