// Internal declarations of the MinJoin CUDA library (sm_103a).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <string>

#include "../../include/minjoin.h"

#define MJ_CUDA_TRY(expr)                                   \
  do {                                                      \
    cudaError_t _e = (expr);                                \
    if (_e != cudaSuccess) {                                \
      mj::set_last_cuda_error(_e, #expr, __FILE__, __LINE__); \
      return MJ_ERR_CUDA;                                   \
    }                                                       \
  } while (0)

// every kernel launch of the library is followed by MJ_KERNEL_DONE(): it
// counts the launch (mj_stats.n_launches) and checks the launch error
#define MJ_KERNEL_DONE()                  \
  do {                                    \
    mj::note_launch();                    \
    MJ_CUDA_TRY(cudaGetLastError());      \
  } while (0)

#define MJ_TRY(expr)          \
  do {                        \
    int _s = (expr);          \
    if (_s != MJ_OK) return _s; \
  } while (0)

namespace mj {

constexpr int kNumSMsHint = 152;

// device-side error flags (mj_stats.device_flags)
enum : uint32_t {
  FLAG_BOUNDS = 1u << 0,       // an index left its buffer (access skipped)
  FLAG_TIMEOUT = 1u << 1,      // a bounded wait gave up
  FLAG_CAPACITY = 1u << 2,     // an output buffer was too small (write skipped)
  FLAG_LENGTH = 1u << 3,       // a string too long for 32-bit column indexing (pair rejected)
};

void set_last_cuda_error(cudaError_t e, const char* expr, const char* file, int line);
void note_launch();
uint64_t launch_count();

// ---------------------------------------------------------------- workspace
// A growable device buffer owned by a context; reallocated (contents
// dropped) only when a larger size is requested.
struct Buf {
  void* p = nullptr;
  size_t bytes = 0;
  int reserve(size_t need, cudaStream_t s);
  // as reserve, but the first `keep` bytes survive a reallocation
  int grow_keep(size_t need, size_t keep, cudaStream_t s);
  template <class T>
  T* as() const { return static_cast<T*>(p); }
  void release();
};

// Derived parameters of one input (host copy).
struct Derived {
  uint32_t sigma = 0, bits = 1, q = 1, T = 1, K = 0;
  int32_t r_min = 1, r_max = 0;
  uint64_t N = 0, seed = 0;
  uint32_t repeats = 1;   // parallel repetition: independent Pi functions
  uint8_t rank[256] = {0};
};

// ---------------------------------------------------------------- kernels (launchers)
// All launchers are stream-ordered and return MJ_OK or MJ_ERR_CUDA.

// a1: out[0 .. 255] non-zero for the byte values present (a sampled count),
// out[256] = the longest string's length, out[257] = the input's size.
int launch_input_stats(const uint8_t* bytes, const int64_t* offsets, uint32_t n, unsigned long long* out,
                       cudaStream_t s);
// *out = max of v[0 .. n-1] (0 when n = 0)
int launch_max_u32(const uint32_t* v, uint64_t n, unsigned int* out, cudaStream_t s);

// A partition record, packed in two 16-byte words: Karp-Rabin key, group
// run (the hash bits of the grouping sort key; 0 until the records are put
// in group order), string length, partition length, string id, position.
struct alignas(16) PRec {
  uint64_t h61;
  uint32_t run, slen, len, sid, pos, pad;
};
static_assert(sizeof(PRec) == 32, "PRec is two 16-byte words");

__device__ __forceinline__ PRec load_rec(const PRec* __restrict__ r, uint64_t u) {
  const uint4* p = reinterpret_cast<const uint4*>(r + u);
  const uint4 a = __ldg(p), b = __ldg(p + 1);
  PRec x;
  x.h61 = (uint64_t)a.x | ((uint64_t)a.y << 32);
  x.run = a.z;
  x.slen = a.w;
  x.len = b.x;
  x.sid = b.y;
  x.pos = b.z;
  x.pad = b.w;
  return x;
}

__device__ __forceinline__ void store_rec(PRec* __restrict__ r, uint64_t u, const PRec& x) {
  uint4* p = reinterpret_cast<uint4*>(r + u);
  p[0] = make_uint4((uint32_t)x.h61, (uint32_t)(x.h61 >> 32), x.run, x.slen);
  p[1] = make_uint4(x.len, x.sid, x.pos, x.pad);
}

// a2-a3: anchor bitmap (1 bit per byte position) and per-tile anchor counts.
struct PartitionArgs {
  const uint8_t* bytes;
  const int64_t* offsets;
  uint32_t n;
  uint64_t nbytes;
  uint32_t q, bits, T;
  int32_t r_min, r_max;
  uint32_t seed32;
  uint64_t seed64;
  const uint64_t* table;  // nullable explicit Pi
  uint8_t rank[256];
  uint8_t* codes = nullptr;  // nullable: also the input's rank codes, one byte per input byte (with the planes)
  // set by the launcher: 2^19 and 2^16, so that x >> 13 and x >> 16 are the
  // high words of x * mul (the mixer's shifts on the multiply pipe)
  uint32_t mul_shr13, mul_shr16;
};
constexpr int kPartTile = 2048;  // byte positions per CTA tile
uint64_t partition_num_tiles(uint64_t nbytes);
// planes (nullable): also writes the rank-code bit-planes of the tile for the
// verifier (plane p's word for positions g .. g+31 at plane_at(guard_words +
// g/32, p)), and
// with a.codes the rank codes themselves (a.codes[g] for position g; the
// buffer covers whole tiles).  With first_call, dev_flags words 0 and 1 and the
// planes' guard words are cleared before.
int launch_anchor_flags(const PartitionArgs& a, uint32_t* bitmap, uint32_t* tile_count,
                        uint32_t* dev_flags, uint32_t* planes, uint64_t plane_words,
                        uint32_t guard_words, uint32_t* tile_first, bool first_call, cudaStream_t s);
// a4: one partition record per anchor, in position order (so string order),
// from the bitmap and the per-tile list offsets; key = (len, H61(substring)).
int launch_partition_records(const PartitionArgs& a, const uint32_t* bitmap, const uint32_t* tile_offset,
                             const uint32_t* tile_first, uint64_t key_base, PRec* recs, cudaStream_t s);
// The fields of n records as separate arrays (any may be null).
int launch_unpack_records(const PRec* recs, uint64_t n, uint32_t* sid, uint32_t* pos, uint32_t* len, uint64_t* key,
                          cudaStream_t s);

// scans (exclusive, in place allowed); temp from scan_temp_bytes
size_t scan_temp_bytes(uint64_t n);
int launch_exclusive_scan_u32(const uint32_t* in, uint32_t* out, uint64_t n, void* temp,
                              uint32_t* total_out, cudaStream_t s);
int launch_exclusive_scan_u64(const uint64_t* in, uint64_t* out, uint64_t n, void* temp,
                              uint64_t* total_out, cudaStream_t s);
int launch_exclusive_scan_u32_to_u64(const uint32_t* in, uint64_t* out, uint64_t n, void* temp,
                                     uint64_t* total_out, cudaStream_t s);

// LSD radix sort of 64-bit keys (optionally with 32-bit values) on bits
// [bit_lo, bit_hi).  Ping-pongs between (keys, keys_alt); *result_in_alt
// tells which buffer holds the sorted data.
size_t radix_temp_bytes(uint64_t n);
int radix_sort_u64(uint64_t* keys, uint64_t* keys_alt, uint32_t* vals, uint32_t* vals_alt,
                   uint64_t n, int bit_lo, int bit_hi, void* temp, bool* result_in_alt,
                   cudaStream_t s);

// The same for 32-bit keys (fewer bytes per pass); temp from radix_temp_bytes.
int radix_sort_u32(uint32_t* keys, uint32_t* keys_alt, uint32_t* vals, uint32_t* vals_alt,
                   uint64_t n, int bit_lo, int bit_hi, void* temp, bool* result_in_alt,
                   cudaStream_t s);

// a5-a7 of a plain join, string by string from the longest (mj_pairs.cu).
// The caller clears every counter these steps add to.
// Ranks: strings from the longest to the shortest (ties by id); short = longest
// - length.  shorts/sid (n entries each and their alternates) end sorted, in the
// alternates if *in_alt; rank_of[id], hi[rank] = the last rank within K of its
// length; short_rank[l] (nullable), l = 0 .. longest = the first rank of short l
// or more; widest[0] = the most ranks above its own that a string can pair with,
// widest[1] = the longest string that can pair at all; *spans += the sum of all
// strings' such ranks, an upper bound on the candidates.
int launch_string_ranks(const int64_t* offsets, uint32_t n, uint32_t K, uint32_t longest, int len_bits,
                        uint32_t* shorts, uint32_t* shorts_alt, uint32_t* sid, uint32_t* sid_alt, void* temp,
                        uint32_t* rank_of, uint32_t* hi, uint32_t* short_rank, unsigned int* widest,
                        unsigned long long* spans, bool* in_alt, cudaStream_t s);
// first[i], i = 0 .. n: base + the anchors before string i in the bitmap
// (`total` anchors in all).
int launch_string_first(const int64_t* offsets, uint32_t n, uint64_t nbytes, const uint32_t* bitmap,
                        const uint32_t* tile_off, uint32_t total, uint32_t base, uint32_t* first, cudaStream_t s);
// delta[k (n + 1) + id] + t = place by rank of record t of repetition k;
// rfirst: n words of scratch.
int launch_rank_order(const uint32_t* first, const uint32_t* sid_of, const uint32_t* rank_of, uint32_t n, uint32_t reps,
                      uint32_t* rfirst, uint32_t* delta, void* temp, cudaStream_t s);
// Sort keys and record indices of records [t0, t1) of one repetition (delta:
// its n + 1 words) at their places by rank.
int launch_rank_keys(const PRec* recs, uint32_t t0, uint32_t t1, const uint32_t* delta, int hash_bits, int pb_bits,
                     uint32_t W, uint32_t* keys, uint32_t* vals, cudaStream_t s);
// Rank bits of a visit word when a visit fits 16 bytes, else 0 (B is then used).
// longest: of the strings that can pair (the words of others are never visited).
int visit_rank_bits(uint64_t longest, uint32_t n);
// From the sorted keys and indices: A, B, skr (n_rec entries) and the windows
// of every record (2 entries each, at the record's own place).
struct RankTables {
  const uint32_t* hi;
  const uint32_t* shorts;
  const uint32_t* short_rank;   // nullable
  uint32_t longest, n;
};
int launch_rank_windows(const uint32_t* idx, const uint32_t* keys, uint32_t n_rec, const PRec* recs,
                        const uint32_t* rank_of, const RankTables& rt, uint32_t K, uint32_t W, int pb_bits, int rb,
                        uint4* A, uint2* B, uint64_t* skr, uint4* win, cudaStream_t s);
// Lower bounds on the edit distance: gram lengths of the two levels and the
// buckets of single symbols (by rank code).
struct SigShape {
  uint32_t q1, q2;
  uint8_t bucket[256];
};
uint32_t signature_grams(uint32_t sigma, uint32_t want);   // the shortest q (<= 8) with sigma^q >= want
SigShape signature_shape(uint32_t sigma, const uint64_t* counts_by_code);
size_t sig1_bytes(uint32_t n);
size_t sig2_bytes(uint32_t n);
// Signatures by rank (sid_of) or id (null).  With sampled (nullable), does
// nothing when *sampled <= min_sampled.
int launch_signatures(const uint8_t* codes, const int64_t* offsets, const uint32_t* sid_of, uint32_t n,
                      const SigShape& g, const unsigned long long* sampled, uint64_t min_sampled, uint4* sig1,
                      uint32_t* sig2, cudaStream_t s);
// The same bounds on listed pairs (signatures by id): rejected[t] = 1 and
// ed[t] = k + 1 where they exceed pair t's band (pk[t], or K when pk is null).
int launch_pair_bounds(const uint32_t* pi, const uint32_t* pj, const uint32_t* pk, uint32_t K, uint64_t m, uint32_t n,
                       const SigShape& g, const uint4* sig1, const uint4* sig2, uint8_t* rejected, uint32_t* ed,
                       cudaStream_t s);
struct PairArgs {
  const PRec* recs;           // in position order
  const uint32_t* first;      // launch_string_first, one row of n + 1 per repetition
  const uint4* win;
  const uint4* A;
  const uint2* B;
  const uint32_t* sid_of;     // by rank
  const uint32_t* shorts;
  uint32_t longest;
  const uint32_t* hi;
  const uint4* sig1;          // read when *sampled > min_sampled
  unsigned long long* sampled;   // candidates of the sampled strings (launch_string_sample)
  uint64_t min_sampled;
  uint32_t stride = 1;        // set by the launcher
  uint32_t n, reps, K, q1;
  int rb;                     // visit_rank_bits
  uint32_t bm_words = 0;      // set by the launcher
  unsigned long long* out_count;   // pairs of ranks that pass the first bound (all counted, the first cap listed)
  unsigned long long* totals;      // out_count + 1: raw pairs, candidates, K-band cells of the candidates
  uint64_t cap = 0;
  uint2* out = nullptr;
};
bool string_pairs_fit(uint32_t widest);   // a string's bitmap fits in shared memory
// Raw pairs from which a join whose widest window holds `widest` ranks goes
// string by string (0: always), and their estimate from one record in
// likely_pairs_step(n_rec): *total sampled pairs, of which likely_pairs makes the
// number.  table: likely_pairs_slots(n_rec) words of scratch.
uint64_t string_pairs_from(uint32_t n, uint32_t widest, int sms);
uint32_t likely_pairs_slots(uint64_t n_rec);
int launch_likely_pairs(const PRec* recs, uint64_t n_rec, uint32_t K, uint32_t* table, unsigned long long* total,
                        cudaStream_t s);
uint64_t likely_pairs(uint64_t n_rec, uint64_t total);
constexpr size_t kStringPairsSmemMax = 160u << 10;
int launch_string_pairs(const PairArgs& a, uint32_t widest, cudaStream_t s);
// *a.sampled += the candidates of about kSampleStrings strings
constexpr uint32_t kSampleStrings = 1024;
int launch_string_sample(const PairArgs& a, uint32_t widest, cudaStream_t s);
// The second bound of the listed pairs: what passes, as pairs of ids (i < j).
struct ListArgs {
  const uint2* in;
  const unsigned long long* in_count;
  uint64_t in_cap;
  const uint4* sig2;          // read when *sampled > min_sampled
  const uint32_t* sid_of;
  const uint32_t* shorts;
  uint32_t longest;
  const unsigned long long* sampled;
  uint64_t min_sampled;
  uint32_t K, q2;
  unsigned long long* out_count;   // all counted, the first cap listed
  uint64_t cap;
  uint32_t* out_i;
  uint32_t* out_j;
};
int launch_listed_pairs(const ListArgs& a, cudaStream_t s);

// a5-a6: grouping keys and pair emission.  A group key is hash_bits (<= 32)
// bits of a hash of (len, Karp-Rabin key), then pb_bits bits of the
// position bucket pos / W (W >= K, so the partner of a record under the
// position filter lies in its bucket or the next), then slen_bits bits of
// string length.
struct GroupKeyShape {
  int hash_bits, pb_bits, slen_bits;
  uint32_t W;
};
int launch_make_group_keys(const PRec* recs, uint32_t n_rec, const GroupKeyShape& g, uint64_t* keys, uint32_t* idx,
                           cudaStream_t s);
// Records in group order: out[t] = recs[idx[t]] with run = the hash bits of
// keys[t] and pad = its position bucket.
int launch_gather_records(const uint32_t* idx, const uint64_t* keys, uint32_t n_rec, const GroupKeyShape& g,
                          const PRec* recs, PRec* out, cudaStream_t s);
int launch_count_pairs(const PRec* r, uint32_t n_rec, uint32_t K, const GroupKeyShape& g, uint32_t* count,
                       cudaStream_t s);
// pairs are packed as (i << nb) | j, i < j
int launch_fill_pairs(const PRec* r, uint32_t n_rec, uint32_t K, const GroupKeyShape& g, int nb,
                      const uint64_t* offs, uint64_t* pairs, cudaStream_t s);
// a7 by the pair bitmap: bit (a, b), a < b < n_str, in row a (ceil((n_str - 1
// - a) / 32) words, rows back to back); pair_bitmap_words(n_str) words in all.
// launch_mark_pairs clears the bitmap (unless `clear` is false: the caller
// knows it is zero), sets the bit of every pair the walk finds and counts
// them (raw pairs, duplicates included) into *raw_total; launch_bitmap_rows
// writes the candidates per row, launch_bitmap_write the candidates (i, j)
// sorted, at the row offsets `off` (exclusive scan of the row counts), and
// with `clear` clears the bitmap's words as it reads them.
uint64_t pair_bitmap_words(uint32_t n_str);
int launch_mark_pairs(const PRec* r, uint32_t n_rec, uint32_t K, const GroupKeyShape& g, uint32_t n_str, uint32_t* bm,
                      unsigned long long* raw_total, bool clear, cudaStream_t s);
int launch_bitmap_rows(const uint32_t* bm, uint32_t n_str, uint32_t* cnt, cudaStream_t s);
int launch_bitmap_write(uint32_t* bm, uint32_t n_str, const uint32_t* off, uint32_t* oi, uint32_t* oj, bool clear,
                        cudaStream_t s);
int launch_key_check(const PRec* r, const uint8_t* bytes, const int64_t* offsets, uint32_t n_rec,
                     unsigned long long* mismatches, cudaStream_t s);
// Sharded join: records from separate arrays, pairs packed for a dedup sort.
int launch_pack_records(const uint32_t* sid, const uint32_t* pos, const uint32_t* len, const uint64_t* key,
                        const uint32_t* slen, uint64_t n, PRec* out, cudaStream_t s);
int launch_pack_pairs(const uint32_t* pi, const uint32_t* pj, uint64_t m, int nb, uint64_t* out, cudaStream_t s);
int launch_unpack_pairs(const uint64_t* packed, uint64_t m, int nb, uint32_t* oi, uint32_t* oj, cudaStream_t s);
// a7: unique of sorted u64 pairs -> flags; then compaction.
int launch_unique_flags(const uint64_t* sorted, uint64_t n, uint32_t* flags, cudaStream_t s);
// run_start (nullable): run_start[u] = index of candidate u's first raw pair
int launch_compact_pairs(const uint64_t* sorted, const uint32_t* flags, const uint32_t* offs, uint64_t n, int nb,
                         uint32_t* out_i, uint32_t* out_j, uint32_t* run_start, cudaStream_t s);

// a8: banded verification (diagonal bit-vector, one thread per pair).
struct RankTable {
  uint8_t r[256];
};
struct VerifyArgs {
  const uint32_t* planes = nullptr;    // bit-planes of rank codes: word w of plane p at w * plane_stride(bits) + p
  uint32_t bits;
  const uint8_t* bytes = nullptr;
  const int64_t* offsets = nullptr;
  uint32_t n_strings;        // pair ids >= n_strings are rejected (flagged, ed = k + 1)
  const uint32_t* pi = nullptr;
  const uint32_t* pj = nullptr;
  const uint32_t* pk = nullptr;        // nullable per-pair band
  const uint32_t* order = nullptr;     // nullable: pair indices in the order to verify them
  const uint32_t* skip_kband = nullptr; // nullable: skip pair t when fed[t] <= skip_kband[t] < K (already settled)
  const uint32_t* first_ed = nullptr;  // nullable: first-pass results fed (else ed itself); a skipped pair copies fed[t] to ed[t]
  const uint32_t* range_lo = nullptr;  // nullable: with range_hi, process order positions [*range_lo, *range_hi) only
  const uint32_t* range_hi = nullptr;
  unsigned long long* skipped = nullptr; // nullable: number of pairs skipped that way
  uint32_t K;
  uint64_t m;
  uint32_t* ed = nullptr;
  unsigned long long* work = nullptr;  // nullable: word-columns processed (columns x W) accumulated
  uint32_t* dev_flags = nullptr;
  const uint4* pair_geo = nullptr;     // nullable: at order position q, (oA, oB, m, n) of pair order[q], A the
                                       // longer string (n = kGeoBadIds: an id out of range); loaded with order[q]
  uint32_t* out_t = nullptr;           // nullable: indices of the pairs with result <= K, appended (order arbitrary)
  const uint8_t* codes = nullptr;      // the input's rank codes, one byte per input byte (digit-table kernels)
  uint64_t nbytes = 0;                 // bytes of the input
  unsigned long long* out_count = nullptr;
};
// The planes' words of the same 32 positions lie side by side, in 2 words for
// codes of up to 2 bits, else in 8 (planes beyond the code's bits are zero), so
// that a lane fetches them by one 8-byte or two 16-byte loads: every lane of
// the verifiers reads at places of its own, and such loads cost one cycle of
// the L1 cache per lane each, whatever their width.  (One array per plane took
// 28 loads per 32 columns of a 3-word band instead of 10: 1.3 M text pairs
// 7.7 -> 5.3 ms, 100,000 byte pairs 691 -> 577 us.)
__host__ __device__ constexpr uint32_t plane_stride(uint32_t bits) { return bits <= 2 ? 2u : 8u; }
int verify_words_for(uint32_t kmax);
inline uint32_t plane_guard_words(uint32_t kmax) { return kmax / 64 + (uint32_t)verify_words_for(kmax) + 4; }
// codes (nullable, nbytes + 32 bytes): also the rank code of every byte.
int launch_build_planes(const uint8_t* bytes, uint64_t nbytes, const RankTable& rt, uint32_t bits,
                        uint32_t* planes, uint64_t plane_words, uint32_t guard_words, uint8_t* codes,
                        cudaStream_t s);
// `next` is a device counter the persistent kernel hands pairs out from.
// kernel: MJ_VERIFY_KERNEL_*; lanes: wavefront lanes per pair (0 = fewest that fit).
// next_is_zero: the caller has cleared it.
int launch_verify(const VerifyArgs& a, uint64_t plane_words, uint32_t guard_words, uint32_t kmax,
                  unsigned long long* next, cudaStream_t s, int kernel = MJ_VERIFY_KERNEL_AUTO, int lanes = 0,
                  bool next_is_zero = false);
// the two-lanes-per-pair verifier (bands of 1 .. 8 words) and the wavefront on
// 2 .. 32 lanes (one warp) or 64 .. 1024 (one CTA per pair); *next is zero
int launch_verify_split(const VerifyArgs& a, uint64_t plane_words, uint32_t guard_words, int words,
                        unsigned long long* next, cudaStream_t s);
int launch_verify_wave(const VerifyArgs& a, uint64_t plane_words, uint32_t guard_words, int lanes,
                       unsigned long long* next, cudaStream_t s);
// the wavefront in the shape (lanes, words per lane) that suits the band and
// the number of pairs
int launch_verify_wave_auto(const VerifyArgs& a, uint64_t plane_words, uint32_t guard_words, uint32_t kmax,
                            unsigned long long* next, cudaStream_t s);
// pairs of bands up to kmax that such a launch has in flight from its start on
uint64_t wave_in_flight(uint32_t kmax, int sms);
int wave_lanes_for(uint32_t kmax);
// whether launch_verify takes bands up to kmax with this kernel choice
bool verify_supported(uint32_t kmax, int kernel, int lanes);
// lanes of the CTA wavefront (several warps per pair) for bands up to kmax,
// and the fewest lanes of either wavefront form; at most kMaxCtaLanes
constexpr int kMaxCtaLanes = 1024;
int cta_lanes_for(uint32_t kmax);
int fewest_lanes_for(uint32_t kmax);

// Verification order: pair indices longest first (by the shorter length), a
// counting sort over 256 length classes; within a class the order is
// arbitrary.  counts[b] and ranges[2b], ranges[2b+1] = [start, end) of the
// pairs whose shorter length has floor(log2) = b (lengths 0 and 1: b = 0),
// the autotuner's length buckets, contiguous and longest first.  scratch:
// kOrderScratchWords words (256 class counts for each of up to 8 blocks per
// SM of the counting sort).
constexpr int kLenBuckets = 32;
constexpr int kOrderScratchWords = 256 * kNumSMsHint * 8;
// cells (nullable): set to the pairs' K-band cells (mj_stats.band_cells).
// geo (nullable): the pairs' geometry at their order positions (VerifyArgs::
// pair_geo).  Pair ids >= n_str count as empty strings here (the verifier
// flags them).
constexpr uint32_t kGeoBadIds = 0xffffffffu;
// sg: n_str entries of scratch for the strings' {offset, length} (inputs
// are under 4 GB).
// rejected (nullable): pairs with rejected[t] != 0 are left out of the order
// and the buckets (not of the cells); *kept (nullable): pairs in the order.
int launch_length_order(const uint32_t* ci, const uint32_t* cj, const int64_t* offsets, uint32_t n_str, uint64_t m,
                        uint32_t K, const uint8_t* rejected, uint32_t* kept, uint32_t* scratch, uint2* sg,
                        uint32_t* order, uint4* geo, uint32_t* counts, uint32_t* ranges, unsigned long long* cells,
                        cudaStream_t s);

// ---- learned first-pass band (MLP 8 -> 64 -> 64 -> 1)
// features of a candidate (i, j), n = min length, d0 = length difference,
// c = matched partition pairs behind the candidate (its multiplicity before
// dedup), pa/pb = partitions of the two strings:
//   log2(1+n)/16, d0/K, c/(T+1), pa/(T+1), pb/(T+1), c/min(pa,pb),
//   log2(1+c)/8, K/(K+100)
constexpr int kBandFeatures = 8;
constexpr int kBandHidden = 64;
constexpr int kBandParams = kBandHidden * kBandFeatures + kBandHidden + kBandHidden * kBandHidden + kBandHidden +
                            kBandHidden + 1;
static_assert(kBandParams == MJ_BAND_PARAMS && kBandFeatures == MJ_BAND_FEATURES, "ABI constants");
int launch_band_features(const uint32_t* ci, const uint32_t* cj, const uint32_t* mult, const uint32_t* parts,
                         const int64_t* offsets, uint64_t m, uint32_t K, uint32_t T, float* X, cudaStream_t s);
int launch_band_forward(const float* P, const float* X, uint64_t m, float* out, cudaStream_t s);
// part: band_grad_part_bytes(batch) of scratch; grad and *loss are overwritten
size_t band_grad_part_bytes(uint64_t batch);
int launch_band_grad(const float* P, const float* X, const float* Y, const uint32_t* ed, uint32_t K, uint64_t m,
                     uint64_t batch, uint64_t seed, float tau, float* part, float* grad, float* loss, cudaStream_t s);
int launch_band_adam(float* P, const float* G, float* M, float* V, float lr, float b1, float b2, float eps, int step,
                     cudaStream_t s);
int launch_band_fused(const float* P, const uint32_t* ci, const uint32_t* cj, const uint32_t* run_start, uint64_t raw,
                      const uint32_t* parts, const int64_t* offsets, uint64_t m, uint32_t K, uint32_t T, uint32_t margin,
                      uint32_t min_mult, const uint8_t* rejected, uint32_t* kband, cudaStream_t s);
int launch_gate_hist(const float* X, const uint32_t* ed, uint64_t m, uint32_t K, unsigned int* hist, cudaStream_t s);
int launch_band_rule(const float* yhat, const uint32_t* ci, const uint32_t* cj, const int64_t* offsets, uint64_t m,
                     uint32_t K, uint32_t margin, uint32_t* kband, cudaStream_t s);

// multiplicity of every candidate from the run starts written by the pair
// compaction; partitions per string counted over the records
int launch_multiplicity(const uint32_t* run_start, uint64_t nc, uint64_t raw, uint32_t* mult, cudaStream_t s);
int launch_partition_counts(const PRec* recs, uint64_t n_rec, uint32_t n, uint32_t* parts, cudaStream_t s);
// Learned first passes: the pairs of every first-pass bucket b = 1 .. nb
// (band widths below band K's word count; bucket 0 = no first pass) listed
// contiguously in list, bucket b at [ranges[2b], ranges[2b+1]); cnt holds
// 2 * (kMaxBandBuckets + 2) words of scratch; *first_total = pairs listed.
constexpr uint32_t kMaxBandBuckets = 16;
int launch_band_buckets(const uint32_t* kband, uint64_t m, uint32_t K, uint32_t nb, uint32_t* cnt, uint32_t* ranges,
                        uint32_t* list, unsigned long long* first_total, cudaStream_t s);

// oa/ob/oc[t] = a/b/c[t], t < n, where the output is non-null
int launch_copy_words(const uint32_t* a, const uint32_t* b, const uint32_t* c, uint64_t n, uint32_t* oa, uint32_t* ob,
                      uint32_t* oc, cudaStream_t s);

// output of the join: the listed pair indices (sorted ascending, which is
// (i, j) order since the candidates are sorted) gathered into (i, j, ED);
// keys/keys_alt: 8 * n bytes each, temp: radix_temp_bytes(n)
int launch_gather_output(const uint32_t* out_t, uint64_t n, uint64_t m, const uint32_t* ci, const uint32_t* cj,
                         const uint32_t* ed, uint64_t* keys, uint64_t* keys_alt, void* temp, uint32_t* oi,
                         uint32_t* oj, uint32_t* oed, cudaStream_t s);

// The same for pairs in any order: sorted by (i, j) (nb bits each); vals and
// vals_alt: 4 * n bytes each.
int launch_gather_output_pairs(const uint32_t* out_t, uint64_t n, int nb, const uint32_t* ci, const uint32_t* cj,
                               const uint32_t* ed, uint64_t* keys, uint64_t* keys_alt, uint32_t* vals,
                               uint32_t* vals_alt, void* temp, uint32_t* oi, uint32_t* oj, uint32_t* oed,
                               cudaStream_t s);

}  // namespace mj
