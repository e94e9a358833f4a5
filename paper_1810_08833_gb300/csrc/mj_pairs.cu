// Steps a5-a7 of a plain join, string by string: grouping of equal
// partitions, the length and position filters of Alg. 3 and the dedup of the
// candidates, with a lower bound on the edit distance tested before a
// candidate is listed for verification.
//
// Strings are ranked from the longest to the shortest (ties by id).  The length
// filter lets a string of rank x pair only with ranks up to hi(x), the last
// string no more than K shorter, so "every pair once" is "every pair from its
// lower rank", and the candidates of x are a bitmap of hi(x) - x bits in shared
// memory: no bitmap over all pairs is cleared, marked at random in DRAM and
// swept.  (Pairs are listed by their longer string, whose bit-planes are most
// of what the verifier reads: neighbouring lanes then read the same words.)
//
// Records are sorted by (hash of the partition, position bucket), stably,
// from an order in which they come by rank: within a bucket ranks ascend.  For
// strings of lengths l and l - L the position filter keeps the partners at
// positions [pos - (K + L) / 2, pos + (K - L) / 2], an interval of K + 1 that
// moves with L.  With buckets of width W >= K / 2, x's partners through one
// record are in four windows of the sorted records: the buckets -2, -1, 0 and
// +1 of its own, each cut to the ranks whose L lets the interval reach it.
// Windows hold about 1 + W / K times the pairs that pass: 1.5 with W = K / 2;
// three whole buckets of width K held 2.5 (protein) to 2.9 (text) times them.
// Lengths are kept by rank as "short" = N - length, N the longest.

// Measured on 300,000 text-like strings (450 MB, 786 M raw pairs, 641 M
// candidates), general path against this one: pairs and dedup 33.8 -> 8.7 ms,
// order of the candidates 8.1 -> 0.1, their verification 182.7 -> 4.4 (1.3 M
// pairs pass the bounds; the signatures take 0.9 ms); 400,000 protein-like
// strings (178 MB, 190 M candidates): 16.1 -> 4.1 + 2.0 (second bound), 2.5 ->
// 0.4, 21.0 -> 3.3.
#include <algorithm>
#include <type_traits>

#include "mj_internal.cuh"


namespace mj {
namespace {

// ---------------------------------------------------------------- strings by length
__global__ void string_lengths_kernel(const int64_t* __restrict__ offsets, uint32_t n, uint32_t* __restrict__ keys,
                                      uint32_t* __restrict__ vals, uint32_t longest) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    keys[i] = longest - (uint32_t)(offsets[i + 1] - offsets[i]);
    vals[i] = (uint32_t)i;
  }
}

// First index in [lo, hi) with a[index] > v, hi if none.
template <class T>
__device__ __forceinline__ uint32_t upper_bound_of(const T* __restrict__ a, uint32_t lo, uint32_t hi, T v) {
  while (lo < hi) {
    const uint32_t mid = lo + (hi - lo) / 2;
    if (__ldg(a + mid) <= v) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// rank_of[sid]; hi[r] = last rank whose short is at most shorts[r] + K;
// widest[0] = the most ranks above its own that a string can pair with, widest[1] = the longest string
// that can pair with another, *spans += all ranks above their own that strings can pair with;
// short_rank[l] (nullable), l = 0 .. longest: first rank of short >= l, n if none.
// Every entry is a search of its own: filled by the rank that ends a run of
// lengths, a gap between two lengths is one thread's loop (20,000 reads and one
// string of 4 M symbols: 50 ms of a join of 108).
__global__ void __launch_bounds__(256) rank_tables_kernel(const uint32_t* __restrict__ shorts, const uint32_t* __restrict__ sid_of, uint32_t n,
                                   uint32_t K, uint32_t longest, uint32_t* __restrict__ rank_of,
                                   uint32_t* __restrict__ hi, uint32_t* __restrict__ short_rank,
                                   unsigned int* __restrict__ widest, unsigned long long* __restrict__ spans) {
  uint32_t w = 0, len = 0;
  unsigned long long sum = 0;
  for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t r = (uint32_t)t;
    rank_of[sid_of[r]] = r;
    const uint32_t L = shorts[r], top = L > 0xffffffffu - K ? 0xffffffffu : L + K;
    const uint32_t h = upper_bound_of(shorts, r + 1, n, top) - 1;
    hi[r] = h;
    w = max(w, h - r);
    if (h > r) len = max(len, longest - L);
    sum += h - r;
  }
  if (short_rank)   // longest < 2^32 - 1: a string's length is below the input's size
    for (uint64_t l = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; l <= longest; l += (uint64_t)gridDim.x * blockDim.x)
      short_rank[l] = l ? upper_bound_of(shorts, 0, n, (uint32_t)l - 1u) : 0u;
  // one block's three results at a time: with a warp's they were 94,000 updates
  // of three words for 1,000,000 strings, 75 us
  __shared__ uint32_t s_w[8], s_len[8];
  __shared__ unsigned long long s_sum[8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  w = __reduce_max_sync(0xffffffffu, w);
  len = __reduce_max_sync(0xffffffffu, len);
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
  if (lane == 0) {
    s_w[wid] = w;
    s_len[wid] = len;
    s_sum[wid] = sum;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < 8; ++k) {
      w = max(w, s_w[k]);
      len = max(len, s_len[k]);
      sum += s_sum[k];
    }
    if (w) {
      atomicMax(widest, w);
      atomicMax(widest + 1, len);
      atomicAdd(spans, sum);
    }
  }
}

// ---------------------------------------------------------------- record order
// first[s] = records of this repetition before byte offsets[s], plus base:
// string s's records are [first[s], first[s + 1]).  One warp per string: the
// tile's list offset plus the anchors before the byte in its tile.
__global__ void string_first_kernel(const int64_t* __restrict__ offsets, uint32_t n, uint64_t nbytes,
                                    const uint32_t* __restrict__ bitmap, const uint32_t* __restrict__ tile_off,
                                    uint32_t total, uint32_t base, uint32_t* __restrict__ first) {
  const int lane = threadIdx.x & 31;
  const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  for (uint64_t s = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; s <= n; s += warps) {
    const uint64_t g = (uint64_t)offsets[s];
    uint32_t v = total;
    if (g < nbytes) {
      const uint64_t tile = g / kPartTile, w0 = tile * (kPartTile / 32), wg = g >> 5;
      uint32_t c = 0;
      for (uint64_t w = w0 + lane; w <= wg; w += 32) {
        uint32_t x = __ldg(bitmap + w);
        if (w == wg) x &= (1u << (g & 31)) - 1u;
        c += __popc(x);
      }
      v = __ldg(tile_off + tile) + __reduce_add_sync(0xffffffffu, c);
    }
    if (lane == 0) first[s] = base + v;
  }
}

// cnt[r] = records of the string of rank r over all repetitions.
__global__ void rank_counts_kernel(const uint32_t* __restrict__ first, const uint32_t* __restrict__ sid_of, uint32_t n,
                                   uint32_t reps, uint32_t* __restrict__ cnt) {
  for (uint64_t r = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t s = sid_of[r];
    uint32_t c = 0;
    for (uint32_t k = 0; k < reps; ++k) {
      const uint32_t* f = first + (uint64_t)k * (n + 1) + s;
      c += f[1] - f[0];
    }
    cnt[r] = c;
  }
}

// delta[k (n + 1) + s] + t = place of record t (string s, repetition k) in the
// order by rank.
__global__ void rank_delta_kernel(const uint32_t* __restrict__ first, const uint32_t* __restrict__ rank_of,
                                  const uint32_t* __restrict__ rfirst, uint32_t n, uint32_t reps,
                                  uint32_t* __restrict__ delta) {
  for (uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t at = rfirst[rank_of[s]];
    for (uint32_t k = 0; k < reps; ++k) {
      const uint64_t x = (uint64_t)k * (n + 1) + s;
      delta[x] = at - first[x];
      at += first[x + 1] - first[x];
    }
  }
}

__device__ __forceinline__ uint64_t mix64(uint64_t k) {  // MurmurHash3 fmix64
  k ^= k >> 33;
  k *= 0xff51afd7ed558ccdull;
  k ^= k >> 33;
  k *= 0xc4ceb9fe1a85ec53ull;
  k ^= k >> 33;
  return k;
}

// Sort keys of records [t0, t1) (one repetition) at their places by rank:
// hash_bits bits of a hash of (len, key), then the position bucket.
__global__ void rank_keys_kernel(const PRec* __restrict__ recs, uint32_t t0, uint32_t t1,
                                 const uint32_t* __restrict__ delta, int hash_bits, int pb_bits, uint32_t W,
                                 uint32_t* __restrict__ keys, uint32_t* __restrict__ vals) {
  const uint32_t pb_max = (1u << pb_bits) - 1u;
  for (uint64_t t = t0 + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < t1;
       t += (uint64_t)gridDim.x * blockDim.x) {
    const PRec r = load_rec(recs, t);
    const uint64_t g = mix64(r.h61 ^ ((uint64_t)r.len * 0x9e3779b97f4a7c15ull));
    const uint32_t d = (uint32_t)t + __ldg(delta + r.sid);
    keys[d] = ((uint32_t)(g >> (64 - hash_bits)) << pb_bits) | min(r.pos / W, pb_max);
    vals[d] = (uint32_t)t;
  }
}

// What a visit compares, in 16 bytes where it fits (PACKED: lengths below
// 2^16 and ranks below 2^rb, rb = min(31, 35 - the length's bits)): both
// distances to the string's ends as halves of x, then rank, partition length
// and the 61-bit key over y, z and w.  Otherwise {pos, rpos, rank, low key
// word} in A and {high key word, partition length} in B.
template <bool PACKED>
__device__ __forceinline__ uint4 visit_word(uint32_t pos, uint32_t rpos, uint32_t rank, uint32_t len, uint64_t h61,
                                            int rb) {
  if (!PACKED) return make_uint4(pos, rpos, rank, (uint32_t)h61);
  return make_uint4(pos | (rpos << 16), rank | (len << rb), (uint32_t)h61,
                    (uint32_t)(h61 >> 32) | ((len >> (32 - rb)) << 29));
}

// The visit words in sorted order, and (sort key, rank) in one word for the
// window searches.
template <bool PACKED>
__global__ void rank_gather_kernel(const uint32_t* __restrict__ idx, const uint32_t* __restrict__ keys, uint32_t n_rec,
                                   const PRec* __restrict__ recs, const uint32_t* __restrict__ rank_of, int rb,
                                   uint4* __restrict__ A, uint2* __restrict__ B, uint64_t* __restrict__ skr) {
  for (uint64_t p = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n_rec;
       p += (uint64_t)gridDim.x * blockDim.x) {
    const PRec r = load_rec(recs, idx[p]);
    const uint32_t x = __ldg(rank_of + r.sid);
    A[p] = visit_word<PACKED>(r.pos, r.slen - r.pos, x, r.len, r.h61, rb);
    if (!PACKED) B[p] = make_uint2((uint32_t)(r.h61 >> 32), r.len);
    skr[p] = ((uint64_t)keys[p] << 32) | x;
  }
}

// First index >= from (<= n) whose word is >= v: galloping, then bisection.
__device__ __forceinline__ uint32_t gallop_up(const uint64_t* __restrict__ a, uint32_t from, uint32_t n, uint64_t v) {
  uint32_t lo = from, step = 1;
  uint64_t hi = from;
  while (hi < n && __ldg(a + hi) < v) {
    lo = (uint32_t)hi + 1;
    hi = (uint64_t)lo + step;
    step <<= 1;
  }
  uint32_t b = hi < n ? (uint32_t)hi : n;
  while (lo < b) {
    const uint32_t mid = lo + (b - lo) / 2;
    if (__ldg(a + mid) < v) lo = mid + 1;
    else b = mid;
  }
  return lo;
}

// First index <= from (from if none lower) whose word is >= v, given that
// a[from] >= v: galloping down, then bisection.
__device__ __forceinline__ uint32_t gallop_down(const uint64_t* __restrict__ a, uint32_t from, uint64_t v) {
  uint32_t hi = from, lo = 0, step = 1;
  while (hi > 0) {
    const uint32_t probe = hi > step ? hi - step : 0u;
    if (__ldg(a + probe) < v) {
      lo = probe + 1;
      break;
    }
    hi = probe;
    step <<= 1;
  }
  while (lo < hi) {
    const uint32_t mid = lo + (hi - lo) / 2;
    if (__ldg(a + mid) < v) lo = mid + 1;
    else hi = mid;
  }
  return hi;
}

// Pairs of sampled records (every step-th) of one partition, position bucket and
// length bucket of K + 1, a third or so of those that pass the filters, counted
// as they meet in a table by hash: a record pairs with those that were counted
// in its slot before.
__global__ void likely_pairs_kernel(const PRec* __restrict__ recs, uint64_t n_rec, uint32_t step, uint32_t K,
                                    uint32_t* __restrict__ table, uint32_t mask,
                                    unsigned long long* __restrict__ total) {
  unsigned long long sum = 0;
  for (uint64_t t = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) * step; t < n_rec;
       t += (uint64_t)gridDim.x * blockDim.x * step) {
    const PRec r = load_rec(recs, t);
    const uint64_t g = mix64(mix64(r.h61 ^ ((uint64_t)r.len * 0x9e3779b97f4a7c15ull)) ^
                             ((uint64_t)(r.pos / (K + 1)) << 32 | r.slen / (K + 1)));
    sum += atomicAdd(table + ((uint32_t)g & mask), 1u);
  }
  __syncwarp();
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
  if ((threadIdx.x & 31) == 0 && sum) atomicAdd(total, sum);
}

// The windows of every record (see the file comment), written at the record's
// own place: win[2 t], win[2 t + 1] = {first, count} of the buckets -2, -1, 0
// and +1.  Threads take the records in sorted order, so that neighbours search
// the same words.
// short_rank: first rank by short (null: no cut by length within a bucket).
__global__ void rank_windows_kernel(const uint64_t* __restrict__ skr, const uint32_t* __restrict__ idx,
                                    const uint4* __restrict__ A, bool packed, uint32_t n_rec, RankTables rt, uint32_t K,
                                    uint32_t W, int pb_bits, uint4* __restrict__ win) {
  const int32_t pb_max = (int32_t)((1u << pb_bits) - 1u);
  for (uint64_t pp = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; pp < n_rec;
       pp += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t p = (uint32_t)pp;
    const uint64_t w = __ldg(skr + p);
    const uint32_t key = (uint32_t)(w >> 32), x = (uint32_t)w, h = __ldg(rt.hi + x);
    uint32_t lo[4] = {0, 0, 0, 0}, cnt[4] = {0, 0, 0, 0};   // buckets 0, +1, -1, -2
    if (h > x) {
      const int64_t pos = packed ? __ldg(&A[p].x) & 0xffffu : __ldg(&A[p].x);
      const uint32_t sh = __ldg(rt.shorts + x);
      const int32_t pb = (int32_t)(key & (uint32_t)pb_max);
      uint32_t up = p, down = p;   // searches go on from here: buckets 0 and +1 upwards, -1 and -2 downwards
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const int e = s < 2 ? s : 1 - s;
        const int32_t bk = pb + e;
        if (bk < 0 || bk > pb_max) continue;
        // ranks (r0, r1] of the lengths from which positions [bk W, bk W + W) can be reached
        uint32_t r0 = x, r1 = h;
        if (e != 0 && rt.short_rank) {
          const int64_t first = (int64_t)bk * W, last = first + W - 1;
          const int64_t lmin = e < 0 ? max((int64_t)0, 2 * (pos - last) - (int64_t)K) : 0;
          const int64_t lmax = e > 0 ? (int64_t)K - 2 * (first - pos) : (int64_t)K;
          if (lmin > lmax) continue;
          const uint64_t l0 = (uint64_t)sh + lmin, l1 = (uint64_t)sh + lmax + 1;
          if (lmin > 0) r0 = max(x, (l0 <= rt.longest ? __ldg(rt.short_rank + l0) : rt.n) - 1u);
          if (lmax < (int64_t)K) r1 = min(h, (l1 <= rt.longest ? __ldg(rt.short_rank + l1) : rt.n) - 1u);
          if (r0 >= r1) continue;
        }
        const uint64_t k = (uint64_t)(key + (uint32_t)e) << 32;
        uint32_t a, b;
        if (e < 0) {
          b = gallop_down(skr, down, (k | r1) + 1u);
          a = gallop_down(skr, b, (k | r0) + 1u);
          down = a;
        } else {
          a = gallop_up(skr, up, n_rec, (k | r0) + 1u);
          b = gallop_up(skr, a, n_rec, (k | r1) + 1u);
          up = b;
        }
        lo[s] = a;
        cnt[s] = b - a;
      }
    }
    const uint64_t t = __ldg(idx + p);
    win[2 * t] = make_uint4(lo[3], cnt[3], lo[2], cnt[2]);
    win[2 * t + 1] = make_uint4(lo[0], cnt[0], lo[1], cnt[1]);
  }
}

// ---------------------------------------------------------------- lower bounds on the edit distance
// Counts of a string's q-grams, hashed to buckets and saturated: an
// edit changes at most 2 q of them by one (a substitution q gone, q new; an
// insertion or deletion one less), and at least d0 = |m - n| of the edits are
// insertions or deletions, so for two strings
//     sum |count_a - count_b| <= 2 q ED - d0,
// and neither hashing nor saturation raises the sum.  A candidate with
// sum + d0 > 2 q K therefore has ED > K and needs no dynamic program.
// Two levels: sig1, 32 bytes (length, then 28 counts up to 255: one sector per
// candidate) and sig2, 128 bytes (256 counts up to 15), for the candidates that
// pass.
constexpr int kSig1 = 28, kSig2 = 256;
constexpr int kSig2Bytes = kSig2 / 2;
// Longer strings are left to the verifier: a warp counts a string's grams, 11 ns
// a symbol, and one of 1,000,000 among 20,000 reads took 11 ms of a join of 35.
constexpr uint32_t kBoundsMaxLen = 1u << 15;

__device__ __forceinline__ uint32_t gram_hash(uint32_t h) {   // MurmurHash3 fmix32
  h ^= h >> 16;
  h *= 0x85ebca6bu;
  h ^= h >> 13;
  h *= 0xc2b2ae35u;
  h ^= h >> 16;
  return h;
}

// Whether a join by strings uses the bounds, from the candidates of a sample of
// its strings (string_pairs_kernel<..., true>), on the device: the host does
// not wait for the sample.
__device__ __forceinline__ bool use_bounds(const unsigned long long* sampled, uint64_t min_sampled) {
  return *sampled > min_sampled;
}

constexpr int kSigWarps = 8;
constexpr int kSigCopies = 4;   // of the first level's few counters, so that a warp's updates spread

// One warp per string: the counts in shared memory, then both signatures at
// the string's rank (sid_of) or id (null).  With sampled, returns at once when
// the bounds are not to be used (use_bounds).  A lane takes the four symbols of an aligned word and
// the words after it for the grams that run on (q <= 8).  Bound by the shared
// memory's updates, two per symbol.
__global__ void __launch_bounds__(32 * kSigWarps) signature_kernel(
    const uint8_t* __restrict__ codes, const int64_t* __restrict__ offsets, const uint32_t* __restrict__ sid_of,
    uint32_t n, SigShape g, const unsigned long long* __restrict__ sampled, uint64_t min_sampled,
    uint4* __restrict__ sig1, uint32_t* __restrict__ sig2) {
  if (sampled && !use_bounds(sampled, min_sampled)) return;
  __shared__ uint32_t s_c1[kSigWarps][kSigCopies * kSig1];
  __shared__ uint32_t s_c2[kSigWarps][kSig2];
  __shared__ uint8_t s_bucket[256];
  for (int c = threadIdx.x; c < 256; c += blockDim.x) s_bucket[c] = g.bucket[c];
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t* c1 = s_c1[wid];
  uint32_t* c1_mine = c1 + kSig1 * (lane & (kSigCopies - 1));
  uint32_t* c2 = s_c2[wid];
  const uint32_t* codes32 = reinterpret_cast<const uint32_t*>(codes);   // whole words: the buffer is longer than the input
  const uint64_t warps = (uint64_t)gridDim.x * kSigWarps;
  for (uint64_t r = (uint64_t)blockIdx.x * kSigWarps + wid; r < n; r += warps) {
    for (int c = lane; c < kSigCopies * kSig1; c += 32) c1[c] = 0;
#pragma unroll
    for (int c = 0; c < kSig2; c += 32) c2[c + lane] = 0;
    __syncwarp();
    const uint32_t s = sid_of ? __ldg(sid_of + r) : (uint32_t)r;
    const uint32_t o = (uint32_t)__ldg(offsets + s), e = (uint32_t)__ldg(offsets + s + 1);   // inputs are under 4 GB
    const uint32_t w1 = e - o < kBoundsMaxLen ? (uint32_t)(((uint64_t)e + 3) >> 2) : 0u;   // no bounds: only the length
#pragma unroll 2
    for (uint32_t w = (o >> 2) + lane; w < w1; w += 32) {
      const uint32_t x0 = __ldg(codes32 + w), x1 = __ldg(codes32 + w + 1);
      const uint32_t x2 = g.q2 > 5 ? __ldg(codes32 + w + 2) : 0u;
#pragma unroll
      for (uint32_t k = 0; k < 4; ++k) {
        const uint32_t p = 4 * w + k;   // below 2^32: w < 2^30
        if (p < o || p >= e) continue;
        const uint32_t left = e - p;
        const uint32_t lo = __funnelshift_r(x0, x1, 8 * k), hi = __funnelshift_r(x1, x2, 8 * k);   // eight symbols from p
        uint32_t v = lo & 255u;
        if (g.q1 == 1) atomicAdd(c1_mine + s_bucket[v], 1u);
        if (g.q2 == 1) atomicAdd(c2 + v, 1u);
        for (uint32_t i = 1; i < g.q2 && i < left; ++i) {   // q1 <= q2
          v = v * 257u + (((i < 4 ? lo >> (8 * i) : hi >> (8 * i - 32)) & 255u) + 1u);
          if (i + 1 == g.q1) atomicAdd(c1_mine + __umulhi(gram_hash(v), (uint32_t)kSig1), 1u);
          if (i + 1 == g.q2) atomicAdd(c2 + (gram_hash(v) >> 24), 1u);
        }
      }
    }
    __syncwarp();
    uint32_t* d1 = reinterpret_cast<uint32_t*>(sig1 + 2 * r);
    if (lane == 0) d1[0] = e - o;
    if (lane < kSig1 / 4) {
      uint32_t v1 = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        uint32_t c = 0;
#pragma unroll
        for (int y = 0; y < kSigCopies; ++y) c += c1[y * kSig1 + 4 * lane + k];
        v1 |= min(c, 255u) << (8 * k);
      }
      d1[1 + lane] = v1;
    }
    uint32_t v2 = 0;   // lane l: buckets 8 l .. 8 l + 7
#pragma unroll
    for (int k = 0; k < 8; ++k) v2 |= min(c2[8 * lane + k], 15u) << (4 * k);
    sig2[r * (kSig2Bytes / 4) + lane] = v2;
    __syncwarp();
  }
}

// sum of |a - b| over the four bytes, added to c
__device__ __forceinline__ uint32_t sad4(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("vabsdiff4.u32.u32.u32.add %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

__device__ __forceinline__ uint64_t band_cells_of(uint32_t M, uint32_t N, uint32_t K) {   // M >= N, M + K < 2^32
  if (N == 0) return 0;
  const uint32_t a = M > K ? min(M - K, N) : 0u;
  const uint64_t smin = (((uint64_t)a * (a + 1u)) >> 1) + (uint64_t)a * K + (uint64_t)(N - a) * M;
  const uint32_t b = min(K, N);
  const uint64_t smax = b + (N > K ? (((uint64_t)(N - K) * (N - K + 1u)) >> 1) : 0ull);
  return smin - smax + N;
}

// Sums of the second level's differences of 32 pairs of strings, one per lane:
// eight lanes read a pair's two records together, 16 bytes each, so that a
// step's loads are four whole records; pair 4 r + i goes to lanes 8 i .. 8 i + 7
// in step r.  The even and odd nibbles are summed apart (the odd ones in
// place, 16 times too large); the partial sums are exchanged by halves, so that
// lane 8 i + r ends with pair 4 r + i.  pair_of(q): the strings of pair q.
template <class F>
__device__ __forceinline__ uint32_t sig2_sums(const uint4* __restrict__ sig2, int lane, F pair_of) {
  constexpr uint32_t kLow = 0x0f0f0f0fu, kHigh = 0xf0f0f0f0u;
  const int g = lane & 7;
  uint32_t v[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const uint2 xy = pair_of(4 * r + (lane >> 3));
    const uint4 m = __ldg(sig2 + (uint64_t)xy.x * 8 + g), p = __ldg(sig2 + (uint64_t)xy.y * 8 + g);
    uint32_t lo = sad4(m.x & kLow, p.x & kLow, sad4(m.y & kLow, p.y & kLow, 0u));
    lo = sad4(m.z & kLow, p.z & kLow, sad4(m.w & kLow, p.w & kLow, lo));
    uint32_t hi = sad4(m.x & kHigh, p.x & kHigh, sad4(m.y & kHigh, p.y & kHigh, 0u));
    hi = sad4(m.z & kHigh, p.z & kHigh, sad4(m.w & kHigh, p.w & kHigh, hi));
    v[r] = lo + (hi >> 4);
  }
#pragma unroll
  for (int w = 4; w >= 1; w >>= 1) {   // lanes with bit w keep the upper half of the steps
    const bool up = lane & w;
#pragma unroll
    for (int k = 0; k < w; ++k) {
      const uint32_t give = up ? v[k] : v[k + w], keep = up ? v[k + w] : v[k];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, give, w);
    }
  }
  return v[0];
}

// The pair that sig2_sums leaves in this lane.
__device__ __forceinline__ int sig2_slot(int lane) { return 4 * (lane & 7) + (lane >> 3); }

// Sum of the first level's differences (sig1 records u, v and p, q) plus the
// length difference.
__device__ __forceinline__ uint32_t sig1_sum(const uint4& u, const uint4& v, const uint4& p, const uint4& q) {
  uint32_t sum = u.x > p.x ? u.x - p.x : p.x - u.x;
  sum = sad4(u.y, p.y, sum);
  sum = sad4(u.z, p.z, sum);
  sum = sad4(u.w, p.w, sum);
  sum = sad4(v.x, q.x, sum);
  sum = sad4(v.y, q.y, sum);
  sum = sad4(v.z, q.z, sum);
  return sad4(v.w, q.w, sum);
}

// rejected[t] = 1 and ed[t] = k + 1 for every pair whose lower bounds exceed
// its band k (pk[t] or K); ids out of range are left to the verifier.
__global__ void __launch_bounds__(256) pair_bounds_kernel(const uint32_t* __restrict__ pi,
                                                          const uint32_t* __restrict__ pj,
                                                          const uint32_t* __restrict__ pk, uint32_t K, uint64_t m,
                                                          uint32_t n, uint32_t q1, uint32_t q2,
                                                          const uint4* __restrict__ sig1,
                                                          const uint4* __restrict__ sig2,
                                                          uint8_t* __restrict__ rejected, uint32_t* __restrict__ ed) {
  const int lane = threadIdx.x & 31;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t t0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; t0 < m; t0 += stride) {
    const uint64_t t = t0 + sig2_slot(lane);
    const uint32_t x = t < m ? pi[t] : n, y = t < m ? pj[t] : n;
    const bool valid = x < n && y < n;
    const uint32_t k = t < m && pk ? min(pk[t], 1u << 20) : K;
    uint32_t d0 = 0;
    bool live = false, too_long = false;
    if (valid) {
      const uint4 u = __ldg(sig1 + 2 * (uint64_t)x), v = __ldg(sig1 + 2 * (uint64_t)x + 1);
      const uint4 p = __ldg(sig1 + 2 * (uint64_t)y), q = __ldg(sig1 + 2 * (uint64_t)y + 1);
      d0 = u.x > p.x ? u.x - p.x : p.x - u.x;
      too_long = max(u.x, p.x) >= kBoundsMaxLen;
      live = d0 <= k && sig1_sum(u, v, p, q) <= 2u * q1 * k;
    }
    if (__any_sync(0xffffffffu, live)) {
      const uint32_t sum = sig2_sums(sig2, lane, [&](int q) {   // pair q of this step is in the lane with that slot
        const int src = 8 * (q & 3) + (q >> 2);
        const uint32_t xx = __shfl_sync(0xffffffffu, live ? x : 0u, src);
        return make_uint2(xx, __shfl_sync(0xffffffffu, live ? y : 0u, src));
      });
      live = live && sum + d0 <= 2u * q2 * k;
    }
    if (t < m) {
      const bool rej = valid && !too_long && !live;
      rejected[t] = rej ? 1 : 0;
      if (rej) ed[t] = k + 1;
    }
  }
}

// ---------------------------------------------------------------- candidates of every string
// One CTA of THREADS threads per string x at a time; the strings are dealt out
// in rank order, so that concurrent CTAs work on neighbouring ranks, which
// share the signatures of their windows in L2.
//   records  its records in batches: non-empty windows listed in shared
//            memory, short ones from the front, long ones from the back;
//   visits   short windows are dealt out 32 items per warp step over 32
//            windows at a time (a scan of their sizes), long ones by the whole
//            CTA; a visit tests the position filter and the key, and sets the
//            partner's bit;
//   list     every warp takes 16 words of the bitmap that hold bits, clears
//            them, pushes their bits on its stack and pops candidates, two per lane, to
//            test them against the first lower bound; what passes is appended
//            to the list of pairs for the second.
// A warp per string has no barriers to wait at; only windows of 2^16 ranks and
// more take four warps per bitmap.  Latency of the scattered loads bounds it:
// on the protein-like workload one warp per string took 4.2 ms, two 6.1; 72
// registers (26 warps per SM) beat both fewer (64: 4.3) and more (94: 4.6).
constexpr uint32_t kLongWindow = 64;       // items from which the whole CTA takes a window
constexpr int kStack = 512 + 64;           // candidates on a warp's stack: 32 half-words' bits on top of an unfinished batch
constexpr int kPassed = 96;                // those that passed the first bound, not yet appended

// WIDE: windows of 2^16 ranks and more.
template <int THREADS, bool WIDE>
struct PairShared {
  static constexpr int kWarps = THREADS / 32;
  using Slot = typename std::conditional<WIDE, uint32_t, uint16_t>::type;   // a rank within the window
  uint4 rec[THREADS];                        // visit words of the string's records
  uint2 rec_b[THREADS];
  uint32_t wlo[4 * THREADS], wcnt[4 * THREADS];
  Slot stack[kWarps][kStack];
  Slot passed[kWarps][kPassed];
  uint8_t wrec[4 * THREADS];
  uint32_t n_short, n_long;
};

__device__ __forceinline__ uint32_t absdiff2(uint32_t a, uint32_t b) {   // |a.lo - b.lo| + |a.hi - b.hi|
  uint32_t d;
  asm("vabsdiff2.u32.u32.u32.add %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(0));
  return d;
}

// SAMPLE: only counts the candidates of every a.stride-th string into *a.sampled.
template <int THREADS, bool WIDE, bool PACKED, bool SAMPLE>
__global__ void __launch_bounds__(THREADS, THREADS == 32 ? 26 : 1) string_pairs_kernel(PairArgs a) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  using Shared = PairShared<THREADS, WIDE>;
  const uint32_t rank_mask = (1u << a.rb) - 1u;   // PACKED: the rank's bits of a visit word's y
  constexpr int kWarps = Shared::kWarps;
  Shared& sh = *reinterpret_cast<Shared*>(smem_raw);
  uint32_t* bm = reinterpret_cast<uint32_t*>(smem_raw + sizeof(Shared));
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  auto sync = [] {
    if (THREADS == 32) __syncwarp();
    else __syncthreads();
  };
  const bool filter = !SAMPLE && use_bounds(a.sampled, a.min_sampled);
  const uint32_t lim1 = 2u * a.q1 * a.K;
  unsigned long long raw = 0, cand = 0, cells = 0;
  if (tid == 0) sh.n_short = sh.n_long = 0;
  for (uint32_t w = tid; w < a.bm_words; w += THREADS) bm[w] = 0;   // cleared again as it is read
  sync();
  for (uint64_t xs = (uint64_t)blockIdx.x * a.stride; xs < a.n; xs += (uint64_t)gridDim.x * a.stride) {
    const uint32_t x = (uint32_t)xs;
    const uint32_t span = __ldg(a.hi + x) - x;
    if (span == 0) continue;
    const uint32_t words = (span + 31) / 32;
    const uint32_t sid = __ldg(a.sid_of + x), len_x = a.longest - __ldg(a.shorts + x);
    uint4 sx = make_uint4(0u, 0u, 0u, 0u), sy = sx;
    if (filter) {
      sx = __ldg(a.sig1 + 2 * (uint64_t)x);
      sy = __ldg(a.sig1 + 2 * (uint64_t)x + 1);
    }
    uint32_t found = 0;
    // E visits of a thread at once: their loads are in flight together
    auto visit = [&](auto ne, const uint32_t* p, const bool* on, const uint4* me, const uint2* me_b) {
      constexpr int E = decltype(ne)::value;
      uint4 o[E];
      uint2 b[E];
      bool ok[E];
#pragma unroll
      for (int e = 0; e < E; ++e)
        if (on[e]) o[e] = __ldg(a.A + p[e]);
#pragma unroll
      for (int e = 0; e < E; ++e) {
        ok[e] = false;
        if (!on[e]) continue;
        if (PACKED) {
          ok[e] = absdiff2(o[e].x, me[e].x) <= a.K &&
                  (((o[e].y ^ me[e].y) & ~rank_mask) | (o[e].z ^ me[e].z) | (o[e].w ^ me[e].w)) == 0;
        } else {
          ok[e] = (uint32_t)(abs((int32_t)(o[e].x - me[e].x)) + abs((int32_t)(o[e].y - me[e].y))) <= a.K &&
                  o[e].w == me[e].w;
          if (ok[e]) b[e] = __ldg(a.B + p[e]);
        }
      }
#pragma unroll
      for (int e = 0; e < E; ++e) {
        if (ok[e] && (PACKED || (b[e].x == me_b[e].x && b[e].y == me_b[e].y))) {
          const uint32_t bit = (PACKED ? o[e].y & rank_mask : o[e].z) - x - 1u;
          atomicOr(bm + (bit >> 5), 1u << (bit & 31u));
          ++found;
        }
      }
    };
    for (uint32_t k = 0; k < a.reps; ++k) {
      const uint32_t* f = a.first + (uint64_t)k * (a.n + 1) + sid;
      const uint32_t t1 = __ldg(f + 1);
      for (uint32_t t0 = __ldg(f); t0 < t1; t0 += THREADS) {
        const uint32_t t = t0 + tid;
        if (t < t1) {
          const uint4 u = __ldg(a.win + 2 * (uint64_t)t), v = __ldg(a.win + 2 * (uint64_t)t + 1);
          const PRec me = load_rec(a.recs, t);
          sh.rec[tid] = visit_word<PACKED>(me.pos, me.slen - me.pos, x, me.len, me.h61, a.rb);
          if (!PACKED) sh.rec_b[tid] = make_uint2((uint32_t)(me.h61 >> 32), me.len);
          const uint32_t lo[4] = {u.x, u.z, v.x, v.z}, cnt[4] = {u.y, u.w, v.y, v.w};
#pragma unroll
          for (int s = 0; s < 4; ++s) {
            if (!cnt[s]) continue;
            const uint32_t at = cnt[s] < kLongWindow ? atomicAdd(&sh.n_short, 1u)
                                                     : 4 * THREADS - 1 - atomicAdd(&sh.n_long, 1u);
            sh.wlo[at] = lo[s];
            sh.wcnt[at] = cnt[s];
            sh.wrec[at] = (uint8_t)tid;
          }
        }
        sync();
        const uint32_t n_short = sh.n_short, n_long = sh.n_long;
        for (uint32_t s0 = 32 * wid; s0 < n_short; s0 += 32 * kWarps) {
          const uint32_t s = s0 + lane;
          const uint32_t cnt = s < n_short ? sh.wcnt[s] : 0u;
          uint32_t incl = cnt;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
          }
          const uint32_t excl = incl - cnt, total = __shfl_sync(0xffffffffu, incl, 31);
          for (uint32_t i0 = 0; i0 < total; i0 += 32) {
            const uint32_t i = i0 + lane;
            int q = 0;   // the last window whose first item is at or before i
#pragma unroll
            for (int step = 16; step > 0; step >>= 1) {
              const uint32_t y = __shfl_sync(0xffffffffu, excl, q + step);
              if (y <= i) q += step;
            }
            const uint32_t e = __shfl_sync(0xffffffffu, excl, q);
            const bool on = i < total;
            const uint32_t pv = sh.wlo[s0 + q] + (i - e), r = sh.wrec[s0 + q] & (THREADS - 1);
            const uint4 me = sh.rec[r];
            const uint2 me_b = PACKED ? make_uint2(0u, 0u) : sh.rec_b[r];
            visit(std::integral_constant<int, 1>(), &pv, &on, &me, &me_b);
          }
        }
        for (uint32_t s = 0; s < n_long; ++s) {
          const uint32_t at = 4 * THREADS - 1 - s;
          const uint32_t lo = sh.wlo[at], cnt = sh.wcnt[at], r = sh.wrec[at];
          const uint4 m = sh.rec[r];
          const uint2 mb = PACKED ? make_uint2(0u, 0u) : sh.rec_b[r];
          const uint4 me[2] = {m, m};
          const uint2 me_b[2] = {mb, mb};
          for (uint32_t i = tid; i < cnt; i += 2 * THREADS) {
            const bool on[2] = {true, i + THREADS < cnt};
            const uint32_t pv[2] = {lo + i, lo + i + THREADS};
            visit(std::integral_constant<int, 2>(), pv, on, me, me_b);
          }
        }
        sync();
        if (tid == 0) sh.n_short = sh.n_long = 0;
        sync();
      }
    }
    raw += found;
    // ---- the candidates
    using Slot = typename Shared::Slot;
    Slot* stack = sh.stack[wid];
    Slot* passed = sh.passed[wid];
    uint32_t depth = 0, waiting = 0;   // warp-uniform
    auto append = [&]() {   // the waiting pairs of ranks go on the list
      unsigned long long base = 0;
      if (lane == 0) base = atomicAdd(a.out_count, (unsigned long long)waiting);
      base = __shfl_sync(0xffffffffu, base, 0);
      for (uint32_t i = lane; i < waiting; i += 32)
        if (base + i < a.cap) a.out[base + i] = make_uint2(x, x + 1u + (uint32_t)passed[i]);
      waiting = 0;
      __syncwarp();   // the entries are read before new ones replace them
    };
    // first bound of the top `take` (at most 32 E) candidates of the stack
    auto test = [&](auto ne, uint32_t take) {
      constexpr int E = decltype(ne)::value;
      depth -= take;
      bool on[E];
      uint32_t slot[E];
      uint4 u[E], v[E];
#pragma unroll
      for (int e = 0; e < E; ++e) {
        on[e] = 32u * e + lane < take;
        slot[e] = on[e] ? (uint32_t)stack[depth + 32u * e + lane] : 0u;
        const uint32_t y = x + 1u + slot[e];
        if (on[e] && filter) {
          u[e] = __ldg(a.sig1 + 2 * (uint64_t)y);
          v[e] = __ldg(a.sig1 + 2 * (uint64_t)y + 1);
        } else if (on[e]) {
          u[e].x = a.longest - __ldg(a.shorts + y);
        }
      }
#pragma unroll
      for (int e = 0; e < E; ++e) {
        bool live = on[e];
        if (live) {
          cells += band_cells_of(len_x, u[e].x, a.K);
          if (filter) live = sig1_sum(u[e], v[e], sx, sy) <= lim1 || len_x >= kBoundsMaxLen;
        }
        const uint32_t mask = __ballot_sync(0xffffffffu, live);
        if (live) passed[waiting + __popc(mask & ((1u << lane) - 1u))] = (Slot)slot[e];
        waiting += __popc(mask);
        __syncwarp();
        if (waiting > kPassed - 32) append();
      }
    };
    // 16 words from half-word h0 on, 32 half-words to a step
    auto take = [&](uint32_t h0) {
      const uint32_t h = h0 + lane;
      const uint32_t both = h < 2 * words ? bm[h >> 1] : 0u;
      if (THREADS != 32 && !__any_sync(0xffffffffu, both != 0)) return;
      uint32_t bits = (both >> (16 * (h & 1))) & 0xffffu;
      __syncwarp();
      if (both && !(h & 1)) bm[h >> 1] = 0;
      const uint32_t c = __popc(bits);
      cand += c;
      if (SAMPLE) return;   // nothing is listed: the stack stays empty
      uint32_t incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t z = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += z;
      }
      uint32_t at = depth + incl - c;
      depth += __shfl_sync(0xffffffffu, incl, 31);
      while (bits) {
        stack[at++] = (Slot)(16u * h + (__ffs(bits) - 1));
        bits &= bits - 1;
      }
      __syncwarp();
      while (depth >= 64) test(std::integral_constant<int, 2>(), 64u);
      __syncwarp();   // the popped entries are read before the next step's pushes
    };
    if (THREADS == 32) {   // a warp looks at 128 words at a time and takes the groups that hold bits
      for (uint32_t w0 = 0; w0 < words; w0 += 128) {
        const uint32_t wl = w0 + 4 * lane;
        const uint4 four = wl < a.bm_words ? *reinterpret_cast<const uint4*>(bm + wl) : make_uint4(0u, 0u, 0u, 0u);
        uint32_t some = __ballot_sync(0xffffffffu, (four.x | four.y | four.z | four.w) != 0);
        while (some) {
          const uint32_t group = (uint32_t)(__ffs(some) - 1) >> 2;
          some &= ~(15u << (4 * group));
          take(2 * (w0 + 16 * group));
        }
      }
    } else {   // wide windows come here with many candidates only: the warps take 16 words in turn
      for (uint32_t h0 = 32 * wid; h0 < 2 * words; h0 += 32 * kWarps) take(h0);
    }
    if (!SAMPLE) {
      if (depth) test(std::integral_constant<int, 2>(), depth);
      if (waiting) append();
    }
    sync();   // the bitmap is clear for the next string
  }
  for (int o = 16; o > 0; o >>= 1) {
    raw += __shfl_down_sync(0xffffffffu, raw, o);
    cand += __shfl_down_sync(0xffffffffu, cand, o);
    cells += __shfl_down_sync(0xffffffffu, cells, o);
  }
  if (SAMPLE) {
    if (lane == 0 && cand) atomicAdd(a.sampled, cand);
    return;
  }
  if (lane == 0) {
    if (raw) atomicAdd(a.totals + 0, raw);
    if (cand) atomicAdd(a.totals + 1, cand);
    if (cells) atomicAdd(a.totals + 2, cells);
  }
}

// Second bound of the listed pairs of ranks (x < y): a warp takes 32 pairs per
// step and appends what passes, as ids.  Without the bounds (few candidates)
// every pair passes.
__global__ void __launch_bounds__(256) listed_pairs_kernel(ListArgs a) {
  const int lane = threadIdx.x & 31;
  const bool filter = use_bounds(a.sampled, a.min_sampled);
  const uint64_t m = min(*a.in_count, (unsigned long long)a.in_cap);
  const uint32_t lim = 2u * a.q2 * a.K;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t t0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; t0 < m; t0 += stride) {
    const uint64_t t = t0 + sig2_slot(lane);
    const uint2 pair = a.in[min(t, m - 1)];
    bool pass = t < m;
    if (filter) {
      const uint32_t sum = sig2_sums(a.sig2, lane, [&](int q) { return a.in[min(t0 + q, m - 1)]; });
      const uint32_t sx = __ldg(a.shorts + pair.x), sy = __ldg(a.shorts + pair.y);
      pass = pass && (sum + (sy - sx) <= lim || a.longest - sx >= kBoundsMaxLen);
    }
    const uint32_t mask = __ballot_sync(0xffffffffu, pass);
    if (!mask) continue;
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(a.out_count, (unsigned long long)__popc(mask));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (pass) {
      const unsigned long long o = base + __popc(mask & ((1u << lane) - 1u));
      if (o < a.cap) {
        const uint32_t i = __ldg(a.sid_of + pair.x), j = __ldg(a.sid_of + pair.y);
        a.out_i[o] = min(i, j);
        a.out_j[o] = max(i, j);
      }
    }
  }
}

template <int THREADS, bool WIDE, bool PACKED, bool SAMPLE>
int launch_string_pairs_t(PairArgs a, uint32_t widest, cudaStream_t s) {
  auto kernel = string_pairs_kernel<THREADS, WIDE, PACKED, SAMPLE>;
  a.bm_words = (widest / 32 + 4) / 4 * 4;   // whole 16-byte words, ceil(widest / 32) or more
  const size_t smem = sizeof(PairShared<THREADS, WIDE>) + (size_t)a.bm_words * 4;
  int dev = 0, sms = 0, per_sm = 0;
  MJ_CUDA_TRY(cudaGetDevice(&dev));
  MJ_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // the limit is the function's, shared by all contexts and threads: the largest
  // size that string_pairs_fit or a 16-bit window allows, never this call's own
  constexpr size_t limit = WIDE ? kStringPairsSmemMax + 32 : sizeof(PairShared<THREADS, WIDE>) + 65536 / 8;
  if (smem > limit) return MJ_ERR_UNSUPPORTED;
  MJ_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit));
  MJ_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, THREADS, smem));
  a.stride = SAMPLE ? std::max<uint32_t>(1, a.n / kSampleStrings) : 1;
  const uint64_t work = (a.n + a.stride - 1) / a.stride;
  const uint64_t grid = std::min<uint64_t>(work, (uint64_t)std::max(1, sms) * std::max(1, per_sm));
  kernel<<<(unsigned)grid, THREADS, smem, s>>>(a);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

template <bool SAMPLE>
int launch_string_pairs_s(const PairArgs& a, uint32_t widest, cudaStream_t s) {
  if (!a.n) return MJ_OK;
  if (widest < 65536 && a.rb) return launch_string_pairs_t<32, false, true, SAMPLE>(a, widest, s);
  if constexpr (!SAMPLE)   // a sample's few strings take longer on one warp each: 5.4 ms against 1.4 on four
    if (widest < 65536) return launch_string_pairs_t<32, false, false, false>(a, widest, s);
  return a.rb ? launch_string_pairs_t<128, true, true, SAMPLE>(a, widest, s)
              : launch_string_pairs_t<128, true, false, SAMPLE>(a, widest, s);
}

unsigned grid_for(uint64_t n, int threads = 256) {
  const uint64_t g = (n + threads - 1) / threads, cap = (uint64_t)kNumSMsHint * 32;
  return (unsigned)(g < 1 ? 1 : (g > cap ? cap : g));
}

}  // namespace

int launch_string_ranks(const int64_t* offsets, uint32_t n, uint32_t K, uint32_t longest, int len_bits,
                        uint32_t* shorts, uint32_t* shorts_alt, uint32_t* sid, uint32_t* sid_alt, void* temp, uint32_t* rank_of, uint32_t* hi,
                        uint32_t* short_rank, unsigned int* widest, unsigned long long* spans, bool* in_alt, cudaStream_t s) {
  *in_alt = false;
  if (!n) return MJ_OK;
  string_lengths_kernel<<<grid_for(n), 256, 0, s>>>(offsets, n, shorts, sid, longest);
  MJ_KERNEL_DONE();
  MJ_TRY(radix_sort_u32(shorts, shorts_alt, sid, sid_alt, n, 0, len_bits, temp, in_alt, s));
  rank_tables_kernel<<<grid_for(std::max<uint64_t>(n, short_rank ? longest + 1ull : 0)), 256, 0, s>>>(
      *in_alt ? shorts_alt : shorts, *in_alt ? sid_alt : sid, n, K, longest, rank_of, hi, short_rank, widest,
      spans);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

int launch_string_first(const int64_t* offsets, uint32_t n, uint64_t nbytes, const uint32_t* bitmap,
                        const uint32_t* tile_off, uint32_t total, uint32_t base, uint32_t* first, cudaStream_t s) {
  string_first_kernel<<<grid_for(((uint64_t)n + 1) * 32), 256, 0, s>>>(offsets, n, nbytes, bitmap, tile_off, total,
                                                                       base, first);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

int launch_rank_order(const uint32_t* first, const uint32_t* sid_of, const uint32_t* rank_of, uint32_t n, uint32_t reps,
                      uint32_t* rfirst, uint32_t* delta, void* temp, cudaStream_t s) {
  rank_counts_kernel<<<grid_for(n), 256, 0, s>>>(first, sid_of, n, reps, rfirst);
  MJ_KERNEL_DONE();
  MJ_TRY(launch_exclusive_scan_u32(rfirst, rfirst, n, temp, nullptr, s));
  rank_delta_kernel<<<grid_for(n), 256, 0, s>>>(first, rank_of, rfirst, n, reps, delta);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

int launch_rank_keys(const PRec* recs, uint32_t t0, uint32_t t1, const uint32_t* delta, int hash_bits, int pb_bits,
                     uint32_t W, uint32_t* keys, uint32_t* vals, cudaStream_t s) {
  if (t1 <= t0) return MJ_OK;
  rank_keys_kernel<<<grid_for(t1 - t0), 256, 0, s>>>(recs, t0, t1, delta, hash_bits, pb_bits, W, keys, vals);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

int launch_rank_windows(const uint32_t* idx, const uint32_t* keys, uint32_t n_rec, const PRec* recs,
                        const uint32_t* rank_of, const RankTables& rt, uint32_t K, uint32_t W, int pb_bits, int rb,
                        uint4* A, uint2* B, uint64_t* skr, uint4* win, cudaStream_t s) {
  if (!n_rec) return MJ_OK;
  if (rb) rank_gather_kernel<true><<<grid_for(n_rec), 256, 0, s>>>(idx, keys, n_rec, recs, rank_of, rb, A, B, skr);
  else rank_gather_kernel<false><<<grid_for(n_rec), 256, 0, s>>>(idx, keys, n_rec, recs, rank_of, rb, A, B, skr);
  MJ_KERNEL_DONE();
  rank_windows_kernel<<<grid_for(n_rec), 256, 0, s>>>(skr, idx, A, rb != 0, n_rec, rt, K, W, pb_bits, win);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

int visit_rank_bits(uint64_t longest, uint32_t n) {
  if (longest >= 65536) return 0;
  int lb = 1;
  while (longest >> lb) ++lb;
  const int rb = std::min(31, 35 - lb);
  return n <= (1u << rb) ? rb : 0;
}

size_t sig1_bytes(uint32_t n) { return (size_t)n * 32; }
size_t sig2_bytes(uint32_t n) { return (size_t)n * kSig2Bytes; }

uint32_t signature_grams(uint32_t sigma, uint32_t want) {
  uint32_t q = 1;
  for (uint64_t c = sigma; c < want && q < 8 && sigma > 1; c *= sigma) ++q;
  return q;
}

// Gram lengths: the shortest q with at least 20 (first level) and 256 (second)
// different grams.  Single symbols of the first level are dealt to its 28
// buckets by their counts in the input, the most frequent first, each to the
// bucket with the smallest total: the sums of differences grow with the
// number of evenly filled buckets.
SigShape signature_shape(uint32_t sigma, const uint64_t* counts_by_code) {
  SigShape g{};
  g.q1 = signature_grams(sigma, 20);
  g.q2 = signature_grams(sigma, kSig2);
  uint32_t order[256];
  for (uint32_t c = 0; c < 256; ++c) order[c] = c;
  std::stable_sort(order, order + sigma, [&](uint32_t a, uint32_t b) { return counts_by_code[a] > counts_by_code[b]; });
  uint64_t load[kSig1] = {0};
  for (uint32_t k = 0; k < sigma; ++k) {
    int best = 0;
    for (int b = 1; b < kSig1; ++b)
      if (load[b] < load[best]) best = b;
    g.bucket[order[k]] = (uint8_t)best;
    load[best] += counts_by_code[order[k]];
  }
  return g;
}

int launch_signatures(const uint8_t* codes, const int64_t* offsets, const uint32_t* sid_of, uint32_t n,
                      const SigShape& g, const unsigned long long* sampled, uint64_t min_sampled, uint4* sig1,
                      uint32_t* sig2, cudaStream_t s) {
  if (!n) return MJ_OK;
  signature_kernel<<<grid_for(n, kSigWarps), 32 * kSigWarps, 0, s>>>(codes, offsets, sid_of, n, g, sampled, min_sampled,
                                                                     sig1, sig2);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

int launch_pair_bounds(const uint32_t* pi, const uint32_t* pj, const uint32_t* pk, uint32_t K, uint64_t m, uint32_t n,
                       const SigShape& g, const uint4* sig1, const uint4* sig2, uint8_t* rejected, uint32_t* ed,
                       cudaStream_t s) {
  if (!m) return MJ_OK;
  pair_bounds_kernel<<<grid_for(m), 256, 0, s>>>(pi, pj, pk, K, m, n, g.q1, g.q2, sig1, sig2, rejected, ed);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

bool string_pairs_fit(uint32_t widest) {
  return sizeof(PairShared<128, true>) + (size_t)widest / 8 <= kStringPairsSmemMax;
}

// Windows of 2^16 ranks and more take a CTA each with up to 142 KB of bitmap, so
// few are resident, and a string costs 6 us of its CTA's place however few
// candidates it has (72,000 / 200,000 / 500,000 / 1,000,000 reads of one length:
// 0.46 / 1.43 / 7.8 / 39 ms for 0.36 / 1.0 / 2.5 / 5.0 M raw pairs).  The general
// path takes 85-130 ps a raw pair of such inputs, and 100-300 ps to verify the
// candidate that it may be.  So strings pay from a raw pair per 0.25 ns of that
// on.  (Whole joins by strings, against this choice, the general path: 0.99 /
// 0.70, 2.21 / 0.94, 9.1 / 1.47, 41.3 / 2.39 ms; 450,000 text-like strings, 1.8 G
// raw pairs, go by strings: 44 ms, some 530 by the general path.)
uint64_t string_pairs_from(uint32_t n, uint32_t widest, int sms) {
  if (widest < 65536) return 0;
  const size_t smem = sizeof(PairShared<128, true>) + (size_t)widest / 8 + 1024;
  const uint64_t resident = std::min<uint64_t>(8, std::max<uint64_t>(1, (227u << 10) / smem));
  return (uint64_t)n * 24000 / ((uint64_t)sms * resident);
}

// About 2^17 records are sampled, whose table stays in L2 (2^20 of 5 M: 176 us).
static uint32_t likely_pairs_step(uint64_t n_rec) { return (uint32_t)std::max<uint64_t>(1, n_rec >> 17); }

uint32_t likely_pairs_slots(uint64_t n_rec) {   // 16 slots and more per sampled record
  uint32_t slots = 1024;
  while (slots < (1u << 22) && slots < 16 * (n_rec / likely_pairs_step(n_rec))) slots <<= 1;
  return slots;
}

int launch_likely_pairs(const PRec* recs, uint64_t n_rec, uint32_t K, uint32_t* table, unsigned long long* total,
                        cudaStream_t s) {
  const uint32_t slots = likely_pairs_slots(n_rec), step = likely_pairs_step(n_rec);
  MJ_CUDA_TRY(cudaMemsetAsync(table, 0, (size_t)slots * 4, s));
  MJ_CUDA_TRY(cudaMemsetAsync(total, 0, sizeof(*total), s));
  if (!n_rec) return MJ_OK;
  likely_pairs_kernel<<<grid_for(n_rec / step + 1), 256, 0, s>>>(recs, n_rec, step, K, table, slots - 1, total);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

uint64_t likely_pairs(uint64_t n_rec, uint64_t total) {
  const double step = likely_pairs_step(n_rec), m = (double)n_rec / step;
  const double met = m * m / 2 / likely_pairs_slots(n_rec);   // different records in one slot
  return (uint64_t)(std::max(0.0, (double)total - met) * step * step);
}

int launch_string_pairs(const PairArgs& a, uint32_t widest, cudaStream_t s) {
  return launch_string_pairs_s<false>(a, widest, s);
}

int launch_string_sample(const PairArgs& a, uint32_t widest, cudaStream_t s) {
  return launch_string_pairs_s<true>(a, widest, s);
}

int launch_listed_pairs(const ListArgs& a, cudaStream_t s) {
  listed_pairs_kernel<<<grid_for(a.in_cap), 256, 0, s>>>(a);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

}  // namespace mj
