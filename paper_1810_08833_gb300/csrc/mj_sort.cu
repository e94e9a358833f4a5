// Device-wide exclusive scans and an LSD radix sort of 64-bit keys with
// optional 32-bit values: the sorting primitives behind grouping the
// partition records (Alg. 3's hash join) and deduplicating candidate pairs
// (the last step of Alg. 3's join).
#include "mj_internal.cuh"

namespace mj {
namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;                          // per thread
constexpr int kScanTile = kScanThreads * kScanItems;   // 2048 per block

template <class T>
__device__ T block_exclusive_scan(T v, T* s_warp, T* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  T x = v;
  for (int o = 1; o < 32; o <<= 1) {
    T y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[wid] = x;
  __syncthreads();
  if (wid == 0) {
    T w = lane < kScanThreads / 32 ? s_warp[lane] : T(0);
    for (int o = 1; o < 32; o <<= 1) {
      T y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < kScanThreads / 32) s_warp[lane] = w;
  }
  __syncthreads();
  T wprefix = wid ? s_warp[wid - 1] : T(0);
  *total = s_warp[kScanThreads / 32 - 1];
  __syncthreads();
  return wprefix + x - v;
}

// Phase 1: per-block sums.
template <class TI, class TO>
__global__ void __launch_bounds__(kScanThreads) scan_reduce_kernel(const TI* __restrict__ in, uint64_t n,
                                                                  TO* __restrict__ block_sum) {
  __shared__ TO s_warp[kScanThreads / 32];
  uint64_t base = (uint64_t)blockIdx.x * kScanTile + (uint64_t)threadIdx.x * kScanItems;
  TO sum = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k)
    if (base + k < n) sum += (TO)in[base + k];
  TO tot;
  block_exclusive_scan<TO>(sum, s_warp, &tot);
  if (threadIdx.x == 0) block_sum[blockIdx.x] = tot;
}

// Phase 3: block-local exclusive scan plus the block's scanned prefix.
template <class TI, class TO>
__global__ void __launch_bounds__(kScanThreads) scan_down_kernel(const TI* __restrict__ in, TO* __restrict__ out,
                                                                uint64_t n, const TO* __restrict__ block_prefix) {
  __shared__ TO s_warp[kScanThreads / 32];
  uint64_t base = (uint64_t)blockIdx.x * kScanTile + (uint64_t)threadIdx.x * kScanItems;
  TO v[kScanItems];
  TO sum = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    v[k] = (base + k < n) ? (TO)in[base + k] : TO(0);
    sum += v[k];
  }
  TO tot;
  TO run = block_exclusive_scan<TO>(sum, s_warp, &tot) + (block_prefix ? block_prefix[blockIdx.x] : TO(0));
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    if (base + k < n) out[base + k] = run;
    run += v[k];
  }
}

// One block scans up to kOneScan elements: short scans are a launch's time
// (about 2 us a piece), so one launch replaces the two or three of the tiled
// form.  Rows of 4,096 elements, four consecutive ones per thread (one 16-byte
// load; up to 32 consecutive ones took a wavefront per lane and load: about
// 20,000 elements 9.0 us, now 3.5), all rows in flight, and one scan over the
// warps' sums of all rows.
constexpr int kOneThreads = 1024, kOneRows = 8;
constexpr uint64_t kOneScan = (uint64_t)kOneThreads * 4 * kOneRows;

template <class TI, class TO>
__global__ void __launch_bounds__(kOneThreads) scan_one_kernel(const TI* __restrict__ in, TO* __restrict__ out,
                                                               uint32_t n, TO* __restrict__ total_out) {
  __shared__ TO s_warp[kOneRows * 32];   // sums before each warp's elements of a row
  __shared__ TO s_group[kOneRows];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int rows = (int)((n + 4 * kOneThreads - 1) / (4 * kOneThreads));
  const bool wide = sizeof(TI) == 4 && ((uintptr_t)in & 15) == 0;
  TI v[kOneRows][4];
  TO sum[kOneRows], x[kOneRows];
#pragma unroll
  for (int k = 0; k < kOneRows; ++k) {
    const uint32_t at = 4 * (k * kOneThreads + threadIdx.x);
    if (wide && at + 4 <= n) {
      const uint4 u = *reinterpret_cast<const uint4*>(in + at);
      v[k][0] = (TI)u.x; v[k][1] = (TI)u.y; v[k][2] = (TI)u.z; v[k][3] = (TI)u.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) v[k][e] = at + e < n ? in[at + e] : TI(0);
    }
  }
#pragma unroll
  for (int k = 0; k < kOneRows; ++k) x[k] = sum[k] = (TO)v[k][0] + (TO)v[k][1] + (TO)v[k][2] + (TO)v[k][3];
  for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
    for (int k = 0; k < kOneRows; ++k) {
      if (k < rows) {
        const TO y = __shfl_up_sync(0xffffffffu, x[k], o);
        if (lane >= o) x[k] += y;
      }
    }
  }
  if (lane == 31) {
#pragma unroll
    for (int k = 0; k < kOneRows; ++k) s_warp[k * 32 + wid] = k < rows ? x[k] : TO(0);
  }
  __syncthreads();
  if (wid < kOneRows) {   // one warp per row of sums
    const TO own = s_warp[wid * 32 + lane];
    TO w = own;
    for (int o = 1; o < 32; o <<= 1) {
      const TO y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    s_warp[wid * 32 + lane] = w - own;
    if (lane == 31) s_group[wid] = w;
  }
  __syncthreads();
  TO before = 0;
#pragma unroll
  for (int k = 0; k < kOneRows; ++k) {
    if (k >= rows) break;
    TO run = before + s_warp[k * 32 + wid] + x[k] - sum[k];
    before += s_group[k];
    const uint32_t at = 4 * (k * kOneThreads + threadIdx.x);
    TO r[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      r[e] = run;
      run += (TO)v[k][e];
    }
    if (sizeof(TO) == 4 && ((uintptr_t)out & 15) == 0 && at + 4 <= n) {
      *reinterpret_cast<uint4*>(out + at) = make_uint4((uint32_t)r[0], (uint32_t)r[1], (uint32_t)r[2], (uint32_t)r[3]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (at + e < n) out[at + e] = r[e];
    }
  }
  if (total_out && threadIdx.x == 0) *total_out = before;
}

uint64_t blocks_for(uint64_t n) { return (n + kScanTile - 1) / kScanTile; }

// temp elements needed by exclusive_scan: 2 per block at every level
size_t scan_temp_elems(uint64_t n) {
  size_t e = 0;
  while (n > kOneScan) {
    uint64_t b = blocks_for(n);
    e += 2 * b;
    n = b;
  }
  return e + 2;
}

// Exclusive scan of `in` (type TI) into `out` (type TO, may alias `in`); the
// total of all inputs goes to the device word total_out if non-null.
// Reduce-then-scan: block sums, a recursive scan of the sums, then a
// block-local scan offset by the scanned sums.
template <class TI, class TO>
int exclusive_scan(const TI* in, TO* out, uint64_t n, TO* temp, TO* total_out, cudaStream_t s) {
  if (n == 0) {
    if (total_out) MJ_CUDA_TRY(cudaMemsetAsync(total_out, 0, sizeof(TO), s));
    return MJ_OK;
  }
  if (n <= kOneScan) {
    scan_one_kernel<TI, TO><<<1, kOneThreads, 0, s>>>(in, out, (uint32_t)n, total_out);
    MJ_KERNEL_DONE();
    return MJ_OK;
  }
  const uint64_t b = blocks_for(n);
  TO* sums = temp;
  TO* sums_scanned = temp + b;
  scan_reduce_kernel<TI, TO><<<(unsigned)b, kScanThreads, 0, s>>>(in, n, sums);
  MJ_KERNEL_DONE();
  MJ_TRY((exclusive_scan<TO, TO>(sums, sums_scanned, b, temp + 2 * b, total_out, s)));
  scan_down_kernel<TI, TO><<<(unsigned)b, kScanThreads, 0, s>>>(in, out, n, sums_scanned);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

// ---------------------------------------------------------------- radix sort
constexpr int kSortThreads = 256;
constexpr int kSortItems = 16;
constexpr int kSortTile = kSortThreads * kSortItems;  // 4096 keys per tile

template <class KT>
__global__ void __launch_bounds__(kSortThreads) radix_hist_kernel(const KT* __restrict__ keys, uint64_t n,
                                                                  int shift, uint32_t num_tiles,
                                                                  uint32_t* __restrict__ hist) {
  __shared__ uint32_t s_hist[256];
  s_hist[threadIdx.x] = 0;
  __syncthreads();
  uint64_t base = (uint64_t)blockIdx.x * kSortTile;
  // all 16 loads in flight: with few tiles the kernel is a load's latency
  uint32_t d[kSortItems];
#pragma unroll
  for (int k = 0; k < kSortItems; ++k) {
    const uint64_t idx = base + (uint64_t)k * kSortThreads + threadIdx.x;
    d[k] = idx < n ? (uint32_t)(keys[idx] >> shift) & 255u : 256u;
  }
#pragma unroll
  for (int k = 0; k < kSortItems; ++k)
    if (d[k] < 256u) atomicAdd(&s_hist[d[k]], 1u);
  __syncthreads();
  hist[(uint64_t)threadIdx.x * num_tiles + blockIdx.x] = s_hist[threadIdx.x];
}

// Stable scatter of one tile.  Warp w owns items [w*512, w*512+512) of the
// tile, taken in 16 rounds of 32 consecutive items; ranks among equal digits
// come from __match_any_sync within a round plus running per-warp counters.
// The tile is first placed in digit order in shared memory, then written out
// item by item in that order: items of one digit go to consecutive global
// addresses, so a warp's stores form a few contiguous runs.
template <class KT>
constexpr size_t kScatterSmem = (size_t)kSortTile * (sizeof(KT) + sizeof(uint32_t));
constexpr int kScatThreads = 512;                       // threads of the scatter kernel
constexpr int kScatItems = kSortTile / kScatThreads;    // items per thread
constexpr int kScatWarps = kScatThreads / 32;

template <class KT>
__global__ void __launch_bounds__(kScatThreads) radix_scatter_kernel(
    const KT* __restrict__ keys, const uint32_t* __restrict__ vals, uint64_t n, int shift,
    uint32_t num_tiles, const uint32_t* __restrict__ offs, KT* __restrict__ keys_out,
    uint32_t* __restrict__ vals_out) {
  extern __shared__ __align__(16) uint8_t smem[];
  KT* s_keys = reinterpret_cast<KT*>(smem);
  uint32_t* s_vals = reinterpret_cast<uint32_t*>(smem + (size_t)kSortTile * sizeof(KT));
  __shared__ uint32_t s_cnt[kScatWarps][256];
  __shared__ uint32_t s_start[256];   // first local position of each digit
  __shared__ uint32_t s_goff[256];    // global position of each digit's first item
  __shared__ uint32_t s_wsum[8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int d = threadIdx.x; d < kScatWarps * 256; d += kScatThreads) (&s_cnt[0][0])[d] = 0;
  if (threadIdx.x < 256) s_goff[threadIdx.x] = offs[(uint64_t)threadIdx.x * num_tiles + blockIdx.x];
  __syncthreads();
  const uint64_t tile0 = (uint64_t)blockIdx.x * kSortTile;
  const uint64_t base = tile0 + (uint64_t)wid * (kSortTile / kScatWarps);
  const uint32_t valid = (uint32_t)min((uint64_t)kSortTile, n - tile0);
  KT k_[kScatItems];
  uint32_t rank_[kScatItems];
  const uint32_t lt = (1u << lane) - 1;
#pragma unroll
  for (int r = 0; r < kScatItems; ++r) {
    const uint64_t idx = base + (uint64_t)r * 32 + lane;
    k_[r] = idx < n ? keys[idx] : ~KT(0);
  }
#pragma unroll
  for (int r = 0; r < kScatItems; ++r) {
    // invalid items sit at the end of the last tile: digit 255 after every
    // valid item, so they take the last local positions
    const uint32_t d = (uint32_t)(k_[r] >> shift) & 255u;
    const uint32_t peers = __match_any_sync(0xffffffffu, d);
    const uint32_t before = __popc(peers & lt);
    const uint32_t cnt = s_cnt[wid][d];
    rank_[r] = cnt + before;
    __syncwarp();
    if (before == 0) s_cnt[wid][d] = cnt + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  // per digit: exclusive prefix over warps; the digit's tile total, then an
  // exclusive scan over digits (threads 0..255, warps 0..7) gives its first
  // local position
  uint32_t run = 0, x = 0;
  if (threadIdx.x < 256) {
    const uint32_t d = threadIdx.x;
    for (int w = 0; w < kScatWarps; ++w) {
      const uint32_t c = s_cnt[w][d];
      s_cnt[w][d] = run;
      run += c;
    }
    x = run;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_wsum[wid] = x;
  }
  __syncthreads();
  if (threadIdx.x < 256) {
    uint32_t pre = 0;
    for (int w = 0; w < wid; ++w) pre += s_wsum[w];
    s_start[threadIdx.x] = pre + x - run;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kScatItems; ++r) {
    const uint32_t d = (uint32_t)(k_[r] >> shift) & 255u;
    const uint32_t pos = s_start[d] + s_cnt[wid][d] + rank_[r];
    s_keys[pos] = k_[r];
    if (vals) {
      const uint64_t idx = base + (uint64_t)r * 32 + lane;
      s_vals[pos] = idx < n ? vals[idx] : 0u;
    }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kScatItems; ++r) {
    const uint32_t i = (uint32_t)r * kScatThreads + threadIdx.x;
    if (i < valid) {
      const KT key = s_keys[i];
      const uint32_t d = (uint32_t)(key >> shift) & 255u;
      const uint32_t dst = s_goff[d] + (i - s_start[d]);
      keys_out[dst] = key;
      if (vals) vals_out[dst] = s_vals[i];
    }
  }
}

// Stable sort of up to kOneSort keys (and values) by one block, all passes in
// shared memory: 3 launches per pass of the tiled form cost more than the
// sort.  Thread t of warp w takes items 512 w + 32 r + lane in round r; the
// ranks are those of radix_scatter_kernel.
constexpr int kOneSortThreads = 1024;
constexpr int kOneSortWarps = kOneSortThreads / 32;
template <class KT>
constexpr uint32_t kOneSort = sizeof(KT) == 4 ? 16384 : 8192;

template <class KT, int ITEMS>
__global__ void __launch_bounds__(kOneSortThreads) radix_one_kernel(KT* __restrict__ keys, uint32_t* __restrict__ vals,
                                                                    uint32_t n, int bit_lo, int bit_hi) {
  extern __shared__ __align__(16) uint8_t smem[];
  KT* s_keys = reinterpret_cast<KT*>(smem);
  uint32_t* s_vals = reinterpret_cast<uint32_t*>(smem + (size_t)kOneSortThreads * ITEMS * sizeof(KT));
  uint32_t(*s_cnt)[256] = reinterpret_cast<uint32_t(*)[256]>(s_vals + (size_t)kOneSortThreads * ITEMS);
  __shared__ uint32_t s_start[256];
  __shared__ uint32_t s_wsum[8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t lt = (1u << lane) - 1;
  KT k_[ITEMS];
  uint32_t v_[ITEMS], rank_[ITEMS];
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const uint32_t i = (uint32_t)(wid * ITEMS + r) * 32 + lane;
    k_[r] = i < n ? keys[i] : ~KT(0);
    v_[r] = i < n && vals ? vals[i] : 0u;
  }
  for (int shift = bit_lo; shift < bit_hi; shift += 8) {
    for (int d = threadIdx.x; d < kOneSortWarps * 256; d += kOneSortThreads) (&s_cnt[0][0])[d] = 0;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {   // items past n have the last digit and come last in the input
      const uint32_t d = (uint32_t)(k_[r] >> shift) & 255u;
      const uint32_t peers = __match_any_sync(0xffffffffu, d);
      const uint32_t before = __popc(peers & lt);
      const uint32_t cnt = s_cnt[wid][d];
      rank_[r] = cnt + before;
      __syncwarp();
      if (before == 0) s_cnt[wid][d] = cnt + __popc(peers);
      __syncwarp();
    }
    __syncthreads();
    uint32_t run = 0, x = 0;
    if (threadIdx.x < 256) {
      for (int w = 0; w < kOneSortWarps; ++w) {
        const uint32_t c = s_cnt[w][threadIdx.x];
        s_cnt[w][threadIdx.x] = run;
        run += c;
      }
      x = run;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (lane == 31) s_wsum[wid] = x;
    }
    __syncthreads();
    if (threadIdx.x < 256) {
      uint32_t pre = 0;
      for (int w = 0; w < wid; ++w) pre += s_wsum[w];
      s_start[threadIdx.x] = pre + x - run;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      const uint32_t d = (uint32_t)(k_[r] >> shift) & 255u;
      const uint32_t pos = s_start[d] + s_cnt[wid][d] + rank_[r];
      s_keys[pos] = k_[r];
      s_vals[pos] = v_[r];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      const uint32_t i = (uint32_t)(wid * ITEMS + r) * 32 + lane;
      k_[r] = s_keys[i];
      v_[r] = s_vals[i];
    }
    __syncthreads();
  }
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const uint32_t i = (uint32_t)(wid * ITEMS + r) * 32 + lane;
    if (i < n) {
      keys[i] = k_[r];
      if (vals) vals[i] = v_[r];
    }
  }
}

template <class KT, int ITEMS>
int launch_radix_one(KT* keys, uint32_t* vals, uint32_t n, int bit_lo, int bit_hi, cudaStream_t s) {
  constexpr size_t smem = (size_t)kOneSortThreads * ITEMS * (sizeof(KT) + 4) + (size_t)kOneSortWarps * 256 * 4;
  MJ_CUDA_TRY(cudaFuncSetAttribute(radix_one_kernel<KT, ITEMS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  radix_one_kernel<KT, ITEMS><<<1, kOneSortThreads, smem, s>>>(keys, vals, n, bit_lo, bit_hi);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

}  // namespace

size_t scan_temp_bytes(uint64_t n) { return scan_temp_elems(n) * sizeof(uint64_t) + 64; }

int launch_exclusive_scan_u32(const uint32_t* in, uint32_t* out, uint64_t n, void* temp, uint32_t* total_out,
                              cudaStream_t s) {
  return exclusive_scan<uint32_t, uint32_t>(in, out, n, static_cast<uint32_t*>(temp), total_out, s);
}

int launch_exclusive_scan_u64(const uint64_t* in, uint64_t* out, uint64_t n, void* temp, uint64_t* total_out,
                              cudaStream_t s) {
  return exclusive_scan<uint64_t, uint64_t>(in, out, n, static_cast<uint64_t*>(temp), total_out, s);
}

int launch_exclusive_scan_u32_to_u64(const uint32_t* in, uint64_t* out, uint64_t n, void* temp,
                                     uint64_t* total_out, cudaStream_t s) {
  return exclusive_scan<uint32_t, uint64_t>(in, out, n, static_cast<uint64_t*>(temp), total_out, s);
}

size_t radix_temp_bytes(uint64_t n) {
  uint64_t tiles = (n + kSortTile - 1) / kSortTile;
  uint64_t h = tiles * 256;
  return 2 * h * sizeof(uint32_t) + scan_temp_bytes(h) + 256;
}

namespace {

template <class KT>
int radix_sort(KT* keys, KT* keys_alt, uint32_t* vals, uint32_t* vals_alt, uint64_t n, int bit_lo, int bit_hi,
               void* temp, bool* result_in_alt, cudaStream_t s) {
  *result_in_alt = false;
  if (n <= 1 || bit_hi <= bit_lo) return MJ_OK;
  if (n >= (1ull << 32)) return MJ_ERR_UNSUPPORTED;
  if (n <= kOneSort<KT>) {
    const uint32_t m = (uint32_t)n;
    if (m <= 1024) return launch_radix_one<KT, 1>(keys, vals, m, bit_lo, bit_hi, s);
    if (m <= 4096) return launch_radix_one<KT, 4>(keys, vals, m, bit_lo, bit_hi, s);
    if (m <= 8192) return launch_radix_one<KT, 8>(keys, vals, m, bit_lo, bit_hi, s);
    if constexpr (sizeof(KT) == 4) {   // 16 items per thread spill registers
      if (m <= 12288) return launch_radix_one<KT, 12>(keys, vals, m, bit_lo, bit_hi, s);
      return launch_radix_one<KT, 16>(keys, vals, m, bit_lo, bit_hi, s);
    }
  }
  const uint32_t tiles = (uint32_t)((n + kSortTile - 1) / kSortTile);
  const uint64_t h = (uint64_t)tiles * 256;
  uint32_t* hist = static_cast<uint32_t*>(temp);
  uint32_t* offs = hist + h;
  void* scan_tmp = offs + h;
  KT* src_k = keys;
  KT* dst_k = keys_alt;
  uint32_t* src_v = vals;
  uint32_t* dst_v = vals_alt;
  bool alt = false;
  MJ_CUDA_TRY(cudaFuncSetAttribute(radix_scatter_kernel<KT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)kScatterSmem<KT>));
  for (int shift = bit_lo; shift < bit_hi; shift += 8) {
    radix_hist_kernel<KT><<<tiles, kSortThreads, 0, s>>>(src_k, n, shift, tiles, hist);
    MJ_KERNEL_DONE();
    MJ_TRY(launch_exclusive_scan_u32(hist, offs, h, scan_tmp, nullptr, s));
    radix_scatter_kernel<KT><<<tiles, kScatThreads, kScatterSmem<KT>, s>>>(src_k, src_v, n, shift, tiles, offs, dst_k,
                                                                    dst_v);
    MJ_KERNEL_DONE();
    std::swap(src_k, dst_k);
    std::swap(src_v, dst_v);
    alt = !alt;
  }
  *result_in_alt = alt;
  return MJ_OK;
}

}  // namespace

int radix_sort_u64(uint64_t* keys, uint64_t* keys_alt, uint32_t* vals, uint32_t* vals_alt, uint64_t n, int bit_lo,
                   int bit_hi, void* temp, bool* result_in_alt, cudaStream_t s) {
  return radix_sort(keys, keys_alt, vals, vals_alt, n, bit_lo, bit_hi, temp, result_in_alt, s);
}

int radix_sort_u32(uint32_t* keys, uint32_t* keys_alt, uint32_t* vals, uint32_t* vals_alt, uint64_t n, int bit_lo,
                   int bit_hi, void* temp, bool* result_in_alt, cudaStream_t s) {
  return radix_sort(keys, keys_alt, vals, vals_alt, n, bit_lo, bit_hi, temp, result_in_alt, s);
}

}  // namespace mj
