// Step a8: verification of candidate pairs: bit-planes of the input, the
// one-lane-per-pair kernel for bands of up to eight words (the recurrence and
// its band: mj_verify_diag.cuh), and the choice among the verifiers.
#include <algorithm>

#include "mj_verify_diag.cuh"

namespace mj {
namespace {

constexpr int kMaxBits = 8;

// One 32-symbol word per thread (two 16-byte loads where aligned).
__global__ void build_planes_kernel(const uint8_t* __restrict__ bytes, uint64_t nbytes, RankTable rt, uint32_t bits,
                                    uint32_t* __restrict__ planes, uint64_t plane_words, uint32_t guard_words,
                                    uint8_t* __restrict__ codes) {
  __shared__ uint8_t s_rank[256];
  s_rank[threadIdx.x] = rt.r[threadIdx.x];
  __syncthreads();
  for (uint64_t w = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; w < plane_words;
       w += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t acc[kMaxBits] = {0};
    const int64_t c0 = ((int64_t)w - (int64_t)guard_words) * 32;
    uint32_t sym[8];
    const bool full = c0 >= 0 && (uint64_t)c0 + 32 <= nbytes && ((uintptr_t)(bytes + c0) & 15) == 0;
    if (full) {
      const uint4 u = __ldg(reinterpret_cast<const uint4*>(bytes + c0));
      const uint4 v = __ldg(reinterpret_cast<const uint4*>(bytes + c0 + 16));
      sym[0] = u.x; sym[1] = u.y; sym[2] = u.z; sym[3] = u.w;
      sym[4] = v.x; sym[5] = v.y; sym[6] = v.z; sym[7] = v.w;
    } else {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        uint32_t x = 0;
        for (int b = 0; b < 4; ++b) {
          const int64_t c = c0 + 4 * q + b;
          if (c >= 0 && (uint64_t)c < nbytes) x |= (uint32_t)__ldg(bytes + c) << (8 * b);
        }
        sym[q] = x;
      }
    }
    uint32_t cw[8] = {0, 0, 0, 0, 0, 0, 0, 0};   // the 32 rank codes, four per word
#pragma unroll
    for (int t = 0; t < 32; ++t) {
      const int64_t c = c0 + t;
      const uint32_t r = (c >= 0 && (uint64_t)c < nbytes) ? s_rank[(sym[t >> 2] >> (8 * (t & 3))) & 255u] : 0u;
      cw[t >> 2] |= r << (8 * (t & 3));
#pragma unroll
      for (int p = 0; p < kMaxBits; ++p) acc[p] |= ((r >> p) & 1u) << t;
    }
    if (codes && c0 >= 0 && (uint64_t)c0 < nbytes) {   // codes + c0 is 32-byte aligned, the buffer nbytes + 32 long
      *reinterpret_cast<uint4*>(codes + c0) = make_uint4(cw[0], cw[1], cw[2], cw[3]);
      *reinterpret_cast<uint4*>(codes + c0 + 16) = make_uint4(cw[4], cw[5], cw[6], cw[7]);
    }
    if (plane_stride(bits) == 2) {
      reinterpret_cast<uint2*>(planes)[w] = make_uint2(acc[0], acc[1]);
    } else {   // codes below 2^bits: the planes beyond are zero
      reinterpret_cast<uint4*>(planes)[2 * w] = make_uint4(acc[0], acc[1], acc[2], acc[3]);
      reinterpret_cast<uint4*>(planes)[2 * w + 1] = make_uint4(acc[4], acc[5], acc[6], acc[7]);
    }
  }
}

// Persistent verifier: every lane keeps one pair in flight and fetches the
// next pair index (warp-aggregated atomic on *next) as soon as its pair is
// decided, so early exits do not leave lanes idle behind slow pairs.
template <int W, int P>
__global__ void __launch_bounds__(128, (P == 7 && W <= 3) ? 7 : ((P == 5 && W <= 2) ? 8 : 1)) verify_diag_kernel(VerifyArgs a, uint64_t PW, uint32_t GW,
                                                          unsigned long long* __restrict__ next) {
  extern __shared__ __align__(16) uint32_t vsm[];   // the digit tables
  uint32_t* tab = vsm;
  const int lane = threadIdx.x & 31;
  const uint64_t q_lo = a.range_lo ? *a.range_lo : 0;
  const uint64_t q_hi = a.range_hi ? *a.range_hi : a.m;
  PairState<W, P> st;
  bool active = false;
  bool more = true;
  uint64_t work = 0, nskip = 0;
  while (true) {
    // lanes without a pair fetch the next indices
    const bool need = !active && more;
    const uint32_t nmask = __ballot_sync(0xffffffffu, need);
    if (nmask) {
      unsigned long long base = 0;
      const int leader = __ffs(nmask) - 1;
      if (lane == leader) base = atomicAdd(next, (unsigned long long)__popc(nmask));
      base = __shfl_sync(0xffffffffu, base, leader);
      if (need) {
        const uint64_t q = q_lo + base + __popc(nmask & ((1u << lane) - 1u));
        if (q >= q_hi) {
          more = false;
        } else {
          const uint64_t t = a.order ? a.order[q] : q;
          // a pair the first pass already decided needs nothing: the lane
          // stays idle and fetches again at the next iteration
          const uint32_t* fed = a.first_ed ? a.first_ed : a.ed;
          const bool settled = a.skip_kband && a.skip_kband[t] < a.K && fed[t] <= a.skip_kband[t];
          if (settled && a.first_ed) put_result(a, t, fed[t]);
          nskip += settled ? 1 : 0;
          if (!settled) {
            uint32_t res;
            if (pair_init<W, P>(st, a, GW, q, t, &res)) {
              active = true;
            } else {
              put_result(a, t, res);
            }
          }
        }
      }
    }
    if (!__any_sync(0xffffffffu, active || more)) break;
    if (active) {
      uint32_t res;
      const int32_t j_before = st.j;
      const bool done = pair_chunk<W, P>(st, a, PW, &res, tab, GW);
      work += (uint64_t)(st.j - j_before) * W;
      if (done) {
        put_result(a, st.t, res);
        active = false;
      }
    }
  }
  if (a.work) {
    for (int o = 16; o > 0; o >>= 1) work += __shfl_down_sync(0xffffffffu, work, o);
    if (lane == 0 && work) atomicAdd(a.work, (unsigned long long)work);
  }
  if (a.skipped) {
    for (int o = 16; o > 0; o >>= 1) nskip += __shfl_down_sync(0xffffffffu, nskip, o);
    if (lane == 0 && nskip) atomicAdd(a.skipped, (unsigned long long)nskip);
  }
}

template <int W, int P>
int launch_wp(const VerifyArgs& a, uint64_t PW, uint32_t GW, unsigned long long* next, cudaStream_t s) {
  int dev = 0, sms = kNumSMsHint, per_sm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const size_t smem = kDigitTables<P> ? digit_smem_bytes<W, P>() : 0;
  if (kDigitTables<P>) {
    if (!a.codes) return MJ_ERR_ARG;
    MJ_CUDA_TRY(cudaFuncSetAttribute(verify_diag_kernel<W, P>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem));
  }
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, verify_diag_kernel<W, P>, 128, smem);
  // at least ~3 pairs per lane, so that the shared queue evens out the early
  // exits (a warp lasts as long as its slowest lane), but at least 3 blocks
  // per SM to hide the recurrence's latency
  const uint64_t per_sm_pairs = (a.m + 3ull * 128 * sms - 1) / (3ull * 128 * sms);
  per_sm = (int)std::min<uint64_t>((uint64_t)per_sm, std::max<uint64_t>(3, per_sm_pairs));
  // Two planes leave registers for 6 blocks at bands of up to 4 words, but a sixth
  // only makes the lanes' rows push each other out of L1: 341,509 pairs of 5,000
  // reads at K = 102 2.63 ms with 6, 2.49 with 5; 700,000 4.34 and 4.19, at K = 60
  // 2.06 and 1.98.
  if (P == 2) per_sm = std::min(per_sm, 5);
  if (per_sm < 1) per_sm = 1;
  uint64_t need = (a.m + 127) / 128;
  uint64_t grid = (uint64_t)sms * per_sm;
  if (need < grid) grid = need;
  verify_diag_kernel<W, P><<<(unsigned)(grid ? grid : 1), 128, smem, s>>>(a, PW, GW, next);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

template <int W>
int launch_w(const VerifyArgs& a, uint64_t PW, uint32_t GW, unsigned long long* next, cudaStream_t s) {
  if (!a.codes) return launch_wp<W, kXnor8>(a, PW, GW, next, s);   // digit tables read B's rank codes
  if (a.bits <= 2) return launch_wp<W, 2>(a, PW, GW, next, s);
  if (a.bits <= 5) return launch_wp<W, 5>(a, PW, GW, next, s);
  if (a.bits == 7) return launch_wp<W, 7>(a, PW, GW, next, s);   // text (65-128 symbols)
  return launch_wp<W, 8>(a, PW, GW, next, s);
}

}  // namespace

int launch_build_planes(const uint8_t* bytes, uint64_t nbytes, const RankTable& rt, uint32_t bits,
                        uint32_t* planes, uint64_t plane_words, uint32_t guard_words, uint8_t* codes,
                        cudaStream_t s) {
  if (bits > (uint32_t)kMaxBits) return MJ_ERR_UNSUPPORTED;
  uint64_t blocks = (plane_words + 255) / 256;
  uint64_t cap = (uint64_t)kNumSMsHint * 32;
  build_planes_kernel<<<(unsigned)(blocks > cap ? cap : blocks), 256, 0, s>>>(bytes, nbytes, rt, bits, planes,
                                                                              plane_words, guard_words, codes);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

int verify_words_for(uint32_t kmax) {
  // widest band: d0 + 2 floor((k - d0) / 2) + 1 <= k + 1 bits
  return (int)((kmax + 1 + 31) / 32);
}

int wave_lanes_for(uint32_t kmax) {
  // blocks of one pair active at one step: floor((w + 30) / 33) + 1, w <= kmax + 1 (>= 64)
  uint32_t w = kmax + 1 < 64 ? 64 : kmax + 1;
  uint32_t cnt = (w + 30) / 33 + 1;
  uint32_t g = 2;
  while (g < cnt) g <<= 1;
  return (int)g;
}

int cta_lanes_for(uint32_t kmax) {
  // a lane's blocks b and b + G are 2G steps apart in the CTA schedule, so
  // G lanes hold bands with 34 G >= 32 + (dhi - dlo), dhi - dlo <= max(kmax, 63)
  const uint32_t w = kmax + 1 < 64 ? 64 : kmax + 1;
  const uint32_t need = (31 + w + 33) / 34;
  uint32_t g = 64;
  while (g < need) g <<= 1;
  return (int)g;
}

int fewest_lanes_for(uint32_t kmax) {
  const int g = wave_lanes_for(kmax);
  return g <= 32 ? g : cta_lanes_for(kmax);
}

bool verify_supported(uint32_t kmax, int kernel, int lanes) {
  if (kmax >= (1u << 16)) return false;
  const int W = verify_words_for(kmax);
  if (kernel == MJ_VERIFY_KERNEL_TUNED) kernel = MJ_VERIFY_KERNEL_AUTO, lanes = 0;
  if (kernel == MJ_VERIFY_KERNEL_AUTO) kernel = W <= 8 ? MJ_VERIFY_KERNEL_DIAGONAL : MJ_VERIFY_KERNEL_WAVEFRONT;
  if (kernel == MJ_VERIFY_KERNEL_DIAGONAL) return W <= 32;
  if (kernel != MJ_VERIFY_KERNEL_WAVEFRONT) return false;
  const bool cta = lanes > 32 || (lanes <= 0 && wave_lanes_for(kmax) > 32);
  const int need = cta ? cta_lanes_for(kmax) : wave_lanes_for(kmax), G = lanes > 0 ? lanes : need;
  return G >= need && G <= (cta ? kMaxCtaLanes : 32) && !(G & (G - 1));
}

int launch_verify(const VerifyArgs& a, uint64_t PW, uint32_t GW, uint32_t kmax, unsigned long long* next,
                  cudaStream_t s, int kernel, int lanes, bool next_is_zero) {
  if (a.m == 0) return MJ_OK;
  const int W = verify_words_for(kmax);
  if (kernel == MJ_VERIFY_KERNEL_AUTO) kernel = W <= 8 ? MJ_VERIFY_KERNEL_DIAGONAL : MJ_VERIFY_KERNEL_WAVEFRONT;
  if (kernel == MJ_VERIFY_KERNEL_WAVEFRONT) {
    if (!verify_supported(kmax, kernel, lanes)) return MJ_ERR_UNSUPPORTED;
    if (!next_is_zero) MJ_CUDA_TRY(cudaMemsetAsync(next, 0, sizeof(unsigned long long), s));
    return lanes > 0 ? launch_verify_wave(a, PW, GW, lanes, next, s)   // one word per lane
                     : launch_verify_wave_auto(a, PW, GW, kmax, next, s);
  }
  if (!next_is_zero) MJ_CUDA_TRY(cudaMemsetAsync(next, 0, sizeof(unsigned long long), s));
  if (kernel != MJ_VERIFY_KERNEL_DIAGONAL) return MJ_ERR_ARG;
  // every pair in flight at once with two lanes each, at three blocks of 128
  // threads per SM: then the longest pair is the kernel's time, and its halves
  // side by side take half of it
  int dev = 0, sms = kNumSMsHint;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (W <= 8 && a.codes && a.m * 2 <= 3ull * 128 * sms) return launch_verify_split(a, PW, GW, W, next, s);
  switch (W) {
    case 1: return launch_w<1>(a, PW, GW, next, s);
    case 2: return launch_w<2>(a, PW, GW, next, s);
    case 3: return launch_w<3>(a, PW, GW, next, s);
    case 4: return launch_w<4>(a, PW, GW, next, s);
    case 5: return launch_w<5>(a, PW, GW, next, s);
    case 6: return launch_w<6>(a, PW, GW, next, s);
    case 7: return launch_w<7>(a, PW, GW, next, s);
    case 8: return launch_w<8>(a, PW, GW, next, s);
    default: break;
  }
  // forced on bands of more than 8 words: the planes' layout goes by the bits
  if (plane_stride(a.bits) == 2)
    return W <= 16 ? launch_wp<16, 2>(a, PW, GW, next, s)
                   : (W <= 32 ? launch_wp<32, 2>(a, PW, GW, next, s) : MJ_ERR_UNSUPPORTED);
  if (W <= 16) return launch_wp<16, kXnor8>(a, PW, GW, next, s);
  if (W <= 32) return launch_wp<32, kXnor8>(a, PW, GW, next, s);
  return MJ_ERR_UNSUPPORTED;
}

}  // namespace mj
