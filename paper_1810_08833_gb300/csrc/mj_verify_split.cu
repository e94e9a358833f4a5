// Step a8 for short lists: verification with two lanes per pair, one for each
// half of the columns (the recurrence and its band: mj_verify_diag.cuh).
#include "mj_verify_diag.cuh"

namespace mj {
namespace {

// D[m][n] of a split pair from its halves' last columns, by the whole warp:
// lane l holds the forward half (column h), lane l + 1 the reversed one (column
// n - h of the reversed strings).  A path of cost <= k crosses from column h
// at some band row h + dlo + s, which is row dhi - dlo - s of the reversed
// half's band, so the distance is the least sum of the two halves' values over
// s (their values are exact along paths in the band, and never too small).
template <int W, int P>
__device__ __forceinline__ uint32_t join_halves(const PairState<W, P>& st, int l, int lane) {
  uint32_t fp[W], fm[W], gp[W], gm[W];
#pragma unroll
  for (int w = 0; w < W; ++w) {
    fp[w] = __shfl_sync(0xffffffffu, st.Pv[w], l);
    fm[w] = __shfl_sync(0xffffffffu, st.Mv[w], l);
    gp[w] = __shfl_sync(0xffffffffu, st.Pv[w], l + 1);
    gm[w] = __shfl_sync(0xffffffffu, st.Mv[w], l + 1);
  }
  const int32_t base = __shfl_sync(0xffffffffu, st.score, l) + __shfl_sync(0xffffffffu, st.score, l + 1);
  const int32_t width = __shfl_sync(0xffffffffu, st.width, l);
  int32_t best = 0x3fffffff;
  for (int32_t s = lane; s <= width; s += 32) {
    int32_t v = base;
    const int32_t u = width - s;
#pragma unroll
    for (int w = 0; w < W; ++w) {   // the deltas of the rows up to s (u)
      const uint32_t ms = s >= 32 * w + 32 ? 0xffffffffu : (s <= 32 * w ? 0u : ((1u << (s - 32 * w)) - 1u));
      const uint32_t mu = u >= 32 * w + 32 ? 0xffffffffu : (u <= 32 * w ? 0u : ((1u << (u - 32 * w)) - 1u));
      v += (int32_t)__popc(fp[w] & ms) - (int32_t)__popc(fm[w] & ms);
      v += (int32_t)__popc(gp[w] & mu) - (int32_t)__popc(gm[w] & mu);
    }
    best = min(best, v);
  }
  return (uint32_t)__reduce_min_sync(0xffffffffu, best);
}

// verify_diag_kernel with two lanes per pair, for lists of at most one pair
// per two lanes: a pair's columns are a serial chain, and with every pair in
// flight at once the longest chain is the kernel's time.  The two halves of
// the columns run at once, one from each end, which halves the chain; a pair
// is rejected as soon as either half alone exceeds its band (a pair that only
// their sum rejects runs to the middle).  Measured, one lane per pair against
// two: 2,200 pairs of 5,000-base reads (4 words) 393 -> 281 us, 4,500 of
// 1,500-symbol text (3 words) 210 -> 143, 1,300 of 700 bytes (2 words) 229 -> 160.
template <int W, int P>
__global__ void __launch_bounds__(128) verify_split_kernel(VerifyArgs a, uint64_t PW, uint32_t GW, int lanes,
                                                           unsigned long long* __restrict__ next) {
  extern __shared__ __align__(16) uint32_t vsm[];
  const int lane = threadIdx.x & 31;
  const bool rev = lane & 1;
  const uint64_t q_lo = a.range_lo ? *a.range_lo : 0;
  const uint64_t q_hi = a.range_hi ? *a.range_hi : a.m;
  PairState<W, P> st;
  bool active = false, running = false;   // the pair is held, this half has columns left
  bool more = lane < lanes;
  uint64_t work = 0, nskip = 0;
  while (true) {
    const bool need = !active && more;   // the same in both lanes of a pair
    const uint32_t nmask = __ballot_sync(0xffffffffu, need && !rev);
    if (nmask) {
      unsigned long long base = 0;
      const int leader = __ffs(nmask) - 1;
      if (lane == leader) base = atomicAdd(next, (unsigned long long)__popc(nmask));
      base = __shfl_sync(0xffffffffu, base, leader);
      if (need) {
        const uint64_t q = q_lo + base + __popc(nmask & ((1u << (lane & ~1)) - 1u));
        if (q >= q_hi) {
          more = false;
        } else {
          const uint64_t t = a.order ? a.order[q] : q;
          const uint32_t* fed = a.first_ed ? a.first_ed : a.ed;
          const bool settled = a.skip_kband && a.skip_kband[t] < a.K && fed[t] <= a.skip_kband[t];
          if (settled) {
            if (a.first_ed && !rev) put_result(a, t, fed[t]);
            nskip += rev ? 0 : 1;
          } else {
            uint32_t res;
            if (pair_init<W, P, true>(st, a, GW, q, t, &res, rev)) {
              active = true;
              running = st.n > 0;
            } else if (!rev) {
              put_result(a, t, res);
            }
          }
        }
      }
    }
    if (!__any_sync(0xffffffffu, active || more)) break;
    uint32_t res = kHalfDone;
    if (running) {
      const int32_t j_before = st.j;
      if (pair_chunk<W, P, true>(st, a, PW, &res, vsm, GW, rev)) running = false;
      work += (uint64_t)(st.j - j_before) * W;
    }
    // both halves of a pair see its state
    const uint32_t rejected = __ballot_sync(0xffffffffu, active && res != kHalfDone);
    const uint32_t busy = __ballot_sync(0xffffffffu, running);
    const bool out = (rejected >> (lane & ~1)) & 3u;
    const bool whole = active && !out && !((busy >> (lane & ~1)) & 3u);
    if (active && out) {
      if (!rev) put_result(a, st.t, st.k + 1);
      active = running = false;
    }
    for (uint32_t rest = __ballot_sync(0xffffffffu, whole && !rev); rest; rest &= rest - 1) {
      const int l = __ffs(rest) - 1;
      const uint32_t d = join_halves<W, P>(st, l, lane);
      if (lane == l) put_result(a, st.t, d > st.k ? st.k + 1 : d);
    }
    if (whole) active = false;
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
int launch_split_wp(const VerifyArgs& a, uint64_t PW, uint32_t GW, unsigned long long* next, cudaStream_t s) {
  if (!a.codes) return MJ_ERR_ARG;
  constexpr size_t smem = digit_smem_bytes<W, P>();
  MJ_CUDA_TRY(cudaFuncSetAttribute(verify_split_kernel<W, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  // The fewest lanes per warp with at most one warp per scheduler: a warp's
  // loads take a wavefront per lane and its chunks last as long as the longest
  // lane's.  2,000 pairs, 8 lanes against 32: 500-symbol protein 76 -> 67 us,
  // 5,000-base reads 258 -> 246; 300 text pairs, 2 lanes: 134 -> 117; more
  // warps than that share a scheduler and take longer (2,000 pairs of reads, 2
  // lanes: 447).
  int dev = 0, sms = kNumSMsHint, lanes = 2;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  while (lanes < 32 && a.m * 2 > (uint64_t)lanes * 4 * sms) lanes *= 2;
  const uint64_t warps = (a.m * 2 + lanes - 1) / lanes;
  verify_split_kernel<W, P><<<(unsigned)((warps + 3) / 4), 128, smem, s>>>(a, PW, GW, lanes, next);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

template <int W>
int launch_split_w(const VerifyArgs& a, uint64_t PW, uint32_t GW, unsigned long long* next, cudaStream_t s) {
  if (a.bits <= 2) return launch_split_wp<W, 2>(a, PW, GW, next, s);
  if (a.bits <= 5) return launch_split_wp<W, 5>(a, PW, GW, next, s);
  if (a.bits == 7) return launch_split_wp<W, 7>(a, PW, GW, next, s);
  return launch_split_wp<W, 8>(a, PW, GW, next, s);
}

}  // namespace

int launch_verify_split(const VerifyArgs& a, uint64_t PW, uint32_t GW, int words, unsigned long long* next,
                        cudaStream_t s) {
  switch (words) {
    case 1: return launch_split_w<1>(a, PW, GW, next, s);
    case 2: return launch_split_w<2>(a, PW, GW, next, s);
    case 3: return launch_split_w<3>(a, PW, GW, next, s);
    case 4: return launch_split_w<4>(a, PW, GW, next, s);
    case 5: return launch_split_w<5>(a, PW, GW, next, s);
    case 6: return launch_split_w<6>(a, PW, GW, next, s);
    case 7: return launch_split_w<7>(a, PW, GW, next, s);
    case 8: return launch_split_w<8>(a, PW, GW, next, s);
    default: return MJ_ERR_UNSUPPORTED;
  }
}

}  // namespace mj
