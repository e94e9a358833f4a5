// Step a8 for wide bands: row-fixed blocks with a skewed wavefront, within one
// warp (G lanes per pair) or one CTA of several warps per pair.
#include <algorithm>
#include <cmath>

#include "mj_verify_diag.cuh"

namespace mj {
namespace {

// ---------------------------------------------------------------- wide bands
// Row-fixed blocks with a skewed wavefront, G lanes per pair.
//
// Rows are cut into blocks of R = 32 V rows (block b = rows Rb+1 .. Rb+R, V
// 32-bit words per vector; below V = 1 unless said); lane b mod G of the pair's group owns block b.  Block b
// advances column j at step s = j + b: it needs the horizontal delta of the
// row just above it in column j, which the lane owning block b-1 produced one
// step earlier and passes on by a shuffle.  A block works on the columns in
// which some of its rows lie in the band [j + dlo, j + dhi]; outside, a block
// entering the band starts from vertical deltas of +1 and the row above a
// retired block gets a horizontal delta of +1 (the same over-estimates as the
// diagonal kernel).  With an incoming horizontal delta hin in {-1, 0, +1}, a
// block step is the recurrence of the diagonal kernel with the top row's
// chain seeded by hin: Xh's carry chain starts set when hin = -1, and the
// shifted-in top bit of Ph (Mh) is set when hin = +1 (-1).  Each block keeps
// D of its bottom row; the bottom row of the block holding row m at column n
// gives D[m][n], and the block holding row j + d0 at column j gives the
// diagonal lower bound used for the early exit.
constexpr int kWaveSteps = 32;   // wavefront steps between refills and votes (<= 32: B's bits per reload)

// Each lane publishes one word per wavefront step for the lane holding the
// next block of rows:
//   bit 31      the block's bottom row gained +1 in this column (hout = +1)
//   bits 1..30  D at the block's bottom row in this column (the score)
//   bit 0       hout = -1
// The next lane reads it only in the columns that block b - 1 shares with
// block b; elsewhere the top row's delta is kIdle, +1 (the band's edge).
constexpr uint32_t kIdle = 0x80000000u;
constexpr int32_t kDeadU = -0x40000000;   // step offset of a lane without a block
constexpr uint32_t kMaxLen = 1u << 27;     // scores must fit bits 1..30

template <int P>
__device__ __forceinline__ void wave_load_bits(const VerifyArgs& a, uint64_t PW, uint64_t pos, uint32_t (&v)[P],
                                               bool reverse) {
  uint32_t lo[P], hi[P];
  load_plane_words<P>(a.planes, (int64_t)(pos >> 5), lo);
  load_plane_words<P>(a.planes, (int64_t)(pos >> 5) + 1, hi);
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const uint32_t x = __funnelshift_r(lo[p], hi[p], (uint32_t)(pos & 31));
    v[p] = reverse ? __brev(x) : x;
  }
}

// One column of a 32-row block (Myers' step in Hyyro's formulation).  wv
// carries the horizontal delta entering the top row (bit 31: +1, bit 0: -1,
// neither: 0); B's symbol is bit 31 of bw[] (consumed, shifted out); T's
// score bits (1..30) follow the bottom row; Ph keeps the bottom row's +1 in
// bit 31 and hn is its -1.  Bit extraction, shifts and disjoint ORs are
// written as integer multiply-adds, which the FMA pipe can take: the logic
// ops already fill the ALU pipe.
__device__ __forceinline__ uint32_t mad_lo(uint32_t a, uint32_t b, uint32_t c) {   // a * b + c on the FMA pipe
  uint32_t d;
  asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

// A block of V words (rows 32 V b + 1 ..) takes the same step, the carry of
// (Eq & Pv) + Pv and the shifted-in bits running through its words.
// pub: the word published to the next lane, ((Ph & 2^31) | T) + hn with the
// updated T (bit 31 and bit 0 of T are clear), formed by multiply-adds as
// T_old + hp (2^31 + 2) - hn.  Ph and hn: of the bottom word.
template <int V>
__device__ __forceinline__ void wave_column(const uint32_t (&Eq)[V], uint32_t wv, uint32_t (&Pv)[V], uint32_t (&Mv)[V],
                                            uint32_t& T, uint32_t& Ph_out, uint32_t& hn, uint32_t& pub) {
  uint32_t EP[V], SUM[V], Ph[V], Mh[V];
  const uint32_t hin_neg = wv & 1u;
  const uint32_t hin_pos = __umulhi(wv, 2u);
#pragma unroll
  for (int w = 0; w < V; ++w) EP[w] = (w == 0 ? Eq[w] | hin_neg : Eq[w]) & Pv[w];
  add_chain<V>::run(EP, Pv, SUM);
#pragma unroll
  for (int w = 0; w < V; ++w) {
    const uint32_t Xh = (SUM[w] ^ Pv[w]) | (w == 0 ? Eq[w] | hin_neg : Eq[w]);
    Ph[w] = Mv[w] | ~(Xh | Pv[w]);
    Mh[w] = Pv[w] & Xh;
  }
  hn = __umulhi(Mh[V - 1], 2u);
  const uint32_t hp = __umulhi(Ph[V - 1], 2u);
  pub = mad_lo(hn, 0xffffffffu, mad_lo(hp, 0x80000002u, T));
  T = mad_lo(hn, 0xfffffffeu, mad_lo(hp, 2u, T));
#pragma unroll
  for (int w = V - 1; w >= 0; --w) {
    const uint32_t Xv = Eq[w] | Mv[w];
    const uint32_t Ph1 = w ? __funnelshift_l(Ph[w - 1], Ph[w], 1) : Ph[w] * 2u + hin_pos;   // (Ph << 1) | hin > 0
    const uint32_t Mh1 = w ? __funnelshift_l(Mh[w - 1], Mh[w], 1) : Mh[w] * 2u + hin_neg;   // (Mh << 1) | hin < 0
    Pv[w] = Mh1 | ~(Xv | Ph1);
    Mv[w] = Ph1 & Xv;
  }
  Ph_out = Ph[V - 1];
}

// Sum of the vertical deltas of a block's rows below row r (0 .. 32 V - 1).
template <int V>
__device__ __forceinline__ int32_t deltas_below(const uint32_t (&Pv)[V], const uint32_t (&Mv)[V], int r) {
  int32_t d = 0;
#pragma unroll
  for (int w = 0; w < V; ++w) {
    const int x = r - 32 * w;
    const uint32_t below = x < 0 ? 0xffffffffu : (x >= 31 ? 0u : (0xffffffffu << (x + 1)));
    d += (int32_t)__popc(Pv[w] & below) - (int32_t)__popc(Mv[w] & below);
  }
  return d;
}

// The planes of the 32 V rows from plane bit pos on.
template <int P, int V>
__device__ __forceinline__ void wave_load_rows(const VerifyArgs& a, uint64_t pos, uint32_t (&pa)[P][V]) {
  uint32_t x0[P];
  load_plane_words<P>(a.planes, (int64_t)(pos >> 5), x0);
#pragma unroll
  for (int w = 0; w < V; ++w) {
    uint32_t x1[P];
    load_plane_words<P>(a.planes, (int64_t)(pos >> 5) + w + 1, x1);
#pragma unroll
    for (int p = 0; p < P; ++p) {
      pa[p][w] = __funnelshift_r(x0[p], x1[p], (uint32_t)(pos & 31));
      x0[p] = x1[p];
    }
  }
}

// Match bits of the block's rows with B's symbol (bit 31 of bw[], consumed).
// From the block's planes:
template <int P, int V>
__device__ __forceinline__ void eq_planes(const uint32_t (&pa)[P][V], uint32_t (&bw)[P], uint32_t (&Eq)[V]) {
#pragma unroll
  for (int w = 0; w < V; ++w) Eq[w] = 0xffffffffu;
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const uint32_t xb = (uint32_t)__mulhi((int32_t)bw[p], 1);   // B's bit p broadcast (sign of bw)
#pragma unroll
    for (int w = 0; w < V; ++w) Eq[w] &= ~(pa[p][w] ^ xb);
    bw[p] *= 2u;
  }
}

// For two planes, from a table in shared memory: a lane's rows for each of the
// four symbols, in units of four words, then two, then one, each unit laid out
// [symbol][lane] (a lane meets no other lane's banks, whatever the symbols).
// The XNORs are 2 of the 12 logic operations per word on the ALU pipe, which
// bounds the kernel (82% busy, the FMA pipe 10%); the loads and their address
// (multiply-adds) take none.  Join of long reads at K = 1000 (5 words) 31.9 ->
// 28.5 ms, 20,000 pairs at K = 4000 (4 words) 15.0 -> 13.4 ms, 300 pairs 1.43 ->
// 1.34 ms; with one or two words a column's chain decides, not the ALU: K =
// 700, 300 pairs 1.21 -> 1.29 ms, so they keep the planes.
constexpr int kTableFrom = 3;
template <int V>
constexpr int kEqTableWords = 4 * 32 * V;   // of a warp

template <int V>
__device__ __forceinline__ void eq_store(uint32_t* tab, int lane, const uint32_t (&pa)[2][V]) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
#pragma unroll
    for (int w = 0; w < V; ++w) {
      const uint32_t e = (c & 1 ? pa[0][w] : ~pa[0][w]) & (c & 2 ? pa[1][w] : ~pa[1][w]);
      const int unit = w < V / 4 * 4 ? 4 : (w < V / 2 * 2 ? 2 : 1);
      const int first = w / unit * unit;   // units before hold words 0 .. first - 1
      tab[first * 128 + (c * 32 + lane) * unit + (w - first)] = e;
    }
  }
}

template <int V>
__device__ __forceinline__ void eq_load(const uint32_t* tab, int lane, uint32_t (&bw)[2], uint32_t (&Eq)[V]) {
  const uint32_t b0 = __umulhi(bw[0], 2u), b1 = __umulhi(bw[1], 2u);
  bw[0] *= 2u;
  bw[1] *= 2u;
  const uint32_t c32 = mad_lo(b1, 64u, mad_lo(b0, 32u, (uint32_t)lane));   // symbol * 32 + lane
#pragma unroll
  for (int w = 0; w + 4 <= V; w += 4) {
    const uint4 x = *reinterpret_cast<const uint4*>(tab + w * 128 + c32 * 4);
    Eq[w] = x.x;
    Eq[w + 1] = x.y;
    Eq[w + 2] = x.z;
    Eq[w + 3] = x.w;
  }
  if constexpr (V % 4 >= 2) {
    constexpr int w = V / 4 * 4;
    const uint2 x = *reinterpret_cast<const uint2*>(tab + w * 128 + c32 * 2);
    Eq[w] = x.x;
    Eq[w + 1] = x.y;
  }
  if constexpr (V % 2) Eq[V - 1] = tab[(V - 1) * 128 + c32];
}

template <int G, int P, int V>
__global__ void __launch_bounds__(128, P <= 2 && V == 1 ? 8 : 1) verify_wave_kernel(VerifyArgs a, uint64_t PW, uint32_t GW,
                                                          unsigned long long* __restrict__ next) {
  constexpr int R = 32 * V;   // rows of a block
    constexpr bool kTable = P == 2 && V >= kTableFrom;
  const int lane = threadIdx.x & 31;
  __shared__ __align__(16) uint32_t tables[kTable ? 4 * kEqTableWords<V> : 4];
  uint32_t* tab = tables + (kTable ? (threadIdx.x >> 5) * kEqTableWords<V> : 0);
  const int gl = lane & (G - 1);
  const int gbase = lane - gl;
  const uint32_t gmask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << gbase);
  const int prev_lane = gbase + ((gl + G - 1) & (G - 1));
  const uint64_t q_lo = a.range_lo ? *a.range_lo : 0;
  const uint64_t q_hi = a.range_hi ? *a.range_hi : a.m;
  // pair state (identical in the G lanes of a group)
  bool has = false, more = true;
  uint64_t t = 0;
  uint32_t k = 0;
  int64_t oA = 0, oB = 0;
  int32_t m = 0, n = 0, d0 = 0, dlo = 0, dhi = 0, bm = 0;
  int32_t sbase = 0;   // wavefront steps done on the pair
  // block state (this lane): block b runs at the steps where 0 <= u <= span
  // (u counts up by one per step); block b - 1 computed the same column one
  // step earlier while u <= u_valid; diagonal d0 crosses it where
  // 0 <= u + dg < R
  int32_t b = 0, u = kDeadU, span = 0, u_valid = -1, dg = 0x40000000;
  uint32_t T = 0;   // score << 1
  uint32_t Pv[V], Mv[V];
  uint32_t pa[P][V], bw[P];
  uint32_t pub = kIdle;
  bool done = false, reject = false;
  int32_t result = 0;
  uint64_t work = 0, nskip = 0;
#pragma unroll
  for (int w = 0; w < V; ++w) {
    Pv[w] = Mv[w] = 0u;
#pragma unroll
    for (int p = 0; p < P; ++p) pa[p][w] = 0u;
  }
  if constexpr (kTable) eq_store<V>(tab, lane, pa);   // lanes without a block compute on it
#pragma unroll
  for (int p = 0; p < P; ++p) bw[p] = 0u;

  // One column: the block step on the match bits, which a table gives one
  // column ahead (they wait for nothing; loaded when used they stand in the
  // chain from hand-over to hand-over).
  uint32_t Eq[V];
#pragma unroll
  for (int w = 0; w < V; ++w) Eq[w] = 0u;
  auto column = [&](uint32_t wv, uint32_t& Ph, uint32_t& hn) {
    if constexpr (!kTable) eq_planes<P, V>(pa, bw, Eq);
    wave_column<V>(Eq, wv, Pv, Mv, T, Ph, hn, pub);
    if constexpr (kTable) eq_load<V>(tab, lane, bw, Eq);
  };

  // Take block nb after step s.  Its columns are [jf, jl]; block nb computes
  // column j at step j + nb.  Blocks past row m never run.
  auto take_block = [&](int32_t nb, int32_t s) {
    b = nb;
    if (b <= bm) {
      const int32_t jf = max(1, R * b + 1 - dhi);
      const int32_t jl = min(n, R * b + R - dlo);
      u = s - (jf + b);
      span = jl - jf;
      u_valid = b == 0 ? -1 : min(n, R * b - dlo) - jf;   // last column of block b - 1
      dg = jf - R * b - 1 + d0;   // row j + d0 is row R b + 1 + (u + dg)
    } else {
      u = kDeadU;
      span = 0;
      u_valid = -1;
      dg = 0x40000000;
    }
  };

  while (true) {
    // ---- groups without a pair take pairs until they hold one that needs
    // the wavefront (one vote while all groups are busy)
    while (true) {
      const bool need = !has && more;
      const uint32_t leaders = __ballot_sync(0xffffffffu, need && gl == 0);
      if (!leaders) break;
      const int first = __ffs(leaders) - 1;
      unsigned long long base = 0;
      if (lane == first) base = atomicAdd(next, (unsigned long long)__popc(leaders));
      base = __shfl_sync(0xffffffffu, base, first);
      const uint64_t q = q_lo + base + __popc(leaders & ((1u << gbase) - 1u));
      if (need) {
        if (q >= q_hi) {
          more = false;
        } else {
          t = a.order ? a.order[q] : q;
          int64_t gm = 0, gn = 0;
          k = a.pk ? a.pk[t] : a.K;
          uint32_t res = 0xffffffffu;
          const uint32_t* fed = a.first_ed ? a.first_ed : a.ed;
          const bool skip = a.skip_kband && a.skip_kband[t] < a.K && fed[t] <= a.skip_kband[t];
          if (skip) {
            if (a.first_ed && gl == 0) put_result(a, t, fed[t]);
            res = 0xfffffffeu;   // settled by the first pass: nothing to do
          } else if (!pair_geometry(a, q, t, oA, oB, gm, gn)) {
            if (gl == 0) atomicOr(a.dev_flags, FLAG_BOUNDS);
            res = k + 1;
          } else {
            const int64_t mm = gm, nn = gn;
            if (mm >= (int64_t)kMaxLen) {
              if (gl == 0) atomicOr(a.dev_flags, FLAG_LENGTH);
              res = k + 1;
            } else if (mm - nn > (int64_t)k) {
              res = k + 1;
            } else if (nn == 0) {
              res = (uint32_t)mm;
            } else {
              m = (int32_t)mm;
              n = (int32_t)nn;
              d0 = m - n;
              dlo = -(int32_t)((k - (uint32_t)d0) >> 1);
              dhi = d0 + (int32_t)((k - (uint32_t)d0) >> 1);
              if (dhi - dlo < 63) dlo = dhi - 63;   // at least 64 band rows (any wider band is exact)
              bm = (m - 1) / R;
              sbase = 0;
              take_block(gl, 0);
              pub = kIdle;
              done = reject = false;
            }
          }
          if (res == 0xfffffffeu) {
            if (gl == 0) ++nskip;
          } else if (res != 0xffffffffu) {
            if (gl == 0) put_result(a, t, res);
          } else {
            has = true;
          }
        }
      }
    }
    if (!__any_sync(0xffffffffu, has || more)) break;

    // ---- kWaveSteps wavefront steps.  Every lane runs the column step; a lane
    // outside its block's steps computes on stale state (rebuilt at the
    // block's first column) that no other lane reads.  First and last
    // columns and the diagonal test take one rarely divergent branch.
    // Steps in which no lane of the warp meets such an event (a block's first
    // or last column, its input word switching from the predecessor's to the
    // band edge's, the window's last step) run in a loop without the tests:
    // their number is the warp's minimum of the steps to each lane's next
    // event.
    int it = 0;
    while (it < kWaveSteps) {
      {
        const int64_t un = (int64_t)u + 1;   // u at the next step
        int64_t fr = kWaveSteps - 1 - it;
        if (un <= 0) fr = min(fr, -un);
        if (un <= span) fr = min(fr, (int64_t)span - un);
        if (un <= u_valid) fr = min(fr, (int64_t)u_valid - un + 1);
        const int free = __reduce_min_sync(0xffffffffu, (int)fr);
        const bool from_prev = un <= u_valid;
        const uint32_t keep_in = from_prev ? 1u : 0u, idle_in = from_prev ? 0u : kIdle;
#pragma unroll(V == 1 ? 4 : 2)
        for (int f = 0; f < free; ++f) {
          const uint32_t w_in = __shfl_sync(0xffffffffu, pub, prev_lane);
          const uint32_t wv = mad_lo(w_in, keep_in, idle_in);   // w_in, or kIdle at the band's edge
          uint32_t Ph, hn;
          column(wv, Ph, hn);
        }
        u += free;
        it += free;
      }
      const uint32_t w_in = __shfl_sync(0xffffffffu, pub, prev_lane);
      ++u;
      const uint32_t wv = u <= u_valid ? w_in : kIdle;
      uint32_t Ph, hn;
      column(wv, Ph, hn);
      const bool diag_here = it == kWaveSteps - 1 && (uint32_t)(u + dg) < (uint32_t)R;
      if (u == 0 || u == span || diag_here) {
        if (u == 0) {   // first column: load the block's symbols, rows start from +1 deltas
          const int32_t jf = sbase + it + 1 - b;
          wave_load_rows<P, V>(a, (uint64_t)(oA + R * (int64_t)b + 32 * (int64_t)GW), pa);
          if constexpr (kTable) eq_store<V>(tab, lane, pa);
          wave_load_bits<P>(a, PW, (uint64_t)(oB + jf - 1 + 32 * (int64_t)GW), bw, true);
          if constexpr (kTable) eq_load<V>(tab, lane, bw, Eq);
#pragma unroll
          for (int w = 0; w < V; ++w) {
            Pv[w] = 0xffffffffu;
            Mv[w] = 0u;
          }
          column(wv, Ph, hn);
          // D of the row above the block in this column, plus the block's deltas
          const int32_t above = b == 0 ? 1 : (int32_t)((w_in >> 1) & 0x3fffffffu);
          const int32_t score = above + deltas_below<V>(Pv, Mv, -1);
          T = (uint32_t)score << 1;
          pub = ((Ph & 0x80000000u) | T) + hn;
        }
        // D at row r of this block = score minus the deltas of the rows below r
        if (diag_here && (uint32_t)u <= (uint32_t)span) {   // row j + d0 of diagonal d0
          const int32_t diag = (int32_t)(T >> 1) - deltas_below<V>(Pv, Mv, u + dg);
          if (diag > (int32_t)k) reject = true;
        }
        if (u == span) {   // the block leaves the band
          if (b == bm) {
            result = (int32_t)(T >> 1) - deltas_below<V>(Pv, Mv, (m - 1) % R);
            done = true;
          }
          work += (uint64_t)(span + 1) * V;
          take_block(b + G, sbase + it + 1);
        }
      }
      ++it;
    }
    sbase += kWaveSteps;
    if ((sbase & 31) == 0 && u >= 0 && u <= span) {   // B's symbols of the next 32 columns, all lanes at once
      wave_load_bits<P>(a, PW, (uint64_t)(oB + (sbase - b) + 32 * (int64_t)GW), bw, true);
      if constexpr (kTable) eq_load<V>(tab, lane, bw, Eq);
    }
    // ---- a group whose pair finished (or was rejected) writes it and frees
    // its lanes; one vote in the common case where none did
    const bool overrun = has && sbase >= n + bm;   // cannot happen: the last block ends at step n + bm
    if (__ballot_sync(0xffffffffu, done || reject || overrun)) {
      const uint32_t dmask = __ballot_sync(0xffffffffu, done) & gmask;
      const uint32_t rmask = __ballot_sync(0xffffffffu, reject) & gmask;
      const int src = dmask ? __ffs(dmask) - 1 : lane;
      const int32_t fin = __shfl_sync(0xffffffffu, result, src);
      bool end = false;
      if (has && (dmask || rmask)) {
        if (gl == 0) put_result(a, t, rmask ? k + 1 : (fin > (int32_t)k ? k + 1 : (uint32_t)fin));
        end = true;
      } else if (overrun) {
        if (gl == 0) {
          atomicOr(a.dev_flags, FLAG_BOUNDS);
          put_result(a, t, k + 1);
        }
        end = true;
      }
      if (end) {
        if (u >= 0 && u <= span) work += (uint64_t)(u + 1) * V;   // block cut short by the exit
        has = false;
        u = kDeadU;
        span = 0;
        u_valid = -1;
        dg = 0x40000000;
        pub = kIdle;
        done = reject = false;
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

// ---------------------------------------------------------------- bands wider than one warp
// One CTA of V warps (G = 32 V lanes) per pair, for bands whose wavefront
// no shape of one warp holds (K > 7968), or with 64 lanes or more asked for.
// Blocks, lanes and the column step are those of verify_wave_kernel with one
// word per lane (lane g owns blocks b = g mod G), with one change to the
// schedule: block b computes column j at step
//     j + b + 32 floor(b / 32),
// i.e. every group of 32 blocks runs one window of kWaveSteps (= 32) steps
// behind the group above it.  Inside a group the predecessor block b - 1 is
// the next lane down in the same warp and hands its word over by a shuffle,
// one step earlier as before.  The first block of a group (lane 0 of its
// warp) takes its predecessor's word from the last lane of the previous warp,
// written 33 steps earlier into a ring in shared memory: the CTA synchronises
// once per window (__syncthreads), after which the previous window's words
// are visible.  The extra skew also spaces a lane's consecutive blocks b and
// b + G by 2G steps instead of G, so G lanes hold any band with
//     34 G >= 32 + (dhi - dlo),  dhi - dlo <= K.
// Pair fetch, the early exit and the result are CTA-wide decisions taken at
// the window barrier; every loop bound is uniform over the CTA.
constexpr int kRing = 128;   // words per warp in the ring: steps s - 128 .. s - 1 (reads reach s - 33)

template <int V, int P>
__global__ void __launch_bounds__(32 * V) verify_cta_kernel(VerifyArgs a, uint64_t PW, uint32_t GW,
                                                            unsigned long long* __restrict__ next) {
  constexpr int G = 32 * V;
  constexpr int S = kWaveSteps;
  static_assert(S == 32 && kRing >= 2 * S + 2 && (kRing & (kRing - 1)) == 0, "window and ring sizes");
  __shared__ uint32_t ring[V][kRing];
  __shared__ unsigned long long s_t;   // pair of the CTA (~0: none left)
  __shared__ longlong2 s_geo;          // its offsets of A and B
  __shared__ int2 s_len;               // and lengths m >= n
  __shared__ int s_flag[3];            // per window (mod 3): 1 = finished, 2 = rejected
  __shared__ int32_t s_result[3];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int prev_warp = (warp + V - 1) % V;
  const uint64_t q_lo = a.range_lo ? *a.range_lo : 0;
  const uint64_t q_hi = a.range_hi ? *a.range_hi : a.m;
  if (tid < 3) s_flag[tid] = 0;
  uint32_t k = 0;
  int64_t oA = 0, oB = 0;
  int32_t m = 0, n = 0, d0 = 0, dlo = 0, dhi = 0, bm = 0;
  int32_t b = 0, u = kDeadU, span = 0, u_valid = -1, dg = 0x40000000, colbase = 0;
  uint32_t T = 0, Pv[1] = {0u}, Mv[1] = {0u};
  uint32_t pa[P][1], bw[P];
  uint32_t pub = kIdle;
  bool done = false, reject = false;
  int32_t result = 0;
  uint32_t win = 0;   // windows run by the CTA (selects the flag slot)
  uint64_t work = 0, nskip = 0;
#pragma unroll
  for (int p = 0; p < P; ++p) pa[p][0] = bw[p] = 0u;

  // Take block nb after s steps.  Its columns are [jf, jl]; it computes
  // column j at step j + colbase (colbase = nb + 32 floor(nb / 32)).
  auto take_block = [&](int32_t nb, int32_t s) {
    b = nb;
    if (b <= bm) {
      const int32_t jf = max(1, 32 * b + 1 - dhi);
      const int32_t jl = min(n, 32 * b + 32 - dlo);
      colbase = b + S * (b >> 5);
      u = s - (jf + colbase);
      span = jl - jf;
      u_valid = b == 0 ? -1 : min(n, 32 * b - dlo) - jf;   // last column of block b - 1
      dg = jf - 32 * b - 1 + d0;
    } else {
      u = kDeadU;
      span = 0;
      u_valid = -1;
      dg = 0x40000000;
      colbase = 0;
    }
  };

  while (true) {
    // ---- thread 0 takes pairs until one needs the wavefront
    if (tid == 0) {
      unsigned long long got = ~0ull;
      while (true) {
        const uint64_t q = q_lo + atomicAdd(next, 1ull);
        if (q >= q_hi) break;
        const uint64_t t = a.order ? a.order[q] : q;
        const uint32_t kt = a.pk ? a.pk[t] : a.K;
        const uint32_t* fed = a.first_ed ? a.first_ed : a.ed;
        if (a.skip_kband && a.skip_kband[t] < a.K && fed[t] <= a.skip_kband[t]) {
          if (a.first_ed) put_result(a, t, fed[t]);
          ++nskip;
          continue;
        }
        int64_t gA, gB, mm, nn;
        if (!pair_geometry(a, q, t, gA, gB, mm, nn)) {
          atomicOr(a.dev_flags, FLAG_BOUNDS);
          put_result(a, t, kt + 1);
          continue;
        }
        if (mm >= (int64_t)kMaxLen) {
          atomicOr(a.dev_flags, FLAG_LENGTH);
          put_result(a, t, kt + 1);
          continue;
        }
        if (mm - nn > (int64_t)kt) {
          put_result(a, t, kt + 1);
          continue;
        }
        if (nn == 0) {
          put_result(a, t, (uint32_t)mm);
          continue;
        }
        got = t;
        s_geo = make_longlong2(gA, gB);
        s_len = make_int2((int32_t)mm, (int32_t)nn);
        break;
      }
      s_t = got;
    }
    __syncthreads();
    const unsigned long long t = s_t;
    if (t == ~0ull) break;
    {
      k = a.pk ? a.pk[t] : a.K;
      const longlong2 geo = s_geo;
      const int2 len = s_len;
      oA = geo.x;
      oB = geo.y;
      m = len.x;
      n = len.y;
      d0 = m - n;
      dlo = -(int32_t)((k - (uint32_t)d0) >> 1);
      dhi = d0 + (int32_t)((k - (uint32_t)d0) >> 1);
      if (dhi - dlo < 63) dlo = dhi - 63;
      bm = (m - 1) >> 5;
    }
    take_block(tid, 0);
    pub = kIdle;
    done = reject = false;
    const int32_t last_step = n + bm + S * (bm >> 5);   // block bm's last column
    int32_t sbase = 0;
    while (true) {
#pragma unroll 8
      for (int it = 0; it < S; ++it) {
        const int32_t s1 = sbase + it + 1;   // this step, counted from 1
        uint32_t w_in = __shfl_up_sync(0xffffffffu, pub, 1);
        if (lane == 0) w_in = ring[prev_warp][(uint32_t)(s1 - 1 - S) & (kRing - 1)];
        ++u;
        const uint32_t wv = u <= u_valid ? w_in : kIdle;
        uint32_t Ph, hn;
        uint32_t Eq[1];
        eq_planes<P, 1>(pa, bw, Eq);
        wave_column<1>(Eq, wv, Pv, Mv, T, Ph, hn, pub);
        const bool diag_here = it == S - 1 && (uint32_t)(u + dg) < 32u;
        if (u == 0 || u == span || diag_here) {
          if (u == 0) {   // first column: load the block's symbols, rows start from +1 deltas
            const int32_t jf = s1 - colbase;
            wave_load_rows<P, 1>(a, (uint64_t)(oA + 32 * (int64_t)b + 32 * (int64_t)GW), pa);
            wave_load_bits<P>(a, PW, (uint64_t)(oB + jf - 1 + 32 * (int64_t)GW), bw, true);
            Pv[0] = 0xffffffffu;
            Mv[0] = 0u;
            eq_planes<P, 1>(pa, bw, Eq);
            wave_column<1>(Eq, wv, Pv, Mv, T, Ph, hn, pub);
            const int32_t above = b == 0 ? 1 : (int32_t)((w_in >> 1) & 0x3fffffffu);
            const int32_t score = above + deltas_below<1>(Pv, Mv, -1);
            T = (uint32_t)score << 1;
            pub = ((Ph & 0x80000000u) | T) + hn;
          }
          if (diag_here && (uint32_t)u <= (uint32_t)span) {   // row j + d0 of diagonal d0
            const int32_t diag = (int32_t)(T >> 1) - deltas_below<1>(Pv, Mv, u + dg);
            if (diag > (int32_t)k) reject = true;
          }
          if (u == span) {   // the block leaves the band
            if (b == bm) {
              result = (int32_t)(T >> 1) - deltas_below<1>(Pv, Mv, (m - 1) & 31);
              done = true;
            }
            work += (uint64_t)(span + 1);
            take_block(b + G, s1);
          }
        }
        if (lane == 31) ring[warp][(uint32_t)s1 & (kRing - 1)] = pub;
      }
      sbase += S;
      if (u >= 0 && u <= span)   // B's symbols of the next 32 columns
        wave_load_bits<P>(a, PW, (uint64_t)(oB + (sbase - colbase) + 32 * (int64_t)GW), bw, true);
      const uint32_t slot = win % 3;
      if (done) {
        s_result[slot] = result;
        atomicOr(&s_flag[slot], 1);
      }
      if (reject) atomicOr(&s_flag[slot], 2);
      __syncthreads();
      const int f = s_flag[slot];
      const int32_t fin = s_result[slot];
      if (tid == 0) s_flag[(win + 2) % 3] = 0;
      ++win;
      const bool overrun = sbase >= last_step;   // finished at the latest in the window of step last_step
      if (f || overrun) {
        if (tid == 0) {
          if (f & 1) {
            put_result(a, t, fin > (int32_t)k ? k + 1 : (uint32_t)fin);
          } else if (f & 2) {
            put_result(a, t, k + 1);
          } else {
            atomicOr(a.dev_flags, FLAG_BOUNDS);
            put_result(a, t, k + 1);
          }
        }
        if (u >= 0 && u <= span) work += (uint64_t)(u + 1);   // block cut short by the exit
        break;
      }
    }
  }
  if (a.work) {
    for (int o = 16; o > 0; o >>= 1) work += __shfl_down_sync(0xffffffffu, work, o);
    if (lane == 0 && work) atomicAdd(a.work, (unsigned long long)work);
  }
  if (tid == 0 && a.skipped && nskip) atomicAdd(a.skipped, (unsigned long long)nskip);
}

// Warps per scheduler that a list is worth, from the warps it fills in all.
// More warps hide more latency, but a pair taken early then runs more slowly
// and cannot move, so the kernel ends with the slowest share: with throughput
// T (1 + a / c) and c L for the longest pairs, c = sqrt(a T / L).  Measured with
// 1 / 2 / 3 / all resident blocks of four warps per SM (pairs of 2,000-20,000
// symbols): K = 3900, 3,000 pairs 3.18 / 2.66 / 3.36 / 4.37 ms, 20,000 pairs
// 19.8 / 15.7 / 15.0 / 15.0; K = 700 (8 lanes), 8,000 pairs 1.65 / 2.42 / 3.42 /
// 3.35, 100,000 pairs 14.0 / 10.5 / 9.9 / 10.3.
inline int wave_blocks_per_sm(uint64_t pairs, int G, int sms) {
  const double x = (double)pairs * G / 32 / (4.0 * sms);
  return std::max(1, (int)std::lround(std::sqrt(x / 2)));
}

template <int G, int P, int V>
int launch_gpv(const VerifyArgs& a, uint64_t PW, uint32_t GW, unsigned long long* next, cudaStream_t s) {
  int dev = 0, sms = kNumSMsHint, per_sm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, verify_wave_kernel<G, P, V>, 128, 0);
  per_sm = std::max(1, std::min(per_sm, wave_blocks_per_sm(a.m, G, sms)));
  uint64_t need = (a.m * G + 127) / 128;
  uint64_t grid = (uint64_t)sms * per_sm;
  if (need < grid) grid = need;
  verify_wave_kernel<G, P, V><<<(unsigned)(grid ? grid : 1), 128, 0, s>>>(a, PW, GW, next);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

template <int G>
int launch_g(const VerifyArgs& a, uint64_t PW, uint32_t GW, unsigned long long* next, cudaStream_t s) {
  if (a.bits <= 2) return launch_gpv<G, 2, 1>(a, PW, GW, next, s);
  if (a.bits <= 5) return launch_gpv<G, 5, 1>(a, PW, GW, next, s);
  return launch_gpv<G, 8, 1>(a, PW, GW, next, s);
}

template <int G, int V>
int launch_gv(const VerifyArgs& a, uint64_t PW, uint32_t GW, unsigned long long* next, cudaStream_t s) {
  return a.bits <= 2 ? launch_gpv<G, 2, V>(a, PW, GW, next, s) : launch_gpv<G, 8, V>(a, PW, GW, next, s);
}

// Shapes: G lanes of V words.  A block of R = 32 V rows is active for
// width + R - 1 columns and its successor starts R + 1 steps later, so
// floor((width + R - 2) / (R + 1)) + 1 <= G blocks must fit.
struct WaveShape {
  int G, V;
  int (*launch)(const VerifyArgs&, uint64_t, uint32_t, unsigned long long*, cudaStream_t);
};
const WaveShape kWaveShapes[] = {
    {2, 1, launch_g<2>}, {4, 1, launch_g<4>}, {8, 1, launch_g<8>}, {16, 1, launch_g<16>},
    {32, 1, launch_g<32>}, {4, 4, launch_gv<4, 4>}, {4, 6, launch_gv<4, 6>}, {8, 2, launch_gv<8, 2>},
    {8, 3, launch_gv<8, 3>}, {8, 4, launch_gv<8, 4>}, {8, 5, launch_gv<8, 5>}, {16, 2, launch_gv<16, 2>},
    {16, 3, launch_gv<16, 3>}, {16, 5, launch_gv<16, 5>}, {32, 2, launch_gv<32, 2>}, {32, 3, launch_gv<32, 3>},
    {32, 4, launch_gv<32, 4>}, {32, 6, launch_gv<32, 6>}, {32, 8, launch_gv<32, 8>},
};

bool shape_holds(const WaveShape& w, uint32_t kmax) {
  const int R = 32 * w.V, width = std::max<int>((int)kmax + 1, 64);
  return (width + R - 2) / (R + 1) + 1 <= w.G;
}

template <int V, int P>
int launch_vp(const VerifyArgs& a, uint64_t PW, uint32_t GW, unsigned long long* next, cudaStream_t s) {
  int dev = 0, sms = kNumSMsHint, per_sm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, verify_cta_kernel<V, P>, 32 * V, 0);
  if (per_sm < 1) per_sm = 1;
  // pairs take about equally long: no more CTAs than give every one the same
  // number of pairs (fewer CTAs per SM run faster, a part-filled last round
  // does not)
  uint64_t grid = (uint64_t)sms * per_sm;
  const uint64_t rounds = (a.m + grid - 1) / grid;
  grid = (a.m + rounds - 1) / rounds;
  verify_cta_kernel<V, P><<<(unsigned)(grid ? grid : 1), 32 * V, 0, s>>>(a, PW, GW, next);
  MJ_KERNEL_DONE();
  return MJ_OK;
}

template <int V>
int launch_v(const VerifyArgs& a, uint64_t PW, uint32_t GW, unsigned long long* next, cudaStream_t s) {
  if (a.bits <= 2) return launch_vp<V, 2>(a, PW, GW, next, s);
  if (a.bits <= 5) return launch_vp<V, 5>(a, PW, GW, next, s);
  return launch_vp<V, 8>(a, PW, GW, next, s);
}

}  // namespace

// The shape with the least estimated time.  Per step, a warp takes about
// 24 + 20 V issue cycles, a step alone 100 + 12 V cycles (K = 950, 50,000
// pairs: 32 lanes of 1 / 2 / 4 / 8 words 10.8 / 13.9 / 22.3 / 39.9 ms; 100 pairs:
// 1.20 ms with one word, 1.42 with four, 2.08 with eight); pairs reject early,
// so the average one takes about 0.3 of the longest one's steps.  Work W
// per scheduler and a longest pair L then overlap to (sqrt W + sqrt L)^2 (see
// wave_blocks_per_sm).  Against one word per lane (for K >= 1025: a CTA per
// pair) and all resident blocks: K = 1000, the band of 2,000 x 10 long noisy
// reads' join: 46.8 -> 31.2 ms; K = 4000, 3,000 pairs: 5.6 -> 2.7 ms; K = 1900
// and 12,000 pairs: 8.4 -> 5.4 ms.
// Codes of more than two planes compare eight, zero or not, with several words
// per lane, and five or eight with one.  10 pairs of 8,000 to 20,000 symbols of
// protein, alone: 1 word (K = 1000) 1.40 ms, 2 (1500) 1.44, 3 (2500) 1.64, 4 (4000)
// 1.81, 6 (5000) 2.42, 8 (7900) 2.93; a CTA per pair 1.55 (1500), 1.56 (2500), 1.60
// (4000), 1.93 (5000), 1.92 (7900).  Two planes, 20,000 to 60,000 bases: 4 words
// (4000) 3.52, 6 (5000) 4.38, 8 (7900) 5.26; a CTA 4.04, 4.55, 4.55.
int launch_verify_wave_auto(const VerifyArgs& a, uint64_t PW, uint32_t GW, uint32_t kmax, unsigned long long* next,
                            cudaStream_t s) {
  int dev = 0, sms = kNumSMsHint;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const WaveShape* best = nullptr;
  double least = 0;
  for (const WaveShape& w : kWaveShapes) {
    // the last block reads up to V words beyond the string: the guard holds them
    if (!shape_holds(w, kmax) || (int)GW <= w.V) continue;
    const double work = 0.3 * (24 + 20 * w.V) * ((double)a.m * w.G / 32 / (4.0 * sms)), longest = 100 + 12 * w.V;
    const double t = std::sqrt(work) + std::sqrt(longest);
    if (!best || t < least) {
      best = &w;
      least = t;
    }
  }
  // At most a pair per SM: every pair runs alone either way, and a CTA's warps
  // take less than the steps of many words (see above).
  if (best && a.m <= (uint64_t)sms && best->V > (a.bits <= 2 ? 6 : 2)) best = nullptr;
  return best ? best->launch(a, PW, GW, next, s) : launch_verify_wave(a, PW, GW, cta_lanes_for(kmax), next, s);
}

uint64_t wave_in_flight(uint32_t kmax, int sms) {
  for (const WaveShape& w : kWaveShapes)
    if (shape_holds(w, kmax)) return 4ull * sms;
  return (uint64_t)sms;
}

int launch_verify_wave(const VerifyArgs& a, uint64_t PW, uint32_t GW, int lanes, unsigned long long* next,
                       cudaStream_t s) {
  switch (lanes) {
    case 2: return launch_g<2>(a, PW, GW, next, s);
    case 4: return launch_g<4>(a, PW, GW, next, s);
    case 8: return launch_g<8>(a, PW, GW, next, s);
    case 16: return launch_g<16>(a, PW, GW, next, s);
    case 32: return launch_g<32>(a, PW, GW, next, s);
    case 64: return launch_v<2>(a, PW, GW, next, s);
    case 128: return launch_v<4>(a, PW, GW, next, s);
    case 256: return launch_v<8>(a, PW, GW, next, s);
    case 512: return launch_v<16>(a, PW, GW, next, s);
    case 1024: return launch_v<32>(a, PW, GW, next, s);
    default: return MJ_ERR_UNSUPPORTED;
  }
}

}  // namespace mj
