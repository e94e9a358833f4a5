// Step a8: verification of candidate pairs (Sec. 3: Ukkonen's banded dynamic
// program) as a bit-parallel computation over a diagonal band.
//
// For a pair, A is the longer string (rows i = 1..m) and B the shorter
// (columns j = 1..n), d0 = m - n <= k.  A path of cost <= k from (0,0) to
// (m,n) never leaves the diagonals d = i - j in
//     [dlo, dhi] = [-floor((k-d0)/2), d0 + floor((k-d0)/2)],
// because reaching diagonal d costs |d| and returning costs |d0 - d|.  The
// kernel holds, for every column j, the vertical deltas D[i][j] - D[i-1][j]
// of the rows i = j + dlo + t (t = 0 .. 32W-1, W 32-bit words, 32W >= width)
// as two bit-vectors (+1 and -1 bits), and advances a column with the
// bit-vector recurrence of Myers (1999) in Hyyro's formulation:
//     Xv = Eq | Mv;  Xh = (((Eq & Pv) + Pv) ^ Pv) | Eq
//     Ph = Mv | ~(Xh | Pv);  Mh = Pv & Xh
//     Ph = (Ph << 1) | hin;  Mh = Mh << 1
//     Pv = Mh | ~(Xv | Ph);  Mv = Ph & Xv
// Between columns the band slides down one row, so the vectors shift right by
// one bit.  Cells outside the band take over-estimates that keep every delta
// in {-1, 0, +1}: the row entering at the bottom gets a vertical delta of +1,
// the row above the top a horizontal delta of +1 (hin).  Rows above row 0 are
// virtual, with D[i][j] = j - i, which reproduces D[0][j] = j exactly.  The
// computed values are then >= the true ones everywhere and exact along any
// path that stays in the band, so D[m][n] is exact whenever ED <= k and > k
// otherwise.
//
// Early exit: along a diagonal, D[i+1][j+1] >= D[i][j], so D[m][n] >=
// D[j+d0][j] for every j; once that cell exceeds k the pair is rejected
// (checked every 32 columns).  The kernel tracks the value of the band's top
// row (bit 0) and recovers the cell on diagonal d0 (bit t0) by summing the
// deltas of bits 1..t0.
//
// Equality bits: rank codes of all bytes are stored as bit-planes over the
// concatenated input (plane p holds bit p of every code).  For column j the
// 32(W+1) plane bits starting at A's row j + dlo are ANDed against the rank of
// B[j-1] (XNOR per plane) and funnel-shifted into band position.  The words of
// all planes for the same 32 symbols lie side by side (plane_stride), so that a
// chunk's rows are a few wide loads.
#pragma once

#include "mj_verify_common.cuh"

namespace mj {
namespace {

// P, the planes a kernel is built for: 2, 5, 7 or 8 with digit tables, which
// need the input's rank codes, or kXnor8: eight planes compared by XNOR.
constexpr int kXnor8 = 9;
template <int P>
constexpr int kPlanes = P == kXnor8 ? 8 : P;

// Per-lane state of one pair in flight.
template <int W, int P>
struct PairState {
  uint32_t Pv[W], Mv[W], M1[W];
  uint64_t abit;           // plane bit index of the band's top row at column 1
  uint64_t bpos;           // plane bit index of B's symbol of column j
  int32_t j, n;            // next column, number of columns
  int32_t score;           // D at the band's top row
  uint32_t k;              // band of this pair
  uint64_t t;              // pair index
  int32_t width;           // split pairs: rows of the band below its top row
};

// Sets up pair t; returns false if the pair is decided without the DP
// (result written to *res).
template <int W, int P, bool SPLIT = false>
__device__ __forceinline__ bool pair_init(PairState<W, P>& st, const VerifyArgs& a, uint32_t GW, uint64_t q, uint64_t t,
                                          uint32_t* res, bool rev = false) {
  const uint32_t k = a.pk ? a.pk[t] : a.K;
  st.t = t;
  st.k = k;
  int64_t oA, oB, m, n;
  if (!pair_geometry(a, q, t, oA, oB, m, n)) {
    atomicOr(a.dev_flags, FLAG_BOUNDS);
    *res = k + 1;
    return false;
  }
  const int64_t d0 = m - n;
  if (d0 > (int64_t)k) {
    *res = k + 1;
    return false;
  }
  if (n == 0) {
    *res = (uint32_t)d0;
    return false;
  }
  if (m >= ((int64_t)1 << 30)) {         // column counters are 32-bit
    atomicOr(a.dev_flags, FLAG_LENGTH);
    *res = k + 1;
    return false;
  }
  const int32_t dlo = -(int32_t)(((int64_t)k - d0) >> 1);
  const int32_t t0 = (int32_t)d0 - dlo;  // bit of diagonal d0
  if (t0 >= 32 * W) {                    // cannot happen with a correct dispatch
    atomicOr(a.dev_flags, FLAG_BOUNDS);
    *res = k + 1;
    return false;
  }
  const int32_t nneg = 1 - dlo;          // band rows dlo..0 (virtual rows and row 0)
#pragma unroll
  for (int w = 0; w < W; ++w) {
    const int lo = 32 * w;
    const uint32_t neg = nneg >= lo + 32 ? 0xffffffffu : (nneg <= lo ? 0u : ((1u << (nneg - lo)) - 1u));
    st.Mv[w] = neg;
    st.Pv[w] = ~neg;
    int32_t a0 = 1 - lo, a1 = t0 + 1 - lo;  // bits 1..t0 within this word: [a0, a1)
    a0 = a0 < 0 ? 0 : a0;
    a1 = a1 > 32 ? 32 : a1;
    const uint32_t hiMask = a1 >= 32 ? 0xffffffffu : (a1 <= 0 ? 0u : ((1u << a1) - 1u));
    const uint32_t loMask = a0 >= 32 ? 0xffffffffu : ((1u << a0) - 1u);
    st.M1[w] = a1 > a0 ? (hiMask & ~loMask) : 0u;
  }
  // the state is kept one row down, ready for the next column: the band's
  // vectors (and the diagonal mask) shifted right by one bit, Pv's new bottom
  // row +1
#pragma unroll
  for (int w = 0; w < W - 1; ++w) {
    st.Pv[w] = __funnelshift_r(st.Pv[w], st.Pv[w + 1], 1);
    st.Mv[w] = __funnelshift_r(st.Mv[w], st.Mv[w + 1], 1);
    st.M1[w] = __funnelshift_r(st.M1[w], st.M1[w + 1], 1);
  }
  st.Pv[W - 1] = (st.Pv[W - 1] >> 1) | 0x80000000u;
  st.Mv[W - 1] >>= 1;
  st.M1[W - 1] >>= 1;
  st.score = -dlo;                       // D[dlo][0] = -dlo
  st.abit = (uint64_t)(oA + dlo + 32 * (int64_t)GW);   // plane bit of row 1 + dlo (column 1)
  st.bpos = (uint64_t)(oB + 32 * (int64_t)GW);
  st.j = 1;
  st.n = (int32_t)n;
  if (SPLIT) {
    // the first half of the columns forwards, the others from the ends of both
    // strings: column j of the reversed strings is B's symbol n - j, row i is
    // A's symbol m - i, and words are read so that their last bit or byte is
    // the first row or column
    const int32_t half = (int32_t)((n + 1) >> 1);
    st.width = (int32_t)d0 - 2 * dlo;   // dhi - dlo
    st.n = rev ? (int32_t)n - half : half;
    if (rev) {
      st.abit = (uint64_t)(oA + m - 1 - dlo - 31 + 32 * (int64_t)GW);
      st.bpos = (uint64_t)(oB + n - 32 + 32 * (int64_t)GW);
    }
  }
  return true;
}

// s = a + b over W 32-bit words (word 0 least significant): one carry chain
// (add.cc / addc) for bands up to 8 words, 64-bit partial sums beyond.
template <int W>
struct add_chain {
  static __device__ __forceinline__ void run(const uint32_t* a, const uint32_t* b, uint32_t* s) {
    uint32_t carry = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const uint64_t sum = (uint64_t)a[w] + b[w] + carry;
      carry = (uint32_t)(sum >> 32);
      s[w] = (uint32_t)sum;
    }
  }
};
template <>
struct add_chain<1> {
  static __device__ __forceinline__ void run(const uint32_t* a, const uint32_t* b, uint32_t* s) { s[0] = a[0] + b[0]; }
};
template <> struct add_chain<2> {
  static __device__ __forceinline__ void run(const uint32_t* a, const uint32_t* b, uint32_t* s) {
    asm("add.cc.u32 %0, %2, %4;\n\taddc.u32 %1, %3, %5;"
        : "=r"(s[0]), "=r"(s[1])
        : "r"(a[0]), "r"(a[1]), "r"(b[0]), "r"(b[1]));
  }
};
template <> struct add_chain<3> {
  static __device__ __forceinline__ void run(const uint32_t* a, const uint32_t* b, uint32_t* s) {
    asm("add.cc.u32 %0, %3, %6;\n\taddc.cc.u32 %1, %4, %7;\n\taddc.u32 %2, %5, %8;"
        : "=r"(s[0]), "=r"(s[1]), "=r"(s[2])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(b[0]), "r"(b[1]), "r"(b[2]));
  }
};
template <> struct add_chain<4> {
  static __device__ __forceinline__ void run(const uint32_t* a, const uint32_t* b, uint32_t* s) {
    asm("add.cc.u32 %0, %4, %8;\n\taddc.cc.u32 %1, %5, %9;\n\taddc.cc.u32 %2, %6, %10;\n\taddc.u32 %3, %7, %11;"
        : "=r"(s[0]), "=r"(s[1]), "=r"(s[2]), "=r"(s[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]));
  }
};
template <> struct add_chain<5> {
  static __device__ __forceinline__ void run(const uint32_t* a, const uint32_t* b, uint32_t* s) {
    asm("add.cc.u32 %0, %5, %10;\n\taddc.cc.u32 %1, %6, %11;\n\taddc.cc.u32 %2, %7, %12;\n\taddc.cc.u32 %3, %8, %13;\n\taddc.u32 %4, %9, %14;"
        : "=r"(s[0]), "=r"(s[1]), "=r"(s[2]), "=r"(s[3]), "=r"(s[4])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]));
  }
};
template <> struct add_chain<6> {
  static __device__ __forceinline__ void run(const uint32_t* a, const uint32_t* b, uint32_t* s) {
    asm("add.cc.u32 %0, %6, %12;\n\taddc.cc.u32 %1, %7, %13;\n\taddc.cc.u32 %2, %8, %14;\n\taddc.cc.u32 %3, %9, %15;\n\taddc.cc.u32 %4, %10, %16;\n\taddc.u32 %5, %11, %17;"
        : "=r"(s[0]), "=r"(s[1]), "=r"(s[2]), "=r"(s[3]), "=r"(s[4]), "=r"(s[5])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]));
  }
};
template <> struct add_chain<7> {
  static __device__ __forceinline__ void run(const uint32_t* a, const uint32_t* b, uint32_t* s) {
    asm("add.cc.u32 %0, %7, %14;\n\taddc.cc.u32 %1, %8, %15;\n\taddc.cc.u32 %2, %9, %16;\n\taddc.cc.u32 %3, %10, %17;\n\taddc.cc.u32 %4, %11, %18;\n\taddc.cc.u32 %5, %12, %19;\n\taddc.u32 %6, %13, %20;"
        : "=r"(s[0]), "=r"(s[1]), "=r"(s[2]), "=r"(s[3]), "=r"(s[4]), "=r"(s[5]), "=r"(s[6])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]));
  }
};
template <> struct add_chain<8> {
  static __device__ __forceinline__ void run(const uint32_t* a, const uint32_t* b, uint32_t* s) {
    asm("add.cc.u32 %0, %8, %16;\n\taddc.cc.u32 %1, %9, %17;\n\taddc.cc.u32 %2, %10, %18;\n\taddc.cc.u32 %3, %11, %19;\n\taddc.cc.u32 %4, %12, %20;\n\taddc.cc.u32 %5, %13, %21;\n\taddc.cc.u32 %6, %14, %22;\n\taddc.u32 %7, %15, %23;"
        : "=r"(s[0]), "=r"(s[1]), "=r"(s[2]), "=r"(s[3]), "=r"(s[4]), "=r"(s[5]), "=r"(s[6]), "=r"(s[7])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]), "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]));
  }
};

// Columns between two early-exit checks: 32 (the most one load of B's bits
// covers).  With the XNORs, bands of one or two words take 16, since their
// pairs are often short and exit early (measured before the digit tables: 32
// was 5% faster at 3-4 words and 8% slower at 2).  With digit tables every
// chunk rebuilds them, and 32 columns won at two words too (protein verify
// 24.9 -> 22.6 ms, with 25% more word-columns advanced).
template <int P>
constexpr bool kDigitTables = P != kXnor8;
template <int W, int P>
constexpr int kChunkFor = (W <= 2 && !kDigitTables<P>) ? 16 : 32;

// Advances up to kChunkFor<W, P> columns; returns true when the pair is decided.
// The chunk's symbols are loaded at its start for every lane at once: A's
// plane words of the rows the band covers in these columns (pre-shifted so
// that column j0 + c needs a shift by c < 32), and B's symbols of the
// columns: with digit tables its rank codes, one byte per column; with the
// XNORs (8 planes) its plane bits, bit-reversed so that the next column's
// bit is the sign bit.
// Equality bits by digit tables.  Per chunk, every
// thread writes to shared memory, for each of A's band words, the masks "rows
// whose rank code has digit value d" for each digit of the code: one digit of
// 2 bits for 2 planes (4 masks), 3 + 2 bits for 5 planes (8 + 4), 3 + 2 + 2
// bits for 7 planes (8 + 4 + 4), 3 + 3 + 2 bits for 8 planes (8 + 8 + 4); a
// column then takes its symbol's rank code
// from the input's code bytes and ANDs one mask of each digit's table (one load per word
// for 2 planes, one three-input logic op per word for 7), instead of an XNOR
// per plane and word.  Tables: word (d * (W + 1) + w) * 128 + thread, the
// digits' tables back to back.  (For 7 planes, two digits of 4 and 3 bits,
// 24 masks a word, take 50% more shared memory: 4 blocks per SM instead of
// 6.)  Bytes (8 planes), 150,000 pairs of 700 random bytes: an XNOR per plane and
// word over planes stored apart took 959 us at K = 60 and 1932 at K = 250, the
// tables 509 and 978.  kXnor8 keeps
// the XNORs where there are no rank codes (the allocation-free entry point)
// and for forced bands of more than 8 words, whose tables would not fit.
template <int P>
constexpr int digit_masks() { return P == 2 ? 4 : (P == 5 ? 12 : (P == 7 ? 16 : 20)); }
template <int W, int P>
constexpr size_t digit_smem_bytes() { return (size_t)digit_masks<P>() * (W + 1) * 128 * 4; }

// The masks of band word w (A's pre-shifted plane words pa) into the tables.
template <int W, int P>
__device__ __forceinline__ void build_digit_tables(const uint32_t (&pa)[kPlanes<P>][W + 1], int w, uint32_t* __restrict__ tab,
                                                   int tid) {
  auto put = [&](int d, uint32_t v) { tab[(d * (W + 1) + w) * 128 + tid] = v; };
  auto two = [&](int p, int base) {   // a 2-bit digit from planes p, p + 1
    const uint32_t x = pa[p][w], y = pa[p + 1][w];
    put(base + 0, ~x & ~y);
    put(base + 1, x & ~y);
    put(base + 2, ~x & y);
    put(base + 3, x & y);
  };
  if constexpr (P == 2) {
    two(0, 0);
  } else {
    auto three = [&](int p, int base) {   // a 3-bit digit from planes p .. p + 2
      const uint32_t a0 = pa[p][w], a1 = pa[p + 1][w], a2 = pa[p + 2][w];
      const uint32_t t2[4] = {~a0 & ~a1, a0 & ~a1, ~a0 & a1, a0 & a1};
#pragma unroll
      for (int d = 0; d < 8; ++d) put(base + d, t2[d & 3] & ((d & 4) ? a2 : ~a2));
    };
    three(0, 0);
    if constexpr (P == 8) {
      three(3, 8);
      two(6, 16);
    } else {
      two(3, 8);
      if constexpr (P == 7) two(5, 12);
    }
  }
}

// The equality bits of a symbol with rank code `code` over the band's words.
template <int W, int P>
__device__ __forceinline__ void digit_lookup(const uint32_t* __restrict__ tab, uint32_t code, int tid,
                                             uint32_t (&EqF)[W + 1]) {
  constexpr int S = (W + 1) * 128;
  if constexpr (P == 2) {
    const uint32_t* t = tab + code * S + tid;
#pragma unroll
    for (int w = 0; w <= W; ++w) EqF[w] = t[w * 128];
  } else if constexpr (P == 5) {
    const uint32_t* ta = tab + (code & 7u) * S + tid;
    const uint32_t* tb = tab + (8u + (code >> 3)) * S + tid;
#pragma unroll
    for (int w = 0; w <= W; ++w) EqF[w] = ta[w * 128] & tb[w * 128];
  } else {
    const uint32_t* ta = tab + (code & 7u) * S + tid;
    const uint32_t* tb = tab + (8u + ((code >> 3) & (P == 7 ? 3u : 7u))) * S + tid;
    const uint32_t* tc = tab + (P == 7 ? 12u + (code >> 5) : 16u + (code >> 6)) * S + tid;
#pragma unroll
    for (int w = 0; w <= W; ++w) EqF[w] = ta[w * 128] & tb[w * 128] & tc[w * 128];
  }
}

// SPLIT: the lane's half of a pair (rev: the reversed half); true when it is
// rejected, or (*res = kHalfDone) its columns are done.
constexpr uint32_t kHalfDone = 0xffffffffu;
template <int W, int P, bool SPLIT = false>
__device__ __forceinline__ bool pair_chunk(PairState<W, P>& st, const VerifyArgs& a, uint64_t PW, uint32_t* res,
                                           uint32_t* __restrict__ tab, uint32_t GW, bool rev = false) {
  constexpr bool kDigits = kDigitTables<P>;
  const int32_t j0 = st.j;
  constexpr int NP = kPlanes<P>;
  uint32_t pa[NP][W + 1];
  uint32_t bw[NP];
  uint32_t bsym[kDigits ? 8 : 1];   // B's rank codes of the chunk's columns, four per word
  {
    const uint64_t ab = SPLIT && rev ? st.abit - (uint64_t)(j0 - 1) : st.abit + (uint64_t)(j0 - 1);
    const uint64_t aw = (ab >> 5) + (SPLIT && rev ? 1 : 0);
    const int64_t step = SPLIT && rev ? -1 : 1;   // the reversed half's words descend
    const uint32_t ash = (uint32_t)(ab & 31);
    const uint64_t wb = st.bpos >> 5;
    const uint32_t sb = (uint32_t)(st.bpos & 31);
    uint32_t x0[NP];
    load_plane_words<NP>(a.planes, (int64_t)aw, x0);
#pragma unroll
    for (int w = 0; w <= W; ++w) {
      uint32_t x1[NP];
      load_plane_words<NP>(a.planes, (int64_t)aw + step * (w + 1), x1);
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        pa[p][w] = SPLIT && rev ? __brev(__funnelshift_r(x1[p], x0[p], ash)) : __funnelshift_r(x0[p], x1[p], ash);
        x0[p] = x1[p];
      }
    }
    if (!kDigits) {
      uint32_t y0[NP], y1[NP];
      load_plane_words<NP>(a.planes, (int64_t)wb, y0);
      load_plane_words<NP>(a.planes, (int64_t)wb + 1, y1);
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        bw[p] = __funnelshift_r(y0[p], y1[p], sb);
        if (!(SPLIT && rev)) bw[p] = __brev(bw[p]);
      }
    }
    if (kDigits) {
      const int tid = threadIdx.x;
#pragma unroll
      for (int w = 0; w <= W; ++w) build_digit_tables<W, P>(pa, w, tab, tid);
      // B's rank codes of columns j0 .. j0 + 31, aligned so that column j0 + c
      // is byte c (words beyond the input read as zero)
      const uint64_t bi = st.bpos - 32 * (uint64_t)GW;   // byte index of column j0's symbol
      const uintptr_t at0 = (uintptr_t)(a.codes + bi);
      const uint32_t sh = 8u * (uint32_t)(at0 & 3);
      const uintptr_t wa = at0 & ~(uintptr_t)15;
      const uintptr_t lo_end = (uintptr_t)a.codes, hi_end = (uintptr_t)(a.codes + a.nbytes);
      uint32_t raw[12];   // the three aligned 16-byte groups holding them
      if (wa >= lo_end && wa + 48 <= hi_end) {   // the common case: all inside the input
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const uint4 v = __ldg(reinterpret_cast<const uint4*>(wa) + k);
          raw[4 * k] = v.x;
          raw[4 * k + 1] = v.y;
          raw[4 * k + 2] = v.z;
          raw[4 * k + 3] = v.w;
        }
      } else {   // near an end of the input: byte by byte, zero outside it
#pragma unroll 1
        for (int k = 0; k < 12; ++k) {
          uint32_t x = 0;
          for (int b = 0; b < 4; ++b) {
            const uintptr_t q = wa + 4 * k + b;
            if (q >= lo_end && q < hi_end) x |= (uint32_t)__ldg(reinterpret_cast<const uint8_t*>(q)) << (8 * b);
          }
#pragma unroll
          for (int r = 0; r < 12; ++r)
            if (r == k) raw[r] = x;
        }
      }
      // the word of the first symbol to the front
      if (at0 & 8) {
#pragma unroll
        for (int k = 0; k < 10; ++k) raw[k] = raw[k + 2];
      }
      if (at0 & 4) {
#pragma unroll
        for (int k = 0; k < 9; ++k) raw[k] = raw[k + 1];
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) bsym[k] = __funnelshift_r(raw[k], raw[k + 1], sh);
      if (SPLIT && rev) {   // the last byte is the first column
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t x = __byte_perm(bsym[k], 0, 0x0123), y = __byte_perm(bsym[7 - k], 0, 0x0123);
          bsym[k] = y;
          bsym[7 - k] = x;
        }
      }
    }
  }
  constexpr int kChunk = kChunkFor<W, P>;
  const int32_t cnt = min(kChunk, st.n - j0 + 1);
  // The top row's D moves along a diagonal, so it rises by 0 or 1 per
  // column: by 1 exactly when the vertical delta entering the row and the
  // horizontal delta leaving it are +1 and 0 or 0 and +1 (the pairs summing
  // to 2 or -2 cannot occur).  Bit 0 of (Pv | Ph) & ~(Mv | Mh) per column,
  // shifted into `rises` (one bit per column, at most 32), and counted at the
  // end of the chunk.
  uint32_t rises = 0;
#pragma unroll 8   // part of the chunk: a smaller body is fetched better (measured)
  for (int c = 0; c < kChunk; ++c) {
    if (c >= cnt) break;
    // equality bits of column j0 + c: A's plane bits XNOR B's, over the planes
    uint32_t EqF[W + 1];
    if constexpr (kDigits) {
      const uint32_t code = (bsym[c >> 2] >> (8 * (c & 3))) & 255u;
      digit_lookup<W, P>(tab, code, threadIdx.x, EqF);
    } else {
#pragma unroll
      for (int w = 0; w <= W; ++w) EqF[w] = 0xffffffffu;
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        if (p < (int)a.bits) {
          const uint32_t xb = (uint32_t)__mulhi((int32_t)bw[p], 1);   // B's bit broadcast (sign)
          bw[p] *= 2u;
#pragma unroll
          for (int w = 0; w <= W; ++w) EqF[w] &= ~(pa[p][w] ^ xb);
        }
      }
    }
    uint32_t Eq[W];
#pragma unroll
    for (int w = 0; w < W; ++w) Eq[w] = __funnelshift_r(EqF[w], EqF[w + 1], (uint32_t)c);


    uint32_t Xv[W], Ph[W], Mh[W], EP[W], SUM[W];
#pragma unroll
    for (int w = 0; w < W; ++w) EP[w] = Eq[w] & st.Pv[w];
    add_chain<W>::run(EP, st.Pv, SUM);   // (Eq & Pv) + Pv across the band's words
#pragma unroll
    for (int w = 0; w < W; ++w) {
      Xv[w] = Eq[w] | st.Mv[w];
      const uint32_t Xh = (SUM[w] ^ st.Pv[w]) | Eq[w];
      Ph[w] = st.Mv[w] | ~(Xh | st.Pv[w]);
      Mh[w] = st.Pv[w] & Xh;
    }
    // the band has slid down one row already (the vectors are kept shifted):
    // bit 0 of Pv / Mv is the vertical delta entering the top row
    rises = __funnelshift_r(rises, (st.Pv[0] | Ph[0]) & ~(st.Mv[0] | Mh[0]), 1);
    // Myers' update Pv' = (Mh << 1) | ~(Xv | (Ph << 1) | 1), Mv' = ((Ph << 1) | 1)
    // & Xv, followed by the next column's slide (>> 1, Pv's new bottom row +1),
    // is Pv = Mh | ~((Xv >> 1) | Ph) | top, Mv = Ph & (Xv >> 1): one shift
    // instead of four per word.
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const uint32_t xs = w + 1 < W ? __funnelshift_r(Xv[w], Xv[w + 1], 1) : Xv[w] >> 1;
      st.Pv[w] = Mh[w] | ~(xs | Ph[w]);
      st.Mv[w] = Ph[w] & xs;
    }
    st.Pv[W - 1] |= 0x80000000u;
  }
  const int32_t jend = j0 + cnt - 1;
  st.j = jend + 1;
  st.bpos = SPLIT && rev ? st.bpos - (uint64_t)cnt : st.bpos + (uint64_t)cnt;
  st.score += __popc(rises);
  // D on diagonal d0 at column jend: a lower bound of D[m][n] (exact at n);
  // M1 (kept shifted like the vectors) selects the rows below the top row
  // down to diagonal d0
  int32_t diag = st.score;
#pragma unroll
  for (int w = 0; w < W; ++w) diag += (int32_t)__popc(st.Pv[w] & st.M1[w]) - (int32_t)__popc(st.Mv[w] & st.M1[w]);
  if (diag > (int32_t)st.k) {
    *res = st.k + 1;
    return true;
  }
  if (jend == st.n) {
    *res = SPLIT ? kHalfDone : (uint32_t)diag;
    return true;
  }
  return false;
}

}  // namespace
}  // namespace mj
