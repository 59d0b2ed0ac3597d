// fx.cuh -- block fixed-point FFT engine of the pass kernels.
//
// GB300 issues about 1.7 FP64 instructions per clock per SM but 64 lanes of
// 32-bit integer additions and of 32 x 32 + 64-bit multiply-adds, so a 64-bit
// integer addition (two instructions) costs a sixteenth of an FP64 one and a
// 64 x 64-bit high product (four multiply-adds) a tenth.  The transforms of
// the pass kernels therefore run on 64-bit integers with one power-of-two
// exponent per sequence: a value is v 2^e.  Additions are exact; a product
// with a twiddle rounds once, at the unit of the sequence's integers.
//
// Error.  A sequence enters a forward transform normalised so that its
// largest component has 62 - log2 G bits, G the largest growth of a component
// over the stages, or over the first stage only where that leaves two bits
// more: the second stage then starts with a measured shift.  A sequence enters
// an inverse transform, whose inputs are spectra with few large coefficients,
// normalised by the sum of its components' magnitudes, which bounds every
// partial sum (inv_shift).  Every rounding is at most one unit, against results whose root mean square is
// 2^54 units or more on the fields of the path (FP64's roundings are 2^-53 of
// the values themselves).
//
// Stages are those of fft.cuh (Stockham, mixed radix, in place, R points per
// butterfly in registers).  The inverse transform runs the plan's radices in
// reverse, so its last radix is the forward transform's first, and the row
// passes hand the data over in registers.  A twiddled stage of
// radix 4 or 8 scales by 1/4, one of radix 2 by 1/2: the twiddles are 62-bit
// integers, and no shift follows the product.
#pragma once
#include <cuda_runtime.h>

#include <cmath>
#include <vector>

#include "fft.cuh"

namespace da {

typedef long long i64;
typedef longlong2 q2;  // complex integer

__host__ __device__ __forceinline__ q2 mkq(i64 x, i64 y) {
  q2 r;
  r.x = x;
  r.y = y;
  return r;
}
__device__ __forceinline__ q2 qadd(q2 a, q2 b) { return mkq(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ q2 qsub(q2 a, q2 b) { return mkq(a.x - b.x, a.y - b.y); }

// (S i) a, S = +-1
template <int S>
__device__ __forceinline__ q2 qmul_si(q2 a) {
  return S > 0 ? mkq(-a.y, a.x) : mkq(a.y, -a.x);
}

// Sum and difference where ZX, ZY mark an operand known to be zero (its
// register holds nothing).
template <bool ZX, bool ZY>
__device__ __forceinline__ q2 qadd_z(q2 x, q2 y) {
  if constexpr (ZX && ZY) return mkq(0, 0);
  else if constexpr (ZY) return x;
  else if constexpr (ZX) return y;
  else return qadd(x, y);
}
template <bool ZX, bool ZY>
__device__ __forceinline__ q2 qsub_z(q2 x, q2 y) {
  if constexpr (ZX && ZY) return mkq(0, 0);
  else if constexpr (ZY) return x;
  else if constexpr (ZX) return mkq(-y.x, -y.y);
  else return qsub(x, y);
}

// d = hi 2^32 + lo with a signed low word (-2^31 <= lo < 2^31), so that both
// words enter signed multiply-adds.  Data are negated before they are split,
// never by words: a low word of -2^31 has no negative.  The words of a
// coefficient may be negated (fx_words leaves that one out).
__device__ __forceinline__ int lo_word(i64 d) { return (int)d; }
__device__ __forceinline__ int hi_word(i64 d) { return (int)(d >> 32) + (int)((unsigned)d >> 31); }

// a b + c as the one instruction it is: written in C++, the compiler reorders
// the sums of a product's parts and needs twice the instructions (a twiddle:
// 50 against 28).
__device__ __forceinline__ i64 madw(int a, int b, i64 c) {
  i64 r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}

constexpr i64 kHalfWord = 0x80000000LL;  // rounds the discarded low word of a middle sum

// a b / 2^64, the product of the low words left out (below one unit).
// |a|, |b| <= 2^62.
__device__ __forceinline__ i64 mul_hi(i64 a, i64 b) {
  const int ah = hi_word(a), al = lo_word(a), bh = hi_word(b), bl = lo_word(b);
  const i64 mid = madw(ah, bl, madw(al, bh, kHalfWord));
  return madw(ah, bh, (i64)(int)(mid >> 32));
}

// A 64-bit factor in words.
struct Words {
  int h, l;
  __device__ __forceinline__ explicit Words(i64 d) : h(hi_word(d)), l(lo_word(d)) {}
  __device__ __forceinline__ Words(int h_, int l_) : h(h_), l(l_) {}
};

// (a b + c d) / 2^64: |.| < 2^62 each, the sum of either pair's magnitudes
// below 2^62.5.
__device__ __forceinline__ i64 mul_hi2(Words a, Words b, Words c, Words d) {
  const i64 mid = madw(c.h, d.l, madw(c.l, d.h, madw(a.h, b.l, madw(a.l, b.h, kHalfWord))));
  return madw(c.h, d.h, madw(a.h, b.h, (i64)(int)(mid >> 32)));
}

// Twiddle: (cos, sin) as 62-bit integers, each split in signed words.
// a w / 4 for S = -1, a conj(w) / 4 for S = +1 (the tables hold S = -1).
template <int S>
__device__ __forceinline__ q2 qtwiddle(q2 a, int4 w) {
  const int xh = hi_word(a.x), xl = lo_word(a.x), yh = hi_word(a.y), yl = lo_word(a.y);
  const int sh = S < 0 ? w.z : -w.z, sl = S < 0 ? w.w : -w.w;  // imaginary part for this sign
  const int nh = S < 0 ? -w.z : w.z, nl = S < 0 ? -w.w : w.w;
  const i64 mr = madw(yh, nl, madw(yl, nh, madw(xh, w.y, madw(xl, w.x, kHalfWord))));
  const i64 mi = madw(yh, w.y, madw(yl, w.x, madw(xh, sl, madw(xl, sh, kHalfWord))));
  return mkq(madw(yh, nh, madw(xh, w.x, (i64)(int)(mr >> 32))), madw(yh, w.x, madw(xh, sh, (i64)(int)(mi >> 32))));
}

// x c for a constant c in (1/2, 1): x + x (c - 1), with c - 1 in 64 bits.
template <unsigned long long CM1>
__device__ __forceinline__ i64 mul_near_one(i64 x) {
  constexpr int cl = (int)(unsigned)CM1;
  constexpr int ch = (int)((i64)CM1 >> 32) + (int)((unsigned)CM1 >> 31);
  const int h = hi_word(x), l = lo_word(x);
  const i64 mid = madw(h, cl, madw(l, ch, kHalfWord));
  return madw(h, ch, x + (i64)(int)(mid >> 32));
}

// 2^64 (cos(pi/4) - 1), 2^64 (cos(pi/8) - 1), 2^64 sin(pi/8), rounded.
constexpr unsigned long long kFxR2m1 = 0xB504F333F9DE6484ULL;
constexpr unsigned long long kFxC8m1 = 0xEC835E79946A3145ULL;
constexpr unsigned long long kFxS8 = 0x61F78A9ABAA58B47ULL;

__device__ __forceinline__ q2 q_r2(q2 a) { return mkq(mul_near_one<kFxR2m1>(a.x), mul_near_one<kFxR2m1>(a.y)); }

// a (cos(pi/8) + S i sin(pi/8))
template <int S>
__device__ __forceinline__ q2 q_rot8(q2 a) {
  constexpr int cl = (int)(unsigned)kFxC8m1, ch = (int)((i64)kFxC8m1 >> 32) + (int)((unsigned)kFxC8m1 >> 31);
  constexpr int sl0 = (int)(unsigned)kFxS8, sh0 = (int)((i64)kFxS8 >> 32) + (int)((unsigned)kFxS8 >> 31);
  constexpr int sl = S > 0 ? sl0 : -sl0, sh = S > 0 ? sh0 : -sh0;
  const int xh = hi_word(a.x), xl = lo_word(a.x), yh = hi_word(a.y), yl = lo_word(a.y);
  const i64 mr = madw(yh, -sl, madw(yl, -sh, madw(xh, cl, madw(xl, ch, kHalfWord))));
  const i64 mi = madw(xh, sl, madw(xl, sh, madw(yh, cl, madw(yl, ch, kHalfWord))));
  return mkq(madw(yh, -sh, madw(xh, ch, a.x + (i64)(int)(mr >> 32))),
             madw(xh, sh, madw(yh, ch, a.y + (i64)(int)(mi >> 32))));
}

template <int S, int Z = 0>
__device__ __forceinline__ void qdft2(q2* a) {
  constexpr bool z0 = Z & 1, z1 = (Z >> 1) & 1;
  const q2 t = a[0];
  a[0] = qadd_z<z0, z1>(t, a[1]);
  a[1] = qsub_z<z0, z1>(t, a[1]);
}

// X_k = sum_m a_m exp(S 2 pi i m k / R), in place; bit m of Z: input m is
// zero (not loaded).
template <int S, int Z = 0>
__device__ __forceinline__ void qdft4(q2* a) {
  constexpr bool z0 = Z & 1, z1 = (Z >> 1) & 1, z2 = (Z >> 2) & 1, z3 = (Z >> 3) & 1;
  constexpr bool ze = z0 && z2, zo = z1 && z3;
  const q2 t0 = qadd_z<z0, z2>(a[0], a[2]), t1 = qsub_z<z0, z2>(a[0], a[2]);
  const q2 t2 = qadd_z<z1, z3>(a[1], a[3]), t3 = qsub_z<z1, z3>(a[1], a[3]);
  a[0] = qadd_z<ze, zo>(t0, t2);
  a[2] = qsub_z<ze, zo>(t0, t2);
  // t1 +- S i t3
  if constexpr (S > 0) {
    a[1] = mkq(t1.x - t3.y, t1.y + t3.x);
    a[3] = mkq(t1.x + t3.y, t1.y - t3.x);
  } else {
    a[1] = mkq(t1.x + t3.y, t1.y - t3.x);
    a[3] = mkq(t1.x - t3.y, t1.y + t3.x);
  }
}

template <int S, int Z = 0>
__device__ __forceinline__ void qdft8(q2* a) {
  q2 e[4] = {a[0], a[2], a[4], a[6]};
  q2 o[4] = {a[1], a[3], a[5], a[7]};
  qdft4<S, even_bits(Z, 8)>(e);
  qdft4<S, odd_bits(Z, 8)>(o);
  a[0] = qadd(e[0], o[0]);
  a[4] = qsub(e[0], o[0]);
  const q2 o2 = qmul_si<S>(o[2]);
  a[2] = qadd(e[2], o2);
  a[6] = qsub(e[2], o2);
  const q2 w1 = q_r2(mkq(S > 0 ? o[1].x - o[1].y : o[1].x + o[1].y, S > 0 ? o[1].y + o[1].x : o[1].y - o[1].x));
  a[1] = qadd(e[1], w1);
  a[5] = qsub(e[1], w1);
  const q2 w3 = q_r2(mkq(S > 0 ? o[3].x + o[3].y : o[3].x - o[3].y, S > 0 ? o[3].y - o[3].x : o[3].y + o[3].x));
  a[3] = qsub(e[3], w3);
  a[7] = qadd(e[3], w3);
}

template <int S, int Z = 0>
__device__ __forceinline__ void qdft16(q2* a) {
  q2 e[8], o[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    e[k] = a[2 * k];
    o[k] = a[2 * k + 1];
  }
  qdft8<S, even_bits(Z, 16)>(e);
  qdft8<S, odd_bits(Z, 16)>(o);
  // o_k exp(S i k pi / 8)
  o[1] = q_rot8<S>(o[1]);
  o[2] = q_r2(mkq(S > 0 ? o[2].x - o[2].y : o[2].x + o[2].y, S > 0 ? o[2].y + o[2].x : o[2].y - o[2].x));
  o[3] = qmul_si<S>(q_rot8<-S>(o[3]));  // 3 pi/8 = pi/2 - pi/8
  o[4] = qmul_si<S>(o[4]);
  o[5] = qmul_si<S>(q_rot8<S>(o[5]));  // 5 pi/8 = pi/2 + pi/8
  o[6] = qmul_si<S>(q_r2(mkq(S > 0 ? o[6].x - o[6].y : o[6].x + o[6].y, S > 0 ? o[6].y + o[6].x : o[6].y - o[6].x)));
  const q2 r7 = q_rot8<-S>(o[7]);  // 7 pi/8 = pi - pi/8
  o[7] = mkq(-r7.x, -r7.y);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    a[k] = qadd(e[k], o[k]);
    a[k + 8] = qsub(e[k], o[k]);
  }
}

template <int R, int S, int Z = 0>
__device__ __forceinline__ void qdftR(q2* a) {
  if constexpr (R == 2) qdft2<S, Z>(a);
  if constexpr (R == 4) qdft4<S, Z>(a);
  if constexpr (R == 8) qdft8<S, Z>(a);
  if constexpr (R == 16) qdft16<S, Z>(a);
}

// ---------------------------------------------------------------------------
// Plans, scaling and twiddle tables
// ---------------------------------------------------------------------------

template <typename P, typename Q> struct ReverseOnto;
template <typename Q> struct ReverseOnto<Radices<>, Q> { using type = Q; };
template <int R, int... Rs, int... Qs> struct ReverseOnto<Radices<R, Rs...>, Radices<Qs...>> {
  using type = typename ReverseOnto<Radices<Rs...>, Radices<R, Qs...>>::type;
};

// log2 of the scaling of one twiddled stage (1/4, radix 2: 1/2)
constexpr int stage_shift(int r) { return r == 2 ? 1 : 2; }

template <int L, typename P> struct FxSum;
template <int L> struct FxSum<L, Radices<>> { static constexpr int shift = 0, entries = 0; };
template <int L, int R, int... Rs> struct FxSum<L, Radices<R, Rs...>> {
  using Next = FxSum<L * R, Radices<Rs...>>;
  static constexpr int shift = (L > 1 ? stage_shift(R) : 0) + Next::shift;
  static constexpr int entries = (L > 1 ? (R - 1) * L : 0) + Next::entries;
};

constexpr int log2c(int n) { return n <= 1 ? 0 : 1 + log2c(n / 2); }

// A plan of N points on TPS threads a sequence; fwd: its radices.
template <int N_, int TPS_, typename Fwd>
struct FxPlanOf {
  static constexpr int N = N_, TPS = TPS_;
  using fwd = Fwd;
  using inv = typename ReverseOnto<fwd, Radices<>>::type;
  // both directions scale by 2^-SHIFT in all
  static constexpr int SHIFT = FxSum<1, fwd>::shift;
  static constexpr int SHIFT_INV = FxSum<1, inv>::shift;
  static constexpr int ENTRIES = FxSum<1, fwd>::entries, ENTRIES_INV = FxSum<1, inv>::entries;
  static constexpr int TABLE = ENTRIES + ENTRIES_INV;  // forward table, then inverse
  // Bits of the largest input component of a forward transform: a component
  // of a partial sum is at most sqrt2 times the largest input component times
  // the product of the radices so far, scaled; it stays below 2^63.
  template <int L, typename P> struct Growth;
  template <int L> struct Growth<L, Radices<>> { static constexpr int most(int) { return 0; } };
  template <int L, int R, int... Rs> struct Growth<L, Radices<R, Rs...>> {
    static constexpr int most(int g) {
      const int here = g + log2c(R) - (L > 1 ? stage_shift(R) : 0);
      const int next = Growth<L * R, Radices<Rs...>>::most(here);
      return here > next ? here : next;
    }
  };
  static constexpr int GROWTH = Growth<1, fwd>::most(0);
  static constexpr int R1 = FirstRadix<fwd>::value;
  static constexpr int GROWTH1 = log2c(R1);                                          // first stage
  static constexpr int GROWTH2 = Growth<R1, typename TailRadices<fwd>::type>::most(0);  // the others
  static constexpr int BITS_FWD = 62 - GROWTH;
  static constexpr int SEQ = N + N / 8;  // q2 of one buffer of a sequence
  static constexpr int WARPS = (TPS + 31) / 32;
};

template <int N, int V = 0>
using FxPlan = FxPlanOf<N, PlanInfo<N, V>::THREADS / 2, typename Plan<N, V>::two>;

// Signed words (hi, lo) of a coefficient; a low word of -2^31, which could
// not be negated, is moved by one unit (2^-62).
__host__ __device__ inline int2 fx_words(i64 v) {
  if ((unsigned)v == 0x80000000u) ++v;
  const int lo = (int)(unsigned)v;
  return make_int2((int)((v - lo) >> 32), lo);
}

template <int L>
inline void fx_fill(int4*, Radices<>) {}

// exp(-2 pi i m k / (L R)) for m = 1..R-1, k < L, entry (m - 1) L + k of each
// twiddled stage: round(2^62 cos), round(2^62 sin), each hi, lo signed words.
template <int L, int R, int... Rs>
inline void fx_fill(int4* out, Radices<R, Rs...>) {
  if (L > 1) {
    const long double pi = 3.141592653589793238462643383279502884L;
    const long double s = 4611686018427387904.0L;
    for (int m = 1; m < R; ++m)
      for (int k = 0; k < L; ++k) {
        const long double th = -2.0L * pi * (long double)(m * k) / (long double)(L * R);
        const i64 c = llroundl(s * cosl(th)), n = llroundl(s * sinl(th));
        const int2 cw = fx_words(c), nw = fx_words(n);
        out[(m - 1) * L + k] = make_int4(cw.x, cw.y, nw.x, nw.y);
      }
    out += (R - 1) * L;
  }
  fx_fill<L * R>(out, Radices<Rs...>{});
}

// The two tables of a plan, computed on first use (a long double cosine is
// software on some hosts: 6 ms for 1024 points).
template <typename P>
inline const std::vector<int4>& fx_table() {
  static const std::vector<int4> table = [] {
    std::vector<int4> t(P::TABLE);
    fx_fill<1>(t.data(), typename P::fwd{});
    fx_fill<1>(t.data() + P::ENTRIES, typename P::inv{});
    return t;
  }();
  return table;
}

// ---------------------------------------------------------------------------
// Exponents and conversions
// ---------------------------------------------------------------------------

// Exponent of a symbol that vanishes or of values that are not there, and of a
// sequence that holds an infinity or a NaN, whose integers are all zero (zeros
// that are data have the exponent of subnormals).  Ordinary exponents are a few
// thousand at most, so that a mark plus any of them stays beyond half the mark,
// and clamp_exp brings it back.  The sum of the two marks lies beyond half the
// bad one: zero times NaN is NaN.
constexpr int kZeroExp = -100000, kBadExp = 400000;
static_assert(kBadExp + kZeroExp - 10000 > kBadExp / 2, "a bad sequence stays bad in a product with a zero one");

__device__ __forceinline__ int clamp_exp(int e) { return e < kZeroExp / 2 ? kZeroExp : e > kBadExp / 2 ? kBadExp : e; }

// Magnitude of an integer's high word: |v| < 2^32 (mag32(v) + 1).
__device__ __forceinline__ int mag32(i64 v) { return abs((int)(v >> 32)); }
__device__ __forceinline__ int max_mag(int m, q2 v) { return max(m, max(mag32(v.x), mag32(v.y))); }
__device__ __forceinline__ int bits32(int m) { return 32 - __clz(m); }
// Bits of a value whose high word has magnitude at most m: |v| < 2^bits64(m).
__device__ __forceinline__ int bits64(int m) { return 32 + bits32(m + 1); }

// v / 2^r, rounded, r >= 0 (62 where r is larger).
struct ShiftRight {
  int r;
  i64 half;
  __device__ __forceinline__ explicit ShiftRight(int r_) : r(min(r_, 62)) { half = (1LL << r) >> 1; }
  __device__ __forceinline__ i64 operator()(i64 v) const { return (v + half) >> r; }
  __device__ __forceinline__ q2 operator()(q2 v) const { return mkq((*this)(v.x), (*this)(v.y)); }
};

// v 2^s: left for s >= 0 (the caller knows that it fits), right with
// rounding for s < 0.
struct Shift {
  int l;
  ShiftRight right;
  __device__ __forceinline__ explicit Shift(int s) : l(min(max(s, 0), 62)), right(max(-s, 0)) {}
  __device__ __forceinline__ i64 operator()(i64 v) const { return right(v << l); }
  __device__ __forceinline__ q2 operator()(q2 v) const { return mkq((*this)(v.x), (*this)(v.y)); }
};

// The threads of one sequence: TPS of them, whole warps or an aligned part of
// one.  Threads of several sequences share a warp where TPS < 32; they run in
// lockstep.  id: the sequence's index in the CTA, 0 or 1 where TPS > 32.  The
// barriers are named by constants: one named by a register reserves all 16 of
// a CTA's, and an SM has 64 (256^2 on 128 threads: 4 CTAs of the 10 that the
// registers allow).
template <int TPS>
__device__ __forceinline__ void seq_sync(int id) {
  if constexpr (TPS <= 32) __syncwarp();
  else if (id == 0) asm volatile("bar.sync 1, %0;" ::"n"(TPS) : "memory");
  else asm volatile("bar.sync 2, %0;" ::"n"(TPS) : "memory");
}

// Reductions over a sequence: put leaves each warp's part in scratch (TPS/32
// ints of the sequence's own; unused where one warp holds the sequence), and
// get, after the next seq_sync, returns the whole.
template <int TPS>
__device__ __forceinline__ unsigned seq_mask(int t) {
  if constexpr (TPS >= 32) return 0xffffffffu;
  else return ((1u << TPS) - 1) << ((threadIdx.x & 31) - t);
}
template <int TPS>
__device__ __forceinline__ int seq_max_put(int v, int t, int* scratch) {
  v = __reduce_max_sync(seq_mask<TPS>(t), v);
  if constexpr (TPS > 32) {
    if ((t & 31) == 0) scratch[t >> 5] = v;
  }
  return v;
}
template <int TPS>
__device__ __forceinline__ int seq_max_get(int v, const int* scratch) {
  if constexpr (TPS > 32) {
    v = scratch[0];
#pragma unroll
    for (int w = 1; w < TPS / 32; ++w) v = max(v, scratch[w]);
  }
  return v;
}
template <int TPS>
__device__ __forceinline__ int seq_sum_put(int v, int t, int* scratch) {
  v = (int)__reduce_add_sync(seq_mask<TPS>(t), (unsigned)v);
  if constexpr (TPS > 32) {
    if ((t & 31) == 0) scratch[t >> 5] = v;
  }
  return v;
}
template <int TPS>
__device__ __forceinline__ int seq_sum_get(int v, const int* scratch) {
  if constexpr (TPS > 32) {
    v = scratch[0];
#pragma unroll
    for (int w = 1; w < TPS / 32; ++w) v += scratch[w];
  }
  return v;
}

// Inputs of an inverse transform have at most BITS bits (columns 60, rows 61); as the first
// stage reads them, they are shifted (right with rounding, or left) until the
// sum of their magnitudes has 62 bits, or up to G more (below).  The sum is
// counted in units of 2^(32 + kSumDrop), one unit more for each group of up to
// four magnitudes, whose low part is dropped.
//
// The second stage scales by 2^-G before it adds, so the sum may have 62 + G
// bits where the first stage's own sums, at most R sqrt2 times the largest
// component, stay below 2^62.5: while the components have 62 - log2 R bits.
// Nor may it have more than 60 + SHIFT_INV bits: the results then have 60,
// and the row passes only ever shift them left (RowBits).
constexpr int kSumDrop = 12;
template <typename P, int BITS>
__device__ __forceinline__ int inv_shift(int sum) {
  using I = typename P::inv;
  constexpr int first = BITS - (62 - log2c(FirstRadix<I>::value));
  constexpr int G0 = stage_shift(FirstRadix<typename TailRadices<I>::type>::value);
  constexpr int G = G0 < P::SHIFT_INV - 2 ? G0 : P::SHIFT_INV - 2;
  const int r = bits32(sum) + 32 + kSumDrop - 62;
  return min(r, max(r - G, first));
}
__device__ __forceinline__ int mag_units(q2 a, q2 b) {
  const unsigned m = (unsigned)mag32(a.x) + (unsigned)mag32(a.y) + (unsigned)mag32(b.x) + (unsigned)mag32(b.y);
  return (int)(m >> kSumDrop) + 1;
}

// v 2^e as a double (one rounding).
__device__ __forceinline__ double pow2_double(int e) {  // 2^e, -1022 <= e <= 1023
  return __hiloint2double((e + 1023) << 20, 0);
}
// The scaling where 2^e is not an ordinary double: in steps, each within a
// double's range.  Out of line: states in the ordinary range never come here.
static __device__ __noinline__ double fx_scale_far(double d, int e) {
  if (e > kBadExp / 2) return __hiloint2double(0x7ff80000, 0);
  if (d == 0.0) return 0.0;
  int left = max(min(e, 2200), -2200);
  while (left != 0) {
    const int s = max(min(left, 900), -900);
    d *= pow2_double(s);
    left -= s;
  }
  return d;
}
__device__ __forceinline__ double fx_to_double(i64 v, int e) {
  const double d = (double)v;
  if (e < -960 || e > 960) return fx_scale_far(d, e);
  // times 2^e by the exponent field: an FP64 product would cost a warp 64 clocks
  return v == 0 ? 0.0 : __hiloint2double(__double2hiint(d) + (e << 20), __double2loint(d));
}

// Two real coefficients of a mode, a and b, as integers of one exponent: the
// larger of |a|, |b| has 62 bits (the smaller may lose what lies below a
// unit); words (a_hi, a_lo, b_hi, b_lo).
struct __align__(16) FxPair {
  int ah, al, bh, bl;
};

// a b / 2^64 of two factors in words.
__device__ __forceinline__ i64 mul_hi(Words a, Words b) {
  const i64 mid = madw(a.h, b.l, madw(a.l, b.h, kHalfWord));
  return madw(a.h, b.h, (i64)(int)(mid >> 32));
}
// (a p + SG b q) / 2^64, |p|, |q| < 2^61.5.
template <int SG>
__device__ __forceinline__ i64 fx_pair_sum(const FxPair& c, i64 p, i64 q) {
  return mul_hi2(Words(p), Words(c.ah, c.al), Words(q), SG > 0 ? Words(c.bh, c.bl) : Words(-c.bh, -c.bl));
}

// Biased exponent field of a double (0: zero or subnormal, whose unit is that
// of field 1; 2047: not finite).
__device__ __forceinline__ int exp_field(double d) { return (__double2hiint(d) >> 20) & 0x7ff; }

// Exponent e for a sequence whose largest exponent field is f, so that every
// component has at most BITS bits: |d| < 2^(f - 1022) = 2^(BITS + e).
template <int BITS>
__device__ __forceinline__ int exp_for(int f) {
  return f == 2047 ? kBadExp : max(f, 1) - 1022 - BITS;
}

// d / 2^e as an integer, rounded towards zero; e from exp_for<BITS> (BITS <=
// 62).
__device__ __forceinline__ i64 double_to_fx(double d, int e) {
  const int hi = __double2hiint(d), lo = __double2loint(d);
  const int f = (hi >> 20) & 0x7ff;
  // significand m of 53 bits (of a subnormal: fewer), value m 2^(max(f, 1) - 1075): m 2^9 >> r
  const i64 m = ((i64)((hi & 0xfffff) | (f ? 0x100000 : 0)) << 32) | (unsigned)lo;
  const int r = (int)min((unsigned)(9 - (max(f, 1) - 1075 - e)), 63u);
  const i64 q = (m << 9) >> r;
  return hi < 0 ? -q : q;
}

// The pair of coefficients a, b and its exponent; a pair of zeros gets zero_e.
__device__ __forceinline__ FxPair fx_pair(double a, double b, int zero_e, int* e) {
  const int f = max(exp_field(a), exp_field(b));
  *e = f == 0 ? zero_e : exp_for<62>(f);
  if (f == 0) return {0, 0, 0, 0};
  const int2 x = fx_words(double_to_fx(a, *e)), y = fx_words(double_to_fx(b, *e));
  return {x.x, x.y, y.x, y.y};
}

// ---------------------------------------------------------------------------
// Stages
// ---------------------------------------------------------------------------

// a / 2^s, rounded
__device__ __forceinline__ i64 shr_round(i64 v, int s) { return (v + (1LL << (s - 1))) >> s; }

// The butterfly of one stage: twiddles (L > 1), then the R-point DFT.
template <int R, int S, int L, int Z>
__device__ __forceinline__ void fx_butterfly(q2* a, const int4* __restrict__ T, int k) {
  if constexpr (L > 1) {
    a[0] = mkq(shr_round(a[0].x, stage_shift(R)), shr_round(a[0].y, stage_shift(R)));
#pragma unroll
    for (int m = 1; m < R; ++m) {
      a[m] = qtwiddle<S>(a[m], __ldg(T + (m - 1) * L + k));
      if constexpr (R == 2) a[m] = mkq(a[m].x * 2, a[m].y * 2);
    }
  }
  qdftR<R, S, Z>(a);
}

// Position of element i of a sequence in its buffer: one element of padding
// after every eight (128 bytes), so that the strided stores of a stage meet
// few bank conflicts.  Every i + m c used below adds pad(m c) exactly.
__host__ __device__ constexpr int pad(int i) { return i + i / 8; }

// Butterflies of a stage of radix R held by one thread: i = t + jb TPS, jb <
// J; where there are fewer butterflies than threads, threads t < N / R hold
// one each.
template <typename P, int R>
struct Bfly {
  static constexpr int NB = P::N / R;
  static constexpr int J = NB >= P::TPS ? NB / P::TPS : 1;
  static constexpr int POINTS = J * R;
  static_assert(NB < P::TPS || NB % P::TPS == 0, "whole butterflies per thread");
  __device__ static __forceinline__ bool active(int t) { return NB >= P::TPS || t < NB; }
};

// Inputs i + m NB of butterfly i, out of buf; Z: inputs left out.
template <typename P, int R, int Z = 0>
__device__ __forceinline__ void fx_load(q2* a, const q2* buf, int i) {
  const q2* s = buf + pad(i);
#pragma unroll
  for (int m = 0; m < R; ++m)
    if (!((Z >> m) & 1)) a[m] = s[pad(m * (P::N / R))];
}

// Outputs of butterfly i of the stage with sub-length L, into buf.
template <typename P, int R, int L>
__device__ __forceinline__ void fx_store(const q2* a, q2* buf, int i) {
  const int k = i & (L - 1);
  q2* d = buf + pad((i - k) * R + k);
#pragma unroll
  for (int m = 0; m < R; ++m) d[pad(m * L)] = a[m];
}

// Middle stages with sub-lengths from L on, in place: every thread holds its
// butterflies in registers across a barrier of the sequence (two buffers and one
// barrier a stage measured the same from 128 to 1024 points).  SHR: the
// first of them starts with a right shift by r.
template <typename P, int S, int L, bool SHR>
__device__ __forceinline__ void fx_middle(q2*, const int4*, int, int, int, Radices<>) {}
template <typename P, int S, int L, bool SHR, int R, int... Rs>
__device__ __forceinline__ void fx_middle(q2* buf, const int4* T, int t, int id, int r, Radices<R, Rs...>) {
  using B = Bfly<P, R>;
  q2 a[B::POINTS];
  if (B::active(t)) {
#pragma unroll
    for (int jb = 0; jb < B::J; ++jb) {
      const int i = t + jb * P::TPS;
      fx_load<P, R>(a + jb * R, buf, i);
      if constexpr (SHR) {
        if (r > 0) {
#pragma unroll
          for (int m = 0; m < R; ++m) a[jb * R + m] = mkq(shr_round(a[jb * R + m].x, r), shr_round(a[jb * R + m].y, r));
        }
      }
      fx_butterfly<R, S, L, 0>(a + jb * R, T, i & (L - 1));
    }
  }
  seq_sync<P::TPS>(id);
  if (B::active(t)) {
#pragma unroll
    for (int jb = 0; jb < B::J; ++jb) fx_store<P, R, L>(a + jb * R, buf, t + jb * P::TPS);
  }
  seq_sync<P::TPS>(id);
  fx_middle<P, S, L * R, false>(buf, T + (R - 1) * L, t, id, r, Radices<Rs...>{});
}

// Inverse transform (S = +1) of the sequence in buf, zero outside the band
// KB: the inputs are shifted right by pre (left by -pre) first, and the result is the transform times 2^-SHIFT_INV, of at most 60 bits.  It
// is left in registers: out[jb R + m] is position t + jb TPS + m N / R for R
// the last radix.  buf is not free before the next sync.
template <typename P, int KB>
__device__ __forceinline__ void fx_inverse(q2* buf, const int4* tw, int t, int id, int pre, q2* out) {
  using I = typename P::inv;
  constexpr int R1 = FirstRadix<I>::value, RL = LastRadix<I>::value;
  constexpr int Z = gap_common(P::N, R1, KB);  // inputs in the gap for every butterfly
  using B1 = Bfly<P, R1>;
  using BL = Bfly<P, RL>;
  const int4* T = tw + P::ENTRIES;
  q2 a[B1::POINTS];
  if (B1::active(t)) {
    const ShiftRight right(max(pre, 0));
#pragma unroll
    for (int jb = 0; jb < B1::J; ++jb) {
      q2* b = a + jb * R1;
      fx_load<P, R1, Z>(b, buf, t + jb * P::TPS);
      if (pre > 0) {
#pragma unroll
        for (int m = 0; m < R1; ++m)
          if (!((Z >> m) & 1)) b[m] = right(b[m]);
      } else if (pre < 0) {
#pragma unroll
        for (int m = 0; m < R1; ++m)
          if (!((Z >> m) & 1)) b[m] = mkq(b[m].x << -pre, b[m].y << -pre);
      }
      qdftR<R1, +1, Z>(b);
    }
  }
  seq_sync<P::TPS>(id);
  if (B1::active(t)) {
#pragma unroll
    for (int jb = 0; jb < B1::J; ++jb) fx_store<P, R1, 1>(a + jb * R1, buf, t + jb * P::TPS);
  }
  seq_sync<P::TPS>(id);
  using Mid = typename InitRadices<typename TailRadices<I>::type>::type;
  fx_middle<P, +1, R1, false>(buf, T, t, id, 0, Mid{});
  constexpr int L = P::N / RL;
  if (BL::active(t)) {
    const int4* Tl = T + P::ENTRIES_INV - (RL - 1) * L;
#pragma unroll
    for (int jb = 0; jb < BL::J; ++jb) {
      const int i = t + jb * P::TPS;
      fx_load<P, RL>(out + jb * RL, buf, i);
      fx_butterfly<RL, +1, L, 0>(out + jb * RL, Tl, i);
    }
  }
}

// Forward transform (S = -1) of the sequence in registers: in[jb R + m] is
// position t + jb TPS + m N / R for R the first radix.  MEASURE: the inputs
// leave room for the first stage only, and a shift measured after it makes
// room for the others, with SPARE bits of the result free; the shift is
// returned.  The result, times 2^-SHIFT, is left in buf, in natural order,
// synchronised; only the band KB is formed.
template <typename P, int KB, bool MEASURE, int SPARE>
__device__ __forceinline__ int fx_forward(q2* in, q2* buf, const int4* tw, int t, int id, int* scratch) {
  using F = typename P::fwd;
  using Tail = typename TailRadices<F>::type;
  constexpr int R1 = FirstRadix<F>::value, RL = LastRadix<F>::value, L = P::N / RL;
  constexpr int C = gap_common(P::N, RL, KB);  // outputs in the gap for every butterfly
  using B1 = Bfly<P, R1>;
  using BL = Bfly<P, RL>;
  int big = 0, r = 0;
  seq_sync<P::TPS>(id);  // the registers may have been loaded from this buffer
  if (B1::active(t)) {
#pragma unroll
    for (int jb = 0; jb < B1::J; ++jb) {
      q2* a = in + jb * R1;
      qdftR<R1, -1, 0>(a);
      if constexpr (MEASURE) {
#pragma unroll
        for (int m = 0; m < R1; ++m) big = max_mag(big, a[m]);
      }
      fx_store<P, R1, 1>(a, buf, t + jb * P::TPS);
    }
  }
  if constexpr (MEASURE) big = seq_max_put<P::TPS>(big, t, scratch);
  seq_sync<P::TPS>(id);
  if constexpr (MEASURE) r = max(0, bits64(seq_max_get<P::TPS>(big, scratch)) - (62 - SPARE - P::GROWTH2));
  using Mid = typename InitRadices<Tail>::type;
  constexpr bool MIDDLE = L > R1;  // there are middle stages
  fx_middle<P, -1, R1, MEASURE && MIDDLE>(buf, tw, t, id, r, Mid{});
  q2 a[BL::POINTS];
  if (BL::active(t)) {
    const int4* Tl = tw + P::ENTRIES - (RL - 1) * L;
#pragma unroll
    for (int jb = 0; jb < BL::J; ++jb) {
      const int i = t + jb * P::TPS;
      q2* b = a + jb * RL;
      fx_load<P, RL>(b, buf, i);
      if constexpr (MEASURE && !MIDDLE) {
        if (r > 0) {
#pragma unroll
          for (int m = 0; m < RL; ++m) b[m] = mkq(shr_round(b[m].x, r), shr_round(b[m].y, r));
        }
      }
      fx_butterfly<RL, -1, L, 0>(b, Tl, i);
    }
  }
  seq_sync<P::TPS>(id);
  if (BL::active(t)) {
#pragma unroll
    for (int jb = 0; jb < BL::J; ++jb) {
      q2* d = buf + pad(t + jb * P::TPS);
#pragma unroll
      for (int m = 0; m < RL; ++m)
        if (!((C >> m) & 1)) d[pad(m * L)] = a[jb * RL + m];
    }
  }
  seq_sync<P::TPS>(id);
  return r;
}

}  // namespace da
