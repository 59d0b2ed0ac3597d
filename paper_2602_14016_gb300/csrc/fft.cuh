// fft.cuh -- radix plans and gap masks of the integer FFT engine (fx.cuh), and
// an FP64 shared-memory FFT for the allocation-free control map.
//
// A CTA transforms a complex sequence of length N held in shared memory, with a mixed-radix Stockham auto-sort algorithm: stage s with
// radix R and current sub-length L loads the R points x[i + m N/R] of
// butterfly i, twiddles them by W_{LR}^{m (i mod L)}, applies an R-point DFT
// in registers and stores them to y[(i - i mod L) R + i mod L + m L].  After
// the last stage (L = N) the output is in natural order.  The FP64 stages work
// in place: every thread holds its butterfly in registers across a barrier.
// fft_sequence takes a plain table of W_N^t = exp(-2 pi i t / N) (conjugated for
// the inverse sign); the allocation-free control map has static scratch and no
// context to keep the integer engine's tables.
#pragma once
#include <cuda_runtime.h>

#include <cmath>

namespace da {

__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cscale(double2 a, double s) { return make_double2(a.x * s, a.y * s); }

// (S i) * a, S = +-1
template <int S>
__device__ __forceinline__ double2 mul_si(double2 a) {
  return S > 0 ? make_double2(-a.y, a.x) : make_double2(a.y, -a.x);
}

// Bits 0, 2, 4, ... (even) or 1, 3, 5, ... (odd) of a zero mask of r inputs,
// packed: the masks of the two half-length DFTs of an even/odd split.
__host__ __device__ constexpr int even_bits(int z, int r) {
  int o = 0;
  for (int j = 0; j < r / 2; ++j) o |= ((z >> (2 * j)) & 1) << j;
  return o;
}
__host__ __device__ constexpr int odd_bits(int z, int r) { return even_bits(z >> 1, r); }

// X_k = sum_m a_m exp(S 2 pi i m k / R), in place, natural order.
template <int S>
__device__ __forceinline__ void dft4(double2* a) {
  const double2 t0 = cadd(a[0], a[2]), t1 = csub(a[0], a[2]);
  const double2 t2 = cadd(a[1], a[3]), t3 = mul_si<S>(csub(a[1], a[3]));
  a[0] = cadd(t0, t2);
  a[2] = csub(t0, t2);
  a[1] = cadd(t1, t3);
  a[3] = csub(t1, t3);
}

// cos(pi/4)
constexpr double kR2 = 0.70710678118654752440;

// Output pair of a radix-2 combination with a scaled twiddle:
// e +- c z, as two FMAs per component.
__device__ __forceinline__ void bfly_scaled(const double2 e, const double2 z, double c, double2& plus, double2& minus) {
  plus = make_double2(fma(c, z.x, e.x), fma(c, z.y, e.y));
  minus = make_double2(fma(-c, z.x, e.x), fma(-c, z.y, e.y));
}

// The twiddles w = (+-1 + S i)/sqrt2 of the internal combinations are written
// as c z with z two adds, so that e +- w o = e +- c z costs four FMAs.
template <int S>
__device__ __forceinline__ void dft8(double2* a) {
  double2 e[4] = {a[0], a[2], a[4], a[6]};
  double2 o[4] = {a[1], a[3], a[5], a[7]};
  dft4<S>(e);
  dft4<S>(o);
  // k = 0
  a[0] = cadd(e[0], o[0]);
  a[4] = csub(e[0], o[0]);
  // k = 2: w = S i
  const double2 o2 = mul_si<S>(o[2]);
  a[2] = cadd(e[2], o2);
  a[6] = csub(e[2], o2);
  // k = 1: w = (1 + S i)/sqrt2
  const double2 z1 = make_double2(o[1].x - S * o[1].y, o[1].y + S * o[1].x);
  bfly_scaled(e[1], z1, kR2, a[1], a[5]);
  // k = 3: w = (-1 + S i)/sqrt2 = -(1 - S i)/sqrt2
  const double2 z3 = make_double2(o[3].x + S * o[3].y, o[3].y - S * o[3].x);
  bfly_scaled(e[3], z3, -kR2, a[3], a[7]);
}

template <int R, int S>
__device__ __forceinline__ void dftR(double2* a) {
  static_assert(R == 4 || R == 8, "the plans of the allocation-free control map");
  if constexpr (R == 4) dft4<S>(a);
  if constexpr (R == 8) dft8<S>(a);
}

// Radix plans: a list of stage radices whose product is N.
template <int... Rs>
struct Radices {};

// Plans: for each size N, a few variants V of the radix list used for two
// concurrent transforms (the pass kernels; `two`) and for a single transform
// (`one`), with the CTA width they run on.  Wide radices keep the
// instruction count low; narrow ones and wider CTAs keep more warps in
// flight.  A stage with more butterflies than threads gives each thread
// several.  Variant 0 is the default; the autotuner (da_autotune) times the
// variants of a grid on the context's own batch and keeps the fastest.  The
// allocation-free control map uses variant 0.
template <int N, int V = 0> struct Plan;
template <> struct Plan<16, 0> { using two = Radices<4, 4>; using one = Radices<4, 4>; static constexpr int threads = 32; };
template <> struct Plan<32, 0> { using two = Radices<4, 8>; using one = Radices<4, 8>; static constexpr int threads = 32; };
template <> struct Plan<64, 0> { using two = Radices<4, 4, 4>; using one = Radices<4, 4, 4>; static constexpr int threads = 32; };
template <> struct Plan<64, 1> { using two = Radices<8, 8>; using one = Radices<8, 8>; static constexpr int threads = 32; };
// Radix-2 plans: more instructions than the radix-4 ones, but a shorter chain a
// thread.  Small grids at small batches, whose pass kernels are bound by that
// chain, run faster on them: 128^2, one member, 5.3 us a pass on plan 0 and 4.2
// on plan 3; 24 members 9.2 and 9.5.
template <> struct Plan<32, 1> { using two = Radices<2, 2, 2, 2, 2>; using one = Radices<2, 2, 2, 2, 2>; static constexpr int threads = 32; };
template <> struct Plan<64, 2> { using two = Radices<2, 2, 2, 2, 2, 2>; using one = Radices<2, 2, 2, 2, 2, 2>; static constexpr int threads = 64; };
template <> struct Plan<128, 0> { using two = Radices<4, 4, 8>; using one = Radices<4, 4, 8>; static constexpr int threads = 64; };
template <> struct Plan<128, 1> { using two = Radices<8, 4, 4>; using one = Radices<8, 4, 4>; static constexpr int threads = 64; };
template <> struct Plan<128, 2> { using two = Radices<4, 4, 8>; using one = Radices<4, 4, 8>; static constexpr int threads = 32; };
template <> struct Plan<128, 3> { using two = Radices<2, 2, 2, 2, 2, 2, 2>; using one = Radices<2, 2, 2, 2, 2, 2, 2>; static constexpr int threads = 128; };
template <> struct Plan<256, 0> { using two = Radices<4, 4, 4, 4>; using one = Radices<4, 4, 4, 4>; static constexpr int threads = 128; };
template <> struct Plan<256, 1> { using two = Radices<8, 8, 4>; using one = Radices<8, 8, 4>; static constexpr int threads = 64; };
template <> struct Plan<256, 2> { using two = Radices<4, 4, 4, 4>; using one = Radices<4, 4, 4, 4>; static constexpr int threads = 64; };
template <> struct Plan<512, 0> { using two = Radices<8, 8, 8>; using one = Radices<8, 8, 8>; static constexpr int threads = 128; };
template <> struct Plan<512, 1> { using two = Radices<8, 4, 4, 4>; using one = Radices<8, 4, 4, 4>; static constexpr int threads = 128; };
template <> struct Plan<512, 2> { using two = Radices<8, 8, 8>; using one = Radices<8, 8, 8>; static constexpr int threads = 64; };
template <> struct Plan<1024, 0> { using two = Radices<16, 8, 8>; using one = Radices<16, 8, 8>; static constexpr int threads = 256; };
template <> struct Plan<1024, 1> { using two = Radices<16, 4, 4, 4>; using one = Radices<16, 4, 4, 4>; static constexpr int threads = 256; };
template <> struct Plan<1024, 2> { using two = Radices<8, 8, 4, 4>; using one = Radices<8, 8, 4, 4>; static constexpr int threads = 256; };

// Number of plan variants of each size (the instantiations in inst_n*.cu).
constexpr int plan_count(int n) {
  return n == 32 ? 2 : n == 64 ? 3 : n == 128 ? 4 : (n == 256 || n == 512 || n == 1024) ? 3 : 1;
}

template <int N, int V = 0>
struct PlanInfo {
  static constexpr int THREADS = Plan<N, V>::threads;
};

// One in-place Stockham stage on the N points in `buf`: every thread loads the
// R points of each of its butterflies, twiddles and transforms them in
// registers, waits for all loads, then stores.
template <int N, int R, int S>
__device__ __forceinline__ void stockham_stage(double2* buf, int L, const double2* __restrict__ tw) {
  constexpr int NB = N / R, T = PlanInfo<N>::THREADS, J = (NB + T - 1) / T;
  double2 a[J][R];
  int dst[J];
#pragma unroll
  for (int jb = 0; jb < J; ++jb) {
    const int i = threadIdx.x + jb * T;
    dst[jb] = 0;
    if (NB % T == 0 || i < NB) {
      const int k = i & (L - 1);
#pragma unroll
      for (int m = 0; m < R; ++m) a[jb][m] = buf[i + m * NB];
      if (L > 1) {
        const int step = N / (L * R);
#pragma unroll
        for (int m = 1; m < R; ++m) {
          double2 w = tw[m * k * step];
          if (S > 0) w.y = -w.y;
          a[jb][m] = cmul(a[jb][m], w);
        }
      }
      dftR<R, S>(a[jb]);
      dst[jb] = (i - k) * R + k;
    }
  }
  __syncthreads();
#pragma unroll
  for (int jb = 0; jb < J; ++jb) {
    const int i = threadIdx.x + jb * T;
    if (NB % T == 0 || i < NB) {
#pragma unroll
      for (int m = 0; m < R; ++m) buf[dst[jb] + m * L] = a[jb][m];
    }
  }
  __syncthreads();
}

template <int N, int S, int L>
__device__ __forceinline__ void run_stages(double2*, const double2*, Radices<>) {}

template <int N, int S, int L, int R, int... Rs>
__device__ __forceinline__ void run_stages(double2* buf, const double2* tw, Radices<R, Rs...>) {
  stockham_stage<N, R, S>(buf, L, tw);
  run_stages<N, S, L * R>(buf, tw, Radices<Rs...>{});
}

// ---------------------------------------------------------------------------
// Band-limited sequences
// ---------------------------------------------------------------------------
//
// The inverse transforms of the pass kernels read sequences that are zero in
// the gap K < q < N - K (the 2/3 rule, K = (N-1)/3), and their forward
// transforms are read back only on the band q <= K, q >= N - K.  Input m of
// butterfly i of the first stage is x[i + m N/R]; output m of butterfly k of
// the last stage is y[k + m N/R].  Where that position lies in the gap for
// every butterfly, the load and the additions the zero would enter (first
// stage), or the output's forming and storing (last stage), are left out
// (gap_common).  The nominal flop counts (da_plan_flops) also leave out what
// lies in the gap for all 32 lanes of a warp (GapMask), which FP64 stages can
// skip and the integer stages of fx.cuh do not.

// positions lo..hi all in the gap of band kb (kb < 0: no band)
__host__ __device__ constexpr bool in_gap(int n, int kb, int lo, int hi) {
  return kb >= 0 && lo >= kb + 1 && hi <= n - kb - 1;
}
// m whose position is in the gap for every butterfly of a stage of radix r
__host__ __device__ constexpr int gap_common(int n, int r, int kb) {
  int c = 0;
  for (int m = 0; m < r; ++m)
    if (in_gap(n, kb, m * (n / r), m * (n / r) + n / r - 1)) c |= 1 << m;
  return c;
}
// m in the gap for all lanes of some warps only
__host__ __device__ constexpr int gap_per_warp(int n, int r, int kb) {
  const int nb = n / r;
  int c = 0;
  if (nb % 32) return 0;
  for (int m = 0; m < r; ++m)
    for (int i0 = 0; i0 < nb; i0 += 32)
      if (!((gap_common(n, r, kb) >> m) & 1) && in_gap(n, kb, i0 + m * nb, i0 + 31 + m * nb)) c |= 1 << m;
  return c;
}
__host__ __device__ constexpr int bit_index(int b) {
  int m = 0;
  while (b > 1) {
    b >>= 1;
    ++m;
  }
  return m;
}
__host__ __device__ constexpr int popcount_c(int b) {
  int c = 0;
  for (; b; b &= b - 1) ++c;
  return c;
}

template <int N, int R, int KB>
struct GapMask {
  static constexpr int NB = N / R;
  static constexpr int C = gap_common(N, R, KB), X = gap_per_warp(N, R, KB);
  static constexpr int A = X & -X, B = X & ~A;  // the per-warp bits
  static_assert((B & (B - 1)) == 0, "at most two per-warp gap positions per butterfly");
  // mask of the warp that holds butterfly i
  __host__ __device__ static int warp(int i) {
    int w = C;
    if constexpr (A != 0) {
      const int i0 = i & ~31;
      constexpr int ma = bit_index(A);
      if (in_gap(N, KB, i0 + ma * NB, i0 + 31 + ma * NB)) w |= A;
      if constexpr (B != 0) {
        constexpr int mb = bit_index(B);
        if (in_gap(N, KB, i0 + mb * NB, i0 + 31 + mb * NB)) w |= B;
      }
    }
    return w;
  }
};

// First and last radix of a plan, the plan without its last stage, and
// without its first.
template <typename P> struct FirstRadix;
template <int R, int... Rs> struct FirstRadix<Radices<R, Rs...>> { static constexpr int value = R; };
template <typename P> struct LastRadix;
template <int R> struct LastRadix<Radices<R>> { static constexpr int value = R; };
template <int R, int R2, int... Rs> struct LastRadix<Radices<R, R2, Rs...>> {
  static constexpr int value = LastRadix<Radices<R2, Rs...>>::value;
};
template <int R, typename P> struct Prepend;
template <int R, int... Rs> struct Prepend<R, Radices<Rs...>> { using type = Radices<R, Rs...>; };
template <typename P> struct InitRadices;
template <int R> struct InitRadices<Radices<R>> { using type = Radices<>; };
template <int R, int R2, int... Rs> struct InitRadices<Radices<R, R2, Rs...>> {
  using type = typename Prepend<R, typename InitRadices<Radices<R2, Rs...>>::type>::type;
};
template <typename P> struct TailRadices;
template <int R, int... Rs> struct TailRadices<Radices<R, Rs...>> { using type = Radices<Rs...>; };

// Host side: nominal flops of one band-limited transform of N points under
// Plan<N, V>: 5 N log2 N less the FP64 operations that warp-wide gap tests
// would skip in the list's first stage (inverse) and last stage (forward); a
// real addition or multiplication counts one, an FMA two.  A measure of the
// work, the same whatever arithmetic does it: the pass kernels run integer
// stages, whose inverse begins with the list's last radix.  Inverse: the zero
// inputs of the first stage; forward: the unformed outputs of the last (two
// FMAs each).

// flops a zero mask z saves in the untwiddled r-point DFT (dft2/4/8/16):
// every add_z / sub_z with a known-zero operand saves one complex addition
constexpr int zero_savings(int r, int z) {
  if (r == 2) return (z & 3) ? 4 : 0;
  if (r == 4) {
    const bool z0 = z & 1, z1 = (z >> 1) & 1, z2 = (z >> 2) & 1, z3 = (z >> 3) & 1;
    return ((z0 || z2) ? 4 : 0) + ((z1 || z3) ? 4 : 0) + (((z0 && z2) || (z1 && z3)) ? 8 : 0);
  }
  return zero_savings(r / 2, even_bits(z, r)) + zero_savings(r / 2, odd_bits(z, r));
}

template <int N, int V, int KB>
inline double band_transform_flops(bool inverse) {
  using P = typename Plan<N, V>::two;
  double saved = 0.0;
  if (inverse) {
    constexpr int R = FirstRadix<P>::value;
    for (int i = 0; i < N / R; ++i) saved += zero_savings(R, GapMask<N, R, KB>::warp(i));
  } else {
    constexpr int R = LastRadix<P>::value;
    for (int i = 0; i < N / R; ++i) saved += 4 * popcount_c(GapMask<N, R, KB>::warp(i));
  }
  return 5.0 * N * std::log2((double)N) - saved;
}

// Transform, in place, the N points in buf.  Called by every thread of a CTA of
// PlanInfo<N>::THREADS threads, with buf already synchronised; returns after a
// final __syncthreads().
template <int N, int S>
__device__ __forceinline__ void fft_sequence(double2* buf, const double2* tw) {
  run_stages<N, S, 1>(buf, tw, typename Plan<N>::one{});
}

}  // namespace da
