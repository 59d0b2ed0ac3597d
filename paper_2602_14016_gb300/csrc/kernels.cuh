// kernels.cuh -- pass kernels of the cost-and-gradient evaluation.
//
// Layout (per member b of a batch):
//   compact spectra  [Kc][Kr] complex, column-major (cidx): the retained
//                    set of the 2/3 rule, kx = 0..K (columns), compact row
//                    r -> ky = r (r <= K) or r - Kr; K = floor((N-1)/3),
//                    Kc = K+1, Kr = 2K+1.  A column pass reads and writes one
//                    contiguous column.
//   mixed fields     physical y, spectral kx (kx = 0..K), two fields: the
//                    column-pass output Mx row-major [2][N][Kc] (a row
//                    pass reads whole rows), the row-pass output Mn
//                    column-major [Kc][2][N] (a column pass reads its
//                    column of both fields as one contiguous block).
//   stage fields     [nsteps][4 stages][N][N] (u, v) of every RK stage
//                    state, written by the forward row pass and read back by
//                    the adjoint row pass.
// Mixed and stage fields are 64-bit integers (fx.cuh) with one exponent per
// column and field (Mx) or per row (Mn, stage fields) beside them; compact
// spectra, observations, controls and gradients are doubles.  (The control
// maps use Mn as a field of doubles.)
//
// The advection term is evaluated in the divergence form of Basdevant
// (1983): for a divergence-free band-limited velocity,
//   u . grad w = (d_xx - d_yy)(u v) + d_xy (v^2 - u^2),
// and with the 2/3 rule both sides are the same retained coefficients (the
// products of retained fields alias nothing onto the retained set), so the
// discrete right-hand side is the one of the advective form, u w_x + v w_y,
// evaluated with four real transforms instead of five and two stored stage
// fields instead of four.
//
// A forward RK stage is two kernels: a ROW pass (inverse transforms along x
// of the packed mixed rows -> u, v; stage-field store; probe gather; the
// products u v and v^2 - u^2; their forward transforms along x, handed over
// in registers: fx_turn) and a COLUMN
// pass (forward transforms along y of the two products, the advection term,
// RK epilogue with viscosity, forcing and the stage update, then the
// inverse column transforms of the next stage's u and v).  The adjoint
// mirrors this with the transposed operators.  Every transform between the
// control and its gradient is an integer FFT from fx.cuh; those of the control
// maps are FP64 FFTs from fft.cuh.  The 1/N^2 of the inverse 2D transform is
// applied once, to the spectral coefficients before the column transform.
// Every inverse transform here reads a sequence that is zero in the gap
// K < q < N - K, and every forward transform is read back only on the band
// q <= K, q >= N - K: the transforms are band-limited (KIN / KOUT = K) and
// skip that work where whole warps allow.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "fx.cuh"

namespace da {

enum : int {
  F_STORE = 1,     // forward row pass: write stage fields
  F_OBS = 2,       // forward row pass: gather probes into the observation slot
  F_OBS_ONLY = 4,  // forward row pass: only gather probes (final state)
  F_NO_NEXT = 8,   // column pass: skip the inverse transforms of the next stage
  F_SRC = 16       // adjoint column pass: add the observation source at this step
};

// Start of the adjoint sweep (k_adj_init): add the observation source of
// the last step, and/or start from the terminal field already in LamBar; or
// resume from the adjoint stage value in KB after a checkpoint recompute.
enum : int { INIT_SRC = 1, INIT_LAMBAR = 2, INIT_RESUME = 4 };

// Multipliers of the generic spectral-to-mixed column pass.
enum : int { M_ONE = 0, M_CTRL = 1, M_FILTERED = 2, M_INV_CTRL = 3 };

// Per-mode constants of the column passes, column-major [Kc][Kr] (entry
// kx * Kr + r), computed once on the host so that no column pass divides or
// converts integers in FP64:
//   fwd: su = ky/k^2/N^2, sv = kx/k^2/N^2 (u, v columns of a state value),
//        cp = (ky^2 - kx^2)/2, cq = -kx ky/2 (advection symbols; the 1/2 is
//        the one the row pass leaves out when it unpacks two real rows);
//   adj: a1 = ky/k^2/2, c1 = kx/k^2/2 (transposed velocity symbols, same
//        1/2), ca = -2 kx ky/N^2, cb = (ky^2 - kx^2)/N^2 (adjoint-field
//        columns; ca carries the 2 of rho_u, rho_v);
//   k2 = k^2 (the column passes multiply it by the member's viscosity).
struct __align__(32) Sym4 {
  double a, b, c, d;
};

// Everything a kernel needs, passed by value.
struct Dev {
  int B, nsteps, every, include_t0, px, nt;  // nsteps: the evaluation's window (global steps)
  double dt, nu;
  int force;
  double amp;
  int nf;
  // Ragged batches: member b runs its own window, end-aligned in the
  // evaluation's -- live from global step mstart[b] to nsteps, its local step
  // n - mstart[b] -- with its own probe lattice, viscosity and forcing switch;
  // a member with mstart[b] > nsteps is idle.  With ragged == 0 every member
  // runs the context's window and the tables are not read.
  int ragged;
  const int* mstart;                         // [B]
  const int* mnt;                            // [B] observation times of member b
  const int* mpx;                            // [B] probes per side of member b
  const double* mnu;                         // [B]
  const int* mforce;                         // [B] Kolmogorov forcing on (1) or off (0)
  size_t obs_stride;                         // doubles from one member's obs, mobs, res to the next
  double2 *W, *Acc, *Y, *KB, *LamBar, *Sum;  // compact [B][Kc][Kr] (cidx)
  q2* Mx;                                    // mixed [B][2][N][Kc]: column-pass output
  int* eX;                                   // [B][2][Kc] exponents of Mx (one per column and field)
  q2* Mn;                                    // mixed [B][Kc][2][N]: row-pass output
  int* eN;                                   // [B][N] exponents of Mn (one per row)
  q2* traj;                                  // [B][traj_steps][4][N][N] (u, v)
  int* eT;                                   // [B][traj_steps][4][N] exponents of traj (one per row)
  int traj_steps;                            // steps the stage-field store holds
  int seg0;                                  // step stored in slot 0 of the store
  double* obs;                               // model observations [B][nt][P2][2]
  const double* mobs;                        // data [B][nt][P2][2]
  double* res;                               // residuals [B][nt][P2][2]
  double* J;                                 // [B]
  const double* mult;                        // control multiplier |k| W^1/2, compact [B][Kc][Kr]
  const double* fold;                        // folded twiddles of Plan<N> (fft.cuh)
  const int4* fxtw;                          // integer twiddles of FxPlan<N> (fx.cuh)
  const double2* twP;                        // W_64^t, t < 64 (W_P^t = W_64^{t 64/P})
  const Sym4* symF;                          // [Kc][Kr] su, sv, cp, cq
  const Sym4* symA;                          // [Kc][Kr] a1, c1, ca, cb
  const double* k2;                          // [Kc][Kr] k^2 (times nu of the member)
  double dt2, dt3, dt6;                      // dt/2, dt/3, dt/6
};

template <int N, int V = 0>
struct Geo {
  static constexpr int K = (N - 1) / 3;
  static constexpr int Kc = K + 1;
  static constexpr int Kr = 2 * K + 1;
  static constexpr int NH = N / 2 + 1;
  // threads: two transforms at a time (fft.cuh)
  static constexpr int THREADS = PlanInfo<N, V>::THREADS;
  // shared memory: folded twiddle table + one buffer of two sequences +
  // probe sums
  static constexpr int PMAX = 64;
  static constexpr int SCRATCH = 4 * 2 * 8;  // ints: four reductions of two values over at most 8 warps
  static constexpr size_t SMEM =
      sizeof(double) * FoldInfo<N, V>::PADDED + sizeof(double2) * (2 * N + 2 * PMAX) + sizeof(int) * SCRATCH;
  // passes that run the integer transforms only: two sequences, probe sums, scratch
  static constexpr size_t SMEM_FX = sizeof(q2) * (2 * N + 2 * PMAX) + sizeof(int) * SCRATCH;
  // column passes load their epilogue inputs before the transforms (about
  // 60 more registers a thread) where a CTA is at most 128 threads
  static constexpr bool PREFETCH = THREADS <= 128;
};

__device__ __forceinline__ int ky_of_row(int r, int K) { return r <= K ? r : r - (2 * K + 1); }

// Index of mode (row r, column kx) of member bm in a compact array.
template <int N>
__host__ __device__ __forceinline__ size_t cidx(int bm, int r, int kx) {
  return ((size_t)bm * Geo<N>::Kc + kx) * Geo<N>::Kr + r;
}

template <int N, int V = 0>
__device__ __forceinline__ void load_fold(double* T, const double* __restrict__ g) {
  for (int i = threadIdx.x; i < FoldInfo<N, V>::DOUBLES; i += blockDim.x) T[i] = g[i];
}

// The window of member bm in this evaluation (see Dev).
struct MemberWindow {
  int start, P;
  double nu;
  bool forced;
};

__device__ __forceinline__ MemberWindow member_window(const Dev& d, int bm) {
  if (!d.ragged) return {0, d.px, d.nu, d.force != 0};
  return {d.mstart[bm], d.mpx[bm], d.mnu[bm], d.force != 0 && d.mforce[bm] != 0};
}

// Observation slot of local step k, or -1.
__device__ __forceinline__ int obs_slot(const Dev& d, int k) {
  if (k == 0) return d.include_t0 ? 0 : -1;
  if (k % d.every) return -1;
  return k / d.every - 1 + (d.include_t0 ? 1 : 0);
}

// Full-length sequence whose inverse transform is a + i b, for two real rows
// a, b given by their mixed half spectra A, B (kx = 0..K): Z(kx) = A + iB,
// Z(-kx) = conj(A) + i conj(B); the DC bin keeps real parts only.  Every
// coefficient is loaded once and written to kx and -kx; the gap
// K < kx < N-K is zeroed.  Coefficient kx of A and Bv is at [kx * STRIDE].
// Loops run over compile-time trip counts so that a thread's loads are
// issued together.
template <int N, int T, int STRIDE = 1>
__device__ __forceinline__ void pack_rows(double2* seq, const double2* __restrict__ A, const double2* __restrict__ Bv) {
  constexpr int K = Geo<N>::K, GAP = N - 2 * K - 1;
#pragma unroll
  for (int t = 0; t < (GAP + T - 1) / T; ++t) {
    const int u = threadIdx.x + t * T;
    if (u < GAP) seq[K + 1 + u] = make_double2(0.0, 0.0);
  }
#pragma unroll
  for (int t = 0; t < (K + 1 + T - 1) / T; ++t) {
    const int kx = threadIdx.x + t * T;
    if (kx <= K) {
      const double2 p = A[(size_t)kx * STRIDE], q = Bv[(size_t)kx * STRIDE];
      if (kx == 0) {
        seq[0] = make_double2(p.x, q.x);
      } else {
        seq[kx] = make_double2(p.x - q.y, p.y + q.x);
        seq[N - kx] = make_double2(p.x + q.y, q.x - p.y);
      }
    }
  }
}

// The two half spectra packed in a forward transform Z of a + i b:
// A(k) = (Z(k) + conj Z(-k))/2, B(k) = -i (Z(k) - conj Z(-k))/2.
template <int N, int V = 0>
__device__ __forceinline__ void unpack_pair(const double2* Z, int kx, double2& A, double2& Bv) {
  const double2 zk = Z[kx], zm = Z[(N - kx) & (N - 1)];
  const double sx = zk.x + zm.x, sy = zk.y - zm.y;
  const double tx = zk.x - zm.x, ty = zk.y + zm.y;
  A = make_double2(0.5 * sx, 0.5 * sy);
  Bv = make_double2(0.5 * ty, -0.5 * tx);
}

// ---------------------------------------------------------------------------
// Generic row transforms (control map, gradient map)
// ---------------------------------------------------------------------------

// Real rows in[b][y][x] -> mixed half rows Mn[b][y][kx], kx <= K (forward,
// unnormalised), two rows per complex transform.  grid (N/2, B).
template <int N, int V = 0>
__global__ void __launch_bounds__(Geo<N, V>::THREADS) k_r2c_rows(Dev d, const double* __restrict__ in) {
  using G = Geo<N, V>;
  extern __shared__ double2 sm[];
  double* T = reinterpret_cast<double*>(sm);
  double2* a = sm + FoldInfo<N, V>::PADDED / 2;
  const int bm = blockIdx.y, y0 = 2 * blockIdx.x;
  load_fold<N, V>(T, d.fold);
  const double* r0 = in + ((size_t)bm * N + y0) * N;
  #pragma unroll
  for (int x = threadIdx.x; x < N; x += G::THREADS) a[x] = make_double2(r0[x], r0[N + x]);
  __syncthreads();
  fft_folded<N, V, -1, 1, -1, G::K>(a, T);
  double2* M = reinterpret_cast<double2*>(d.Mn) + (size_t)bm * G::Kc * 2 * N + y0;  // field 0, rows y0 and y0 + 1
  #pragma unroll
  for (int kx = threadIdx.x; kx < G::Kc; kx += G::THREADS) {
    double2 A, Bv;
    unpack_pair<N>(a, kx, A, Bv);
    M[(size_t)kx * 2 * N] = A;
    M[(size_t)kx * 2 * N + 1] = Bv;
  }
}

// Mixed half rows Mn[b][y][kx] -> real rows out[b][y][x] (the inverse along
// x; the 1/N^2 is already in Mn), two rows per complex transform.
template <int N, int V = 0>
__global__ void __launch_bounds__(Geo<N, V>::THREADS) k_c2r_rows(Dev d, double* __restrict__ out) {
  using G = Geo<N, V>;
  extern __shared__ double2 sm[];
  double* T = reinterpret_cast<double*>(sm);
  double2* a = sm + FoldInfo<N, V>::PADDED / 2;
  const int bm = blockIdx.y, y0 = 2 * blockIdx.x;
  load_fold<N, V>(T, d.fold);
  const double2* M = reinterpret_cast<const double2*>(d.Mn) + (size_t)bm * G::Kc * 2 * N + y0;  // field 0, rows y0 and y0 + 1
  pack_rows<N, G::THREADS, 2 * N>(a, M, M + 1);
  __syncthreads();
  fft_folded<N, V, +1, 1, G::K>(a, T);
  double* r0 = out + ((size_t)bm * N + y0) * N;
  #pragma unroll
  for (int x = threadIdx.x; x < N; x += G::THREADS) {
    r0[x] = a[x].x;
    r0[N + x] = a[x].y;
  }
}

// Compact spectrum src[b] times a multiplier (and 1/N^2), transformed along
// y -> mixed Mn[b] (first field).  grid (Kc, B).
template <int N, int V = 0>
__global__ void __launch_bounds__(Geo<N, V>::THREADS) k_spec_to_mixed(Dev d, const double2* __restrict__ src, int mode) {
  using G = Geo<N, V>;
  extern __shared__ double2 sm[];
  double* T = reinterpret_cast<double*>(sm);
  double2* a = sm + FoldInfo<N, V>::PADDED / 2;
  const int kx = blockIdx.x, bm = blockIdx.y;
  load_fold<N, V>(T, d.fold);
  const double s = 1.0 / ((double)N * N);
  #pragma unroll
  for (int q = threadIdx.x; q < N; q += G::THREADS) {
    const int ky = q < N / 2 ? q : q - N;
    double2 v = make_double2(0.0, 0.0);
    if (ky >= -G::K && ky <= G::K) {
      const int r = ky >= 0 ? ky : ky + G::Kr;
      const size_t idx = cidx<N>(bm, r, kx);
      const double m = d.mult[idx];
      double f;
      if (mode == M_ONE) f = 1.0;
      else if (mode == M_CTRL) f = m;
      else if (mode == M_FILTERED) f = (kx == 0 && ky == 0) ? 0.0 : m * m / sqrt((double)(kx * kx + ky * ky));
      else f = m != 0.0 ? 1.0 / m : 0.0;
      v = cscale(src[idx], f * s);
    }
    a[q] = v;
  }
  __syncthreads();
  fft_folded<N, V, +1, 1, G::K>(a, T);
  double2* M = reinterpret_cast<double2*>(d.Mn) + ((size_t)bm * G::Kc + kx) * 2 * N;  // field 0 of column kx
  #pragma unroll
  for (int y = threadIdx.x; y < N; y += G::THREADS) M[y] = a[y];
}

// Compact <-> half-spectrum copies.  grid (ceil(N*NH/256), B), block 256.
template <int N, int V = 0>
__global__ void k_compact_to_half(const double2* __restrict__ src, double2* __restrict__ out) {
  using G = Geo<N, V>;
  const int bm = blockIdx.y;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N * G::NH; i += gridDim.x * blockDim.x) {
    const int q = i / G::NH, p = i - q * G::NH;
    const int ky = q < N / 2 ? q : q - N;
    double2 v = make_double2(0.0, 0.0);
    if (p <= G::K && ky >= -G::K && ky <= G::K) {
      const int r = ky >= 0 ? ky : ky + G::Kr;
      v = src[cidx<N>(bm, r, p)];
    }
    out[(size_t)bm * N * G::NH + i] = v;
  }
}

template <int N, int V = 0>
__global__ void k_half_to_compact(const double2* __restrict__ in, double2* __restrict__ dst) {
  using G = Geo<N, V>;
  const int bm = blockIdx.y;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < G::Kr * G::Kc; i += gridDim.x * blockDim.x) {
    const int kx = i / G::Kr, r = i - kx * G::Kr;
    const int ky = ky_of_row(r, G::K);
    dst[(size_t)bm * G::Kr * G::Kc + i] = in[((size_t)bm * N + (ky & (N - 1))) * G::NH + kx];
  }
}

// ---------------------------------------------------------------------------
// Control map and the inverse column transforms of a stage state
// ---------------------------------------------------------------------------

// Shared memory of the pass kernels: the two sequences, the probe sums and
// the scratch of the reductions.
template <int N>
struct FxSmem {
  q2* a;
  double2 *Tu, *Tv;
  int* scratch;
  __device__ __forceinline__ explicit FxSmem(void* base) {
    a = static_cast<q2*>(base);
    Tu = reinterpret_cast<double2*>(a + 2 * N);
    Tv = Tu + Geo<N>::PMAX;
    scratch = reinterpret_cast<int*>(Tv + Geo<N>::PMAX);
  }
};

// A column under construction: complex doubles, as raw bits, at the retained
// positions of two sequences, and the largest exponent field of each.
template <int N>
struct ColumnPut {
  q2* a;
  int f0 = 0, f1 = 0;
  __device__ __forceinline__ explicit ColumnPut(q2* a_) : a(a_) {}
  __device__ __forceinline__ void put(int q, double2 v0, double2 v1) {
    a[q] = mkq(__double_as_longlong(v0.x), __double_as_longlong(v0.y));
    a[N + q] = mkq(__double_as_longlong(v1.x), __double_as_longlong(v1.y));
    f0 = max(f0, max(exp_field(v0.x), exp_field(v0.y)));
    f1 = max(f1, max(exp_field(v1.x), exp_field(v1.y)));
  }
};

// The two column values u = i ky/k^2 Yv, v = -i kx/k^2 Yv (scaled by 1/N^2;
// f = symF entry of the mode) at position q.
template <int N>
__device__ __forceinline__ void put_stage_columns(ColumnPut<N>& c, int q, const Sym4& f, double2 Yv) {
  c.put(q, make_double2(-f.a * Yv.y, f.a * Yv.x),  // u:  i ky / k^2
        make_double2(f.b * Yv.y, -f.b * Yv.x));    // v: -i kx / k^2
}

// The two column values of the adjoint fields of an adjoint stage value kb:
// 2a = 2 d_xy kb = -2 kx ky kb and b = (d_xx - d_yy) kb = (ky^2 - kx^2) kb,
// scaled by 1/N^2 (g = symA entry of the mode), at q.
template <int N>
__device__ __forceinline__ void put_adjoint_columns(ColumnPut<N>& c, int q, const Sym4& g, double2 kb) {
  c.put(q, cscale(kb, g.c), cscale(kb, g.d));
}

// Zeroes the positions outside the retained set in both sequences.
template <int N, int V>
__device__ __forceinline__ void zero_outside(q2* seq) {
  constexpr int K = Geo<N, V>::K, GAP = N - 2 * K - 1;
  for (int u = threadIdx.x; u < 2 * GAP; u += Geo<N, V>::THREADS) {
    const int f = u / GAP, q = K + 1 + (u - f * GAP);
    seq[f * N + q] = mkq(0, 0);
  }
}

// Both columns put in c by this CTA (each thread its rows rr = threadIdx.x +
// t THREADS, as in the loops that put them): to integers, inverse transform
// along y, into column kx of both fields of Mx.
template <int N, int V>
__device__ __forceinline__ void finish_columns(const Dev& d, const ColumnPut<N>& c, int bm, int kx, int* scratch) {
  using G = Geo<N, V>;
  using P = FxPlan<N, V>;
  q2* a = c.a;
  const int2 f = block_max2<G::THREADS>(c.f0, c.f1, scratch);
  const int e0 = exp_for<kInvBits>(f.x), e1 = exp_for<kInvBits>(f.y);
  unsigned s0 = 0, s1 = 0;
#pragma unroll
  for (int t = 0; t < (G::Kr + G::THREADS - 1) / G::THREADS; ++t) {
    const int rr = threadIdx.x + t * G::THREADS;
    if (rr >= G::Kr) break;
    const int q = ky_of_row(rr, G::K) & (N - 1);
    const q2 x = a[q], y = a[N + q];
    const q2 u = mkq(double_to_fx(__longlong_as_double(x.x), e0), double_to_fx(__longlong_as_double(x.y), e0));
    const q2 v = mkq(double_to_fx(__longlong_as_double(y.x), e1), double_to_fx(__longlong_as_double(y.y), e1));
    s0 += mag_units(u);
    s1 += mag_units(v);
    a[q] = u;
    a[N + q] = v;
  }
  zero_outside<N, V>(a);
  block_sum2_put(s0, s1, scratch + 16);
  __syncthreads();
  const int2 sum = block_sum2_get<G::THREADS>(scratch + 16);
  const int2 pre = make_int2(inv_shift<N, V>(sum.x), inv_shift<N, V>(sum.y));
  fx_inverse<N, V, G::K>(a, d.fxtw, pre);
  q2* M = d.Mx + (size_t)bm * 2 * N * G::Kc + kx;
#pragma unroll
  for (int t = 0; t < (2 * N + G::THREADS - 1) / G::THREADS; ++t) {
    const int u = threadIdx.x + t * G::THREADS;
    if (u < 2 * N) M[(size_t)u * G::Kc] = a[u];
  }
  if (threadIdx.x < 2)
    d.eX[(bm * 2 + threadIdx.x) * G::Kc + kx] = clamp_exp((threadIdx.x ? e1 + pre.y : e0 + pre.x) + P::SHIFT_INV);
}

// Column kx of both fields of the column-major Mn (M points at the column,
// eN at the member's row exponents) into a, forward transform along y.
// Returns the exponents of the two results.  `between` runs after the loads
// are issued.
template <int N, int V, typename Between>
__device__ __forceinline__ int2 forward_columns(const q2* __restrict__ M, const int* __restrict__ eN, q2* a,
                                                const int4* tw, int* scratch, Between between) {
  using G = Geo<N, V>;
  using P = FxPlan<N, V>;
  constexpr int T = G::THREADS, J = (2 * N + T - 1) / T;
  q2 v[J];
  int e[J], k0 = kZeroExp, k1 = kZeroExp;
#pragma unroll
  for (int t = 0; t < J; ++t) {
    const int u = threadIdx.x + t * T;
    if (u < 2 * N) {
      v[t] = M[u];
      e[t] = eN[u & (N - 1)];
    }
  }
  between();
#pragma unroll
  for (int t = 0; t < J; ++t) {
    const int u = threadIdx.x + t * T;
    if (u < 2 * N) {
      const int k = bits32(max(mag32(v[t].x), mag32(v[t].y))) + 32 + e[t];
      if (u < N) k0 = max(k0, k);
      else k1 = max(k1, k);
    }
  }
  const int2 k = block_max2<T>(k0, k1, scratch);
  const int e0 = k.x - P::BITS_FWD, e1 = k.y - P::BITS_FWD;
#pragma unroll
  for (int t = 0; t < J; ++t) {
    const int u = threadIdx.x + t * T;
    if (u < 2 * N) a[u] = Shift(e[t] - (u < N ? e0 : e1))(v[t]);
  }
  __syncthreads();
  fx_forward<N, V, G::K>(a, tw);
  return make_int2(clamp_exp(e0 + P::SHIFT), clamp_exp(e1 + P::SHIFT));
}

// Integers of one exponent to doubles, with the power of two folded into the
// caller's coefficients where it is an ordinary double: value = s (*this)(v).
struct FxScale {
  int e;
  bool plain;
  double s;
  __device__ __forceinline__ explicit FxScale(int e_) : e(e_), plain(e_ >= -960 && e_ <= 960) {
    s = plain ? pow2_double(e) : 1.0;
  }
  __device__ __forceinline__ double operator()(i64 v) const { return plain ? (double)v : fx_to_double(v, e); }
};

// s_hat = forward transform along y of the mixed rows in Mn (doubles here,
// from k_r2c_rows); w0 = mult s_hat into W (and Y); then, unless F_NO_NEXT,
// the inverse column transforms of u and v of stage 1.  grid (Kc, B).
template <int N, int V = 0>
__global__ void __launch_bounds__(Geo<N, V>::THREADS) k_ctrl_cols(Dev d, int flags) {
  using G = Geo<N, V>;
  extern __shared__ double2 sm[];
  double* T = reinterpret_cast<double*>(sm);
  double2* a = sm + FoldInfo<N, V>::PADDED / 2;
  const FxSmem<N> fs(a);
  const int kx = blockIdx.x, bm = blockIdx.y;
  load_fold<N, V>(T, d.fold);
  const double2* M = reinterpret_cast<const double2*>(d.Mn) + ((size_t)bm * G::Kc + kx) * 2 * N;
#pragma unroll
  for (int y = threadIdx.x; y < N; y += G::THREADS) a[y] = M[y];
  __syncthreads();
  fft_folded<N, V, -1, 1, -1, G::K>(a, T);
  ColumnPut<N> put(fs.a);
  // each retained position is read and rewritten by one thread only
  #pragma unroll
  for (int rr = threadIdx.x; rr < G::Kr; rr += G::THREADS) {
    const int ky = ky_of_row(rr, G::K);
    const size_t idx = cidx<N>(bm, rr, kx);
    const double2 w0 = cscale(a[ky & (N - 1)], d.mult[idx]);
    d.W[idx] = w0;
    d.Y[idx] = w0;
    put_stage_columns<N>(put, ky & (N - 1), d.symF[kx * G::Kr + rr], w0);
  }
  if (flags & F_NO_NEXT) return;
  finish_columns<N, V>(d, put, bm, kx, fs.scratch);
}

// Restart from the compact state in W (a checkpoint): Y = W and the inverse
// column transforms of u and v of stage 1.  grid (Kc, B).
template <int N, int V = 0>
__global__ void __launch_bounds__(Geo<N, V>::THREADS) k_state_cols(Dev d) {
  using G = Geo<N, V>;
  extern __shared__ double2 sm[];
  const FxSmem<N> fs(sm);
  const int kx = blockIdx.x, bm = blockIdx.y;
  ColumnPut<N> put(fs.a);
  #pragma unroll
  for (int rr = threadIdx.x; rr < G::Kr; rr += G::THREADS) {
    const int ky = ky_of_row(rr, G::K);
    const size_t idx = cidx<N>(bm, rr, kx);
    const double2 w = d.W[idx];
    d.Y[idx] = w;
    put_stage_columns<N>(put, ky & (N - 1), d.symF[kx * G::Kr + rr], w);
  }
  finish_columns<N, V>(d, put, bm, kx, fs.scratch);
}

// ---------------------------------------------------------------------------
// Row passes
// ---------------------------------------------------------------------------

// Rows y0, y0 + 1 of the two fields of Mx, packed for the inverse transform
// along x as field 0 + i field 1: Z(kx) = A + iB, Z(-kx) = conj(A) + i conj(B)
// for the mixed half spectra A, B (kx = 0..K); the DC bin keeps real parts
// only; the gap is zeroed.  Ends with a barrier.
struct RowLoad {
  int e;     // exponent of both rows as they stand in a
  int2 pre;  // right shifts their inverse transforms start with
};
template <int N, int V>
__device__ __forceinline__ RowLoad load_row_pair(const Dev& d, int bm, int y0, q2* a, int* scratch) {
  using G = Geo<N, V>;
  constexpr int T = G::THREADS, K = G::K, Kc = G::Kc, GAP = N - 2 * K - 1, J = (2 * Kc + T - 1) / T;
  const q2* M = d.Mx + (size_t)bm * 2 * N * Kc;
  const int* eX = d.eX + (size_t)bm * 2 * Kc;
  q2 p[J], q[J];
  int ep[J], eq[J], key = kZeroExp;
#pragma unroll
  for (int t = 0; t < J; ++t) {
    const int u = threadIdx.x + t * T;
    if (u < 2 * Kc) {
      const int rr = u / Kc, kx = u - rr * Kc;
      p[t] = M[(size_t)(y0 + rr) * Kc + kx];
      q[t] = M[((size_t)N + y0 + rr) * Kc + kx];
      ep[t] = eX[kx];
      eq[t] = eX[Kc + kx];
    }
  }
  for (int u = threadIdx.x; u < 2 * GAP; u += T) {
    const int rr = u / GAP;
    a[rr * N + K + 1 + (u - rr * GAP)] = mkq(0, 0);
  }
#pragma unroll
  for (int t = 0; t < J; ++t) {
    const int u = threadIdx.x + t * T;
    if (u < 2 * Kc) {
      key = max(key, bits32(max(mag32(p[t].x), mag32(p[t].y))) + 32 + ep[t]);
      key = max(key, bits32(max(mag32(q[t].x), mag32(q[t].y))) + 32 + eq[t]);
    }
  }
  const int e = block_max2<T>(key, key, scratch).x - (kInvBits - 1);  // sums of two below kInvBits bits
  unsigned s0 = 0, s1 = 0;
#pragma unroll
  for (int t = 0; t < J; ++t) {
    const int u = threadIdx.x + t * T;
    if (u < 2 * Kc) {
      const int rr = u / Kc, kx = u - rr * Kc;
      const q2 A = Shift(ep[t] - e)(p[t]), B = Shift(eq[t] - e)(q[t]);
      q2* seq = a + rr * N;
      const unsigned units = 2 * (mag_units(A) + mag_units(B));  // of Z(kx) and Z(-kx)
      if (rr == 0) s0 += units;
      else s1 += units;
      if (kx == 0) {
        seq[0] = mkq(A.x, B.x);
      } else {
        seq[kx] = mkq(A.x - B.y, A.y + B.x);
        seq[N - kx] = mkq(A.x + B.y, B.x - A.y);
      }
    }
  }
  block_sum2_put(s0, s1, scratch + 16);
  __syncthreads();
  const int2 sum = block_sum2_get<T>(scratch + 16);
  return {e, make_int2(inv_shift<N, V>(sum.x), inv_shift<N, V>(sum.y))};
}

// Forward transforms along x of rows y0, y0+1, sequence rr packed as
// (field 0 of row y0+rr) + i (field 1 of row y0+rr) -> twice the two fields
// of both rows (A = Z(k) + conj Z(-k), B = -i (Z(k) - conj Z(-k)); the column
// pass's symbols carry the 1/2) in the column-major Mn of the member: entry
// (kx, f, y) at (kx * 2 + f) * N + y, with the rows' exponents e0, e1.
template <int N, int V>
__device__ __forceinline__ void store_row_pair(const Dev& d, int bm, int y0, const q2* a, int e0, int e1) {
  using G = Geo<N, V>;
  q2* O = d.Mn + (size_t)bm * G::Kc * 2 * N;
#pragma unroll
  for (int t = 0; t < (2 * G::Kc + G::THREADS - 1) / G::THREADS; ++t) {
    const int u = threadIdx.x + t * G::THREADS;
    if (u < 2 * G::Kc) {
      const int rr = u & 1, kx = u >> 1;
      const q2 zk = a[rr * N + kx], zm = a[rr * N + ((N - kx) & (N - 1))];
      q2* o = O + (size_t)kx * 2 * N + y0 + rr;
      o[0] = mkq(zk.x + zm.x, zk.y - zm.y);
      o[N] = mkq(zk.y + zm.y, zm.x - zk.x);
    }
  }
  if (threadIdx.x < 2) d.eN[bm * N + y0 + threadIdx.x] = clamp_exp(threadIdx.x ? e1 : e0);
}

// Bits that a row pass brings u, v and 2a, b to, so that the products, less
// the 64 bits dropped, enter the forward transform with one bit to spare for
// the sums of store_row_pair: room for all its stages, or (MEASURE, where it
// gives the products at least two bits more) for the first one.
template <int N, int V>
struct RowBits {
  using P = FxPlan<N, V>;
  static constexpr int F = P::BITS_FWD - 1;
  static constexpr int UV0 = (64 + F) / 2;  // u v and v^2 - u^2: 2 UV - 64 <= F
  static constexpr int AB0 = 63 + F - UV0;  // sums of two products: UV + AB - 63 <= F
  static constexpr int UV1 = 61, AB1 = P::GROWTH1 <= 3 ? 61 : 60;
  static constexpr bool MEASURE = UV1 + AB1 >= UV0 + AB0 + 2;
  static constexpr int UV = MEASURE ? UV1 : UV0, AB = MEASURE ? AB1 : AB0;
};

// Row pass of stage `stage` (1..4) of step n: u, v of rows y0, y0+1; the
// stage-field store and probe gather; the products u v and v^2 - u^2 of
// each row (packed as P + i Q) and their forward transforms along x into
// Mn.  grid (N/2, B).
template <int N, int V = 0>
__global__ void __launch_bounds__(Geo<N, V>::THREADS) k_fwd_rows(Dev d, int n, int stage, int flags) {
  using G = Geo<N, V>;
  using P = FxPlan<N, V>;
  extern __shared__ double2 sm[];
  const FxSmem<N> fs(sm);
  const int bm = blockIdx.y, y0 = 2 * blockIdx.x;
  const MemberWindow mw = member_window(d, bm);
  if (n < mw.start) return;  // the member's window has not begun
  const RowLoad in = load_row_pair<N, V>(d, bm, y0, fs.a, fs.scratch);
  const int Pp = mw.P, st = N / Pp;
  const int slot = (flags & (F_OBS | F_OBS_ONLY)) ? obs_slot(d, n - mw.start) : -1;
  const size_t trow = (((size_t)bm * d.traj_steps + (n - d.seg0)) * 4 + (stage - 1)) * N + y0;
  const bool store = (flags & F_STORE) != 0;
  int ex[2];  // exponents of u, v of the two rows, once normalised
  int sh[2];
  auto prep = [&](int m0, int m1) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int m = r ? m1 : m0;
      sh[r] = m == 0 ? 0 : RowBits<N, V>::UV - 32 - bits32(m);
      ex[r] = clamp_exp(in.e + (r ? in.pre.y : in.pre.x) + P::SHIFT_INV - sh[r]);
    }
    if (store && threadIdx.x < 2) d.eT[trow + threadIdx.x] = threadIdx.x ? ex[1] : ex[0];
  };
  // (u, v) at column x of row y0 + rr: stage-field store, probe gather, and
  // the products P = u v, Q = v^2 - u^2 as P + i Q
  auto products = [&](int rr, int x, q2 uv) {
    const int y = y0 + rr;
    uv = Shift(rr ? sh[1] : sh[0])(uv);
    if (store) d.traj[(trow + rr) * N + x] = uv;
    if (slot >= 0 && (y % st) == 0 && (x % st) == 0) {
      const int p = (y / st) * Pp + x / st;
      double* o = d.obs + bm * d.obs_stride + ((size_t)slot * Pp * Pp + p) * 2;
      o[0] = fx_to_double(uv.x, rr ? ex[1] : ex[0]);
      o[1] = fx_to_double(uv.y, rr ? ex[1] : ex[0]);
    }
    return mkq(mul_hi(uv.x, uv.y), mul_hi(uv.y - uv.x, uv.y + uv.x));
  };
  if (flags & F_OBS_ONLY) {  // the final state: probes only
    fx_inverse<N, V, G::K>(fs.a, d.fxtw, in.pre);
    sh[0] = sh[1] = 0;
    ex[0] = clamp_exp(in.e + in.pre.x + P::SHIFT_INV);
    ex[1] = clamp_exp(in.e + in.pre.y + P::SHIFT_INV);
    for (int u = threadIdx.x; u < 2 * N; u += G::THREADS) products(u / N, u & (N - 1), fs.a[u]);
    return;
  }
  const int2 r = fx_turn<N, V, G::K, RowBits<N, V>::MEASURE>(fs.a, d.fxtw, in.pre, fs.scratch + 32, prep, products);
  store_row_pair<N, V>(d, bm, y0, fs.a, 2 * ex[0] + 64 + P::SHIFT + r.x, 2 * ex[1] + 64 + P::SHIFT + r.y);
}

// ---------------------------------------------------------------------------
// Forward RK stage: column pass
// ---------------------------------------------------------------------------

// Column pass of stage `stage`: the advection term
//   n_hat = (ky^2 - kx^2) DFT(u v) - kx ky DFT(v^2 - u^2),
// k_j = -n_hat - nu k^2 y_j + f_hat, the RK4 update, and the inverse column
// transforms of u and v of the next stage state.  Acc holds k1 + 2 k2 +
// 2 k3 (+ k4).  grid (Kc, B).
template <int N, int V = 0>
__global__ void __launch_bounds__(Geo<N, V>::THREADS) k_fwd_cols(Dev d, int n, int stage, int flags) {
  using G = Geo<N, V>;
  extern __shared__ double2 sm[];
  const FxSmem<N> fs(sm);
  q2* a = fs.a;
  const int kx = blockIdx.x, bm = blockIdx.y;
  const MemberWindow mw = member_window(d, bm);
  if (n < mw.start) return;
  // the epilogue's inputs for this thread's modes; where registers allow
  // (G::PREFETCH), loaded early so that their latency hides behind the
  // column transforms
  constexpr int MT = (G::Kr + G::THREADS - 1) / G::THREADS;
  double2 yv[MT], wv[MT], accv[MT];
  Sym4 f[MT];
  double nk2[MT];
  auto load_inputs = [&](int t) {
    const int rr = threadIdx.x + t * G::THREADS;
    if (rr < G::Kr) {
      const size_t idx = cidx<N>(bm, rr, kx);
      yv[t] = d.Y[idx];
      wv[t] = d.W[idx];
      accv[t] = stage > 1 ? d.Acc[idx] : make_double2(0.0, 0.0);
      f[t] = d.symF[kx * G::Kr + rr];
      nk2[t] = mw.nu * d.k2[kx * G::Kr + rr];
    }
  };
  const int2 e = forward_columns<N, V>(d.Mn + ((size_t)bm * G::Kc + kx) * 2 * N, d.eN + bm * N, a, d.fxtw, fs.scratch,
                                       [&] {
                                         if constexpr (G::PREFETCH) {
#pragma unroll
                                           for (int t = 0; t < MT; ++t) load_inputs(t);
                                         }
                                       });
  const FxScale s0(e.x), s1(e.y);
  const double dt = d.dt;
  const double fval = -d.amp * d.nf * (double)N * N / 2.0;
  ColumnPut<N> put(a);
  // each retained position is read and rewritten (both sequences) by one
  // thread only
#pragma unroll
  for (int t = 0; t < MT; ++t) {
    const int rr = threadIdx.x + t * G::THREADS;
    if (rr >= G::Kr) break;
    if constexpr (!G::PREFETCH) load_inputs(t);
    const int ky = ky_of_row(rr, G::K);
    const int qi = ky & (N - 1);
    const size_t idx = cidx<N>(bm, rr, kx);
    const q2 pq = a[qi], qq = a[N + qi];
    const double2 ph = make_double2(s0(pq.x), s0(pq.y)), qh = make_double2(s1(qq.x), s1(qq.y));
    const double cp = f[t].c * s0.s, cq = f[t].d * s1.s;
    // F = -(cp P + cq Q) - nu k^2 y
    double2 F = make_double2(-fma(cp, ph.x, fma(cq, qh.x, nk2[t] * yv[t].x)),
                             -fma(cp, ph.y, fma(cq, qh.y, nk2[t] * yv[t].y)));
    if (mw.forced && kx == 0 && (ky == d.nf || ky == -d.nf)) F.x += fval;
    const double2 w = wv[t], acc = accv[t];
    double2 ynext;
    if (stage == 1) {
      d.Acc[idx] = F;
      ynext = make_double2(fma(d.dt2, F.x, w.x), fma(d.dt2, F.y, w.y));
    } else if (stage == 2) {
      d.Acc[idx] = make_double2(fma(2.0, F.x, acc.x), fma(2.0, F.y, acc.y));
      ynext = make_double2(fma(d.dt2, F.x, w.x), fma(d.dt2, F.y, w.y));
    } else if (stage == 3) {
      d.Acc[idx] = make_double2(fma(2.0, F.x, acc.x), fma(2.0, F.y, acc.y));
      ynext = make_double2(fma(dt, F.x, w.x), fma(dt, F.y, w.y));
    } else {
      ynext = make_double2(fma(d.dt6, acc.x + F.x, w.x), fma(d.dt6, acc.y + F.y, w.y));
      d.W[idx] = ynext;
    }
    d.Y[idx] = ynext;
    put_stage_columns<N>(put, qi, f[t], ynext);
  }
  if (flags & F_NO_NEXT) return;
  finish_columns<N, V>(d, put, bm, kx, fs.scratch + 16);
}

// r = model observations - data and J = 1/2 sum r^2 per member, in a fixed
// order (deterministic).  grid B, block 256.  Defined in residual.cu.
__global__ void k_residual(Dev d);

// Regularisation of Eq. (4): J[b] += lambda/2 sum_grid w0^2, from the compact
// initial spectrum w0 (sum_grid w^2 = 1/N^2 sum over the full spectrum).
// grid B, block 256.  Defined in residual.cu.
__global__ void k_sobolev_cost(double* J, const double2* w0, double lambda, int N, int Kr, int Kc);

// Shell energies of the adjoint velocity, per member and of the ensemble
// mean.  Defined in residual.cu.
__global__ void k_shell_member(const double2* lam, const int* off, const int* mode, const double* wgt, int nmodes,
                               double* out, int nshell);
__global__ void k_shell_mean(const double2* lam, int B, const int* off, const int* mode, const double* wgt, int nmodes,
                             double* out);

// LamBar[b] += lambda w0[b] on the compact set.  Defined in residual.cu.
__global__ void k_sobolev_grad(double2* lam, const double2* w0, double lambda, int count);

// ---------------------------------------------------------------------------
// Adjoint
// ---------------------------------------------------------------------------
//
// The tangent of the advection term at (u, v) is
//   dn = (d_xx - d_yy)(u dv + v du) + d_xy (2 v dv - 2 u du),
// so its transpose applied to kbar is, with a = IDFT(d_xy kbar) and
// b = IDFT((d_xx - d_yy) kbar) on the grid,
//   rho_u = v b - 2 u a,   rho_v = u b + 2 v a,
//   J^T kbar = -P[(-i ky/k^2) DFT(rho_u) + (i kx/k^2) DFT(rho_v)] - nu k^2 kbar,
// the transposes of du = IDFT(i ky/k^2 dw), dv = IDFT(-i kx/k^2 dw).

// Separable DFT of the residual at observation slot `slot` on the probe
// lattice: for each lattice row, T(kx) = sum_q r[row][q] W_P^{kx q}; the
// column pass then sums over rows with W_P^{ky row}.  Fills Tu, Tv [P].
__device__ __forceinline__ void probe_row_sums(const Dev& d, int bm, int P, int slot, int kx, double2* Tu,
                                               double2* Tv) {
  const double* r = d.res + bm * d.obs_stride + (size_t)slot * P * P * 2;
  const int tws = 64 / P;
  for (int row = threadIdx.x; row < P; row += blockDim.x) {
    double2 su = make_double2(0.0, 0.0), sv = make_double2(0.0, 0.0);
    for (int qq = 0; qq < P; ++qq) {
      const double2 w = d.twP[((kx * qq) % P) * tws];
      const double ru = r[(row * P + qq) * 2], rv = r[(row * P + qq) * 2 + 1];
      su = make_double2(fma(ru, w.x, su.x), fma(ru, w.y, su.y));
      sv = make_double2(fma(rv, w.x, sv.x), fma(rv, w.y, sv.y));
    }
    Tu[row] = su;
    Tv[row] = sv;
  }
}

// H^T r at (kx, ky): (-i ky/k^2) R_u + (i kx/k^2) R_v with R the DFT of the
// probe residual scattered onto the grid.
__device__ __forceinline__ double2 probe_source(const Dev& d, int P, int kx, int ky, const double2* Tu,
                                                const double2* Tv) {
  double2 Ru = make_double2(0.0, 0.0), Rv = make_double2(0.0, 0.0);
  const int kyp = ((ky % P) + P) % P;
  const int tws = 64 / P;
  for (int row = 0; row < P; ++row) {
    const double2 w = d.twP[((kyp * row) % P) * tws];
    Ru = cadd(Ru, cmul(Tu[row], w));
    Rv = cadd(Rv, cmul(Tv[row], w));
  }
  const double k2 = (double)(kx * kx + ky * ky);
  const double ik2 = k2 > 0.0 ? 1.0 / k2 : 0.0;
  const double a = ky * ik2, c = kx * ik2;
  // (-i a) Ru + (i c) Rv
  return make_double2(a * Ru.y - c * Rv.y, -a * Ru.x + c * Rv.x);
}

// Start of the adjoint sweep: LamBar = (terminal field in LamBar, with
// INIT_LAMBAR) + (H^T r at the last step, with INIT_SRC), KB = dt/6 LamBar;
// with INIT_RESUME, KB as it stands (after a checkpoint recompute).  Then
// the inverse column transforms of the adjoint fields a, b of KB into Mx.
// grid (Kc, B).
template <int N, int V = 0>
__global__ void __launch_bounds__(Geo<N, V>::THREADS) k_adj_init(Dev d, int mode) {
  using G = Geo<N, V>;
  extern __shared__ double2 sm[];
  const FxSmem<N> fs(sm);
  double2 *Tu = fs.Tu, *Tv = fs.Tv;
  const int kx = blockIdx.x, bm = blockIdx.y;
  const MemberWindow mw = member_window(d, bm);
  // an idle member starts (and stays) at lambda = 0
  if (mw.start > d.nsteps) mode = 0;
  const bool resume = (mode & INIT_RESUME) != 0;
  const int slot = (!resume && (mode & INIT_SRC)) ? obs_slot(d, d.nsteps - mw.start) : -1;
  if (slot >= 0) probe_row_sums(d, bm, mw.P, slot, kx, Tu, Tv);
  __syncthreads();
  ColumnPut<N> put(fs.a);
  #pragma unroll
  for (int rr = threadIdx.x; rr < G::Kr; rr += G::THREADS) {
    const int ky = ky_of_row(rr, G::K);
    const size_t idx = cidx<N>(bm, rr, kx);
    double2 kb;
    if (resume) {
      kb = d.KB[idx];
    } else {
      double2 lam = (mode & INIT_LAMBAR) ? d.LamBar[idx] : make_double2(0.0, 0.0);
      if (slot >= 0) lam = cadd(lam, probe_source(d, mw.P, kx, ky, Tu, Tv));
      d.LamBar[idx] = lam;
      kb = cscale(lam, d.dt6);
      d.KB[idx] = kb;
    }
    put_adjoint_columns<N>(put, ky & (N - 1), d.symA[kx * G::Kr + rr], kb);
  }
  finish_columns<N, V>(d, put, bm, kx, fs.scratch);
}

// Adjoint row pass of stage `stage` of step n: 2a, b of rows y0, y0+1
// (inverse transforms along x), rho_u and rho_v with the stored u, v (each
// row packed as rho_u + i rho_v), and their forward transforms along x into
// Mn (twice, as in the forward row pass).  grid (N/2, B).
template <int N, int V = 0>
__global__ void __launch_bounds__(Geo<N, V>::THREADS) k_adj_rows(Dev d, int n, int stage) {
  using P = FxPlan<N, V>;
  using G = Geo<N, V>;
  extern __shared__ double2 sm[];
  const FxSmem<N> fs(sm);
  const int bm = blockIdx.y, y0 = 2 * blockIdx.x;
  if (d.ragged && n < d.mstart[bm]) return;
  const RowLoad in = load_row_pair<N, V>(d, bm, y0, fs.a, fs.scratch);
  const size_t trow = (((size_t)bm * d.traj_steps + (n - d.seg0)) * 4 + (stage - 1)) * N + y0;
  int sh[2], ex[2];
  auto prep = [&](int m0, int m1) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int m = r ? m1 : m0;
      sh[r] = m == 0 ? 0 : RowBits<N, V>::AB - 32 - bits32(m);
      ex[r] = clamp_exp(in.e + (r ? in.pre.y : in.pre.x) + P::SHIFT_INV - sh[r]);
    }
  };
  // (2a, b) at column x of row y0 + rr -> rho_u + i rho_v with the stored
  // u, v: rho_u = v b - u 2a, rho_v = u b + v 2a
  auto rho = [&](int rr, int x, q2 ab) {
    const q2 uv = d.traj[(trow + rr) * N + x];
    ab = Shift(rr ? sh[1] : sh[0])(ab);
    const int uh = hi_word(uv.x), ul = lo_word(uv.x), vh = hi_word(uv.y), vl = lo_word(uv.y);
    const int ah = hi_word(ab.x), al = lo_word(ab.x), bh = hi_word(ab.y), bl = lo_word(ab.y);
    return mkq(mul_hi2<-1>(vh, vl, bh, bl, uh, ul, ah, al), mul_hi2<+1>(uh, ul, bh, bl, vh, vl, ah, al));
  };
  const int2 r = fx_turn<N, V, G::K, RowBits<N, V>::MEASURE>(fs.a, d.fxtw, in.pre, fs.scratch + 32, prep, rho);
  store_row_pair<N, V>(d, bm, y0, fs.a, clamp_exp(ex[0] + d.eT[trow]) + 64 + P::SHIFT + r.x,
                       clamp_exp(ex[1] + d.eT[trow + 1]) + 64 + P::SHIFT + r.y);
}

// Adjoint column pass of stage `stage` of step n:
//   ybar_j = -P[(-i ky/k^2) DFT(rho_u) + (i kx/k^2) DFT(rho_v)] - nu k^2 kbar_j,
// the transposed RK4 combination, the observation source at step n (on
// stage 1), and the inverse column transforms of a, b of the next kbar.
// grid (Kc, B).
template <int N, int V = 0>
__global__ void __launch_bounds__(Geo<N, V>::THREADS) k_adj_cols(Dev d, int n, int stage, int flags) {
  using G = Geo<N, V>;
  extern __shared__ double2 sm[];
  const FxSmem<N> fs(sm);
  q2* a = fs.a;
  double2 *Tu = fs.Tu, *Tv = fs.Tv;
  const int kx = blockIdx.x, bm = blockIdx.y;
  const MemberWindow mw = member_window(d, bm);
  if (n < mw.start) return;
  // the epilogue's inputs for this thread's modes (before the column
  // transforms where registers allow, as in k_fwd_cols)
  constexpr int MT = (G::Kr + G::THREADS - 1) / G::THREADS;
  double2 kbv[MT], lbv[MT], sumv[MT];
  Sym4 g[MT];
  double nk2[MT];
  auto load_inputs = [&](int t) {
    const int rr = threadIdx.x + t * G::THREADS;
    if (rr < G::Kr) {
      const size_t idx = cidx<N>(bm, rr, kx);
      kbv[t] = d.KB[idx];
      lbv[t] = d.LamBar[idx];
      sumv[t] = stage < 4 ? d.Sum[idx] : make_double2(0.0, 0.0);
      g[t] = d.symA[kx * G::Kr + rr];
      nk2[t] = mw.nu * d.k2[kx * G::Kr + rr];
    }
  };
  const int slot = (flags & F_SRC) ? obs_slot(d, n - mw.start) : -1;
  const int2 e = forward_columns<N, V>(d.Mn + ((size_t)bm * G::Kc + kx) * 2 * N, d.eN + bm * N, a, d.fxtw, fs.scratch,
                                       [&] {
                                         if constexpr (G::PREFETCH) {
#pragma unroll
                                           for (int t = 0; t < MT; ++t) load_inputs(t);
                                         }
                                         if (slot >= 0) probe_row_sums(d, bm, mw.P, slot, kx, Tu, Tv);
                                       });
  const FxScale s0(e.x), s1(e.y);
  const double dt = d.dt;
  ColumnPut<N> put(a);
  // each retained position is read and rewritten (both sequences) by one
  // thread only
#pragma unroll
  for (int t = 0; t < MT; ++t) {
    const int rr = threadIdx.x + t * G::THREADS;
    if (rr >= G::Kr) break;
    if constexpr (!G::PREFETCH) load_inputs(t);
    const int ky = ky_of_row(rr, G::K);
    const int qi = ky & (N - 1);
    const size_t idx = cidx<N>(bm, rr, kx);
    const q2 qu = a[qi], qv = a[N + qi];
    const double2 Ru = make_double2(s0(qu.x), s0(qu.y)), Rv = make_double2(s1(qv.x), s1(qv.y));
    const double a1 = g[t].a * s0.s, c1 = g[t].b * s1.s;
    // t = (-i ky/k^2) Ru + (i kx/k^2) Rv (the 1/2 of the row unpack in a1, c1)
    const double2 tt = make_double2(fma(a1, Ru.y, -c1 * Rv.y), fma(-a1, Ru.x, c1 * Rv.x));
    const double2 kb = kbv[t], lb = lbv[t];
    double2 yb;
    yb.x = -fma(nk2[t], kb.x, tt.x);
    yb.y = -fma(nk2[t], kb.y, tt.y);
    double2 nk;
    if (stage == 4) {
      d.Sum[idx] = yb;
      nk = make_double2(fma(d.dt3, lb.x, dt * yb.x), fma(d.dt3, lb.y, dt * yb.y));
    } else if (stage == 3) {
      d.Sum[idx] = cadd(sumv[t], yb);
      nk = make_double2(fma(d.dt3, lb.x, d.dt2 * yb.x), fma(d.dt3, lb.y, d.dt2 * yb.y));
    } else if (stage == 2) {
      d.Sum[idx] = cadd(sumv[t], yb);
      nk = make_double2(fma(d.dt6, lb.x, d.dt2 * yb.x), fma(d.dt6, lb.y, d.dt2 * yb.y));
    } else {
      const double2 sum = cadd(sumv[t], yb);
      double2 lam = cadd(lb, sum);
      if (slot >= 0) lam = cadd(lam, probe_source(d, mw.P, kx, ky, Tu, Tv));
      d.LamBar[idx] = lam;
      nk = cscale(lam, d.dt6);
    }
    d.KB[idx] = nk;
    put_adjoint_columns<N>(put, qi, g[t], nk);
  }
  if (stage == 1 && n == mw.start) return;  // the member's first step: lambda_0 stays in LamBar
  finish_columns<N, V>(d, put, bm, kx, fs.scratch + 16);
}

// Control multipliers m(k) = |k| W(k)^{1/2} on the retained set (0 at k = 0),
// per member.  grid (ceil(Kr*Kc/256), B), block 256.
template <int N, int V = 0>
__global__ void k_make_mult(double* __restrict__ mult, const int* __restrict__ kind, const double* __restrict__ param,
                            const double* __restrict__ table, const double* __restrict__ nu) {
  using G = Geo<N, V>;
  const int bm = blockIdx.y;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < G::Kr * G::Kc; i += gridDim.x * blockDim.x) {
    const int kx = i / G::Kr, r = i - kx * G::Kr;
    const int ky = ky_of_row(r, G::K);
    const double k2 = (double)(kx * kx + ky * ky);
    const double k = sqrt(k2);
    double W;
    const double a = param[bm];
    switch (kind[bm]) {
      case 0: W = 1.0; break;
      case 1: W = exp(-a * k); break;
      case 2: W = pow(k, -2.0 * a); break;
      case 3: W = exp(-nu[bm] * a * k2); break;
      default: W = table[((size_t)bm * N + (ky & (N - 1))) * G::NH + kx]; break;
    }
    mult[(size_t)bm * G::Kr * G::Kc + i] = (kx == 0 && ky == 0) ? 0.0 : k * sqrt(W);
  }
}

}  // namespace da
