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
// spectra, observations, controls and gradients are doubles.
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
// in registers) and a COLUMN
// pass (forward transforms along y of the two products, the advection term,
// RK epilogue with viscosity, forcing and the stage update, then the
// inverse column transforms of the next stage's u and v).  The adjoint
// mirrors this with the transposed operators.  Every transform is an integer
// FFT from fx.cuh.  The 1/N^2 of the inverse 2D transform is
// applied once, to the spectral coefficients before the column transform.
// Every inverse transform here reads a sequence that is zero in the gap
// K < q < N - K, and every forward transform is read back only on the band
// q <= K, q >= N - K: the transforms are band-limited and skip the inputs and
// outputs that lie in the gap for every butterfly of a stage.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "fx.cuh"

namespace da {

enum : int {
  F_STORE = 1,     // forward row pass: write stage fields
  F_OBS = 2,       // forward row pass: gather probes into the observation slot
  F_OBS_ONLY = 4,  // forward row pass: only gather probes (final state)
  F_SRC = 8       // adjoint column pass: add the observation source at this step
};

// Whole windows in one kernel (window.cuh).
enum : int {
  W_OBS = 1,    // forward: gather probes at the observation steps
  W_STORE = 2,  // forward: write stage fields of the steps from seg0 on
  W_FINAL = 4   // forward: gather the probes of the state after the last step
};

// Start of the adjoint sweep (k_adj_init): add the observation source of
// the last step, and/or start from the terminal field already in LamBar; or
// resume from the adjoint stage value in KB after a checkpoint recompute.
enum : int { INIT_SRC = 1, INIT_LAMBAR = 2, INIT_RESUME = 4 };

// Multipliers of the generic spectral-to-mixed column pass.
enum : int { M_ONE = 0, M_CTRL = 1, M_FILTERED = 2, M_INV_CTRL = 3 };

// Per-mode constants of the column passes, column-major [Kc][Kr] (entry
// kx * Kr + r), computed once (k_make_symbols): pairs of real symbols as integers
// of one exponent (fx_pair), since an FP64 product costs a warp 64 clocks of
// its SM's quarter and the integer one a fifth of that:
//   fwd: put = su = ky/k^2/N^2, sv = kx/k^2/N^2 (u, v columns of a state
//        value); get = cp = (ky^2 - kx^2)/2, cq = -kx ky/2 (advection symbols;
//        the 1/2 is the one the row pass leaves out when it unpacks two real
//        rows);
//   adj: put = ca = -2 kx ky/N^2, cb = (ky^2 - kx^2)/N^2 (adjoint-field
//        columns; ca carries the 2 of rho_u, rho_v); get = a1 = ky/k^2/2, c1 =
//        kx/k^2/2 (transposed velocity symbols, same 1/2).
struct __align__(16) ModeSym {
  FxPair get, put;
  int get_e, put_e, pad0, pad1;
};

// Everything a kernel needs, passed by value.
struct Dev {
  int B, nsteps, every, include_t0, px, nt;  // nsteps: the evaluation's window (global steps)
  int b0;                                    // first member of an RK stage pass (else 0), which works on B
  int early;                                 // launchers: column passes of an undivided batch may load early
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
  const int4* fxtw;                          // integer twiddles of FxPlan<N> (fx.cuh)
  const double2* twP;                        // W_64^t, t < 64 (W_P^t = W_64^{t 64/P})
  const ModeSym* symF;                       // [Kc][Kr] forward
  const ModeSym* symA;                       // [Kc][Kr] adjoint
  const double* k2;                          // [Kc][Kr] k^2
  const double* nuk2;                        // [Kc][Kr] nu k^2, the context's nu
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
  static constexpr int PMAX = 64;
  static constexpr size_t SMEM = sizeof(double2) * 2 * N;  // static_ctrl.cu: plain table and one sequence
  // passes that run the integer transforms: the buffers of two sequences,
  // scratch of the reductions (Place), and probe sums (adjoint column passes)
  static constexpr int SCRATCH = ((3 * 2 + 2 * 4) * FxPlan<N, V>::WARPS + 3) / 4 * 4;
  static constexpr size_t SMEM_FX = sizeof(q2) * (2 * FxPlan<N, V>::SEQ) + sizeof(int) * SCRATCH;
  static constexpr size_t SMEM_FXP = SMEM_FX + sizeof(double2) * 2 * PMAX;
  // Column passes load their epilogue inputs before the transforms (EARLY:
  // about 60 more registers a thread) where a warp's own latency counts, and
  // after them, at 768 threads an SM or more, where other warps hide it.  us a
  // stage pass by captured graphs, early / late: 256^2 1 member 4.99 / 5.13, 3
  // members 7.01 / 7.22, 16 members 17.0 / 16.0; 512^2 1 member 10.1 / 10.6, 2
  // members 16.0 / 14.0, 4 members in parts 20.8 / 19.0; 1024^2 1 member 34.3 / 29.2;
  // 128^2 on 64 threads 8 members 6.06 / 6.19, on 128 threads 4 members 5.28 / 4.91.
  // So: early where a whole, undivided batch is at most 256 threads an SM
  // (Columns::early); on 64 threads and fewer up to 128^2 always, on 128 never.
  // 768 threads an SM leave 80 registers, and the late kernels spill (ptxas, bytes
  // stored a thread, without / with the observation source): forward 256^2 32 to
  // 76, 512^2 92 to 332, 1024^2 88 to 148; adjoint 256^2 0 to 80 / 84 to 136,
  // 512^2 60 to 272 / 136 to 656, 1024^2 64 to 144 / 144 to 664, 128^2 on 128
  // threads 0 / 52.  Bounds between 512 and 768 have not been measured.
  static constexpr int EARLY_CTAS = N > 128 ? 152 * 256 / THREADS : THREADS < 128 ? 1 << 30 : 0;
  static constexpr int COL_CTAS = 768 / THREADS;
  // Row passes: registers for 768 threads an SM on plans of up to 128 threads;
  // for 512 on radix-16 plans, whose rows took up to 178 registers and left
  // room for one CTA of 256 threads (1024^2 plan 0: 35.9 -> 33.1 us a pass, with
  // adj_rows spilling 188 to 260 bytes a thread; for 768 38.5); free on 1024^2
  // plan 2 (28.9, for 1 CTA or 512 29.2).  256^2: 1 member 5.39 -> 5.15, 7
  // members 10.0 -> 9.8, 16 members 15.7 -> 16.0.
  static constexpr int ROW_CTAS = N <= 128                        ? 1
                                  : THREADS <= 128                ? 768 / THREADS
                                  : FirstRadix<typename Plan<N, V>::two>::value == 16 ? 512 / THREADS
                                                                  : 0;
};

__device__ __forceinline__ int ky_of_row(int r, int K) { return r <= K ? r : r - (2 * K + 1); }

// Index of mode (row r, column kx) of member bm in a compact array.
template <int N>
__host__ __device__ __forceinline__ size_t cidx(int bm, int r, int kx) {
  return ((size_t)bm * Geo<N>::Kc + kx) * Geo<N>::Kr + r;
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
// Column passes: parts, and the inverse column transforms of a stage state
// ---------------------------------------------------------------------------

// A thread's place in a column pass: sequence f of its column, thread t of
// the sequence and pt of the column's PT threads; the buffer of its sequence
// (the other's lies OTHER away); scratch of
// the sequence's reductions (three of WARPS ints) and of the column's (two of
// PAIR ints).  In a row pass the two sequences are rows.
template <typename P_>
struct Place {
  using P = P_;
  static constexpr int PT = 2 * P::TPS;
  static constexpr int OTHER = P::SEQ;
  static constexpr int PAIR = PT > 32 ? 2 * (PT / 32) : 0;
  static constexpr int SCRATCH = 2 * 3 * P::WARPS + 2 * PAIR;  // ints of the pair
  int t, f, pt;
  q2* src;
  int *scratch, *pscratch;
  // pair: index of the pair of sequences in the CTA; thread: index in the pair
  __device__ __forceinline__ Place(q2* bufs, int* ints, int pair, int thread) : pt(thread) {
    f = thread / P::TPS;
    t = thread - f * P::TPS;
    src = bufs + (pair * 2 + f) * OTHER;
    int* s = ints + pair * SCRATCH;
    scratch = s + f * 3 * P::WARPS;
    pscratch = s + 2 * 3 * P::WARPS;
  }
  __device__ __forceinline__ q2* first(q2* p) const { return f ? p - OTHER : p; }
  // scratch of the pair's sequence g
  __device__ __forceinline__ int* seq_scratch(int g) const { return scratch + (g - f) * 3 * P::WARPS; }
};

// Barrier of a pair: its warp, or the CTA.
template <typename P>
__device__ __forceinline__ void pair_sync() {
  if constexpr (Place<P>::PT <= 32) __syncwarp();
  else __syncthreads();
}

// Two reductions over a pair at once.  scratch: PAIR ints, not in use since
// the barrier before last.  Ends with the pair's barrier.
template <typename P, bool SUM>
__device__ __forceinline__ int2 pair_reduce2(int a, int b, int pt, int* scratch) {
  constexpr int PT = Place<P>::PT;
  const unsigned mask = seq_mask<(PT < 32 ? PT : 32)>(PT < 32 ? pt : 0);
  if constexpr (SUM) {
    a = (int)__reduce_add_sync(mask, (unsigned)a);
    b = (int)__reduce_add_sync(mask, (unsigned)b);
  } else {
    a = __reduce_max_sync(mask, a);
    b = __reduce_max_sync(mask, b);
  }
  if constexpr (PT > 32) {
    if ((pt & 31) == 0) {
      scratch[(pt >> 5) * 2] = a;
      scratch[(pt >> 5) * 2 + 1] = b;
    }
    pair_sync<P>();
    a = scratch[0];
    b = scratch[1];
#pragma unroll
    for (int w = 1; w < PT / 32; ++w) {
      a = SUM ? a + scratch[2 * w] : max(a, scratch[2 * w]);
      b = SUM ? b + scratch[2 * w + 1] : max(b, scratch[2 * w + 1]);
    }
  } else {
    pair_sync<P>();
  }
  return make_int2(a, b);
}

// A column under construction: the integers a thread puts at its retained rows
// rr = pt + j PT of the two fields, each mode at its own exponent, and the
// largest of those.
template <typename P>
struct ColumnPut {
  static constexpr int PT = Place<P>::PT;
  static constexpr int MT = (Geo<P::N>::Kr + PT - 1) / PT;
  q2 v0[MT], v1[MT];
  int e[MT];
  int top = 2 * kZeroExp;
  __device__ __forceinline__ void zero(int j) {
    v0[j] = v1[j] = mkq(0, 0);
    e[j] = 2 * kZeroExp;
  }
  // the pair c times the value y: (a y.x, a y.y), (b y.x, b y.y), of at most
  // 60 bits
  __device__ __forceinline__ void times(int j, const FxPair& c, int ce, double2 y) {
    const int em = exp_for<62>(max(exp_field(y.x), exp_field(y.y)));
    const Words yx(double_to_fx(y.x, em)), yy(double_to_fx(y.y, em)), a(c.ah, c.al), b(c.bh, c.bl);
    v0[j] = mkq(mul_hi(yx, a), mul_hi(yy, a));
    v1[j] = mkq(mul_hi(yx, b), mul_hi(yy, b));
    e[j] = em + 64 + ce;
    top = max(top, e[j]);
  }
};

// The two column values u = i ky/k^2 y, v = -i kx/k^2 y of a state value y
// (scaled by 1/N^2) as entry j.
template <typename P>
__device__ __forceinline__ void put_stage_columns(ColumnPut<P>& c, int j, const ModeSym& s, double2 y) {
  c.times(j, s.put, s.put_e, y);
  c.v0[j] = mkq(-c.v0[j].y, c.v0[j].x);  // i a y
  c.v1[j] = mkq(c.v1[j].y, -c.v1[j].x);  // -i b y
}

// The two column values of the adjoint fields of an adjoint stage value kb:
// 2a = 2 d_xy kb = -2 kx ky kb and b = (d_xx - d_yy) kb = (ky^2 - kx^2) kb,
// scaled by 1/N^2.
template <typename P>
__device__ __forceinline__ void put_adjoint_columns(ColumnPut<P>& c, int j, const ModeSym& s, double2 kb) {
  c.times(j, s.put, s.put_e, kb);
}

// Both columns put in c: at one exponent into the pair's src buffers (free to
// write after a barrier), inverse transform along y; store(y, value) gets this
// thread's results of its own sequence.  Returns the sequence's exponent.
template <typename P, typename Store>
__device__ __forceinline__ int finish_columns(const ColumnPut<P>& c, Place<P>& x, const int4* tw, Store store) {
  using G = Geo<P::N>;
  constexpr int N = P::N, PT = Place<P>::PT, GAP = N - 2 * G::K - 1;
  const int e0 = pair_reduce2<P, false>(c.top, c.top, x.pt, x.pscratch).x;
  q2 *a0 = x.first(x.src), *a1 = a0 + x.OTHER;
  unsigned s0 = 0, s1 = 0;
#pragma unroll
  for (int j = 0; j < c.MT; ++j) {
    const int rr = x.pt + j * PT;
    if (rr >= G::Kr) break;
    const int q = pad(ky_of_row(rr, G::K) & (N - 1));
    const ShiftRight down(e0 - c.e[j]);
    const q2 u = down(c.v0[j]), v = down(c.v1[j]);
    s0 += mag_units(u, mkq(0, 0));
    s1 += mag_units(v, mkq(0, 0));
    a0[q] = u;
    a1[q] = v;
  }
  for (int u = x.t; u < GAP; u += P::TPS) x.src[pad(G::K + 1 + u)] = mkq(0, 0);
  const int2 sum = pair_reduce2<P, true>(s0, s1, x.pt, x.pscratch + x.PAIR);
  const int pre = inv_shift<P, 60>(x.f ? sum.y : sum.x);
  constexpr int R = LastRadix<typename P::inv>::value;
  using B = Bfly<P, R>;
  q2 out[B::POINTS];
  fx_inverse<P, G::K>(x.src, tw, x.t, x.f, pre, out);
  if (B::active(x.t)) {
#pragma unroll
    for (int jb = 0; jb < B::J; ++jb)
#pragma unroll
      for (int m = 0; m < R; ++m) store(x.t + jb * P::TPS + m * B::NB, out[jb * R + m]);
  }
  return clamp_exp(e0 + pre + P::SHIFT_INV);
}

// finish_columns into column kx of both fields of Mx.
template <typename P>
__device__ __forceinline__ void finish_to_mixed(const Dev& d, const ColumnPut<P>& c, Place<P>& x, int bm, int kx) {
  constexpr int N = P::N, Kc = Geo<N>::Kc;
  q2* M = d.Mx + ((size_t)bm * 2 + x.f) * N * Kc + kx;
  const int e = finish_columns<P>(c, x, d.fxtw, [&](int y, q2 z) { M[(size_t)y * Kc] = z; });
  if (x.t == 0) d.eX[(bm * 2 + x.f) * Kc + kx] = e;
}

// Forward transform along y of a sequence of the pair (M: its N values; eN:
// the exponents of the N rows), left in the src buffers with one exponent for
// both sequences (COMMON; else one each), which is returned, and one bit to
// spare; synchronised over the pair.  `between` runs after the loads are
// issued.
template <typename P, bool COMMON = true, typename Between>
__device__ __forceinline__ int forward_columns(const q2* __restrict__ M, const int* __restrict__ eN, Place<P>& x,
                                               const int4* __restrict__ tw, Between between) {
  using G = Geo<P::N>;
  constexpr int N = P::N, R = FirstRadix<typename P::fwd>::value;
  // the first stage only must leave room where that gives a bit more
  constexpr bool MEASURE = P::GROWTH >= P::GROWTH1 + 1;
  constexpr int BITS = MEASURE ? 62 - P::GROWTH1 : P::BITS_FWD - 1;
  using B = Bfly<P, R>;
  q2 v[B::POINTS];
  int e[B::POINTS], e0 = 2 * kZeroExp, big = 0;
  if (B::active(x.t)) {
#pragma unroll
    for (int j = 0; j < B::POINTS; ++j) {
      const int y = x.t + (j / R) * P::TPS + (j % R) * B::NB;
      v[j] = M[y];
      e[j] = eN[y];
    }
  }
  between();
  // to the largest row exponent (the same for both sequences), then left
  // until the largest component of either has BITS bits
  if (B::active(x.t)) {
#pragma unroll
    for (int j = 0; j < B::POINTS; ++j) e0 = max(e0, e[j]);
  }
  e0 = seq_max_put<P::TPS>(e0, x.t, x.scratch);
  if constexpr (P::TPS > 32) seq_sync<P::TPS>(x.f);
  e0 = seq_max_get<P::TPS>(e0, x.scratch);
  if (B::active(x.t)) {
#pragma unroll
    for (int j = 0; j < B::POINTS; ++j) {
      v[j] = ShiftRight(e0 - e[j])(v[j]);
      big = max_mag(big, v[j]);
    }
  }
  if constexpr (COMMON) {
    big = pair_reduce2<P, false>(big, big, x.pt, x.pscratch).x;
  } else {
    big = seq_max_put<P::TPS>(big, x.t, x.scratch + 2 * P::WARPS);
    if constexpr (P::TPS > 32) seq_sync<P::TPS>(x.f);
    big = seq_max_get<P::TPS>(big, x.scratch + 2 * P::WARPS);
  }
  const int sh = BITS - bits64(big);
  e0 -= sh;
  if (B::active(x.t)) {
    if (sh >= 0) {
#pragma unroll
      for (int j = 0; j < B::POINTS; ++j) v[j] = mkq(v[j].x << sh, v[j].y << sh);
    } else {
#pragma unroll
      for (int j = 0; j < B::POINTS; ++j) v[j] = ShiftRight(-sh)(v[j]);
    }
  }
  const int r = fx_forward<P, G::K, MEASURE, 1>(v, x.src, tw, x.t, x.f, x.scratch + P::WARPS);
  if constexpr (MEASURE && COMMON) {  // results of two shifts: bring both to the larger one
    if (x.t == 0) x.scratch[0] = r;
    pair_sync<P>();
    const int rm = max(x.seq_scratch(0)[0], x.seq_scratch(1)[0]);
    if (r < rm) {
      for (int q = x.t; q < N; q += P::TPS) {
        const q2 z = x.src[pad(q)];
        x.src[pad(q)] = mkq(shr_round(z.x, rm - r), shr_round(z.y, rm - r));
      }
    }
    pair_sync<P>();
    return clamp_exp(e0 + rm + P::SHIFT);
  } else {
    pair_sync<P>();
    return clamp_exp(e0 + r + P::SHIFT);
  }
}

// nu k^2 of mode i for a member.
__device__ __forceinline__ double mode_nuk2(const Dev& d, const MemberWindow& mw, int i) {
  return d.ragged ? mw.nu * d.k2[i] : d.nuk2[i];
}

// One mode of the forward column pass: p, q the transforms of u v and v^2 -
// u^2 at exponent e; w the state at the step's start, y the stage value, acc
// the RK sum.  Updates w (stage 4), y and acc.  forced: the mode carries the
// force's coefficient fval.
__device__ __forceinline__ void rk_mode(const Dev& d, int stage, const ModeSym& m, double nk2, q2 p, q2 q, int e,
                                        bool forced, double fval, double2& w, double2& y, double2& acc) {
  // F = -(cp P + cq Q) - nu k^2 y
  const int eF = e + 64 + m.get_e;
  const double ax = fx_to_double(fx_pair_sum<1>(m.get, p.x, q.x), eF);
  const double ay = fx_to_double(fx_pair_sum<1>(m.get, p.y, q.y), eF);
  double2 F = make_double2(-fma(nk2, y.x, ax), -fma(nk2, y.y, ay));
  if (forced) F.x += fval;
  if (stage == 1) {
    acc = F;
    y = make_double2(fma(d.dt2, F.x, w.x), fma(d.dt2, F.y, w.y));
  } else if (stage == 2) {
    acc = make_double2(fma(2.0, F.x, acc.x), fma(2.0, F.y, acc.y));
    y = make_double2(fma(d.dt2, F.x, w.x), fma(d.dt2, F.y, w.y));
  } else if (stage == 3) {
    acc = make_double2(fma(2.0, F.x, acc.x), fma(2.0, F.y, acc.y));
    y = make_double2(fma(d.dt, F.x, w.x), fma(d.dt, F.y, w.y));
  } else {
    y = make_double2(fma(d.dt6, acc.x + F.x, w.x), fma(d.dt6, acc.y + F.y, w.y));
    w = y;
  }
}

// One mode of the adjoint column pass of stage 4..1: ru, rv the transforms of
// rho_u, rho_v at exponent e; kb the stage value, lb lambda at the step's end,
// sum the stages' sum.  Updates sum, kb (the next stage's) and, on stage 1, lb
// (lambda at the step's start; src: the observation source there).
__device__ __forceinline__ void adj_mode(const Dev& d, int stage, const ModeSym& m, double nk2, q2 ru, q2 rv, int e,
                                         bool has_src, double2 src, double2& kb, double2& lb, double2& sum) {
  // t = (-i ky/k^2) Ru + (i kx/k^2) Rv (the 1/2 of the row unpack in a1, c1)
  const int eR = e + 64 + m.get_e;
  const double2 tt = make_double2(fx_to_double(fx_pair_sum<-1>(m.get, ru.y, rv.y), eR),
                                  -fx_to_double(fx_pair_sum<-1>(m.get, ru.x, rv.x), eR));
  double2 yb;
  yb.x = -fma(nk2, kb.x, tt.x);
  yb.y = -fma(nk2, kb.y, tt.y);
  if (stage == 4) {
    sum = yb;
    kb = make_double2(fma(d.dt3, lb.x, d.dt * yb.x), fma(d.dt3, lb.y, d.dt * yb.y));
  } else if (stage == 3) {
    sum = cadd(sum, yb);
    kb = make_double2(fma(d.dt3, lb.x, d.dt2 * yb.x), fma(d.dt3, lb.y, d.dt2 * yb.y));
  } else if (stage == 2) {
    sum = cadd(sum, yb);
    kb = make_double2(fma(d.dt6, lb.x, d.dt2 * yb.x), fma(d.dt6, lb.y, d.dt2 * yb.y));
  } else {
    lb = cadd(lb, cadd(sum, yb));
    if (has_src) lb = cadd(lb, src);
    kb = cscale(lb, d.dt6);
  }
}

// Whether mode (kx, ky) carries the Kolmogorov force, and its coefficient.
__device__ __forceinline__ bool forced_mode(const Dev& d, const MemberWindow& mw, int kx, int ky) {
  return mw.forced && kx == 0 && (ky == d.nf || ky == -d.nf);
}
template <int N>
__device__ __forceinline__ double force_value(const Dev& d) {
  return -d.amp * d.nf * (double)N * N / 2.0;
}

// The place of a thread of a pass kernel, whose CTA is one pair, in its
// dynamic shared memory; the probe sums after it (adjoint column passes).
template <int N, int V>
__device__ __forceinline__ Place<FxPlan<N, V>> pass_place(void* base) {
  using X = Place<FxPlan<N, V>>;
  q2* a = static_cast<q2*>(base);
  return X(a, reinterpret_cast<int*>(a + 2 * X::OTHER), 0, threadIdx.x);
}
template <int N, int V>
__device__ __forceinline__ double2* pass_probe_sums(void* base) {
  return reinterpret_cast<double2*>(static_cast<char*>(base) + Geo<N, V>::SMEM_FX);
}

// Restart from the compact state in W (a checkpoint): Y = W and the inverse
// column transforms of u and v of stage 1.  grid (Kc, B).
template <int N, int V = 0>
__global__ void __launch_bounds__(Geo<N, V>::THREADS) k_state_cols(Dev d) {
  using G = Geo<N, V>;
  extern __shared__ double2 sm[];
  const int kx = blockIdx.x, bm = blockIdx.y;
  ColumnPut<FxPlan<N, V>> put;
#pragma unroll
  for (int j = 0; j < put.MT; ++j) {
    const int rr = threadIdx.x + j * G::THREADS;
    if (rr >= G::Kr) break;
    const size_t idx = cidx<N>(bm, rr, kx);
    const double2 w = d.W[idx];
    d.Y[idx] = w;
    put_stage_columns(put, j, d.symF[kx * G::Kr + rr], w);
  }
  Place<FxPlan<N, V>> x = pass_place<N, V>(sm);
  finish_to_mixed(d, put, x, bm, kx);
}

// ---------------------------------------------------------------------------
// Row passes
// ---------------------------------------------------------------------------

// A row of each of two mixed fields (MA, MB: Kc values each; eA, eB: the
// exponents of the Kc columns), packed for the inverse transform along x as
// the first + i the second: Z(kx) = A + iB, Z(-kx) = conj(A) + i conj(B) for the
// mixed half spectra A, B (kx = 0..K); the DC bin keeps real parts only; the
// gap is zeroed.  Into the sequence's src buffer, synchronised.
constexpr int kRowBits = 61;
struct RowLoad {
  int e;    // exponent of the row as it stands in src
  int pre;  // shift its inverse transform starts with
};
template <typename P>
__device__ __forceinline__ RowLoad load_row(const q2* __restrict__ MA, const q2* __restrict__ MB,
                                            const int* __restrict__ eA, const int* __restrict__ eB, Place<P>& x) {
  using G = Geo<P::N>;
  constexpr int N = P::N, K = G::K, Kc = G::Kc, GAP = N - 2 * K - 1, J = (Kc + P::TPS - 1) / P::TPS;
  q2 p[J], q[J];
  int ep[J], eq[J], e = 2 * kZeroExp;
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const int kx = x.t + j * P::TPS;
    if (kx < Kc) {
      p[j] = MA[kx];
      q[j] = MB[kx];
      ep[j] = eA[kx];
      eq[j] = eB[kx];
    }
  }
  for (int u = x.t; u < GAP; u += P::TPS) x.src[pad(K + 1 + u)] = mkq(0, 0);
  // one exponent for the row, at which its largest component has kRowBits - 1
  // bits (sums of two have one more): the columns' own exponents would leave
  // the small ones to be rounded at the unit of the largest
#pragma unroll
  for (int j = 0; j < J; ++j) {
    if (x.t + j * P::TPS < Kc) {
      e = max(e, bits64(max_mag(0, p[j])) + ep[j]);
      e = max(e, bits64(max_mag(0, q[j])) + eq[j]);
    }
  }
  e = seq_max_put<P::TPS>(e, x.t, x.scratch);
  if constexpr (P::TPS > 32) seq_sync<P::TPS>(x.f);
  e = seq_max_get<P::TPS>(e, x.scratch) - (kRowBits - 1);
  int sum = 0;
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const int kx = x.t + j * P::TPS;
    if (kx < Kc) {
      const q2 A = Shift(ep[j] - e)(p[j]), B = Shift(eq[j] - e)(q[j]);
      sum += 2 * mag_units(A, B);  // of Z(kx) and Z(-kx)
      if (kx == 0) {
        x.src[0] = mkq(A.x, B.x);
      } else {
        x.src[pad(kx)] = mkq(A.x - B.y, A.y + B.x);
        x.src[pad(N - kx)] = mkq(A.x + B.y, B.x - A.y);
      }
    }
  }
  sum = seq_sum_put<P::TPS>(sum, x.t, x.scratch + P::WARPS);
  seq_sync<P::TPS>(x.f);
  return {e, inv_shift<P, kRowBits>(seq_sum_get<P::TPS>(sum, x.scratch + P::WARPS))};
}

// Forward transforms along x of rows y0, y0+1, sequence f packed as (field 0
// of row y0+f) + i (field 1 of row y0+f) -> twice the two fields of both rows
// (A = Z(k) + conj Z(-k), B = -i (Z(k) - conj Z(-k)); the column pass's
// symbols carry the 1/2) in the column-major Mn of the member: entry
// (kx, f, y) at (kx * 2 + f) * N + y; e: this sequence's exponent.
template <int N, int V>
__device__ __forceinline__ void store_row_pair(const Dev& d, int bm, int y0, const Place<FxPlan<N, V>>& x, int e) {
  using G = Geo<N, V>;
  __syncthreads();  // both rows are in
  const q2* a = x.first(x.src);
  q2* O = d.Mn + (size_t)bm * G::Kc * 2 * N;
#pragma unroll
  for (int j = 0; j < (2 * G::Kc + G::THREADS - 1) / G::THREADS; ++j) {
    const int u = threadIdx.x + j * G::THREADS;
    if (u < 2 * G::Kc) {
      const int rr = u & 1, kx = u >> 1;
      const q2 zk = a[rr * x.OTHER + pad(kx)], zm = a[rr * x.OTHER + pad((N - kx) & (N - 1))];
      q2* o = O + (size_t)kx * 2 * N + y0 + rr;
      o[0] = mkq(zk.x + zm.x, zk.y - zm.y);
      o[N] = mkq(zk.y + zm.y, zm.x - zk.x);
    }
  }
  if (x.t == 0) d.eN[bm * N + y0 + x.f] = clamp_exp(e);
}

// Bits that a row pass brings u, v and 2a, b to, so that the products, less
// the 64 bits dropped, enter the forward transform with one bit to spare for
// the sums of store_row_pair: room for all its stages, or (MEASURE, where it
// gives the products at least two bits more) for the first one.
template <typename P>
struct RowBits {
  static constexpr int F = P::BITS_FWD - 1;
  static constexpr int UV0 = (64 + F) / 2;  // u v and v^2 - u^2: 2 UV - 64 <= F
  static constexpr int AB0 = 63 + F - UV0;  // sums of two products: UV + AB - 63 <= F
  static constexpr int UV1 = 61, AB1 = P::GROWTH1 <= 3 ? 61 : 60;
  static constexpr bool MEASURE = UV1 + AB1 >= UV0 + AB0 + (P::N >= 1024 ? 1 : 2);
  static constexpr int UV = MEASURE ? UV1 : UV0, AB = MEASURE ? AB1 : AB0;
};

// Inverse transform along x of a loaded row, brought to BITS bits: z[j] at x =
// row_x(j).  between runs before the results are measured.  Returns the row's
// exponent.
template <typename P>
struct RowPoints {
  static constexpr int R = LastRadix<typename P::inv>::value;
  using B = Bfly<P, R>;
  static constexpr int POINTS = B::POINTS;
  __device__ static __forceinline__ int x(int t, int j) { return t + (j / R) * P::TPS + (j % R) * B::NB; }
};
template <typename P, int BITS, typename Between>
__device__ __forceinline__ int row_fields(const RowLoad& in, Place<P>& x, const int4* tw, q2* z, Between between) {
  using RP = RowPoints<P>;
  fx_inverse<P, Geo<P::N>::K>(x.src, tw, x.t, x.f, in.pre, z);
  between();
  int m = 0;
  if (RP::B::active(x.t)) {
#pragma unroll
    for (int j = 0; j < RP::POINTS; ++j) m = max_mag(m, z[j]);
  }
  m = seq_max_put<P::TPS>(m, x.t, x.scratch + 2 * P::WARPS);
  if constexpr (P::TPS > 32) seq_sync<P::TPS>(x.f);
  m = seq_max_get<P::TPS>(m, x.scratch + 2 * P::WARPS);
  const int sh = max(0, BITS - bits64(m));  // at most 60 bits: never right
  if (RP::B::active(x.t)) {
#pragma unroll
    for (int j = 0; j < RP::POINTS; ++j) z[j] = mkq(z[j].x << sh, z[j].y << sh);
  }
  return clamp_exp(in.e + in.pre + P::SHIFT_INV - sh);
}

// (u, v) -> P + i Q, P = u v, Q = v^2 - u^2 (less 64 bits).
__device__ __forceinline__ q2 uv_products(q2 z) {
  return mkq(mul_hi(z.x, z.y), mul_hi(z.y - z.x, z.y + z.x));
}
// (2a, b) with the stored u, v -> rho_u + i rho_v, rho_u = v b - u 2a, rho_v =
// u b + v 2a (less 64 bits).
__device__ __forceinline__ q2 rho_products(q2 uv, q2 ab) {
  const Words u(uv.x), v(uv.y), a(ab.x), b(ab.y), na(-ab.x);
  return mkq(mul_hi2(v, b, u, na), mul_hi2(u, b, v, a));
}

// Velocity at a probe into its place o of the observations.  Out of line: few
// steps have probes, and few threads one.
static __device__ __noinline__ void put_probe(double* o, i64 u, i64 v, int e) {
  o[0] = fx_to_double(u, e);
  o[1] = fx_to_double(v, e);
}
// Place of the probe of row y, column xx of a member's slot (P probes a side,
// st points apart).
__device__ __forceinline__ double* probe_place(const Dev& d, int bm, int slot, int P, int st, int y, int xx) {
  return d.obs + bm * d.obs_stride + ((size_t)slot * P * P + (y / st) * P + xx / st) * 2;
}

// First value of the stored stage fields of stage `stage` of step n, row y of
// member bm, over N: index of the row (times N: of its values).
template <int N>
__device__ __forceinline__ size_t stored_row(const Dev& d, int bm, int n, int stage, int y) {
  return (((size_t)bm * d.traj_steps + (n - d.seg0)) * 4 + (stage - 1)) * N + y;
}

// Row pass of stage `stage` (1..4) of step n: u, v of rows y0, y0+1; the
// stage-field store and probe gather; the products u v and v^2 - u^2 of
// each row (packed as P + i Q) and their forward transforms along x into
// Mn.  OBS: with the probe gather.  grid (N/2, B).
template <int N, int V, bool OBS>
__global__ void __launch_bounds__(Geo<N, V>::THREADS, Geo<N, V>::ROW_CTAS) k_fwd_rows(Dev d, int n, int stage, int flags) {
  using P = FxPlan<N, V>;
  using RP = RowPoints<P>;
  extern __shared__ double2 sm[];
  Place<P> x = pass_place<N, V>(sm);
  const int bm = d.b0 + blockIdx.y, y0 = 2 * blockIdx.x, y = y0 + x.f;
  const MemberWindow mw = member_window(d, bm);
  if (n < mw.start) return;  // the member's window has not begun
  constexpr int Kc = Geo<N>::Kc;
  const q2* MA = d.Mx + ((size_t)bm * 2 * N + y) * Kc;
  const int* eX = d.eX + (size_t)bm * 2 * Kc;
  const RowLoad in = load_row<P>(MA, MA + (size_t)N * Kc, eX, eX + Kc, x);
  q2 z[RP::POINTS];
  const int ex = row_fields<P, RowBits<P>::UV>(in, x, d.fxtw, z, [] {});
  const size_t trow = stored_row<N>(d, bm, n, stage, y);
  const bool store = (flags & F_STORE) != 0;
  if (store && x.t == 0) d.eT[trow] = ex;
  if (RP::B::active(x.t)) {
    if constexpr (OBS) {
      const int st = N / mw.P, slot = obs_slot(d, n - mw.start);
      if (slot >= 0 && (y % st) == 0) {
#pragma unroll
        for (int j = 0; j < RP::POINTS; ++j) {
          const int xx = RP::x(x.t, j);
          if ((xx % st) == 0) put_probe(probe_place(d, bm, slot, mw.P, st, y, xx), z[j].x, z[j].y, ex);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < RP::POINTS; ++j) {
      if (store) d.traj[trow * N + RP::x(x.t, j)] = z[j];
      z[j] = uv_products(z[j]);
    }
  }
  if constexpr (OBS) {
    if (flags & F_OBS_ONLY) return;  // the final state: probes only
  }
  const int r = fx_forward<P, Geo<N>::K, RowBits<P>::MEASURE, 1>(z, x.src, d.fxtw, x.t, x.f, x.scratch);
  store_row_pair<N, V>(d, bm, y0, x, 2 * ex + 64 + P::SHIFT + r);
}

// ---------------------------------------------------------------------------
// Control map, its inverse and the gradient map
// ---------------------------------------------------------------------------
//
// One real field: two rows make one complex sequence, and the two sequences of
// a CTA are two pairs of rows, or two columns (the second of the last pair a
// copy of the first where Kc is odd).

// Real rows in[b][y][x] -> mixed half rows in field 0 of Mn (forward along x,
// unnormalised).  grid (N/4, B).
template <int N, int V = 0>
__global__ void __launch_bounds__(Geo<N, V>::THREADS) k_r2c_rows(Dev d, const double* __restrict__ in) {
  using P = FxPlan<N, V>;
  using G = Geo<N>;
  extern __shared__ double2 sm[];
  Place<P> x = pass_place<N, V>(sm);
  const int bm = blockIdx.y, y0 = 4 * blockIdx.x + 2 * x.f;
  constexpr int R = FirstRadix<typename P::fwd>::value;
  constexpr bool MEASURE = P::GROWTH >= P::GROWTH1 + 1;
  constexpr int BITS = MEASURE ? 62 - P::GROWTH1 : P::BITS_FWD - 1;
  using B = Bfly<P, R>;
  const double* r0 = in + ((size_t)bm * N + y0) * N;
  double2 v[B::POINTS];
  int f = 0;
  if (B::active(x.t)) {
#pragma unroll
    for (int j = 0; j < B::POINTS; ++j) {
      const int xx = x.t + (j / R) * P::TPS + (j % R) * B::NB;
      v[j] = make_double2(r0[xx], r0[N + xx]);
      f = max(f, max(exp_field(v[j].x), exp_field(v[j].y)));
    }
  }
  f = seq_max_put<P::TPS>(f, x.t, x.scratch);
  if constexpr (P::TPS > 32) seq_sync<P::TPS>(x.f);
  const int e = exp_for<BITS>(seq_max_get<P::TPS>(f, x.scratch));
  q2 z[B::POINTS];
  if (B::active(x.t)) {
#pragma unroll
    for (int j = 0; j < B::POINTS; ++j) z[j] = mkq(double_to_fx(v[j].x, e), double_to_fx(v[j].y, e));
  }
  const int r = fx_forward<P, G::K, MEASURE, 1>(z, x.src, d.fxtw, x.t, x.f, x.scratch + P::WARPS);
  q2* M = d.Mn + (size_t)bm * G::Kc * 2 * N + y0;
  for (int kx = x.t; kx < G::Kc; kx += P::TPS) {
    const q2 zk = x.src[pad(kx)], zm = x.src[pad((N - kx) & (N - 1))];
    q2* o = M + (size_t)kx * 2 * N;
    o[0] = mkq(zk.x + zm.x, zk.y - zm.y);
    o[1] = mkq(zk.y + zm.y, zm.x - zk.x);
  }
  if (x.t < 2) d.eN[bm * N + y0 + x.t] = clamp_exp(e + r + P::SHIFT - 1);  // the sums are twice the spectra
}

// s_hat = forward transform along y of field 0 of Mn; w0 = mult s_hat into W.
// NEXT: also into Y, and the inverse column transforms of u and v of stage 1;
// a CTA then has one column, which both its sequences transform.
// grid ((Kc + 1) / 2, B), with NEXT (Kc, B).
template <int N, int V, bool NEXT>
__global__ void __launch_bounds__(Geo<N, V>::THREADS) k_ctrl_cols(Dev d) {
  using P = FxPlan<N, V>;
  using G = Geo<N, V>;
  extern __shared__ double2 sm[];
  Place<P> x = pass_place<N, V>(sm);
  const int bm = blockIdx.y, kx = NEXT ? (int)blockIdx.x : min(2 * (int)blockIdx.x + x.f, G::Kc - 1);
  const int e =
      forward_columns<P, false>(d.Mn + ((size_t)bm * G::Kc + kx) * 2 * N, d.eN + bm * N, x, d.fxtw, [] {});
  auto w0 = [&](int rr, const q2* a) {
    const size_t idx = cidx<N>(bm, rr, kx);
    const q2 z = a[pad(ky_of_row(rr, G::K) & (N - 1))];
    const double2 w = cscale(make_double2(fx_to_double(z.x, e), fx_to_double(z.y, e)), d.mult[idx]);
    d.W[idx] = w;
    if constexpr (NEXT) d.Y[idx] = w;
    return w;
  };
  if constexpr (NEXT) {
    ColumnPut<P> put;
#pragma unroll
    for (int j = 0; j < put.MT; ++j) {
      const int rr = threadIdx.x + j * G::THREADS;
      if (rr >= G::Kr) break;
      put_stage_columns(put, j, d.symF[kx * G::Kr + rr], w0(rr, x.first(x.src)));
    }
    finish_to_mixed(d, put, x, bm, kx);
  } else {
    for (int rr = x.t; rr < G::Kr; rr += P::TPS) w0(rr, x.src);
  }
}

// Compact spectrum src[b] times a multiplier (and 1/N^2), transformed along
// y -> field 0 of Mx.  grid ((Kc + 1) / 2, B).
template <int N, int V = 0>
__global__ void __launch_bounds__(Geo<N, V>::THREADS) k_spec_to_mixed(Dev d, const double2* __restrict__ src, int mode) {
  using P = FxPlan<N, V>;
  using G = Geo<N>;
  extern __shared__ double2 sm[];
  Place<P> x = pass_place<N, V>(sm);
  const int bm = blockIdx.y, kx = min(2 * (int)blockIdx.x + x.f, G::Kc - 1);
  constexpr int MT = (G::Kr + P::TPS - 1) / P::TPS, GAP = N - 2 * G::K - 1;
  const double s = 1.0 / ((double)N * N);
  double2 v[MT];
  int top = 0;
#pragma unroll
  for (int j = 0; j < MT; ++j) {
    const int rr = x.t + j * P::TPS;
    if (rr >= G::Kr) break;
    const int ky = ky_of_row(rr, G::K);
    const size_t idx = cidx<N>(bm, rr, kx);
    const double m = d.mult[idx];
    double f;
    if (mode == M_ONE) f = 1.0;
    else if (mode == M_CTRL) f = m;
    else if (mode == M_FILTERED) f = (kx == 0 && ky == 0) ? 0.0 : m * m / sqrt((double)(kx * kx + ky * ky));
    else f = m != 0.0 ? 1.0 / m : 0.0;
    v[j] = cscale(src[idx], f * s);
    top = max(top, max(exp_field(v[j].x), exp_field(v[j].y)));
  }
  top = seq_max_put<P::TPS>(top, x.t, x.scratch);
  if constexpr (P::TPS > 32) seq_sync<P::TPS>(x.f);
  const int e = exp_for<60>(seq_max_get<P::TPS>(top, x.scratch));
  int sum = 0;
#pragma unroll
  for (int j = 0; j < MT; ++j) {
    const int rr = x.t + j * P::TPS;
    if (rr >= G::Kr) break;
    const q2 z = mkq(double_to_fx(v[j].x, e), double_to_fx(v[j].y, e));
    sum += mag_units(z, mkq(0, 0));
    x.src[pad(ky_of_row(rr, G::K) & (N - 1))] = z;
  }
  for (int u = x.t; u < GAP; u += P::TPS) x.src[pad(G::K + 1 + u)] = mkq(0, 0);
  sum = seq_sum_put<P::TPS>(sum, x.t, x.scratch + P::WARPS);
  seq_sync<P::TPS>(x.f);
  const int pre = inv_shift<P, 60>(seq_sum_get<P::TPS>(sum, x.scratch + P::WARPS));
  using RP = RowPoints<P>;
  q2 z[RP::POINTS];
  fx_inverse<P, G::K>(x.src, d.fxtw, x.t, x.f, pre, z);
  q2* M = d.Mx + (size_t)bm * 2 * N * G::Kc + kx;
  if (RP::B::active(x.t)) {
#pragma unroll
    for (int j = 0; j < RP::POINTS; ++j) M[(size_t)RP::x(x.t, j) * G::Kc] = z[j];
  }
  if (x.t == 0) d.eX[bm * 2 * G::Kc + kx] = clamp_exp(e + pre + P::SHIFT_INV);
}

// Mixed half rows of field 0 of Mx -> real rows out[b][y][x] (the inverse
// along x; the 1/N^2 is already in Mx).  grid (N/4, B).
template <int N, int V = 0>
__global__ void __launch_bounds__(Geo<N, V>::THREADS) k_c2r_rows(Dev d, double* __restrict__ out) {
  using P = FxPlan<N, V>;
  using G = Geo<N>;
  using RP = RowPoints<P>;
  extern __shared__ double2 sm[];
  Place<P> x = pass_place<N, V>(sm);
  const int bm = blockIdx.y, y0 = 4 * blockIdx.x + 2 * x.f;
  const q2* M = d.Mx + ((size_t)bm * 2 * N + y0) * G::Kc;
  const int* eX = d.eX + (size_t)bm * 2 * G::Kc;
  const RowLoad in = load_row<P>(M, M + G::Kc, eX, eX, x);
  q2 z[RP::POINTS];
  fx_inverse<P, G::K>(x.src, d.fxtw, x.t, x.f, in.pre, z);
  const int e = clamp_exp(in.e + in.pre + P::SHIFT_INV);
  double* r0 = out + ((size_t)bm * N + y0) * N;
  if (RP::B::active(x.t)) {
#pragma unroll
    for (int j = 0; j < RP::POINTS; ++j) {
      r0[RP::x(x.t, j)] = fx_to_double(z[j].x, e);
      r0[N + RP::x(x.t, j)] = fx_to_double(z[j].y, e);
    }
  }
}

// ---------------------------------------------------------------------------
// Forward RK stage: column pass
// ---------------------------------------------------------------------------

// Column pass of stage `stage`: the advection term
//   n_hat = (ky^2 - kx^2) DFT(u v) - kx ky DFT(v^2 - u^2),
// k_j = -n_hat - nu k^2 y_j + f_hat, the RK4 update, and the inverse column
// transforms of u and v of the next stage state.  Acc holds k1 + 2 k2 +
// 2 k3 (+ k4).  grid (Kc, B).
template <int N, int V, bool EARLY>
__global__ void __launch_bounds__(Geo<N, V>::THREADS, EARLY ? 1 : Geo<N, V>::COL_CTAS) k_fwd_cols(Dev d, int n, int stage) {
  using G = Geo<N, V>;
  using P = FxPlan<N, V>;
  extern __shared__ double2 sm[];
  Place<P> x = pass_place<N, V>(sm);
  const int kx = blockIdx.x, bm = d.b0 + blockIdx.y;
  const MemberWindow mw = member_window(d, bm);
  if (n < mw.start) return;
  // the epilogue's inputs for this thread's modes (EARLY: loaded before the transforms)
  ColumnPut<P> put;
  double2 yv[put.MT], wv[put.MT], accv[put.MT];
  ModeSym mc[put.MT];
  double nk2[put.MT];
  auto load_inputs = [&](int t) {
    const int rr = threadIdx.x + t * G::THREADS;
    if (rr < G::Kr) {
      const size_t idx = cidx<N>(bm, rr, kx);
      yv[t] = d.Y[idx];
      wv[t] = d.W[idx];
      accv[t] = stage > 1 ? d.Acc[idx] : make_double2(0.0, 0.0);
      mc[t] = d.symF[kx * G::Kr + rr];
      nk2[t] = mode_nuk2(d, mw, kx * G::Kr + rr);
    }
  };
  const int e = forward_columns<P>(d.Mn + (((size_t)bm * G::Kc + kx) * 2 + x.f) * N, d.eN + bm * N, x, d.fxtw, [&] {
    if constexpr (EARLY) {
#pragma unroll
      for (int t = 0; t < put.MT; ++t) load_inputs(t);
    }
  });
  const q2 *a0 = x.first(x.src), *a1 = a0 + x.OTHER;
  const double fval = force_value<N>(d);
#pragma unroll
  for (int t = 0; t < put.MT; ++t) {
    const int rr = threadIdx.x + t * G::THREADS;
    if (rr >= G::Kr) break;
    if constexpr (!EARLY) load_inputs(t);
    const int ky = ky_of_row(rr, G::K);
    const int qi = pad(ky & (N - 1));
    const size_t idx = cidx<N>(bm, rr, kx);
    rk_mode(d, stage, mc[t], nk2[t], a0[qi], a1[qi], e, forced_mode(d, mw, kx, ky), fval, wv[t], yv[t],
            accv[t]);
    if (stage < 4) d.Acc[idx] = accv[t];
    else d.W[idx] = wv[t];
    d.Y[idx] = yv[t];
    put_stage_columns(put, t, mc[t], yv[t]);
  }
  finish_to_mixed(d, put, x, bm, kx);
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
__device__ __forceinline__ void probe_row_sums(const Dev& d, int bm, int P, int slot, int kx, int thread, int threads,
                                               double2* Tu, double2* Tv) {
  const double* r = d.res + bm * d.obs_stride + (size_t)slot * P * P * 2;
  const int tws = 64 / P;
  for (int row = thread; row < P; row += threads) {
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
  Place<FxPlan<N, V>> x = pass_place<N, V>(sm);
  double2 *Tu = pass_probe_sums<N, V>(sm), *Tv = Tu + G::PMAX;
  const int kx = blockIdx.x, bm = blockIdx.y;
  const MemberWindow mw = member_window(d, bm);
  // an idle member starts (and stays) at lambda = 0
  if (mw.start > d.nsteps) mode = 0;
  const bool resume = (mode & INIT_RESUME) != 0;
  const int slot = (!resume && (mode & INIT_SRC)) ? obs_slot(d, d.nsteps - mw.start) : -1;
  if (slot >= 0) probe_row_sums(d, bm, mw.P, slot, kx, threadIdx.x, G::THREADS, Tu, Tv);
  __syncthreads();
  ColumnPut<FxPlan<N, V>> put;
#pragma unroll
  for (int j = 0; j < put.MT; ++j) {
    const int rr = threadIdx.x + j * G::THREADS;
    if (rr >= G::Kr) break;
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
    put_adjoint_columns(put, j, d.symA[kx * G::Kr + rr], kb);
  }
  finish_to_mixed(d, put, x, bm, kx);
}

// Adjoint row pass of stage `stage` of step n: 2a, b of rows y0, y0+1
// (inverse transforms along x), rho_u and rho_v with the stored u, v (each
// row packed as rho_u + i rho_v), and their forward transforms along x into
// Mn (twice, as in the forward row pass).  grid (N/2, B).
template <int N, int V = 0>
__global__ void __launch_bounds__(Geo<N, V>::THREADS, Geo<N, V>::ROW_CTAS) k_adj_rows(Dev d, int n, int stage) {
  using P = FxPlan<N, V>;
  using RP = RowPoints<P>;
  extern __shared__ double2 sm[];
  Place<P> x = pass_place<N, V>(sm);
  const int bm = d.b0 + blockIdx.y, y0 = 2 * blockIdx.x, y = y0 + x.f;
  if (d.ragged && n < d.mstart[bm]) return;
  constexpr int Kc = Geo<N>::Kc;
  const q2* MA = d.Mx + ((size_t)bm * 2 * N + y) * Kc;
  const int* eX = d.eX + (size_t)bm * 2 * Kc;
  const RowLoad in = load_row<P>(MA, MA + (size_t)N * Kc, eX, eX + Kc, x);
  const size_t trow = stored_row<N>(d, bm, n, stage, y);
  q2 z[RP::POINTS], uv[RP::POINTS];
  const int ex = row_fields<P, RowBits<P>::AB>(in, x, d.fxtw, z, [&] {
    if (RP::B::active(x.t)) {
#pragma unroll
      for (int j = 0; j < RP::POINTS; ++j) uv[j] = d.traj[trow * N + RP::x(x.t, j)];
    }
  });
  if (RP::B::active(x.t)) {
#pragma unroll
    for (int j = 0; j < RP::POINTS; ++j) z[j] = rho_products(uv[j], z[j]);
  }
  const int eT = d.eT[trow];
  const int r = fx_forward<P, Geo<N>::K, RowBits<P>::MEASURE, 1>(z, x.src, d.fxtw, x.t, x.f, x.scratch);
  store_row_pair<N, V>(d, bm, y0, x, clamp_exp(ex + eT) + 64 + P::SHIFT + r);
}

// Adjoint column pass of stage `stage` of step n:
//   ybar_j = -P[(-i ky/k^2) DFT(rho_u) + (i kx/k^2) DFT(rho_v)] - nu k^2 kbar_j,
// the transposed RK4 combination, the observation source at step n (on
// stage 1), and the inverse column transforms of a, b of the next kbar.
// SRC: with the observation source, which few steps have and whose code would
// double the kernel.  grid (Kc, B).
template <int N, int V, bool SRC, bool EARLY>
__global__ void __launch_bounds__(Geo<N, V>::THREADS, EARLY ? 1 : Geo<N, V>::COL_CTAS) k_adj_cols(Dev d, int n, int stage) {
  using G = Geo<N, V>;
  using P = FxPlan<N, V>;
  extern __shared__ double2 sm[];
  Place<P> x = pass_place<N, V>(sm);
  double2 *Tu = pass_probe_sums<N, V>(sm), *Tv = Tu + G::PMAX;
  const int kx = blockIdx.x, bm = d.b0 + blockIdx.y;
  const MemberWindow mw = member_window(d, bm);
  if (n < mw.start) return;
  // the epilogue's inputs for this thread's modes (EARLY: loaded before the transforms)
  ColumnPut<P> put;
  double2 kbv[put.MT], lbv[put.MT], sumv[put.MT];
  ModeSym mc[put.MT];
  double nk2[put.MT];
  auto load_inputs = [&](int t) {
    const int rr = threadIdx.x + t * G::THREADS;
    if (rr < G::Kr) {
      const size_t idx = cidx<N>(bm, rr, kx);
      kbv[t] = d.KB[idx];
      lbv[t] = d.LamBar[idx];
      sumv[t] = stage < 4 ? d.Sum[idx] : make_double2(0.0, 0.0);
      mc[t] = d.symA[kx * G::Kr + rr];
      nk2[t] = mode_nuk2(d, mw, kx * G::Kr + rr);
    }
  };
  const int slot = SRC ? obs_slot(d, n - mw.start) : -1;
  const int e = forward_columns<P>(d.Mn + (((size_t)bm * G::Kc + kx) * 2 + x.f) * N, d.eN + bm * N, x, d.fxtw, [&] {
    if constexpr (EARLY) {
#pragma unroll
      for (int t = 0; t < put.MT; ++t) load_inputs(t);
    }
    if constexpr (SRC) {
      if (slot >= 0) probe_row_sums(d, bm, mw.P, slot, kx, threadIdx.x, G::THREADS, Tu, Tv);
    }
  });
  const q2 *a0 = x.first(x.src), *a1 = a0 + x.OTHER;
#pragma unroll
  for (int t = 0; t < put.MT; ++t) {
    const int rr = threadIdx.x + t * G::THREADS;
    if (rr >= G::Kr) break;
    if constexpr (!EARLY) load_inputs(t);
    const int ky = ky_of_row(rr, G::K);
    const int qi = pad(ky & (N - 1));
    const size_t idx = cidx<N>(bm, rr, kx);
    double2 src = make_double2(0.0, 0.0);
    if constexpr (SRC) {
      if (slot >= 0) src = probe_source(d, mw.P, kx, ky, Tu, Tv);
    }
    adj_mode(d, stage, mc[t], nk2[t], a0[qi], a1[qi], e, slot >= 0, src, kbv[t], lbv[t], sumv[t]);
    if (stage > 1) d.Sum[idx] = sumv[t];
    else d.LamBar[idx] = lbv[t];
    d.KB[idx] = kbv[t];
    put_adjoint_columns(put, t, mc[t], kbv[t]);
  }
  if (stage == 1 && n == mw.start) return;  // the member's first step: lambda_0 stays in LamBar
  finish_to_mixed(d, put, x, bm, kx);
}

// Per-mode constants of the column passes (ModeSym), k^2 and nu k^2.
// grid ceil(Kr*Kc/256), block 256.
template <int N, int V = 0>
__global__ void k_make_symbols(ModeSym* __restrict__ F, ModeSym* __restrict__ A, double* __restrict__ k2out,
                               double* __restrict__ nuk2, double nu) {
  using G = Geo<N, V>;
  const double s2 = 1.0 / ((double)N * N);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < G::Kr * G::Kc; i += gridDim.x * blockDim.x) {
    const int kx = i / G::Kr, r = i - kx * G::Kr;
    const int ky = ky_of_row(r, G::K);
    const double k2 = (double)(kx * kx + ky * ky);
    const double ik2 = k2 > 0.0 ? 1.0 / k2 : 0.0;
    ModeSym f{}, a{};
    // a mode whose put symbols vanish must not set its column's exponent
    f.put = fx_pair(ky * ik2 * s2, kx * ik2 * s2, kZeroExp, &f.put_e);
    f.get = fx_pair(0.5 * (ky * ky - kx * kx), -0.5 * kx * ky, 0, &f.get_e);
    a.put = fx_pair(-2.0 * kx * ky * s2, (double)(ky * ky - kx * kx) * s2, kZeroExp, &a.put_e);
    a.get = fx_pair(0.5 * ky * ik2, 0.5 * kx * ik2, 0, &a.get_e);
    F[i] = f;
    A[i] = a;
    k2out[i] = k2;
    nuk2[i] = nu * k2;
  }
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
