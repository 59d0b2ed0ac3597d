// window.cuh -- whole windows of small grids in one kernel.
//
// A pass of a small grid is a microsecond of work that the launch-per-pass
// sequence surrounds with a kernel boundary, cold instruction and data caches
// and a trip of every field through L2: 3.9 us a pass at 64^2.  Here one
// cluster of CTAs runs a member's whole window: every CTA owns some rows and
// some columns, the mixed fields go from the one to the other through
// distributed shared memory, a cluster barrier ends each pass, and the RK and
// adjoint states of the columns stay in registers.  Members are independent
// clusters.  Stage fields, observations and the state at the ends of a window
// are in global memory as in the pass kernels, and the arithmetic is theirs,
// value by value (the same functions on the same plan), so that the results
// are bitwise the same whichever path a batch takes.
#pragma once
#include <cooperative_groups.h>

#include "kernels.cuh"

namespace da {

namespace cg = cooperative_groups;

// Cluster of CTAs of one member: N = 64 on 16, so that a CTA's four rows are
// four warps' work at most; a 16^2 window fits one CTA.
template <int N, int V>
struct WinGeo {
  using G = Geo<N>;
  static constexpr bool SUPPORTED = N <= 64;
  static constexpr int C = N == 16 ? 1 : N == 32 ? 4 : 16;
  // Largest batch that runs this way: beyond it the pass kernels, which spread
  // a batch over the whole chip, are the faster ones.  us a pass by captured
  // graphs, this way / pass kernels: 64^2 plans 0, 1, 2 at 13 members 4.4/5.3,
  // 6.6/6.6, 3.8/4.5, at 24 members 5.4/5.5, 7.9/6.8, 6.4/5.2; 32^2 plans 0, 1
  // at 64 members 5.6/5.2, 3.6/4.4, at 256 members 12.5/10.7, 8.1/7.8; 16^2 at
  // 1 member 3.9/3.8, at 256 members 4.1/5.2.  Launched directly, a pass
  // kernel costs the host 6 us, which decides for this way at 16^2 and 32^2.
  static constexpr int BATCH = N == 16 ? 1 << 30 : N == 32 ? 128 : V == 1 ? 4 : 16;
  static constexpr int ROWS = N / C, COLS = (G::Kc + C - 1) / C;
  static constexpr int RMAX = FirstRadix<typename Plan<N, V>::two>::value;
  static constexpr int TPS = N / (RMAX < 4 ? 2 : 4) < 32 ? N / (RMAX < 4 ? 2 : 4) : 32;
  using P = FxPlanOf<N, TPS, typename Plan<N, V>::two>;
  using X = Place<P>;
  static constexpr int SLOTS = ROWS;  // sequences a CTA works on at once
  static_assert(!SUPPORTED || (2 * COLS <= SLOTS && SLOTS % 2 == 0), "columns fit the rows' slots");
  static constexpr int THREADS = SLOTS * TPS;
  static constexpr int WORK = SLOTS * P::SEQ, ROWBUF = ROWS * 2 * G::Kc, COLBUF = COLS * 2 * N;  // q2
  static constexpr int INTS = 2 * G::Kc + N + SLOTS / 2 * X::SCRATCH;
  static constexpr size_t SMEM = sizeof(q2) * (WORK + ROWBUF + COLBUF + COLS * 2 * G::PMAX) + sizeof(int) * INTS;
};

// The shared memory of a CTA and its thread's places.
template <int N, int V>
struct Win {
  using W = WinGeo<N, V>;
  using G = Geo<N>;
  using P = typename W::P;
  static constexpr int C = W::C, MT = ColumnPut<P>::MT;
  q2 *rowbuf, *colbuf;  // [ROWS][2][Kc], [COLS][2][N]
  int *rowexp, *colexp; // [2][Kc] exponents of the columns, [N] of the rows
  double2* probes;      // [COLS][2][PMAX]
  Place<P> x;
  int rank, pair;
  int kx, kxs;   // this pair's column, and a valid one to read constants of
  bool column;   // kx is a column

  __device__ __forceinline__ static int* ints(void* base) {
    return reinterpret_cast<int*>(static_cast<q2*>(base) + W::WORK + W::ROWBUF + W::COLBUF + W::COLS * 2 * G::PMAX);
  }
  __device__ __forceinline__ explicit Win(void* base)
      : x(static_cast<q2*>(base), ints(base) + 2 * G::Kc + N, threadIdx.x / Place<P>::PT, threadIdx.x % Place<P>::PT) {
    rowbuf = static_cast<q2*>(base) + W::WORK;
    colbuf = rowbuf + W::ROWBUF;
    probes = reinterpret_cast<double2*>(colbuf + W::COLBUF);
    rowexp = ints(base);
    colexp = rowexp + 2 * G::Kc;
    rank = blockIdx.x % C;
    pair = threadIdx.x / Place<P>::PT;
    kx = rank + pair * C;
    column = pair < W::COLS && kx < G::Kc;
    kxs = column ? kx : 0;
  }
  __device__ __forceinline__ int row() const { return rank * W::ROWS + pair * 2 + x.f; }
  // row rr of this thread's entry j of its column, or none
  __device__ __forceinline__ int mode(int j) const { return x.pt + j * Place<P>::PT; }
  __device__ __forceinline__ bool has(int j) const { return column && mode(j) < G::Kr; }

  template <typename T>
  __device__ __forceinline__ static T* on(T* p, int r) {
    if constexpr (C == 1) return p;
    else return cg::this_cluster().map_shared_rank(p, r);
  }
  // all of the pass's writes are visible to the whole cluster afterwards
  __device__ __forceinline__ static void sync() {
    if constexpr (C == 1) __syncthreads();
    else cg::this_cluster().sync();
  }

  // This pair's columns to the rows' owners.
  __device__ __forceinline__ void send_columns(const ColumnPut<P>& put, const int4* tw) {
    const int e = finish_columns<P>(put, x, tw, [&](int y, q2 z) {
      if (column) on(rowbuf + ((y % W::ROWS) * 2 + x.f) * G::Kc + kx, y / W::ROWS)[0] = z;
    });
    if (column)
      for (int r = x.t; r < C; r += P::TPS) on(rowexp + x.f * G::Kc + kx, r)[0] = e;
  }
  __device__ __forceinline__ RowLoad take_row() {
    const q2* M = rowbuf + (pair * 2 + x.f) * 2 * G::Kc;
    return load_row<P>(M, M + G::Kc, rowexp, rowexp + G::Kc, x);
  }
  // The transformed row in src, twice its two fields, to the columns' owners.
  __device__ __forceinline__ void send_row(int e) {
    const int y = row();
    for (int k = x.t; k < G::Kc; k += P::TPS) {
      const q2 zk = x.src[pad(k)], zm = x.src[pad((N - k) & (N - 1))];
      q2* o = on(colbuf + (k / C) * 2 * N + y, k % C);
      o[0] = mkq(zk.x + zm.x, zk.y - zm.y);
      o[N] = mkq(zk.y + zm.y, zm.x - zk.x);
    }
    const int ec = clamp_exp(e);
    for (int r = x.t; r < C; r += P::TPS) on(colexp + y, r)[0] = ec;
  }
  // Forward transform of this pair's column; its exponent.
  __device__ __forceinline__ int take_columns(const int4* tw) {
    return forward_columns<P>(colbuf + ((pair < W::COLS ? pair : 0) * 2 + x.f) * N, colexp, x, tw, [] {});
  }
};

// RK steps k0..k1-1 of every member whose window they reach, from the state
// in W, to W.  grid B clusters of C CTAs.
template <int N, int V>
__global__ void __launch_bounds__(WinGeo<N, V>::THREADS) k_window_fwd(Dev d, int k0, int k1, int flags) {
  using Wn = Win<N, V>;
  using P = typename Wn::P;
  using G = Geo<N>;
  using RP = RowPoints<P>;
  extern __shared__ double2 sm[];
  Wn w(sm);
  Place<P>& x = w.x;
  const int bm = blockIdx.x / Wn::C;
  const MemberWindow mw = member_window(d, bm);
  const int first = max(k0, mw.start);
  const bool final_probes = (flags & W_FINAL) != 0;
  if (first > k1 || (first == k1 && !final_probes)) return;  // nothing of the member's window here
  double2 ws[Wn::MT], ys[Wn::MT], acc[Wn::MT];
  ModeSym mc[Wn::MT];
  double nk2[Wn::MT];
  ColumnPut<P> put;
#pragma unroll
  for (int j = 0; j < Wn::MT; ++j) {
    const int rr = w.has(j) ? w.mode(j) : 0;
    mc[j] = d.symF[w.kxs * G::Kr + rr];
    nk2[j] = mode_nuk2(d, mw, w.kxs * G::Kr + rr);
    ws[j] = w.has(j) ? d.W[cidx<N>(bm, rr, w.kx)] : make_double2(0.0, 0.0);
    ys[j] = ws[j];
    acc[j] = make_double2(0.0, 0.0);
    put_stage_columns(put, j, mc[j], ys[j]);
  }
  Wn::sync();  // every CTA of the cluster runs
  w.send_columns(put, d.fxtw);
  Wn::sync();
  const int Pp = mw.P, st = N / Pp, y = w.row();
  const double fval = force_value<N>(d);
  for (int n = first; n <= k1; ++n) {
    if (n == k1 && !final_probes) break;
    const bool store = (flags & W_STORE) != 0 && n >= d.seg0 && n < k1;
#pragma unroll 1
    for (int stage = 1; stage <= 4; ++stage) {
      // row pass
      const RowLoad in = w.take_row();
      const int slot = stage == 1 && (flags & W_OBS) ? obs_slot(d, n - mw.start) : -1;
      q2 z[RP::POINTS];
      const int ex = row_fields<P, RowBits<P>::UV>(in, x, d.fxtw, z, [] {});
      const size_t trow = stored_row<N>(d, bm, n, stage, y);
      if (store && x.t == 0) d.eT[trow] = ex;
      const bool probes = slot >= 0 && (y % st) == 0;
      if (RP::B::active(x.t)) {
#pragma unroll
        for (int j = 0; j < RP::POINTS; ++j) {
          const int xx = RP::x(x.t, j);
          if (store) d.traj[trow * N + xx] = z[j];
          if (probes && (xx % st) == 0) put_probe(probe_place(d, bm, slot, Pp, st, y, xx), z[j].x, z[j].y, ex);
          z[j] = uv_products(z[j]);
        }
      }
      if (n == k1) break;  // the final state: probes only
      const int r = fx_forward<P, G::K, RowBits<P>::MEASURE, 1>(z, x.src, d.fxtw, x.t, x.f, x.scratch);
      w.send_row(2 * ex + 64 + P::SHIFT + r);
      Wn::sync();
      // column pass
      const int e = w.take_columns(d.fxtw);
      const q2 *a0 = x.first(x.src), *a1 = a0 + x.OTHER;
      put.top = 2 * kZeroExp;
#pragma unroll
      for (int j = 0; j < Wn::MT; ++j) {
        if (!w.has(j)) {
          put.zero(j);
          continue;
        }
        const int ky = ky_of_row(w.mode(j), G::K);
        const int qi = pad(ky & (N - 1));
        rk_mode(d, stage, mc[j], nk2[j], a0[qi], a1[qi], e, forced_mode(d, mw, w.kx, ky), fval, ws[j], ys[j],
                acc[j]);
        put_stage_columns(put, j, mc[j], ys[j]);
      }
      if (stage == 4 && n == k1 - 1 && !final_probes) break;  // nothing reads the columns
      w.send_columns(put, d.fxtw);
      Wn::sync();
    }
  }
#pragma unroll
  for (int j = 0; j < Wn::MT; ++j)
    if (w.has(j)) d.W[cidx<N>(bm, w.mode(j), w.kx)] = ws[j];
}

// Adjoint steps k1-1..k0 of every member whose window they reach, from and to
// LamBar and KB.  sources: add the observation source at the observation
// steps.  grid B clusters of C CTAs.
template <int N, int V>
__global__ void __launch_bounds__(WinGeo<N, V>::THREADS) k_window_adj(Dev d, int k1, int k0, int sources) {
  using Wn = Win<N, V>;
  using P = typename Wn::P;
  using G = Geo<N>;
  using RP = RowPoints<P>;
  extern __shared__ double2 sm[];
  Wn w(sm);
  Place<P>& x = w.x;
  const int bm = blockIdx.x / Wn::C;
  const MemberWindow mw = member_window(d, bm);
  const int last = max(k0, mw.start);
  if (last >= k1) return;  // nothing of the member's window here
  double2 kb[Wn::MT], lb[Wn::MT], sum[Wn::MT];
  ModeSym mc[Wn::MT];
  double nk2[Wn::MT];
  ColumnPut<P> put;
#pragma unroll
  for (int j = 0; j < Wn::MT; ++j) {
    const int rr = w.has(j) ? w.mode(j) : 0;
    mc[j] = d.symA[w.kxs * G::Kr + rr];
    nk2[j] = mode_nuk2(d, mw, w.kxs * G::Kr + rr);
    const size_t idx = cidx<N>(bm, rr, w.kxs);
    kb[j] = w.has(j) ? d.KB[idx] : make_double2(0.0, 0.0);
    lb[j] = w.has(j) ? d.LamBar[idx] : make_double2(0.0, 0.0);
    sum[j] = make_double2(0.0, 0.0);
    put_adjoint_columns(put, j, mc[j], kb[j]);
  }
  Wn::sync();  // every CTA of the cluster runs
  w.send_columns(put, d.fxtw);
  Wn::sync();
  const int y = w.row();
  double2 *Tu = w.probes + (w.pair < WinGeo<N, V>::COLS ? w.pair : 0) * 2 * G::PMAX, *Tv = Tu + G::PMAX;
  for (int n = k1 - 1; n >= last; --n) {
#pragma unroll 1
    for (int stage = 4; stage >= 1; --stage) {
      // row pass
      const size_t trow = stored_row<N>(d, bm, n, stage, y);
      q2 uv[RP::POINTS];
      if (RP::B::active(x.t)) {
#pragma unroll
        for (int j = 0; j < RP::POINTS; ++j) uv[j] = d.traj[trow * N + RP::x(x.t, j)];
      }
      const int eT = d.eT[trow];
      const RowLoad in = w.take_row();
      q2 z[RP::POINTS];
      const int ex = row_fields<P, RowBits<P>::AB>(in, x, d.fxtw, z, [] {});
      if (RP::B::active(x.t)) {
#pragma unroll
        for (int j = 0; j < RP::POINTS; ++j) z[j] = rho_products(uv[j], z[j]);
      }
      const int r = fx_forward<P, G::K, RowBits<P>::MEASURE, 1>(z, x.src, d.fxtw, x.t, x.f, x.scratch);
      w.send_row(clamp_exp(ex + eT) + 64 + P::SHIFT + r);
      Wn::sync();
      // column pass
      const int slot = sources && stage == 1 ? obs_slot(d, n - mw.start) : -1;
      if (slot >= 0 && w.column) probe_row_sums(d, bm, mw.P, slot, w.kx, x.pt, Place<P>::PT, Tu, Tv);
      const int e = w.take_columns(d.fxtw);  // ends with the pair's barrier
      const q2 *a0 = x.first(x.src), *a1 = a0 + x.OTHER;
      put.top = 2 * kZeroExp;
#pragma unroll
      for (int j = 0; j < Wn::MT; ++j) {
        if (!w.has(j)) {
          put.zero(j);
          continue;
        }
        const int ky = ky_of_row(w.mode(j), G::K);
        const int qi = pad(ky & (N - 1));
        double2 src = make_double2(0.0, 0.0);
        if (slot >= 0) src = probe_source(d, mw.P, w.kx, ky, Tu, Tv);
        adj_mode(d, stage, mc[j], nk2[j], a0[qi], a1[qi], e, slot >= 0, src, kb[j], lb[j], sum[j]);
        put_adjoint_columns(put, j, mc[j], kb[j]);
      }
      if (stage == 1 && n == last) break;  // nothing reads the columns
      w.send_columns(put, d.fxtw);
      Wn::sync();
    }
  }
#pragma unroll
  for (int j = 0; j < Wn::MT; ++j) {
    if (!w.has(j)) continue;
    const size_t idx = cidx<N>(bm, w.mode(j), w.kx);
    d.LamBar[idx] = lb[j];
    d.KB[idx] = kb[j];
  }
}

}  // namespace da
