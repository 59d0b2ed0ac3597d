// ops_impl.cuh -- launch configurations of the pass kernels for one N.
#pragma once
#include "ops.h"
#include "window.cuh"

namespace da {

// One cluster of C CTAs per member.
template <int C, typename... A>
inline void launch_clusters(void (*f)(A...), int members, int threads, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = C;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(members * C);
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = &at;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, f, args...);
}

// The column kernels that a batch may run (Geo::EARLY_CTAS): those of one kind
// are not built where no batch, or every batch, loads early.
template <int N, int V>
struct Columns {
  using G = Geo<N, V>;
  static constexpr bool SOME_EARLY = G::EARLY_CTAS >= G::Kc, ALL_EARLY = N <= 128 && SOME_EARLY;
  static bool early(const Dev& d) {
    return ALL_EARLY || (SOME_EARLY && d.early && (long long)d.B * G::Kc <= G::EARLY_CTAS);
  }
  static auto fwd(const Dev& d) {
    return early(d) ? k_fwd_cols<N, V, SOME_EARLY> : k_fwd_cols<N, V, ALL_EARLY>;
  }
  template <bool SRC>
  static auto adj(const Dev& d) {
    return early(d) ? k_adj_cols<N, V, SRC, SOME_EARLY> : k_adj_cols<N, V, SRC, ALL_EARLY>;
  }
};

template <int N, int V>
Ops make_ops() {
  using G = Geo<N, V>;
  Ops o{};
  o.n = N;
  o.K = G::K;
  o.Kc = G::Kc;
  o.Kr = G::Kr;
  o.variant = V;
  o.threads = G::THREADS;
  o.flops_inverse = band_transform_flops<N, V, G::K>(true);
  o.flops_forward = band_transform_flops<N, V, G::K>(false);
  o.fx_entries = FxPlan<N, V>::TABLE;
  o.fx_table = []() -> const std::vector<int4>& { return fx_table<FxPlan<N, V>>(); };
  o.setup = []() -> cudaError_t {
    cudaError_t e = cudaSuccess;
    auto set = [&](const void* f, size_t s = G::SMEM_FX) {
      if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s);
    };
    set((const void*)k_r2c_rows<N, V>);
    set((const void*)k_c2r_rows<N, V>);
    set((const void*)k_spec_to_mixed<N, V>);
    set((const void*)k_ctrl_cols<N, V, false>);
    set((const void*)k_ctrl_cols<N, V, true>);
    set((const void*)k_fwd_rows<N, V, false>);
    set((const void*)k_fwd_rows<N, V, true>);
    set((const void*)k_fwd_cols<N, V, Columns<N, V>::ALL_EARLY>);
    set((const void*)k_fwd_cols<N, V, Columns<N, V>::SOME_EARLY>);
    set((const void*)k_state_cols<N, V>);
    set((const void*)k_adj_init<N, V>, G::SMEM_FXP);
    set((const void*)k_adj_rows<N, V>);
    set((const void*)k_adj_cols<N, V, false, Columns<N, V>::ALL_EARLY>, G::SMEM_FXP);
    set((const void*)k_adj_cols<N, V, true, Columns<N, V>::ALL_EARLY>, G::SMEM_FXP);
    set((const void*)k_adj_cols<N, V, false, Columns<N, V>::SOME_EARLY>, G::SMEM_FXP);
    set((const void*)k_adj_cols<N, V, true, Columns<N, V>::SOME_EARLY>, G::SMEM_FXP);
    if constexpr (WinGeo<N, V>::SUPPORTED) {
      for (const void* f : {(const void*)k_window_fwd<N, V>, (const void*)k_window_adj<N, V>}) {
        set(f, WinGeo<N, V>::SMEM);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      }
    }
    return e;
  };
  o.r2c_rows = [](const Dev& d, const double* in, cudaStream_t st) {
    k_r2c_rows<N, V><<<dim3(N / 4, d.B), G::THREADS, G::SMEM_FX, st>>>(d, in);
  };
  o.c2r_rows = [](const Dev& d, double* out, cudaStream_t st) {
    k_c2r_rows<N, V><<<dim3(N / 4, d.B), G::THREADS, G::SMEM_FX, st>>>(d, out);
  };
  o.spec_to_mixed = [](const Dev& d, const double2* src, int mode, cudaStream_t st) {
    k_spec_to_mixed<N, V><<<dim3((G::Kc + 1) / 2, d.B), G::THREADS, G::SMEM_FX, st>>>(d, src, mode);
  };
  o.compact_to_half = [](const Dev& d, const double2* src, double2* out, cudaStream_t st) {
    k_compact_to_half<N, V><<<dim3((N * G::NH + 255) / 256, d.B), 256, 0, st>>>(src, out);
  };
  o.half_to_compact = [](const Dev& d, const double2* in, double2* dst, cudaStream_t st) {
    k_half_to_compact<N, V><<<dim3((G::Kr * G::Kc + 255) / 256, d.B), 256, 0, st>>>(in, dst);
  };
  o.ctrl_cols = [](const Dev& d, bool next, cudaStream_t st) {
    if (next) k_ctrl_cols<N, V, true><<<dim3(G::Kc, d.B), G::THREADS, G::SMEM_FX, st>>>(d);
    else k_ctrl_cols<N, V, false><<<dim3((G::Kc + 1) / 2, d.B), G::THREADS, G::SMEM_FX, st>>>(d);
  };
  o.fwd_rows = [](const Dev& d, int n, int stage, int flags, cudaStream_t st) {
    if (flags & (F_OBS | F_OBS_ONLY))
      k_fwd_rows<N, V, true><<<dim3(N / 2, d.B), G::THREADS, G::SMEM_FX, st>>>(d, n, stage, flags);
    else
      k_fwd_rows<N, V, false><<<dim3(N / 2, d.B), G::THREADS, G::SMEM_FX, st>>>(d, n, stage, flags);
  };
  o.fwd_cols = [](const Dev& d, int n, int stage, cudaStream_t st) {
    Columns<N, V>::fwd(d)<<<dim3(G::Kc, d.B), G::THREADS, G::SMEM_FX, st>>>(d, n, stage);
  };
  o.state_cols = [](const Dev& d, cudaStream_t st) {
    k_state_cols<N, V><<<dim3(G::Kc, d.B), G::THREADS, G::SMEM_FX, st>>>(d);
  };
  o.adj_init = [](const Dev& d, int mode, cudaStream_t st) {
    k_adj_init<N, V><<<dim3(G::Kc, d.B), G::THREADS, G::SMEM_FXP, st>>>(d, mode);
  };
  o.adj_rows = [](const Dev& d, int n, int stage, cudaStream_t st) {
    k_adj_rows<N, V><<<dim3(N / 2, d.B), G::THREADS, G::SMEM_FX, st>>>(d, n, stage);
  };
  o.adj_cols = [](const Dev& d, int n, int stage, int flags, cudaStream_t st) {
    using C = Columns<N, V>;
    const auto f = flags & F_SRC ? C::template adj<true>(d) : C::template adj<false>(d);
    f<<<dim3(G::Kc, d.B), G::THREADS, G::SMEM_FXP, st>>>(d, n, stage);
  };
  o.window_batch = 0;
  o.window_fwd = nullptr;
  o.window_adj = nullptr;
  if constexpr (WinGeo<N, V>::SUPPORTED) {
    using W = WinGeo<N, V>;
    o.window_batch = W::BATCH;
    o.window_fwd = [](const Dev& d, int k0, int k1, int flags, cudaStream_t st) {
      launch_clusters<W::C>(k_window_fwd<N, V>, d.B, W::THREADS, W::SMEM, st, d, k0, k1, flags);
    };
    o.window_adj = [](const Dev& d, int k1, int k0, int sources, cudaStream_t st) {
      launch_clusters<W::C>(k_window_adj<N, V>, d.B, W::THREADS, W::SMEM, st, d, k1, k0, sources);
    };
  }
  o.make_symbols = [](const Dev& d, double nu, cudaStream_t st) {
    k_make_symbols<N, V><<<dim3((G::Kr * G::Kc + 255) / 256), 256, 0, st>>>((ModeSym*)d.symF, (ModeSym*)d.symA,
                                                                          (double*)d.k2, (double*)d.nuk2, nu);
  };
  o.make_mult = [](const Dev& d, double* mult, const int* kind, const double* param, const double* table, const double* nu,
                   cudaStream_t st) {
    k_make_mult<N, V><<<dim3((G::Kr * G::Kc + 255) / 256, d.B), 256, 0, st>>>(mult, kind, param, table, nu);
  };
  return o;
}

}  // namespace da

#define DA_INSTANTIATE(NN, VV)                  \
  namespace da {                                \
  const Ops* ops_n##NN##_v##VV() {              \
    static const Ops o = make_ops<NN, VV>();    \
    return &o;                                  \
  }                                             \
  }
