// ctx.h -- the context behind the C ABI of include/da.h and the host
// helpers shared by the files that implement it (da_api.cu: creation,
// forward, cost and gradient, adjoint variants; plans.cu: FFT plan variants
// and the autotuner; lbfgs.cu: the optimiser).  Internal: nothing here is
// part of the ABI.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <string>
#include <type_traits>
#include <utility>
#include <vector>

#include "../../include/da.h"
#include "ops.h"

using da::Dev;
using da::Ops;

struct da_ctx {
  int device = 0;
  int n = 0, nsteps = 0, ckpt = 0, B = 1;
  double dt = 0, nu = 0;
  da_forcing force{};
  da_obs_operator obs{};
  int nt = 0, P = 0;
  // ragged batches (da_set_member): per-member windows, end-aligned in each
  // evaluation's window of eval_steps steps (the longest live member's)
  bool ragged = false;
  std::vector<int> m_nsteps, m_px, m_force;
  std::vector<double> m_nu;
  int eval_steps = 0;
  int* d_mstart = nullptr;   // device tables read by the kernels (Dev)
  int* d_mnt = nullptr;
  int* d_mpx = nullptr;
  int* d_mforce = nullptr;
  double* d_mnu = nullptr;
  int* d_kind = nullptr;     // member kernels, for re-making the multiplier
  double *d_param = nullptr, *d_table = nullptr;
  std::vector<int> h_kind;
  std::vector<double> h_param;
  const Ops* ops = nullptr;
  Dev dev{};
  std::vector<void*> allocs;
  unsigned long long bytes = 0;
  unsigned long long launches = 0;
  bool have_obs = false;
  bool have_adj = false;
  bool have_fwd = false;  // a stored forward (stage fields / checkpoints) is valid
  int nckpt = 0;          // checkpoints held (ckpt > 0)
  double2* ckpt_buf = nullptr;
  double sobolev = 0.0;   // lambda of the regularisation term of Eq. (4)
  // shell lists of the adjoint spectra (built on the first da_adjoint_spectra)
  int nshell = 0;
  int *shell_off = nullptr, *shell_mode = nullptr;
  double *shell_wgt = nullptr, *shell_scratch = nullptr;
  double2* w0 = nullptr;  // compact initial state kept for that term
  std::string err;
  // optimiser buffers (allocated on the first da_assimilate; blas.cuh)
  double* lb_V = nullptr;      // vector banks [5 + 2 (mem + 1)][B][n^2]
  double* lb_scal = nullptr;   // device scalars [B][SC_COUNT]
  double* lb_J = nullptr;      // costs [B]
  int* lb_iargs = nullptr;     // argument tables of the vector kernels
  double* lb_dargs = nullptr;
  double* lb_host = nullptr;   // pinned mirror of lb_scal and lb_J
  int mem = 0;
  // optimiser state per member (lbfgs.cu), freed by free_optimiser
  void* lb_state = nullptr;
  // CUDA-graph replay of da_cost_grad (captured per evaluation window)
  bool use_graph = false;
  struct CapturedEval {
    int steps;                    // the evaluation window it was captured for
    cudaGraphExec_t exec;
    unsigned long long launches;  // kernel nodes in it
  };
  std::vector<CapturedEval> cg_cache;  // newest last, at most kMaxCapturedEvals
  cudaStream_t gstream = nullptr;
  cudaEvent_t ev_in = nullptr, ev_out = nullptr;
  double *sbuf = nullptr, *gbuf = nullptr;
  // CUDA-graph replay of da_adjoint_spectra (captured per save_every and outputs)
  cudaGraphExec_t sp_exec = nullptr;
  unsigned long long sp_launches = 0;
  int sp_key = -1;
  double *sp_lbuf = nullptr, *sp_member = nullptr, *sp_mean = nullptr;
  // the batch's parts but the first run their RK stages on these streams (Parts)
  std::vector<cudaStream_t> side;
  std::vector<cudaEvent_t> side_done;
  cudaEvent_t side_go = nullptr;
  // event timing of one kernel class
  int timed_class = 0;
  std::vector<cudaEvent_t> ev;
  size_t ev_used = 0;
};

// Captured evaluations kept per context: one per evaluation window that a
// ragged batch's live members produce (a window is the longest live horizon).
constexpr size_t kMaxCapturedEvals = 16;

// Drops every captured evaluation (their kernel arguments or launch sequence
// changed).
inline void drop_graphs(da_ctx* c) {
  for (auto& g : c->cg_cache) cudaGraphExecDestroy(g.exec);
  c->cg_cache.clear();
}

// A captured sequence made ready for replay, and its replay.  A graph holds 2.5 KB
// of device memory a launch, which no context counts: where the device has not
// that much left, the evaluations captured before give theirs up, and if that is
// not enough *exec becomes NULL with DA_OK, and the caller launches directly.
da_status instantiate_graph(da_ctx* c, cudaGraph_t g, cudaGraphExec_t* exec);
da_status launch_graph(da_ctx* c, cudaGraphExec_t* exec, cudaStream_t st);

// Message of the last failed da_create (no context to hold it).
extern std::string g_create_error;

#define DA_TRY_CUDA(ctx, call)                                                                    \
  do {                                                                                            \
    cudaError_t e_ = (call);                                                                      \
    if (e_ != cudaSuccess) return fail((ctx), DA_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

inline da_status fail(da_ctx* c, da_status s, const std::string& msg) {
  if (c)
    c->err = msg;
  else
    g_create_error = msg;
  return s;
}

inline da_status check_launch(da_ctx* c, unsigned long long nlaunch = 1) {
  c->launches += nlaunch;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(c, DA_ECUDA, std::string("kernel launch: ") + cudaGetErrorString(e));
  return DA_OK;
}

// Brackets one launch of kernel class `cls` with events when that class is timed.
struct Timed {
  da_ctx* c;
  bool on;
  cudaStream_t st;
  Timed(da_ctx* c_, int cls, cudaStream_t s) : c(c_), on(c_->timed_class == cls), st(s) {
    if (!on) return;
    if (c->ev_used + 2 > c->ev.size()) {
      for (int i = 0; i < 256; ++i) {
        cudaEvent_t e;
        if (cudaEventCreate(&e) != cudaSuccess) {
          on = false;
          return;
        }
        c->ev.push_back(e);
      }
    }
    cudaEventRecord(c->ev[c->ev_used], st);
  }
  ~Timed() {
    if (!on) return;
    cudaEventRecord(c->ev[c->ev_used + 1], st);
    c->ev_used += 2;
  }
};

template <typename T>
da_status dalloc(da_ctx* c, T** p, size_t count) {
  *p = nullptr;
  if (count == 0) return DA_OK;
  void* v = nullptr;
  cudaError_t e = cudaMalloc(&v, count * sizeof(T));
  if (e != cudaSuccess) {
    cudaGetLastError();
    char buf[160];
    snprintf(buf, sizeof buf, "cudaMalloc of %.3f GB failed: %s", count * sizeof(T) / 1e9, cudaGetErrorString(e));
    return fail(c, DA_ENOMEM, buf);
  }
#ifdef DA_POISON_ALLOCATIONS
  // debugging builds: every fresh allocation holds NaNs (0xff bytes), so a
  // read of device memory that nothing wrote shows up as NaN in the results
  cudaMemset(v, 0xff, count * sizeof(T));
#endif
  c->allocs.push_back(v);
  c->bytes += count * sizeof(T);
  *p = static_cast<T*>(v);
  return DA_OK;
}

// Arrays of a context that share one device allocation (a cudaMalloc costs the
// host 0.1 ms): add each, then alloc sets their pointers, 256 bytes aligned.
class DeviceGroup {
 public:
  template <typename T>
  void add(T** p, size_t count) {
    *p = nullptr;
    parts_.push_back({reinterpret_cast<void**>(const_cast<std::remove_const_t<T>**>(p)), total_});
    bytes_ += count * sizeof(T);
    total_ += (count * sizeof(T) + 255) / 256 * 256;
  }
  da_status alloc(da_ctx* c) {
    char* base = nullptr;
    da_status r = dalloc(c, &base, total_);
    if (r) return r;
    c->bytes -= total_ - bytes_;  // what the arrays hold, not the padding
    for (auto& p : parts_) *p.first = base + p.second;
    return DA_OK;
  }

 private:
  std::vector<std::pair<void**, size_t>> parts_;
  size_t total_ = 0, bytes_ = 0;
};

// Whether global step k of the evaluation window can be an observation step
// of some member (every member's window is a whole number of observation
// intervals and ends with the evaluation's, so its observation steps fall on
// multiples of obs.every; the kernels find each member's slot).
inline bool obs_step_host(const da_ctx* c, int k) { return k % c->obs.every == 0; }

// Whether this context's windows run as single kernels (window.cuh): small
// grids and batches, unless a class of pass kernels is being timed.
inline bool whole_windows(const da_ctx* c) {
  return c->ops->window_fwd && c->B <= c->ops->window_batch && c->timed_class == 0;
}

// Parts that a batch's RK stages are split into, each a chain of kernels on a
// stream of its own: a pass ends with SMs that have nothing left to do while
// its last rows and columns finish, and begins with loads that nothing covers;
// the other parts' passes fill both.  From 512 threads an SM on: us for a stage
// pass of all members, replayed as a graph, in one part and in four: 256^2 on 128
// threads, batch 5 (539 threads an SM) 8.60 and 8.37, 7 9.93 and 9.68, 8 12.0 and
// 10.3, 16 20.6 and 16.0; on 64 threads batch 16 19.8 and 17.5; 512^2 batch 3 17.6
// and 15.8 (three parts); 128^2 batch 16 9.08 and 8.12; 1024^2 batch 2 49.5 and
// 43.4 (two parts).  Below the line there is little to gain and four times the
// launches: 512^2 batch 2 (431) 14.0 and 13.5, 128^2 batch 8 6.6 and 6.9.  Three
// parts: 0 to 4 % more (256^2 batch 7 9.88, 16 16.0); six: batch 7 9.4, but 16 17.3.
// These are replays: launched directly, a divided batch takes its launches' time
// where that is longer (256^2 batch 5, forward: 1600 launches in 4.2 ms, 10.5 us
// a pass of all members).
constexpr int kMaxParts = 4;
constexpr int kSplitThreads = 152 * 512;
inline int batch_parts(const Ops& o, int B) {
  return (long long)B * (o.n / 2) * o.threads >= kSplitThreads ? std::min(B, kMaxParts) : 1;
}

// The batch of a context in parts between fork and join: part p's stage passes
// are launched with dev(p) on stream(p).  The first part runs on the caller's
// stream, which the others wait for in fork and which waits for them in join,
// so that to the caller all of it is on that stream, captured or not.
class Parts {
 public:
  Parts(da_ctx* c, cudaStream_t st) : c_(c), st_(st), n_(c->timed_class == 0 ? batch_parts(*c->ops, c->B) : 1) {}
  ~Parts() { join(); }
  int count() const { return n_; }
  int begin(int p) const { return (int)((long long)c_->B * p / n_); }
  Dev dev(int p) const {
    Dev d = c_->dev;
    d.b0 = begin(p);
    d.early = n_ == 1;
    d.B = begin(p + 1) - d.b0;
    return d;
  }
  cudaStream_t stream(int p) const { return p == 0 ? st_ : c_->side[p - 1]; }
  da_status fork() {
    if (n_ == 1 || forked_) return DA_OK;
    DA_TRY_CUDA(c_, cudaEventRecord(c_->side_go, st_));
    forked_ = true;
    for (int p = 1; p < n_; ++p) DA_TRY_CUDA(c_, cudaStreamWaitEvent(stream(p), c_->side_go, 0));
    return DA_OK;
  }
  da_status join() {
    if (!forked_) return DA_OK;
    forked_ = false;
    cudaError_t e = cudaSuccess;
    for (int p = 1; p < n_; ++p) {
      cudaError_t ep = cudaEventRecord(c_->side_done[p - 1], stream(p));
      if (ep == cudaSuccess) ep = cudaStreamWaitEvent(st_, c_->side_done[p - 1], 0);
      if (e == cudaSuccess) e = ep;
    }
    DA_TRY_CUDA(c_, e);
    return DA_OK;
  }

 private:
  da_ctx* c_;
  cudaStream_t st_;
  int n_;
  bool forked_ = false;
};

// The RK stages of step k and of its adjoint, part by part (da_api.cu).
da_status forward_step(da_ctx* c, const Parts& parts, int k, int store_flag, int obs_flag);
da_status adjoint_step(da_ctx* c, const Parts& parts, int k, int flags);

// Sets the evaluation window for the members marked in `live` (all members
// with a non-empty window if live is NULL): eval_steps = the longest live
// window, each live member end-aligned in it, the others idle; uploads the
// start table of a ragged batch on stream st.  Homogeneous contexts always
// evaluate every member over the context's window.
da_status set_eval_window(da_ctx* c, const std::vector<char>* live, cudaStream_t st);

// Cost and gradient of the members marked in `live` (lbfgs.cu's evaluations).
da_status cost_grad_members(da_ctx* c, const double* s, double* J, double* grad_s, const std::vector<char>* live,
                            cudaStream_t st);

// Frees the optimiser state of lbfgs.cu (da_destroy).
void free_optimiser(da_ctx* c);

// Plan variant the autotuner chose for (n, batch) in this process, or 0
// (plans.cu).
int cached_plan(int n, int B);
