// plans.cu -- FFT plan variants of the pass kernels and the autotuner
// (da_plan_count, da_get_plan, da_set_plan, da_autotune of include/da.h).
#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

#include "ctx.h"

// Plan variant chosen by the autotuner per (grid size, batch), for the
// contexts created afterwards in this process.
static std::mutex g_plan_mu;
static std::map<std::pair<int, int>, int> g_plan_choice;

int cached_plan(int n, int B) {
  std::lock_guard<std::mutex> lock(g_plan_mu);
  auto it = g_plan_choice.find({n, B});
  return it == g_plan_choice.end() ? 0 : it->second;
}

// Switches the context's pass kernels to plan variant v: launchers, twiddle
// tables, shared-memory attributes.  A captured graph holds the old
// kernels and is dropped; a stored forward trajectory is invalidated.
static da_status set_plan(da_ctx* c, int v) {
  const Ops* o = da::ops_for(c->n, v);
  if (!o) return fail(c, DA_EINVAL, "plan variant out of range (da_plan_count)");
  if (o == c->ops) return DA_OK;
  const std::vector<int4>& fxtw = o->fx_table();
  DA_TRY_CUDA(c, cudaMemcpy((void*)c->dev.fxtw, fxtw.data(), fxtw.size() * sizeof(int4), cudaMemcpyHostToDevice));
  DA_TRY_CUDA(c, o->setup());
  c->ops = o;
  drop_graphs(c);
  if (c->sp_exec) {
    cudaGraphExecDestroy(c->sp_exec);
    c->sp_exec = nullptr;
    c->sp_key = -1;
  }
  c->have_fwd = false;
  return DA_OK;
}

extern "C" int da_plan_count(int n) { return da::ops_for(n) ? da::plan_count(n) : 0; }

extern "C" int da_get_plan(const da_ctx* c) { return c ? c->ops->variant : -1; }

extern "C" da_status da_plan_flops(int n, int variant, double* inverse, double* forward) {
  const Ops* o = da::ops_for(n, variant);
  if (!o) return fail(nullptr, DA_EINVAL, "unsupported size or plan variant (da_plan_count)");
  if (!inverse || !forward) return fail(nullptr, DA_EINVAL, "inverse and forward must not be NULL");
  *inverse = o->flops_inverse;
  *forward = o->flops_forward;
  return DA_OK;
}

extern "C" da_status da_set_plan(da_ctx* c, int variant) {
  if (!c) return fail(c, DA_EINVAL, "ctx must not be NULL");
  // the twiddle tables and the launchers change under any work in flight
  DA_TRY_CUDA(c, cudaDeviceSynchronize());
  return set_plan(c, variant);
}

// Zeroes the working state that the tuning passes run over.
static da_status clear_state(da_ctx* c, cudaStream_t st) {
  const Dev& d = c->dev;
  const size_t comp = (size_t)c->B * c->ops->Kr * c->ops->Kc * sizeof(double2);
  const size_t mixed = (size_t)c->B * 2 * c->n * c->ops->Kc * sizeof(double2);
  for (void* p : {(void*)d.W, (void*)d.Acc, (void*)d.Y, (void*)d.KB, (void*)d.LamBar, (void*)d.Sum})
    DA_TRY_CUDA(c, cudaMemsetAsync(p, 0, comp, st));
  DA_TRY_CUDA(c, cudaMemsetAsync(d.Mx, 0, mixed, st));
  DA_TRY_CUDA(c, cudaMemsetAsync(d.Mn, 0, mixed, st));
  DA_TRY_CUDA(c, cudaMemsetAsync(d.eX, 0, (size_t)c->B * 2 * c->ops->Kc * sizeof(int), st));
  DA_TRY_CUDA(c, cudaMemsetAsync(d.eN, 0, (size_t)c->B * c->n * sizeof(int), st));
  return DA_OK;
}

// A state and an adjoint field of ordinary size for the tuning passes, real and
// even in k, slow enough (velocities of 1e-3) to stay so over any tuning run:
// values that are zero or not finite take another path in the conversions.
__global__ void k_tuning_fields(double2* W, double2* LamBar, double amp, int Kr, int Kc) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Kr * Kc; i += gridDim.x * blockDim.x) {
    const int kx = i / Kr, r = i - kx * Kr, ky = r < Kc ? r : r - Kr;
    const double2 v = make_double2(i == 0 ? 0.0 : amp / (1 + kx * kx + ky * ky), 0.0);
    W[(size_t)blockIdx.y * Kr * Kc + i] = LamBar[(size_t)blockIdx.y * Kr * Kc + i] = v;
  }
}

// `steps` RK steps of the context's batch as an evaluation runs them (its
// route, its parts; forward, and the adjoint when the context stores stage
// fields), in windows that the store holds.
static da_status tuning_steps(da_ctx* c, int steps, cudaStream_t st) {
  const Ops* o = c->ops;
  const Dev& d = c->dev;
  const bool store = d.traj != nullptr, whole = whole_windows(c);
  const int most = store ? d.traj_steps : steps;
  Parts parts(c, st);
  da_status r = DA_OK;
  for (int i = 0; i < steps; i += most) {
    const int n = std::min(most, steps - i);
    if (whole) {
      o->window_fwd(d, 0, n, store ? da::W_STORE : 0, st);
    } else {
      o->state_cols(d, st);
      if ((r = parts.fork())) return r;
      for (int k = 0; k < n; ++k)
        if ((r = forward_step(c, parts, k, store ? da::F_STORE : 0, 0))) return r;
      if ((r = parts.join())) return r;
    }
    if ((r = check_launch(c))) return r;
    if (!store) continue;
    o->adj_init(d, da::INIT_LAMBAR, st);
    if (whole) {
      o->window_adj(d, n, 0, 0, st);
    } else {
      if ((r = parts.fork())) return r;
      for (int k = n - 1; k >= 0; --k)
        if ((r = adjoint_step(c, parts, k, 0))) return r;
      if ((r = parts.join())) return r;
    }
    if ((r = check_launch(c, whole ? 2 : 1))) return r;
  }
  return DA_OK;
}

// The tuning steps as a graph that is on the device, captured on *cap_stream
// (made on first use); *exec stays NULL where another thread's device-wide calls
// broke every capture (da_cost_grad's note on that) or the device has no memory
// for it.
static da_status capture_tuning(da_ctx* c, int steps, cudaStream_t st, cudaStream_t* cap_stream, cudaGraphExec_t* exec,
                                unsigned long long* launches) {
  if (!*cap_stream) DA_TRY_CUDA(c, cudaStreamCreateWithFlags(cap_stream, cudaStreamNonBlocking));
  const cudaStream_t cap = *cap_stream;
  for (int attempt = 0; attempt < 4; ++attempt) {
    cudaGraph_t g = nullptr;
    const unsigned long long l0 = c->launches;
    DA_TRY_CUDA(c, cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal));
    da_status r = tuning_steps(c, steps, cap);
    cudaError_t e = cudaStreamEndCapture(cap, &g);
    *launches = c->launches - l0;
    c->launches = l0;
    if (!r && e == cudaSuccess) {
      r = instantiate_graph(c, g, exec);
      cudaGraphDestroy(g);
      if (*exec && cudaGraphUpload(*exec, st) != cudaSuccess) {
        cudaGetLastError();
        cudaGraphExecDestroy(*exec);
        *exec = nullptr;
      }
      return r;
    }
    if (g) cudaGraphDestroy(g);
    cudaGetLastError();
    if (e != cudaErrorStreamCaptureInvalidated && (r != DA_ECUDA || e == cudaSuccess))
      return r ? r : fail(c, DA_ECUDA, std::string("graph capture: ") + cudaGetErrorString(e));
  }
  return DA_OK;
}

// Milliseconds of a step on the context's plan, replayed as a graph of at most
// 32 steps unless whole windows run in one kernel.  Launched directly, the 16
// launches of a step (64 of a batch in four parts) would be what is timed, 2.5
// us each, wherever a pass takes less: 256^2, batch 5, 0.173 ms a step where
// evaluations take 0.140, and batch 2 0.147 where they take 0.105.
static da_status time_plan(da_ctx* c, int steps, cudaStream_t st, cudaStream_t* cap, cudaEvent_t e0, cudaEvent_t e1,
                           float* ms) {
  cudaGraphExec_t exec = nullptr;
  unsigned long long launches = 0;
  const int part = std::min(steps, 32), parts = (steps + part - 1) / part;
  da_status r = tuning_steps(c, 1, st);  // warm-up
  if (r) return r;
  if (!whole_windows(c) && (r = capture_tuning(c, part, st, cap, &exec, &launches))) return r;
  auto run = [&]() -> da_status {
    DA_TRY_CUDA(c, cudaEventRecord(e0, st));
    for (int j = 0; j < parts; ++j) {
      da_status q = exec ? launch_graph(c, &exec, st) : DA_OK;
      if (exec) c->launches += launches;
      else if (!q) q = tuning_steps(c, part, st);
      if (q) return q;
    }
    DA_TRY_CUDA(c, cudaEventRecord(e1, st));
    DA_TRY_CUDA(c, cudaEventSynchronize(e1));
    DA_TRY_CUDA(c, cudaEventElapsedTime(ms, e0, e1));
    *ms /= part * parts;
    return DA_OK;
  };
  r = run();
  if (exec) cudaGraphExecDestroy(exec);
  return r;
}

extern "C" da_status da_autotune(da_ctx* c, int steps, int* chosen, double* ms_per_step) {
  if (!c) return fail(c, DA_EINVAL, "ctx must not be NULL");
  if (steps < 1) return fail(c, DA_EINVAL, "steps must be >= 1");
  // the tuning passes overwrite the working state: let every evaluation in
  // flight on any stream finish first
  DA_TRY_CUDA(c, cudaDeviceSynchronize());
  // the device is idle now; the tuning runs on the legacy default stream, which
  // cannot be captured: that takes a stream of its own (cap)
  cudaStream_t st = nullptr, cap = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  da_status r = DA_OK;
  int best = 0;
  float best_ms = 0.f;
  auto cuda = [&](cudaError_t e, const char* what) {
    if (r == DA_OK && e != cudaSuccess) r = fail(c, DA_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
  };
  cuda(cudaEventCreate(&e0), "event");
  cuda(cudaEventCreate(&e1), "event");
  // every member works, whatever windows a ragged batch holds, on the routes
  // that evaluations take, whatever is being timed
  const int ragged = c->dev.ragged, timed = c->timed_class;
  c->dev.ragged = 0;
  c->timed_class = 0;
  c->dev.seg0 = 0;
  const int modes = c->ops->Kr * c->ops->Kc;
  for (int v = 0; r == DA_OK && v < da::plan_count(c->n); ++v) {
    if ((r = set_plan(c, v))) break;
    if ((r = clear_state(c, st))) break;
    k_tuning_fields<<<dim3((modes + 255) / 256, c->B), 256, 0, st>>>(c->dev.W, c->dev.LamBar, 1e-3 * c->n * c->n,
                                                                  c->ops->Kr, c->ops->Kc);
    float ms = 0.f;
    if ((r = check_launch(c))) break;
    if ((r = time_plan(c, steps, st, &cap, e0, e1, &ms))) break;
    if (ms_per_step) ms_per_step[v] = ms;
    if (v == 0 || ms < best_ms) {
      best = v;
      best_ms = ms;
    }
  }
  c->dev.ragged = ragged;
  c->timed_class = timed;
  if (r == DA_OK) r = set_plan(c, best);
  if (r == DA_OK) r = clear_state(c, st);
  if (r == DA_OK) cuda(cudaStreamSynchronize(st), "stream synchronize");
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  if (cap) cudaStreamDestroy(cap);
  if (r) return r;
  {
    std::lock_guard<std::mutex> lock(g_plan_mu);
    g_plan_choice[{c->n, c->B}] = best;
  }
  c->have_fwd = false;
  if (chosen) *chosen = best;
  return DA_OK;
}
