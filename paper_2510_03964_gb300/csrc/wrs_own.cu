// Batches pushed through each stream's own kernel (wrs_own.h): host code only.
#include "wrs_own.h"

#include <cstring>

// Microseconds per million pixels that a stream takes longer as a part of the
// batched kernel for all forms than through its own kernel, which holds one
// form only (unrolled for its slot count, fold inputs ahead, stages of its own
// size). Fitted to batches of eight streams (two each of 4K, VR, 1440 x 1600 and
// HD, of K and min(K, 4) slots, back to back) at 34.5 and 8.3 Mpx in all, for
// instance, batched and own kernels, us: literal FP16 569 and 295, 145 and 102;
// K = 3 FP16 953 and 770, 240 and 219; K = 6 FP32 895 and 862, 228 and 247; K = 8
// and 4 of different colours 895 and 899; foveated K = 6 FP16 1255 and 945.
static double own_gain(const wrs_config& c, bool fov, bool one_cta) {
  const bool f16 = c.color_fp16 != 0;
  if (c.update_rule == WRS_RULE_LITERAL) return fov ? 5.5 : 8.5;
  if (c.K >= 9) return fov ? 8.0 : 6.0;
  // own kernels keep two CTAs on an SM where one large stream leaves the
  // batched kernel one: K = 16 and 4 FP16 2004 and 1499 us
  const double alone = one_cta ? (fov ? 18.0 : 13.0) : 0.0;
  switch (c.K) {
    case 1: return alone + (fov ? 10.0 : 12.0);
    case 2: return alone + (fov ? 10.0 : f16 ? 10.0 : 9.0);
    case 3: return alone + (fov ? 11.0 : 6.0);
    case 4: return alone + (fov ? 8.0 : f16 ? 3.0 : 1.5);
    case 8: return alone + (fov ? 3.0 : 0.0);
    default: return alone + (fov ? 12.0 : f16 ? 7.0 : 3.0);
  }
}

bool wrs_own_faster(int n, wrs_ctx* const* ctxs, bool fov, bool one_cta) {
  double gain = 0.0;
  bool few = true;
  for (int i = 0; i < n; ++i) {
    const wrs_config& c = ctxs[i]->cfg;
    gain += 1e-6 * c.width * static_cast<double>(c.height) * own_gain(c, fov, one_cta);
    few = few && c.K <= 3;
  }
  // what each kernel after the first costs: its start and its last tiles (the
  // same fits; a 4K K = 16 stream and 15 of 256 x 256: 695 us batched, 718)
  return gain > (n - 1) * (fov ? 6.0 : few ? 4.5 : 5.5);
}

void wrs_own_drop(wrs_own* o) {
  if (o->exec) cudaGraphExecDestroy(o->exec);
  if (o->graph) cudaGraphDestroy(o->graph);
  o->exec = nullptr;
  o->graph = nullptr;
  o->nodes = 0;
}

// The kernel node parameters of a planned push.
static cudaKernelNodeParams node_params(wrs_pipe_plan& p) {
  cudaKernelNodeParams kp;
  std::memset(&kp, 0, sizeof kp);
  kp.func = const_cast<void*>(p.fn);
  kp.gridDim = dim3(p.grid);
  kp.blockDim = dim3(p.threads);
  kp.sharedMemBytes = static_cast<unsigned>(p.smem);
  kp.kernelParams = p.params;
  return kp;
}

// A graph of the plans as a chain of kernel nodes, each of which may start
// while the one before it ends (programmatic edges).
static cudaError_t build_graph(wrs_own* o, int n) {
  cudaError_t e = cudaGraphCreate(&o->graph, 0);
  for (int i = 0; e == cudaSuccess && i < n; ++i) {
    const cudaKernelNodeParams kp = node_params(o->plan[i]);
    e = cudaGraphAddKernelNode(&o->node[i], o->graph, nullptr, 0, &kp);
    if (e == cudaSuccess && i > 0) {
      cudaGraphEdgeData early;
      std::memset(&early, 0, sizeof early);
      early.from_port = cudaGraphKernelNodePortProgrammatic;
      early.type = cudaGraphDependencyTypeProgrammatic;
      e = cudaGraphAddDependencies(o->graph, &o->node[i - 1], &o->node[i], &early, 1);
    }
  }
  if (e == cudaSuccess) e = cudaGraphInstantiate(&o->exec, o->graph, 0);
  if (e == cudaSuccess) o->nodes = n;
  return e;
}

// One graph launch for the whole batch, so that nothing is launched on error
// (a launch per stream, refused half-way, left the streams before it
// advanced). On the GPU it takes the time of the single launches, and 2 us more
// for the smallest batches (HD literal 19.2 us alone, 22.6 as a graph: one
// stream is launched directly); on the host 36 us instead of 52 for eight
// streams.
int wrs_own_push(wrs_own* o, int n, wrs_ctx* const* ctxs, const BatchEntry* entries, bool fov, int filter,
                 cudaStream_t st) {
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < n; ++i) {
    const wrs_ctx* x = ctxs[i];
    const BatchEntry& in = entries[i];
    const bool f16 = x->cfg.color_fp16 != 0;
    int px, stages;
    wrs_pipe_shape(x, fov, &px, &stages);
    e = fov ? wrs_plan_pipe_fov(in.s, in.f, in.fv, filter, f16, stages, x->sms, x->pipe_ctas, in.status,
                                x->timeout_ns, x->test_extra_tx, &o->plan[i])
            : wrs_plan_pipe(in.s, in.f, f16, px, stages, x->sms, x->pipe_ctas, in.status, x->timeout_ns,
                            x->test_extra_tx, &o->plan[i]);
    if (e != cudaSuccess) return wrs_cuda_fail(e, "push_batch: launch shape");
  }
  // a capture takes the launches themselves (building a graph would end it) and
  // runs nothing before it is complete
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  e = cudaStreamIsCapturing(st, &capture);
  if (e != cudaSuccess) return wrs_cuda_fail(e, "push_batch: capture status");
  if (n == 1 || capture != cudaStreamCaptureStatusNone) {
    for (int i = 0; i < n && e == cudaSuccess; ++i) e = wrs_launch_plan(o->plan[i], st);
    if (e != cudaSuccess) return wrs_cuda_fail(e, "push_batch: launch");
  } else {
    bool ready = o->exec != nullptr && o->nodes == n;
    for (int i = 0; ready && i < n; ++i) {
      const cudaKernelNodeParams kp = node_params(o->plan[i]);
      ready = cudaGraphExecKernelNodeSetParams(o->exec, o->node[i], &kp) == cudaSuccess;
    }
    if (!ready) {
      (void)cudaGetLastError();  // an in-place update that was refused: built anew
      wrs_own_drop(o);
      e = build_graph(o, n);
      if (e != cudaSuccess) {
        wrs_own_drop(o);
        return wrs_cuda_fail(e, "push_batch: graph build");
      }
    }
    e = cudaGraphLaunch(o->exec, st);
    if (e != cudaSuccess) return wrs_cuda_fail(e, "push_batch: graph launch");
  }
  for (int i = 0; i < n; ++i) ctxs[i]->t += 1;
  return WRS_OK;
}
