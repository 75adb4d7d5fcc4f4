// Batches pushed through each stream's own kernel (wrs_own.h): host code only.
#include "wrs_own.h"

#include <cstring>

// The streams' bytes per push (mean over the batch: frame, output, sums and
// slots) from which their own kernels are taken: the general batched kernel
// lacks the forms for one, two and up to 8 slots, but a kernel more per stream
// costs about 4 us. Eight streams (two each of 4K, VR, 1440 x 1600 and HD),
// batched kernel and own kernels: literal 551 and 310 us, K = 1 751 and 381,
// K = 3 939 and 774, K = 6 928 and 828; with an eighth of the pixels K = 1 100
// and 80, K = 3 125 and 132, K = 6 127 and 145.
constexpr int64_t kOwnKernelBytes = 112ll << 20, kOwnKernelBytesFew = 24ll << 20;

bool wrs_own_faster(int n, wrs_ctx* const* ctxs) {
  int64_t bytes = 0;
  int most_slots = 0;
  for (int i = 0; i < n; ++i) {
    const wrs_config& c = ctxs[i]->cfg;
    if (c.K > most_slots) most_slots = c.K;
    bytes += static_cast<int64_t>(c.width) * c.height * (40 + c.K * (c.color_fp16 ? 14 : 20));
  }
  return bytes >= (most_slots <= 2 ? kOwnKernelBytesFew : kOwnKernelBytes) * n;
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
