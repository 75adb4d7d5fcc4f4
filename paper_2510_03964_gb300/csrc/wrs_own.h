// Batches pushed through each stream's own kernel instead of the batched one.
#pragma once

#include <cuda_runtime.h>

#include "wrs_batch_kernel.cuh"
#include "wrs_internal.h"

// The streams' planned pushes and the graph that launches them as a whole.
struct wrs_own {
  wrs_pipe_plan plan[WRS_MAX_BATCH];
  cudaGraph_t graph;
  cudaGraphExec_t exec;
  cudaGraphNode_t node[WRS_MAX_BATCH];
  int nodes;
};

// Whether a batch outside the batched kernel's two families (other slot counts,
// the literal rule, mixed colours) is faster through the streams' own kernels.
// one_cta: the batched kernel's stages, sized for the largest stream, leave
// room for one CTA on an SM.
bool wrs_own_faster(int n, wrs_ctx* const* ctxs, bool fov, bool one_cta);
// Pushes the validated entries; WRS_OK, or WRS_ERR_CUDA with nothing launched.
int wrs_own_push(wrs_own* o, int n, wrs_ctx* const* ctxs, const BatchEntry* e, bool fov, int filter,
                 cudaStream_t st);
void wrs_own_drop(wrs_own* o);
