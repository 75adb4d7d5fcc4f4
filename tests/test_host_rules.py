"""Rules that the kernels and the host share, compiled for the host and run there (no GPU)."""
import ctypes as C
import glob
import os
import re
import subprocess

import numpy as np
import pytest

from paper_2510_03964_gb300 import build

SRC = r"""
#include <cuda_runtime.h>

// a runtime that refuses every launch, with the last-error state of the real one
static cudaError_t g_last = cudaSuccess;
static cudaError_t last_error() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
template <typename... T>
cudaError_t refuse(const T&...) {
  return g_last = cudaErrorInvalidConfiguration;
}
#define cudaGetLastError last_error
#define cudaLaunchKernelExC refuse

#include "wrs_batch_kernel.cuh"
#include "wrs_internal.h"

extern "C" void entries(int n, const unsigned* tile0, int tiles, const unsigned* order, int* entry) {
  BatchArgs* a = new BatchArgs();
  a->n = n;
  for (int i = 0; i < n; ++i) a->e[i].tile0 = tile0[i];
  int e = 0;
  for (int i = 0; i < tiles; ++i) entry[i] = e = entry_of(*a, order[i], e);
  delete a;
}

__global__ void nothing(int) {}

// a refused launch, then what the next launch's cudaGetLastError would report
extern "C" void refused(int* refusal, int* left) {
  *refusal = wrs_launch_early(nothing, dim3(1), 32, 0, nullptr, 0);
  *left = last_error();
}
"""

OWN = r"""
#include <cuda_runtime.h>

// a runtime that counts launches of kernels and graphs and refuses one of them
static int g_launches = 0, g_refused = -1;
static cudaError_t launch() { return g_launches++ == g_refused ? cudaErrorLaunchFailure : cudaSuccess; }
template <typename... T>
cudaError_t fine(const T&...) {
  return cudaSuccess;
}
template <typename... T>
cudaError_t launch_graph(const T&...) {
  return launch();
}
template <typename... T>
cudaError_t instantiate(cudaGraphExec_t* exec, const T&...) {
  *exec = reinterpret_cast<cudaGraphExec_t>(exec);
  return cudaSuccess;
}
#define cudaGetLastError fine
#define cudaStreamIsCapturing fine
#define cudaGraphCreate fine
#define cudaGraphAddKernelNode fine
#define cudaGraphAddDependencies fine
#define cudaGraphInstantiate instantiate
#define cudaGraphExecKernelNodeSetParams fine
#define cudaGraphExecDestroy fine
#define cudaGraphDestroy fine
#define cudaGraphLaunch launch_graph

#include "wrs_own.cu"

int wrs_cuda_fail(cudaError_t, const char*) { return WRS_ERR_CUDA; }
void wrs_pipe_shape(const wrs_ctx*, bool, int*, int*) {}
cudaError_t wrs_plan_pipe(const wrs::StreamDev&, const wrs::FrameDev&, bool, int, int, int, int, uint32_t*,
                          uint64_t, uint32_t, wrs_pipe_plan*) {
  return cudaSuccess;
}
cudaError_t wrs_plan_pipe_fov(const wrs::StreamDev&, const wrs::FrameDev&, const wrs::FovDev&, int, bool, int,
                              int, int, uint32_t*, uint64_t, uint32_t, wrs_pipe_plan*) {
  return cudaSuccess;
}
cudaError_t wrs_launch_plan(const wrs_pipe_plan&, cudaStream_t) { return launch(); }

// pushes a batch of n streams twice; the launch of that number is refused
extern "C" int push_twice(int n, int refuse, unsigned* frames) {
  static wrs_ctx ctx[WRS_MAX_BATCH];
  static BatchEntry entry[WRS_MAX_BATCH];
  static wrs_own own;
  wrs_ctx* ctxs[WRS_MAX_BATCH];
  own = wrs_own();
  for (int i = 0; i < n; ++i) {
    ctx[i] = wrs_ctx();
    ctxs[i] = &ctx[i];
  }
  g_launches = 0;
  g_refused = refuse;
  int rc = wrs_own_push(&own, n, ctxs, entry, false, 0, nullptr);
  if (rc == WRS_OK) rc = wrs_own_push(&own, n, ctxs, entry, false, 0, nullptr);
  for (int i = 0; i < n; ++i) frames[i] = ctx[i].t;
  return rc;
}

extern "C" int faster(int n, const int* w, const int* h, const int* K, const int* literal, const int* f16, int fov,
                      int one_cta) {
  static wrs_ctx ctx[WRS_MAX_BATCH];
  wrs_ctx* ctxs[WRS_MAX_BATCH];
  for (int i = 0; i < n; ++i) {
    ctxs[i] = &ctx[i];
    ctx[i].cfg.width = w[i];
    ctx[i].cfg.height = h[i];
    ctx[i].cfg.K = K[i];
    ctx[i].cfg.update_rule = literal[i] ? WRS_RULE_LITERAL : WRS_RULE_KEYS;
    ctx[i].cfg.color_fp16 = f16[i];
  }
  return wrs_own_faster(n, ctxs, fov != 0, one_cta != 0);
}
"""


def _compile(d, name, source):
    (d / f"{name}.cu").write_text(source)
    subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-O1", "-shared", "-cudart", "static",
                    "-o", str(d / f"{name}.so"), str(d / f"{name}.cu")], check=True)
    return C.CDLL(str(d / f"{name}.so"))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return _compile(tmp_path_factory.mktemp("rules"), "rules", SRC)


@pytest.fixture(scope="module")
def own(tmp_path_factory):
    return _compile(tmp_path_factory.mktemp("own"), "own", OWN)


@pytest.mark.parametrize("order", ["ascending", "descending", "shuffled"])
@pytest.mark.parametrize("sizes", [[1], [5, 1, 1, 7], [1, 300, 2, 2, 40, 1], [3] * 64])
def test_tile_entries_in_any_order(lib, sizes, order):
    """The work queue names a tile that no CTA has taken; which one is not part of its contract."""
    tile0 = np.cumsum([0] + sizes[:-1]).astype(np.uint32)
    tiles = np.arange(sum(sizes), dtype=np.uint32)
    if order == "descending":
        tiles = tiles[::-1].copy()
    elif order == "shuffled":
        np.random.default_rng(7).shuffle(tiles)
    got = np.full(tiles.size, -1, np.int32)
    lib.entries(len(sizes), tile0.ctypes.data_as(C.c_void_p), tiles.size, tiles.ctypes.data_as(C.c_void_p),
                got.ctypes.data_as(C.c_void_p))
    assert np.array_equal(got, np.repeat(np.arange(len(sizes)), sizes)[tiles])


def test_a_refused_launch_leaves_no_error_behind(lib):
    """The next launch of the thread must not be taken for refused: the host would not count a
    frame that the device has pushed."""
    refusal, left = C.c_int(0), C.c_int(-1)
    lib.refused(C.byref(refusal), C.byref(left))
    assert refusal.value != 0 and left.value == 0


def test_no_noncoherent_loads():
    """Kernels that start before the previous one of their stream has ended (grid_begin) read what
    that kernel writes: a load through the read-only path may pass the wait, and needs memory that
    stays as it is for as long as the kernel runs."""
    early = 0
    for path in glob.glob(os.path.join(build.CSRC, "*.cu*")):
        code = re.sub(r"/\*.*?\*/|//[^\n]*", "", open(path).read(), flags=re.S)
        early += len(re.findall(r"\bgrid_begin\(\);", code))
        assert not re.findall(r"__ldg\b|\bld\.global[\w.]*\.nc\b|\bconst\s+[\w:]+\s*\*\s*(?:const\s+)?__restrict__", code), path
    assert early >= 5


@pytest.mark.parametrize("n", [1, 2, 8])
def test_a_batch_through_own_kernels_is_launched_whole_or_not_at_all(own, n):
    frames = (C.c_uint * n)()
    assert own.push_twice(n, -1, frames) == 0 and list(frames) == [2] * n
    for refused in (0, 1):
        assert own.push_twice(n, refused, frames) != 0 and list(frames) == [refused] * n


def _mix(scale, K, literal=False, f16=True):
    """Two streams of each size, K and min(K, 4) slots; f16 None: colours mixed."""
    out = []
    for w, h in ((3840, 2160), (2064, 2208), (1440, 1600), (1920, 1080)):
        for i, k in enumerate((K, min(4, K))):
            out.append((round(w * scale / 4) * 4, round(h * scale), k, literal, f16 if f16 is not None else i == 0))
    return out


@pytest.mark.parametrize("streams,fov,one_cta,faster", [
    # measured, us: the batched kernel, a graph of own kernels
    (_mix(1.0, 1, True), 0, 0, True),                # 569, 295
    (_mix(0.347, 1, True), 0, 0, True),              # 78, 70
    (_mix(0.245, 1, True), 0, 0, False),             # 43, 47
    (_mix(0.49, 3), 0, 0, True),                     # 240, 219
    (_mix(0.347, 3), 0, 0, False),                   # 127, 132
    (_mix(1.0, 6, f16=False), 0, 0, True),           # 895, 862
    (_mix(0.49, 6, f16=False), 0, 0, False),         # 228, 247
    (_mix(0.49, 12), 0, 0, False),                   # 294, 300
    (_mix(0.347, 16), 0, 1, True),                   # 254, 229
    (_mix(1.0, 8, f16=None), 0, 0, False),           # 895, 899
    (_mix(1.0, 8, f16=None), 1, 0, True),            # 1085, 924
    (_mix(0.347, 1, True), 1, 0, False),             # 123, 130
    ([(3840, 2160, 16, 0, 1)] + [(256, 256, 16, 0, 1)] * 15, 0, 1, False),  # 695, 718
    ([(3840, 2160, 1, 1, 1)] + [(256, 256, 1, 1, 1)] * 15, 0, 0, True),     # 160, 130
    ([(3840, 2160, 1, 1, 1)] + [(256, 256, 1, 1, 1)] * 40, 0, 0, False),    # 191, 231
    ([(1920, 1080, 3, 0, 1)], 0, 0, True),           # 67, 50
])
def test_general_batches_take_the_measured_faster_form(own, streams, fov, one_cta, faster):
    cols = [(C.c_int * len(streams))(*[int(v) for v in col]) for col in zip(*streams)]
    assert bool(own.faster(len(streams), *cols, fov, one_cta)) == faster


def test_a_tuned_launch_shape_belongs_to_the_sources_it_was_tuned_with(tmp_path, monkeypatch):
    import torch
    from paper_2510_03964_gb300 import autotune
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda: "GB300")
    src = tmp_path / "kernel.cu"
    src.write_text("// one tile per CTA\n")
    monkeypatch.setattr(build, "CSRC", str(tmp_path))
    keys = [autotune._key("stream", [(64, 32, 4, 0)]), autotune._key("stream", [(64, 32, 4, 0)])]
    src.write_text("// a fixed deal\n")
    keys.append(autotune._key("stream", [(64, 32, 4, 0)]))
    assert keys[0] == keys[1] != keys[2]
