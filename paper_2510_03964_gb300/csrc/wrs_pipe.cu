// Pipelined persistent form of the fused update + resolve (sm_103a).
//
// The CTAs that fit on the GPU take the image's tiles of T = 256 * PX pixels in
// ascending order from the hardware's work queue (request_tile). A copying warp
// streams the planes a tile needs (frame RGB, W, P, the K key planes and, for
// the fused resolve, the K slot records) into a ring of S shared-memory stages with 1-D bulk asynchronous copies
// (cp.async.bulk) that complete on one transaction-count "full" mbarrier per
// stage; a drawing warp adds the tile's uniforms (one Philox block per 4
// pixels). With one warp doing both, the draw (about 220 dependent
// instructions a tile) held back the copies: 4K K = 8 FP16 244 -> 238 us, 4K
// literal rule 73.8 -> 69.7 us, 8-stream FP16 batch 990 -> 932 us when the
// drawing moved to its own warp. Eight consumer warps compute each
// landed tile from shared memory with the plain kernel's arithmetic
// (push_staged: bit-identical results), write straight to global memory and free
// the stage through its "empty" mbarrier. No block-wide barrier sits inside
// the loop.
//
// Every wait is bounded by %globaltimer. A wait that runs out records
// WRS_ERR_TIMEOUT in the stream's status word, waits (again bounded) for the
// copies this CTA still has in flight, and returns; the host reads the word
// with wrs_check_status.
#include <cuda_runtime.h>

#include <mutex>

#include "wrs.h"
#include "wrs_async.cuh"
#include "wrs_device.cuh"
#include "wrs_internal.h"

using wrs::FovDev;
using wrs::FrameDev;
using wrs::StageLayout;
using wrs::StreamDev;

namespace {

using PipeArgs = wrs_pipe_args;

constexpr int kConsumerWarps = 8;
// FOVF >= 0: the frame is not copied but foveated from `fv` with filter FOVF
// (WRS_FILTER_*) by two more warps; FOVF < 0: `fv` is unused.
constexpr int producers(int fovf) { return fovf >= 0 ? 2 + wrs::kFovWarps : 2; }
constexpr int pipe_threads(int fovf) { return (kConsumerWarps + producers(fovf)) * 32; }

// Warp-specialised: warps 0..7 compute (consumers, PX pixels per thread), warp 8
// issues copies and warp 9 draws uniforms. They meet only at the per-stage
// full/empty barriers, never at a block-wide barrier.
// Resident CTAs per SM the compiler is asked to fit: three for one or two
// slots and one pixel per thread and for the literal rule at up to two (their
// stages are small, and the extra warps hide the per-pixel arithmetic's
// latency: 4K literal rule, 24 against 16 consumer warps per SM, 68.7 -> 63.9
// us), two for one pixel per thread, else one.
template <int KT, int PX, bool LIT, int FOVF>
constexpr int pipe_min_blocks() {
  if (FOVF >= 0) return 2;
  if (LIT ? PX <= 2 : (KT == 1 || KT == 2) && PX == 1) return 3;
  return PX == 1 ? 2 : 1;
}

template <int KT, bool F16, int PX, bool LIT, int FOVF = -1>
__global__ void __launch_bounds__(pipe_threads(FOVF), pipe_min_blocks<KT, PX, LIT, FOVF>())
    pipe_kernel(const __grid_constant__ StreamDev s, const __grid_constant__ FrameDev f,
                const PipeArgs a, const __grid_constant__ FovDev fv) {
  extern __shared__ __align__(128) uint8_t smem[];
  constexpr int T = kConsumerWarps * 32 * PX;
  constexpr int cs = F16 ? 2 : 4;
  const int K = KT > 0 ? KT : s.K;
  const bool resolve = a.resolve != 0;
  const StageLayout L = wrs::stage_layout(T, K, cs, resolve, LIT);
  const wrs::Ring r = wrs::make_ring(smem, L.bytes, T, a.stages, a.queue != 0, f.fov != nullptr);
  const int tid = threadIdx.x;
  const int warp = tid >> 5;
  const int lane = tid & 31;
  __shared__ uint32_t failed;
  if (warp == 0) wrs::init_ring(r, kConsumerWarps, producers(FOVF), lane);
  wrs::grid_begin();
  // not for grids that fit (their planes are in the L2 already: 256 x 256 K = 4
  // 4.5 -> 4.7 us with it) nor for one or two slots (4K literal rule +0.4%)
  if (KT != 1 && KT != 2 && r.queue && warp == kConsumerWarps)
    wrs::prefetch_tile<T>(s, f, K, cs, resolve, static_cast<int64_t>(blockIdx.x) * T, lane);
  if (tid == 0) {
    // a wait of an earlier push gave up and the host has not yet seen it: the
    // reservoirs are undefined, so leave them (and the waits) alone
    failed = *reinterpret_cast<volatile const uint32_t*>(a.status);
  }
  __syncthreads();
  if (failed != 0) return;

  int issued = 0;
  int replaced = 0;
  if (warp == kConsumerWarps) {
    issued = wrs::produce<true>(r, a.timeout_ns, lane,
                                [&](uint32_t tile, uint8_t* st, float*, uint64_t* full, int ln) {
                                  wrs::issue_tile_copies<T, true>(s, f, K, cs, resolve, L, st, full,
                                                            static_cast<int64_t>(tile) * T, a.extra_tx,
                                                            ln, FOVF < 0, r.stage_bytes);
                                });
  } else if (warp == kConsumerWarps + 1) {
    wrs::produce<false>(r, a.timeout_ns, lane,
                        [&](uint32_t tile, uint8_t*, float* u, uint64_t* full, int ln) {
                          wrs::draw_tile<T>(s, f, static_cast<int64_t>(tile) * T, u, full, ln);
                        });
  } else if (FOVF >= 0 && warp >= kConsumerWarps + 2) {
    if constexpr (FOVF >= 0)
      wrs::produce<false>(r, a.timeout_ns, lane,
                          [&](uint32_t tile, uint8_t* st, float*, uint64_t* full, int ln) {
                            wrs::foveate_tile<FOVF>(s, f, fv, tile, st, full, warp - kConsumerWarps - 2, ln);
                          });
  } else {
    constexpr int KM = wrs::FoldCap<KT>::value;
    const float d_f = wrs::fovea_density(s);
    wrs::TilePx<KM> px;
    wrs::consume(
        r, a.timeout_ns, lane,
        [&](uint32_t tile) {
          px.p = tile * T + tid * PX;
          wrs::row_col(s, static_cast<int>(px.p), px.y, px.x);
          wrs::tile_ahead<KM, PX, (KT > 2 || KT == wrs::kUpTo8)>(s, f, px);
        },
        [&](uint8_t* st, const float* u) {
          replaced += wrs::compute_tile<KT, F16, PX, T, LIT>(s, f, st, u, px, d_f, tid);
        });
  }
  __syncthreads();
  if (warp < kConsumerWarps) wrs::add_warp_count(s.replacements, replaced, lane);
  if (wrs::flag_raised(r)) {
    if (warp == kConsumerWarps) wrs::drain(r, issued, a.timeout_ns);
    if (tid == 0) atomicExch(a.status, static_cast<uint32_t>(WRS_ERR_TIMEOUT));
  }
}

const FovDev kNoSource{};

template <int KT, bool F16, int PX, bool LIT = false, int FOVF = -1>
cudaError_t plan_pipe_t(const StreamDev& s, const FrameDev& f, PipeArgs a, int sms, int ctas_per_sm,
                        wrs_pipe_plan* plan, const FovDev& fv = kNoSource) {
  constexpr int T = kConsumerWarps * 32 * PX;
  const StageLayout L = wrs::stage_layout(T, s.K, F16 ? 2 : 4, a.resolve != 0, LIT);
  if (f.fov != nullptr) a.stages = wrs::stages_with_maps(L.bytes, T, a.stages);
  size_t smem = wrs::ring_bytes(L.bytes, T, a.stages, f.fov != nullptr);
  // per instantiation and device: the whole budget allowed once, and how many
  // CTAs of the last shared-memory size fit on the device
  struct Fit {
    size_t smem = 0;
    int ctas = 0;
  };
  static Fit fits[64];
  static std::mutex lock;
  const auto kernel = pipe_kernel<KT, F16, PX, LIT, FOVF>;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  int fit;
  {
    std::lock_guard<std::mutex> hold(lock);
    Fit& known = fits[dev];
    if (known.smem == 0) {
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSmemBudget));
      if (e != cudaSuccess) return e;
    }
    if (known.smem != smem) {
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&known.ctas, kernel, pipe_threads(FOVF), smem);
      if (e != cudaSuccess) return e;
      known.smem = smem;
    }
    fit = known.ctas;
  }
  if (fit < 1) return cudaErrorInvalidConfiguration;
  // fewer CTAs per SM than fit: a larger shared-memory request keeps the others out
  if (ctas_per_sm > 0 && ctas_per_sm < fit) {
    smem = wrs::smem_for_ctas(smem, ctas_per_sm);
    fit = ctas_per_sm;
  }
  const int64_t tiles = (static_cast<int64_t>(s.hw) + T - 1) / T;
  a.queue = tiles > static_cast<int64_t>(fit) * sms ? 1 : 0;
  plan->fn = reinterpret_cast<const void*>(kernel);
  plan->grid = static_cast<unsigned>(tiles);
  plan->threads = pipe_threads(FOVF);
  plan->smem = smem;
  plan->a = a;
  plan->params[0] = const_cast<StreamDev*>(&s);
  plan->params[1] = const_cast<FrameDev*>(&f);
  plan->params[2] = &plan->a;
  plan->params[3] = const_cast<FovDev*>(&fv);
  return cudaSuccess;
}

// The foveating form: one pixel per thread (the default tile), K = 4, 8 or
// any other through the generic instantiation, and the literal rule.
template <bool F16, int FILTER>
cudaError_t plan_pipe_fov_k(const StreamDev& s, const FrameDev& f, const FovDev& fv,
                            const PipeArgs& a, int sms, int ctas, wrs_pipe_plan* plan) {
  if (s.literal) return plan_pipe_t<1, F16, 1, true, FILTER>(s, f, a, sms, ctas, plan, fv);
  switch (s.K) {
    case 4: return plan_pipe_t<4, F16, 1, false, FILTER>(s, f, a, sms, ctas, plan, fv);
    case 8: return plan_pipe_t<8, F16, 1, false, FILTER>(s, f, a, sms, ctas, plan, fv);
    default:
      if (s.K <= 8) return plan_pipe_t<wrs::kUpTo8, F16, 1, false, FILTER>(s, f, a, sms, ctas, plan, fv);
      return plan_pipe_t<0, F16, 1, false, FILTER>(s, f, a, sms, ctas, plan, fv);
  }
}

template <int KT, bool F16, bool LIT = false>
cudaError_t plan_pipe_px(const StreamDev& s, const FrameDev& f, const PipeArgs& a, int px, int sms, int ctas,
                         wrs_pipe_plan* plan) {
  switch (px) {
    case 4: return plan_pipe_t<KT, F16, 4, LIT>(s, f, a, sms, ctas, plan);
    case 2: return plan_pipe_t<KT, F16, 2, LIT>(s, f, a, sms, ctas, plan);
    default: return plan_pipe_t<KT, F16, 1, LIT>(s, f, a, sms, ctas, plan);
  }
}

template <bool F16>
cudaError_t plan_pipe_k(const StreamDev& s, const FrameDev& f, const PipeArgs& a, int px, int sms, int ctas,
                        wrs_pipe_plan* plan) {
  if (s.literal) return plan_pipe_px<1, F16, true>(s, f, a, px, sms, ctas, plan);
  switch (s.K) {
    case 1: return plan_pipe_px<1, F16>(s, f, a, px, sms, ctas, plan);
    case 2: return plan_pipe_px<2, F16>(s, f, a, px, sms, ctas, plan);
    case 4: return plan_pipe_px<4, F16>(s, f, a, px, sms, ctas, plan);
    case 8: return plan_pipe_px<8, F16>(s, f, a, px, sms, ctas, plan);
    default:
      // other slot counts: up to 8 unrolled with a test per slot, 9 to 16
      // through run-time loops (184 x 143, K = 6: 4.8 us against 10.6)
      if (px == 1 && s.K <= 8) return plan_pipe_t<wrs::kUpTo8, F16, 1>(s, f, a, sms, ctas, plan);
      return plan_pipe_px<0, F16>(s, f, a, px, sms, ctas, plan);
  }
}

}  // namespace

// Shared memory one CTA of the pipelined kernel needs (the literal rule: less).
size_t wrs_pipe_smem_bytes(int K, bool f16, int px, int stages, bool resolve) {
  const int T = kConsumerWarps * 32 * px;
  return wrs::ring_bytes(wrs::stage_layout(T, K, f16 ? 2 : 4, resolve, false).bytes, T, stages, false);
}

// Frames the bulk copies can read: rows without padding, 16-byte aligned.
// Threads with several pixels need them in one row (width % 4 == 0); one
// pixel per thread takes any width. Against the plain kernel, which odd widths
// took before, the staged update of a 1365 x 767 K = 4 stream with flushes
// needs 33.4 us instead of 38.5.
bool wrs_pipe_supported(const wrs_ctx* x, const float* frame, int64_t pitch, const float* out) {
  const auto al = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
  return pitch == 3 * static_cast<int64_t>(x->cfg.width) && al(frame) && (out == nullptr || al(out));
}

cudaError_t wrs_plan_pipe_fov(const StreamDev& s, const FrameDev& f, const FovDev& fv, int filter,
                              bool f16, int stages, int sms, int ctas_per_sm, uint32_t* status,
                              uint64_t timeout_ns, uint32_t extra_tx, wrs_pipe_plan* plan) {
  PipeArgs a;
  a.stages = stages;
  a.resolve = (f.out != nullptr || s.bias == 2) ? 1 : 0;  // records: resolve or Delta L
  a.status = status;
  a.timeout_ns = timeout_ns;
  a.extra_tx = extra_tx;
  if (filter == WRS_FILTER_BOX)
    return f16 ? plan_pipe_fov_k<true, WRS_FILTER_BOX>(s, f, fv, a, sms, ctas_per_sm, plan)
               : plan_pipe_fov_k<false, WRS_FILTER_BOX>(s, f, fv, a, sms, ctas_per_sm, plan);
  return f16 ? plan_pipe_fov_k<true, WRS_FILTER_BILINEAR>(s, f, fv, a, sms, ctas_per_sm, plan)
             : plan_pipe_fov_k<false, WRS_FILTER_BILINEAR>(s, f, fv, a, sms, ctas_per_sm, plan);
}

cudaError_t wrs_plan_pipe(const StreamDev& s, const FrameDev& f, bool f16, int px, int stages,
                          int sms, int ctas_per_sm, uint32_t* status, uint64_t timeout_ns,
                          uint32_t extra_tx, wrs_pipe_plan* plan) {
  PipeArgs a;
  a.stages = stages;
  a.resolve = (f.out != nullptr || s.bias == 2) ? 1 : 0;  // records: resolve or Delta L
  a.status = status;
  a.timeout_ns = timeout_ns;
  a.extra_tx = extra_tx;
  return f16 ? plan_pipe_k<true>(s, f, a, px, sms, ctas_per_sm, plan)
             : plan_pipe_k<false>(s, f, a, px, sms, ctas_per_sm, plan);
}

cudaError_t wrs_launch_plan(const wrs_pipe_plan& plan, cudaStream_t st) {
  return wrs_launch_early_params(plan.fn, dim3(plan.grid), plan.threads, plan.smem, st,
                                 const_cast<void**>(plan.params));
}
