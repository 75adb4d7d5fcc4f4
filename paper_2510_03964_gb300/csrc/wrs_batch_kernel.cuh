// The batched persistent kernel (template), shared by the translation unit of
// the plain batches (wrs_batch.cu, frames in memory) and that of the
// foveating batches (wrs_batch_fov.cu, frames foveated on read), which each
// instantiate their own variants.
#pragma once

#include <cuda_runtime.h>

#include "wrs.h"
#include "wrs_async.cuh"
#include "wrs_device.cuh"
#include "wrs_fov.cuh"

using wrs::FrameDev;
using wrs::StageLayout;
using wrs::StreamDev;

// One stream of a batch and its frame.
struct BatchEntry {
  StreamDev s;
  FrameDev f;
  wrs::FovDev fv;  // the stream's rendered image and mip levels (foveating batches only)
  uint32_t* status;
  uint32_t tile0;  // first global tile of this stream
  int code;    // arithmetic variant: 0 K=4 f16, 1 K=8 f16, 2 K=4 f32, 3 K=8 f32, 4 any K f16,
               // 5 any K f32, 6 literal f16, 7 literal f32
};

namespace {

constexpr int kMaxBatch = WRS_MAX_BATCH;

// The slot records are staged when the fused resolve needs them or the full
// temporal bias forms the history's resolved colour from them.
__device__ __forceinline__ bool stage_records(const BatchEntry& e) {
  return e.f.out != nullptr || e.s.bias == 2;
}

struct BatchArgs {
  int n;
  int queue;             // more tiles than CTAs that fit: see Ring::queue
  int maps;              // some frame has a flush map: see Ring
  int stages;
  uint32_t stage_bytes;  // largest stage of any stream in the batch
  uint64_t timeout_ns;
  uint32_t extra_tx;     // added to the expected bytes: > 0 only to test the timeout path
  BatchEntry e[kMaxBatch];
};
// kernel parameters may take up to 32764 bytes on sm_70 and later (CUDA 12.1+)
static_assert(sizeof(BatchArgs) <= 32000, "batch descriptor too large for a kernel parameter");

// The entry (stream) of global tile g: the last entry with tile0 <= g, searched
// from the entry `e` of the warp's previous tile. The work queue hands tiles
// out in ascending order (a few steps per stream boundary instead of a search
// per tile), but its contract only names some tile not yet taken, so a lower
// one is looked for as well.
__host__ __device__ __forceinline__ int entry_of(const BatchArgs& a, uint32_t g, int e) {
  while (e > 0 && a.e[e].tile0 > g) --e;
  while (e + 1 < a.n && a.e[e + 1].tile0 <= g) ++e;
  return e;
}

__device__ __forceinline__ bool entry_f16(const BatchEntry& e) {
  return e.code == 0 || e.code == 1 || e.code == 4 || e.code == 6;
}

constexpr int kConsumerWarps = 8;
// the copying and the drawing warp, and two that foveate frames on read
constexpr int batch_producers(bool fov) { return fov ? 2 + wrs::kFovWarps : 2; }
constexpr int batch_threads(bool fov) { return (kConsumerWarps + batch_producers(fov)) * 32; }

// Adds a warp's running count of replacements in entry ei to the CTA's
// per-stream total and clears it: once per stream a warp leaves, not per tile.
__device__ __forceinline__ void flush_count(unsigned long long* replaced_s, int ei, int& count,
                                            int lane) {
  const unsigned c = __reduce_add_sync(0xffffffffu, static_cast<unsigned>(count));
  if (lane == 0 && c != 0) atomicAdd(&replaced_s[ei], static_cast<unsigned long long>(c));
  count = 0;
}

// Arithmetic families: a batch whose streams all use FP16 colour with K = 4
// or 8 (the serving mix) or all FP32 colour with K = 4 or 8 gets a kernel
// holding only those two variants; any other mix gets the kernel with all.
constexpr int kFamF16K48 = 0, kFamF32K48 = 1, kFamAll = 2;

// One tile of entry e. The fold inputs are held for up to 8 slots
// whatever the stream's K (no narrowed copy, which would have to live in local
// memory); the generic-K and literal forms load their own.
template <int KT, bool F16, int PX, int T, bool LIT>
__device__ __forceinline__ int tile(const BatchEntry& e, uint8_t* st, const float* u,
                                    const wrs::TilePx<8>& px, float d_f, int tid) {
  return wrs::compute_tile<KT, F16, PX, T, LIT>(e.s, e.f, st, u, px, d_f, tid);
}

// The copying warp's work for one tile of entry e. KT, CS > 0 fix the slot
// count and colour bytes at compile time (the K = 4 / 8 families), so the copy
// sizes and stage offsets fold to constants.
template <int T, int KT, int CS, bool COPY_FRAME>
__device__ __forceinline__ void produce_tile(const BatchEntry& e, int64_t p0, uint8_t* st,
                                             uint64_t* full, int ln, uint32_t stage_cap,
                                             uint32_t extra_tx) {
  const int K = KT > 0 ? KT : e.s.K;
  const int cs = CS > 0 ? CS : (entry_f16(e) ? 2 : 4);
  const bool resolve = stage_records(e);
  const StageLayout L = wrs::stage_layout(T, K, cs, resolve, KT == 0 && e.s.literal != 0);
  wrs::issue_tile_copies<T, false>(e.s, e.f, K, cs, resolve, L, st, full, p0, extra_tx, ln, COPY_FRAME,
                                   stage_cap);
}

// Warp-specialised like the single-stream pipelined kernel: warp 8 issues each
// tile's copies, warp 9 draws its uniforms, warps 0..7 compute it. FOVF >= 0:
// no frame is copied; two more warps foveate each tile from the stream's
// image and mip levels (filter FOVF, WRS_FILTER_*) into the stage.
template <int PX, int FAM, int FOVF = -1>
__global__ void __launch_bounds__(batch_threads(FOVF >= 0), PX == 1 ? 2 : 1)
    batch_kernel(const __grid_constant__ BatchArgs a) {
  static_assert(FOVF < 0 || PX == 1, "foveating batches take one pixel per thread");
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ unsigned long long replaced_s[kMaxBatch];  // per stream, this CTA
  __shared__ float d_f_s[kMaxBatch];                    // per stream: density at the fovea edge
  __shared__ uint32_t failed_s[kMaxBatch];              // per stream: an earlier wait gave up
  constexpr int T = kConsumerWarps * 32 * PX;
  const wrs::Ring r = wrs::make_ring(smem, a.stage_bytes, T, a.stages, a.queue != 0, a.maps != 0);
  const int tid = threadIdx.x;
  const int warp = tid >> 5;
  const int lane = tid & 31;
  if (warp == 0) wrs::init_ring(r, kConsumerWarps, batch_producers(FOVF >= 0), lane);
  if (tid < kMaxBatch) replaced_s[tid] = 0;
  // each stream's Eq. (phat) normaliser, once per CTA instead of once per tile
  bool usable = false;
  if (tid < a.n) {
    d_f_s[tid] = wrs::fovea_density(a.e[tid].s);
    // a stream whose earlier push timed out (not yet seen by the host) has
    // undefined reservoirs: its tiles are copied but not computed or written
    const uint32_t failed = *reinterpret_cast<volatile const uint32_t*>(a.e[tid].status);
    failed_s[tid] = failed;
    usable = failed == 0;
  }
  // nothing to compute: among others the CTAs that start after a wait of this
  // launch has given up, which then add no waits of their own
  if (!__syncthreads_or(usable)) return;

  int issued = 0;
  if (warp == kConsumerWarps) {
    int pe = 0;  // entry of the copying warp's current tile
    issued = wrs::produce<true>(r, a.timeout_ns, lane,
                                [&](uint32_t g, uint8_t* st, float*, uint64_t* full, int ln) {
      pe = entry_of(a, g, pe);
      const BatchEntry& e = a.e[pe];
      const int64_t p0 = static_cast<int64_t>(g - e.tile0) * T;
      constexpr bool cf = FOVF < 0;
      if constexpr (FAM == kFamF16K48) {
        if (e.code == 0) produce_tile<T, 4, 2, cf>(e, p0, st, full, ln, r.stage_bytes, a.extra_tx);
        else produce_tile<T, 8, 2, cf>(e, p0, st, full, ln, r.stage_bytes, a.extra_tx);
      } else if constexpr (FAM == kFamF32K48) {
        if (e.code == 2) produce_tile<T, 4, 4, cf>(e, p0, st, full, ln, r.stage_bytes, a.extra_tx);
        else produce_tile<T, 8, 4, cf>(e, p0, st, full, ln, r.stage_bytes, a.extra_tx);
      } else {
        produce_tile<T, 0, 0, cf>(e, p0, st, full, ln, r.stage_bytes, a.extra_tx);
      }
    });
  } else if (warp == kConsumerWarps + 1) {
    int pe = 0;
    wrs::produce<false>(r, a.timeout_ns, lane,
                        [&](uint32_t g, uint8_t*, float* u, uint64_t* full, int ln) {
      pe = entry_of(a, g, pe);
      const BatchEntry& e = a.e[pe];
      wrs::draw_tile<T>(e.s, e.f, static_cast<int64_t>(g - e.tile0) * T, u, full, ln);
    });
  } else if (FOVF >= 0 && warp >= kConsumerWarps + 2) {
    int pe = 0;
    if constexpr (FOVF >= 0)
      wrs::produce<false>(r, a.timeout_ns, lane,
                          [&](uint32_t g, uint8_t* st, float*, uint64_t* full, int ln) {
        pe = entry_of(a, g, pe);
        const BatchEntry& e = a.e[pe];
        wrs::foveate_tile<FOVF>(e.s, e.f, e.fv, g - e.tile0, st, full, warp - kConsumerWarps - 2, ln);
      });
  } else {
    wrs::TilePx<8> px;
    int ei = 0;        // entry of the consumer's current tile
    int replaced = 0;  // this thread's replacements in entry ei so far
    wrs::consume(r, a.timeout_ns, lane, [&](uint32_t g) {
      const int next = entry_of(a, g, ei);
      if (next != ei) {
        flush_count(replaced_s, ei, replaced, lane);
        ei = next;
      }
      const BatchEntry& e = a.e[ei];
      px.p = (g - e.tile0) * T + tid * PX;
      wrs::row_col(e.s, static_cast<int>(px.p), px.y, px.x);
      // fold inputs only for entries that compute with K = 4 or 8
      if (e.code < 4) {
        wrs::tile_ahead<8, PX, true>(e.s, e.f, px);
      } else {
        wrs::tile_ahead<8, PX, false>(e.s, e.f, px);
      }
    }, [&](uint8_t* st, const float* u) {
      const BatchEntry& e = a.e[ei];
      const float d_f = d_f_s[ei];
      if (failed_s[ei] != 0) return;
      int rc;
      if constexpr (FAM == kFamF16K48) {
        rc = e.code == 0 ? tile<4, true, PX, T, false>(e, st, u, px, d_f, tid)
                         : tile<8, true, PX, T, false>(e, st, u, px, d_f, tid);
      } else if constexpr (FAM == kFamF32K48) {
        rc = e.code == 2 ? tile<4, false, PX, T, false>(e, st, u, px, d_f, tid)
                         : tile<8, false, PX, T, false>(e, st, u, px, d_f, tid);
      } else {
        switch (e.code) {
          case 0: rc = tile<4, true, PX, T, false>(e, st, u, px, d_f, tid); break;
          case 1: rc = tile<8, true, PX, T, false>(e, st, u, px, d_f, tid); break;
          case 2: rc = tile<4, false, PX, T, false>(e, st, u, px, d_f, tid); break;
          case 3: rc = tile<8, false, PX, T, false>(e, st, u, px, d_f, tid); break;
          case 4: rc = tile<0, true, PX, T, false>(e, st, u, px, d_f, tid); break;
          case 6: rc = tile<1, true, PX, T, true>(e, st, u, px, d_f, tid); break;
          case 7: rc = tile<1, false, PX, T, true>(e, st, u, px, d_f, tid); break;
          default: rc = tile<0, false, PX, T, false>(e, st, u, px, d_f, tid); break;
        }
      }
      replaced += rc;
    });
    flush_count(replaced_s, ei, replaced, lane);
  }
  __syncthreads();
  if (tid < a.n && replaced_s[tid] != 0) atomicAdd(a.e[tid].s.replacements, replaced_s[tid]);
  if (wrs::flag_raised(r)) {
    if (warp == kConsumerWarps) wrs::drain(r, issued, a.timeout_ns);
    // the batch ran out of time as a whole: report it on every stream
    if (tid < a.n) atomicExch(a.e[tid].status, static_cast<uint32_t>(WRS_ERR_TIMEOUT));
  }
}

}  // namespace
