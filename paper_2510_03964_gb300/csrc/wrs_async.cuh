// Bulk asynchronous copies and transaction-count barriers (sm_90+ PTX, used on
// sm_103a), and the tile pipeline shared by the single-stream and batched
// persistent kernels.
#pragma once

#include <stdint.h>

#include "wrs_device.cuh"
#include "wrs_fov.cuh"
#include "wrs_staged.cuh"

namespace wrs {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
               : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// global -> shared bulk copy of `bytes` (multiple of 16, both addresses 16-byte
// aligned), completing `bytes` transactions on `bar`
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes,
                                         uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// `bytes` (multiple of 16, 16-byte aligned) of global memory into the L2
__device__ __forceinline__ void bulk_prefetch(const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Waits for phase `parity` of `bar` to complete; false once limit_ns has passed.
// The call that finds the phase complete (the common one) stays inline.
static __device__ __noinline__ bool mbar_wait_slow(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
  const uint64_t t0 = global_ns();
  for (;;) {
    if (mbar_try_wait(bar, parity)) return true;
    if (global_ns() - t0 > limit_ns) return false;
  }
}

__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
  return mbar_try_wait(bar, parity) || mbar_wait_slow(bar, parity, limit_ns);
}

// Warp-wide: lane 0 arms `bar` for the tile's bytes (plus extra_tx, which is
// non-zero only to test the timeout path), then the lanes issue one bulk copy
// per plane segment. The tile starts at pixel p0 (a multiple of T >= 256);
// requires frame rows without padding and 16-byte aligned frame and state
// planes. A bulk copy moves whole 16 bytes, four pixels of the frame: up to
// three last pixels of an image come by plain loads. copy_frame = false leaves
// the frame segment to the warps that foveate the frame into it.
// AHEAD: also bring what the tile's fold will read into the L2.
template <int T, bool AHEAD>
__device__ __forceinline__ void issue_tile_copies(const StreamDev& s, const FrameDev& f, int K,
                                                  int cs, bool resolve, const StageLayout& L,
                                                  uint8_t* stage, uint64_t* bar, int64_t p0,
                                                  uint32_t extra_tx, int lane,
                                                  bool copy_frame = true,
                                                  uint32_t stage_cap = 0xFFFFFFFFu) {
  const int64_t rem_plane = s.plane - p0, rem_px = s.hw - p0;
  const uint32_t n = static_cast<uint32_t>(rem_plane < T ? rem_plane : T);  // plane entries (x64)
  const uint32_t np = static_cast<uint32_t>(rem_px < T ? rem_px : T);       // pixels
#ifdef WRS_CHECKED
  // every copy's global range inside its plane or the frame, and the stage's
  // layout inside the ring's stage; otherwise no copy is issued and the
  // barrier completes empty (the consumers then compute stale data, flagged)
  {
    bool ok = WRS_IN(s, p0 >= 0 && p0 < s.hw && p0 + n <= s.plane && p0 + np <= s.hw &&
                            n % 64 == 0 && K >= 1 && K <= WRS_MAX_K,
                     kChkCopy);
    ok = WRS_IN(s, L.bytes <= stage_cap, kChkStageSize) && ok;
    if (!ok) {
      if (lane == 0) mbar_arrive_expect_tx(bar, 0u);
      __syncwarp();
      return;
    }
  }
#else
  (void)stage_cap;
#endif
  const uint32_t np4 = np & ~3u;
  if (copy_frame && np4 != np) {
    if (static_cast<uint32_t>(lane) < 3u * (np - np4))
      reinterpret_cast<float*>(stage + L.frame)[3u * np4 + lane] = f.frame[3 * (p0 + np4) + lane];
    __syncwarp();
  }
  // the literal rule (K = 1) reads no P and no key plane: copies 2 and 3 are skipped
  const int skip = s.literal ? 2 : 0;
  const int ncopy = 3 + K + (resolve ? (cs == 2 ? 2 * K : K) : 0);
  if (lane == 0) {
    uint32_t bytes = (copy_frame ? 12u * np4 : 0u) + 8u * n + 4u * K * n;
    if (skip) bytes -= 4u * n + 4u * K * n;
    if (resolve) bytes += cs == 2 ? (2u * K * n + 8u * K * n) : 16u * K * n;
    mbar_arrive_expect_tx(bar, bytes + extra_tx);
  }
  __syncwarp();
  const int64_t pl = s.plane;
  for (int c = lane; c < ncopy; c += 32) {
    if (skip && (c == 2 || c == 3)) continue;
    if (c == 0 && (!copy_frame || np4 == 0u)) continue;
    if (c == 0) {
      bulk_g2s(stage + L.frame, f.frame + 3 * p0, 12u * np4, bar);
    } else if (c == 1) {
      bulk_g2s(stage + L.W, s.W + p0, 4u * n, bar);
    } else if (c == 2) {
      bulk_g2s(stage + L.P, s.P + p0, 4u * n, bar);
    } else if (c < 3 + K) {
      const int j = c - 3;
      bulk_g2s(stage + L.key + 4u * T * j, s.key + j * pl + p0, 4u * n, bar);
    } else if (cs == 4) {
      const int j = c - 3 - K;  // FP32 colour: record plane j
      bulk_g2s(stage + L.col + 16u * T * j,
               static_cast<const float4*>(s.col) + j * pl + p0, 16u * n, bar);
    } else if (c < 3 + 2 * K) {
      const int j = c - 3 - K;
      bulk_g2s(stage + L.wt + 2u * T * j, s.wt + j * pl + p0, 2u * n, bar);
    } else {
      const int j = c - 3 - 2 * K;  // FP16 colour: record plane j
      bulk_g2s(stage + L.col + 8u * T * j, static_cast<const uint2*>(s.col) + j * pl + p0,
               8u * n, bar);
    }
  }
  if constexpr (T == 256 && AHEAD) {
    if (K > 2 && folds_now(f, p0)) {
      // the code rows of the last 15 frames and the K index rows: the consumers
      // load them when they come to the tile, S tiles later (HD K = 4 43.9 ->
      // 42.6 us)
      const int c = lane < kRingFrames - 1 ? lane : lane - (kRingFrames - 1);
      if (lane < kRingFrames - 1)
        bulk_prefetch(s.maps + static_cast<int64_t>((f.t - 1u - c) & kRingMask) * pl + p0, n);
      else if (c < K)
        bulk_prefetch(s.idx + c * pl + p0, 4u * n);
    }
  }
}

// The planes of the CTA's first tile into the L2 (the copies proper wait for
// the stream's status word, a read of about 0.7 us: HD K = 4 42.8 -> 42.2 us).
template <int T>
__device__ __forceinline__ void prefetch_tile(const StreamDev& s, const FrameDev& f, int K, int cs,
                                              bool resolve, int64_t p0, int lane) {
  const int64_t pl = s.plane;
  const int64_t rem = pl - p0;
  if (p0 >= s.hw) return;
  const uint32_t n = static_cast<uint32_t>(rem < T ? rem : T);
  const int64_t rem_px = s.hw - p0;
  const uint32_t np4 = static_cast<uint32_t>(rem_px < T ? rem_px : T) & ~3u;
  if (lane == 0) {
    if (f.frame != nullptr && np4 != 0u) bulk_prefetch(f.frame + 3 * p0, 12u * np4);
    bulk_prefetch(s.W + p0, 4u * n);
    if (!s.literal) bulk_prefetch(s.P + p0, 4u * n);
  }
  for (int j = lane; j < K; j += 32) {
    if (!s.literal) bulk_prefetch(s.key + j * pl + p0, 4u * n);
    if (!resolve) continue;
    if (cs == 2) {
      bulk_prefetch(s.wt + j * pl + p0, 2u * n);
      bulk_prefetch(static_cast<const uint2*>(s.col) + j * pl + p0, 8u * n);
    } else {
      bulk_prefetch(static_cast<const float4*>(s.col) + j * pl + p0, 16u * n);
    }
  }
}

// The tile's uniforms, drawn by one warp: one Philox block per 4 pixels,
// written to u[0 .. T-1]; with a flush map its entries of the tile go to the T
// bytes behind them. Then the warp's arrival on `bar`. The consumers loaded
// their own flush-map bytes before: a wait on DRAM in every tile that the wait
// for the stage seldom covered, 1365 x 767 K = 4 with flushes 29.7 -> 27.5 us.
template <int T>
__device__ __forceinline__ void draw_tile(const StreamDev& s, const FrameDev& f, int64_t p0, float* u,
                                          uint64_t* bar, int lane) {
  uint8_t fov[T / 32];
  if (f.fov != nullptr) {
#pragma unroll
    for (int i = 0; i < T / 32; ++i) {
      const int64_t p = p0 + 32 * i + lane;
      fov[i] = p < s.hw ? f.fov[p] : 0u;
    }
  }
#pragma unroll
  for (int q = lane; q < T / 4; q += 32) {
    const uint32_t blk = static_cast<uint32_t>((p0 >> 2) + q);
    const uint4 b = philox4x32_10(make_uint4(blk, f.t, s.stream_id, 0u), s.seed_lo, s.seed_hi);
    float4 v;
    v.x = unit_uniform(b.x);
    v.y = unit_uniform(b.y);
    v.z = unit_uniform(b.z);
    v.w = unit_uniform(b.w);
    reinterpret_cast<float4*>(u)[q] = v;
  }
  if (f.fov != nullptr) {
    uint8_t* flags = reinterpret_cast<uint8_t*>(u + T);
#pragma unroll
    for (int i = 0; i < T / 32; ++i) flags[32 * i + lane] = fov[i];
  }
  __syncwarp();
  if (lane == 0) mbar_arrive(bar);
}

// What a consumer thread of a tile knows before the tile has landed: its first
// pixel p = (x, y) (no pixel if p >= hw) and, in the band this frame folds, the
// fold's inputs, loaded ahead of the wait, so that their latency passes while
// the tile is still in flight.
template <int KM>
struct TilePx {
  uint32_t p;
  int x, y;
  bool folding;
  FoldIn<KM> fold;
};

// Fills t for the pixels at t.p (t.x and t.y already set).
template <int KM, int PX, bool FOLD>
__device__ __forceinline__ void tile_ahead(const StreamDev& s, const FrameDev& f, TilePx<KM>& t) {
  t.folding = false;
  if (t.p >= static_cast<uint32_t>(s.hw)) return;
  if constexpr (FOLD && PX == 1) {
    if (s.K > 2 && s.K <= KM && folds_now(f, t.p)) {
      fold_load(s, s.idx, s.K, f.t, t.p, t.fold);
      t.folding = true;
    }
  }
}

// Computes consumer thread `tid`'s PX pixels of a landed tile from shared
// memory; returns how many of them replaced a slot. LIT: the literal n = 1
// rule (KT = 1).
template <int KT, bool F16, int PX, int T, bool LIT, int KM>
__device__ __forceinline__ int compute_tile(const StreamDev& s, const FrameDev& f, uint8_t* st,
                                            const float* u, const TilePx<KM>& t, float d_f, int tid) {
  if (t.p >= static_cast<uint32_t>(s.hw)) return 0;
  uint32_t flush = 0;
  if (f.fov != nullptr) {
    const uint8_t* flags = reinterpret_cast<const uint8_t*>(u + T) + tid * PX;
#pragma unroll
    for (int i = 0; i < PX; ++i) flush |= flags[i] == 0xFFu ? 1u << i : 0u;
  }
  if constexpr (LIT)
    return push_staged_literal<F16, PX, T>(s, f, st, u, t.p, t.x, t.y, d_f, tid, flush);
  else
    return push_staged<KT, F16, PX, T, KM>(s, f, st, u, t.p, t.x, t.y, d_f, tid, flush,
                                           t.folding ? &t.fold : nullptr);
}

// Frames foveated on read: two warps (w = 0, 1) write the 256-pixel tile's
// foveated colours into the stage's frame segment, four pixels per lane, and
// arrive on `bar`. With the consumers foveating their own pixels one by one, a
// 4K K = 8 FP16 frame (mip levels and update) takes 261 us instead of 259.
constexpr int kFovWarps = 2;
template <int FILTER>
__device__ __forceinline__ void foveate_tile(const StreamDev& s, const FrameDev& f, const FovDev& fv,
                                             uint32_t tile, uint8_t* stage, uint64_t* bar, int w,
                                             int lane) {
  const uint32_t q = 4u * (32u * w + lane);  // the lane's first pixel in the tile
  const uint32_t p = tile * 256u + q;
  if (p < static_cast<uint32_t>(s.hw)) {
    int y, x;
    row_col(s, static_cast<int>(p), y, x);
    float rgb[12];
    fov_quad<FILTER>(fv, f.gx, f.gy, x, y, rgb);
    float4* o = reinterpret_cast<float4*>(stage) + 3 * (q / 4);
    o[0] = make_float4(rgb[0], rgb[1], rgb[2], rgb[3]);
    o[1] = make_float4(rgb[4], rgb[5], rgb[6], rgb[7]);
    o[2] = make_float4(rgb[8], rgb[9], rgb[10], rgb[11]);
  }
  __syncwarp();
  if (lane == 0) mbar_arrive(bar);
}

// Adds a warp's counts to a running total: one atomic per warp.
__device__ __forceinline__ void add_warp_count(unsigned long long* total, int count, int lane) {
  const unsigned c = __reduce_add_sync(0xffffffffu, static_cast<unsigned>(count));
  if (lane == 0 && c != 0) atomicAdd(total, static_cast<unsigned long long>(c));
}

// ---------------------------------------------------------------- warp-specialised loop

// Tiles are handed out by the hardware's work queue (cluster launch control):
// the grid has one CTA per tile, the CTAs that fit start, and each of them,
// instead of ending after its own tile, cancels a CTA that has not started and
// takes its tile, in ascending order. A fixed deal (tile it * grid + CTA) let
// CTAs near the memory run ahead; the tiles in flight then spread over the
// planes, and at 4K K = 8 FP16 the same 1.5 GB of traffic took 250 to 267 us,
// depending on the box, where tiles handed out in order take 224 (FP32: 275 and
// 267).

// Asks for the tile of a CTA that has not started: 16 bytes to `resp`,
// completing 16 transactions on `bar`. One thread; at most one request in
// flight, and none after one has been refused.
__device__ __forceinline__ void request_tile(uint4* resp, uint64_t* bar) {
  mbar_arrive_expect_tx(bar, 16u);
  asm volatile(
      "clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];" ::
          "r"(smem_u32(resp)),
      "r"(smem_u32(bar))
      : "memory");
}

// Whether the landed answer at `resp` gives a tile, and which.
__device__ __forceinline__ bool answered_tile(const uint4* resp, uint32_t& tile) {
  uint32_t ok, x;
  asm volatile(
      "{\n .reg .pred p;\n .reg .b128 h;\n ld.shared.b128 h, [%2];\n"
      " clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, h;\n selp.u32 %0, 1, 0, p;\n"
      " mov.u32 %1, 0;\n @p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %1, h;\n}\n"
      : "=r"(ok), "=r"(x)
      : "r"(smem_u32(resp))
      : "memory");
  tile = x;
  return ok != 0;
}

// Shared memory a CTA asks for so that at most `n` of them fit on an SM
// (`smem` or more).
__host__ inline size_t smem_for_ctas(size_t smem, int n) {
  constexpr size_t kSmPerSm = 228 * 1024, kReservedPerCta = 1024;
  const size_t least = (kSmPerSm / (n + 1) - kReservedPerCta + 16 + 127) / 128 * 128;
  return smem > least ? smem : least;
}

constexpr int kMaxStages = 8;
// answers kept: of the tiles in the S stages, the next one and the one asked for
constexpr int kAnswers = kMaxStages + 2;

// Shared-memory ring of S stages, each holding one tile's planes followed by
// its uniforms and, if some frame has a flush map, its flush-map entries; then
// the answers of the work queue, the S "full" and S "empty" barriers, the
// answers' barriers and a flag word.
struct Ring {
  uint8_t* base;
  uint32_t stage_bytes;  // planes of the largest tile layout used
  uint32_t stride;       // stage_bytes + 4 * T (+ T with flush maps)
  int S;
  bool queue;            // the grid has more tiles than CTAs that fit: ask for more
  uint64_t* full;
  uint64_t* empty;
  uint64_t* told;        // [kAnswers]
  uint4* answer;         // [kAnswers]
  int* flag;             // non-zero once some wait gave up

  __device__ uint8_t* stage(int i) const { return base + i * stride; }
  __device__ float* u(int i) const { return reinterpret_cast<float*>(base + i * stride + stage_bytes); }
};

__host__ __device__ __forceinline__ size_t ring_bytes(uint32_t stage_bytes, int T, int S, bool maps) {
  return static_cast<size_t>(S) * (stage_bytes + (maps ? 5u : 4u) * T) + 16u * S + 24u * kAnswers + 16u;
}

// Stages that keep as many CTAs of a ring with flush maps on an SM as fit
// without them (one CTA at least).
__host__ inline int stages_with_maps(uint32_t stage_bytes, int T, int S) {
  constexpr size_t kSmPerSm = 228 * 1024, kReservedPerCta = 2048, kMost = 226 * 1024;
  const size_t plain = ring_bytes(stage_bytes, T, S, false);
  const size_t ctas = kSmPerSm / (plain + kReservedPerCta);
  while (S > 1) {
    const size_t smem = ring_bytes(stage_bytes, T, S, true);
    if (smem <= kMost && kSmPerSm / (smem + kReservedPerCta) >= ctas) break;
    --S;
  }
  return S;
}

__device__ __forceinline__ Ring make_ring(uint8_t* smem, uint32_t stage_bytes, int T, int S,
                                          bool queue, bool maps) {
  Ring r;
  r.queue = queue;
  r.base = smem;
  r.stage_bytes = stage_bytes;
  r.stride = stage_bytes + (maps ? 5u : 4u) * T;
  r.S = S;
  r.answer = reinterpret_cast<uint4*>(smem + static_cast<size_t>(S) * r.stride);
  r.full = reinterpret_cast<uint64_t*>(r.answer + kAnswers);
  r.empty = r.full + S;
  r.told = r.empty + S;
  r.flag = reinterpret_cast<int*>(r.told + kAnswers);
  return r;
}

// One warp initialises the barriers (full: one arrival per producing warp, the
// copying, the drawing and any foveating ones; empty: one arrival per consumer
// warp; told: the request's) and the flag; the caller then synchronises the
// block.
__device__ __forceinline__ void init_ring(const Ring& r, int consumer_warps, int producer_warps, int lane) {
  if (lane < r.S) {
    mbar_init(&r.full[lane], producer_warps);
    mbar_init(&r.empty[lane], consumer_warps);
  }
  if (lane < kAnswers) mbar_init(&r.told[lane], 1);
  if (lane == 0) *r.flag = 0;
  fence_mbar_init();
}

__device__ __forceinline__ void raise_flag(const Ring& r) {
  atomicExch(r.flag, 1);
}

__device__ __forceinline__ bool flag_raised(const Ring& r) {
  return *reinterpret_cast<volatile int*>(r.flag) != 0;
}

// A warp's place in the CTA's sequence of tiles: its current tile and the next
// answer it reads.
struct TileWalk {
  uint32_t tile;
  int slot = 0;
  uint32_t phase = 0;
  __device__ explicit TileWalk(uint32_t first) : tile(first) {}

  // Moves to the next tile; false when there is none or the wait gave up.
  __device__ __forceinline__ bool next(const Ring& r, uint64_t timeout_ns) {
    if (!r.queue) return false;
    if (!mbar_wait_bounded(&r.told[slot], phase, timeout_ns)) {
      raise_flag(r);
      return false;
    }
    const bool ok = answered_tile(&r.answer[slot], tile);
    if (++slot == kAnswers) {
      slot = 0;
      phase ^= 1u;
    }
    return ok;
  }
};

// A producer warp: for each of the CTA's tiles, waits until the stage is free
// and runs `tile_fn(tile, stage, u, full_bar, lane)`, which issues the tile's
// copies (the copying warp), draws its uniforms or foveates its frame, and
// arrives on the stage's full barrier. The copying warp (ASK) also asks for
// the tiles, one ahead of the one it copies: the answer it overwrites is that
// of a tile whose stage has since been freed. Returns the number of tiles
// produced.
template <bool ASK, typename TileFn>
__device__ __forceinline__ int produce(const Ring& r, uint64_t timeout_ns, int lane, TileFn tile_fn) {
  TileWalk at(blockIdx.x);
  int it = 0, stg = 0, ask = 0;
  uint32_t phase = 1;  // of the stage's last release; the first S tiles wait for none
  if (ASK && r.queue && lane == 0) request_tile(&r.answer[0], &r.told[0]);
  do {
    if (it >= r.S && !mbar_wait_bounded(&r.empty[stg], phase, timeout_ns)) {
      raise_flag(r);
      break;
    }
    if (flag_raised(r)) break;
    tile_fn(at.tile, r.stage(stg), r.u(stg), &r.full[stg], lane);
    ++it;
    if (++stg == r.S) {
      stg = 0;
      phase ^= 1u;
    }
    if (!at.next(r, timeout_ns)) break;
    if (ASK) {
      if (++ask == kAnswers) ask = 0;
      __syncwarp();
      if (lane == 0) request_tile(&r.answer[ask], &r.told[ask]);
    }
  } while (true);
  // a wait gave up: an answer still on its way lands before the CTA may end
  if (ASK && r.queue && flag_raised(r)) mbar_wait_bounded(&r.told[at.slot], at.phase, timeout_ns);
  return it;
}

// Consumer warp: for each tile, runs `before_fn(tile)` (loads that need not
// wait for the stage), waits for its stage to land, computes it
// (`compute_fn(stage, u)`), and releases the stage.
template <typename BeforeFn, typename ComputeFn>
__device__ __forceinline__ void consume(const Ring& r, uint64_t timeout_ns, int lane,
                                        BeforeFn before_fn, ComputeFn compute_fn) {
  TileWalk at(blockIdx.x);
  int stg = 0;
  uint32_t phase = 0;
  do {
    before_fn(at.tile);
    if (!mbar_wait_bounded(&r.full[stg], phase, timeout_ns)) {
      raise_flag(r);
      break;
    }
    compute_fn(r.stage(stg), r.u(stg));
    fence_stage_writes();
    __syncwarp();
    if (lane == 0) mbar_arrive(&r.empty[stg]);
    if (++stg == r.S) {
      stg = 0;
      phase ^= 1u;
    }
  } while (at.next(r, timeout_ns));
}

// After the loops (and a block barrier): if a wait gave up, the copying warp
// waits (bounded) on the full barriers of the last S tiles it issued, giving
// their copies time to land before the CTA exits. A barrier whose expected
// bytes can never all arrive (the test_extra_tx fault injection) does not
// complete even after its copies have landed, so there this wait only spends
// the limit once per stage: the guarantee then rests on the copies finishing
// within that time (they take microseconds; the limit is milliseconds), not on
// observing the barrier.
__device__ __forceinline__ void drain(const Ring& r, int issued, uint64_t timeout_ns) {
  const int from = issued > r.S ? issued - r.S : 0;
  for (int j = from; j < issued; ++j)
    mbar_wait_bounded(&r.full[j % r.S], (j / r.S) & 1u, timeout_ns);
}

}  // namespace wrs
