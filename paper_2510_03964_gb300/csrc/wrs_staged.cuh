// The per-pixel update of a tile that has landed in shared memory: what the
// consumer warps of the pipelined and the batched kernels run. The arithmetic
// is push_group's (wrs_device.cuh), step for step and bit for bit.
//
// What bounds it: instruction issue and its latency, with DRAM close behind.
// An SM holds 16 consumer warps (shared memory allows no more pixels in flight),
// so each pixel's instructions set the time of the forms that move little per
// pixel (HD K = 4, the literal rule, flushes, the full bias); 4K K = 8 is at its
// DRAM traffic. Hence, against push_group:
//  * a thread owns its pixels' columns of the stage, so the rare events (a
//    flush, a rescale of the keys, the replaced slot) are written into the
//    columns and the loops over the slots then read them as they are: no
//    select per slot for what seldom or never happens;
//  * the race takes the largest key first and looks for its slot only where
//    the candidate has won.
// Measured against push_group on the same stages: 4K K = 8 FP16 286 -> 247 us,
// 4K K = 8 FP32 295 -> 282 us (mostly DRAM), HD K = 4 FP32 55.5 -> 48.7 us, 4K
// literal rule 82.8 -> 73.8 us; executed instructions per pixel 770 -> 610
// (K = 8 FP16), 540 -> 450 (K = 4 FP32), and 570 and 425 with the folds by
// shifts and the flush maps in the stage.
#pragma once

#include <stdint.h>

#include "wrs_device.cuh"

namespace wrs {

// Byte offsets of one stage's planes in shared memory (tile of T pixels).
// cs = 2 (FP16 colour: K planes of the weights' low 16 bits, then K planes of
// 8-byte records {r, g, b, w_hi}) or 4 (FP32 colour: K float4 {w, r, g, b}
// record planes, starting at `col`; `wt` == `col`). The literal rule has no P
// and no key planes: its 512-pixel stages of 18 KB let three CTAs with four
// stages share an SM.
struct StageLayout {
  uint32_t frame, W, P, key, wt, col, bytes;
};

__host__ __device__ __forceinline__ StageLayout stage_layout(int T, int K, int cs, bool resolve,
                                                              bool literal) {
  StageLayout L;
  L.frame = 0;
  L.W = 12u * T;
  L.P = L.W + 4u * T;
  L.key = L.P + (literal ? 0u : 4u * T);
  const uint32_t keys = literal ? 0u : 4u * K * T;
  if (cs == 2) {
    L.wt = L.key + keys;
    L.col = L.wt + (resolve ? 2u * K * T : 0u);
    L.bytes = L.col + (resolve ? 8u * K * T : 0u);
  } else {
    L.wt = L.col = L.key + keys;
    L.bytes = L.col + (resolve ? 16u * K * T : 0u);
  }
  return L;
}

// Orders a thread's own writes to a stage before the bulk copy that refills it.
__device__ __forceinline__ void fence_stage_writes() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Checked build: the entries a thread's PX pixels at p (tile entry tl) use.
template <int PX, int T>
__device__ __forceinline__ bool staged_in_bounds(const StreamDev& s, uint32_t p, int tl, int x, int y) {
#ifdef WRS_CHECKED
  const int64_t q = p;
  bool ok = WRS_IN(s, q + PX <= s.plane, kChkPlane);
  ok = WRS_IN(s, tl >= 0 && tl + PX <= T, kChkStage) && ok;
  ok = WRS_IN(s, y >= 0 && y < s.height && x >= 0 && x + PX <= s.width &&
                     static_cast<int64_t>(y) * s.width + x == q,
              kChkFrame) && ok;
  return WRS_IN(s, q + PX <= s.hw, kChkOut) && ok;
#else
  (void)s; (void)p; (void)tl; (void)x; (void)y;
  return true;
#endif
}

// The key race for thread `tid`'s PX pixels p .. p+PX-1 = (x, y) .. (x+PX-1, y)
// of the tile staged at `st` with its uniforms at `u`; flush: the pixels'
// flush bits. Returns how many of them replaced a slot.
template <int KT, bool F16, int PX, int T, int KM>
__device__ __forceinline__ int push_staged(const StreamDev& s, const FrameDev& f, uint8_t* st,
                                           const float* u, uint32_t p, int x, int y, float d_f,
                                           int tid, uint32_t flush, const FoldIn<KM>* pre) {
  static_assert(4 % PX == 0, "pixels per thread must divide 4");
  const int K = KT > 0 ? KT : s.K;
  const int n = KT == kUpTo8 ? 8 : K;  // bound of the unrolled loops
  const int64_t pl = s.plane;
  const int tl = tid * PX;
  if (!staged_in_bounds<PX, T>(s, p, tl, x, y)) return 0;
  const StageLayout L = stage_layout(T, K, F16 ? 2 : 4, true, false);
  float* key = reinterpret_cast<float*>(st + L.key) + tl;
  uint16_t* wt = reinterpret_cast<uint16_t*>(st + L.wt);
  uint8_t* col = st + L.col;
  const bool records = f.out != nullptr || s.bias == 2;  // the stage holds the slot records
  const bool direct = direct_index<KT>(s);

  float rgb[PX][3], Wv[PX], Pv[PX], w[PX], ks[PX], gl[PX];
  load_rgb<PX>(reinterpret_cast<const float*>(st + L.frame) + 3 * tl, rgb);
  load_f<PX>(reinterpret_cast<const float*>(st + L.W) + tl, Wv);
  load_f<PX>(reinterpret_cast<const float*>(st + L.P) + tl, Pv);
#pragma unroll
  for (int i = 0; i < PX; ++i) gl[i] = 1.0f;
  if (s.bias == 2) {
    // Eq. (full-temporal-bias): resolved colour of the slots before the push
    float n0[PX], n1[PX], n2[PX], dn[PX];
#pragma unroll
    for (int i = 0; i < PX; ++i) { n0[i] = n1[i] = n2[i] = dn[i] = 0.0f; }
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
      if (KT == kUpTo8 && j >= K) break;
      float a[PX], r[PX], g[PX], b[PX];
      load_slot<F16, PX>(wt, col, K, j, T, tl, a, r, g, b);
#pragma unroll
      for (int i = 0; i < PX; ++i) {
        n0[i] = __fmaf_rn(a[i], r[i], n0[i]);
        n1[i] = __fmaf_rn(a[i], g[i], n1[i]);
        n2[i] = __fmaf_rn(a[i], b[i], n2[i]);
        dn[i] = fadd(dn[i], a[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < PX; ++i) {
      if (((flush >> i) & 1u) || !(Wv[i] > 0.0f)) continue;
      gl[i] = lightness_factor(n0[i], n1[i], n2[i], dn[i], rgb[i]);
      if (gl[i] <= 0.0f) flush |= 1u << i;  // no weight left in the history
    }
  }

  // weight (Eq. phat), A-ES key -ln(u)/w, Eq. (temporal-bias), Alg. 2's sum
#pragma unroll
  for (int i = 0; i < PX; ++i) {
    const int64_t q = static_cast<int64_t>(p) + i;
    w[i] = pixel_weight(s, d_f, x + i, y, f.gx, f.gy);
    const float k = fdiv(-log_pos(u[tl + i]), w[i]);
    if ((flush >> i) & 1u) {
      // every slot of the pixel empty, in its column and in the planes
      Wv[i] = 0.0f;
      Pv[i] = 1.0f;
      for (int j = 0; j < K; ++j) {
        key[j * T + i] = kInf;
        s.key[j * pl + q] = kInf;
        if (direct) s.idx[j * pl + q] = kEmpty;
        if (records) store_slot<F16>(wt, col, K, j, T, tl + i, 0.0f, 0.0f, 0.0f, 0.0f);
        store_slot<F16>(s.wt, s.col, K, j, pl, q, 0.0f, 0.0f, 0.0f, 0.0f);
      }
    }
    bool rescale;
    ks[i] = bias_and_sum(s.bias, w[i], k, Wv[i], Pv[i], rescale, gl[i]);
    if (rescale) {
      for (int j = 0; j < K; ++j) {
        float kj = key[j * T + i];
        if (kj == kInf) continue;
        kj = fminf(fmul(kj, kPScale), kFltMax);
        key[j * T + i] = kj;
        s.key[j * pl + q] = kj;
      }
    }
  }
  store_f<PX>(s.W + p, Wv);
  store_f<PX>(s.P + p, Pv);

  // key race: the slot holding the largest key (lowest index on ties; an empty
  // slot holds +inf) is replaced iff the new key is strictly smaller
  float kmax[PX];
#pragma unroll
  for (int i = 0; i < PX; ++i) kmax[i] = -1.0f;
#pragma unroll 8
  for (int j = 0; j < n; ++j) {
    if (KT == kUpTo8 && j >= K) break;
    float kv[PX];
    load_f<PX>(key + j * T, kv);
#pragma unroll
    for (int i = 0; i < PX; ++i) kmax[i] = fmaxf(kmax[i], kv[i]);
  }
  int replaced = 0;
#pragma unroll
  for (int i = 0; i < PX; ++i) {
    const int64_t q = static_cast<int64_t>(p) + i;
    const uint32_t dropped = (flush >> i) & 1u ? kCodeFlush : 0u;
    uint32_t code = dropped ? kCodeFlush : kCodeKeep;
    if (ks[i] < kmax[i]) {
      int jm = 0;
#pragma unroll 8
      for (int j = n - 1; j >= 0; --j)
        if ((KT != kUpTo8 || j < K) && key[j * T + i] == kmax[i]) jm = j;
      replaced += 1;
      code = jm | dropped;
      s.key[jm * pl + q] = ks[i];
      if (direct) s.idx[jm * pl + q] = f.t;
      if (records) store_slot<F16>(wt, col, K, jm, T, tl + i, w[i], rgb[i][0], rgb[i][1], rgb[i][2]);
      store_slot<F16>(s.wt, s.col, K, jm, pl, q, w[i], rgb[i][0], rgb[i][1], rgb[i][2]);
    }
    if (!direct) record_code<KT, KM>(s, f, q, static_cast<uint8_t>(code), PX == 1 ? pre : nullptr);
  }

  // fused resolve over the slots as they are after this push
  if (f.out != nullptr) {
    float num[PX][3], den[PX], o[PX][3];
#pragma unroll
    for (int i = 0; i < PX; ++i) num[i][0] = num[i][1] = num[i][2] = den[i] = 0.0f;
#pragma unroll 8
    for (int j = 0; j < n; ++j) {
      if (KT == kUpTo8 && j >= K) break;
      float a[PX], r[PX], g[PX], b[PX];
      load_slot<F16, PX>(wt, col, K, j, T, tl, a, r, g, b);
#pragma unroll
      for (int i = 0; i < PX; ++i) {
        num[i][0] = __fmaf_rn(a[i], r[i], num[i][0]);
        num[i][1] = __fmaf_rn(a[i], g[i], num[i][1]);
        num[i][2] = __fmaf_rn(a[i], b[i], num[i][2]);
        den[i] = fadd(den[i], a[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < PX; ++i) {
      const float inv = den[i] > 0.0f ? __frcp_rn(den[i]) : 0.0f;
      o[i][0] = fmul(num[i][0], inv);
      o[i][1] = fmul(num[i][1], inv);
      o[i][2] = fmul(num[i][2], inv);
    }
    store_rgb<PX>(f.out + 3 * static_cast<int64_t>(p), o);
  }
  return replaced;
}

// The literal n = 1 rule (push_group_literal) for a staged tile.
template <bool F16, int PX, int T>
__device__ __forceinline__ int push_staged_literal(const StreamDev& s, const FrameDev& f,
                                                   const uint8_t* st, const float* u, uint32_t p,
                                                   int x, int y, float d_f, int tid,
                                                   uint32_t flush) {
  const int tl = tid * PX;
  if (!staged_in_bounds<PX, T>(s, p, tl, x, y)) return 0;
  const StageLayout L = stage_layout(T, 1, F16 ? 2 : 4, true, true);
  const bool records = f.out != nullptr || s.bias == 2;
  float rgb[PX][3], Wv[PX], a[PX], r[PX], g[PX], b[PX], o[PX][3];
  load_rgb<PX>(reinterpret_cast<const float*>(st + L.frame) + 3 * tl, rgb);
  load_f<PX>(reinterpret_cast<const float*>(st + L.W) + tl, Wv);
  if (records)
    load_slot<F16, PX>(reinterpret_cast<const uint16_t*>(st + L.wt), st + L.col, 1, 0, T, tl, a, r, g, b);
  int taken = 0;
#pragma unroll
  for (int i = 0; i < PX; ++i) {
    const int64_t q = static_cast<int64_t>(p) + i;
    const float w = pixel_weight(s, d_f, x + i, y, f.gx, f.gy);
    bool drop = ((flush >> i) & 1u) != 0;
    float gl = 1.0f;
    if (s.bias == 2 && !drop && Wv[i] > 0.0f) {
      // Eq. (full-temporal-bias): Delta L against the resident sample
      gl = lightness_factor(__fmaf_rn(a[i], r[i], 0.0f), __fmaf_rn(a[i], g[i], 0.0f),
                            __fmaf_rn(a[i], b[i], 0.0f), fadd(0.0f, a[i]), rgb[i]);
      drop = gl <= 0.0f;
    }
    if (drop) Wv[i] = 0.0f;
    if (s.bias && Wv[i] > 0.0f) {
      float fb = fdiv(Wv[i], fadd(Wv[i], w));
      if (s.bias == 2) fb = fmul(fb, gl);
      Wv[i] = fmul(Wv[i], fb);
    }
    const float tot = fadd(Wv[i], w);
    const bool take = !(fmul(u[tl + i], tot) <= Wv[i]);  // Alg. 2: R1 kept on <=
    Wv[i] = tot;
    if (take) {
      s.idx[q] = f.t;  // one slot: the index is written directly (direct_index)
      store_slot<F16>(s.wt, s.col, 1, 0, s.plane, q, w, rgb[i][0], rgb[i][1], rgb[i][2]);
      a[i] = w;
      r[i] = stored_colour<F16>(rgb[i][0]);
      g[i] = stored_colour<F16>(rgb[i][1]);
      b[i] = stored_colour<F16>(rgb[i][2]);
      taken += 1;
    }
    if (f.out != nullptr) {
      const float den = fadd(0.0f, a[i]);
      const float inv = den > 0.0f ? __frcp_rn(den) : 0.0f;
      o[i][0] = fmul(__fmaf_rn(a[i], r[i], 0.0f), inv);
      o[i][1] = fmul(__fmaf_rn(a[i], g[i], 0.0f), inv);
      o[i][2] = fmul(__fmaf_rn(a[i], b[i], 0.0f), inv);
    }
  }
  store_f<PX>(s.W + p, Wv);
  if (f.out != nullptr) store_rgb<PX>(f.out + 3 * static_cast<int64_t>(p), o);
  return taken;
}

}  // namespace wrs
