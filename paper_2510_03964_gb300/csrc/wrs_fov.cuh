// The per-pixel foveation post-process (Sec. 4.3, "Implementation"), shared
// by the standalone foveation kernels and the push kernel that foveates the
// frame as it reads it. Every arithmetic step that decides a bit of the
// result is one round-to-nearest intrinsic.
#pragma once

#include <stdint.h>

#include "wrs.h"

namespace wrs {

// Programmatic dependent launch: a kernel of this library (wrs_launch_early)
// starts on the SMs that the previous kernel of the stream has left and sets up
// its barriers there; grid_begin then waits until that kernel has completed and
// its writes are visible. Nothing before grid_begin touches global memory, and every CTA
// calls it. A kernel that calls it reads with ordinary loads: what the previous
// kernel writes changes while this one runs, and the compiler may move a
// non-coherent load (__ldg) across the wait.
__device__ __forceinline__ void grid_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// One stored mip level: [hb][wb] texels {r, g, b, 0}.
struct MipLevelDev {
  const float4* texels;
  int32_t wb, hb;
};

// A rendered image, its mip levels and the ring radii (squared, FP32).
struct FovDev {
  const float* img;                     // [H][pitch] RGB triples
  int64_t pitch;
  float r2[WRS_MAX_MIP_LEVELS - 1];     // r_i * r_i, rounded once; infinite past the last radius
  MipLevelDev lev[WRS_MAX_MIP_LEVELS];  // one per radius from [1]; [0] unused (the image)
};

// Level coordinate of pixel index i at level L: u = (i + 0.5) * 2^-L - 0.5
// clamped to [0, nb - 1]; integer part, right neighbour (clamped) and fraction.
__device__ __forceinline__ void texel_coord(int32_t i, int L, int32_t nb, int32_t* i0,
                                            int32_t* i1, float* f) {
  const float inv_b = __int_as_float((127 - L) << 23);  // 2^-L, exact
  float u = __fsub_rn(__fmul_rn(__fadd_rn((float)i, 0.5f), inv_b), 0.5f);
  u = fminf(fmaxf(u, 0.0f), (float)(nb - 1));
  const float fl = floorf(u);
  *i0 = (int32_t)fl;
  *i1 = *i0 + 1 < nb ? *i0 + 1 : nb - 1;
  *f = __fsub_rn(u, fl);
}

__device__ __forceinline__ float lerp2(float a, float b, float one_minus_f, float f) {
  return __fadd_rn(__fmul_rn(a, one_minus_f), __fmul_rn(b, f));
}

// Ring level of pixel x of a row whose squared vertical offset is dy2: the
// number of radii with (x + 0.5 - gx)^2 + dy2 > r^2 (FP32).
__device__ __forceinline__ int ring_level(const FovDev& a, float gx, float dy2, int32_t x) {
  const float dx = __fsub_rn(__fadd_rn((float)x, 0.5f), gx);
  const float d2 = __fadd_rn(__fmul_rn(dx, dx), dy2);
  int L = 0;
#pragma unroll
  for (int i = 0; i < WRS_MAX_MIP_LEVELS - 1; ++i) L += d2 > a.r2[i] ? 1 : 0;
  return L;
}

__device__ __forceinline__ float row_dy2(float gy, int32_t y) {
  const float dy = __fsub_rn(__fadd_rn((float)y, 0.5f), gy);
  return __fmul_rn(dy, dy);
}

// Colour of pixel (x, y) of the foveated frame at ring level L: level 0
// copies the image pixel; level L takes the level's texel (box) or the
// bilinear blend of its four nearest texel centres.
template <int FILTER>
__device__ __forceinline__ void level_colour(const FovDev& a, int L, int32_t x, int32_t y,
                                             float* rgb) {
  if (L == 0) {
    const float* s = a.img + (int64_t)y * a.pitch + 3 * (int64_t)x;
    rgb[0] = s[0];
    rgb[1] = s[1];
    rgb[2] = s[2];
  } else {
    const MipLevelDev lv = a.lev[L];
    if (FILTER == WRS_FILTER_BOX) {
      const float4 t = lv.texels[(int64_t)(y >> L) * lv.wb + (x >> L)];
      rgb[0] = t.x;
      rgb[1] = t.y;
      rgb[2] = t.z;
    } else {
      int32_t x0, x1, y0, y1;
      float fx, fy;
      texel_coord(x, L, lv.wb, &x0, &x1, &fx);
      texel_coord(y, L, lv.hb, &y0, &y1, &fy);
      const float4 t00 = lv.texels[(int64_t)y0 * lv.wb + x0];
      const float4 t01 = lv.texels[(int64_t)y0 * lv.wb + x1];
      const float4 t10 = lv.texels[(int64_t)y1 * lv.wb + x0];
      const float4 t11 = lv.texels[(int64_t)y1 * lv.wb + x1];
      const float gx_ = __fsub_rn(1.0f, fx), gy_ = __fsub_rn(1.0f, fy);
      rgb[0] = lerp2(lerp2(t00.x, t01.x, gx_, fx), lerp2(t10.x, t11.x, gx_, fx), gy_, fy);
      rgb[1] = lerp2(lerp2(t00.y, t01.y, gx_, fx), lerp2(t10.y, t11.y, gx_, fx), gy_, fy);
      rgb[2] = lerp2(lerp2(t00.z, t01.z, gx_, fx), lerp2(t10.z, t11.z, gx_, fx), gy_, fy);
    }
  }
}

// Colour of pixel (x, y) of the foveated frame for gaze (gx, gy), and its ring
// level (see ring_level and level_colour).
template <int FILTER>
__device__ __forceinline__ int fov_pixel(const FovDev& a, float gx, float gy, int32_t x,
                                         int32_t y, float* rgb) {
  const int L = ring_level(a, gx, row_dy2(gy, y), x);
  level_colour<FILTER>(a, L, x, y, rgb);
  return L;
}

// ---------------------------------------------------------------- four pixels

// Two floats in one register pair, each half rounded to nearest as the scalar
// operation rounds it.
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
  return v;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
// a * one_minus_f + b * f in both halves (lerp2). The sum is a fused
// multiply-add by `one`, a 1.0 that the compiler cannot see: it contracts a
// packed product and a packed sum (also a fused one by a literal 1.0) into one
// rounding, whatever their rounding modifiers.
__device__ __forceinline__ uint64_t lerp2x2(uint64_t a, uint64_t b, uint64_t one_minus_f, uint64_t f,
                                            uint64_t one) {
  uint64_t p, q;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(p) : "l"(a), "l"(one_minus_f));
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(q) : "l"(b), "l"(f));
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(p) : "l"(p), "l"(one), "l"(q));
  return p;
}

struct Texel {
  uint64_t rg, b0;
};
__device__ __forceinline__ Texel load_texel(const float4* t) {
  const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(t);
  return {v.x, v.y};
}

// Bilinear colours of four pixels whose left texel columns are o0 .. o3 among
// the N + 1 columns starting at row0, row1, with fractions f[0..3].
template <int N, int O0, int O1, int O2, int O3>
__device__ __forceinline__ void blend_quad(const float4* row0, const float4* row1,
                                           const float (&f)[4], float fy, float* rgb) {
  constexpr int off[4] = {O0, O1, O2, O3};
  Texel top[N + 1], bot[N + 1];
#pragma unroll
  for (int c = 0; c <= N; ++c) {
    top[c] = load_texel(row0 + c);
    bot[c] = load_texel(row1 + c);
  }
  const float gy = __fsub_rn(1.0f, fy);
  const float one = __fadd_rn(gy, fy);  // fy has few bits: exactly 1
  const uint64_t fy2 = pack2(fy, fy), gy2 = pack2(gy, gy), one2 = pack2(one, one);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float g = __fsub_rn(1.0f, f[i]);
    const uint64_t fx2 = pack2(f[i], f[i]), gx2 = pack2(g, g);
    const Texel &t0 = top[off[i]], &t1 = top[off[i] + 1], &b0 = bot[off[i]], &b1 = bot[off[i] + 1];
    const uint64_t rg = lerp2x2(lerp2x2(t0.rg, t1.rg, gx2, fx2, one2), lerp2x2(b0.rg, b1.rg, gx2, fx2, one2),
                                gy2, fy2, one2);
    const uint64_t b = lerp2x2(lerp2x2(t0.b0, t1.b0, gx2, fx2, one2), lerp2x2(b0.b0, b1.b0, gx2, fx2, one2),
                               gy2, fy2, one2);
    float pad;
    unpack2(rg, rgb[3 * i], rgb[3 * i + 1]);
    unpack2(b, rgb[3 * i + 2], pad);
  }
}

// Four adjacent pixels x0 .. x0+3 (x0 % 4 == 0) of row y: the same colours and
// levels as fov_pixel, bit for bit. What bounds it is instruction issue (435
// instructions per quad with the pixels treated one by one), so the quad
// shares what its pixels share: its levels are found from its two ends where
// the distance is monotone over it; pixels of one level > 0 away from the
// level's borders read each texel column once (four columns at level 1, three
// at level 2, two beyond, where x0 % 4 == 0 puts the columns' borders between
// fixed pixels) with their fractions known, and blend two channels per
// instruction: 320 instructions per quad, and 4K with three radii takes 31.5 us
// instead of 35 under the profiler, 29.2 instead of 36.6 back to back.
// Returns the four levels, one per byte.
template <int FILTER>
__device__ __forceinline__ uint32_t fov_quad(const FovDev& a, float gx, float gy, int32_t x0,
                                             int32_t y, float* rgb) {
  const float dy2 = row_dy2(gy, y);
  const int first = ring_level(a, gx, dy2, x0), last = ring_level(a, gx, dy2, x0 + 3);
  // (x + 0.5 - gx)^2 grows or falls over the whole quad unless gx lies within it
  const bool monotone = gx <= static_cast<float>(x0) || gx >= static_cast<float>(x0 + 4);
  if (first == last && monotone) {
    const int l = first;
    if (l == 0) {
      const float* s = a.img + (int64_t)y * a.pitch + 3 * (int64_t)x0;
      if (((reinterpret_cast<uintptr_t>(a.img) | (uintptr_t)(4 * a.pitch)) & 15u) == 0) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          const float4 v = reinterpret_cast<const float4*>(s)[i];
          rgb[4 * i] = v.x;
          rgb[4 * i + 1] = v.y;
          rgb[4 * i + 2] = v.z;
          rgb[4 * i + 3] = v.w;
        }
      } else {
#pragma unroll
        for (int i = 0; i < 12; ++i) rgb[i] = s[i];
      }
      return 0u;
    }
    const uint32_t levels = 0x01010101u * (uint32_t)l;
    const MipLevelDev lv = a.lev[l];
    if (FILTER == WRS_FILTER_BOX) {
      const float4* row = lv.texels + (int64_t)(y >> l) * lv.wb + (x0 >> l);
      const float4 t = row[0], u = l == 1 ? row[1] : t;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 c = i < 2 ? t : u;
        rgb[3 * i] = c.x;
        rgb[3 * i + 1] = c.y;
        rgb[3 * i + 2] = c.z;
      }
      return levels;
    }
    int32_t xa, xb, y0, y1;
    float fx, fy;
    texel_coord(x0, l, lv.wb, &xa, &xb, &fx);
    texel_coord(y, l, lv.hb, &y0, &y1, &fy);
    const int n = l == 1 ? 3 : (l == 2 ? 2 : 1);  // columns to the right of xa
    if (x0 >= (1 << l) && xa + n < lv.wb && x0 < (1 << 21) && y < (1 << 21)) {
      const float4* row0 = lv.texels + (int64_t)y0 * lv.wb + xa;
      const float4* row1 = lv.texels + (int64_t)y1 * lv.wb + xa;
      if (l == 1) {
        const float f[4] = {0.75f, 0.25f, 0.75f, 0.25f};
        blend_quad<3, 0, 1, 1, 2>(row0, row1, f, fy, rgb);
      } else if (l == 2) {
        const float f[4] = {0.625f, 0.875f, 0.125f, 0.375f};
        blend_quad<2, 0, 0, 1, 1>(row0, row1, f, fy, rgb);
      } else {
        const float d = __int_as_float((127 - l) << 23);
        const float f[4] = {fx, fx + d, fx + 2.0f * d, fx + 3.0f * d};  // exact
        blend_quad<1, 0, 0, 0, 0>(row0, row1, f, fy, rgb);
      }
      return levels;
    }
  }
  // a quad on a ring's or the image's border: pixel by pixel
  uint32_t levels = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int l = ring_level(a, gx, dy2, x0 + i);
    level_colour<FILTER>(a, l, x0 + i, y, rgb + 3 * i);
    levels |= (uint32_t)l << (8 * i);
  }
  return levels;
}

}  // namespace wrs
