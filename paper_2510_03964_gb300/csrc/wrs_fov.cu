// Foveation post-process (Sec. 4.3, "Implementation"): the rendered frame is
// mip-mapped and each ring around the gaze is reconstructed from a coarser
// level, by nearest lookup or bilinear filtering. Two kernels:
//
//  mip_kernel     one pass over the image builds every stored level: the level
//                 sums are formed bottom-up in registers with the quad-tree
//                 order (s00 + s01) + (s10 + s11) and each level's means are
//                 written as 16-byte texels. The image is read once; levels
//                 >= 1 are written once.
//  foveate4_kernel four adjacent pixels per thread (foveate_kernel: one, for
//                 widths not divisible by 4 or unaligned frames): FP32 ring
//                 test, then a copy of the image pixel (level 0) or one (box)
//                 or four (bilinear) texel reads, which the 129 MB L2 serves
//                 for the coarse levels; writes the colours as 16-byte stores
//                 and the ring levels as one word.
//
// Every arithmetic step that decides a bit of the output is a single
// round-to-nearest intrinsic, so the results are reproducible on any IEEE
// FP32 implementation of the same sequence.
#include <cmath>
#include <cstring>

#include "wrs_fov.cuh"
#include "wrs_internal.h"

using wrs::FovDev;
using wrs::MipLevelDev;

namespace {

constexpr int kMipThreads = 256;
constexpr int kMipTileW = 64, kMipTileH = 32;  // pixels per CTA
constexpr int kFovThreads = 256;

// The four-pixel form: quads and rows per warp, pixels per CTA of 2 x 4 warps.
// Bilinear filtering takes 8 quads of 4 rows (32 x 4 pixels): fewer warps
// straddle a ring's border, where a warp runs the code of both levels, than
// with strips of one row (4K, back to back, 29.2 against 31.7 us). The box
// filter has little code to repeat and writes its strips faster (4K, cold L2,
// 29.3 against 31.3 us).
template <int FILTER>
struct FovTile {
  static constexpr int kQuadsX = FILTER == WRS_FILTER_BOX ? 32 : 8, kQuadsY = 32 / kQuadsX;
  static constexpr int kW = 2 * 4 * kQuadsX, kH = kFovThreads / 64 * kQuadsY;
};


// Writable view of a stored level, for the build.
struct MipLevelOut {
  float4* texels;
  int32_t wb, hb;
};

struct MipArgs {
  const float* img;
  int64_t pitch;
  int32_t width, height;
  MipLevelOut lev[WRS_MAX_MIP_LEVELS];  // [0] unused
};

struct FovArgs {
  FovDev fv;
  float* frame;
  int64_t frame_pitch;
  uint8_t* ring;
  int32_t width, height;
  float gx, gy;
};

// Pixels of level-L block i along an axis of n pixels.
__device__ __forceinline__ int32_t block_extent(int32_t n, int32_t i, int L) {
  const int64_t lo = (int64_t)i << L;
  const int64_t hi = lo + ((int64_t)1 << L);
  return (int32_t)((hi < n ? hi : n) - lo);
}

// Writes texel (x, y) of level L from its block's sums, if the level has it.
// A whole block's count is a power of two: its division is a multiplication.
template <int L>
__device__ __forceinline__ void store_mean(const MipArgs& a, uint32_t x, int32_t y, const float (&sum)[3]) {
  const MipLevelOut& lv = a.lev[L];
  if (x >= (uint32_t)lv.wb || y >= lv.hb) return;
  float4 m;
  if (((x + 1) << L) <= (uint32_t)a.width && ((y + 1) << L) <= a.height) {
    constexpr float inv = 1.0f / (1 << (2 * L));
    m = make_float4(__fmul_rn(sum[0], inv), __fmul_rn(sum[1], inv), __fmul_rn(sum[2], inv), 0.0f);
  } else {
    const float n = (float)(block_extent(a.height, y, L) * block_extent(a.width, (int32_t)x, L));
    m = make_float4(__fdiv_rn(sum[0], n), __fdiv_rn(sum[1], n), __fdiv_rn(sum[2], n), 0.0f);
  }
  lv.texels[(int64_t)y * lv.wb + x] = m;
}

// A CTA builds every level of a 64 x 32 pixel tile: eight warps of 32 x 8
// pixels, a lane four pixels of two rows. A lane's registers hold its pixels,
// its two level-1 sums and, after one exchange per axis (shuffles), the sums of
// levels 2 and 3; only levels 4 and 5 meet in shared memory. Sums are the
// quad-tree order's, (s00 + s01) + (s10 + s11). Bound by DRAM and the L2: the
// form that staged the strip in shared memory waited on its barriers and
// strided reads, 26.7 us for a 4K image's three levels; this one 21.
template <int M, bool VEC>
__global__ void __launch_bounds__(kMipThreads) mip_kernel(MipArgs a) {
  __shared__ float s_sum[4][8][3];  // level-3 sums of the tile (M > 3)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rp = lane >> 3, cq = lane & 7;  // row pair and column quad in the warp's 8 x 32
  wrs::grid_begin();
  const uint32_t x0 = blockIdx.x * kMipTileW + (warp & 1) * 32 + 4 * cq;
  const int32_t y0 = blockIdx.y * kMipTileH + (warp >> 1) * 8 + 2 * rp;
  // pixels from x0 to the end of the row (none past it)
  const int32_t left = (int32_t)((uint32_t)a.width - x0);

  float v[2][12];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int32_t y = y0 + r;
    const float* src = a.img + (int64_t)y * a.pitch + 3 * (int64_t)x0;
    if (VEC && y < a.height && left >= 4) {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const float4 t = reinterpret_cast<const float4*>(src)[i];
        v[r][4 * i] = t.x;
        v[r][4 * i + 1] = t.y;
        v[r][4 * i + 2] = t.z;
        v[r][4 * i + 3] = t.w;
      }
    } else {
      // pixels outside the image count as 0
      const int in_row = y < a.height ? 3 * (left < 4 ? left : 4) : 0;
#pragma unroll
      for (int i = 0; i < 12; ++i) v[r][i] = i < in_row ? src[i] : 0.0f;
    }
  }

  float s[2][3];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
#pragma unroll
    for (int ch = 0; ch < 3; ++ch)
      s[c][ch] = __fadd_rn(__fadd_rn(v[0][6 * c + ch], v[0][6 * c + 3 + ch]),
                           __fadd_rn(v[1][6 * c + ch], v[1][6 * c + 3 + ch]));
    store_mean<1>(a, (x0 >> 1) + c, y0 >> 1, s[c]);
  }
  if constexpr (M >= 2) {
    float t[3];
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
      t[ch] = __fadd_rn(s[0][ch], s[1][ch]);
      t[ch] = __fadd_rn(t[ch], __shfl_xor_sync(0xffffffffu, t[ch], 8));
    }
    if ((rp & 1) == 0) store_mean<2>(a, x0 >> 2, y0 >> 2, t);
    if constexpr (M >= 3) {
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) {
        t[ch] = __fadd_rn(t[ch], __shfl_xor_sync(0xffffffffu, t[ch], 1));
        t[ch] = __fadd_rn(t[ch], __shfl_xor_sync(0xffffffffu, t[ch], 16));
      }
      const bool top = rp == 0 && (cq & 1) == 0;
      if (top) store_mean<3>(a, x0 >> 3, y0 >> 3, t);
      if constexpr (M >= 4) {
        if (top) {
#pragma unroll
          for (int ch = 0; ch < 3; ++ch) s_sum[warp >> 1][(warp & 1) * 4 + (cq >> 1)][ch] = t[ch];
        }
        __syncthreads();
        if (warp == 0) {
          // lanes 0..7: the tile's 2 x 4 level-4 texels, then 1 x 2 of level 5
          const int r = (lane >> 2) & 1, c = lane & 3;
#pragma unroll
          for (int ch = 0; ch < 3; ++ch)
            t[ch] = __fadd_rn(__fadd_rn(s_sum[2 * r][2 * c][ch], s_sum[2 * r][2 * c + 1][ch]),
                              __fadd_rn(s_sum[2 * r + 1][2 * c][ch], s_sum[2 * r + 1][2 * c + 1][ch]));
          const uint32_t gx = blockIdx.x * (kMipTileW >> 4) + c;
          const int32_t gy = blockIdx.y * (kMipTileH >> 4) + r;
          if (lane < 8) store_mean<4>(a, gx, gy, t);
          if constexpr (M >= 5) {
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) {
              t[ch] = __fadd_rn(t[ch], __shfl_xor_sync(0xffffffffu, t[ch], 1));
              t[ch] = __fadd_rn(t[ch], __shfl_xor_sync(0xffffffffu, t[ch], 4));
            }
            if (lane < 4 && (lane & 1) == 0) store_mean<5>(a, gx >> 1, gy >> 1, t);
          }
        }
      }
    }
  }
}

// One pixel per thread (any width, pitch and alignment).
template <int FILTER>
__global__ void __launch_bounds__(kFovThreads) foveate_kernel(FovArgs a) {
  wrs::grid_begin();
  const int64_t n = (int64_t)a.width * a.height;
  for (int64_t p = (int64_t)blockIdx.x * kFovThreads + threadIdx.x; p < n;
       p += (int64_t)gridDim.x * kFovThreads) {
    const int32_t y = (int32_t)(p / a.width);
    const int32_t x = (int32_t)(p - (int64_t)y * a.width);
    float rgb[3];
    const int L = wrs::fov_pixel<FILTER>(a.fv, a.gx, a.gy, x, y, rgb);
    float* o = a.frame + (int64_t)y * a.frame_pitch + 3 * (int64_t)x;
    o[0] = rgb[0];
    o[1] = rgb[1];
    o[2] = rgb[2];
    if (a.ring) a.ring[p] = (uint8_t)L;
  }
}

// Four horizontally adjacent pixels per thread: width % 4 == 0, the frame's
// rows 16-byte aligned and the ring map 4-byte aligned, so a thread writes
// its 48 bytes of colour as three 16-byte stores and its levels as one word.
// Five CTAs per SM: it waits on texels and stores (32.8 -> 31.3 us at 4K, with
// ring levels that compare all radii instead of counting them).
template <int FILTER>
__global__ void __launch_bounds__(kFovThreads, 5) foveate4_kernel(FovArgs a) {
  using Tile = FovTile<FILTER>;
  wrs::grid_begin();
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t tiles_x = ((uint32_t)a.width + Tile::kW - 1) / Tile::kW;
  const uint32_t tiles = tiles_x * (((uint32_t)a.height + Tile::kH - 1) / Tile::kH);
  for (uint32_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const uint32_t ty = t / tiles_x;
    const int32_t x0 = (int32_t)((t - ty * tiles_x) * Tile::kW + (warp & 1) * 4 * Tile::kQuadsX +
                                 4 * (lane % Tile::kQuadsX));
    const int32_t y = (int32_t)(ty * Tile::kH + (warp >> 1) * Tile::kQuadsY + lane / Tile::kQuadsX);
    if (x0 >= a.width || y >= a.height) continue;
    float rgb[12];
    const uint32_t lv = wrs::fov_quad<FILTER>(a.fv, a.gx, a.gy, x0, y, rgb);
    float4* o = reinterpret_cast<float4*>(a.frame + (int64_t)y * a.frame_pitch + 3 * (int64_t)x0);
    o[0] = make_float4(rgb[0], rgb[1], rgb[2], rgb[3]);
    o[1] = make_float4(rgb[4], rgb[5], rgb[6], rgb[7]);
    o[2] = make_float4(rgb[8], rgb[9], rgb[10], rgb[11]);
    if (a.ring) *reinterpret_cast<uint32_t*>(a.ring + (int64_t)y * a.width + x0) = lv;
  }
}

bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

int check_image(int32_t width, int32_t height) {
  if (width < 1 || height < 1)
    return wrs_fail(WRS_ERR_ARG, "image size must be >= 1 x 1 (got %d x %d)", width, height);
  if ((int64_t)width * height >= ((int64_t)1 << 31))
    return wrs_fail(WRS_ERR_ARG, "width * height must be below 2^31");
  return WRS_OK;
}

template <typename Level>
void fill_levels(const wrs_mip_layout& L, const void* base, Level* lev) {
  for (int l = 1; l < L.levels; ++l) {
    lev[l].texels = reinterpret_cast<float4*>(const_cast<uint8_t*>(
        static_cast<const uint8_t*>(base) + L.offset[l]));
    lev[l].wb = L.width[l];
    lev[l].hb = L.height[l];
  }
}

int device_sms(int* sms) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
  return e == cudaSuccess ? WRS_OK : wrs_cuda_fail(e, "device query");
}

}  // namespace

extern "C" int wrs_mip_layout_get(int32_t width, int32_t height, int32_t levels,
                                  wrs_mip_layout* out) {
  wrs_clear_error();
  if (!out) return wrs_fail(WRS_ERR_ARG, "layout output is NULL");
  if (int rc = check_image(width, height)) return rc;
  if (levels < 1 || levels > WRS_MAX_MIP_LEVELS)
    return wrs_fail(WRS_ERR_ARG, "levels must be in 1..%d (got %d)", WRS_MAX_MIP_LEVELS, levels);
  std::memset(out, 0, sizeof(*out));
  out->levels = levels;
  out->width[0] = width;
  out->height[0] = height;
  out->offset[0] = -1;
  int64_t off = 0;
  for (int l = 1; l < levels; ++l) {
    out->width[l] = (int32_t)(((int64_t)width + (1 << l) - 1) >> l);
    out->height[l] = (int32_t)(((int64_t)height + (1 << l) - 1) >> l);
    out->offset[l] = off;
    off += ((int64_t)out->width[l] * out->height[l] * 16 + 255) / 256 * 256;
  }
  out->total_bytes = off;
  return WRS_OK;
}

extern "C" int wrs_mip_build(const float* d_img, int64_t pitch, int32_t width, int32_t height,
                             int32_t levels, void* d_mip, size_t mip_bytes, wrs_stream_t stream) {
  wrs_clear_error();
  wrs_mip_layout L;
  if (int rc = wrs_mip_layout_get(width, height, levels, &L)) return rc;
  if (levels == 1) return WRS_OK;
  if (!d_img || !aligned(d_img, 4)) return wrs_fail(WRS_ERR_ARG, "d_img is NULL or unaligned");
  if (pitch < 3 * (int64_t)width)
    return wrs_fail(WRS_ERR_ARG, "img_pitch_elems %lld is below 3 * width", (long long)pitch);
  if (!d_mip || !aligned(d_mip, 256))
    return wrs_fail(WRS_ERR_ARG, "d_mip is NULL or not 256-byte aligned");
  if ((int64_t)mip_bytes < L.total_bytes)
    return wrs_fail(WRS_ERR_BUDGET, "mip buffer holds %zu bytes, the layout needs %lld", mip_bytes,
                    (long long)L.total_bytes);
  MipArgs a{};
  a.img = d_img;
  a.pitch = pitch;
  a.width = width;
  a.height = height;
  fill_levels(L, d_mip, a.lev);
  const int M = levels - 1;
  const dim3 grid((unsigned)(((int64_t)width + kMipTileW - 1) / kMipTileW),
                  (unsigned)(((int64_t)height + kMipTileH - 1) / kMipTileH));
  if ((((int64_t)height + (1 << M) - 1) >> M) > 65535)
    return wrs_fail(WRS_ERR_ARG, "image too tall for the mip build");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const bool vec = pitch % 4 == 0 && aligned(d_img, 16);
  cudaError_t e;
#define WRS_MIP_LAUNCH(m)                                                    \
  (e = vec ? wrs_launch_early(mip_kernel<m, true>, grid, kMipThreads, 0, st, a) \
           : wrs_launch_early(mip_kernel<m, false>, grid, kMipThreads, 0, st, a))
  switch (M) {
    case 1: WRS_MIP_LAUNCH(1); break;
    case 2: WRS_MIP_LAUNCH(2); break;
    case 3: WRS_MIP_LAUNCH(3); break;
    case 4: WRS_MIP_LAUNCH(4); break;
    default: WRS_MIP_LAUNCH(5); break;
  }
#undef WRS_MIP_LAUNCH
  return e == cudaSuccess ? WRS_OK : wrs_cuda_fail(e, "wrs_mip_build: launch");
}

int wrs_fov_check_source(const float* d_img, int64_t pitch, const void* d_mip, size_t mip_bytes,
                   int32_t width, int32_t height, int32_t nradii, const float* radii,
                   int32_t filter, FovDev* out) {
  if (int rc = check_image(width, height)) return rc;
  if (nradii < 1 || nradii > WRS_MAX_MIP_LEVELS - 1 || !radii)
    return wrs_fail(WRS_ERR_ARG, "nradii must be in 1..%d with a radii array",
                    WRS_MAX_MIP_LEVELS - 1);
  if (filter != WRS_FILTER_BOX && filter != WRS_FILTER_BILINEAR)
    return wrs_fail(WRS_ERR_ARG, "filter must be WRS_FILTER_BOX or WRS_FILTER_BILINEAR");
  if (!d_img || !aligned(d_img, 4)) return wrs_fail(WRS_ERR_ARG, "d_img is NULL or unaligned");
  if (pitch < 3 * (int64_t)width)
    return wrs_fail(WRS_ERR_ARG, "img_pitch_elems %lld is below 3 * width", (long long)pitch);
  if (!d_mip || !aligned(d_mip, 256))
    return wrs_fail(WRS_ERR_ARG, "d_mip is NULL or not 256-byte aligned");
  FovDev fv{};
  for (float& r2 : fv.r2) r2 = HUGE_VALF;
  for (int i = 0; i < nradii; ++i) {
    if (!std::isfinite(radii[i]) || !(radii[i] > 0.0f) || (i > 0 && radii[i] < radii[i - 1]))
      return wrs_fail(WRS_ERR_ARG, "radii must be finite, positive and ascending");
    fv.r2[i] = radii[i] * radii[i];
  }
  wrs_mip_layout L;
  if (int rc = wrs_mip_layout_get(width, height, nradii + 1, &L)) return rc;
  if ((int64_t)mip_bytes < L.total_bytes)
    return wrs_fail(WRS_ERR_BUDGET, "mip buffer holds %zu bytes, %d levels need %lld", mip_bytes,
                    nradii + 1, (long long)L.total_bytes);
  fv.img = d_img;
  fv.pitch = pitch;
  fill_levels(L, d_mip, fv.lev);
  *out = fv;
  return WRS_OK;
}

extern "C" int wrs_foveate(const float* d_img, int64_t pitch, const void* d_mip, size_t mip_bytes,
                           int32_t width, int32_t height, int32_t nradii, const float* radii,
                           float gx, float gy, int32_t filter, float* d_frame,
                           int64_t frame_pitch, uint8_t* d_ring, wrs_stream_t stream) {
  wrs_clear_error();
  if (!std::isfinite(gx) || !std::isfinite(gy)) return wrs_fail(WRS_ERR_ARG, "gaze must be finite");
  if (!d_frame || !aligned(d_frame, 4))
    return wrs_fail(WRS_ERR_ARG, "d_frame must be non-NULL and 4-byte aligned");
  if (frame_pitch < 3 * (int64_t)width)
    return wrs_fail(WRS_ERR_ARG, "pitches must be >= 3 * width");
  FovArgs a{};
  if (int rc = wrs_fov_check_source(d_img, pitch, d_mip, mip_bytes, width, height, nradii, radii, filter,
                              &a.fv))
    return rc;
  a.frame = d_frame;
  a.frame_pitch = frame_pitch;
  a.ring = d_ring;
  a.width = width;
  a.height = height;
  a.gx = gx;
  a.gy = gy;
  int sms = 0;
  if (int rc = device_sms(&sms)) return rc;
  const bool quad = width % 4 == 0 && frame_pitch % 4 == 0 && aligned(d_frame, 16) &&
                    (!d_ring || aligned(d_ring, 4));
  const bool box = filter == WRS_FILTER_BOX;
  const int64_t tw = box ? FovTile<WRS_FILTER_BOX>::kW : FovTile<WRS_FILTER_BILINEAR>::kW;
  const int64_t th = box ? FovTile<WRS_FILTER_BOX>::kH : FovTile<WRS_FILTER_BILINEAR>::kH;
  const int64_t want = quad ? ((width + tw - 1) / tw) * ((height + th - 1) / th)
                            : ((int64_t)width * height + kFovThreads - 1) / kFovThreads;
  const int64_t cap = (int64_t)sms * 128;  // about 25 waves of the five CTAs per SM
  const unsigned grid = (unsigned)(want < cap ? want : cap);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const auto kernel = quad ? (box ? foveate4_kernel<WRS_FILTER_BOX>
                                                       : foveate4_kernel<WRS_FILTER_BILINEAR>)
                           : (box ? foveate_kernel<WRS_FILTER_BOX>
                                                       : foveate_kernel<WRS_FILTER_BILINEAR>);
  const cudaError_t e = wrs_launch_early(kernel, dim3(grid), kFovThreads, 0, st, a);
  return e == cudaSuccess ? WRS_OK : wrs_cuda_fail(e, "wrs_foveate: launch");
}
