// K1: depth-ordered over-compositing of cached per-partition RGBA renders into F and B.
// Section 2 builds, per camera, the foreground and background images from the stored renders
// of the frozen partitions in the camera's depth order; by associativity of 'over' the frozen
// blocks in front of the active partition collapse into F, those behind it into B.
//
// Pure streaming work: every layer is read once (16-byte streaming loads, evict-first), the
// accumulator stays in registers across layers, F and B are written once.  Four layers are
// loaded before they are folded, the last one to three of a side together too.  What bounds it is
// the loads an SM has in flight, so the CTAs on an SM count as much as the loads of a thread: fp16
// layers and single pixels keep to 32 registers, eight CTAs, so the grid of eight per SM (which
// strides over the pixel pairs) is resident at once; pairs of 32-bit layers take 40, six CTAs.
// 64 fp16 layers at 1080p take 154 us (6.8 TB/s), 27 at 1236x822 31.8, at 864x600 15.4, at 640x480
// 14.2 (bound by the host); 33 32-bit layers at 1080p 159.5, 27 at 1236x822 65.7.  At seven CTAs
// (36 registers) the fp16 figures are 182, 40.5, 24.8 and 14.0; with a predicated tail of four
// loads (58 registers, pairs of 32-bit layers 86) 174, 41.9, 20.4 and 14.0, and the 32-bit ones 239
// and 97.  Eight layers in flight are slower (215 us at 1080p), one pixel per thread on small
// images too.
#include <algorithm>

#include "abcd_internal.cuh"

namespace abcd {
namespace {

struct LayerTable {
  const void* p[kMaxLayers];   // front layers in order, then back layers in order
};

__device__ __forceinline__ void unpack_h8(uint4 r, float* f) {
  const unsigned w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&w[k]));
    f[2 * k] = v.x;
    f[2 * k + 1] = v.y;
  }
}

__device__ __forceinline__ void unpack_h4(uint2 r, float* f) {
  const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&r.x));
  const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&r.y));
  f[0] = a.x; f[1] = a.y; f[2] = b.x; f[3] = b.y;
}

// acc (premultiplied RGBA x PIX pixels) = acc over layer
template <int PIX>
__device__ __forceinline__ void fold(float* acc, const float* L) {
#pragma unroll
  for (int q = 0; q < PIX; ++q) {
    const float k = 1.f - acc[4 * q + 3];
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[4 * q + c] = __fmaf_rn(k, L[4 * q + c], acc[4 * q + c]);
  }
}

// PIX pixels (4 channels each) of a layer at pixel group g, as loaded.
template <int PIX, bool F16>
struct Raw {
  uint4 r[F16 ? 1 : PIX];
  __device__ __forceinline__ void load(const void* ptr, long long g) {
    if (F16) {
      if (PIX == 2) {
        r[0] = __ldcs(reinterpret_cast<const uint4*>(ptr) + g);
      } else {
        const uint2 v = __ldcs(reinterpret_cast<const uint2*>(ptr) + g);
        r[0] = make_uint4(v.x, v.y, 0u, 0u);
      }
    } else {
#pragma unroll
      for (int q = 0; q < PIX; ++q) r[q] = __ldcs(reinterpret_cast<const uint4*>(ptr) + g * PIX + q);
    }
  }
  __device__ __forceinline__ void unpack(float* f) const {
    if (F16) {
      if (PIX == 2) unpack_h8(r[0], f);
      else unpack_h4(make_uint2(r[0].x, r[0].y), f);
    } else {
#pragma unroll
      for (int q = 0; q < (F16 ? 1 : PIX); ++q) {
        f[4 * q] = __uint_as_float(r[q].x); f[4 * q + 1] = __uint_as_float(r[q].y);
        f[4 * q + 2] = __uint_as_float(r[q].z); f[4 * q + 3] = __uint_as_float(r[q].w);
      }
    }
  }
};

// acc = acc over layers [k, k + N), their loads in flight together.
template <int N, int PIX, bool F16>
__device__ __forceinline__ void fold_n(const LayerTable& lt, int k, long long g, float* acc) {
  Raw<PIX, F16> v[N];
#pragma unroll
  for (int j = 0; j < N; ++j) v[j].load(lt.p[k + j], g);
#pragma unroll
  for (int j = 0; j < N; ++j) {
    float f[4 * PIX];
    v[j].unpack(f);
    fold<PIX>(acc, f);
  }
}

template <int PIX, bool F16>
__device__ __forceinline__ void fold_range(const LayerTable& lt, int k0, int k1, long long g,
                                           float* acc) {
  int k = k0;
  for (; k + 4 <= k1; k += 4) fold_n<4, PIX, F16>(lt, k, g, acc);
  const int rest = k1 - k;
  if (rest == 3) fold_n<3, PIX, F16>(lt, k, g, acc);
  else if (rest == 2) fold_n<2, PIX, F16>(lt, k, g, acc);
  else if (rest == 1) fold_n<1, PIX, F16>(lt, k, g, acc);
}

template <int PIX>
__device__ __forceinline__ void store_group(void* out, int f16, long long g, const float* acc) {
  if (!out) return;
  if (f16) {
    unsigned w[2 * PIX];
#pragma unroll
    for (int k = 0; k < 2 * PIX; ++k) {
      const __half2 h = __floats2half2_rn(acc[2 * k], acc[2 * k + 1]);
      w[k] = *reinterpret_cast<const unsigned*>(&h);
    }
    if (PIX == 2) reinterpret_cast<uint4*>(out)[g] = make_uint4(w[0], w[1], w[2], w[3]);
    else reinterpret_cast<uint2*>(out)[g] = make_uint2(w[0], w[1]);
  } else {
#pragma unroll
    for (int q = 0; q < PIX; ++q)
      reinterpret_cast<float4*>(out)[g * PIX + q] =
          make_float4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]);
  }
}

// (0 CTAs: left to the compiler, which takes 40 registers; six asked for cost it two spills)
template <int PIX, bool F16>
__global__ void __launch_bounds__(256, PIX == 1 || F16 ? 8 : 0)
composite_kernel(const __grid_constant__ LayerTable lt, int nf, int nb, long long groups,
                 void* Fout, void* Bout, int out_f16) {
  pdl_wait();
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < groups;
       g += (long long)gridDim.x * blockDim.x) {
    float acc[4 * PIX];
    if (Fout) {
#pragma unroll
      for (int c = 0; c < 4 * PIX; ++c) acc[c] = 0.f;
      fold_range<PIX, F16>(lt, 0, nf, g, acc);
      store_group<PIX>(Fout, out_f16, g, acc);
    }
    if (Bout) {
#pragma unroll
      for (int c = 0; c < 4 * PIX; ++c) acc[c] = 0.f;
      fold_range<PIX, F16>(lt, nf, nf + nb, g, acc);
      store_group<PIX>(Bout, out_f16, g, acc);
    }
  }
}

}  // namespace
}  // namespace abcd

using namespace abcd;

extern "C" abcd_status abcd_composite_cache(abcd_ctx* ctx, const void* const* layers, int L,
                                            int layer_dtype, const int* order, int split,
                                            int width, int height, void* F_out, void* B_out,
                                            int out_dtype) {
  if (!ctx) return ABCD_ERR_INVALID_ARG;
  if (L < 0 || L > kMaxLayers || (L > 0 && (!layers || !order)) || split < 0 || split > L ||
      width <= 0 || height <= 0)
    return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_composite_cache: bad layer list, split or size");
  if ((layer_dtype != ABCD_F16 && layer_dtype != ABCD_F32) || (out_dtype != ABCD_F16 && out_dtype != ABCD_F32))
    return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_composite_cache: bad dtype");
  LayerTable lt;
  int nf = 0, nb = 0;
  bool al16 = true;
  for (int k = 0; k < L; ++k) {
    if (k == split) continue;
    if (order[k] < 0 || order[k] >= L) return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_composite_cache: order[%d] out of range", k);
    const void* p = layers[order[k]];
    if (!p) return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_composite_cache: layer %d is NULL", order[k]);
    if ((uintptr_t)p & 15) al16 = false;
    if ((uintptr_t)p & (layer_dtype == ABCD_F16 ? 7 : 15))
      return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_composite_cache: layer %d misaligned", order[k]);
    if (k < split) lt.p[nf++] = p;
  }
  for (int k = split + 1; k < L; ++k) lt.p[nf + nb++] = layers[order[k]];
  const long long npix = (long long)width * height;
  const uintptr_t oal = out_dtype == ABCD_F16 ? 7 : 15;
  if (((uintptr_t)F_out & oal) || ((uintptr_t)B_out & oal))
    return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_composite_cache: misaligned output");
  if (((uintptr_t)F_out & 15) || ((uintptr_t)B_out & 15)) al16 = false;
  if (!F_out && !B_out) return ABCD_OK;
  const int grid = ctx->num_sms * 8;
  const bool pairs = al16 && (npix % 2 == 0);
  const bool o16 = out_dtype == ABCD_F16;
  const long long units = pairs ? npix / 2 : npix;
  cudaError_t e;
  if (layer_dtype == ABCD_F16)
    e = pairs ? launch_pdl(composite_kernel<2, true>, dim3(grid), dim3(256), 0, ctx->stream, lt, nf, nb, units, F_out, B_out, o16)
              : launch_pdl(composite_kernel<1, true>, dim3(grid), dim3(256), 0, ctx->stream, lt, nf, nb, units, F_out, B_out, o16);
  else
    e = pairs ? launch_pdl(composite_kernel<2, false>, dim3(grid), dim3(256), 0, ctx->stream, lt, nf, nb, units, F_out, B_out, o16)
              : launch_pdl(composite_kernel<1, false>, dim3(grid), dim3(256), 0, ctx->stream, lt, nf, nb, units, F_out, B_out, o16);
  return check_launch(ctx, "composite_kernel", e);
}

// ---- K1 over packed layers (the cache's tile-sparse format, see abcd_render_refresh_packed):
// one CTA per 16x16 tile, two pixels per thread; a layer whose tile is not stored is transparent,
// and folding (0, 0, 0, 0) leaves the accumulator unchanged, so skipping it gives the dense result
// bit for bit.  Only the stored tiles are read.
namespace abcd {
namespace {

struct PackedTable {
  const int* map[kMaxLayers];       // front layers in order, then back layers in order
  const uint4* data[kMaxLayers];    // 2 KB blocks of 16-byte units: two fp16 RGBA pixels
};

constexpr int kPackedThreads = kTileThreads / 2;
constexpr int kPackedInFlight = 8;
// What bounds the composite is latency -- the tile's map entries, then its layers -- against the
// CTAs that hide it.  Two warps list the layers that store the tile, one per side, so that all eight
// loads a thread has in flight are real; 56 registers keep nine CTAs on an SM.  32 layers at 1237x822
// (16 front, 15 back), 0.1 / 0.4 / 0.9 of the tiles stored: 8.4 / 18.1 / 34.7 us (0.4: 6.6 TB/s) against
// 12.6 / 23.2 / 41.6 without the list (eight layers at a time, the unstored ones masked, eight CTAs).
// F and B by two halves of a 256-thread CTA took 11.6 / 21.1 / 36.2 and left half the CTA idle when
// one side is empty: 16 front layers at 1080p, a tenth stored, 17.7 us against 12.3 here and 15.6
// without the list.  The list as packed words or as addresses is no better; the next grid launched
// early is worse (640x480, 16 and 16 layers, 0.9 stored: 9.3 against 8.7 us).
constexpr int kListCtas = 9;
// Sides of up to kShortLayers layers are folded without the list (F, then B, no shared memory): one
// round of loads of the tile's map entries, one of its layers.  Against the list at 1080p, 0.4 / 0.9
// of the tiles stored: 1 and 1 layers 11.1 / 12.5 against 12.1 / 16.3 us, 4 and 4 15.0 / 22.1 against
// 16.7 / 24.0.  With 5 and 5 a second round of both follows: 15.8 us against 11.8 (a tenth stored).
// A fold of one layer into the accumulator, 0.9 stored: 13.2 against 15.6 us.  Four loads in flight
// and 12 CTAs per SM (40 registers): eight take 8.2 against 6.9 us for 3 layers, 16 CTAs spill.
constexpr int kShortLayers = 4;
constexpr int kShortInFlight = 4;
constexpr int kShortCtas = 12;

// The positions k in [k0, k1) with s_map[k] >= 0, in order, into s_list, and how many into
// *s_count; warp 0 of the calling threads (thread: 0 for the first) compacts with ballots, and
// the caller's next __syncthreads publishes both.
__device__ __forceinline__ void compact_stored(const int* s_map, int k0, int k1, int thread,
                                               int* s_list, int* s_count) {
  if (thread >= 32) return;
  int run = 0;
  for (int b = k0; b < k1; b += 32) {
    const bool st = b + thread < k1 && s_map[b + thread] >= 0;
    const unsigned m = __ballot_sync(0xffffffffu, st);
    if (st) s_list[run + __popc(m & ((1u << thread) - 1u))] = b + thread;
    run += __popc(m);
  }
  if (thread == 0) *s_count = run;
}

// Calls fn(k, v) in order for the listed positions s_list[j0 .. j1) (v: this thread's 16-byte
// unit of layer k's block at the tile), the loads of kPackedInFlight blocks in flight before
// they are used.
template <typename Fn>
__device__ __forceinline__ void for_each_listed(const uint4* const* data, const int* s_map,
                                                const int* s_list, int j0, int j1, int unit,
                                                Fn fn) {
  int j = j0;
  for (; j + kPackedInFlight <= j1; j += kPackedInFlight) {
    uint4 r[kPackedInFlight];
#pragma unroll
    for (int i = 0; i < kPackedInFlight; ++i) {
      const int k = s_list[j + i];
      r[i] = __ldcs(data[k] + (size_t)s_map[k] * kPackedThreads + unit);
    }
#pragma unroll
    for (int i = 0; i < kPackedInFlight; ++i) fn(s_list[j + i], r[i]);
  }
  if (j < j1) {
    uint4 r[kPackedInFlight];
#pragma unroll
    for (int i = 0; i < kPackedInFlight; ++i) {
      if (j + i >= j1) break;
      const int k = s_list[j + i];
      r[i] = __ldcs(data[k] + (size_t)s_map[k] * kPackedThreads + unit);
    }
#pragma unroll
    for (int i = 0; i < kPackedInFlight; ++i) {
      if (j + i >= j1) break;
      fn(s_list[j + i], r[i]);
    }
  }
}

__device__ __forceinline__ void store_pixel_out(void* out, int f16, long long p, const float* acc) {
  if (f16) {
    const __half2 lo = __floats2half2_rn(acc[0], acc[1]), hi = __floats2half2_rn(acc[2], acc[3]);
    reinterpret_cast<uint2*>(out)[p] = make_uint2(*reinterpret_cast<const unsigned*>(&lo),
                                                  *reinterpret_cast<const unsigned*>(&hi));
  } else {
    reinterpret_cast<float4*>(out)[p] = make_float4(acc[0], acc[1], acc[2], acc[3]);
  }
}

// Layers [k0, k1) folded into acc without the list: each thread reads the tile's map entries
// itself, then has the stored layers' loads in flight together, kShortInFlight layers at a time.
__device__ __forceinline__ void fold_short(const PackedTable& pt, int k0, int k1, int tile, int unit,
                                           float* acc) {
  for (; k0 < k1; k0 += kShortInFlight) {
    int m[kShortInFlight];
    uint4 r[kShortInFlight];
#pragma unroll
    for (int i = 0; i < kShortInFlight; ++i) m[i] = k0 + i < k1 ? __ldg(pt.map[k0 + i] + tile) : -1;
#pragma unroll
    for (int i = 0; i < kShortInFlight; ++i)
      if (m[i] >= 0) r[i] = __ldcs(pt.data[k0 + i] + (size_t)m[i] * kPackedThreads + unit);
#pragma unroll
    for (int i = 0; i < kShortInFlight; ++i) {
      if (m[i] < 0) continue;
      float f[8];
      unpack_h8(r[i], f);
      fold<2>(acc, f);
    }
  }
}

// A layer that stores the tile: its position in the table and the tile's block.
struct Stored {
  int layer, block;
};

// The layers of [k0, k1) that store the tile, in order, into list (one warp); returns how many.
__device__ __forceinline__ int list_stored(const PackedTable& pt, int k0, int k1, int tile, Stored* list) {
  constexpr int kMaps = 4;                             // map entries a lane has in flight
  const int lane = threadIdx.x & 31;
  int run = 0;
  for (int b = k0; b < k1; b += 32 * kMaps) {
    int m[kMaps];
#pragma unroll
    for (int i = 0; i < kMaps; ++i) {
      const int k = b + 32 * i + lane;
      m[i] = k < k1 ? __ldg(pt.map[k] + tile) : -1;
    }
#pragma unroll
    for (int i = 0; i < kMaps; ++i) {
      const unsigned st = __ballot_sync(0xffffffffu, m[i] >= 0);
      if (m[i] >= 0) list[run + __popc(st & ((1u << lane) - 1u))] = {b + 32 * i + lane, m[i]};
      run += __popc(st);
    }
  }
  return run;
}

// acc (2 pixels) = acc over the listed layers [j, j1), the loads of kPackedInFlight in flight together.
__device__ __forceinline__ void fold_listed(const PackedTable& pt, const Stored* list, int j, int j1,
                                            int unit, float* acc) {
  for (; j < j1; j += kPackedInFlight) {
    uint4 r[kPackedInFlight];
#pragma unroll
    for (int i = 0; i < kPackedInFlight; ++i) {
      if (j + i >= j1) continue;
      const Stored e = list[j + i];
      r[i] = __ldcs(pt.data[e.layer] + (size_t)e.block * kPackedThreads + unit);
    }
#pragma unroll
    for (int i = 0; i < kPackedInFlight; ++i) {
      if (j + i >= j1) break;
      float f[8];
      unpack_h8(r[i], f);
      fold<2>(acc, f);
    }
  }
}

// F, then B, by 128 threads; SHORT: sides of at most kShortLayers layers.
template <bool SHORT>
__global__ void __launch_bounds__(kPackedThreads, SHORT ? kShortCtas : kListCtas)
composite_packed_kernel(const __grid_constant__ PackedTable pt, int nf, int nb, int width,
                        int height, int tiles_x, void* Fout, void* Bout, int out_f16) {
  pdl_wait();
  __shared__ Stored s_list[SHORT ? 1 : kMaxLayers];
  __shared__ int s_end[2];
  const int tile = blockIdx.x;
  const int unit = threadIdx.x;                       // pixels 2 unit, 2 unit + 1 of the tile
  const int r = unit / (kTile / 2), c = 2 * (unit % (kTile / 2));
  const int y = (tile / tiles_x) * kTile + r, x = (tile % tiles_x) * kTile + c;
  if (!SHORT) {
    if (unit < 64) {
      const int side = unit >> 5, k0 = side ? nf : 0, k1 = side ? nf + nb : nf;
      const int n = list_stored(pt, k0, k1, tile, s_list + k0);
      if ((unit & 31) == 0) s_end[side] = k0 + n;
    }
    __syncthreads();
  }
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    void* out = side ? Bout : Fout;
    if (!out) continue;
    float acc[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[q] = 0.f;
    if (SHORT) fold_short(pt, side ? nf : 0, side ? nf + nb : nf, tile, unit, acc);
    else fold_listed(pt, s_list, side ? nf : 0, s_end[side], unit, acc);
    if (y >= height) continue;
    if (x < width) store_pixel_out(out, out_f16, (long long)y * width + x, acc);
    if (x + 1 < width) store_pixel_out(out, out_f16, (long long)y * width + x + 1, acc + 4);
  }
}

// One side's left fold continued from an fp32 accumulator: acc = acc over the listed layers, in
// order (acc_in NULL: from transparent); the accumulator goes back in fp32 (acc_out) and/or as
// its fp16 rounding (out16).  The fold runs the same fp32 operations in the same order as
// composite_packed_kernel, so folding the layers in pieces gives its result bit for bit; SHORT as there.
template <bool SHORT>
__global__ void __launch_bounds__(kPackedThreads, SHORT ? kShortCtas : kListCtas)
fold_packed_kernel(const __grid_constant__ PackedTable pt, int n, int width, int height,
                   int tiles_x, const float4* acc_in, float4* acc_out, uint2* out16) {
  pdl_wait();
  __shared__ Stored s_list[SHORT ? 1 : kMaxLayers];
  __shared__ int s_end;
  const int tile = blockIdx.x;
  const int unit = threadIdx.x;
  if (!SHORT && unit < 32) {
    const int k = list_stored(pt, 0, n, tile, s_list);
    if (unit == 0) s_end = k;
  }
  const int r = unit / (kTile / 2), c = 2 * (unit % (kTile / 2));
  const int y = (tile / tiles_x) * kTile + r, x = (tile % tiles_x) * kTile + c;
  const long long p0 = (long long)y * width + x;
  const bool in0 = y < height && x < width, in1 = y < height && x + 1 < width;
  float acc[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) acc[q] = 0.f;
  if (acc_in) {
    if (in0) { const float4 a = acc_in[p0]; acc[0] = a.x; acc[1] = a.y; acc[2] = a.z; acc[3] = a.w; }
    if (in1) { const float4 a = acc_in[p0 + 1]; acc[4] = a.x; acc[5] = a.y; acc[6] = a.z; acc[7] = a.w; }
  }
  if (SHORT) {
    fold_short(pt, 0, n, tile, unit, acc);
  } else {
    __syncthreads();
    fold_listed(pt, s_list, 0, s_end, unit, acc);
  }
  if (in0) {
    if (acc_out) acc_out[p0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
    if (out16) store_pixel_out(out16, 1, p0, acc);
  }
  if (in1) {
    if (acc_out) acc_out[p0 + 1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
    if (out16) store_pixel_out(out16, 1, p0 + 1, acc + 4);
  }
}

}  // namespace
}  // namespace abcd

extern "C" abcd_status abcd_composite_fold_packed(abcd_ctx* ctx, const int* const* tile_maps,
                                                  const void* const* packed, int count,
                                                  int width, int height, const float* acc_in,
                                                  float* acc_out, void* out16) {
  if (!ctx) return ABCD_ERR_INVALID_ARG;
  if (count < 0 || count > kMaxLayers || (count > 0 && (!tile_maps || !packed)) || width <= 0 ||
      height <= 0)
    return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_composite_fold_packed: bad layer list or size");
  if (((uintptr_t)acc_in & 15) || ((uintptr_t)acc_out & 15) || ((uintptr_t)out16 & 7))
    return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_composite_fold_packed: misaligned accumulator or output");
  PackedTable pt;
  for (int k = 0; k < count; ++k) {
    const int* m = tile_maps[k];
    const void* d = packed[k];
    if (!m || !d) return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_composite_fold_packed: layer %d is NULL", k);
    if (((uintptr_t)d & 15) || ((uintptr_t)m & 3))
      return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_composite_fold_packed: layer %d misaligned", k);
    pt.map[k] = m;
    pt.data[k] = (const uint4*)d;
  }
  if (!acc_out && !out16) return ABCD_OK;
  const int tiles_x = (width + kTile - 1) / kTile, tiles_y = (height + kTile - 1) / kTile;
  return check_launch(ctx, "fold_packed_kernel",
                      launch_pdl(count <= kShortLayers ? fold_packed_kernel<true> : fold_packed_kernel<false>,
                                 dim3(tiles_x * tiles_y), dim3(kPackedThreads), 0, ctx->stream, pt, count,
                                 width, height, tiles_x,
                                 (const float4*)acc_in, (float4*)acc_out, (uint2*)out16));
}

extern "C" abcd_status abcd_composite_cache_packed(abcd_ctx* ctx, const int* const* tile_maps,
                                                   const void* const* packed, int L,
                                                   const int* order, int split, int width,
                                                   int height, void* F_out, void* B_out,
                                                   int out_dtype) {
  if (!ctx) return ABCD_ERR_INVALID_ARG;
  if (L < 0 || L > kMaxLayers || (L > 0 && (!tile_maps || !packed || !order)) || split < 0 ||
      split > L || width <= 0 || height <= 0)
    return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_composite_cache_packed: bad layer list, split or size");
  if (out_dtype != ABCD_F16 && out_dtype != ABCD_F32)
    return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_composite_cache_packed: bad dtype");
  PackedTable pt;
  int nf = 0, nb = 0;
  for (int k = 0; k < L; ++k) {
    if (k == split) continue;
    if (order[k] < 0 || order[k] >= L)
      return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_composite_cache_packed: order[%d] out of range", k);
    const int* m = tile_maps[order[k]];
    const void* d = packed[order[k]];
    if (!m || !d) return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_composite_cache_packed: layer %d is NULL", order[k]);
    if (((uintptr_t)d & 15) || ((uintptr_t)m & 3))
      return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_composite_cache_packed: layer %d misaligned", order[k]);
    const int slot = k < split ? nf++ : -1;
    if (slot >= 0) { pt.map[slot] = m; pt.data[slot] = (const uint4*)d; }
  }
  for (int k = split + 1; k < L; ++k) {
    pt.map[nf + nb] = tile_maps[order[k]];
    pt.data[nf + nb] = (const uint4*)packed[order[k]];
    ++nb;
  }
  const uintptr_t oal = out_dtype == ABCD_F16 ? 7 : 15;
  if (((uintptr_t)F_out & oal) || ((uintptr_t)B_out & oal))
    return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_composite_cache_packed: misaligned output");
  if (!F_out && !B_out) return ABCD_OK;
  const int tiles_x = (width + kTile - 1) / kTile, tiles_y = (height + kTile - 1) / kTile;
  const int out_f16 = out_dtype == ABCD_F16 ? 1 : 0;
  const bool few = std::max(nf, nb) <= kShortLayers;
  return check_launch(ctx, "composite_packed_kernel",
                      launch_pdl(few ? composite_packed_kernel<true> : composite_packed_kernel<false>,
                                 dim3(tiles_x * tiles_y), dim3(kPackedThreads), 0, ctx->stream, pt,
                                 nf, nb, width, height, tiles_x, F_out, B_out, out_f16));
}

// ---- visibility of the layers of one camera's depth order (Section 4: visibility thresholds
// and occlusion culling of camera-partition pairs).  For the layer at position k, with alpha_k
// its alpha and T_k the product of (1 - alpha) over the layers before it, visible = mean over
// pixels of alpha_k T_k and coverage = mean of alpha_k.  Leaving a set D of layers out of the
// composite changes every channel of every pixel by at most the sum over D of alpha_j T_j
// (colours premultiplied and at most alpha), so the dropped layers' visible shares bound the
// mean error of a culled composite.
// One CTA per 16x16 tile at a time (a grid that strides over tiles), two pixels per thread, T
// in registers across the order.  Sums are exact: every value is rounded to 24-bit fixed point
// and added as an integer (a warp reduction, then 64-bit shared and global accumulators), so
// the result does not depend on the order of the additions; CTAs add to one of kVisCopies
// copies of the global sums (fewer atomics on one address) and the last CTA to finish adds the
// copies, converts them to means and clears them for the next call.
namespace abcd {
namespace {

constexpr float kVisScale = 16777216.f;       // 2^24
constexpr int kVisInFlight = 8;               // layers whose loads are in flight together
// Most positions with sums per thread.  A position takes 1 KB of a CTA's shared memory, and what that
// leaves bounds the rest: packed layers, streamed past the L1, need the five CTAs that 32 positions
// allow on an SM; dense ones, of which the two loads of a pixel pair share cache lines, need the L1
// that eight CTAs of 14 leave.  Above, a warp reduction and a shared atomic per layer, tile and sum
// (both forms are bound by latency: 3.4 of 6.8 TB/s).  At 1237x822 (us, sums per thread / reduction):
// packed, 0.4 of the tiles stored, 20 layers 17 / 23, 32: 27 / 32, 33: 33 / 33, 64: 87 / 53; at 1080p,
// a tenth stored, 32: 22 / 28, 33: 34 / 30.  Dense 12 layers 23 / 29, 14: 26 / 32, 16: 44 / 35,
// 32: 85 / 61.
constexpr int kVisOwnPacked = 32;
constexpr int kVisOwnDense = 14;
constexpr int kVisCopies = kVisSumCopies;     // global accumulators (CTA b adds to copy b % 8)

struct VisTable {
  const int* map[kMaxLayers];                 // packed: tile map per position of the order
  const uint4* data[kMaxLayers];              // packed: 2 KB blocks; dense: half [H][W][4]
  int layer[kMaxLayers];                      // layer index at each position
};

// Adds one layer's contribution at the thread's two pixels (alphas a0, a1) to the sums of position
// k, then takes the layer's transmittance factor into T0, T1.  OWN: into the thread's own pair of
// 32-bit sums (no reduction and no atomic per layer and tile); else into the CTA's, through a warp
// reduction.  Warp-uniform k.
template <bool OWN>
__device__ __forceinline__ void vis_accumulate(float a0, float a1, float& T0, float& T1, int k,
                                               unsigned long long (*s_sum)[kMaxLayers], uint2* s_own) {
  const unsigned vf = __float2uint_rn(a0 * T0 * kVisScale) + __float2uint_rn(a1 * T1 * kVisScale);
  const unsigned cf = __float2uint_rn(a0 * kVisScale) + __float2uint_rn(a1 * kVisScale);
  T0 *= 1.f - a0;
  T1 *= 1.f - a1;
  if (OWN) {
    uint2& o = s_own[k * kPackedThreads + threadIdx.x];
    o = make_uint2(o.x + vf, o.y + cf);
    return;
  }
  const unsigned vs = __reduce_add_sync(0xffffffffu, vf);
  const unsigned cs = __reduce_add_sync(0xffffffffu, cf);
  if ((threadIdx.x & 31) == 0) {
    if (vs) atomicAdd(&s_sum[0][k], (unsigned long long)vs);
    if (cs) atomicAdd(&s_sum[1][k], (unsigned long long)cs);
  }
}

__device__ __forceinline__ float alpha_hi(unsigned w) {
  return __high2float(*reinterpret_cast<const __half2*>(&w));
}

template <bool PACKED, bool OWN>
__global__ void __launch_bounds__(kPackedThreads, 10)
visibility_kernel(const __grid_constant__ VisTable vt, int count, int L, int width, int height,
                  int tiles_x, int n_tiles, unsigned long long* sums, unsigned* ticket,
                  double* visible, double* coverage) {
  pdl_wait();
  __shared__ unsigned long long s_sum[2][kMaxLayers];
  __shared__ int s_map[kMaxLayers];
  __shared__ int s_list[kMaxLayers];
  __shared__ int s_count;
  __shared__ bool s_last;
  extern __shared__ uint2 s_own[];                     // OWN: [count][kPackedThreads]
  for (int k = threadIdx.x; k < count; k += blockDim.x) { s_sum[0][k] = 0ull; s_sum[1][k] = 0ull; }
  if (OWN)
    for (int k = 0; k < count; ++k) s_own[k * kPackedThreads + threadIdx.x] = make_uint2(0u, 0u);
  const int unit = threadIdx.x;
  const int r = unit / (kTile / 2), c = 2 * (unit % (kTile / 2));
  for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    __syncthreads();                                   // s_map, s_list of the previous tile done
    if (PACKED) {
      for (int k = threadIdx.x; k < count; k += blockDim.x) s_map[k] = __ldg(vt.map[k] + tile);
      __syncthreads();
      compact_stored(s_map, 0, count, unit, s_list, &s_count);
    }
    __syncthreads();
    const int y = (tile / tiles_x) * kTile + r, x = (tile % tiles_x) * kTile + c;
    const bool in0 = y < height && x < width, in1 = y < height && x + 1 < width;
    float T0 = 1.f, T1 = 1.f;
    if (PACKED) {
      for_each_listed(vt.data, s_map, s_list, 0, s_count, unit, [&](int k, uint4 u) {
        vis_accumulate<OWN>(in0 ? alpha_hi(u.y) : 0.f, in1 ? alpha_hi(u.w) : 0.f, T0, T1, k, s_sum, s_own);
      });
      continue;
    }
    const long long p = (long long)y * width + x;
    for (int k0 = 0; k0 < count; k0 += kVisInFlight) {
      // the loads of kVisInFlight layers are issued before any is used (they do not depend on
      // T), so a tile waits for memory once per group instead of once per layer
      unsigned w0[kVisInFlight], w1[kVisInFlight];
#pragma unroll
      for (int j = 0; j < kVisInFlight; ++j) {
        w0[j] = w1[j] = 0u;
        const int k = k0 + j;
        if (k >= count) continue;
        const uint2* d = reinterpret_cast<const uint2*>(vt.data[k]);
        if (in0) w0[j] = __ldcs(d + p).y;
        if (in1) w1[j] = __ldcs(d + p + 1).y;
      }
#pragma unroll
      for (int j = 0; j < kVisInFlight; ++j)
        if (k0 + j < count)
          vis_accumulate<OWN>(alpha_hi(w0[j]), alpha_hi(w1[j]), T0, T1, k0 + j, s_sum, s_own);
    }
  }
  __syncthreads();
  if (OWN) {                                           // the threads' sums of each position: one warp
    const int lane = threadIdx.x & 31;
    for (int k = threadIdx.x >> 5; k < count; k += kPackedThreads / 32) {
      unsigned long long v = 0ull, cv = 0ull;
#pragma unroll
      for (int q = 0; q < kPackedThreads / 32; ++q) {
        const uint2 o = s_own[k * kPackedThreads + q * 32 + lane];
        v += o.x;
        cv += o.y;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        v += __shfl_xor_sync(0xffffffffu, v, o);
        cv += __shfl_xor_sync(0xffffffffu, cv, o);
      }
      if (lane == 0) { s_sum[0][k] = v; s_sum[1][k] = cv; }
    }
    __syncthreads();
  }
  unsigned long long* mine = sums + (size_t)(blockIdx.x % kVisCopies) * 2 * kMaxLayers;
  for (int k = threadIdx.x; k < count; k += blockDim.x) {
    if (s_sum[0][k]) atomicAdd(mine + k, s_sum[0][k]);
    if (s_sum[1][k]) atomicAdd(mine + kMaxLayers + k, s_sum[1][k]);
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const double inv = 1.0 / ((double)kVisScale * (double)width * (double)height);
  for (int j = threadIdx.x; j < L; j += blockDim.x) {
    visible[j] = 0.0;
    if (coverage) coverage[j] = 0.0;
  }
  __syncthreads();
  for (int k = threadIdx.x; k < count; k += blockDim.x) {
    unsigned long long v = 0ull, cv = 0ull;
    for (int cp = 0; cp < kVisCopies; ++cp) {
      v += atomicExch(sums + (size_t)cp * 2 * kMaxLayers + k, 0ull);
      cv += atomicExch(sums + (size_t)cp * 2 * kMaxLayers + kMaxLayers + k, 0ull);
    }
    visible[vt.layer[k]] = (double)v * inv;
    if (coverage) coverage[vt.layer[k]] = (double)cv * inv;
  }
  if (threadIdx.x == 0) *ticket = 0u;
}

// Checks the order and the outputs, fills vt.layer and launches.
abcd_status visibility_launch(abcd_ctx* ctx, const char* who, VisTable& vt, bool packed, int L,
                              const int* order, int count, int width, int height,
                              double* visible, double* coverage) {
  if (!visible || ((uintptr_t)visible & 7) || ((uintptr_t)coverage & 7))
    return fail(ctx, ABCD_ERR_INVALID_ARG, "%s: null or misaligned output", who);
  const int tiles_x = (width + kTile - 1) / kTile, tiles_y = (height + kTile - 1) / kTile;
  const int n_tiles = tiles_x * tiles_y;
  // per-thread sums while they leave enough CTAs and L1 (kVisOwnPacked, kVisOwnDense), and cannot
  // overflow: a tile adds at most 2^25 to a 32-bit sum
  const size_t own_bytes = sizeof(uint2) * kPackedThreads * (size_t)count;
  const int own_ctas = std::max(1, std::min<int>(8, (int)((200u << 10) / (own_bytes + (8u << 10)))));
  const bool own = count <= (packed ? kVisOwnPacked : kVisOwnDense) &&
                   n_tiles <= 64LL * own_ctas * ctx->num_sms;
  const int grid = std::max(1, std::min(n_tiles, (own ? own_ctas : 8) * ctx->num_sms));
  const size_t smem = own ? own_bytes : 0;
  const auto kernel = packed ? (own ? visibility_kernel<true, true> : visibility_kernel<true, false>)
                             : (own ? visibility_kernel<false, true> : visibility_kernel<false, false>);
  const cudaError_t e = allow_smem(ctx, (const void*)kernel);
  if (e != cudaSuccess) return fail(ctx, ABCD_ERR_CUDA, "%s smem: %s", who, cudaGetErrorString(e));
  return check_launch(ctx, "visibility_kernel",
                      launch_pdl(kernel, dim3(grid), dim3(kPackedThreads), smem, ctx->stream, vt,
                                 count, L, width, height, tiles_x, n_tiles, ctx->ws.vis_sums,
                                 ctx->ws.vis_ticket, visible, coverage));
}

// The order: count distinct indices below L.
bool valid_order(const int* order, int count, int L) {
  unsigned char seen[kMaxLayers] = {0};
  for (int k = 0; k < count; ++k) {
    if (order[k] < 0 || order[k] >= L || seen[order[k]]) return false;
    seen[order[k]] = 1;
  }
  return true;
}

}  // namespace
}  // namespace abcd

extern "C" abcd_status abcd_layer_visibility(abcd_ctx* ctx, const void* const* layers, int L,
                                             const int* order, int count, int width, int height,
                                             double* visible, double* coverage) {
  if (!ctx) return ABCD_ERR_INVALID_ARG;
  if (!has_workspace(ctx)) return fail(ctx, ABCD_ERR_WORKSPACE, "abcd_layer_visibility: no workspace");
  if (L < 0 || L > kMaxLayers || count < 0 || count > L || (count > 0 && (!layers || !order)) ||
      width <= 0 || height <= 0 || !valid_order(order, count, L))
    return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_layer_visibility: bad layer list, order or size");
  VisTable vt;
  for (int k = 0; k < count; ++k) {
    const void* p = layers[order[k]];
    if (!p || ((uintptr_t)p & 7))
      return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_layer_visibility: layer %d is NULL or misaligned", order[k]);
    vt.map[k] = nullptr;
    vt.data[k] = static_cast<const uint4*>(p);
    vt.layer[k] = order[k];
  }
  return visibility_launch(ctx, "abcd_layer_visibility", vt, false, L, order, count, width,
                           height, visible, coverage);
}

extern "C" abcd_status abcd_layer_visibility_packed(abcd_ctx* ctx, const int* const* tile_maps,
                                                    const void* const* packed, int L,
                                                    const int* order, int count, int width,
                                                    int height, double* visible,
                                                    double* coverage) {
  if (!ctx) return ABCD_ERR_INVALID_ARG;
  if (!has_workspace(ctx)) return fail(ctx, ABCD_ERR_WORKSPACE, "abcd_layer_visibility_packed: no workspace");
  if (L < 0 || L > kMaxLayers || count < 0 || count > L ||
      (count > 0 && (!tile_maps || !packed || !order)) || width <= 0 || height <= 0 ||
      !valid_order(order, count, L))
    return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_layer_visibility_packed: bad layer list, order or size");
  VisTable vt;
  for (int k = 0; k < count; ++k) {
    const int* m = tile_maps[order[k]];
    const void* d = packed[order[k]];
    if (!m || !d || ((uintptr_t)d & 15) || ((uintptr_t)m & 3))
      return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_layer_visibility_packed: layer %d is NULL or misaligned", order[k]);
    vt.map[k] = m;
    vt.data[k] = static_cast<const uint4*>(d);
    vt.layer[k] = order[k];
  }
  return visibility_launch(ctx, "abcd_layer_visibility_packed", vt, true, L, order, count,
                           width, height, visible, coverage);
}
