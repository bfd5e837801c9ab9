// K5 (blend + composite forward, also the cache refresh K10) and K7 (its backward).
//
// Per pixel, front to back over its tile's list (3DGS blending): sigma = 1/2 d^T Q d with
// d = pixel centre - uv, alpha = min(alpha_max, o exp(-sigma)), skip alpha < alpha_min (and
// sigma < 0), stop before T (1 - alpha) < t_min; A = (sum T_i alpha_i c_i, 1 - T).  Then the
// frozen partitions enter through out = F over (A over B) (Section 2), over meaning
// X + (1 - X.a) Y on premultiplied RGBA, and out.rgb += (1 - out.a) bg.
//
// One warp per 8x8 block of pixels (four per 16x16 binning tile), two pixels per lane --
// (x, y) and (x + 4, y), which share the shared-memory loads and the dy terms of sigma -- so
// the few heavily covered tiles of a small active block spread over four times as many CTAs,
// each lane runs two independent blend chains, and each CTA stops as soon as its own 64
// pixels have terminated.  List entries are staged in shared memory; an entry whose opacity
// cannot reach alpha_min anywhere on the CTA's pixel-centre box (analytic minimum of the
// quadratic form over the box, with a margin far above fp32 rounding) is dropped while
// staging -- every pixel would skip it, so results are unchanged -- and 64 list positions are
// loaded at a time, so the blocks that walk a long list whose entries mostly miss them are not
// bound by one load round trip per few entries.  What decides whether an entry counts at a pixel
// (sigma and its limit) is computed with explicit round-to-nearest intrinsics in one shared
// function, so the backward kernel retraces exactly the forward's contributors (the forward's
// position of the last one says where a pixel ended).
//
// Work is very uneven across blocks (lists of a few entries next to lists of 15,000), so both
// kernels take their tiles in the order bin_sort left in the workspace (decreasing list
// length) when it was made for the ranges they are given: the longest blocks start in the
// first wave instead of trailing the launch.  The order changes no result (CTAs are
// independent; the backward's gradient sums are atomic either way).
#include "abcd_internal.cuh"

namespace abcd {
namespace {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kHalfLog2e = 0.7213475204444817f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr float kFarSigma = 1e30f;               // 2^-kFarSigma is 0

constexpr int kSub = 8;                          // CTA pixel block edge
constexpr int kSubThreads = 32;                  // one warp, two pixels per lane
constexpr int kSubPerTile = (kTile / kSub) * (kTile / kSub);
static_assert(kSubPerTile == kRenderSubPerTile, "tile order expands to kRenderSubPerTile CTAs per tile");
constexpr int kRounds = 2;                       // list entries per lane per staging group
constexpr int kGroup = kSubThreads * kRounds;    // 64 entries loaded together
constexpr int kFwdUnroll = 4;                    // staged entries per iteration
constexpr int kFwdRounds = 2;
constexpr int kFwdGroup = kFwdRounds * kSubThreads;   // list positions the forward stages together
constexpr int kCkChunk = 128;                    // list positions per backward chunk
constexpr int kBwdUnroll = 5;                    // staged entries per iteration of the backward
constexpr int kItemCtasPerSm = 16;               // backward CTAs that replay listed chunks
static_assert(kCkChunk % kGroup == 0 && kCkChunk % kFwdGroup == 0,
              "checkpoints fall on staging group boundaries");

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Conic scaled for base-2 exponentials: (a/2, b, c/2) * log2(e), opacity kept.
__device__ __forceinline__ float4 scaled_conic(float4 c) {
  return make_float4(__fmul_rn(kHalfLog2e, c.x), __fmul_rn(kLog2e, c.y), __fmul_rn(kHalfLog2e, c.z), c.w);
}

// sigma * log2(e) = dx (a/2 dx + b dy) + c/2 dy^2 at the lane's two pixels (fx.x, fy) and
// (fx.y, fy), nm the negated mean; the dy terms are shared.  Both kernels take every branch
// decision from these bits.  The two pixels go through the packed two-lane fp32 instructions,
// whose every component is rounded exactly as the scalar instruction would round it.
__device__ __forceinline__ void sigma_pair(float4 s, float4 nm, float2 fx, float fy, float2& dx,
                                           float& dy, float2& sg) {
  dy = __fadd_rn(fy, nm.y);
  dx = __fadd2_rn(fx, make_float2(nm.x, nm.x));
  const float bdy = __fmul_rn(s.y, dy);
  const float cdy2 = __fmaf_rn(__fmul_rn(s.z, dy), dy, 0.f);   // + 0: sigma is never -0
  const float2 in = __ffma2_rn(make_float2(s.x, s.x), dx, make_float2(bdy, bdy));
  sg = __ffma2_rn(dx, in, make_float2(cdy2, cdy2));
}

__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Least value of sigma * log2(e) over the box [X0, X0 + 7] x [Y0, Y0 + 7] of offsets d = pixel -
// uv.  For a positive definite conic it lies on an edge that faces d = 0 (on any other edge q
// falls towards d = 0), so at most one edge of each direction counts: x = Xe, the x of the box
// nearest to 0, with the other coordinate's minimiser clamped into the box, and y = Ye likewise
// (when 0 lies in the x range, Xe = 0 is no edge but a point of the box, which does no harm).
__device__ __forceinline__ float box_min_sigma2(float4 s, float X0, float Y0) {
  const float X1 = X0 + (kSub - 1), Y1 = Y0 + (kSub - 1);
  const float Xe = fmaxf(X0, fminf(X1, 0.f)), Ye = fmaxf(Y0, fminf(Y1, 0.f));
  const float hb = -0.5f * s.y;
  const float yx = fminf(fmaxf(hb * rcp_approx(s.z) * Xe, Y0), Y1);
  const float xy = fminf(fmaxf(hb * rcp_approx(s.x) * Ye, X0), X1);
  const float q0 = Xe * (s.x * Xe + s.y * yx) + s.z * yx * yx;
  const float q1 = xy * (s.x * xy + s.y * Ye) + s.z * Ye * Ye;
  return fminf(q0, q1);
}

// Whether an entry of opacity o has alpha >= alpha_min at the sigma * log2(e) of these bits.
__device__ __forceinline__ bool passes(float o, int bits, const Opts& op) {
  return __fmul_rn(o, ex2_approx(-__int_as_float(bits))) >= op.alpha_min;
}

// Largest sigma * log2(e) at which an entry of opacity o still has alpha >= alpha_min, or -1 for
// an entry that never does.  A pixel takes the entry iff 0 <= sigma' <= the limit, one unsigned
// comparison of the two values' bits (a negative or NaN sigma' is above every limit).  The limit
// is the last float at which the alpha itself, o ex2.approx(-sigma'), passes (ex2.approx never rises
// as its argument falls), so a pixel is decided as its alpha would decide it.  It is looked for within
// two floats of log2(o / alpha_min) as lg2.approx gives it, which finds it for every float opacity
// from 4 alpha_min on (tried with ten alpha_min from 1e-36 to 0.3); for a fainter one limit_of_faint
// makes it exact.
__device__ __forceinline__ float sigma_limit(float o, const Opts& op) {
  const float l = fmaxf(__log2f(o * op.inv_alpha_min), 0.f);
  const int bits = max(__float_as_int(l), 2);
  float lim = __int_as_float(bits - 2);
#pragma unroll
  for (int k = -1; k <= 2; ++k)
    if (passes(o, bits + k, op)) lim = __int_as_float(bits + k);
  return ((o >= op.alpha_min) & (op.alpha_max >= op.alpha_min)) ? fmaxf(lim, op.least_limit) : -1.f;
}

// The exact limit of a staged entry below 4 alpha_min (lim >= 0: what sigma_limit gave).  There the
// logarithm is below 2 and its floats come closer than the 3e-7 by which it and ex2.approx are off:
// 13% of the opacities from 1.5 to 2 alpha_min and 77% from 1.01 to 1.2 need the bisection, of about
// 5 and 12 steps.  (The block cull's margin is far above what it changes.)
__device__ __forceinline__ float limit_of_faint(float lim, float o, const Opts& op) {
  const int bits = __float_as_int(lim);
  if (!(o < op.faint) || (passes(o, bits, op) && !passes(o, bits + 1, op))) return lim;
  constexpr float kErr = 4.76837158203125e-7f;         // 2^-21
  const float l = __log2f(o * op.inv_alpha_min);
  const int a = __float_as_int(fmaxf(l - kErr, 0.f)), b = __float_as_int(fmaxf(l, 0.f) + kErr);
  int lo = passes(o, a, op) ? a : 0, hi = passes(o, b, op) ? 0x7f800000 : b;   // alpha: o at 0, 0 at inf
  while (hi - lo > 1) {
    const int m = lo + ((hi - lo) >> 1);
    if (passes(o, m, op)) lo = m;
    else hi = m;
  }
  return __int_as_float(lo);
}

__device__ __forceinline__ bool takes(float sg, float lim) {
  return __float_as_uint(sg) <= __float_as_uint(lim);
}

// True when no pixel centre of the CTA's box can reach the limit (sigma_limit); the margin (0.02
// + 0.2% in log2 units) is orders of magnitude above the fp32 error of either evaluation.  A
// conic that is not positive definite is never culled.
__device__ __forceinline__ bool cull(float4 s, float2 m, float bx0, float by0, float lim) {
  const bool pd = (s.x > 0.f) & (s.z > 0.f) & (4.f * s.x * s.z > s.y * s.y);
  const bool out = box_min_sigma2(s, bx0 - m.x, by0 - m.y) * 0.998f > lim + 0.02f;
  return !(lim >= 0.f) | (pd & out);
}

__device__ __forceinline__ float4 load_px(const void* img, int dtype, long long p) {
  if (dtype == ABCD_F16) {
    const uint2 r = reinterpret_cast<const uint2*>(img)[p];
    const __half2 a = *reinterpret_cast<const __half2*>(&r.x);
    const __half2 b = *reinterpret_cast<const __half2*>(&r.y);
    const float2 fa = __half22float2(a), fb = __half22float2(b);
    return make_float4(fa.x, fa.y, fb.x, fb.y);
  }
  return reinterpret_cast<const float4*>(img)[p];
}

// Stages the entries of the kGroup list positions from `next` on (below n), all loads in flight
// together; survivors of the CTA-box cull are compacted in list order, each with its sigma limit,
// its list position + 1 (bits) and its Gaussian id.  Returns the number staged (warp-uniform);
// clamp: some staged opacity exceeds alpha_max.
__device__ __forceinline__ int stage_fill(const unsigned* ids, unsigned start, int n, int& next,
                                          const float2* uv, const float4* co, const float* rgb,
                                          float bx0, float by0, const Opts& op, float4* s_co,
                                          float4* s_m, float4* s_rgb, unsigned* s_id, bool& clamp) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  int total = 0;
  bool over = false;
  unsigned g[kRounds];
  float2 m[kRounds];
  float4 c[kRounds];
  float col[kRounds][3];
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    const int pos = next + lane + r * kSubThreads;
    g[r] = pos < n ? __ldg(ids + start + pos) : 0xffffffffu;
  }
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    if (g[r] != 0xffffffffu) {
      m[r] = __ldg(uv + g[r]);
      c[r] = __ldg(co + g[r]);
      col[r][0] = __ldg(rgb + 3 * (size_t)g[r]);
      col[r][1] = __ldg(rgb + 3 * (size_t)g[r] + 1);
      col[r][2] = __ldg(rgb + 3 * (size_t)g[r] + 2);
    }
  }
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    bool keep = false;
    float4 sc = make_float4(0.f, 0.f, 0.f, 0.f);
    float lim = -1.f;
    if (g[r] != 0xffffffffu) {
      sc = scaled_conic(c[r]);
      lim = sigma_limit(sc.w, op);
      keep = !cull(sc, m[r], bx0, by0, lim);
    }
    const unsigned b = __ballot_sync(0xffffffffu, keep);
    if (keep) {
      const int slot = total + __popc(b & lt);
      s_co[slot] = make_float4(sc.x, sc.y, sc.z, -sc.w);
      s_m[slot] = make_float4(-m[r].x, -m[r].y, limit_of_faint(lim, sc.w, op),
                              __uint_as_float((unsigned)(next + lane + r * kSubThreads + 1)));
      s_rgb[slot] = make_float4(col[r][0], col[r][1], col[r][2], 0.f);
      s_id[slot] = g[r];
      over = over || !(sc.w <= op.alpha_max);
    }
    total += __popc(b);
  }
  next += kGroup;
  // the loop over the survivors reads past the last: a NaN sigma is taken by no pixel, and the
  // rest must be finite (a zero weight times a non-finite value is not zero)
  if (lane < kBwdUnroll - 1) {
    s_co[total + lane] = make_float4(__int_as_float(0x7fffffff), 0.f, 0.f, 0.f);
    s_m[total + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
    s_rgb[total + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  clamp = __any_sync(0xffffffffu, over);
  __syncwarp();
  return total;
}

// Render CTA b handles the 8x8 block tile_order[b / 4] * 4 + b % 4 (tile_order: a permutation
// of the tiles, longest list first), or block b.
__device__ __forceinline__ int block_index(const unsigned* tile_order, int b) {
  if (tile_order) return (int)tile_order[b / kSubPerTile] * kSubPerTile + b % kSubPerTile;
  return b;
}

// Index, within its 8x8 block, of the lane's first pixel (the second is 4 further).
__device__ __forceinline__ int block_pixel(int lane) { return (lane >> 2) * kSub + (lane & 3); }

// The CTA's 8x8 pixel block and the lane's two pixels (qx0, py), (qx1 = qx0 + 4, py).
struct Block {
  int tile, px0, py0, qx0, qx1, py;
  bool in0, in1;
};

__device__ __forceinline__ Block block_of(const Cam& cam, int blk) {
  Block b;
  b.tile = blk / kSubPerTile;
  const int sub = blk % kSubPerTile;
  const int tx = b.tile % cam.tiles_x, ty = b.tile / cam.tiles_x;
  b.px0 = tx * kTile + (sub % (kTile / kSub)) * kSub;
  b.py0 = ty * kTile + (sub / (kTile / kSub)) * kSub;
  const int lane = threadIdx.x & 31;
  b.qx0 = b.px0 + (lane & 3);
  b.qx1 = b.qx0 + 4;
  b.py = b.py0 + (lane >> 2);
  b.in0 = b.qx0 < cam.width && b.py < cam.height;
  b.in1 = b.qx1 < cam.width && b.py < cam.height;
  return b;
}

struct FwdArgs {
  Cam cam;
  Opts op;
  const float2* uv;
  const float4* co;
  const float* rgb;
  const unsigned* ids;
  const uint2* ranges;
  const void* F;
  const void* B;
  int fb_dtype;
  float bg[3];
  float4* out;
  float4* state_at;
  unsigned* n_last;
  uint2* refresh;      // fp16 x4 per pixel
  uint2* refresh_packed;        // fp16 x4 per pixel of the tiles tile_map lists (packed layer)
  const int* tile_map;
  const unsigned* tile_order;   // tiles, longest list first (nullptr: launch order)
  float4* ckpt;                 // render checkpoints (nullptr: none), see the workspace
  uint4* ck_items;
  unsigned* ck_count;
  unsigned* ck_first;
  int ck_cap;
  const unsigned* status;       // the context's status word: after a timed-out wait the lists
                                // may hold stale ids, so every list reads as empty
};

// Blend state of one pixel.
struct PixF {
  float T, c0, c1, c2;
  unsigned last;       // one past the list position of the last contributor
};

// Blend state of the lane's two pixels, the first in .x, the second in .y.  A pixel that has
// ended (or lies outside the image) has a NaN for its x: every sigma there is NaN and no entry
// is taken, at no cost per entry.
struct PixF2 {
  float2 T, fx;
  float2 nc0, nc1, nc2;     // the colour so far, negated
  float fy;
  unsigned last0, last1;
  __device__ __forceinline__ bool on() const { return fx.x == fx.x || fx.y == fx.y; }
};

// One staged list entry as the backward's loop reads it.
struct Entry {
  float4 s;            // scaled conic, opacity negated
  float4 m;            // uv negated, sigma limit, list position + 1 (bits)
  float4 col;          // rgb
};

__device__ __forceinline__ Entry load_entry(const float4* s_co, const float4* s_m,
                                            const float4* s_rgb, int j) {
  Entry e;
  e.s = s_co[j];
  e.m = s_m[j];
  e.col = s_rgb[j];
  return e;
}

// Front-to-back step of the lane's two pixels over U staged entries.  The alphas come first
// (negated, 0 where an entry is not taken), then the transmittances after each entry, linked by
// one multiplication per entry; when no pixel of the warp falls below t_min among them (a vote), the
// colours are added without another test.  Otherwise the entries are taken one by one: the entry
// that takes a pixel below t_min ends it and does not contribute.  CLAMP: some staged opacity
// exceeds alpha_max (else o 2^-sigma' cannot).
template <int U, bool CLAMP>
__device__ __forceinline__ void blend(PixF2& p, const float4* s_co, const float4* s_m,
                                      const float4* s_rgb, const Opts& op) {
  float2 na[U], Tb[U], T = p.T;
  unsigned l0 = p.last0, l1 = p.last1;
#pragma unroll
  for (int k = 0; k < U; ++k) {
    const float4 s = s_co[k], m = s_m[k];
    float2 dx, sg;
    float dy;
    sigma_pair(s, m, p.fx, p.fy, dx, dy, sg);
    float2 raw = __fmul2_rn(make_float2(s.w, s.w), make_float2(ex2_approx(-sg.x), ex2_approx(-sg.y)));
    if (CLAMP) raw = make_float2(fmaxf(-op.alpha_max, raw.x), fmaxf(-op.alpha_max, raw.y));
    const bool t0 = takes(sg.x, m.z), t1 = takes(sg.y, m.z);
    na[k] = make_float2(t0 ? raw.x : 0.f, t1 ? raw.y : 0.f);
    l0 = t0 ? __float_as_uint(m.w) : l0;
    l1 = t1 ? __float_as_uint(m.w) : l1;
  }
#pragma unroll
  for (int k = 0; k < U; ++k) {
    Tb[k] = T;
    T = __fmul2_rn(T, __fadd2_rn(make_float2(1.f, 1.f), na[k]));
  }
  if (!__any_sync(0xffffffffu, fminf(T.x, T.y) < op.t_min)) {
    p.T = T;
    p.last0 = l0;
    p.last1 = l1;
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const float4 col = s_rgb[k];
      const float2 w = __fmul2_rn(na[k], Tb[k]);
      p.nc0 = __ffma2_rn(w, make_float2(col.x, col.x), p.nc0);
      p.nc1 = __ffma2_rn(w, make_float2(col.y, col.y), p.nc1);
      p.nc2 = __ffma2_rn(w, make_float2(col.z, col.z), p.nc2);
    }
    return;
  }
  bool on0 = p.fx.x == p.fx.x, on1 = p.fx.y == p.fx.y;
#pragma unroll
  for (int k = 0; k < U; ++k) {
    const float4 col = s_rgb[k];
    const unsigned pos = __float_as_uint(s_m[k].w);
    const float2 Tn = __fmul2_rn(p.T, __fadd2_rn(make_float2(1.f, 1.f), na[k]));
    const bool t0 = on0 && na[k].x < 0.f, t1 = on1 && na[k].y < 0.f;
    const bool u0 = t0 && !(Tn.x < op.t_min), u1 = t1 && !(Tn.y < op.t_min);
    on0 = on0 && (u0 || !t0);
    on1 = on1 && (u1 || !t1);
    const float2 wf = __fmul2_rn(na[k], p.T);
    const float2 w = make_float2(u0 ? wf.x : 0.f, u1 ? wf.y : 0.f);
    p.nc0 = __ffma2_rn(w, make_float2(col.x, col.x), p.nc0);
    p.nc1 = __ffma2_rn(w, make_float2(col.y, col.y), p.nc1);
    p.nc2 = __ffma2_rn(w, make_float2(col.z, col.z), p.nc2);
    p.T = make_float2(u0 ? Tn.x : p.T.x, u1 ? Tn.y : p.T.y);
    p.last0 = u0 ? pos : p.last0;
    p.last1 = u1 ? pos : p.last1;
  }
  const float nan = __int_as_float(0x7fffffff);
  p.fx = make_float2(on0 ? p.fx.x : nan, on1 ? p.fx.y : nan);
}

// Blends staged entries [0, cnt), padded to a multiple of kFwdUnroll.
template <bool CLAMP>
__device__ __forceinline__ void blend_staged(PixF2& p, const float4* s_co, const float4* s_m,
                                             const float4* s_rgb, int cnt, const Opts& op) {
  for (int j = 0; j < cnt; j += kFwdUnroll)
    blend<kFwdUnroll, CLAMP>(p, s_co + j, s_m + j, s_rgb + j, op);
}

__device__ __forceinline__ void store_pixel(const FwdArgs& a, long long p, const PixF& s, int qx,
                                            int qy, int tile) {
  const float Aa = 1.f - s.T;
  if (a.refresh || a.refresh_packed) {
    const __half2 lo = __floats2half2_rn(s.c0, s.c1), hi = __floats2half2_rn(s.c2, Aa);
    uint2 r;
    r.x = *reinterpret_cast<const unsigned*>(&lo);
    r.y = *reinterpret_cast<const unsigned*>(&hi);
    if (a.refresh) a.refresh[p] = r;
    if (a.refresh_packed) {
      const int m = a.tile_map[tile];
      if (m >= 0) a.refresh_packed[(size_t)m * kTileThreads + (qy % kTile) * kTile + qx % kTile] = r;
    }
  }
  if (a.state_at) {
    a.state_at[p] = make_float4(s.c0, s.c1, s.c2, s.T);
    a.n_last[p] = s.last;
  }
  if (a.out) {
    const float4 Bv = a.B ? load_px(a.B, a.fb_dtype, p) : make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 Fv = a.F ? load_px(a.F, a.fb_dtype, p) : make_float4(0.f, 0.f, 0.f, 0.f);
    const float kb = 1.f - Aa;      // A over B
    const float m0 = s.c0 + kb * Bv.x, m1 = s.c1 + kb * Bv.y, m2 = s.c2 + kb * Bv.z, ma = Aa + kb * Bv.w;
    const float kf = 1.f - Fv.w;    // F over (A over B)
    float4 o = make_float4(Fv.x + kf * m0, Fv.y + kf * m1, Fv.z + kf * m2, Fv.w + kf * ma);
    const float kg = 1.f - o.w;
    o.x += kg * a.bg[0];
    o.y += kg * a.bg[1];
    o.z += kg * a.bg[2];
    a.out[p] = o;
  }
}

template <int BYTES>
__device__ __forceinline__ void copy_async(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
               "l"(src), "n"(BYTES) : "memory");
}

// The raw entries of a staging group, as the asynchronous copies bring them in.
struct RawGroup {
  float4 co[kFwdGroup];
  float2 uv[kFwdGroup];
  float rgb[3][kFwdGroup];
};

__device__ __forceinline__ void fetch_group(const FwdArgs& a, const unsigned (&g)[kFwdRounds],
                                            RawGroup& raw) {
#pragma unroll
  for (int r = 0; r < kFwdRounds; ++r) {
    const int k = (threadIdx.x & 31) + 32 * r;
    if (g[r] == 0xffffffffu) continue;
    copy_async<16>(&raw.co[k], a.co + g[r]);
    copy_async<8>(&raw.uv[k], a.uv + g[r]);
    const float* col = a.rgb + 3 * (size_t)g[r];
#pragma unroll
    for (int c = 0; c < 3; ++c) copy_async<4>(&raw.rgb[c][k], col + c);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// What bounds it: the longest walks.  A small active block covers a quarter of the tiles, so
// every non-empty 8x8 block is resident at once (about 30 one-warp CTAs per SM at 1237x822) and
// the kernel lasts as long as its longest walk (700 staged entries there, 81,000 of its 137,000
// cycles blending, at 116 cycles per entry).  The walk is therefore built for one warp's
// instructions and latency: the entries of the next 64 list positions are copied to shared
// memory, and the ids of the 64 after them loaded, while the current ones are blended; the block
// cull takes both lanes' rounds side by side without branches; four entries are evaluated
// together whose states are linked by one multiplication, with the end-of-pixel test voted on once per
// four.  Against two entries at a time with their selects and 64 entries loaded when needed:
// 33 -> 23 us (2,000 Gaussians, 128x128), 84 -> 62 us (100,000, 1237x822), 218 -> 189 us (2M,
// 1920x1080); the refresh at 1237x822 77-98 -> 53-68 us.  Eight entries per iteration need 120
// registers and gave 61 and 207 us; 32 positions per group 29 us and 72 us.  24 CTAs per SM (80
// registers, no spills) against 28: 61 against 63 us and 189 against 199 us.
__global__ void __launch_bounds__(kSubThreads, 24) render_fwd_kernel(const __grid_constant__ FwdArgs a) {
  pdl_wait();
  __shared__ RawGroup raw;
  __shared__ float4 s_co[kFwdGroup];
  __shared__ float4 s_m[kFwdGroup];
  __shared__ float4 s_rgb[kFwdGroup];
  const int blk = block_index(a.tile_order, (int)blockIdx.x);
  const Block bk = block_of(a.cam, blk);
  const int lane = threadIdx.x & 31;
  const uint2 rg = a.ranges[bk.tile];
  const int n = (rg.y > rg.x && !(*a.status & kStatusTimeout)) ? (int)(rg.y - rg.x) : 0;
  const float bx0 = (float)bk.px0 + 0.5f, by0 = (float)bk.py0 + 0.5f;
  const float nan = __int_as_float(0x7fffffff);
  PixF2 pp;
  pp.T = make_float2(1.f, 1.f);
  pp.nc0 = pp.nc1 = pp.nc2 = make_float2(0.f, 0.f);
  pp.fx = make_float2(bk.in0 ? (float)bk.qx0 + 0.5f : nan, bk.in1 ? (float)bk.qx1 + 0.5f : nan);
  pp.fy = (float)bk.py + 0.5f;
  pp.last0 = pp.last1 = 0u;
  bool ck_on = a.ckpt != nullptr;          // warp-uniform
  int n_items = 0;
  unsigned my_slot = 0u;                   // lane k: the slot of this block's item k
  const unsigned* ids = a.ids + rg.x;
  unsigned g[kFwdRounds];
#pragma unroll
  for (int r = 0; r < kFwdRounds; ++r) g[r] = lane + 32 * r < n ? __ldg(ids + lane + 32 * r) : 0xffffffffu;
  if (n > 0) fetch_group(a, g, raw);
#pragma unroll
  for (int r = 0; r < kFwdRounds; ++r) {
    const int pos = kFwdGroup + lane + 32 * r;
    g[r] = pos < n ? __ldg(ids + pos) : 0xffffffffu;
  }
  for (int base = 0; base < n; base += kFwdGroup) {
    if (!__any_sync(0xffffffffu, pp.on())) break;
    asm volatile("cp.async.wait_all;" ::: "memory");
    // the survivors of the block cull, compacted in list order (a lane reads the entries that it
    // copied itself)
    int cnt = 0;
    bool over = false;
    float4 sc[kFwdRounds];
    float2 m[kFwdRounds];
    float lim[kFwdRounds], col[kFwdRounds][3];
    bool keep[kFwdRounds];
#pragma unroll
    for (int r = 0; r < kFwdRounds; ++r) {
      const int k = lane + 32 * r;
      sc[r] = scaled_conic(raw.co[k]);
      m[r] = raw.uv[k];
#pragma unroll
      for (int c = 0; c < 3; ++c) col[r][c] = raw.rgb[c][k];
      lim[r] = sigma_limit(sc[r].w, a.op);
      keep[r] = (base + k < n) & !cull(sc[r], m[r], bx0, by0, lim[r]);
    }
#pragma unroll
    for (int r = 0; r < kFwdRounds; ++r) {
      const unsigned kept = __ballot_sync(0xffffffffu, keep[r]);
      const int slot = cnt + __popc(kept & ((1u << lane) - 1u));
      if (keep[r]) {
        s_co[slot] = make_float4(sc[r].x, sc[r].y, sc[r].z, -sc[r].w);
        s_m[slot] = make_float4(-m[r].x, -m[r].y, limit_of_faint(lim[r], sc[r].w, a.op),
                                __uint_as_float((unsigned)(base + lane + 32 * r + 1)));
        s_rgb[slot] = make_float4(col[r][0], col[r][1], col[r][2], 0.f);
      }
      over = over | (keep[r] & !(sc[r].w <= a.op.alpha_max));
      cnt += __popc(kept);
    }
    const bool clamp = __any_sync(0xffffffffu, over);
    // unused slots of the last iteration: a NaN sigma is taken by no pixel
    if (lane < (-cnt & (kFwdUnroll - 1))) {
      s_co[cnt + lane] = make_float4(nan, 0.f, 0.f, 0.f);
      s_m[cnt + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
      s_rgb[cnt + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (base + kFwdGroup < n) fetch_group(a, g, raw);
#pragma unroll
    for (int r = 0; r < kFwdRounds; ++r) {
      const int pos = base + 2 * kFwdGroup + lane + 32 * r;
      g[r] = pos < n ? __ldg(ids + pos) : 0xffffffffu;
    }
    const int end = base + kFwdGroup;
    // at a checkpoint: ask for its slot now, the answer comes while the group is blended
    const bool ck_here = ck_on && end % kCkChunk == 0 && end < n;
    unsigned slot = 0u;
    if (ck_here && lane == 0) slot = atomicAdd(a.ck_count, 1u);
    __syncwarp();
    if (!clamp) blend_staged<false>(pp, s_co, s_m, s_rgb, cnt, a.op);
    else blend_staged<true>(pp, s_co, s_m, s_rgb, cnt, a.op);
    __syncwarp();
    if (ck_here) {
      // the state after every position below `end`, for the backward's chunk starting there
      slot = __shfl_sync(0xffffffffu, slot, 0);
      const bool room = slot < (unsigned)a.ck_cap;
      if (__any_sync(0xffffffffu, pp.on())) {
        if (room) {
          float4* ck = a.ckpt + (size_t)slot * (kSub * kSub);
          const int k0 = block_pixel(lane);
          ck[k0] = make_float4(0.f - pp.nc0.x, 0.f - pp.nc1.x, 0.f - pp.nc2.x, pp.T.x);
          ck[k0 + 4] = make_float4(0.f - pp.nc0.y, 0.f - pp.nc1.y, 0.f - pp.nc2.y, pp.T.y);
          if (lane == n_items) my_slot = slot;
          ++n_items;
        }
        // past 32 items or a full buffer the last item listed runs to the end of the walk
        ck_on = room && n_items < 32;
      } else if (room && lane == 0) {
        a.ck_items[slot] = make_uint4(0u, 0u, 0u, 0u);   // the walk ended: nothing to replay
      }
    }
  }
  const PixF p0 = {pp.T.x, 0.f - pp.nc0.x, 0.f - pp.nc1.x, 0.f - pp.nc2.x, pp.last0};
  const PixF p1 = {pp.T.y, 0.f - pp.nc0.y, 0.f - pp.nc1.y, 0.f - pp.nc2.y, pp.last1};
  if (a.ckpt) {
    if (lane == 0) a.ck_first[blk] = n_items > 0 ? (unsigned)kCkChunk : 0xffffffffu;
    if (lane < n_items) {
      const unsigned start = (unsigned)((lane + 1) * kCkChunk);
      a.ck_items[my_slot] = make_uint4((unsigned)blk, start, lane == n_items - 1 ? 0xffffffffu : start + kCkChunk, 0u);
    }
  }
  if (bk.in0) store_pixel(a, (long long)bk.py * a.cam.width + bk.qx0, p0, bk.qx0, bk.py, bk.tile);
  if (bk.in1) store_pixel(a, (long long)bk.py * a.cam.width + bk.qx1, p1, bk.qx1, bk.py, bk.tile);
  asm volatile("cp.async.wait_all;" ::: "memory");   // a walk that ended early has copies in flight
}

struct BwdArgs {
  Cam cam;
  Opts op;
  const float2* uv;
  const float4* co;
  const float* rgb;
  const unsigned* ids;
  const uint2* ranges;
  const void* F;
  const void* B;
  int fb_dtype;
  float bg[3];
  const float4* state_at;
  const unsigned* n_last;
  const float* dl_dout;
  float* grad2d;
  const unsigned* tile_order;   // tiles, longest list first (nullptr: launch order)
  const float4* ckpt;           // the forward's checkpoints (nullptr: every block walks whole)
  const uint4* ck_items;
  const unsigned* ck_count;
  const unsigned* ck_first;
  int ck_cap;
  int n_item_ctas;              // the first CTAs of the launch replay the listed chunks
  const unsigned* status;       // as in FwdArgs
};

// Backward state of one pixel.  With G = dL/dA.rgb and G_a = dL/dA.a, the derivative of the
// loss w.r.t. an entry's alpha is
//   sum_ch G_ch (T col_ch - (A_ch - C_ch) / (1 - alpha)) + G_a T_final / (1 - alpha)
//   = T (G . col) - (K - G . C) / (1 - alpha),   K = G . A - G_a T_final,
// C the colour accumulated up to and including the entry: only the scalar G . C is replayed.
struct PixB {
  float T, Gc;                  // transmittance and G . C replayed up to the current entry
  float Gr, Gg, Gb, K;          // dL/dA.rgb; G . A - G_a T_final
  unsigned last;                // replay only list positions below this
};

__device__ __forceinline__ void load_pixel_grad(const BwdArgs& a, long long p, int n, PixB& q) {
  q.last = min(a.n_last[p], (unsigned)n);
  const float4 at = a.state_at[p];
  const float g0 = a.dl_dout[3 * p], g1 = a.dl_dout[3 * p + 1], g2 = a.dl_dout[3 * p + 2];
  const float4 Fv = a.F ? load_px(a.F, a.fb_dtype, p) : make_float4(0.f, 0.f, 0.f, 0.f);
  const float4 Bv = a.B ? load_px(a.B, a.fb_dtype, p) : make_float4(0.f, 0.f, 0.f, 0.f);
  const float kf = 1.f - Fv.w;
  q.Gr = kf * g0; q.Gg = kf * g1; q.Gb = kf * g2;
  // d final / d A.a = -(1 - F.a) (B.rgb + (1 - B.a) bg)
  const float Ga = -kf * (g0 * (Bv.x + (1.f - Bv.w) * a.bg[0]) + g1 * (Bv.y + (1.f - Bv.w) * a.bg[1]) +
                          g2 * (Bv.z + (1.f - Bv.w) * a.bg[2]));
  q.K = q.Gr * at.x + q.Gg * at.y + q.Gb * at.z - Ga * at.w;
}

// Backward of the lane's two pixels for one list entry (selects, no branches): when the entry
// contributed to a pixel (live: a position up to the pixel's last contributor; sigma within the
// limit) adds up over the two pixels, into v: the opacity gradient, dL/dsigma dx, dL/dsigma dx^2
// and the colour gradients, and advances the replayed transmittance.  (dL/dsigma is -opacity
// times the opacity gradient's summand, and dy is the same along a row of the block, so these
// six sums hold all nine gradients, see bwd_staged.)  With
// G = dL/dA.rgb and G_a = dL/dA.a, the derivative of the loss w.r.t. an entry's alpha is
//   T (G . col) - (K - G . C) / (1 - alpha),   K = G . A - G_a T_final,
// C the colour accumulated up to and including the entry.  The two pixels' arithmetic is paired
// through the packed two-lane fp32 instructions, which have no negated operands: the staged
// opacity is negated, and so is the replayed G . C, so that none is needed.  The decisions
// (sigma, its limit) are rounded exactly as the forward rounds them.  An entry that a pixel does not
// take adds zeros by its weight of 0, which an infinite or NaN gradient of the pixel would turn into
// NaN: blocks with such a pixel run with WILD, which selects the zeros.  Returns whether the entry
// contributed to either pixel.
constexpr int kSums = 6;              // sums per entry

struct PixB2 {
  float2 T, nGc, Gr, Gg, Gb, K;
};

template <bool CLAMP, bool WILD>
__device__ __forceinline__ bool pixel_backward2(PixB2& p, const Entry& e, float2 sg, float2 dx,
                                                bool live0, bool live1, const Opts& op,
                                                float (&v)[kSums]) {
  const bool ok0 = live0 && takes(sg.x, e.m.z);
  const bool ok1 = live1 && takes(sg.y, e.m.z);
  // an entry that is not taken gets a sigma whose exponential is 0, and with it alpha and every
  // gradient
  const float2 G = make_float2(ex2_approx(-(ok0 ? sg.x : kFarSigma)), ex2_approx(-(ok1 ? sg.y : kFarSigma)));
  const float2 nraw = __fmul2_rn(make_float2(e.s.w, e.s.w), G);      // -o 2^-sigma'
  float2 na = nraw;                                                  // -alpha
  if (CLAMP) na = make_float2(fmaxf(-op.alpha_max, nraw.x), fmaxf(-op.alpha_max, nraw.y));
  const float2 nw = __fmul2_rn(na, p.T);                             // -alpha T
  const float2 gcol = __ffma2_rn(p.Gb, make_float2(e.col.z, e.col.z),
                                 __ffma2_rn(p.Gg, make_float2(e.col.y, e.col.y),
                                            __fmul2_rn(p.Gr, make_float2(e.col.x, e.col.x))));
  const float2 nGc = __ffma2_rn(nw, gcol, p.nGc);                    // -G . C including the entry
  p.nGc = WILD ? make_float2(ok0 ? nGc.x : p.nGc.x, ok1 ? nGc.y : p.nGc.y) : nGc;
  const float2 oma = __fadd2_rn(make_float2(1.f, 1.f), na);
  const float2 nioma = make_float2(rcp_approx(-oma.x), rcp_approx(-oma.y));
  const float2 km = __fadd2_rn(p.K, p.nGc);
  float2 da = __ffma2_rn(km, nioma, __fmul2_rn(p.T, gcol));
  // d alpha / d opacity = G, d alpha / d sigma = -alpha; none of either where alpha was clamped
  if (CLAMP) da = make_float2(nraw.x >= -op.alpha_max ? da.x : 0.f, nraw.y >= -op.alpha_max ? da.y : 0.f);
  if (WILD) da = make_float2(ok0 ? da.x : 0.f, ok1 ? da.y : 0.f);
  const float2 dg = __fmul2_rn(da, G);
  const float2 t = __fmul2_rn(__fmul2_rn(da, nraw), dx);             // dL/dsigma dx
  v[0] = dg.x + dg.y;
  v[1] = t.x + t.y;
  v[2] = fmaf(t.x, dx.x, t.y * dx.y);
  if (WILD) {
    v[3] = (ok0 ? p.Gr.x * -nw.x : 0.f) + (ok1 ? p.Gr.y * -nw.y : 0.f);
    v[4] = (ok0 ? p.Gg.x * -nw.x : 0.f) + (ok1 ? p.Gg.y * -nw.y : 0.f);
    v[5] = (ok0 ? p.Gb.x * -nw.x : 0.f) + (ok1 ? p.Gb.y * -nw.y : 0.f);
  } else {
    v[3] = fmaf(p.Gr.x, -nw.x, p.Gr.y * -nw.y);
    v[4] = fmaf(p.Gg.x, -nw.x, p.Gg.y * -nw.y);
    v[5] = fmaf(p.Gb.x, -nw.x, p.Gb.y * -nw.y);
  }
  p.T = __fmul2_rn(p.T, oma);
  return ok0 || ok1;
}

// Backward of the staged entries [0, cnt) at the lane's two pixels, kBwdUnroll entries per
// iteration (past cnt a NaN sigma is taken by no pixel).  Each lane writes an entry's six sums to shared memory as row 6 i + k (pitch 36: no
// bank conflicts in either direction); lane l then reads row l, whose float4 q holds the four
// lanes of pixel row q, and takes the row's sum S = sum s_q and its moments S1 = sum s_q dy_q and
// S2 = sum s_q dy_q^2 over the rows.  With (ca, cb, cc) = ln 2 (2 a', b', 2 c') of the scaled
// conic, D = dL/dsigma = -o (the opacity gradient's summands):
//   d/du = -(ca sum D dx + cb sum D dy),  d/dv = -(cb sum D dx + cc sum D dy),
//   d/da = sum D dx^2 / 2,  d/db = sum D dx dy,  d/dc = sum D dy^2 / 2.
constexpr int kRedPitch = 36;
static_assert(kBwdUnroll * kSums <= 32, "one row per lane");

template <bool CLAMP, bool WILD>
__device__ __forceinline__ void bwd_staged(const BwdArgs& a, PixB2& pp, float2 fx, float fy,
                                           float by0, unsigned last0, unsigned last1, int cnt,
                                           const float4* s_co, const float4* s_m,
                                           const float4* s_rgb, const unsigned* s_id,
                                           float* s_red) {
  const int lane = threadIdx.x & 31;
  const int ei = min(lane / kSums, kBwdUnroll - 1), comp = lane - kSums * ei;
  for (int j = 0; j < cnt; j += kBwdUnroll) {
    unsigned who = 0u;                               // bit i: entry j + i counts for some pixel
#pragma unroll
    for (int i = 0; i < kBwdUnroll; ++i) {
      const Entry e = load_entry(s_co, s_m, s_rgb, j + i);
      const unsigned nxt = __float_as_uint(e.m.w);
      float2 dx, sg;
      float dy, v[kSums];
      sigma_pair(e.s, e.m, fx, fy, dx, dy, sg);
      const bool c = pixel_backward2<CLAMP, WILD>(pp, e, sg, dx, nxt <= last0, nxt <= last1, a.op, v);
      if (__any_sync(0xffffffffu, c)) who |= 1u << i;
#pragma unroll
      for (int k = 0; k < kSums; ++k) s_red[(kSums * i + k) * kRedPitch + lane] = v[k];
    }
    if (who == 0u) continue;
    __syncwarp();
    const float4 sc = s_co[j + ei];    // a', b', c', -o
    const float dy0 = by0 + s_m[j + ei].y;
    const float4* row = reinterpret_cast<const float4*>(s_red + min(lane, kSums * kBwdUnroll - 1) * kRedPitch);
    float S = 0.f, S1 = 0.f, S2 = 0.f;
#pragma unroll
    for (int q = 0; q < kSub; ++q) {
      const float4 r = row[q];
      const float2 h = __fadd2_rn(make_float2(r.x, r.y), make_float2(r.z, r.w));
      const float sq = h.x + h.y, dyq = dy0 + (float)q, sd = sq * dyq;
      S += sq;
      S1 += sd;
      S2 = fmaf(sd, dyq, S2);
    }
    __syncwarp();
    const float sx = __shfl_sync(0xffffffffu, S, kSums * ei + 1);             // sum D dx
    const float sy = sc.w * __shfl_sync(0xffffffffu, S1, kSums * ei);         // sum D dy
    if (lane < kSums * kBwdUnroll && ((who >> ei) & 1u)) {
      const float ca = 2.f * kLn2 * sc.x, cb = kLn2 * sc.y, cc = 2.f * kLn2 * sc.z;
      float* g = a.grad2d + 9 * (size_t)s_id[j + ei];
      const float g0 = comp == 1 ? -(ca * sx + cb * sy) : (comp == 2 ? 0.5f * S : S);
      const int c0 = comp == 0 ? 5 : (comp == 1 ? 0 : (comp == 2 ? 2 : comp + 3));
      atomicAdd(g + c0, g0);                         // o, u, a, r, g, b
      if (comp < 3) {
        const float g1 = comp == 0 ? 0.5f * sc.w * S2 : (comp == 1 ? S1 : -(cb * sx + cc * sy));
        const int c1 = comp == 0 ? 4 : (comp == 1 ? 3 : 1);
        atomicAdd(g + c1, g1);                       // c, b, v
      }
    }
  }
}

// Backward of list positions [start, end) of block blk (clipped to the block's walk), from the
// forward's checkpoint `ck` when start > 0.
__device__ __forceinline__ void bwd_chunk(const BwdArgs& a, int blk, int start, unsigned end,
                                          const float4* ck, float4* s_co, float4* s_m,
                                          float4* s_rgb, unsigned* s_id, float* s_red) {
  const Block bk = block_of(a.cam, blk);
  const int lane = threadIdx.x & 31;
  const uint2 rg = a.ranges[bk.tile];
  const int n = (rg.y > rg.x && !(*a.status & kStatusTimeout)) ? (int)(rg.y - rg.x) : 0;
  const float2 fx = make_float2((float)bk.qx0 + 0.5f, (float)bk.qx1 + 0.5f);
  const float fy = (float)bk.py + 0.5f;
  const float bx0 = (float)bk.px0 + 0.5f, by0 = (float)bk.py0 + 0.5f;
  PixB p0 = {}, p1 = {};
  p0.T = p1.T = 1.f;
  if (bk.in0) load_pixel_grad(a, (long long)bk.py * a.cam.width + bk.qx0, n, p0);
  if (bk.in1) load_pixel_grad(a, (long long)bk.py * a.cam.width + bk.qx1, n, p1);
  if (ck) {
    const int k0 = block_pixel(lane);
    const float4 c0 = ck[k0], c1 = ck[k0 + 4];
    p0.T = c0.w; p0.Gc = p0.Gr * c0.x + p0.Gg * c0.y + p0.Gb * c0.z;
    p1.T = c1.w; p1.Gc = p1.Gr * c1.x + p1.Gg * c1.y + p1.Gb * c1.z;
  }
  const int span = (int)min((unsigned)__reduce_max_sync(0xffffffffu, max(p0.last, p1.last)), end);
  PixB2 pp;
  pp.T = make_float2(p0.T, p1.T);
  pp.nGc = make_float2(-p0.Gc, -p1.Gc);
  pp.Gr = make_float2(p0.Gr, p1.Gr);
  pp.Gg = make_float2(p0.Gg, p1.Gg);
  pp.Gb = make_float2(p0.Gb, p1.Gb);
  pp.K = make_float2(p0.K, p1.K);
  const unsigned last0 = p0.last, last1 = p1.last;
  const float size0 = fabsf(p0.Gr) + fabsf(p0.Gg) + fabsf(p0.Gb) + fabsf(p0.K);
  const float size1 = fabsf(p1.Gr) + fabsf(p1.Gg) + fabsf(p1.Gb) + fabsf(p1.K);
  const bool wild = __any_sync(0xffffffffu, !(size0 + size1 < 3.402823466e38f));
  int next = start;
  while (next < span) {
    __syncwarp();
    bool clamp;
    const int cnt = stage_fill(a.ids, rg.x, span, next, a.uv, a.co, a.rgb, bx0, by0, a.op, s_co,
                               s_m, s_rgb, s_id, clamp);
    if (wild) bwd_staged<true, true>(a, pp, fx, fy, by0, last0, last1, cnt, s_co, s_m, s_rgb, s_id, s_red);
    else if (clamp) bwd_staged<true, false>(a, pp, fx, fy, by0, last0, last1, cnt, s_co, s_m, s_rgb, s_id, s_red);
    else bwd_staged<false, false>(a, pp, fx, fy, by0, last0, last1, cnt, s_co, s_m, s_rgb, s_id, s_red);
  }
}

// What bounds it: shared memory and the gathers (the L1's data stage 65% busy at 1237x822, 84% for
// dense tiles before the sums went by rows) and instruction issue (55%).  With nine sums per entry
// in three entries per iteration: 95 and 79 us (two cameras, 100,000 Gaussians at 1237x822) and
// 450 us (2M at 1920x1080); with six sums in five entries 87, 72 and 406 us; four entries 90, 75
// and 427 us; staging through asynchronous copies 100, 80 and 467 us (more shared-memory traffic).
// 20 CTAs per SM leave 96 registers, so nothing spills; 16 CTAs 94, 76 and 434 us.
__global__ void __launch_bounds__(kSubThreads, 20) render_bwd_kernel(BwdArgs a) {
  pdl_wait();
  __shared__ float4 s_co[kGroup + kBwdUnroll - 1];
  __shared__ float4 s_m[kGroup + kBwdUnroll - 1];
  __shared__ float4 s_rgb[kGroup + kBwdUnroll - 1];
  __shared__ unsigned s_id[kGroup];
  __shared__ __align__(16) float s_red[kSums * kBwdUnroll * kRedPitch];
  // the first n_item_ctas CTAs replay the listed chunks after the first of the long walks, the
  // others each a block's walk up to its first checkpoint
  const int b = (int)blockIdx.x;
  const bool item_cta = b < a.n_item_ctas;
  const unsigned items = item_cta ? min(*a.ck_count, (unsigned)a.ck_cap) : 0u;
  for (unsigned i = b; !item_cta || i < items; i += a.n_item_ctas) {
    int blk, start = 0;
    unsigned end = 0xffffffffu;
    const float4* ck = nullptr;
    if (item_cta) {
      const uint4 it = a.ck_items[i];
      if (it.z == 0u) continue;                // a walk that ended before its checkpoint
      blk = (int)it.x; start = (int)it.y; end = it.z;
      ck = a.ckpt + (size_t)i * (kSub * kSub);
    } else {
      blk = block_index(a.tile_order, b - a.n_item_ctas);
      if (a.ckpt) end = a.ck_first[blk];
    }
    __syncwarp();
    bwd_chunk(a, blk, start, end, ck, s_co, s_m, s_rgb, s_id, s_red);
    if (!item_cta) break;
  }
}

// The tile order bin_sort left in the workspace, if it was made for these ranges.
const unsigned* tile_order_for(const abcd_ctx* ctx, const abcd_tiles* tiles, long long n_tiles) {
  return (has_workspace(ctx) && ctx->order_ranges == tiles->ranges && ctx->order_tiles == n_tiles)
             ? ctx->ws.tile_order : nullptr;
}

// Checkpoints need the workspace and room for a first-chunk end per block.
bool ckpt_ok(const abcd_ctx* ctx, long long n_blocks) {
  return has_workspace(ctx) && ctx->ws.ckpt && n_blocks <= kSubPerTile * ctx->ws.max_tiles;
}

bool fb_ok(const void* F, const void* B, int dtype) {
  if (dtype != ABCD_F16 && dtype != ABCD_F32) return false;
  const uintptr_t al = dtype == ABCD_F16 ? 7 : 15;
  return (((uintptr_t)F & al) == 0) && (((uintptr_t)B & al) == 0);
}

bool proj_ok(const abcd_projected* p) {
  return p && p->uv && p->conic_opacity && p->rgb && ((uintptr_t)p->uv & 7) == 0 &&
         ((uintptr_t)p->conic_opacity & 15) == 0;
}

}  // namespace
}  // namespace abcd

using namespace abcd;

abcd_status abcd::render_composite_fwd(abcd_ctx* ctx, const abcd_camera* cam,
                                       const abcd_render_opts* opts, const abcd_projected* proj,
                                       const abcd_tiles* tiles, const void* F, const void* B,
                                       int fb_dtype, const float* bg, float* out_rgba,
                                       abcd_fwd_state* state, void* refresh_f16,
                                       bool count_cleared) {
  if (!ctx) return ABCD_ERR_INVALID_ARG;
  if (!cam || cam->width <= 0 || cam->height <= 0 || !tiles || !tiles->ids || !tiles->ranges)
    return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_render_composite_fwd: bad camera or tiles");
  if (!proj_ok(proj)) return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_render_composite_fwd: bad projected buffers");
  if (!fb_ok(F, B, fb_dtype)) return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_render_composite_fwd: bad F/B dtype or alignment");
  if (state && (!state->A_T || !state->n_last || ((uintptr_t)state->A_T & 15)))
    return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_render_composite_fwd: bad state buffers");
  if (((uintptr_t)out_rgba & 15) || ((uintptr_t)refresh_f16 & 7))
    return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_render_composite_fwd: misaligned output");
  FwdArgs a;
  a.status = ctx->ws.status;
  a.cam = make_cam(cam, opts);
  a.op = make_opts(opts);
  a.uv = (const float2*)proj->uv;
  a.co = (const float4*)proj->conic_opacity;
  a.rgb = proj->rgb;
  a.ids = tiles->ids;
  a.ranges = (const uint2*)tiles->ranges;
  a.F = F; a.B = B; a.fb_dtype = fb_dtype;
  for (int c = 0; c < 3; ++c) a.bg[c] = bg ? bg[c] : 0.f;
  a.out = (float4*)out_rgba;
  a.state_at = state ? (float4*)state->A_T : nullptr;
  a.n_last = state ? state->n_last : nullptr;
  a.refresh = (uint2*)refresh_f16;
  a.refresh_packed = nullptr;
  a.tile_map = nullptr;
  const int n_tiles = a.cam.tiles_x * a.cam.tiles_y, n_blocks = n_tiles * kSubPerTile;
  a.tile_order = tile_order_for(ctx, tiles, n_tiles);
  a.ckpt = nullptr; a.ck_items = nullptr; a.ck_count = nullptr; a.ck_first = nullptr;
  a.ck_cap = 0;
  if (state && ckpt_ok(ctx, n_blocks)) {
    if (!count_cleared) {
      const abcd_status z = zero_async(ctx, ctx->ws.ck_count, sizeof(unsigned), "checkpoint count clear");
      if (z != ABCD_OK) return z;
    }
    a.ckpt = ctx->ws.ckpt; a.ck_items = ctx->ws.ck_items; a.ck_count = ctx->ws.ck_count;
    a.ck_first = ctx->ws.ck_first; a.ck_cap = ctx->ws.ck_cap;
    ctx->ck_state = state->A_T;
    ctx->ck_blocks = n_blocks;
    ctx->ck_ranges = tiles->ranges;
  } else if (state && ctx->ck_state == state->A_T) {
    ctx->ck_state = nullptr;               // this state's checkpoints are gone
  }
  return check_launch(ctx, "render_fwd_kernel",
                      launch_pdl(render_fwd_kernel, dim3(n_blocks), dim3(kSubThreads), 0, ctx->stream, a));
}

extern "C" abcd_status abcd_render_composite_fwd(abcd_ctx* ctx, const abcd_camera* cam,
                                                 const abcd_render_opts* opts,
                                                 const abcd_projected* proj,
                                                 const abcd_tiles* tiles, const void* F,
                                                 const void* B, int fb_dtype, const float* bg,
                                                 float* out_rgba, abcd_fwd_state* state,
                                                 void* refresh_f16) {
  return render_composite_fwd(ctx, cam, opts, proj, tiles, F, B, fb_dtype, bg, out_rgba, state,
                              refresh_f16, false);
}

abcd_status abcd::render_backward(abcd_ctx* ctx, const abcd_camera* cam,
                                  const abcd_render_opts* opts, const abcd_projected* proj,
                                  const abcd_tiles* tiles, const void* F, const void* B,
                                  int fb_dtype, const float* bg, const abcd_fwd_state* state,
                                  const float* dL_dout, int n, float* grad2d, bool grad_cleared) {
  if (!ctx) return ABCD_ERR_INVALID_ARG;
  if (!cam || cam->width <= 0 || cam->height <= 0 || !tiles || !tiles->ids || !tiles->ranges)
    return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_render_backward: bad camera or tiles");
  if (!proj_ok(proj)) return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_render_backward: bad projected buffers");
  if (!fb_ok(F, B, fb_dtype)) return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_render_backward: bad F/B dtype or alignment");
  if (!state || !state->A_T || !state->n_last || !dL_dout || n < 0 || (n > 0 && !grad2d))
    return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_render_backward: null state, gradient or output");
  if (n == 0) return ABCD_OK;
  if (!grad_cleared) {
    const abcd_status z = zero_async(ctx, grad2d, sizeof(float) * 9 * (size_t)n, "grad2d clear");
    if (z != ABCD_OK) return z;
  }
  BwdArgs a;
  a.status = ctx->ws.status;
  a.cam = make_cam(cam, opts);
  a.op = make_opts(opts);
  a.uv = (const float2*)proj->uv;
  a.co = (const float4*)proj->conic_opacity;
  a.rgb = proj->rgb;
  a.ids = tiles->ids;
  a.ranges = (const uint2*)tiles->ranges;
  a.F = F; a.B = B; a.fb_dtype = fb_dtype;
  for (int c = 0; c < 3; ++c) a.bg[c] = bg ? bg[c] : 0.f;
  a.state_at = (const float4*)state->A_T;
  a.n_last = state->n_last;
  a.dl_dout = dL_dout;
  a.grad2d = grad2d;
  const int n_tiles = a.cam.tiles_x * a.cam.tiles_y, n_blocks = n_tiles * kSubPerTile;
  a.tile_order = tile_order_for(ctx, tiles, n_tiles);
  a.ckpt = nullptr; a.ck_items = nullptr; a.ck_count = nullptr; a.ck_first = nullptr;
  a.ck_cap = 0; a.n_item_ctas = 0;
  if (ckpt_ok(ctx, n_blocks) && ctx->ck_state == state->A_T && ctx->ck_blocks == n_blocks &&
      ctx->ck_ranges == tiles->ranges) {
    a.ckpt = ctx->ws.ckpt; a.ck_items = ctx->ws.ck_items; a.ck_count = ctx->ws.ck_count;
    a.ck_first = ctx->ws.ck_first; a.ck_cap = ctx->ws.ck_cap;
    a.n_item_ctas = std::min(ctx->ws.ck_cap, kItemCtasPerSm * ctx->num_sms);
  }
  return check_launch(ctx, "render_bwd_kernel",
                      launch_pdl(render_bwd_kernel, dim3(a.n_item_ctas + n_blocks), dim3(kSubThreads),
                                 0, ctx->stream, a));
}

extern "C" abcd_status abcd_render_backward(abcd_ctx* ctx, const abcd_camera* cam,
                                            const abcd_render_opts* opts,
                                            const abcd_projected* proj, const abcd_tiles* tiles,
                                            const void* F, const void* B, int fb_dtype,
                                            const float* bg, const abcd_fwd_state* state,
                                            const float* dL_dout, int n, float* grad2d) {
  return render_backward(ctx, cam, opts, proj, tiles, F, B, fb_dtype, bg, state, dL_dout, n, grad2d,
                         false);
}

// ---- packed layers (the cache's tile-sparse format): tile t of a layer is stored iff its
// list is non-empty (a tile with no entry renders (0, 0, 0, 0) exactly), as the block
// tile_map[t] of 16 x 16 fp16 RGBA pixels in row-major order; blocks are numbered in tile order.
namespace abcd {
namespace {

__global__ void __launch_bounds__(1024)
tile_map_kernel(const uint2* ranges, int n_tiles, int* tile_map, int* count) {
  pdl_prologue();
  const int per = (n_tiles + (int)blockDim.x - 1) / (int)blockDim.x;
  const int lo = min(n_tiles, (int)threadIdx.x * per), hi = min(n_tiles, lo + per);
  unsigned long long s = 0;
  for (int t = lo; t < hi; ++t) s += ranges[t].y > ranges[t].x ? 1u : 0u;
  unsigned long long total = 0;
  __shared__ unsigned long long warp_sums[32];
  // exclusive block scan of s
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned long long x = s;
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sums[wid] = x;
  __syncthreads();
  if (wid == 0) {
    const int nw = blockDim.x >> 5;
    unsigned long long v = lane < nw ? warp_sums[lane] : 0ull;
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += y;
    }
    if (lane < nw) warp_sums[lane] = v;
  }
  __syncthreads();
  unsigned long long run = (wid > 0 ? warp_sums[wid - 1] : 0ull) + x - s;
  total = warp_sums[(blockDim.x >> 5) - 1];
  for (int t = lo; t < hi; ++t) {
    const bool used = ranges[t].y > ranges[t].x;
    tile_map[t] = used ? (int)run : -1;
    run += used ? 1u : 0u;
  }
  if (threadIdx.x == 0) *count = (int)total;
}

}  // namespace
}  // namespace abcd

extern "C" abcd_status abcd_render_refresh_packed(abcd_ctx* ctx, const abcd_camera* cam,
                                                  const abcd_render_opts* opts,
                                                  const abcd_projected* proj,
                                                  const abcd_tiles* tiles, int* tile_map,
                                                  void* packed, int* count) {
  if (!ctx) return ABCD_ERR_INVALID_ARG;
  if (!cam || cam->width <= 0 || cam->height <= 0 || !tiles || !tiles->ids || !tiles->ranges)
    return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_render_refresh_packed: bad camera or tiles");
  if (!proj_ok(proj)) return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_render_refresh_packed: bad projected buffers");
  if (!tile_map || !packed || !count || ((uintptr_t)packed & 15) || ((uintptr_t)tile_map & 3))
    return fail(ctx, ABCD_ERR_INVALID_ARG, "abcd_render_refresh_packed: bad or misaligned output");
  FwdArgs a;
  a.status = ctx->ws.status;
  a.cam = make_cam(cam, opts);
  a.op = make_opts(opts);
  a.uv = (const float2*)proj->uv;
  a.co = (const float4*)proj->conic_opacity;
  a.rgb = proj->rgb;
  a.ids = tiles->ids;
  a.ranges = (const uint2*)tiles->ranges;
  a.F = nullptr; a.B = nullptr; a.fb_dtype = ABCD_F16;
  for (int c = 0; c < 3; ++c) a.bg[c] = 0.f;
  a.out = nullptr;
  a.state_at = nullptr;
  a.n_last = nullptr;
  a.refresh = nullptr;
  a.refresh_packed = (uint2*)packed;
  a.tile_map = tile_map;
  const int n_tiles = a.cam.tiles_x * a.cam.tiles_y, n_blocks = n_tiles * kSubPerTile;
  a.tile_order = tile_order_for(ctx, tiles, n_tiles);
  a.ckpt = nullptr; a.ck_items = nullptr; a.ck_count = nullptr; a.ck_first = nullptr;
  a.ck_cap = 0;
  abcd_status s = check_launch(ctx, "tile_map_kernel",
                               launch_pdl(tile_map_kernel, dim3(1), dim3(1024), 0, ctx->stream,
                                          (const uint2*)tiles->ranges, n_tiles, tile_map, count));
  if (s) return s;
  return check_launch(ctx, "render_fwd_kernel",
                      launch_pdl(render_fwd_kernel, dim3(n_blocks), dim3(kSubThreads), 0, ctx->stream, a));
}
