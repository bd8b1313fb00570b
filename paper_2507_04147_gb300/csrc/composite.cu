// composite.cu -- foveated front-to-back compositing of every tile of every eye (Sec. 2.3
// "Rasterization"; Sec. 3.4 AMR; Sec. 3.5 implementation details).
//
// The paper splits a tile into one group per label of its 2x2 blocks (TL 1, BR 2, TR 3, BL 4), and a
// level-k tile runs only the groups of labels 1..k.  Here a label's pixels are assigned to lanes or
// not at all.  plan_kernel computes every tile's level from the gaze in the device mailbox (Eq. 1: the
// distance from the gaze to the tile's nearest pixel centre against r_k = f tan(theta_k)) and lists
// the tiles, or halves of them, as work items by the length of their Gaussian lists; composite_px is
// one persistent launch that takes the items, the heaviest first.
//
// Per batch, a CTA gathers the tile's next Gaussians (indices from the sorted values) into shared
// memory; each warp lists those that reach its patch and blends them front to back with the 1/255
// skip, the 0.99 clamp and the 1e-4 transmittance stop, until all its pixels are done.  The exp of
// the falloff uses the MUFU ex2 unit with log2(e) folded into the conic.  The blend is branch-free,
// so a warp whose lanes disagree on the accept test does not run both sides.
#include <algorithm>

#include "blend.cuh"
#include "common.cuh"

namespace a3fr {
namespace {

// Level of tile `tile` of eye `eye` (exactly rounded; the same decision as the definition).
__device__ __forceinline__ int tile_level(const CompositeParams &p, int eye, int tile,
                                          const float *gaze) {
  const int tx = tile % p.tiles_x, ty = tile / p.tiles_x;
  const float gx = gaze[2 * eye], gy = gaze[2 * eye + 1];
  const float x0 = (float)(tx * p.tile), y0 = (float)(ty * p.tile);
  const float x1 = (float)(min((tx + 1) * p.tile, p.width) - 1);
  const float y1 = (float)(min((ty + 1) * p.tile, p.height) - 1);
  const float dx = fmaxf(fmaxf(fs(x0, gx), fs(gx, x1)), 0.0f);
  const float dy = fmaxf(fmaxf(fs(y0, gy), fs(gy, y1)), 0.0f);
  const float d2 = fa(fm(dx, dx), fm(dy, dy));
  int layer = p.n_layers - 1;
  for (int k = p.n_layers - 2; k >= 0; --k)
    if (d2 <= p.r2[eye][k]) layer = k;
  return p.level[layer];
}

// Count-based tile levels (Sec. 3.6, 4.6): per eye (one CTA each), the instance count tau of the k-th
// heaviest tile, k = floor(count_frac * tiles), by an exact radix select (four 8-bit digits,
// most significant first) over the tiles' range lengths; tau = UINT32_MAX when k < 1 (no tile is
// heavy).  A digit is found by one warp's scan of the 256 counts from the top: read one after
// another by one thread, for the eyes in turn, they took 46 us on 2 x 2,835 tiles (ncu), 6.4 us now.
__global__ void __launch_bounds__(1024)
tile_threshold_kernel(const CompositeParams *__restrict__ pp, const uint2 *__restrict__ ranges,
                      uint32_t *__restrict__ thresholds) {
  pdl_begin();
  const CompositeParams &p = *pp;
  __shared__ uint32_t s_hist[256];
  __shared__ uint32_t s_prefix, s_k;
  const int t = threadIdx.x, e = blockIdx.x;
  const uint32_t k0 = (uint32_t)floorf(p.count_frac * (float)p.n_tiles);
  if (k0 < 1u) {
    if (t == 0) thresholds[e] = 0xffffffffu;
    return;
  }
  if (t == 0) {
    s_prefix = 0u;
    s_k = min(k0, (uint32_t)p.n_tiles);
  }
  for (int shift = 24; shift >= 0; shift -= 8) {
    if (t < 256) s_hist[t] = 0u;
    __syncthreads();
    const uint32_t prefix = s_prefix;
    for (int i = t; i < p.n_tiles; i += blockDim.x) {
      const uint2 r = ranges[e * p.n_tiles + i];
      const uint32_t c = r.y - r.x;
      const bool match = shift == 24 || (c >> (shift + 8)) == prefix;
      if (match) atomicAdd(&s_hist[(c >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (t < 32) {
      // lane l: digits 255 - 8 l down to 248 - 8 l; at least k tiles match the prefix
      uint32_t n[8], sum = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        n[j] = s_hist[255 - 8 * t - j];
        sum += n[j];
      }
      uint32_t incl = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if (t >= o) incl += v;
      }
      uint32_t k = s_k;
      __syncwarp();
      if (incl >= k && incl - sum < k) {   // the k-th heaviest is among this lane's digits
        k -= incl - sum;
        int j = 0;
        while (j < 7 && n[j] < k) k -= n[j++];
        s_k = k;
        s_prefix = (prefix << 8) | (uint32_t)(255 - 8 * t - j);
      }
    }
    __syncthreads();
  }
  if (t == 0) thresholds[e] = s_prefix;
}

// Label interval (lo, hi] a composite renders in tile gt (eye-major global tile index), and
// the tile's bookkeeping (cur, levels).  Three uses:
//   * a normal foveated render: lo = 0, hi = the tile's level from the gaze mailbox (Eq. 1),
//     lowered for heavy tiles by the count-based rule when count_frac > 0;
//   * a uniform render (uniform > 0): lo = 0, hi = uniform for every tile (the first round of
//     a frame, and the full-resolution render with uniform = 4);
//   * a later round (round != nullptr): hi = the level from the round's gaze and radii, lo =
//     the level already rendered (cur); tiles with hi <= lo render nothing; cur becomes hi.
__device__ __forceinline__ void tile_interval(const CompositeParams &p, int gt, const float *gaze,
                                              const RoundPlan *round, int uniform, uint8_t *cur,
                                              uint8_t *levels, const uint2 *ranges,
                                              const uint32_t *thresholds, int *lo_out, int *hi_out) {
  const int eye = gt / p.n_tiles;
  const int tile = gt - eye * p.n_tiles;
  int lo = 0, hi;
  if (uniform > 0) {
    hi = uniform;
  } else if (round != nullptr) {
    hi = 0;
    if (round->active) {
      CompositeParams q = p;
      for (int k = 0; k < 3; ++k) q.r2[eye][k] = round->r2[eye][k];
      hi = tile_level(q, eye, tile, &round->gaze[0][0]);
    }
    lo = cur[gt];
  } else {
    hi = tile_level(p, eye, tile, gaze);
    if (p.count_frac > 0.0f && (hi == 2 || hi == 3)) {
      // a heavy tile (count >= the k-th largest count of its eye) drops one level
      const uint2 r = ranges[gt];
      const uint32_t c = r.y - r.x;
      if (c > 0u && c >= thresholds[eye]) hi -= 1;
    }
  }
  if (cur != nullptr && hi > lo) cur[gt] = (uint8_t)hi;
  levels[gt] = (uint8_t)(hi > lo ? hi : lo);
  *lo_out = lo;
  *hi_out = hi;
}

// Work plan of one composite launch (composite_px_kernel).  A tile rendering the P = hi - lo
// labels (lo, hi] is `parts` work items (halves of the tile, or the whole of it); a tile with no
// instances is one item that only writes background.  Items go into kItemClasses classes by the
// tile's instance count (class 0: none; class c: 4^(c-1) <= count < 4^c; the last class unbounded)
// and the composite takes the heaviest class first, so the longest items start first and the
// short ones fill in behind them.  items[c * 4 * n_ranges + slot] = gt << 6 | (P - 1) << 4 |
// region << 2 | lo, class sizes in class_counts[0..kItemClasses).
constexpr int kItemClasses = 8;

__global__ void __launch_bounds__(256)
plan_kernel(const CompositeParams *__restrict__ pp, const float *__restrict__ gaze_ring,
            const RoundPlan *__restrict__ round, int uniform, int parts, uint8_t *__restrict__ cur,
            uint8_t *__restrict__ levels, uint32_t *__restrict__ items,
            uint32_t *__restrict__ class_counts, const uint2 *__restrict__ ranges,
            const uint32_t *__restrict__ thresholds) {
  pdl_begin();
  const CompositeParams &p = *pp;
  const float *gaze = gaze_ring + 4 * p.gaze_slot;
  const int n_ranges = p.n_eyes * p.n_tiles;
  const int gt = blockIdx.x * blockDim.x + threadIdx.x;
  if (gt >= n_ranges) return;
  int lo, hi;
  tile_interval(p, gt, gaze, round, uniform, cur, levels, ranges, thresholds, &lo, &hi);
  if (hi <= lo) return;
  const int P = hi - lo;
  const uint2 r = ranges[gt];
  const uint32_t count = r.y > r.x ? r.y - r.x : 0u;
  const int n_items = count == 0u ? 1 : parts;
  const int cls = count == 0u ? 0 : min(kItemClasses - 1, 1 + (31 - __clz(count)) / 2);
  const uint32_t slot = atomicAdd(class_counts + cls, (uint32_t)n_items);
  uint32_t *dst = items + (size_t)cls * 4 * n_ranges + slot;
  for (int k = 0; k < n_items; ++k)
    dst[k] = ((uint32_t)gt << 6) | ((uint32_t)(P - 1) << 4) | ((uint32_t)k << 2) | (uint32_t)lo;
}

// A tile of labels (lo, hi] renders those P = hi - lo labels of every 2 x 2 block and no others (the
// paper's groups above the level exit; here their pixels are never assigned).  One persistent
// launch renders every item of the plan (plan_kernel) -- both eyes, every layer -- taking items
// heaviest class first from an atomic counter, so the longest lists start first and the short
// ones fill in behind them.  A 128-thread CTA renders one item.  Per batch it stages the tile's
// next Gaussians in shared memory with the box where each can reach alpha = 1/255; every warp
// builds the hit list of its patch (box test, then the exact falloff over the patch: a Gaussian
// left out has alpha < 1/255 at every pixel of the patch, so no output bit changes) and blends
// only those, front to back, with the 1/255 skip, the 0.99 clamp and the 1e-4 stop.  The per-pixel
// arithmetic is the same in every shape, so images do not depend on how tiles are cut into items.
// A tile rendered from label 0 also writes its inherited pixels (the labels above hi take the
// top-left value).  Three shapes:
//   kTile32       32-pixel tiles (the paper's, Sec. 3.5): an item is half a tile, a lane the P
//                 pixels of one block, so a staged Gaussian is set up once for them; a warp's
//                 patch is 16 x 8 pixels.
//   kTile16       16-pixel tiles: an item is a tile, a warp's patch 8 x 8 pixels, two pixels a lane.
//                 Bound by issue, as kTile32; every warp walking the whole list of its tile, one
//                 pixel a lane, took 254 us on the 1M-Gaussian 1920 x 1080 full render (ncu), this
//                 shape 111 us.
//   kTile16Split  the same in half tiles, a patch 8 x 4 pixels, one pixel a lane: for renders with
//                 too few tiles to fill the device, which are bound by the longest list's chain of
//                 blends; fewer Gaussians reach the smaller patch.
enum : int { kTile32 = 0, kTile16 = 1, kTile16Split = 2 };
constexpr int kHalfThreads = 128;
constexpr int kBatch = 256;   // Gaussians staged per batch (times the staging multiple)
// 16-pixel tiles are split in halves up to this many tiles per SM (of 7 CTAs resident).  Whole
// render, split / not: 256 tiles 163 / 188 us, 825 tiles (training step) 420 / 451 us, 4,096 tiles
// (training step) 896 / 889 us, 5,670 tiles 241 / 227 us, 8,160 tiles 616 / 567 us.
constexpr int kSplitTilesPerSm = 16;

__device__ __forceinline__ int label_dx(int L) { return (L == 1 || L == 2) ? 1 : 0; }
__device__ __forceinline__ int label_dy(int L) { return (L == 1 || L == 3) ? 1 : 0; }

template <int kMult>
struct ItemSmem {
  // one slot past the batch: a Gaussian of opacity 0, which fails the 1/255 test everywhere
  float4 geo[kBatch * kMult + 1];
  float2 cz[kBatch * kMult + 1];
  float4 rgb[kBatch * kMult + 1];
  short4 box[kBatch * kMult];        // support box, outward-rounded pixels
  float thr[kBatch * kMult];         // log2 falloff needed for alpha = 1/255
  // per warp: batch slots that reach its patch, padded to a multiple of 4 with the empty slot
  uint16_t hits[kHalfThreads / 32][kBatch * kMult + 4];
  int done[kHalfThreads / 32];
  uint32_t prefix[kItemClasses + 1];  // item index ranges, heaviest class first
  uint32_t item;
};

// The pixels of one lane: P pixel centres (in pairs), which of them are to be rendered, and the
// warp's patch -- the span of the pixel centres of all its lanes.
template <int P>
struct LanePixels {
  float x[P], y[P];
  bool inside[P];
  float wx0, wx1, wy0, wy1;
};

// One item, by the whole CTA: the Gaussians of a tile's list blended into every lane's pixels.
// A finished pixel is marked by T = 0 (a live pixel keeps T >= 1e-4): skipped Gaussians then blend
// with alpha 0, which leaves T and the colour bit for bit as they were, and every later Gaussian of
// a finished pixel stops with weight 0.  With the auxiliary outputs a finished pixel keeps its final
// transmittance negated instead, and the loop also keeps the last contributor and the evaluation and
// blend counts: one select each and no flags (500k stereo 158 -> 137 us under ncu; 16-pixel tiles, at
// 5 CTAs per SM, 1M at 1024 x 1024 76 -> 71 us).  inherit: pixel 0 is the top-left one of the block at (px0, py0), and the labels from
// hi on take its value.
template <int P, bool kAux, int kMult>
__device__ __forceinline__ void render_pixels(ItemSmem<kMult> &sm, const CompositeParams &p, const float *rec,
                                              int n, int eye, uint2 range, const LanePixels<P> &lp,
                                              bool inherit, int hi, int px0, int py0,
                                              const uint32_t *vals,
                                              float *t_final, uint32_t *n_contrib, float *depth,
                                              unsigned long long &ev, unsigned long long &bl,
                                              unsigned long long &staged) {
  constexpr int NB = kBatch * kMult;
  float *out = p.out;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const float (&fpx)[P] = lp.x, (&fpy)[P] = lp.y;
  const bool (&inside)[P] = lp.inside;
  const float wx0 = lp.wx0, wx1 = lp.wx1, wy0 = lp.wy0, wy1 = lp.wy1;
  const float *rec_eye = rec + (size_t)eye * n * kRec;

  float T[P], C0[P], C1[P], C2[P], Z[P];
  uint32_t last[P], stop[P], blended = 0;
#pragma unroll
  for (int k = 0; k < P; ++k) {
    T[k] = inside[k] ? 1.0f : (kAux ? -1.0f : 0.0f);
    C0[k] = C1[k] = C2[k] = Z[k] = 0.0f;
    last[k] = stop[k] = 0u;
  }
  auto all_done = [&]() {
    bool a = true;
#pragma unroll
    for (int k = 0; k < P; ++k) a = a && T[k] <= 0.0f;
    return a;
  };
  // the auxiliary outputs' bookkeeping of pixel k at list position pos, and its new T: alpha a is
  // blended unless it would end the pixel or the pixel had ended (tt, T (1 - a), below 1e-4 or negative)
  auto note = [&](int k, float a, float tt, uint32_t pos) {
    const bool go = tt >= 0.0001f, upd = go && a > 0.0f;
    last[k] = upd ? pos : last[k];
    blended += upd ? 1u : 0u;
    stop[k] = !go && T[k] > 0.0f ? pos : stop[k];
    T[k] = go ? tt : -fabsf(T[k]);
  };
  for (uint32_t start = range.x; start < range.y; start += NB) {
    const bool wdone = __all_sync(0xffffffffu, all_done());
    if (lane == 0) sm.done[warp] = wdone;
    __syncthreads();
    bool all = true;
#pragma unroll
    for (int w = 0; w < kHalfThreads / 32; ++w) all = all && sm.done[w];
    if (all) break;
    const uint32_t cnt = min((uint32_t)NB, range.y - start);
    if (t == 0) staged += cnt;
#pragma unroll
    for (int j = 0; j < NB / kHalfThreads; ++j) {
      const uint32_t slot = (uint32_t)(t + j * kHalfThreads);
      if (slot < cnt) {
        const uint32_t gidx = min(vals[start + slot], (uint32_t)(n - 1));   // in range unless a sort failed
        const float4 *r4 = reinterpret_cast<const float4 *>(rec_eye + (size_t)gidx * kRec);
        const float4 a = __ldg(r4), b = __ldg(r4 + 1), c = __ldg(r4 + 2);
        sm.geo[slot] = make_float4(a.x, a.y, __fmul_rn(-0.5f * kLog2e, a.z), __fmul_rn(-kLog2e, a.w));
        sm.cz[slot] = make_float2(__fmul_rn(-0.5f * kLog2e, b.x), c.y);
        sm.rgb[slot] = make_float4(b.z, b.w, c.x, b.y);
        sm.box[slot] = int_box(support_box(a.x, a.y, a.z, a.w, b.x, b.y));
        sm.thr[slot] = -__log2f(255.0f * b.y) - 0.01f;
      }
    }
    __syncthreads();
    if (!__all_sync(0xffffffffu, all_done())) {
      // the warp's hit list: 32 Gaussians tested per step (support box, then the falloff
      // over the patch), slots kept in list order
      int n_hit = 0;
      for (uint32_t base = 0; base < cnt; base += 32) {
        const uint32_t k = base + (uint32_t)lane;
        bool hit = false;
        if (k < cnt) {
          const short4 box = sm.box[k];
          hit = !((float)box.y < wx0 || (float)box.x > wx1 || (float)box.w < wy0 || (float)box.z > wy1);
        }
        const unsigned m = __ballot_sync(0xffffffffu, hit);
        if (hit) sm.hits[warp][n_hit + __popc(m & ((1u << lane) - 1u))] = (uint16_t)k;
        n_hit += __popc(m);
      }
      __syncwarp();
      {
        int n_keep = 0;
        for (int base = 0; base < n_hit; base += 32) {
          const int i = base + lane;
          int k = 0;
          bool keep = false;
          if (i < n_hit) {
            k = sm.hits[warp][i];
            const float4 geo = sm.geo[k];
            keep = falloff_reaches(geo.z, geo.w, sm.cz[k].x, sm.thr[k], wx0 - geo.x, wx1 - geo.x,
                                   wy0 - geo.y, wy1 - geo.y);
          }
          __syncwarp();
          const unsigned m = __ballot_sync(0xffffffffu, keep);
          if (keep) sm.hits[warp][n_keep + __popc(m & ((1u << lane) - 1u))] = (uint16_t)k;
          n_keep += __popc(m);
        }
        n_hit = n_keep;
        // padding: the steps of four below have no exit inside them, so their loads overlap
        // (with one after each: 500k stereo composite 107 -> 99 us, the longest chain of the 20k
        // 256 x 256 view 96 -> 75 us)
        if (lane < 3) sm.hits[warp][n_hit + lane] = (uint16_t)NB;
      }
      __syncwarp();
      const uint32_t pos0 = start - range.x + 1;
      for (int i = 0; i < n_hit; i += 4) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          // four of these at once would spill (248 bytes; 500k stereo frame 407 -> 425 us)
          if (kAux && P > 2 && i + j >= n_hit) break;
          const int e = sm.hits[warp][i + j];
          const float4 geo = sm.geo[e];
          const float2 cz = sm.cz[e];
          const float4 rgb = sm.rgb[e];
          const uint32_t pos = pos0 + (uint32_t)e;
          if constexpr (P >= 2) {
            // pixel pairs (0, 1) and (2, 3): the same operations as the scalar loop below, two
            // pixels per instruction wherever both take the same one
            const f32x2 gx = f2_pack(geo.x, geo.x), gy = f2_pack(geo.y, geo.y);
            const f32x2 ca = f2_pack(geo.z, geo.z), cb = f2_pack(geo.w, geo.w), cc = f2_pack(cz.x, cz.x);
            const f32x2 op = f2_pack(rgb.w, rgb.w);
            const f32x2 cr = f2_pack(rgb.x, rgb.x), cg = f2_pack(rgb.y, rgb.y), cbl = f2_pack(rgb.z, rgb.z);
            const f32x2 one = f2_pack(1.0f, 1.0f), mone = f2_pack(-1.0f, -1.0f);
#pragma unroll
            for (int k = 0; k + 1 < P; k += 2) {
              const f32x2 dx = f2_add(gx, f2_pack(-fpx[k], -fpx[k + 1]));
              const f32x2 dy = f2_add(gy, f2_pack(-fpy[k], -fpy[k + 1]));
              // falloff_log2: (A dx + B dy) dx + (C dy) dy, rounded step by step
              const f32x2 pw2 = f2_fma(f2_fma(ca, dx, f2_mul(cb, dy)), dx, f2_mul(f2_mul(cc, dy), dy));
              float pw0, pw1;
              f2_unpack(pw2, pw0, pw1);
              float oe0, oe1;
              f2_unpack(f2_mul(op, f2_pack(ex2_approx(pw0), ex2_approx(pw1))), oe0, oe1);
              const float al0 = fminf(0.99f, oe0), al1 = fminf(0.99f, oe1);
              const float a0 = (pw0 <= 0.0f && al0 >= 1.0f / 255.0f) ? al0 : 0.0f;
              const float a1 = (pw1 <= 0.0f && al1 >= 1.0f / 255.0f) ? al1 : 0.0f;
              const f32x2 a2 = f2_pack(a0, a1), t2 = f2_pack(T[k], T[k + 1]);
              const f32x2 tt2 = f2_mul(t2, f2_fma(a2, mone, one));   // T (1 - a)
              float tt0, tt1;
              f2_unpack(tt2, tt0, tt1);
              // 1 while the pixel goes on, 0 once this Gaussian would end it (or it ended):
              // multiplying by it equals the scalar path's selects bit for bit (T, a T >= 0)
              const f32x2 keep = f2_pack(ge_factor(tt0, 0.0001f), ge_factor(tt1, 0.0001f));
              const f32x2 w2 = f2_mul(f2_mul(a2, t2), keep);
              f2_unpack(f2_fma(cr, w2, f2_pack(C0[k], C0[k + 1])), C0[k], C0[k + 1]);
              f2_unpack(f2_fma(cg, w2, f2_pack(C1[k], C1[k + 1])), C1[k], C1[k + 1]);
              f2_unpack(f2_fma(cbl, w2, f2_pack(C2[k], C2[k + 1])), C2[k], C2[k + 1]);
              if constexpr (kAux) {
                f2_unpack(f2_fma(f2_pack(cz.y, cz.y), w2, f2_pack(Z[k], Z[k + 1])), Z[k], Z[k + 1]);
                note(k, a0, tt0, pos);
                note(k + 1, a1, tt1, pos);
              } else {
                f2_unpack(f2_mul(tt2, keep), T[k], T[k + 1]);
              }
            }
          }
#pragma unroll
          for (int k = 0; k < P; ++k) {
            if constexpr (P >= 2) {
              if (k + 1 < P || P % 2 == 0) continue;   // done in pairs above (all but an odd last)
            }
            const float dx = __fsub_rn(geo.x, fpx[k]), dy = __fsub_rn(geo.y, fpy[k]);
            const float pw = falloff_log2(geo.z, geo.w, cz.x, dx, dy);
            const float alpha = blend_alpha(rgb.w, pw);
            const float a = (pw <= 0.0f && alpha >= 1.0f / 255.0f) ? alpha : 0.0f;
            const float tt = __fmul_rn(T[k], __fsub_rn(1.0f, a));
            const bool fin = tt < 0.0001f;   // this Gaussian would end the pixel, or it ended
            const float w = fin ? 0.0f : __fmul_rn(a, T[k]);
            C0[k] = __fmaf_rn(rgb.x, w, C0[k]);
            C1[k] = __fmaf_rn(rgb.y, w, C1[k]);
            C2[k] = __fmaf_rn(rgb.z, w, C2[k]);
            if constexpr (kAux) {
              Z[k] = __fmaf_rn(cz.y, w, Z[k]);
              note(k, a, tt, pos);
            } else {
              T[k] = fin ? 0.0f : tt;
            }
          }
        }
        if (__all_sync(0xffffffffu, all_done())) break;
      }
    }
    __syncthreads();   // the next batch overwrites the staged Gaussians
  }
#pragma unroll
  for (int k = 0; k < P; ++k) {
    if (!inside[k]) continue;
    if (kAux) {
      if (T[k] > 0.0f) stop[k] = range.y - range.x;
      T[k] = fabsf(T[k]);
      ev += stop[k];
    }
    const size_t pix = ((size_t)eye * p.height + (size_t)fpy[k]) * p.width + (size_t)fpx[k];
    out[3 * pix] = C0[k];
    out[3 * pix + 1] = C1[k];
    out[3 * pix + 2] = C2[k];
    if (kAux) {
      t_final[pix] = T[k];
      n_contrib[pix] = last[k];
      depth[pix] = Z[k];
    }
  }
  bl += blended;
  if (inherit && inside[0]) {
    for (int L = hi; L < 4; ++L) {
      const int x = px0 + label_dx(L), y = py0 + label_dy(L);
      if (x >= p.width || y >= p.height) continue;
      const size_t q = ((size_t)eye * p.height + y) * p.width + x;
      out[3 * q] = C0[0];
      out[3 * q + 1] = C1[0];
      out[3 * q + 2] = C2[0];
      if (kAux) {
        t_final[q] = T[0];
        n_contrib[q] = last[0];
        depth[q] = Z[0];
      }
    }
  }
}

// 32-pixel tiles: labels lo .. lo + P - 1 of the 16 x 8 blocks of half `half` of the tile, a lane
// the P pixels of one block, a warp 8 x 4 blocks (kLo0: lo is 0, so the lane's pixel offsets are
// known at compile time).
template <int P, bool kLo0>
__device__ __forceinline__ LanePixels<P> pixels32(const CompositeParams &p, int tx, int ty, int half, int lo,
                                                  int &px0, int &py0) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bx = (lane & 7) + 8 * (warp & 1), by = 8 * half + 4 * (warp >> 1) + (lane >> 3);
  px0 = tx * 32 + 2 * bx;
  py0 = ty * 32 + 2 * by;   // the block's top-left pixel
  LanePixels<P> lp;
  int any_ox = 0, all_ox = 1, any_oy = 0, all_oy = 1;
#pragma unroll
  for (int k = 0; k < P; ++k) {
    const int L = kLo0 ? k : lo + k;
    const int ox = label_dx(L), oy = label_dy(L);
    any_ox |= ox;
    all_ox &= ox;
    any_oy |= oy;
    all_oy &= oy;
    lp.inside[k] = px0 + ox < p.width && py0 + oy < p.height;
    lp.x[k] = (float)(px0 + ox);
    lp.y[k] = (float)(py0 + oy);
  }
  // the warp's patch: the span of its pixels (one label: every other pixel of 16 x 8)
  const int wxb = tx * 32 + 16 * (warp & 1), wyb = ty * 32 + 16 * half + 8 * (warp >> 1);
  lp.wx0 = (float)(wxb + all_ox);
  lp.wx1 = (float)(wxb + 14 + any_ox);
  lp.wy0 = (float)(wyb + all_oy);
  lp.wy1 = (float)(wyb + 6 + any_oy);
  return lp;
}

// 16-pixel tiles: labels lo .. lo + P - 1 of a warp's patch of 4 x BH blocks (BH 4: the CTA's four
// warps cover the tile; BH 2: half `half` of it).  The lanes are the patch's blocks times 8 / BH
// label slots; a slot is Q consecutive labels (Q 2 with BH 4 when P > 2, else 1).
template <int Q, int BH>
__device__ __forceinline__ LanePixels<Q> pixels16(const CompositeParams &p, int tx, int ty, int half, int lo, int P,
                                                  int &px0, int &py0) {
  constexpr int NB = 4 * BH;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wxb = tx * 16 + 8 * (warp & 1), wyb = ty * 16 + (BH == 4 ? 0 : 8 * half) + 2 * BH * (warp >> 1);
  const int blk = lane % NB, slot = lane / NB;
  px0 = wxb + 2 * (blk & 3);
  py0 = wyb + 2 * (blk >> 2);
  LanePixels<Q> lp;
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    const int L = lo + slot * Q + k;
    const int x = px0 + label_dx(L), y = py0 + label_dy(L);
    lp.inside[k] = slot * Q + k < P && x < p.width && y < p.height;
    lp.x[k] = (float)x;
    lp.y[k] = (float)y;
  }
  int any_ox = 0, all_ox = 1, any_oy = 0, all_oy = 1;
  for (int L = lo; L < lo + P; ++L) {
    any_ox |= label_dx(L);
    all_ox &= label_dx(L);
    any_oy |= label_dy(L);
    all_oy &= label_dy(L);
  }
  lp.wx0 = (float)(wxb + all_ox);
  lp.wx1 = (float)(wxb + 6 + any_ox);
  lp.wy0 = (float)(wyb + all_oy);
  lp.wy1 = (float)(wyb + 2 * (BH - 1) + any_oy);
  return lp;
}

template <bool kAux, int kMult, int kShape>
__global__ void __launch_bounds__(kHalfThreads, kAux ? (kShape == kTile32 ? 6 : 5) : 7)
composite_px_kernel(const CompositeParams *__restrict__ pp, const float *__restrict__ rec, int n,
                    const uint2 *__restrict__ ranges, const uint32_t *__restrict__ kept,
                    const uint32_t *__restrict__ vals, const uint32_t *__restrict__ items,
                    const uint32_t *__restrict__ class_counts, uint32_t *__restrict__ work,
                    int incremental, float *__restrict__ t_final,
                    uint32_t *__restrict__ n_contrib, float *__restrict__ depth,
                    unsigned long long *__restrict__ counters) {
  pdl_begin();
  __shared__ ItemSmem<kMult> sm;
  const CompositeParams &p = *pp;
  float *out = p.out;
  const int t = threadIdx.x, lane = t & 31;
  const int n_ranges = p.n_eyes * p.n_tiles;
  const size_t cap = 4 * (size_t)n_ranges;
  if (t == 0) {
    sm.geo[kBatch * kMult] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    sm.cz[kBatch * kMult] = make_float2(0.0f, 0.0f);
    sm.rgb[kBatch * kMult] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    sm.prefix[0] = 0u;
    for (int i = 0; i < kItemClasses; ++i)
      sm.prefix[i + 1] = sm.prefix[i] + class_counts[kItemClasses - 1 - i];
  }
  __syncthreads();
  const uint32_t total = sm.prefix[kItemClasses];
  const uint32_t n_kept = *kept;   // fewer than the instances only after a capacity overflow
  unsigned long long ev = 0, bl = 0, staged = 0;

  for (;;) {
    if (t == 0) sm.item = atomicAdd(work, 1u);
    __syncthreads();
    const uint32_t w = sm.item;
    if (w >= total) break;
    int ci = 0;
    while (w >= sm.prefix[ci + 1]) ++ci;
    const uint32_t item = items[(size_t)(kItemClasses - 1 - ci) * cap + (w - sm.prefix[ci])];
    const int gtile = (int)(item >> 6);
    const int P = (int)((item >> 4) & 3u) + 1;
    const int half = (int)((item >> 2) & 3u);
    const int lo = (int)(item & 3u), hi = lo + P;
    uint2 range = ranges[gtile];
    range.x = min(range.x, n_kept);
    range.y = min(range.y, n_kept);
    const bool inherit = !incremental && lo == 0 && hi < 4;
    constexpr int TS = kShape == kTile32 ? 32 : 16;
    const int eye = gtile / p.n_tiles;
    const int tile = gtile - eye * p.n_tiles;
    const int tx = tile % p.tiles_x, ty = tile / p.tiles_x;
    if (range.y <= range.x) {
      // no Gaussian reaches the tile: background (0) for every pixel the tile's items would
      // write (this is the tile's only item)
      for (int b = t; b < TS * TS / 4; b += kHalfThreads) {
        const int px0 = tx * TS + 2 * (b % (TS / 2)), py0 = ty * TS + 2 * (b / (TS / 2));
        for (int L = lo; L < 4; ++L) {
          if (L >= hi && !inherit) break;
          const int x = px0 + label_dx(L), y = py0 + label_dy(L);
          if (x >= p.width || y >= p.height) continue;
          const size_t pix = ((size_t)eye * p.height + y) * p.width + x;
          out[3 * pix] = 0.0f;
          out[3 * pix + 1] = 0.0f;
          out[3 * pix + 2] = 0.0f;
          if (kAux) {
            t_final[pix] = 1.0f;
            n_contrib[pix] = 0u;
            depth[pix] = 0.0f;
          }
        }
      }
    } else {
      int px0, py0;
#define A3FR_RENDER(PP, INHERIT, HI)                                                                             \
  render_pixels<PP, kAux, kMult>(sm, p, rec, n, eye, range, lp, INHERIT, HI, px0, py0, vals, t_final, n_contrib, \
                                 depth, ev, bl, staged)
#define A3FR_HALF(PP, LO0)                                            \
  {                                                                   \
    const auto lp = pixels32<PP, LO0>(p, tx, ty, half, lo, px0, py0); \
    A3FR_RENDER(PP, inherit, LO0 ? PP : hi);                          \
  }
      if constexpr (kShape != kTile32) {
        // the lanes of slot 0 hold label lo
        const bool mine = inherit && lane < (kShape == kTile16 ? 16 : 8);
        if (kShape == kTile16 && P > 2) {
          const auto lp = pixels16<2, 4>(p, tx, ty, half, lo, P, px0, py0);
          A3FR_RENDER(2, mine, hi);
        } else {
          const auto lp = pixels16<1, kShape == kTile16 ? 4 : 2>(p, tx, ty, half, lo, P, px0, py0);
          A3FR_RENDER(1, mine, hi);
        }
      } else if (lo == 0) {
        switch (P) {
          case 1: A3FR_HALF(1, true); break;
          case 2: A3FR_HALF(2, true); break;
          case 3: A3FR_HALF(3, true); break;
          default: A3FR_HALF(4, true); break;
        }
      } else {   // later rounds: labels above the ones already rendered (lo + P <= 4)
        switch (P) {
          case 1: A3FR_HALF(1, false); break;
          case 2: A3FR_HALF(2, false); break;
          default: A3FR_HALF(3, false); break;
        }
      }
#undef A3FR_HALF
#undef A3FR_RENDER
    }
    __syncthreads();   // every thread has read sm.item and is done with the staging arrays
  }
  // statistics: records staged (thread 0 counts its CTA's); with the auxiliary outputs also
  // the evaluations and the blends
  if (kAux) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      ev += __shfl_xor_sync(0xffffffffu, ev, o);
      bl += __shfl_xor_sync(0xffffffffu, bl, o);
    }
    if (lane == 0) {
      if (ev) atomicAdd(counters, ev);
      if (bl) atomicAdd(counters + 2, bl);
    }
  }
  if (t == 0 && staged) atomicAdd(counters + 1, staged);
}

}  // namespace

// The plan buffer: the items [kItemClasses * 4 * n_ranges], then their class counts [kItemClasses]
// and the work counter.
size_t plan_bytes(int n_ranges) {
  return sizeof(uint32_t) * ((size_t)kItemClasses * 4 * (size_t)n_ranges + kItemClasses + 8);
}

cudaError_t launch_composite(const CompositeParams &p, const CompositeParams *p_dev,
                             const float *rec, int n, const uint2 *ranges, const uint32_t *kept,
                             const uint32_t *vals, const float *gaze, const RoundPlan *round,
                             int uniform, uint8_t *cur, uint32_t *plan, uint8_t *levels,
                             float *t_final, uint32_t *n_contrib, float *depth,
                             unsigned long long *counters, int batch_mult, uint32_t *thresholds,
                             cudaStream_t s, int *kernels) {
  const int n_ranges = p.n_eyes * p.n_tiles;
  if (kernels) *kernels = 0;
  if (n_ranges <= 0) return cudaSuccess;
  const int inc = round != nullptr ? 1 : 0;
  const bool aux = t_final != nullptr;
  const int mult = batch_mult == 2 ? 2 : 1;
  const bool by_count = !p.full && p.count_frac > 0.0f && round == nullptr && uniform == 0;
  // shared memory preferred so that registers, not the carveout, set residency
  auto prefer_smem = [](auto kern, int variant) {
    static bool carve[64][16] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 && variant >= 0 && variant < 16 &&
        !carve[dev][variant]) {
      cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                           cudaSharedmemCarveoutMaxShared);
      carve[dev][variant] = true;
    }
  };
  if (by_count) {
    {
      const cudaError_t e_ = launch_pdl(tile_threshold_kernel, p.n_eyes, 1024, 0, s, p_dev, ranges, thresholds);
      if (e_ != cudaSuccess) return e_;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (kernels) ++*kernels;
  }
  // plan (every tile, also for the full render: uniform level 4) + one persistent composite
  uint32_t *items = plan;
  uint32_t *class_counts = plan + (size_t)kItemClasses * 4 * n_ranges;
  uint32_t *work = class_counts + kItemClasses;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 1;
  const int shape = p.tile == 32 ? kTile32 : (n_ranges <= kSplitTilesPerSm * sms ? kTile16Split : kTile16);
  const int parts = shape == kTile16 ? 1 : 2;
  cudaError_t e = cudaMemsetAsync(class_counts, 0, sizeof(uint32_t) * (kItemClasses + 1), s);
  if (e != cudaSuccess) return e;
  e = launch_pdl(plan_kernel, (n_ranges + 255) / 256, 256, 0, s, p_dev, gaze, round, p.full ? 4 : uniform, parts, cur,
                 levels, items, class_counts, ranges, thresholds);
  if (e != cudaSuccess) return e;
  auto go = [&](auto kern, int variant) -> cudaError_t {
    prefer_smem(kern, variant);
    static int per_sm[64][16] = {};
    int occ = (dev >= 0 && dev < 64) ? per_sm[dev][variant] : 0;
    if (occ == 0) {
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kHalfThreads, 0) != cudaSuccess || occ < 1)
        occ = 1;
      if (dev >= 0 && dev < 64) per_sm[dev][variant] = occ;
    }
    const int grid = (int)std::min<long>((long)sms * occ, (long)parts * n_ranges);
    return launch_pdl(kern, grid, kHalfThreads, 0, s, p_dev, rec, n, ranges, kept, vals, items, class_counts, work,
                      inc, t_final, n_contrib, depth, counters);
  };
  if (kernels) *kernels += 2;
  switch (shape) {
    case kTile32:
      return aux ? (mult == 2 ? go(composite_px_kernel<true, 2, kTile32>, 0) : go(composite_px_kernel<true, 1, kTile32>, 1))
                 : (mult == 2 ? go(composite_px_kernel<false, 2, kTile32>, 2) : go(composite_px_kernel<false, 1, kTile32>, 3));
    case kTile16:
      return aux ? (mult == 2 ? go(composite_px_kernel<true, 2, kTile16>, 4) : go(composite_px_kernel<true, 1, kTile16>, 5))
                 : (mult == 2 ? go(composite_px_kernel<false, 2, kTile16>, 6) : go(composite_px_kernel<false, 1, kTile16>, 7));
    default:
      return aux ? (mult == 2 ? go(composite_px_kernel<true, 2, kTile16Split>, 8) : go(composite_px_kernel<true, 1, kTile16Split>, 9))
                 : (mult == 2 ? go(composite_px_kernel<false, 2, kTile16Split>, 10) : go(composite_px_kernel<false, 1, kTile16Split>, 11));
  }
}

}  // namespace a3fr
