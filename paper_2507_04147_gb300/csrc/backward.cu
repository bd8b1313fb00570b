// backward.cu -- gradients of the 3DGS forward pass (Sec. 2.3: projection, rasterization)
// with respect to the scene parameters, for a loss whose gradient with respect to the
// rendered image is given (L = sum(dl_drgb * image)).
//
// composite_backward: one CTA per 16 x 16 quadrant of an (eye, tile), or per half of one.  A pixel
// walks its tile's Gaussians back to front from its last contributor (n_contrib), recovering the
// transmittance before each contributor from the stored final one (T_before = T_after /
// (1 - alpha)) instead of storing it per Gaussian.  The colour accumulated behind a
// contributor enters the alpha gradient only through its dot product with dL/dC, so one
// scalar D carries it:  dL/dalpha_i = T_i (c_i . g - D_i),  D_{i-1} = alpha_i c_i . g +
// (1 - alpha_i) D_i.  Alpha is recomputed exactly as the forward computed it (shared
// helpers, explicitly rounded), so every skip / accept decision is the forward's.  Nine sums over
// the pixels -- w g (three), dL/dopacity, and with p = dL/dpower and the falloff's A, B, C those of
// p (2 A dx + B dy), p (2 C dy + B dx), p dx^2, p dx dy, p dy^2 -- go to a per-(eye, Gaussian) buffer.  A foveated render's inherited pixels pass their gradient to the top-left
// pixel of their block.
//
// preprocess_backward: one thread per Gaussian, summing the eyes: conic -> 2-D covariance
// -> (3-D covariance, Jacobian) -> camera-space position -> mean; 3-D covariance ->
// scales (through exp) and rotation -> quaternion (through the normalisation); opacity
// through the sigmoid; colour -> SH coefficients and, through the view direction, mean.
#include <type_traits>

#include "blend.cuh"
#include "common.cuh"
#include "stage.cuh"

namespace a3fr {
namespace {

constexpr int kTile = 16;
constexpr int kThreads = 128;            // four warps
constexpr int kBatch = 128;              // Gaussians staged per batch
constexpr int kG2 = 9;                   // sums per (eye, Gaussian): eight side by side, the ninth apart
constexpr int kPreBwdThreads = 128;
constexpr int kPreBwdCtas = 6;           // CTAs per SM
// Quadrants are split in halves up to this many per SM, as the forward's 16-pixel tiles are: split /
// not, 825 quadrants 102 / 145 us, 4,096 quadrants 160 / 146 us (ncu, before the first-order sums
// were formed per pixel).
constexpr int kSplitQuadsPerSm = 16;
constexpr float kTame = 1e15f;           // a few products of two such values are far from overflow

// Where the sums of (eye, Gaussian) entry q of n_entries lie: [n_entries][8] -- the five of p,
// dopacity, dr, dg (one 32-byte sector) -- then [n_entries] db.
__device__ __forceinline__ float *sums8(float *g2d, size_t q) { return g2d + 8 * q; }
__device__ __forceinline__ float *sum9(float *g2d, size_t q, size_t n_entries) { return g2d + 8 * n_entries + q; }

// Each warp owns a patch of 8 x 8 pixels (Q = 2: lanes are 4 x 4 blocks of 2 x 2 pixels times two
// label pairs) or of 8 x 4 (Q = 1: 4 x 2 blocks times four labels); per batch it lists the
// Gaussians that can reach alpha = 1/255 in its patch (falloff_reaches: the others contribute to no
// pixel of it) and walks only those, two at a time, so that the warp sums of one overlap the
// other's.  A pixel that a listed Gaussian does not touch takes alpha 0 through the same products,
// which is exact while they are finite; a CTA with an image gradient or a colour that is not below kTame
// skips such pixels instead, so that a NaN or an infinity reaches only the Gaussians blended at its
// pixels.  The sums of a batch meet in shared memory, one row per warp and Gaussian, and
// leave as one reduction per value, Gaussian and quadrant.
// Bound by issue, and by the longest list's chain on small images.  1M Gaussians at 1024 x 1024 (ncu):
// 281 us with every warp (16 x 2 pixels) walking the whole list and adding its own nine sums to
// memory, 152 us now; 50k at 517 x 389: 247, 106 us.
template <int Q>
__global__ void __launch_bounds__(kThreads, 6)
composite_backward_kernel(BackwardParams p, const float *__restrict__ rec, const uint2 *__restrict__ ranges,
                          const uint32_t *__restrict__ kept, const uint32_t *__restrict__ vals,
                          const uint8_t *__restrict__ levels, const float *__restrict__ t_final,
                          const uint32_t *__restrict__ n_contrib, const float *__restrict__ dl_drgb,
                          float *__restrict__ g2d) {
  constexpr int BH = Q == 2 ? 4 : 2;   // blocks down a patch
  constexpr int W = kThreads / 32;
  // slot kBatch: a Gaussian of opacity 0, which pads odd hit lists
  __shared__ float4 s_geo[kBatch + 1];   // u, v, A, B (base-2 falloff coefficients)
  __shared__ float4 s_crg[kBatch + 1];   // C, opacity, r, g
  __shared__ float s_b[kBatch + 1];
  __shared__ uint32_t s_gid[kBatch];
  __shared__ short4 s_box[kBatch];
  __shared__ float s_thr[kBatch];
  __shared__ uint8_t s_hits[W][kBatch + 4];
  __shared__ uint32_t s_mask[W][kBatch / 32];   // slots with sums of this warp
  __shared__ float s_sum[W][kBatch + 1][kG2];
  __shared__ uint32_t s_max[W];
  __shared__ __align__(16) uint32_t s_wild[4];   // 1: a pixel of the warp, or a record it has staged, is not below kTame
  static_assert(W == 4, "s_wild is read as one vector");

  const int qn = p.tile / kTile, parts = Q == 2 ? 1 : 2;
  const int gtile = blockIdx.x / (qn * qn * parts);
  const int rest = blockIdx.x - gtile * qn * qn * parts, quad = rest / parts, half = rest - quad * parts;
  const int eye = gtile / p.n_tiles;
  const int tile = gtile - eye * p.n_tiles;
  const int tx = tile % p.tiles_x, ty = tile / p.tiles_x;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int wx = tx * p.tile + (quad % qn) * kTile + 8 * (warp & 1);
  const int wy = ty * p.tile + (quad / qn) * kTile + (Q == 2 ? 0 : 8 * half) + 2 * BH * (warp >> 1);
  const int blk = lane % (4 * BH), slot0 = lane / (4 * BH) * Q;
  const int px0 = wx + 2 * (blk & 3), py0 = wy + 2 * (blk >> 2);
  const int level = levels ? levels[gtile] : 4;
  uint2 range = ranges[gtile];
  const uint32_t n_kept = *kept;
  range.x = min(range.x, n_kept);
  range.y = min(range.y, n_kept);

  float T[Q], D[Q], g[Q][3], fpx[Q], fpy[Q];   // D: colour accumulated behind, normalised by T, . dL/dC
  uint32_t last[Q];
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    // labels of the 2x2 block: top-left 0, bottom-right 1, top-right 2, bottom-left 3
    const int L = slot0 + k;
    const int px = px0 + ((L == 1 || L == 2) ? 1 : 0), py = py0 + ((L == 1 || L == 3) ? 1 : 0);
    fpx[k] = (float)px;
    fpy[k] = (float)py;
    T[k] = 1.0f;
    D[k] = g[k][0] = g[k][1] = g[k][2] = 0.0f;
    last[k] = 0u;
    if (L < level && px < p.width && py < p.height) {
      const size_t pix = ((size_t)eye * p.height + py) * p.width + px;
      T[k] = t_final[pix];
      last[k] = min(n_contrib[pix], range.y - range.x);
#pragma unroll
      for (int c = 0; c < 3; ++c) g[k][c] = dl_drgb[3 * pix + c];
      if (L == 0 && level < 4) {
        // inherited pixels of the block copy this one: BR (label 2), TR (label 3), BL (label 4)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const int dx = j < 2 ? 1 : 0, dy = j == 1 ? 0 : 1;
          if (level < j + 2 && px + dx < p.width && py + dy < p.height) {
            const size_t q = pix + (size_t)dy * p.width + dx;
#pragma unroll
            for (int c = 0; c < 3; ++c) g[k][c] += dl_drgb[3 * q + c];
          }
        }
      }
    }
  }
  bool wild_px = false;
#pragma unroll
  for (int k = 0; k < Q; ++k)
    wild_px = wild_px || !(fabsf(g[k][0]) + fabsf(g[k][1]) + fabsf(g[k][2]) <= kTame);
  wild_px = __any_sync(0xffffffffu, wild_px);
  // the deepest last contributor bounds the walk: the warp's for its lists, the CTA's for the batches
  uint32_t wlast = last[0];
  if (Q == 2) wlast = max(wlast, last[Q - 1]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) wlast = max(wlast, __shfl_xor_sync(0xffffffffu, wlast, o));
  if (lane == 0) {
    s_max[warp] = wlast;
    s_wild[warp] = wild_px ? 1u : 0u;
  }
  if (t == 0) {
    s_geo[kBatch] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    s_crg[kBatch] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    s_b[kBatch] = 0.0f;
  }
  __syncthreads();
  uint32_t max_last = 0;
#pragma unroll
  for (int w = 0; w < W; ++w) max_last = max(max_last, s_max[w]);

  const float wx0 = (float)wx, wx1 = (float)(wx + 7), wy0 = (float)wy, wy1 = (float)(wy + 2 * BH - 1);
  const float *rec_eye = rec + (size_t)eye * p.n * kRec;
  const size_t n_entries = (size_t)p.n_eyes * p.n, q0 = (size_t)eye * p.n;

  // the nine sums of the Gaussian in slot e over this lane's pixels, and the pixels' state behind it
  auto evaluate = [&](int e, int hi, float (&v)[kG2], auto guard) {
    const float4 geo = s_geo[e], crg = s_crg[e];
    const float cb = s_b[e];
    const uint32_t pos = (uint32_t)(hi - e);
#pragma unroll
    for (int j = 0; j < kG2; ++j) v[j] = 0.0f;
    if constexpr (decltype(guard)::value) {
#pragma unroll
      for (int k = 0; k < Q; ++k) {
        const float dx = __fsub_rn(geo.x, fpx[k]), dy = __fsub_rn(geo.y, fpy[k]);
        const float pw = falloff_log2(geo.z, geo.w, crg.x, dx, dy);
        const float G = ex2_approx(pw), araw = __fmul_rn(crg.y, G), a = fminf(0.99f, araw);
        if (!(pos <= last[k] && pw <= 0.0f && a >= 1.0f / 255.0f)) continue;
        const float om = __fsub_rn(1.0f, a);
        T[k] = T[k] / om;
        const float w = a * T[k], cdot = crg.z * g[k][0] + crg.w * g[k][1] + cb * g[k][2];
        const float dal = T[k] * (cdot - D[k]);
        D[k] = a * cdot + om * D[k];
#pragma unroll
        for (int c = 0; c < 3; ++c) v[6 + c] += w * g[k][c];
        if (!(araw <= 0.99f)) continue;   // the clamp passes no gradient
        const float dpow = dal * araw;
        v[0] += dpow * (2.0f * geo.z * dx + geo.w * dy);
        v[1] += dpow * (2.0f * crg.x * dy + geo.w * dx);
        v[2] += dpow * dx * dx;
        v[3] += dpow * dx * dy;
        v[4] += dpow * dy * dy;
        v[5] += dal * G;
      }
    } else if constexpr (Q == 2) {
      // both pixels per instruction where the arithmetic is the same
      const f32x2 dx = f2_add(f2_pack(geo.x, geo.x), f2_pack(-fpx[0], -fpx[Q - 1]));
      const f32x2 dy = f2_add(f2_pack(geo.y, geo.y), f2_pack(-fpy[0], -fpy[Q - 1]));
      const f32x2 pw = f2_fma(f2_fma(f2_pack(geo.z, geo.z), dx, f2_mul(f2_pack(geo.w, geo.w), dy)), dx,
                              f2_mul(f2_mul(f2_pack(crg.x, crg.x), dy), dy));
      float pw0, pw1, ar0, ar1;
      f2_unpack(pw, pw0, pw1);
      const float G0 = ex2_approx(pw0), G1 = ex2_approx(pw1);
      f2_unpack(f2_mul(f2_pack(crg.y, crg.y), f2_pack(G0, G1)), ar0, ar1);
      const float al0 = fminf(0.99f, ar0), al1 = fminf(0.99f, ar1);
      const bool ok0 = pos <= last[0] && pw0 <= 0.0f && al0 >= 1.0f / 255.0f;
      const bool ok1 = pos <= last[Q - 1] && pw1 <= 0.0f && al1 >= 1.0f / 255.0f;
      // a pixel this Gaussian does not touch takes alpha 0: T and D keep their bits
      const float a0 = ok0 ? al0 : 0.0f, a1 = ok1 ? al1 : 0.0f;
      const bool free0 = ok0 && ar0 <= 0.99f, free1 = ok1 && ar1 <= 0.99f;   // the clamp passes no gradient
      const f32x2 a2 = f2_pack(a0, a1), om = f2_pack(__fsub_rn(1.0f, a0), __fsub_rn(1.0f, a1));
      T[0] = T[0] / __fsub_rn(1.0f, a0);   // transmittance in front of this Gaussian
      T[Q - 1] = T[Q - 1] / __fsub_rn(1.0f, a1);
      const f32x2 T2 = f2_pack(T[0], T[Q - 1]), D2 = f2_pack(D[0], D[Q - 1]);
      const f32x2 g0 = f2_pack(g[0][0], g[Q - 1][0]), g1 = f2_pack(g[0][1], g[Q - 1][1]),
                  g2 = f2_pack(g[0][2], g[Q - 1][2]);
      const f32x2 w2 = f2_mul(a2, T2);
      const f32x2 cdot = f2_fma(f2_pack(crg.z, crg.z), g0,
                                f2_fma(f2_pack(crg.w, crg.w), g1, f2_mul(f2_pack(cb, cb), g2)));
      const f32x2 dal = f2_mul(T2, f2_fma(D2, f2_pack(-1.0f, -1.0f), cdot));
      f2_unpack(f2_fma(a2, cdot, f2_mul(om, D2)), D[0], D[Q - 1]);
      const f32x2 dpow = f2_mul(dal, f2_pack(free0 ? ar0 : 0.0f, free1 ? ar1 : 0.0f));
      const f32x2 px2 = f2_mul(dpow, dx), py2 = f2_mul(dpow, dy);
      // 2 A dx + B dy and 2 C dy + B dx per pixel, before the sum: in an elongated Gaussian the
      // two terms nearly cancel
      const f32x2 bx = f2_pack(geo.w, geo.w);
      const float A2 = geo.z + geo.z, C2 = crg.x + crg.x;
      v[0] = f2_sum(f2_mul(dpow, f2_fma(f2_pack(A2, A2), dx, f2_mul(bx, dy))));
      v[1] = f2_sum(f2_mul(dpow, f2_fma(f2_pack(C2, C2), dy, f2_mul(bx, dx))));
      v[2] = f2_sum(f2_mul(px2, dx));
      v[3] = f2_sum(f2_mul(px2, dy));
      v[4] = f2_sum(f2_mul(py2, dy));
      v[5] = f2_sum(f2_mul(dal, f2_pack(free0 ? G0 : 0.0f, free1 ? G1 : 0.0f)));
      v[6] = f2_sum(f2_mul(w2, g0));
      v[7] = f2_sum(f2_mul(w2, g1));
      v[8] = f2_sum(f2_mul(w2, g2));
    } else {
      const float dx = __fsub_rn(geo.x, fpx[0]), dy = __fsub_rn(geo.y, fpy[0]);
      const float pw = falloff_log2(geo.z, geo.w, crg.x, dx, dy);
      const float G = ex2_approx(pw);
      const float araw = __fmul_rn(crg.y, G);
      const float al = fminf(0.99f, araw);
      const bool ok = pos <= last[0] && pw <= 0.0f && al >= 1.0f / 255.0f;
      const float a = ok ? al : 0.0f;
      const bool open = ok && araw <= 0.99f;   // the clamp passes no gradient
      const float om = __fsub_rn(1.0f, a);
      T[0] = T[0] / om;   // transmittance in front of this Gaussian
      const float w = a * T[0];
      const float cdot = crg.z * g[0][0] + crg.w * g[0][1] + cb * g[0][2];
      const float dal = T[0] * (cdot - D[0]);
      D[0] = a * cdot + om * D[0];
      const float dpow = dal * (open ? araw : 0.0f);
      v[0] = dpow * (2.0f * geo.z * dx + geo.w * dy);
      v[1] = dpow * (2.0f * crg.x * dy + geo.w * dx);
      v[2] = dpow * dx * dx;
      v[3] = dpow * dx * dy;
      v[4] = dpow * dy * dy;
      v[5] = dal * (open ? G : 0.0f);
      v[6] = w * g[0][0];
      v[7] = w * g[0][1];
      v[8] = w * g[0][2];
    }
  };

  for (int hi = (int)max_last; hi >= 1; hi -= kBatch) {
    const int cnt = min(hi, kBatch);   // slot k: 1-based position hi - k of the tile's list
    __syncthreads();                   // the previous batch's sums have left
    if (t < cnt) {
      const uint32_t gidx = min(vals[range.x + (uint32_t)(hi - t) - 1u], (uint32_t)(p.n - 1));
      const float4 *r4 = reinterpret_cast<const float4 *>(rec_eye + (size_t)gidx * kRec);
      const float4 a = __ldg(r4), b = __ldg(r4 + 1);
      s_geo[t] = make_float4(a.x, a.y, __fmul_rn(-0.5f * kLog2e, a.z), __fmul_rn(-kLog2e, a.w));
      s_crg[t] = make_float4(__fmul_rn(-0.5f * kLog2e, b.x), b.y, b.z, b.w);
      const float blue = __ldg(rec_eye + (size_t)gidx * kRec + 8);
      s_b[t] = blue;
      if (!(b.z + b.w + blue <= kTame)) s_wild[warp] = 1u;   // stays: D keeps what it has met
      s_gid[t] = gidx;
      s_box[t] = int_box(support_box(a.x, a.y, a.z, a.w, b.x, b.y));
      s_thr[t] = -__log2f(255.0f * b.y) - 0.01f;
    }
    __syncthreads();
    const uint4 wild4 = *reinterpret_cast<const uint4 *>(s_wild);
    const bool wild = (wild4.x | wild4.y | wild4.z | wild4.w) != 0u;
    int n_hit = 0;
    for (int base = 0; base < kBatch; base += 32) {
      const int k = base + lane;
      bool hit = k < cnt && hi - k <= (int)wlast;
      if (hit) {
        const short4 box = s_box[k];
        hit = !((float)box.y < wx0 || (float)box.x > wx1 || (float)box.w < wy0 || (float)box.z > wy1);
        if (hit) {
          const float4 geo = s_geo[k];
          hit = falloff_reaches(geo.z, geo.w, s_crg[k].x, s_thr[k], wx0 - geo.x, wx1 - geo.x, wy0 - geo.y,
                                wy1 - geo.y);
        }
      }
      const unsigned m = __ballot_sync(0xffffffffu, hit);
      if (hit) s_hits[warp][n_hit + __popc(m & ((1u << lane) - 1u))] = (uint8_t)k;
      if (lane == 0) s_mask[warp][base / 32] = m;
      n_hit += __popc(m);
    }
    if (lane == 0) s_hits[warp][n_hit] = (uint8_t)kBatch;
    __syncwarp();
    auto walk = [&](auto guard) {
      for (int i = 0; i < n_hit; i += 2) {
        float v[2][kG2];
#pragma unroll
        for (int u = 0; u < 2; ++u) evaluate(s_hits[warp][i + u], hi, v[u], guard);
        // warp sums by recursive halving: at each of the first four steps a lane keeps half of its
        // values and sends its partner the other half, so the sixteen cost 8 + 4 + 2 + 1 + 1 shuffles;
        // lane bit 4 ends as the Gaussian, bits 3..1 as the value; the ninth values 1 + 4
        float h[8];
        const bool b4 = (lane & 16) != 0, b3 = (lane & 8) != 0, b2 = (lane & 4) != 0, b1 = (lane & 2) != 0;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          h[j] = (b4 ? v[1][j] : v[0][j]) + __shfl_xor_sync(0xffffffffu, b4 ? v[0][j] : v[1][j], 16);
        float h9 = (b4 ? v[1][8] : v[0][8]) + __shfl_xor_sync(0xffffffffu, b4 ? v[0][8] : v[1][8], 16);
#pragma unroll
        for (int j = 0; j < 4; ++j)
          h[j] = (b3 ? h[j + 4] : h[j]) + __shfl_xor_sync(0xffffffffu, b3 ? h[j] : h[j + 4], 8);
#pragma unroll
        for (int j = 0; j < 2; ++j)
          h[j] = (b2 ? h[j + 2] : h[j]) + __shfl_xor_sync(0xffffffffu, b2 ? h[j] : h[j + 2], 4);
        h[0] = (b1 ? h[1] : h[0]) + __shfl_xor_sync(0xffffffffu, b1 ? h[0] : h[1], 2);
        h[0] += __shfl_xor_sync(0xffffffffu, h[0], 1);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) h9 += __shfl_xor_sync(0xffffffffu, h9, o);
        float *row = s_sum[warp][s_hits[warp][i + (b4 ? 1 : 0)]];
        if (!(lane & 1)) row[(lane >> 1) & 7] = h[0];
        else if ((lane & 15) == 1) row[8] = h9;
      }
    };
    if (!wild) walk(std::false_type{});
    else walk(std::true_type{});
    __syncthreads();
    // the batch's sums over the warps, eight values of a Gaussian to a sector
    for (int e = t; e < cnt * 8; e += kThreads) {
      const int k = e >> 3, j = e & 7;
      float sum = 0.0f;
      bool any = false;
#pragma unroll
      for (int w = 0; w < W; ++w)
        if ((s_mask[w][k >> 5] >> (k & 31)) & 1u) {
          sum += s_sum[w][k][j];
          any = true;
        }
      if (any) atomicAdd(sums8(g2d, q0 + s_gid[k]) + j, sum);
    }
    if (t < cnt) {
      float sum = 0.0f;
      bool any = false;
#pragma unroll
      for (int w = 0; w < W; ++w)
        if ((s_mask[w][t >> 5] >> (t & 31)) & 1u) {
          sum += s_sum[w][t][8];
          any = true;
        }
      if (any) atomicAdd(sum9(g2d, q0 + s_gid[t], n_entries), sum);
    }
  }
}

// Real SH basis (3DGS order and signs) at the unit direction (x, y, z) and its gradient
// contracted with per-coefficient weights wk: returns sum_k wk * dY_k/d(x, y, z).
template <int K>
__device__ __forceinline__ void sh_basis_eval(const ShConsts &c, float x, float y, float z, float *Y) {
  Y[0] = c.c0;
  if constexpr (K > 1) {
    Y[1] = -c.c1 * y;
    Y[2] = c.c1 * z;
    Y[3] = -c.c1 * x;
  }
  if constexpr (K > 4) {
    const float xx = x * x, yy = y * y, zz = z * z;
    Y[4] = c.c2a * x * y;
    Y[5] = -c.c2a * y * z;
    Y[6] = c.c2b * (2.0f * zz - xx - yy);
    Y[7] = -c.c2a * x * z;
    Y[8] = c.c2c * (xx - yy);
    if constexpr (K > 9) {
      Y[9] = -c.c3a * y * (3.0f * xx - yy);
      Y[10] = c.c3b * x * y * z;
      Y[11] = -c.c3c * y * (4.0f * zz - xx - yy);
      Y[12] = c.c3d * z * (2.0f * zz - 3.0f * xx - 3.0f * yy);
      Y[13] = -c.c3c * x * (4.0f * zz - xx - yy);
      Y[14] = c.c3e * z * (xx - yy);
      Y[15] = -c.c3a * x * (xx - 3.0f * yy);
    }
  }
}

template <int K>
__device__ __forceinline__ void sh_basis_vjp(const ShConsts &c, float x, float y, float z,
                                             const float *wk, float &gx, float &gy, float &gz) {
  gx = gy = gz = 0.0f;
  if constexpr (K > 1) {
    gy += -c.c1 * wk[1];
    gz += c.c1 * wk[2];
    gx += -c.c1 * wk[3];
  }
  if constexpr (K > 4) {
    // Y4 = c2a x y, Y5 = -c2a y z, Y6 = c2b (2zz - xx - yy), Y7 = -c2a x z, Y8 = c2c (xx - yy)
    gx += c.c2a * y * wk[4];
    gy += c.c2a * x * wk[4];
    gy += -c.c2a * z * wk[5];
    gz += -c.c2a * y * wk[5];
    gx += -2.0f * c.c2b * x * wk[6];
    gy += -2.0f * c.c2b * y * wk[6];
    gz += 4.0f * c.c2b * z * wk[6];
    gx += -c.c2a * z * wk[7];
    gz += -c.c2a * x * wk[7];
    gx += 2.0f * c.c2c * x * wk[8];
    gy += -2.0f * c.c2c * y * wk[8];
    if constexpr (K > 9) {
      const float xx = x * x, yy = y * y, zz = z * z;
      // Y9 = -c3a y (3xx - yy)
      gx += -6.0f * c.c3a * x * y * wk[9];
      gy += -3.0f * c.c3a * (xx - yy) * wk[9];
      // Y10 = c3b x y z
      gx += c.c3b * y * z * wk[10];
      gy += c.c3b * x * z * wk[10];
      gz += c.c3b * x * y * wk[10];
      // Y11 = -c3c y (4zz - xx - yy)
      gx += 2.0f * c.c3c * x * y * wk[11];
      gy += -c.c3c * (4.0f * zz - xx - 3.0f * yy) * wk[11];
      gz += -8.0f * c.c3c * y * z * wk[11];
      // Y12 = c3d z (2zz - 3xx - 3yy)
      gx += -6.0f * c.c3d * x * z * wk[12];
      gy += -6.0f * c.c3d * y * z * wk[12];
      gz += c.c3d * (6.0f * zz - 3.0f * xx - 3.0f * yy) * wk[12];
      // Y13 = -c3c x (4zz - xx - yy)
      gx += -c.c3c * (4.0f * zz - 3.0f * xx - yy) * wk[13];
      gy += 2.0f * c.c3c * x * y * wk[13];
      gz += -8.0f * c.c3c * x * z * wk[13];
      // Y14 = c3e z (xx - yy)
      gx += 2.0f * c.c3e * x * z * wk[14];
      gy += -2.0f * c.c3e * y * z * wk[14];
      gz += c.c3e * (xx - yy) * wk[14];
      // Y15 = -c3a x (xx - 3yy)
      gx += -3.0f * c.c3a * (xx - yy) * wk[15];
      gy += 6.0f * c.c3a * x * y * wk[15];
    }
  }
}

// Calls f(index, element) for the 3K elements of thread t's SH row in shared memory (the layouts of
// stage.cuh), four to a 16-byte access where rows are whole chunks; kStore writes them back.
template <int K, bool kStore, typename F>
__device__ __forceinline__ void each_sh(float *rows, int t, F f) {
  if constexpr (sh_chunked<K>()) {
    float4 *row4 = reinterpret_cast<float4 *>(rows + t * 3 * K);
#pragma unroll
    for (int m = 0; m < 3 * K / 4; ++m) {
      const float4 v = row4[sh_swz<K>(m, t)];
      float e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) f(4 * m + j, e[j]);
      if (kStore) row4[sh_swz<K>(m, t)] = make_float4(e[0], e[1], e[2], e[3]);
    }
  } else {
    float *row = rows + t * sh_stride<K>();
#pragma unroll
    for (int j = 0; j < 3 * K; ++j) f(j, row[j]);
  }
}

// One thread per Gaussian.  The block's SH rows are copied into shared memory asynchronously while
// the threads load the rest; a row is read for every eye, then overwritten by its gradient (the
// eyes' directions and colour gradients are kept, their bases evaluated again), and the rows are
// written back coalesced.
// Bound by memory: 1M Gaussians, SH degree 3 (556 MB) 125 us under ncu; 196 us with the rows and
// their gradients in separate arrays copied by plain loads (50 KB and 127 registers: 16 warps per SM,
// waiting on memory).
template <int K>
__global__ void __launch_bounds__(kPreBwdThreads, kPreBwdCtas)
preprocess_backward_kernel(const PreParams *__restrict__ pp, int n, const float *__restrict__ means,
                           const float *__restrict__ log_scales, const float *__restrict__ quats,
                           const float *__restrict__ opacity_logits, const float *__restrict__ sh,
                           const float *__restrict__ rec, const float *__restrict__ g2d,
                           float *__restrict__ d_means, float *__restrict__ d_log_scales,
                           float *__restrict__ d_quats, float *__restrict__ d_logits,
                           float *__restrict__ d_sh) {
  constexpr int ROW = 3 * K;
  __shared__ PreParams s_p;
  __shared__ __align__(16) float s_sh[kPreBwdThreads * sh_stride<K>()];
  static_assert(sizeof(PreParams) % 4 == 0 && sizeof(PreParams) / 4 <= kPreBwdThreads, "PreParams copy");
  const int i0 = blockIdx.x * kPreBwdThreads;
  const int rows = min(kPreBwdThreads, n - i0);
  const int t = threadIdx.x;
  if constexpr (sh_chunked<K>()) stage_sh_async<K>(s_sh, sh + (size_t)ROW * i0, rows);
  if (t < sizeof(PreParams) / 4)
    reinterpret_cast<uint32_t *>(&s_p)[t] = reinterpret_cast<const uint32_t *>(pp)[t];
  if constexpr (!sh_chunked<K>()) stage(s_sh, sh + (size_t)ROW * i0, rows * ROW, ROW, sh_stride<K>());
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  const PreParams &p = s_p;
  const int i = i0 + t;
  if (i < n) {

  const float mx = means[3 * i], my = means[3 * i + 1], mz = means[3 * i + 2];
  float s2[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const float s = expf(log_scales[3 * i + j]);
    s2[j] = s * s;
  }
  const float q0 = quats[4 * i], q1 = quats[4 * i + 1], q2 = quats[4 * i + 2], q3 = quats[4 * i + 3];
  const float qn = sqrtf(q0 * q0 + q1 * q1 + q2 * q2 + q3 * q3);
  const float qw = q0 / qn, qx = q1 / qn, qy = q2 / qn, qz = q3 / qn;
  float R[3][3];
  R[0][0] = 1.0f - 2.0f * (qy * qy + qz * qz);
  R[0][1] = 2.0f * (qx * qy - qw * qz);
  R[0][2] = 2.0f * (qx * qz + qw * qy);
  R[1][0] = 2.0f * (qx * qy + qw * qz);
  R[1][1] = 1.0f - 2.0f * (qx * qx + qz * qz);
  R[1][2] = 2.0f * (qy * qz - qw * qx);
  R[2][0] = 2.0f * (qx * qz - qw * qy);
  R[2][1] = 2.0f * (qy * qz + qw * qx);
  R[2][2] = 1.0f - 2.0f * (qx * qx + qy * qy);
  float S[3][3];
#pragma unroll
  for (int j = 0; j < 3; ++j)
#pragma unroll
    for (int k = 0; k < 3; ++k)
      S[j][k] = R[j][0] * s2[0] * R[k][0] + R[j][1] * s2[1] * R[k][1] + R[j][2] * s2[2] * R[k][2];
  const float opacity = 1.0f / (1.0f + expf(-opacity_logits[i]));

  float dmu[3] = {0.f, 0.f, 0.f};
  float dS[3][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
  float dlogit = 0.0f;
  float dir[kMaxEyes][3], gcol[kMaxEyes][3];   // per eye: direction, gradient of the colour

#pragma unroll
  for (int e = 0; e < kMaxEyes; ++e) {
#pragma unroll
    for (int k = 0; k < 3; ++k) dir[e][k] = gcol[e][k] = 0.0f;
    if (e >= p.n_eyes) continue;
    const size_t q = (size_t)e * n + i;
    if (__ldg(rec + q * kRec + 11) == 0.0f) continue;   // culled for this eye
    const float4 s0 = __ldg(reinterpret_cast<const float4 *>(g2d + 8 * q));
    const float4 s1 = __ldg(reinterpret_cast<const float4 *>(g2d + 8 * q) + 1);
    // power = -0.5 (a dx^2 + c dy^2) - b dx dy with dx = u - x, dy = v - y; in base 2, as
    // composite_backward sums it, A = -0.5 log2(e) a, B = -log2(e) b, C = -0.5 log2(e) c
    const float gu = s0.x * (1.0f / kLog2e), gv = s0.y * (1.0f / kLog2e);
    const float gca = -0.5f * s0.z, gcb = -s0.w, gcc = -0.5f * s1.x, gop = s1.y;
    const float gr[3] = {s1.z, s1.w, __ldg(g2d + 8 * (size_t)p.n_eyes * n + q)};
    const CamParams &c = p.cam[e];
    const float *W = c.R;
    const float tx = W[0] * mx + W[1] * my + W[2] * mz + c.t[0];
    const float ty = W[3] * mx + W[4] * my + W[5] * mz + c.t[1];
    const float tz = W[6] * mx + W[7] * my + W[8] * mz + c.t[2];
    const float txz = tx / tz, tyz = ty / tz;
    const bool clx = txz < -c.limx || txz > c.limx;
    const bool cly = tyz < -c.limy || tyz > c.limy;
    const float xc = fminf(c.limx, fmaxf(-c.limx, txz)) * tz;
    const float yc = fminf(c.limy, fmaxf(-c.limy, tyz)) * tz;
    const float tz2 = tz * tz;
    const float J00 = c.fx / tz, J02 = -c.fx * xc / tz2;
    const float J11 = c.fy / tz, J12 = -c.fy * yc / tz2;
    float T[2][3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      T[0][j] = J00 * W[j] + J02 * W[6 + j];
      T[1][j] = J11 * W[3 + j] + J12 * W[6 + j];
    }
    float U[2][3];   // T Sigma
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int l = 0; l < 3; ++l) U[r][l] = T[r][0] * S[0][l] + T[r][1] * S[1][l] + T[r][2] * S[2][l];
    const float a = U[0][0] * T[0][0] + U[0][1] * T[0][1] + U[0][2] * T[0][2] + 0.3f;
    const float b = U[0][0] * T[1][0] + U[0][1] * T[1][1] + U[0][2] * T[1][2];
    const float cc = U[1][0] * T[1][0] + U[1][1] * T[1][1] + U[1][2] * T[1][2] + 0.3f;
    const float det = a * cc - b * b;
    const float id2 = 1.0f / (det * det);
    // conic (cc, -b, a) / det -> covariance entries
    const float ga = (-cc * cc * gca + b * cc * gcb - b * b * gcc) * id2;
    const float gb = (2.0f * b * cc * gca - (a * cc + b * b) * gcb + 2.0f * a * b * gcc) * id2;
    const float gc = (-b * b * gca + a * b * gcb - a * a * gcc) * id2;
    // cov = T Sigma T^T with G2 = [[ga, gb/2], [gb/2, gc]]: dSigma += T^T G2 T, dT = 2 G2 T Sigma
    const float G2[2][2] = {{ga, 0.5f * gb}, {0.5f * gb, gc}};
    float GT[2][3];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int j = 0; j < 3; ++j) GT[r][j] = G2[r][0] * T[0][j] + G2[r][1] * T[1][j];
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int k = 0; k < 3; ++k) dS[j][k] += T[0][j] * GT[0][k] + T[1][j] * GT[1][k];
    float dT[2][3];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int j = 0; j < 3; ++j)
        dT[r][j] = 2.0f * (G2[r][0] * U[0][j] + G2[r][1] * U[1][j]);
    // T = J W
    float dJ00 = 0.f, dJ02 = 0.f, dJ11 = 0.f, dJ12 = 0.f;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      dJ00 += dT[0][j] * W[j];
      dJ02 += dT[0][j] * W[6 + j];
      dJ11 += dT[1][j] * W[3 + j];
      dJ12 += dT[1][j] * W[6 + j];
    }
    float dtx = 0.f, dty = 0.f, dtz = 0.f;
    dtz += -c.fx / tz2 * dJ00 - c.fy / tz2 * dJ11;
    // J02 = -fx x' / tz^2 with x' = tx (inside the clamp) or +-limx tz (outside)
    if (!clx) {
      dtx += -c.fx / tz2 * dJ02;
      dtz += 2.0f * c.fx * tx / (tz2 * tz) * dJ02;
    } else {
      dtz += c.fx * (xc / tz) / tz2 * dJ02;
    }
    if (!cly) {
      dty += -c.fy / tz2 * dJ12;
      dtz += 2.0f * c.fy * ty / (tz2 * tz) * dJ12;
    } else {
      dtz += c.fy * (yc / tz) / tz2 * dJ12;
    }
    // u = fx tx / tz + cx, v = fy ty / tz + cy
    dtx += c.fx / tz * gu;
    dty += c.fy / tz * gv;
    dtz += -c.fx * tx / tz2 * gu - c.fy * ty / tz2 * gv;
    // t = W mu + t_c
#pragma unroll
    for (int j = 0; j < 3; ++j) dmu[j] += W[j] * dtx + W[3 + j] * dty + W[6 + j] * dtz;
    // opacity
    dlogit += gop * opacity * (1.0f - opacity);
    // colour: the unit direction from the eye centre -W^T t_c to the mean
    float C[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) C[j] = -(W[j] * c.t[0] + W[3 + j] * c.t[1] + W[6 + j] * c.t[2]);
    const float ddx = mx - C[0], ddy = my - C[1], ddz = mz - C[2];
    const float dn = sqrtf(ddx * ddx + ddy * ddy + ddz * ddz);
    const float x = ddx / dn, y = ddy / dn, z = ddz / dn;
    dir[e][0] = x;
    dir[e][1] = y;
    dir[e][2] = z;
    float acc[3] = {0.5f, 0.5f, 0.5f};
    {
      float Y[K];
      sh_basis_eval<K>(p.shc, x, y, z, Y);
      each_sh<K, false>(s_sh, t, [&](int f, float &c) { acc[f % 3] += Y[f / 3] * c; });
    }
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) gcol[e][ch] = acc[ch] > 0.0f ? gr[ch] : 0.0f;   // max(0, .): where positive
    float wk[K];
#pragma unroll
    for (int k = 0; k < K; ++k) wk[k] = 0.0f;
    each_sh<K, false>(s_sh, t, [&](int f, float &c) { wk[f / 3] += c * gcol[e][f % 3]; });
    float gx, gy, gz;
    sh_basis_vjp<K>(p.shc, x, y, z, wk, gx, gy, gz);
    const float dot = x * gx + y * gy + z * gz;
    dmu[0] += (gx - x * dot) / dn;
    dmu[1] += (gy - y * dot) / dn;
    dmu[2] += (gz - z * dot) / dn;
  }
  // Sigma = R diag(s2) R^T (dS symmetric): ds2_k = (R^T dS R)_kk, dR = 2 dS R diag(s2)
  float dR[3][3];
#pragma unroll
  for (int j = 0; j < 3; ++j)
#pragma unroll
    for (int k = 0; k < 3; ++k)
      dR[j][k] = 2.0f * (dS[j][0] * R[0][k] + dS[j][1] * R[1][k] + dS[j][2] * R[2][k]) * s2[k];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    float v = 0.0f;
#pragma unroll
    for (int j = 0; j < 3; ++j)
      v += R[j][k] * (dS[j][0] * R[0][k] + dS[j][1] * R[1][k] + dS[j][2] * R[2][k]);
    d_log_scales[3 * i + k] = 2.0f * s2[k] * v;   // s2 = exp(2 log s)
  }
  // R of the unit quaternion (w, x, y, z)
  const float dw = 2.0f * (-qz * dR[0][1] + qy * dR[0][2] + qz * dR[1][0] - qx * dR[1][2] -
                           qy * dR[2][0] + qx * dR[2][1]);
  const float dx = 2.0f * (qy * dR[0][1] + qz * dR[0][2] + qy * dR[1][0] - 2.0f * qx * dR[1][1] -
                           qw * dR[1][2] + qz * dR[2][0] + qw * dR[2][1] - 2.0f * qx * dR[2][2]);
  const float dy = 2.0f * (-2.0f * qy * dR[0][0] + qx * dR[0][1] + qw * dR[0][2] + qx * dR[1][0] +
                           qz * dR[1][2] - qw * dR[2][0] + qz * dR[2][1] - 2.0f * qy * dR[2][2]);
  const float dz = 2.0f * (-2.0f * qz * dR[0][0] - qw * dR[0][1] + qx * dR[0][2] + qw * dR[1][0] -
                           2.0f * qz * dR[1][1] + qy * dR[1][2] + qx * dR[2][0] + qy * dR[2][1]);
  // through q / |q|
  const float qd = qw * dw + qx * dx + qy * dy + qz * dz;
  d_quats[4 * i] = (dw - qw * qd) / qn;
  d_quats[4 * i + 1] = (dx - qx * qd) / qn;
  d_quats[4 * i + 2] = (dy - qy * qd) / qn;
  d_quats[4 * i + 3] = (dz - qz * qd) / qn;
  d_means[3 * i] = dmu[0];
  d_means[3 * i + 1] = dmu[1];
  d_means[3 * i + 2] = dmu[2];
  d_logits[i] = dlogit;
  // the SH gradient in place of the row
  {
    float Y[K];
    sh_basis_eval<K>(p.shc, dir[0][0], dir[0][1], dir[0][2], Y);
    each_sh<K, true>(s_sh, t, [&](int f, float &c) { c = Y[f / 3] * gcol[0][f % 3]; });
    if (p.n_eyes > 1) {
      sh_basis_eval<K>(p.shc, dir[1][0], dir[1][1], dir[1][2], Y);
      each_sh<K, true>(s_sh, t, [&](int f, float &c) { c += Y[f / 3] * gcol[1][f % 3]; });
    }
  }
  }
  __syncthreads();
  float *dst = d_sh + (size_t)ROW * i0;
  if constexpr (sh_chunked<K>()) {
    if ((reinterpret_cast<uintptr_t>(d_sh) & 15u) == 0u) {
      for (int c = t; c < rows * (ROW / 4); c += kPreBwdThreads) {
        const int r = c / (ROW / 4), m = c - r * (ROW / 4);
        reinterpret_cast<float4 *>(dst)[c] = reinterpret_cast<const float4 *>(s_sh + r * ROW)[sh_swz<K>(m, r)];
      }
      return;
    }
  }
  for (int f = t; f < rows * ROW; f += kPreBwdThreads) {
    const int r = f / ROW, c = f % ROW;
    if constexpr (sh_chunked<K>()) dst[f] = s_sh[r * ROW + 4 * sh_swz<K>(c >> 2, r) + (c & 3)];
    else dst[f] = s_sh[r * sh_stride<K>() + c];
  }
}

}  // namespace

size_t backward_g2d_floats(int n_eyes, int n) { return (size_t)n_eyes * n * kG2; }

cudaError_t launch_backward(const BackwardParams &bp, const PreParams *pre_dev, int sh_degree,
                            const float *means, const float *log_scales, const float *quats,
                            const float *opacity_logits, const float *sh, const float *rec,
                            const uint2 *ranges, const uint32_t *kept, const uint32_t *vals,
                            const uint8_t *levels, const float *t_final, const uint32_t *n_contrib,
                            const float *dl_drgb, float *g2d, float *d_means, float *d_log_scales,
                            float *d_quats, float *d_logits, float *d_sh, cudaStream_t s) {
  if (bp.n <= 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(g2d, 0, sizeof(float) * backward_g2d_floats(bp.n_eyes, bp.n), s);
  if (e != cudaSuccess) return e;
  const int quads = bp.n_eyes * bp.n_tiles * (bp.tile / kTile) * (bp.tile / kTile);
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (quads <= kSplitQuadsPerSm * sms)
    composite_backward_kernel<1><<<2 * quads, kThreads, 0, s>>>(bp, rec, ranges, kept, vals, levels, t_final,
                                                                n_contrib, dl_drgb, g2d);
  else
    composite_backward_kernel<2><<<quads, kThreads, 0, s>>>(bp, rec, ranges, kept, vals, levels, t_final, n_contrib,
                                                            dl_drgb, g2d);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int blocks = (bp.n + kPreBwdThreads - 1) / kPreBwdThreads;
  auto go = [&](auto kern) -> cudaError_t {
    kern<<<blocks, kPreBwdThreads, 0, s>>>(pre_dev, bp.n, means, log_scales, quats, opacity_logits, sh, rec, g2d,
                                           d_means, d_log_scales, d_quats, d_logits, d_sh);
    return cudaGetLastError();
  };
  switch (sh_degree) {
    case 0: return go(preprocess_backward_kernel<1>);
    case 1: return go(preprocess_backward_kernel<4>);
    case 2: return go(preprocess_backward_kernel<9>);
    default: return go(preprocess_backward_kernel<16>);
  }
}

}  // namespace a3fr
