// cnn.cu -- tensor-core (tcgen05) kernels of the learned periphery: small CNNs in BF16 with
// FP32 accumulation that reconstruct full-resolution RGB from the quarter-density peripheral
// layer (the level-1 pixels of Sec. 3.4) and its depth -- a residual network of ten 3x3
// convolutions, and a compact one (a 3x3 convolution and two per-block layers) whose whole
// fill is one fused kernel.
//
// This file starts with the single-tile GEMM that validates the operand encodings (shared-
// memory descriptors, instruction descriptor, tensor-memory round trip) before the
// convolution kernels use them.
#include "../../include/a3fr.h"
#include "common.cuh"
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <new>

#include "tc.cuh"

namespace a3fr {
namespace {

constexpr int kProbeSmem = 96 * 1024;
constexpr int kProbeB = 48 * 1024;   // offset of the B tile

// D[128][N] = A[128][K] B[N][K]^T for one tile.  variant 0: leading byte offset = distance
// of K-adjacent core matrices, stride byte offset = distance of M/N-adjacent ones; variant
// 1: the two swapped.  Either way every address the tensor core can form stays inside the
// zeroed 96 KB of shared memory.
__global__ void __launch_bounds__(128)
tc_tile_gemm_kernel(const uint16_t *__restrict__ A, const uint16_t *__restrict__ B,
                    float *__restrict__ D, int N, int K, int variant, uint32_t *__restrict__ status) {
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ uint32_t s_tmem;
  __shared__ __align__(8) uint64_t s_bar;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  for (int i = t; i < kProbeSmem / 16; i += 128) reinterpret_cast<uint4 *>(smem)[i] = make_uint4(0, 0, 0, 0);
  if (warp == 0) tc::tmem_alloc(&s_tmem, 256);
  __syncthreads();
  const uint32_t sbo = (uint32_t)(K / 8) * 128u;   // a row group holds K/8 core matrices
  for (int idx = t; idx < 128 * K; idx += 128) {
    const int m = idx / K, k = idx - m * K;
    const uint32_t off = (m >> 3) * sbo + (k >> 3) * 128u + (m & 7) * 16u + (k & 7) * 2u;
    *reinterpret_cast<uint16_t *>(smem + off) = A[idx];
  }
  for (int idx = t; idx < N * K; idx += 128) {
    const int nn = idx / K, k = idx - nn * K;
    const uint32_t off = (nn >> 3) * sbo + (k >> 3) * 128u + (nn & 7) * 16u + (k & 7) * 2u;
    *reinterpret_cast<uint16_t *>(smem + kProbeB + off) = B[idx];
  }
  tc::fence_proxy_async();
  if (t == 0) tc::mbar_init(&s_bar, 1);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = s_tmem;
  if (t == 0) {
    const uint32_t a0 = tc::smem_u32(smem), b0 = tc::smem_u32(smem + kProbeB);
    const uint32_t idesc = tc::idesc_bf16_f32(128, N);
    for (int kk = 0; kk < K / 16; ++kk) {
      const uint32_t lbo = variant == 0 ? 128u : sbo, s2 = variant == 0 ? sbo : 128u;
      const uint64_t ad = tc::smem_desc(a0 + kk * 256u, lbo, s2);
      const uint64_t bd = tc::smem_desc(b0 + kk * 256u, lbo, s2);
      tc::mma_bf16(tmem, ad, bd, idesc, kk > 0);
    }
    tc::mma_commit(&s_bar);
  }
  const bool ok = tc::mbar_wait(&s_bar, 0);
  if (!ok && lane == 0) atomicOr(status, kStatusTimeout);
  tc::fence_after_sync();
  float v[32];
  const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16);
  if (N == 32) tc::tmem_ld32(taddr, v);
  else tc::tmem_ld16(taddr, v);
  const int row = warp * 32 + lane;
  for (int nn = 0; nn < N; ++nn) D[row * N + nn] = v[nn];
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 256);
}


// ---------------------------------------------------------------- convolution kernels
// Activations are NHWC BF16 with 16 or 32 channels (32 or 64 bytes per pixel); a 3x3 "same"
// convolution is an implicit GEMM  D[pixel][cout] = sum over (tap, cin) of X[pixel + tap][cin]
// W[cout][cin][tap].  The A operand is never expanded: the tile's input halo sits in shared
// memory as [channel group of 8][row][column][8 channels], which is exactly the K-major core-
// matrix layout (8 pixels x 16 bytes) with the column direction inside a core matrix, so the
// operand of tap (ky, kx) is the same halo seen from a start address shifted by ky rows and kx
// columns.  Weights come pre-packed as [tap][cin group][cout][8 cin].

constexpr int kConvTW = 8;    // output tile width (pixels)
constexpr int kConvTH = 16;   // output tile height: 128 pixels = the MMA's M

struct ConvDims {
  int B, H, W;
};

enum : int { kEpiBias = 1, kEpiRelu = 2, kEpiResid = 4, kEpiMask = 8, kEpiF32 = 16, kBiasRelu = kEpiBias | kEpiRelu };

// The image side of the learned fill, for the two convolutions that touch it when the fill
// runs fused: the first reads its input straight from the render (kSrcImage), the last
// composes the skipped pixels in its epilogue (kDstCompose) -- the same values the separate
// gather and compose kernels produce, without their intermediate tensors.
struct FillIO {
  const float *depth;     // [B][H][W] expected depth of the render
  float *img;             // [B][H][W][3]: top-left pixels read, skipped pixels written
  const uint8_t *levels;  // tile levels [B][n_tiles]
  int H, W, tile, tiles_x, n_tiles;
};
enum : int { kSrcTensor = 0, kSrcImage = 1 };
enum : int { kDstTensor = 0, kDstCompose = 1 };

// The first eight of a block's 16 input channels: r, g, b of its top-left pixel and depth / 8 in
// BF16, then zeros (as are the other eight).
__device__ __forceinline__ uint4 block_operand(float4 v) {
  uint4 lo;
  __nv_bfloat162 *l2 = reinterpret_cast<__nv_bfloat162 *>(&lo);
  l2[0] = __floats2bfloat162_rn(v.x, v.y);
  l2[1] = __floats2bfloat162_rn(v.z, v.w * 0.125f);
  l2[2] = __floats2bfloat162_rn(0.0f, 0.0f);
  l2[3] = l2[2];
  return lo;
}
__device__ __forceinline__ uint4 block_input(const float *__restrict__ img, const float *__restrict__ depth,
                                             int b, int H, int W, int y2, int x2) {
  const size_t src = ((size_t)b * H + 2 * y2) * W + 2 * x2;
  return block_operand(make_float4(img[3 * src], img[3 * src + 1], img[3 * src + 2], depth[src]));
}

// Final image of a foveated render at block (y2, x2) from its 12 residuals res[c][2 dy + dx]:
// rendered pixels kept, the skipped sub-pixels -- top-right (label 3), bottom-left (4),
// bottom-right (2) -- set to the bilinear base of the blocks' top-left pixels (the last block
// repeated past the edge) plus the residual.  The base reads only top-left pixels, which every
// level renders and nobody writes.
__device__ __forceinline__ void compose_block(float *__restrict__ img, int b, int H, int W, int y2, int x2, int lv,
                                              const float (&res)[3][4]) {
  const int H2 = (H + 1) / 2, W2 = (W + 1) / 2;
  const int x = 2 * x2, y = 2 * y2;
  const int xr = min(x2 + 1, W2 - 1), yd = min(y2 + 1, H2 - 1);
  auto tl = [&](int yy, int xx, int c) { return img[3 * (((size_t)b * H + 2 * yy) * W + 2 * xx) + c]; };
  float a[3], right[3], down[3], diag[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    a[c] = tl(y2, x2, c);
    right[c] = tl(y2, xr, c);
    down[c] = lv <= 3 ? tl(yd, x2, c) : 0.0f;
    diag[c] = lv <= 1 ? tl(yd, xr, c) : 0.0f;
  }
  auto put = [&](int dy, int dx, const float *base) {
    if (y + dy >= H || x + dx >= W) return;
    float *o = img + 3 * (((size_t)b * H + y + dy) * W + x + dx);
#pragma unroll
    for (int c = 0; c < 3; ++c) o[c] = base[c] + res[c][2 * dy + dx];
  };
  float bt[3], bb[3], bd[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    bt[c] = __fmul_rn(__fadd_rn(a[c], right[c]), 0.5f);                                   // top-right
    bb[c] = __fmul_rn(__fadd_rn(a[c], down[c]), 0.5f);                                    // bottom-left
    bd[c] = __fmul_rn(__fadd_rn(__fadd_rn(__fadd_rn(a[c], right[c]), down[c]), diag[c]), 0.25f);   // bottom-right
  }
  if (lv <= 2) put(0, 1, bt);   // top-right: label 3, rendered from level 3
  if (lv <= 3) put(1, 0, bb);   // bottom-left: label 4, rendered at level 4
  if (lv <= 1) put(1, 1, bd);   // bottom-right: label 2, rendered from level 2
}

// Lane j of four has a[0..4): afterwards a[i] is what lane i had as a[j].
__device__ __forceinline__ void transpose4(uint4 (&a)[4]) {
  const bool b0 = threadIdx.x & 1, b1 = threadIdx.x & 2;
  auto swap = [](uint4 &p, uint4 &q, bool up, int mask) {   // up: p is what the partner wants, else q
    const uint4 s = up ? p : q;
    uint4 r;
    r.x = __shfl_xor_sync(0xffffffffu, s.x, mask);
    r.y = __shfl_xor_sync(0xffffffffu, s.y, mask);
    r.z = __shfl_xor_sync(0xffffffffu, s.z, mask);
    r.w = __shfl_xor_sync(0xffffffffu, s.w, mask);
    if (up) p = r;
    else q = r;
  };
  swap(a[0], a[1], b0, 1);
  swap(a[2], a[3], b0, 1);
  swap(a[0], a[2], b1, 2);
  swap(a[1], a[3], b1, 2);
}

// The tiles blockIdx.x, + gridDim.x, + 2 gridDim.x ... of B x tiles_y x tiles_x, by additions.
struct TileWalk {
  int tx, ty, b;
  __device__ __forceinline__ TileWalk(int tiles_x, int tiles_y) : nx(tiles_x), ny(tiles_y) {
    split((int)blockIdx.x, tx, ty, b);
    split((int)gridDim.x, dx, dy, db);
  }
  __device__ __forceinline__ void next() {
    tx += dx;
    ty += dy;
    b += db;
    if (tx >= nx) {
      tx -= nx;
      ++ty;
    }
    if (ty >= ny) {
      ty -= ny;
      ++b;
    }
  }

 private:
  int nx, ny, dx, dy, db;
  __device__ __forceinline__ void split(int i, int &x, int &y, int &z) const {
    x = i % nx;
    y = i / nx % ny;
    z = i / nx / ny;
  }
};

// Persistent over 8 x 16 output tiles, one CTA per SM, warp-specialised: eight warps copy input
// halos into a ring of stages; two warps issue the 9 x (CIN/16) MMAs of a tile, in turn, into the stage's own
// 32-column accumulator, so that one commit frees the halo and hands over the accumulator; two groups
// of four warps take the tiles in turn for the epilogue (tensor-memory read, bias, ReLU, residual,
// mask, store; one output pixel a thread), each loading its next tile's residual and mask before the
// current one's accumulator is complete.  What the epilogue does is a template parameter.
//
// kSrcImage (16 input channels): the halo is formed from the render (block_operand) instead of copied
// from a tensor.  kDstCompose (16 output channels): the epilogue composes the block's skipped pixels
// into the image (compose_block) instead of storing the residuals.
//
// What the parts do for a tile is short (18 MMAs of about 32 clocks, 11 KB loaded, 8 KB stored), so
// the time goes to latencies and the rings' depth decides: with residual on 2 x 1104 x 1032 pixels
// (32 -> 32, 438 MB, 65 us at the measured copy rate) 92 us under ncu with 12 stages, 108 us with 6;
// 131 us with one MMA warp and copies straight to shared memory, 140 us with five CTAs of 128 threads
// per SM that each loaded, multiplied and stored in turn.  Without it 102 -> 80 us; 16 x 128 x 128
// pixels 22 -> 15 us.  MMAs of several tiles interleaved in one issue stream: no faster.
//
// Twelve accumulators take all 512 columns of an SM's tensor memory (allocations are powers of two), so
// a kernel of another stream that needs some (a compact fill) shares no SM with this one: its CTA waits
// in its allocation until this one's ends.
constexpr int kConvStages = 12;                    // even: see the parities below; 32 accumulator columns each
constexpr int kConvThreads = 2 * 128 + 2 * 128 + 2 * 32;   // epilogue groups, copying groups, MMA warps
constexpr int kConvHR = kConvTH + 2, kConvHC = kConvTW + 2;
// one plane of 8 channels; the padding puts a pixel's groups in different banks (CIN 32)
constexpr int kConvPlane = kConvHR * kConvHC * 16 + 96;

template <int CIN, int COUT>
constexpr int conv_smem_bytes() { return kConvStages * (CIN / 8) * kConvPlane + 9 * (CIN / 8) * COUT * 16; }

template <int CIN, int COUT, int FLAGS, int SRC, int DST>
__global__ void __launch_bounds__(kConvThreads, 1)
conv3x3_tc_kernel(ConvDims d, const __nv_bfloat16 *__restrict__ X, const uint4 *__restrict__ Wpk,
                  const float *__restrict__ bias, const __nv_bfloat16 *__restrict__ R,
                  const __nv_bfloat16 *__restrict__ Mk, void *__restrict__ Y, uint32_t *__restrict__ status,
                  FillIO io) {
  static_assert(SRC == kSrcTensor || CIN == 16, "the image input has 16 channels");
  static_assert(DST == kDstTensor || COUT == 16, "the composed residuals have 16 channels");
  constexpr int CG = CIN / 8, HR = kConvHR, HC = kConvHC, S = kConvStages;
  constexpr int HALO = CG * kConvPlane, WBYTES = 9 * CG * COUT * 16;
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t *const ws = smem + S * HALO;
  __shared__ uint32_t s_tmem;
  __shared__ __align__(8) uint64_t s_full[S], s_done[S], s_free[S];   // halo landed, MMAs done, accumulator read
  __shared__ __align__(16) float s_bias[32];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int tiles_x = (d.W + kConvTW - 1) / kConvTW, tiles_y = (d.H + kConvTH - 1) / kConvTH;
  const int n_tiles = d.B * tiles_x * tiles_y;
  const int my_n = (n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;   // grid <= n_tiles
  if (warp == 16) tc::tmem_alloc(&s_tmem, 512);
  if (t == 0) {
    for (int k = 0; k < S; ++k) {
      tc::mbar_init(&s_full[k], 4);
      tc::mbar_init(&s_done[k], 1);
      tc::mbar_init(&s_free[k], 4);
    }
  }
  pdl_begin();
  for (int i = t; i < WBYTES / 16; i += kConvThreads) reinterpret_cast<uint4 *>(ws)[i] = __ldg(Wpk + i);
  if (t < COUT) s_bias[t] = (FLAGS & kEpiBias) ? bias[t] : 0.0f;
  if constexpr (SRC == kSrcImage) {
    for (int i = t; i < S * HR * HC; i += kConvThreads) {   // the second input group is zero
      const int st = i / (HR * HC), q = i - st * (HR * HC);
      *reinterpret_cast<uint4 *>(smem + st * HALO + kConvPlane + q * 16) = make_uint4(0u, 0u, 0u, 0u);
    }
  }
  tc::fence_proxy_async();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = s_tmem;

  if (warp >= 16) {
    // two warps take the tiles in turn (one's waits overlap the other's issue); a whole warp runs the
    // loop, so that descriptors stay in uniform registers, and one lane issues
    const bool leader = tc::elect_one();
    const uint32_t idesc = tc::idesc_bf16_f32(128, COUT), w0 = tc::smem_u32(ws), h00 = tc::smem_u32(smem);
    for (int k = warp - 16, st = warp - 16, ph = 0; k < my_n; k += 2) {
      bool ok = tc::mbar_wait(&s_full[st], ph);
      if (k >= S) ok = tc::mbar_wait(&s_free[st], ph ^ 1) && ok;
      if (!ok && leader) atomicOr(status, kStatusTimeout);
      tc::fence_after_sync();
      const uint32_t h0 = h00 + st * HALO;
#pragma unroll
      for (int tap = 0; tap < 9; ++tap)
#pragma unroll
        for (int cb = 0; cb < CIN / 16; ++cb) {
          const int ky = tap / 3, kx = tap - 3 * ky;
          tc::mma_bf16_if(leader, tmem + 32 * st,
                          tc::smem_desc(h0 + (2 * cb) * kConvPlane + ky * (HC * 16) + kx * 16, kConvPlane, HC * 16),
                          tc::smem_desc(w0 + tap * (CG * COUT * 16) + (2 * cb) * (COUT * 16), COUT * 16, 128), idesc,
                          tap > 0 || cb > 0);
        }
      if (leader) tc::mma_commit(&s_done[st]);
      __syncwarp();
      st += 2;   // S is even: a warp or group keeps its parity of stages
      if (st >= S) {
        st -= S;
        ph ^= 1;
      }
    }
  } else if (warp >= 8) {
    // Two groups of four warps take the tiles in turn, each with three register sets: a tile's loads
    // are issued two of the group's tiles before they are stored, so that five tiles are in flight.  (Copies straight to shared memory would be one L2 request per 16
    // bytes here -- neighbouring 16 bytes go to different planes -- and fetch every sector twice.)
    const int group = (warp - 8) >> 2, lt = t & 127;
    TileWalk at(tiles_x, tiles_y);
    if (group == 1) at.next();
    // image: two halo pixels a thread (180 of them), r g b depth; tensor: 120 threads, a column and
    // channel group each, every (12 / CG)-th row
    constexpr int RSTEP = 12 / CG, NV = SRC == kSrcImage ? 2 : HR / RSTEP;
    const int lg = lt % CG, lc = (lt / CG) % HC, lrow = lt / (CG * HC);
    auto load = [&](uint4 (&v)[NV]) {
      if constexpr (SRC == kSrcImage) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int q = lt + 128 * j, r = q / HC, c = q - r * HC;
          const int y = at.ty * kConvTH - 1 + r, x = at.tx * kConvTW - 1 + c;
          v[j] = make_uint4(0u, 0u, 0u, 0u);
          if (q < HR * HC && y >= 0 && y < d.H && x >= 0 && x < d.W) {
            const size_t src = ((size_t)at.b * io.H + 2 * y) * io.W + 2 * x;
            v[j] = make_uint4(__float_as_uint(io.img[3 * src]), __float_as_uint(io.img[3 * src + 1]),
                              __float_as_uint(io.img[3 * src + 2]), __float_as_uint(io.depth[src]));
          }
        }
      } else {
        const int x = at.tx * kConvTW - 1 + lc;
        int y = at.ty * kConvTH - 1 + lrow;
        const bool in_x = lrow < RSTEP && x >= 0 && x < d.W;
        const uint4 *src = reinterpret_cast<const uint4 *>(X + (((ptrdiff_t)at.b * d.H + y) * d.W + x) * CIN + lg * 8);
#pragma unroll
        for (int j = 0; j < NV; ++j) {
          v[j] = in_x && y >= 0 && y < d.H ? __ldg(src) : make_uint4(0u, 0u, 0u, 0u);
          y += RSTEP;
          src += (ptrdiff_t)RSTEP * d.W * CG;
        }
      }
      at.next();
      at.next();
    };
    int sst = group, sph = 1;
    auto store = [&](int k, const uint4 (&v)[NV]) {
      if (k >= S && !tc::mbar_wait(&s_done[sst], sph) && lane == 0) atomicOr(status, kStatusTimeout);
      uint8_t *hs = smem + sst * HALO;
      if constexpr (SRC == kSrcImage) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int q = lt + 128 * j;
          if (q < HR * HC)
            *reinterpret_cast<uint4 *>(hs + q * 16) = block_operand(
                make_float4(__uint_as_float(v[j].x), __uint_as_float(v[j].y), __uint_as_float(v[j].z),
                            __uint_as_float(v[j].w)));
        }
      } else if (lrow < RSTEP) {
#pragma unroll
        for (int j = 0; j < NV; ++j)
          *reinterpret_cast<uint4 *>(hs + lg * kConvPlane + ((lrow + j * RSTEP) * HC + lc) * 16) = v[j];
      }
      tc::fence_proxy_async();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&s_full[sst]);
      sst += 2;
      if (sst >= S) {
        sst -= S;
        sph ^= 1;
      }
    };
    uint4 va[NV], vb[NV], vc[NV];
    if (group < my_n) load(va);
    if (group + 2 < my_n) load(vb);
    for (int k = group; k < my_n; k += 6) {
      if (k + 4 < my_n) load(vc);
      store(k, va);
      if (k + 2 >= my_n) break;
      if (k + 6 < my_n) load(va);
      store(k + 2, vb);
      if (k + 4 >= my_n) break;
      if (k + 8 < my_n) load(vb);
      store(k + 4, vc);
    }
  } else {
    const int group = warp >> 2, m = t & 127;   // accumulator row = output pixel of the tile
    const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    uint4 rv[COUT / 8], mv[COUT / 8];
    size_t pix = 0;
    int b = 0, y = 0, x = 0;
    bool inside = false;
    TileWalk at(tiles_x, tiles_y);
    if (group == 1) at.next();
    auto prefetch = [&]() {   // the next tile of this group
      b = at.b;
      y = at.ty * kConvTH + m / kConvTW;
      x = at.tx * kConvTW + (m % kConvTW);
      inside = y < d.H && x < d.W;
      pix = inside ? ((size_t)b * d.H + y) * d.W + x : 0;
#pragma unroll
      for (int g = 0; g < COUT / 8; ++g) {
        if (FLAGS & kEpiResid)
          rv[g] = inside ? __ldg(reinterpret_cast<const uint4 *>(R + pix * COUT) + g) : make_uint4(0u, 0u, 0u, 0u);
        if (FLAGS & kEpiMask)
          mv[g] = inside ? __ldg(reinterpret_cast<const uint4 *>(Mk + pix * COUT) + g) : make_uint4(0u, 0u, 0u, 0u);
      }
      at.next();
      at.next();
    };
    if (group < my_n) prefetch();
    for (int k = group, st = group, ph = 0; k < my_n; k += 2) {
      if (!tc::mbar_wait(&s_done[st], ph) && lane == 0) atomicOr(status, kStatusTimeout);
      tc::fence_after_sync();
      float v[32];
      if (COUT == 32) tc::tmem_ld32(taddr + 32 * st, v);
      else tc::tmem_ld16(taddr + 32 * st, v);
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&s_free[st]);
      st += 2;
      if (st >= S) {
        st -= S;
        ph ^= 1;
      }
      if constexpr ((FLAGS & kEpiBias) != 0) {
#pragma unroll
        for (int c = 0; c < COUT; c += 4) {
          const float4 bv = *reinterpret_cast<const float4 *>(s_bias + c);
          v[c] += bv.x;
          v[c + 1] += bv.y;
          v[c + 2] += bv.z;
          v[c + 3] += bv.w;
        }
      }
      if constexpr (DST == kDstCompose) {
        if (inside) {
          const int lv = io.levels[b * io.n_tiles + ((2 * y) / io.tile) * io.tiles_x + (2 * x) / io.tile];
          if (lv < 4) {   // else every pixel of the block was rendered
            // residual of colour c, sub-pixel s = 2 dy + dx: channel 4 c + s (12..15 unused)
            float res[3][4];
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
              for (int q = 0; q < 4; ++q) res[c][q] = v[4 * c + q];
            compose_block(io.img, b, io.H, io.W, y, x, lv, res);
          }
        }
      } else {
        uint4 out[4];   // the pixel's 64 bytes: 32 BF16 or 16 FP32 channels
        static_assert(COUT * ((FLAGS & kEpiF32) ? 4 : 2) == 64 || DST == kDstCompose, "64 bytes a pixel");
#pragma unroll
        for (int g = 0; g < COUT / 8; ++g) {
          float o[8];
#pragma unroll
          for (int c = 0; c < 8; ++c) o[c] = (FLAGS & kEpiRelu) ? fmaxf(v[g * 8 + c], 0.0f) : v[g * 8 + c];
          if constexpr ((FLAGS & kEpiResid) != 0) {
            const __nv_bfloat16 *rb = reinterpret_cast<const __nv_bfloat16 *>(&rv[g]);
#pragma unroll
            for (int c = 0; c < 8; ++c) o[c] += __bfloat162float(rb[c]);
          }
          if constexpr ((FLAGS & kEpiMask) != 0) {
            const __nv_bfloat16 *mb = reinterpret_cast<const __nv_bfloat16 *>(&mv[g]);
#pragma unroll
            for (int c = 0; c < 8; ++c) o[c] = __bfloat162float(mb[c]) > 0.0f ? o[c] : 0.0f;
          }
          if constexpr ((FLAGS & kEpiF32) != 0) {
            out[2 * g] = make_uint4(__float_as_uint(o[0]), __float_as_uint(o[1]), __float_as_uint(o[2]),
                                    __float_as_uint(o[3]));
            out[2 * g + 1] = make_uint4(__float_as_uint(o[4]), __float_as_uint(o[5]), __float_as_uint(o[6]),
                                        __float_as_uint(o[7]));
          } else {
            __nv_bfloat162 *p2 = reinterpret_cast<__nv_bfloat162 *>(&out[g]);
#pragma unroll
            for (int c = 0; c < 4; ++c) p2[c] = __floats2bfloat162_rn(o[2 * c], o[2 * c + 1]);
          }
        }
        // four lanes hold four pixels of one row: exchanged so that every store covers whole pixels
        // (16 bytes a lane at a 64-byte stride would write every 32-byte sector in two halves)
        transpose4(out);
        const int xq = x & ~3;
        const bool in_y = y < d.H;
        uint4 *yo = static_cast<uint4 *>(Y) + (((size_t)b * d.H + y) * d.W + xq) * 4 + (lane & 3);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (in_y && xq + i < d.W) yo[4 * i] = out[i];
      }
      if (k + 2 < my_n) prefetch();
    }
    tc::fence_before_sync();
  }
  __syncthreads();
  tc::fence_after_sync();
  if (warp == 16) tc::tmem_dealloc(tmem, 512);
}

// The compact network's whole fill in one persistent kernel, per 16 x 16 block tile made of two
// halves of 8 x 16 blocks side by side, each half one MMA of M = 128 rows (row m of half h =
// block (y0 + m / 8, x0 + 8 h + m % 8)); thread t holds row t of both halves in the epilogues:
//   layer 0: the 3x3 convolution 16 -> 32 on the tile's 18 x 18 input halo, formed from the
//            render: per half 9 MMAs, N 32, K 16;
//   layer 1: the per-block layer 32 -> 32: per half 2 MMAs (K 32);
//   layer 2: the per-block layer 32 -> 16: per half 2 MMAs, the epilogue composing the block's
//            skipped pixels.
// The halo sits in shared memory as [row][column][8 channels] (16 bytes per block): a half's A
// operand for tap (ky, kx) starts ky rows, kx + 8 h columns in, its core matrices (8 blocks of
// one row) one halo row apart (SBO).  Input channels 8..15 are zero: the MMA's second K group
// reads the first group's blocks again (leading byte offset 0) against a zero block of weights,
// so those products are exactly zero.  The epilogues of layers 0 and 1 read the accumulators
// from tensor memory, add the bias, apply the ReLU, round to BF16 and write the next layer's A
// operands to shared memory as [half][K group of 8][row][8 channels] -- K-major core matrices,
// rows 16 bytes apart (SBO 128), K groups 2,048 bytes apart (LBO) -- so no activation leaves
// the SM.  The per-block layers' weights are the centre taps of their 3x3 packs.  The halo's
// FP32 colours stay beside it, so the compose step reads its top-left pixels in shared memory.
// The three layers of a tile reuse two 32-column accumulators (one per half); the CTAs sharing
// an SM overlap one another's serial chains, and the next tile's halo and levels load into
// registers while this tile's layers run.  Tiles whose blocks are all fully rendered (level 4)
// skip the network.
constexpr int kCmpTW = 2 * kConvTW, kCmpTH = kConvTH;   // 16 x 16 blocks
constexpr int kCmpHR = kCmpTH + 2, kCmpHC = kCmpTW + 2;
constexpr int kCmpHalo = kCmpHR * kCmpHC * 16;       // input group 0 (BF16) per halo block
constexpr int kCmpRgb = kCmpHR * kCmpHC * 16;        // FP32 r, g, b (and a pad) per halo block
constexpr int kCmpW0 = 9 * 32 * 16;                  // [tap][cout][8 cin] of input group 0
constexpr int kCmpZero = 32 * 16;                    // zero weights of input group 1
constexpr int kCmpW1 = 4 * 32 * 16;                  // [cin group][cout][8 cin]
constexpr int kCmpW2 = 4 * 16 * 16;
constexpr int kCmpAct = 2 * 4 * 128 * 16;            // [half][K group][row][8]
constexpr int kCmpSmem = kCmpHalo + kCmpRgb + kCmpW0 + kCmpZero + kCmpW1 + kCmpW2 + kCmpAct;
constexpr int kCmpCtas = 6;                          // CTAs per SM
static_assert(kCmpHalo % 16 == 0 && kCmpRgb % 16 == 0 && kCmpW0 % 16 == 0 && kCmpZero % 16 == 0 &&
              kCmpW1 % 16 == 0 && kCmpW2 % 16 == 0, "operands start on 16-byte boundaries");

__global__ void __launch_bounds__(128, kCmpCtas)
compact_fill_tc_kernel(ConvDims d, const uint4 *__restrict__ W0, const uint4 *__restrict__ W1,
                       const uint4 *__restrict__ W2, const float *__restrict__ bias,
                       uint32_t *__restrict__ status, FillIO io) {
  constexpr int HR = kCmpHR, HC = kCmpHC;
  constexpr int kGPer = (HR * HC + 127) / 128;
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t *const halo = smem;
  float4 *const rgb = reinterpret_cast<float4 *>(smem + kCmpHalo);
  uint8_t *const w0s = smem + kCmpHalo + kCmpRgb;
  uint8_t *const zs = w0s + kCmpW0;
  uint8_t *const w1s = zs + kCmpZero;
  uint8_t *const w2s = w1s + kCmpW1;
  uint8_t *const act = w2s + kCmpW2;
  __shared__ uint32_t s_tmem;
  __shared__ __align__(8) uint64_t s_bar;
  __shared__ float s_bias[80];   // b0 [32], b1 [32], b2 [16]
  const int t = threadIdx.x, warp = t >> 5;
  const int ty = t / kConvTW, tx = t % kConvTW;   // this thread's block within a half
  if (t < 80) s_bias[t] = bias[t];
  const int tiles_x = (d.W + kCmpTW - 1) / kCmpTW, tiles_y = (d.H + kCmpTH - 1) / kCmpTH;
  const int n_tiles = d.B * tiles_x * tiles_y;
  const int my_n = (int)blockIdx.x < n_tiles ? (n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
  const int lsh = io.tile == 32 ? 5 : 4;   // pixel -> tile shift (tiles of 16 or 32 pixels)
  // a tile's origin, halo blocks (r, g, b of the top-left pixel, depth; zero outside the image)
  // and the levels of this thread's two blocks (4 outside the image), loaded into registers
  float4 gv[kGPer];
  int nb = 0, ny0 = 0, nx0 = 0, lv_next[2] = {4, 4};
  auto gather_load = [&](int k) {
    const int tt = (int)blockIdx.x + k * (int)gridDim.x;
    const int r = tt / tiles_x;
    nx0 = (tt - r * tiles_x) * kCmpTW;
    nb = r / tiles_y;
    ny0 = (r - nb * tiles_y) * kCmpTH;
    const float *img = io.img + (size_t)nb * io.H * io.W * 3;
    const float *dep = io.depth + (size_t)nb * io.H * io.W;
#pragma unroll
    for (int j = 0; j < kGPer; ++j) {
      const int q = t + 128 * j, rr = q / HC, c = q - rr * HC;
      const int y = ny0 - 1 + rr, x = nx0 - 1 + c;
      gv[j] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (q < HR * HC && y >= 0 && y < d.H && x >= 0 && x < d.W) {
        const unsigned src = (unsigned)(2 * y) * (unsigned)io.W + (unsigned)(2 * x);
        gv[j] = make_float4(img[3 * src], img[3 * src + 1], img[3 * src + 2], dep[src]);
      }
    }
    const uint8_t *lrow = io.levels + nb * io.n_tiles + ((2 * (ny0 + ty)) >> lsh) * io.tiles_x;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int y = ny0 + ty, x = nx0 + 8 * h + tx;
      lv_next[h] = y < d.H && x < d.W ? lrow[(2 * x) >> lsh] : 4;
    }
  };
  // the BF16 operand ...
  auto store_operand = [&]() {
#pragma unroll
    for (int j = 0; j < kGPer; ++j) {
      const int q = t + 128 * j;
      if (q < HR * HC) *reinterpret_cast<uint4 *>(halo + (size_t)q * 16) = block_operand(gv[j]);
    }
  };
  // ... and the FP32 colours
  auto store_colours = [&]() {
#pragma unroll
    for (int j = 0; j < kGPer; ++j) {
      const int q = t + 128 * j;
      if (q < HR * HC) rgb[q] = gv[j];
    }
  };
  if (warp == 0) tc::tmem_alloc(&s_tmem, 64);
  for (int i = t; i < kCmpW0 / 16; i += 128) {   // input group 0 of each tap: the first 32 of 64 rows
    const int tap = i / 32, row = i - tap * 32;
    reinterpret_cast<uint4 *>(w0s)[i] = __ldg(W0 + tap * 64 + row);
  }
  for (int i = t; i < kCmpZero / 16; i += 128) reinterpret_cast<uint4 *>(zs)[i] = make_uint4(0u, 0u, 0u, 0u);
  for (int i = t; i < kCmpW1 / 16; i += 128) reinterpret_cast<uint4 *>(w1s)[i] = __ldg(W1 + i);
  for (int i = t; i < kCmpW2 / 16; i += 128) reinterpret_cast<uint4 *>(w2s)[i] = __ldg(W2 + i);
  if (my_n > 0) {
    gather_load(0);
    store_operand();
  }
  tc::fence_proxy_async();
  if (t == 0) tc::mbar_init(&s_bar, 1);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = s_tmem;
  const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16);
  const uint32_t h0 = tc::smem_u32(halo), a0 = tc::smem_u32(act);
  const uint32_t b0 = tc::smem_u32(w0s), b1 = tc::smem_u32(w1s), b2 = tc::smem_u32(w2s);
  uint32_t phase = 0;
  // one thread waits for the MMAs (bounded); the others wait at the barrier, issuing nothing
  auto wait_mma = [&]() {
    if (t == 0) {
      if (!tc::mbar_wait(&s_bar, phase)) atomicOr(status, kStatusTimeout);
      tc::fence_before_sync();
    }
    phase ^= 1u;
    __syncthreads();
    tc::fence_after_sync();
  };
  // bias (+ ReLU) of both halves' 32-column accumulators, rounded to BF16 as the next layer's
  // A operands
  auto to_act = [&](int boff) {
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      float v[32];
      tc::tmem_ld32(taddr + 32 * h, v);
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        uint4 pk;
        __nv_bfloat162 *p2 = reinterpret_cast<__nv_bfloat162 *>(&pk);
#pragma unroll
        for (int c = 0; c < 4; ++c)
          p2[c] = __floats2bfloat162_rn(fmaxf(v[g * 8 + 2 * c] + s_bias[boff + g * 8 + 2 * c], 0.0f),
                                        fmaxf(v[g * 8 + 2 * c + 1] + s_bias[boff + g * 8 + 2 * c + 1], 0.0f));
        *reinterpret_cast<uint4 *>(act + h * 8192 + g * 2048 + t * 16) = pk;
      }
    }
    tc::fence_proxy_async();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
  };
  // the per-block layer (N = 16 or 32) of both halves, issued by thread 0
  auto issue_block_layer = [&](uint32_t bw0, int n) {
    const uint32_t idesc = tc::idesc_bf16_f32(128, n);
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int kk = 0; kk < 2; ++kk)
        tc::mma_bf16(tmem + 32 * h, tc::smem_desc(a0 + h * 8192 + kk * 4096, 2048, 128),
                     tc::smem_desc(bw0 + kk * (2 * n * 16), n * 16, 128), idesc, kk > 0);
    tc::mma_commit(&s_bar);
  };
  const int bh = (io.H + 1) / 2, bw = (io.W + 1) / 2;   // blocks per column and row
  for (int k = 0; k < my_n; ++k) {
    const int b = nb, y0 = ny0, x0 = nx0, lv0 = lv_next[0], lv1 = lv_next[1];
    // operand k stored and fenced by every thread; the last tile's tensor-memory reads and
    // colour reads done
    const bool need = __syncthreads_or(lv0 < 4 || lv1 < 4) != 0;
    tc::fence_after_sync();
    store_colours();   // read by this tile's compose, after the barriers below
    if (need && t == 0) {
      const uint32_t idesc = tc::idesc_bf16_f32(128, 32);
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
          const int ky = tap / 3, kx = tap - 3 * ky;
          tc::mma_bf16(tmem + 32 * h, tc::smem_desc(h0 + (ky * HC + kx + 8 * h) * 16, 0, HC * 16),
                       tc::smem_desc(b0 + tap * 512, (9 - tap) * 512, 128), idesc, tap > 0);
        }
      tc::mma_commit(&s_bar);
    }
    if (k + 1 < my_n) gather_load(k + 1);   // in flight while this tile's layers run
    if (need) {
      wait_mma();
      to_act(0);
      if (t == 0) issue_block_layer(b1, 32);
      wait_mma();
      to_act(32);
      if (t == 0) issue_block_layer(b2, 16);
      wait_mma();
      const int y = y0 + ty, rd = min(y + 1, bh - 1) - y0 + 1, Y = 2 * y;
      float *const img = io.img + (size_t)b * io.H * io.W * 3;
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        const int lv = h ? lv1 : lv0;
        float v[16];
        tc::tmem_ld16(taddr + 32 * h, v);
        if (lv >= 4) continue;   // outside the image or every pixel of the block rendered
        // the top-left pixels of the block, its right and lower neighbours and the diagonal one
        // (the last block repeated past the edge) from the halo's colours; then the same
        // arithmetic as compose_block
        const int cx = tx + 8 * h, x = x0 + cx;
        const int cr = min(x + 1, bw - 1) - x0 + 1;
        const float4 a = rgb[(ty + 1) * HC + cx + 1], right = rgb[(ty + 1) * HC + cr];
        const float4 down = rgb[rd * HC + cx + 1], diag = rgb[rd * HC + cr];
        const float av[3] = {a.x, a.y, a.z}, rv[3] = {right.x, right.y, right.z};
        const float dv[3] = {down.x, down.y, down.z}, gv3[3] = {diag.x, diag.y, diag.z};
        const int X = 2 * x;
        auto put = [&](int dy, int dx, const float *base, int s) {
          if (Y + dy >= io.H || X + dx >= io.W) return;
          float *o = img + 3 * ((unsigned)(Y + dy) * (unsigned)io.W + (unsigned)(X + dx));
#pragma unroll
          for (int c = 0; c < 3; ++c) o[c] = base[c] + (v[4 * c + s] + s_bias[64 + 4 * c + s]);
        };
        float bt[3], bb[3], bd[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          bt[c] = __fmul_rn(__fadd_rn(av[c], rv[c]), 0.5f);
          bb[c] = __fmul_rn(__fadd_rn(av[c], dv[c]), 0.5f);
          bd[c] = __fmul_rn(__fadd_rn(__fadd_rn(__fadd_rn(av[c], rv[c]), dv[c]), gv3[c]), 0.25f);
        }
        if (lv <= 2) put(0, 1, bt, 1);   // top-right: label 3, rendered from level 3
        float *const o1 = img + 3 * ((unsigned)(Y + 1) * (unsigned)io.W + (unsigned)X);
        if (lv <= 1 && Y + 1 < io.H && X + 1 < io.W && (reinterpret_cast<uintptr_t>(o1) & 7u) == 0) {
          // bottom-left and bottom-right: six consecutive floats, three 8-byte stores
          float2 *o2 = reinterpret_cast<float2 *>(o1);
          auto res = [&](int c, int s) { return v[4 * c + s] + s_bias[64 + 4 * c + s]; };
          o2[0] = make_float2(bb[0] + res(0, 2), bb[1] + res(1, 2));
          o2[1] = make_float2(bb[2] + res(2, 2), bd[0] + res(0, 3));
          o2[2] = make_float2(bd[1] + res(1, 3), bd[2] + res(2, 3));
        } else {
          if (lv <= 3) put(1, 0, bb, 2);   // bottom-left: label 4, rendered at level 4
          if (lv <= 1) put(1, 1, bd, 3);   // bottom-right: label 2, rendered from level 2
        }
      }
    }
    if (k + 1 < my_n) store_operand();   // layer 0 of this tile, if any, has completed
    tc::fence_proxy_async();
    tc::fence_before_sync();
  }
  __syncthreads();
  tc::fence_after_sync();
  if (warp == 0) tc::tmem_dealloc(tmem, 64);
}

// Weight gradient  dW[cout][cin][tap] += sum over pixels of X[q + tap][cin] dY[q][cout]  as one
// accumulator  D[(ky, cout)][(kx, cin)] += A[(ky, cout)][pixel] B[(kx, cin)][pixel]^T  with K =
// the pixels p of X: the row of A for tap row ky is dY one row below, at or above p, the row of B
// for tap column kx is X one column left of, at or right of the column of dY.  Both operands are
// read as they lie in memory, channels innermost (MN-major descriptors: a core matrix is 8 pixels
// of one image row x 8 channels, 16 bytes a pixel), so a tile is staged by 16-byte asynchronous
// copies alone and nothing is transposed:
//   dY as [row][cout group][column]: the rows are 8 COUT / 8 core matrices apart, so the M groups
//      (2 - ky, cout group) of one MMA are one core matrix apart (M = 128; 3 COUT rows used);
//   X as planes [kx][cin group][row][column], three copies a column apart; then a plane of ones in
//      channel 0, whose accumulator column for ky = 1 is the sum of dY: the bias gradient.
// Rows and columns past those read whatever follows in shared memory and are never read back.
// One CTA per SM, warp-specialised: four warps copy tiles into a ring of stages, one thread issues
// the 8 MMAs of a tile (K = 16: two image rows).  The partial sums go to a scratch gradient
// [tap][cout][cin] (bias after the weights) in 16-byte reductions, two lanes to a 32-byte sector;
// unpack_grads_kernel lays it out as the parameters.
// All nine taps in one MMA, because what bounds it is the operands' shared-memory reads: one MMA
// per tap row, (kx, cin) x cout, reads A three times (2.2 times the time per tile), and one CTA per
// SM, because every CTA ends with the whole gradient in reductions (5 us of a launch at two per SM).
// 32 -> 32 on 16 x 128 x 128 pixels under ncu: 318 us with both operands transposed into K-major
// tiles by 2-byte stores and scalar reductions at a 36-byte stride; 18 us now.
constexpr int kWgTW = 8, kWgTH = 16;               // K = 128 pixels per tile
constexpr int kWgStages = 4;
constexpr int kWgThreads = 160;                    // four copying warps and the MMA warp
template <int C> constexpr int wg_pad() { return 16 * (64 / C); }   // a pixel's groups in different banks
template <int CIN> constexpr int wg_plane() { return kWgTH * kWgTW * 16 + wg_pad<CIN>(); }
template <int COUT> constexpr int wg_core() { return kWgTW * 16 + wg_pad<COUT>(); }
template <int CIN, int COUT>
constexpr int wgrad_stage_bytes() {
  return (3 * (CIN / 8) + 1) * wg_plane<CIN>() + (kWgTH + 2) * (COUT / 8) * wg_core<COUT>();
}
// the last core matrices of the last stage's A operand end past its rows
template <int CIN, int COUT>
constexpr int wgrad_smem_bytes() { return kWgStages * wgrad_stage_bytes<CIN, COUT>() + 16 * wg_core<COUT>(); }

__device__ __forceinline__ void red_add4(float *p, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

// Adds v[0..N), of this lane's row, to row[0..N) of every lane (rows of adjacent lanes exchange
// quarters so that two lanes cover one 32-byte sector of one row per instruction).  Whole warps;
// row may be null in adjacent pairs of lanes only.
template <int N>
__device__ __forceinline__ void red_add_rows(float *row, const float *v) {
  const bool odd = threadIdx.x & 1;
  const unsigned long long mine = reinterpret_cast<unsigned long long>(row);
  float *const other = reinterpret_cast<float *>(__shfl_xor_sync(0xffffffffu, mine, 1));
  float *const even_row = odd ? other : row, *const odd_row = odd ? row : other;
#pragma unroll
  for (int c = 0; c < N; c += 8) {
    float r[4];   // even lanes: the odd row's first half sector; odd lanes: the even row's second
#pragma unroll
    for (int j = 0; j < 4; ++j) r[j] = __shfl_xor_sync(0xffffffffu, odd ? v[c + j] : v[c + 4 + j], 1);
    if (row) {
      if (odd) {
        red_add4(even_row + c + 4, r[0], r[1], r[2], r[3]);
        red_add4(odd_row + c + 4, v[c + 4], v[c + 5], v[c + 6], v[c + 7]);
      } else {
        red_add4(even_row + c, v[c], v[c + 1], v[c + 2], v[c + 3]);
        red_add4(odd_row + c, r[0], r[1], r[2], r[3]);
      }
    }
  }
}

template <int CIN, int COUT>
__global__ void __launch_bounds__(kWgThreads, 1)
conv3x3_wgrad_tc_kernel(ConvDims d, const __nv_bfloat16 *__restrict__ X, const __nv_bfloat16 *__restrict__ dY,
                        float *__restrict__ dW, float *__restrict__ db, uint32_t *__restrict__ status) {
  constexpr int CG = CIN / 8, OG = COUT / 8, XG = 3 * CG, HR = kWgTH + 2, S = kWgStages;
  constexpr int XP = wg_plane<CIN>(), YC = wg_core<COUT>(), XROW = kWgTW * 16, YROW = OG * YC;
  constexpr int STAGE = wgrad_stage_bytes<CIN, COUT>(), YOFF = (XG + 1) * XP;
  constexpr int N = 3 * CIN + 16;   // the plane of ones and one of nothing: N is a multiple of 16
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ uint32_t s_tmem;
  __shared__ __align__(8) uint64_t s_full[S], s_empty[S], s_done;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int tx_n = (d.W + kWgTW - 1) / kWgTW, ty_n = (d.H + kWgTH - 1) / kWgTH;
  const int n_tiles = d.B * tx_n * ty_n;
  const int my_n = (n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;   // grid <= n_tiles
  for (int i = t; i < S * kWgTH * kWgTW; i += kWgThreads) {
    const int stage = i / (kWgTH * kWgTW), q = i - stage * (kWgTH * kWgTW);
    *reinterpret_cast<uint4 *>(smem + stage * STAGE + XG * XP + q * 16) = make_uint4(0x3f80u, 0u, 0u, 0u);
  }
  if (warp == 4) tc::tmem_alloc(&s_tmem, 128);
  if (t == 0) {
    for (int k = 0; k < S; ++k) {
      tc::mbar_init(&s_full[k], 4);
      tc::mbar_init(&s_empty[k], 1);
    }
    tc::mbar_init(&s_done, 1);
  }
  tc::fence_proxy_async();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = s_tmem;
  pdl_begin();
  if (warp == 4) {
    const bool leader = tc::elect_one();   // as in conv3x3_tc_kernel
    constexpr uint32_t idesc = tc::idesc_bf16_f32(128, N) | tc::kIdescMnMajorA | tc::kIdescMnMajorB;
    const uint32_t s0 = tc::smem_u32(smem);
    for (int k = 0; k < my_n; ++k) {
      const int st = k % S;
      if (!tc::mbar_wait(&s_full[st], (k / S) & 1) && leader) atomicOr(status, kStatusTimeout);
      tc::fence_after_sync();
      const uint32_t b0 = s0 + st * STAGE, a0 = b0 + YOFF;
#pragma unroll
      for (int r = 0; r < kWgTH / 2; ++r)
        tc::mma_bf16_if(leader, tmem, tc::smem_desc(a0 + 2 * r * YROW, YROW, YC),
                        tc::smem_desc(b0 + 2 * r * XROW, XROW, XP), idesc, k > 0 || r > 0);
      if (leader) tc::mma_commit(&s_empty[st]);
      __syncwarp();
    }
    if (leader) tc::mma_commit(&s_done);
    __syncwarp();
  } else {
    // threads 0..95 copy X (24 CG of them one row of the three copies), threads 96..127 dY (8 OG a
    // row): each thread one (shift, column, group) down the rows, so a copy costs a few additions
    const bool mine_x = t < 96;
    const int lt = mine_x ? t : t - 96;
    const int lg = mine_x ? lt % CG : lt % OG, lc = (mine_x ? lt / CG : lt / OG) % kWgTW;
    const int lkx = (lt / (CG * kWgTW)) % 3;                                             // X only
    const int lrow = mine_x ? lt / (CG * kWgTW * 3) : lt / (OG * kWgTW), lstep = mine_x ? 4 / CG : 4 / OG;
    const uint32_t ldst = mine_x ? (lkx * CG + lg) * XP + lrow * XROW + lc * 16
                                 : YOFF + lrow * YROW + lg * YC + lc * 16;
    TileWalk at(tx_n, ty_n);
    for (int k = 0; k < my_n + 2; ++k) {
      const int st = k % S;
      if (k >= S && k < my_n && !tc::mbar_wait(&s_empty[st], (k / S - 1) & 1) && lane == 0)
        atomicOr(status, kStatusTimeout);
      if (k < my_n) {
        const int x0 = at.tx * kWgTW, y0 = at.ty * kWgTH;
        const ptrdiff_t img = (ptrdiff_t)at.b * d.H * d.W;
        at.next();
        uint32_t dst = tc::smem_u32(smem + st * STAGE) + ldst;
        if (mine_x) {
          const int x = x0 - 1 + lkx + lc;
          const bool in_x = x >= 0 && x < d.W;
          int y = y0 + lrow;
          const __nv_bfloat16 *src = X + (img + (ptrdiff_t)y * d.W + x) * CIN + lg * 8;
          const ptrdiff_t step = (ptrdiff_t)lstep * d.W * CIN;
#pragma unroll 8
          for (int row = lrow; row < kWgTH; row += lstep) {
            const bool in = in_x && y < d.H;
            // the three copies of a row read the same lines: through L1
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(in ? src : X),
                         "r"(in ? 16 : 0)
                         : "memory");
            dst += lstep * XROW;
            src += step;
            y += lstep;
          }
        } else {
          const int x = x0 + lc;
          int y = y0 - 1 + lrow;
          const __nv_bfloat16 *src = dY + (img + (ptrdiff_t)y * d.W + x) * COUT + lg * 8;
          const ptrdiff_t step = (ptrdiff_t)lstep * d.W * COUT;
#pragma unroll 6
          for (int row = lrow; row < HR; row += lstep) {
            const bool in = x < d.W && y >= 0 && y < d.H;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(in ? src : dY),
                         "r"(in ? 16 : 0)
                         : "memory");
            dst += lstep * YROW;
            src += step;
            y += lstep;
          }
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      if (k >= 2) {   // tile k - 2 has landed
        asm volatile("cp.async.wait_group 2;" ::: "memory");
        tc::fence_proxy_async();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&s_full[(k - 2) % S]);
      }
    }
    if (!tc::mbar_wait(&s_done, 0) && lane == 0) atomicOr(status, kStatusTimeout);
    tc::fence_after_sync();
    // accumulator rows (2 - ky, cout), columns (kx, cin), then the ones
    const int row = warp * 32 + lane, ky = 2 - row / COUT, co = row % COUT;
    const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16);
    if (warp * 32 < 3 * COUT) {   // whole warps: 3 COUT is 96, or 48 with the rest skipped below
#pragma unroll 1
      for (int kx = 0; kx < 3; ++kx) {
        float v[32];
        if (CIN == 32) tc::tmem_ld32(taddr + kx * CIN, v);
        else tc::tmem_ld16(taddr + kx * CIN, v);
        red_add_rows<CIN>(ky >= 0 ? dW + (size_t)((ky * 3 + kx) * COUT + co) * CIN : nullptr, v);
      }
      float v[16];
      tc::tmem_ld16(taddr + 3 * CIN, v);
      if (ky == 1) atomicAdd(db + co, v[0]);
    }
    tc::fence_before_sync();
  }
  __syncthreads();
  tc::fence_after_sync();
  if (warp == 4) tc::tmem_dealloc(tmem, 128);
}

// ------------------------------------------------------- CUDA-core helpers of the network
// x0[b][y2][x2] = (r, g, b, depth / 8, 0 ...) of the top-left pixel of each 2x2 block.
__global__ void gather_input_kernel(const float *__restrict__ img, const float *__restrict__ depth, int B,
                                    int H, int W, __nv_bfloat16 *__restrict__ x0) {
  pdl_begin();
  const int H2 = (H + 1) / 2, W2 = (W + 1) / 2;
  const size_t n = (size_t)B * H2 * W2;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int x2 = (int)(i % W2);
    const size_t r = i / W2;
    const int y2 = (int)(r % H2), b = (int)(r / H2);
    uint4 *dst = reinterpret_cast<uint4 *>(x0 + i * 16);
    dst[0] = block_input(img, depth, b, H, W, y2, x2);
    dst[1] = make_uint4(0u, 0u, 0u, 0u);
  }
}

// Base of sub-pixel (dx, dy) of block (x2, y2), colour c: the bilinear interpolation of the
// blocks' top-left pixels of img [B][H][W][3] -- a, right = (x2 + 1), down = (y2 + 1), diag --
// with the last block repeated past the edge: a; (a + right) / 2; (a + down) / 2;
// (((a + right) + down) + diag) / 4.  Where only top-left pixels are rendered it is the
// interpolating fill (Sec. 3.4 "inherit or interpolate").
__device__ __forceinline__ float base_px(const float *__restrict__ img, int b, int H, int W, int y2,
                                         int x2, int dy, int dx, int c) {
  const int H2 = (H + 1) / 2, W2 = (W + 1) / 2;
  const int xr = min(x2 + 1, W2 - 1), yd = min(y2 + 1, H2 - 1);
  auto tl = [&](int yy, int xx) { return img[3 * (((size_t)b * H + 2 * yy) * W + 2 * xx) + c]; };
  const float a = tl(y2, x2);
  if (dx == 0 && dy == 0) return a;
  if (dy == 0) return __fmul_rn(__fadd_rn(a, tl(y2, xr)), 0.5f);
  if (dx == 0) return __fmul_rn(__fadd_rn(a, tl(yd, x2)), 0.5f);
  return __fmul_rn(__fadd_rn(__fadd_rn(__fadd_rn(a, tl(y2, xr)), tl(yd, x2)), tl(yd, xr)), 0.25f);
}

// Prediction = bilinear base + residual of the sub-pixel; loss = mean squared error against
// the target; g_r = dL/dr (BF16, channels 12..15 zero).  loss_acc accumulates the sum of
// squared errors.
__global__ void loss_kernel(const float *__restrict__ r, const float *__restrict__ img,
                            const float *__restrict__ target, int B, int H, int W, float inv_count,
                            __nv_bfloat16 *__restrict__ g_r, float *__restrict__ loss_acc) {
  pdl_begin();
  const int H2 = (H + 1) / 2, W2 = (W + 1) / 2;
  const size_t n = (size_t)B * H2 * W2;
  float acc = 0.0f;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int x2 = (int)(i % W2);
    const size_t rr = i / W2;
    const int y2 = (int)(rr % H2), b = (int)(rr / H2);
    float g[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) g[k] = 0.0f;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const int dy = s >> 1, dx = s & 1;
      const int y = 2 * y2 + dy, x = 2 * x2 + dx;
      if (y >= H || x >= W) continue;
      const size_t q = ((size_t)b * H + y) * W + x;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float e = base_px(img, b, H, W, y2, x2, dy, dx, c) + r[i * 16 + c * 4 + s] - target[3 * q + c];
        acc += e * e;
        g[c * 4 + s] = 2.0f * e * inv_count;
      }
    }
    uint4 *dst = reinterpret_cast<uint4 *>(g_r + i * 16);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint4 pk;
      __nv_bfloat162 *p2 = reinterpret_cast<__nv_bfloat162 *>(&pk);
#pragma unroll
      for (int c = 0; c < 4; ++c) p2[c] = __floats2bfloat162_rn(g[h * 8 + 2 * c], g[h * 8 + 2 * c + 1]);
      dst[h] = pk;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(loss_acc, acc);
}

// Adam on the fp32 master parameters.
__global__ void adam_kernel(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, int n, float lr, float b1, float b2, float eps,
                            float c1, float c2) {
  pdl_begin();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + eps);
  }
}

// BF16 packs of one layer's weights W[cout][cin][9]: forward [tap][cin/8][cout][8 cin] and the
// data-gradient conv's [tap'][cout/8][cin][8 cout] with W'[cin][cout][tap'] = W[cout][cin][8 - tap'].
// A per-block (1x1) layer, W[cout][cin] with taps = 1, is the centre tap (4) of a 3x3 pack whose
// other taps stay zero, so the 3x3 kernels train it unchanged.
__global__ void pack_kernel(const float *__restrict__ w, int cin, int cout, int taps,
                            __nv_bfloat16 *__restrict__ fwd, __nv_bfloat16 *__restrict__ bwd) {
  pdl_begin();
  const int n = cin * cout * taps;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int tap = taps == 9 ? i % 9 : 4, rest = taps == 9 ? i / 9 : i;
    const int ci = rest % cin, co = rest / cin;
    const __nv_bfloat16 v = __float2bfloat16_rn(w[i]);
    fwd[((size_t)(tap * (cin / 8) + ci / 8) * cout + co) * 8 + (ci & 7)] = v;
    if (bwd) bwd[((size_t)((8 - tap) * (cout / 8) + co / 8) * cin + ci) * 8 + (co & 7)] = v;
  }
}

// Layer tables.  Residual network: ten 3x3 convolutions (16 -> 32, eight 32 -> 32, 32 -> 16).
// Compact network: 3x3 16 -> 32, then the per-block layers 32 -> 32 and 32 -> 16.
constexpr int kLayers = 10;   // the most layers of either network
int n_layers(int arch) { return arch == A3FR_CNN_COMPACT ? 3 : kLayers; }
int layer_in(int arch, int l) { return l == 0 ? 16 : 32; }
int layer_out(int arch, int l) { return l == n_layers(arch) - 1 ? 16 : 32; }
int layer_taps(int arch, int l) { return arch == A3FR_CNN_COMPACT && l > 0 ? 1 : 9; }

size_t weight_offset(int arch, int l) {
  size_t o = 0;
  for (int k = 0; k < l; ++k) o += (size_t)layer_in(arch, k) * layer_out(arch, k) * layer_taps(arch, k);
  return o;
}
size_t bias_offset(int arch, int l) {
  size_t o = weight_offset(arch, n_layers(arch));
  for (int k = 0; k < l; ++k) o += layer_out(arch, k);
  return o;
}
size_t n_params(int arch) { return bias_offset(arch, n_layers(arch)); }

// The scratch gradient of the weight-gradient kernels: per layer [9 taps][cout][cin], then [cout].
size_t scratch_offset(int arch, int l) {
  size_t o = 0;
  for (int k = 0; k < l; ++k) o += ((size_t)9 * layer_in(arch, k) + 1) * layer_out(arch, k);
  return o;
}

struct GradMap {   // per layer: parameters and scratch offsets
  int n_layers, n_params;
  int w[kLayers], b[kLayers], scratch[kLayers], cin[kLayers], cout[kLayers], taps[kLayers];
};

GradMap grad_map(int arch) {
  GradMap m{};
  m.n_layers = n_layers(arch);
  m.n_params = (int)n_params(arch);
  for (int l = 0; l < m.n_layers; ++l) {
    m.w[l] = (int)weight_offset(arch, l);
    m.b[l] = (int)bias_offset(arch, l);
    m.scratch[l] = (int)scratch_offset(arch, l);
    m.cin[l] = layer_in(arch, l);
    m.cout[l] = layer_out(arch, l);
    m.taps[l] = layer_taps(arch, l);
  }
  return m;
}

// The flat gradient, laid out as the parameters (W[cout][cin][taps] per layer, then the biases),
// from the scratch gradient; a per-block layer takes the centre tap.
__global__ void unpack_grads_kernel(GradMap m, const float *__restrict__ scratch, float *__restrict__ grads) {
  pdl_begin();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m.n_params; i += gridDim.x * blockDim.x) {
    int l = m.n_layers - 1;
    if (i < m.b[0]) {
      while (i < m.w[l]) --l;
      const int j = i - m.w[l], tap = m.taps[l] == 9 ? j % 9 : 4, rest = j / m.taps[l];
      const int ci = rest % m.cin[l], co = rest / m.cin[l];
      grads[i] = scratch[m.scratch[l] + (tap * m.cout[l] + co) * m.cin[l] + ci];
    } else {
      while (i < m.b[l]) --l;
      grads[i] = scratch[m.scratch[l] + 9 * m.cin[l] * m.cout[l] + (i - m.b[l])];
    }
  }
}

int grid_1d(size_t n) {
  const size_t b = (n + 255) / 256;
  const size_t most = 16 * (size_t)sm_count();
  return (int)(b < most ? (b > 0 ? b : 1) : most);
}

}  // namespace
}  // namespace a3fr

struct a3fr_cnn {
  int arch = A3FR_CNN_RESIDUAL;
  float *params = nullptr, *grads = nullptr, *adam_m = nullptr, *adam_v = nullptr;
  float *wscratch = nullptr;   // the gradients as the weight-gradient kernels leave them (scratch_offset)
  __nv_bfloat16 *wf[a3fr::kLayers] = {}, *wb[a3fr::kLayers] = {};
  size_t cap_px = 0;
  __nv_bfloat16 *x0 = nullptr, *h[5] = {}, *t[4] = {}, *g_r = nullptr, *gA = nullptr, *gB = nullptr, *gT = nullptr;
  float *r = nullptr;
  float *loss_acc = nullptr;
  uint32_t *status = nullptr;
  int step = 0;
};

namespace a3fr {
namespace {

template <typename T>
void dfree2(T *&p) {
  if (p) cudaFree(p);
  p = nullptr;
}

void free_acts(a3fr_cnn *n) {
  dfree2(n->x0);
  for (auto &p : n->h) dfree2(p);
  for (auto &p : n->t) dfree2(p);
  dfree2(n->g_r);
  dfree2(n->gA);
  dfree2(n->gB);
  dfree2(n->gT);
  dfree2(n->r);
  n->cap_px = 0;
}

int ensure_acts(a3fr_cnn *n, size_t px) {
  if (px <= n->cap_px) return A3FR_OK;
  free_acts(n);
  const size_t b16 = sizeof(__nv_bfloat16);
  bool ok = cudaMalloc(&n->x0, px * 16 * b16) == cudaSuccess &&
            cudaMalloc(&n->g_r, px * 16 * b16) == cudaSuccess &&
            cudaMalloc(&n->gA, px * 32 * b16) == cudaSuccess &&
            cudaMalloc(&n->gB, px * 32 * b16) == cudaSuccess &&
            cudaMalloc(&n->gT, px * 32 * b16) == cudaSuccess &&
            cudaMalloc(&n->r, px * 16 * sizeof(float)) == cudaSuccess;
  for (auto &p : n->h) ok = ok && cudaMalloc(&p, px * 32 * b16) == cudaSuccess;
  for (auto &p : n->t) ok = ok && cudaMalloc(&p, px * 32 * b16) == cudaSuccess;
  if (!ok) {
    free_acts(n);
    return A3FR_ERR_OOM;
  }
  n->cap_px = px;
  return A3FR_OK;
}

template <int CIN, int COUT, int FLAGS, int SRC = kSrcTensor, int DST = kDstTensor>
cudaError_t conv(const ConvDims &d, const __nv_bfloat16 *X, const __nv_bfloat16 *W, const float *bias,
                 const __nv_bfloat16 *R, const __nv_bfloat16 *M, void *Y, uint32_t *status, cudaStream_t s,
                 const FillIO &io = FillIO{}) {
  constexpr int smem = conv_smem_bytes<CIN, COUT>();
  static bool attr[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !attr[dev]) {
    cudaError_t e = cudaFuncSetAttribute(conv3x3_tc_kernel<CIN, COUT, FLAGS, SRC, DST>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    attr[dev] = true;
  }
  const int tiles = d.B * ((d.W + kConvTW - 1) / kConvTW) * ((d.H + kConvTH - 1) / kConvTH);
  return launch_pdl(conv3x3_tc_kernel<CIN, COUT, FLAGS, SRC, DST>, std::min(tiles, sm_count()), kConvThreads, smem, s,
                    d, X, reinterpret_cast<const uint4 *>(W), bias, R, M, Y, status, io);
}

cudaError_t compact_fill(const ConvDims &d, const a3fr_cnn *n, uint32_t *status, cudaStream_t s, const FillIO &io) {
  static bool attr[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !attr[dev]) {
    cudaError_t e = cudaFuncSetAttribute(compact_fill_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kCmpSmem);
    if (e != cudaSuccess) return e;
    attr[dev] = true;
  }
  const int tiles = d.B * ((d.W + kCmpTW - 1) / kCmpTW) * ((d.H + kCmpTH - 1) / kCmpTH);
  const int grid = std::min(tiles, sm_count() * kCmpCtas);
  const int A = A3FR_CNN_COMPACT;
  // the per-block layers' weights: the centre tap (4) of their 3x3 packs [tap][cin/8][cout][8]
  const uint4 *w1 = reinterpret_cast<const uint4 *>(n->wf[1] + 4 * 32 * 32);
  const uint4 *w2 = reinterpret_cast<const uint4 *>(n->wf[2] + 4 * 32 * 16);
  compact_fill_tc_kernel<<<grid, 128, kCmpSmem, s>>>(d, reinterpret_cast<const uint4 *>(n->wf[0]), w1, w2,
                                                     n->params + bias_offset(A, 0), status, io);
  return cudaGetLastError();
}

// Adds layer l's weight and bias gradients to the scratch gradient.
template <int CIN, int COUT>
cudaError_t wgrad(const a3fr_cnn *n, int l, const ConvDims &d, const __nv_bfloat16 *X, const __nv_bfloat16 *dY,
                  cudaStream_t s) {
  constexpr int smem = wgrad_smem_bytes<CIN, COUT>();
  static bool attr[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !attr[dev]) {
    cudaError_t e = cudaFuncSetAttribute(conv3x3_wgrad_tc_kernel<CIN, COUT>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    attr[dev] = true;
  }
  const int tiles = d.B * ((d.H + kWgTH - 1) / kWgTH) * ((d.W + kWgTW - 1) / kWgTW);
  float *dW = n->wscratch + scratch_offset(n->arch, l);
  return launch_pdl(conv3x3_wgrad_tc_kernel<CIN, COUT>, std::min(tiles, sm_count()), kWgThreads, smem, s, d, X, dY,
                    dW, dW + 9 * CIN * COUT, n->status);
}

#define CNN_CHECK(call)                                  \
  do {                                                   \
    cudaError_t e_ = (call);                             \
    if (e_ != cudaSuccess) return A3FR_ERR_CUDA;         \
  } while (0)

int pack_all(a3fr_cnn *n, cudaStream_t s) {
  for (int l = 0; l < n_layers(n->arch); ++l) {
    const int cin = layer_in(n->arch, l), cout = layer_out(n->arch, l), taps = layer_taps(n->arch, l);
    pack_kernel<<<grid_1d((size_t)cin * cout * taps), 256, 0, s>>>(n->params + weight_offset(n->arch, l), cin,
                                                                  cout, taps, n->wf[l], l > 0 ? n->wb[l] : nullptr);
    CNN_CHECK(cudaGetLastError());
  }
  return A3FR_OK;
}

// The prediction r (training, a3fr_cnn_forward: io null) or, for the fill (io set), the
// composed image.  Residual network, fill: the first convolution reads its input from the
// render and the last composes the skipped pixels, with neither x0 nor r stored.  Compact
// network, fill: one fused kernel (no activation tensors at all); training: the 3x3 kernels,
// the per-block layers as centre-tap packs.
int forward(a3fr_cnn *n, const float *img, const float *depth, int B, int H, int W, cudaStream_t s,
            const FillIO *io = nullptr) {
  const ConvDims d{B, (H + 1) / 2, (W + 1) / 2};
  const size_t px = (size_t)d.B * d.H * d.W;
  const int A = n->arch;
  if (A == A3FR_CNN_COMPACT && io) {
    CNN_CHECK(compact_fill(d, n, n->status, s, *io));
    return A3FR_OK;
  }
  const int rc = ensure_acts(n, px);
  if (rc != A3FR_OK) return rc;
  const float *P = n->params;
  if (io) {
    CNN_CHECK((conv<16, 32, kBiasRelu, kSrcImage>(d, nullptr, n->wf[0], P + bias_offset(A, 0), nullptr, nullptr,
                                                  n->h[0], n->status, s, *io)));
  } else {
    CNN_CHECK(launch_pdl(gather_input_kernel, grid_1d(px), 256, 0, s, img, depth, B, H, W, n->x0));
    CNN_CHECK((conv<16, 32, kBiasRelu>(d, n->x0, n->wf[0], P + bias_offset(A, 0), nullptr, nullptr, n->h[0], n->status,
                                       s)));
  }
  if (A == A3FR_CNN_COMPACT) {
    CNN_CHECK((conv<32, 32, kBiasRelu>(d, n->h[0], n->wf[1], P + bias_offset(A, 1), nullptr, nullptr, n->t[0],
                                       n->status, s)));
    CNN_CHECK((conv<32, 16, kEpiBias | kEpiF32>(d, n->t[0], n->wf[2], P + bias_offset(A, 2), nullptr, nullptr, n->r,
                                                n->status, s)));
    return A3FR_OK;
  }
  for (int b = 0; b < 4; ++b) {
    CNN_CHECK((conv<32, 32, kBiasRelu>(d, n->h[b], n->wf[1 + 2 * b], P + bias_offset(A, 1 + 2 * b), nullptr, nullptr,
                                       n->t[b], n->status, s)));
    CNN_CHECK((conv<32, 32, kEpiBias | kEpiResid>(d, n->t[b], n->wf[2 + 2 * b], P + bias_offset(A, 2 + 2 * b), n->h[b],
                                                  nullptr, n->h[b + 1], n->status, s)));
  }
  if (io) {
    CNN_CHECK((conv<32, 16, kEpiBias, kSrcTensor, kDstCompose>(d, n->h[4], n->wf[9], P + bias_offset(A, 9), nullptr,
                                                               nullptr, nullptr, n->status, s, *io)));
  } else {
    CNN_CHECK((conv<32, 16, kEpiBias | kEpiF32>(d, n->h[4], n->wf[9], P + bias_offset(A, 9), nullptr, nullptr, n->r,
                                                n->status, s)));
  }
  return A3FR_OK;
}

// Gradients of the mean squared error of the prediction against target into n->grads.
int backward(a3fr_cnn *n, const float *img, const float *target, int B, int H, int W, cudaStream_t s) {
  const ConvDims d{B, (H + 1) / 2, (W + 1) / 2};
  const size_t px = (size_t)d.B * d.H * d.W;
  const int A = n->arch;
  CNN_CHECK(cudaMemsetAsync(n->wscratch, 0, sizeof(float) * scratch_offset(A, n_layers(A)), s));
  CNN_CHECK(cudaMemsetAsync(n->loss_acc, 0, sizeof(float), s));
  CNN_CHECK(launch_pdl(loss_kernel, grid_1d(px), 256, 0, s, n->r, img, target, B, H, W, 1.0f / (3.0f * B * H * W),
                       n->g_r, n->loss_acc));
  if (A == A3FR_CNN_COMPACT) {
    // r = W2 t + b2;  t = ReLU(W1 h + b1);  h = ReLU(conv0(x0) + b0)
    CNN_CHECK((wgrad<32, 16>(n, 2, d, n->t[0], n->g_r, s)));
    CNN_CHECK((conv<16, 32, kEpiMask>(d, n->g_r, n->wb[2], nullptr, nullptr, n->t[0], n->gA, n->status, s)));
    CNN_CHECK((wgrad<32, 32>(n, 1, d, n->h[0], n->gA, s)));
    CNN_CHECK((conv<32, 32, kEpiMask>(d, n->gA, n->wb[1], nullptr, nullptr, n->h[0], n->gB, n->status, s)));
    CNN_CHECK((wgrad<16, 32>(n, 0, d, n->x0, n->gB, s)));
  } else {
    CNN_CHECK((wgrad<32, 16>(n, 9, d, n->h[4], n->g_r, s)));
    CNN_CHECK((conv<16, 32, 0>(d, n->g_r, n->wb[9], nullptr, nullptr, nullptr, n->gA, n->status, s)));
    __nv_bfloat16 *cur = n->gA, *nxt = n->gB;
    for (int b = 3; b >= 0; --b) {
      const int l2 = 2 + 2 * b, l1 = 1 + 2 * b;
      CNN_CHECK((wgrad<32, 32>(n, l2, d, n->t[b], cur, s)));
      CNN_CHECK((conv<32, 32, kEpiMask>(d, cur, n->wb[l2], nullptr, nullptr, n->t[b], n->gT, n->status, s)));
      CNN_CHECK((wgrad<32, 32>(n, l1, d, n->h[b], n->gT, s)));
      if (b == 0)
        CNN_CHECK((conv<32, 32, kEpiResid | kEpiMask>(d, n->gT, n->wb[l1], nullptr, cur, n->h[0], nxt, n->status, s)));
      else
        CNN_CHECK((conv<32, 32, kEpiResid>(d, n->gT, n->wb[l1], nullptr, cur, nullptr, nxt, n->status, s)));
      __nv_bfloat16 *tmp = cur;
      cur = nxt;
      nxt = tmp;
    }
    CNN_CHECK((wgrad<16, 32>(n, 0, d, n->x0, cur, s)));
  }
  CNN_CHECK(launch_pdl(unpack_grads_kernel, grid_1d(n_params(A)), 256, 0, s, grad_map(A), n->wscratch, n->grads));
  return A3FR_OK;
}

int read_status(a3fr_cnn *n, cudaStream_t s) {
  uint32_t h = 0;
  CNN_CHECK(cudaMemcpyAsync(&h, n->status, sizeof h, cudaMemcpyDeviceToHost, s));
  CNN_CHECK(cudaStreamSynchronize(s));
  return h ? A3FR_ERR_TIMEOUT : A3FR_OK;
}

}  // namespace
}  // namespace a3fr

using namespace a3fr;

extern "C" int a3fr_tc_tile_gemm(const uint16_t *A, const uint16_t *B, float *D, int n, int k,
                                 int variant, void *stream) {
  if (!A || !B || !D || (n != 16 && n != 32) || k < 16 || k > 64 || k % 16 != 0 ||
      (variant != 0 && variant != 1))
    return A3FR_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint32_t *status = nullptr;
  if (cudaMalloc(&status, sizeof(uint32_t)) != cudaSuccess) return A3FR_ERR_OOM;
  cudaError_t e = cudaMemsetAsync(status, 0, sizeof(uint32_t), st);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(tc_tile_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kProbeSmem);
  if (e == cudaSuccess) {
    tc_tile_gemm_kernel<<<1, 128, kProbeSmem, st>>>(A, B, D, n, k, variant, status);
    e = cudaGetLastError();
  }
  uint32_t h = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, status, sizeof h, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(status);
  if (e != cudaSuccess) return A3FR_ERR_CUDA;
  return h ? A3FR_ERR_TIMEOUT : A3FR_OK;
}

extern "C" {

size_t a3fr_cnn_param_count(void) { return n_params(A3FR_CNN_RESIDUAL); }

size_t a3fr_cnn_arch_param_count(int arch) {
  return arch == A3FR_CNN_RESIDUAL || arch == A3FR_CNN_COMPACT ? n_params(arch) : 0;
}

int a3fr_cnn_create(a3fr_cnn **out) { return a3fr_cnn_create_arch(out, A3FR_CNN_RESIDUAL); }

int a3fr_cnn_create_arch(a3fr_cnn **out, int arch) {
  if (!out || (arch != A3FR_CNN_RESIDUAL && arch != A3FR_CNN_COMPACT)) return A3FR_ERR_INVALID_ARG;
  *out = nullptr;
  a3fr_cnn *n = new (std::nothrow) a3fr_cnn();
  if (!n) return A3FR_ERR_OOM;
  n->arch = arch;
  const size_t np = n_params(arch);
  bool ok = cudaMalloc(&n->params, np * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&n->grads, np * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&n->adam_m, np * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&n->adam_v, np * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&n->wscratch, scratch_offset(arch, n_layers(arch)) * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&n->loss_acc, sizeof(float)) == cudaSuccess &&
            cudaMalloc(&n->status, sizeof(uint32_t)) == cudaSuccess;
  for (int l = 0; l < n_layers(arch) && ok; ++l) {   // 3x3 packs (a per-block layer: its centre tap)
    const size_t w = (size_t)layer_in(arch, l) * layer_out(arch, l) * 9 * sizeof(__nv_bfloat16);
    ok = cudaMalloc(&n->wf[l], w) == cudaSuccess && cudaMalloc(&n->wb[l], w) == cudaSuccess &&
         cudaMemset(n->wf[l], 0, w) == cudaSuccess && cudaMemset(n->wb[l], 0, w) == cudaSuccess;
  }
  if (ok) ok = cudaMemset(n->params, 0, np * sizeof(float)) == cudaSuccess &&
               cudaMemset(n->adam_m, 0, np * sizeof(float)) == cudaSuccess &&
               cudaMemset(n->adam_v, 0, np * sizeof(float)) == cudaSuccess &&
               cudaMemset(n->status, 0, sizeof(uint32_t)) == cudaSuccess;
  if (ok) ok = pack_all(n, nullptr) == A3FR_OK && cudaDeviceSynchronize() == cudaSuccess;
  if (!ok) {
    a3fr_cnn_destroy(n);
    return A3FR_ERR_OOM;
  }
  *out = n;
  return A3FR_OK;
}

int a3fr_cnn_destroy(a3fr_cnn *n) {
  if (!n) return A3FR_ERR_INVALID_ARG;
  cudaDeviceSynchronize();
  free_acts(n);
  dfree2(n->params);
  dfree2(n->grads);
  dfree2(n->adam_m);
  dfree2(n->adam_v);
  dfree2(n->wscratch);
  dfree2(n->loss_acc);
  dfree2(n->status);
  for (int l = 0; l < kLayers; ++l) {
    dfree2(n->wf[l]);
    dfree2(n->wb[l]);
  }
  delete n;
  return A3FR_OK;
}

int a3fr_cnn_set_params(a3fr_cnn *n, const float *host, size_t count) {
  if (!n || !host || count != n_params(n->arch)) return A3FR_ERR_INVALID_ARG;
  CNN_CHECK(cudaMemcpy(n->params, host, count * sizeof(float), cudaMemcpyHostToDevice));
  CNN_CHECK(cudaMemset(n->adam_m, 0, count * sizeof(float)));
  CNN_CHECK(cudaMemset(n->adam_v, 0, count * sizeof(float)));
  n->step = 0;
  const int rc = pack_all(n, nullptr);
  if (rc != A3FR_OK) return rc;
  CNN_CHECK(cudaDeviceSynchronize());
  return A3FR_OK;
}

int a3fr_cnn_get_params(a3fr_cnn *n, float *host, size_t count) {
  if (!n || !host || count != n_params(n->arch)) return A3FR_ERR_INVALID_ARG;
  CNN_CHECK(cudaDeviceSynchronize());
  CNN_CHECK(cudaMemcpy(host, n->params, count * sizeof(float), cudaMemcpyDeviceToHost));
  return A3FR_OK;
}

int a3fr_cnn_forward(a3fr_cnn *n, const float *img, const float *depth, int b, int h, int w,
                     float *residual_out, void *stream) {
  if (!n || !img || !depth || b < 1 || h < 2 || w < 2) return A3FR_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int rc = forward(n, img, depth, b, h, w, s);
  if (rc != A3FR_OK) return rc;
  if (residual_out) {
    const size_t px = (size_t)b * ((h + 1) / 2) * ((w + 1) / 2);
    CNN_CHECK(cudaMemcpyAsync(residual_out, n->r, px * 16 * sizeof(float), cudaMemcpyDeviceToDevice, s));
  }
  return A3FR_OK;
}

int a3fr_cnn_grads(a3fr_cnn *n, const float *img, const float *depth, const float *target, int b, int h,
                   int w, float *host_grads, float *loss, void *stream) {
  if (!n || !img || !depth || !target || !host_grads || b < 1 || h < 2 || w < 2) return A3FR_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int rc = forward(n, img, depth, b, h, w, s);
  if (rc == A3FR_OK) rc = backward(n, img, target, b, h, w, s);
  if (rc != A3FR_OK) return rc;
  CNN_CHECK(cudaMemcpyAsync(host_grads, n->grads, n_params(n->arch) * sizeof(float), cudaMemcpyDeviceToHost, s));
  float acc = 0.0f;
  CNN_CHECK(cudaMemcpyAsync(&acc, n->loss_acc, sizeof(float), cudaMemcpyDeviceToHost, s));
  rc = read_status(n, s);
  if (loss) *loss = acc / (3.0f * b * h * w);
  return rc;
}

int a3fr_cnn_train_step(a3fr_cnn *n, const float *img, const float *depth, const float *target, int b, int h,
                        int w, float lr, float *loss, void *stream) {
  if (!n || !img || !depth || !target || b < 1 || h < 2 || w < 2 || !(lr > 0.0f)) return A3FR_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int rc = forward(n, img, depth, b, h, w, s);
  if (rc == A3FR_OK) rc = backward(n, img, target, b, h, w, s);
  if (rc != A3FR_OK) return rc;
  n->step++;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.0f / (1.0f - powf(b1, (float)n->step)), c2 = 1.0f / (1.0f - powf(b2, (float)n->step));
  adam_kernel<<<grid_1d(n_params(n->arch)), 256, 0, s>>>(n->params, n->grads, n->adam_m, n->adam_v,
                                                         (int)n_params(n->arch), lr, b1, b2, 1e-8f, c1, c2);
  CNN_CHECK(cudaGetLastError());
  rc = pack_all(n, s);
  if (rc != A3FR_OK) return rc;
  if (loss) {
    float acc = 0.0f;
    CNN_CHECK(cudaMemcpyAsync(&acc, n->loss_acc, sizeof(float), cudaMemcpyDeviceToHost, s));
    rc = read_status(n, s);
    *loss = acc / (3.0f * b * h * w);
    return rc;
  }
  return A3FR_OK;
}

int a3fr_cnn_fill(a3fr_cnn *n, a3fr_scene *scene, float *out_rgb, void *stream) {
  if (!n || !scene || !out_rgb) return A3FR_ERR_INVALID_ARG;
  FillView v{};
  if (!scene_fill_view(scene, &v)) return A3FR_ERR_NOT_READY;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const FillIO io{v.depth, out_rgb, v.levels, v.height, v.width, v.tile, v.tiles_x, v.n_tiles};
  return forward(n, out_rgb, v.depth, v.eyes, v.height, v.width, s, &io);
}

}  // extern "C"
