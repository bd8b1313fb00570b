// stage.cuh -- staging of a block's slices of the scene arrays in shared memory, shared by the
// projection and its backward, and the 16-byte asynchronous copy.
#pragma once

#include <cuda_runtime.h>

namespace a3fr {

// SH rows whose 3K floats are whole 16-byte chunks (degrees 1 and 3) are staged by cp.async
// without padding; with an even number of chunks per row (degree 3: 12) chunk m of thread t's
// row sits at m ^ ((t >> 1) & 3), so the eight threads of a quarter warp reading the same
// chunk index hit eight different 16-byte bank groups.
template <int K>
constexpr bool sh_chunked() { return (3 * K) % 4 == 0; }

template <int K>
__device__ __forceinline__ int sh_swz(int m, int t) {
  return ((3 * K / 4) % 2 == 0) ? (m ^ ((t >> 1) & 3)) : m;
}

// Shared-memory stride of one Gaussian's SH row: 3K floats (chunked rows), else rounded up to
// an odd count so the per-thread scalar reads are free of bank conflicts.
template <int K>
constexpr int sh_stride() { return sh_chunked<K>() ? 3 * K : ((3 * K) % 2 == 0 ? 3 * K + 1 : 3 * K); }

// Cooperative coalesced copy of `count` floats starting at src into shared memory,
// laid out as rows of `row` floats at stride `stride`.  src is 16-byte aligned.
__device__ __forceinline__ void stage(float *dst, const float *__restrict__ src, int count,
                                      int row, int stride) {
  const int n4 = count >> 2;
  const float4 *src4 = reinterpret_cast<const float4 *>(src);
  // four independent 16-byte loads in flight per thread before the shared-memory stores
  for (int i0 = threadIdx.x; i0 < n4; i0 += 4 * blockDim.x) {
    float4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = i0 + u * blockDim.x;
      v[u] = i < n4 ? __ldg(src4 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = i0 + u * blockDim.x;
      if (i < n4) {
        const float e[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int f = 4 * i + j;
          dst[(f / row) * stride + (f % row)] = e[j];
        }
      }
    }
  }
  for (int f = 4 * n4 + threadIdx.x; f < count; f += blockDim.x)
    dst[(f / row) * stride + (f % row)] = __ldg(src + f);
}

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
}

// Asynchronous copy of `count` floats from src to dst (both 16-byte aligned); a tail of
// fewer than four floats is copied with plain loads.
__device__ __forceinline__ void stage_async(float *dst, const float *__restrict__ src, int count) {
  const int n4 = count >> 2;
  for (int i = threadIdx.x; i < n4; i += blockDim.x) cp_async16(dst + 4 * i, src + 4 * i);
  for (int f = 4 * n4 + threadIdx.x; f < count; f += blockDim.x) dst[f] = __ldg(src + f);
}

// Asynchronous copy of `cnt` chunked SH rows into the swizzled shared-memory layout.
template <int K>
__device__ __forceinline__ void stage_sh_async(float *dst, const float *__restrict__ src, int cnt) {
  constexpr int kChunks = 3 * K / 4;
  for (int g = threadIdx.x; g < cnt * kChunks; g += blockDim.x) {
    const int t = g / kChunks, m = g - t * kChunks;
    cp_async16(dst + 4 * (t * kChunks + sh_swz<K>(m, t)), src + 4 * g);
  }
}

}  // namespace a3fr
