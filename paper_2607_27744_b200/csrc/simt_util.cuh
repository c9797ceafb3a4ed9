// Helpers of the plain (non tensor-core) kernels.
#pragma once
#include <cuda_bf16.h>
#include <cstdint>

#include "rocs_internal.h"

namespace rocs {

// Copies `rows` dense rows of `d` elements (fp32 or bf16, global memory) into shared memory as fp32
// with row stride `ds`.  Where rows are whole 16-byte vectors the block issues four vector loads per
// thread before it touches shared memory, so a request's operand arrives after about one memory
// latency instead of one per element (measured on the request-side kernels of the interaction
// operators: 16 dependent scalar loads per thread cost more than all of their arithmetic).
template <typename T>
__device__ __forceinline__ void rows_to_shared(const T* __restrict__ src, float* __restrict__ dst, int rows, int d,
                                               int ds) {
  constexpr int kVec = 16 / (int)sizeof(T);
  const int total = rows * d;
  if (d % kVec == 0 && (reinterpret_cast<uintptr_t>(src) & 15u) == 0) {
    const int n_vec = total / kVec;
    constexpr int kBatch = 4;
    for (int base = threadIdx.x; base < n_vec; base += kBatch * blockDim.x) {
      uint4 raw[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int v = base + u * blockDim.x;
        if (v < n_vec) raw[u] = __ldg(reinterpret_cast<const uint4*>(src) + v);
      }
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int v = base + u * blockDim.x;
        if (v >= n_vec) continue;
        const int e = v * kVec;
        float* out = dst + (e / d) * ds + e % d;
        if constexpr (sizeof(T) == 4) {
          out[0] = __uint_as_float(raw[u].x);
          out[1] = __uint_as_float(raw[u].y);
          out[2] = __uint_as_float(raw[u].z);
          out[3] = __uint_as_float(raw[u].w);
        } else {
          const uint32_t w[4] = {raw[u].x, raw[u].y, raw[u].z, raw[u].w};
#pragma unroll
          for (int j = 0; j < 4; ++j) {  // bf16 -> fp32 is a shift into the high half
            out[2 * j] = __uint_as_float(w[j] << 16);
            out[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
          }
        }
      }
    }
  } else {
    for (int e = threadIdx.x; e < total; e += blockDim.x) {
      if constexpr (sizeof(T) == 4)
        dst[(e / d) * ds + e % d] = reinterpret_cast<const float*>(src)[e];
      else
        dst[(e / d) * ds + e % d] = __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(src)[e]);
    }
  }
}

// Entry i of the list of tiles of at most `per` consecutive candidates of one request, in the order
// request, head, tile (heads = 1: request, tile), found by the block itself from the offsets of R <= THREADS
// requests: one request per thread and one scan.  A list in memory is one more launch and allocation in
// front of the kernel (4 us of a 68 us pass over 4 tiny requests); where there are more requests than
// threads the caller brings the plan's list.  All threads of the block call this.
struct FoundTile {
  int32_t req, cand0, count, head;
};
template <int THREADS>
__device__ __forceinline__ FoundTile find_tile_in_block(int32_t R, int32_t per, int32_t heads,
                                                        const int32_t* __restrict__ off, int32_t i) {
  __shared__ int32_t warp_sum[THREADS / 32];
  __shared__ FoundTile found;
  const int32_t t = threadIdx.x, lane = t % 32;
  const int32_t c0 = t < R ? off[t] : 0, n = t < R ? off[t + 1] - c0 : 0;
  const int32_t tiles = tiles_of(n, per), entries = tiles * heads;
  int32_t incl = entries;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += up;
  }
  if (lane == 31) warp_sum[t / 32] = incl;
  __syncthreads();
  int32_t first = incl - entries;
  for (int w = 0; w < t / 32; ++w) first += warp_sum[w];
  if (first <= i && i < first + entries) {
    const int32_t local = i - first, h = local / tiles, c = (local - h * tiles) * per;
    found = FoundTile{t, c0 + c, min(per, n - c), h};
  }
  __syncthreads();
  return found;
}

__device__ __forceinline__ void cp_async_16(uint32_t smem_dst, const void* src, int bytes) {  // the rest of the 16 is zeros
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
}

// Eight bf16 values of one 16-byte vector as fp32.
__device__ __forceinline__ void bf16x8_to_f32(const uint4& raw, float4& lo, float4& hi) {
  lo = make_float4(__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xffff0000u), __uint_as_float(raw.y << 16),
                   __uint_as_float(raw.y & 0xffff0000u));
  hi = make_float4(__uint_as_float(raw.z << 16), __uint_as_float(raw.z & 0xffff0000u), __uint_as_float(raw.w << 16),
                   __uint_as_float(raw.w & 0xffff0000u));
}

// A tile of `rows` rows of up to COLS columns into shared memory as fp32 (row stride `stride` floats, a
// multiple of 4), zeros beyond `valid` rows and beyond d columns.  Rows are `ld` elements apart in
// global memory and start on 16-byte boundaries; d is a multiple of a 16-byte vector.  fp32 goes by
// cp.async (the caller commits and waits), bf16 through registers.
template <typename T, int COLS>
__device__ __forceinline__ void rows_to_shared_async(const T* __restrict__ src, int64_t ld, int valid, int rows, int d,
                                                     float* __restrict__ dst, int stride, int tid, int threads) {
  constexpr int kVec = 16 / (int)sizeof(T), kPerRow = COLS / kVec;
#pragma unroll 4
  for (int v = tid; v < rows * kPerRow; v += threads) {
    const int r = v / kPerRow, c = (v % kPerRow) * kVec;
    const bool in = r < valid && c < d;
    const T* from = src + (in ? r * ld + c : 0);
    float* to = dst + r * stride + c;
    if constexpr (sizeof(T) == 4) {
      cp_async_16((uint32_t)__cvta_generic_to_shared(to), from, in ? 16 : 0);
    } else {
      float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
      if (in) bf16x8_to_f32(__ldg(reinterpret_cast<const uint4*>(from)), lo, hi);
      *reinterpret_cast<float4*>(to) = lo;
      *reinterpret_cast<float4*>(to + 4) = hi;
    }
  }
}

// `rows` dense rows of d elements (d a multiple of a 16-byte vector) into shared memory as fp32 with row
// stride `stride` floats; fp32 by cp.async, bf16 through registers.
template <typename T>
__device__ __forceinline__ void dense_rows_to_shared_async(const T* __restrict__ src, int rows, int d,
                                                           float* __restrict__ dst, int stride, int tid, int threads) {
  constexpr int kVec = 16 / (int)sizeof(T);
  const int per_row = d / kVec, dr = threads / per_row, dc = threads - dr * per_row;
  int r = tid / per_row, c = tid - r * per_row;
#pragma unroll 4
  for (int v = tid; v < rows * per_row; v += threads) {
    float* to = dst + r * stride + c * kVec;
    r += dr;
    c += dc;
    if (c >= per_row) {
      c -= per_row;
      ++r;
    }
    if constexpr (sizeof(T) == 4) {
      cp_async_16((uint32_t)__cvta_generic_to_shared(to), src + (int64_t)v * kVec, 16);
    } else {
      float4 lo, hi;
      bf16x8_to_f32(__ldg(reinterpret_cast<const uint4*>(src) + v), lo, hi);
      *reinterpret_cast<float4*>(to) = lo;
      *reinterpret_cast<float4*>(to + 4) = hi;
    }
  }
}

// Component c (a constant after unrolling) of a vector.
__device__ __forceinline__ float lane_of(const float4& v, int c) { return c == 0 ? v.x : c == 1 ? v.y : c == 2 ? v.z : v.w; }

__device__ __forceinline__ void store_pair(float* p, float a, float b) { *reinterpret_cast<float2*>(p) = make_float2(a, b); }
__device__ __forceinline__ void store_pair(__nv_bfloat16* p, float a, float b) {
  *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(a, b);
}

}  // namespace rocs
