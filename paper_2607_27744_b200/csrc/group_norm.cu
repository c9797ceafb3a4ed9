// Group-local normalisation (Eq. 7): every row of ONE group's tensor X [M, d] is normalised over
// its own d coordinates, so no statistic spans two groups (request rows and candidate rows are
// separate tensors and separate calls).
//   LayerNorm:  y = (x - mean) / sqrt(var + eps) * gamma + beta     (biased variance)
//   RMSNorm:    y = x / sqrt(mean(x^2) + eps) * gamma
// Pure streaming work (read once, write once), bound by memory: a row on 4 to 32 lanes of one
// warp, held in registers as 16-byte vectors, statistics in fp32 by shuffles among them, the
// variance taken around the mean from the registers (no E[x^2] - E[x]^2 cancellation).  Rows
// of more than 256 vectors or a width that is no whole number of them run on a kernel that
// re-reads the row element by element (from L1/L2).
#include <algorithm>

#include "rocs_internal.h"
#include "sm100_ptx.cuh"

namespace rocs {
namespace {

constexpr int kWarpsPerBlock = 8;

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <typename T>
struct Vec;  // 16 bytes of T
template <>
struct Vec<float> {
  static constexpr int kElems = 4;
  static __device__ __forceinline__ void load(const float* p, float (&f)[4]) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
  }
  static __device__ __forceinline__ void store(float* p, const float (&f)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(f[0], f[1], f[2], f[3]);
  }
};
template <>
struct Vec<__nv_bfloat16> {
  static constexpr int kElems = 8;
  static __device__ __forceinline__ void load(const __nv_bfloat16* p, float (&f)[8]) {
    const uint4 v = *reinterpret_cast<const uint4*>(p);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      f[2 * i] = __uint_as_float(w[i] << 16);
      f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
  }
  static __device__ __forceinline__ void store(__nv_bfloat16* p, const float (&f)[8]) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
      w[i] = *reinterpret_cast<const uint32_t*>(&h);
    }
    *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
  }
};

// Rows of whole 16-byte vectors, at most NV * G of them (FULL: exactly): G lanes per row, lane l of them owns vectors
// l, l + G, ...; a warp has 32 / G rows at a time.  Lanes without a row or a vector add nothing.
template <typename T, int NV, int G, bool FULL>
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
group_norm_rows_kernel(int kind, int64_t M, int32_t d_arg, const T* __restrict__ X, int64_t ld_x, const T* __restrict__ gamma,
                       const T* __restrict__ beta, float eps, T* __restrict__ Y, int64_t ld_y) {
  constexpr int E = Vec<T>::kElems;
  constexpr int kRows = 32 / G;
  ptx::griddep_wait_for(X, gamma, beta);
  ptx::griddep_launch_dependents();
  const int d = FULL ? NV * G * E : d_arg;
  // d as a divisor of fp32 rows: 1 / d is up to 2^-24 off, which shows beside their rounding (d = 1000: error 6.3e-8 against
  // 64 bits, 5.8e-8 divided).  bf16 rows are rounded to 2^-9, and the division would be on their path: 9.0 us at [40000,
  // 200] and 10.1 divided.
  auto per_d = [inv_d = 1.f / (float)d, d](float v) { return sizeof(T) == 4 ? v / (float)d : v * inv_d; };
  const int lane = threadIdx.x % G, sub = threadIdx.x % 32 / G;
  const int64_t warp = (int64_t)blockIdx.x * kWarpsPerBlock + threadIdx.x / 32;
  const int64_t n_warps = (int64_t)gridDim.x * kWarpsPerBlock;
  auto group_sum = [](float v) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  for (int64_t first = warp * kRows; first < M; first += n_warps * kRows) {
    const int64_t row = first + sub;
    const bool have = kRows == 1 || row < M;
    float x[NV][E];
    float s = 0.f;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int col = (v * G + lane) * E;
      if (have && (FULL || col < d)) {
        Vec<T>::load(X + row * ld_x + col, x[v]);
      } else {
#pragma unroll
        for (int e = 0; e < E; ++e) x[v][e] = 0.f;
      }
#pragma unroll
      for (int e = 0; e < E; ++e) s += x[v][e];
    }
    float mean = 0.f;
    if (kind == ROCS_NORM_LAYER) mean = per_d(group_sum(s));
    float sq = 0.f;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      if (!FULL && (v * G + lane) * E >= d) continue;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        x[v][e] -= mean;
        sq = fmaf(x[v][e], x[v][e], sq);
      }
    }
    const float inv = rsqrtf(per_d(group_sum(sq)) + eps);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int col = (v * G + lane) * E;
      if (!have || (!FULL && col >= d)) continue;
      float g[E], b[E];
#pragma unroll
      for (int e = 0; e < E; ++e) {
        g[e] = 1.f;
        b[e] = 0.f;
      }
      if (gamma) Vec<T>::load(gamma + col, g);
      if (beta && kind == ROCS_NORM_LAYER) Vec<T>::load(beta + col, b);
#pragma unroll
      for (int e = 0; e < E; ++e) x[v][e] = fmaf(x[v][e] * inv, g[e], b[e]);
      Vec<T>::store(Y + row * ld_y + col, x[v]);
    }
  }
}

__device__ __forceinline__ float ld_f(const float* p, int64_t i) { return p[i]; }
__device__ __forceinline__ float ld_f(const __nv_bfloat16* p, int64_t i) { return __bfloat162float(p[i]); }
__device__ __forceinline__ void st_f(float* p, int64_t i, float v) { p[i] = v; }
__device__ __forceinline__ void st_f(__nv_bfloat16* p, int64_t i, float v) { p[i] = __float2bfloat16_rn(v); }

// any d: the row is read three times (sum, centred squares, output), scalar accesses
template <typename T>
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
group_norm_general_kernel(int kind, int64_t M, int32_t d, const T* __restrict__ X, int64_t ld_x,
                          const T* __restrict__ gamma, const T* __restrict__ beta, float eps, T* __restrict__ Y,
                          int64_t ld_y) {
  ptx::griddep_wait_for(X, gamma, beta);
  ptx::griddep_launch_dependents();
  const int lane = threadIdx.x % 32;
  const int64_t warp = (int64_t)blockIdx.x * kWarpsPerBlock + threadIdx.x / 32;
  const int64_t n_warps = (int64_t)gridDim.x * kWarpsPerBlock;
  for (int64_t row = warp; row < M; row += n_warps) {
    const T* x = X + row * ld_x;
    float mean = 0.f;
    if (kind == ROCS_NORM_LAYER) {
      float s = 0.f;
      for (int e = lane; e < d; e += 32) s += ld_f(x, e);
      mean = warp_sum(s) / d;
    }
    float sq = 0.f;
    for (int e = lane; e < d; e += 32) {
      const float c = ld_f(x, e) - mean;
      sq = fmaf(c, c, sq);
    }
    const float inv = rsqrtf(warp_sum(sq) / d + eps);
    for (int e = lane; e < d; e += 32) {
      const float g = gamma ? ld_f(gamma, e) : 1.f;
      const float b = (beta && kind == ROCS_NORM_LAYER) ? ld_f(beta, e) : 0.f;
      st_f(Y, row * ld_y + e, fmaf((ld_f(x, e) - mean) * inv, g, b));
    }
  }
}

int sm_count_norm() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  }
  return n;
}

template <typename T>
rocs_status_t launch_norm(int kind, int64_t M, int32_t d, const void* X, int64_t ld_x, const void* gamma,
                          const void* beta, float eps, void* Y, int64_t ld_y, cudaStream_t stream) {
  if (M == 0) return ROCS_OK;
  constexpr int E = Vec<T>::kElems;
  const int threads = kWarpsPerBlock * 32;
  auto blocks = [&](int rows_per_warp) {  // 64 resident warps per SM at most
    const int64_t per_block = (int64_t)kWarpsPerBlock * rows_per_warp;
    return dim3((unsigned)std::min<int64_t>((M + per_block - 1) / per_block, (int64_t)sm_count_norm() * 8));
  };
  // Lanes per row and vectors per lane by the width: the fewest that hold the row, so that few lanes idle.  A width that
  // is no multiple of a warp's 512 bytes on the element-wise kernel below took 34.1 us at [51922, 384] bf16 where
  // three vectors on 16 lanes take 13.2 (6.0 TB/s), 20.0 against 8.8 at [40000, 200] and 12.8 against 4.0 at [40000, 64].
  // Two rows in flight per lane group measured 5.4 us for 5.9 at [40000, 128] and 11.2 for 10.4 at [46262, 256]: not taken.
  const int vecs = d % E == 0 && ld_x % E == 0 && ld_y % E == 0 ? d / E : 0;
#define ROCS_NORM_LAUNCH(NV_, G_, FULL_)                                                                              \
  return launch_dependent(group_norm_rows_kernel<T, NV_, G_, FULL_>, blocks(32 / G_), threads, 0, stream, kind, M, d, \
                          (const T*)X, ld_x, (const T*)gamma, (const T*)beta, eps, (T*)Y, ld_y)
#define ROCS_NORM_WIDTH(NV_, G_)                            \
  if (vecs == NV_ * G_) ROCS_NORM_LAUNCH(NV_, G_, true);    \
  if (vecs > 0 && vecs < NV_ * G_) ROCS_NORM_LAUNCH(NV_, G_, false)
  ROCS_NORM_WIDTH(1, 4);
  ROCS_NORM_WIDTH(1, 8);
  ROCS_NORM_WIDTH(1, 16);
  ROCS_NORM_WIDTH(1, 32);
  ROCS_NORM_WIDTH(3, 16);
  ROCS_NORM_WIDTH(2, 32);
  ROCS_NORM_WIDTH(3, 32);
  ROCS_NORM_WIDTH(4, 32);
  ROCS_NORM_WIDTH(6, 32);
  ROCS_NORM_WIDTH(8, 32);
#undef ROCS_NORM_WIDTH
#undef ROCS_NORM_LAUNCH
  return launch_dependent(group_norm_general_kernel<T>, blocks(1), threads, 0, stream, kind, M, d, (const T*)X,
                          ld_x, (const T*)gamma, (const T*)beta, eps, (T*)Y, ld_y);
}

}  // namespace

rocs_status_t group_norm(rocs_dtype_t dt, int kind, int64_t M, int32_t d, const void* X, int64_t ld_x,
                         const void* gamma, const void* beta, float eps, void* Y, int64_t ld_y, cudaStream_t stream) {
  if (dt == ROCS_F32) return launch_norm<float>(kind, M, d, X, ld_x, gamma, beta, eps, Y, ld_y, stream);
  return launch_norm<__nv_bfloat16>(kind, M, d, X, ld_x, gamma, beta, eps, Y, ld_y, stream);
}

}  // namespace rocs
