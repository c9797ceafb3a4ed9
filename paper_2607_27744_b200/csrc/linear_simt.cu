// Linear layer on the CUDA cores (Eq. 4 / Eq. 14):
//     Y[i, n] = act( sum_k X[i, k] W[n, k] + bias[n] + add[map.of(i), n] )
// in fp32 FMA on fp32 or bf16 storage: the fp32 path, and bf16 shapes the tensor-core kernels do not take.
//
// A block computes a BM x BN tile.  Its threads form KS groups of 64 (8 x 8 threads, TM x TN outputs each)
// that take the 16-wide slices of K in turn, each through a three-stage cp.async ring of its own with a
// barrier of its own, and add their partial tiles up in shared memory in a fixed order at the end.
// Operands stay row-major in shared memory (20-float rows): a thread reads four k of a row at once, the
// eight rows a quarter-warp reads hit eight different bank groups.
//
// Which tile (`simt_linear`): the largest that still gives every SM work, since the FMAs per shared-memory
// read fall with it (8 x 8 outputs: 16 FMAs per 16-byte read, 4 x 4: 8, 2 x 2: 4) and what bounds the large
// shapes is the FMA pipe and those reads, while a small batch (the request half at R rows) is bound by the
// length of its K chain on a few SMs.  Measured, fp32: 24 requests x 768 -> 1024 with 2613 candidates x
// 256 -> 1024 behind it, 46 us for both (56 us with the request rows of the epilogue read one at a time and a part's rows
// on the same banks; one 64 x 64 tile of 16-wide synchronous slices for every shape:
// 160 us, half of it the 16 blocks of the request half).
// Every output is produced by a sequence that depends on the batch's shape only, so results are deterministic and
// independent of the other rows' values (Eq. 1).
#include "rocs_internal.h"
#include "simt_util.cuh"
#include "sm100_ptx.cuh"

namespace rocs {
namespace {

constexpr int kBk = 16, kRow = kBk + 4;  // k per slice; floats per shared-memory row
constexpr int kGroup = 64, kStages = 3;

template <int BM, int BN, int KS, bool BOTH>
constexpr int smem_bytes() {
  constexpr int ring = KS * kStages * (BM + BN) * kRow, tiles = (BOTH ? 2 : 1) * KS * BM * (BN + 8);
  return (ring > tiles ? ring : tiles) * (int)sizeof(float);
}

__device__ __forceinline__ float ld_f(const __nv_bfloat16* p) { return __bfloat162float(*p); }
__device__ __forceinline__ void st_f(float* p, float v) { *p = v; }
__device__ __forceinline__ void st_f(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

// 16 columns from k0 of `rows` rows starting at row0 of a matrix, zeros outside it.
__device__ __forceinline__ void load_slice(const float* __restrict__ src, int64_t ld, int64_t row0, int64_t n_rows,
                                           int rows, int32_t k0, int32_t d, float* dst, int t) {
  // thread t has the same four columns of every 16th row
  const int k = k0 + t % 4 * 4, in_row = min(max(d - k, 0), 4);
  const float* from = src + (row0 + t / 4) * ld + k;
  const uint32_t to = (uint32_t)__cvta_generic_to_shared(dst + t / 4 * kRow + t % 4 * 4);
  const int64_t left_rows = n_rows - row0 - t / 4;
#pragma unroll
  for (int r = 0; r < rows; r += kGroup / 4) {
    const int left = r < left_rows ? in_row : 0;
    cp_async_16(to + r * kRow * 4, left > 0 ? from + r * ld : src, left * 4);
  }
}
__device__ __forceinline__ void load_slice(const __nv_bfloat16* __restrict__ src, int64_t ld, int64_t row0,
                                           int64_t n_rows, int rows, int32_t k0, int32_t d, float* dst, int t) {
  for (int v = t; v < rows * (kBk / 8); v += kGroup) {
    const int r = v / (kBk / 8), k = k0 + (v % (kBk / 8)) * 8;
    const int left = row0 + r < n_rows ? min(max(d - k, 0), 8) : 0;
    const __nv_bfloat16* from = src + (row0 + r) * ld + k;
    float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
    if (left == 8) {
      bf16x8_to_f32(__ldg(reinterpret_cast<const uint4*>(from)), lo, hi);
    } else if (left > 0) {
      float f[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) f[e] = e < left ? ld_f(from + e) : 0.f;
      lo = make_float4(f[0], f[1], f[2], f[3]);
      hi = make_float4(f[4], f[5], f[6], f[7]);
    }
    float* to = dst + r * kRow + (v % (kBk / 8)) * 8;
    *reinterpret_cast<float4*>(to) = lo;
    *reinterpret_cast<float4*>(to + 4) = hi;
  }
}

// The request half of a split layer in the same launch (BOTH): rows of X are gathered by request, its sums kept apart.
struct RequestHalf {
  const float *X, *W;
  int64_t ld_x, ld_w;
  int32_t d_in;
};

template <typename TIn, typename TOut, int TM, int TN, int KS, bool BOTH>
__global__ void __launch_bounds__(kGroup* KS, TM == 8 ? 3 : 1) linear_simt_kernel(
    int64_t M, int32_t d_in, int32_t d_out, const TIn* __restrict__ X, int64_t ld_x, const TIn* __restrict__ W,
    int64_t ld_w, const float* __restrict__ bias, const float* __restrict__ add, int64_t ld_add,
    const RequestMap map, int act, TOut* __restrict__ Y, int64_t ld_y, const RequestHalf half) {
  constexpr int BM = 8 * TM, BN = 8 * TN;
  extern __shared__ __align__(16) float sm[];
  __shared__ int32_t req[BM];  // request of each row of the tile
  RequestMap requests = map;
  ptx::griddep_wait_for(X, W, bias, add, requests.row2req, requests.offsets);
  ptx::griddep_launch_dependents();
  const int group = threadIdx.x / kGroup, t = threadIdx.x % kGroup;
  const int tx = t % 8, ty = t / 8;
  const int64_t m0 = (int64_t)blockIdx.x * BM;
  const int32_t n0 = blockIdx.y * BN;
  const int32_t slices = (d_in + kBk - 1) / kBk;
  const int32_t mine = (slices - group + KS - 1) / KS;  // slices group, group + KS, ...
  float* ring = sm + group * kStages * (BM + BN) * kRow;
  // BOTH: the group's slices of the request half come behind those
  const int32_t all = BOTH ? mine + ((half.d_in + kBk - 1) / kBk - group + KS - 1) / KS : mine;
  if constexpr (BOTH) {
    if (threadIdx.x < BM) req[threadIdx.x] = requests.of(min(m0 + threadIdx.x, M - 1));
    __syncthreads();
  }
  auto fetch = [&](int32_t it) {
    if (BOTH && it >= mine && it < all) {
      float* st = ring + (it % kStages) * (BM + BN) * kRow;
      const int32_t k = (group + (it - mine) * KS) * kBk + t % 4 * 4, in_row = min(max(half.d_in - k, 0), 4);
#pragma unroll
      for (int r = 0; r < BM; r += kGroup / 4)
        cp_async_16((uint32_t)__cvta_generic_to_shared(st + (r + t / 4) * kRow + t % 4 * 4),
                    in_row > 0 ? half.X + req[r + t / 4] * half.ld_x + k : half.X, in_row * 4);
      load_slice(half.W, half.ld_w, n0, d_out, BN, k - t % 4 * 4, half.d_in, st + BM * kRow, t);
    } else if (it < mine) {
      float* st = ring + (it % kStages) * (BM + BN) * kRow;
      const int32_t k0 = (group + it * KS) * kBk;
      load_slice(X, ld_x, m0, M, BM, k0, d_in, st, t);
      load_slice(W, ld_w, n0, d_out, BN, k0, d_in, st + BM * kRow, t);
    }
    cp_async_commit();
  };
  auto group_sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(kGroup) : "memory"); };

  float acc[TM][TN], acc_r[BOTH ? TM : 1][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      acc[i][j] = 0.f;
      acc_r[BOTH ? i : 0][j] = 0.f;
    }
  auto multiply = [&](int32_t it, auto& sums) {
    cp_async_wait<kStages - 2>();
    group_sync();  // slice `it` has landed for the group, and everybody is done with slice it - 1
    fetch(it + kStages - 1);
    const float* a_s = ring + (it % kStages) * (BM + BN) * kRow + ty * kRow;
    const float* b_s = ring + (it % kStages) * (BM + BN) * kRow + (BM + tx) * kRow;
#pragma unroll
    for (int k = 0; k < kBk; k += 4) {
      float4 a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = *reinterpret_cast<const float4*>(a_s + i * 8 * kRow + k);
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = *reinterpret_cast<const float4*>(b_s + j * 8 * kRow + k);
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN; ++j) sums[i][j] = fmaf(lane_of(a[i], c), lane_of(b[j], c), sums[i][j]);
    }
  };
#pragma unroll
  for (int s = 0; s < kStages - 1; ++s) fetch(s);
  for (int32_t it = 0; it < mine; ++it) multiply(it, acc);
  if constexpr (BOTH)
    for (int32_t it = mine; it < all; ++it) multiply(it, acc_r);
  if (add && threadIdx.x < BM && m0 + threadIdx.x < M) req[threadIdx.x] = requests.of(m0 + threadIdx.x);
  cp_async_wait<0>();
  __syncthreads();  // the rings become the groups' partial tiles
  constexpr int PS = BN + 8;  // row stride of a partial tile: the 8 x 4 threads of a warp hit 32 different banks
  float* part = sm + group * BM * PS;
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      part[(ty + 8 * i) * PS + tx + 8 * j] = acc[i][j];
      if constexpr (BOTH) part[(KS * BM + ty + 8 * i) * PS + tx + 8 * j] = acc_r[i][j];
    }
  __syncthreads();
  static_assert(!BOTH || BM * BN <= kGroup * KS, "the request half's sums are added up below only");
  if constexpr (BM * BN <= kGroup * KS) {
    // a value per thread: a chain of four-wide sums on few threads was longer (1850 candidates, 64|32 -> 64, fp32:
    // 9.1 us, 8.8 so)
    const int32_t r = threadIdx.x / BN, c = threadIdx.x % BN, n = n0 + c;
    if (r >= BM || m0 + r >= M || n >= d_out) return;
    const float z = add ? add[(int64_t)req[r] * ld_add + n] : 0.f, b = bias ? bias[n] : 0.f;
    float v = sm[r * PS + c], zr = 0.f;
#pragma unroll
    for (int g = 1; g < KS; ++g) v += sm[(g * BM + r) * PS + c];
    if constexpr (BOTH) {
#pragma unroll
      for (int g = 0; g < KS; ++g) zr += sm[((KS + g) * BM + r) * PS + c];
      v += zr + b;
    } else {
      v += b;
      v += z;
    }
    if (act == ROCS_ACT_RELU) v = fmaxf(v, 0.f);
    st_f(Y + (m0 + r) * ld_y + n, v);
  } else {
    // Four neighbouring columns of kRowsEach rows per thread.  The request rows are all asked for before the first is
    // used: one at a time, every row of a tile waited for the L2 cache.
    constexpr int kPerRow = BN / 4, kThreads = kGroup * KS, kRowStep = kThreads / kPerRow, kRowsEach = BM / kRowStep;
    static_assert(kThreads % kPerRow == 0 && BM % kRowStep == 0, "rows of a tile over the threads");
    const int32_t c4 = threadIdx.x % kPerRow * 4, r0 = threadIdx.x / kPerRow, n = n0 + c4;
    const int32_t cols = min(d_out - n, 4);
    if (cols <= 0) return;
    float4 z[kRowsEach];
#pragma unroll
    for (int u = 0; u < kRowsEach; ++u) {
      const int32_t r = r0 + u * kRowStep;
      z[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (add && m0 + r < M) {
        const float* from = add + (int64_t)req[r] * ld_add + n;
        if (cols == 4 && ld_add % 4 == 0) {
          z[u] = *reinterpret_cast<const float4*>(from);
        } else {
          z[u].x = from[0];
          if (cols > 1) z[u].y = from[1];
          if (cols > 2) z[u].z = from[2];
          if (cols > 3) z[u].w = from[3];
        }
      }
    }
    float b4[4] = {0.f, 0.f, 0.f, 0.f};
    if (bias)
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (c < cols) b4[c] = bias[n + c];
#pragma unroll
    for (int u = 0; u < kRowsEach; ++u) {
      const int32_t r = r0 + u * kRowStep;
      if (m0 + r >= M) break;
      float4 v4 = *reinterpret_cast<const float4*>(sm + r * PS + c4);
#pragma unroll
      for (int g = 1; g < KS; ++g) {
        const float4 o = *reinterpret_cast<const float4*>(sm + (g * BM + r) * PS + c4);
        v4.x += o.x; v4.y += o.y; v4.z += o.z; v4.w += o.w;
      }
      float v[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (bias) v[c] += b4[c];
        if (add) v[c] += lane_of(z[u], c);
        if (act == ROCS_ACT_RELU) v[c] = fmaxf(v[c], 0.f);
      }
      TOut* out = Y + (m0 + r) * ld_y + n;  // rows start on 16-byte boundaries and n is a multiple of 4
      if (cols == 4) {
        store_pair(out, v[0], v[1]);
        store_pair(out + 2, v[2], v[3]);
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (c < cols) st_f(out + c, v[c]);
      }
    }
  }
}

template <typename TIn, typename TOut>
rocs_status_t launch_linear(int64_t M, int32_t d_in, int32_t d_out, const void* X, int64_t ld_x, const void* W,
                            int64_t ld_w, const float* bias, const float* add, int64_t ld_add,
                            const RequestMap& map, int act, void* Y, int64_t ld_y, cudaStream_t stream,
                            const RequestHalf* half = nullptr) {
  if (M == 0 || d_out == 0) return ROCS_OK;
  auto tiles = [&](int b) { return ((M + b - 1) / b) * ((d_out + b - 1) / b); };
#define ROCS_LAUNCH(T_, KS_, BOTH_)                                                                               \
  do {                                                                                                            \
    constexpr int smem = smem_bytes<8 * T_, 8 * T_, KS_, BOTH_>();                                                \
    auto kernel = linear_simt_kernel<TIn, TOut, T_, T_, KS_, BOTH_>;                                              \
    ROCS_ALLOW_SMEM(kernel, smem);                                                                                \
    const dim3 grid((unsigned)((M + 8 * T_ - 1) / (8 * T_)), (unsigned)((d_out + 8 * T_ - 1) / (8 * T_)));        \
    return launch_dependent(kernel, grid, kGroup * KS_, smem, stream, M, d_in, d_out, (const TIn*)X, ld_x,        \
                            (const TIn*)W, ld_w, bias, add, ld_add, map, act, (TOut*)Y, ld_y,                     \
                            half ? *half : RequestHalf{});                                                        \
  } while (0)
  if constexpr (sizeof(TIn) == 4) {
    if (half != nullptr) ROCS_LAUNCH(2, 8, true);
  }
  if (tiles(64) >= 296) ROCS_LAUNCH(8, 2, false);
  else if (tiles(32) >= 148) ROCS_LAUNCH(4, 4, false);
  else ROCS_LAUNCH(2, 8, false);
#undef ROCS_LAUNCH
}

}  // namespace

rocs_status_t simt_linear(rocs_dtype_t dt, int64_t M, int32_t d_in, int32_t d_out, const void* X, int64_t ld_x,
                          const void* W, int64_t ld_w, const float* bias, const float* add, int64_t ld_add,
                          const RequestMap& map, int act, void* Y, int64_t ld_y, bool out_f32, cudaStream_t stream) {
  if (dt == ROCS_F32)
    return launch_linear<float, float>(M, d_in, d_out, X, ld_x, W, ld_w, bias, add, ld_add, map, act, Y, ld_y,
                                       stream);
  if (out_f32)
    return launch_linear<__nv_bfloat16, float>(M, d_in, d_out, X, ld_x, W, ld_w, bias, add, ld_add, map, act, Y,
                                               ld_y, stream);
  return launch_linear<__nv_bfloat16, __nv_bfloat16>(M, d_in, d_out, X, ld_x, W, ld_w, bias, add, ld_add, map, act,
                                                     Y, ld_y, stream);
}

// The request half is computed for every candidate: worth it while that is less than a launch.  In a chain, two launches and
// one: 25 x 80 | 64 -> 64 3.6 and 2.5 us (5.7 and 2.8 with the host in front), 341 x 112 | 256 -> 512 9.4 and 11.7.  Nor where a
// request's row is fetched by too many at the same time, its candidates in every block of columns: 64 | 32 -> 64, 800 of 20
// requests 6.2 and 5.3, 64 of one 4.0 and 2.8, 700 of one 5.1 and 8.3; 128 | 64 -> 512, 48 of two 4.6 and 6.7.
bool simt_linear_both_supported(int64_t N, int32_t R, int32_t d_req, int32_t d_out) {
  constexpr int64_t kMost = 1 << 22;
  return N > 0 && N <= kSearchRows && N * d_out <= 4096 * (int64_t)R && N * d_req * d_out <= kMost &&
         ((N + 31) / 32) * ((d_out + 31) / 32) < 148;
}
rocs_status_t simt_linear_both(const rocs_plan* plan, int32_t d_req, int32_t d_cand, int32_t d_out, const void* XR, int64_t ld_xr,
                               const void* XC, int64_t ld_xc, const void* W_CR, int64_t ld_wcr, const void* W_CC, int64_t ld_wcc,
                               const float* bias, int act, void* Y, int64_t ld_y, cudaStream_t stream) {
  const RequestHalf half{(const float*)XR, (const float*)W_CR, ld_xr, ld_wcr, d_req};
  return launch_linear<float, float>(plan->N, d_cand, d_out, XC, ld_xc, W_CC, ld_wcc, bias, nullptr, 0,
                                     RequestMap{nullptr, plan->cand_offsets, plan->R}, act, Y, ld_y, stream, &half);
}

}  // namespace rocs
