// General CUDA-core kernels: fp32 FMA arithmetic on fp32 or bf16 storage.  They accept every
// legal shape, carry the fp32 path, and serve bf16 shapes the tensor-core kernels do not take.
// Every output row is produced by a fixed instruction sequence over that row's own inputs, so
// results are bitwise deterministic and independent of neighbouring candidates (Eq. 1).
#include <algorithm>

#include "rocs_internal.h"
#include "simt_util.cuh"
#include "sm100_ptx.cuh"

namespace rocs {
namespace {

constexpr int kGlmThreads = 128;

__device__ __forceinline__ float ld_f(const float* p, int64_t i) { return p[i]; }
__device__ __forceinline__ float ld_f(const __nv_bfloat16* p, int64_t i) { return __bfloat162float(p[i]); }
__device__ __forceinline__ void st_f(float* p, int64_t i, float v) { p[i] = v; }
__device__ __forceinline__ void st_f(__nv_bfloat16* p, int64_t i, float v) { p[i] = __float2bfloat16_rn(v); }

// ---------------------------------------------------------------------------------------------
// GLM factorization machine (Eq. 9-10) and row-axis compression (Eq. 5-6).
// Request kernel (one block per request): YR = [X^R X^R^T, 0], OR = W_RR YR, and the request
// term ZR = W_CR YR that the candidate kernel adds to every candidate of the request.
// Candidate kernel (one block per tile of candidates): YC = [X^C X^R^T, X^C X^C^T], OC = ZR + W_CC YC.
// ---------------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) glm_request_simt_kernel(
    int32_t n_r, int32_t n_c, int32_t d, const T* __restrict__ XR, const T* __restrict__ W,
    int32_t n_ro, int32_t n_co, T* __restrict__ YR, T* __restrict__ OR_, float* __restrict__ ZR) {
  extern __shared__ float sm[];
  const int32_t n = n_r + n_c;
  const int32_t ds = d + 1;                    // padded row stride: rows land in different banks
  float* xr = sm;                              // [n_r, d + 1]
  float* g = xr + (size_t)n_r * ds;            // [n_r, n_r]
  float* w = g + (size_t)n_r * n_r;            // [n_ro + n_co, n_r]: the request columns of W
  const int32_t r = blockIdx.x;
  // the candidate kernel launched behind this one may start now: it streams its own operands and waits for this
  // grid only before it reads ZR
  ptx::griddep_wait_for(XR, W);
  ptx::griddep_launch_dependents();
  rows_to_shared(XR + (int64_t)r * n_r * d, xr, n_r, d, ds);
  if (W)
    for (int e = threadIdx.x; e < (n_ro + n_co) * n_r; e += blockDim.x)
      w[e] = ld_f(W, (int64_t)(e / n_r) * n + e % n_r);
  __syncthreads();
  // four neighbouring columns of one row per thread: four independent accumulation chains
  const int n_r4 = (n_r + 3) / 4;
  for (int idx = threadIdx.x; idx < n_r * n_r4; idx += blockDim.x) {
    const int a = idx / n_r4, b0 = (idx % n_r4) * 4;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    const float* xa = xr + a * ds;
    const float* xb[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) xb[u] = xr + min(b0 + u, n_r - 1) * ds;
#pragma unroll 4
    for (int e = 0; e < d; ++e) {
      const float va = xa[e];
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[u] = fmaf(va, xb[u][e], acc[u]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (b0 + u < n_r) g[a * n_r + b0 + u] = acc[u];
  }
  __syncthreads();
  if (YR)
    for (int idx = threadIdx.x; idx < n_r * n; idx += blockDim.x) {
      const int a = idx / n, b = idx % n;
      st_f(YR, (int64_t)r * n_r * n + idx, b < n_r ? g[a * n_r + b] : 0.f);
    }
  if (W) {
    for (int idx = threadIdx.x; idx < (n_ro + n_co) * n; idx += blockDim.x) {
      const int o = idx / n, b = idx % n;
      float acc = 0.f;
      if (b < n_r) {
        float acc1 = 0.f;  // two chains: the sum is short but each step waits for two shared-memory reads
        int a = 0;
        for (; a + 1 < n_r; a += 2) {
          acc = fmaf(w[o * n_r + a], g[a * n_r + b], acc);
          acc1 = fmaf(w[o * n_r + a + 1], g[(a + 1) * n_r + b], acc1);
        }
        if (a < n_r) acc = fmaf(w[o * n_r + a], g[a * n_r + b], acc);
        acc += acc1;
      }
      if (o < n_ro) {
        if (OR_) st_f(OR_, ((int64_t)r * n_ro + o) * n + b, acc);
      } else if (ZR) {
        ZR[((int64_t)r * n_co + (o - n_ro)) * n + b] = acc;
      }
    }
  }
}

// Candidate side: one block per tile of up to `cands_per_tile` candidates of one request, about 64 rows of
// X^C.  The request's rows are staged once per tile, not once per candidate, and a thread computes 4 x 4
// products at a time (eight 16-byte shared-memory reads per 64 FMAs); the products of a candidate's rows
// with the request's rows and with its own are one list of such work items.  What bounds it: the FMA pipe
// and the shared-memory reads on wide rows, HBM only for short ones.  With a
// block per candidate (request rows staged for each, one product per thread and step) 2613 candidates of
// 24 + 8 embeddings x 128, fp32, with compression took 45 us; a pass that holds this kernel is 29 us shorter.
template <typename T>
__global__ void __launch_bounds__(kGlmThreads) glm_candidate_simt_kernel(
    int32_t R, int32_t cands_per_tile, const int32_t* __restrict__ cand_offsets, const Tile* __restrict__ tiles,
    int32_t n_r, int32_t n_c, int32_t d, const T* __restrict__ XR, const T* __restrict__ XC,
    const T* __restrict__ W, int32_t n_ro, int32_t n_co, int32_t w_shared, const float* __restrict__ ZR,
    T* __restrict__ YC, T* __restrict__ OC) {
  extern __shared__ __align__(16) float sm[];
  const int32_t n = n_r + n_c;
  const int32_t ds = d + 4;                                    // row stride: eight rows hit eight bank groups
  float* xr = sm;                                              // [n_r, d + 4]
  float* xc = xr + (size_t)n_r * ds;                           // [cands_per_tile * n_c, d + 4]
  float* yc = xc + (size_t)cands_per_tile * n_c * ds;          // [cands_per_tile * n_c, n]
  float* wc = yc + (size_t)cands_per_tile * n_c * n;           // [n_c, n_co]: W_CC transposed (if w_shared)
  const int tid = threadIdx.x;
  Tile tile;
  if (tiles != nullptr) {
    tile = tiles[blockIdx.x];
  } else {
    const FoundTile f = find_tile_in_block<kGlmThreads>(R, cands_per_tile, 1, cand_offsets, blockIdx.x);
    tile = Tile{f.req, f.cand0, f.count, 0};
  }
  const int32_t rows = tile.count * n_c;
  dense_rows_to_shared_async(XR + (int64_t)tile.req * n_r * d, n_r, d, xr, ds, tid, kGlmThreads);
  dense_rows_to_shared_async(XC + (int64_t)tile.cand0 * n_c * d, rows, d, xc, ds, tid, kGlmThreads);
  cp_async_commit();
  const bool compress = W != nullptr && OC != nullptr && n_co > 0;
  if (compress && w_shared)
    for (int e = tid; e < n_c * n_co; e += kGlmThreads) wc[e] = ld_f(W, (int64_t)(n_ro + e % n_co) * n + n_r + e / n_co);
  cp_async_wait<0>();
  __syncthreads();
  // work items of 4 x 4 products: rows i0 + 4-strided groups keep neighbouring threads on neighbouring rows
  const int32_t rg = (rows + 3) / 4, cg = (n_r + 3) / 4, og = (n_c + 3) / 4;
  const int32_t request_items = rg * cg, items = request_items + tile.count * og * og;
  for (int32_t it = tid; it < items; it += kGlmThreads) {
    // row u of the item is a0 + u * a_step, counted in xc; column v is b0 + v * b_step of xb
    int32_t a0, a_step, a_end, b0, b_step, b_end, col0;
    const float* xb;
    if (it < request_items) {
      a0 = it / cg; a_step = rg; a_end = rows;
      b0 = it % cg; b_step = cg; b_end = n_r; col0 = 0;
      xb = xr;
    } else {
      const int32_t e = it - request_items, c = e / (og * og), o = e % (og * og);
      a0 = c * n_c + o / og; a_step = og; a_end = (c + 1) * n_c;
      b0 = o % og; b_step = og; b_end = n_c; col0 = n_r;
      xb = xc + (size_t)c * n_c * ds;
    }
    const float *pa[4], *pb[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      pa[u] = xc + (size_t)min(a0 + u * a_step, a_end - 1) * ds;
      pb[u] = xb + (size_t)min(b0 + u * b_step, b_end - 1) * ds;
    }
    float acc[4][4] = {};
#pragma unroll 2
    for (int e = 0; e < d; e += 4) {
      float4 a[4], b[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = *reinterpret_cast<const float4*>(pa[u] + e);
#pragma unroll
      for (int u = 0; u < 4; ++u) b[u] = *reinterpret_cast<const float4*>(pb[u] + e);
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          acc[u][v] = fmaf(a[u].x, b[v].x, acc[u][v]);
          acc[u][v] = fmaf(a[u].y, b[v].y, acc[u][v]);
          acc[u][v] = fmaf(a[u].z, b[v].z, acc[u][v]);
          acc[u][v] = fmaf(a[u].w, b[v].w, acc[u][v]);
        }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v)
        if (a0 + u * a_step < a_end && b0 + v * b_step < b_end)
          yc[(a0 + u * a_step) * n + col0 + b0 + v * b_step] = acc[u][v];
  }
  __syncthreads();
  if (YC) {  // the tile's rows are contiguous in the output
    T* out = YC + (int64_t)tile.cand0 * n_c * n;
    for (int32_t e = tid; e < rows * n; e += kGlmThreads) st_f(out, e, yc[e]);
  }
  // Launched beside the request kernel: its ZR is read from here on, and whoever waits for this grid counts on both.
  ptx::griddep_wait();
  if (!compress) return;
  const float* zr = ZR + (int64_t)tile.req * n_co * n;
  T* out = OC + (int64_t)tile.cand0 * n_co * n;
  for (int32_t e = tid; e < tile.count * n; e += kGlmThreads) {
    const int32_t c = e / n, b = e % n;
    const float* y = yc + (size_t)c * n_c * n + b;
    for (int32_t o0 = 0; o0 < n_co; o0 += 4) {
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
      for (int32_t a = 0; a < n_c; ++a) {
        const float v = y[a * n];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int32_t o = min(o0 + u, n_co - 1);
          acc[u] = fmaf(w_shared ? wc[a * n_co + o] : ld_f(W, (int64_t)(n_ro + o) * n + n_r + a), v, acc[u]);
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (o0 + u < n_co) st_f(out, ((int64_t)c * n_co + o0 + u) * n + b, acc[u] + zr[(o0 + u) * n + b]);
    }
  }
}

}  // namespace

template <typename T>
static rocs_status_t launch_glm(const rocs_plan* plan, int32_t n_r, int32_t n_c, int32_t d,
                                const void* XR, const void* XC, const void* W, int32_t n_ro,
                                int32_t n_co, void* YR, void* YC, void* OR_, void* OC, float* zr, cudaStream_t stream) {
  const int32_t n = n_r + n_c;
  const size_t smem_r = ((size_t)n_r * (d + 1) + (size_t)n_r * n_r + (size_t)(n_ro + n_co) * n_r) * sizeof(float);
  int32_t w_shared = 1;  // an unusually large W_CC that does not fit beside the rest stays in global memory
  auto smem_c = [&](int32_t cands) {
    const size_t rows = (size_t)cands * n_c;
    return ((n_r + rows) * (d + 4) + rows * n + (w_shared ? (size_t)n_c * n_co : 0)) * sizeof(float);
  };
  // about 64 rows per tile, fewer where the rows are so wide that less than three blocks would fit an SM
  int32_t cands = n_c > 0 ? std::max(1, 64 / n_c) : 1;
  while (cands > 1 && smem_c(cands) > 72 * 1024) cands /= 2;
  constexpr size_t kMaxSmem = 200 * 1024, kMaxSmemC = 227 * 1024 - 64;  // 64: the tile search's own
  if (smem_c(cands) > kMaxSmemC) w_shared = 0;
  if (smem_r > kMaxSmem || smem_c(cands) > kMaxSmemC) return ROCS_ERR_UNSUPPORTED;
  const bool candidate_side = plan->N > 0 && (YC || OC);
  // the tile list in front of the request kernel: the candidate kernel may start beside that one
  TileList tiles;
  if (candidate_side && plan->R > kGlmThreads) {
    const rocs_status_t st = plan_tiles(plan, cands, stream, &tiles);
    if (st != ROCS_OK) return st;
  } else if (candidate_side) {
    const int64_t total = plan_entries(plan, cands);  // the blocks find their tiles themselves
    tiles.num = (int32_t)total;
  }
  if (plan->R > 0) {
    ROCS_ALLOW_SMEM(glm_request_simt_kernel<T>, kMaxSmem);
    const rocs_status_t st = launch_dependent(glm_request_simt_kernel<T>, dim3((unsigned)plan->R), 256, smem_r, stream, n_r, n_c, d,
                                              (const T*)XR, (const T*)W, n_ro, n_co, (T*)YR, (T*)OR_, zr);
    if (st != ROCS_OK) return st;
  }
  if (candidate_side) {
    auto kernel = glm_candidate_simt_kernel<T>;
    ROCS_ALLOW_SMEM(kernel, kMaxSmemC);
    return launch_dependent(kernel, dim3((unsigned)tiles.num), kGlmThreads, smem_c(cands), stream, plan->R, cands,
                            plan->cand_offsets, (const Tile*)tiles.dev, n_r, n_c, d, (const T*)XR, (const T*)XC, (const T*)W,
                            n_ro, n_co, w_shared, (const float*)zr, (T*)YC, (T*)OC);
  }
  return ROCS_OK;
}

// YC == OC == nullptr runs only the request side (used in front of the tensor-core candidate
// kernel); XC == nullptr is then allowed.
rocs_status_t simt_glm(rocs_dtype_t dt, const rocs_plan* plan, int32_t n_r, int32_t n_c, int32_t d,
                       const void* XR, const void* XC, const void* W, int32_t n_ro, int32_t n_co,
                       void* YR, void* YC, void* OR_, void* OC, float* zr_workspace,
                       cudaStream_t stream) {
  if (dt == ROCS_F32)
    return launch_glm<float>(plan, n_r, n_c, d, XR, XC, W, n_ro, n_co, YR, YC, OR_, OC, zr_workspace, stream);
  return launch_glm<__nv_bfloat16>(plan, n_r, n_c, d, XR, XC, W, n_ro, n_co, YR, YC, OR_, OC,
                                   zr_workspace, stream);
}

}  // namespace rocs
