// General CUDA-core kernels: fp32 FMA arithmetic on fp32 or bf16 storage.  They accept every
// legal shape, carry the fp32 path, and serve bf16 shapes the tensor-core kernels do not take.
// Every output row is produced by a fixed instruction sequence over that row's own inputs, so
// results are bitwise deterministic and independent of neighbouring candidates (Eq. 1).
#include "rocs_internal.h"
#include "simt_util.cuh"
#include "sm100_ptx.cuh"

namespace rocs {
namespace {

__device__ __forceinline__ float ld_f(const float* p, int64_t i) { return p[i]; }
__device__ __forceinline__ float ld_f(const __nv_bfloat16* p, int64_t i) { return __bfloat162float(p[i]); }
__device__ __forceinline__ void st_f(float* p, int64_t i, float v) { p[i] = v; }
__device__ __forceinline__ void st_f(__nv_bfloat16* p, int64_t i, float v) { p[i] = __float2bfloat16_rn(v); }

// ---------------------------------------------------------------------------------------------
// GLM factorization machine (Eq. 9-10) and row-axis compression (Eq. 5-6).
// Request kernel (one block per request): YR = [X^R X^R^T, 0], OR = W_RR YR, and the request
// term ZR = W_CR YR that the candidate kernel adds to every candidate of the request.
// Candidate kernel (one block per candidate): YC = [X^C X^R^T, X^C X^C^T], OC = ZR + W_CC YC.
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
  // a candidate kernel launched behind this one as a programmatic dependent may start now: it streams
  // its own operands and waits for this grid only before it reads ZR
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

template <typename T>
__global__ void __launch_bounds__(128) glm_candidate_simt_kernel(
    int32_t n_r, int32_t n_c, int32_t d, const T* __restrict__ XR, const T* __restrict__ XC,
    const T* __restrict__ W, int32_t n_ro, int32_t n_co, const int32_t* __restrict__ row2req,
    const float* __restrict__ ZR, T* __restrict__ YC, T* __restrict__ OC) {
  extern __shared__ float sm[];
  const int32_t n = n_r + n_c;
  const int32_t ds = d + 1;          // padded row stride: rows land in different banks
  float* x = sm;                     // [n, d + 1]: request rows then candidate rows
  float* yc = sm + (size_t)n * ds;   // [n_c, n]
  const int64_t i = blockIdx.x;
  const int32_t r = row2req[i];
  for (int e = threadIdx.x; e < n_r * d; e += blockDim.x) x[(e / d) * ds + e % d] = ld_f(XR, (int64_t)r * n_r * d + e);
  for (int e = threadIdx.x; e < n_c * d; e += blockDim.x)
    x[(n_r + e / d) * ds + e % d] = ld_f(XC, i * n_c * d + e);
  __syncthreads();
  for (int idx = threadIdx.x; idx < n_c * n; idx += blockDim.x) {
    const int a = idx / n, b = idx % n;
    const float* xa = x + (size_t)(n_r + a) * ds;
    const float* xb = x + (size_t)b * ds;
    float acc = 0.f;
    for (int e = 0; e < d; ++e) acc = fmaf(xa[e], xb[e], acc);
    yc[idx] = acc;
    if (YC) st_f(YC, i * n_c * n + idx, acc);
  }
  if (!W || !OC) return;
  __syncthreads();
  for (int idx = threadIdx.x; idx < n_co * n; idx += blockDim.x) {
    const int o = idx / n, b = idx % n;
    float acc = 0.f;
    for (int a = 0; a < n_c; ++a) acc = fmaf(ld_f(W, (int64_t)(n_ro + o) * n + n_r + a), yc[a * n + b], acc);
    acc += ZR[((int64_t)r * n_co + o) * n + b];
    st_f(OC, (i * n_co + o) * n + b, acc);
  }
}

}  // namespace

template <typename T>
static rocs_status_t launch_glm(const rocs_plan* plan, int32_t n_r, int32_t n_c, int32_t d,
                                const void* XR, const void* XC, const void* W, int32_t n_ro,
                                int32_t n_co, void* YR, void* YC, void* OR_, void* OC, float* zr,
                                bool request_side, bool candidate_side, cudaStream_t stream) {
  const int32_t n = n_r + n_c;
  const size_t smem_r = ((size_t)n_r * (d + 1) + (size_t)n_r * n_r + (size_t)(n_ro + n_co) * n_r) * sizeof(float);
  const size_t smem_c = ((size_t)n * (d + 1) + (size_t)n_c * n) * sizeof(float);
  constexpr size_t kMaxSmem = 200 * 1024;
  if (smem_r > kMaxSmem || smem_c > kMaxSmem) return ROCS_ERR_UNSUPPORTED;
  if (request_side && plan->R > 0) {
    ROCS_CUDA_TRY(cudaFuncSetAttribute(glm_request_simt_kernel<T>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem));
    glm_request_simt_kernel<T><<<plan->R, 256, smem_r, stream>>>(
        n_r, n_c, d, (const T*)XR, (const T*)W, n_ro, n_co, (T*)YR, (T*)OR_, zr);
    ROCS_CUDA_TRY(cudaGetLastError());
  }
  if (candidate_side && plan->N > 0 && (YC || OC)) {
    const int32_t* row2req = nullptr;
    const rocs_status_t st = plan_row2req(plan, stream, &row2req);
    if (st != ROCS_OK) return st;
    ROCS_CUDA_TRY(cudaFuncSetAttribute(glm_candidate_simt_kernel<T>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem));
    glm_candidate_simt_kernel<T><<<(unsigned)plan->N, 128, smem_c, stream>>>(
        n_r, n_c, d, (const T*)XR, (const T*)XC, (const T*)W, n_ro, n_co, row2req, zr, (T*)YC,
        (T*)OC);
    ROCS_CUDA_TRY(cudaGetLastError());
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
    return launch_glm<float>(plan, n_r, n_c, d, XR, XC, W, n_ro, n_co, YR, YC, OR_, OC, zr_workspace,
                             true, true, stream);
  return launch_glm<__nv_bfloat16>(plan, n_r, n_c, d, XR, XC, W, n_ro, n_co, YR, YC, OR_, OC,
                                   zr_workspace, true, true, stream);
}

}  // namespace rocs
