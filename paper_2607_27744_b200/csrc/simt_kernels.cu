// General CUDA-core kernels: fp32 FMA arithmetic on fp32 or bf16 storage.  They accept every
// legal shape, carry the fp32 path, and serve bf16 shapes the tensor-core kernels do not take.
// An output row is produced from its own inputs alone, in a sequence that the batch's shape fixes (how many lanes share a product,
// and whether the request term is W (X X^T) or (W X) X^T, follow from the number of candidates): for a batch of given shape
// results are bitwise deterministic and independent of the other candidates' values (Eq. 1).
#include <algorithm>

#include "rocs_internal.h"
#include "simt_util.cuh"
#include "sm100_ptx.cuh"

namespace rocs {
namespace {

constexpr int kGlmThreads = 128;
// Tiles (of about 64 rows) of a small batch, whose blocks have tiles of fewer candidates and share the lanes out over K, and
// of one whose request side is not worth a launch of its own (2613 candidates of 24 requests, 24 + 8 x 128, compression to
// 4 + 4, 337 tiles: 14.1 us with that launch, 17.0 without).  fp32, 25 candidates of one request, 32 + 2 embeddings x 128,
// compression to 8 + 8: 15.7 us before both, 6.1 us; 288 candidates of 32 + 8: 15.2 and 8.6 us.
constexpr int32_t kGlmSmallTiles = 296, kGlmFusedTiles = 148;

__device__ __forceinline__ float ld_f(const float* p, int64_t i) { return p[i]; }
__device__ __forceinline__ float ld_f(const __nv_bfloat16* p, int64_t i) { return __bfloat162float(p[i]); }
__device__ __forceinline__ void st_f(float* p, int64_t i, float v) { p[i] = v; }
__device__ __forceinline__ void st_f(__nv_bfloat16* p, int64_t i, float v) { p[i] = __float2bfloat16_rn(v); }

// ---------------------------------------------------------------------------------------------
// GLM factorization machine (Eq. 9-10) and row-axis compression (Eq. 5-6).
// Request side (one block per request): YR = [X^R X^R^T, 0], OR = W_RR YR, and the request
// term ZR = W_CR YR that the candidate side adds to every candidate of the request.
// Candidate side (one block per tile of candidates): YC = [X^C X^R^T, X^C X^C^T], OC = ZR + W_CC YC.
// ---------------------------------------------------------------------------------------------

// 4 x 4 products over d: rows pa[0..3] by rows pb[0..3], both in shared memory (eight 16-byte reads per 64 FMAs).
// KS > 1: `ks` neighbouring lanes share the item, each takes every ks-th 16 bytes, and all of them get the sums.
template <bool KS>
__device__ __forceinline__ void products_4x4(const float* const (&pa)[4], const float* const (&pb)[4], int32_t d, int32_t ks,
                                             int32_t part, float (&acc)[4][4]) {
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[u][v] = 0.f;
#pragma unroll 2
  for (int32_t e = KS ? 4 * part : 0; e < d; e += KS ? 4 * ks : 4) {
    float4 a[4], b[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) a[u] = *reinterpret_cast<const float4*>(pa[u] + e);
#pragma unroll
    for (int u = 0; u < 4; ++u) b[u] = *reinterpret_cast<const float4*>(pb[u] + e);
#pragma unroll
    for (int c = 0; c < 4; ++c)  // 16 independent FMAs per column
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(lane_of(a[u], c), lane_of(b[v], c), acc[u][v]);
  }
  if constexpr (KS) {
    for (int o = ks / 2; o > 0; o /= 2)
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] += __shfl_xor_sync(0xffffffffu, acc[u][v], o);
  }
}
// Lanes per item of 4 x 4 products, so that about all threads of the block have some.
__host__ __device__ inline int32_t lanes_per_item(int32_t items, int32_t threads) {
  int32_t ks = 1;
  while (ks < 8 && items * ks * 2 <= threads) ks *= 2;
  return ks;
}

// The request side of request r, by all THREADS threads of a block.  sm: xr [n_r, d + 4], g [n_r, n_r],
// w [n_ro + n_co, n_r].  One 4 x 4 item per 1 to 8 lanes and four outputs of a column of W YR per thread: with one
// product per thread and step over d, and one output at a time, a request of 32 embeddings x 128 took about 6 us.
template <typename T, int THREADS>
__device__ void glm_request_side(int32_t r, int32_t n_r, int32_t n_c, int32_t d, const T* __restrict__ XR,
                                 const T* __restrict__ W, int32_t n_ro, int32_t n_co, T* __restrict__ YR,
                                 T* __restrict__ OR_, float* __restrict__ ZR, float* sm) {
  const int32_t n = n_r + n_c, ds = d + 4, tid = threadIdx.x;
  const int32_t n_o = W != nullptr ? (ZR != nullptr ? n_ro + n_co : n_ro) : 0;  // rows of W that are asked for
  float* xr = sm;
  float* g = xr + (size_t)n_r * ds;
  float* w = g + (size_t)n_r * n_r;
  dense_rows_to_shared_async(XR + (int64_t)r * n_r * d, n_r, d, xr, ds, tid, THREADS);
  cp_async_commit();
  for (int32_t e = tid; e < n_o * n_r; e += THREADS) w[e] = ld_f(W, (int64_t)(e / n_r) * n + e % n_r);
  cp_async_wait<0>();
  __syncthreads();
  const int32_t q = (n_r + 3) / 4, items = q * q, ks = lanes_per_item(items, THREADS), part = tid % ks;
  for (int32_t i0 = 0; i0 < items; i0 += THREADS / ks) {
    const int32_t it = min(i0 + tid / ks, items - 1), a0 = it / q, b0 = it % q;
    const float *pa[4], *pb[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      pa[u] = xr + (size_t)min(a0 + u * q, n_r - 1) * ds;
      pb[u] = xr + (size_t)min(b0 + u * q, n_r - 1) * ds;
    }
    float acc[4][4];
    products_4x4<true>(pa, pb, d, ks, part, acc);
    if (i0 + tid / ks < items)
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v)
          if ((u * 4 + v) % ks == part && a0 + u * q < n_r && b0 + v * q < n_r) g[(a0 + u * q) * n_r + b0 + v * q] = acc[u][v];
  }
  __syncthreads();
  if (YR)
    for (int32_t idx = tid; idx < n_r * n; idx += THREADS) {
      const int32_t a = idx / n, b = idx % n;
      st_f(YR, (int64_t)r * n_r * n + idx, b < n_r ? g[a * n_r + b] : 0.f);
    }
  for (int32_t idx = tid; idx < (n_o + 3) / 4 * n; idx += THREADS) {
    const int32_t o0 = idx / n * 4, b = idx % n;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    if (b < n_r) {
      const float* wo[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) wo[u] = w + min(o0 + u, n_o - 1) * n_r;
#pragma unroll 4
      for (int32_t a = 0; a < n_r; ++a) {
        const float v = g[a * n_r + b];
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[u] = fmaf(wo[u][a], v, acc[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int32_t o = o0 + u;
      if (o >= n_o) break;
      if (o < n_ro) {
        if (OR_) st_f(OR_, ((int64_t)r * n_ro + o) * n + b, acc[u]);
      } else {
        ZR[((int64_t)r * n_co + (o - n_ro)) * n + b] = acc[u];
      }
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(256) glm_request_simt_kernel(
    int32_t n_r, int32_t n_c, int32_t d, const T* __restrict__ XR, const T* __restrict__ W,
    int32_t n_ro, int32_t n_co, T* __restrict__ YR, T* __restrict__ OR_, float* __restrict__ ZR) {
  extern __shared__ __align__(16) float sm[];
  // the candidate kernel launched behind this one may start now: it streams its own operands and waits for this
  // grid only before it reads ZR
  ptx::griddep_wait_for(XR, W);
  ptx::griddep_launch_dependents();
  glm_request_side<T, 256>(blockIdx.x, n_r, n_c, d, XR, W, n_ro, n_co, YR, OR_, ZR, sm);
}

// Candidate side: one block per tile of up to `cands_per_tile` candidates of one request, about 64 rows of
// X^C.  The request's rows are staged once per tile, not once per candidate, and a thread computes 4 x 4
// products at a time; the products of a candidate's rows with the request's rows and with its own are one list of
// such work items.  What bounds it: the FMA pipe
// and the shared-memory reads on wide rows, HBM only for short ones.  With a
// block per candidate (request rows staged for each, one product per thread and step) 2613 candidates of
// 24 + 8 embeddings x 128, fp32, with compression took 45 us; a pass that holds this kernel is 29 us shorter.
//
// FUSED: the first R blocks are the request side, and a tile makes the request term of its own request:
// ZR = W_CR (X^R X^R^T) = (W_CR X^R) X^R^T, where the n_co rows W_CR X^R stand behind the tile's rows of X^C and are
// multiplied like them.  One launch instead of two, at 2 n_co n_r d more products per tile.
template <typename T, bool FUSED, bool KS>
__global__ void __launch_bounds__(kGlmThreads) glm_candidate_simt_kernel(
    int32_t R, int32_t cands_per_tile, const int32_t* __restrict__ cand_offsets, const Tile* __restrict__ tiles,
    int32_t n_r, int32_t n_c, int32_t d, const T* __restrict__ XR, const T* __restrict__ XC,
    const T* __restrict__ W, int32_t n_ro, int32_t n_co, int32_t w_shared, const float* __restrict__ ZR,
    T* __restrict__ YR, T* __restrict__ YC, T* __restrict__ OR_, T* __restrict__ OC) {
  extern __shared__ __align__(16) float sm[];
  const int32_t n = n_r + n_c;
  const bool compress = W != nullptr && OC != nullptr && n_co > 0;
  const int32_t extra = FUSED && compress ? n_co : 0;          // rows of W_CR X^R
  const int32_t ds = d + 4;                                    // row stride: eight rows hit eight bank groups
  const int32_t max_rows = cands_per_tile * n_c + extra;
  float* xr = sm;                                              // [n_r, d + 4]
  float* xc = xr + (size_t)n_r * ds;                           // [max_rows, d + 4]
  float* yc = xc + (size_t)max_rows * ds;                      // [max_rows, n]
  float* wc = yc + (size_t)max_rows * n;                       // [n_c, n_co]: W_CC transposed (if w_shared)
  float* wr = wc + (w_shared ? (size_t)n_c * n_co : 0);        // [n_co, n_r]: W_CR (extra)
  const int tid = threadIdx.x;
  int32_t block = blockIdx.x;
  if constexpr (FUSED) {  // the call's first launch: the one in front may be what writes its inputs
    ptx::griddep_wait_for(XR, XC, W, cand_offsets, tiles);
    ptx::griddep_launch_dependents();
    if (block < R) {
      glm_request_side<T, kGlmThreads>(block, n_r, n_c, d, XR, W, n_ro, n_co, YR, OR_, nullptr, sm);
      return;
    }
    block -= R;
  }
  Tile tile;
  if (tiles != nullptr) {
    tile = tiles[block];
  } else {
    const FoundTile f = find_tile_in_block<kGlmThreads>(R, cands_per_tile, 1, cand_offsets, block);
    tile = Tile{f.req, f.cand0, f.count, 0};
  }
  const int32_t rows = tile.count * n_c;
  dense_rows_to_shared_async(XR + (int64_t)tile.req * n_r * d, n_r, d, xr, ds, tid, kGlmThreads);
  dense_rows_to_shared_async(XC + (int64_t)tile.cand0 * n_c * d, rows, d, xc, ds, tid, kGlmThreads);
  cp_async_commit();
  if (compress && w_shared)
    for (int e = tid; e < n_c * n_co; e += kGlmThreads) wc[e] = ld_f(W, (int64_t)(n_ro + e % n_co) * n + n_r + e / n_co);
  if (extra > 0)
    for (int e = tid; e < extra * n_r; e += kGlmThreads) wr[e] = ld_f(W, (int64_t)(n_ro + e / n_r) * n + e % n_r);
  cp_async_wait<0>();
  __syncthreads();
  if (extra > 0) {  // two rows by four columns of W_CR X^R per thread
    const int32_t d4 = d / 4;
    for (int32_t it = tid; it < (extra + 1) / 2 * d4; it += kGlmThreads) {
      const int32_t o = it / d4 * 2, e = it % d4 * 4;
      const float *w0 = wr + o * n_r, *w1 = wr + min(o + 1, extra - 1) * n_r;
      float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0;
#pragma unroll 4
      for (int32_t a = 0; a < n_r; ++a) {
        const float4 x = *reinterpret_cast<const float4*>(xr + (size_t)a * ds + e);
        const float u = w0[a], v = w1[a];
        s0.x = fmaf(u, x.x, s0.x); s0.y = fmaf(u, x.y, s0.y); s0.z = fmaf(u, x.z, s0.z); s0.w = fmaf(u, x.w, s0.w);
        s1.x = fmaf(v, x.x, s1.x); s1.y = fmaf(v, x.y, s1.y); s1.z = fmaf(v, x.z, s1.z); s1.w = fmaf(v, x.w, s1.w);
      }
      float* to = xc + (size_t)(rows + o) * ds + e;
      *reinterpret_cast<float4*>(to) = s0;
      if (o + 1 < extra) *reinterpret_cast<float4*>(to + ds) = s1;
    }
    __syncthreads();
  }
  // work items of 4 x 4 products: rows i0 + 4-strided groups keep neighbouring threads on neighbouring rows
  const int32_t all_rows = rows + extra;
  const int32_t rg = (all_rows + 3) / 4, cg = (n_r + 3) / 4, og = (n_c + 3) / 4;
  const int32_t request_items = rg * cg, items = request_items + tile.count * og * og;
  const int32_t ks = KS ? lanes_per_item(items, kGlmThreads) : 1, part = KS ? tid % ks : 0, per_round = kGlmThreads / ks;
  for (int32_t i0 = 0; i0 < items; i0 += per_round) {
    const bool mine = i0 + tid / ks < items;
    if (!KS && !mine) break;
    const int32_t it = min(i0 + tid / ks, items - 1);
    // row u of the item is a0 + u * a_step, counted in xc; column v is b0 + v * b_step of xb
    int32_t a0, a_step, a_end, b0, b_step, b_end, col0;
    const float* xb;
    if (it < request_items) {
      a0 = it / cg; a_step = rg; a_end = all_rows;
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
    float acc[4][4];
    products_4x4<KS>(pa, pb, d, ks, part, acc);
    if (mine)
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v)
          if ((!KS || (u * 4 + v) % ks == part) && a0 + u * a_step < a_end && b0 + v * b_step < b_end)
            yc[(a0 + u * a_step) * n + col0 + b0 + v * b_step] = acc[u][v];
  }
  __syncthreads();
  if (YC) {  // the tile's rows are contiguous in the output
    T* out = YC + (int64_t)tile.cand0 * n_c * n;
    for (int32_t e = tid; e < rows * n; e += kGlmThreads) st_f(out, e, yc[e]);
  }
  // Launched beside the request kernel: its ZR is read from here on, and whoever waits for this grid counts on both.
  if constexpr (!FUSED) ptx::griddep_wait_for(ZR);
  if (!compress) return;
  const float* zr = FUSED ? yc + (size_t)rows * n : ZR + (int64_t)tile.req * n_co * n;  // FUSED: columns of requests only
  const int32_t zr_cols = FUSED ? n_r : n;
  T* out = OC + (int64_t)tile.cand0 * n_co * n;
  const int32_t n_og = FUSED ? (n_co + 3) / 4 : 1;  // few candidates: a thread per four outputs of a column
  for (int32_t e = tid; e < tile.count * n * n_og; e += kGlmThreads) {
    const int32_t c = e / (n * n_og), x = e % (n * n_og), b = x % n;
    const float* y = yc + (size_t)c * n_c * n + b;
    for (int32_t o0 = x / n * 4; o0 < (FUSED ? x / n * 4 + 4 : n_co); o0 += 4) {
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
        if (o0 + u < n_co) st_f(out, ((int64_t)c * n_co + o0 + u) * n + b, b < zr_cols ? acc[u] + zr[(o0 + u) * n + b] : acc[u]);
    }
  }
}

}  // namespace

template <typename T>
static rocs_status_t launch_glm(const rocs_plan* plan, int32_t n_r, int32_t n_c, int32_t d,
                                const void* XR, const void* XC, const void* W, int32_t n_ro,
                                int32_t n_co, void* YR, void* YC, void* OR_, void* OC, float* zr, cudaStream_t stream) {
  const int32_t n = n_r + n_c;
  const size_t smem_r = ((size_t)n_r * (d + 4) + (size_t)n_r * n_r + (size_t)(n_ro + n_co) * n_r) * sizeof(float);
  const bool candidate_side = plan->N > 0 && (YC || OC);
  const bool compress = W != nullptr && OC != nullptr && n_co > 0;
  int32_t w_shared = 1;  // an unusually large W_CC that does not fit beside the rest stays in global memory
  auto smem_c = [&](int32_t cands, bool fused) {
    const size_t extra = fused && compress ? n_co : 0, rows = (size_t)cands * n_c + extra;
    return ((n_r + rows) * (d + 4) + rows * n + (w_shared ? (size_t)n_c * n_co : 0) + extra * n_r) * sizeof(float);
  };
  // about 64 rows per tile, fewer where the rows are so wide that less than three blocks would fit an SM
  int32_t cands = n_c > 0 ? std::max(1, 64 / n_c) : 1;
  while (cands > 1 && smem_c(cands, false) > 72 * 1024) cands /= 2;
  // the limit of the request side counts rows of d + 1 values, which they once had
  constexpr size_t kMaxSmem = 200 * 1024, kMaxSmemC = 227 * 1024 - 64;  // 64: the tile search's own
  if (smem_c(cands, false) > kMaxSmemC) w_shared = 0;
  if (smem_r - 12 * (size_t)n_r > kMaxSmem || smem_c(cands, false) > kMaxSmemC) return ROCS_ERR_UNSUPPORTED;
  // A small batch: tiles of fewer candidates while SMs are left over, the lanes of a block shared out over K.
  const int32_t full = cands;
  const bool small = plan->N < (int64_t)kGlmSmallTiles * full;
  while (cands > 1 && plan->N < (int64_t)kGlmSmallTiles / 2 * cands) cands /= 2;
  const bool fused = candidate_side && plan->R > 0 && plan->R <= kGlmThreads && w_shared != 0 && (!compress || plan->N < (int64_t)kGlmFusedTiles * full) &&
                     std::max(smem_c(cands, true), smem_r) <= kMaxSmemC;
  // the tile list in front of the request kernel: the candidate kernel may start beside that one
  TileList tiles;
  if (candidate_side && plan->R > kGlmThreads) {
    const rocs_status_t st = plan_tiles(plan, cands, stream, &tiles);
    if (st != ROCS_OK) return st;
  } else if (candidate_side) {
    const int64_t total = plan_entries(plan, cands);  // the blocks find their tiles themselves
    tiles.num = (int32_t)total;
  }
  if (plan->R > 0 && !fused) {
    ROCS_ALLOW_SMEM(glm_request_simt_kernel<T>, kMaxDynamicSmem);
    const rocs_status_t st = launch_dependent(glm_request_simt_kernel<T>, dim3((unsigned)plan->R), 256, smem_r, stream, n_r, n_c, d,
                                              (const T*)XR, (const T*)W, n_ro, n_co, (T*)YR, (T*)OR_, zr);
    if (st != ROCS_OK) return st;
  }
  if (!candidate_side) return ROCS_OK;
#define ROCS_LAUNCH(FUSED_, KS_)                                                                                       \
  do {                                                                                                                 \
    auto kernel = glm_candidate_simt_kernel<T, FUSED_, KS_>;                                                           \
    ROCS_ALLOW_SMEM(kernel, kMaxSmemC);                                                                                \
    return launch_dependent(kernel, dim3((unsigned)(tiles.num + (FUSED_ ? plan->R : 0))), kGlmThreads,                 \
                            FUSED_ ? std::max(smem_c(cands, true), smem_r) : smem_c(cands, false), stream, plan->R, cands,  \
                            plan->cand_offsets, (const Tile*)tiles.dev, n_r, n_c, d, (const T*)XR, (const T*)XC,       \
                            (const T*)W, n_ro, n_co, w_shared, (const float*)zr, (T*)YR, (T*)YC, (T*)OR_, (T*)OC);     \
  } while (0)
  if (fused && small) ROCS_LAUNCH(true, true);
  if (fused) ROCS_LAUNCH(true, false);
  if (small) ROCS_LAUNCH(false, true);
  ROCS_LAUNCH(false, false);
#undef ROCS_LAUNCH
}

// Where a small bf16 batch is faster here than on the tensor-core kernels, which are two launches: few products, and none of the
// chains long that a block's lanes make of a request's own products or of a candidate's (with compression W_CR X^R and its products
// too).  Plan kept, tensor cores and general kernels, us: 20 / 320 / 640 candidates of 24 + 8 embeddings x 128, raw (0.6 / 10 / 20 M
// products), 6.9 / 7.0 / 6.8 and 4.6 / 5.7 / 7.9; 40 / 160 / 320 of 20 + 12 x 64 to 4 + 4 (0.9 / 3.8 / 7.5 M) 6.8 / 6.8 / 6.8 and 5.7 / 6.1 /
// 7.3; 640 of 8 + 4 x 64, raw (1.9 M), 6.8 and 4.1.  Chains, a candidate each of one / of 100 requests, raw: 32 embeddings x 64 / 128 / 192 (32 /
// 64 / 96 steps) 4.9 / 5.1 / 4.5 and 3.9 / 4.7 / 5.7, 6.2 / 6.8 / 6.8 and 4.6 / 6.0 / 7.0; 40 x 64 (64) 5.1 and 5.1, 7.2 and 6.0; 48 x 64 (128) 4.5
// and 7.2, 7.4 and 8.3; 48 x 192 (384) 5.6 and 13.4, 9.2 and 16.2.  To 8 + 8, 8 of one request: 16 + 8 x 128 (32) 6.2 and 6.0, 16 + 16 x
// 128 (64) 5.6 and 7.1, 32 + 16 x 128 7.1 and 7.7.
bool simt_glm_pays(const rocs_plan* plan, int32_t n_r, int32_t n_c, int32_t d, int32_t n_co, bool compress) {
  constexpr int64_t kFewProducts = 1 << 22;
  if (plan->R > kGlmThreads || plan->N * n_c * (n_r + n_c) * d > kFewProducts) return false;
  auto steps = [&](int32_t items) {
    const int32_t ks = lanes_per_item(items, kGlmThreads);
    return (int64_t)((items + kGlmThreads / ks - 1) / (kGlmThreads / ks)) * (d / ks);
  };
  const int32_t q = (n_r + 3) / 4, own = (n_c + 3) / 4, rows = (n_c + (compress ? n_co : 0) + 3) / 4;
  return steps(q * q) <= 64 && steps(rows * q + own * own) <= (compress ? 32 : 64) && (!compress || (int64_t)n_r * d <= 2048);
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
