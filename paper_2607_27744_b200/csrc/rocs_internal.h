// Internal declarations shared by the translation units of librocs.so.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "../../include/rocs.h"

namespace rocs {

// One unit of work of the attention / interaction kernels: `count` consecutive candidates
// of request `req`, starting at candidate row `cand0`.  A tile never crosses a request.
struct Tile {
  int32_t req;
  int32_t cand0;
  int32_t count;
  int32_t pad;
};

struct TileList {
  Tile* dev = nullptr;
  int32_t num = 0;
};

// A list of a plan in device memory, of whatever kind its key says.
struct DeviceList {
  void* dev = nullptr;
  int32_t num = 0;
  bool common = false;  // complete, or made on the plan's stream: for whoever is ordered behind the plan
};

// One unit of work of the attention kernels: one head of `count` consecutive candidates of a request.
struct DcaItem {
  int32_t req;
  int32_t cand0;
  int32_t count;
  int32_t head;
};

struct DcaItemList {
  DcaItem* dev = nullptr;
  int32_t num = 0;
};

}  // namespace rocs

struct rocs_plan {
  int32_t R = 0;
  int64_t N = 0;
  const int32_t* cand_offsets = nullptr;  // device, borrowed
  std::vector<int32_t> offsets_host;      // [R+1]
  mutable std::mutex mu;
  // Device lists, made on first use and kept per stream (its id, which is never reused; 0: complete when it was made):
  // a list is only ever read on the stream whose order puts its making in front of the reader, or, if it is a common one,
  // by a graph captured later.
  // Key: stream id, candidates per tile (0: the candidate -> request map), heads (0: no head dimension).
  using ListKey = std::tuple<unsigned long long, int32_t, int32_t>;
  mutable std::map<ListKey, rocs::DeviceList> lists;
  // The same of calls inside the capture that the plan was created in (by stream: ids cannot be asked for there).  They
  // are memory of the graph, which exists while it runs, and serve no call outside it.
  mutable std::map<ListKey, rocs::DeviceList> captured;
  // List entries by candidates per tile, added up once: a walk over all offsets (540 us for 100000 requests, in a call that
  // tiles them twice), which a plan kept for many calls would take in each of them.
  mutable std::map<int32_t, int64_t> entries;
  int device = 0;
  cudaStream_t stream = nullptr;  // stream the plan was created on; its memory is freed there
  unsigned long long capture = 0; // the capture the plan was created in; 0: none
};

namespace rocs {

#define ROCS_CUDA_TRY(expr)                    \
  do {                                         \
    cudaError_t _e = (expr);                   \
    if (_e != cudaSuccess) return ROCS_ERR_CUDA; \
  } while (0)

// Id of the calling thread's current CUDA context, 0 if it has none yet.  Never reused: what is known about a context
// (an address, an attribute, a pool) goes with its id, and so does not outlive a reset of the device.
unsigned long long context_id();

// Raises a kernel's limit of dynamic shared memory to `bytes` (a constant of the kernel), once per context: the
// attribute stays with the function (setting it again took 0.1 us of every launch, this takes 0.02).
#define ROCS_ALLOW_SMEM(kernel, bytes)                                                                     \
  do {                                                                                                     \
    static std::atomic<unsigned long long> _done{0};                                                       \
    const unsigned long long _context = rocs::context_id();                                                \
    if (_context == 0 || _done.load(std::memory_order_acquire) != _context) {                              \
      ROCS_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(bytes))); \
      _done.store(_context, std::memory_order_release);                                                    \
    }                                                                                                      \
  } while (0)
// Launches a kernel as a programmatic dependent of the one in front of it on the stream.  The kernel must wait for
// that one (griddep_wait) before it touches global memory, and may then release the next, in this order: what is
// released relies on everything in front of its predecessor being complete.  A kernel may read, or write, before its
// wait what was complete, or free, in front of a kernel of the same call that kept to this order (the request half or
// request kernel in front of a candidate kernel).  The request table made beside a request half releases first; nothing
// but that call's candidate half relies on it, and on the request half only.  Every grid waits before it completes.
template <typename... P, typename... A>
inline rocs_status_t launch_dependent(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t stream,
                                      A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  ROCS_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...));
  return ROCS_OK;
}

constexpr int kMaxDynamicSmem = 227 * 1024;  // per block on sm_100

inline size_t elem_size(rocs_dtype_t dt) { return dt == ROCS_BF16 ? 2 : 4; }
inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline size_t round_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Tiles of at most `per` of n candidates.  Unsigned: a request may have all of nearly 2^31.
__host__ __device__ inline int32_t tiles_of(int32_t n, int32_t per) {
  return (int32_t)(((uint32_t)n + (uint32_t)per - 1u) / (uint32_t)per);
}

// Tiles of at most `cands_per_tile` candidates that the batch's requests are cut into; the plan keeps the number.
int64_t plan_entries(const rocs_plan* plan, int32_t cands_per_tile);

// m_i of Section 4.1: a table of all rows, or the offsets to search in; neither: row i is its own request.
struct RequestMap {
  const int32_t* row2req = nullptr;  // [N]
  const int32_t* offsets = nullptr;  // [R + 1]
  int32_t R = 0;
#ifdef __CUDACC__
  __device__ __forceinline__ int32_t of(int64_t row) const {
    if (row2req != nullptr) return row2req[row];
    if (offsets == nullptr) return (int32_t)row;
    int32_t lo = 0, hi = R;  // largest r with offsets[r] <= row
    while (hi - lo > 1) {
      const int32_t mid = lo + (hi - lo) / 2;
      if (offsets[mid] <= row) lo = mid; else hi = mid;
    }
    return lo;
  }
#endif
};
// The same for a thread whose rows ascend.  The end of the request behind is loaded with a request's own, long before
// it is compared with: no load is waited for unless a request is skipped, which takes a search.  For the streaming
// interaction kernel in place of a table, which is a launch of its own: plan and projected interaction of 112 requests
// x 454 candidates 31.8 us with the table, 24.4 us with this (a load of the next end when it is needed: 24.7 us).
struct RequestWalk {
  const int32_t* offsets;  // [R + 1]
  int32_t R;
  int32_t r = -1, end = 0, next_end = -1;
#ifdef __CUDACC__
  __device__ __forceinline__ int32_t of(int64_t row) {
    if (row >= end) {
      if (row < next_end) {
        ++r;
        end = next_end;
      } else {
        r = RequestMap{nullptr, offsets, R}.of(row);
        end = offsets[r + 1];
      }
      next_end = offsets[min(r + 2, R)];
    }
    return r;
  }
#endif
};
// A run of consecutive interaction tiles found in the offsets and walked like the above, in place of the plan's list.
// Making the list is a launch in front of the request kernel, which a small batch feels and a large one does not: a
// block of 8 requests x 697 candidates (attention's list made in its kernel too) 40.0 us with lists and 35.4 without,
// one of 2 x 17 36.4 and 26.0; 128 x 1024 candidates (16384 tiles) 127.0 us with the list and 130.7 walked, the walk
// being on every warp's path from tile to tile (with a third group of epilogue warps 120.7 and 120.5: it is no longer the longest).  (One kernel for both ran the list in 136.4 us for 132.0: two instantiations.)
// Plan and interaction with compression, 32 + 16 embeddings x 128, walked and with the list: 64 requests with 627 / 1230 /
// 2432 / 4826 / 9628 tiles 14.0 / 18.6 / 27.5 / 43.9 / 85.9 us and 17.0 / 20.6 / 28.6 / 44.3 / 82.0 us.  About 2200 tiles of
// 256 / 512 / 768 / 1024 requests 28.3 / 30.9 / 34.0 / 42.1 and 28.8 / 30.8 / 34.5 / 39.0; with 12 embeddings 39.1 / 44.0 /
// - / 62.5 and 39.5 / 42.5 / - / 53.7.
constexpr int32_t kMaxTileWalk = 2400;         // tiles: 16 per CTA, for about half of what the launch costs
constexpr int32_t kMaxTileWalkRequests = 512;  // the first tile takes two loads per 32 requests
struct TileWalk {
  const int32_t* offsets;  // [R + 1]
  int32_t R, per;          // requests, candidates per tile
  Tile next = {0, 0, 0, 0};
  int32_t end = 0, next_end = 0;
#ifdef __CUDACC__
  // Finds tile t; all lanes of a warp take part.
  __device__ __forceinline__ void start(int32_t t, int lane) {
    const int32_t chunk = (R + 31) / 32, r0 = min(lane * chunk, R), r1 = min(r0 + chunk, R);
    int32_t sum = 0;
    for (int32_t r = r0; r < r1; ++r) sum += tiles_of(offsets[r + 1] - offsets[r], per);
    int32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t up = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += up;
    }
    const uint32_t hit = __ballot_sync(0xffffffffu, incl - sum <= t && t < incl);
    if (hit == 0) return;
    const int src = __ffs(hit) - 1;
    int32_t r = __shfl_sync(0xffffffffu, r0, src), local = t - __shfl_sync(0xffffffffu, incl - sum, src), first, n;
    while (true) {
      first = offsets[r];
      end = offsets[r + 1];
      n = tiles_of(end - first, per);
      if (local < n) break;
      local -= n;
      ++r;
    }
    next_end = offsets[min(r + 2, R)];
    const int32_t c = first + local * per;
    next = Tile{r, c, min(per, end - c), 0};
  }
  // The same by all THREADS threads of a block, each with its share of the requests; scratch: THREADS / 32 + 2 words.
  template <int THREADS>
  __device__ __forceinline__ void start_in_block(int32_t t, int32_t* scratch) {
    int32_t *found = scratch, *warp_sum = scratch + 2;
    const int32_t chunk = (R + THREADS - 1) / THREADS, r0 = min((int32_t)threadIdx.x * chunk, R), r1 = min(r0 + chunk, R);
    const int32_t lane = threadIdx.x % 32, w = threadIdx.x / 32;
    int32_t sum = 0;
#pragma unroll 4
    for (int32_t r = r0; r < r1; ++r) sum += tiles_of(offsets[r + 1] - offsets[r], per);
    int32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t up = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += up;
    }
    if (lane == 31) warp_sum[w] = incl;
    __syncthreads();
    int32_t local = t - (incl - sum);
    for (int x = 0; x < w; ++x) local -= warp_sum[x];
    if (0 <= local && local < sum) {
      int32_t r = r0, n;
      while (local >= (n = tiles_of(offsets[r + 1] - offsets[r], per))) {
        local -= n;
        ++r;
      }
      found[0] = r;
      found[1] = offsets[r] + local * per;
    }
    __syncthreads();
    next = Tile{found[0], found[1], 0, 0};
    end = offsets[next.req + 1];
    next_end = offsets[min(next.req + 2, R)];
    next.count = min(per, end - next.cand0);
  }
  // The tile at hand; moves on to the next one if there is `more`.
  __device__ __forceinline__ Tile take(bool more) {
    const Tile t = next;
    if (!more) return t;
    next.cand0 += per;
    while (next.cand0 >= end) {  // the end of a request: on to the next that has candidates
      ++next.req;
      next.cand0 = end;
      end = next_end;
      next_end = offsets[min(next.req + 2, R)];
    }
    next.count = min(per, end - next.cand0);
    return t;
  }
#endif
};
// Up to this many candidates the kernels search for a row's request themselves: the table is a launch of its own (and
// host time), the search a handful of cached loads per row and slice of 256 columns; with more rows the loads add up and the
// launch does not.  Plan and split layer 512|256, about 400 candidates per request, searched and with the table: to 1024
// columns 2048 / 8192 / 16384 / 32768 candidates 11.5 / 15.1 / 20.9 / 33.6 us and 15.6 / 15.1 / 18.4 / 27.4 us, to 512 columns
// 8192 / 12000 / 16384 candidates 11.4 / 15.3 / 16.2 and 15.1 / 15.1 / 15.3, to 256 columns 16384 candidates 11.3 and 15.1.
// The line is between the widths' crossings (8500, 12000 and beyond 16384).
constexpr int64_t kSearchRows = 16384;
rocs_status_t plan_request_map(const rocs_plan* plan, cudaStream_t stream, RequestMap* out);
// The same around a launch that waits for everything in front of itself before it releases the next (a request half):
// begin in front of it, and behind it, where begin gave memory for a table, fill.  The table is made while that kernel runs
// (normalised tower on 46262 candidates of 96 requests: 106.4 us behind it, 105.0 beside it).  The kernel behind must wait
// before it reads the map.
rocs_status_t plan_request_map_begin(const rocs_plan* plan, cudaStream_t stream, RequestMap* out, void** memory);
rocs_status_t plan_request_map_fill(const rocs_plan* plan, cudaStream_t stream, void* memory, RequestMap* out);

// The tiles of a launch whose CTAs take contiguous runs of them: `out` without a list where they can be walked.
rocs_status_t plan_tile_runs(const rocs_plan* plan, int32_t cands_per_tile, cudaStream_t stream, TileList* out);
// Returns the cached tile list for `cands_per_tile`, building it on first use.
rocs_status_t plan_tiles(const rocs_plan* plan, int32_t cands_per_tile, cudaStream_t stream,
                         TileList* out);

// Work items for the attention kernels, ordered request, head, tile; cached in the plan.
rocs_status_t plan_dca_items(const rocs_plan* plan, int32_t cands_per_tile, int32_t heads, cudaStream_t stream,
                             DcaItemList* out);

// ---- general (CUDA-core) kernels: simt_kernels.cu -------------------------------------
// Y[i, :] = act(add[map.of(i), :] + X[i, :] W^T + bias).  out_f32 selects an
// fp32 output regardless of the storage type (used for the request half Z).
rocs_status_t simt_linear(rocs_dtype_t dt, int64_t M, int32_t d_in, int32_t d_out, const void* X,
                          int64_t ld_x, const void* W, int64_t ld_w, const float* bias,
                          const float* add, int64_t ld_add, const RequestMap& map, int act,
                          void* Y, int64_t ld_y, bool out_f32, cudaStream_t stream);
// Both halves of an fp32 split layer in one launch, for few candidates.
bool simt_linear_both_supported(int64_t N, int32_t R, int32_t d_req, int32_t d_out);
rocs_status_t simt_linear_both(const rocs_plan* plan, int32_t d_req, int32_t d_cand, int32_t d_out, const void* XR, int64_t ld_xr,
                               const void* XC, int64_t ld_xc, const void* W_CR, int64_t ld_wcr, const void* W_CC, int64_t ld_wcc,
                               const float* bias, int act, void* Y, int64_t ld_y, cudaStream_t stream);
rocs_status_t simt_dca(rocs_dtype_t dt, const rocs_plan* plan, int32_t n_q, int32_t H, int32_t dh,
                       float scale, const void* Q, const void* K, const void* V,
                       const int32_t* seq_offsets, int64_t T, void* O, cudaStream_t stream);
bool simt_glm_pays(const rocs_plan* plan, int32_t n_r, int32_t n_c, int32_t d, int32_t n_co, bool compress);
rocs_status_t simt_glm(rocs_dtype_t dt, const rocs_plan* plan, int32_t n_r, int32_t n_c, int32_t d,
                       const void* XR, const void* XC, const void* W, int32_t n_ro, int32_t n_co,
                       void* YR, void* YC, void* OR_, void* OC, float* zr_workspace,
                       cudaStream_t stream);

// ---- group-local normalisation (Eq. 7): group_norm.cu -------------------------------------
rocs_status_t group_norm(rocs_dtype_t dt, int kind, int64_t M, int32_t d, const void* X, int64_t ld_x,
                         const void* gamma, const void* beta, float eps, void* Y, int64_t ld_y, cudaStream_t stream);

// ---- projected factorization machine: fm_projection.cu ----------------------------------
// F = G P on the request-once form; tt_workspace [R, k, d] fp32 receives P_R^T X^R per request.
// allow_fast: use the bf16 streaming kernel for the candidate side where the shape allows it.
bool fm_projection_fast_supported(int32_t n_c, int32_t d, int32_t k);
// Candidate rows on tcgen05 (fm_umma.cu), for the shapes above.
bool fm_umma_pays(const rocs_plan* plan, int32_t n_c, int32_t d, int32_t k);
rocs_status_t fm_umma(const rocs_plan* plan, int32_t n_r, int32_t n_c, int32_t d, int32_t k, const void* XC, const void* P,
                      const float* TT, void* FC, cudaStream_t stream);
rocs_status_t fm_projection(rocs_dtype_t dt, const rocs_plan* plan, int32_t n_r, int32_t n_c, int32_t d, int32_t k,
                            const void* XR, const void* XC, const void* P, void* FR, void* FC, float* tt_workspace,
                            bool allow_fast, cudaStream_t stream);

// ---- tcgen05 tensor-core kernels (bf16): umma_*.cu -------------------------------------
bool umma_linear_supported(int64_t M, int32_t d_in, int32_t d_out, int64_t ld_x, int64_t ld_w,
                           int64_t ld_y, bool out_f32);
// add_rows: number of rows of `add` (the requests of the batch); 0 means one row per output row.
// add_from_previous_launch: `add` is written by the launch directly in front of this one on the
// stream (the request half) and nothing else this call reads is; the kernel may then overlap its
// set-up with that launch and waits for it only before it reads `add`.
rocs_status_t umma_linear(int64_t M, int32_t d_in, int32_t d_out, const void* X, int64_t ld_x,
                          const void* W, int64_t ld_w, const float* bias, const float* add,
                          int64_t ld_add, const RequestMap& map, int act, void* Y, int64_t ld_y,
                          bool out_f32, cudaStream_t stream, bool add_from_previous_launch = false,
                          float2* stat_partials = nullptr, int64_t add_rows = 0);
// Both halves of a split layer in one launch, for few candidates; `taken` says whether the batch is one of those.
rocs_status_t umma_linear_both(const rocs_plan* plan, int32_t d_req, int32_t d_cand, int32_t d_out, const void* XR, int64_t ld_xr,
                               const void* XC, int64_t ld_xc, const void* W_CR, int64_t ld_wcr, const void* W_CC, int64_t ld_wcc,
                               const float* bias, int act, void* Y, int64_t ld_y, cudaStream_t stream, bool* taken);
// Weight-stationary kernel on CTA pairs (cta_group::2) for d_in <= 256 and bf16 output: half a weight
// slice per SM, TMA-store epilogue (umma_linear picks it when it applies).
bool umma_linear_ws2_supported(int64_t M, int32_t d_in, int32_t d_out, bool out_f32);
rocs_status_t umma_linear_ws2(int64_t M, int32_t d_in, int32_t d_out, const void* X, int64_t ld_x,
                              const void* W, int64_t ld_w, const float* bias, const float* add,
                              int64_t ld_add, const RequestMap& map, int act, void* Y, int64_t ld_y,
                              cudaStream_t stream, bool add_from_previous_launch = false,
                              float2* stat_partials = nullptr, int64_t add_rows = 0);
// The same with the request half in its launch, where the rows of each CTA pair are of few requests (`taken`).
rocs_status_t umma_linear_ws2_both(const rocs_plan* plan, int32_t d_req, int32_t d_cand, int32_t d_out, const void* XR,
                                   int64_t ld_xr, const void* XC, int64_t ld_xc, const void* W_CR, int64_t ld_wcr, const void* W_CC,
                                   int64_t ld_wcc, const float* bias, int act, void* Y, int64_t ld_y, float2* stat_partials,
                                   cudaStream_t stream, bool* taken);
// Number of (sum, sum of squares) partials per row the kernel above writes when asked to.
inline int32_t umma_linear_ws2_stat_partials(int32_t d_out) { return 2 * ((d_out + 255) / 256); }
// K-ring GEMM on CTA pairs for wide plain layers (no request term, bf16 output, many rows).
bool umma_linear_pair_supported(int64_t M, int32_t d_in, int32_t d_out, bool out_f32, bool has_add);
// norm (optional): the rows of X are to be normalised (Eq. 7) before the product; the kernel applies the
// row's scale and shift to its accumulators instead (see rocs_linear_normed).
struct RowNorm {
  const float2* row_stats = nullptr;  // [M] (sum, sum of squares) over the d_in columns of each row of X
  int kind = 0;                       // ROCS_NORM_LAYER / ROCS_NORM_RMS
  float eps = 0.f;
  const float* wbar = nullptr;        // [d_out] row sums of W (LayerNorm only)
};
rocs_status_t umma_linear_pair(int64_t M, int32_t d_in, int32_t d_out, const void* X, int64_t ld_x,
                               const void* W, int64_t ld_w, const float* bias, int act, void* Y,
                               int64_t ld_y, cudaStream_t stream, const RowNorm* norm = nullptr);

// ---- per-row sums for a normalisation fused into the next layer: row_stats.cu ---------------------
rocs_status_t row_stats_from_partials(int64_t M, int32_t partials_per_row, const float2* partials, float2* row_stats,
                                      cudaStream_t stream);
rocs_status_t row_stats_direct(rocs_dtype_t dt, int64_t M, int32_t d, const void* Y, int64_t ld_y, float2* row_stats,
                               cudaStream_t stream);
rocs_status_t weight_row_sums(rocs_dtype_t dt, int32_t d_out, int32_t d_in, const void* W, int64_t ld_w, float* wbar,
                              cudaStream_t stream);
bool umma_dca_supported(int32_t n_q, int32_t H, int32_t dh);
rocs_status_t umma_dca(const rocs_plan* plan, int32_t n_q, int32_t H, int32_t dh, float scale,
                       const void* Q, const void* K, const void* V, const int32_t* seq_offsets,
                       int64_t T, void* O, cudaStream_t stream);
// Candidate side of the interaction operator (bf16).  glm_mma: warp-level tensor cores, 4 to 16 embeddings per
// candidate; its tile list can be made in front of the request kernel.  umma_glm: 8, 16 or 32, the faster of the two.
bool glm_mma_supported(int32_t n_r, int32_t n_c, int32_t d, int32_t n_co);
rocs_status_t glm_mma_tiles(const rocs_plan* plan, int32_t n_r, int32_t n_c, int32_t d, cudaStream_t stream, TileList* out);
rocs_status_t glm_mma(const rocs_plan* plan, int32_t n_r, int32_t n_c, int32_t d, const void* XR, const void* XC,
                      const void* W, int32_t n_ro, int32_t n_co, void* YC, void* OC, const float* zr_workspace,
                      cudaStream_t stream);
bool umma_glm_supported(int32_t n_r, int32_t n_c, int32_t d, int32_t n_ro, int32_t n_co);
rocs_status_t umma_glm(const rocs_plan* plan, int32_t n_r, int32_t n_c, int32_t d, const void* XR,
                       const void* XC, const void* W, int32_t n_ro, int32_t n_co, void* YC,
                       void* OC, const float* zr_workspace, cudaStream_t stream);

// Request side of the interaction operator on warp-level tensor cores (bf16): YR, OR and the request
// term ZR of the compression, one block per request.
bool glm_request_mma_supported(int32_t n_r, int32_t d, int32_t n_ro, int32_t n_co);
rocs_status_t glm_request_mma(const rocs_plan* plan, int32_t n_r, int32_t n_c, int32_t d, const void* XR,
                              const void* W, int32_t n_ro, int32_t n_co, void* YR, void* OR_, float* zr,
                              cudaStream_t stream);

// Device status word written by bounded waits of the tensor-core kernels.
uint32_t* device_status_word();

}  // namespace rocs
