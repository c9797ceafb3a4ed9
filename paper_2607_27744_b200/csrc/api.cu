// C ABI of librocs.so: argument validation, the segment plan, and dispatch to the kernels.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <map>
#include <mutex>
#include <new>

#include "rocs_internal.h"
#include "sm100_ptx.cuh"

namespace rocs {
namespace {

std::atomic<int> g_path{ROCS_PATH_AUTO};

// m_i of Section 4.1 from the segment offsets: one thread per candidate, binary search.
// beside: kernels in front may still run, of this call and of other threads' calls that share the stream.  One of them,
// the request half, waited for everything in front of itself before it released the next: the offsets, and all that ever
// used the table's memory, are complete.  (The memory is taken in front of the request half: taken behind it, it could be
// that of another thread's plan whose last kernel still reads it.)  This grid completes behind the kernels in front, so
// that the next need wait for this one only.
__global__ void fill_row2req_kernel(int32_t R, int64_t N, const int32_t* __restrict__ off,
                                    int32_t* __restrict__ row2req, bool beside) {
  if (!beside) ptx::griddep_wait_for(off);
  ptx::griddep_launch_dependents();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N) {
    int32_t lo = 0, hi = R;  // largest r with off[r] <= i
    while (hi - lo > 1) {
      const int32_t mid = lo + (hi - lo) / 2;
      if (off[mid] <= i) lo = mid; else hi = mid;
    }
    row2req[i] = lo;
  }
  if (beside) ptx::griddep_wait();
}

bool row_stride_ok(int64_t ld, int64_t min_cols, rocs_dtype_t dt) {
  return ld >= min_cols && (ld * (int64_t)elem_size(dt)) % 16 == 0;
}

__device__ uint32_t g_device_status;

}  // namespace

// Stream-ordered allocations of the plan's lists (request ids, tiles, items) come from a pool of the library's
// own that keeps up to 1 GiB of freed memory instead of returning it to the driver at the next synchronisation: a
// serving loop builds and drops one plan per batch, and with the default pool's zero release
// threshold every batch would pay the driver's allocation path again.
static cudaError_t pool_alloc(void** ptr, size_t bytes, cudaStream_t stream) {
  static std::mutex mu;
  static std::map<unsigned long long, cudaMemPool_t> pools;  // by context: a reset takes its pool along
  unsigned long long context = context_id();
  cudaError_t e;
  if (context == 0) {  // the thread's first CUDA call: this makes the device's context its own
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess || (e = cudaSetDevice(dev)) != cudaSuccess) return e;
    context = context_id();
  }
  cudaMemPool_t pool = nullptr;
  {
    std::lock_guard<std::mutex> lock(mu);
    auto it = pools.find(context);
    if (it == pools.end()) {
      cudaMemPoolProps props = {};
      props.allocType = cudaMemAllocationTypePinned;
      props.handleTypes = cudaMemHandleTypeNone;
      props.location.type = cudaMemLocationTypeDevice;
      if ((e = cudaGetDevice(&props.location.id)) != cudaSuccess) return e;
      e = cudaMemPoolCreate(&pool, &props);
      if (e != cudaSuccess) return e;
      uint64_t keep = 1ull << 30;
      cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
      pools[context] = pool;
    } else {
      pool = it->second;
    }
  }
  return cudaMallocFromPoolAsync(ptr, bytes, pool, stream);
}

uint32_t* device_status_word() {
  uint32_t* p = nullptr;
  if (cudaGetSymbolAddress((void**)&p, g_device_status) != cudaSuccess) return nullptr;
  return p;
}

// Work lists are expanded on the device from the offsets alone: every block adds up the list entries
// ceil(n_r / cands_per_tile) of the R requests into a prefix array in its shared memory, every entry then
// finds its request by binary search in it.  One launch and no host copy per list: adding up on the host
// also takes a staged copy to the device and an allocation for it (plan + query projection + attention of
// 3 requests x 574 candidates: 49.5 us that way, 42.3 us this way; plan + interaction of 128 x 1024
// candidates: 159.6 and 156.4 us).  All blocks read the same R offsets, from L2; beyond kMaxScan requests
// (the 48 KB of shared memory a block has without asking for more) one block adds up for all, into global
// memory in front of them: under a capture a copy from the host would read this call's host memory at every replay.
constexpr int kListThreads = 256;
constexpr int32_t kMaxScan = 12000;
constexpr int32_t kAddUpRequests = 64;  // requests that are walked sooner than a number is looked up

// Prefix sums of the entries per request in the block's memory; all threads of the block take part.
__device__ void scan_entries(int32_t R, int32_t cands_per_tile, const int32_t* __restrict__ off, int32_t* pre) {
  __shared__ int32_t warp_sum[kListThreads / 32];
  for (int32_t r = threadIdx.x; r < R; r += kListThreads) pre[r] = tiles_of(off[r + 1] - off[r], cands_per_tile);
  __syncthreads();
  const int32_t chunk = (R + kListThreads - 1) / kListThreads;
  const int32_t r0 = min((int32_t)threadIdx.x * chunk, R), r1 = min(r0 + chunk, R);
  int32_t sum = 0;
  for (int32_t r = r0; r < r1; ++r) sum += pre[r];
  int32_t incl = sum;
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += up;
  }
  if (lane == 31) warp_sum[warp] = incl;
  __syncthreads();
  int32_t acc = incl - sum;
  for (int w = 0; w < warp; ++w) acc += warp_sum[w];
  for (int32_t r = r0; r < r1; ++r) {
    const int32_t n = pre[r];
    pre[r] = acc;
    acc += n;
  }
  if (r1 == R && r0 < R) pre[R] = acc;
  __syncthreads();
}

// Entry i of the list is entry `local` of request `req`, which has `per_head` of them for every head.
__device__ __forceinline__ void find_entry(int32_t R, int32_t heads, const int32_t* __restrict__ base, int32_t i,
                                           int32_t& req, int32_t& local, int32_t& per_head) {
  int32_t lo = 0, hi = R;  // largest r with base[r] * heads <= i
  while (hi - lo > 1) {
    const int32_t mid = lo + (hi - lo) / 2;
    if ((int64_t)base[mid] * heads <= i) lo = mid; else hi = mid;
  }
  req = lo;
  local = i - base[lo] * heads;
  per_head = base[lo + 1] - base[lo];
}

// heads == 0: interaction tiles, in the order request, tile.  heads > 0: attention items, in the order
// request, head, tile.  base: prefix sums of the entries per request, or null to add them up here.
__global__ void __launch_bounds__(kListThreads) expand_list_kernel(int32_t R, int32_t total, int32_t cands_per_tile,
                                                                   int32_t heads, const int32_t* __restrict__ off,
                                                                   const int32_t* __restrict__ base,
                                                                   void* __restrict__ out) {
  extern __shared__ int32_t pre[];
  ptx::griddep_wait_for(off, base);
  ptx::griddep_launch_dependents();
  if (base == nullptr) {
    scan_entries(R, cands_per_tile, off, pre);
    base = pre;
  }
  const uint32_t i = blockIdx.x * (uint32_t)kListThreads + threadIdx.x;  // the last block of nearly 2^31 entries reaches past them
  if (i >= (uint32_t)total) return;
  int32_t req, local, per_head;
  find_entry(R, max(heads, 1), base, (int32_t)i, req, local, per_head);
  const int32_t h = local / per_head, t = local % per_head;
  const int32_t c = off[req] + t * cands_per_tile;
  const int32_t count = min(cands_per_tile, off[req + 1] - c);
  if (heads == 0)
    static_cast<Tile*>(out)[i] = Tile{req, c, count, 0};
  else
    static_cast<DcaItem*>(out)[i] = DcaItem{req, c, count, h};
}

__global__ void __launch_bounds__(kListThreads) scan_entries_kernel(int32_t R, int32_t cands_per_tile,
                                                                    const int32_t* __restrict__ off, int32_t* base) {
  ptx::griddep_wait_for(off);
  ptx::griddep_launch_dependents();
  scan_entries(R, cands_per_tile, off, base);
}

static int64_t add_up_entries(const rocs_plan* plan, int32_t cands_per_tile) {
  int64_t entries = 0;
  for (int32_t r = 0; r < plan->R; ++r) entries += tiles_of(plan->offsets_host[r + 1] - plan->offsets_host[r], cands_per_tile);
  return entries;
}
// The caller holds plan->mu.
static int64_t entries_locked(const rocs_plan* plan, int32_t cands_per_tile) {
  if (plan->R <= kAddUpRequests) return add_up_entries(plan, cands_per_tile);
  const auto known = plan->entries.find(cands_per_tile);
  if (known != plan->entries.end()) return known->second;
  return plan->entries[cands_per_tile] = add_up_entries(plan, cands_per_tile);
}

int64_t plan_entries(const rocs_plan* plan, int32_t cands_per_tile) {
  if (plan->R <= kAddUpRequests) return add_up_entries(plan, cands_per_tile);
  std::lock_guard<std::mutex> lock(plan->mu);
  return entries_locked(plan, cands_per_tile);
}

static rocs_status_t fill_table(const rocs_plan* plan, const int32_t* off, int32_t* table, cudaStream_t stream, bool beside) {
  return launch_dependent(fill_row2req_kernel, dim3((unsigned)((plan->N + 255) / 256)), 256, 0, stream, plan->R, plan->N, off,
                          table, beside);
}

// Allocates and fills one list of the plan (key as in rocs_plan::lists) in the order of `stream`, from the
// offsets at `off`.  The caller holds plan->mu.
static rocs_status_t make_list(const rocs_plan* plan, int32_t cands_per_tile, int32_t heads, const int32_t* off,
                               cudaStream_t stream, DeviceList* out) {
  static_assert(sizeof(Tile) == 16 && sizeof(DcaItem) == 16, "list entries");
  DeviceList list;
  if (plan->N > 0 && cands_per_tile == 0) {
    ROCS_CUDA_TRY(pool_alloc(&list.dev, sizeof(int32_t) * (size_t)plan->N, stream));
    if (fill_table(plan, off, static_cast<int32_t*>(list.dev), stream, false) != ROCS_OK) {
      cudaFreeAsync(list.dev, stream);
      return ROCS_ERR_CUDA;
    }
  } else if (plan->N > 0) {
    const int32_t R = plan->R;
    const int64_t total = entries_locked(plan, cands_per_tile) * std::max(heads, 1);
    if (total > 0x7fffffffLL) return ROCS_ERR_UNSUPPORTED;
    list.num = (int32_t)total;
    ROCS_CUDA_TRY(pool_alloc(&list.dev, sizeof(Tile) * (size_t)total, stream));
    int32_t* base_dev = nullptr;
    cudaError_t e = cudaSuccess;
    if (R > kMaxScan) {
      e = pool_alloc((void**)&base_dev, sizeof(int32_t) * ((size_t)R + 1), stream);
      if (e == cudaSuccess &&
          launch_dependent(scan_entries_kernel, dim3(1), kListThreads, 0, stream, R, cands_per_tile, off, base_dev) != ROCS_OK)
        e = cudaErrorUnknown;
    }
    if (e == cudaSuccess &&
        launch_dependent(expand_list_kernel, dim3((unsigned)((total + kListThreads - 1) / kListThreads)), kListThreads,
                         base_dev ? 0 : sizeof(int32_t) * ((size_t)R + 1), stream, R, list.num, cands_per_tile, heads, off,
                         base_dev, list.dev) != ROCS_OK)
      e = cudaErrorUnknown;
    if (base_dev) cudaFreeAsync(base_dev, stream);
    if (e != cudaSuccess) {
      cudaFreeAsync(list.dev, stream);
      return ROCS_ERR_CUDA;
    }
  }
  *out = list;
  return ROCS_OK;
}

// The same list outside any stream capture, complete on return: on a stream of its own, from the plan's host
// copy of the offsets (work in front of the plan's stream may itself be captured and never run).
static rocs_status_t make_list_now(const rocs_plan* plan, int32_t cands_per_tile, int32_t heads, DeviceList* out) {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  ROCS_CUDA_TRY(cudaThreadExchangeStreamCaptureMode(&mode));
  rocs_status_t st = ROCS_ERR_CUDA;
  cudaStream_t own = nullptr;
  int32_t* off = nullptr;
  const size_t bytes = sizeof(int32_t) * plan->offsets_host.size();
  if (cudaStreamCreateWithFlags(&own, cudaStreamNonBlocking) == cudaSuccess) {
    if (pool_alloc((void**)&off, bytes, own) == cudaSuccess) {
      if (cudaMemcpyAsync(off, plan->offsets_host.data(), bytes, cudaMemcpyHostToDevice, own) == cudaSuccess)
        st = make_list(plan, cands_per_tile, heads, off, own, out);
      cudaFreeAsync(off, own);
    }
    if (cudaStreamSynchronize(own) != cudaSuccess) st = ROCS_ERR_CUDA;
    cudaStreamDestroy(own);
  }
  out->common = true;
  cudaThreadExchangeStreamCaptureMode(&mode);
  return st;
}

static unsigned long long capture_of(cudaStream_t stream) {  // 0: the stream is not being captured
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  unsigned long long id = 0;
  if (cudaStreamGetCaptureInfo(stream, &status, &id) != cudaSuccess || status != cudaStreamCaptureStatusActive) {
    cudaGetLastError();
    return 0;
  }
  return id;
}

// The list that a call on `stream` may read, if there is one (`found`), and where one that is made on the stream is kept.
// Under a capture that the plan was not created in there always is one.  The caller holds plan->mu.
struct ListPlace {
  std::map<rocs_plan::ListKey, DeviceList>* lists;
  rocs_plan::ListKey key;
  bool common;
  void keep(DeviceList& list) const {
    list.common = common;
    (*lists)[key] = list;
  }
};
static rocs_status_t find_list(const rocs_plan* plan, int32_t cands_per_tile, int32_t heads, unsigned long long capture,
                               cudaStream_t stream, ListPlace* place, bool* found, DeviceList* out) {
  *found = true;
  if (capture == 0 || capture != plan->capture) {
    // what was complete when it was made serves everybody; a graph that outlives this call, and is launched behind the
    // plan, also takes a list made on the plan's stream, and otherwise one made now and not one that its own replays
    // would allocate
    for (const auto& kv : plan->lists)
      if (std::get<1>(kv.first) == cands_per_tile && std::get<2>(kv.first) == heads && kv.second.common &&
          (capture != 0 || std::get<0>(kv.first) == 0)) {
        *out = kv.second;
        return ROCS_OK;
      }
    if (capture != 0) {
      const rocs_status_t st = make_list_now(plan, cands_per_tile, heads, out);
      if (st == ROCS_OK) plan->lists[std::make_tuple(0ull, cands_per_tile, heads)] = *out;
      return st;
    }
  }
  unsigned long long id = (unsigned long long)reinterpret_cast<uintptr_t>(stream);
  place->lists = &plan->captured;
  place->common = false;
  if (capture == 0) {
    ROCS_CUDA_TRY(cudaStreamGetId(stream, &id));
    place->lists = &plan->lists;
    place->common = plan->capture == 0 && stream == plan->stream;
  }
  place->key = std::make_tuple(id, cands_per_tile, heads);
  auto it = place->lists->find(place->key);
  *found = it != place->lists->end();
  if (*found) *out = it->second;
  return ROCS_OK;
}

static rocs_status_t plan_list(const rocs_plan* plan, int32_t cands_per_tile, int32_t heads, cudaStream_t stream,
                               DeviceList* out) {
  const unsigned long long capture = capture_of(stream);
  std::lock_guard<std::mutex> lock(plan->mu);
  ListPlace place;
  bool found;
  rocs_status_t st = find_list(plan, cands_per_tile, heads, capture, stream, &place, &found, out);
  if (st != ROCS_OK || found) return st;
  st = make_list(plan, cands_per_tile, heads, plan->cand_offsets, stream, out);
  if (st == ROCS_OK) place.keep(*out);
  return st;
}

rocs_status_t plan_request_map(const rocs_plan* plan, cudaStream_t stream, RequestMap* out) {
  *out = RequestMap{};
  if (plan->N <= kSearchRows) {
    out->offsets = plan->cand_offsets;
    out->R = plan->R;
    return ROCS_OK;
  }
  DeviceList list;
  const rocs_status_t st = plan_list(plan, 0, 0, stream, &list);
  out->row2req = static_cast<const int32_t*>(list.dev);
  return st;
}

rocs_status_t plan_request_map_begin(const rocs_plan* plan, cudaStream_t stream, RequestMap* out, void** memory) {
  *memory = nullptr;
  if (plan->N <= kSearchRows) return plan_request_map(plan, stream, out);
  *out = RequestMap{};
  const unsigned long long capture = capture_of(stream);
  {
    std::lock_guard<std::mutex> lock(plan->mu);
    ListPlace place;
    bool found;
    DeviceList list;
    const rocs_status_t st = find_list(plan, 0, 0, capture, stream, &place, &found, &list);
    out->row2req = static_cast<const int32_t*>(list.dev);
    if (st != ROCS_OK || found) return st;
  }
  ROCS_CUDA_TRY(pool_alloc(memory, sizeof(int32_t) * (size_t)plan->N, stream));
  return ROCS_OK;
}

rocs_status_t plan_request_map_fill(const rocs_plan* plan, cudaStream_t stream, void* memory, RequestMap* out) {
  const unsigned long long capture = capture_of(stream);
  std::lock_guard<std::mutex> lock(plan->mu);
  ListPlace place;
  bool found = false;
  DeviceList list;
  rocs_status_t st = find_list(plan, 0, 0, capture, stream, &place, &found, &list);
  if (st == ROCS_OK && !found) {
    st = fill_table(plan, plan->cand_offsets, static_cast<int32_t*>(memory), stream, /*beside=*/true);
    if (st == ROCS_OK) {
      list.dev = memory;
      place.keep(list);
      memory = nullptr;
    }
  }
  if (memory != nullptr) cudaFreeAsync(memory, stream);  // not used: a call of another thread was in front of this one
  out->row2req = static_cast<const int32_t*>(list.dev);
  return st;
}

rocs_status_t plan_tiles(const rocs_plan* plan, int32_t cands_per_tile, cudaStream_t stream, TileList* out) {
  if (cands_per_tile < 1) return ROCS_ERR_INVALID_ARG;
  DeviceList list;
  const rocs_status_t st = plan_list(plan, cands_per_tile, 0, stream, &list);
  *out = TileList{static_cast<Tile*>(list.dev), list.num};
  return st;
}

rocs_status_t plan_tile_runs(const rocs_plan* plan, int32_t cands_per_tile, cudaStream_t stream, TileList* out) {
  if (plan->R > kMaxTileWalkRequests) return plan_tiles(plan, cands_per_tile, stream, out);
  const int64_t total = plan_entries(plan, cands_per_tile);
  if (total > kMaxTileWalk) return plan_tiles(plan, cands_per_tile, stream, out);
  *out = TileList{nullptr, (int32_t)total};
  return ROCS_OK;
}

rocs_status_t plan_dca_items(const rocs_plan* plan, int32_t cands_per_tile, int32_t heads, cudaStream_t stream,
                             DcaItemList* out) {
  if (cands_per_tile < 1 || heads < 1) return ROCS_ERR_INVALID_ARG;
  DeviceList list;
  const rocs_status_t st = plan_list(plan, cands_per_tile, heads, stream, &list);
  *out = DcaItemList{static_cast<DcaItem*>(list.dev), list.num};
  return st;
}

}  // namespace rocs

using namespace rocs;

extern "C" {

const char* rocs_status_string(rocs_status_t s) {
  switch (s) {
    case ROCS_OK: return "ok";
    case ROCS_ERR_INVALID_ARG: return "invalid argument";
    case ROCS_ERR_ALIGNMENT: return "pointer or row stride not 16-byte aligned";
    case ROCS_ERR_UNSUPPORTED: return "unsupported shape";
    case ROCS_ERR_SEGMENTS: return "malformed segment offsets";
    case ROCS_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
    case ROCS_ERR_CUDA: return "CUDA call failed";
    case ROCS_ERR_TIMEOUT: return "bounded device-side wait expired";
    case ROCS_ERR_STATIC_LIMIT: return "problem larger than the fixed scratch array of the no-allocation entry point";
  }
  return "unknown status";
}

int64_t rocs_padded_ld(int64_t n, rocs_dtype_t dtype) {
  const int64_t per16 = 16 / (int64_t)elem_size(dtype);
  return n <= 0 ? 0 : (n + per16 - 1) / per16 * per16;
}

rocs_status_t rocs_set_path(rocs_path_t path) {
  if (path != ROCS_PATH_AUTO && path != ROCS_PATH_GENERAL) return ROCS_ERR_INVALID_ARG;
  g_path.store(path);
  return ROCS_OK;
}

rocs_status_t rocs_plan_create(rocs_plan_t** out, int32_t R, int64_t N, const int32_t* cand_offsets,
                               const int32_t* cand_offsets_host, void* stream_) {
  if (!out) return ROCS_ERR_INVALID_ARG;
  *out = nullptr;
  if (R < 0 || N < 0 || N > 0x7fffffffLL || !cand_offsets) return ROCS_ERR_INVALID_ARG;
  if (R == 0 && N != 0) return ROCS_ERR_SEGMENTS;
  cudaStream_t stream = (cudaStream_t)stream_;
  rocs_plan* p = new (std::nothrow) rocs_plan();
  if (!p) return ROCS_ERR_INVALID_ARG;
  p->R = R;
  p->N = N;
  p->cand_offsets = cand_offsets;
  p->offsets_host.resize((size_t)R + 1);
  if (cand_offsets_host) {
    std::copy(cand_offsets_host, cand_offsets_host + R + 1, p->offsets_host.begin());
  } else {
    if (cudaMemcpyAsync(p->offsets_host.data(), cand_offsets, sizeof(int32_t) * ((size_t)R + 1),
                        cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
        cudaStreamSynchronize(stream) != cudaSuccess) {
      delete p;
      return ROCS_ERR_CUDA;
    }
  }
  const auto& off = p->offsets_host;
  bool ok = off[0] == 0 && off[R] == N;
  for (int32_t r = 0; ok && r < R; ++r) ok = off[r + 1] >= off[r];
  if (!ok) {
    delete p;
    return ROCS_ERR_SEGMENTS;
  }
  if (cudaGetDevice(&p->device) != cudaSuccess) {
    delete p;
    return ROCS_ERR_CUDA;
  }
  {
    // Keep freed plan memory in the device's default pool instead of returning it to the driver
    // at every synchronisation (a per-process setting of the CUDA context, not of the GPU).
    static std::once_flag once[64];
    if (p->device >= 0 && p->device < 64)
      std::call_once(once[p->device], [&] {
        cudaMemPool_t pool;
        if (cudaDeviceGetDefaultMemPool(&pool, p->device) == cudaSuccess) {
          uint64_t keep = 1ull << 30;
          cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
        }
      });
  }
  p->stream = stream;
  p->capture = capture_of(stream);
  *out = p;
  return ROCS_OK;
}

rocs_status_t rocs_plan_destroy(rocs_plan_t* plan) {
  if (!plan) return ROCS_OK;
  rocs_status_t st = ROCS_OK;
  // Freed in stream order behind whatever the caller enqueued on the plan's stream.
  for (const auto* lists : {&plan->captured, &plan->lists})
    for (const auto& kv : *lists)
      if (kv.second.dev && cudaFreeAsync(kv.second.dev, plan->stream) != cudaSuccess) {
        cudaGetLastError();  // of a graph that has not run, or has ended already: not the next call's error
        st = ROCS_ERR_CUDA;
      }
  delete plan;
  return st;
}

size_t rocs_ikbo_linear_workspace(const rocs_plan_t* plan, int32_t d_out) {
  if (!plan || d_out <= 0) return 0;
  return round_up((size_t)plan->R * (size_t)d_out * sizeof(float), 256);
}

static rocs_status_t linear_dispatch(rocs_dtype_t dt, int64_t M, int32_t d_in, int32_t d_out,
                                     const void* X, int64_t ld_x, const void* W, int64_t ld_w,
                                     const float* bias, const float* add, int64_t ld_add,
                                     const RequestMap& map, int act, void* Y, int64_t ld_y,
                                     bool out_f32, cudaStream_t stream,
                                     bool add_from_previous_launch = false, float2* stat_partials = nullptr,
                                     int64_t add_rows = 0) {
  if (dt == ROCS_BF16 && g_path.load() == ROCS_PATH_AUTO &&
      umma_linear_supported(M, d_in, d_out, ld_x, ld_w, ld_y, out_f32))
    return umma_linear(M, d_in, d_out, X, ld_x, W, ld_w, bias, add, ld_add, map, act, Y, ld_y,
                       out_f32, stream, add_from_previous_launch, stat_partials, add_rows);
  return simt_linear(dt, M, d_in, d_out, X, ld_x, W, ld_w, bias, add, ld_add, map, act, Y, ld_y,
                     out_f32, stream);
}

// row_stats (optional): per-row (sum, sum of squares) of the output, for a normalisation folded into
// the next layer; its partials follow Z in the workspace.
static rocs_status_t ikbo_linear_impl(const rocs_plan_t* plan, rocs_dtype_t dtype, int32_t d_req,
                                      int32_t d_cand, int32_t d_out, const void* XR, int64_t ld_xr,
                                      const void* XC, int64_t ld_xc, const void* W_CR, int64_t ld_wcr,
                                      const void* W_CC, int64_t ld_wcc, const float* bias, rocs_act_t act,
                                      void* Y, int64_t ld_y, float* row_stats, void* workspace,
                                      size_t workspace_bytes, void* stream_) {
  if (!plan || (dtype != ROCS_BF16 && dtype != ROCS_F32)) return ROCS_ERR_INVALID_ARG;
  if (d_req < 0 || d_cand < 0 || d_out <= 0 || d_req + d_cand <= 0) return ROCS_ERR_INVALID_ARG;
  if (act != ROCS_ACT_NONE && act != ROCS_ACT_RELU) return ROCS_ERR_INVALID_ARG;
  if ((plan->N > 0 && (!Y || (d_cand > 0 && !XC))) || (d_cand > 0 && !W_CC) ||
      (d_req > 0 && (!W_CR || (plan->R > 0 && !XR))))
    return ROCS_ERR_INVALID_ARG;
  if (!aligned16(Y) || !aligned16(bias) || !row_stride_ok(ld_y, d_out, dtype)) return ROCS_ERR_ALIGNMENT;
  if (d_cand > 0 && (!aligned16(XC) || !aligned16(W_CC) || !row_stride_ok(ld_xc, d_cand, dtype) ||
                     !row_stride_ok(ld_wcc, d_cand, dtype)))
    return ROCS_ERR_ALIGNMENT;
  if (d_req > 0 && (!aligned16(XR) || !aligned16(W_CR) || !row_stride_ok(ld_xr, d_req, dtype) ||
                    !row_stride_ok(ld_wcr, d_req, dtype)))
    return ROCS_ERR_ALIGNMENT;
  cudaStream_t stream = (cudaStream_t)stream_;
  const float* Z = nullptr;
  const size_t z_bytes = d_req > 0 ? rocs_ikbo_linear_workspace(plan, d_out) : 0;
  if (row_stats != nullptr) {
    if (!aligned16(row_stats) || d_cand <= 0) return row_stats && d_cand <= 0 ? ROCS_ERR_INVALID_ARG : ROCS_ERR_ALIGNMENT;
    const size_t need = rocs_ikbo_linear_stats_workspace(plan, d_out);
    if (!workspace || workspace_bytes < need || (reinterpret_cast<uintptr_t>(workspace) & 255u))
      return ROCS_ERR_WORKSPACE;
  }
  RequestMap map;
  if (d_req > 0) {
    const size_t need = z_bytes;
    if (!workspace || workspace_bytes < need || (reinterpret_cast<uintptr_t>(workspace) & 255u))
      return ROCS_ERR_WORKSPACE;
    // Both halves in one launch where the batch allows it: otherwise the candidate half waits for the request half in its
    // epilogue, and the request half holds SMs that the candidate half then starts late on.
    if (dtype == ROCS_BF16 && d_cand > 0 && g_path.load() == ROCS_PATH_AUTO) {
      bool taken = false;
      rocs_status_t st = ROCS_OK;
      if (row_stats == nullptr) {
        st = umma_linear_both(plan, d_req, d_cand, d_out, XR, ld_xr, XC, ld_xc, W_CR, ld_wcr, W_CC, ld_wcc, bias, act, Y, ld_y,
                              stream, &taken);
        if (taken) return st;
      }
      float2* partials = row_stats ? reinterpret_cast<float2*>(static_cast<uint8_t*>(workspace) + z_bytes) : nullptr;
      st = umma_linear_ws2_both(plan, d_req, d_cand, d_out, XR, ld_xr, XC, ld_xc, W_CR, ld_wcr, W_CC, ld_wcc, bias, act, Y, ld_y,
                                partials, stream, &taken);
      if (taken && st == ROCS_OK && row_stats != nullptr)
        st = row_stats_from_partials(plan->N, umma_linear_ws2_stat_partials(d_out), partials, reinterpret_cast<float2*>(row_stats),
                                     stream);
      if (taken) return st;
    }
    if (row_stats == nullptr && dtype == ROCS_F32 && d_cand > 0 && simt_linear_both_supported(plan->N, plan->R, d_req, d_out))
      return simt_linear_both(plan, d_req, d_cand, d_out, XR, ld_xr, XC, ld_xc, W_CR, ld_wcr, W_CC, ld_wcc, bias, act, Y, ld_y, stream);
    // Request half, once per request (Section 4.1): Z = X^R W_CR^T + bias, fp32.  The map, where a table of it has to be
    // made, beside it on the SMs that it leaves idle; the candidate kernel waits for both before it reads either.
    void* table = nullptr;
    rocs_status_t st = plan_request_map_begin(plan, stream, &map, &table);
    if (st != ROCS_OK) return st;
    st = linear_dispatch(dtype, plan->R, d_req, d_out, XR, ld_xr, W_CR, ld_wcr, bias, nullptr, 0, RequestMap{}, ROCS_ACT_NONE,
                         workspace, d_out, /*out_f32=*/true, stream);
    if (st != ROCS_OK && table != nullptr) cudaFreeAsync(table, stream);
    if (st == ROCS_OK && table != nullptr) st = plan_request_map_fill(plan, stream, table, &map);
    if (st != ROCS_OK) return st;
    Z = (const float*)workspace;
    bias = nullptr;
  }
  // Candidate half with the request term gathered in the epilogue (Eq. 14, Section 4.2.1).
  // The request half was enqueued directly in front: the candidate kernel may overlap its set-up
  // with it (it waits for it before reading Z).  Only meaningful when both went to tensor cores.
  const bool request_half_on_umma = Z != nullptr && dtype == ROCS_BF16 && g_path.load() == ROCS_PATH_AUTO &&
                                    umma_linear_supported(plan->R, d_req, d_out, ld_xr, ld_wcr, d_out, true);
  // Row sums for a following normalisation: left as partials by the candidate kernel's epilogue where
  // the CTA-pair kernel runs (and added up by a small kernel), otherwise taken from the stored output.
  float2* partials = nullptr;
  if (row_stats != nullptr && dtype == ROCS_BF16 && g_path.load() == ROCS_PATH_AUTO &&
      umma_linear_supported(plan->N, d_cand, d_out, ld_xc, ld_wcc, ld_y, false) &&
      umma_linear_ws2_supported(plan->N, d_cand, d_out, false))
    partials = reinterpret_cast<float2*>(static_cast<uint8_t*>(workspace) + z_bytes);
  rocs_status_t st = linear_dispatch(dtype, plan->N, d_cand, d_out, XC, ld_xc, W_CC, ld_wcc, bias, Z, d_out,
                                     map, act, Y, ld_y, /*out_f32=*/false, stream,
                                     request_half_on_umma, partials, plan->R);
  if (st != ROCS_OK || row_stats == nullptr) return st;
  if (partials != nullptr)
    return row_stats_from_partials(plan->N, umma_linear_ws2_stat_partials(d_out), partials,
                                   reinterpret_cast<float2*>(row_stats), stream);
  return row_stats_direct(dtype, plan->N, d_out, Y, ld_y, reinterpret_cast<float2*>(row_stats), stream);
}

rocs_status_t rocs_ikbo_linear(const rocs_plan_t* plan, rocs_dtype_t dtype, int32_t d_req,
                               int32_t d_cand, int32_t d_out, const void* XR, int64_t ld_xr,
                               const void* XC, int64_t ld_xc, const void* W_CR, int64_t ld_wcr,
                               const void* W_CC, int64_t ld_wcc, const float* bias, rocs_act_t act,
                               void* Y, int64_t ld_y, void* workspace, size_t workspace_bytes,
                               void* stream_) {
  return ikbo_linear_impl(plan, dtype, d_req, d_cand, d_out, XR, ld_xr, XC, ld_xc, W_CR, ld_wcr, W_CC, ld_wcc, bias,
                          act, Y, ld_y, nullptr, workspace, workspace_bytes, stream_);
}

size_t rocs_ikbo_linear_stats_workspace(const rocs_plan_t* plan, int32_t d_out) {
  if (!plan || d_out <= 0) return 0;
  return rocs_ikbo_linear_workspace(plan, d_out) +
         round_up((size_t)plan->N * (size_t)umma_linear_ws2_stat_partials(d_out) * sizeof(float2), 256);
}

rocs_status_t rocs_ikbo_linear_stats(const rocs_plan_t* plan, rocs_dtype_t dtype, int32_t d_req,
                                     int32_t d_cand, int32_t d_out, const void* XR, int64_t ld_xr,
                                     const void* XC, int64_t ld_xc, const void* W_CR, int64_t ld_wcr,
                                     const void* W_CC, int64_t ld_wcc, const float* bias, rocs_act_t act,
                                     void* Y, int64_t ld_y, float* row_stats, void* workspace,
                                     size_t workspace_bytes, void* stream_) {
  if (!row_stats && plan && plan->N > 0) return ROCS_ERR_INVALID_ARG;
  return ikbo_linear_impl(plan, dtype, d_req, d_cand, d_out, XR, ld_xr, XC, ld_xc, W_CR, ld_wcr, W_CC, ld_wcc, bias,
                          act, Y, ld_y, row_stats, workspace, workspace_bytes, stream_);
}

rocs_status_t rocs_weight_row_sums(rocs_dtype_t dtype, int32_t d_out, int32_t d_in, const void* W, int64_t ld_w,
                                   float* wbar, void* stream_) {
  if ((dtype != ROCS_BF16 && dtype != ROCS_F32) || d_out <= 0 || d_in <= 0 || !W || !wbar) return ROCS_ERR_INVALID_ARG;
  if (!aligned16(W) || !aligned16(wbar) || !row_stride_ok(ld_w, d_in, dtype)) return ROCS_ERR_ALIGNMENT;
  return weight_row_sums(dtype, d_out, d_in, W, ld_w, wbar, (cudaStream_t)stream_);
}

rocs_status_t rocs_linear_normed(rocs_dtype_t dtype, rocs_norm_t kind, int64_t M, int32_t d_in, int32_t d_out,
                                 const void* X, int64_t ld_x, const float* row_stats, float eps, const void* W,
                                 int64_t ld_w, const float* wbar, const float* bias, rocs_act_t act, void* Y,
                                 int64_t ld_y, void* stream_) {
  if ((dtype != ROCS_BF16 && dtype != ROCS_F32) || (kind != ROCS_NORM_LAYER && kind != ROCS_NORM_RMS))
    return ROCS_ERR_INVALID_ARG;
  if (M < 0 || d_in <= 0 || d_out <= 0 || !X || !W || !Y || !row_stats || !(eps >= 0.f)) return ROCS_ERR_INVALID_ARG;
  if (kind == ROCS_NORM_LAYER && !wbar) return ROCS_ERR_INVALID_ARG;
  if (act != ROCS_ACT_NONE && act != ROCS_ACT_RELU) return ROCS_ERR_INVALID_ARG;
  if (!aligned16(X) || !aligned16(W) || !aligned16(Y) || !aligned16(bias) || !aligned16(wbar) || !aligned16(row_stats) ||
      !row_stride_ok(ld_x, d_in, dtype) || !row_stride_ok(ld_w, d_in, dtype) || !row_stride_ok(ld_y, d_out, dtype))
    return ROCS_ERR_ALIGNMENT;
  // The folded form lives in the epilogue of the wide-layer kernel; other shapes normalise with
  // rocs_group_norm and call rocs_linear.
  if (dtype != ROCS_BF16 || g_path.load() != ROCS_PATH_AUTO || d_out % 4 != 0 ||
      !umma_linear_pair_supported(M, d_in, d_out, false, false))
    return ROCS_ERR_UNSUPPORTED;
  RowNorm norm;
  norm.row_stats = reinterpret_cast<const float2*>(row_stats);
  norm.kind = (int)kind;
  norm.eps = eps;
  norm.wbar = wbar;
  return umma_linear_pair(M, d_in, d_out, X, ld_x, W, ld_w, bias, (int)act, Y, ld_y, (cudaStream_t)stream_, &norm);
}

rocs_status_t rocs_linear(rocs_dtype_t dtype, int64_t M, int32_t d_in, int32_t d_out, const void* X,
                          int64_t ld_x, const void* W, int64_t ld_w, const float* bias,
                          rocs_act_t act, void* Y, int64_t ld_y, void* stream_) {
  if (dtype != ROCS_BF16 && dtype != ROCS_F32) return ROCS_ERR_INVALID_ARG;
  if (M < 0 || d_in <= 0 || d_out <= 0 || !X || !W || !Y) return ROCS_ERR_INVALID_ARG;
  if (act != ROCS_ACT_NONE && act != ROCS_ACT_RELU) return ROCS_ERR_INVALID_ARG;
  if (!aligned16(X) || !aligned16(W) || !aligned16(Y) || !aligned16(bias) || !row_stride_ok(ld_x, d_in, dtype) ||
      !row_stride_ok(ld_w, d_in, dtype) || !row_stride_ok(ld_y, d_out, dtype))
    return ROCS_ERR_ALIGNMENT;
  return linear_dispatch(dtype, M, d_in, d_out, X, ld_x, W, ld_w, bias, nullptr, 0, RequestMap{}, act, Y,
                         ld_y, false, (cudaStream_t)stream_);
}

size_t rocs_dca_attention_workspace(const rocs_plan_t*, int32_t, int32_t, int32_t) { return 0; }

rocs_status_t rocs_dca_attention(const rocs_plan_t* plan, rocs_dtype_t dtype, int32_t n_q, int32_t H,
                                 int32_t dh, float scale, const void* Q, const void* K,
                                 const void* V, int64_t T, const int32_t* seq_offsets, void* O,
                                 void* workspace, size_t workspace_bytes, void* stream_) {
  (void)workspace;
  (void)workspace_bytes;
  if (!plan || (dtype != ROCS_BF16 && dtype != ROCS_F32)) return ROCS_ERR_INVALID_ARG;
  if (n_q <= 0 || H <= 0 || dh <= 0 || T < 0 || T > 0x7fffffffLL || !seq_offsets) return ROCS_ERR_INVALID_ARG;
  if (plan->N > 0 && (!Q || !O)) return ROCS_ERR_INVALID_ARG;
  if (T > 0 && (!K || !V)) return ROCS_ERR_INVALID_ARG;
  if (!aligned16(Q) || !aligned16(K) || !aligned16(V) || !aligned16(O) ||
      ((int64_t)dh * (int64_t)elem_size(dtype)) % 16 != 0)
    return ROCS_ERR_ALIGNMENT;
  if (dh > 256) return ROCS_ERR_UNSUPPORTED;
  if (!(scale > 0.f)) scale = 1.0f / sqrtf((float)dh);
  cudaStream_t stream = (cudaStream_t)stream_;
  if (dtype == ROCS_BF16 && g_path.load() == ROCS_PATH_AUTO && umma_dca_supported(n_q, H, dh))
    return umma_dca(plan, n_q, H, dh, scale, Q, K, V, seq_offsets, T, O, stream);
  return simt_dca(dtype, plan, n_q, H, dh, scale, Q, K, V, seq_offsets, T, O, stream);
}

size_t rocs_glm_interaction_workspace(const rocs_plan_t* plan, int32_t n_r, int32_t n_c, int32_t n_co) {
  if (!plan || n_r < 0 || n_c < 0 || n_co <= 0) return 0;
  return round_up((size_t)plan->R * (size_t)n_co * (size_t)(n_r + n_c) * sizeof(float), 256);
}

rocs_status_t rocs_glm_interaction(const rocs_plan_t* plan, rocs_dtype_t dtype, int32_t n_r,
                                   int32_t n_c, int32_t d, const void* XR, const void* XC,
                                   const void* W, int32_t n_ro, int32_t n_co, void* YR, void* YC,
                                   void* OR_, void* OC, void* workspace, size_t workspace_bytes,
                                   void* stream_) {
  if (!plan || (dtype != ROCS_BF16 && dtype != ROCS_F32)) return ROCS_ERR_INVALID_ARG;
  if (n_r < 0 || n_c < 0 || n_r + n_c <= 0 || d <= 0 || n_ro < 0 || n_co < 0) return ROCS_ERR_INVALID_ARG;
  if ((n_r > 0 && plan->R > 0 && !XR) || (n_c > 0 && plan->N > 0 && !XC)) return ROCS_ERR_INVALID_ARG;
  if (!W && (n_ro != 0 || n_co != 0 || OR_ || OC)) return ROCS_ERR_INVALID_ARG;
  if (W && n_ro + n_co <= 0) return ROCS_ERR_INVALID_ARG;
  if (!aligned16(XR) || !aligned16(XC) || !aligned16(W) || !aligned16(YR) || !aligned16(YC) ||
      !aligned16(OR_) || !aligned16(OC) || ((int64_t)d * (int64_t)elem_size(dtype)) % 16 != 0)
    return ROCS_ERR_ALIGNMENT;
  cudaStream_t stream = (cudaStream_t)stream_;
  float* zr = nullptr;
  if (W && n_co > 0) {
    const size_t need = rocs_glm_interaction_workspace(plan, n_r, n_c, n_co);
    if (!workspace || workspace_bytes < need || (reinterpret_cast<uintptr_t>(workspace) & 255u))
      return ROCS_ERR_WORKSPACE;
    zr = (float*)workspace;
  }
  // Few products: the general kernels, whose request side is in the candidates' launch.
  if (dtype == ROCS_BF16 && g_path.load() == ROCS_PATH_AUTO && (YC || OC) &&
      simt_glm_pays(plan, n_r, n_c, d, n_co, OC != nullptr && n_co > 0)) {
    const rocs_status_t st = simt_glm(dtype, plan, n_r, n_c, d, XR, XC, W, n_ro, n_co, YR, YC, OR_, OC, zr, stream);
    if (st != ROCS_ERR_UNSUPPORTED) return st;
  }
  const bool mma = !umma_glm_supported(n_r, n_c, d, n_ro, n_co) && glm_mma_supported(n_r, n_c, d, n_co);
  if (dtype == ROCS_BF16 && g_path.load() == ROCS_PATH_AUTO && (mma || umma_glm_supported(n_r, n_c, d, n_ro, n_co))) {
    // The candidate kernel's tile list first: that kernel then starts beside the request kernel.
    TileList tiles;
    rocs_status_t st = !YC && !OC ? ROCS_OK
                       : mma      ? glm_mma_tiles(plan, n_r, n_c, d, stream, &tiles)
                                  : plan_tile_runs(plan, 128 / n_c, stream, &tiles);
    if (st != ROCS_OK) return st;
    // Request side once per request (tiny), candidate side on tensor cores.
    st = glm_request_mma_supported(n_r, d, n_ro, n_co)
             ? glm_request_mma(plan, n_r, n_c, d, XR, W, n_ro, n_co, YR, OR_, zr, stream)
             : simt_glm(dtype, plan, n_r, n_c, d, XR, nullptr, W, n_ro, n_co, YR, nullptr, OR_, nullptr, zr, stream);
    if (st != ROCS_OK) return st;
    if (!YC && !OC) return ROCS_OK;
    return mma ? glm_mma(plan, n_r, n_c, d, XR, XC, W, n_ro, n_co, YC, OC, zr, stream)
               : umma_glm(plan, n_r, n_c, d, XR, XC, W, n_ro, n_co, YC, OC, zr, stream);
  }
  return simt_glm(dtype, plan, n_r, n_c, d, XR, XC, W, n_ro, n_co, YR, YC, OR_, OC, zr, stream);
}

size_t rocs_glm_fm_projection_workspace(const rocs_plan_t* plan, int32_t d, int32_t k) {
  if (!plan || d <= 0 || k <= 0) return 0;
  return round_up((size_t)std::max(plan->R, 1) * (size_t)k * (size_t)d * sizeof(float), 256);
}

rocs_status_t rocs_glm_fm_projection(const rocs_plan_t* plan, rocs_dtype_t dtype, int32_t n_r, int32_t n_c,
                                     int32_t d, int32_t k, const void* XR, const void* XC, const void* P,
                                     void* FR, void* FC, void* workspace, size_t workspace_bytes, void* stream_) {
  if (!plan || (dtype != ROCS_BF16 && dtype != ROCS_F32)) return ROCS_ERR_INVALID_ARG;
  if (n_r <= 0 || n_c <= 0 || d <= 0 || k <= 0 || !P) return ROCS_ERR_INVALID_ARG;
  if ((plan->R > 0 && !XR) || (plan->N > 0 && FC && !XC)) return ROCS_ERR_INVALID_ARG;
  if (!aligned16(XR) || !aligned16(XC) || !aligned16(P) || !aligned16(FR) || !aligned16(FC) ||
      ((int64_t)d * (int64_t)elem_size(dtype)) % 16 != 0)
    return ROCS_ERR_ALIGNMENT;
  const size_t need = rocs_glm_fm_projection_workspace(plan, d, k);
  if (!workspace || workspace_bytes < need || (reinterpret_cast<uintptr_t>(workspace) & 255u))
    return ROCS_ERR_WORKSPACE;
  return fm_projection(dtype, plan, n_r, n_c, d, k, XR, XC, P, FR, FC, (float*)workspace,
                       g_path.load() == ROCS_PATH_AUTO, (cudaStream_t)stream_);
}

rocs_status_t rocs_group_norm(rocs_dtype_t dtype, rocs_norm_t kind, int64_t M, int32_t d, const void* X,
                              int64_t ld_x, const void* gamma, const void* beta, float eps, void* Y, int64_t ld_y,
                              void* stream_) {
  if ((dtype != ROCS_BF16 && dtype != ROCS_F32) || (kind != ROCS_NORM_LAYER && kind != ROCS_NORM_RMS))
    return ROCS_ERR_INVALID_ARG;
  if (M < 0 || d <= 0 || ld_x < d || ld_y < d || !(eps >= 0.f)) return ROCS_ERR_INVALID_ARG;
  if (M > 0 && (!X || !Y)) return ROCS_ERR_INVALID_ARG;
  const int64_t es = (int64_t)elem_size(dtype);
  if (!aligned16(X) || !aligned16(Y) || !aligned16(gamma) || !aligned16(beta) || (ld_x * es) % 16 != 0 ||
      (ld_y * es) % 16 != 0)
    return ROCS_ERR_ALIGNMENT;
  return group_norm(dtype, (int)kind, M, d, X, ld_x, gamma, beta, eps, Y, ld_y, (cudaStream_t)stream_);
}

rocs_status_t rocs_last_device_status(uint32_t* detail_host) {
  uint32_t* word = device_status_word();
  if (!word) return ROCS_ERR_CUDA;
  uint32_t v = 0;
  ROCS_CUDA_TRY(cudaDeviceSynchronize());
  ROCS_CUDA_TRY(cudaMemcpy(&v, word, sizeof v, cudaMemcpyDeviceToHost));
  if (v != 0) {
    const uint32_t zero = 0;
    ROCS_CUDA_TRY(cudaMemcpy(word, &zero, sizeof zero, cudaMemcpyHostToDevice));
  }
  if (detail_host) *detail_host = v;
  return v == 0 ? ROCS_OK : ROCS_ERR_TIMEOUT;
}

}  // extern "C"
