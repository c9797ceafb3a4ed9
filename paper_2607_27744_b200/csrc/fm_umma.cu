// Projected factorization machine, candidate rows, on the 5th-generation tensor cores:
//     FC[i] = X^C_i T[m_i] + (X^C_i X^C_i^T) P_C
// with T[r] = X^R_r^T P_R as a bf16 pair (value rounded to bf16 and rounded remainder), which the request kernel in front
// writes transposed, [R, 2, k, d].
//
// Tile = 128 / NC consecutive candidates of ONE request, NC = 4, 8 or 16 rows each: the box of the tensor map is NC rows of a
// candidate high, and the rows behind its last embedding arrive as zeros.  Per 64-wide slice of d shared memory holds
// [T^T values ; T^T remainders ; X^C tile] back to back, so that a single tcgen05.mma per 16-deep K step computes
//     D[128, 2 kp + 128] = X^C_tile * [T^T ; T^T remainders ; X^C_tile]^T
// whose first columns are the two parts of X^C T and whose 128 x 128 tail holds every candidate's Gram matrix on the diagonal.
// A thread of the epilogue owns a row: it adds the parts up and its NC Gram values times P_C in fp32 FMA.
//
// Bound by HBM, and in small batches by what a short run of tiles takes to start and end.  In place of a candidate per warp
// on mma.sync, whose products were what took the time (some 25 cycles of a scheduler each): 18400 candidates of 12
// embeddings x 128, k = 16, 28.7 -> 20.2 us with their request kernel; 56721 of 12 x 192, k = 24, 205 -> 66; 32768 of 16 x 64,
// k = 24, 50 -> 32.5; 19236 of 4 x 128, k = 16, 24.9 -> 11.1.  T kept in a ring of its own, loaded once per request and multiplied
// apart from the Gram matrix, was slower (23.1 us for 18400 to 21000 candidates of 12 x 128 as above, 26.9 us so).  The tiles are
// walked and not listed, in any number: the walk is short against a tile (2700 tiles 25.3 us with the list, 23.0 walked).
#include <algorithm>

#include "rocs_internal.h"
#include "sm100_ptx.cuh"

namespace rocs {
namespace {

using namespace ptx;

constexpr uint32_t kStatusFmUmma = 0x900;
constexpr uint32_t kTmemCols = 512;
constexpr int kMaxStages = 6;

struct FmUmmaParams {
  const int32_t* offsets;  // [R + 1]
  int32_t R, num_tiles;
  int32_t n_r, n_c, d, k, kp;  // kp: k rounded up to 8
  int32_t stages, stage_bytes;
  const __nv_bfloat16 *P, *XC, *TT;  // [n_r + n_c, k], [N, n_c, d], [R, 2, k, d]
  __nv_bfloat16* FC;                 // [N, n_c, k]
  uint32_t* status;
};

// KP: columns computed per row, 16 or 32.  Three accumulators and groups of epilogue warps fit with 16, two with 32.
template <int KP>
struct FmUmmaCfg {
  static constexpr int kGroups = KP == 16 ? 3 : 2;
  static constexpr int kAccStride = KP == 16 ? 160 : 256;
  static constexpr int kThreads = 64 + 128 * kGroups;
};

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// One row in plain fp32, the request's and the candidate's own term added up before the row's product: for values that the
// pair or the Gram matrix cannot hold (an infinity, a square past fp32), where the result has to be what fp32 arithmetic gives.
__device__ __noinline__ void row_by_hand(const __nv_bfloat16* xc, const __nv_bfloat16* row, const __nv_bfloat16* tt,
                                         const __nv_bfloat16* pc, int32_t n_c, int32_t d, int32_t k, __nv_bfloat16* out) {
#pragma unroll 1
  for (int32_t c = 0; c < k; ++c) {
    float acc = 0.f;
#pragma unroll 1
    for (int32_t e = 0; e < d; ++e) {
      float h = __bfloat162float(tt[c * d + e]) + __bfloat162float(tt[(k + c) * d + e]);
#pragma unroll 1
      for (int32_t a = 0; a < n_c; ++a) h = fmaf(__bfloat162float(pc[a * k + c]), __bfloat162float(xc[a * d + e]), h);
      acc = fmaf(__bfloat162float(row[e]), h, acc);
    }
    out[c] = __float2bfloat16_rn(acc);
  }
}

template <int NC, int KP>
__global__ void __launch_bounds__(FmUmmaCfg<KP>::kThreads, 1)
fm_umma_kernel(const __grid_constant__ CUtensorMap map_tt, const __grid_constant__ CUtensorMap map_xc, const FmUmmaParams p) {
  constexpr int G = FmUmmaCfg<KP>::kGroups, kAccStride = FmUmmaCfg<KP>::kAccStride;
  extern __shared__ __align__(1024) uint8_t smem[];
  float* pc = reinterpret_cast<float*>(smem + p.stages * p.stage_bytes);  // [NC][KP], zero beyond n_c rows and k columns
  uint64_t* full = reinterpret_cast<uint64_t*>(pc + NC * KP);
  uint64_t* empty = full + kMaxStages;
  uint64_t* tmem_full = empty + kMaxStages;
  uint64_t* tmem_empty = tmem_full + G;
  uint64_t* drain = tmem_empty + G;
  uint32_t* tmem_ptr = reinterpret_cast<uint32_t*>(drain + 1);
  AbortFlag* abort_flag = reinterpret_cast<AbortFlag*>(tmem_ptr + 1);
  int32_t* scratch = reinterpret_cast<int32_t*>(tmem_ptr + 2);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if ((smem_u32(smem) & 1023u) != 0) {  // the swizzled tiles assume a 1024-byte aligned base
    if (threadIdx.x == 0) atomicCAS(p.status, 0u, kStatusFmUmma | 15);
    return;
  }
  const int32_t k_slices = p.d / 64;
  const int32_t tt_bytes = 2 * p.kp * 128, slice_bytes = tt_bytes + 128 * 128;
  // a contiguous run of tiles per CTA: consecutive tiles mostly share a request, whose T stays in L2
  const int32_t t_begin = (int32_t)((int64_t)blockIdx.x * p.num_tiles / gridDim.x);
  const int32_t t_end = (int32_t)((int64_t)(blockIdx.x + 1) * p.num_tiles / gridDim.x);

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < G; ++a) {
      mbar_init(&tmem_full[a], 1);
      mbar_init(&tmem_empty[a], 4);
    }
    mbar_init(drain, 1);
    abort_flag->v = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_ptr, kTmemCols);
    tmem_relinquish();
  }
  for (int e = threadIdx.x; e < NC * KP; e += FmUmmaCfg<KP>::kThreads) {
    const int a = e / KP, c = e % KP;
    pc[e] = a < p.n_c && c < p.k ? __bfloat162float(p.P[(int64_t)(p.n_r + a) * p.k + c]) : 0.f;
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_ptr;
  TileWalk walk{p.offsets, p.R, 128 / NC};
  walk.start_in_block<FmUmmaCfg<KP>::kThreads>(t_begin, scratch);

  if (warp == 0) {
    // ------------------------------ TMA producer ------------------------------------------
    if (elect_one()) {
      prefetch_tensormap(&map_xc);
      prefetch_tensormap(&map_tt);
      auto load_x = [&](int s, const Tile& tile) {
        mbar_expect_tx(&full[s], p.stage_bytes);
        for (int32_t ks = 0; ks < k_slices; ++ks)
          tma_load_3d(smem + s * p.stage_bytes + ks * slice_bytes + tt_bytes, &map_xc, &full[s], ks * 64, 0, tile.cand0);
      };
      auto load_t = [&](int s, const Tile& tile) {
        for (int32_t ks = 0; ks < k_slices; ++ks)
          tma_load_3d(smem + s * p.stage_bytes + ks * slice_bytes, &map_tt, &full[s], ks * 64, 0, 2 * tile.req);
      };
      // the first tiles of X^C beside the request kernel, which writes T
      TileWalk behind = walk;
      const int32_t ahead = min(p.stages, t_end - t_begin);
      for (int32_t i = 0; i < ahead; ++i) load_x(i, walk.take(t_begin + i + 1 < t_end));
      griddep_wait();
      for (int32_t i = 0; i < ahead; ++i) load_t(i, behind.take(t_begin + i + 1 < t_end));
      uint32_t it = (uint32_t)ahead;
      bool ok = true;
      for (int32_t t = t_begin + ahead; t < t_end; ++t, ++it) {
        const Tile tile = walk.take(t + 1 < t_end);
        const int s = it % p.stages;
        if (!mbar_wait(&empty[s], ((it / p.stages) & 1) ^ 1, abort_flag, p.status, kStatusFmUmma | 1)) { ok = false; break; }
        load_x(s, tile);
        load_t(s, tile);
      }
      if (!ok) {
        for (int s = 0; s < p.stages; ++s) {
          const uint32_t n_issued = it / p.stages + (((int)(it % p.stages) > s) ? 1 : 0);
          if (n_issued == 0) continue;
          const uint64_t t0 = globaltimer_ns();
          while (!mbar_try_wait(&full[s], (n_issued - 1) & 1) && globaltimer_ns() - t0 < kWaitLimitNs) {}
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------ MMA issuer ---------------------------------------------
    if (elect_one()) {
      const uint32_t idesc = umma_idesc_bf16(128, (uint32_t)(2 * p.kp + 128), false, false);
      uint32_t it = 0;
      bool ok = true;
      for (int32_t t = t_begin; t < t_end; ++t, ++it) {
        const uint32_t acc = it % G;
        const int s = it % p.stages;
        if (!mbar_wait(&tmem_empty[acc], ((it / G) & 1) ^ 1, abort_flag, p.status, kStatusFmUmma | 2)) { ok = false; break; }
        if (!mbar_wait(&full[s], (it / p.stages) & 1, abort_flag, p.status, kStatusFmUmma | 3)) { ok = false; break; }
        tc_fence_after_sync();
        const uint32_t d_tmem = tmem_base + acc * kAccStride;
        const uint32_t st = smem_u32(smem + s * p.stage_bytes);
        for (int32_t ks = 0; ks < k_slices; ++ks) {
          const uint64_t b_desc = smem_desc_sw128(st + ks * slice_bytes, 1024, 16);             // [T^T ; T^T ; X^C]
          const uint64_t a_desc = smem_desc_sw128(st + ks * slice_bytes + tt_bytes, 1024, 16);  // X^C
#pragma unroll
          for (int k = 0; k < 4; ++k) umma_ss(d_tmem, a_desc + 2 * k, b_desc + 2 * k, idesc, (ks | k) != 0 ? 1u : 0u);
        }
        umma_commit(&empty[s]);
        umma_commit(&tmem_full[acc]);
      }
      if (!ok) {
        umma_commit(drain);
        const uint64_t t0 = globaltimer_ns();
        while (!mbar_try_wait(drain, 0) && globaltimer_ns() - t0 < kWaitLimitNs) {}
      }
    }
  } else {
    // ------------------------------ epilogue groups ----------------------------------------
    const int g = (warp - 2) / 4;  // group 0: warps 2-5, group 1: warps 6-9, ...
    const int q = warp % 4;        // TMEM lane quadrant = rows 32q .. 32q+31 of the tile
    const int cand_l = (q * 32 + lane) / NC, a_row = lane % NC, sub = lane / NC;
    uint32_t it = 0;
    for (int32_t t = t_begin; t < t_end; ++t, ++it) {
      const Tile tile = walk.take(t + 1 < t_end);
      if ((int)(it % G) != g) continue;
      if (!mbar_wait(&tmem_full[g], (it / G) & 1, abort_flag, p.status, kStatusFmUmma | 4)) break;
      tc_fence_after_sync();
      const uint32_t t_row = tmem_base + g * kAccStride + ((uint32_t)(q * 32) << 16);
      uint32_t val[KP], rem[KP], vcc[32];
      if constexpr (KP == 16) {
        tmem_ld_32x32b_x16(t_row, val);
        tmem_ld_32x32b_x16(t_row + p.kp, rem);
      } else {
        tmem_ld_32x32b_x32(t_row, val);
        tmem_ld_32x32b_x32(t_row + p.kp, rem);
      }
      tmem_ld_32x32b_x32(t_row + 2 * p.kp + q * 32, vcc);
      tmem_ld_wait();
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tmem_empty[g]);
      if (a_row < p.n_c && cand_l < tile.count) {
        uint64_t out[KP / 2];
#pragma unroll
        for (int c = 0; c < KP; c += 2)
          out[c / 2] = pack2(__uint_as_float(val[c]) + __uint_as_float(rem[c]), __uint_as_float(val[c + 1]) + __uint_as_float(rem[c + 1]));
        float probe = 0.f;  // not 0 behind an infinity or a NaN among this row's values
#pragma unroll
        for (int j = 0; j < NC; ++j) {
          if (j >= p.n_c) break;
          // of the diagonal block the columns of the row's own candidate
          uint32_t x = vcc[j];
#pragma unroll
          for (int s = 1; s < 32 / NC; ++s) x = sub == s ? vcc[s * NC + j] : x;
          const float gram = __uint_as_float(x);
          probe = fmaf(gram, 0.f, probe);
          const uint64_t gram2 = pack2(gram, gram);
#pragma unroll
          for (int c = 0; c < KP; c += 4) {
            const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(pc + j * KP + c);
            out[c / 2] = ffma2(gram2, w.x, out[c / 2]);
            out[c / 2 + 1] = ffma2(gram2, w.y, out[c / 2 + 1]);
          }
        }
        float f[KP];
#pragma unroll
        for (int c = 0; c < KP; c += 2) {
          unpack2(out[c / 2], f[c], f[c + 1]);
          if (c < p.k) probe = fmaf(f[c], 0.f, fmaf(f[c + 1], 0.f, probe));  // (k is even)
        }
        const int64_t cand = (int64_t)tile.cand0 + cand_l;
        __nv_bfloat16* dst = p.FC + (cand * p.n_c + a_row) * p.k;
        if (probe != 0.f) {
          const __nv_bfloat16* xc = p.XC + cand * p.n_c * p.d;
          row_by_hand(xc, xc + a_row * p.d, p.TT + (int64_t)tile.req * 2 * p.k * p.d, p.P + (int64_t)p.n_r * p.k, p.n_c, p.d, p.k, dst);
        } else if (p.k % 8 == 0) {
#pragma unroll
          for (int c = 0; c < KP; c += 8)
            if (c < p.k)
              *reinterpret_cast<uint4*>(dst + c) = make_uint4(pack_bf16(f[c], f[c + 1]), pack_bf16(f[c + 2], f[c + 3]),
                                                              pack_bf16(f[c + 4], f[c + 5]), pack_bf16(f[c + 6], f[c + 7]));
        } else {
#pragma unroll
          for (int c = 0; c < KP; c += 2)
            if (c < p.k) *reinterpret_cast<uint32_t*>(dst + c) = pack_bf16(f[c], f[c + 1]);
        }
      }
      __syncwarp();
    }
  }

  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

int sm_count_fm_umma() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  }
  return n;
}

template <int NC, int KP>
rocs_status_t launch(int smem, const CUtensorMap& map_tt, const CUtensorMap& map_xc, const FmUmmaParams& p, cudaStream_t stream) {
  ROCS_ALLOW_SMEM((fm_umma_kernel<NC, KP>), kMaxDynamicSmem);
  return launch_dependent(fm_umma_kernel<NC, KP>, dim3((unsigned)std::min(p.num_tiles, sm_count_fm_umma())), FmUmmaCfg<KP>::kThreads,
                          (size_t)smem, stream, map_tt, map_xc, p);
}

int rows_of(int32_t n_c) { return n_c <= 4 ? 4 : n_c <= 8 ? 8 : 16; }

}  // namespace

// Where this kernel is the faster one of the two on bf16 rows.  fm_projection.cu's has as many candidates at work on an SM as
// warps and takes a candidate's bytes alone; this one takes a tile's 128 rows however few of them a request fills, and its run of
// tiles starts and ends slower.  Request kernel included, on a plan that is kept, that one and this one, in us:
//   few candidates per tile, of 1000 requests 4 x 128, k = 16: one / two / eight each 13.4 / 16.4 / 24.5 and 17.4 / 17.4 / 17.6;
//   12000 x 2 of 8 x 64, k = 8, 77 and 96; 100 x 3 of 12 x 128, k = 16, 7.0 and 7.9; of 12 x 192, k = 24, 1000 x 1 / 2 24.2 / 28.9 and
//   27.4 / 27.6
//   d = 64, few requests, their products being short: 12 embeddings, k = 8, 1 x 3000 / 5000 / 10000 6.6 / 7.6 / 9.8 and 8.4 / 9.6 / 11.9,
//   100 x 10 / 30 / 100 7.1 / 8.2 / 12.0 and 8.0 / 8.8 / 12.3, 1000 x 8 / 30 17.0 / 27.8 and 14.8 / 25.6; 8 embeddings, 1 x 300 /
//   3000 / 5000 / 10000 5.3 / 6.6 / 7.6 / 9.8 and 5.5 / 7.6 / 8.2 / 9.5, 100 x 30 8.2 and 7.8
//   d = 128, k = 16, 12 embeddings in two or three rounds of tiles of a request or a few: 3000 8.4 and 9.2, 5000 11.1 and 10.9
// 16 embeddings to 8 or 16 columns take H rounded once there (103 and 106 us on 131072 x 128, k = 16; 5.6 and 6.3 on 29).
bool fm_umma_pays(const rocs_plan* plan, int32_t n_c, int32_t d, int32_t k) {
  if (n_c == 16 && (k == 8 || k == 16)) return false;
  const int64_t N = plan->N, R = plan->R, tiles = plan_entries(plan, 128 / rows_of(n_c));
  if (R > 64 && (d <= 128 ? N <= 3 * tiles : N < 2 * tiles)) return false;
  if (d == 64 && k <= 16 && n_c > 4 && (n_c > 8 ? R <= 128 && N <= 16384 : R <= 32 && N <= 6144)) return false;
  if (d == 128 && k <= 16 && n_c > 8 && R <= 4 && tiles > 148 && tiles <= 3 * 148) return false;
  return true;
}

rocs_status_t fm_umma(const rocs_plan* plan, int32_t n_r, int32_t n_c, int32_t d, int32_t k, const void* XC, const void* P,
                      const void* TT, void* FC, cudaStream_t stream) {
  const int nc = rows_of(n_c);
  const int64_t tiles = plan_entries(plan, 128 / nc);
  if (tiles == 0) return ROCS_OK;
  if (tiles > 0x7fffffffLL) return ROCS_ERR_UNSUPPORTED;
  FmUmmaParams p{};
  p.offsets = plan->cand_offsets;
  p.R = plan->R;
  p.num_tiles = (int32_t)tiles;
  p.n_r = n_r; p.n_c = n_c; p.d = d; p.k = k;
  p.kp = (k + 7) / 8 * 8;
  p.stage_bytes = (2 * p.kp + 128) * d * 2;
  constexpr int kFixed = 16 * 32 * 4 + (2 * kMaxStages + 7) * 8 + 8 + 16 * 4;
  p.stages = std::min(kMaxStages, (kMaxDynamicSmem - kFixed) / p.stage_bytes);
  p.P = (const __nv_bfloat16*)P; p.XC = (const __nv_bfloat16*)XC; p.TT = (const __nv_bfloat16*)TT;
  p.FC = (__nv_bfloat16*)FC;
  p.status = device_status_word();
  if (!p.status) return ROCS_ERR_CUDA;
  CUtensorMap map_tt, map_xc;
  if (!make_tensor_map_3d(&map_tt, TT, (uint64_t)d, (uint64_t)k, 2 * (uint64_t)plan->R, 64, (uint32_t)p.kp, 2) ||
      !make_tensor_map_3d(&map_xc, XC, (uint64_t)d, (uint64_t)n_c, (uint64_t)plan->N, 64, (uint32_t)nc, (uint32_t)(128 / nc)))
    return ROCS_ERR_CUDA;
  const int smem = p.stages * p.stage_bytes + kFixed;
#define ROCS_LAUNCH(NC_, KP_) return launch<NC_, KP_>(smem, map_tt, map_xc, p, stream)
  if (k <= 16) {
    if (nc == 4) ROCS_LAUNCH(4, 16);
    if (nc == 8) ROCS_LAUNCH(8, 16);
    ROCS_LAUNCH(16, 16);
  }
  if (nc == 4) ROCS_LAUNCH(4, 32);
  if (nc == 8) ROCS_LAUNCH(8, 32);
  ROCS_LAUNCH(16, 32);
#undef ROCS_LAUNCH
}

}  // namespace rocs
