// Linear layer on the 5th-generation tensor cores (Eq. 4 / Eq. 14):
//     Y[i, n] = act( sum_k X[i, k] W[n, k] + bias[n] + add[map.of(i), n] )
// `add` is the request half Z of the split layer; it is gathered per output row in the epilogue
// through the candidate->request map (the in-kernel broadcast of Section 4.2.1), so the broadcast
// tensor never exists.
//
// One persistent CTA per SM, 6 warps:
//   warp 0   TMA producer: TM x 64 tiles of X and BN x 64 tiles of W into a shared-memory ring
//   warp 1   issues tcgen05.mma (128 x BN x 16, bf16 -> fp32) into one of two TMEM accumulators (TM rows of it used)
//   warps 2-5 epilogue: TMEM -> registers, + Z[m_i] (+ bias), ReLU, round to the output type,
//            128-byte-swizzled staging in shared memory, TMA store (clipped at the edges)
// The two accumulators let the epilogue of tile t overlap the main loop of tile t + 1.
// A split layer on few candidates is one launch (BOTH): a tile computes the request half of its own requests, at most TM
// consecutive rows of X^R, into the second accumulator, from where it goes through shared memory to the candidates' rows.  In a
// chain, two launches and one: 500 candidates of one request, 512|256 -> 1024, 6.6 and 5.5 us; 926 of 28, 736|200 -> 512,
// 11.0 and 6.9; 12 of one, 96|200 -> 512, 4.1 and 3.0 (and a launch less for the host, 5.4 and 3.5 us).
// Tiles are ordered with the output-column index fastest, so CTAs working at the same time share
// the same rows of X in L2.  M tiles may span several requests: each row looks up its own request.
#include <algorithm>
#include <type_traits>

#include "rocs_internal.h"
#include "sm100_ptx.cuh"

namespace rocs {
namespace {

using namespace ptx;

constexpr int BM = 128;           // rows of an MMA = TMEM lanes
constexpr int BK = 64;            // 64 bf16 = one 128-byte swizzle row
constexpr int kThreads = 192;
constexpr int kEpiWarps = 4;
constexpr uint32_t kStatusLinear = 0x100;

// TM x BN outputs per tile.  With TM < 128 the MMA still has 128 rows: those behind the tile's hold whatever lies behind
// its slot of X in shared memory, and their outputs are not stored.
template <int TM, int BN>
struct LinearCfg {
  static constexpr int kABytes = TM * BK * 2;
  static constexpr int kBBytes = BN * BK * 2;
  static constexpr int kStages = BN == 256 ? 4 : TM + BN >= 192 ? 6 : TM + BN >= 128 ? 8 : 12;
  static constexpr int kOffB = kStages * kABytes;  // slots of X, then of W
  static constexpr int kOffStaging = kOffB + kStages * kBBytes;
  static constexpr int kStagingBytes = kEpiWarps * 2 * 4096;  // per warp: two buffers of 32 rows x 128 bytes at most
  static constexpr int kTmemCols = 2 * BN;
  static constexpr int kSmemBytes = kOffStaging + kStagingBytes + 512 /*barriers*/ + 1024 /*align*/;
  static constexpr int kZStride = BN + 4;  // BOTH: floats per request row, eight rows hit eight different bank groups
  static constexpr int kZBytes = TM * kZStride * 4;
  static_assert(BN > 64 || kSmemBytes + kZBytes <= kMaxDynamicSmem, "shared memory of an SM");
  static_assert(kOffB - kABytes + BM * BK * 2 <= kOffStaging + kStagingBytes, "rows behind the last slot");
};

struct LinearParams {
  int64_t M;
  int32_t d_in, d_out;
  const float* bias;
  const float* add;
  int64_t ld_add;
  RequestMap map;
  int32_t act;
  int32_t x_rows;     // rows of an X tile that are loaded
  int32_t wait_late;  // `add` is written by the launch in front and nothing else this kernel reads is
  uint32_t* status;
};

// The request half of a split layer in the same launch: one tile per CTA.
constexpr int kMaxTilesBoth = 192;
struct RequestHalf {
  int32_t k_blocks;                // 64-wide blocks of d_req
  int32_t rows;                    // rows of X^R that a tile loads
  int32_t first[kMaxTilesBoth];    // the first of them, by row tile
};
struct NoRequestHalf {};

template <int TM, int BN, typename OutT, bool BOTH>
__global__ void __launch_bounds__(kThreads, 1)
linear_umma_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w,
                   const __grid_constant__ CUtensorMap map_y, const LinearParams p, const __grid_constant__ CUtensorMap map_xr,
                   const __grid_constant__ CUtensorMap map_wr,
                   const __grid_constant__ std::conditional_t<BOTH, RequestHalf, NoRequestHalf> rh) {
  using Cfg = LinearCfg<TM, BN>;
  constexpr int kStages = Cfg::kStages;
  constexpr int CH = BN * (int)sizeof(OutT) < 128 ? BN : 128 / (int)sizeof(OutT);  // output columns per staging row
  constexpr int kChunks16 = CH * (int)sizeof(OutT) / 16;                           // 16-byte chunks of a staging row

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* staging = smem + Cfg::kOffStaging;
  float* z_rows = reinterpret_cast<float*>(staging + Cfg::kStagingBytes);  // BOTH: [rh.rows][kZStride]
  uint64_t* full = reinterpret_cast<uint64_t*>(staging + Cfg::kStagingBytes + (BOTH ? Cfg::kZBytes : 0));
  uint64_t* empty = full + kStages;
  uint64_t* tmem_full = empty + kStages;
  uint64_t* tmem_empty = tmem_full + 2;
  uint64_t* drain = tmem_empty + 2;
  uint32_t* tmem_ptr = reinterpret_cast<uint32_t*>(drain + 1);
  AbortFlag* abort_flag = reinterpret_cast<AbortFlag*>(tmem_ptr + 1);

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int32_t m_tiles = (int32_t)((p.M + TM - 1) / TM);
  const int32_t n_tiles = (p.d_out + BN - 1) / BN;
  const int32_t k_blocks = (p.d_in + BK - 1) / BK;
  const int64_t num_tiles = (int64_t)m_tiles * n_tiles;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&tmem_full[a], 1);
      mbar_init(&tmem_empty[a], kEpiWarps);
    }
    mbar_init(drain, 1);
    abort_flag->v = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_ptr, Cfg::kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_ptr;
  // Launched as a programmatic dependent: the set-up above may overlap the end of the kernel in front;
  // nothing below touches global memory before that kernel is complete.  Then the kernel behind this one
  // (the candidate half behind the request half) may begin its own set-up; it waits for this grid before
  // it reads our output, and since it is released only after the wait above, everything in front of this
  // kernel is complete by the time it starts.
  if (warp == 0 && lane == 0) {  // parameters of the launch: no need to wait
    prefetch_tensormap(&map_x);
    prefetch_tensormap(&map_w);
    prefetch_tensormap(&map_y);
    if constexpr (BOTH) {
      prefetch_tensormap(&map_xr);
      prefetch_tensormap(&map_wr);
    }
  }
  // A candidate half in front of which only the request half is still running streams X and W at once; its
  // epilogue waits.
  if (!p.wait_late) {
    griddep_wait();
    griddep_launch_dependents();
  }

  if (warp == 0) {
    // ------------------------------ TMA producer ------------------------------------------
    if (elect_one()) {
      uint32_t it = 0;
      bool ok = true;
      if constexpr (BOTH) {  // the longer half first: its way to the rows overlaps the other's products
        const int32_t r0 = rh.first[blockIdx.x / n_tiles], n0 = (int32_t)(blockIdx.x % n_tiles) * BN;
        for (int32_t kb = 0; kb < rh.k_blocks; ++kb, ++it) {
          const int s = it % kStages;
          if (!mbar_wait(&empty[s], ((it / kStages) & 1) ^ 1, abort_flag, p.status, kStatusLinear | 1)) { ok = false; break; }
          mbar_expect_tx(&full[s], rh.rows * (BK * 2) + Cfg::kBBytes);
          tma_load_2d(smem + s * Cfg::kABytes, &map_xr, &full[s], kb * BK, r0);
          tma_load_2d(smem + Cfg::kOffB + s * Cfg::kBBytes, &map_wr, &full[s], kb * BK, n0);
        }
      }
      for (int64_t t = blockIdx.x; t < num_tiles && ok; t += gridDim.x) {
        const int32_t m0 = (int32_t)(t / n_tiles) * TM, n0 = (int32_t)(t % n_tiles) * BN;
        for (int32_t kb = 0; kb < k_blocks; ++kb, ++it) {
          const int s = it % kStages;
          const uint32_t ph = (it / kStages) & 1;
          if (!mbar_wait(&empty[s], ph ^ 1, abort_flag, p.status, kStatusLinear | 1)) { ok = false; break; }
          mbar_expect_tx(&full[s], p.x_rows * (BK * 2) + Cfg::kBBytes);
          tma_load_2d(smem + s * Cfg::kABytes, &map_x, &full[s], kb * BK, m0);
          tma_load_2d(smem + Cfg::kOffB + s * Cfg::kBBytes, &map_w, &full[s], kb * BK, n0);
        }
      }
      if (!ok) {
        // Aborting: let the copies already in flight land before the CTA gives up its shared memory.
        for (int s = 0; s < kStages; ++s) {
          const uint32_t n_issued = it / kStages + (((int)(it % kStages) > s) ? 1 : 0);  // loads issued to stage s
          if (n_issued == 0) continue;
          const uint32_t ph = (n_issued - 1) & 1;
          const uint64_t t0 = globaltimer_ns();
          while (!mbar_try_wait(&full[s], ph) && globaltimer_ns() - t0 < kWaitLimitNs) {}
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------ MMA issuer ---------------------------------------------
    if (elect_one()) {
      constexpr uint32_t idesc = umma_idesc_bf16(BM, BN, false, false);
      uint32_t it = 0, lt = 0;
      bool ok = true;
      auto products = [&](uint32_t d_tmem, int32_t blocks) {
        for (int32_t kb = 0; kb < blocks; ++kb, ++it) {
          const int s = it % kStages;
          if (!mbar_wait(&full[s], (it / kStages) & 1, abort_flag, p.status, kStatusLinear | 3)) return false;
          tc_fence_after_sync();
          const uint64_t a_desc = smem_desc_sw128(smem_u32(smem + s * Cfg::kABytes), 1024, 16);
          const uint64_t b_desc = smem_desc_sw128(smem_u32(smem + Cfg::kOffB + s * Cfg::kBBytes), 1024, 16);
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)  // +32 bytes = 16 bf16 along K, in 16-byte units
            umma_ss(d_tmem, a_desc + 2 * k, b_desc + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
          umma_commit(&empty[s]);  // frees the stage once these MMAs have read it
        }
        return true;
      };
      if constexpr (BOTH) {
        ok = products(tmem_base + BN, rh.k_blocks);
        if (ok) umma_commit(&tmem_full[1]);
      }
      for (int64_t t = blockIdx.x; t < num_tiles && ok; t += gridDim.x, ++lt) {
        const uint32_t acc = lt & 1;
        if (!mbar_wait(&tmem_empty[acc], ((lt >> 1) & 1) ^ 1, abort_flag, p.status, kStatusLinear | 2)) { ok = false; break; }
        tc_fence_after_sync();
        ok = products(tmem_base + acc * BN, k_blocks);
        if (ok) umma_commit(&tmem_full[acc]);
      }
      if (!ok) {
        umma_commit(drain);
        const uint64_t t0 = globaltimer_ns();
        while (!mbar_try_wait(drain, 0) && globaltimer_ns() - t0 < kWaitLimitNs) {}
      }
    }
  } else {
    // ------------------------------ epilogue -----------------------------------------------
    const int q = warp % 4;  // TMEM lane quadrant this warp may read
    uint8_t* my_stage = staging + (warp - 2) * 8192;
    uint32_t lt = 0, stores = 0;
    bool ok = true;
    if (p.wait_late) {
      griddep_wait();
      griddep_launch_dependents();
    }
    if constexpr (BOTH) {
      // the request half, bias included, to shared memory: row by row of X^R
      const int32_t n0 = (int32_t)(blockIdx.x % n_tiles) * BN;
      ok = mbar_wait(&tmem_full[1], 0, abort_flag, p.status, kStatusLinear | 4);
      tc_fence_after_sync();
      if (ok && q * 32 < rh.rows) {
        float* z = z_rows + (q * 32 + lane) * Cfg::kZStride;
#pragma unroll 1
        for (int c = 0; c < BN; c += 32) {
          uint32_t v[32];
          tmem_ld_32x32b_x32(tmem_base + BN + c + ((uint32_t)(q * 32) << 16), v);
          tmem_ld_wait();
          if (q * 32 + lane < rh.rows) {
#pragma unroll
            for (int i = 0; i < 32; i += 4) {
              float4 f = make_float4(__uint_as_float(v[i]), __uint_as_float(v[i + 1]), __uint_as_float(v[i + 2]), __uint_as_float(v[i + 3]));
              if (p.bias != nullptr && n0 + c + i < p.d_out) {
                const float4 b = __ldg(reinterpret_cast<const float4*>(p.bias + n0 + c + i));
                f.x += b.x; f.y += b.y; f.z += b.z; f.w += b.w;
              }
              *reinterpret_cast<float4*>(z + c + i) = f;
            }
          }
        }
      }
      asm volatile("bar.sync 1, %0;" ::"n"(kEpiWarps * 32) : "memory");
    }
    for (int64_t t = blockIdx.x; t < num_tiles && ok; t += gridDim.x, ++lt) {
      const uint32_t acc = lt & 1;
      const int32_t m0 = (int32_t)(t / n_tiles) * TM, n0 = (int32_t)(t % n_tiles) * BN;
      const int64_t row = (int64_t)m0 + q * 32 + lane;
      const bool mine = TM == BM || q * 32 < TM;  // rows of the tile among this warp's
      const float* add_row = nullptr;
      if constexpr (BOTH) {
        if (mine && row < p.M) add_row = z_rows + (p.map.of(row) - rh.first[t / n_tiles]) * Cfg::kZStride - n0;
      } else {
        if (p.add != nullptr && mine && row < p.M) add_row = p.add + (int64_t)p.map.of(row) * p.ld_add;
      }
      if (!mbar_wait(&tmem_full[acc], (lt >> 1) & 1, abort_flag, p.status, kStatusLinear | 4)) { ok = false; break; }
      tc_fence_after_sync();
      const uint32_t t_row = tmem_base + acc * BN + ((uint32_t)(q * 32) << 16);
      constexpr int kChunks = BN / CH;
      if (!mine) {
        __syncwarp();
        if (lane == 0) mbar_arrive(&tmem_empty[acc]);
        continue;
      }
#pragma unroll 1
      for (int c = 0; c < kChunks; ++c) {
        const int32_t col0 = n0 + c * CH;
        if (col0 >= p.d_out) break;
        uint32_t v[CH];
        tmem_ld_32x32b_x32(t_row + c * CH, v);
        if constexpr (CH == 64) tmem_ld_32x32b_x32(t_row + c * CH + 32, v + 32);
        tmem_ld_wait();
        if (c == kChunks - 1 || col0 + CH >= p.d_out) {
          // last read of this accumulator: hand it back to the MMA warp before finishing the math
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(&tmem_empty[acc]);
        }
        float f[CH];
#pragma unroll
        for (int i = 0; i < CH; ++i) f[i] = __uint_as_float(v[i]);
        if (add_row != nullptr) {
#pragma unroll
          for (int i = 0; i < CH; i += 4) {
            if (col0 + i < p.d_out) {
              const float4* from = reinterpret_cast<const float4*>(add_row + col0 + i);
              const float4 z = BOTH ? *from : __ldg(from);
              f[i] += z.x; f[i + 1] += z.y; f[i + 2] += z.z; f[i + 3] += z.w;
            }
          }
        }
        if (!BOTH && p.bias != nullptr) {
#pragma unroll
          for (int i = 0; i < CH; i += 4) {
            if (col0 + i < p.d_out) {
              const float4 b = __ldg(reinterpret_cast<const float4*>(p.bias + col0 + i));
              f[i] += b.x; f[i + 1] += b.y; f[i + 2] += b.z; f[i + 3] += b.w;
            }
          }
        }
        if (p.act == ROCS_ACT_RELU) {
#pragma unroll
          for (int i = 0; i < CH; ++i) f[i] = fmaxf(f[i], 0.f);
        }
        // staging buffer (two per warp): make sure the TMA store that last read it has finished
        uint8_t* buf = my_stage + (stores & 1) * 4096;
        if (elect_one()) tma_store_wait_read<1>();
        __syncwarp();
        uint8_t* row_ptr = buf + lane * (kChunks16 * 16);
        const int swizzle = kChunks16 == 8 ? lane & 7 : lane / 2 & 3;  // of 128- and 64-byte rows
#pragma unroll
        for (int j = 0; j < kChunks16; ++j) {  // 16-byte chunks, XOR-swizzled by row
          uint4 w;
          if constexpr (sizeof(OutT) == 2) {
            __nv_bfloat162 h0 = __floats2bfloat162_rn(f[8 * j + 0], f[8 * j + 1]);
            __nv_bfloat162 h1 = __floats2bfloat162_rn(f[8 * j + 2], f[8 * j + 3]);
            __nv_bfloat162 h2 = __floats2bfloat162_rn(f[8 * j + 4], f[8 * j + 5]);
            __nv_bfloat162 h3 = __floats2bfloat162_rn(f[8 * j + 6], f[8 * j + 7]);
            w.x = *reinterpret_cast<uint32_t*>(&h0);
            w.y = *reinterpret_cast<uint32_t*>(&h1);
            w.z = *reinterpret_cast<uint32_t*>(&h2);
            w.w = *reinterpret_cast<uint32_t*>(&h3);
          } else {
            w.x = __float_as_uint(f[4 * j + 0]);
            w.y = __float_as_uint(f[4 * j + 1]);
            w.z = __float_as_uint(f[4 * j + 2]);
            w.w = __float_as_uint(f[4 * j + 3]);
          }
          *reinterpret_cast<uint4*>(row_ptr + ((j ^ swizzle) << 4)) = w;
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (elect_one()) {
          tma_store_2d(&map_y, buf, col0, m0 + q * 32);
          tma_store_commit();
        }
        ++stores;
      }
    }
    if (elect_one()) tma_store_wait_all<0>();
  }

  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, Cfg::kTmemCols);
  }
}

int sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  }
  return n;
}

// What the request half of a split layer reads, and where its rows begin for each row tile.
struct RequestArgs {
  const void *XR, *W;
  int64_t ld_xr, ld_w;
  int32_t R, d_req;
  RequestHalf half;
};

template <int TM, int BN, typename OutT, bool BOTH = false>
rocs_status_t launch(int64_t M, int32_t d_in, int32_t d_out, const void* X, int64_t ld_x, const void* W,
                     int64_t ld_w, const float* bias, const float* add, int64_t ld_add, const RequestMap& map,
                     int act, void* Y, int64_t ld_y, cudaStream_t stream, bool wait_late, const RequestArgs* request = nullptr) {
  using Cfg = LinearCfg<TM, BN>;
  constexpr int CH = BN * (int)sizeof(OutT) < 128 ? BN : 128 / (int)sizeof(OutT);
  // A batch of fewer rows than a tile loads no more than it has: the loads of a small batch, 64 bytes per clock and
  // SM whatever they bring, are its time (K = 1024 on one row: 408 cycles per 64-deep block with 128 rows of X and
  // 64 of W).  The other rows of the operand hold whatever the buffer held; so do their outputs, which are not stored.
  const int32_t x_rows = (int32_t)std::min<int64_t>(TM, (M + 7) / 8 * 8);
  CUtensorMap map_x, map_w, map_y;
  if (!make_tensor_map_2d(&map_x, X, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)M, (uint64_t)d_in, (uint64_t)ld_x,
                          (uint32_t)x_rows, BK, true) ||
      !make_tensor_map_2d(&map_w, W, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)d_out, (uint64_t)d_in,
                          (uint64_t)ld_w, BN, BK, true) ||
      !make_tensor_map_2d(&map_y, Y, sizeof(OutT) == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                          sizeof(OutT), (uint64_t)M, (uint64_t)d_out, (uint64_t)ld_y, 32, CH, CH * sizeof(OutT) == 128,
                          CH * sizeof(OutT) == 64))
    return ROCS_ERR_CUDA;
  CUtensorMap map_xr = map_x, map_wr = map_w;
  std::conditional_t<BOTH, RequestHalf, NoRequestHalf> rh{};
  if constexpr (BOTH) {
    rh = request->half;
    if (!make_tensor_map_2d(&map_xr, request->XR, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)request->R, (uint64_t)request->d_req,
                            (uint64_t)request->ld_xr, (uint32_t)rh.rows, BK, true) ||
        !make_tensor_map_2d(&map_wr, request->W, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)d_out, (uint64_t)request->d_req,
                            (uint64_t)request->ld_w, BN, BK, true))
      return ROCS_ERR_CUDA;
  }
  uint32_t* status = device_status_word();
  if (!status) return ROCS_ERR_CUDA;
  constexpr int kSmem = Cfg::kSmemBytes + (BOTH ? Cfg::kZBytes : 0);
  auto kernel = linear_umma_kernel<TM, BN, OutT, BOTH>;
  ROCS_ALLOW_SMEM(kernel, kSmem);
  const int64_t tiles = ((M + TM - 1) / TM) * ((d_out + BN - 1) / BN);
  const int grid = (int)std::min<int64_t>(tiles, sm_count());
  LinearParams p{M, d_in, d_out, bias, add, ld_add, map, act, x_rows, wait_late ? 1 : 0, status};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  ROCS_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, map_x, map_w, map_y, p, map_xr, map_wr, rh));
  ROCS_CUDA_TRY(cudaGetLastError());
  return ROCS_OK;
}

// Few tiles: the one that loads least (its rows of X and of W) among those that give every tile an SM of its own.
// An SM loads 64 bytes per clock, which is the time of such a layer, down to about 240 cycles per K block (the
// products of 128 rows, however few are used, and their hand-over).  In a chain of the same layer, with 128 x 64
// tiles and with these: 500 x 1024 -> 1024 4.80 and 4.48 us (64 x 64), 500 x 1024 -> 256 4.63 and 4.09 (32 x 32),
// 741 x 512 -> 512 3.69 and 3.40, 96 x 512 -> 1024 3.54 and 3.04, 128 x 256 -> 256 2.90 and 2.43.  Measured and not
// taken: a tile's K blocks split over a cluster of 2 to 8 CTAs (5.64, 6.6, 4.86, 4.24, 4.26: clusters start later
// and hold up the next launch), the two loads of a K block issued by two warps (4.53, 4.15, 3.43, 3.09, 2.49).
bool small_tile(int64_t M, int32_t d_out, int* tm, int* bn) {
  const int sms = sm_count();
  int64_t least = INT64_MAX;
  for (int t = 32; t <= 128; t *= 2)
    for (int b = 32; b <= 64; b *= 2) {
      const int64_t rows = std::min<int64_t>(t, (M + 7) / 8 * 8) + b;
      if (((M + t - 1) / t) * ((d_out + b - 1) / b) <= sms && rows < least) { least = rows; *tm = t; *bn = b; }
    }
  return least != INT64_MAX;
}

}  // namespace

bool umma_linear_supported(int64_t M, int32_t d_in, int32_t d_out, int64_t ld_x, int64_t ld_w, int64_t ld_y,
                           bool out_f32) {
  (void)ld_x; (void)ld_w; (void)ld_y;  // row strides are already multiples of 16 bytes at the ABI
  if (M < 1 || M > 0x7fffff00LL || d_in < 8 || d_out < 8) return false;
  if (d_out % 4 != 0) return false;  // fp32 request rows are read as float4
  (void)out_f32;
  return true;
}

rocs_status_t umma_linear(int64_t M, int32_t d_in, int32_t d_out, const void* X, int64_t ld_x, const void* W,
                          int64_t ld_w, const float* bias, const float* add, int64_t ld_add,
                          const RequestMap& map, int act, void* Y, int64_t ld_y, bool out_f32,
                          cudaStream_t stream, bool add_from_previous_launch, float2* stat_partials,
                          int64_t add_rows) {
  if (umma_linear_ws2_supported(M, d_in, d_out, out_f32))
    return umma_linear_ws2(M, d_in, d_out, X, ld_x, W, ld_w, bias, add, ld_add, map, act, Y, ld_y, stream,
                           add_from_previous_launch, stat_partials, add_rows);
  if (stat_partials != nullptr) return ROCS_ERR_UNSUPPORTED;  // the caller asks for them only where the kernel above applies
  if (umma_linear_pair_supported(M, d_in, d_out, out_f32, add != nullptr))
    return umma_linear_pair(M, d_in, d_out, X, ld_x, W, ld_w, bias, act, Y, ld_y, stream);
  const bool wait_late = add_from_previous_launch && add != nullptr;
#define ROCS_LAUNCH(TM_, BN_)                                                                                         \
  (out_f32 ? launch<TM_, BN_, float>(M, d_in, d_out, X, ld_x, W, ld_w, bias, add, ld_add, map, act, Y, ld_y, stream,  \
                                     wait_late)                                                                      \
           : launch<TM_, BN_, __nv_bfloat16>(M, d_in, d_out, X, ld_x, W, ld_w, bias, add, ld_add, map, act, Y, ld_y, \
                                             stream, wait_late))
  const int sms = sm_count();
  int tm, bn;
  if (small_tile(M, d_out, &tm, &bn)) {
    if (bn == 32) return tm == 32 ? ROCS_LAUNCH(32, 32) : tm == 64 ? ROCS_LAUNCH(64, 32) : ROCS_LAUNCH(128, 32);
    return tm == 32 ? ROCS_LAUNCH(32, 64) : tm == 64 ? ROCS_LAUNCH(64, 64) : ROCS_LAUNCH(128, 64);
  }
  // Otherwise the widest tile that still gives every SM something to do.
  bn = d_out > 128 ? 256 : (d_out > 64 ? 128 : 64);
  while (bn > 64 && ((M + 127) / 128) * ((d_out + bn - 1) / bn) < sms) bn /= 2;
  if (bn == 256) return ROCS_LAUNCH(128, 256);
  if (bn == 128) return ROCS_LAUNCH(128, 128);
  return ROCS_LAUNCH(128, 64);
#undef ROCS_LAUNCH
}

// One launch for both halves where every tile has an SM of its own and its candidates' requests (their rows of X^R are
// consecutive) are no more than its rows.
rocs_status_t umma_linear_both(const rocs_plan* plan, int32_t d_req, int32_t d_cand, int32_t d_out, const void* XR, int64_t ld_xr,
                               const void* XC, int64_t ld_xc, const void* W_CR, int64_t ld_wcr, const void* W_CC, int64_t ld_wcc,
                               const float* bias, int act, void* Y, int64_t ld_y, cudaStream_t stream, bool* taken) {
  *taken = false;
  int tm, bn;
  if (plan->N < 1 || plan->N > kSearchRows || d_req < 8 || d_cand < 8 || d_out < 8 || d_out % 4 != 0 || !small_tile(plan->N, d_out, &tm, &bn))
    return ROCS_OK;
  const int32_t m_tiles = (int32_t)((plan->N + tm - 1) / tm);
  if (m_tiles > kMaxTilesBoth) return ROCS_OK;
  RequestArgs request{XR, W_CR, ld_xr, ld_wcr, plan->R, d_req, {}};
  const int32_t* off = plan->offsets_host.data();
  int32_t r = 0, most = 1;  // r: the request that holds a row, the last one that does not begin behind it
  for (int32_t t = 0; t < m_tiles; ++t) {
    const int32_t row0 = t * tm, last = std::min(row0 + tm, (int32_t)plan->N) - 1;
    while (off[r + 1] <= row0) ++r;
    request.half.first[t] = r;
    while (off[r + 1] <= last && r - request.half.first[t] < tm) ++r;
    most = std::max(most, r - request.half.first[t] + 1);
    if (most > tm) return ROCS_OK;  // requests without candidates in between
  }
  request.half.rows = (most + 7) / 8 * 8;
  request.half.k_blocks = (d_req + BK - 1) / BK;
  const RequestMap map{nullptr, plan->cand_offsets, plan->R};
  *taken = true;
#define ROCS_LAUNCH(TM_, BN_)                                                                                             \
  launch<TM_, BN_, __nv_bfloat16, true>(plan->N, d_cand, d_out, XC, ld_xc, W_CC, ld_wcc, bias, nullptr, 0, map, act, Y, ld_y, \
                                        stream, false, &request)
  if (bn == 32) return tm == 32 ? ROCS_LAUNCH(32, 32) : tm == 64 ? ROCS_LAUNCH(64, 32) : ROCS_LAUNCH(128, 32);
  return tm == 32 ? ROCS_LAUNCH(32, 64) : tm == 64 ? ROCS_LAUNCH(64, 64) : ROCS_LAUNCH(128, 64);
#undef ROCS_LAUNCH
}

}  // namespace rocs
