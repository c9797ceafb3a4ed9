// Cross attention (Eq. 13) on the CUDA cores: fp32 FMA arithmetic on fp32 or bf16 storage.  Carries the
// fp32 path and the head dimensions the tensor-core kernel does not take.
//
// One block per (tile of 32 query rows of one request, head): the tile's queries stay in shared memory,
// the request's keys and values come through it in blocks of 64, read once per tile and in place (never
// copied per candidate).  128 threads as 8 x 16; a thread owns 4 query rows and, of a block, 4 keys for
// the scores and DHP / 16 columns for the output, so eight 16-byte shared-memory reads feed 64 FMAs.  The
// running maximum and normaliser of a row live in the 16 neighbouring lanes that share it.  K_{j+1} is
// fetched while the softmax and P V of block j run, V_{j+1} while the scores of block j + 1 do.
//
// What bounds it: shared-memory reads and the FMA pipe about equally (ncu: L1/shared 67 %, FMA 48 % of
// active cycles), and the last blocks (1.3 waves at the size below).  Measured on 2613 candidates of 24
// requests x 8 heads of 64 over 64..384 keys, fp32: 69 us; one warp per query row, which re-read the keys
// for every row, 1450 us.  32 rows and not 64: ragged requests leave less of a tile empty (74 us with 64);
// 8 x 4 scores per thread 71-90 us, packed fma.rn.f32x2 68 us: the reads, not the issue slots, are the limit.
// Every row is computed by a fixed sequence over its own request's keys, so results are deterministic
// and independent of neighbouring candidates (Eq. 1).
#include <algorithm>

#include "rocs_internal.h"
#include "sm100_ptx.cuh"
#include "simt_util.cuh"

namespace rocs {
namespace {

constexpr int kRows = 32, kKeys = 64, kThreads = 128;
constexpr int kPStride = kKeys + 4;

template <int DHP>
constexpr int smem_floats() {
  return (kRows + 2 * kKeys) * (DHP + 4) + kRows * kPStride;
}

template <typename T, int DHP>
__global__ void __launch_bounds__(kThreads, DHP <= 64 ? 4 : DHP <= 128 ? 2 : 1) dca_simt_kernel(
    int32_t n_q, int32_t H, int32_t dh, float scale, const T* __restrict__ Q, const T* __restrict__ K,
    const T* __restrict__ V, int32_t R, int32_t cands_per_tile, const int32_t* __restrict__ cand_offsets,
    const DcaItem* __restrict__ items, const int32_t* __restrict__ seq_offsets, T* __restrict__ O) {
  constexpr int S = DHP + 4;           // row stride in floats: 16-byte reads of 8 rows hit 8 different bank groups
  constexpr int C = DHP / 16;          // output columns per thread
  extern __shared__ __align__(16) float sm[];
  float* qs = sm;                      // [32][S]
  float* ks = qs + kRows * S;          // [64][S]
  float* vs = ks + kKeys * S;          // [64][S]
  float* ps = vs + kKeys * S;          // [32][kPStride]
  ptx::griddep_wait_for(Q, K, V, cand_offsets, items, seq_offsets);
  ptx::griddep_launch_dependents();
  DcaItem item;
  if (items != nullptr) {
    item = items[blockIdx.x];
  } else {
    const FoundTile f = find_tile_in_block<kThreads>(R, cands_per_tile, H, cand_offsets, blockIdx.x);
    item = DcaItem{f.req, f.cand0, f.count, f.head};
  }
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  const int64_t hd = (int64_t)H * dh;
  const int32_t s0 = seq_offsets[item.req];
  const int32_t L = seq_offsets[item.req + 1] - s0;
  const T* kg = K + (int64_t)s0 * hd + (int64_t)item.head * dh;
  const T* vg = V + (int64_t)s0 * hd + (int64_t)item.head * dh;

  // a candidate with more query tokens than a tile has rows takes several row tiles
  const int32_t item_rows = item.count * n_q;
  for (int32_t row0 = blockIdx.y * kRows; row0 < item_rows; row0 += gridDim.y * kRows) {
    const int32_t rows = min(kRows, item_rows - row0);
    const int64_t q0 = ((int64_t)item.cand0 * n_q + row0) * hd + (int64_t)item.head * dh;
    float acc[4][C];
    float m[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      m[i] = -INFINITY;
      l[i] = 0.f;
#pragma unroll
      for (int c = 0; c < C; ++c) acc[i][c] = 0.f;
    }
    if (L > 0) {
      rows_to_shared_async<T, DHP>(Q + q0, hd, rows, kRows, dh, qs, S, tid, kThreads);
      rows_to_shared_async<T, DHP>(kg, hd, min(kKeys, L), kKeys, dh, ks, S, tid, kThreads);
      cp_async_commit();
      rows_to_shared_async<T, DHP>(vg, hd, min(kKeys, L), kKeys, dh, vs, S, tid, kThreads);
      cp_async_commit();
    }
    for (int32_t j0 = 0; j0 < L; j0 += kKeys) {
      const int32_t next = L - j0 - kKeys;  // keys behind this block
      cp_async_wait<1>();                   // K_j (and Q) have landed, V_j may still be on its way
      __syncthreads();
      float s[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) s[i][j] = 0.f;
#pragma unroll 4
      for (int e = 0; e < DHP; e += 4) {
        float4 a[4], b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(qs + (ty * 4 + i) * S + e);
#pragma unroll
        for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const float4*>(ks + (tx + 16 * j) * S + e);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            s[i][j] = fmaf(a[i].x, b[j].x, s[i][j]);
            s[i][j] = fmaf(a[i].y, b[j].y, s[i][j]);
            s[i][j] = fmaf(a[i].z, b[j].z, s[i][j]);
            s[i][j] = fmaf(a[i].w, b[j].w, s[i][j]);
          }
      }
      __syncthreads();  // K_j is read: its buffer takes K_{j+1}
      if (next > 0) rows_to_shared_async<T, DHP>(kg + (int64_t)(j0 + kKeys) * hd, hd, min(kKeys, next), kKeys, dh, ks, S, tid, kThreads);
      cp_async_commit();
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float mx = -INFINITY;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          s[i][j] = j0 + tx + 16 * j < L ? s[i][j] * scale : -INFINITY;
          mx = fmaxf(mx, s[i][j]);
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const float m_new = fmaxf(m[i], mx);
        const float corr = m[i] == -INFINITY ? 0.f : expf(m[i] - m_new);
        float sum = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float p = j0 + tx + 16 * j < L ? expf(s[i][j] - m_new) : 0.f;
          sum += p;
          ps[(ty * 4 + i) * kPStride + tx + 16 * j] = p;
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        l[i] = l[i] * corr + sum;
        m[i] = m_new;
#pragma unroll
        for (int c = 0; c < C; ++c) acc[i][c] *= corr;
      }
      cp_async_wait<1>();  // V_j
      __syncthreads();     // V_j for everybody; the P rows of a warp are its own
#pragma unroll 2
      for (int k = 0; k < kKeys; k += 4) {
        float4 a[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(ps + (ty * 4 + i) * kPStride + k);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          float b[C];
          const float* vr = vs + (k + kk) * S;
          if constexpr (C == 2) {
            const float2 t = *reinterpret_cast<const float2*>(vr + tx * 2);
            b[0] = t.x; b[1] = t.y;
          } else {
#pragma unroll
            for (int c = 0; c < C; c += 4) {
              const float4 t = *reinterpret_cast<const float4*>(vr + c * 16 + tx * 4);
              b[c] = t.x; b[c + 1] = t.y; b[c + 2] = t.z; b[c + 3] = t.w;
            }
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float p = kk == 0 ? a[i].x : kk == 1 ? a[i].y : kk == 2 ? a[i].z : a[i].w;
#pragma unroll
            for (int c = 0; c < C; ++c) acc[i][c] = fmaf(p, b[c], acc[i][c]);
          }
        }
      }
      __syncthreads();  // V_j is read: its buffer takes V_{j+1}
      if (next > 0) rows_to_shared_async<T, DHP>(vg + (int64_t)(j0 + kKeys) * hd, hd, min(kKeys, next), kKeys, dh, vs, S, tid, kThreads);
      cp_async_commit();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int row = ty * 4 + i;
      if (row >= rows) continue;
      const float inv = L > 0 ? 1.f / l[i] : 0.f;
      T* out = O + q0 + (int64_t)row * hd;
      constexpr int W = C == 2 ? 2 : 4;  // neighbouring columns
#pragma unroll
      for (int c = 0; c < C; c += W) {
        const int col = c * 16 + tx * W;
        if (col < dh) {                  // dh is a multiple of 4 (8 for bf16): whole groups
#pragma unroll
          for (int w = 0; w < W; w += 2) store_pair(out + col + w, acc[i][c + w] * inv, acc[i][c + w + 1] * inv);
        }
      }
    }
  }
}

template <typename T, int DHP>
rocs_status_t launch(const rocs_plan* plan, int32_t n_q, int32_t H, int32_t dh, float scale, const void* Q,
                     const void* K, const void* V, const int32_t* seq_offsets, void* O, cudaStream_t stream) {
  const int32_t cands = std::max(1, kRows / n_q);
  DcaItemList items;
  if (plan->R > kThreads) {
    const rocs_status_t st = plan_dca_items(plan, cands, H, stream, &items);
    if (st != ROCS_OK) return st;
  } else {
    const int64_t total = plan_entries(plan, cands) * H;  // the blocks find their tiles themselves
    if (total > 0x7fffffffLL) return ROCS_ERR_UNSUPPORTED;
    items.num = (int32_t)total;
  }
  constexpr int smem = smem_floats<DHP>() * (int)sizeof(float);
  auto kernel = dca_simt_kernel<T, DHP>;
  ROCS_ALLOW_SMEM(kernel, smem);
  const dim3 grid((unsigned)items.num, (unsigned)std::min<int64_t>(((int64_t)cands * n_q + kRows - 1) / kRows, 65535));
  return launch_dependent(kernel, grid, kThreads, smem, stream, n_q, H, dh, scale, (const T*)Q, (const T*)K, (const T*)V,
                          plan->R, cands, plan->cand_offsets, (const DcaItem*)items.dev, seq_offsets, (T*)O);
}

template <typename T>
rocs_status_t dispatch(const rocs_plan* plan, int32_t n_q, int32_t H, int32_t dh, float scale, const void* Q,
                       const void* K, const void* V, const int32_t* seq_offsets, void* O, cudaStream_t stream) {
  // smallest compiled width that holds the head: columns beyond dh are zeros in shared memory
  if (dh <= 32) return launch<T, 32>(plan, n_q, H, dh, scale, Q, K, V, seq_offsets, O, stream);
  if (dh <= 64) return launch<T, 64>(plan, n_q, H, dh, scale, Q, K, V, seq_offsets, O, stream);
  if (dh <= 128) return launch<T, 128>(plan, n_q, H, dh, scale, Q, K, V, seq_offsets, O, stream);
  return launch<T, 256>(plan, n_q, H, dh, scale, Q, K, V, seq_offsets, O, stream);
}

}  // namespace

rocs_status_t simt_dca(rocs_dtype_t dt, const rocs_plan* plan, int32_t n_q, int32_t H, int32_t dh, float scale,
                       const void* Q, const void* K, const void* V, const int32_t* seq_offsets, void* O,
                       cudaStream_t stream) {
  if (dh > 256) return ROCS_ERR_UNSUPPORTED;
  if (plan->N == 0) return ROCS_OK;
  if (dt == ROCS_F32) return dispatch<float>(plan, n_q, H, dh, scale, Q, K, V, seq_offsets, O, stream);
  return dispatch<__nv_bfloat16>(plan, n_q, H, dh, scale, Q, K, V, seq_offsets, O, stream);
}

}  // namespace rocs
