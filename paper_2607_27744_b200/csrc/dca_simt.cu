// Cross attention (Eq. 13) on the CUDA cores: fp32 FMA arithmetic on fp32 or bf16 storage.  Carries the
// fp32 path and the head dimensions the tensor-core kernel does not take.
//
// One block per (tile of 32 query rows of one request, head): the tile's queries stay in shared memory,
// the request's keys and values come through it in blocks of 64, read once per tile and in place (never
// copied per candidate).  A group of 128 threads as 8 x 16, two groups with every other block where a request has several;
// a thread owns 4 query rows and, of a block, 4 keys for
// the scores and DHP / 16 columns for the output, so eight 16-byte shared-memory reads feed 64 FMAs.  The
// running maximum and normaliser of a row live in the 16 neighbouring lanes that share it.  K_{j+1} is
// fetched while the softmax and P V of block j run, V_{j+1} while the scores of block j + 1 do.
//
// What bounds it: shared-memory reads and the FMA pipe about equally (ncu: L1/shared 67 %, FMA 48 % of
// active cycles), and the last blocks (1.3 waves at the size below).  Measured on 2613 candidates of 24
// requests x 8 heads of 64 over 64..384 keys, fp32: 69 us; one warp per query row, which re-read the keys
// for every row, 1450 us.  32 rows and not 64: ragged requests leave less of a tile empty (74 us with 64);
// 8 x 4 scores per thread 71-90 us, packed fma.rn.f32x2 68 us: the reads, not the issue slots, are the limit.
// A row is computed from its own request's keys alone, in a sequence that the batch's shape fixes (whether its blocks of keys go to
// one group or two follows from the average length and the number of tiles): for a batch of given shape results are deterministic
// and independent of the other candidates' values (Eq. 1), in batches of different shape the last bits can differ.
#include <algorithm>

#include "rocs_internal.h"
#include "sm100_ptx.cuh"
#include "simt_util.cuh"

namespace rocs {
namespace {

constexpr int kRows = 32, KEYS = 64, kGroup = 128;

template <int DHP, int KS>
constexpr int smem_floats() {
  constexpr int S = DHP + 4, group = 2 * KEYS * S + kRows * (KEYS + 4);
  constexpr int part = kRows * S;  // what a group leaves for the first one, over its keys and values
  static_assert(KS == 1 || part <= 2 * KEYS * S, "a part fits the group's keys and values");
  return kRows * S + KS * group;
}

// KS groups of 128 threads take the blocks of keys in turn.
template <typename T, int DHP, int KS>
__global__ void __launch_bounds__(kGroup* KS, KS == 1 ? (DHP <= 64 ? 4 : DHP <= 128 ? 2 : 1) : KS == 2 && DHP <= 64 ? 2 : 1) dca_simt_kernel(
    int32_t n_q, int32_t H, int32_t dh, float scale, const T* __restrict__ Q, const T* __restrict__ K,
    const T* __restrict__ V, int32_t R, int32_t cands_per_tile, const int32_t* __restrict__ cand_offsets,
    const DcaItem* __restrict__ items, const int32_t* __restrict__ seq_offsets, T* __restrict__ O) {
  constexpr int S = DHP + 4;           // row stride in floats: 16-byte reads of 8 rows hit 8 different bank groups
  constexpr int C = DHP / 16;          // output columns per thread
  constexpr int J = KEYS / 16;         // keys of a block per thread
  constexpr int kPStride = KEYS + 4;
  constexpr int kThreads = kGroup * KS;
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x % kGroup, group = threadIdx.x / kGroup, tx = tid % 16, ty = tid / 16;
  float* qs = sm;                      // [32][S]
  float* ks = qs + kRows * S + group * (2 * KEYS * S + kRows * kPStride);  // [KEYS][S]
  float* vs = ks + KEYS * S;           // [KEYS][S]
  float* ps = vs + KEYS * S;           // [32][kPStride]
  ptx::griddep_wait_for(Q, K, V, cand_offsets, items, seq_offsets);
  ptx::griddep_launch_dependents();
  DcaItem item;
  if (items != nullptr) {
    item = items[blockIdx.x];
  } else {
    const FoundTile f = find_tile_in_block<kThreads>(R, cands_per_tile, H, cand_offsets, blockIdx.x);
    item = DcaItem{f.req, f.cand0, f.count, f.head};
  }
  auto group_sync = [&]() {
    if constexpr (KS == 1) __syncthreads(); else asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(kGroup) : "memory");
  };
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
    const int32_t first = group * KEYS;
    if (L > 0) rows_to_shared_async<T, DHP>(Q + q0, hd, rows, kRows, dh, qs, S, threadIdx.x, kThreads);
    if (first < L) rows_to_shared_async<T, DHP>(kg + first * hd, hd, min(KEYS, L - first), KEYS, dh, ks, S, tid, kGroup);
    cp_async_commit();
    if (first < L) rows_to_shared_async<T, DHP>(vg + first * hd, hd, min(KEYS, L - first), KEYS, dh, vs, S, tid, kGroup);
    cp_async_commit();
    if constexpr (KS > 1) {  // everybody's share of Q
      cp_async_wait<1>();
      __syncthreads();
    }
    for (int32_t j0 = first; j0 < L; j0 += KS * KEYS) {
      const int32_t next = L - j0 - KS * KEYS;  // keys from the group's next block on
      cp_async_wait<1>();                       // K_j (and Q) have landed, V_j may still be on its way
      group_sync();
      float s[4][J];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < J; ++j) s[i][j] = 0.f;
#pragma unroll 4
      for (int e = 0; e < DHP; e += 4) {
        float4 a[4], b[J];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(qs + (ty * 4 + i) * S + e);
#pragma unroll
        for (int j = 0; j < J; ++j) b[j] = *reinterpret_cast<const float4*>(ks + (tx + 16 * j) * S + e);
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < J; ++j) s[i][j] = fmaf(lane_of(a[i], c), lane_of(b[j], c), s[i][j]);
      }
      group_sync();  // K_j is read: its buffer takes the group's next
      if (next > 0)
        rows_to_shared_async<T, DHP>(kg + (int64_t)(j0 + KS * KEYS) * hd, hd, min(KEYS, next), KEYS, dh, ks, S, tid, kGroup);
      cp_async_commit();
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float mx = -INFINITY;
#pragma unroll
        for (int j = 0; j < J; ++j) {
          s[i][j] = j0 + tx + 16 * j < L ? s[i][j] * scale : -INFINITY;
          mx = fmaxf(mx, s[i][j]);
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const float m_new = fmaxf(m[i], mx);
        const float corr = m[i] == -INFINITY ? 0.f : expf(m[i] - m_new);
        float sum = 0.f;
#pragma unroll
        for (int j = 0; j < J; ++j) {
          // (scores that are all -inf so far have no weight: finite ones may follow, or be another group's)
          const float p = j0 + tx + 16 * j < L && (mx != -INFINITY || s[i][j] != -INFINITY) ? expf(s[i][j] - m_new) : 0.f;
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
      group_sync();        // V_j for everybody; the P rows of a warp are its own
#pragma unroll 2
      for (int k = 0; k < KEYS; k += 4) {
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
      group_sync();  // V_j is read: its buffer takes the group's next
      if (next > 0)
        rows_to_shared_async<T, DHP>(vg + (int64_t)(j0 + KS * KEYS) * hd, hd, min(KEYS, next), KEYS, dh, vs, S, tid, kGroup);
      cp_async_commit();
    }
    constexpr int W = C == 2 ? 2 : 4;  // neighbouring columns
    if constexpr (KS > 1) {
      // the groups' parts, added up by the first in the order of the groups: row by row S floats, maximum and
      // normaliser behind the columns
      cp_async_wait<0>();
      if (group > 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float* part = ks + (ty * 4 + i) * S;
#pragma unroll
          for (int c = 0; c < C; c += W)
#pragma unroll
            for (int w = 0; w < W; ++w) part[c * 16 + tx * W + w] = acc[i][c + w];
          if (tx == 0) {
            part[DHP] = m[i];
            part[DHP + 1] = l[i];
          }
        }
      }
      __syncthreads();
      if (group == 0) {
#pragma unroll
        for (int g = 1; g < KS; ++g) {
          const float* other = ks + g * (2 * KEYS * S + kRows * kPStride);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float* part = other + (ty * 4 + i) * S;
            const float m_o = part[DHP], l_o = part[DHP + 1], m_new = fmaxf(m[i], m_o);
            // a part whose scores are all -inf, or that has no keys, adds nothing
            const float a = m[i] == -INFINITY ? 0.f : expf(m[i] - m_new), b = m_o == -INFINITY ? 0.f : expf(m_o - m_new);
            l[i] = l[i] * a + l_o * b;
            m[i] = m_new;
#pragma unroll
            for (int c = 0; c < C; c += W)
#pragma unroll
              for (int w = 0; w < W; ++w) acc[i][c + w] = acc[i][c + w] * a + part[c * 16 + tx * W + w] * b;
          }
        }
      }
    }
    if (group == 0) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int row = ty * 4 + i;
        if (row >= rows) continue;
        const float inv = L > 0 ? 1.f / l[i] : 0.f;
        T* out = O + q0 + (int64_t)row * hd;
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
    if constexpr (KS > 1) __syncthreads();  // the next rows' operands come where the parts are
  }
}

template <typename T, int DHP, int KS>
rocs_status_t launch(const rocs_plan* plan, int32_t n_q, int32_t H, int32_t dh, float scale, const void* Q,
                     const void* K, const void* V, const int32_t* seq_offsets, void* O, const DcaItemList& items,
                     int32_t cands, cudaStream_t stream) {
  constexpr int smem = smem_floats<DHP, KS>() * (int)sizeof(float);
  static_assert(smem <= kMaxDynamicSmem - 256, "shared memory of an SM, less what the search for the tile takes");
  auto kernel = dca_simt_kernel<T, DHP, KS>;
  ROCS_ALLOW_SMEM(kernel, smem);
  const dim3 grid((unsigned)items.num, (unsigned)std::min<int64_t>(((int64_t)cands * n_q + kRows - 1) / kRows, 65535));
  return launch_dependent(kernel, grid, kGroup * KS, smem, stream, n_q, H, dh, scale, (const T*)Q, (const T*)K, (const T*)V,
                          plan->R, cands, plan->cand_offsets, (const DcaItem*)items.dev, seq_offsets, (T*)O);
}

template <typename T>
rocs_status_t dispatch(const rocs_plan* plan, int32_t n_q, int32_t H, int32_t dh, float scale, const void* Q,
                       const void* K, const void* V, const int32_t* seq_offsets, int64_t T_rows, void* O, cudaStream_t stream) {
  const int32_t cands = std::max(1, kRows / n_q);
  DcaItemList items;
  if (plan->R > kGroup) {
    const rocs_status_t st = plan_dca_items(plan, cands, H, stream, &items);
    if (st != ROCS_OK) return st;
  } else {
    const int64_t total = plan_entries(plan, cands) * H;  // the blocks find their tiles themselves
    if (total > 0x7fffffffLL) return ROCS_ERR_UNSUPPORTED;
    items.num = (int32_t)total;
  }
#define ROCS_LAUNCH(DHP_, KS_) return launch<T, DHP_, KS_>(plan, n_q, H, dh, scale, Q, K, V, seq_offsets, O, items, cands, stream)
  // Two groups share the blocks of a request that has more than one.  One group and two, 1 x 25 candidates x 2 heads of 64
  // over 72..144 keys 9.9 and 8.5 us, 1 x 288 x 16 heads of 32 over 58..116 8.4 and 6.9 us, 24 x 109 x 8 heads of 64 over
  // 64..384 the same; four groups with blocks of 32 keys 9.3, 7.8 and 83 us for 69: an SM's FMAs are then the limit.
  // 64 wide they also pay in long grids (100 x 27 candidates x 8 heads over 200..400 keys 101 and 93 us, 20 x 60 over 70..140
  // 28.7 and 26.1); 32 wide, where twice the blocks of one group fit an SM, not (76 x 9 x 16 heads over 51..103 29.7 and 38.1).
  const int64_t keys = T_rows / plan->R;  // of an average request
  constexpr int32_t kOneRound = 296;  // blocks of two groups
  const bool two = keys > KEYS && (dh > 32 || items.num <= kOneRound);
  // smallest compiled width that holds the head: columns beyond dh are zeros in shared memory
  if (dh <= 32) {
    if (two) ROCS_LAUNCH(32, 2);
    ROCS_LAUNCH(32, 1);
  }
  if (dh <= 64) {
    if (two) ROCS_LAUNCH(64, 2);
    ROCS_LAUNCH(64, 1);
  }
  if (dh <= 128) ROCS_LAUNCH(128, 1);
  ROCS_LAUNCH(256, 1);
#undef ROCS_LAUNCH
}

}  // namespace

rocs_status_t simt_dca(rocs_dtype_t dt, const rocs_plan* plan, int32_t n_q, int32_t H, int32_t dh, float scale,
                       const void* Q, const void* K, const void* V, const int32_t* seq_offsets, int64_t T, void* O,
                       cudaStream_t stream) {
  if (dh > 256) return ROCS_ERR_UNSUPPORTED;
  if (plan->N == 0) return ROCS_OK;
  if (dt == ROCS_F32) return dispatch<float>(plan, n_q, H, dh, scale, Q, K, V, seq_offsets, T, O, stream);
  return dispatch<__nv_bfloat16>(plan, n_q, H, dh, scale, Q, K, V, seq_offsets, T, O, stream);
}

}  // namespace rocs
