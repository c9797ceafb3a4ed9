// Projected factorization machine, candidate rows, on the 5th-generation tensor cores:
//     FC[i] = X^C_i T[m_i] + (X^C_i X^C_i^T) P_C
// with T[r] = X^R_r^T P_R in fp32, which the request kernel in front writes transposed, [R, k, d].
//
// Tile = 128 / NC consecutive candidates of ONE request, NC = 4, 8 or 16 rows each: the box of the tensor map is NC rows of a
// candidate high, and the rows behind its last embedding arrive as zeros.  T goes in as three bf16 parts, the upper 16 bits of
// T, of what is left and of what is left then, which add up to its 24 bits: four warps split it into the tile's stage, where it
// stays as long as the stage's tiles are of that request.  (Two parts, 17 bits, are as exact on independent inputs; where X^C T is
// what little its values do not cancel of each other they are not.)  Both terms are fp32 sums and meet behind their
// products; rows in which they cancel to less than a 256th are computed by hand, both terms added up in front of the product.
// Per 64-wide slice of d shared memory holds [T_3 ; T_2 ; T_1 ; X^C tile] back to back, each part k rows (to a multiple of 8),
// so that a single tcgen05.mma per 16-deep K step computes
//     D[128, 3 kp + 128] = X^C_tile * [T_3 ; T_2 ; T_1 ; X^C_tile]^T
// whose first columns are the parts of X^C T and whose 128 x 128 tail holds every candidate's Gram matrix on the diagonal.
// A thread of the epilogue owns a row: it adds the parts up and its NC Gram values times P_C in fp32 FMA.
//
// Bound by HBM, and in small batches by what a short run of tiles takes to start and end.  In place of a candidate per warp
// on mma.sync, whose products were what took the time (some 25 cycles of a scheduler each), request kernel included: 18400
// candidates of 12 embeddings x 128, k = 16, 26.0 -> 20.2 us; 56736 of 12 x 192, k = 24, 202 -> 69.7; 32768 of 16 x 64, k = 24,
// 46.6 -> 34.7; 19200 of 4 x 128, k = 16, 24.7 -> 11.5.  The split of T is some of that: with two parts, written by the request kernel
// and loaded, 18.7 us on the first; with three so, in half as much workspace again, 20.2; split by two warps 23.1, one 29.4.
// The last product of T by itself, 16 columns for every K step, 22.2.  The tiles are walked and not listed, in any number: the
// walk is short against a tile (2700 tiles 25.3 us with the list, 23.0 walked).
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
  const __nv_bfloat16 *P, *XC;  // [n_r + n_c, k], [N, n_c, d]
  const float* TT;              // [R, k, d]
  __nv_bfloat16* FC;            // [N, n_c, k]
  uint32_t* status;
};

// KP: columns computed per row, 16 or 32.  Groups of epilogue warps: three fit the registers with 16, two with 32; they take
// tiles in turn, and the two accumulators also, which are free again as soon as a group has read them.
constexpr int kAccs = 2, kAccStride = 256;
template <int KP>
struct FmUmmaCfg {
  static constexpr int kGroups = KP == 16 ? 3 : 2;
  static constexpr int kTermWarps = 4;  // they split T
  static constexpr int kTermWarp0 = 2 + 4 * kGroups;
  static constexpr int kThreads = 32 * (kTermWarp0 + kTermWarps);
};

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// Rows whose products with their candidate's rows are all below this are computed by hand: what fp32's range cuts off of them
// may count where P_C is large.
constexpr float kSmallProduct = 0x1p-90f;
// And rows in which the two terms cancel to less than this part of the request's: what fp32 sums lose of the terms (some 2^-21 of them)
// stays below 2^-13 of the row then, a sixteenth of its rounding to bf16.  (With 64 in place of 256 independent values meet it often
// enough with two columns, one row in some thousands, to cost a batch of one round of tiles 2.8 us.)
constexpr float kCancelled = 256.f;

// The upper halves of two values as a bf16 pair, and what is left of them.
__device__ __forceinline__ uint32_t take_upper(float& a, float& b) {
  const uint32_t ua = __float_as_uint(a), ub = __float_as_uint(b);
  a -= __uint_as_float(ua & 0xffff0000u);  // exact; NaN behind an infinity, whose rows are computed by hand
  b -= __uint_as_float(ub & 0xffff0000u);
  return __byte_perm(ua, ub, 0x7632);
}

// Rows of a warp's candidates in plain fp32, by the whole warp, the request's and the candidate's own term added up before a row's
// product: for values that the parts or the Gram matrix cannot hold (an infinity, a square out of fp32's range), where the result
// has to be what fp32 arithmetic gives.  A NaN in the request's term or among a candidate's values is one either way and is not
// computed again.  Where the term or a value is infinite the sum of both terms is so at that position of d, for every row: what
// the other positions add does not show.  Half a warp per column: its lanes sum both terms up for 16 positions, and every
// lane takes all 16 into its row.  18400 candidates of 12 x 128, k = 16, with a NaN / an infinity in two of their 100 requests: 37 / 148
// us, on the warp-level kernel 40 / 40; with a thread per row, k d n_c steps one after another, 20.7 ms.
template <int NC>
__device__ __noinline__ void rows_by_hand(uint32_t rows, const __nv_bfloat16* x, const float* tt, const __nv_bfloat16* pc,
                                          int32_t n_c, int32_t d, int32_t k, __nv_bfloat16* out, int lane) {
  uint32_t nan_columns = 0, inf_columns = 0, term_blocks = 0;  // columns of the term with one, blocks of 16 positions with an infinity
#pragma unroll 4
  for (int32_t c = 0; c < k; ++c) {
    bool nan = false, inf = false;
    for (int32_t e = lane; e < d; e += 32) {
      const float t = tt[c * d + e];
      nan = nan || isnan(t);
      inf = inf || isinf(t);
      if (isinf(t)) term_blocks |= 1u << (e / 16);
    }
    if (__any_sync(0xffffffffu, nan)) nan_columns |= 1u << c;
    if (__any_sync(0xffffffffu, inf)) inf_columns |= 1u << c;
  }
  term_blocks = __reduce_or_sync(0xffffffffu, term_blocks);
  const uint32_t all_columns = k == 32 ? ~0u : (1u << k) - 1u, all_blocks = (1u << (d / 16)) - 1u;
  if (nan_columns == all_columns) return;
  const int half = lane / 16, at = lane % 16, row = min(at, n_c - 1);
#pragma unroll 1
  for (; rows != 0; rows >>= NC, x += n_c * d, out += n_c * k) {
    const uint32_t mine = rows & ((1u << NC) - 1u);
    if (mine == 0) continue;
    bool nan = false;
    uint32_t row_blocks = 0;
#pragma unroll 4
    for (int32_t v = lane; v < n_c * d / 8; v += 32) {
      const uint4 raw = reinterpret_cast<const uint4*>(x)[v];
      const uint32_t pair[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const uint32_t magnitude = pair[u / 2] >> (u % 2 * 16) & 0x7fffu;
        nan = nan || magnitude > 0x7f80u;
        if (magnitude == 0x7f80u) row_blocks |= 1u << (v * 8 % d / 16);
      }
    }
    if (__any_sync(0xffffffffu, nan)) continue;
    row_blocks = __reduce_or_sync(0xffffffffu, row_blocks);
#pragma unroll 1
    for (int32_t c0 = 0; c0 < k; c0 += 2) {  // (k is even)
      if ((nan_columns >> c0 & 3u) == 3u) continue;
      const int32_t c = c0 + half;
      uint32_t blocks = row_blocks != 0 || (inf_columns >> c0 & 3u) == 3u ? row_blocks | term_blocks : all_blocks;
      float sum = 0.f;
#pragma unroll 1
      for (; blocks != 0; blocks &= blocks - 1) {
        const int32_t e0 = 16 * (__ffs(blocks) - 1);
        float h = tt[c * d + e0 + at];
#pragma unroll 4
        for (int32_t a = 0; a < n_c; ++a) h = fmaf(__bfloat162float(pc[a * k + c]), __bfloat162float(x[a * d + e0 + at]), h);
        const uint4* of_row = reinterpret_cast<const uint4*>(x + row * d + e0);
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          const uint4 raw = of_row[v];
          const uint32_t pair[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            sum = fmaf(__uint_as_float(pair[u] << 16), __shfl_sync(0xffffffffu, h, half * 16 + v * 8 + 2 * u), sum);
            sum = fmaf(__uint_as_float(pair[u] & 0xffff0000u), __shfl_sync(0xffffffffu, h, half * 16 + v * 8 + 2 * u + 1), sum);
          }
        }
      }
      if (at < n_c && (mine >> at & 1u) != 0) out[at * k + c] = __float2bfloat16_rn(sum);
    }
  }
}

template <int NC, int KP>
__global__ void __launch_bounds__(FmUmmaCfg<KP>::kThreads, 1)
fm_umma_kernel(const __grid_constant__ CUtensorMap map_xc, const FmUmmaParams p) {
  using Cfg = FmUmmaCfg<KP>;
  constexpr int G = Cfg::kGroups;
  extern __shared__ __align__(1024) uint8_t smem[];
  float* pc = reinterpret_cast<float*>(smem + p.stages * p.stage_bytes);  // [NC][kp], zero beyond n_c rows and k columns
  uint64_t* full = reinterpret_cast<uint64_t*>(pc + NC * p.kp);
  uint64_t* empty = full + kMaxStages;
  uint64_t* tmem_full = empty + kMaxStages;
  uint64_t* tmem_empty = tmem_full + G;
  uint64_t* drain = tmem_empty + kAccs;
  uint32_t* tmem_ptr = reinterpret_cast<uint32_t*>(drain + 1);
  AbortFlag* abort_flag = reinterpret_cast<AbortFlag*>(tmem_ptr + 1);
  int32_t* scratch = reinterpret_cast<int32_t*>(tmem_ptr + 2);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if ((smem_u32(smem) & 1023u) != 0) {  // the swizzled tiles assume a 1024-byte aligned base
    if (threadIdx.x == 0) atomicCAS(p.status, 0u, kStatusFmUmma | 15);
    return;
  }
  const int32_t k_slices = p.d / 64;
  const int32_t part_bytes = p.kp * 128, slice_bytes = 3 * part_bytes + 128 * 128;
  // a contiguous run of tiles per CTA: consecutive tiles mostly share a request, whose T stays in L2
  const int32_t t_begin = (int32_t)((int64_t)blockIdx.x * p.num_tiles / gridDim.x);
  const int32_t t_end = (int32_t)((int64_t)(blockIdx.x + 1) * p.num_tiles / gridDim.x);

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(&full[s], 1 + Cfg::kTermWarps);
      mbar_init(&empty[s], 1);
    }
    for (int g = 0; g < G; ++g) mbar_init(&tmem_full[g], 1);
    for (int a = 0; a < kAccs; ++a) mbar_init(&tmem_empty[a], 4);
    mbar_init(drain, 1);
    abort_flag->v = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_ptr, kTmemCols);
    tmem_relinquish();
  }
  for (int e = threadIdx.x; e < NC * p.kp; e += Cfg::kThreads) {
    const int a = e / p.kp, c = e % p.kp;
    pc[e] = a < p.n_c && c < p.k ? __bfloat162float(p.P[(int64_t)(p.n_r + a) * p.k + c]) : 0.f;
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_ptr;
  TileWalk walk{p.offsets, p.R, 128 / NC};
  walk.start_in_block<Cfg::kThreads>(t_begin, scratch);

  if (warp == 0) {
    // ------------------------------ TMA producer ------------------------------------------
    if (elect_one()) {
      prefetch_tensormap(&map_xc);
      // X^C alone, which the request kernel in front does not write
      uint32_t it = 0;
      bool ok = true;
      for (int32_t t = t_begin; t < t_end; ++t, ++it) {
        const Tile tile = walk.take(t + 1 < t_end);
        const int s = it % p.stages;
        if (!mbar_wait(&empty[s], ((it / p.stages) & 1) ^ 1, abort_flag, p.status, kStatusFmUmma | 1)) { ok = false; break; }
        mbar_expect_tx(&full[s], k_slices * (128 * 128));
        for (int32_t ks = 0; ks < k_slices; ++ks)
          tma_load_3d(smem + s * p.stage_bytes + ks * slice_bytes + 3 * part_bytes, &map_xc, &full[s], ks * 64, 0, tile.cand0);
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
      // (to a multiple of 16: the rows behind the tile give columns that nobody reads)
      const uint32_t idesc = umma_idesc_bf16(128, (uint32_t)((3 * p.kp + 128 + 15) / 16 * 16), false, false);
      uint32_t it = 0;
      bool ok = true;
      for (int32_t t = t_begin; t < t_end; ++t, ++it) {
        const uint32_t acc = it % kAccs;
        const int s = it % p.stages;
        if (!mbar_wait(&tmem_empty[acc], ((it / kAccs) & 1) ^ 1, abort_flag, p.status, kStatusFmUmma | 2)) { ok = false; break; }
        if (!mbar_wait(&full[s], (it / p.stages) & 1, abort_flag, p.status, kStatusFmUmma | 3)) { ok = false; break; }
        tc_fence_after_sync();
        const uint32_t d_tmem = tmem_base + acc * kAccStride;
        const uint32_t st = smem_u32(smem + s * p.stage_bytes);
        for (int32_t ks = 0; ks < k_slices; ++ks) {
          const uint64_t b_desc = smem_desc_sw128(st + ks * slice_bytes, 1024, 16);                   // [T_3 ; T_2 ; T_1 ; X^C]
          const uint64_t a_desc = smem_desc_sw128(st + ks * slice_bytes + 3 * part_bytes, 1024, 16);  // X^C
#pragma unroll
          for (int k = 0; k < 4; ++k) umma_ss(d_tmem, a_desc + 2 * k, b_desc + 2 * k, idesc, (ks | k) != 0 ? 1u : 0u);
        }
        umma_commit(&empty[s]);
        umma_commit(&tmem_full[it % G]);
      }
      if (!ok) {
        umma_commit(drain);
        const uint64_t t0 = globaltimer_ns();
        while (!mbar_try_wait(drain, 0) && globaltimer_ns() - t0 < kWaitLimitNs) {}
      }
    }
  } else if (warp >= Cfg::kTermWarp0) {
    // ------------------------------ the request's term, in three parts ---------------------
    griddep_wait();  // T comes from the request kernel launched just before
    const int32_t per_row = p.d / 8, items = p.k * per_row;  // eight values of a row each; rows from k on are in no column that is kept
    constexpr int kStep = 32 * Cfg::kTermWarps, kBatch = 4;    // all loads of a batch in front of its first use
    const int32_t first = threadIdx.x - 32 * Cfg::kTermWarp0, dr = kStep / per_row, dc = kStep - dr * per_row;
    float4 v[kBatch][2];
    auto load = [&](int32_t req, int32_t i0) {
      const float4* from = reinterpret_cast<const float4*>(p.TT + (int64_t)req * p.k * p.d) + 2 * i0;
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        if (i0 + u * kStep >= items) break;
        v[u][0] = from[2 * u * kStep];
        v[u][1] = from[2 * u * kStep + 1];
      }
    };
    Tile next = walk.take(t_begin + 1 < t_end);
    load(next.req, first);
    uint32_t it = 0, since = 0;  // since: the first tile of the request
    for (int32_t t = t_begin; t < t_end; ++t, ++it) {
      const Tile tile = next;
      const uint32_t s = it % p.stages;
      const bool ok = mbar_wait(&empty[s], ((it / p.stages) & 1) ^ 1, abort_flag, p.status, kStatusFmUmma | 5);
      if (!__all_sync(0xffffffffu, ok)) break;
      if (it - since < (uint32_t)p.stages) {  // otherwise the parts are in the stage already
        uint8_t* st = smem + s * p.stage_bytes;
        int32_t row = first / per_row, chunk = first - row * per_row;
        for (int32_t i0 = first; i0 < items; i0 += kBatch * kStep) {
          if (items > kBatch * kStep && (i0 != first || it != since)) load(tile.req, i0);
#pragma unroll
          for (int u = 0; u < kBatch; ++u) {
            if (i0 + u * kStep >= items) break;
            float4 a = v[u][0], b = v[u][1];
            uint8_t* to = st + (chunk / 8) * slice_bytes + row * 128 + (((chunk % 8) ^ (row & 7)) << 4);
#pragma unroll
            for (int part = 2; part >= 0; --part)
              *reinterpret_cast<uint4*>(to + part * part_bytes) =
                  make_uint4(take_upper(a.x, a.y), take_upper(a.z, a.w), take_upper(b.x, b.y), take_upper(b.z, b.w));
            row += dr;
            chunk += dc;
            if (chunk >= per_row) {
              chunk -= per_row;
              ++row;
            }
          }
        }
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[s]);
      if (t + 1 < t_end) next = walk.take(t + 2 < t_end);
      if (next.req != tile.req) {  // asked for while this tile is on its way
        since = it + 1;
        load(next.req, first);
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
      const uint32_t acc = it % kAccs, t_row = tmem_base + acc * kAccStride + ((uint32_t)(q * 32) << 16);
      uint32_t val[KP], rem[KP], vcc[32];  // T_1, then T_2 and T_3 added up
      auto load = [&](uint32_t at, uint32_t(&r)[KP]) {
        if constexpr (KP == 16) tmem_ld_32x32b_x16(at, r); else tmem_ld_32x32b_x32(at, r);
      };
      load(t_row, val);
      load(t_row + p.kp, rem);
      tmem_ld_wait();
#pragma unroll
      for (int c = 0; c < KP; ++c) rem[c] = __float_as_uint(__uint_as_float(rem[c]) + __uint_as_float(val[c]));
      load(t_row + 2 * p.kp, val);
      tmem_ld_32x32b_x32(t_row + 3 * p.kp + q * 32, vcc);
      tmem_ld_wait();
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tmem_empty[acc]);
      bool by_hand = false;
      if (a_row < p.n_c && cand_l < tile.count) {
        uint64_t out[KP / 2];
        uint64_t square_t = 0, square_f = 0;  // of the request's term and of the sum, two chains each
#pragma unroll
        for (int c = 0; c < KP; c += 2) {
          out[c / 2] = pack2(__uint_as_float(val[c]) + __uint_as_float(rem[c]), __uint_as_float(val[c + 1]) + __uint_as_float(rem[c + 1]));
          if (c < p.k) square_t = ffma2(out[c / 2], out[c / 2], square_t);  // (k is even)
        }
        float most = 0.f;  // the largest of the row's products with its candidate's rows
#pragma unroll
        for (int j = 0; j < NC; ++j) {
          if (j >= p.n_c) break;
          // of the diagonal block the columns of the row's own candidate
          uint32_t x = vcc[j];
#pragma unroll
          for (int s = 1; s < 32 / NC; ++s) x = sub == s ? vcc[s * NC + j] : x;
          const float gram = __uint_as_float(x);
          most = fmaxf(most, fabsf(gram));
          const uint64_t gram2 = pack2(gram, gram);
#pragma unroll
          for (int c = 0; c < KP; c += 4) {
            const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(pc + j * p.kp + c);
            out[c / 2] = ffma2(gram2, w.x, out[c / 2]);
            out[c / 2 + 1] = ffma2(gram2, w.y, out[c / 2 + 1]);
          }
        }
        float f[KP];
#pragma unroll
        for (int c = 0; c < KP; c += 2) {
          unpack2(out[c / 2], f[c], f[c + 1]);
          if (c < p.k) square_f = ffma2(out[c / 2], out[c / 2], square_f);
        }
        const int64_t cand = (int64_t)tile.cand0 + cand_l;
        __nv_bfloat16* dst = p.FC + (cand * p.n_c + a_row) * p.k;
        if (p.k % 8 == 0) {
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
        float t0, t1, f0, f1;
        unpack2(square_t, t0, t1);
        unpack2(square_f, f0, f1);
        // not finite behind an infinity or a NaN among this row's values, which one of its products also gives
        by_hand = !(f0 + f1 < INFINITY) || (f0 + f1) * (kCancelled * kCancelled) < t0 + t1;
        if (most < kSmallProduct) {
          bool zeros = most == 0.f;  // a row of zeros
#pragma unroll
          for (int c = 0; c < KP; ++c) zeros = zeros && (c >= p.k || f[c] == 0.f);
          by_hand = !zeros;
        }
      }
      const uint32_t rows = __ballot_sync(0xffffffffu, by_hand);
      if (rows != 0) {
        griddep_wait();  // T is read here by threads that have not waited for it themselves
        __syncwarp();  // their values are written again
        const int64_t first = (int64_t)tile.cand0 + q * 32 / NC;  // the warp's candidates
        rows_by_hand<NC>(rows, p.XC + first * p.n_c * p.d, p.TT + (int64_t)tile.req * p.k * p.d, p.P + (int64_t)p.n_r * p.k, p.n_c, p.d, p.k,
                         p.FC + first * p.n_c * p.k, lane);
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
rocs_status_t launch(int smem, const CUtensorMap& map_xc, const FmUmmaParams& p, cudaStream_t stream) {
  ROCS_ALLOW_SMEM((fm_umma_kernel<NC, KP>), kMaxDynamicSmem);
  return launch_dependent(fm_umma_kernel<NC, KP>, dim3((unsigned)std::min(p.num_tiles, sm_count_fm_umma())), FmUmmaCfg<KP>::kThreads,
                          (size_t)smem, stream, map_xc, p);
}

int rows_of(int32_t n_c) { return n_c <= 4 ? 4 : n_c <= 8 ? 8 : 16; }

}  // namespace

// Where this kernel is the faster one of the two on bf16 rows.  fm_projection.cu's has as many candidates at work on an SM as
// warps and takes a candidate's bytes alone; this one takes a tile's 128 rows however few of them a request fills, and its run of
// tiles starts and ends slower.  Request kernel included, on a plan that is kept, that one and this one, in us:
//   few candidates per tile: 1000 requests of 4 x 128, k = 16, one / two / eight each, 13.3 / 16.4 / 24.5 and 18.8 / 18.8 / 18.9;
//   12000 x 2 of 8 x 64, k = 8, 76 and 119; 100 x 3 of 12 x 128, k = 16, 7.0 and 8.4; 1000 x 1 / 2 of 12 x 192, k = 24, 24.2 / 28.9 and
//   29.6 / 29.7
//   d = 64, the products of a candidate being short: 12 embeddings, k = 8, 1 x 3000 / 10000 / 40000 6.6 / 9.7 / 24.6 and 8.9 / 12.9 / 27.7,
//   128 x 1024 72 and 77, 100 x 10 / 100 7.0 / 11.9 and 8.6 / 13.3, 1000 x 8 / 30 17.0 / 28.0 and 16.2 / 30.1; 8 embeddings, 1 x 3000 / 5000 /
//   10000 6.4 / 7.6 / 9.8 and 8.0 / 8.6 / 10.0, 100 x 10 / 30 7.1 / 8.4 and 7.6 / 8.4
//   d = 128, k = 16, 12 embeddings in a few rounds of tiles: 1 x 1000 / 3000 / 5000 / 10000 7.0 / 8.4 / 11.1 / 15.2 and 6.8 / 9.7 / 11.4 /
//   14.3, 100 x 10 / 30 8.7 / 11.6 and 9.2 / 10.2
// 16 embeddings to 8 or 16 columns take H rounded once there (104 and 127 us on 131072 x 128, k = 16; 5.8 and 6.8 on 29).
bool fm_umma_pays(const rocs_plan* plan, int32_t n_c, int32_t d, int32_t k) {
  if (n_c == 16 && (k == 8 || k == 16)) return false;
  const int64_t N = plan->N, R = plan->R, tiles = plan_entries(plan, 128 / rows_of(n_c));
  if (R > 64 && N <= (d <= 128 ? 3 : 2) * tiles) return false;
  if (d == 64 && k <= 16 && n_c > 8 && (R <= 128 || N >= 12 * R)) return false;
  if (d == 64 && k <= 16 && n_c > 4 && n_c <= 8 && (R <= 32 ? N <= 6144 : R <= 128 && N <= 1024)) return false;
  if (d == 128 && k <= 16 && n_c > 8 && tiles > 148 && (R <= 16 ? tiles <= 5 * 148 : R <= 128 && tiles <= 256)) return false;
  return true;
}

rocs_status_t fm_umma(const rocs_plan* plan, int32_t n_r, int32_t n_c, int32_t d, int32_t k, const void* XC, const void* P,
                      const float* TT, void* FC, cudaStream_t stream) {
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
  p.stage_bytes = (3 * p.kp + 128) * d * 2;
  // (behind the last stage at least the eight rows that the products read past it)
  const int fixed = std::max(nc * p.kp * 4 + (2 * kMaxStages + 6) * 8 + 8 + 20 * 4, 1024);
  p.stages = std::min(kMaxStages, (kMaxDynamicSmem - fixed) / p.stage_bytes);
  p.P = (const __nv_bfloat16*)P; p.XC = (const __nv_bfloat16*)XC; p.TT = TT;
  p.FC = (__nv_bfloat16*)FC;
  p.status = device_status_word();
  if (!p.status) return ROCS_ERR_CUDA;
  CUtensorMap map_xc;
  if (!make_tensor_map_3d(&map_xc, XC, (uint64_t)d, (uint64_t)n_c, (uint64_t)plan->N, 64, (uint32_t)nc, (uint32_t)(128 / nc)))
    return ROCS_ERR_CUDA;
  const int smem = p.stages * p.stage_bytes + fixed;
#define ROCS_LAUNCH(NC_, KP_) return launch<NC_, KP_>(smem, map_xc, p, stream)
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
