// GLM factorization machine, candidate rows (Eq. 10, bottom row) with the optional row-axis compression
// (Eq. 6), bf16, on warp-level tensor cores:
//     YC[i] = [ X^C_i X^R_r^T , X^C_i X^C_i^T ]        r = request of candidate i
//     OC[i] = ZR[r] + W_CC YC[i]                       ZR[r] = W_CR YR[r], once per request (fp32)
//
// Takes what the tcgen05 kernel (umma_glm.cu) does not: 4 or 12 embeddings per candidate, request sides that are
// no multiple of 8.  Bound by the fixed latencies of its short chains (mma.sync, ldmatrix) with four warps per
// scheduler.  100 requests x 184 candidates, 20 + 12 embeddings x 128 with compression to 4: 32.4 us; the general
// kernel 286 us.  The compression takes the fp32 block as a bf16 pair (value and remainder) through two products, as
// exact as that kernel: error of OC against 64 bits 1.6573e-3 on 128 requests x 1024 candidates, 32 + 12 embeddings x
// 128 to 8, at 187 us; 1.9116e-3 and 140 us with the block rounded first.  The tcgen05 kernel rounds it: where both
// apply it is the faster also without the pair (128 x 1024 candidates, 32 + 16 embeddings with compression: 118 us,
// this one 145 us with 15 compute warps, 161 us with 8 that take two fragments each).
//
// A persistent CTA takes a contiguous run of tiles (tiles never cross a request); a producer warp streams the
// tiles through a TMA ring and each request's X^R, once per run of tiles of that request, through two slots.
// Fifteen compute warps take a 16-row fragment each (16 / n_c whole candidates per fragment; unused rows are
// computed and dropped).  Per 16-deep step of d a fragment is one ldmatrix, which serves as the row operand
// and, the registers being the same, as the column operand of the fragment's products with itself.
//
// Rows are permuted inside a fragment (and inside 16 rows of X^R) so that a thread ends up with four
// neighbouring columns, in either order, and the eight rows of an ldmatrix block differ modulo 8 (no bank
// conflicts under the 128-byte swizzle).  Outputs leave as 8-byte stores that fill whole 32-byte sectors.
// With compression the products are formed transposed, so that an accumulator, split into bf16 parts, is the K x N
// operand of OC = ZR + W_CC YC as it stands; W_CC is repeated for every candidate of the fragment, and the other
// candidates' rows are masked out of both operands (a NaN of one candidate must not reach another).  The raw block, if
// wanted too, is turned by movmatrix.
#include <algorithm>
#include <type_traits>

#include "rocs_internal.h"
#include "sm100_ptx.cuh"

namespace rocs {
namespace {

using namespace ptx;

constexpr int kWarps = 15;
constexpr int kThreads = (kWarps + 1) * 32;
constexpr int kMaxStages = 8;
constexpr int kGroups = 2;  // 16-column groups of the request block per pass
constexpr uint32_t kStatusGlmMma = 0x800;

struct GlmMmaParams {
  const Tile* tiles;       // the list, or null
  const int32_t* offsets;  // [R + 1]
  int32_t R, tile_cands, num_tiles;
  int32_t n_r, n_c, d, n_ro, n_co;
  int32_t frags, frag_cands;  // fragments per tile, whole candidates per fragment
  int32_t stages, stage_bytes, tx_bytes, slab_bytes, xr_bytes, xr_slab_bytes;
  const __nv_bfloat16* W;  // [n_ro + n_co, n]
  const float* ZR;         // [R, n_co, n]
  __nv_bfloat16* YC;       // [N, n_c, n] or null
  __nv_bfloat16* OC;       // [N, n_co, n]
  uint32_t* status;
};

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}
// Two fp32 values as bf16 pairs that add up to them.  Rounded value and rounded remainder: 17 bits.
__device__ __forceinline__ void split(float a, float b, uint32_t (&part)[2]) {
  part[0] = pack(a, b);
  float ra, rb;  // one packed subtraction
  asm("{\n.reg .b64 v, h;\nmov.b64 v, {%2, %3};\nmov.b64 h, {%4, %5};\nadd.rn.f32x2 v, v, h;\nmov.b64 {%0, %1}, v;\n}"
      : "=f"(ra), "=f"(rb)
      : "f"(a), "f"(b), "f"(-__uint_as_float(part[0] << 16)), "f"(-__uint_as_float(part[0] & 0xffff0000u)));
  part[1] = pack(ra, rb);
}
// Upper halves of the values, of what is left and of what is left then: every bit.  An infinity is infinite in every part,
// and what is left of a value is never 0 unless the value is, so that products with an infinity stay what they are.
__device__ __forceinline__ void split(float a, float b, uint32_t (&part)[3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const uint32_t ua = __float_as_uint(a), ub = __float_as_uint(b);
    part[i] = __byte_perm(ua, ub, 0x7632);
    const float ra = a - __uint_as_float(ua & 0xffff0000u), rb = b - __uint_as_float(ub & 0xffff0000u);
    const uint32_t least = 0x10000u;  // the smallest positive bf16
    a = fabsf(a) == INFINITY || a == 0.f ? a : ra == 0.f ? __uint_as_float((ua & 0x80000000u) | least) : ra;
    b = fabsf(b) == INFINITY || b == 0.f ? b : rb == 0.f ? __uint_as_float((ub & 0x80000000u) | least) : rb;
  }
}
__device__ __forceinline__ uint32_t transpose8x8(uint32_t v) {
  uint32_t r;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(v));
  return r;
}
// Row of index m: 4 t + {0, 1} for m = 2 t + {0, 1} and 2 further on for m + 8; the other way round from t = 2.
__device__ __forceinline__ int perm(int m) {
  const int t = (m & 7) / 2;
  return 4 * t + 2 * ((m >> 3) ^ (t >> 1)) + (m & 1);
}

// The 16 x 16 product of a 16-row fragment and 16 columns, as two 16 x 8 accumulators.
struct Acc {
  float v[2][4];
};

// COMPRESS: transposed, rows of the accumulator are columns of YC.
template <bool COMPRESS>
__device__ __forceinline__ void product(Acc& acc, const uint32_t (&frag)[4], const uint32_t (&cols)[4]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if constexpr (COMPRESS)
      mma_bf16(acc.v[h], cols, frag[h], frag[h + 2]);
    else
      mma_bf16(acc.v[h], frag, cols[h], cols[h + 2]);
  }
}

// CO8: blocks of 8 compressed outputs (0: no compression).
// WALK: the tiles are found in the offsets, otherwise read from the list.
template <int CO8, bool RAW, bool WALK>
__global__ void __launch_bounds__(kThreads, 1)
glm_mma_kernel(const __grid_constant__ CUtensorMap map_xr, const __grid_constant__ CUtensorMap map_xc,
               const GlmMmaParams p) {
  constexpr bool COMPRESS = CO8 > 0;
  extern __shared__ __align__(1024) uint8_t smem[];
  // [stages][d / 64 slabs][rows][128 bytes], [2][d / 64 slabs][n_r rounded up to 16][128 bytes]; a last fragment
  // reads up to 15 rows past its slab, which is inside what follows
  uint8_t* xr_smem = smem + p.stages * p.stage_bytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(xr_smem + 2 * p.xr_bytes + 2048);
  uint64_t* empty = full + kMaxStages;
  uint64_t* xr_full = empty + kMaxStages;
  uint64_t* xr_empty = xr_full + 2;
  AbortFlag* abort_flag = reinterpret_cast<AbortFlag*>(xr_empty + 2);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if ((smem_u32(smem) & 1023u) != 0) {  // the swizzled tiles assume a 1024-byte aligned base
    if (threadIdx.x == 0) atomicCAS(p.status, 0u, kStatusGlmMma | 15);
    return;
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], kWarps);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&xr_full[s], 1);
      mbar_init(&xr_empty[s], kWarps);
    }
    abort_flag->v = 0;
    fence_mbar_init();
  }
  __syncthreads();
  const int32_t slabs = p.d / 64;
  const int32_t t_begin = (int32_t)((int64_t)blockIdx.x * p.num_tiles / gridDim.x);
  const int32_t t_end = (int32_t)((int64_t)(blockIdx.x + 1) * p.num_tiles / gridDim.x);
  TileWalk walk{p.offsets, p.R, p.tile_cands};
  if constexpr (WALK) walk.start(t_begin, lane);

  if (warp == kWarps) {
    // ------------------------------ TMA producer ------------------------------------------
    if (elect_one()) {
      prefetch_tensormap(&map_xr);
      prefetch_tensormap(&map_xc);
      int s = 0;
      uint32_t phase = 0, it = 0, n_req = 0;
      int32_t req = -1;
      Tile next = !WALK && t_begin < t_end ? p.tiles[t_begin] : Tile{};
      for (int32_t t = t_begin; t < t_end; ++t, ++it) {
        const Tile tile = WALK ? walk.take(t + 1 < t_end) : next;
        if (!WALK && t + 1 < t_end) next = p.tiles[t + 1];
        if (tile.req != req) {
          const uint32_t x = n_req & 1;
          if (!mbar_wait(&xr_empty[x], ((n_req >> 1) & 1) ^ 1, abort_flag, p.status, kStatusGlmMma | 1)) break;
          mbar_expect_tx(&xr_full[x], p.xr_bytes);
          for (int32_t sl = 0; sl < slabs; ++sl)
            tma_load_2d(xr_smem + x * p.xr_bytes + sl * p.xr_slab_bytes, &map_xr, &xr_full[x], sl * 64, tile.req * p.n_r);
          req = tile.req;
          ++n_req;
        }
        if (!mbar_wait(&empty[s], phase ^ 1, abort_flag, p.status, kStatusGlmMma | 2)) break;
        mbar_expect_tx(&full[s], p.tx_bytes);
        for (int32_t sl = 0; sl < slabs; ++sl)
          tma_load_2d(smem + s * p.stage_bytes + sl * p.slab_bytes, &map_xc, &full[s], sl * 64, tile.cand0 * p.n_c);
        if (++s == p.stages) { s = 0; phase ^= 1; }
      }
      // loads in flight land in this CTA's shared memory: wait for them before the CTA may exit
      auto landed = [&](uint64_t* bar, uint32_t issued) {
        if (issued == 0) return;
        const uint64_t t0 = globaltimer_ns();
        while (!mbar_try_wait(bar, (issued - 1) & 1) && globaltimer_ns() - t0 < kWaitLimitNs) {}
      };
      for (int st = 0; st < p.stages; ++st) landed(&full[st], it / p.stages + (((int)(it % p.stages) > st) ? 1 : 0));
      for (uint32_t x = 0; x < 2; ++x) landed(&xr_full[x], n_req / 2 + (n_req % 2 > x ? 1 : 0));
    }
    return;
  }

  // ------------------------------ compute warps --------------------------------------------
  const int g = lane / 4, tq = lane % 4;
  const int32_t n_r = p.n_r, n_c = p.n_c, n = n_r + n_c;
  const int32_t frag_rows = p.frag_cands * n_c;  // rows of a fragment that are candidates of its own
  // ldmatrix: lane l gives the address of row l % 8 of block l / 8; blocks (m lo, k lo), (m hi, k lo), (m lo, k hi), (m hi, k hi)
  const int lrow = perm((lane & 7) + ((lane >> 3) & 1) * 8);
  const int lk = lane >> 4;
  // the two rows of an accumulator that this thread holds, and the four columns 4 tq ..
  const int rows[2] = {perm(g), perm(g + 8)};
  const int row_cand[2] = {rows[0] / n_c, rows[1] / n_c};  // candidate of the fragment they belong to
  const int col_cand = 4 * tq < frag_rows ? 4 * tq / n_c : -1;  // and that of fragment rows 4 tq .. as columns
  const int32_t own_col = n_r + 4 * tq - col_cand * n_c;   // output column of those
  const bool swap = tq >= 2;  // the first of the two accumulators holds columns 4 tq + 2, 4 tq + 3
  auto in_order = [&](uint32_t a, uint32_t b) { return swap ? make_uint2(b, a) : make_uint2(a, b); };
  // rows of YC that this thread holds as an operand of the compression: which candidate's
  const int k_cand[2] = {perm(2 * tq) / n_c, perm(2 * tq + 8) / n_c};
  uint32_t wa[4] = {0u, 0u, 0u, 0u};  // W_CC: rows = outputs, k = rows of the fragment in permuted order
  if constexpr (COMPRESS) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int o = g + (i & 1) * 8;
      const int a = perm(2 * tq + (i >> 1) * 8);  // and a + 1
      if (o < p.n_co && a < frag_rows) {
        const __nv_bfloat16* w = p.W + (int64_t)(p.n_ro + o) * n + n_r + a % n_c;
        wa[i] = pack(__bfloat162float(w[0]), __bfloat162float(w[1]));
      }
    }
  }
  bool zr_ready = false;
  int s = 0;
  uint32_t phase = 0, n_req = 0;
  int32_t req = -1;
  uint32_t xr_slot = 0;
  Tile next = !WALK && t_begin < t_end ? p.tiles[t_begin] : Tile{};
  for (int32_t t = t_begin; t < t_end; ++t) {
    const Tile tile = WALK ? walk.take(t + 1 < t_end) : next;
    if (!WALK && t + 1 < t_end) next = p.tiles[t + 1];
    if (tile.req != req) {
      __syncwarp();
      if (req >= 0 && lane == 0) mbar_arrive(&xr_empty[xr_slot]);
      xr_slot = n_req & 1;
      if (!mbar_wait(&xr_full[xr_slot], (n_req >> 1) & 1, abort_flag, p.status, kStatusGlmMma | 3)) break;
      ++n_req;
      req = tile.req;
    }
    const int32_t cand_first = warp * p.frag_cands;  // of this warp, in the tile
    const bool active = warp < p.frags && cand_first < tile.count;
    if (COMPRESS && !zr_ready && active) {
      griddep_wait();  // the request kernel must have finished before its result is read
      zr_ready = true;
    }
    if (!mbar_wait(&full[s], phase, abort_flag, p.status, kStatusGlmMma | 4)) break;
    if (active) {
      const uint32_t xc = smem_u32(smem + s * p.stage_bytes), xr = smem_u32(xr_smem + xr_slot * p.xr_bytes);
      const uint32_t xr_row = xr + lrow * 128;
      const int xc_r = warp * frag_rows + lrow;
      const uint32_t xc_row = xc + xc_r * 128;
      const int xc_sw = xc_r & 7;
      const int xr_sw = lrow & 7;
      const float* zr = COMPRESS ? p.ZR + (int64_t)tile.req * p.n_co * n : nullptr;
      // request term of outputs g (and g + 8) at four columns from col
      auto load_z = [&](float4 (&z)[CO8 > 0 ? CO8 : 1], int32_t col, bool in) {
#pragma unroll
        for (int b = 0; b < CO8; ++b) {
          z[b] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (in && g + 8 * b < p.n_co) z[b] = *reinterpret_cast<const float4*>(zr + (g + 8 * b) * n + col);
        }
      };
      // One 16-column group: columns from col0.  self: the columns are the fragment's own rows, of
      // which each candidate keeps its own.
      // parts: bf16 parts of a value in the compression.  redo: the candidates to do (a bit each; ~0: all, and the raw block).
      // nan: those with a NaN among their outputs.
      uint32_t nan = 0;
      auto emit = [&](const Acc& acc, const float4 (&z)[CO8 > 0 ? CO8 : 1], int32_t col0, bool self, auto parts, uint32_t redo) {
        const int32_t last = min(p.frag_cands, tile.count - cand_first);
        const int64_t cand = tile.cand0 + cand_first;
        const int32_t col = self ? own_col : col0 + 4 * tq;
        const bool in_cols = self ? col_cand >= 0 : col < n_r;
        auto store_raw = [&](int h, uint32_t first, uint32_t second) {
          if (in_cols && row_cand[h] < last && (!self || col_cand == row_cand[h]))
            *reinterpret_cast<uint2*>(p.YC + (cand * n_c + rows[h]) * n + col) = in_order(first, second);
        };
        if constexpr (!COMPRESS) {
#pragma unroll
          for (int h = 0; h < 2; ++h)
            store_raw(h, pack(acc.v[0][2 * h], acc.v[0][2 * h + 1]), pack(acc.v[1][2 * h], acc.v[1][2 * h + 1]));
        } else {
          // of yt[j][h]: columns of index 8 j + g of YC, fragment rows of index 8 h + 2 tq, + 1
          constexpr int kParts = decltype(parts)::value;
          if (RAW && kParts == 2) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const uint32_t first = transpose8x8(pack(acc.v[h][0], acc.v[h][1])),
                             second = transpose8x8(pack(acc.v[h][2], acc.v[h][3]));
              store_raw(h, first, second);
            }
          }
          for (int c = 0; c < last; ++c) {
            if ((redo >> c & 1u) == 0u) continue;
            const uint32_t k0 = k_cand[0] == c ? 0xffffffffu : 0u, k1 = k_cand[1] == c ? 0xffffffffu : 0u;
            const uint32_t w[4] = {wa[0] & k0, wa[1] & k0, wa[2] & k1, wa[3] & k1};
            float o[2][4];
#pragma unroll
            for (int b = 0; b < 2; ++b) {
              const float4 zb = b < CO8 ? z[b < CO8 ? b : 0] : make_float4(0.f, 0.f, 0.f, 0.f);
              o[0][2 * b] = swap ? zb.z : zb.x;
              o[0][2 * b + 1] = swap ? zb.w : zb.y;
              o[1][2 * b] = swap ? zb.x : zb.z;
              o[1][2 * b + 1] = swap ? zb.y : zb.w;
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              uint32_t yt[2][kParts];
              split(acc.v[0][2 * j], acc.v[0][2 * j + 1], yt[0]);
              split(acc.v[1][2 * j], acc.v[1][2 * j + 1], yt[1]);
#pragma unroll
              for (int i = 0; i < kParts; ++i) mma_bf16(o[j], w, yt[0][i] & k0, yt[1][i] & k1);
            }
            const bool in = in_cols && (!self || col_cand == c);
            float sum = 0.f;
#pragma unroll
            for (int b = 0; b < CO8; ++b)
              if (in && g + 8 * b < p.n_co) sum += (o[0][2 * b] + o[0][2 * b + 1]) + (o[1][2 * b] + o[1][2 * b + 1]);
            if (isnan(sum)) nan |= 1u << c;
            __nv_bfloat16* oc = p.OC + (cand + c) * p.n_co * n + col;
#pragma unroll
            for (int b = 0; b < CO8; ++b)
              if (in && g + 8 * b < p.n_co)
                *reinterpret_cast<uint2*>(oc + (g + 8 * b) * n) =
                    in_order(pack(o[0][2 * b], o[0][2 * b + 1]), pack(o[1][2 * b], o[1][2 * b + 1]));
          }
        }
      };
      // request columns in passes of kGroups groups of 16, the fragment's own block in the first of them
      auto columns = [&](auto parts, uint32_t redo) {
        for (int32_t col0 = 0; col0 < n_r; col0 += 16 * kGroups) {
          // in front of the products, which hide the latency (with the loads behind them they took half of the time)
          float4 z[kGroups][CO8 > 0 ? CO8 : 1], z_own[CO8 > 0 ? CO8 : 1];
          if constexpr (COMPRESS) {
#pragma unroll
            for (int q = 0; q < kGroups; ++q) load_z(z[q], col0 + 16 * q + 4 * tq, col0 + 16 * q + 4 * tq < n_r);
            load_z(z_own, own_col, col0 == 0 && col_cand >= 0);
          }
          Acc acc[kGroups] = {}, own = {};
          const bool second = col0 + 16 < n_r;
          auto step = [&](int32_t sl, int k, bool first) {
            const int chunk = 2 * k + lk;
            uint32_t xf[4], xq[kGroups][4];
            ldsm_x4(xc_row + sl * p.slab_bytes + ((chunk ^ xc_sw) << 4), xf);
            const uint32_t at = xr_row + col0 * 128 + sl * p.xr_slab_bytes + ((chunk ^ xr_sw) << 4);
            ldsm_x4(at, xq[0]);
            if (second) ldsm_x4(at + 2048, xq[1]);
            product<COMPRESS>(acc[0], xf, xq[0]);
            if (second) product<COMPRESS>(acc[1], xf, xq[1]);
            if (first) product<COMPRESS>(own, xf, xf);
          };
          if (col0 == 0) {
            for (int32_t sl = 0; sl < slabs; ++sl)
#pragma unroll
              for (int k = 0; k < 4; ++k) step(sl, k, true);
          } else {
            for (int32_t sl = 0; sl < slabs; ++sl)
#pragma unroll
              for (int k = 0; k < 4; ++k) step(sl, k, false);
          }
          emit(acc[0], z[0], col0, false, parts, redo);
          if (second) emit(acc[1], z[1], col0 + 16, false, parts, redo);
          if (col0 == 0) emit(own, z_own, n_r, true, parts, redo);
        }
      };
      columns(std::integral_constant<int, 2>(), ~0u);
      if constexpr (COMPRESS) {
        // Perhaps of an infinity, or of a value that rounds to one.  Decided from a candidate's own outputs, for it alone.
        const uint32_t redo = __reduce_or_sync(0xffffffffu, nan);
        if (redo != 0u) columns(std::integral_constant<int, 3>(), redo);
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[s]);
    if (++s == p.stages) { s = 0; phase ^= 1; }
  }
  if (!zr_ready) griddep_wait();  // complete only behind the request kernel, for whoever waits for this grid
}

int sm_count_glm_mma() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  }
  return n;
}

struct Layout {
  int32_t frags, frag_cands, tile_cands, tile_rows, stages, stage_bytes, tx_bytes, slab_bytes, xr_bytes, xr_slab_bytes, smem;
};

Layout layout(int32_t n_r, int32_t n_c, int32_t d) {
  Layout L{};
  L.frag_cands = 16 / n_c;
  L.frags = std::min(kWarps, 64 * 1024 / (L.frag_cands * n_c * d * 2));  // wide rows: fewer, so that stages stay <= 64 KB
  L.tile_cands = L.frags * L.frag_cands;
  L.tile_rows = L.tile_cands * n_c;
  L.slab_bytes = (L.tile_rows * 128 + 1023) / 1024 * 1024;  // the swizzle repeats every 1024 bytes
  L.stage_bytes = d / 64 * L.slab_bytes;
  L.tx_bytes = d / 64 * L.tile_rows * 128;
  L.xr_slab_bytes = (n_r + 15) / 16 * 16 * 128;
  L.xr_bytes = d / 64 * L.xr_slab_bytes;
  const int32_t fixed = 2 * L.xr_bytes + 2048 + (2 * kMaxStages + 4) * 8 + 16;
  L.stages = std::min(kMaxStages, (kMaxDynamicSmem - fixed) / L.stage_bytes);
  L.smem = fixed + L.stages * L.stage_bytes;
  return L;
}

}  // namespace

bool glm_mma_supported(int32_t n_r, int32_t n_c, int32_t d, int32_t n_co) {
  if (n_c < 4 || n_c > 16 || n_c % 4 != 0 || n_r < 4 || n_r > 128 || n_r % 4 != 0) return false;
  if (d % 64 != 0 || d < 64 || d > 256 || n_co > 16) return false;
  return layout(n_r, n_c, d).stages >= 2;
}

rocs_status_t glm_mma_tiles(const rocs_plan* plan, int32_t n_r, int32_t n_c, int32_t d, cudaStream_t stream, TileList* out) {
  return plan_tile_runs(plan, layout(n_r, n_c, d).tile_cands, stream, out);
}

rocs_status_t glm_mma(const rocs_plan* plan, int32_t n_r, int32_t n_c, int32_t d, const void* XR, const void* XC,
                      const void* W, int32_t n_ro, int32_t n_co, void* YC, void* OC, const float* zr_workspace,
                      cudaStream_t stream) {
  if (plan->N == 0) return ROCS_OK;
  const bool compress = W != nullptr && OC != nullptr && n_co > 0;
  if (!compress && YC == nullptr) return ROCS_OK;
  const Layout L = layout(n_r, n_c, d);
  TileList tl;
  const rocs_status_t st = plan_tile_runs(plan, L.tile_cands, stream, &tl);
  if (st != ROCS_OK) return st;
  if (tl.num == 0) return ROCS_OK;
  CUtensorMap map_xr, map_xc;
  if (!make_tensor_map_2d(&map_xr, XR, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)plan->R * n_r, (uint64_t)d,
                          (uint64_t)d, (uint32_t)(L.xr_slab_bytes / 128), 64, true) ||
      !make_tensor_map_2d(&map_xc, XC, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)plan->N * n_c, (uint64_t)d,
                          (uint64_t)d, (uint32_t)L.tile_rows, 64, true))
    return ROCS_ERR_CUDA;
  uint32_t* status = device_status_word();
  if (!status) return ROCS_ERR_CUDA;
  GlmMmaParams p{};
  p.tiles = tl.dev;
  p.offsets = plan->cand_offsets;
  p.R = plan->R;
  p.tile_cands = L.tile_cands;
  p.num_tiles = tl.num;
  p.n_r = n_r; p.n_c = n_c; p.d = d; p.n_ro = n_ro; p.n_co = n_co;
  p.frags = L.frags; p.frag_cands = L.frag_cands;
  p.stages = L.stages; p.stage_bytes = L.stage_bytes; p.tx_bytes = L.tx_bytes; p.slab_bytes = L.slab_bytes;
  p.xr_bytes = L.xr_bytes; p.xr_slab_bytes = L.xr_slab_bytes;
  p.W = (const __nv_bfloat16*)W; p.ZR = zr_workspace;
  p.YC = (__nv_bfloat16*)YC; p.OC = (__nv_bfloat16*)OC;
  p.status = status;
  // The request kernel runs directly in front on the same stream and releases its dependents at once:
  // this kernel streams X^C beside it and waits for it only before it reads ZR, if it does.
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)std::min(tl.num, sm_count_glm_mma()));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = (size_t)L.smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
#define ROCS_GLM_LAUNCH_AS(...)                                                  \
  do {                                                                           \
    auto kernel = glm_mma_kernel<__VA_ARGS__>;                                   \
    ROCS_ALLOW_SMEM(kernel, kMaxDynamicSmem);                                    \
    ROCS_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, map_xr, map_xc, p));          \
    return ROCS_OK;                                                              \
  } while (0)
#define ROCS_GLM_LAUNCH(C_, R_)                                                  \
  do {                                                                           \
    if (tl.dev == nullptr) ROCS_GLM_LAUNCH_AS(C_, R_, true);                     \
    ROCS_GLM_LAUNCH_AS(C_, R_, false);                                           \
  } while (0)
  if (!compress) ROCS_GLM_LAUNCH(0, true);
  if (n_co <= 8 && YC) ROCS_GLM_LAUNCH(1, true);
  if (n_co <= 8) ROCS_GLM_LAUNCH(1, false);
  if (YC) ROCS_GLM_LAUNCH(2, true);
  ROCS_GLM_LAUNCH(2, false);
#undef ROCS_GLM_LAUNCH
#undef ROCS_GLM_LAUNCH_AS
}

}  // namespace rocs
