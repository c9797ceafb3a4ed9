// Group-wise cross attention, candidate side (Eq. 13), with the request's K/V shared inside the
// kernel (Section 4.3.1):  O[i,t,h,:] = softmax_j(scale <Q[i,t,h,:], K[r,j,h,:]>) V[r,j,h,:],  r = m_i.
//
// Candidates of one request are stacked in the tile M dimension: a work item is one head of one
// 128-row query tile of a request; K/V are addressed per request through seq_offsets and read in
// 128-key blocks, nothing is replicated per candidate (tiles of the same request and head are
// consecutive items, so their K/V blocks are read from L2 at about the same time).
//
// Head dimensions 64 (128-key blocks), 128 (64-key blocks: tensor memory holds S, P and O of both
// sides in 512 columns either way) and 32 (128-key blocks, operand rows of 64 bytes under the 64-byte
// swizzle); the description below gives the figures of the first.
//
// One persistent CTA per SM runs TWO independent item streams (sides A and B), 20 warps:
//   warps 16,19 TMA producers of sides A, B: the Q tile of the item, then its K and V blocks through a ring of
//               slots that hold one block each, in the order of their use (K_0, K_1, V_0, K_2, V_1, ...): a K
//               block gives its slot back when its S is done, half a block before its V does.  With a stage
//               per (K_j, V_j) pair two stages were all that fits at dh = 128 and the issuer waited for them
//               (821 candidates x 32 query tokens, 4 heads of 128, 500..1500 keys: 113 us, 90 us with slots)
//   warps 17,18 tcgen05.mma issuers of sides A, B:  S = Q K_j^T (128x128x64, operands in shared memory)
//               and O += P V_j (128x64x128, P read from tensor memory, V from shared memory); the last block's
//               products end at the next multiple of 16 keys
//   warps 0-15  softmax: 8 warps per side, TWO threads per query row, each owning 64 of the 128 key
//               columns of a block: S from TMEM into registers (one read), exp2 on scaled scores,
//               fp32 partial sums, P rounded to bf16 and stored to tensor memory.
// Tensor memory per side (256 columns): S [0,128) fp32, P [128,192) bf16 pairs, O [192,256) fp32.
// P has its own columns, so S_{j+1} is issued as soon as S_j sits in registers, and the wait on
// P V_{j-1} comes in the middle of block j, just before P_j starts to overwrite P_{j-1}.
//
// A batch with no more items than SMs would leave most of them idle and run an item's key blocks in one chain: there
// a cluster of 1 to 8 CTAs takes one item (SPLIT), each of its 2 to 16 sides a run of the item's key blocks with a
// reference of its own.  The sides leave their unnormalised outputs, references and sums in shared memory and the
// cluster adds them up, each CTA a share of the rows, through distributed shared memory.  1721 candidates of 3
// requests x 8 heads, 1000 to 2048 keys (120 items): whole pass with the projection 32.7 us unsplit, 22.2 us split.
//
// Reference of the softmax: the maximum over the row's FIRST 32 keys, rounded up to an integer, found
// by both threads of the row (each scans those columns, so they agree bit for bit without
// talking) and never moved: later blocks need no maximum, no rescaling of O and no exchange.
// fp32 holds 2^x up to x = 128, so a row overflows only if a later score exceeds that maximum by about
// 88 nats; such a row shows Inf/NaN in its sums at the end of the item and is then
// computed again by its two threads alone in plain fp32 loops (slow, correct, reached only by inputs
// whose scores span more than fp32's exponent range).  Every decision inside a row is taken from that row's own values,
// so in a batch of given shape a row's bits do not depend on its neighbours' values.  They do depend on the shape: whether
// items are split, and over how many CTAs, follows from the number of items and the average sequence, and a split has
// references and an order of summation of its own.
#include <algorithm>

#include "rocs_internal.h"
#include "sm100_ptx.cuh"


namespace rocs {
namespace {

using namespace ptx;

constexpr int BQ = 128;           // query rows per tile
constexpr int kSoftmaxWarps = 16; // 8 per side
constexpr int kControlWarp0 = kSoftmaxWarps;   // warps 16, 19: TMA producers of sides A, B; 17, 18: their MMA issuers
constexpr int kThreads = (kSoftmaxWarps + 4) * 32;
constexpr int kTmemCols = 512;
constexpr uint32_t kStatusDca = 0x400;
constexpr int kSideTmemStride = 256;

// Everything that depends on the head dimension DH and the keys per block BKV.  Operand tiles are kept
// as boxes of 64 columns (128-byte rows, 128-byte swizzle): a tile of DH columns is DH / 64 boxes; a head
// dimension of 32 is one box of 32 columns (64-byte rows, 64-byte swizzle).
template <int DH_, int BKV_>
struct DcaCfg {
  static constexpr int DH = DH_, BKV = BKV_;
  static constexpr int kBoxCols = DH < 64 ? DH : 64;         // columns of a box = output columns per P V product
  static constexpr int kRowBytes = kBoxCols * 2;             // 128 or 64: also the swizzle span
  static constexpr int kBoxes = DH / kBoxCols;
  static_assert(kRowBytes == 128 || kRowBytes == 64, "operand rows");
  static constexpr int kCols = BKV / 2;                      // score columns per softmax thread
  static constexpr int kOutCols = DH / 2;                    // output columns per softmax thread
  static constexpr int kKvSlots = DH == 128 ? 5 : DH == 64 ? 6 : 8;  // per side, one K or V block each
  static constexpr int kQBoxBytes = BQ * kRowBytes, kQBytes = kBoxes * kQBoxBytes;
  static constexpr int kKvBoxBytes = BKV * kRowBytes, kKBytes = kBoxes * kKvBoxBytes;
  // operand descriptor of a tile of 8-row groups, rows of kRowBytes
  __device__ static uint64_t desc(uint32_t addr) {
    return kRowBytes == 128 ? smem_desc_sw128(addr, 1024, 16) : smem_desc_sw64(addr, 512, 16);
  }
  // V block as the N x K operand of P V: rows are keys, boxes of output columns kKvBoxBytes apart
  __device__ static uint64_t desc_v(uint32_t addr) {
    return kRowBytes == 128 ? smem_desc_sw128(addr, 1024, kBoxes > 1 ? kKvBoxBytes : 16) : smem_desc_sw64(addr, 512, 16);
  }
  // tensor memory per side: S [0, BKV) fp32, P (one or two buffers of BKV / 2) bf16 pairs, O [.., + DH) fp32.
  // Two P buffers where they fit (dh = 128): P_j then replaces P_{j-2}, whose P V was issued in front of S_j, so the
  // arrival of S_j says that it is done and the wait in the middle of a block goes.  That wait also kept a fast warp
  // from announcing P_{j+1} before a slow one had announced P_j: each buffer has a barrier of its own instead (P_{j+2}
  // comes after S_{j+2}, which is issued when every warp has read S_{j+1}, i.e. has announced P_j).
  // 821 candidates x 32 query tokens, 4 heads of 128, 500..1500 keys: 86 us with one buffer, 79 us with two.
  static constexpr int kPBuffers = BKV + BKV + DH <= kSideTmemStride ? 2 : 1;
  static constexpr int kPColOffset = BKV, kOColOffset = BKV + kPBuffers * (BKV / 2);
  static_assert(kOColOffset + DH <= kSideTmemStride, "tensor memory columns of a side");
  static_assert(kCols == 32 || kCols == 64, "score columns per thread");
  // Shared-memory map (byte offsets from the 1024-byte aligned base); per side: one Q tile (freed when
  // the item's last S is issued, a block before its end) and a ring of K / V slots.
  static constexpr uint32_t kOffQ = 0;                                          // [2 sides][boxes][128][64] bf16
  static constexpr uint32_t kOffKv = kOffQ + 2 * kQBytes;                       // [2 sides][slots]
  static constexpr uint32_t kOffL = kOffKv + 2 * kKvSlots * kKBytes;     // partial sums [2 sides][2 halves][128] fp32
  static constexpr uint32_t kOffBar = kOffL + 2 * 2 * BQ * 4;
  // barriers, 8 bytes each, [side] innermost where there are two
  static constexpr uint32_t kBarQFull = kOffBar;                    // [2]
  static constexpr uint32_t kBarQEmpty = kBarQFull + 16;            // [2]
  static constexpr uint32_t kBarKvFull = kBarQEmpty + 16;           // [2][slots]
  static constexpr uint32_t kBarKvEmpty = kBarKvFull + 16 * kKvSlots;
  static constexpr uint32_t kBarSFull = kBarKvEmpty + 16 * kKvSlots;  // [2]
  static constexpr uint32_t kBarSEmpty = kBarSFull + 16;
  static constexpr uint32_t kBarPFull = kBarSEmpty + 16;            // [2][2 buffers]
  static constexpr uint32_t kBarOFull = kBarPFull + 32;
  static constexpr uint32_t kBarPair = kBarOFull + 16;              // [8]: the two warps that share 32 query rows
  static constexpr uint32_t kBarDrain = kBarPair + 64;              // [2]
  static constexpr uint32_t kBarInfoFull = kBarDrain + 16;          // [2][2 slots]
  static constexpr uint32_t kBarInfoEmpty = kBarInfoFull + 32;      // [2][2 slots]
  static constexpr uint32_t kBarTail = kBarInfoEmpty + 32;          // [2]
  static constexpr uint32_t kOffInfo = (kBarTail + 16 + 15) / 16 * 16;  // [2][2 slots][2] int4
  static constexpr uint32_t kOffClaim = kOffInfo + 128;          // struct Claims
  static constexpr uint32_t kOffTmemPtr = kOffClaim + 32;
  // SPLIT: a side's unnormalised output, row by row with reference and sum of the row's halves behind it, over its K / V slots
  static constexpr int kPartStride = DH + 4;  // floats
  static_assert(BQ * kPartStride * 4 <= kKvSlots * kKBytes, "a part fits the side's slots");
  __device__ static constexpr uint32_t part_offset(int side) { return kOffKv + side * kKvSlots * kKBytes; }
  static constexpr uint32_t kOffAbort = kOffTmemPtr + 4;
  static constexpr int kSmemBytes = kOffAbort + 12;
  static_assert(kSmemBytes <= 232448, "shared memory of one SM");
};

struct DcaParams {
  const DcaItem* items;  // null: the producers find their item in the offsets
  const int32_t* cand_offsets;
  int32_t R;
  int32_t n_q, H;
  float scale_log2e;  // scale * log2(e)
  float per_key;      // 1 / average keys of a request where items go by length, otherwise 0
  const int32_t* seq_offsets;
  const __nv_bfloat16 *Q, *K, *V;  // plain pointers for rows that are computed by hand
  __nv_bfloat16* O;
  uint32_t* status;
};

__host__ __device__ constexpr int32_t round16(int32_t x) { return (x + 15) / 16 * 16; }

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Packed sum of two pairs, and the three-input maximum.
__device__ __forceinline__ uint64_t fadd2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ uint32_t bf16x2_bits(float lo, float hi) {
  const __nv_bfloat162 h2 = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h2);
}

// D[tmem] (+)= A[tmem] * B[smem]: A holds bf16 pairs in 32-bit columns (16 keys = 8 columns).
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void tmem_st_32x32b_x8(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(r[0]),
               "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}

// One query row of one head, half of its DH output columns, unnormalised, in plain fp32 with the row's true maximum
// m as reference and l as sum (a score of -inf has weight 0 whatever the maximum: these keys may be a part of the row's
// only, and the others' scores finite): q and k point at the head's DH values of the row / of the first key, v at the
// DH / 2 columns wanted; consecutive keys are `stride` elements apart.  Inlined on purpose: as a called
// function it forces the caller's hot loop to keep its registers where the calling convention wants
// them, and the loop spills.
template <int DH>
__device__ __forceinline__ void row_by_hand(const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                                            int32_t stride, int32_t L, float scale_log2e, float& m, float& l,
                                            float (&acc)[DH / 2]) {
  auto score = [&](int32_t j) {
    float s = 0.f;
    for (int d = 0; d < DH; ++d) s = fmaf(__bfloat162float(q[d]), __bfloat162float(k[(int64_t)j * stride + d]), s);
    return s * scale_log2e;
  };
  m = -INFINITY;
  for (int32_t j = 0; j < L; ++j) m = fmaxf(m, score(j));
  l = 0.f;
  for (int d = 0; d < DH / 2; ++d) acc[d] = 0.f;
  for (int32_t j = 0; j < L; ++j) {
    const float s = score(j), pj = s == -INFINITY ? 0.f : exp2f(s - m);
    l += pj;
    for (int d = 0; d < DH / 2; ++d) acc[d] = fmaf(pj, __bfloat162float(v[(int64_t)j * stride + d]), acc[d]);
  }
}

// Classes of requests by their number of keys, most keys first, an eighth of the average apart: the order of the items where
// they are a few rounds of the chip, so that the last to be claimed are short ones.  Lane c of a warp has the index of class
// c's first item and the number of its items.
constexpr int kLengthClasses = 8;
__device__ __forceinline__ int length_class(int32_t L, float per_key) {
  return min(max((int)((1.5f - (float)L * per_key) * 8.f), 0), kLengthClasses - 1);
}
struct ClassItems {
  int32_t first, count;
};
__device__ __forceinline__ ClassItems count_classes(const int32_t* __restrict__ off, const int32_t* __restrict__ seq, int32_t R,
                                                    int32_t per, int32_t heads, float per_key, int lane) {
  int32_t count = 0;
  for (int32_t r0 = 0; r0 < R; r0 += 32) {
    const int32_t r = r0 + lane;
    const int32_t entries = r < R ? tiles_of(off[r + 1] - off[r], per) * heads : 0;
    const int c = r < R ? length_class(seq[r + 1] - seq[r], per_key) : 0;
#pragma unroll
    for (int x = 0; x < kLengthClasses; ++x) {
      const int32_t sum = __reduce_add_sync(0xffffffffu, c == x ? entries : 0);
      if (lane == x) count += sum;
    }
  }
  int32_t incl = count;
#pragma unroll
  for (int o = 1; o < kLengthClasses; o <<= 1) {
    const int32_t up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += up;
  }
  return ClassItems{incl - count, lane < kLengthClasses ? count : 0};
}

// The item of index i in the order class, request, head, tile, found by one warp from the offsets, with its request's keys: their
// offsets are loaded with the candidates' and not behind them, a second trip to memory in front of the item's first loads.
template <bool BY_LENGTH>
__device__ __forceinline__ DcaItem find_item(const int32_t* __restrict__ off, const int32_t* __restrict__ seq, int32_t R, int32_t per,
                                             int32_t heads, float per_key, const ClassItems& classes, int32_t i, int lane,
                                             int32_t& s0, int32_t& L) {
  int32_t base = 0;
  int cls = 0;
  const bool by_length = BY_LENGTH && per_key != 0.f;
  if (by_length) {
    const uint32_t in_class = __ballot_sync(0xffffffffu, classes.first <= i && i - classes.first < classes.count);
    if (in_class == 0) return DcaItem{-1, 0, 0, 0};
    cls = __ffs(in_class) - 1;
    base = __shfl_sync(0xffffffffu, classes.first, cls);
  }
  for (int32_t r0 = 0; r0 < R; r0 += 32) {
    const int32_t r = r0 + lane;
    const int32_t c0 = r < R ? off[r] : 0, n = r < R ? off[r + 1] - c0 : 0;
    const int32_t k0 = r < R ? seq[r] : 0, k1 = r < R ? seq[r + 1] : 0;
    const int32_t tiles = tiles_of(n, per);
    const int32_t entries = !by_length || length_class(k1 - k0, per_key) == cls ? tiles * heads : 0;
    int32_t incl = entries;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t up = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += up;
    }
    const int32_t first = base + incl - entries;
    const uint32_t hit = __ballot_sync(0xffffffffu, first <= i && i < first + entries);
    if (hit != 0) {
      const int32_t local = i - first, h = tiles > 0 ? local / tiles : 0, c = (local - h * tiles) * per;
      const int src = __ffs(hit) - 1;
      s0 = __shfl_sync(0xffffffffu, k0, src);
      L = __shfl_sync(0xffffffffu, k1, src) - s0;
      return DcaItem{__shfl_sync(0xffffffffu, r, src), __shfl_sync(0xffffffffu, c0 + c, src),
                     __shfl_sync(0xffffffffu, min(per, n - c), src), __shfl_sync(0xffffffffu, h, src)};
    }
    base += __shfl_sync(0xffffffffu, incl, 31);
  }
  return DcaItem{-1, 0, 0, 0};
}

// Claims a CTA of the grid that has not started yet and returns its index, or -1 when there is none left
// (cluster launch control: the hardware's own list of waiting CTAs).  One thread of each side calls this; a lock
// keeps the sides' requests apart, since after one that failed there must be no other.
struct Claims {
  uint4 response;
  uint64_t bar;
  uint32_t lock;   // 1: taken
  uint32_t state;  // bit 0: phase of the barrier, bit 1: nothing left
};
static_assert(sizeof(Claims) == 32, "space in shared memory");
__device__ __forceinline__ int32_t claim_cta(Claims* c, AbortFlag* abort_flag, uint32_t* status, uint32_t code) {
  const uint64_t t0 = globaltimer_ns();
  while (atomicCAS(&c->lock, 0u, 1u) != 0u) {
    if (abort_flag->v) return -1;
    if (globaltimer_ns() - t0 > 2 * kWaitLimitNs) {
      abort_flag->v = 1;
      atomicCAS(status, 0u, code);
      return -1;
    }
  }
  __threadfence_block();
  int32_t index = -1;
  const uint32_t state = *reinterpret_cast<volatile uint32_t*>(&c->state);
  if ((state & 2u) == 0u) {
    const uint32_t bar = smem_u32(&c->bar), at = smem_u32(&c->response);
    mbar_expect_tx(bar, 16);
    asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];" ::"r"(at),
                 "r"(bar)
                 : "memory");
    uint32_t got = 0, x = 0;
    if (mbar_wait_paced(bar, state & 1u, abort_flag, status, code)) {
      asm volatile(
          "{\n.reg .pred p;\n.reg .b128 r;\nld.shared.b128 r, [%2];\n"
          "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, r;\nselp.u32 %0, 1, 0, p;\nmov.u32 %1, 0;\n"
          "@p clusterlaunchcontrol.query_cancel.get_first_ctaid.v4.b32.b128 {%1, _, _, _}, r;\n}\n"
          : "=&r"(got), "=&r"(x)
          : "r"(at)
          : "memory");
      fence_proxy_async_smem();  // the next response may overwrite what was read
    }
    if (got) index = (int32_t)x;
    *reinterpret_cast<volatile uint32_t*>(&c->state) = ((state & 1u) ^ 1u) | (got ? 0u : 2u);
  }
  __threadfence_block();
  atomicExch(&c->lock, 0u);
  return index;
}

__device__ __forceinline__ float4 ld_cluster_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}

// A short burst of probes before the paced wait: for hand-offs that are usually complete already.
__device__ __forceinline__ bool mbar_wait_spin(uint32_t bar, uint32_t parity, AbortFlag* abort_flag, uint32_t* status,
                                               uint32_t code) {
#pragma unroll 1
  for (int i = 0; i < 64; ++i)
    if (mbar_try_wait_brief(bar, parity)) return true;
  return mbar_wait_paced(bar, parity, abort_flag, status, code);
}


template <int DH, int BKV, bool SPLIT>
__global__ void __launch_bounds__(kThreads, 1)
dca_umma_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                const __grid_constant__ CUtensorMap map_v, const DcaParams p) {
  using C = DcaCfg<DH, BKV>;
  constexpr int kKvSlots = C::kKvSlots, kBoxes = C::kBoxes, kCols = C::kCols, kOutCols = C::kOutCols;
  constexpr int kQBytes = C::kQBytes, kKBytes = C::kKBytes;
  constexpr int kPColOffset = C::kPColOffset, kOColOffset = C::kOColOffset;
  constexpr uint32_t kOffQ = C::kOffQ, kOffKv = C::kOffKv, kOffL = C::kOffL, kBarQFull = C::kBarQFull,
                     kBarQEmpty = C::kBarQEmpty, kBarKvFull = C::kBarKvFull, kBarKvEmpty = C::kBarKvEmpty,
                     kBarSFull = C::kBarSFull, kBarSEmpty = C::kBarSEmpty, kBarPFull = C::kBarPFull,
                     kBarOFull = C::kBarOFull, kBarPair = C::kBarPair, kBarDrain = C::kBarDrain, kBarInfoFull = C::kBarInfoFull,
                     kBarInfoEmpty = C::kBarInfoEmpty, kBarTail = C::kBarTail, kOffInfo = C::kOffInfo,
                     kOffTmemPtr = C::kOffTmemPtr, kOffAbort = C::kOffAbort;
  extern __shared__ __align__(1024) uint8_t smem[];     // swizzled operand tiles need 1024-byte alignment
  const uint32_t sb = smem_u32(smem);                   // every shared-memory address below is sb + constant
  AbortFlag* abort_flag = reinterpret_cast<AbortFlag*>(smem + kOffAbort);

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if ((sb & 1023u) != 0) {  // the swizzled tiles assume a 1024-byte aligned base
    if (threadIdx.x == 0) atomicCAS(p.status, 0u, kStatusDca | 15);
    return;
  }

  if (threadIdx.x == 0) {
    auto init = [&](uint32_t off, int n, uint32_t count) {
      for (int x = 0; x < n; ++x) mbar_init(reinterpret_cast<uint64_t*>(smem + off + 8 * x), count);
    };
    init(kBarQFull, 2, 1);
    init(kBarQEmpty, 2, 1);
    init(kBarKvFull, 2 * kKvSlots, 1);
    init(kBarKvEmpty, 2 * kKvSlots, 1);
    init(kBarSFull, 2, 1);
    init(kBarSEmpty, 2, kSoftmaxWarps / 2);
    init(kBarPFull, 4, kSoftmaxWarps / 2);
    init(kBarOFull, 2, 1);
    init(kBarPair, 8, 2);
    init(kBarDrain, 2, 1);
    init(kBarInfoFull, 4, 1);
    init(kBarInfoEmpty, 4, kSoftmaxWarps / 2 + 1);
    init(kBarTail, 2, 1);
    init(C::kOffClaim + 16, 1, 1);
    reinterpret_cast<Claims*>(smem + C::kOffClaim)->lock = 0;
    reinterpret_cast<Claims*>(smem + C::kOffClaim)->state = 0;
    abort_flag->v = 0;
    fence_mbar_init();
  }
  if (warp == kControlWarp0 + 1) {
    tmem_alloc(reinterpret_cast<uint32_t*>(smem + kOffTmemPtr), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = *reinterpret_cast<const uint32_t*>(smem + kOffTmemPtr);
  // launched as a programmatic dependent: the set-up above may overlap the end of the kernel in front;
  // global memory is touched only from here on, and the kernel behind this one is released after the wait
  if (warp == kControlWarp0 && lane == 0) {  // parameters of the launch: no need to wait
    prefetch_tensormap(&map_q);
    prefetch_tensormap(&map_k);
    prefetch_tensormap(&map_v);
  }
  griddep_wait();
  griddep_launch_dependents();
  const int32_t row_width = p.H * DH;  // elements per query / key row over all heads
  const uint32_t cluster_size = SPLIT ? cluster_ctas() : 1;

  if (warp == kControlWarp0 || warp == kControlWarp0 + 3) {
    // ------------------------------ TMA producers: one warp per side --------------------------
    // Also the side's item reader: it claims an item, looks it up in global memory and hands it to the other warps
    // through two slots in shared memory, so that nobody else waits for global memory between two items.
    // Items are claimed and not dealt out by position: with few items per side their number and length differ
    // (100 requests x 300 candidates, 100..200 keys: 31.8 us dealt out, 29.6 us claimed; 40 requests x 400, 300..700
    // keys: 43.1 and 40.5 us), and long streams end more evenly too (103 024 items: 3.79 and 3.71 ms).
    const int side = warp == kControlWarp0 ? 0 : 1;
    const uint32_t q_full = sb + kBarQFull + 8 * side, q_empty = sb + kBarQEmpty + 8 * side;
    const uint32_t kv_full = sb + kBarKvFull + 8 * kKvSlots * side, kv_empty = sb + kBarKvEmpty + 8 * kKvSlots * side;
    const uint32_t info_full = sb + kBarInfoFull + 16 * side, info_empty = sb + kBarInfoEmpty + 16 * side;
    const uint32_t q_dst = sb + kOffQ + side * kQBytes, kv_dst = sb + kOffKv + side * kKvSlots * kKBytes;
    int4* info = reinterpret_cast<int4*>(smem + kOffInfo) + side * 4;
    uint32_t kv_it = 0, n_work = 0, n_item = 0;
    bool ok = true;
    auto wait = [&](uint32_t bar, uint32_t parity, uint32_t code) {  // the same answer for the whole warp
      return __all_sync(0xffffffffu, mbar_wait_paced(bar, parity, abort_flag, p.status, kStatusDca | code)) != 0;
    };
    // The last block of a sequence may reach past it into the next request's rows (or past the
    // tensor, where TMA fills zeros).  Scores of such keys are masked to -inf by the softmax warps,
    // so P is exactly 0 there; the V rows are zeroed here so that 0 x (Inf or NaN of a foreign
    // request) cannot reach this request's output.  (The products go no further than the next multiple of 16
    // keys, so at most 15 rows.)  Done once the next item's Q load is out, i.e. after the last S of this item
    // was issued and while its softmax runs; P V waits for it.
    int32_t tail_valid = 0;  // valid keys of a block that waits to be zeroed; 0: none
    uint32_t tail_slot = 0, tail_phase = 0;
    auto zero_tail = [&]() {
      if (tail_valid == 0) return true;
      if (!wait(kv_full + 8 * tail_slot, tail_phase, 4)) return false;
      uint8_t* v = smem + kOffKv + (side * kKvSlots + tail_slot) * kKBytes;
      for (int bx = 0; bx < kBoxes; ++bx)
        for (int idx = tail_valid * (C::kRowBytes / 16) + lane; idx < round16(tail_valid) * (C::kRowBytes / 16); idx += 32)
          *reinterpret_cast<uint4*>(v + bx * C::kKvBoxBytes + idx * 16) = make_uint4(0u, 0u, 0u, 0u);
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(sb + kBarTail + 8 * side);
      tail_valid = 0;
      return true;
    };
    Claims* claims = reinterpret_cast<Claims*>(smem + C::kOffClaim);
    int32_t i = SPLIT ? (int32_t)(blockIdx.x / cluster_size) : (int32_t)blockIdx.x;  // -1: no more
    ClassItems classes{0, 0};
    constexpr bool kByLength = DH == 128 && !SPLIT;
    if (kByLength && p.per_key != 0.f) classes = count_classes(p.cand_offsets, p.seq_offsets, p.R, BQ / p.n_q, p.H, p.per_key, lane);
    DcaItem next{-1, 0, 0, 0};
    int32_t next_s0 = 0, next_L = 0, total_L = 0;
    auto read_next = [&]() {
      if (i >= 0) {
        if (p.items == nullptr) {
          next = find_item<kByLength>(p.cand_offsets, p.seq_offsets, p.R, BQ / p.n_q, p.H, p.per_key, classes, i, lane, next_s0, next_L);
        } else {
          next = p.items[i];
          next_s0 = p.seq_offsets[next.req];
          next_L = p.seq_offsets[next.req + 1] - next_s0;
        }
        if constexpr (SPLIT) {  // this side's run of the item's key blocks
          const int32_t nblk = (next_L + BKV - 1) / BKV, parts = 2 * (int32_t)cluster_size;
          const int32_t part = 2 * (int32_t)cluster_ctarank() + side;
          const int32_t k0 = nblk * part / parts * BKV, k1 = min(nblk * (part + 1) / parts * BKV, next_L);
          total_L = next_L;
          next_s0 += k0;
          next_L = max(k1 - k0, 0);
        }
      } else {
        next.req = -1;
        next_L = 0;
      }
    };
    // An item is claimed when the loads of the one in front are out, no earlier: what is claimed ahead cannot go to
    // a side that is done before.  In SPLIT every side has its part of the CTA's item and no other.
    auto claim_next = [&]() {
      int32_t c = -1;
      if (!SPLIT && lane == 0) c = claim_cta(claims, abort_flag, p.status, kStatusDca | 16);
      i = __shfl_sync(0xffffffffu, c, 0);
    };
    if (!SPLIT && side == 1) claim_next();  // the CTA's own item goes to side A
    for (bool first = true;; first = false) {
      if (!first) claim_next();
      read_next();
      const DcaItem item = next;
      const int32_t s0 = next_s0, L = next_L;
      const uint32_t slot = n_item & 1;
      // (a slot comes free only if the items in front of it can finish, the last one included when this one
      // has no loads behind which its tail would be zeroed)
      if (L == 0 && tail_valid != 0) {
        // not before that item's last S, as in the ordinary case: the issuer is then past the tail in front of it,
        // and two arrivals never meet one wait
        if (!wait(q_empty, (n_work & 1) ^ 1, 1) || !zero_tail()) { ok = false; break; }
      }
      if (!wait(info_empty + 8 * slot, ((n_item >> 1) & 1) ^ 1, 12)) { ok = false; break; }
      if (lane == 0) {
        info[2 * slot] = make_int4(item.req, item.cand0, item.count * p.n_q, item.head);
        info[2 * slot + 1] = make_int4(L, s0, total_L, 0);
        mbar_arrive(info_full + 8 * slot);
      }
      ++n_item;
      if (item.req < 0) break;
      if (L == 0) continue;  // nobody touches another barrier for an item without keys
      if (!wait(q_empty, (n_work & 1) ^ 1, 1)) { ok = false; break; }
      ++n_work;
      if (elect_one()) {
        mbar_expect_tx(q_full, kQBytes);
#pragma unroll
        for (int bx = 0; bx < kBoxes; ++bx)
          tma_load_2d(q_dst + bx * C::kQBoxBytes, &map_q, q_full, item.head * DH + bx * C::kBoxCols, item.cand0 * p.n_q);
      }
      __syncwarp();
      if (!zero_tail()) { ok = false; break; }
      const int32_t nblk = (L + BKV - 1) / BKV;
      auto load_block = [&](const CUtensorMap* map, int32_t j) {
        const uint32_t s = kv_it % kKvSlots;
        if (!wait(kv_empty + 8 * s, ((kv_it / kKvSlots) & 1) ^ 1, 2)) return false;
        if (elect_one()) {
          mbar_expect_tx(kv_full + 8 * s, kKBytes);
#pragma unroll
          for (int bx = 0; bx < kBoxes; ++bx)
            tma_load_2d(kv_dst + s * kKBytes + bx * C::kKvBoxBytes, map, kv_full + 8 * s, item.head * DH + bx * C::kBoxCols,
                        s0 + j * BKV);
        }
        __syncwarp();
        ++kv_it;
        return true;
      };
      // in the order of their use, which is the order they come free in: K_0, K_1, V_0, K_2, V_1, ...
      ok = load_block(&map_k, 0);
      for (int32_t j = 0; j < nblk && ok; ++j) {
        if (j + 1 < nblk) ok = load_block(&map_k, j + 1);
        if (ok) ok = load_block(&map_v, j);
      }
      if (!ok) break;
      tail_valid = L % 16 == 0 ? 0 : L % BKV;
      tail_slot = (kv_it - 1) % kKvSlots;
      tail_phase = ((kv_it - 1) / kKvSlots) & 1;
    }
    if (!ok) {
      // let the loads in flight land before the CTA's shared memory goes away
      for (uint32_t s = 0; s < kKvSlots; ++s) {
        const uint32_t n_issued = kv_it / kKvSlots + ((kv_it % kKvSlots > s) ? 1 : 0);
        if (n_issued == 0) continue;
        const uint64_t t0 = globaltimer_ns();
        while (!mbar_try_wait_brief(kv_full + 8 * s, (n_issued - 1) & 1) && globaltimer_ns() - t0 < kWaitLimitNs) {}
      }
    }
  } else if (warp >= kControlWarp0) {
    // ------------------------------ MMA issuers: one thread per side -------------------------
    // (a whole loop under one elected lane: with the products alone under it, in a loop of the whole warp,
    // issuing S and P V of a block took 780 cycles instead of the 180 here)
    if (elect_one()) {
      const int side = warp - (kControlWarp0 + 1);
      constexpr uint32_t idesc_o = umma_idesc_bf16(BQ, DH, false, true);    // O = P V, V is MN-major
      const uint32_t q_full = sb + kBarQFull + 8 * side, q_empty = sb + kBarQEmpty + 8 * side;
      const uint32_t kv_full = sb + kBarKvFull + 8 * kKvSlots * side, kv_empty = sb + kBarKvEmpty + 8 * kKvSlots * side;
      const uint32_t s_full = sb + kBarSFull + 8 * side, s_empty = sb + kBarSEmpty + 8 * side;
      const uint32_t p_full = sb + kBarPFull + 16 * side, o_full = sb + kBarOFull + 8 * side;
      const uint32_t tail_done = sb + kBarTail + 8 * side;
      const uint32_t info_full = sb + kBarInfoFull + 16 * side, info_empty = sb + kBarInfoEmpty + 16 * side;
      const int4* info = reinterpret_cast<const int4*>(smem + kOffInfo) + side * 4;
      uint32_t kv_it = 0, n_work = 0, n_tail = 0, n_item = 0;  // phases of kv_full, q_full, tail_done, info_full
      uint32_t cnt_p = 0, cnt_se = 0;                          // phases of p_full and s_empty
      bool ok = true;
      const uint32_t t_s = tmem_base + side * kSideTmemStride;
      // Q tile of this side; slot 0 as a K and as a V block (a slot is kKBytes >> 4 further on)
      const uint64_t dq = C::desc(sb + kOffQ + side * kQBytes);
      const uint64_t dk0 = C::desc(sb + kOffKv + side * kKvSlots * kKBytes);
      const uint64_t dv0 = C::desc_v(sb + kOffKv + side * kKvSlots * kKBytes);
      // `keys`: of the block, a multiple of 16
      auto issue_s = [&](uint32_t slot, int32_t keys) {
        const uint64_t dk = dk0 + slot * (kKBytes >> 4);
        const uint32_t idesc_s = umma_idesc_bf16(BQ, (uint32_t)keys, false, false);  // S = Q K^T, both K-major
#pragma unroll
        for (int k = 0; k < DH / 16; ++k) {  // 16 columns of dh per step: box k / kPerBox, 32 bytes further on inside it
          constexpr int kPerBox = C::kBoxCols / 16;
          umma_ss(t_s, dq + (k / kPerBox) * (C::kQBoxBytes >> 4) + 2 * (k % kPerBox),
                  dk + (k / kPerBox) * (C::kKvBoxBytes >> 4) + 2 * (k % kPerBox), idesc_s, k != 0 ? 1u : 0u);
        }
        umma_commit(s_full);
        umma_commit(kv_empty + 8 * slot);
      };
      auto issue_pv = [&](uint32_t slot, uint32_t buf, int32_t keys, int32_t j, bool last) {
        const uint64_t dv = dv0 + slot * (kKBytes >> 4);
        const uint32_t t_p = t_s + kPColOffset + buf * (BKV / 2);
        // P: 16 keys = 8 columns of bf16 pairs in tensor memory; V: rows are keys, 16 keys = 16 rows further on
#pragma unroll
        for (int k = 0; k < BKV / 16; ++k)
          if (k * 16 < keys)
            umma_ts(t_s + kOColOffset, t_p + k * 8, dv + k * (16 * C::kRowBytes / 16), idesc_o, (k | j) != 0 ? 1u : 0u);
        if (C::kPBuffers == 1 || last) umma_commit(o_full);
        umma_commit(kv_empty + 8 * slot);
      };
      auto next_slot = [&](uint32_t code) {  // the next block in the order of loading, landed
        if (!mbar_wait_paced(kv_full + 8 * (kv_it % kKvSlots), (kv_it / kKvSlots) & 1, abort_flag, p.status, kStatusDca | code)) return false;
        ++kv_it;
        return true;
      };
      while (ok) {
        const uint32_t slot = n_item & 1;
        if (!mbar_wait_paced(info_full + 8 * slot, (n_item >> 1) & 1, abort_flag, p.status, kStatusDca | 13)) { ok = false; break; }
        ++n_item;
        const int32_t req = info[2 * slot].x, L = info[2 * slot + 1].x;
        mbar_arrive(info_empty + 8 * slot);
        if (req < 0) break;
        if (L == 0) continue;
        const int32_t nblk = (L + BKV - 1) / BKV;
        const int32_t tail_keys = round16(L - (nblk - 1) * BKV);  // products of the last block
        if (!mbar_wait_paced(q_full, n_work & 1, abort_flag, p.status, kStatusDca | 3)) { ok = false; break; }
        ++n_work;
        // first key block (the S tile was drained at the end of the previous item)
        if (!next_slot(4)) { ok = false; break; }
        tc_fence_after_sync();
        issue_s((kv_it - 1) % kKvSlots, nblk == 1 ? tail_keys : BKV);
        if (nblk == 1) umma_commit(q_empty);
        for (int32_t j = 0; j < nblk; ++j) {
          if (j + 1 < nblk && !next_slot(5)) { ok = false; break; }
          // S_{j+1} as soon as the side has pulled S_j into registers
          if (!mbar_wait_paced(s_empty, cnt_se & 1, abort_flag, p.status, kStatusDca | 11)) { ok = false; break; }
          ++cnt_se;
          if (j + 1 < nblk) {
            tc_fence_after_sync();
            issue_s((kv_it - 1) % kKvSlots, j + 2 == nblk ? tail_keys : BKV);
            if (j + 2 == nblk) umma_commit(q_empty);  // last S of the item: the Q tile is free
          }
          if (!next_slot(8)) { ok = false; break; }
          if (j + 1 == nblk && L % 16 != 0) {  // V rows past the sequence are zero
            if (!mbar_wait_paced(tail_done, n_tail & 1, abort_flag, p.status, kStatusDca | 10)) { ok = false; break; }
            ++n_tail;
          }
          // P_j of this side is in tensor memory
          const uint32_t buf = cnt_p & (C::kPBuffers - 1);
          if (!mbar_wait_paced(p_full + 8 * buf, (cnt_p / C::kPBuffers) & 1, abort_flag, p.status, kStatusDca | 6)) { ok = false; break; }
          ++cnt_p;
          tc_fence_after_sync();
          issue_pv((kv_it - 1) % kKvSlots, buf, j + 1 == nblk ? tail_keys : BKV, j, j + 1 == nblk);
        }
      }
      if (!ok) {
        umma_commit(sb + kBarDrain + 8 * side);
        const uint64_t t0 = globaltimer_ns();
        while (!mbar_try_wait_brief(sb + kBarDrain + 8 * side, 0) && globaltimer_ns() - t0 < kWaitLimitNs) {}
      }
    }
  } else {
    // ------------------------------ softmax warps ------------------------------------------
    const int side = warp >> 3;
    const int half = (warp >> 2) & 1;       // which half of the block's key columns
    const int q = warp & 3;                 // TMEM lane quadrant this warp may touch
    const int row = q * 32 + lane;          // query row of the tile = TMEM lane
    const uint32_t t_row = tmem_base + side * kSideTmemStride + ((uint32_t)(q * 32) << 16);  // S columns of the row
    const uint32_t t_s = t_row + half * kCols;
    const uint32_t t_p = t_row + kPColOffset + half * (kCols / 2);
    const uint32_t t_o = t_row + kOColOffset + half * kOutCols;
    const uint32_t s_full = sb + kBarSFull + 8 * side, s_empty = sb + kBarSEmpty + 8 * side;
    const uint32_t p_full = sb + kBarPFull + 16 * side, o_full = sb + kBarOFull + 8 * side;
    const uint32_t my_pair = sb + kBarPair + 8 * (side * 4 + q);
    uint32_t cnt_s = 0, cnt_o = 0, cnt_pair = 0;
    const uint32_t info_full = sb + kBarInfoFull + 16 * side, info_empty = sb + kBarInfoEmpty + 16 * side;
    const int4* info = reinterpret_cast<const int4*>(smem + kOffInfo) + side * 4;
    for (uint32_t n_item = 0;; ++n_item) {
      const uint32_t slot = n_item & 1;
      if (!mbar_wait_spin(info_full + 8 * slot, (n_item >> 1) & 1, abort_flag, p.status, kStatusDca | 13)) break;
      const int4 item = info[2 * slot];  // request, first candidate, query rows, head
      const int32_t L = info[2 * slot + 1].x, s0 = info[2 * slot + 1].y;
      __syncwarp();
      if (lane == 0) mbar_arrive(info_empty + 8 * slot);
      if (item.x < 0) break;
      const int32_t rows_valid = item.z;
      // this thread's half of the output columns of its row
      auto out_ptr = [&]() { return p.O + ((int64_t)item.y * p.n_q + row) * row_width + item.w * DH + half * kOutCols; };
      bool aborted = false;
      if (L > 0) {
        const int32_t nblk = (L + BKV - 1) / BKV;
        // ---- reference of the row: the maximum over its first 32 keys, rounded up to an integer
        if (!mbar_wait_spin(s_full, cnt_s & 1, abort_flag, p.status, kStatusDca | 7)) break;
        tc_fence_after_sync();
        float m_ref;
        {
          float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
          uint32_t ov[32];
          tmem_ld_32x32b_x32(t_row, ov);
          tmem_ld_wait();
          if (L < 32) {
#pragma unroll
            for (int e = 0; e < 32; ++e)
              if (e >= L) ov[e] = 0xff800000u;  // -inf: the key does not exist
          }
#pragma unroll
          for (int e = 0; e < 32; e += 2)  // four short chains of three-input maxima
            mx4[(e >> 1) & 3] = fmax3(mx4[(e >> 1) & 3], __uint_as_float(ov[e]), __uint_as_float(ov[e + 1]));
          m_ref = ceilf(fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * p.scale_log2e);
        }
        const uint64_t c2 = pack2(p.scale_log2e, p.scale_log2e), m2 = pack2(-m_ref, -m_ref);
        uint64_t sum2 = pack2(0.f, 0.f);
        for (int32_t j = 0; j < nblk; ++j) {
          if (j > 0) {
            if (!mbar_wait_spin(s_full, cnt_s & 1, abort_flag, p.status, kStatusDca | 7)) { aborted = true; break; }
            tc_fence_after_sync();
          }
          ++cnt_s;
          uint32_t sv[kCols];  // this thread's scores of the block
#pragma unroll
          for (int c = 0; c < kCols; c += 32) tmem_ld_32x32b_x32(t_s + c, sv + c);
          tmem_ld_wait();
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(s_empty);  // S_{j+1} may overwrite the tile now
          const int32_t valid = L - j * BKV - half * kCols;  // columns of this thread's half that are keys of the request
          if (valid < kCols) {
#pragma unroll
            for (int e = 0; e < kCols; ++e)
              if (e >= valid) sv[e] = 0xff800000u;  // -inf: the key does not exist
          }
          uint32_t pk[kCols / 4];  // P of half of this thread's keys, bf16 pairs; stored in two halves
          auto store_p = [&](uint32_t taddr) {
            if constexpr (kCols == 64) tmem_st_32x32b_x16(taddr, pk); else tmem_st_32x32b_x8(taddr, pk);
          };
          auto exp_pair = [&](int e) {
            float x0, x1;
            unpack2(ffma2(pack2(__uint_as_float(sv[e]), __uint_as_float(sv[e + 1])), c2, m2), x0, x1);
            const float p0 = ex2(x0), p1 = ex2(x1);
            sum2 = fadd2(sum2, pack2(p0, p1));
            pk[(e / 2) % (kCols / 4)] = bf16x2_bits(p0, p1);
          };
          // P V of the previous block has read P_{j-1} (it was issued most of a block ago): from there on this
          // thread's P columns may be rewritten
          auto previous_pv_done = [&]() {
            if (C::kPBuffers == 2) return true;
            if (j > 0) {
              if (!mbar_wait_spin(o_full, (cnt_o & 1) ^ 1, abort_flag, p.status, kStatusDca | 9)) return false;
              tc_fence_after_sync();
            }
            ++cnt_o;
            return true;
          };
          const uint32_t buf = (cnt_s - 1) & (C::kPBuffers - 1), t_pj = t_p + buf * (BKV / 2);
          if (valid > 0) {
#pragma unroll
            for (int e = 0; e < kCols / 2; e += 2) exp_pair(e);
            if (!previous_pv_done()) { aborted = true; break; }
            store_p(t_pj);
#pragma unroll
            for (int e = kCols / 2; e < kCols; e += 2) exp_pair(e);
            store_p(t_pj + kCols / 4);
          } else if (!previous_pv_done()) {  // no key in this half of the last block: P V stops in front of it
            aborted = true;
            break;
          }
          tmem_st_wait();
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(p_full + 8 * buf);
        }
        if (aborted) break;
        if (C::kPBuffers == 2) ++cnt_o;  // one arrival per item
        float sum_lo, sum_hi;
        unpack2(sum2, sum_lo, sum_hi);
        const float l_run = sum_lo + sum_hi;
        float* l_x = reinterpret_cast<float*>(smem + kOffL);
        l_x[(side * 2 + half) * BQ + row] = l_run;
        __syncwarp();
        if (lane == 0) mbar_arrive(my_pair);
        if (!mbar_wait_paced(my_pair, cnt_pair & 1, abort_flag, p.status, kStatusDca | 14) ||
            !mbar_wait_paced(o_full, (cnt_o & 1) ^ 1, abort_flag, p.status, kStatusDca | 9))
          break;
        ++cnt_pair;
        tc_fence_after_sync();
        const float l_o = l_x[(side * 2 + (half ^ 1)) * BQ + row];
        const float l_tot = half == 0 ? l_run + l_o : l_o + l_run;  // same order in both halves
        const float inv = 1.f / l_tot;
        uint32_t v[kOutCols];
        if constexpr (kOutCols == 16) {
          tmem_ld_32x32b_x16(t_o, v);
        } else {
#pragma unroll
          for (int c = 0; c < kOutCols; c += 32) tmem_ld_32x32b_x32(t_o + c, v + c);
        }
        tmem_ld_wait();
        // Scores that outgrow the first block's maximum by 2^128 or so overflow fp32 (and so can
        // a sum of products with huge values): the row then holds Inf or NaN instead of a result.
        float probe = l_tot * 0.f;
#pragma unroll
        for (int e = 0; e < kOutCols; ++e) probe = fmaf(__uint_as_float(v[e]), 0.f, probe);
        // such a row is computed again by its two threads, with its true maximum as reference
        float hand_m, hand_l, hand[kOutCols];
        auto by_hand = [&]() {
          const int64_t q_row = (int64_t)item.y * p.n_q + row;
          const int64_t kv0 = ((int64_t)s0 * p.H + item.w) * DH;
          row_by_hand<DH>(p.Q + q_row * row_width + item.w * DH, p.K + kv0, p.V + kv0 + half * kOutCols, row_width, L,
                          p.scale_log2e, hand_m, hand_l, hand);
        };
        if constexpr (SPLIT) {
          if (row < rows_valid) {
            float* part = reinterpret_cast<float*>(smem + C::part_offset(side)) + row * C::kPartStride;
            if (probe == 0.f) {
#pragma unroll
              for (int e = 0; e < kOutCols; e += 4)
                *reinterpret_cast<float4*>(part + half * kOutCols + e) =
                    make_float4(__uint_as_float(v[e]), __uint_as_float(v[e + 1]), __uint_as_float(v[e + 2]), __uint_as_float(v[e + 3]));
              part[DH + 2 * half] = m_ref;  // each half its own: one may have overflowed and been redone, the other not
              part[DH + 2 * half + 1] = l_tot;
            } else {
              by_hand();
              for (int e = 0; e < kOutCols; ++e) part[half * kOutCols + e] = hand[e];
              part[DH + 2 * half] = hand_m;
              part[DH + 2 * half + 1] = hand_l;
            }
          }
        } else if (row < rows_valid) {
          __nv_bfloat16* out = out_ptr();
          if (probe == 0.f) {
#pragma unroll
            for (int e = 0; e < kOutCols; e += 8) {
              uint4 w;
              w.x = bf16x2_bits(__uint_as_float(v[e + 0]) * inv, __uint_as_float(v[e + 1]) * inv);
              w.y = bf16x2_bits(__uint_as_float(v[e + 2]) * inv, __uint_as_float(v[e + 3]) * inv);
              w.z = bf16x2_bits(__uint_as_float(v[e + 4]) * inv, __uint_as_float(v[e + 5]) * inv);
              w.w = bf16x2_bits(__uint_as_float(v[e + 6]) * inv, __uint_as_float(v[e + 7]) * inv);
              *reinterpret_cast<uint4*>(out + e) = w;
            }
          } else {
            by_hand();
            const float hand_inv = 1.f / hand_l;
            for (int e = 0; e < kOutCols; ++e) out[e] = __float2bfloat16_rn(hand[e] * hand_inv);
          }
        }
      } else if (SPLIT) {
        // no key blocks for this side: it adds nothing
        float* part = reinterpret_cast<float*>(smem + C::part_offset(side)) + row * C::kPartStride;
        part[DH + 2 * half] = -INFINITY;
        part[DH + 2 * half + 1] = 0.f;
      } else if (row < rows_valid) {
        // a request without keys: zero rows
        __nv_bfloat16* out = out_ptr();
#pragma unroll
        for (int c = 0; c < kOutCols; c += 8) *reinterpret_cast<uint4*>(out + c) = make_uint4(0u, 0u, 0u, 0u);
      }
      tc_fence_before_sync();  // the next item's first P V overwrites O
    }
  }

  tc_fence_before_sync();
  __syncthreads();
  if (warp == kControlWarp0 + 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, kTmemCols);
  }
  if constexpr (SPLIT) {
    // O = sum_s 2^(m_s - M) O_s / sum_s 2^(m_s - M) l_s over the parts s of the item, M the largest reference.  Every
    // weight is 2^-kScaleDown of that, in both sums: up to 16 parts that are finite each, perhaps close to 2^128, have
    // a finite sum.
    constexpr float kScaleDown = 5.f;
    cluster_sync_all();
    const int4* info = reinterpret_cast<const int4*>(smem + kOffInfo);  // slot 0 of side A: the item
    const int4 item = info[0];
    const int32_t total = info[1].z;
    const int32_t share = BQ / (int32_t)cluster_size, row0 = (int32_t)cluster_ctarank() * share;
    constexpr int kVecs = DH / 4;
    for (int32_t x = threadIdx.x; x < share * kVecs; x += kThreads) {
      const int32_t row = row0 + x / kVecs, col = x % kVecs * 4;
      if (row >= item.z) continue;
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
      float M = -INFINITY, l = 0.f;
      for (uint32_t c = 0; c < cluster_size; ++c)
#pragma unroll
        for (int side = 0; side < 2; ++side) {
          const uint32_t part = map_to_cta(sb + C::part_offset(side) + row * (C::kPartStride * 4), c);
          const float4 both = ld_cluster_f4(part + DH * 4);  // reference and sum of either half of the columns
          const float m = col < DH / 2 ? both.x : both.z, l_part = col < DH / 2 ? both.y : both.w;
          if (m == -INFINITY && l_part == 0.f) continue;  // a side without keys, or whose scores are all -inf
          const float m_new = fmaxf(M, m);
          const float a = M == -INFINITY ? 0.f : exp2f(M - m_new), b = exp2f(m - m_new - kScaleDown);
          const float4 o = ld_cluster_f4(part + col * 4);
          acc.x = acc.x * a + o.x * b;
          acc.y = acc.y * a + o.y * b;
          acc.z = acc.z * a + o.z * b;
          acc.w = acc.w * a + o.w * b;
          l = l * a + l_part * b;
          M = m_new;
        }
      const float inv = total > 0 ? 1.f / l : 0.f;
      *reinterpret_cast<uint2*>(p.O + ((int64_t)item.y * p.n_q + row) * row_width + item.w * DH + col) =
          make_uint2(bf16x2_bits(acc.x * inv, acc.y * inv), bf16x2_bits(acc.z * inv, acc.w * inv));
    }
    __syncwarp();
    cluster_sync_all();  // nobody leaves while another CTA reads its part
  }
}

int sm_count_dca() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  }
  return n;
}

}  // namespace

bool umma_dca_supported(int32_t n_q, int32_t H, int32_t dh) {
  return (dh == 32 || dh == 64 || dh == 128) && n_q >= 1 && n_q <= BQ && H >= 1 && H <= 65535;
}

template <int DH, int BKV>
static rocs_status_t launch_dca(const rocs_plan* plan, int32_t n_q, int32_t H, float scale, const void* Q,
                                const void* K, const void* V, const int32_t* seq_offsets, int64_t T, void* O,
                                cudaStream_t stream) {
  using C = DcaCfg<DH, BKV>;
  const int32_t sms = sm_count_dca();
  const int64_t num = plan_entries(plan, BQ / n_q) * H;
  if (num > 0x7fffffffLL) return ROCS_ERR_UNSUPPORTED;
  if (num == 0) return ROCS_OK;
  // Items that fit the SMs once are split along their keys (SPLIT): over the two sides of a CTA, and over the CTAs
  // of the largest cluster of which every item still gets one at the same time.  Short
  // sequences are not worth it.  How many clusters run at once differs from chip to chip (a cluster stays inside one of
  // its partitions, of which each chip has other SMs: 74 pairs, 33 of 4 and 15 of 8 on one), and an item more than that
  // takes a second round: 16 items of 4096 keys 26.1 us over clusters of 8 there, 14.6 us over 4.  The numbers below are a
  // little less, and constants, so that results do not depend on which GPU they were computed.
  const int64_t blocks = (T + plan->R - 1) / plan->R / BKV + 1;  // of an average sequence
  const bool split = num <= sms && blocks >= 3;
  int32_t cluster = 1;
  const int32_t most[4] = {sms, 70, 32, 14};
  // Blocks of 128 keys: one per CTA is enough (its sides then do not compete for the SM).  40 candidates of one request x 8
  // heads of 64, in a chain, with two per side and this: 300 / 520 / 1000 keys 8.4 / 9.7 / 9.7 and 7.7 / 8.2 / 8.7 us; 2000 keys
  // over 4 and 8 CTAs 10.6 and 11.2.  Blocks of 64 keys: 8 requests x 4 heads of 128, 300 / 520 keys, two per side and one per
  // CTA 9.2 / 10.3 and 10.3 / 11.6.
  auto worth = [&](int i) { return (4 << i) <= blocks || (BKV == 128 && (1 << i) <= blocks && (i < 3 || blocks < 12)); };
  for (int i = 1; i < 4 && split; ++i)
    if (num <= most[i] && worth(i)) cluster = 1 << i;
  // Requests that a producer warp looks through itself, at every item; the list is a launch in front.  What looking
  // costs grows with the requests times the items.  Plan and attention, 8 heads of 64, 200 to 400 keys, without and with
  // the list: 27 candidates of each of 64 / 256 / 288 / 512 requests 15.9 / 44.4 / 54.1 / 105 us and 18.4 / 46.2 / 52.2 /
  // 90 us; 150 candidates of 128 / 256 requests 40.2 / 81.7 and 43.3 / 77.3; 600 candidates of 64 / 128 / 256 requests
  // 60.8 / 115.0 / 242 and 62.7 / 114.6 / 220.  The line is where small requests cross.
  constexpr int32_t kMaxFind = 256;
  DcaItemList items;
  if (plan->R > kMaxFind) {
    const rocs_status_t st = plan_dca_items(plan, BQ / n_q, H, stream, &items);
    if (st != ROCS_OK) return st;
  }
  const uint64_t width = (uint64_t)H * DH;
  CUtensorMap map_q, map_k, map_v;
  constexpr bool sw64 = C::kRowBytes == 64;
  if (!make_tensor_map_2d(&map_q, Q, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)plan->N * n_q, width, width, BQ,
                          C::kBoxCols, true, sw64))
    return ROCS_ERR_CUDA;
  if (T > 0) {
    if (!make_tensor_map_2d(&map_k, K, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)T, width, width, BKV, C::kBoxCols,
                            true, sw64) ||
        !make_tensor_map_2d(&map_v, V, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)T, width, width, BKV, C::kBoxCols,
                            true, sw64))
      return ROCS_ERR_CUDA;
  } else {
    map_k = map_q;  // every sequence is empty: the kernel only writes zeros
    map_v = map_q;
  }
  uint32_t* status = device_status_word();
  if (!status) return ROCS_ERR_CUDA;
  DcaParams p{};
  p.items = items.dev;
  p.cand_offsets = plan->cand_offsets;
  p.R = plan->R;
  p.n_q = n_q;
  p.H = H;
  p.scale_log2e = scale * 1.4426950408889634f;
  // Items of the longest requests first where a side takes one to three and a half of them and they are long: 40 requests x
  // about 20 candidates of 32 query tokens x 4 heads of 128 over 500..1500 keys 68.4 -> 63.2 us, 40 x 500 candidates over 1000..2000 73.1 ->
  // 68.5, 20 x 600 over 750..1500 42.6 -> 40.2.  Not with many requests or short ones, which pay for the counting (60 x 200 over
  // 200..400 23.9 -> 24.4, 120 x 100 over 60..120 19.4 -> 21.5), nor with heads of 64, where sides of an SM in step with one
  // another cost more than the end gains (80 x 200 over 500..1000 54.8 -> 57.3, 64 x 300 over 150..300 30.8 -> 32.7).
  const bool by_length = BKV == 64 && plan->R <= 64 && blocks >= 10 && num > 2 * sms && num <= 7 * sms;
  p.per_key = by_length ? (float)plan->R / (float)T : 0.f;
  p.seq_offsets = seq_offsets;
  p.Q = (const __nv_bfloat16*)Q;
  p.K = (const __nv_bfloat16*)K;
  p.V = (const __nv_bfloat16*)V;
  p.O = (__nv_bfloat16*)O;
  p.status = status;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = C::kSmemBytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (split) {
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.numAttrs = 2;
    cfg.gridDim = dim3((unsigned)(num * cluster));
    auto kernel = dca_umma_kernel<DH, BKV, true>;
    ROCS_ALLOW_SMEM(kernel, C::kSmemBytes);
    ROCS_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, map_q, map_k, map_v, p));
  } else {
    cfg.gridDim = dim3((unsigned)num);  // one CTA per item; those that get an SM claim the others' items
    auto kernel = dca_umma_kernel<DH, BKV, false>;
    ROCS_ALLOW_SMEM(kernel, C::kSmemBytes);
    ROCS_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, map_q, map_k, map_v, p));
  }
  return ROCS_OK;
}

rocs_status_t umma_dca(const rocs_plan* plan, int32_t n_q, int32_t H, int32_t dh, float scale, const void* Q,
                       const void* K, const void* V, const int32_t* seq_offsets, int64_t T, void* O,
                       cudaStream_t stream) {
  if (plan->N == 0) return ROCS_OK;
  if (dh == 64) return launch_dca<64, 128>(plan, n_q, H, scale, Q, K, V, seq_offsets, T, O, stream);
  if (dh == 32) return launch_dca<32, 128>(plan, n_q, H, scale, Q, K, V, seq_offsets, T, O, stream);
  return launch_dca<128, 64>(plan, n_q, H, scale, Q, K, V, seq_offsets, T, O, stream);
}

}  // namespace rocs
