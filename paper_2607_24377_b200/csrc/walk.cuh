// The walking attention kernel: MXFP4 and NVFP4 forward, one query tile per work item (paper Algorithm 2, lines 6-19; launched by
// forward_walk.cu and forward_nvfp4.cu).  MXFP4: value for value the arithmetic of forward.cu.
//
// One CTA per SM walks work items of one query tile (128 rows of one head); the tiles of all its items form one stream
// f = 0, 1, 2, ... (KV tiles of 128 keys in ascending order within an item), and barriers, tensor memory and the pipelines
// run on across items.  Up to 48 KV tiles (kStaticTiles; NVFP4 3) a CTA's items are fixed at the launch, every 148th.  Above, the grid has
// a CTA per item, and a CTA that is done with an item takes over one that has not started (kTake): with fixed shares a launch
// beside that holds a few SMs for long leaves whole shares to come last.  Whole call, us, beside 4 CTAs that stay, fixed / taken:
// 24 x 8192 937 / 550 (direct row sum 1023 / 589), NVFP4 40 x 4096 453 / 293 (490 / 318), 40 x 8192 x 1024 272 / 178.  Alone, NVFP4, fixed /
// taken: 40 x 18900 at 1, 2, 3, 4 tiles 136.1 / 141.5, 160.1 / 167.2, 190.6 / 194.4, 219.0 / 220.9, 24 x 8192 at 4, 16, 48 66.4 / 66.4, 172.8 /
// 169.2, 445.3 / 433.5; up to 3 tiles a call whose last share comes late still takes less than with two query tiles per CTA (297 us at
// 40 x 18900 x 384).  MXFP4 below 49 tiles stays with fixed shares: alone, taken ones are up to 2 % behind (24 x 30000 at 24 tiles, fp32
// output; direct row sum, 24 to 48 tiles, up to 1 %), beside a launch that holds SMs they would be ahead (40 x 4096 393 / 248).
// Roles (736 threads):
//   warps 0-15   softmax, two teams of eight: team f & 1 takes tile f.  Two threads a row, one half of 64 keys each.  A team
//                has a score buffer of its own, so that neither waits for the other to take its scores; what passes from
//                team to team is the maxima of a tile, two floats a row (a named barrier at which the owners of the next tile
//                wait and the posters only arrive).  They are posted before the exponentials, but the others are let on only
//                behind three quarters of them: teams that take their exponentials at the same time also wait at the same time.
//   warps 16-19  scaling: alpha, the accumulator's rescaling (Algorithm 2 line 15) and the epilogue, one warp per quarter of
//                tensor memory.  The softmax warps never touch the accumulator and go straight on to the next item.
//   warp 20      score products S(f) = Q K_f^T;   warp 21  output products O += P(f) [V_f | 1];   warp 22  copies
//
// What bounds it: the exponential unit (1024 cycles per 128 x 128 tile and SM if it had to take all) and the latency around it: a
// memory or barrier instruction queues behind the exponentials of its SM sub-partition, and every tile waits for the slowest of
// the four.  Cycles per tile, 16 x 32768, PNQ 1315 -> 1205 (launch 4741 -> 4345 us), 24 x 8192 1443 -> 1343, 40 x 18900 x 512
// 1641 -> 1440, x 250 2035 -> 1705; direct sum 1433 -> 1391, 1557 -> 1524, 1706 -> 1580, 2100 -> 1719.  What gave it, in these figures:
//  - With the row sum from P-hat, which needs a probability's code and not its value, three or (MXFP4, items taken) four pairs of
//    exponentials in sixteen are a polynomial on the multipliers (exp2_poly): 16 x 32768 at 0, 2, 3, 4, 5 pairs 1343, 1256, 1225, 1205, 1204, 24 x
//    8192 1467, 1386, 1357, 1343, 1361, 40 x 4096 1502, 1416, 1390, 1395, 1421, 40 x 18900 x 512 at 1 to 4 1509, 1470, 1460, 1545: the
//    scaling warps multiply as well, in nearly every tile of a short sequence.  So three where shares are fixed, four elsewhere;
//    NVFP4 three (four: 24 x 8192 x 512 66.6 -> 67.4, 24 x 8192 560 -> 563, 40 x 16384 3207 -> 3215 us for the call).
//  - The issuing warps wait at named barriers, which neither side's memory queue delays: from the last read of a score buffer to its next
//    product took 600 cycles with an mbarrier, 50 so.  The compiler has to leave the arrival where it is (here()).
//  - The scaling warps load 16 columns while they multiply or convert 16 others, and let the next item's first product go as soon as
//    the last ones are in registers, in front of the fence and the output copies (40 x 18900 x 512 1542 -> 1474 in one series).
//  - What a scaling or issuing warp takes from shared memory (the next item) is made uniform by a shuffle: otherwise the compiler
//    takes everything behind it for divergent, and each tile of the scaling warps took 200 cycles longer.
// An issuing warp slows the softmax warps of its own SM sub-partition, hence two issuers and the copies on three different ones.
// The scores stay in tensor memory until they are used (each half is read for its maximum and once more for its exponentials), so
// that a thread holds 32 of them and 23 warps fit the register file at 80 (at 72 registers and 28 warps 16 x 32768 takes 5 %
// longer, direct 12 %).  Per-tile work of a warp is kept short by immediate offsets (the parity of the team's tile count is a template argument).
// Not kept: four more warps that take the maxima of the next tile, two or four softmax threads a row (1380, 1414), shared exponents
// of the second block behind the first one's exponentials (no change), larger batches of exponentials in a row (1410-1470).
//
// Tensor memory (512 columns): scores [0,128) and [128,256), accumulator and row sum [256,400), scales behind it: Q 4 slots,
// K 4, V 8, P 4.  Slots are as many as it takes that a copy never follows a product that still reads the slot.
//
// NVFP4 (kNv; E2M1 in blocks of 16, E4M3 block scale, one fp32 scale per head and operand; include/mxattn.h has the recipe):
//  - tcgen05.mma kind::mxf4nvf4, block16: an operand tile has two scale atoms, 8 columns a slot.  Q 2 slots, K 3, V 4, P 4 fit, if V's
//    slots hold no scales of ones: the row sum P-hat 1 (PNQ) is a product of its own with a tile of 16 rows of ones.  Q's scales are
//    copied behind the wait for the score buffer, V's behind a wait for O(f - 4).
//  - The tensor scales stay outside the tensor core: s_T(Q) s_T(K) softmax_scale is the exponent's multiplier, s_T(V) and, with the
//    direct placement, s_T(P) = fl32(1/2688) (the softmax tile's maximum is known to be 1) the output's factor; under PNQ s_T(P) cancels
//    against the row sum.  The copy warp leaves both factors of an item in shared memory, eight items deep: what reads them
//    last, the scaling warps, is at most six tiles behind the scores.
//  - Per block of 16: M = its largest p = exp2(s_max c - m c), d = E4M3(fl32(fl32(M 2688) fl32(1/6))), scale byte d; per element
//    E2M1(exp2(s c - m c + log2(2688 / d))): the multiplier folded into the exponent differs from the recipe's fl32(p r) by
//    about 2e-7 relative for the blocks that carry a row, d > 168, the order of ex2.approx itself, and by up to 1.5e-6 for the smallest
//    scales, whose logarithm is a larger number; a block with d = 0 keeps r = 1, its codes are 0 either way.
// Whole call, us, two query tiles per CTA as in forward.cu, which it was before / walking, the outputs bit for bit the same: PNQ
// 40 x 16384 3801 / 3199, 40 x 4096 331 / 267, direct 40 x 16384 3990 / 3623, 24 x 8192 719 / 623, 24 x 2000 74 / 59, 24 x 20000 x 512 228 / 157.
//
// Every wait at an mbarrier is bounded (mbar_wait_soft / role_wait), and none is stranded at a named barrier.  A softmax warp keeps its
// meetings with the other team to the end (team_tiles).  An issuing warp looks at the abort flag before it waits for softmax
// and scaling warps; if it is not up, the tile's scores have been issued, and all of them come: they go on when a wait of theirs runs
// out, and when they leave they come once more (leave(), the epilogue).  They come to a tile no earlier than the issuing warp can
// be there: in a healthy run the scores of tile f + 2 (f + 4) need the product that is issued behind the wait, afterwards a wait
// that is given up takes 4 us.  An item whose accumulator was still to be read when the flag went up is not stored.  tests/test_give_up_protocol.py has a model of all this.
#pragma once
#include <cuda_fp16.h>

#include "common.cuh"
#include "tc_helpers.cuh"

namespace mxattn {
namespace walk {
using namespace fwd;

constexpr int kSoftmaxWarps = 16, kScaleWarps = 4, kTeamWarps = kSoftmaxWarps / 2;
constexpr int kIssuer1 = kSoftmaxWarps + kScaleWarps, kIssuer2 = kIssuer1 + 1, kProducer = kIssuer2 + 1;
constexpr int kThreads = 32 * (kProducer + 1);
constexpr int kStages = 6;
constexpr int kXSlot = 128 * 2 * 4;
enum Bar { BAR_Q = 0, BAR_QEMPTY = 2, BAR_KFULL = 4, BAR_ODONE = BAR_KFULL + kStages, BAR_SFULL = BAR_ODONE + kStages,
           BAR_X = BAR_SFULL + 2 /* [quarter][tile & 3]: maxima posted */, BAR_NEXT = BAR_X + 16,
           BAR_ITEM = BAR_NEXT + 1 /* items n & 7 are known (kTake) */, kNumBars = BAR_ITEM + 8 };

template <bool kNv> struct Lay {                                  // shared memory, tensor memory
  static constexpr int kSF = (kNv ? 2 : 1) * kTileScaleBytes;     // scale bytes of an operand tile: one or two atoms
  static constexpr int kN2 = kNv ? 128 : 144;                     // GEMM 2 N: 128 channels and, MXFP4, 16 rows of ones (column 128 = row sum of P-hat)
  static constexpr int kVStageBytes = kN2 * 64;
  static constexpr int kOffQ = 0;                                 // 2 buffers
  static constexpr int kOffK = kOffQ + 2 * kTileCodeBytes;
  static constexpr int kOffV = kOffK + kStages * kTileCodeBytes;
  static constexpr int kOffP = kOffV + kStages * kVStageBytes;    // 4 buffers
  static constexpr int kOffOnes = kOffP + 4 * kTileCodeBytes;     // NVFP4: the rows of ones, a tile of their own
  static constexpr int kOffOut = kOffOnes + (kNv ? 1024 : 0);     // two boxes per scaling warp
  static constexpr int kOffSFQ = kOffOut + 2 * kScaleWarps * kOutBoxBytes;
  static constexpr int kOffSFK = kOffSFQ + 2 * kSF;
  static constexpr int kOffSFV = kOffSFK + kStages * kSF;
  static constexpr int kOffSFP = kOffSFV + kStages * kSF;         // 4 buffers
  static constexpr int kOffSFOnes = kOffSFP + 4 * kSF;
  static constexpr int kOffX = kOffSFOnes + kTileScaleBytes;      // half-row maxima: [4 slots][row 128][half 2] floats
  static constexpr int kOffXL = kOffX + 4 * kXSlot;               // row sums of a tile by half (direct placement): 8 slots, laid out alike
  static constexpr int kOffTab = kOffXL + 8 * kXSlot;             // NVFP4, per E4M3 code: log2(2688 / d), d / 2688
  static constexpr int kOffC = kOffTab + (kNv ? 128 * 8 : 0);     // NVFP4, items n & 7: the exponent's multiplier, the output's factor
  static constexpr int kOffBar = kOffC + (kNv ? 8 * 8 : 0);
  static constexpr int kOffMisc = (kOffBar + kNumBars * 8 + 15) & ~15;    // tensor memory's start; abort flag, number of tiles, status on entry
  static constexpr int kOffNext = kOffMisc + 32, kOffItems = kOffNext + 16;     // answer to the request for an item; items n & 7 (-1: there is none)
  static constexpr int kSmemBytes = kOffItems + 32 + 1024;
  static_assert(kOffOut % 1024 == 0 && kSmemBytes <= 227 * 1024, "shared memory per CTA");
  // Columns of scale factors behind the accumulator, and how many an operand tile has.
  static constexpr uint32_t kSlot = kNv ? 8 : 4, kColSFQ = 400, kColSFK = 416, kColSFV = kNv ? 440 : 432, kColSFP = kNv ? 472 : 496, kColSFOnes = 504;
};
constexpr uint32_t kColS = 0, kColO = 256;
// Named barriers: 1 + quarter + 4 team: the quarter's warps of both teams (maxima); the issuing warps wait at the others, to which
// 9 + team: the team's warps come when they have read their score buffer, 11 + (tile & 3): the team's and the scaling warps when
// P-hat is in place and the accumulator scaled.
constexpr int kBarMax = 1, kBarFree = 9, kBarP = 11;
constexpr int kFreeThreads = 32 * (kTeamWarps + 1), kPThreads = 32 * (kTeamWarps + kScaleWarps + 1);
constexpr float kTensorRangeP = 2688.0f;                   // NVFP4: 448 * 6, encode scale of the softmax tile (tensor maximum 1)
constexpr float kOneSixth = 0.16666667163372040f;          // fl32(1/6)
constexpr float kInvTensorRangeP = 3.7202381e-4f;          // fl32(1/2688)

struct Params {
  const uint8_t* q_codes; const uint8_t* q_scales;
  const uint8_t* k_codes; const uint8_t* k_scales;
  const uint8_t* v_codes; const uint8_t* v_scales;
  const float* ts_q; const float* ts_k; const float* ts_v;       // NVFP4: tensor decode scales, one per head
  int* status;
  int64_t Nq, Nkv;
  int q_tiles, kv_tiles, first_item, total_items;                // items from first_item on; their number
  float scale_log2e;
  float softmax_scale;                                           // kDump
  uint8_t* dump;                                                 // per tile P-hat's image, scales and running maxima, then the row sums (include/mxattn.h)
};
constexpr int kDumpTileBytes = kTileCodeBytes + kTileScaleBytes + kTile * 4;

// Shared-memory accesses at a register plus a constant: addresses formed in front of each access cost the softmax warps
// instructions, and kept ones registers.
template <int kOff> __device__ __forceinline__ void sts128o(uint32_t a, const uint32_t (&w)[4]) {
  asm volatile("st.shared.v4.b32 [%0+%5], {%1, %2, %3, %4};" ::"r"(a), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "n"(kOff) : "memory");
}
template <int kOff> __device__ __forceinline__ void sts32o(uint32_t a, float v) { asm volatile("st.shared.f32 [%0+%2], %1;" ::"r"(a), "f"(v), "n"(kOff) : "memory"); }
template <int kOff> __device__ __forceinline__ void sts16o(uint32_t a, uint32_t v) { asm volatile("st.shared.b16 [%0+%2], %1;" ::"r"(a), "h"((uint16_t)v), "n"(kOff) : "memory"); }
template <int kOff> __device__ __forceinline__ float2 lds64o(uint32_t a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2+%3];" : "=f"(v.x), "=f"(v.y) : "r"(a), "n"(kOff) : "memory");
  return v;
}
template <int kOff> __device__ __forceinline__ void arrive_if(uint32_t b, bool me) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p mbarrier.arrive.shared::cta.b64 _, [%0+%1];\n\t}" ::"r"(b), "n"(kOff), "r"((uint32_t)me) : "memory");
}
// Takes over the work of a CTA of this grid that has not started yet.  The answer (16 bytes) and its bytes' completion arrive
// asynchronously; the index of the CTA that will not be launched, or -1 if all have been (after which nothing more may be asked).
__device__ __forceinline__ void ask_for_cta(uint32_t answer, uint32_t bar) {
  asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];" ::"r"(answer), "r"(bar) : "memory");
}
__device__ __forceinline__ int cta_taken(uint32_t answer) {
  int cta;
  asm volatile("{\n\t.reg .b128 a;\n\t.reg .pred p;\n\tld.shared.b128 a, [%1];\n\tmov.s32 %0, -1;\n\t"
               "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, a;\n\t"
               "@p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %0, a;\n\t}" : "=r"(cta) : "r"(answer) : "memory");
  return cta;
}
__device__ __forceinline__ bool role_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status, int code) {
  return __all_sync(0xFFFFFFFFu, mbar_test(bar, parity)) || mbar_wait_warp(bar, parity, abort_flag, status, code);
}

__device__ __forceinline__ bool given_up(uint32_t abort_addr) { return __any_sync(0xFFFFFFFFu, lds_volatile(abort_addr) != 0); }
// What stands in front stays in front: an exit that is never taken (a count of tiles is not negative).  An arrival at a barrier
// has no result that anything waits for, and the compiler moves it behind the exponentials that follow, 500 cycles and more.
__device__ __forceinline__ void here(int tiles) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.s32 p, %0, -5;\n\t@p exit;\n\t}" ::"r"(tiles) : "memory");
}
// Whether there is no tile f: from its item's barrier, which is also completed when no item is left.
static __device__ __noinline__ bool no_tile(uint32_t bar_item, uint32_t parity, uint32_t abort_addr, int f) {
  mbar_wait_soft<36, 0, true>(bar_item, parity, abort_addr);
  int up, all;
  asm volatile("ld.volatile.shared.v2.s32 {%0, %1}, [%2];" : "=r"(up), "=r"(all) : "r"(abort_addr) : "memory");
  return f >= all || up != 0;
}
// A scaling warp's 32 rows of the accumulator times inv_l, as bf16 into its two boxes (store_half_rows' form); `o0` holds the first 16
// columns, and the next 16 are loaded while the last ones are converted (40 x 18900 x 512: 124 -> 121 us for the launch).
__device__ __forceinline__ void drain_rows_bf16(uint32_t t_o, uint32_t box, int lane, float inv_l, uint32_t (&o0)[16]) {
  const uint64_t il2 = dup2(inv_l);
  const uint32_t x7 = (lane & 7) << 4;
  uint32_t o1[16];
  auto put = [&](const uint32_t (&v)[16], uint32_t a0, uint32_t a1) {
    uint32_t w[8];
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
      uint32_t x = v[i], y = v[i + 1];
      mul2(x, y, il2);
      asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w[i / 2]) : "f"(__uint_as_float(y)), "f"(__uint_as_float(x)));
    }
    sts128(a0, make_uint4(w[0], w[1], w[2], w[3]));
    sts128(a1, make_uint4(w[4], w[5], w[6], w[7]));
  };
#pragma unroll 1
  for (int c0 = 0; c0 < 128; c0 += 32) {
    const uint32_t a = box + (c0 >> 6) * kOutBoxBytes + lane * 128, c = (c0 & 32) << 1;      // 16-byte chunks of the row: 4 of them from byte c on
    TMEM_LD16(t_o + c0 + 16, o1);
    put(o0, a + (c ^ x7), a + ((c + 16) ^ x7));
    TMEM_LD_WAIT16(o1);
    TMEM_LD16(t_o + ((c0 + 32) & 127), o0);
    put(o1, a + ((c + 32) ^ x7), a + ((c + 48) ^ x7));
    TMEM_LD_WAIT16(o0);
  }
}
// The two boxes to the output.
__device__ __forceinline__ void copy_out(uint32_t box, int lane, const CUtensorMap* map, int row0, int bh, bool inside) {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
  if (lane == 0 && inside) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
      asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];"
                   ::"l"(map), "r"(64 * h), "r"(row0), "r"(bh), "r"(box + h * kOutBoxBytes) : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
  }
}

// instruction descriptor of kind::mxf4nvf4.block_scale.block16: A, B = E2M1 (K-major), scales UE4M3, M = 128
__device__ __forceinline__ constexpr uint32_t make_idesc_nv(int n) {
  return (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24);
}
__device__ __forceinline__ void tc_mma_nv_if(uint32_t leader, uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                             uint32_t sfa, uint32_t sfb, uint32_t accumulate) {
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %7, 0;\n\t"
               "@q tcgen05.mma.cta_group::1.kind::mxf4nvf4.block_scale.block16 [%0], %1, %2, %3, [%5], [%6], p;\n\t}"
               ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(sfa), "r"(sfb), "r"(leader) : "memory");
}
__device__ __forceinline__ float e4m3_decode(uint32_t code) {
  uint32_t h2;
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"((uint16_t)code));
  return __half2float(__ushort_as_half((unsigned short)(h2 & 0xFFFFu)));
}
// The scale atoms of an operand tile to tensor memory, and a product of K = 128 in two instructions.  MXFP4: one atom holds the scales
// of both; NVFP4: an atom each (kStepB: columns from B's first to its second).
template <bool kNv> __device__ __forceinline__ void copy_scales(uint32_t leader, uint32_t taddr, uint32_t saddr) {
  tc_cp_sf_if(leader, taddr, saddr);
  if (kNv) tc_cp_sf_if(leader, taddr + 4, saddr + kTileScaleBytes);
}
template <bool kNv, int kN, int kStepB = 4>
__device__ __forceinline__ void mma2(uint32_t leader, uint32_t d, uint64_t a, uint64_t b, uint32_t sfa, uint32_t sfb, uint32_t accumulate) {
  if constexpr (kNv) {
    tc_mma_nv_if(leader, d, a, b, make_idesc_nv(kN), sfa, sfb, accumulate);
    tc_mma_nv_if(leader, d, a + 2, b + 2, make_idesc_nv(kN), sfa + 4, sfb + kStepB, 1u);
  } else {
    tc_mma_if(leader, d, a, b, make_idesc(kN, 0), sfa, sfb, accumulate);
    tc_mma_if(leader, d, a + 2, b + 2, make_idesc(kN, 1), sfa, sfb, 1u);
  }
}
__device__ __forceinline__ float max16(const uint32_t* s) {
#define SFL(i) __uint_as_float(s[i])
  const float a = max3(SFL(0), SFL(1), SFL(2)), b = max3(SFL(3), SFL(4), SFL(5)), c = max3(SFL(6), SFL(7), SFL(8)), d = max3(SFL(9), SFL(10), SFL(11));
  const float e = max3(SFL(12), SFL(13), SFL(14));
  return fmaxf(max3(a, b, c), max3(d, e, SFL(15)));
#undef SFL
}

// Barriers, rows of ones, tables: all threads of the CTA.
template <bool kNv>
__device__ __forceinline__ void set_up(uint8_t* smem, int tid) {
  using L = Lay<kNv>;
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar0 = sbase + L::kOffBar;
  auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::kOffMisc + 8);
  volatile int* tiles_in_all = abort_flag + 1;
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar(BAR_Q + i), 1); mbar_init(bar(BAR_QEMPTY + i), 1);
      mbar_init(bar(BAR_SFULL + i), 1);
    }
    for (int s = 0; s < kStages; ++s) { mbar_init(bar(BAR_KFULL + s), 1); mbar_init(bar(BAR_ODONE + s), 1); }
    for (int i = 0; i < 16; ++i) mbar_init(bar(BAR_X + i), 1);
    mbar_init(bar(BAR_NEXT), 1);
    for (int i = 0; i < 8; ++i) mbar_init(bar(BAR_ITEM + i), 1);
    abort_flag[0] = 0;
    *tiles_in_all = 0x7FFFFFFF;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = tid; i < (kNv ? 1 : kStages) * 64; i += kThreads)  // rows of ones (code 2 = 1.0), MXFP4: behind every V stage; their scales
    reinterpret_cast<uint4*>(smem + (kNv ? L::kOffOnes : L::kOffV + (i >> 6) * L::kVStageBytes + kTileCodeBytes))[i & 63] =
        make_uint4(0x22222222u, 0x22222222u, 0x22222222u, 0x22222222u);
  constexpr uint32_t kOneScales = kNv ? 0x38383838u : 0x7F7F7F7Fu;
  if (tid < kTileScaleBytes / 16) reinterpret_cast<uint4*>(smem + L::kOffSFOnes)[tid] = make_uint4(kOneScales, kOneScales, kOneScales, kOneScales);
  // NVFP4: what a softmax thread needs of a block's scale code (E4M3, never negative): the logarithm of the element multiplier, and
  // for the direct placement its inverse.  d = 0 keeps multiplier 1.
  if (kNv && tid < 128) {
    const float d = e4m3_decode((uint32_t)tid);
    reinterpret_cast<float2*>(smem + L::kOffTab)[tid] = (tid == 0 || tid == 127) ? make_float2(0.0f, 1.0f) : make_float2(log2f(kTensorRangeP / d), d * kInvTensorRangeP);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// The part of one warp, between the setup and the teardown.  kDump (MXFP4): what the softmax warps hand to the output products, and the row
// sums, are written out as well.
template <bool kNv, bool kUos, bool kPnq, bool kOutF32, bool kTake, bool kDump = false>
__device__ __forceinline__ void play(const Params& p, const CUtensorMap& out_map, uint8_t* smem, int role, int warp, int lane) {
  using L = Lay<kNv>;
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar0 = sbase + L::kOffBar;
  auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::kOffMisc + 8);
  const uint32_t abort_addr = sbase + L::kOffMisc + 8;
  volatile int* tiles_in_all = abort_flag + 1;                   // kTake: written once, when no item is left
  volatile int* items = reinterpret_cast<volatile int*>(smem + L::kOffItems);
  constexpr uint32_t tmem = 0;
  const int T = p.kv_tiles;

  // Items of this CTA: every gridDim.x-th one, or (kTake) its own and then those of CTAs that have not started, one after another.
  // The producer asks for them; the others learn of item n from a barrier of its own, of which there are eight: scores are at most four
  // tiles ahead of the last warp to look, and the producer two items ahead of the scores.
  const int n_items = kTake ? 0x7FFFFFFF : (p.total_items - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
  const int F = kTake ? 0x7FFFFFFF : n_items * T;                // tiles of this CTA

  if (role == kProducer) {
    // =============================== producer ===============================================
    if (lane == 0) {
      bool ok = true;
      int f = 0, n = 0, s = 0;
      uint32_t ph = 0;
      for (int item = p.first_item + blockIdx.x; n < n_items && ok; ++n) {
        const int bh = item / p.q_tiles;
        const int qb = n & 1;
        if (n >= 2) ok = mbar_wait1(bar(BAR_QEMPTY + qb), (uint32_t)(((n - 2) >> 1) & 1), abort_flag, p.status, 13);
        if (!ok) break;
        if (kTake) {
          items[n & 7] = item;
          if (item < 0) {
            *tiles_in_all = n * T;
            mbar_arrive(bar(BAR_Q + qb));
            mbar_arrive(bar(BAR_ITEM + (n & 7)));
            if (T == 1) mbar_arrive(bar(BAR_ITEM + ((n + 1) & 7)));     // where the other team looks
            break;
          }
        }
        if (kNv) {                                               // read behind the item's first scores
          const float c = p.scale_log2e * ld_global(p.ts_q + bh) * ld_global(p.ts_k + bh), v = ld_global(p.ts_v + bh);
          reinterpret_cast<volatile float*>(smem + L::kOffC)[2 * (n & 7)] = c;
          reinterpret_cast<volatile float*>(smem + L::kOffC)[2 * (n & 7) + 1] = kPnq ? v : v * __fdiv_rn(1.0f, kTensorRangeP);
        }
        if (kTake) mbar_arrive(bar(BAR_ITEM + (n & 7)));
        mbar_expect_tx(bar(BAR_Q + qb), kTileCodeBytes + L::kSF);
        bulk_g2s(sbase + L::kOffQ + qb * kTileCodeBytes, p.q_codes + (int64_t)item * kTileCodeBytes, kTileCodeBytes, bar(BAR_Q + qb));
        bulk_g2s(sbase + L::kOffSFQ + qb * L::kSF, p.q_scales + (int64_t)item * L::kSF, L::kSF, bar(BAR_Q + qb));
        const int64_t kv0 = (int64_t)bh * T;
        for (int j = 0; j < T; ++j, ++f) {
          if (f >= kStages) ok = mbar_wait1(bar(BAR_ODONE + s), ph ^ 1u, abort_flag, p.status, 11);
          if (!ok) break;
          mbar_expect_tx(bar(BAR_KFULL + s), 2 * (kTileCodeBytes + L::kSF));
          bulk_g2s(sbase + L::kOffK + s * kTileCodeBytes, p.k_codes + (kv0 + j) * kTileCodeBytes, kTileCodeBytes, bar(BAR_KFULL + s));
          bulk_g2s(sbase + L::kOffSFK + s * L::kSF, p.k_scales + (kv0 + j) * L::kSF, L::kSF, bar(BAR_KFULL + s));
          bulk_g2s(sbase + L::kOffV + s * L::kVStageBytes, p.v_codes + (kv0 + j) * kTileCodeBytes, kTileCodeBytes, bar(BAR_KFULL + s));
          bulk_g2s(sbase + L::kOffSFV + s * L::kSF, p.v_scales + (kv0 + j) * L::kSF, L::kSF, bar(BAR_KFULL + s));
          if (++s == kStages) { s = 0; ph ^= 1u; }
        }
        if (!kTake) {
          item += gridDim.x;
        } else if (ok) {                                         // now, not earlier: an item taken while another is far from done may end last
          mbar_expect_tx(bar(BAR_NEXT), 16);
          ask_for_cta(sbase + L::kOffNext, bar(BAR_NEXT));
          if (!mbar_wait1(bar(BAR_NEXT), (uint32_t)(n & 1), abort_flag, p.status, 14)) {
            const long long t0 = clock64();
            while (!mbar_try(bar(BAR_NEXT), (uint32_t)(n & 1)) && clock64() - t0 < 200000000LL) {}
            ok = false;
          } else {
            item = cta_taken(sbase + L::kOffNext);
            if (item >= 0) item += p.first_item;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // read before the next answer is written
          }
        }
      }
      if (kTake && *tiles_in_all == 0x7FFFFFFF) *tiles_in_all = n * T;       // gave up; n: items begun
      if (!ok || *abort_flag) {                                  // gave up: let copies in flight land before shared memory is released
        const long long t0 = clock64();
        for (int g = (f > kStages ? f - kStages : 0); g < f; ++g)
          while (!mbar_try(bar(BAR_KFULL + g % kStages), (uint32_t)((g / kStages) & 1)) && clock64() - t0 < 200000000LL) {}
        for (int g = (n > 2 ? n - 2 : 0); g < n; ++g)
          while (!mbar_try(bar(BAR_Q + (g & 1)), (uint32_t)((g >> 1) & 1)) && clock64() - t0 < 200000000LL) {}
      }
    }
  } else if (role == kIssuer1) {
    // =============================== score products (converged warp) ========================
    const uint32_t leader = elect_one();
    constexpr uint32_t kDescHiTile = (512u >> 4) | (1u << 14) | (4u << 29);   // 64-byte swizzle, K-major
    auto desc = [](uint32_t saddr) { return ((uint64_t)kDescHiTile << 32) | (saddr >> 4); };
    int j = 0, n = 0, s = 0, sd = 0, k3 = 0;
    uint32_t ph = 0, phd = 0;
    bool ok = true;
    for (int f = 0; f < F && ok; ++f) {
      const int qb = n & 1;
      if (j == 0) {
        if (!role_wait(bar(BAR_Q + qb), (uint32_t)((n >> 1) & 1), abort_flag, p.status, 21)) break;
        if (kTake && __shfl_sync(0xFFFFFFFFu, items[n & 7], 0) < 0) break;
        tc_fence_after();
        if (!kNv) tc_cp_sf_if(leader, tmem + L::kColSFQ + 4 * (n & 3), sbase + L::kOffSFQ + qb * L::kSF);
      }
      if (!role_wait(bar(BAR_KFULL + s), ph, abort_flag, p.status, 22)) break;
      tc_fence_after();
      const uint32_t d = tmem + kColS + 128 * (f & 1), sfb = tmem + L::kColSFK + (kNv ? 8 * k3 : 4 * (f & 3)), sfa = tmem + L::kColSFQ + (kNv ? 8 * (n & 1) : 4 * (n & 3));
      const uint32_t a = sbase + L::kOffQ + qb * kTileCodeBytes, b = sbase + L::kOffK + s * kTileCodeBytes;
      copy_scales<kNv>(leader, sfb, sbase + L::kOffSFK + s * L::kSF);
      if (f >= 4) {                                              // the scores of tile f also say that its P buffer is free
        if (!role_wait(bar(BAR_ODONE + sd), phd, abort_flag, p.status, 25)) break;
        if (++sd == kStages) { sd = 0; phd ^= 1u; }
      }
      if (f >= 2) {                                              // S(f - 2) has been read
        if (given_up(abort_addr)) break;
        asm volatile("bar.sync %0, %1;" ::"r"(kBarFree + (f & 1)), "n"(kFreeThreads) : "memory");
        tc_fence_after();
      }
      if (kNv && j == 0) copy_scales<true>(leader, sfa, sbase + L::kOffSFQ + qb * L::kSF);     // the slot's last products are complete
      mma2<kNv, 128>(leader, d, desc(a), desc(b), sfa, sfb, 0u);
      if (kNv) k3 = k3 == 2 ? 0 : k3 + 1;
      tc_commit_if(leader, bar(BAR_SFULL + (f & 1)));
      if (++j == T) {
        tc_commit_if(leader, bar(BAR_QEMPTY + qb));
        j = 0; ++n;
      }
      if (++s == kStages) { s = 0; ph ^= 1u; }
    }
  } else if (role == kIssuer2) {
    // =============================== output products (converged warp) =======================
    const uint32_t leader = elect_one();
    constexpr uint32_t kDescHiTile = (512u >> 4) | (1u << 14) | (4u << 29);   // 64-byte swizzle, K-major
    auto desc = [](uint32_t saddr) { return ((uint64_t)kDescHiTile << 32) | (saddr >> 4); };
    if constexpr (kNv) tc_cp_sf_if(leader, tmem + L::kColSFOnes, sbase + L::kOffSFOnes);
    else for (int i = 0; i < 8; ++i) tc_cp_sf_if(leader, tmem + L::kColSFV + 8 * i + 4, sbase + L::kOffSFOnes);
    int j = 0, s = 0, n = 0, sd = 0;
    uint32_t ph = 0, phd = 0;
    for (int f = 0; f < F; ++f) {
      if (kTake && j == 0) {
        if (!role_wait(bar(BAR_ITEM + (n & 7)), (uint32_t)((n >> 3) & 1), abort_flag, p.status, 27) || __shfl_sync(0xFFFFFFFFu, items[n & 7], 0) < 0) break;
        ++n;
      }
      if (!role_wait(bar(BAR_KFULL + s), ph, abort_flag, p.status, 26)) break;
      tc_fence_after();
      if (kNv && f >= 4) {                                       // O(f - 4) is complete: V's slot is free
        if (!role_wait(bar(BAR_ODONE + sd), phd, abort_flag, p.status, 28)) break;
        if (++sd == kStages) { sd = 0; phd ^= 1u; }
      }
      const uint32_t sfa = tmem + L::kColSFP + L::kSlot * (f & 3), sfb = tmem + L::kColSFV + 8 * (f & (kNv ? 3 : 7));
      const uint32_t pa = sbase + L::kOffP + (f & 3) * kTileCodeBytes, vb = sbase + L::kOffV + s * L::kVStageBytes;
      copy_scales<kNv>(leader, sfb, sbase + L::kOffSFV + s * L::kSF);
      if (given_up(abort_addr)) break;
      asm volatile("bar.sync %0, %1;" ::"r"(kBarP + (f & 3)), "n"(kPThreads) : "memory");
      tc_fence_after();
      copy_scales<kNv>(leader, sfa, sbase + L::kOffSFP + (f & 3) * L::kSF);
      mma2<kNv, L::kN2>(leader, tmem + kColO, desc(pa), desc(vb), sfa, sfb, j > 0 ? 1u : 0u);
      if constexpr (kNv && kPnq)                                 // the row sum P-hat 1 (both K halves of the ones have the same scales)
        mma2<true, 16, 0>(leader, tmem + kColO + 128, desc(pa), desc(sbase + L::kOffOnes), sfa, tmem + L::kColSFOnes, j > 0 ? 1u : 0u);
      tc_commit_if(leader, bar(BAR_ODONE + s));
      if (++j == T) j = 0;
      if (++s == kStages) { s = 0; ph ^= 1u; }
    }
  } else if (role >= kSoftmaxWarps && role < kSoftmaxWarps + kScaleWarps) {
    // =============================== scaling warps: alpha, the accumulator, the epilogue ====
    const int q = warp - kSoftmaxWarps;
    const uint32_t t_o = tmem + ((uint32_t)q << 21) + kColO;
    const uint32_t aX = sbase + L::kOffX + (q * 32 + lane) * 8;
    float c = p.scale_log2e, o_scale = 1.0f;
    float m_run = -INFINITY, lA = 0.0f, lB = 0.0f, alpha1 = 1.0f, alpha2 = 1.0f;
    int f = 0, s_prev = kStages - 1;
    uint32_t ph_prev = 1;                                        // stage and parity of tile f - 1
    auto add_sums = [&](int g, float alpha) {                    // line 14 (direct), Eq. 12: tile g
      const float2 v = lds64o<L::kOffXL - L::kOffX>(aX + (g & 7) * kXSlot);
      lA = fmaf(alpha, lA, v.x);
      lB = fmaf(alpha, lB, v.y);
    };
    auto ready = [&]() {                                         // tile f: the accumulator may be written
      tc_fence_before();
      __syncwarp();
      asm volatile("bar.arrive %0, %1;" ::"r"(kBarP + (f & 3)), "n"(kPThreads) : "memory");
      if (++s_prev == kStages) { s_prev = 0; ph_prev ^= 1u; }
      ++f;
    };
    auto first_tile = [&](int n) {                               // of item n: nothing to rescale
      mbar_wait_soft<34>(bar(BAR_X + q * 4 + (f & 3)), (uint32_t)((f >> 2) & 1), abort_addr);
      if (kNv) {
        const float2 v = lds64o<0>(sbase + L::kOffC + 8 * (n & 7));
        c = v.x;
        o_scale = v.y;
      }
      const float2 mx = lds64o<0>(aX + (f & 3) * kXSlot);
      m_run = max3(mx.x, mx.y, -INFINITY);                       // a tile without a number leaves -inf, as in forward.cu
      if (!kPnq) { alpha2 = alpha1; alpha1 = 1.0f; }
      ready();
    };
    int item = p.first_item + blockIdx.x;
    bool more = true;
    auto next_item = [&](int n) {                                // whether there is an item n, and which
      if (kTake) {
        mbar_wait_soft<35, 0, true>(bar(BAR_ITEM + (n & 7)), (uint32_t)((n >> 3) & 1), abort_addr);
        item = __shfl_sync(0xFFFFFFFFu, items[n & 7], 0);        // the same for all lanes, which the compiler has to know; anything if the CTA has given up: nothing is stored then
        more = item >= 0;
      } else {
        if (n > 0) item += gridDim.x;
        more = n < n_items;
      }
      if (more) first_tile(n);
    };
    next_item(0);
    for (int n = 0; more; ++n) {
      for (int j = 1; j < T; ++j) {
        mbar_wait_soft<34>(bar(BAR_X + q * 4 + (f & 3)), (uint32_t)((f >> 2) & 1), abort_addr);
        const float2 mx = lds64o<0>(aX + (f & 3) * kXSlot);
        const float m_old = m_run;
        const float m_new = max3(mx.x, mx.y, m_old);
        m_run = m_new;
        if (!kPnq && j >= 2) add_sums(f - 2, alpha2);
        float alpha = 1.0f;
        if (__any_sync(0xFFFFFFFFu, m_new != m_old)) {
          alpha = ex2((m_old - m_new) * c);
          mbar_wait_soft<32>(bar(BAR_ODONE + s_prev), ph_prev, abort_addr);
          tc_fence_after();
          const uint64_t al2 = dup2(alpha);
          uint32_t lr = 0;
          if (kPnq) asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(lr) : "r"(t_o + 128) : "memory");
          uint32_t o0[16], o1[16];
          TMEM_LD16(t_o, o0);
          TMEM_LD_WAIT16(o0);
#pragma unroll 1
          for (int c0 = 0; c0 < 128; c0 += 32) {                 // one half is loaded while the other is multiplied
            TMEM_LD16(t_o + c0 + 16, o1);
#pragma unroll
            for (int i = 0; i < 16; i += 2) mul2(o0[i], o0[i + 1], al2);
            TMEM_ST16(t_o + c0, o0);
            TMEM_LD_WAIT16(o1);
            TMEM_LD16(t_o + ((c0 + 32) & 127), o0);              // (behind the last one nothing uses it)
#pragma unroll
            for (int i = 0; i < 16; i += 2) mul2(o1[i], o1[i + 1], al2);
            TMEM_ST16(t_o + c0 + 16, o1);
            TMEM_LD_WAIT16(o0);
          }
          if (kPnq) {
            asm volatile("" : "+r"(lr));
            lr = __float_as_uint(__uint_as_float(lr) * alpha);
            asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%1], {%0};" ::"r"(lr), "r"(t_o + 128) : "memory");
          }
          tmem_st_wait();
        }
        if (!kPnq) { alpha2 = alpha1; alpha1 = alpha; }
        ready();
      }
      // ---- epilogue: O = O~ / l (line 18) ----
      const int bh = item / p.q_tiles, row0 = (item - bh * p.q_tiles) * kTile + q * 32;
      const bool inside = row0 < p.Nq;
      if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");      // the previous item's copies have left the boxes
      __syncwarp();
      mbar_wait_soft<33>(bar(BAR_ODONE + s_prev), ph_prev, abort_addr);
      tc_fence_after();
      float l;
      uint32_t lr = 0, o0[16];
      if (kPnq) asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(lr) : "r"(t_o + 128) : "memory");
      TMEM_LD16(t_o, o0);
      if (!kPnq) {
        if (T >= 2) add_sums(f - 2, alpha2);
        add_sums(f - 1, alpha1);
        l = lA + lB;
        lA = lB = 0.0f;
      }
      TMEM_LD_WAIT16(o0);
      if (kPnq) {
        asm volatile("" : "+r"(lr));
        l = __uint_as_float(lr);
      }
      const float inv_l = (kNv ? o_scale : 1.0f) / l;
      if (kDump) reinterpret_cast<float*>(p.dump + (int64_t)p.total_items * T * kDumpTileBytes)[(int64_t)item * kTile + q * 32 + lane] = l;
      if (lds_volatile(abort_addr) != 0) {                       // given up: this item and later ones are not stored, and the output products wait for this warp once more at most
        asm volatile("bar.arrive %0, %1;" ::"r"(kBarP + (f & 3)), "n"(kPThreads) : "memory");
        break;
      }
      const uint32_t box = sbase + L::kOffOut + 2 * q * kOutBoxBytes;
      if constexpr (kOutF32) {
#pragma unroll 1
        for (int h = 0; h < 2; ++h) store_half_rows<true>(t_o + 64 * h, box + h * kOutBoxBytes, lane, inv_l, &out_map, 64 * h, row0, bh, inside);
        next_item(n + 1);
      } else {
        drain_rows_bf16(t_o, box, lane, inv_l, o0);
        next_item(n + 1);
        copy_out(box, lane, &out_map, row0, bh, inside);
      }
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
  } else if (role < kSoftmaxWarps) {
    // =============================== softmax warps ==========================================
    // Two teams of eight warps take the tiles in turn (tile f: team f & 1); two threads a row, 64 keys each.
    const int quarter = warp & 3, h = (warp >> 2) & 1, t = warp >> 3, row = quarter * 32 + lane;
    const uint32_t t_s = tmem + ((uint32_t)quarter << 21) + 128 * t + 64 * h;
    const uint32_t aM = sbase + L::kOffX + row * 8 + t * kXSlot;                                // own maxima (+ 2 slots on every other own tile)
    const uint32_t aMp0 = sbase + L::kOffX + row * 8 + (t ? 0 : 3) * kXSlot;                    // the tile before, at even own tiles
    const uint32_t aMp1 = sbase + L::kOffX + row * 8 + (t ? 2 : 1) * kXSlot;                    // ... at odd ones
    const uint32_t aP0 = sbase + L::kOffP + t * kTileCodeBytes + tile_code_offset(row, 2 * h);
    const uint32_t aP1 = sbase + L::kOffP + t * kTileCodeBytes + tile_code_offset(row, 2 * h + 1);
    const uint32_t aSF = sbase + L::kOffSFP + t * L::kSF + (kNv ? h * kTileScaleBytes + tile_scale_offset(row, 0) : tile_scale_offset(row, 2 * h));
    const uint32_t barT = bar0 + 8 * t, barX = bar0 + 32 * quarter + 8 * t;
    const int idOwn = kBarMax + quarter + 4 * t, idOther = kBarMax + quarter + 4 * (t ^ 1);
    const int ragged = (int)(p.Nkv & (kTile - 1)) != 0 ? (int)(p.Nkv & (kTile - 1)) - 64 * h : 64;     // keys of this half in an item's last tile
    float c = p.scale_log2e;                                     // NVFP4: with Q's and K's tensor scales, another one for each head
    uint64_t cc2 = dup2(c);
    float m_run = -INFINITY;                                     // of the team's last tile
    int jn = t % T, n_own = t / T;                               // index of tile f in its item, and the item's
    uint32_t xl = 0;                                             // slot of the row sums
    if (t == 1) asm volatile("bar.arrive %0, 128;" ::"r"(idOther) : "memory");     // nothing comes before tile 0
    auto max32 = [&](const uint32_t (&s)[32]) {
#define SFL(i) __uint_as_float(s[i])
      float q[10];
#pragma unroll
      for (int i = 0; i < 10; ++i) q[i] = max3(SFL(3 * i), SFL(3 * i + 1), SFL(3 * i + 2));
      q[0] = max3(q[0], q[1], q[2]); q[3] = max3(q[3], q[4], q[5]); q[6] = max3(q[6], q[7], q[8]); q[9] = max3(q[9], SFL(30), SFL(31));
#undef SFL
      return fmaxf(max3(q[0], q[3], q[6]), q[9]);
    };
    auto exponent = [&](float bmax, float m_new, uint64_t& nb, uint32_t& sf) {
      const float d = (bmax - m_new) * c;
      const float fl = __fadd_rd(d, 12582912.0f) - 12582912.0f;                    // floor(d)
      float ef = fl + ((kUos && (d - fl) > 0.85798097f) ? -1.0f : -2.0f);
      ef = fmaxf(ef, -127.0f);
      if (d < -126.0f) ef = 0.0f;
      sf = __float_as_uint(ef + 12582912.0f) - (0x4B400000u - 127u);               // e + 127
      nb = dup2(-(m_new * c) - ef);
    };
    // NVFP4, two blocks of 16: scale codes, constant terms of the exponents, and the inverse multipliers.  The block's largest
    // probability by the elements' own expression, then the two-level recipe, two blocks per conversion; the element multiplier
    // 2688 / d is folded into the exponent as its logarithm, from a table of the 127 codes (log2f of the rounded quotient: within a unit
    // in the last place plus the quotient's 9e-8; computed per block it was 22 instructions instead of 8).  A block whose scale
    // rounds to zero keeps multiplier 1: its probabilities are below 2.2e-6 and round to code 0 either way, and the direct
    // placement still sums them.
    auto block_scales = [&](const float (&bmax)[2], float m_new, float (&nb)[2], float (&inv_r)[2]) {
      const float nmc = -(m_new * c);
      const float y0 = __fmul_rn(__fmul_rn(ex2(fmaf(bmax[0], c, nmc)), kTensorRangeP), kOneSixth);
      const float y1 = __fmul_rn(__fmul_rn(ex2(fmaf(bmax[1], c, nmc)), kTensorRangeP), kOneSixth);
      uint16_t code2;
      asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(code2) : "f"(y1), "f"(y0));
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const float2 v = lds64o<L::kOffTab>(sbase + ((u ? (uint32_t)code2 >> 8 : (uint32_t)code2 & 0xFFu) << 3));
        nb[u] = fmaf(-m_new, c, v.x);                            // one rounding: -(m_new c) + log2(2688 / d)
        inv_r[u] = v.y;
      }
      return (uint32_t)code2;
    };
    auto codes = [&](const uint32_t (&s)[32], int g, uint64_t nb, float& sx, float inv_r) {     // eight exponentials, their codes
      float x[8];
#pragma unroll
      for (int i = 0; i < 8; i += 2) {
        fma2(s[8 * g + i], s[8 * g + i + 1], cc2, nb, x[i], x[i + 1]);
        const bool poly = kTake && !kNv ? i == ((g & 1) ? 2 : 6) : g != 0 && i == ((g & 1) ? 6 : 4);     // which pairs: 1 % between the placements tried
        if (kPnq && poly) {
          exp2_poly(x[i], x[i + 1]);
        } else {
          x[i] = ex2(x[i]);
          x[i + 1] = ex2(x[i + 1]);
        }
      }
      if constexpr (kPnq) {
        return pack_e2m1x8_relu(x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7]);
      } else {
        float s0, s1;
        add2x2(x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7], s0, s1);
        sx = kNv ? fmaf(s0 + s1, inv_r, sx) : sx + (s0 + s1);
        return pack_e2m1x8(x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7]);
      }
    };
    auto meet_others = [&]() { asm volatile("bar.arrive %0, 128;" ::"r"(idOther) : "memory"); };
    auto tile = [&](auto kk) {                                   // kk: parity of the team's tile count
      constexpr int k = decltype(kk)::value;
      mbar_wait_soft<31, 8 * BAR_SFULL, true>(barT, (uint32_t)k, abort_addr);
      tc_fence_after();
      if (kNv && jn < 2) {                                       // the team's first tile of an item
        c = lds32f(sbase + L::kOffC + 8 * (n_own & 7));
        cc2 = dup2(c);
      }
      if (jn == T - 1 && ragged < 64) mask_scores(t_s, ragged, 64);
      float b0, b1, bm0[2], bm1[2];
      uint32_t s[32];
      {
        uint32_t s1[32];
        TMEM_LD32(t_s + 32, s1);
        TMEM_LD_WAIT32(s1);
        if constexpr (kNv) {
          bm1[0] = max16(s1); bm1[1] = max16(s1 + 16);
          asm volatile("" : "+f"(bm1[0]), "+f"(bm1[1]));
          b1 = fmaxf(bm1[0], bm1[1]);
        } else {
          b1 = max32(s1);
          asm volatile("" : "+f"(b1));
        }
        TMEM_LD32(t_s, s);
      }
      TMEM_LD_WAIT32(s);
      if constexpr (kNv) {
        bm0[0] = max16(s); bm0[1] = max16(s + 16);
        b0 = fmaxf(bm0[0], bm0[1]);
      } else {
        b0 = max32(s);
      }
      sts32o<2 * k * kXSlot>(aM + 4 * h, fmaxf(b0, b1));
      asm volatile("bar.sync %0, 128;" ::"r"(idOwn) : "memory");
      const float2 mo = lds64o<2 * k * kXSlot>(aM), mp = lds64o<0>(k ? aMp1 : aMp0);
      arrive_if<8 * BAR_X + 16 * k>(barX, h == 0 && lane == 0);
      const float prev = jn >= 1 ? fmaxf(mp.x, mp.y) : -INFINITY, run = jn >= 2 ? m_run : -INFINITY;
      const float m_new = max3(fmaxf(mo.x, mo.y), prev, run);    // line 10
      m_run = m_new;
      uint8_t* image = nullptr;                                  // kDump: of this tile
      if (kDump) {
        const int item = kTake ? items[n_own & 7] : (int)blockIdx.x + n_own * (int)gridDim.x;
        image = p.dump + ((int64_t)item * T + jn) * kDumpTileBytes;
        if (h == 0) reinterpret_cast<float*>(image + kTileCodeBytes + kTileScaleBytes)[row] = m_new * p.softmax_scale;     // (m is kept in unscaled score units)
      }
      jn += 2;
      if (jn >= T) { jn -= T; if (kNv || kDump) ++n_own; }
      if (jn >= T) { jn -= T; if (kNv || kDump) ++n_own; }                // T = 1; left out where T is larger, PNQ takes 9 % longer (24 x 8192)
      // NVFP4, the scales of the other 32 keys (two exponentials, a table): in front of the first exponentials, or in the gap where
      // their scores are loaded.  There the score buffer is given back later, which short sequences with PNQ do not make up for.
      // Whole call, us, in front / in the gap: direct 40 x 16384 3770 / 3710, 24 x 8192 646 / 636, 40 x 4096 299.7 / 297.7, 40 x 18900 x
      // 512 232.2 / 230.6, PNQ 40 x 16384 3321 / 3293, with fixed shares 40 x 4096 275.3 / 279.5, 24 x 8192 x 2000 175.3 / 177.5.
      constexpr bool kLate = kNv && (!kPnq || kTake);
      uint64_t nb0, nb1;
      uint32_t sf0, sf1;
      float e0[2], e1[2], r0[2], r1[2];                          // NVFP4: of the first 32 keys' two blocks, and of the others
      if constexpr (kNv) {
        sf0 = block_scales(bm0, m_new, e0, r0);
        if (!kLate) {
          sf1 = block_scales(bm1, m_new, e1, r1);
          sts32o<2 * k * L::kSF>(aSF, __uint_as_float(sf0 | (sf1 << 16)));
        }
      } else {
        exponent(b0, m_new, nb0, sf0);
        exponent(b1, m_new, nb1, sf1);
        sts16o<2 * k * L::kSF>(aSF, sf0 | (sf1 << 8));
        if (kDump) *reinterpret_cast<uint16_t*>(image + kTileCodeBytes + tile_scale_offset(row, 2 * h)) = (uint16_t)(sf0 | (sf1 << 8));
      }
      float sx0 = 0.0f, sx1 = 0.0f;
      uint32_t w[4];
#pragma unroll
      for (int g = 0; g < 4; ++g) w[g] = codes(s, g, kNv ? dup2(e0[g >> 1]) : nb0, sx0, kNv ? r0[g >> 1] : 1.0f);
      uint32_t s1[32];
      TMEM_LD32(t_s + 32, s1);
      if (kLate) {
        sf1 = block_scales(bm1, m_new, e1, r1);
        sts32o<2 * k * L::kSF>(aSF, __uint_as_float(sf0 | (sf1 << 16)));
      }
      sts128o<2 * k * kTileCodeBytes>(aP0, w);
      if (kDump) *reinterpret_cast<uint4*>(image + tile_code_offset(row, 2 * h)) = make_uint4(w[0], w[1], w[2], w[3]);
      TMEM_LD_WAIT32(s1);
      tc_fence_before();
      __syncwarp();
      asm volatile("bar.arrive %0, %1;" ::"r"(kBarFree + t), "n"(kFreeThreads) : "memory");      // the score buffer may be overwritten
      here(p.kv_tiles);
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        w[g] = codes(s1, g, kNv ? dup2(e1[g >> 1]) : nb1, kNv ? sx0 : sx1, kNv ? r1[g >> 1] : 1.0f);
        if (g == 1) { meet_others(); here(p.kv_tiles); }
      }
      sts128o<2 * k * kTileCodeBytes>(aP1, w);
      if (kDump) *reinterpret_cast<uint4*>(image + tile_code_offset(row, 2 * h + 1)) = make_uint4(w[0], w[1], w[2], w[3]);
      if (!kPnq) {
        sts32o<L::kOffXL - L::kOffX>(aM + 4 * h + xl, kNv ? sx0 : fmaf(sx1, __uint_as_float(sf1 << 23), fmaf(sx0, __uint_as_float(sf0 << 23), 0.0f)));   // Eq. 12
        xl = (xl + 2 * kXSlot) & (8 * kXSlot - 1);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      asm volatile("bar.arrive %0, %1;" ::"r"(kBarP + t + 2 * k), "n"(kPThreads) : "memory");
    };
    // Gives up at its tile f: the issuing warps, which look at the flag before they wait for this team, may have begun to wait
    // for that tile, no later one; the pause lets them begin before this warp comes.
    auto leave = [&](int f) {
      const long long t0 = clock64();
      while (clock64() - t0 < 40000) {}
      asm volatile("bar.arrive %0, %1;" ::"r"(kBarFree + t), "n"(kFreeThreads) : "memory");
      asm volatile("bar.arrive %0, %1;" ::"r"(kBarP + (f & 3)), "n"(kPThreads) : "memory");
    };
    if (!kTake) {
      team_tiles(t, F, abort_addr, idOwn, idOther, tile, leave);
    } else {
      // At the team's first tile of item n: whether there is one.  If the CTA has given up, the meetings that are kept are those of the
      // tiles that the producer says it has begun (it watches the flag too): whole items, so that no warp is beyond them.
      // NVFP4 counts items anyway (n_own, jn); with counters of its own the loop spilled a register.
      int f = t, n = 0, known = 0;                               // known: tiles of the items up to n
      auto ends = [&]() {
        if constexpr (kNv) {
          if (jn >= 2) return false;
          n = n_own + 1;
          f = n_own * T + jn;
        } else {
          if (f < known) return false;
          known += T;
          ++n;
        }
        return (bool)__any_sync(0xFFFFFFFFu, no_tile(bar(BAR_ITEM + ((n - 1) & 7)), (uint32_t)(((n - 1) >> 3) & 1), abort_addr, f));
      };
      for (;; f += 2) {
        if (ends()) break;
        tile(std::integral_constant<int, 0>{});
        f += 2;
        if (ends()) break;
        tile(std::integral_constant<int, 1>{});
      }
      if (lds_volatile(abort_addr) != 0) {
        leave(f);
        int all = *tiles_in_all;
        for (int i = 0; all == 0x7FFFFFFF && i < (1 << 28); ++i) all = *tiles_in_all;
        if (all != 0x7FFFFFFF) team_meetings(f, all, idOwn, idOther);
      }
    }
  }
}

// Items p.first_item .. + p.total_items - 1 of `bh` heads, by a kernel that takes them from CTAs that have not started, or has fixed shares.
using Kernel = void (*)(const Params, const CUtensorMap);
template <bool kNv> inline bool takes(const Params& p, int64_t n_sm) { return p.kv_tiles > (kNv ? kStaticTilesNv : kStaticTiles) && p.total_items > n_sm; }
inline int launch(Kernel kern, int smem_bytes, const Params& p, bool take, int64_t n_sm, int64_t bh, void* o, unsigned flags, cudaStream_t stream) {
  CUtensorMap out_map;
  const int map_rc = encode_output_map(&out_map, o, bh, p.Nq, flags & MXATTN_FLAG_OUT_FP32);
  if (map_rc != MXATTN_OK) return map_rc;
  if (!ensure_dynamic_smem((const void*)kern, smem_bytes)) return MXATTN_ECUDA;
  return launch_pdl(kern, dim3((unsigned)(take || p.total_items < n_sm ? p.total_items : n_sm)), kThreads, smem_bytes, stream, p, out_map) == cudaSuccess ? MXATTN_OK : MXATTN_ECUDA;
}

}  // namespace walk
}  // namespace mxattn
