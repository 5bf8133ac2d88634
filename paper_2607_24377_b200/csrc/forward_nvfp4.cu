// NVFP4 variant of the fused attention forward: the paper's comparison baseline "NVFP4" (Section 5.2) -- Q, K, V and
// the softmax tile in NVFP4 (E2M1 in blocks of 16, E4M3 block scale, fp32 tensor scale), nothing else changed -- run by
// the same CTA structure, pipeline and online-softmax recurrence as the MXFP4 kernel in forward.cu (Algorithm 2 with
// the quantizer exchanged), so that the two formats can be compared at equal kernel design.
//
//   GEMM 1  S_raw = Q-hat_t K-hat_j^T            tcgen05.mma kind::mxf4nvf4, block16, UE4M3 scales; M = 128, N = 128
//   GEMM 2  O_t  += P-hat_t [V-hat_j | 1]        N = 144: the 16 extra rows hold the constant 1 (code 2, scale 1.0),
//                                                so column 128 accumulates the row sum of the quantized probabilities
// The tensor-level scales are applied outside the tensor core: S = S_raw * s_T(Q) s_T(K) * softmax_scale (folded into
// the exponent's multiplier), O = O_raw * s_T(V) * s_T(P) / l with s_T(P) = fl32(1/2688) (the softmax tile's maximum
// is known to be 1); under PNQ l = l_raw * s_T(P) and s_T(P) cancels.
//
// Per KV tile a softmax thread (two threads per query row, 64 key columns = 4 blocks of 16 each):
//   per block: M = its largest p = exp2(s_max * c - m_new * c), d = E4M3(fl32(fl32(M * 2688) * fl32(1/6))), scale byte = d
//   per element: codes = E2M1(exp2(s_i * c - m_new * c + log2(2688 / d)))      half a packed fma + one ex2
// which is the library's NVFP4 recipe (include/mxattn.h) with the tensor maximum 1, the element multiplier
// r = 2688 / d folded into the exponent (the recipe's fl32(p_i * r) differs from this by about 2e-7 relative for the blocks
// that carry a row, d > 168, the order of ex2.approx itself, and by up to 1.5e-6 for the smallest scales, whose logarithm
// is a larger number; a block with d = 0 keeps r = 1, its codes are 0 either way).
//
// One CTA per work item: two query tiles of one head, or one where the last wave would leave half of the SMs idle
// (common.cuh; 2 heads of 1024: 29 -> 23 us, 40 heads of 16384: 4090 -> 4033).  The output leaves as tensor copies
// (store_half_rows; 40 heads of 4096 x 512: 92.1 -> 87.9 us, fp32 105.6 -> 96.5).  Tensor-memory map:
// S [0,128), O_0 [128,272), O_1 [272,416), scale factors from 416 (8 columns per operand tile: two atoms).
// Every mbarrier wait is bounded; a softmax warp that gives up keeps its partner's appointments (tc_helpers.cuh).
#include <cuda_fp16.h>

#include <type_traits>

#include "common.cuh"
#include "tc_helpers.cuh"

namespace mxattn {
namespace fwdnv {
using namespace fwd;

constexpr int kCols = 64;                        // key columns per softmax thread
constexpr int kSoftmaxWarps = 16;
constexpr int kThreads = 32 * (kSoftmaxWarps + 2);
constexpr int kStages = 4;
constexpr int kNV = 144;
constexpr int kVStageBytes = kNV * 64;
constexpr int kSF = 2 * kTileScaleBytes;         // scale bytes per operand tile: two atoms (8 blocks of 16 per row)

constexpr int kOffQ = 0;                                   // 2 tiles
constexpr int kOffK = kOffQ + 2 * kTileCodeBytes;          // 4 stages
constexpr int kOffV = kOffK + kStages * kTileCodeBytes;    // 4 stages of 144 rows
constexpr int kOffP = kOffV + kStages * kVStageBytes;      // 2 tiles
constexpr int kOffSFQ = kOffP + 2 * kTileCodeBytes;        // 2 x 1024
constexpr int kOffSFK = kOffSFQ + 2 * kSF;                 // 4 x 1024
constexpr int kOffSFV = kOffSFK + kStages * kSF;           // 4 x 1024
constexpr int kOffSFOnes = kOffSFV + kStages * kSF;        // 512 (one atom serves both K halves)
constexpr int kOffSFP = kOffSFOnes + kTileScaleBytes;      // 2 x 1024
constexpr int kOffBar = kOffSFP + 2 * kSF;
enum Bar { BAR_Q = 0, BAR_KFULL = 1, BAR_KEMPTY = BAR_KFULL + kStages, BAR_SFULL = BAR_KEMPTY + kStages, BAR_SFREE = BAR_SFULL + 2,
           BAR_PFULL = BAR_SFREE + 1, BAR_ODONE = BAR_PFULL + 2, kNumBars = BAR_ODONE + 2 };
constexpr int kOffMisc = kOffBar + kNumBars * 8;
constexpr int kOffMax = kOffMisc + 64;                     // half-row exchange: [parity 2][tile 2][half 2][128] floats
constexpr int kOffTab = kOffMax + 2 * 2 * 2 * 128 * 4;           // per E4M3 code: log2(2688 / d), d / 2688
constexpr int kOffOut = (kOffTab + 128 * 8 + 1023) & ~1023;           // output staging: one box per softmax warp
constexpr int kSmemBytes = kOffOut + kSoftmaxWarps * kOutBoxBytes + 1024;
static_assert(kSmemBytes <= 227 * 1024, "shared memory per CTA");

// tensor-memory columns: per operand tile 8 scale columns (atom of K half 0, atom of K half 1); a V slot interleaves
// the atoms of the ones rows: [V half 0][ones][V half 1][ones]
constexpr uint32_t kColS = 0, kColO0 = 128, kColO1 = 272, kColSFQ = 416, kColSFK = 432, kColSFV = 448, kColSFP = 480;

constexpr float kTensorRangeP = 2688.0f;                   // 448 * 6: encode scale of the softmax tile (tensor maximum 1)
constexpr float kOneSixth = 0.16666667163372040f;          // fl32(1/6)
constexpr float kInvTensorRangeP = 3.7202381e-4f;          // fl32(1/2688)

struct Params {
  const uint8_t* q_codes; const uint8_t* q_scales;
  const uint8_t* k_codes; const uint8_t* k_scales;
  const uint8_t* v_codes; const uint8_t* v_scales;
  const float* ts_q; const float* ts_k; const float* ts_v;   // tensor decode scales, one per head
  int* status;
  int64_t Nq, Nkv;
  int q_tiles, kv_tiles, q_pairs;
  int pair_ctas;        // CTAs before this one take two query tiles, the others one (TileSplit)
  float scale_log2e;
};

// instruction descriptor of kind::mxf4nvf4.block_scale.block16: A, B = E2M1 (K-major), scales UE4M3, M = 128
__device__ __forceinline__ constexpr uint32_t make_idesc_nv(int n) {
  return (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24);
}
__device__ __forceinline__ void tc_mma_nv(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t sfa, uint32_t sfb, uint32_t accumulate) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
               "tcgen05.mma.cta_group::1.kind::mxf4nvf4.block_scale.block16 [%0], %1, %2, %3, [%5], [%6], p;\n\t}"
               ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(sfa), "r"(sfb) : "memory");
}
__device__ __forceinline__ float e4m3_decode(uint32_t code) {
  uint32_t h2;
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"((uint16_t)code));
  return __half2float(__ushort_as_half((unsigned short)(h2 & 0xFFFFu)));
}

template <bool kPnq, bool kOutF32>
__global__ void __launch_bounds__(kThreads, 1) attention_nvfp4_kernel(const Params p, const __grid_constant__ CUtensorMap out_map) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar0 = sbase + kOffBar;
  auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kOffMisc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kOffMisc + 8);

  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const int T = p.kv_tiles;
  const TileOfCta at((int)blockIdx.x, p.pair_ctas, p.q_pairs, p.q_tiles);
  const int bh = at.bh, qtile0 = at.qtile;
  const bool two = at.two;                           // a second query tile: softmax group 1 has work

  if (tid == 0) {
    mbar_init(bar(BAR_Q), 1);
    for (int s = 0; s < kStages; ++s) { mbar_init(bar(BAR_KFULL + s), 1); mbar_init(bar(BAR_KEMPTY + s), 1); }
    mbar_init(bar(BAR_SFULL + 0), 1); mbar_init(bar(BAR_SFULL + 1), 1);
    mbar_init(bar(BAR_SFREE), 8);
    mbar_init(bar(BAR_PFULL + 0), 8); mbar_init(bar(BAR_PFULL + 1), 8);
    mbar_init(bar(BAR_ODONE + 0), 1); mbar_init(bar(BAR_ODONE + 1), 1);
    abort_flag[0] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // rows of ones appended to every V stage (E2M1 code 2 = 1.0) and their scale atom (E4M3 1.0 = 0x38)
  for (int i = tid; i < kStages * 16 * 64 / 16; i += kThreads) {
    const int s = i / 64, c = i % 64;
    reinterpret_cast<uint4*>(smem + kOffV + s * kVStageBytes + kTileCodeBytes)[c] =
        make_uint4(0x22222222u, 0x22222222u, 0x22222222u, 0x22222222u);
  }
  for (int i = tid; i < kTileScaleBytes / 16; i += kThreads)
    reinterpret_cast<uint4*>(smem + kOffSFOnes)[i] = make_uint4(0x38383838u, 0x38383838u, 0x38383838u, 0x38383838u);
  // what a softmax thread needs of a block's scale code (E4M3, never negative): the logarithm of the element multiplier, and
  // for the direct placement its inverse.  d = 0 keeps multiplier 1 (see below).
  if (tid < 128) {
    const float d = e4m3_decode((uint32_t)tid);
    reinterpret_cast<float2*>(smem + kOffTab)[tid] = (tid == 0 || tid == 127) ? make_float2(0.0f, 1.0f) : make_float2(log2f(2688.0f / d), d * kInvTensorRangeP);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == kSoftmaxWarps + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  pdl_wait();                                        // the operands and the status word are ready
  if (tid == 0) abort_flag[1] = *reinterpret_cast<volatile int*>(p.status);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_trigger();
  const uint32_t tmem = *tmem_slot;
  const int role = (abort_flag[1] != 0 || at.empty || (!two && warp >= 8 && warp < kSoftmaxWarps)) ? kSoftmaxWarps + 2 : warp;     // an earlier CTA gave up: drain the grid quickly

  // Waits of the single-thread roles.  Loops out of line keep their code short, but the call's register conventions reach the
  // softmax warps: with the direct row sum that is worth it (37 x 16384: 3492 us against 3665), with the PNQ row sum it makes
  // short key sequences slower (12 x 9000 x 100: 43.2 us against 41.5) and long ones no faster.
  auto role_wait = [&](uint32_t b, uint32_t parity, volatile int* flag, int* status, int code) {
    return kPnq ? mbar_wait(b, parity, flag, status, code) : mbar_wait1(b, parity, flag, status, code);
  };

  if (role == kSoftmaxWarps) {
    // =============================== producer ===============================================
    if (lane == 0) {
      const int64_t qt0 = (int64_t)bh * p.q_tiles + qtile0;
      mbar_expect_tx(bar(BAR_Q), (two ? 2 : 1) * (kTileCodeBytes + kSF));
      for (int i = 0; i < (two ? 2 : 1); ++i) {
        bulk_g2s(sbase + kOffQ + i * kTileCodeBytes, p.q_codes + (qt0 + i) * kTileCodeBytes, kTileCodeBytes, bar(BAR_Q));
        bulk_g2s(sbase + kOffSFQ + i * kSF, p.q_scales + (qt0 + i) * kSF, kSF, bar(BAR_Q));
      }
      const int64_t kv0 = (int64_t)bh * T;
      bool ok = true;
      int j = 0;
      for (; j < T && ok; ++j) {
        const int s = j % kStages;
        if (j >= kStages) ok = role_wait(bar(BAR_KEMPTY + s), (uint32_t)(((j / kStages) & 1) ^ 1), abort_flag, p.status, 11);
        if (!ok) break;
        mbar_expect_tx(bar(BAR_KFULL + s), 2 * (kTileCodeBytes + kSF));
        bulk_g2s(sbase + kOffK + s * kTileCodeBytes, p.k_codes + (kv0 + j) * kTileCodeBytes, kTileCodeBytes, bar(BAR_KFULL + s));
        bulk_g2s(sbase + kOffSFK + s * kSF, p.k_scales + (kv0 + j) * kSF, kSF, bar(BAR_KFULL + s));
        bulk_g2s(sbase + kOffV + s * kVStageBytes, p.v_codes + (kv0 + j) * kTileCodeBytes, kTileCodeBytes, bar(BAR_KFULL + s));
        bulk_g2s(sbase + kOffSFV + s * kSF, p.v_scales + (kv0 + j) * kSF, kSF, bar(BAR_KFULL + s));
      }
      if (!ok || *abort_flag) {                        // gave up: let copies in flight land before shared memory is released
        const long long t0 = clock64();
        for (int f = (j > kStages ? j - kStages : 0); f < j; ++f)
          while (!mbar_try(bar(BAR_KFULL + f % kStages), (uint32_t)((f / kStages) & 1)) && clock64() - t0 < 200000000LL) {}
        while (!mbar_try(bar(BAR_Q), 0u) && clock64() - t0 < 200000000LL) {}
      }
    }
  } else if (role == kSoftmaxWarps + 1) {
    // =============================== MMA issuer =============================================
    if (lane == 0) {
      bool ok = role_wait(bar(BAR_Q), 0, abort_flag, p.status, 21);
      uint32_t sfree_n = 0;
      constexpr uint32_t kDescHiTile = (512u >> 4) | (1u << 14) | (4u << 29);   // 64-byte swizzle, K-major
      const uint32_t q_lo = (sbase + kOffQ) >> 4, k_lo = (sbase + kOffK) >> 4;
      const uint32_t v_lo = (sbase + kOffV) >> 4, p_lo = (sbase + kOffP) >> 4;
      auto desc = [](uint32_t lo) { return ((uint64_t)kDescHiTile << 32) | lo; };
      auto gemm1 = [&](int t, int j) {                 // S = Q_t K_j^T
        const uint32_t a = q_lo + (uint32_t)t * (kTileCodeBytes >> 4);
        const uint32_t b = k_lo + (uint32_t)(j % kStages) * (kTileCodeBytes >> 4);
        const uint32_t sfa = tmem + kColSFQ + 8 * t, sfb = tmem + kColSFK + 8 * (j & 1);
        tc_mma_nv(tmem + kColS, desc(a), desc(b), make_idesc_nv(128), sfa, sfb, 0u);
        tc_mma_nv(tmem + kColS, desc(a + 2), desc(b + 2), make_idesc_nv(128), sfa + 4, sfb + 4, 1u);
        tc_commit(bar(BAR_SFULL + t));
      };
      auto gemm2 = [&](int t, int j) {                 // O_t += P_t [V_j | 1]
        tc_cp_sf(tmem + kColSFP + 8 * t, sbase + kOffSFP + t * kSF);
        tc_cp_sf(tmem + kColSFP + 8 * t + 4, sbase + kOffSFP + t * kSF + kTileScaleBytes);
        const uint32_t a = p_lo + (uint32_t)t * (kTileCodeBytes >> 4);
        const uint32_t b = v_lo + (uint32_t)(j % kStages) * (kVStageBytes >> 4);
        const uint32_t d = tmem + (t ? kColO1 : kColO0);
        const uint32_t sfa = tmem + kColSFP + 8 * t, sfb = tmem + kColSFV + 16 * (j & 1);
        tc_mma_nv(d, desc(a), desc(b), make_idesc_nv(kNV), sfa, sfb, j > 0 ? 1u : 0u);
        tc_mma_nv(d, desc(a + 2), desc(b + 2), make_idesc_nv(kNV), sfa + 4, sfb + 8, 1u);
        tc_commit(bar(BAR_ODONE + t));
      };
      auto wait_sfree = [&]() {
        const bool r = role_wait(bar(BAR_SFREE), sfree_n & 1u, abort_flag, p.status, 23);
        ++sfree_n;
        tc_fence_after();
        return r;
      };
      // K of tile j has landed: its scale atoms go to tensor memory (slot j & 1 was last read by the score products of tile
      // j - 2, issued before), apart from the wait for the score buffer, so that nothing but that wait stands between "the
      // other group has taken its scores" and the next score product.  V's atoms (same stage) follow behind the products.
      auto k_ready = [&](int j) {
        const int s = j % kStages;
        if (!role_wait(bar(BAR_KFULL + s), (uint32_t)((j / kStages) & 1), abort_flag, p.status, 22)) return false;
        tc_fence_after();
        tc_cp_sf(tmem + kColSFK + 8 * (j & 1), sbase + kOffSFK + s * kSF);
        tc_cp_sf(tmem + kColSFK + 8 * (j & 1) + 4, sbase + kOffSFK + s * kSF + kTileScaleBytes);
        return true;
      };
      auto v_scales = [&](int j) {
        tc_cp_sf(tmem + kColSFV + 16 * (j & 1), sbase + kOffSFV + (j % kStages) * kSF);
        tc_cp_sf(tmem + kColSFV + 16 * (j & 1) + 8, sbase + kOffSFV + (j % kStages) * kSF + kTileScaleBytes);
      };
      if (ok) {
        tc_fence_after();
        for (int t = 0; t < (two ? 2 : 1); ++t) {
          tc_cp_sf(tmem + kColSFQ + 8 * t, sbase + kOffSFQ + t * kSF);
          tc_cp_sf(tmem + kColSFQ + 8 * t + 4, sbase + kOffSFQ + t * kSF + kTileScaleBytes);
        }
        for (int slot = 0; slot < 2; ++slot) {           // scales of the ones rows, both slots and both K halves
          tc_cp_sf(tmem + kColSFV + 16 * slot + 4, sbase + kOffSFOnes);
          tc_cp_sf(tmem + kColSFV + 16 * slot + 12, sbase + kOffSFOnes);
        }
      }
      ok = ok && k_ready(0);
      if (ok) { v_scales(0); gemm1(0, 0); }
      for (int j = 0; !two && j < T && ok; ++j) {      // one query tile: its next scores go ahead of the output product
        if (j + 1 < T) {
          ok = k_ready(j + 1) && wait_sfree();
          if (!ok) break;
          gemm1(0, j + 1);
          v_scales(j + 1);
        }
        ok = role_wait(bar(BAR_PFULL + 0), (uint32_t)(j & 1), abort_flag, p.status, 24);
        if (!ok) break;
        tc_fence_after();
        gemm2(0, j);
        tc_commit(bar(BAR_KEMPTY + j % kStages));
      }
      if (two) {
        // the issue order of forward.cu: G2(0,j) G1(1,j+1) G2(1,j) G1(0,j+2)
        ok = ok && wait_sfree();
        if (ok) gemm1(1, 0);
        if (T > 1) {
          ok = ok && k_ready(1);
          if (ok) v_scales(1);
          ok = ok && wait_sfree();
          if (ok) gemm1(0, 1);
        }
#pragma unroll 2
        for (int j = 0; j < T && ok; ++j) {
          ok = role_wait(bar(BAR_PFULL + 0), (uint32_t)(j & 1), abort_flag, p.status, 24);
          if (!ok) break;
          tc_fence_after();
          gemm2(0, j);
          if (j + 1 < T) {
            ok = wait_sfree();
            if (!ok) break;
            gemm1(1, j + 1);
          }
          if (j + 2 < T) {                             // off the critical chain: the thread would wait for P here anyway
            ok = k_ready(j + 2);
            if (!ok) break;
          }
          ok = role_wait(bar(BAR_PFULL + 1), (uint32_t)(j & 1), abort_flag, p.status, 26);
          if (!ok) break;
          tc_fence_after();
          gemm2(1, j);
          if (j + 2 < T) {
            ok = wait_sfree();
            if (!ok) break;
            gemm1(0, j + 2);
          }
          tc_commit(bar(BAR_KEMPTY + j % kStages));
          if (j + 2 < T) v_scales(j + 2);
        }
      }
    }
  } else if (role < kSoftmaxWarps) {
    // =============================== softmax groups =========================================
    const int t = warp >> 3;
    const int h = (warp >> 2) & 1;
    const int row = (warp & 3) * 32 + lane;
    const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t t_s = tmem + kColS + lane_addr + kCols * h;
    const uint32_t t_o = tmem + (t ? kColO1 : kColO0) + lane_addr;
    // S_raw carries neither tensor scale: both go into the exponent's multiplier
    const float c = p.scale_log2e * p.ts_q[bh] * p.ts_k[bh];
    float m_run = -INFINITY, l_run = 0.0f;
    const uint32_t aP0 = sbase + kOffP + t * kTileCodeBytes + tile_code_offset(row, 2 * h);
    const uint32_t aP1 = sbase + kOffP + t * kTileCodeBytes + tile_code_offset(row, 2 * h + 1);
    const uint32_t aSF = sbase + kOffSFP + t * kSF + h * kTileScaleBytes + tile_scale_offset(row, 0);   // atom h: this thread's 4 blocks
    const uint32_t aMaxOwn = sbase + kOffMax + (t * 256 + h * 128 + row) * 4;
    const uint32_t aMaxPartner = sbase + kOffMax + (t * 256 + (h ^ 1) * 128 + row) * 4;
    const uint32_t aTab = sbase + kOffTab;
    const int pair_bar = 1 + (warp & 3) + 4 * t;
    volatile int* const own_limit_only = abort_flag + 1;
    bool ok = true;
    int j = 0;
    for (; j < T; ++j) {
      ok = __all_sync(0xFFFFFFFFu, mbar_wait(bar(BAR_SFULL + t), (uint32_t)(j & 1), own_limit_only, p.status, 31, kWaitLimitCycles, abort_flag));
      if (!ok) break;
      tc_fence_after();
      uint32_t sr[kCols];
      TMEM_LD64(t_s, sr);
      tmem_ld_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(BAR_SFREE));
      if (j == T - 1) {
        const int valid = (int)(p.Nkv - (int64_t)j * kTile) - kCols * h;
#pragma unroll
        for (int i = 0; i < kCols; ++i)
          if (i >= valid) sr[i] = 0xFF800000u;
      }
      float bmax[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        float q2[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const uint32_t* v = sr + 16 * b + 8 * u;
          float mx = max3(__uint_as_float(v[0]), __uint_as_float(v[1]), __uint_as_float(v[2]));
          mx = max3(mx, __uint_as_float(v[3]), __uint_as_float(v[4]));
          mx = max3(mx, __uint_as_float(v[5]), __uint_as_float(v[6]));
          q2[u] = fmaxf(mx, __uint_as_float(v[7]));
        }
        bmax[b] = fmaxf(q2[0], q2[1]);
      }
      const float own_max = fmaxf(fmaxf(bmax[0], bmax[1]), fmaxf(bmax[2], bmax[3]));
      const uint32_t par = (uint32_t)(j & 1) * 2048u;
      sts32f(aMaxOwn + par, own_max);
      asm volatile("bar.sync %0, 64;" ::"r"(pair_bar) : "memory");
      const float partner_max = lds32f(aMaxPartner + par);
      const bool o_ready = (j == 0) || mbar_test(bar(BAR_ODONE + t), (uint32_t)((j - 1) & 1));
      const float m_new = max3(m_run, own_max, partner_max);
      const bool moved = (m_new != m_run) && (j > 0);
      const float m_old = m_run;
      m_run = m_new;
      const float nmc = -(m_new * c);
      if (!__all_sync(0xFFFFFFFFu, o_ready)) {
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(bar(BAR_ODONE + t), (uint32_t)((j - 1) & 1), own_limit_only, p.status, 32, kWaitLimitCycles, abort_flag));
        if (!ok) { ++j; break; }
      }
      tc_fence_after();
      const bool rescale = __any_sync(0xFFFFFFFFu, moved);
      float alpha = 1.0f;
      // Block scales: the block's largest probability by the elements' own expression, then the two-level recipe, two blocks
      // per conversion.  The element multiplier 2688 / d_b is folded into the exponent as its logarithm, which (like
      // d_b / 2688) comes from a table of the 127 codes: log2f of the rounded quotient, within a unit in the last place of the
      // logarithm plus the quotient's 9e-8.  (Computed per block -- decode, lg2.approx on the mantissa, two additions and the selections for
      // subnormal and zero codes -- it was 22 instructions per block instead of 8.)  A block whose scale rounds to zero
      // keeps multiplier 1: its probabilities are below 2.2e-6 and round to code 0 either way, and the direct placement
      // still sums them.
      float nb[4], inv_r[4];
      uint32_t sf4 = 0;
#pragma unroll
      for (int b = 0; b < 4; b += 2) {
        const float y0 = __fmul_rn(__fmul_rn(ex2(fmaf(bmax[b], c, nmc)), kTensorRangeP), kOneSixth);
        const float y1 = __fmul_rn(__fmul_rn(ex2(fmaf(bmax[b + 1], c, nmc)), kTensorRangeP), kOneSixth);
        uint16_t code2;
        asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(code2) : "f"(y1), "f"(y0));
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          float lr;
          asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(lr), "=f"(inv_r[b + u]) : "r"(aTab + ((u ? (uint32_t)code2 >> 8 : (uint32_t)code2 & 0xFFu) << 3)));
          nb[b + u] = fmaf(-m_new, c, lr);         // one rounding: -(m_new c) + log2(2688 / d)
        }
        sf4 |= (uint32_t)code2 << (8 * b);
      }
      asm volatile("st.shared.b32 [%0], %1;" ::"r"(aSF), "r"(sf4) : "memory");
      float l_tile = 0.0f;
      const uint64_t cc2 = dup2(c);
      auto tile_body = [&](auto resc_tag) {
        constexpr bool kResc = decltype(resc_tag)::value;
        if (kResc) alpha = ex2((m_old - m_new) * c);
        const uint64_t al2 = dup2(alpha);
#pragma unroll
        for (int b32 = 0; b32 < 2; ++b32) {           // one 16-byte chunk of codes = 32 elements = two blocks
          uint4 w;
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            uint32_t oc[8];
            const uint32_t t_oc = t_o + kCols * h + 32 * b32 + 8 * g;
            if (kResc) TMEM_LD8(t_oc, oc);
            const uint64_t nb2 = dup2(nb[2 * b32 + (g >> 1)]);
            float x[8];
#pragma unroll
            for (int i = 0; i < 8; i += 2) {           // x = exp2(s * c + nb) = p~ * 2688 / d_b, two elements per multiply-add
              fma2(sr[32 * b32 + 8 * g + i], sr[32 * b32 + 8 * g + i + 1], cc2, nb2, x[i], x[i + 1]);
              x[i] = ex2(x[i]);
              x[i + 1] = ex2(x[i + 1]);
            }
            if (!kPnq) {
              float s0, s1;
              add2x2(x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7], s0, s1);
              l_tile = fmaf(s0 + s1, inv_r[2 * b32 + (g >> 1)], l_tile);
            }
            const uint32_t pk = pack_e2m1x8(x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7]);
            if (g == 0) w.x = pk; else if (g == 1) w.y = pk; else if (g == 2) w.z = pk; else w.w = pk;
            if (kResc) {
              tmem_ld_wait();
#pragma unroll
              for (int i = 0; i < 8; i += 2) mul2(oc[i], oc[i + 1], al2);
              TMEM_ST8(t_oc, oc);
            }
          }
          sts128(b32 == 0 ? aP0 : aP1, w);
        }
        if (kResc) {
          if (kPnq && h == 0) {                        // column 128: the running row sum of the quantized probabilities
            uint32_t lr;
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(lr) : "r"(t_o + 128) : "memory");
            tmem_ld_wait();
            lr = __float_as_uint(__uint_as_float(lr) * alpha);
            asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%1], {%0};" ::"r"(lr), "r"(t_o + 128) : "memory");
          }
          tmem_st_wait();
        }
      };
      if (rescale) tile_body(std::true_type{}); else tile_body(std::false_type{});
      if (!kPnq) l_run = fmaf(alpha, l_run, l_tile);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(BAR_PFULL + t));
    }
    if (!ok) pair_keep_company(pair_bar, T - j);

    // ---- epilogue ----
    if (ok) ok = __all_sync(0xFFFFFFFFu, mbar_wait(bar(BAR_ODONE + t), (uint32_t)((T - 1) & 1), own_limit_only, p.status, 33, kWaitLimitCycles, abort_flag));
    float l = l_run;
    if (!kPnq) {
      const uint32_t par = (uint32_t)(T & 1) * 2048u;
      sts32f(aMaxOwn + par, l_run);
      asm volatile("bar.sync %0, 64;" ::"r"(pair_bar) : "memory");
      l = l_run + lds32f(aMaxPartner + par);
    }
    if (ok) {
      tc_fence_after();
      float o_scale = p.ts_v[bh];                      // O = O_raw s_T(V) s_T(P) / l; under PNQ l = l_raw s_T(P)
      if (kPnq) {
        uint32_t lr;
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(lr) : "r"(t_o + 128) : "memory");
        tmem_ld_wait();
        l = __uint_as_float(lr);
      } else {
        o_scale *= __fdiv_rn(1.0f, kTensorRangeP);
      }
      const float inv_l = o_scale / l;
      // coordinates computed afresh: with those of the loop the kernel took 760 us instead of 715 at 24 x 8192 (registers)
      const uint32_t tid2 = fresh_tid(), w = tid2 >> 5;
      const TileOfCta at2((int)blockIdx.x, p.pair_ctas, p.q_pairs, p.q_tiles);
      const int row0 = (at2.qtile + (int)(w >> 3)) * kTile + (int)(w & 3) * 32, col = kCols * ((w >> 2) & 1);
      store_half_rows<kOutF32>((w >> 3 ? kColO1 : kColO0) + ((w & 3) << 21) + col, ((smem_u32(smem_raw) + 1023u) & ~1023u) + kOffOut + w * kOutBoxBytes,
                               (int)(tid2 & 31), inv_l, &out_map, col, row0, at2.bh, row0 < p.Nq);
    }
  }

  if (warp < kSoftmaxWarps && lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");     // the output copies have left shared memory
  tc_fence_before();
  __syncthreads();
  if (warp == kSoftmaxWarps + 1) {
    tc_fence_after();
    check_tmem_base(*tmem_slot, lane, p.status);
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}

struct Layout { size_t status, amax, tscale, q_codes, q_scales, k_codes, k_scales, v_codes, v_scales, total; };

static inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

static bool carve(int B, int H, int64_t Nq, int64_t Nkv, Layout* w) {
  if (B <= 0 || H <= 0 || Nq <= 0 || Nkv <= 0) return false;
  const size_t bh = (size_t)B * H;
  const size_t qt = (size_t)((Nq + kTile - 1) / kTile), kt = (size_t)((Nkv + kTile - 1) / kTile);
  size_t off = 0;
  w->status = off;   off += 256;
  w->amax = off;     off += align_up(3 * bh * sizeof(float), 256);
  w->tscale = off;   off += align_up(3 * bh * sizeof(float), 256);
  w->q_codes = off;  off += align_up(bh * qt * kTileCodeBytes, 256);
  w->q_scales = off; off += align_up(bh * qt * kSF, 256);
  w->k_codes = off;  off += align_up(bh * kt * kTileCodeBytes, 256);
  w->k_scales = off; off += align_up(bh * kt * kSF, 256);
  w->v_codes = off;  off += align_up(bh * kt * kTileCodeBytes, 256);
  w->v_scales = off; off += align_up(bh * kt * kSF, 256);
  w->total = off;
  return true;
}

}  // namespace fwdnv

size_t nvfp4_workspace_bytes(int B, int H, int64_t Nq, int64_t Nkv) {
  fwdnv::Layout w;
  return fwdnv::carve(B, H, Nq, Nkv, &w) ? w.total : 0;
}

int launch_forward_nvfp4(const void* q, const void* k, const void* v, void* o, int B, int H, int64_t Nq, int64_t Nkv,
                         float softmax_scale, unsigned flags, void* workspace, size_t workspace_bytes, cudaStream_t stream) {
  using namespace fwdnv;
  Layout w;
  if (!carve(B, H, Nq, Nkv, &w)) return MXATTN_EINVAL;
  if (workspace_bytes < w.total) return MXATTN_EWORKSPACE;
  const int64_t bh = (int64_t)B * H;
  const int64_t qt = (Nq + kTile - 1) / kTile, kt = (Nkv + kTile - 1) / kTile;
  const int64_t pairs = (qt + 1) / 2, grid = bh * pairs;
  if (qt > 0x3FFFFFFF || kt > 0x3FFFFFFF || grid > 0x7FFFFFFF) return MXATTN_EUNSUPPORTED;
  const int n_sm = sm_count();
  if (n_sm == 0) return MXATTN_ECUDA;
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  float* amax = reinterpret_cast<float*>(ws + w.amax);
  float* ts = reinterpret_cast<float*>(ws + w.tscale);
  if (launch_zero(reinterpret_cast<uint32_t*>(ws + w.status), (int64_t)(w.tscale - w.status) / 4, stream) != MXATTN_OK) return MXATTN_ECUDA;      // status word and tensor maxima
  const int rc = launch_nvfp4_operands(q, ws + w.q_codes, ws + w.q_scales, k, ws + w.k_codes, ws + w.k_scales, v, ws + w.v_codes, ws + w.v_scales,
                                       amax, ts, bh, Nq, Nkv, stream);
  if (rc != MXATTN_OK) return rc;
  Params p;
  p.q_codes = ws + w.q_codes; p.q_scales = ws + w.q_scales; p.k_codes = ws + w.k_codes; p.k_scales = ws + w.k_scales;
  p.v_codes = ws + w.v_codes; p.v_scales = ws + w.v_scales;
  p.ts_q = ts; p.ts_k = ts + bh; p.ts_v = ts + 2 * bh;
  p.status = reinterpret_cast<int*>(ws + w.status);
  p.Nq = Nq; p.Nkv = Nkv; p.q_tiles = (int)qt; p.kv_tiles = (int)kt; p.q_pairs = (int)pairs;
  const TileSplit split(grid, n_sm);
  p.pair_ctas = (int)split.pair_ctas;
  p.scale_log2e = softmax_scale * 1.4426950408889634f;
  const bool pnq = flags & MXATTN_FLAG_PNQ, f32 = flags & MXATTN_FLAG_OUT_FP32;
  CUtensorMap out_map;
  const int map_rc = encode_output_map(&out_map, o, bh, Nq, f32);
  if (map_rc != MXATTN_OK) return map_rc;
  void (*kern)(const Params, const CUtensorMap) = pnq ? (f32 ? attention_nvfp4_kernel<true, true> : attention_nvfp4_kernel<true, false>)
                                   : (f32 ? attention_nvfp4_kernel<false, true> : attention_nvfp4_kernel<false, false>);
  if (!ensure_dynamic_smem((const void*)kern, kSmemBytes)) return MXATTN_ECUDA;
  return launch_pdl(kern, dim3((unsigned)split.ctas), kThreads, kSmemBytes, stream, p, out_map) == cudaSuccess ? MXATTN_OK : MXATTN_ECUDA;
}

}  // namespace mxattn
