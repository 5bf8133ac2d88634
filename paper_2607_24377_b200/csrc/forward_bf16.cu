// bf16 variant of the fused attention forward: the online-softmax recurrence (paper Section 2, the FlashAttention-2 form:
// Eq. 2-3) with NO quantization: Q, K, V stay bf16, the exponentials are rounded to bf16 for the second GEMM, and the row
// sum is taken from the fp32 exponentials.  It is the "high precision" reference point the MXFP4 variants are reported
// against (paper Section 5.2, "FP16" baseline; bf16 here).
//
//   GEMM 1  S_t  = Q_t K_j^T         tcgen05.mma kind::f16, M=128, N=128, 8 instructions of K=16, operands in shared memory
//   GEMM 2  O_t += P_t V_j           A = P_t from tensor memory, B = V_j as it lies in memory (token-major, "MN-major" operand)
//
// One CTA = two query tiles of 128 rows of one head (or one, see below); the roles are those of forward.cu (16 softmax
// warps in two groups, a producer, an MMA issuer).  Q, K and V tiles are fetched straight from the [B H][N][128] tensors by tensor copies with the
// 128-byte swizzle (two 64-channel halves of 16 KiB per tile; rows beyond the sequence arrive as zeros), so there is no
// re-tiling pass over the inputs.
//
// What bounds it: the tensor cores, and the shared memory that feeds them.  Per 256 x 128 tile the four products take 2048
// cycles at the dense bf16 rate, and their operands 2 x 64 KiB (GEMM 1) + 2 x 32 KiB (GEMM 2) of shared-memory reads plus
// 64 KiB of fills, 2048 cycles at 128 B per clock.  P therefore goes through tensor memory: in shared memory, writing it and
// reading it back costs another 1024 cycles.  Tensor memory: P_0 [0,64), S [64,192) shared by both groups, P_1 [192,256),
// O_0, O_1 [256,512).  (A score buffer per group that P overwrites in place leaves the next scores behind the output
// product: 1385 cycles from P to the next scores, 8 % slower.)
// Measured (B200): H=24, N=8192 970 -> 755 us, H=40, N=16384 5.40 -> 4.5 ms; the former version re-tiled its inputs
// (60 us), kept P in shared memory and issued its 32 multiplies per tile from a single thread, which had to move every
// descriptor word to a uniform register in front of each of them (966 -> 800 us by the converged issuer alone).
// The output leaves as tensor copies (store_half_rows) from the query tiles' own shared memory: 69.8 -> 65.6 us at
// H=40, 4096 x 512 (fp32 84.3 -> 71.9), 123 -> 115 at H=24, 8192 x 1024.
// The issuer waits for the softmax groups at named barriers, which no memory queue delays (an mbarrier arrival waits behind the exponentials):
// 24 x 2000 71.3 -> 64.1 us, 40 x 16384 4727 -> 4608, 24 x 8192 673 -> 668, 2 x 1024 15.6 -> 15.1.  It looks at the abort flag before; the
// softmax warps come to every tile's, also when their own waits run out.
// A last wave that would leave half of the SMs idle runs with one query tile per CTA (common.cuh): 755 -> 646 us at
// H=24, N=8192 (5.19 waves), 25 -> 19 us at 2 heads of 1024.  (All figures in series of a few calls at full clock; under the power
// limit the same 24 x 8192 takes 674 us in the mean of 20 calls back to back, 706 to 721 of some hundred, 787 of 2000.)
#include <string.h>

#include <type_traits>

#include "common.cuh"
#include "tc_helpers.cuh"

namespace mxattn {
namespace fwd16 {

using namespace fwd;

constexpr int kThreads = 576;
constexpr int kSoftmaxWarps = 16;
constexpr int kStages = 4;                                 // one ring for K and V tiles, in the order K0 V0 K1 V1 ...
constexpr int kTileBytes = 32768;                          // 128 x 128 bf16: two halves of 64 channels
constexpr int kHalfBytes = 16384;                          // 128 rows x 128 bytes, 128-byte swizzle

constexpr int kOffQ = 0;                                   // 2 tiles
constexpr int kOffKV = kOffQ + 2 * kTileBytes;
constexpr int kOffMax = kOffKV + kStages * kTileBytes;     // half-row exchange: [parity 2][tile 2][half 2][128] floats
constexpr int kOffBar = kOffMax + 2 * 2 * 2 * 128 * 4;
enum Bar { BAR_Q = 0, BAR_FULL = 1, BAR_EMPTY = BAR_FULL + kStages, BAR_SFULL = BAR_EMPTY + kStages, BAR_ODONE = BAR_SFULL + 2, kNumBars = BAR_ODONE + 2 };
constexpr int kOffMisc = kOffBar + kNumBars * 8;           // tmem slot, abort flag, "an earlier CTA gave up"
constexpr int kSmemBytes = kOffMisc + 32 + 1024;           // + slack for the 1024 alignment
static_assert(kSmemBytes <= 232448, "shared memory budget");

constexpr int kBarFree = 9, kBarP = 11;                    // named barriers: group t has read its scores, P_t is in place
constexpr uint32_t kColP = 0, kColS = 64, kColO = 256;      // P_t at 192 t (64 columns), S between them, O_t at 256 + 128 t

__device__ __forceinline__ void tc_mma_ss(uint32_t leader, uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"
               "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
               ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(leader) : "memory");
}
__device__ __forceinline__ void tc_mma_ts(uint32_t leader, uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"
               "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
               ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(leader) : "memory");
}
__device__ __forceinline__ void tensor_g2s(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
  asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
               ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar) : "memory");
}

struct Params {
  int* status;
  int64_t Nq, Nkv;
  int q_tiles_n, kv_tiles, q_pairs;
  int pair_ctas;        // CTAs before this one take two query tiles, the others one (TileSplit)
  float scale_log2e;
};

// ---------------------------------------------------------------------------------------------
template <bool kOutF32>
__global__ void __launch_bounds__(kThreads, 1) attention_bf16_kernel(const Params p, const __grid_constant__ CUtensorMap q_map,
                                                                     const __grid_constant__ CUtensorMap k_map,
                                                                     const __grid_constant__ CUtensorMap v_map,
                                                                     const __grid_constant__ CUtensorMap out_map) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar0 = sbase + kOffBar;
  auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kOffMisc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kOffMisc + 8);

  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const uint32_t abort_addr = bar0 + (kOffMisc + 8 - kOffBar);
  const TileOfCta at((int)blockIdx.x, p.pair_ctas, p.q_pairs, p.q_tiles_n);
  const int bh = at.bh, qtile0 = at.qtile;
  const bool two = at.two;                           // a second query tile: softmax group 1 has work
  const int T = p.kv_tiles;

  if (tid == 0) {
    mbar_init(bar(BAR_Q), 1);
    for (int s = 0; s < kStages; ++s) { mbar_init(bar(BAR_FULL + s), 1); mbar_init(bar(BAR_EMPTY + s), 1); }
    for (int t = 0; t < 2; ++t) { mbar_init(bar(BAR_SFULL + t), 1); mbar_init(bar(BAR_ODONE + t), 1); }
    abort_flag[0] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kSoftmaxWarps + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  pdl_wait();
  if (tid == 0) abort_flag[1] = *reinterpret_cast<volatile int*>(p.status);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_trigger();
  constexpr uint32_t tmem = 0;
  if (*tmem_slot != 0) *abort_flag = kCodeTmemBase;
  const int role = (abort_flag[1] != 0 || *tmem_slot != 0 || at.empty || (!two && warp >= 8 && warp < kSoftmaxWarps)) ? kSoftmaxWarps + 2 : warp;     // an earlier CTA gave up: drain the grid quickly

  if (role == kSoftmaxWarps) {
    // =============================== producer ===============================================
    if (lane == 0) {
      auto fetch = [&](uint32_t dst, const CUtensorMap* map, int row, uint32_t b) {
        tensor_g2s(dst, map, 0, row, bh, b);
        tensor_g2s(dst + kHalfBytes, map, 64, row, bh, b);
      };
      mbar_expect_tx(bar(BAR_Q), (two ? 2 : 1) * kTileBytes);
      fetch(sbase + kOffQ, &q_map, qtile0 * kTile, bar(BAR_Q));
      if (two) fetch(sbase + kOffQ + kTileBytes, &q_map, (qtile0 + 1) * kTile, bar(BAR_Q));
      bool ok = true;
      int n = 0;
      for (; n < 2 * T; ++n) {                         // load n: K_j for n = 2 j, V_j for n = 2 j + 1
        const int s = n % kStages;
        if (n >= kStages) ok = mbar_wait1(bar(BAR_EMPTY + s), (uint32_t)((n / kStages) & 1) ^ 1u, abort_flag, p.status, 11);
        if (!ok) break;
        mbar_expect_tx(bar(BAR_FULL + s), kTileBytes);
        fetch(sbase + kOffKV + s * kTileBytes, (n & 1) ? &v_map : &k_map, (n >> 1) * kTile, bar(BAR_FULL + s));
      }
      if (!ok || *abort_flag) {                        // let copies in flight land before shared memory is released
        const long long t0 = clock64();
        for (int i = (n > kStages ? n - kStages : 0); i < n; ++i)
          while (!mbar_try(bar(BAR_FULL + i % kStages), (uint32_t)((i / kStages) & 1)) && clock64() - t0 < 400000000LL) {}
        while (!mbar_try(bar(BAR_Q), 0) && clock64() - t0 < 400000000LL) {}
      }
    }
  } else if (role == kSoftmaxWarps + 1) {
    // =============================== MMA issuer (converged warp) ============================
    const uint32_t leader = elect_one();
    constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);       // 8-row (8-token) groups 1024 B apart, 128-byte swizzle
    constexpr uint32_t kIdescBase = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);  // f32 accum, bf16 x bf16, N=128, M=128
    constexpr uint32_t kIdescV = kIdescBase | (1u << 16);                      // B is MN-major (channels contiguous)
    const uint32_t q_lo = (sbase + kOffQ) >> 4, kv_lo = (sbase + kOffKV) >> 4;
    auto landed = [&](int n) {
      const bool r = mbar_wait_warp(bar(BAR_FULL + n % kStages), (uint32_t)((n / kStages) & 1), abort_flag, p.status, 22);
      tc_fence_after();
      return r;
    };
    auto gemm1 = [&](int t, int j) {                   // S_t = Q_t K_j^T; K = 16 channels per instruction: 4 steps of 32 bytes per half
      const uint32_t a = q_lo + (uint32_t)t * (kTileBytes >> 4), b = kv_lo + (uint32_t)(2 * j % kStages) * (kTileBytes >> 4);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const uint32_t off = (uint32_t)(k >> 2) * (kHalfBytes >> 4) + (uint32_t)(k & 3) * 2;
        tc_mma_ss(leader, tmem + kColS, ((uint64_t)kDescHi << 32) | (a + off), ((uint64_t)kDescHi << 32) | (b + off), kIdescBase, k > 0 ? 1u : 0u);
      }
      tc_commit_if(leader, bar(BAR_SFULL + t));
      if (t == 1 || !two) tc_commit_if(leader, bar(BAR_EMPTY + 2 * j % kStages));      // K_j: both groups' products are issued
    };
    auto gemm2 = [&](int t, int j) {                   // O_t += P_t V_j; K = 16 tokens per instruction: 8 columns of P, 2048 bytes of V
      const uint32_t b = kv_lo + (uint32_t)((2 * j + 1) % kStages) * (kTileBytes >> 4);
#pragma unroll
      for (int k = 0; k < 8; ++k)                      // leading-dimension offset: the other 64 channels, 16 KiB on
        tc_mma_ts(leader, tmem + kColO + 128 * t, tmem + kColP + 192 * t + 8 * k,
                  ((uint64_t)kDescHi << 32) | ((uint64_t)(kHalfBytes >> 4) << 16) | (b + (uint32_t)k * 128), kIdescV, (j > 0 || k > 0) ? 1u : 0u);
      tc_commit_if(leader, bar(BAR_ODONE + t));
      if (t == 1 || !two) tc_commit_if(leader, bar(BAR_EMPTY + (2 * j + 1) % kStages));
    };
    auto join = [&](int id) {                          // the eight warps of a softmax group
      if (__any_sync(0xFFFFFFFFu, lds_volatile(abort_addr) != 0)) return false;
      asm volatile("bar.sync %0, 288;" ::"r"(id) : "memory");
      tc_fence_after();
      return true;
    };
    auto wait_p = [&](int t) { return join(kBarP + t); };
    bool ok = mbar_wait_warp(bar(BAR_Q), 0, abort_flag, p.status, 21);
    // the issue order of forward.cu: G2(0,j) G1(1,j+1) G2(1,j) G1(0,j+2), which keeps the two groups half a tile apart
    auto wait_sfree = [&](int t) { return join(kBarFree + t); };      // group t has taken its scores
    ok = ok && landed(0);
    if (ok) gemm1(0, 0);
    for (int j = 0; !two && j < T && ok; ++j) {        // one query tile: its next scores go ahead of the output product
      if (j + 1 < T) {
        ok = landed(2 * j + 2) && wait_sfree(0);
        if (!ok) break;
        gemm1(0, j + 1);
      }
      ok = landed(2 * j + 1) && wait_p(0);
      if (ok) gemm2(0, j);
    }
    if (two) {
      ok = ok && wait_sfree(0);
      if (ok) gemm1(1, 0);
      if (T > 1) {
        ok = ok && landed(2) && wait_sfree(1);
        if (ok) gemm1(0, 1);
      }
      for (int j = 0; j < T && ok; ++j) {
        ok = landed(2 * j + 1) && wait_p(0);
        if (!ok) break;
        gemm2(0, j);
        if (j + 1 < T) {
          ok = wait_sfree(0);
          if (!ok) break;
          gemm1(1, j + 1);
        }
        if (j + 2 < T) ok = landed(2 * j + 4);
        ok = ok && wait_p(1);
        if (!ok) break;
        gemm2(1, j);
        if (j + 2 < T) {
          ok = wait_sfree(1);
          if (!ok) break;
          gemm1(0, j + 2);
        }
      }
    }
  } else if (role < kSoftmaxWarps) {
    // =============================== softmax groups =========================================
    // Two threads per query row (64 key columns each).  Their waits never leave the loop early (mbar_wait_soft), so that the
    // two warps of a pair, which meet at a named barrier in every tile, keep all their meetings.
    const int t = warp >> 3;
    const int h = (warp >> 2) & 1;
    const int row = (warp & 3) * 32 + lane;
    const uint32_t t_row = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t t_s = t_row + kColS + 64 * h;
    const uint32_t t_p = t_row + kColP + 192 * t + 32 * h;             // P: two bf16 per column, this thread's 64 keys in 32 columns
    const uint32_t t_o = t_row + kColO + 128 * t + 64 * h;             // this thread's 64 output channels
    const float c = p.scale_log2e;
    float m_run = -INFINITY, l_run = 0.0f;
    const uint32_t aMaxOwn = sbase + kOffMax + (t * 256 + h * 128 + row) * 4;
    const uint32_t aMaxPartner = sbase + kOffMax + (t * 256 + (h ^ 1) * 128 + row) * 4;
    const int pair_bar = 1 + (warp & 3) + 4 * t;

    for (int j = 0; j < T; ++j) {
      mbar_wait_soft<31>(bar(BAR_SFULL + t), (uint32_t)(j & 1), abort_addr);
      tc_fence_after();
      uint32_t sr[64];
      TMEM_LD64(t_s, sr);
      tmem_ld_wait();
      tc_fence_before();
      __syncwarp();
      asm volatile("bar.arrive %0, 288;" ::"r"(kBarFree + t) : "memory");
      if (j == T - 1) {
        const int valid = (int)(p.Nkv - (int64_t)j * kTile) - 64 * h;
#pragma unroll
        for (int i = 0; i < 64; ++i)
          if (i >= valid) sr[i] = 0xFF800000u;
      }
      float q8[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const uint32_t* v = sr + 8 * u;
        float mx = max3(__uint_as_float(v[0]), __uint_as_float(v[1]), __uint_as_float(v[2]));
        mx = max3(mx, __uint_as_float(v[3]), __uint_as_float(v[4]));
        mx = max3(mx, __uint_as_float(v[5]), __uint_as_float(v[6]));
        q8[u] = fmaxf(mx, __uint_as_float(v[7]));
      }
      const float hmax = fmaxf(max3(q8[0], q8[1], q8[2]), max3(max3(q8[3], q8[4], q8[5]), q8[6], q8[7]));
      const uint32_t par = (uint32_t)(j & 1) * 2048u;
      sts32f(aMaxOwn + par, hmax);
      asm volatile("bar.sync %0, 64;" ::"r"(pair_bar) : "memory");
      const float m_old = m_run;
      const float m_new = max3(m_old, hmax, lds32f(aMaxPartner + par));
      m_run = m_new;
      const bool rescale = __any_sync(0xFFFFFFFFu, (m_new != m_old) && (j > 0));
      if (j > 0) mbar_wait_soft<32>(bar(BAR_ODONE + t), (uint32_t)((j - 1) & 1), abort_addr);   // P has been read, O updated
      tc_fence_after();
      float alpha = 1.0f;
      float l_tile = 0.0f;
      const uint64_t cc2 = dup2(c), nm2 = dup2(-(m_new * c));
      auto tile_body = [&](auto resc_tag) {
        constexpr bool kResc = decltype(resc_tag)::value;
        if (kResc) alpha = ex2((m_old - m_new) * c);
        const uint64_t al2 = dup2(alpha);
#pragma unroll
        for (int g = 0; g < 8; ++g) {                  // 8 keys per step = 4 columns of P; 8 accumulator columns
          uint32_t oc[8];
          if (kResc) TMEM_LD8(t_o + 8 * g, oc);
          float x[8];
#pragma unroll
          for (int i = 0; i < 8; i += 2) {
            fma2(sr[8 * g + i], sr[8 * g + i + 1], cc2, nm2, x[i], x[i + 1]);
            x[i] = ex2(x[i]);
            x[i + 1] = ex2(x[i + 1]);
          }
          float s0, s1;
          add2x2(x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7], s0, s1);
          l_tile += s0 + s1;
          uint32_t w[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w[i]) : "f"(x[2 * i + 1]), "f"(x[2 * i]));
          asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%4], {%0, %1, %2, %3};" ::"r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(t_p + 4 * g) : "memory");
          if (kResc) {
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 8; i += 2) mul2(oc[i], oc[i + 1], al2);
            TMEM_ST8(t_o + 8 * g, oc);
          }
        }
      };
      if (rescale) tile_body(std::true_type{}); else tile_body(std::false_type{});
      l_run = fmaf(alpha, l_run, l_tile);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      asm volatile("bar.arrive %0, 288;" ::"r"(kBarP + t) : "memory");
    }

    const uint32_t par = (uint32_t)(T & 1) * 2048u;
    sts32f(aMaxOwn + par, l_run);
    asm volatile("bar.sync %0, 64;" ::"r"(pair_bar) : "memory");
    const float inv_l = 1.0f / (l_run + lds32f(aMaxPartner + par));
    mbar_wait_soft<33>(bar(BAR_ODONE + t), (uint32_t)((T - 1) & 1), abort_addr);
    tc_fence_after();
    const int qtile = qtile0 + t;
    // the query tile's own 32 KiB are the boxes of its eight warps: its last scores have been computed
    const int row0 = qtile * kTile + (row & ~31);
    if (lds_volatile(abort_addr) == 0)
      store_half_rows<kOutF32>(t_o, sbase + kOffQ + t * kTileBytes + (warp & 7) * kOutBoxBytes, lane, inv_l, &out_map, 64 * h, row0, bh, row0 < p.Nq);
  }

  if (warp < kSoftmaxWarps && lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");     // the output copies have left shared memory
  tc_fence_before();
  __syncthreads();
  if (tid == 0 && *abort_flag != 0) atomicCAS(p.status, 0, *abort_flag);
  if (warp == kSoftmaxWarps + 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(*tmem_slot) : "memory");
  }
}

}  // namespace fwd16

// The status word, and room for copies of Q, K and V (whole tiles), which are made where the output overlaps them.
size_t bf16_workspace_bytes(int B, int H, int64_t Nq, int64_t Nkv) {
  const size_t bh = (size_t)B * H;
  const size_t qt = (size_t)((Nq + kTile - 1) / kTile), kt = (size_t)((Nkv + kTile - 1) / kTile);
  return 256 + bh * (qt + 2 * kt) * fwd16::kTileBytes;
}

// an operand as a [B H][N][128] bf16 tensor, fetched in boxes of 128 rows x 64 channels with the 128-byte swizzle
static int encode_operand_map(CUtensorMap* map, const void* x, int64_t bh, int64_t n) {
  const auto encode = tensor_map_encoder();
  if (!encode) return MXATTN_ECUDA;
  if (n > 0x7FFFFFFFLL || (uint64_t)n * kHeadDim * 2 >= (1ULL << 40)) return MXATTN_EUNSUPPORTED;
  const cuuint64_t dims[3] = {(cuuint64_t)kHeadDim, (cuuint64_t)n, (cuuint64_t)bh};
  const cuuint64_t strides[2] = {(cuuint64_t)kHeadDim * 2, (cuuint64_t)n * kHeadDim * 2};     // bytes, dimensions 1 and 2
  const cuuint32_t box[3] = {64u, (cuuint32_t)kTile, 1u};
  const cuuint32_t estr[3] = {1u, 1u, 1u};
  return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(x), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? MXATTN_OK : MXATTN_ECUDA;
}

int launch_forward_bf16(const void* q, const void* k, const void* v, void* o, int B, int H, int64_t Nq, int64_t Nkv,
                        float softmax_scale, unsigned flags, void* workspace, size_t workspace_bytes, cudaStream_t stream) {
  using namespace fwd16;
  if (workspace_bytes < bf16_workspace_bytes(B, H, Nq, Nkv)) return MXATTN_EWORKSPACE;
  const int64_t bh = (int64_t)B * H;
  const int64_t qt = (Nq + kTile - 1) / kTile, kt = (Nkv + kTile - 1) / kTile;
  const int64_t pairs = (qt + 1) / 2, grid = bh * pairs;
  if (qt > 0x3FFFFFFF || kt > 65535 || qt > 0x7FFFFFFF || bh > 65535 || grid > 0x7FFFFFFF) return MXATTN_EUNSUPPORTED;
  const int n_sm = sm_count();
  if (n_sm == 0) return MXATTN_ECUDA;
  CUtensorMap q_map, k_map, v_map, out_map;
  const bool f32 = flags & MXATTN_FLAG_OUT_FP32;
  // The kernel reads its inputs while its first CTAs write the output.  An operand that the output overlaps is copied to the
  // workspace first -- other than Q exactly in place, of which a CTA reads the rows that it writes, and before it does.
  const size_t row = kHeadDim * 2, nq = (size_t)bh * Nq * row, nkv = (size_t)bh * Nkv * row, no = f32 ? 2 * nq : nq;
  uint8_t* spare = static_cast<uint8_t*>(workspace) + 256;
  auto apart = [&](const void*& x, size_t n, int64_t tiles, bool in_place) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(x), b = reinterpret_cast<uintptr_t>(o);
    if (a < b + no && b < a + n && !(in_place && a == b)) {
      if (cudaMemcpyAsync(spare, x, n, cudaMemcpyDeviceToDevice, stream) != cudaSuccess) return false;
      x = spare;
    }
    spare += (size_t)(bh * tiles) * kTileBytes;
    return true;
  };
  const void *q_in = q, *k_in = k, *v_in = v;
  if (!apart(q_in, nq, qt, !f32) || !apart(k_in, nkv, kt, false) || !apart(v_in, nkv, kt, false)) return MXATTN_ECUDA;
  int rc;
  if ((rc = encode_operand_map(&q_map, q_in, bh, Nq)) || (rc = encode_operand_map(&k_map, k_in, bh, Nkv)) || (rc = encode_operand_map(&v_map, v_in, bh, Nkv)) ||
      (rc = encode_output_map(&out_map, o, bh, Nq, f32)))
    return rc;
  if (launch_zero(static_cast<uint32_t*>(workspace), 4, stream) != MXATTN_OK) return MXATTN_ECUDA;
  Params p;
  p.status = static_cast<int*>(workspace);
  p.Nq = Nq; p.Nkv = Nkv; p.q_tiles_n = (int)qt; p.kv_tiles = (int)kt; p.q_pairs = (int)pairs;
  const TileSplit split(grid, n_sm);
  p.pair_ctas = (int)split.pair_ctas;
  p.scale_log2e = softmax_scale * 1.4426950408889634f;
  auto kern = f32 ? attention_bf16_kernel<true> : attention_bf16_kernel<false>;
  if (!ensure_dynamic_smem((const void*)kern, kSmemBytes)) return MXATTN_ECUDA;
  return launch_pdl(kern, dim3((unsigned)split.ctas), kThreads, kSmemBytes, stream, p, q_map, k_map, v_map, out_map) == cudaSuccess ? MXATTN_OK : MXATTN_ECUDA;
}

}  // namespace mxattn
