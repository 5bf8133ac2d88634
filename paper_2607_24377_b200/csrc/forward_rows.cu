// MXFP4 attention forward for few query rows (paper Algorithm 2, lines 6-19): the kernel for a problem whose query tiles cannot fill the
// GPU, or not its last wave (forward_plan in forward_walk.cu says where).
//
// KV tiles must be visited one after the other (P-hat depends on the history of the running maximum), so what counts for a
// short problem is the latency of one tile, and the only way to use idle SMs is to give each CTA fewer query rows.  A CTA of
// the walking kernel takes 128 rows and 1200 cycles per tile and more; most of that is the exponentials, 1024 cycles per 128 x 128 tile
// and SM.  A tensor-core product has 128 rows, and the 32 rows of a tensor-memory lane quarter belong to one SM sub-partition, so
// fewer rows per CTA alone would only leave sub-partitions idle.  Here the CTA's 128/R query rows are REPLICATED R times down
// the operand tile: every quarter (or pair of quarters) then sees the same rows' scores, and each takes its own share of the
// KEYS.  R = 4: 32 rows, each sub-partition one block of 32 keys, 256 cycles of exponentials per tile; R = 2: 64 rows, two
// warps of one block each, 512 cycles.  P-hat is written to all R replicas, so each replica's accumulator is complete, and a
// warp rescales and stores only its own 32 output channels of its replica.  The arithmetic per row is that of forward.cu,
// value for value.
//
// Warp w works on the tensor-memory quarter w % 4 (row group rg = w % (4/R) of 32 rows) and the keys (and output channels)
// of block kb: one thread per row and block.  The four warps of a row group exchange their block maxima through shared
// memory at a named barrier once per tile.  S is double-buffered, so the next tile's scores are ready when a warp gets
// there (loading them before the hand-over instead makes the hand-over's fence wait for the load: 5 % slower).  Measured
// (B200, 1965 MHz, all exponentials on their unit): 1200 cycles per tile with R = 4, 1530 with R = 2; 2 heads of 1024 x 1024: attention
// launch 14 -> 6 us (from 256 rows per CTA).  With R = 4 a sub-partition has one softmax warp, which alone keeps the
// exponential unit busy for half of the time: where only the codes count (PNQ) every other pair is a polynomial (exp2_poly), 1200 ->
// 1085 cycles (1 x 4096 x 40000, whole call, none, a quarter, three eighths, half: 182.7, 172.6, 166.2, 165.0 us; 2 x 1024 10.6 -> 10.35).
// With R = 2, which runs few tiles only, half is ahead as well (attention launch, none, a quarter, half: 2 x 4096 at 1, 2, 3 tiles 3.78, 3.71,
// 3.67, 4.58, 4.45, 4.40, 5.40, 5.22, 5.14, 1 x 9000 x 512 6.35, 6.13, 6.04).  R = 1 (128 rows, 16 warps) was behind the walking kernel at
// every length (74 x 256 queries x 128: 5.02 / 4.82, 37 x 256 x 8192: 64.9 / 45.6) and is gone.
// Not kept: the accumulator loaded for its rescaling before the last exponentials (184) or before P-hat is stored (173), a test_wait in
// front of the wait for the scores (192).
#include <string.h>

#include "common.cuh"
#include "tc_helpers.cuh"

namespace mxattn {
namespace rows {
using namespace fwd;

constexpr int kStages = 4;
constexpr int kNV = 144;                         // GEMM 2 N: 128 channels + 16 rows of ones (column 128 = row sum of P-hat)
constexpr int kVStageBytes = kNV * 64;

constexpr int kOffQ = 0;
constexpr int kOffK = kOffQ + kTileCodeBytes;
constexpr int kOffV = kOffK + kStages * kTileCodeBytes;
constexpr int kOffP = kOffV + kStages * kVStageBytes;            // 2 buffers
constexpr int kOffSFQ = kOffP + 2 * kTileCodeBytes;
constexpr int kOffSFK = kOffSFQ + kTileScaleBytes;
constexpr int kOffSFV = kOffSFK + kStages * kTileScaleBytes;
constexpr int kOffSFP = kOffSFV + kStages * kTileScaleBytes;     // 2 buffers
constexpr int kOffSFOnes = kOffSFP + 2 * kTileScaleBytes;
constexpr int kOffX = kOffSFOnes + kTileScaleBytes;              // block maxima: [2 buffers][row group 4][block 4][32] floats
constexpr int kXBuf = 4 * 4 * 32 * 4;
constexpr int kOffXL = kOffX + 2 * kXBuf;               // row sums of a tile by block (direct placement), laid out alike
constexpr int kOffBar = kOffXL + 2 * kXBuf;
enum Bar { BAR_Q = 0, BAR_KFULL = 1, BAR_KEMPTY = BAR_KFULL + kStages, BAR_SFULL = BAR_KEMPTY + kStages, BAR_PFULL = BAR_SFULL + 2,
           BAR_ODONE = BAR_PFULL + 2, kNumBars = BAR_ODONE + 2 };
constexpr int kOffMisc = kOffBar + kNumBars * 8;                 // tmem slot, abort flag, "an earlier CTA gave up"
// More than half of an SM's shared memory, so that no two CTAs share an SM: the second one would wait in its tensor-memory
// allocation until the first has finished, while other SMs stand idle (placed behind a draining predecessor, CTAs do land
// like that: 1.5 us per tile instead of 0.7).
constexpr int kSmemBytes = 120 * 1024;
static_assert(kOffMisc + 32 + 1024 <= kSmemBytes, "shared memory per CTA");
constexpr uint32_t kColS = 0, kColO = 256, kColSFQ = 400, kColSFK = 404, kColSFV = 412, kColSFP = 428;

struct Params {
  const uint8_t* q_codes; const uint8_t* q_scales;
  const uint8_t* k_codes; const uint8_t* k_scales;
  const uint8_t* v_codes; const uint8_t* v_scales;
  void* out;
  int* status;
  int64_t Nq, Nkv;
  int q_tiles, kv_tiles, groups;   // groups of 128/R rows per head
  int first;                       // the first CTA's group, counted over all heads
  float scale_log2e;
};

template <int R, bool kUos, bool kPnq, bool kOutF32>      // R = 4 or 2
__global__ void __launch_bounds__(32 * (16 / R + 2), 1) attention_rows_kernel(const Params p) {
  constexpr int kWarps = 16 / R, kRG = 4 / R;                    // softmax warps, row groups of 32
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar0 = sbase + kOffBar;
  auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kOffMisc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kOffMisc + 8);

  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const int T = p.kv_tiles;
  const int bh = ((int)blockIdx.x + p.first) / p.groups, grp = (int)blockIdx.x + p.first - bh * p.groups;
  const int qtile = grp / R, slab = (grp % R) * kRG;             // 128-row tile and first 32-row group in it

  // ---- setup -------------------------------------------------------------------------------
  if (tid == 0) {
    mbar_init(bar(BAR_Q), 1);
    for (int s = 0; s < kStages; ++s) { mbar_init(bar(BAR_KFULL + s), 1); mbar_init(bar(BAR_KEMPTY + s), 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(bar(BAR_SFULL + i), 1); mbar_init(bar(BAR_PFULL + i), kWarps); mbar_init(bar(BAR_ODONE + i), 1); }
    abort_flag[0] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = tid; i < kStages * 64; i += 32 * (kWarps + 2))    // rows of ones behind every V stage (code 2 = 1.0), their scales
    reinterpret_cast<uint4*>(smem + kOffV + (i >> 6) * kVStageBytes + kTileCodeBytes)[i & 63] =
        make_uint4(0x22222222u, 0x22222222u, 0x22222222u, 0x22222222u);
  if (tid < kTileScaleBytes / 16) reinterpret_cast<uint4*>(smem + kOffSFOnes)[tid] = make_uint4(0x7F7F7F7Fu, 0x7F7F7F7Fu, 0x7F7F7F7Fu, 0x7F7F7F7Fu);
  if (warp == kWarps + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  pdl_wait();                                                    // the operands and the status word are ready
  const int64_t qt = (int64_t)bh * p.q_tiles + qtile;
  if (warp == 0) {                                               // Q's scales, replicated: the four bytes of row i of a 32-row group
    uint32_t w[4];                                               // sit at 16 i + 4 (group), one 16-byte line per i
#pragma unroll
    for (int g = 0; g < 4; ++g) w[g] = ld_global(reinterpret_cast<const uint32_t*>(p.q_scales + qt * kTileScaleBytes) + lane * 4 + slab + g % kRG);
    *reinterpret_cast<uint4*>(smem + kOffSFQ + lane * 16) = make_uint4(w[0], w[1], w[2], w[3]);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (tid == 0) abort_flag[1] = *reinterpret_cast<volatile int*>(p.status);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_trigger();
  constexpr uint32_t tmem = 0;
  if (*tmem_slot != 0) *abort_flag = kCodeTmemBase;
  const int role = (abort_flag[1] != 0 || *tmem_slot != 0) ? kWarps + 2 : warp;     // an earlier CTA gave up: drain the grid quickly

  if (role == kWarps) {
    // =============================== producer ===============================================
    if (lane == 0) {
      mbar_expect_tx(bar(BAR_Q), kTileCodeBytes);
      for (int r = 0; r < R; ++r)                                // the rows' codes, R times down the tile (the swizzle has a period of 8 rows)
        bulk_g2s(sbase + kOffQ + r * (kTileCodeBytes / R), p.q_codes + qt * kTileCodeBytes + slab * 2048, kTileCodeBytes / R, bar(BAR_Q));
      const int64_t kv0 = (int64_t)bh * T;
      bool ok = true;
      int j = 0;
      for (; j < T; ++j) {
        const int s = j % kStages;
        if (j >= kStages) ok = mbar_wait1(bar(BAR_KEMPTY + s), (uint32_t)((j / kStages) & 1) ^ 1u, abort_flag, p.status, 11);
        if (!ok) break;
        mbar_expect_tx(bar(BAR_KFULL + s), 2 * (kTileCodeBytes + kTileScaleBytes));
        bulk_g2s(sbase + kOffK + s * kTileCodeBytes, p.k_codes + (kv0 + j) * kTileCodeBytes, kTileCodeBytes, bar(BAR_KFULL + s));
        bulk_g2s(sbase + kOffSFK + s * kTileScaleBytes, p.k_scales + (kv0 + j) * kTileScaleBytes, kTileScaleBytes, bar(BAR_KFULL + s));
        bulk_g2s(sbase + kOffV + s * kVStageBytes, p.v_codes + (kv0 + j) * kTileCodeBytes, kTileCodeBytes, bar(BAR_KFULL + s));
        bulk_g2s(sbase + kOffSFV + s * kTileScaleBytes, p.v_scales + (kv0 + j) * kTileScaleBytes, kTileScaleBytes, bar(BAR_KFULL + s));
      }
      if (!ok || *abort_flag) {                                  // gave up: let copies in flight land before shared memory is released
        const long long t0 = clock64();
        for (int f = (j > kStages ? j - kStages : 0); f < j; ++f)
          while (!mbar_try(bar(BAR_KFULL + f % kStages), (uint32_t)((f / kStages) & 1)) && clock64() - t0 < 200000000LL) {}
        while (!mbar_try(bar(BAR_Q), 0u) && clock64() - t0 < 200000000LL) {}
      }
    }
  } else if (role == kWarps + 1) {
    // =============================== MMA issuer (converged warp) ============================
    const uint32_t leader = elect_one();
    constexpr uint32_t kDescHiTile = (512u >> 4) | (1u << 14) | (4u << 29);   // 64-byte swizzle, K-major
    auto desc = [](uint32_t saddr) { return ((uint64_t)kDescHiTile << 32) | (saddr >> 4); };
    auto gemm1 = [&](int f) {                                    // S(f) = Q K_f^T into score buffer f & 1
      const int s = f % kStages;
      if (!mbar_wait_warp(bar(BAR_KFULL + s), (uint32_t)((f / kStages) & 1), abort_flag, p.status, 22)) return false;
      tc_fence_after();
      const uint32_t d = tmem + kColS + 128 * (f & 1), sfb = tmem + kColSFK + 4 * (f & 1), a = sbase + kOffQ, b = sbase + kOffK + s * kTileCodeBytes;
      tc_cp_sf_if(leader, sfb, sbase + kOffSFK + s * kTileScaleBytes);
      tc_mma_if(leader, d, desc(a), desc(b), make_idesc(128, 0), tmem + kColSFQ, sfb, 0u);
      tc_mma_if(leader, d, desc(a + 32), desc(b + 32), make_idesc(128, 1), tmem + kColSFQ, sfb, 1u);
      tc_commit_if(leader, bar(BAR_SFULL + (f & 1)));
      tc_cp_sf_if(leader, tmem + kColSFV + 8 * (f & 1), sbase + kOffSFV + s * kTileScaleBytes);
      return true;
    };
    bool ok = mbar_wait_warp(bar(BAR_Q), 0u, abort_flag, p.status, 21);
    if (ok) {
      tc_fence_after();
      tc_cp_sf_if(leader, tmem + kColSFQ, sbase + kOffSFQ);
      tc_cp_sf_if(leader, tmem + kColSFV + 4, sbase + kOffSFOnes);
      tc_cp_sf_if(leader, tmem + kColSFV + 12, sbase + kOffSFOnes);
      ok = gemm1(0) && (T < 2 || gemm1(1));
    }
    for (int f = 0; f < T && ok; ++f) {
      const int s = f % kStages, b = f & 1;
      ok = mbar_wait_warp(bar(BAR_PFULL + b), (uint32_t)((f >> 1) & 1), abort_flag, p.status, 24);
      if (!ok) break;
      tc_fence_after();
      const uint32_t sfa = tmem + kColSFP + 4 * b, sfb = tmem + kColSFV + 8 * b;
      const uint32_t pa = sbase + kOffP + b * kTileCodeBytes, vb = sbase + kOffV + s * kVStageBytes;
      tc_cp_sf_if(leader, sfa, sbase + kOffSFP + b * kTileScaleBytes);
      tc_mma_if(leader, tmem + kColO, desc(pa), desc(vb), make_idesc(kNV, 0), sfa, sfb, f > 0 ? 1u : 0u);
      tc_mma_if(leader, tmem + kColO, desc(pa + 32), desc(vb + 32), make_idesc(kNV, 1), sfa, sfb, 1u);
      tc_commit_if(leader, bar(BAR_ODONE + b));
      tc_commit_if(leader, bar(BAR_KEMPTY + s));
      // the hand-over of P-hat(f) also says that the scores of tile f have been read
      if (f + 2 < T) ok = gemm1(f + 2);
    }
  } else if (role < kWarps) {
    // =============================== softmax warps ==========================================
    const int quarter = warp & 3, rg = quarter % kRG, kb = (quarter / kRG) * kRG + (warp >> 2);
    const uint32_t t_s = tmem + ((uint32_t)(quarter * 32) << 16) + 32 * kb;       // this block's scores (buffer 0)
    constexpr uint32_t kToO = kColO - kColS;                                       // ... and from there its output channels
    const uint32_t t_l = tmem + ((uint32_t)(quarter * 32) << 16) + kColO + 128;    // the row sum P-hat 1
    const uint32_t abort_addr = bar0 + (kOffMisc + 8 - kOffBar);
    const uint32_t aX = sbase + kOffX + (rg * 4 * 32 + lane) * 4;
    const bool ragged = (p.Nkv & (kTile - 1)) != 0;
    const float c = p.scale_log2e;
    float m_run = -INFINITY;
    // Direct placement: the row sum of a pair of blocks (64 keys, the share of a thread of forward.cu, so that the sums round
    // alike) is accumulated by both warps of the pair, one tile behind: the partner's part comes with the next meeting.
    float l_run = 0.0f, l_own = 0.0f, alpha = 1.0f;
    auto add_sums = [&](int b) {
      l_run = fmaf(alpha, l_run, l_own + lds32f(aX + (kOffXL - kOffX) + b * kXBuf + (kb ^ 1) * 128));     // line 14 (direct), Eq. 12
    };
    for (int j = 0; j < T; ++j) {
      const int b = j & 1;
      mbar_wait_soft<31>(bar(BAR_SFULL + b), (uint32_t)((j >> 1) & 1), abort_addr);
      tc_fence_after();
      uint32_t s[32];
      TMEM_LD32(t_s + 128 * b, s);
      TMEM_LD_WAIT32(s);
      if (ragged && j == T - 1) {                                // keys beyond Nkv do not exist
        const int valid = (int)(p.Nkv - (int64_t)j * kTile) - 32 * kb;
#pragma unroll
        for (int i = 0; i < 32; ++i)
          if (i >= valid) s[i] = 0xFF800000u;                    // -inf
      }
      float q4[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t* v = s + 8 * u;
        float mx = max3(__uint_as_float(v[0]), __uint_as_float(v[1]), __uint_as_float(v[2]));
        mx = max3(mx, __uint_as_float(v[3]), __uint_as_float(v[4]));
        mx = max3(mx, __uint_as_float(v[5]), __uint_as_float(v[6]));
        q4[u] = fmaxf(mx, __uint_as_float(v[7]));
      }
      const float bmax = fmaxf(max3(q4[0], q4[1], q4[2]), q4[3]);
      const uint32_t ax = aX + b * kXBuf;
      sts32f(ax + kb * 128, bmax);
      asm volatile("bar.sync %0, 128;" ::"r"(1 + rg) : "memory");                  // the four warps of these rows
      if (!kPnq && j > 0) add_sums(b ^ 1);
      const float m_old = m_run;
      const float m_new = fmaxf(max3(lds32f(ax), lds32f(ax + 128), lds32f(ax + 256)), fmaxf(lds32f(ax + 384), m_old));   // line 10
      m_run = m_new;
      const bool rescale = __any_sync(0xFFFFFFFFu, m_new != m_old) && j > 0;       // line 15
      // block exponent, as in forward.cu
      const float d = (bmax - m_new) * c;
      const float fl = __fadd_rd(d, 12582912.0f) - 12582912.0f;                    // floor(d)
      float ef = fl + ((kUos && (d - fl) > 0.85798097f) ? -1.0f : -2.0f);
      ef = fmaxf(ef, -127.0f);
      if (d < -126.0f) ef = 0.0f;
      const uint32_t sfb = __float_as_uint(ef + 12582912.0f) - (0x4B400000u - 127u);   // e + 127
      const float nmc = -(m_new * c);
      const uint64_t cc2 = dup2(c), nb2 = dup2(nmc - ef);
      uint32_t w[4];
      float sx = 0.0f;
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        float x[8];
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
          fma2(s[8 * g + i], s[8 * g + i + 1], cc2, nb2, x[i], x[i + 1]);
          if (kPnq && i >= 4) {
            exp2_poly(x[i], x[i + 1]);
          } else {
            x[i] = ex2(x[i]);
            x[i + 1] = ex2(x[i + 1]);
          }
        }
        if constexpr (kPnq) {
          w[g] = pack_e2m1x8_relu(x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7]);
        } else {
          w[g] = pack_e2m1x8(x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7]);
          float s0, s1;
          add2x2(x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7], s0, s1);
          sx += s0 + s1;
        }
      }
      // P buffer b was read by the output product of tile j - 2, behind which the scores of tile j were committed
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int row = (r * kRG + rg) * 32 + lane;
        sts128(sbase + kOffP + b * kTileCodeBytes + tile_code_offset(row, kb), make_uint4(w[0], w[1], w[2], w[3]));
        sts8(sbase + kOffSFP + b * kTileScaleBytes + tile_scale_offset(row, kb), sfb);
      }
      alpha = 1.0f;
      if (!kPnq) {
        l_own = sx * __uint_as_float(sfb << 23);
        sts32f(ax + (kOffXL - kOffX) + kb * 128, l_own);
      }
      if (rescale) {
        alpha = ex2((m_old - m_new) * c);
        mbar_wait_soft<32>(bar(BAR_ODONE + (b ^ 1)), (uint32_t)(((j - 1) >> 1) & 1), abort_addr);
        tc_fence_after();
        const uint64_t al2 = dup2(alpha);
        uint32_t o[32], lr = 0;
        TMEM_LD32(t_s + kToO, o);
        const bool sum = kPnq && (warp >> 2) == 0;               // one warp per quarter rescales the row sum
        if (sum) asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(lr) : "r"(t_l) : "memory");
        TMEM_LD_WAIT32(o);
#pragma unroll
        for (int i = 0; i < 32; i += 2) mul2(o[i], o[i + 1], al2);
        TMEM_ST32(t_s + kToO, o);
        if (sum) {
          asm volatile("" : "+r"(lr));
          lr = __float_as_uint(__uint_as_float(lr) * alpha);
          asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%1], {%0};" ::"r"(lr), "r"(t_l) : "memory");
        }
        tmem_st_wait();
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(BAR_PFULL + b));
    }
    // ---- epilogue: O = O~ / l (line 18), this block's 32 channels ----
    float l = 0.0f;
    if (!kPnq) {
      asm volatile("bar.sync %0, 128;" ::"r"(1 + rg) : "memory");
      add_sums((T - 1) & 1);
      const uint32_t ax = aX + (T & 1) * kXBuf;
      sts32f(ax + kb * 128, l_run);
      asm volatile("bar.sync %0, 128;" ::"r"(1 + rg) : "memory");
      l = l_run + lds32f(ax + (kb ^ 2) * 128);                   // the other pair's sum
    }
    mbar_wait_soft<33>(bar(BAR_ODONE + ((T - 1) & 1)), (uint32_t)(((T - 1) >> 1) & 1), abort_addr);
    tc_fence_after();
    uint32_t o[32], lr = 0;
    if (kPnq) asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(lr) : "r"(t_l) : "memory");
    TMEM_LD32(t_s + kToO, o);
    TMEM_LD_WAIT32(o);
    if (kPnq) { asm volatile("" : "+r"(lr)); l = __uint_as_float(lr); }
    const uint64_t inv2 = dup2(1.0f / l);
    const int64_t grow = (int64_t)qtile * kTile + (slab + rg) * 32 + lane;
    if (grow < p.Nq && lds_volatile(abort_addr) == 0) {
#pragma unroll
      for (int i = 0; i < 32; i += 2) mul2(o[i], o[i + 1], inv2);
      const int64_t at = ((int64_t)bh * p.Nq + grow) * kHeadDim + 32 * kb;
      if (kOutF32) {
        uint4* dst = reinterpret_cast<uint4*>(static_cast<float*>(p.out) + at);
#pragma unroll
        for (int i = 0; i < 8; ++i) dst[i] = make_uint4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
      } else {
        uint4* dst = reinterpret_cast<uint4*>(static_cast<uint16_t*>(p.out) + at);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          uint32_t hh[4];
#pragma unroll
          for (int k = 0; k < 4; ++k)
            asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(hh[k]) : "f"(__uint_as_float(o[8 * i + 2 * k + 1])), "f"(__uint_as_float(o[8 * i + 2 * k])));
          dst[i] = make_uint4(hh[0], hh[1], hh[2], hh[3]);
        }
      }
    }
  }

  // ---- teardown ------------------------------------------------------------------------------
  tc_fence_before();
  __syncthreads();
  if (tid == 0 && *abort_flag != 0) atomicCAS(p.status, 0, *abort_flag);
  if (warp == kWarps + 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(*tmem_slot) : "memory");
  }
}

}  // namespace rows

int launch_forward_rows(int R, int64_t first_pair, const void* q_codes, const void* q_scales, const void* k_codes, const void* k_scales,
                        const void* v_codes, const void* v_scales, void* o, int B, int H, int64_t Nq, int64_t Nkv,
                        float softmax_scale, unsigned flags, int* status, cudaStream_t stream) {
  using namespace rows;
  Params p;
  p.q_codes = (const uint8_t*)q_codes; p.q_scales = (const uint8_t*)q_scales;
  p.k_codes = (const uint8_t*)k_codes; p.k_scales = (const uint8_t*)k_scales;
  p.v_codes = (const uint8_t*)v_codes; p.v_scales = (const uint8_t*)v_scales;
  p.out = o; p.status = status; p.Nq = Nq; p.Nkv = Nkv;
  p.q_tiles = (int)((Nq + kTile - 1) / kTile); p.kv_tiles = (int)((Nkv + kTile - 1) / kTile);
  p.groups = (int)((Nq + kTile / R - 1) / (kTile / R));
  const int64_t pairs = (p.q_tiles + 1) / 2, first = first_pair / pairs * p.groups + (first_pair % pairs) * 2 * R, total = (int64_t)B * H * p.groups;
  if (total > 0x7FFFFFFF) return MXATTN_EUNSUPPORTED;
  p.first = (int)first;
  p.scale_log2e = softmax_scale * 1.4426950408889634f;
  const bool uos = flags & MXATTN_FLAG_UOS, pnq = flags & MXATTN_FLAG_PNQ, f32 = flags & MXATTN_FLAG_OUT_FP32;
  void (*kern)(const Params) = nullptr;
#define PICK(U, P, F) if (uos == U && pnq == P && f32 == F) kern = R == 4 ? attention_rows_kernel<4, U, P, F> : attention_rows_kernel<2, U, P, F>;
  PICK(false, false, false) PICK(false, false, true) PICK(false, true, false) PICK(false, true, true)
  PICK(true, false, false) PICK(true, false, true) PICK(true, true, false) PICK(true, true, true)
#undef PICK
  if (!ensure_dynamic_smem((const void*)kern, kSmemBytes)) return MXATTN_ECUDA;
  return launch_pdl(kern, dim3((unsigned)(total - first)), 32 * (16 / R + 2), kSmemBytes, stream, p) == cudaSuccess ? MXATTN_OK : MXATTN_ECUDA;
}

}  // namespace mxattn
