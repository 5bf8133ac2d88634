// MXFP4 launches of the walking attention kernel (walk.cuh), and which problems it takes.
#include "walk.cuh"

namespace mxattn {
namespace walk {

template <bool kUos, bool kPnq, bool kOutF32, bool kTake, bool kDump>
__global__ void __launch_bounds__(kThreads, 1) attention_walk_kernel(const Params p, const __grid_constant__ CUtensorMap out_map) {
  using L = Lay<false>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::kOffMisc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::kOffMisc + 8);
  volatile int* status_before = abort_flag + 2;
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  set_up<false>(smem, tid);
  if (warp == kIssuer1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  pdl_wait();                                                    // the operands and the status word are ready
  if (tid == 0) *status_before = *reinterpret_cast<volatile int*>(p.status);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_trigger();
  if (*tmem_slot != 0) *abort_flag = kCodeTmemBase;
  const int role = __shfl_sync(0xFFFFFFFFu, (*status_before != 0 || *tmem_slot != 0) ? kThreads / 32 : warp, 0);     // an earlier launch gave up
  play<false, kUos, kPnq, kOutF32, kTake, kDump>(p, out_map, smem, role, warp, lane);
  tc_fence_before();
  __syncthreads();
  if (tid == 0 && *abort_flag != 0) atomicCAS(p.status, 0, *abort_flag);
  if (warp == kIssuer1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(*tmem_slot) : "memory");
  }
}

}  // namespace walk

// How a problem is divided between the kernels.  All figures are attention launches with the PNQ row sum / the direct one, in us.
//
// A launch that has the GPU to itself: the walking kernel, but
//  - CTAs of 32 rows where they are one wave at most: they take two thirds to nine tenths of the time whatever the length (18 x 256 queries, 1,
//    4, 16, 64, 300 KV tiles, walked 4.59 6.63 14.7 45.4 187 / 4.79 7.11 16.1 50.7 214, 32 rows 3.37 5.30 12.5 39.1 158 / 3.39 5.41 13.1 41.8
//    175).  A second wave of them never pays (37 x 256, 64 tiles: 45.6 / 50.9, 32 rows 76.7 / 82.7).
//  - CTAs of 64 rows where those are one wave, up to 6 KV tiles (direct 14; 37 x 256, 1, 4, 8, 16, 32 tiles: walked 4.62 6.69 9.40 14.8 25.4 /
//    4.81 7.18 10.2 16.1 28.0, 64 rows 3.82 6.04 9.02 14.9 26.5 / 3.94 6.42 9.78 16.2 29.1).  In a whole call the operand launch's last CTAs decide
//    as well: of 21 problems with PNQ at 5 tiles one takes longer with 64 rows (by 1 %), at 7 and 9 tiles they are 3 and 2 % ahead in the
//    mean, but five behind by up to 4 % (6 x 889 x 889 11.3 / 11.9).
//  - Whole waves of pairs walked and the rest in one wave of CTAs of 32 rows, a second launch, if that is estimated to take less than the
//    rounds of single tiles it saves.  A round: T x 1150 + 4500 cycles (direct 1335, 3500); the second launch with the wait for the first's last
//    CTAs: T x 1045 + 12000 (1175, 8000).  152 x 256, 32, 64, 128, 300 tiles: all walked 67.9 127.7 244.1 548.9 / 75.6 144.4 279.0 635.5,
//    divided 69.8 128.4 241.0 536.9 / 75.5 141.4 270.7 613.2; 758 x 256, 64, 128: 455.4 879.5 / 517.4 1009.6, divided 458.4 879.5 / 517.1 1003.9.
//    64 rows there were behind in all cases (185 x 256, 64 and 300 tiles: 136.9 576 / 154.2 671 for 128.1 550 / 144.9 638).
//  - The kernel for pairs beyond 2^31 tiles, which a CTA of the walking kernel counts in 32 bits (where it takes items from others it may get
//    them all): a single tile takes 1200-1290 cycles here (direct row sum 1390-1450), a pair 2570-2700 there (3050).
//
// Beside other launches (the stages of a forward from host tensors) nothing is left idle that small CTAs could use, and CTAs that hold their
// SMs longer, as those of pairs do not, keep the next stage's waiting.  Up to 48 tiles: walked, unless a wave of pairs makes two rounds of tiles.
// Above 128 tiles: walked, unless the query tiles are fewer than half of the KV tiles.  Between, the kernel for pairs.  Whole call, medians of 22, kernel
// for pairs / walked: 24 x 8192 3253 3270 / 3292 3296, 8 x 16000 2235 2292 / 2259 2282, 24 x 6200 2542 2528 / 2502 2545, 12 x 13000 2684 2687 / 2637
// 2660, 24 x 14000 5473 5476 / 5392 5450, but 10 x 10000 1849 1808 / 1853 1827, 16 x 12000 3302 3271 / 3314 3296; 24 x 7000 x 30000 7891 7934 / 7977
// 7957; above 128 tiles, at an earlier state, 12 x 20000 4061 3908, 8 x 40000 5934 5588 / 6039 5817, 10 x 75600 16875 15673, 2 x 60000 3608 3157.
ForwardPlan forward_plan(int64_t n_sm, int64_t bh, int64_t Nq, int64_t Nkv, bool pnq, bool followed) {
  const int64_t T = (Nkv + kTile - 1) / kTile, tiles = (Nq + kTile - 1) / kTile, pairs = (tiles + 1) / 2, total = bh * pairs;
  auto rounds = [&](int64_t n) { return (n + n_sm - 1) / n_sm; };
  const bool counts = (T > kStaticTiles ? bh * tiles : rounds(bh * tiles)) * T <= 0x7FFFFF00;      // (the last few are for the teams' steps beyond the end)
  if (followed) {
    const bool walk = T <= 48 ? rounds(bh * tiles) < 2 * rounds(total) || rounds(total) > 1 : T > 128 && 2 * tiles >= T;
    return ForwardPlan{counts && walk, total, 0};
  }
  auto groups = [&](int64_t R, int64_t from) {        // of 128 / R rows, behind the first `from` pairs
    const int64_t per_head = (Nq + kTile / R - 1) / (kTile / R);
    return bh * per_head - from / pairs * per_head - from % pairs * 2 * R;
  };
  const int64_t at = total / n_sm * n_sm;
  if (at == 0) {
    if (groups(4, 0) <= n_sm) return ForwardPlan{true, 0, 4};
    if (groups(2, 0) <= n_sm && T <= (pnq ? 6 : 14)) return ForwardPlan{true, 0, 2};
  }
  if (!counts) return ForwardPlan{false, total, 0};
  if (at > 0 && at < total && groups(4, at) <= n_sm) {
    const int64_t saved = rounds(bh * tiles) - rounds(at / pairs * tiles + at % pairs * 2);
    if (T * (pnq ? 1045 : 1175) + (pnq ? 12000 : 8000) < saved * (T * (pnq ? 1150 : 1335) + (pnq ? 4500 : 3500))) return ForwardPlan{true, at, 4};
  }
  return ForwardPlan{true, total, 0};
}

size_t forward_dump_bytes(int B, int H, int64_t Nq, int64_t Nkv) {
  const int64_t qt = (Nq + kTile - 1) / kTile, kt = (Nkv + kTile - 1) / kTile;
  return (size_t)((int64_t)B * H * qt * kt * walk::kDumpTileBytes + (int64_t)B * H * qt * kTile * 4);
}

// The first `pairs` pairs of query tiles, counted over all heads.  `dump`: all of them.
int launch_forward_walk(int64_t n_sm, int64_t pairs, const void* q_codes, const void* q_scales, const void* k_codes, const void* k_scales,
                        const void* v_codes, const void* v_scales, void* o, int B, int H, int64_t Nq, int64_t Nkv,
                        float softmax_scale, unsigned flags, int* status, cudaStream_t stream, void* dump) {
  using namespace walk;
  Params p = {};
  p.q_codes = (const uint8_t*)q_codes; p.q_scales = (const uint8_t*)q_scales;
  p.k_codes = (const uint8_t*)k_codes; p.k_scales = (const uint8_t*)k_scales;
  p.v_codes = (const uint8_t*)v_codes; p.v_scales = (const uint8_t*)v_scales;
  p.status = status; p.Nq = Nq; p.Nkv = Nkv;
  p.q_tiles = (int)((Nq + kTile - 1) / kTile); p.kv_tiles = (int)((Nkv + kTile - 1) / kTile);
  const int64_t per_head = (p.q_tiles + 1) / 2, items = pairs / per_head * p.q_tiles + (pairs % per_head) * 2;
  if (items > 0x7FFFFFFF) return MXATTN_EUNSUPPORTED;
  p.total_items = (int)items;
  p.scale_log2e = softmax_scale * 1.4426950408889634f; p.softmax_scale = softmax_scale; p.dump = (uint8_t*)dump;
  const bool uos = flags & MXATTN_FLAG_UOS, pnq = flags & MXATTN_FLAG_PNQ, f32 = flags & MXATTN_FLAG_OUT_FP32, take = takes<false>(p, n_sm);
  Kernel kern = nullptr;
#define PICK(U, P, F) if (uos == U && pnq == P && f32 == F) kern = take ? attention_walk_kernel<U, P, F, true, false> : attention_walk_kernel<U, P, F, false, false>;
  PICK(false, false, false) PICK(false, false, true) PICK(false, true, false) PICK(false, true, true)
  PICK(true, false, false) PICK(true, false, true) PICK(true, true, false) PICK(true, true, true)
#undef PICK
  if (dump) {
    if (!f32) return MXATTN_EINVAL;
#define PICK(U, P) if (uos == U && pnq == P) kern = take ? attention_walk_kernel<U, P, true, true, true> : attention_walk_kernel<U, P, true, false, true>;
    PICK(false, false) PICK(false, true) PICK(true, false) PICK(true, true)
#undef PICK
  }
  return launch(kern, Lay<false>::kSmemBytes, p, take, n_sm, (int64_t)B * H, o, flags, stream);
}

}  // namespace mxattn
