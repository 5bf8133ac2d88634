// MXFP4 launches of the walking attention kernel (walk.cuh), and which problems it takes.
#include "walk.cuh"

namespace mxattn {
namespace walk {

template <bool kUos, bool kPnq, bool kOutF32, bool kTake>
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
  play<false, kUos, kPnq, kOutF32, kTake>(p, out_map, smem, role, warp, lane);
  tc_fence_before();
  __syncthreads();
  if (tid == 0 && *abort_flag != 0) atomicCAS(p.status, 0, *abort_flag);
  if (warp == kIssuer1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(*tmem_slot) : "memory");
  }
}

}  // namespace walk

// Which problems this kernel takes, and how many of their pairs of query tiles (the rest goes to the small CTAs that
// `split` names).  Attention launch, us, kernel of forward.cu (in a form that walked its items up to 48 tiles) / this one, PNQ:
// 37 x 16384 queries, KV tiles 1, 4, 128: 52.8 / 45.7, 122.0 / 108.2, 2800 / 2753; 40 x 16384, 2 tiles: 84.6 / 73.3;
// 40 x 4096, 32: 235 / 206; 64 x 8192, 8: 188 / 169; 40 x 8192, 48, 64: 631 / 603, 825 / 795; 16 x 32768, 256: 4736 / 4733;
// 12 x 75600, 591: 18376 / 18456.  With the direct row sum, 1, 4, 32, 48 tiles: 58.2 / 46.0, 136.7 / 112.3, 262 / 228,
// 711 / 668, and whole calls: 37 x 4096, 100: 695 / 672; 16 x 32768, 256: 5402 / 5293; 12 x 40000, 400: 7647 / 7554; 12 x 75600,
// 591: 20726 / 20574; 24 x 16384, 591: 9405 / 9109.  (These figures, and those below, are of both kernels before the polynomial and
// the named barriers; what these changed stands at forward_walk_rest, which has the last word.)
// - A few whole waves of pairs that single tiles do not round better.  PNQ: one wave, whole call at 2, 7, 12, 49, 100 tiles: 37 x
//   1000 13.2 / 12.8, 22.7 / 22.5, 31.2 / 31.3, 105.4 / 106.8, 194.6 / 196.4 (14 x 1300 x 777, fp32: 20.7 / 20.5).  Direct: up to
//   four waves above 256 tiles; one wave (37 x 1000) at 2, 12, 48, 100, 256, 400 tiles: 13.8 / 12.9, 34.8 / 32.1, 115.4 / 111.0,
//   215.3 / 209.9, 506.8 / 506.4, 774.7 / 780.0; two (37 x 2048), 1016: 3369 / 3412; four (37 x 4096), 256, 469: 1658 / 1646,
//   2961 / 2970.
// - Launches that run beside others (`followed`) keep to short sequences: CTAs with fixed shares hold their SMs to the end
//   (24 x 8192 from host tensors: 3225 us for 3246); forward_walk_rest adds the long ones.
// - A CTA counts its tiles in 32 bits (the last few are left for the teams' steps beyond the end).  Where it takes items from
//   others it may get them all: one head of 6 million queries and keys has more.
// - Small CTAs for the last wave cost a launch and 1200 to 2125 cycles per tile and CTA, a round of single tiles T x 1390
//   cycles (direct 1500) + 1000.  All in one walk / last wave in small CTAs, whole call: 24 x 8192 529 / 541 (direct 568 / 589),
//   40 x 4096 241 / 261, 38 x 8192 x 3000 330 / 337, x 1000 134.8 / 139.7 (direct 140.4 / 145.3), 38 x 1000 x 700 25.0 / 27.7,
//   51 x 700 x 300 18.3 / 21.2.
WalkSplit forward_walk_split(int64_t n_sm, int64_t bh, int64_t Nq, int64_t Nkv, bool pnq, bool followed, const RowSplit& split) {
  const int64_t T = (Nkv + kTile - 1) / kTile, tiles = (Nq + kTile - 1) / kTile, pairs = (tiles + 1) / 2;
  if ((pnq && T > 256) || (followed && T > kBesideTiles)) return WalkSplit{false, 0};
  if ((T > kStaticTiles ? bh * tiles : (bh * tiles + n_sm - 1) / n_sm) * T > 0x7FFFFF00) return WalkSplit{false, 0};
  if (split.R == 0) {
    const int64_t rounds = (bh * tiles + n_sm - 1) / n_sm, waves = (bh * pairs + n_sm - 1) / n_sm;
    const bool pairs_ahead = pnq || followed ? waves == 1 : waves <= 4 && T > 256;
    return WalkSplit{rounds < 2 * waves || !pairs_ahead, bh * pairs};
  }
  auto walk = [&](int64_t items) { return (items + n_sm - 1) / n_sm * (T * (pnq ? 1390 : 1500) + 1000) + 4400; };
  const int64_t per_head = (Nq + kTile / split.R - 1) / (kTile / split.R), at = split.pairs_256;
  const int64_t done = at / pairs * per_head + (at % pairs) * 2 * split.R, before = at / pairs * tiles + (at % pairs) * 2;
  const int64_t small = (bh * per_head - done + n_sm - 1) / n_sm * (T * (split.R == 4 ? 1200 : split.R == 2 ? 1530 : 2125) + 4500);
  const bool all = walk(bh * tiles) <= (before > 0 ? walk(before) + 4000 : 0) + small;
  return WalkSplit{true, all ? bh * pairs : at};
}

// A launch that has the GPU to itself leaves none of the rest to the kernel of forward.cu: a single tile takes 1200-1290 cycles here
// (direct row sum 1390-1450), a pair 2570-2700 there (3050), so that two rounds of tiles are less than one wave of pairs.  Whole call, us,
// that kernel (and small CTAs for its last wave) / this one, PNQ: one wave of pairs, 37 x 1000 at 2, 8, 12, 49, 100, 313 KV tiles 13.2 / 12.3,
// 24.0 / 23.0, 31.2 / 29.9, 104.8 / 101.3, 193.8 / 185.8, 561.8 / 532.7, 14 x 1300 x 777 19.6 / 18.5 (fp32 output 20.5 / 19.8), x 6200
// 83.0 / 78.0, 74 x 500 x 3000 70.9 / 68.9; above 256 tiles 12 x 75600 18517 / 16972, 40 x 20000 x 40000 9183 / 8298, 24 x 16384 x 75600
// 8477 / 7565, 5 x 4000 x 40000 441 / 411, 20 x 2000 x 40000 682 / 657, 1 x 9000 x 40000 237 / 202, 2 x 5000 x 40000 334 / 206.  Direct, one to four
// waves of pairs above 256 tiles: 37 x 1000 x 33000 515 / 494, x 52000 795 / 765, 37 x 2048 x 130000 3411 / 3278, 37 x 4096 x 33000 1684 / 1590,
// x 60000 2994 / 2846, 20 x 1000 x 65536 881 / 851, 18 x 4096 x 65536 1622 / 1551.  Small CTAs of 32
// rows keep what they would do alone (1200 cycles per tile; 1 x 4096 x 40000 183).
// Beside other launches (the stages of a forward from host tensors) above 128 tiles, with either row sum: CTAs that take items leave an
// SM when none is left, and the next stage's come there.  us: 12 x 20000 4061 / 3908, 8 x 40000 5934 / 5588 (direct 6039 / 5817), 10 x 75600
// 16875 / 15673, 2 x 60000 3608 / 3157.  Where the link is the bound only the last stage counts: 24 x 8192 3196 / 3210, 12 x 13000 2679 / 2686
// (direct 2647 / 2664), 24 x 14000 5445 / 5430, and with fewer query tiles than half of T 24 x 7000 x 30000 7900 / 7930.
bool forward_walk_rest(int64_t n_sm, int64_t bh, int64_t Nq, int64_t Nkv, bool pnq, bool followed, const RowSplit& split) {
  const int64_t T = (Nkv + kTile - 1) / kTile, tiles = (Nq + kTile - 1) / kTile;
  if (followed && (T <= 128 || 2 * tiles < T)) return false;
  if ((T > kStaticTiles ? bh * tiles : (bh * tiles + n_sm - 1) / n_sm) * T > 0x7FFFFF00) return false;
  return !(split.R == 4 && split.pairs_256 == 0);
}

// The first `pairs` pairs of query tiles, counted over all heads.
int launch_forward_walk(int64_t n_sm, int64_t pairs, const void* q_codes, const void* q_scales, const void* k_codes, const void* k_scales,
                        const void* v_codes, const void* v_scales, void* o, int B, int H, int64_t Nq, int64_t Nkv,
                        float softmax_scale, unsigned flags, int* status, cudaStream_t stream) {
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
  p.scale_log2e = softmax_scale * 1.4426950408889634f;
  const bool uos = flags & MXATTN_FLAG_UOS, pnq = flags & MXATTN_FLAG_PNQ, f32 = flags & MXATTN_FLAG_OUT_FP32, take = takes<false>(p, n_sm);
  Kernel kern = nullptr;
#define PICK(U, P, F) if (uos == U && pnq == P && f32 == F) kern = take ? attention_walk_kernel<U, P, F, true> : attention_walk_kernel<U, P, F, false>;
  PICK(false, false, false) PICK(false, false, true) PICK(false, true, false) PICK(false, true, true)
  PICK(true, false, false) PICK(true, false, true) PICK(true, true, false) PICK(true, true, true)
#undef PICK
  return launch(kern, Lay<false>::kSmemBytes, p, take, n_sm, (int64_t)B * H, o, flags, stream);
}

}  // namespace mxattn
