// NVFP4 variant of the fused attention forward: the paper's comparison baseline "NVFP4" (Section 5.2) -- Q, K, V and
// the softmax tile in NVFP4 (E2M1 in blocks of 16, E4M3 block scale, fp32 tensor scale), nothing else changed -- run by
// the walking attention kernel (walk.cuh; Algorithm 2 with the quantizer exchanged), so that the two formats can be compared at
// equal kernel design.
#include "walk.cuh"

namespace mxattn {
namespace fwdnv {
using namespace walk;

template <bool kPnq, bool kOutF32, bool kTake>
__global__ void __launch_bounds__(kThreads, 1) attention_nvfp4_kernel(const Params p, const __grid_constant__ CUtensorMap out_map) {
  using L = Lay<true>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::kOffMisc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::kOffMisc + 8);
  volatile int* status_before = abort_flag + 2;
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  set_up<true>(smem, tid);
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
  play<true, false, kPnq, kOutF32, kTake>(p, out_map, smem, role, warp, lane);
  tc_fence_before();
  __syncthreads();
  if (tid == 0 && *abort_flag != 0) atomicCAS(p.status, 0, *abort_flag);
  if (warp == kIssuer1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(*tmem_slot) : "memory");
  }
}

constexpr int kScaleBytes = Lay<true>::kSF;    // per operand tile: two atoms (8 blocks of 16 per row)

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
  w->q_scales = off; off += align_up(bh * qt * kScaleBytes, 256);
  w->k_codes = off;  off += align_up(bh * kt * kTileCodeBytes, 256);
  w->k_scales = off; off += align_up(bh * kt * kScaleBytes, 256);
  w->v_codes = off;  off += align_up(bh * kt * kTileCodeBytes, 256);
  w->v_scales = off; off += align_up(bh * kt * kScaleBytes, 256);
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
  if (qt > 0x3FFFFFFF || kt > 0x3FFFFFFF || bh * qt > 0x7FFFFFFF) return MXATTN_EUNSUPPORTED;
  const int n_sm = sm_count();
  if (n_sm == 0) return MXATTN_ECUDA;
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  float* amax = reinterpret_cast<float*>(ws + w.amax);
  float* ts = reinterpret_cast<float*>(ws + w.tscale);
  if (launch_zero(reinterpret_cast<uint32_t*>(ws + w.status), (int64_t)(w.tscale - w.status) / 4, stream) != MXATTN_OK) return MXATTN_ECUDA;      // status word and tensor maxima
  const int rc = launch_nvfp4_operands(q, ws + w.q_codes, ws + w.q_scales, k, ws + w.k_codes, ws + w.k_scales, v, ws + w.v_codes, ws + w.v_scales,
                                       amax, ts, bh, Nq, Nkv, stream);
  if (rc != MXATTN_OK) return rc;
  Params p = {};
  p.q_codes = ws + w.q_codes; p.q_scales = ws + w.q_scales; p.k_codes = ws + w.k_codes; p.k_scales = ws + w.k_scales;
  p.v_codes = ws + w.v_codes; p.v_scales = ws + w.v_scales;
  p.ts_q = ts; p.ts_k = ts + bh; p.ts_v = ts + 2 * bh;
  p.status = reinterpret_cast<int*>(ws + w.status);
  p.Nq = Nq; p.Nkv = Nkv; p.q_tiles = (int)qt; p.kv_tiles = (int)kt;
  p.scale_log2e = softmax_scale * 1.4426950408889634f;
  const bool pnq = flags & MXATTN_FLAG_PNQ, f32 = flags & MXATTN_FLAG_OUT_FP32;
  // A CTA counts its tiles in 32 bits, and one that takes items from others may get them all: more come in several launches.
  const int64_t items = bh * qt, most = 0x7FFFFF00 / kt;
  for (int64_t first = 0; first < items; first += most) {
    p.first_item = (int)first;
    p.total_items = (int)(items - first < most ? items - first : most);
    const bool take = takes<true>(p, n_sm);
    Kernel kern = nullptr;
#define PICK(P, F) if (pnq == P && f32 == F) kern = take ? attention_nvfp4_kernel<P, F, true> : attention_nvfp4_kernel<P, F, false>;
    PICK(false, false) PICK(false, true) PICK(true, false) PICK(true, true)
#undef PICK
    const int rc2 = launch(kern, Lay<true>::kSmemBytes, p, take, n_sm, bh, o, flags, stream);
    if (rc2 != MXATTN_OK) return rc2;
  }
  return MXATTN_OK;
}

}  // namespace mxattn
