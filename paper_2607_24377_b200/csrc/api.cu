// C-ABI entry points that orchestrate the kernels: workspace carving, the operand launches (one to
// three) and the fused attention (one or two; paper Algorithm 2, lines 3-19), and the host-buffer
// end-to-end form.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <vector>

#include "common.cuh"
#include <nvtx3/nvToolsExt.h>      // header-only: the ranges cost nothing unless a profiling tool is attached

namespace mxattn {

// NVTX range for the lifetime of the object: the host-side enqueue of a launch or of a pipeline stage, so that a
// timeline shows which call and which stage queued which kernels.
struct TraceRange {
  explicit TraceRange(const char* name) { nvtxRangePushA(name); }
  ~TraceRange() { nvtxRangePop(); }
  TraceRange(const TraceRange&) = delete;
  TraceRange& operator=(const TraceRange&) = delete;
};

// Kernel launches of the last forward call.  Every launch counts itself for its thread; a forward call reports the difference.
static thread_local int t_launches = 0;
static std::atomic<int> g_last_launches{0};
void count_launch() { ++t_launches; }
struct CountedCall {
  const int before = t_launches;
  ~CountedCall() { g_last_launches.store(t_launches - before, std::memory_order_relaxed); }
};

static void* g_workspace = nullptr;
static size_t g_workspace_bytes = 0;

constexpr int kMaxDevices = 64;
static int current_device() {
  int dev = -1;
  return (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kMaxDevices) ? dev : -1;
}

int sm_count() {
  static std::atomic<int> n[kMaxDevices];
  const int dev = current_device();
  if (dev < 0) return 0;
  int v = n[dev].load(std::memory_order_relaxed);
  if (v == 0) {
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) return 0;
    n[dev].store(v, std::memory_order_relaxed);
  }
  return v;
}

// A kernel's attributes belong to a context, of which a device may have
// several (and a new one after a reset); numbers, unlike handles, are never used twice.
uint64_t current_context() {
  static std::atomic<void*> fn{nullptr};
  void* get = fn.load(std::memory_order_acquire);
  if (!get) {
    cudaDriverEntryPointQueryResult found;
    if (cudaGetDriverEntryPoint("cuCtxGetId", &get, cudaEnableDefault, &found) != cudaSuccess || found != cudaDriverEntryPointSuccess || !get) return 0;
    fn.store(get, std::memory_order_release);
  }
  unsigned long long id = 0;
  return reinterpret_cast<PFN_cuCtxGetId>(get)(nullptr, &id) == CUDA_SUCCESS ? (uint64_t)id : 0;
}

bool ensure_attribute(const void* kern, cudaFuncAttribute attribute, int value) {
  // one entry per kernel (a few dozen): the contexts in which it has been set, each at its number mod 16
  struct Entry { std::atomic<const void*> kern; std::atomic<uint64_t> contexts[16]; };
  static Entry table[128];
  const uint64_t context = current_context();
  if (context != 0) {
    for (Entry& e : table) {
      const void* k = e.kern.load(std::memory_order_acquire);
      if (k == nullptr && e.kern.compare_exchange_strong(k, kern, std::memory_order_acq_rel)) k = kern;
      if (k != kern) continue;                        // (a failed exchange left another thread's kernel in k)
      std::atomic<uint64_t>& at = e.contexts[context & 15];
      if (at.load(std::memory_order_acquire) == context) return true;
      if (cudaFuncSetAttribute(kern, attribute, value) != cudaSuccess) return false;
      at.store(context, std::memory_order_release);
      return true;
    }
  }
  return cudaFuncSetAttribute(kern, attribute, value) == cudaSuccess;
}
bool ensure_dynamic_smem(const void* kern, int bytes) { return ensure_attribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); }

struct WorkspaceLayout {
  size_t q_codes, q_scales, k_codes, k_scales, v_codes, v_scales, status, total;
};

static inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

static bool carve(int B, int H, int64_t Nq, int64_t Nkv, int d, WorkspaceLayout* w) {
  if (B <= 0 || H <= 0 || Nq <= 0 || Nkv <= 0 || d != kHeadDim) return false;
  const size_t bh = (size_t)B * H;
  const size_t qt = (size_t)((Nq + kTile - 1) / kTile), kt = (size_t)((Nkv + kTile - 1) / kTile);
  size_t off = 0;
  w->status = off;   off += 256;
  w->q_codes = off;  off += align_up(bh * qt * kTileCodeBytes, 256);
  w->q_scales = off; off += align_up(bh * qt * kTileScaleBytes, 256);
  w->k_codes = off;  off += align_up(bh * kt * kTileCodeBytes, 256);
  w->k_scales = off; off += align_up(bh * kt * kTileScaleBytes, 256);
  w->v_codes = off;  off += align_up(bh * kt * kTileCodeBytes, 256);
  w->v_scales = off; off += align_up(bh * kt * kTileScaleBytes, 256);
  w->total = off;
  return true;
}

// `qstream` / `qdone`: if given, the quantize launches go to `qstream`, `qdone` is recorded behind them and
// the attention launch on `stream` waits for it (the host pipeline uses this to quantize the next stage's
// operands while the current stage's attention kernel drains).  `followed`: other attention launches run at the same time.
static int forward_ws(const void* q, const void* k, const void* v, void* o, int B, int H, int64_t Nq,
                      int64_t Nkv, int d, float softmax_scale, unsigned flags, void* workspace,
                      size_t workspace_bytes, cudaStream_t stream, void* dump = nullptr,
                      cudaStream_t qstream = nullptr, cudaEvent_t qdone = nullptr, void* profile = nullptr, bool followed = false) {
  if (!q || !k || !v || !o) return MXATTN_EINVAL;
  if (B <= 0 || H <= 0 || Nq <= 0 || Nkv <= 0) return MXATTN_EINVAL;
  if (flags & ~(unsigned)(MXATTN_FLAG_UOS | MXATTN_FLAG_PNQ | MXATTN_FLAG_OUT_FP32 | MXATTN_FLAG_HADAMARD)) return MXATTN_EINVAL;
  if (!(softmax_scale > 0.0f) || !(softmax_scale < 3.0e38f)) return MXATTN_EINVAL;
  if (d != kHeadDim) return MXATTN_EUNSUPPORTED;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o)) return MXATTN_EALIGN;
  WorkspaceLayout w;
  if (!carve(B, H, Nq, Nkv, d, &w)) return MXATTN_EUNSUPPORTED;
  if (!workspace || workspace_bytes < w.total) return MXATTN_EWORKSPACE;
  if (!aligned16(workspace)) return MXATTN_EALIGN;
  CountedCall counted;
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  const int mode = (flags & MXATTN_FLAG_UOS) ? MXATTN_MODE_UOS : MXATTN_MODE_OCP;
  const int qk_mode = mode | ((flags & MXATTN_FLAG_HADAMARD) ? MXATTN_MODE_HADAMARD : 0);   // Algorithm 2 lines 1-2
  const int64_t bh = (int64_t)B * H;
  cudaStream_t qs = qstream ? qstream : stream;
  // Algorithm 2 lines 3-5: Q-hat, K-hat (blocks along d), V-hat (blocks along tokens); the launch clears the status word
  {
    TraceRange tr("mxattn quantize Q K V");
    const int rc = launch_quantize_qkv(q, ws + w.q_codes, ws + w.q_scales, k, ws + w.k_codes, ws + w.k_scales, v, ws + w.v_codes,
                                       ws + w.v_scales, bh, Nq, Nkv, qk_mode, reinterpret_cast<int*>(ws + w.status), qs);
    if (rc != MXATTN_OK) return rc;
  }
  if (qstream) {
    if (cudaEventRecord(qdone, qstream) != cudaSuccess || cudaStreamWaitEvent(stream, qdone, 0) != cudaSuccess) return MXATTN_ECUDA;
  }
  // lines 6-19
  TraceRange tr("mxattn attention");
  return launch_forward(ws + w.q_codes, ws + w.q_scales, ws + w.k_codes, ws + w.k_scales, ws + w.v_codes,
                        ws + w.v_scales, o, B, H, Nq, Nkv, softmax_scale, flags,
                        reinterpret_cast<int*>(ws + w.status), stream, dump, profile, followed);
}

}  // namespace mxattn

using namespace mxattn;

extern "C" size_t mxattn_forward_workspace_bytes(int B, int H, int64_t Nq, int64_t Nkv, int d) {
  WorkspaceLayout w;
  return carve(B, H, Nq, Nkv, d, &w) ? w.total : 0;
}

extern "C" int mxattn_set_workspace(void* dev_ptr, size_t bytes) {
  if (dev_ptr && !aligned16(dev_ptr)) return MXATTN_EALIGN;
  g_workspace = dev_ptr;
  g_workspace_bytes = dev_ptr ? bytes : 0;
  return MXATTN_OK;
}

extern "C" int mxattn_forward(const void* q, const void* k, const void* v, void* o, int B, int H,
                              int64_t Nq, int64_t Nkv, int d, float softmax_scale, unsigned flags,
                              void* stream) {
  return forward_ws(q, k, v, o, B, H, Nq, Nkv, d, softmax_scale, flags, g_workspace, g_workspace_bytes,
                    (cudaStream_t)stream);
}

extern "C" int mxattn_forward_ws(const void* q, const void* k, const void* v, void* o, int B, int H,
                                 int64_t Nq, int64_t Nkv, int d, float softmax_scale, unsigned flags,
                                 void* workspace, size_t workspace_bytes, void* stream) {
  return forward_ws(q, k, v, o, B, H, Nq, Nkv, d, softmax_scale, flags, workspace, workspace_bytes,
                    (cudaStream_t)stream);
}

extern "C" int mxattn_rowsum_diagnostic(const void* q, const void* k, void* out, int B, int H, int64_t Nq,
                                        int64_t Nkv, int d, float softmax_scale, unsigned flags,
                                        void* workspace, size_t workspace_bytes, void* stream_) {
  cudaStream_t stream = (cudaStream_t)stream_;
  if (!q || !k || !out) return MXATTN_EINVAL;
  if (B <= 0 || H <= 0 || Nq <= 0 || Nkv <= 0) return MXATTN_EINVAL;
  if (flags & ~(unsigned)(MXATTN_FLAG_UOS | MXATTN_FLAG_HADAMARD)) return MXATTN_EINVAL;
  if (!(softmax_scale > 0.0f) || !(softmax_scale < 3.0e38f)) return MXATTN_EINVAL;
  if (d != kHeadDim) return MXATTN_EUNSUPPORTED;
  if (!aligned16(q) || !aligned16(k) || !aligned16(out)) return MXATTN_EALIGN;
  WorkspaceLayout w;
  if (!carve(B, H, Nq, Nkv, d, &w)) return MXATTN_EUNSUPPORTED;
  if (!workspace || workspace_bytes < w.total) return MXATTN_EWORKSPACE;
  if (!aligned16(workspace)) return MXATTN_EALIGN;
  CountedCall counted;
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  const int mode = (flags & MXATTN_FLAG_UOS) ? MXATTN_MODE_UOS : MXATTN_MODE_OCP;
  const int qk_mode = mode | ((flags & MXATTN_FLAG_HADAMARD) ? MXATTN_MODE_HADAMARD : 0);
  const int64_t bh = (int64_t)B * H;
  const int rc = launch_quantize_qkv(q, ws + w.q_codes, ws + w.q_scales, k, ws + w.k_codes, ws + w.k_scales, nullptr, nullptr, nullptr,
                                     bh, Nq, Nkv, qk_mode, reinterpret_cast<int*>(ws + w.status), stream);
  if (rc != MXATTN_OK) return rc;
  return launch_rowsum_diag(ws + w.q_codes, ws + w.q_scales, ws + w.k_codes, ws + w.k_scales, out, B, H, Nq, Nkv,
                            softmax_scale, (flags & MXATTN_FLAG_UOS) ? kRuleUos : kRuleOcp,
                            reinterpret_cast<int*>(ws + w.status), stream);
}

extern "C" size_t mxattn_forward_debug_dump_bytes(int B, int H, int64_t Nq, int64_t Nkv, int d) {
  if (B <= 0 || H <= 0 || Nq <= 0 || Nkv <= 0 || d != kHeadDim) return 0;
  return forward_dump_bytes(B, H, Nq, Nkv);
}

extern "C" int mxattn_forward_debug_dump(const void* q, const void* k, const void* v, void* o, int B, int H,
                                         int64_t Nq, int64_t Nkv, int d, float softmax_scale, unsigned flags,
                                         void* workspace, size_t workspace_bytes, void* dump,
                                         size_t dump_bytes, void* stream) {
  if (!dump) return MXATTN_EINVAL;
  if (!(flags & MXATTN_FLAG_OUT_FP32)) return MXATTN_EINVAL;
  if (B <= 0 || H <= 0 || Nq <= 0 || Nkv <= 0) return MXATTN_EINVAL;
  if (d != kHeadDim) return MXATTN_EUNSUPPORTED;
  const size_t need = forward_dump_bytes(B, H, Nq, Nkv);
  if (need > ((size_t)1 << 30)) return MXATTN_EUNSUPPORTED;      // a debugging aid for small problems
  if (dump_bytes < need) return MXATTN_EWORKSPACE;
  if (!aligned16(dump)) return MXATTN_EALIGN;
  return forward_ws(q, k, v, o, B, H, Nq, Nkv, d, softmax_scale, flags, workspace, workspace_bytes,
                    (cudaStream_t)stream, dump);
}

extern "C" size_t mxattn_forward_cycle_profile_bytes(int B, int H, int64_t Nq, int64_t Nkv, int d) {
  if (B <= 0 || H <= 0 || Nq <= 0 || Nkv <= 0 || d != kHeadDim) return 0;
  return forward_profile_bytes(B, H, Nq, Nkv);
}

extern "C" int mxattn_forward_cycle_profile(const void* q, const void* k, const void* v, void* o, int B, int H,
                                            int64_t Nq, int64_t Nkv, int d, float softmax_scale, unsigned flags,
                                            void* workspace, size_t workspace_bytes, void* profile,
                                            size_t profile_bytes, void* stream) {
  if (!profile) return MXATTN_EINVAL;
  if (flags != (unsigned)(MXATTN_FLAG_UOS | MXATTN_FLAG_PNQ)) return MXATTN_EINVAL;
  if (B <= 0 || H <= 0 || Nq <= 0 || Nkv <= 0) return MXATTN_EINVAL;
  if (d != kHeadDim) return MXATTN_EUNSUPPORTED;
  if (profile_bytes < forward_profile_bytes(B, H, Nq, Nkv)) return MXATTN_EWORKSPACE;
  if (!aligned16(profile)) return MXATTN_EALIGN;
  return forward_ws(q, k, v, o, B, H, Nq, Nkv, d, softmax_scale, flags, workspace, workspace_bytes,
                    (cudaStream_t)stream, nullptr, nullptr, nullptr, profile);
}

extern "C" int mxattn_forward_prequantized(const void* q_codes, const void* q_scales, const void* k_codes,
                                           const void* k_scales, const void* v_codes, const void* v_scales,
                                           void* o, int B, int H, int64_t Nq, int64_t Nkv, int d,
                                           float softmax_scale, unsigned flags, void* status, void* stream) {
  if (!q_codes || !q_scales || !k_codes || !k_scales || !v_codes || !v_scales || !o || !status) return MXATTN_EINVAL;
  if (B <= 0 || H <= 0 || Nq <= 0 || Nkv <= 0) return MXATTN_EINVAL;
  if (flags & ~(unsigned)(MXATTN_FLAG_UOS | MXATTN_FLAG_PNQ | MXATTN_FLAG_OUT_FP32 | MXATTN_FLAG_HADAMARD)) return MXATTN_EINVAL;
  if (!(softmax_scale > 0.0f) || !(softmax_scale < 3.0e38f)) return MXATTN_EINVAL;
  if (d != kHeadDim) return MXATTN_EUNSUPPORTED;
  if (!aligned16(q_codes) || !aligned16(q_scales) || !aligned16(k_codes) || !aligned16(k_scales) ||
      !aligned16(v_codes) || !aligned16(v_scales) || !aligned16(o) || !aligned16(status))
    return MXATTN_EALIGN;
  CountedCall counted;
  return launch_forward(q_codes, q_scales, k_codes, k_scales, v_codes, v_scales, o, B, H, Nq, Nkv,
                        softmax_scale, flags, static_cast<int*>(status), (cudaStream_t)stream);
}

// ---------------------------------------------------------------------------------------------
// Host-buffer form.  Heads are independent, so the call is pipelined in stages of one or more heads over five
// streams -- the caller's and four helper streams (copies in, quantization, a second attention stream, copies out):
// host->device copies of the next stage and the device->host copy of the previous one overlap the kernels of the
// current stage (PCIe is full duplex).  The helper streams and the events are created on first use, once per
// device, and kept for the life of the process; no device memory is allocated.
struct HostPipe {
  cudaStream_t in = nullptr, quant = nullptr, out = nullptr, attn = nullptr;
  std::vector<cudaEvent_t> ev;
};
static HostPipe g_pipe[64];

static HostPipe* host_pipe(size_t n_events) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  HostPipe& hp = g_pipe[dev];
  if (!hp.in && cudaStreamCreateWithFlags(&hp.in, cudaStreamNonBlocking) != cudaSuccess) return nullptr;
  if (!hp.out && cudaStreamCreateWithFlags(&hp.out, cudaStreamNonBlocking) != cudaSuccess) return nullptr;
  if (!hp.quant) {
    // the quantize launches are short and feed the next attention launch: they go first when SMs free up
    int lo = 0, hi = 0;
    if (cudaDeviceGetStreamPriorityRange(&lo, &hi) != cudaSuccess) return nullptr;
    if (cudaStreamCreateWithPriority(&hp.quant, cudaStreamNonBlocking, hi) != cudaSuccess) return nullptr;
  }
  if (!hp.attn && cudaStreamCreateWithFlags(&hp.attn, cudaStreamNonBlocking) != cudaSuccess) return nullptr;
  while (hp.ev.size() < n_events) {
    cudaEvent_t e;
    if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) return nullptr;
    hp.ev.push_back(e);
  }
  return &hp;
}

namespace mxattn {
// First heads of the pipeline stages of mxattn_forward_host; the last entry is bh.  last_alone: the attention of earlier
// stages is done when the last stage's operands arrive.  The link bounds the call (a head of N tokens arrives in 14 us per
// 1000 tokens, and its attention takes less than that below some 50000 tokens), and a stage costs it about 20 us: three
// copies of some 6 us each on top of their bytes.  So there should be few stages.
//   - Nothing hides the last stage's attention and copy out, so that stage is small, and the stages before it grow by
//     the ratio at which a stage's attention and copy out are just done when the smaller one behind it has arrived
//     (55 GB/s in and out, attention at 1.6 PFLOP/s).  It is kept between 1.5 and 3, beyond which nothing is gained.
//   - Where the copies in are the bound the first stages may be large: they start at an eighth of the heads and double.
//     Where the copies out weigh as much (Nkv small) or the attention does (long sequences) the first stage has to be
//     small, and a stage that grows leaves the other two idle while it arrives: equal ones then, of the size at which
//     the wait for one stage is what all stages' fixed cost is.
//   - No stage is below 2.5 MB in, which is 45 us of the link, unless the call is.
// Against one head followed by stages of equal size, us: 24 x 8192 3310 -> 3249 (copying in alone takes 2731), 40 x 4096
// 2858 -> 2712 (2280), 160 x 5000 13170 -> 12230, 160 x 300 1134 -> 912, 2 x 1024 (one stage now) 195 -> 164, 12 x 20000
// 4084 -> 4011; 40 heads of 10000 x 512 3024 -> 3023, of 75600 x 512 18460 -> 18060.
//   - Up to eight heads of which one fits the SMs and two do not (256 query rows per CTA): a stage of two leaves a second
//     wave, which is late when the last stage follows right behind.  There the sizes grow by the ratio itself, kept above
//     1.25, and not by what it rounds to, and the larger stages come first (2, 1, 1 instead of 1, 2, 1).  Direct row sum /
//     PNQ, 21070 x 21070: 4 heads 1811 / 1735 -> 1653 / 1651, 6 heads 2447 / 2390 -> 2286 / 2321, 8 heads 3159 / 3076 -> 2998 / 3037;
//     28000 x 28000, 4 heads 2420 / 2287 -> 2149 / 2134.  Where two heads fit (18000 x 18000) it is 3 to 8 % slower, from
//     twelve heads on as fast.
// first[0 .. stages] receives the first heads (room for bh + 1); the number of stages is returned.
size_t host_stages(size_t bh, int64_t Nq, int64_t Nkv, size_t in_bytes_per_head, size_t out_bytes_per_head, int n_sm, size_t* first, bool* last_alone) {
  const double t_in = (double)in_bytes_per_head / 55e9, t_out = (double)out_bytes_per_head / 55e9;
  const double t_attn = 4.0 * (double)Nq * (double)Nkv * kHeadDim / 1.6e15;
  const double ratio = 1.1 * t_in / (t_out + t_attn);
  const size_t least = (size_t)(2.5e6 / (double)in_bytes_per_head) + 1;
  const double t_other = std::max(t_out, t_attn);
  const bool in_bound = t_in > 1.5 * t_other;
  const int64_t ctas = (Nq + 2 * kTile - 1) / (2 * kTile);       // of a head
  const bool late = in_bound && ratio < 1.5 && bh <= 8 && ctas <= n_sm && 2 * ctas > n_sm;
  const double shrink = std::min(3.0, std::max(late ? 1.25 : 1.5, ratio));
  const size_t most = in_bound ? bh : std::max(least, (size_t)std::ceil(std::sqrt((double)bh * 20e-6 / t_other)));
  *last_alone = in_bound || bh <= least;
  size_t next_head = in_bound ? std::max(least, bh / 8) : least, next_tail = least;
  double size_tail = (double)least;
  std::vector<size_t> head, tail;
  for (size_t left = bh; left > 0;) {
    const bool at_head = next_head < next_tail && !(late && left <= next_tail);
    size_t& next = at_head ? next_head : next_tail;
    // what would be left over and too small for a stage of its own joins this one
    const size_t n = 4 * left < 5 * next || left < next + least ? left : next;
    (at_head ? head : tail).push_back(n);
    if (!at_head) size_tail = shrink * (late ? size_tail : (double)n);
    next = std::min(most, at_head ? 2 * n : (size_t)std::lround(size_tail));
    left -= n;
  }
  size_t stages = 0;
  first[0] = 0;
  auto add = [&](size_t n) { first[stages + 1] = first[stages] + n; ++stages; };
  for (size_t n : head) add(n);
  for (size_t k = tail.size(); k-- > 0;) add(tail[k]);
  return stages;
}
}  // namespace mxattn

extern "C" size_t mxattn_forward_host_arena_bytes(int B, int H, int64_t Nq, int64_t Nkv, int d, unsigned flags) {
  WorkspaceLayout w;
  if (!carve(1, 1, Nq, Nkv, d, &w) || B <= 0 || H <= 0) return 0;     // one workspace slice per head
  const size_t bh = (size_t)B * H;
  const size_t qb = align_up(bh * (size_t)Nq * d * 2, 256), kb = align_up(bh * (size_t)Nkv * d * 2, 256);
  const size_t ob = align_up(bh * (size_t)Nq * d * ((flags & MXATTN_FLAG_OUT_FP32) ? 4 : 2), 256);
  return qb + 2 * kb + ob + bh * w.total;
}

extern "C" int mxattn_forward_host(const void* q_host, const void* k_host, const void* v_host, void* o_host,
                                   int B, int H, int64_t Nq, int64_t Nkv, int d, float softmax_scale,
                                   unsigned flags, void* device_arena, size_t arena_bytes, void* stream_) {
  if (!q_host || !k_host || !v_host || !o_host) return MXATTN_EINVAL;
  const size_t need = mxattn_forward_host_arena_bytes(B, H, Nq, Nkv, d, flags);
  if (need == 0) return (d != kHeadDim) ? MXATTN_EUNSUPPORTED : MXATTN_EINVAL;
  if (!device_arena || arena_bytes < need) return MXATTN_EWORKSPACE;
  if (!aligned16(device_arena)) return MXATTN_EALIGN;
  cudaStream_t stream = (cudaStream_t)stream_;
  const size_t bh = (size_t)B * H;
  const size_t osz = (flags & MXATTN_FLAG_OUT_FP32) ? 4 : 2;
  const size_t qh = (size_t)Nq * d * 2, kh = (size_t)Nkv * d * 2, oh = (size_t)Nq * d * osz;   // bytes per head
  WorkspaceLayout w;
  carve(1, 1, Nq, Nkv, d, &w);
  uint8_t* a = static_cast<uint8_t*>(device_arena);
  uint8_t* dq = a;
  uint8_t* dk = dq + align_up(bh * qh, 256);
  uint8_t* dv = dk + align_up(bh * kh, 256);
  uint8_t* dout = dv + align_up(bh * kh, 256);
  uint8_t* ws = dout + align_up(bh * oh, 256);
  bool last_alone;
  std::vector<size_t> first_head(bh + 1);
  const size_t stages = host_stages(bh, Nq, Nkv, qh + 2 * kh, oh, sm_count(), first_head.data(), &last_alone);
  HostPipe* hp = host_pipe(3 * stages + 2);
  if (!hp) return MXATTN_ECUDA;
  cudaEvent_t* ev = hp->ev.data();
  bool fail = false;
  auto ck = [&](cudaError_t e) { if (e != cudaSuccess) fail = true; };
  ck(cudaEventRecord(ev[3 * stages], stream));                   // work already queued on the caller's stream comes first
  ck(cudaStreamWaitEvent(hp->in, ev[3 * stages], 0));
  ck(cudaStreamWaitEvent(hp->attn, ev[3 * stages], 0));
  CountedCall counted;
  int rc = MXATTN_OK;
  for (size_t st = 0; st < stages && !fail && rc == MXATTN_OK; ++st) {
    TraceRange tr("mxattn host stage");
    const size_t i = first_head[st], n = first_head[st + 1] - i;  // heads of the stage; heads are contiguous in memory
    // attention launches alternate between the caller's stream and one of the pipeline's, so that the CTAs of a
    // stage start on the SMs the previous stage's last CTAs leave (no tail, no launch gap between stages)
    cudaStream_t as = (st & 1) ? hp->attn : stream;
    ck(cudaMemcpyAsync(dq + i * qh, static_cast<const char*>(q_host) + i * qh, n * qh, cudaMemcpyHostToDevice, hp->in));
    ck(cudaMemcpyAsync(dk + i * kh, static_cast<const char*>(k_host) + i * kh, n * kh, cudaMemcpyHostToDevice, hp->in));
    ck(cudaMemcpyAsync(dv + i * kh, static_cast<const char*>(v_host) + i * kh, n * kh, cudaMemcpyHostToDevice, hp->in));
    ck(cudaEventRecord(ev[3 * st], hp->in));
    ck(cudaStreamWaitEvent(hp->quant, ev[3 * st], 0));
    // the stage's workspace starts at its first head's slice (n slices are at least as large as one workspace for
    // n heads); its operands are quantized on a stream of their own, behind the copies and ahead of the attention
    // launch, so that they fill the SMs the previous stage's attention kernel frees as it drains
    rc = forward_ws(dq + i * qh, dk + i * kh, dv + i * kh, dout + i * oh, 1, (int)n, Nq, Nkv, d, softmax_scale, flags,
                    ws + i * w.total, n * w.total, as, nullptr, hp->quant, ev[3 * st + 1], nullptr, st + 1 < stages || !last_alone);
    ck(cudaEventRecord(ev[3 * st + 2], as));
    ck(cudaStreamWaitEvent(hp->out, ev[3 * st + 2], 0));
    ck(cudaMemcpyAsync(static_cast<char*>(o_host) + i * oh, dout + i * oh, n * oh, cudaMemcpyDeviceToHost, hp->out));
  }
  ck(cudaEventRecord(ev[3 * stages + 1], hp->out));
  ck(cudaStreamWaitEvent(stream, ev[3 * stages + 1], 0));
  // everything enqueued so far must drain before returning, also on an error path
  ck(cudaStreamSynchronize(hp->in));
  ck(cudaStreamSynchronize(hp->quant));
  ck(cudaStreamSynchronize(stream));
  ck(cudaStreamSynchronize(hp->attn));
  ck(cudaStreamSynchronize(hp->out));
  if (rc != MXATTN_OK) return rc;
  if (fail) return MXATTN_ECUDA;
  // one status word per stage, at the start of the workspace slice of the stage's first head
  std::vector<int> word(bh, 0);
  if (cudaMemcpy2D(word.data(), sizeof(int), ws, w.total, sizeof(int), bh, cudaMemcpyDeviceToHost) != cudaSuccess) return MXATTN_ECUDA;
  for (size_t st = 0; st < stages; ++st)
    if (word[first_head[st]]) return MXATTN_ETIMEOUT;
  return MXATTN_OK;
}

// ---------------------------------------------------------------------------------------------
// Forward pass for callers that cannot allocate device memory.
//
// Some hosts of this library may not call cudaMalloc at all: code running inside another
// framework's memory plan where every byte is pre-assigned, plugins loaded into a process that
// forbids allocation after start-up, or latency-critical loops where an allocator call (and the
// implicit synchronization it can bring) is not acceptable.  For them the scratch that
// mxattn_forward needs lives in the library image itself: a fixed array in device global memory,
// present on every GPU that loads the library for as long as the process lives.
static __device__ __align__(256) unsigned char g_static_scratch[MXATTN_STATIC_SCRATCH_BYTES];

// In host code `g_static_scratch` is only a handle for the runtime, not a device address, so the
// address is looked up once per device (with that device current) and cached.
static void* g_static_scratch_ptr[kMaxDevices] = {nullptr};

extern "C" int mxattn_forward_static(const void* q, const void* k, const void* v, void* o, int B, int H,
                                     int64_t Nq, int64_t Nkv, int d, float softmax_scale, unsigned flags,
                                     void* stream) {
  const size_t need = mxattn_forward_workspace_bytes(B, H, Nq, Nkv, d);
  if (need == 0) return (d != kHeadDim) ? MXATTN_EUNSUPPORTED : MXATTN_EINVAL;
  if (need > (size_t)MXATTN_STATIC_SCRATCH_BYTES) return MXATTN_ESCRATCH_TOO_SMALL;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return MXATTN_ECUDA;
  if (!g_static_scratch_ptr[dev]) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess || !ptr) return MXATTN_ECUDA;
    g_static_scratch_ptr[dev] = ptr;
  }
  return forward_ws(q, k, v, o, B, H, Nq, Nkv, d, softmax_scale, flags, g_static_scratch_ptr[dev],
                    (size_t)MXATTN_STATIC_SCRATCH_BYTES, (cudaStream_t)stream);
}

extern "C" size_t mxattn_forward_bf16_workspace_bytes(int B, int H, int64_t Nq, int64_t Nkv, int d) {
  if (B <= 0 || H <= 0 || Nq <= 0 || Nkv <= 0 || d != kHeadDim) return 0;
  return bf16_workspace_bytes(B, H, Nq, Nkv);
}

extern "C" int mxattn_forward_bf16(const void* q, const void* k, const void* v, void* o, int B, int H, int64_t Nq,
                                   int64_t Nkv, int d, float softmax_scale, unsigned flags, void* workspace,
                                   size_t workspace_bytes, void* stream) {
  if (!q || !k || !v || !o) return MXATTN_EINVAL;
  if (B <= 0 || H <= 0 || Nq <= 0 || Nkv <= 0) return MXATTN_EINVAL;
  if (flags & ~(unsigned)MXATTN_FLAG_OUT_FP32) return MXATTN_EINVAL;
  if (!(softmax_scale > 0.0f) || !(softmax_scale < 3.0e38f)) return MXATTN_EINVAL;
  if (d != kHeadDim) return MXATTN_EUNSUPPORTED;
  if (!workspace) return MXATTN_EWORKSPACE;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o) || !aligned16(workspace)) return MXATTN_EALIGN;
  CountedCall counted;
  return launch_forward_bf16(q, k, v, o, B, H, Nq, Nkv, softmax_scale, flags, workspace, workspace_bytes,
                             (cudaStream_t)stream);
}

extern "C" size_t mxattn_forward_nvfp4_workspace_bytes(int B, int H, int64_t Nq, int64_t Nkv, int d) {
  if (B <= 0 || H <= 0 || Nq <= 0 || Nkv <= 0 || d != kHeadDim) return 0;
  return nvfp4_workspace_bytes(B, H, Nq, Nkv);
}

extern "C" int mxattn_forward_nvfp4(const void* q, const void* k, const void* v, void* o, int B, int H, int64_t Nq,
                                    int64_t Nkv, int d, float softmax_scale, unsigned flags, void* workspace,
                                    size_t workspace_bytes, void* stream) {
  if (!q || !k || !v || !o) return MXATTN_EINVAL;
  if (B <= 0 || H <= 0 || Nq <= 0 || Nkv <= 0) return MXATTN_EINVAL;
  if (flags & ~(unsigned)(MXATTN_FLAG_PNQ | MXATTN_FLAG_OUT_FP32)) return MXATTN_EINVAL;
  if (!(softmax_scale > 0.0f) || !(softmax_scale < 3.0e38f)) return MXATTN_EINVAL;
  if (d != kHeadDim) return MXATTN_EUNSUPPORTED;
  if (!workspace) return MXATTN_EWORKSPACE;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o) || !aligned16(workspace)) return MXATTN_EALIGN;
  CountedCall counted;
  return launch_forward_nvfp4(q, k, v, o, B, H, Nq, Nkv, softmax_scale, flags, workspace, workspace_bytes,
                              (cudaStream_t)stream);
}

extern "C" int mxattn_device_status(const void* workspace, int* host_out, void* stream) {
  if (!workspace || !host_out) return MXATTN_EINVAL;
  if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return MXATTN_ECUDA;
  if (cudaMemcpy(host_out, workspace, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return MXATTN_ECUDA;
  return MXATTN_OK;
}

extern "C" int mxattn_selftest_bounded_wait(void* status, int64_t limit_cycles, void* stream) {
  if (!status || limit_cycles <= 0 || limit_cycles > 2000000000LL) return MXATTN_EINVAL;
  if (!aligned16(status)) return MXATTN_EALIGN;
  return launch_bounded_wait_selftest(static_cast<int*>(status), (long long)limit_cycles, (cudaStream_t)stream);
}

extern "C" int mxattn_selftest_pair_abandon(void* status, int64_t limit_cycles, int meetings, void* stream) {
  if (!status || limit_cycles <= 0 || limit_cycles > 2000000000LL || meetings <= 0 || meetings > 100000) return MXATTN_EINVAL;
  if (!aligned16(status)) return MXATTN_EALIGN;
  return launch_pair_abandon_selftest(static_cast<int*>(status), (long long)limit_cycles, meetings, (cudaStream_t)stream);
}

extern "C" int mxattn_selftest_exp2_codes(void* status, void* stream) {
  if (!status) return MXATTN_EINVAL;
  if (!aligned16(status)) return MXATTN_EALIGN;
  return launch_exp2_codes_selftest(static_cast<int*>(status), (cudaStream_t)stream);
}

extern "C" int mxattn_last_launch_count(void) { return g_last_launches.load(std::memory_order_relaxed); }

extern "C" const char* mxattn_strerror(int status) {
  switch (status) {
    case MXATTN_OK: return "ok";
    case MXATTN_EINVAL: return "invalid argument";
    case MXATTN_EUNSUPPORTED: return "unsupported shape";
    case MXATTN_EALIGN: return "pointer not 16-byte aligned";
    case MXATTN_EWORKSPACE: return "workspace missing or too small";
    case MXATTN_ECUDA: return "CUDA runtime error";
    case MXATTN_ETIMEOUT: return "device-side bounded wait expired";
    case MXATTN_ESCRATCH_TOO_SMALL:
      return "problem needs more scratch than the built-in static array holds (MXATTN_STATIC_SCRATCH_BYTES); "
             "use mxattn_forward_ws with caller-provided memory";
    default: return "unknown status";
  }
}
