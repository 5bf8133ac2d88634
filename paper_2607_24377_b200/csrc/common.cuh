// Device helpers shared by the quantize and attention kernels (sm_100a only).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <cuda.h>              // CUtensorMap and the enumerations of its encoder (types only: nothing links libcuda)
#include <cudaTypedefs.h>

#include "../../include/mxattn.h"

namespace mxattn {

constexpr int kBlock = 32;       // elements per MXFP4 block (paper Section 2)
constexpr int kHeadDim = 128;    // supported head dimension
constexpr int kTile = 128;       // rows per operand tile and keys per KV tile (B_c)
constexpr int kTileCodeBytes = kTile * kHeadDim / 2;   // 8192
constexpr int kTileScaleBytes = kTile * kHeadDim / kBlock;  // 512

// Shared exponent e of a block whose maximum magnitude has fp32 bit pattern `u` (sign cleared).
// OCP: floor(log2 M) - 2 (paper Eq. 5).  UOS: ceil(log2(M / 7.25)) (paper Eq. 13, Algorithm 1).
// With M = mu * 2^E, mu in [1, 2): 7.25 = 1.8125 * 2^2, so the ceiling equals E - 2 when
// mu <= 1.8125 and E - 1 otherwise; in fp32 bits "mu > 1.8125" is "mantissa field > 0x680000".
// log2 is never evaluated.  M == 0 gives e = 0 (sigma = 1); e is clamped to [-127, 127]
// (subnormal M always clamps to -127; the upper clamp cannot be reached by a finite fp32).
__device__ __forceinline__ int shared_exponent(uint32_t u, bool uos) {
  if (u == 0u) return 0;
  const int eb = (int)(u >> 23);
  if (eb == 0) return -127;
  const int raise = (uos && (u & 0x7FFFFFu) > 0x680000u) ? 1 : 0;
  const int e = eb - 129 + raise;
  return e < -127 ? -127 : e;
}

// The ceiling family e = ceil(log2(M / q)) for an arbitrary boundary q > 0 (paper Eq. 7; TFS is q = 6,
// OAS at block 32 is q = 7, UOS is q = 7.25): with M = mu * 2^E and q = mu_q * 2^Eq,
// e = E - Eq + [mu > mu_q], decided on the bit patterns.  `q_bits` is the fp32 pattern of q.
__device__ __forceinline__ int shared_exponent_ceil(uint32_t u, uint32_t q_bits) {
  if (u == 0u) return 0;
  const int eb = (int)(u >> 23);
  if (eb == 0) return -127;
  const int e = eb - (int)(q_bits >> 23) + (((u & 0x7FFFFFu) > (q_bits & 0x7FFFFFu)) ? 1 : 0);
  return e < -127 ? -127 : (e > 127 ? 127 : e);
}

// Rule word used by the quantize kernels: 0 = OCP floor rule, otherwise the fp32 bit pattern of the
// ceiling-family boundary q (UOS: 7.25f).  For q = 7.25 this is exactly shared_exponent(u, true).
constexpr uint32_t kRuleOcp = 0u;
constexpr uint32_t kRuleUos = 0x40E80000u;   // 7.25f
__device__ __forceinline__ int shared_exponent_rule(uint32_t u, uint32_t rule) {
  return rule == kRuleOcp ? shared_exponent(u, false) : shared_exponent_ceil(u, rule);
}

// 2^-e as fp32 for e in [-127, 126] (exact, normal number).
__device__ __forceinline__ float pow2_neg(int e) {
  return __uint_as_float((uint32_t)(127 - e) << 23);
}

// Eight fp32 values -> eight E2M1 codes packed little-end first (x0 in bits 0-3).
// cvt.rn.satfinite rounds to nearest-even and saturates at +-6; its first source operand goes to
// the upper nibble.
__device__ __forceinline__ uint32_t pack_e2m1x8(float x0, float x1, float x2, float x3,
                                                float x4, float x5, float x6, float x7) {
  uint32_t out;
  asm("{\n\t"
      ".reg .b8 b0, b1, b2, b3;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b0, %2, %1;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b1, %4, %3;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b2, %6, %5;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b3, %8, %7;\n\t"
      "mov.b32 %0, {b0, b1, b2, b3};\n\t"
      "}"
      : "=r"(out)
      : "f"(x0), "f"(x1), "f"(x2), "f"(x3), "f"(x4), "f"(x5), "f"(x6), "f"(x7));
  return out;
}

__device__ __forceinline__ float bf16lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// Byte offset of the 16-byte code chunk of block c (0..3) of row r (0..127) inside an 8 KiB
// operand tile: rows of 64 bytes, 16-byte chunks XOR-swizzled with bits 1-2 of the row
// (the tensor core's 64-byte swizzle mode for a K-major operand).
__device__ __host__ __forceinline__ int tile_code_offset(int r, int c) {
  return r * 64 + ((c ^ ((r >> 1) & 3)) << 4);
}
// Byte offset of the scale of (row r, block c) inside a 512-byte scale-factor atom.
__device__ __host__ __forceinline__ int tile_scale_offset(int r, int c) {
  return (r & 31) * 16 + (r >> 5) * 4 + c;
}

// Programmatic dependent launch.  Every kernel of this library that is launched with launch_pdl starts with pdl_wait():
// nothing is read or written before all work queued earlier on the stream has completed and is visible, so the launch
// behaves as in plain stream order.  What overlaps is the launch itself: the CTAs are placed, and their set-up that
// touches no global memory runs, while the predecessor drains (pdl_trigger lets the successor's CTAs be placed as soon as
// every CTA of this grid has started).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// Loads of what an earlier launch may have written: ordinary, coherent ones behind the wait.  The read-only path (__ldg, or a
// load that the compiler takes for one because its pointer is const and __restrict__) asks that nobody writes the data while
// the kernel runs, which its predecessor may still do, and nothing holds such a load behind the wait.
__device__ __forceinline__ uint4 ld_global(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t ld_global(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float ld_global(const float* p) { return __uint_as_float(ld_global(reinterpret_cast<const uint32_t*>(p))); }
void count_launch();         // called at every kernel launch of a forward call (mxattn_last_launch_count)
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, unsigned block, size_t smem, cudaStream_t stream, Args... args) {
  count_launch();
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = dim3(block); cfg.dynamicSmemBytes = smem; cfg.stream = stream;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, KArgs(args)...);
}
// The same with clusters of `cluster` CTAs along x.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl_cluster(void (*kern)(KArgs...), dim3 grid, unsigned block, unsigned cluster, cudaStream_t stream, Args... args) {
  count_launch();
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = dim3(block); cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, KArgs(args)...);
}
uint64_t current_context();       // its number, 0 if there is none yet
// Sets a kernel's attribute, once per kernel and context (a driver call per launch otherwise).  One attribute per kernel.
bool ensure_attribute(const void* kern, cudaFuncAttribute attribute, int value);
bool ensure_dynamic_smem(const void* kern, int bytes);       // its limit of dynamic shared memory
PFN_cuTensorMapEncodeTiled tensor_map_encoder();      // null if the driver has none
// an attention output as a [bh][Nq][128] tensor that is written in boxes of 32 rows x 128 bytes with the 128-byte swizzle
int encode_output_map(CUtensorMap* map, void* o, int64_t bh, int64_t Nq, bool f32);
int sm_count();              // of the current device (0 on error)

// Division of an attention kernel's work (pairs of query tiles of 128 rows, one pair per CTA and wave): where the last wave
// of pairs fills at most half of the SMs, each of its tiles gets a CTA of its own, which takes less time than a pair.
struct TileSplit {
  int64_t pair_ctas, ctas;
  TileSplit(int64_t pairs, int64_t n_sm) {
    const int64_t rest = pairs % n_sm;
    pair_ctas = 2 * rest <= n_sm ? pairs - rest : pairs;
    ctas = pair_ctas + 2 * (pairs - pair_ctas);
  }
};
struct TileOfCta {
  int bh, qtile;               // head, first query tile
  bool two, empty;             // whether the CTA has a second one / has none (an odd head's missing tile)
  __device__ __forceinline__ TileOfCta(int cta, int pair_ctas, int q_pairs, int q_tiles) {
    const bool single = cta >= pair_ctas;
    const int pair = single ? pair_ctas + ((cta - pair_ctas) >> 1) : cta;
    bh = pair / q_pairs;
    qtile = 2 * (pair - bh * q_pairs) + (single ? (cta - pair_ctas) & 1 : 0);
    empty = qtile >= q_tiles;
    two = !single && qtile + 1 < q_tiles;
  }
};

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Internal launchers (defined in quantize.cu / forward.cu); all return an mxattn_status.
int launch_quantize(const void* in, void* codes, void* scales, int64_t batch, int64_t rows,
                    int64_t cols, int block_axis, int mode, int layout, cudaStream_t stream,
                    uint32_t rule_override = 0xFFFFFFFFu);
// Q, K (block axis 1) and V (block axis 0) of `bh` heads in tile layout; mode may carry MXATTN_MODE_HADAMARD for Q and K.
// v may be null (two operands).  Also clears status[0..3].
int launch_quantize_qkv(const void* q, void* q_codes, void* q_scales, const void* k, void* k_codes, void* k_scales,
                        const void* v, void* v_codes, void* v_scales, int64_t bh, int64_t Nq, int64_t Nkv, int mode,
                        int* status, cudaStream_t stream);
// NVFP4 operands of a forward call in tile layout: tensor maxima (amax[3 bh], zero on entry) and quantization of Q, K, V.
int launch_nvfp4_operands(const void* q, void* q_codes, void* q_scales, const void* k, void* k_codes, void* k_scales,
                          const void* v, void* v_codes, void* v_scales, float* amax, float* tensor_scale, int64_t bh,
                          int64_t Nq, int64_t Nkv, cudaStream_t stream);
int launch_zero(uint32_t* words, int64_t n, cudaStream_t stream);      // a few words: status, tensor maxima
bool amax_by_cluster(int64_t batch, int64_t chunks, bool fits);      // `fits`: a cluster of 16 CTAs can run
int launch_tensor_amax(const void* in, float* amax, int64_t batch, int64_t rows, int64_t cols, cudaStream_t stream);
int launch_quantize_nvfp4(const void* in, void* codes, void* scales, const float* amax, float* tensor_scale, int64_t batch,
                          int64_t rows, int64_t cols, int block_axis, int layout, cudaStream_t stream);
int launch_forward(const void* q_codes, const void* q_scales, const void* k_codes,
                   const void* k_scales, const void* v_codes, const void* v_scales, void* o,
                   int B, int H, int64_t Nq, int64_t Nkv, float softmax_scale, unsigned flags,
                   int* status, cudaStream_t stream, void* dump = nullptr, void* profile = nullptr, bool followed = false);
constexpr int kStaticTiles = 48, kStaticTilesNv = 3;     // KV tiles up to which a CTA of the walking kernel (walk.cuh) has its items from the start: MXFP4, NVFP4
// The first `pairs` pairs of query tiles, counted over all heads, go to the walking kernel (walk) or to the kernel for pairs, the rest to CTAs of
// 128 / R rows (R = 0: there is none).  `followed`: other attention launches run beside.
struct ForwardPlan { bool walk; int64_t pairs; int R; };
ForwardPlan forward_plan(int64_t n_sm, int64_t bh, int64_t Nq, int64_t Nkv, bool pnq, bool followed);
int launch_forward_rows(int R, int64_t first_pair, const void* q_codes, const void* q_scales, const void* k_codes, const void* k_scales,
                        const void* v_codes, const void* v_scales, void* o, int B, int H, int64_t Nq, int64_t Nkv,
                        float softmax_scale, unsigned flags, int* status, cudaStream_t stream);
int launch_forward_walk(int64_t n_sm, int64_t pairs, const void* q_codes, const void* q_scales, const void* k_codes, const void* k_scales,
                        const void* v_codes, const void* v_scales, void* o, int B, int H, int64_t Nq, int64_t Nkv,
                        float softmax_scale, unsigned flags, int* status, cudaStream_t stream, void* dump = nullptr);
size_t forward_dump_bytes(int B, int H, int64_t Nq, int64_t Nkv);
size_t forward_profile_bytes(int B, int H, int64_t Nq, int64_t Nkv);
size_t bf16_workspace_bytes(int B, int H, int64_t Nq, int64_t Nkv);
int launch_forward_bf16(const void* q, const void* k, const void* v, void* o, int B, int H, int64_t Nq, int64_t Nkv,
                        float softmax_scale, unsigned flags, void* workspace, size_t workspace_bytes, cudaStream_t stream);
size_t nvfp4_workspace_bytes(int B, int H, int64_t Nq, int64_t Nkv);
int launch_forward_nvfp4(const void* q, const void* k, const void* v, void* o, int B, int H, int64_t Nq, int64_t Nkv,
                         float softmax_scale, unsigned flags, void* workspace, size_t workspace_bytes, cudaStream_t stream);
int launch_rowsum_diag(const void* q_codes, const void* q_scales, const void* k_codes, const void* k_scales,
                       void* out, int B, int H, int64_t Nq, int64_t Nkv, float softmax_scale, uint32_t rule,
                       int* status, cudaStream_t stream);
int launch_bounded_wait_selftest(int* status, long long limit_cycles, cudaStream_t stream);
int launch_exp2_codes_selftest(int* status, cudaStream_t stream);
int launch_pair_abandon_selftest(int* status, long long limit_cycles, int meetings, cudaStream_t stream);

}  // namespace mxattn
