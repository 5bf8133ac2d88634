// NVFP4 block quantization for sm_100a: the comparison format of the paper (named in its Introduction; Section 5.2,
// baseline "NVFP4"): E2M1 elements in blocks of 16 with an E4M3 block scale and one fp32 tensor-level scale.
//
// Two-level recipe, every step in IEEE fp32 (the order is part of the definition because the results are codes):
//   g   = fl32(2688 / A)       A = largest magnitude of the tensor (one per matrix of the batch), 2688 = 448 * 6
//   s_T = fl32(1 / g)          decode scale of the tensor
//   y_b = fl32(fl32(M_b * g) * fl32(1/6))          M_b = largest magnitude of the block
//   d_b = E4M3(y_b), round-to-nearest-even, saturating at 448
//   r_b = fl32(g / d_b)        (0 when d_b = 0)
//   code = sign | E2M1(fl32(|x| * r_b))
// Three HBM-bound passes: the tensor maximum (2 B/element read), then the quantizer (2 B read, 0.5 + 1/16 B written).
#include <cuda_fp16.h>

#include <atomic>

#include "common.cuh"

namespace mxattn {
namespace nv {

constexpr int kThreads = 256;
constexpr float kOneSixth = 0.16666667163372040f;      // fl32(1/6)
constexpr int kNvTileScaleBytes = 2 * kTileScaleBytes;   // two scale-factor atoms per 128 x 128 tile (8 blocks of 16 per row)

__device__ __forceinline__ uint32_t absmax_bf16x8(const uint4& v) {
  const uint32_t m = 0x7FFF7FFFu;
  uint32_t a = __vmaxu2(__vmaxu2(v.x & m, v.y & m), __vmaxu2(v.z & m, v.w & m));
  return max(a & 0xFFFFu, a >> 16);
}

// fp32 -> E4M3 code (round-to-nearest-even, saturating to 448) and back
__device__ __forceinline__ uint32_t e4m3_encode(float y) {
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(0.0f), "f"(y));     // second source -> low byte
  return (uint32_t)(r & 0xFFu);
}
__device__ __forceinline__ float e4m3_decode(uint32_t code) {
  uint32_t h2;
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"((uint16_t)code));
  return __half2float(__ushort_as_half((unsigned short)(h2 & 0xFFFFu)));
}

__device__ __forceinline__ float encode_scale(float amax) { return amax == 0.0f ? 1.0f : __fdiv_rn(2688.0f, amax); }

// Block scale code and element multiplier of a block whose maximum magnitude is `m` (fp32, >= 0).
__device__ __forceinline__ float block_scale(float m, float g, uint32_t* code_out) {
  const float y = __fmul_rn(__fmul_rn(m, g), kOneSixth);
  const uint32_t code = e4m3_encode(y);
  *code_out = code;
  const float d = e4m3_decode(code);
  return d == 0.0f ? 0.0f : __fdiv_rn(g, d);
}

__device__ __forceinline__ uint32_t quantize_bf16x8(const uint4& v, float r) {
  return pack_e2m1x8(__fmul_rn(bf16lo(v.x), r), __fmul_rn(bf16hi(v.x), r), __fmul_rn(bf16lo(v.y), r), __fmul_rn(bf16hi(v.y), r),
                     __fmul_rn(bf16lo(v.z), r), __fmul_rn(bf16hi(v.z), r), __fmul_rn(bf16lo(v.w), r), __fmul_rn(bf16hi(v.w), r));
}

// ------------------------------------------------------------------------------------------
// Largest magnitude of each matrix of the batch: amax[b] (fp32; must be zero on entry).  grid = (chunks, batch); a forward
// call takes the matrices of Q, K and V in one grid of three operands.  Eight loads of 16 bytes are in flight per thread.
// The grids walk the tensors from their end to their start: the block quantizer, which begins at the start, then finds
// what was read last still in L2.  Maximum and quantizer of 105 / 128 / 268 MB: 41.6 -> 40.9, 50.5
// -> 49.9, 105.2 -> 103.5 us.
constexpr int kAmaxUnroll = 8;
struct AmaxOperand { const uint4* in; uint32_t* amax; int64_t chunks; };       // chunks of 16 bytes per matrix
template <bool kFromEnd>
__device__ __forceinline__ uint32_t thread_amax(const uint4* src, int64_t chunks, int64_t first, int64_t step) {
  if (kFromEnd) src += chunks - 1;
  auto load = [&](int64_t i) { return ld_global(kFromEnd ? src - i : src + i); };
  uint32_t m = 0;
  int64_t i = first;
  for (; i + (kAmaxUnroll - 1) * step < chunks; i += kAmaxUnroll * step) {
    uint4 v[kAmaxUnroll];
#pragma unroll
    for (int u = 0; u < kAmaxUnroll; ++u) v[u] = load(i + u * step);
#pragma unroll
    for (int u = 0; u < kAmaxUnroll; ++u) m = max(m, absmax_bf16x8(v[u]));
  }
  for (; i < chunks; i += step) m = max(m, absmax_bf16x8(load(i)));
  return __reduce_max_sync(0xFFFFFFFFu, m);           // over the warp
}
__device__ __forceinline__ void tensor_amax_part(const AmaxOperand& o, int64_t b, int part, int parts) {
  uint32_t m = thread_amax<true>(o.in + b * o.chunks, o.chunks, (int64_t)part * kThreads + threadIdx.x, (int64_t)parts * kThreads);
  __shared__ uint32_t s[kThreads / 32];
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 1; w < kThreads / 32; ++w) m = max(m, s[w]);
    atomicMax(o.amax + b, m << 16);                 // non-negative floats order like their bit patterns
  }
}
__global__ void __launch_bounds__(kThreads) tensor_amax_kernel(const AmaxOperand o) {
  pdl_wait(); pdl_trigger();
  tensor_amax_part(o, gridDim.y - 1 - blockIdx.y, blockIdx.x, gridDim.x);
}
// The same with one cluster of 16 CTAs per matrix: the maxima meet in the first CTA's shared memory, which then simply writes
// the result -- nothing has to be zeroed before (a memset and the gap behind it are 2 us of a 10 us call).
constexpr int kClusterCtas = 16, kClusterThreads = 512;
__global__ void __launch_bounds__(kClusterThreads) tensor_amax_cluster_kernel(const AmaxOperand o) {
  __shared__ uint32_t s[kClusterCtas * kClusterThreads / 32];       // of CTA 0: one slot per warp of the cluster
  // Another CTA's shared memory may be written only once that CTA has started, which being scheduled together does not say.
  // Every thread arrives here and waits in front of its store below, so that the loads hide the barrier.
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  pdl_wait(); pdl_trigger();
  const uint32_t rank = blockIdx.x;                                 // gridDim.x == cluster size
  const uint32_t m = thread_amax<false>(o.in + blockIdx.y * o.chunks, o.chunks, (int64_t)rank * kClusterThreads + threadIdx.x, (int64_t)kClusterCtas * kClusterThreads);
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");             // every CTA of the cluster has started
  if ((threadIdx.x & 31) == 0) {
    uint32_t dst;
    asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(dst) : "r"((uint32_t)__cvta_generic_to_shared(&s[rank * (kClusterThreads / 32) + (threadIdx.x >> 5)])));
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(dst), "r"(m) : "memory");
  }
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (rank == 0 && threadIdx.x < 32) {
    uint32_t v = 0;
#pragma unroll
    for (int i = 0; i < kClusterCtas * kClusterThreads / 32; i += 32) v = max(v, s[i + threadIdx.x]);
    v = __reduce_max_sync(0xFFFFFFFFu, v);
    if (threadIdx.x == 0) o.amax[blockIdx.y] = v << 16;
  }
}
__global__ void __launch_bounds__(kThreads) tensor_amax_qkv_kernel(const AmaxOperand q, const AmaxOperand k, const AmaxOperand v) {
  pdl_wait(); pdl_trigger();
  tensor_amax_part(blockIdx.z == 0 ? v : blockIdx.z == 1 ? k : q, gridDim.y - 1 - blockIdx.y, blockIdx.x, gridDim.x);
}

// ------------------------------------------------------------------------------------------
// Axis 1 (Q, K: blocks of 16 along the row).  The CTA's four chunks of 16 bytes per thread arrive in shared memory by
// asynchronous copies (chunk c at position c ^ ((c >> 3) & 7) within its group of eight: copies and reads both touch
// every bank group once per quarter warp); a thread then owns four consecutive chunks = two blocks: block maxima
// without shuffles, one division per block, one 16-byte store of codes and one 2-byte store of scales.
// Canonical layout: chunks = rows * cols / 8 per matrix; tile layout (cols == 128): chunks = rows_pad * 16, rows beyond
// `rows` read as zero.  As a kernel of its own it runs in CTAs of 128 threads (grid = (ceil(chunks / 512), batch)): a CTA
// alternates between loading and computing, and sixteen small ones per SM keep the loads flowing better than eight of
// 256 threads (quantizer alone, 8 matrices of 128 columns, 2^24 / 2^25 / 2^27 elements: 8.7 -> 8.0, 15.0 -> 14.2, 55.9 -> 53.7 us).
constexpr int kA1Threads = 128;
template <bool kTileLayout, int kT>
__device__ __forceinline__ void quantize_nvfp4_axis1_part(uint4* s_v, const uint4* __restrict__ in, uint8_t* __restrict__ codes, uint8_t* __restrict__ scales,
                                                          const float* amax, float* __restrict__ tensor_scale, int64_t rows, int64_t cols,
                                                          int64_t rows_pad, int64_t part, int64_t b) {
  const int tid = threadIdx.x;
  const int64_t chunks_per_row = cols / 8;
  const int64_t n_valid = rows * chunks_per_row;                                  // chunks that exist in the input
  const int64_t n_out = (kTileLayout ? rows_pad : rows) * chunks_per_row;         // chunks that are written
  const uint4* src = in + b * n_valid;
  const int64_t base = part * (4 * kT);
  auto pos = [](int c) { return c ^ ((c >> 3) & 7); };
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int c = u * kT + tid;
    const bool inside = base + c < n_valid;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(&s_v[pos(c)])),
                 "l"(inside ? src + base + c : in), "r"(inside ? 16 : 0) : "memory");
  }
  const float g = encode_scale(ld_global(amax + b));
  if (part == 0 && tid == 0 && tensor_scale) tensor_scale[b] = __fdiv_rn(1.0f, g);
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  const int64_t i = base + 4 * tid;                 // first of this thread's four chunks (n_out is even: whole blocks only)
  if (i >= n_out) return;
  uint4 v[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) v[k] = s_v[pos(4 * tid + k)];
  uint32_t sc[2], w[4];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t m = max(absmax_bf16x8(v[2 * h]), absmax_bf16x8(v[2 * h + 1]));
    const float r = block_scale(__uint_as_float(m << 16), g, &sc[h]);
    w[2 * h] = quantize_bf16x8(v[2 * h], r);
    w[2 * h + 1] = quantize_bf16x8(v[2 * h + 1], r);
  }
  const bool both = i + 2 < n_out;                  // the matrix may end after this thread's first block
  if (kTileLayout) {                                // 16 chunks per row: the four chunks are one 32-column group of one row
    const int64_t row = i >> 4;
    const int q = (int)(i & 15) >> 2;
    const int64_t tile = b * (rows_pad / kTile) + row / kTile;
    const int rr = (int)(row % kTile);
    *reinterpret_cast<uint4*>(codes + tile * kTileCodeBytes + tile_code_offset(rr, q)) = make_uint4(w[0], w[1], w[2], w[3]);
    // blocks 2q and 2q + 1 of the row: adjacent bytes of one scale-factor atom
    *reinterpret_cast<uint16_t*>(scales + tile * kNvTileScaleBytes + (q >> 1) * kTileScaleBytes + tile_scale_offset(rr, (2 * q) & 3)) =
        (uint16_t)(sc[0] | (sc[1] << 8));
  } else {
    uint32_t* cdst = reinterpret_cast<uint32_t*>(codes) + b * n_out + i;
    uint8_t* sdst = scales + b * (n_out / 2) + (i >> 1);
    if (both && (((b * n_out) & 3) == 0)) {
      *reinterpret_cast<uint4*>(cdst) = make_uint4(w[0], w[1], w[2], w[3]);
    } else {
      *reinterpret_cast<uint2*>(cdst) = make_uint2(w[0], w[1]);
      if (both) *reinterpret_cast<uint2*>(cdst + 2) = make_uint2(w[2], w[3]);
    }
    if (both && (((b * (n_out / 2)) & 1) == 0)) {
      *reinterpret_cast<uint16_t*>(sdst) = (uint16_t)(sc[0] | (sc[1] << 8));
    } else {
      sdst[0] = (uint8_t)sc[0];
      if (both) sdst[1] = (uint8_t)sc[1];
    }
  }
}

template <bool kTileLayout>
__global__ void __launch_bounds__(kA1Threads)
quantize_nvfp4_axis1_kernel(const uint4* __restrict__ in, uint8_t* __restrict__ codes, uint8_t* __restrict__ scales,
                            const float* amax, float* __restrict__ tensor_scale, int64_t rows, int64_t cols,
                            int64_t rows_pad) {
  __shared__ uint4 s_v[4 * kA1Threads];
  pdl_wait(); pdl_trigger();
  quantize_nvfp4_axis1_part<kTileLayout, kA1Threads>(s_v, in, codes, scales, amax, tensor_scale, rows, cols, rows_pad, blockIdx.x, blockIdx.y);
}

// ------------------------------------------------------------------------------------------
// Axis 0 (V: blocks of 16 along the rows = tokens), outputs transposed (column-major, token-contiguous).
// A CTA stages a 32 KiB slab; thread -> (column pair, chunk of 32 tokens = two blocks).
//   tile layout:  128 tokens x 128 columns, one tile image; grid = (1, rows_pad / 128, batch)
//   canonical:    256 tokens x 64 columns, so that a column leaves as one 128-byte segment of codes and none of the slab is
//                 empty at 64 columns; grid = (ceil(cols / 64), ceil(rows_pad / 256), batch).
//                 Against 128 x 128: 12 x 50000 x 64 27.8 -> 18.4 us, 2^27 elements in 128 columns 62.2 -> 61.3
struct __align__(16) Axis0Smem {
  uint16_t in[kTile * kTile];
  uint8_t codes[kTileCodeBytes];
  uint8_t scales[kNvTileScaleBytes];
};
template <bool kTileLayout>
__device__ __forceinline__ void quantize_nvfp4_axis0_slab(Axis0Smem& sm, const uint16_t* __restrict__ in, uint8_t* __restrict__ codes, uint8_t* __restrict__ scales,
                                                          const float* amax, float* __restrict__ tensor_scale, int64_t rows, int64_t cols,
                                                          int64_t rows_pad, int64_t cx, int64_t ry, int64_t b) {
  constexpr int kTok = kTileLayout ? 128 : 256;                   // tokens per slab
  constexpr int kCol = kTileLayout ? 128 : 64;                    // columns per slab
  constexpr int kColBytes = kTok / 2;                             // code bytes per column of the slab
  uint16_t(*s_in)[kCol] = reinterpret_cast<uint16_t(*)[kCol]>(sm.in);
  uint8_t* s_codes = sm.codes;
  uint8_t* s_scales = sm.scales;
  const int tid = threadIdx.x;
  const int64_t col0 = cx * kCol, row0 = ry * kTok;
  const uint16_t* src = in + b * rows * cols;
  // staging offset of the 16-byte chunk c of column n: the tile image's own swizzle, or (canonical) the chunk index XORed
  // with the column pair so that the 8 threads of a store phase hit 8 different bank groups
  auto code_off = [](int n, int c) { return kTileLayout ? tile_code_offset(n, c) : n * kColBytes + ((c ^ ((n >> 1) & 7)) << 4); };
#pragma unroll
  for (int k = 0; k < (kTile * kTile / 8) / kThreads; ++k) {
    const int chunk = k * kThreads + tid;
    const int t = chunk / (kCol / 8), cc = (chunk % (kCol / 8)) << 3;
    // asynchronous 16-byte copy straight into shared memory; nothing is read (and zeros are written) beyond the edges
    const bool inside = row0 + t < rows && col0 + cc < cols;
    const uint16_t* gsrc = inside ? src + (row0 + t) * cols + col0 + cc : src;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(&s_in[t][cc])), "l"(gsrc), "r"(inside ? 16 : 0) : "memory");
  }
  const float g = encode_scale(ld_global(amax + b));
  if (cx == 0 && ry == 0 && tid == 0 && tensor_scale) tensor_scale[b] = __fdiv_rn(1.0f, g);
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  {
    const int np = tid % (kCol / 2), c = tid / (kCol / 2);      // column pair, chunk of 32 tokens
    const uint32_t* s32 = reinterpret_cast<const uint32_t*>(&s_in[0][0]);
    uint32_t w[32], m2[2] = {0u, 0u};
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      w[i] = s32[(c * 32 + i) * (kCol / 2) + np];
      m2[i >> 4] = __vmaxu2(m2[i >> 4], w[i] & 0x7FFF7FFFu);
    }
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const int n = 2 * np + side;
      uint32_t o[4];
#pragma unroll
      for (int hb = 0; hb < 2; ++hb) {                  // the two blocks of 16 tokens
        const uint32_t m = side ? (m2[hb] >> 16) : (m2[hb] & 0xFFFFu);
        uint32_t sc;
        const float r = block_scale(__uint_as_float(m << 16), g, &sc);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          float f[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const uint32_t ww = w[16 * hb + 8 * q + i];
            f[i] = __fmul_rn(side ? bf16hi(ww) : bf16lo(ww), r);
          }
          o[2 * hb + q] = pack_e2m1x8(f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7]);
        }
        const int blk = 2 * c + hb;                      // block of 16 tokens within the slab
        s_scales[kTileLayout ? ((blk >> 2) * kTileScaleBytes + tile_scale_offset(n, blk & 3)) : (n * (kTok / 16) + blk)] = (uint8_t)sc;
      }
      *reinterpret_cast<uint4*>(&s_codes[code_off(n, c)]) = make_uint4(o[0], o[1], o[2], o[3]);
    }
  }
  __syncthreads();
  if (kTileLayout) {
    const int64_t tile = b * (rows_pad / kTile) + ry;
    uint4* dst = reinterpret_cast<uint4*>(codes + tile * kTileCodeBytes);
#pragma unroll
    for (int k = 0; k < kTileCodeBytes / 16 / kThreads; ++k)
      dst[k * kThreads + tid] = reinterpret_cast<const uint4*>(s_codes)[k * kThreads + tid];
    if (tid < kNvTileScaleBytes / 16)
      reinterpret_cast<uint4*>(scales + tile * kNvTileScaleBytes)[tid] = reinterpret_cast<const uint4*>(s_scales)[tid];
  } else {
    // column n owns kColBytes contiguous bytes of this slab (the second 128 tokens only if they are inside rows_pad, which
    // is a multiple of 128, not of 256)
    uint8_t* cdst = codes + b * cols * (rows_pad / 2);
    uint8_t* sdst = scales + b * cols * (rows_pad / 16);
    const bool second = row0 + 128 < rows_pad;
#pragma unroll
    for (int k = 0; k < kTileCodeBytes / 16 / kThreads; ++k) {
      const int chunk = k * kThreads + tid;
      const int n = chunk / (kColBytes / 16), q = chunk % (kColBytes / 16);
      if (col0 + n < cols && (q < 4 || second))
        *reinterpret_cast<uint4*>(cdst + (col0 + n) * (rows_pad / 2) + row0 / 2 + q * 16) =
            *reinterpret_cast<const uint4*>(&s_codes[code_off(n, q)]);
    }
    if (tid < 2 * kCol) {
      const int n = tid >> 1, half = tid & 1;
      if (col0 + n < cols && (half == 0 || second))
        *reinterpret_cast<uint2*>(sdst + (col0 + n) * (rows_pad / 16) + row0 / 16 + 8 * half) = reinterpret_cast<const uint2*>(s_scales)[tid];
    }
  }
}

template <bool kTileLayout>
__global__ void __launch_bounds__(kThreads)
quantize_nvfp4_axis0_kernel(const uint16_t* __restrict__ in, uint8_t* __restrict__ codes, uint8_t* __restrict__ scales,
                            const float* amax, float* __restrict__ tensor_scale, int64_t rows, int64_t cols,
                            int64_t rows_pad) {
  __shared__ Axis0Smem sm;
  pdl_wait(); pdl_trigger();
  quantize_nvfp4_axis0_slab<kTileLayout>(sm, in, codes, scales, amax, tensor_scale, rows, cols, rows_pad, blockIdx.x, blockIdx.y, blockIdx.z);
}

// Q, K (axis 1) and V (axis 0) of a forward call in one launch (tile layout), as in quantize.cu; amax and tensor_scale are
// indexed by operand and head.
struct QkvOperand { const void* in; uint8_t* codes; uint8_t* scales; const float* amax; float* tensor_scale; int64_t rows, tiles, ctas; };
__global__ void __launch_bounds__(kThreads) quantize_nvfp4_qkv_kernel(const QkvOperand q, const QkvOperand k, const QkvOperand v) {
  __shared__ Axis0Smem sm;
  pdl_wait(); pdl_trigger();
  int64_t i = blockIdx.x;
  if (i < q.ctas + k.ctas) {                       // half a tile per CTA
    const QkvOperand& o = i < q.ctas ? q : k;
    if (i >= q.ctas) i -= q.ctas;
    const int64_t b = i / (2 * o.tiles);
    quantize_nvfp4_axis1_part<true, kThreads>(reinterpret_cast<uint4*>(sm.in), (const uint4*)o.in, o.codes, o.scales, o.amax, o.tensor_scale, o.rows, kHeadDim,
                                    o.tiles * kTile, i - b * 2 * o.tiles, b);
  } else if (i < q.ctas + k.ctas + v.ctas) {
    i -= q.ctas + k.ctas;
    const int64_t b = i / v.tiles;
    quantize_nvfp4_axis0_slab<true>(sm, (const uint16_t*)v.in, v.codes, v.scales, v.amax, v.tensor_scale, v.rows, kHeadDim, v.tiles * kTile, 0, i - b * v.tiles, b);
  }
}

}  // namespace nv

int launch_nvfp4_operands(const void* q, void* q_codes, void* q_scales, const void* k, void* k_codes, void* k_scales,
                          const void* v, void* v_codes, void* v_scales, float* amax, float* tensor_scale, int64_t bh,
                          int64_t Nq, int64_t Nkv, cudaStream_t stream) {
  using namespace nv;
  const int64_t qt = (Nq + kTile - 1) / kTile, kt = (Nkv + kTile - 1) / kTile;
  if (bh > 65535 || bh * (2 * qt + 3 * kt) > 0x7FFFFFFF) return MXATTN_EUNSUPPORTED;
  const int n_sm = sm_count();
  if (n_sm == 0) return MXATTN_ECUDA;
  // one tensor-level scale per head matrix (Q, K, V each), then the block quantizers
  const int64_t cq = Nq * kHeadDim / 8, ck = Nkv * kHeadDim / 8;
  int64_t parts = ((cq > ck ? cq : ck) + kThreads * kAmaxUnroll - 1) / (kThreads * kAmaxUnroll);
  const int64_t most = (8 * n_sm + 3 * bh - 1) / (3 * bh) > 1 ? (8 * n_sm + 3 * bh - 1) / (3 * bh) : 1;    // about one wave of CTAs
  if (parts > most) parts = most;
  if (launch_pdl(tensor_amax_qkv_kernel, dim3((unsigned)parts, (unsigned)bh, 3), kThreads, 0, stream, AmaxOperand{(const uint4*)q, (uint32_t*)amax, cq},
                 AmaxOperand{(const uint4*)k, (uint32_t*)amax + bh, ck}, AmaxOperand{(const uint4*)v, (uint32_t*)amax + 2 * bh, ck}) != cudaSuccess) return MXATTN_ECUDA;
  QkvOperand oq{q, (uint8_t*)q_codes, (uint8_t*)q_scales, amax, tensor_scale, Nq, qt, 2 * bh * qt};
  QkvOperand ok{k, (uint8_t*)k_codes, (uint8_t*)k_scales, amax + bh, tensor_scale + bh, Nkv, kt, 2 * bh * kt};
  QkvOperand ov{v, (uint8_t*)v_codes, (uint8_t*)v_scales, amax + 2 * bh, tensor_scale + 2 * bh, Nkv, kt, bh * kt};
  // Long problems: a kernel of their own for Q and K (quantize.cu has the reason).  The sides cross later than there, but
  // within 1 % of one another: 40 heads against 128 keys, us, one launch / apart: 1280 queries (6 per SM) 22.7 / 26.7, 8192
  // (35) 110.1 / 111.2, 16384 (70) 208.7 / 206.8; 24 x 8192 (42) 720.0 / 719.4.
  if (oq.ctas + ok.ctas > 24 * (int64_t)n_sm) {
    for (const QkvOperand* o : {&oq, &ok})
      if (launch_pdl(quantize_nvfp4_axis1_kernel<true>, dim3((unsigned)(kTile * kHeadDim / 32 / kA1Threads * o->tiles), (unsigned)bh), kA1Threads, 0, stream, (const uint4*)o->in, o->codes, o->scales,
                     o->amax, o->tensor_scale, o->rows, (int64_t)kHeadDim, o->tiles * kTile) != cudaSuccess) return MXATTN_ECUDA;
    oq.ctas = ok.ctas = 0;
  }
  if (launch_pdl(quantize_nvfp4_qkv_kernel, dim3((unsigned)(oq.ctas + ok.ctas + ov.ctas)), kThreads, 0, stream, oq, ok, ov) != cudaSuccess) return MXATTN_ECUDA;
  return MXATTN_OK;
}

// One cluster per matrix up to 4 MB each and 11 MB in all: what 16 SMs per matrix take longer than a full grid is less
// than what the launch that zeroes the results costs.  With the block quantizer behind, us against the full grid: one
// matrix of 1 MB 7.0 / 9.2, one of 4.2 MB 7.0 / 9.2, 40 of 0.26 MB 8.4 / 9.2; beyond, three of 4.2 MB 10.3 / 9.2, six
// 11.8 / 11.0, 40 of 0.8 MB 16.5 / 14.9, two of 8.4 MB 10.7 / 9.4.
bool amax_by_cluster(int64_t batch, int64_t chunks, bool fits) {
  return fits && chunks <= (4 << 20) / 16 && batch * chunks <= (11 << 20) / 16;
}

// Whether a cluster of 16 CTAs can run in the current context (a part of a device may be too small for one): asked once per
// context.
static bool cluster_fits() {
  static std::atomic<uint64_t> answers[16];                          // context's number and the answer in the lowest bit
  const uint64_t context = current_context();
  std::atomic<uint64_t>& at = answers[context & 15];
  const uint64_t seen = at.load(std::memory_order_relaxed);
  if (context != 0 && seen >> 1 == context) return seen & 1;
  bool fits = ensure_attribute((const void*)nv::tensor_amax_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nv::kClusterCtas); cfg.blockDim = dim3(nv::kClusterThreads);
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = nv::kClusterCtas; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
  cfg.attrs = &attr; cfg.numAttrs = 1;
  int n = 0;
  if (fits && (cudaOccupancyMaxActiveClusters(&n, nv::tensor_amax_cluster_kernel, &cfg) != cudaSuccess || n < 1)) fits = false;
  if (!fits) (void)cudaGetLastError();                               // an answer, not an error of the call
  if (context != 0) at.store(context << 1 | (fits ? 1 : 0), std::memory_order_relaxed);
  return fits;
}

int launch_tensor_amax(const void* in, float* amax, int64_t batch, int64_t rows, int64_t cols, cudaStream_t stream) {
  if (!in || !amax) return MXATTN_EINVAL;
  if (batch <= 0 || rows <= 0 || cols <= 0) return MXATTN_EINVAL;
  if ((rows * cols) % 8 != 0) return MXATTN_EUNSUPPORTED;
  if (!aligned16(in) || (reinterpret_cast<uintptr_t>(amax) & 3u)) return MXATTN_EALIGN;
  if (batch > 65535) return MXATTN_EUNSUPPORTED;
  const int64_t chunks = rows * cols / 8;
  const nv::AmaxOperand op{(const uint4*)in, reinterpret_cast<uint32_t*>(amax), chunks};
  if (amax_by_cluster(batch, chunks, cluster_fits())) {
    return launch_pdl_cluster(nv::tensor_amax_cluster_kernel, dim3(nv::kClusterCtas, (unsigned)batch), nv::kClusterThreads, nv::kClusterCtas, stream, op) == cudaSuccess
               ? MXATTN_OK : MXATTN_ECUDA;
  }
  int64_t blocks = (chunks + nv::kThreads * 8 - 1) / (nv::kThreads * 8);
  if (blocks > 1184) blocks = 1184;                 // 8 CTAs per SM at most: the loop strides over the rest
  if (launch_zero(op.amax, batch, stream) != MXATTN_OK) return MXATTN_ECUDA;
  return launch_pdl(nv::tensor_amax_kernel, dim3((unsigned)blocks, (unsigned)batch), nv::kThreads, 0, stream,
                    op) == cudaSuccess ? MXATTN_OK : MXATTN_ECUDA;
}

int launch_quantize_nvfp4(const void* in, void* codes, void* scales, const float* amax, float* tensor_scale, int64_t batch,
                          int64_t rows, int64_t cols, int block_axis, int layout, cudaStream_t stream) {
  if (!in || !codes || !scales || !amax) return MXATTN_EINVAL;
  if (batch <= 0 || rows <= 0 || cols <= 0) return MXATTN_EINVAL;
  if (block_axis != 0 && block_axis != 1) return MXATTN_EINVAL;
  if (layout != MXATTN_LAYOUT_CANONICAL && layout != MXATTN_LAYOUT_TILE) return MXATTN_EINVAL;
  if (layout == MXATTN_LAYOUT_TILE && cols != kHeadDim) return MXATTN_EUNSUPPORTED;
  if (block_axis == 1 && cols % 16 != 0) return MXATTN_EUNSUPPORTED;
  if (block_axis == 0 && cols % 8 != 0) return MXATTN_EUNSUPPORTED;
  if (!aligned16(in) || !aligned16(codes) || !aligned16(scales)) return MXATTN_EALIGN;
  if ((reinterpret_cast<uintptr_t>(amax) & 3u) || (reinterpret_cast<uintptr_t>(tensor_scale) & 3u)) return MXATTN_EALIGN;
  if (batch > 65535) return MXATTN_EUNSUPPORTED;
  const int64_t rows_pad = (rows + kTile - 1) / kTile * kTile;
  const bool tile = (layout == MXATTN_LAYOUT_TILE);
  cudaError_t e = cudaSuccess;
  if (block_axis == 1) {
    const int64_t n_out = (tile ? rows_pad : rows) * (cols / 8);
    const int64_t blocks = (n_out + 4 * nv::kA1Threads - 1) / (4 * nv::kA1Threads);
    if (blocks > 0x7FFFFFFF) return MXATTN_EUNSUPPORTED;
    dim3 grid((unsigned)blocks, (unsigned)batch);
    if (tile)
      e = launch_pdl(nv::quantize_nvfp4_axis1_kernel<true>, grid, nv::kA1Threads, 0, stream, (const uint4*)in, (uint8_t*)codes, (uint8_t*)scales,
                                                                               amax, tensor_scale, rows, cols, rows_pad);
    else
      e = launch_pdl(nv::quantize_nvfp4_axis1_kernel<false>, grid, nv::kA1Threads, 0, stream, (const uint4*)in, (uint8_t*)codes, (uint8_t*)scales,
                                                                                amax, tensor_scale, rows, cols, rows_pad);
  } else {
    const int64_t ct = tile ? 1 : (cols + 63) / 64, rt = tile ? rows_pad / kTile : (rows_pad + 255) / 256;   // tile layout: cols == 128
    if (ct > 0x7FFFFFFF || rt > 65535) return MXATTN_EUNSUPPORTED;
    dim3 grid((unsigned)ct, (unsigned)rt, (unsigned)batch);
    if (tile)
      e = launch_pdl(nv::quantize_nvfp4_axis0_kernel<true>, grid, nv::kThreads, 0, stream, (const uint16_t*)in, (uint8_t*)codes, (uint8_t*)scales,
                                                                               amax, tensor_scale, rows, cols, rows_pad);
    else
      e = launch_pdl(nv::quantize_nvfp4_axis0_kernel<false>, grid, nv::kThreads, 0, stream, (const uint16_t*)in, (uint8_t*)codes, (uint8_t*)scales,
                                                                                amax, tensor_scale, rows, cols, rows_pad);
  }
  return e == cudaSuccess ? MXATTN_OK : MXATTN_ECUDA;
}

}  // namespace mxattn

extern "C" int mxattn_tensor_amax(const void* in, void* amax, int64_t batch, int64_t rows, int64_t cols, void* stream) {
  return mxattn::launch_tensor_amax(in, static_cast<float*>(amax), batch, rows, cols, (cudaStream_t)stream);
}

extern "C" int mxattn_quantize_nvfp4(const void* in, void* codes, void* e4m3_scales, const void* tensor_amax,
                                     void* tensor_scale, int64_t batch, int64_t rows, int64_t cols, int block_axis,
                                     int layout, void* stream) {
  return mxattn::launch_quantize_nvfp4(in, codes, e4m3_scales, static_cast<const float*>(tensor_amax),
                                       static_cast<float*>(tensor_scale), batch, rows, cols, block_axis, layout,
                                       (cudaStream_t)stream);
}
