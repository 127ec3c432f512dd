// Shared device helpers: NVFP4 block quantization primitives and small utilities.
// sm_100a only.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/quads.h"

namespace quads {

constexpr int kBlock = 16;          // elements per scale block
constexpr float kGlobalDiv = 2688.f; // 6 * 448

// Launch bookkeeping (host side, per thread).
extern thread_local int g_launch_count;
inline void note_launch() { ++g_launch_count; }

#define QUADS_CUDA_OK(expr)                              \
  do {                                                   \
    cudaError_t _e = (expr);                             \
    if (_e != cudaSuccess) return QUADS_ERR_CUDA;        \
  } while (0)

// Programmatic dependent launch: every kernel of the MoE chain starts with this.  It blocks
// until the preceding kernel of the stream has completed and its writes are visible, then
// lets the following kernel begin its own launch (that one blocks at the same point), so
// launch latencies overlap instead of adding up.  A no-op for ordinary launches.
__device__ __forceinline__ void pdl_sync() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Host side: launch with the programmatic-stream-serialization attribute (or plainly).
bool pdl_enabled();
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                 Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 1 : 0;
  note_launch();
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// The same for a grid of n_cta CTAs in clusters of `cluster`, and for a grid that is one cluster.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_clusters(void (*kernel)(KArgs...), int n_cta, int cluster, int threads, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_cta);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cluster; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 2 : 1;
  note_launch();
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_cluster(void (*kernel)(KArgs...), int n_cta, int threads, size_t smem, cudaStream_t st, Args&&... args) {
  return launch_clusters(kernel, n_cta, n_cta, threads, smem, st, static_cast<Args&&>(args)...);
}

// Raise a kernel's dynamic shared-memory limit once per device (the attribute is per device; a
// process may drive several).  `Kernel` must be a distinct function per instantiation.
template <auto Kernel>
inline cudaError_t set_max_dynamic_smem(int bytes) {
  static bool done[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
  e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = true;
  return e;
}

__device__ __forceinline__ float bf16_bits_to_float(uint32_t b16) { return __uint_as_float(b16 << 16); }

// Two packed floats: one instruction where two would take two issue slots (the arithmetic units' time is the same).
__device__ __forceinline__ uint64_t f32x2_pack(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void f32x2_unpack(uint64_t v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ uint64_t f32x2_mul(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f32x2_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// Unpack 8 bf16 (one 16-byte vector) to float.  As an addition to -0 it runs in the FMA pipe, one cycle per
// value; a shift or a mask takes two in the integer pipe, which bounds the quantizer.
__device__ __forceinline__ void unpack2(uint32_t w, float& lo, float& hi) {
  asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %2;\n\tadd.f32.bf16 %0, l, %3;\n\tadd.f32.bf16 %1, h, %3;\n\t}"
      : "=f"(lo), "=f"(hi) : "r"(w), "f"(-0.0f));
}
__device__ __forceinline__ void unpack8(const uint4& v, float* f) {
  unpack2(v.x, f[0], f[1]);
  unpack2(v.y, f[2], f[3]);
  unpack2(v.z, f[4], f[5]);
  unpack2(v.w, f[6], f[7]);
}

// 32-byte read-only global load (two 16-byte halves of one scale block).
__device__ __forceinline__ void ldg256(const void* p, uint4& a, uint4& b) {
  asm volatile("ld.global.nc.L1::no_allocate.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
               : "l"(p));
}

// The same, asking L2 to keep the lines for a second pass (evict_last) or to drop them (evict_first).
__device__ __forceinline__ void ldg256_keep(const void* p, uint4& a, uint4& b) {
  asm volatile("ld.global.L2::evict_last.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w) : "l"(p));
}
__device__ __forceinline__ void ldg256_stream(const void* p, uint4& a, uint4& b) {
  asm volatile("ld.global.L2::evict_first.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w) : "l"(p));
}
// Largest magnitudes of eight bf16 values, two per word.
__device__ __forceinline__ uint32_t absmax8(const uint4& v) {
  return __vmaxu2(__vmaxu2(v.x & 0x7FFF7FFFu, v.y & 0x7FFF7FFFu), __vmaxu2(v.z & 0x7FFF7FFFu, v.w & 0x7FFF7FFFu));
}
// Order-preserving map float -> uint32 (larger float <=> larger uint).
__device__ __forceinline__ uint32_t float_key(float v) {
  const uint32_t b = __float_as_uint(v);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ uint32_t ld_acquire_u32(const void* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t ld_relaxed_u32(const void* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float gs_from_amax_bits(uint32_t bits) {
  const float amax = __uint_as_float(bits);
  return amax > 0.f ? __fdiv_rn(amax, kGlobalDiv) : 1.0f;
}

// float -> E4M3 byte, round-to-nearest-even, saturating to 448.
__device__ __forceinline__ uint32_t f32_to_e4m3(float v) {
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(0.f), "f"(v));
  return r & 0xFFu;
}

// E4M3 byte -> float (exact).
__device__ __forceinline__ float e4m3_to_f32(uint32_t b) {
  uint32_t h2;
  uint16_t in = (uint16_t)b;
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"(in));
  return __half2float(__ushort_as_half((unsigned short)(h2 & 0xFFFFu)));
}

// Eight floats -> eight E2M1 codes in one 32-bit word (element i in nibble i),
// round-to-nearest-even, saturating to 6.  The hardware convert keeps the sign bit of
// values that round to zero (-0, small negatives), which is the convention of this
// library; the exhaustive quantizer test pins it.
__device__ __forceinline__ uint32_t f32x8_to_e2m1x8(float v0, float v1, float v2, float v3, float v4, float v5,
                                                    float v6, float v7) {
  uint32_t r;
  asm("{\n\t.reg .b8 b0, b1, b2, b3;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b0, %2, %1;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b1, %4, %3;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b2, %6, %5;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b3, %8, %7;\n\t"
      "mov.b32 %0, {b0, b1, b2, b3};\n\t}"
      : "=r"(r) : "f"(v0), "f"(v1), "f"(v2), "f"(v3), "f"(v4), "f"(v5), "f"(v6), "f"(v7));
  return r;
}

// Eight E2M1 codes (element i in nibble i) -> eight floats (exact).  The conversion wants its byte alone in a register.
__device__ __forceinline__ void e2m1x8_to_f32x8(uint32_t codes, float* f) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    uint32_t h2;
    const uint16_t in = (uint16_t)__byte_perm(codes, 0u, 0x4440 + i);
    asm("{ .reg .b8 t; cvt.u8.u16 t, %1; cvt.rn.f16x2.e2m1x2 %0, t; }" : "=r"(h2) : "h"(in));
    const float2 v = __half22float2(*reinterpret_cast<__half2*>(&h2));
    f[2 * i] = v.x;
    f[2 * i + 1] = v.y;
  }
}

struct BlockQ {
  uint32_t lo, hi;   // 16 codes: elements 0..7 in lo, 8..15 in hi
  uint32_t sf8;      // E4M3 scale byte
  float d;           // decoded block scale sf * gs
};

// Per-tensor constants of the quantizer.  `r6` is the correctly rounded reciprocal of d6 and
// `inv_lut[c]` = 1 / (E4M3(c) * gs) (0 for c = 0), both computed with IEEE operations, so that
// the per-block arithmetic below reproduces the documented single-operation recipe bit for bit
// without a division routine per block.
struct QuantCtx {
  float gs, d6, r6;
  const float* inv_lut;   // 128 entries (shared memory)
};

__device__ __forceinline__ void quant_ctx_scalars(QuantCtx& c, float gs) {
  c.gs = gs;
  c.d6 = __fmul_rn(6.0f, gs);
  c.r6 = __frcp_rn(c.d6);
}
// Entry `code` of the reciprocal table for per-tensor scale gs.
__device__ __forceinline__ float quant_inv_entry(uint32_t code, float gs) {
  const float sf = e4m3_to_f32(code & 0x7Fu);
  return (sf == 0.f || code == 0x7Fu) ? 0.f : __fdiv_rn(1.0f, __fmul_rn(sf, gs));
}

// Largest magnitude of three values (NaN ignored).
__device__ __forceinline__ float absmax3(float a, float b, float c) {
  float r;
  asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// Quantize one block of 16 floats.  u = amax / d6 is formed as q0 = amax * r6 followed by one
// fused correction step (residual amax - q0 * d6 is exact in an FMA), which yields the correctly
// rounded quotient given a correctly rounded reciprocal; the 1 / d of the element scaling comes
// from the table (kLut) or from the table's own formula evaluated in place.
// What it costs a warp (32 blocks, eight warps per scheduler, with the loads and a checksum): 107 cycles, of which the
// sixteen values' conversions to E2M1 are 32 (an instruction for two values takes four cycles) and the integer
// pipe, two cycles per instruction, most of the rest; with scalar products, two-input maxima and shifts for
// the unpacking 116; with the decode to bf16 behind it 179 (215), with residual, its squares and its
// quantization 240 (276).  Calls, before and now: fake-quant of 128 x 1536 x 2048 390.7 -> 373.9 us, quantizer 8192 x
// 2048 15.9 -> 15.1.
template <bool kLut = true>
__device__ __forceinline__ BlockQ quantize_block(const float* v, const QuantCtx& c) {
  const float a = absmax3(absmax3(absmax3(v[0], v[1], v[2]), absmax3(v[3], v[4], v[5]), absmax3(v[6], v[7], v[8])),
                          absmax3(absmax3(v[9], v[10], v[11]), absmax3(v[12], v[13], v[14]), v[15]), 0.f);
  const float q0 = __fmul_rn(a, c.r6);
  const float u = __fmaf_rn(__fmaf_rn(-q0, c.d6, a), c.r6, q0);
  BlockQ r;
  r.sf8 = f32_to_e4m3(u);
  r.d = __fmul_rn(e4m3_to_f32(r.sf8), c.gs);
  // without the table: the same quotient, one division per block
  const float inv = kLut ? c.inv_lut[r.sf8] : quant_inv_entry(r.sf8, c.gs);
  const uint64_t inv2 = f32x2_pack(inv, inv);
  float y[16];
#pragma unroll
  for (int i = 0; i < 8; ++i) f32x2_unpack(f32x2_mul(f32x2_pack(v[2 * i], v[2 * i + 1]), inv2), y[2 * i], y[2 * i + 1]);
  r.lo = f32x8_to_e2m1x8(y[0], y[1], y[2], y[3], y[4], y[5], y[6], y[7]);
  r.hi = f32x8_to_e2m1x8(y[8], y[9], y[10], y[11], y[12], y[13], y[14], y[15]);
  return r;
}

// Dequantize the 16 codes of a block: value(code) * d, one float32 multiply.
__device__ __forceinline__ void dequant_block(const BlockQ& q, float* out) {
  float f[16];
  e2m1x8_to_f32x8(q.lo, f);
  e2m1x8_to_f32x8(q.hi, f + 8);
  const uint64_t d2 = f32x2_pack(q.d, q.d);
#pragma unroll
  for (int i = 0; i < 8; ++i) f32x2_unpack(f32x2_mul(f32x2_pack(f[2 * i], f[2 * i + 1]), d2), out[2 * i], out[2 * i + 1]);
}

// Residual of a block, Q_A(v) - v (one float32 subtraction: the product with -1 is exact).
__device__ __forceinline__ void residual_block(const BlockQ& q, const float* v, float* out) {
  dequant_block(q, out);
  const uint64_t minus1 = f32x2_pack(-1.f, -1.f);
#pragma unroll
  for (int i = 0; i < 8; ++i)
    f32x2_unpack(f32x2_fma(f32x2_pack(v[2 * i], v[2 * i + 1]), minus1, f32x2_pack(out[2 * i], out[2 * i + 1])), out[2 * i], out[2 * i + 1]);
}
// acc += r * r, 16 sums.
__device__ __forceinline__ void add_squares(const float* r, float* acc) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint64_t v = f32x2_pack(r[2 * i], r[2 * i + 1]);
    f32x2_unpack(f32x2_fma(v, v, f32x2_pack(acc[2 * i], acc[2 * i + 1])), acc[2 * i], acc[2 * i + 1]);
  }
}

__device__ __forceinline__ uint32_t f32x2_to_bf16x2(float lo, float hi) {
  __nv_bfloat162 b = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&b);
}

// Mask bytes m[0..7] in {0, 1} -> 0xF per selected nibble.
__device__ __forceinline__ uint32_t nibble_mask8(const uint2& v) {
  uint32_t out = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    out |= ((v.x >> (8 * i)) & 1u) * (0xFu << (4 * i));
    out |= ((v.y >> (8 * i)) & 1u) * (0xFu << (16 + 4 * i));
  }
  return out;
}
__device__ __forceinline__ uint32_t nibble_mask8(const uint8_t* m) { return nibble_mask8(*reinterpret_cast<const uint2*>(m)); }

// Byte offset of scale (row, blk) in the tiled layout with kt_count = ceil(K/64) atoms per row tile.
__host__ __device__ __forceinline__ size_t sf_tiled_offset(int64_t row, int64_t blk, int64_t kt_count) {
  return ((size_t)(row >> 7) * (size_t)kt_count + (size_t)(blk >> 2)) * 512u +
         (size_t)((row & 31) * 16 + ((row >> 5) & 3) * 4 + (blk & 3));
}

__device__ __forceinline__ void stg256(void* addr, const uint32_t* v) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(addr), "r"(v[0]), "r"(v[1]), "r"(v[2]),
               "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}

// The same, telling L2 that nobody reads it soon.  Fake-quantized weights leave by it: two 16-byte streaming stores
// per thread write every sector in two halves (16 tensors of 3072 x 4096: 212 us, 203 with this one; 8 of
// 1536 x 2048: 35 and 33), and without the hint the written lines push the tensor that is still to be quantized out
// of L2 (220 us).  (The decoded operand of the one-sided mode W16A4 leaves by it too, although the product behind it reads
// it back: not measured without the hint.)
__device__ __forceinline__ void stg256_stream(void* addr, const uint32_t* v) {
  asm volatile("st.global.L2::evict_first.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(addr), "r"(v[0]), "r"(v[1]), "r"(v[2]),
               "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}

// Store a warp's 32 rows x 64 accumulator columns (thread = row) as bf16, scaled, to rows of
// `n_out` elements starting at `dst`, rows >= rows_valid skipped.  The 32-byte chunks are first
// transposed inside every group of 4 lanes (two butterfly exchanges), so that each store
// instruction of the warp writes eight complete 128-byte lines instead of a 32-byte piece of 32
// different lines.  All 32 lanes must call it.  kHalves: `dst` is 16-byte, not 32-byte aligned.
template <bool kHalves = false>
__device__ __forceinline__ void store_y_rows(const float* acc, float scale, uint16_t* dst, int n_out, int rows_valid,
                                             int lane) {
  uint32_t w[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) w[i] = f32x2_to_bf16x2(acc[2 * i] * scale, acc[2 * i + 1] * scale);
  // chunk c = w[8c .. 8c+7]; after the exchanges chunk slot c of lane (g, j) holds chunk j of lane (g, c)
#pragma unroll
  for (int s = 1; s < 4; s <<= 1) {
    const bool up = (lane & s) != 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (c & s) continue;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const uint32_t lo = w[8 * c + k], hi = w[8 * (c | s) + k];
        const uint32_t got = __shfl_xor_sync(0xFFFFFFFFu, up ? lo : hi, s);
        w[8 * c + k] = up ? got : lo;
        w[8 * (c | s) + k] = up ? hi : got;
      }
    }
  }
  const int g = lane >> 2, j = lane & 3;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = 4 * g + i;
    if (r >= rows_valid) continue;
    uint16_t* d = dst + (size_t)r * n_out + 16 * j;
    if (!kHalves) {
      stg256(d, w + 8 * i);
    } else {
      reinterpret_cast<uint4*>(d)[0] = make_uint4(w[8 * i], w[8 * i + 1], w[8 * i + 2], w[8 * i + 3]);
      reinterpret_cast<uint4*>(d)[1] = make_uint4(w[8 * i + 4], w[8 * i + 5], w[8 * i + 6], w[8 * i + 7]);
    }
  }
}

// One partial column score of site 2 (a float32 sum of squared residuals over at most 32 rows, >= 0) as a fixed-point
// integer with `bits` fractional bits in units of gs^2, capped at 2^(23 + bits): where the scale covers the value a
// residual is at most half a quantization step, 448 gs, so 32 rows stay below 2^23 gs^2; sums of rows that a
// scale several times too small clips reach the cap and count as equal.  Added to the column's total with an integer
// reduction, whose result does not depend on the order of the additions.
__device__ __forceinline__ void add_score(unsigned long long* total, float partial, float gs, int bits) {
  constexpr int kCapBits = 23;
  const float u = __fdiv_rn(__fdiv_rn(partial, gs), gs);
  const float cap = __uint_as_float((uint32_t)(127 + kCapBits + bits) << 23);
  const float v = fminf(u * __uint_as_float((uint32_t)(127 + bits) << 23), cap);
  const unsigned long long q = __float2ull_rd(v);
  if (q) asm volatile("red.global.add.u64 [%0], %1;" ::"l"(total), "l"(q) : "memory");
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
  return v;
}

}  // namespace quads
