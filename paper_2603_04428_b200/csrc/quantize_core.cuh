// The quantizer of Section 3.2 as a device function shared by the kernels that write the cache: affine 4-bit
// codes over groups of 64, 16-bit scale and bias (binary16, or bfloat16: the section names both).  Every arithmetic
// step is a single rounded binary32 operation in a fixed order, so that codes, scales and biases are reproducible
// bit for bit:
//   bias = RD_16(min) (-0 -> +0), scale = RU_16((max - bias) / 15), code = clamp(rne((x - bias) / scale), 0, 15),
//   all codes 0 when scale = 0; RD_16 / RU_16 round toward -inf / +inf into the 16-bit type.
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

namespace q4kv {

struct QuantOut { uint32_t word; uint32_t sb; };         // sb: scale in the low 16 bits, bias in the high 16 bits

// bfloat16 is the upper half of binary32: dropping the lower half rounds toward zero, and a value that lost bits on
// the far side of zero from the rounding direction moves one step away from zero.
__device__ inline uint32_t bf16_bits_rd(float x) {
  const uint32_t u = __float_as_uint(x);
  return (u >> 16) + (((u & 0xFFFFu) != 0u && (u >> 31) != 0u) ? 1u : 0u);
}
__device__ inline uint32_t bf16_bits_ru(float x) {
  const uint32_t u = __float_as_uint(x);
  return (u >> 16) + (((u & 0xFFFFu) != 0u && (u >> 31) == 0u) ? 1u : 0u);
}

// Scale and bias of one group from its minimum and maximum (the fixed binary32 sequence of the header comment):
// their 16-bit patterns and their values.
struct GroupScale { uint32_t hs, hb; float sf, bf; };
__device__ inline GroupScale group_scale(float mn, float mx, bool bf16) {
  GroupScale gs;
  if (bf16) {
    gs.hb = bf16_bits_rd(mn);
    if ((gs.hb & 0x7FFFu) == 0u) gs.hb = 0u;                                      // -0 -> +0
    gs.bf = __uint_as_float(gs.hb << 16);
    gs.hs = bf16_bits_ru(__fdiv_rn(__fsub_rn(mx, gs.bf), 15.0f));
    gs.sf = __uint_as_float(gs.hs << 16);
  } else {
    __half hb = __float2half_rd(mn);
    if (__half2float(hb) == 0.0f) hb = __ushort_as_half((unsigned short)0);       // -0 -> +0
    gs.hb = __half_as_ushort(hb);
    gs.bf = __half2float(hb);
    const __half hs = __float2half_ru(__fdiv_rn(__fsub_rn(mx, gs.bf), 15.0f));
    gs.hs = __half_as_ushort(hs);
    gs.sf = __half2float(hs);
  }
  return gs;
}

// code = clamp(rne(fl((x - b) / s))), inv = fl(1 / s), s != 0.  The IEEE division would dominate the quantizer, so the
// quotient is taken as q = t * inv with one correction by its residual.  The residual t - s q is exact, since s has at most 11
// significant bits, and with inv correctly rounded the corrected quotient is within 2^-46 of itself of t / s before its own
// rounding, while t / s, unless it is a binary32 number, is at least 2^-36 of itself away from the midpoint of two of them: it
// is the correctly rounded quotient, ties of the code included.  Only a scale without a finite reciprocal (a bfloat16 scale
// below 2^-128) is divided by.
__device__ inline uint32_t quantize_code(float x, const GroupScale& gs, float inv) {
  const float t = __fsub_rn(x, gs.bf);
  float q = __fmul_rn(t, inv);
  q = __fmaf_rn(__fmaf_rn(-gs.sf, q, t), inv, q);
  if (inv > 3.0e38f) q = __fdiv_rn(t, gs.sf);
  return (uint32_t)min(max(__float2int_rn(q), 0), 15);
}

// One group of 64 elements by one warp, two elements per lane (`two`: their bf16 bits): eight words of codes and the pair.
__device__ __forceinline__ void quantize_row_group(uint32_t two, bool bf16, int lane, uint32_t* words, uint32_t* sb) {
  const float x0 = __uint_as_float(two << 16), x1 = __uint_as_float(two & 0xffff0000u);
  float mn = fminf(x0, x1), mx = fmaxf(x0, x1);
  asm("redux.sync.min.f32 %0, %0, 0xffffffff;" : "+f"(mn));
  asm("redux.sync.max.f32 %0, %0, 0xffffffff;" : "+f"(mx));
  const GroupScale gs = group_scale(mn, mx, bf16);
  uint32_t w = 0u;
  if (gs.sf != 0.f) {
    const float inv = __frcp_rn(gs.sf);
    w = (quantize_code(x0, gs, inv) | (quantize_code(x1, gs, inv) << 4)) << (8 * (lane & 3));
  }
  w |= __shfl_xor_sync(0xffffffffu, w, 1);
  w |= __shfl_xor_sync(0xffffffffu, w, 2);
  if ((lane & 3) == 0) words[lane >> 2] = w;
  if (lane == 0) *sb = gs.hs | (gs.hb << 16);
}

// A (scale, bias) pair of the cache as two binary32 numbers.
template <bool kBf16>
__device__ __forceinline__ float2 sb_to_f2(uint32_t u) {
  if (kBf16) return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xFFFF0000u));
  return __half22float2(*reinterpret_cast<const __half2*>(&u));
}

// x[8]: eight consecutive elements owned by this lane; the 8 lanes of a group cooperate.
__device__ inline QuantOut quantize_eight(const float x[8], bool bf16) {
  float mn = x[0], mx = x[0];
#pragma unroll
  for (int i = 1; i < 8; ++i) { mn = fminf(mn, x[i]); mx = fmaxf(mx, x[i]); }
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  const GroupScale gs = group_scale(mn, mx, bf16);
  uint32_t w = 0;
  if (gs.sf != 0.0f) {
    const float inv = __frcp_rn(gs.sf);
#pragma unroll
    for (int i = 0; i < 8; ++i) w |= quantize_code(x[i], gs, inv) << (4 * i);
  }
  QuantOut o;
  o.word = w;
  o.sb = gs.hs | (gs.hb << 16);
  return o;
}

__device__ inline void load_eight_bf16(const void* base, size_t elem_index, float x[8]) {
  const uint4 v = *reinterpret_cast<const uint4*>((const uint16_t*)base + elem_index);
  const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    x[2 * i] = __uint_as_float(u[i] << 16);
    x[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u);
  }
}

}  // namespace q4kv
