// Conversions that several attention kernels share: packed codes, scale and bias pairs and probabilities into binary16.
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

namespace q4kv {

constexpr float kLog2e = 1.4426950408889634f;

// Eight codes of one packed word -> eight binary16 values c * s + b, as the pairs (0,4) (1,5) (2,6)
// (3,7) with the scale and bias pair given for each.  Masking a nibble into the mantissa of 1024
// (ulp 1) or of 64 (ulp 1/16, for a nibble sitting four bits up) gives 1024 + c or 64 + c exactly.  The masks are kernel
// parameters, so that the compiler does not know them: (w & mask) | magic is then one instruction with one immediate operand,
// where two immediates take two (prefill in short runs: d = 256 391 -> 379 us, 192 / 128 321 -> 303, latent 231 -> 227, d = 128 1310 -> 1290).
struct CodeMasks { uint32_t lo = 0x000F000Fu, hi = 0x00F000F0u; };
__device__ inline uint4 dequant8(uint32_t w, uint32_t s04, uint32_t b04, uint32_t s15, uint32_t b15, uint32_t s26,
                                 uint32_t b26, uint32_t s37, uint32_t b37, const CodeMasks& m) {
  const uint32_t wh = w >> 8;
  const __half2 k1024 = __half2half2(__ushort_as_half((unsigned short)0x6400));
  const __half2 k64 = __half2half2(__ushort_as_half((unsigned short)0x5400));
  auto as_h2 = [](uint32_t u) { return *reinterpret_cast<__half2*>(&u); };
  auto as_u = [](__half2 h) { return *reinterpret_cast<uint32_t*>(&h); };
  const __half2 c04 = __hsub2(as_h2((w & m.lo) | 0x64006400u), k1024);
  const __half2 c15 = __hsub2(as_h2((w & m.hi) | 0x54005400u), k64);
  const __half2 c26 = __hsub2(as_h2((wh & m.lo) | 0x64006400u), k1024);
  const __half2 c37 = __hsub2(as_h2((wh & m.hi) | 0x54005400u), k64);
  return make_uint4(as_u(__hfma2(c04, as_h2(s04), as_h2(b04))), as_u(__hfma2(c15, as_h2(s15), as_h2(b15))),
                    as_u(__hfma2(c26, as_h2(s26), as_h2(b26))), as_u(__hfma2(c37, as_h2(s37), as_h2(b37))));
}
// the same with one (scale, bias) for all: s2 = (s, s), b2 = (b, b)
__device__ inline uint4 dequant8(uint32_t w, uint32_t s2, uint32_t b2, const CodeMasks& m) {
  return dequant8(w, s2, b2, s2, b2, s2, b2, s2, b2, m);
}
// position inside a row's eight elements of element u (the inverse of 0,4,1,5,2,6,3,7)
__host__ __device__ constexpr int slot_of(int u) { return ((u & 3) << 1) | (u >> 2); }
// element held by slot j of a row
__host__ __device__ constexpr int elem_of(int j) { return ((j & 1) << 2) | (j >> 1); }
__device__ inline float fast_exp2(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ inline uint32_t f32x2_to_h2(float lo, float hi) {
  const __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}
// A bfloat16 (scale, bias) pair as a binary16 pair: exact while the magnitude is a binary16 normal number (bfloat16
// has 8 significant bits), within 2^-25 below that; a magnitude beyond binary16's largest number is reported.
__device__ inline uint32_t bf16_pair_to_h2(uint32_t u, bool& overflow) {
  const uint32_t h = f32x2_to_h2(__uint_as_float(u << 16), __uint_as_float(u & 0xFFFF0000u));
  overflow |= (((h & 0x7C007C00u) + 0x04000400u) & 0x80008000u) != 0u;     // an exponent field of all ones
  return h;
}

}  // namespace q4kv
