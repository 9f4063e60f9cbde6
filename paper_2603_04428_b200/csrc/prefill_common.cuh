// What the tcgen05 prefill kernels share.
#pragma once
#include "convert.cuh"
#include "f32x2.cuh"
#include "q4kv_layout.cuh"
#include "tcgen05.cuh"

namespace q4kv {
namespace prefill {

constexpr float kLazy = 8.f;                             // rescale when the row maximum grew by more than this (log2)

// the largest magnitude of eight bf16 numbers
__device__ inline float max_abs8(uint4 v) {
  auto two = [](uint32_t u) { return fmaxf(fabsf(__uint_as_float(u << 16)), fabsf(__uint_as_float(u & 0xffff0000u))); };
  return fmaxf(fmaxf(two(v.x), two(v.y)), fmaxf(two(v.z), two(v.w)));
}
// eight bf16 numbers times sf (a power of two) as binary16, in the order 0,4,1,5,2,6,3,7
__device__ inline uint4 query8(uint4 v, float sf) {
  auto lo = [&](uint32_t u) { return __uint_as_float(u << 16) * sf; };
  auto hi = [&](uint32_t u) { return __uint_as_float(u & 0xffff0000u) * sf; };
  return make_uint4(f32x2_to_h2(lo(v.x), lo(v.z)), f32x2_to_h2(hi(v.x), hi(v.z)), f32x2_to_h2(lo(v.y), lo(v.w)),
                    f32x2_to_h2(hi(v.y), hi(v.w)));
}

// The agents that bring one query in a batch where others bring more are left to the decode kernel, which is launched next
// on the same stream; its arrival counters are cleared here, so that the caller need not hand over a cleared workspace.
__device__ inline void clear_tickets(const PrefillExtra& x) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  for (int i = threadIdx.x; i < x.n_tickets; i += blockDim.x) x.tickets[i] = 0;
}

}  // namespace prefill
}  // namespace q4kv
