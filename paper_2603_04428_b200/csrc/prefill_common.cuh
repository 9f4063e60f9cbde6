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

// What a CTA reads first, asked of L2 while the preceding kernel drains: a prefetch returns nothing, and L2 is where the writes of the
// preceding kernels land, so it may come before the wait for them.  Lane l of one warp asks for the 64-key block it0 + l (block tables are
// inputs that no kernel writes; the table entries are then in L1 for the loader), the threads of the tile's rows for their query row.
// Latent cache, 3 agents of 250 to 512 on 2000 to 4000 tokens, with the append: 210.3 -> 206.3 us a layer, blocks and rows.  d = 256 and
// 192 / 128: rows only.  Their blocks come by bulk copies that a loader issues at once; asked for beforehand as well, four layers with the
// append, 44 tokens on 107 72.5 -> 75.1 us, 2 x (2000 + 203) 183.3 -> 184.6, 6 x (3000 + 400) in a window 422.8 -> 424.7.  Not at d = 128,
// whose tiles' steps are long beside it: one agent 1377.0 / 1375.6, injection pass 5135 / 5145.
template <class Par>
__device__ __forceinline__ void ask_for_blocks(const Par& P, int a, int hk, int it0, int count, uint32_t chunk_bytes) {
  const int l = threadIdx.x & 31;
  if (l >= count) return;
  const int c = 2 * (it0 + l), blk = P.tables[(size_t)a * P.max_blocks + (c >> 3)];
  if (blk >= 0 && blk < P.n_blocks)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(head_block(P.pool, P.y, P.layer, blk, hk) + (size_t)(c & 7) * chunk_bytes),
                 "r"(2 * chunk_bytes) : "memory");
}
template <int kElements>
__device__ __forceinline__ void ask_for_row(const uint16_t* row) {
#pragma unroll
  for (int e = 0; e < kElements; e += 64) asm volatile("prefetch.global.L2 [%0];" ::"l"(row + e) : "memory");
}
// A warp's 32 rows and global memory.  A thread owns a row, but rows lie kilobytes apart: threads that load or store their own rows
// touch 32 lines with every instruction, which made 4 us of a tile's start and 3 to 4 of its end.  So the lanes share lines -- eight
// rows x four 16-byte pieces in a load, whole 64- or 128-byte parts of rows in a store -- and what is stored passes through 4 KB of
// shared memory per warp, where piece j of row r lies at j ^ r % 8 (no bank conflicts either way).  8 x (8192 + 1024) tokens at
// d = 128: 1156 -> 1112 us; d = 256 (stores alone: its queries go to tensor memory, and the exchange on the way there cost 1.1 us of a
// tile's start through a buffer that has to be added): 501 -> 495 us a pass over windowed layers; latent: 212 -> 204 us.
constexpr int kRowsBytes = 32 * 128;
__device__ __forceinline__ uint32_t piece_at(int row, int piece) { return (uint32_t)(row * 128 + ((piece ^ (row & 7)) << 4)); }
// The query rows 8 g + lane % 8, g < 4, of the warp's 32 (nullptr: no such query).  Row r of a tile is query r % tile_q of head r / tile_q.
struct RowsIn { const uint16_t* row[4]; };
__device__ __forceinline__ RowsIn rows_in(const uint16_t* q, int tile_row, int tile_q, int i_first, int q0, int q_len, int Hq, int head0, int n_rep,
                                          int d, bool none) {
  RowsIn in;
  const float per = __fdividef(1.f, (float)tile_q);
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    const int r = tile_row + 8 * g + ((int)threadIdx.x & 7), h = (int)(((float)r + 0.5f) * per), i = i_first + r - h * tile_q;   // r < 256: exact
    in.row[g] = i < q_len && h < n_rep && !none ? q + ((size_t)(q0 + i) * Hq + head0 + h) * d : nullptr;
  }
  return in;
}
__device__ __forceinline__ uint4 piece_of(const uint16_t* row, int p) {
  return row ? *reinterpret_cast<const uint4*>(row + 8 * p) : make_uint4(0u, 0u, 0u, 0u);
}
// The first kCount pieces of all rows, shared out: w[k] is piece 4 (k / 4) + lane / 8 of row 8 (k % 4) + lane % 8.
template <int kCount>
__device__ __forceinline__ void load_rows(const RowsIn& in, uint4* w) {
#pragma unroll
  for (int k = 0; k < kCount; ++k) w[k] = piece_of(in.row[k & 3], 4 * (k >> 2) + (((int)threadIdx.x & 31) >> 3));
}
// Where a warp's rows go: element `at` on of the output for this lane's row, if it is `mine` to write.  A store covers 8 rows of
// bfloat16 or 4 of binary32.
struct RowsOut { size_t base; int rel[8]; unsigned there; bool bf16; };
__device__ __forceinline__ RowsOut rows_out(size_t at, bool mine, bool bf16) {
  const int lane = threadIdx.x & 31;
  const unsigned rows = __ballot_sync(0xffffffffu, mine);
  RowsOut o;
  o.bf16 = bf16;
  o.base = __shfl_sync(0xffffffffu, (unsigned long long)at, rows ? __ffs(rows) - 1 : 0);
  o.there = 0u;
  const int rel = (int)(long long)(at - o.base);         // inside a tile's output
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int r = bf16 ? 8 * (k & 3) + (lane >> 2) : 4 * k + (lane >> 3);
    o.rel[k] = __shfl_sync(0xffffffffu, rel, r) + (bf16 ? 8 * (lane & 3) : 4 * (lane & 7));
    o.there |= ((rows >> r) & 1u) << k;
  }
  return o;
}
// 32 elements of every row, from `first` on: x is this lane's.
__device__ __forceinline__ void store_rows(uint8_t* buf, const float (&x)[32], const RowsOut& o, void* out, int first) {
  const int lane = threadIdx.x & 31;
  __syncwarp();                                          // what was in the buffer has been read
  if (o.bf16) {
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      uint32_t w[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const __nv_bfloat162 b = __floats2bfloat162_rn(x[8 * p + 2 * e], x[8 * p + 2 * e + 1]);
        w[e] = *reinterpret_cast<const uint32_t*>(&b);
      }
      *reinterpret_cast<uint4*>(buf + piece_at(lane, p)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint4 v = *reinterpret_cast<const uint4*>(buf + piece_at(8 * k + (lane >> 2), lane & 3));
      if ((o.there >> k) & 1u) *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(out) + o.base + first + o.rel[k]) = v;
    }
  } else {
#pragma unroll
    for (int p = 0; p < 8; ++p) *reinterpret_cast<float4*>(buf + piece_at(lane, p)) = make_float4(x[4 * p], x[4 * p + 1], x[4 * p + 2], x[4 * p + 3]);
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float4 v = *reinterpret_cast<const float4*>(buf + piece_at(4 * k + (lane >> 3), lane & 7));
      if ((o.there >> k) & 1u) *reinterpret_cast<float4*>(reinterpret_cast<float*>(out) + o.base + first + o.rel[k]) = v;
    }
  }
}

// The agents that bring one query in a batch where others bring more are left to the decode kernel, which is launched next
// on the same stream; its arrival counters are cleared here, so that the caller need not hand over a cleared workspace.
__device__ inline void clear_tickets(const PrefillExtra& x) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  for (int i = threadIdx.x; i < x.n_tickets; i += blockDim.x) x.tickets[i] = 0;
}

}  // namespace prefill
}  // namespace q4kv
