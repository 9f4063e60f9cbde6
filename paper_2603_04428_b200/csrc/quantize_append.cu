// q4kv_quantize_append: affine 4-bit group quantization of new K/V rows, written in place
// into the agents' pool blocks (Section 3.2 format; Section 3.4 "update" step).
//
// Work unit = one "octet": the (up to) eight cache positions of one agent that share
// position/8, for one KV head.  An octet is the unit because the V codes are stored
// token-packed (eight tokens per word): one CTA owns every word it read-modify-writes.
// Eight consecutive lanes own one 64-element group (eight elements each) and reduce
// min/max with three shuffles.  Every arithmetic step is a single rounded binary32
// operation in the documented order so that codes/scales/biases are reproducible.
#include <algorithm>

#include "f32x2.cuh"
#include "q4kv_layout.cuh"
#include "quantize_core.cuh"

namespace q4kv {

namespace {

constexpr int kThreads = 256;
constexpr int kItemBytes = 8 * 4 * 128;                  // eight positions, four groups (see the bulk kernel)

struct UnitInfo { int agent, first, cnt, row0, block; };

// Warp 0: find the (agent, octet) of unit u: agent a has ceil((pos%8 + n_a)/8) octets.  The lanes look at 32
// agents at a time, so the lengths arrive in one round trip instead of one per agent.
__device__ inline void find_unit(int u, int n_agents, int max_blocks, int n_blocks, const int32_t* __restrict__ tables,
                                 const int32_t* __restrict__ pos, const int32_t* __restrict__ new_offs, int32_t* flags,
                                 bool report_bad_len, UnitInfo* out) {
  const int lane = threadIdx.x & 31;
  int cum = 0;
  bool found = false;
  for (int base = 0; base < n_agents && !found; base += 32) {
    const int a = base + lane;
    int p = 0, r0 = 0, n = 0, octs = 0;
    bool bad_len = false;
    if (a < n_agents) {
      p = pos[a]; r0 = new_offs[a]; n = new_offs[a + 1] - r0;
      if (n > 0) {
        if (p < 0 || (long long)p + n > (long long)max_blocks * kBlockTokens) bad_len = true;
        else octs = ((p & 7) + n + 7) >> 3;
      }
    }
    if (__any_sync(0xffffffffu, bad_len) && lane == 0 && report_bad_len) raise_flag(flags, Q4KV_FLAG_BAD_LENGTH);
    int inc = octs;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    const int tot = __shfl_sync(0xffffffffu, inc, 31);
    if (u < cum + tot) {
      found = true;
      const unsigned bal = __ballot_sync(0xffffffffu, cum + inc > u);
      if (lane == __ffs(bal) - 1) {
        const int uu = u - (cum + inc - octs);
        const int lo = max(p, ((p >> 3) + uu) << 3);
        const int hi = min(p + n, (((p >> 3) + uu) << 3) + 8);
        int who = a;
        const int blk = tables[(size_t)a * max_blocks + (lo >> 8)];
        if (blk < 0 || blk >= n_blocks) { raise_flag(flags, Q4KV_FLAG_BAD_BLOCK); who = -1; }
        out->agent = who; out->first = lo; out->cnt = hi - lo; out->row0 = r0 + (lo - p); out->block = blk;
      }
    }
    cum += tot;
  }
  if (!found && lane == 0) out->agent = -1;
}

// grid: (unit upper bound, Hkv); a CTA handles one octet.  Dynamic smem: 8 * Dv bytes of V codes (one byte per code).  Phases of
// many tokens per agent take the bulk kernel further down; this kernel serves the appends of a few tokens per agent.  Its time is a
// chain of latencies -- the predecessor's end, the rows, the quantizer, the value words --, so the value words that are patched are
// fetched beside the rows, and only the tokens there are get threads.  One token of each of 12 agents, us a launch: 8 KV heads
// 2.9 -> 2.2, d = 256 3.7 -> 2.0, 16 heads at 192 / 128 4.6 -> 2.3, latent cache 2.7 -> 1.8 (before: a thread for every word that eight tokens
// would have, two divisions each, the value words fetched at the end, a grid for two octets more per agent).  Several octets per CTA, and
// one octet for all KV heads per CTA, were slower on phases: 37 -> 63 us for the latter on 8 x 1024 tokens.
constexpr int kMaxDv = 512;
__global__ void __launch_bounds__(kThreads)
quantize_append_kernel(Layout y, uint8_t* pool, int n_blocks, int layer, int n_agents, int max_blocks,
                       const int32_t* __restrict__ tables, const int32_t* __restrict__ pos,
                       const int32_t* __restrict__ new_offs, const void* k_new, const void* v_new, int32_t* flags) {
  extern __shared__ uint8_t vcodes[];       // [8][Dv]
  __shared__ UnitInfo s_unit;
  // (k_new, v_new carry no __restrict__: the preceding kernel may write them while this one is resident, and read-only loads are
  // not defined for such data.)
  // let the next kernel of the stream start its prologue; the unit is found from the lengths and block tables (inputs
  // that no kernel writes) while the preceding kernels drain, and the wait comes before the new rows and the pool
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (threadIdx.x < 32)
    find_unit(blockIdx.x, n_agents, max_blocks, n_blocks, tables, pos, new_offs, flags, blockIdx.x == 0 && blockIdx.y == 0, &s_unit);
  __syncthreads();
  const UnitInfo un = s_unit;
  const int hk = blockIdx.y;
  const int kw = y.D / 8, per = kw + (y.alias ? 0 : y.Dv / 8);           // words of a token: K, then V
  const int slot0 = un.first & 255;                     // the octet lies inside one 32-token chunk
  uint8_t* const chunk = head_block(pool, y, layer, un.agent < 0 ? 0 : un.block, hk) + (size_t)(slot0 >> 5) * y.chunk_bytes;
  uint32_t* const vc = reinterpret_cast<uint32_t*>(chunk + y.off_vc);
  // while the preceding kernel drains, L2 is asked for the first token's rows and the value words (a prefetch returns nothing)
  if (un.agent >= 0) {
    const size_t row = (size_t)un.row0 * y.Hkv + hk;
    const int lines_k = y.D / 64, lines = y.alias ? lines_k : lines_k + y.Dv / 64 + y.Dv / 8;
    for (int i = threadIdx.x; i < lines; i += kThreads) {
      const void* at = i < lines_k ? (const void*)((const uint16_t*)k_new + row * y.D + 64 * i)
                     : i < lines_k + y.Dv / 64 ? (const void*)((const uint16_t*)v_new + row * y.Dv + 64 * (i - lines_k))
                                               : (const void*)(vc + 32 * (i - lines_k - y.Dv / 64));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(at));
    }
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (un.agent < 0) return;                             // uniform over the CTA
  uint32_t old[kMaxDv / kThreads] = {};
  if (!y.alias && un.cnt < 8) {
#pragma unroll
    for (int r = 0; r < kMaxDv / kThreads; ++r) {
      const int d = threadIdx.x + kThreads * r;
      if (d < y.Dv) old[r] = vc[v_word_offset((slot0 & 31) >> 3, d)];
    }
  }
  // ---- K and V rows in one sweep: items (token i, word w), eight lanes per group.  K words and
  // scale/bias pairs go straight to the pool; V codes go to shared memory as bytes for the transposition. ----
  const int n_items = un.cnt * per;
  for (int base = 0; base < n_items; base += kThreads) {
    const int idx = base + threadIdx.x;
    const bool live = idx < n_items;
    const int i = un.cnt == 1 ? 0 : idx / per, ww = idx - i * per;       // (eight lanes of a group: per is a multiple of eight)
    const bool is_v = ww >= kw;
    const int w = is_v ? ww - kw : ww;
    float x[8];
    if (live) {
      const size_t row = (size_t)(un.row0 + i) * y.Hkv + hk;
      if (is_v) load_eight_bf16(v_new, row * y.Dv + 8 * w, x);
      else load_eight_bf16(k_new, row * y.D + 8 * w, x);
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) x[e] = 0.f;
    }
    const QuantOut o = quantize_eight(x, y.sb_bf16 != 0);
    if (!live) continue;
    const int tau = (slot0 & 31) + i;
    if (is_v) {
#pragma unroll
      for (int e = 0; e < 8; ++e) vcodes[i * y.Dv + 8 * w + e] = (o.word >> (4 * e)) & 15u;
      if ((w & 7) == 0) reinterpret_cast<uint32_t*>(chunk + y.off_vsb)[sb_offset(tau, w >> 3, y.Gv)] = o.sb;
    } else {
      reinterpret_cast<uint32_t*>(chunk + y.off_kc)[k_word_offset(tau, w, y.G)] = o.word;
      if ((w & 7) == 0) reinterpret_cast<uint32_t*>(chunk + y.off_ksb)[sb_offset(tau, w >> 3, y.G)] = o.sb;
    }
  }
  if (y.alias) return;
  __syncthreads();
  // ---- token-packed V words: one word = one head-dim element of the octet's 8 positions ----
  const int k0 = un.first & 7;                           // nibble of the first new token inside the word
  const uint32_t mask = un.cnt == 8 ? 0xffffffffu : ((1u << (4 * un.cnt)) - 1u) << (4 * k0);
#pragma unroll
  for (int r = 0; r < kMaxDv / kThreads; ++r) {
    const int d = threadIdx.x + kThreads * r;
    if (d >= y.Dv) break;
    uint32_t bits = 0;
    for (int i = 0; i < un.cnt; ++i) bits |= (uint32_t)vcodes[i * y.Dv + d] << (4 * (k0 + i));
    vc[v_word_offset((slot0 & 31) >> 3, d)] = (old[r] & ~mask) | bits;
  }
}

// ---------------------------------------------------------------------------------------------
// Bulk form (a prefill phase: many new tokens per agent).  kWpc warps own one (32-token chunk, KV head) unit and walk its
// items -- four (octet of eight positions, group) pairs, K groups first, then V groups -- with the next item's rows on their way
// into shared memory while the current one is quantized.  Within an item a lane owns one of the eight positions and
// one 64-element group: it reads its 64 elements as eight 16-byte words, takes minimum and maximum with packed bf16
// instructions (no cross-lane step at all), and quantizes them two at a time (packed binary32; see quantize_code for why the
// codes equal those of the fixed sequence bit for bit).  V words
// are first exchanged between the eight lanes of a group (an 8 x 8 transposition of words by twelve shuffles), which leaves
// in each lane the 8 positions x 8 elements block of nibbles that an in-register transposition turns into eight token-packed
// words.  The chunk is assembled in shared memory and stored as whole 16-byte pieces; a chunk that the phase fills only in
// part (an unaligned start or end) starts from its present bytes.
// Bound by instruction issue (about 16 instructions an element) with the sixteen warps an SM has room for.  Measured, each lane
// loading its own rows (32 lines per load) -> rows copied whole lines at a time: d = 128, 8 KV heads, 8 x 1024 tokens 16.6 -> 15.8 us,
// 8 x 4096 55.8 -> 48.7; d = 256 97.7 -> 84.4; 192 / 128, where an item was four groups of one octet, 16 KV heads, 8 x 1024 53.1 ->
// 37.4; latent cache 8 x 4096 21.2 -> 18.3.  Three CTAs per SM of 80 registers: 21.8 us on the first.  kWpc = 1 where the units fill the
// GPU and two CTAs' chunks fit an SM; 4 otherwise and for smaller phases, whose time is one unit's chain of items: 5 x 64 tokens 12.8 ->
// 4.7 us.
// ---------------------------------------------------------------------------------------------
__device__ inline void transpose_nibbles_8x8_regs(uint32_t (&r)[8]) {
  // rows = registers, columns = nibbles: three rounds of block swaps
#pragma unroll
  for (int s = 1; s < 8; s <<= 1) {
    const uint32_t m = s == 1 ? 0x0F0F0F0Fu : s == 2 ? 0x00FF00FFu : 0x0000FFFFu;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      if (t & s) continue;
      const uint32_t x = ((r[t] >> (4 * s)) ^ r[t + s]) & m;
      r[t + s] ^= x;
      r[t] ^= x << (4 * s);
    }
  }
}

// The eight codes of a word for a (bfloat16) scale without a finite reciprocal.
__device__ __noinline__ uint32_t divided_word(uint4 raw, GroupScale gs, float inv) {
  const uint32_t wv[4] = {raw.x, raw.y, raw.z, raw.w};
  uint32_t word = 0u;
#pragma unroll
  for (int e = 0; e < 4; ++e)
    word |= (quantize_code(__uint_as_float(wv[e] << 16), gs, inv) | (quantize_code(__uint_as_float(wv[e] & 0xffff0000u), gs, inv) << 4)) << (8 * e);
  return word;
}

// Unit of the bulk kernel: one 32-token chunk of one agent's new range (up to four octets, all in one pool block).
struct ChunkUnit { int agent, p, n, r0, chunk, block; };

// Warp-wide: find the (agent, chunk) of unit u; agent a has chunk(p + n - 1) - chunk(p) + 1 units.
__device__ inline void find_chunk_unit(int u, int n_agents, int max_blocks, int n_blocks, const int32_t* __restrict__ tables,
                                       const int32_t* __restrict__ pos, const int32_t* __restrict__ new_offs, int32_t* flags,
                                       bool report_bad_len, ChunkUnit* out) {
  const int lane = threadIdx.x & 31;
  int cum = 0;
  bool found = false;
  for (int base = 0; base < n_agents && !found; base += 32) {
    const int a = base + lane;
    int p = 0, r0 = 0, n = 0, cnt = 0;
    bool bad_len = false;
    if (a < n_agents) {
      p = pos[a]; r0 = new_offs[a]; n = new_offs[a + 1] - r0;
      if (n > 0) {
        if (p < 0 || (long long)p + n > (long long)max_blocks * kBlockTokens) bad_len = true;
        else cnt = ((p + n - 1) >> 5) - (p >> 5) + 1;
      }
    }
    if (__any_sync(0xffffffffu, bad_len) && lane == 0 && report_bad_len) raise_flag(flags, Q4KV_FLAG_BAD_LENGTH);
    int inc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    const int tot = __shfl_sync(0xffffffffu, inc, 31);
    if (u < cum + tot) {
      found = true;
      const unsigned bal = __ballot_sync(0xffffffffu, cum + inc > u);
      if (lane == __ffs(bal) - 1) {
        const int c = (p >> 5) + (u - (cum + inc - cnt));
        int who = a;
        const int blk = tables[(size_t)a * max_blocks + (c >> 3)];
        if (blk < 0 || blk >= n_blocks) { raise_flag(flags, Q4KV_FLAG_BAD_BLOCK); who = -1; }
        out->agent = who; out->p = p; out->n = n; out->r0 = r0; out->chunk = c; out->block = blk;
      }
    }
    cum += tot;
  }
  if (!found && lane == 0) out->agent = -1;
}

// kFour: four groups per token, so that an item is one octet (fewer instructions for the common shape).  kRing: the rows come through
// shared memory; else (few units) a lane loads its own.
template <int kWpc, bool kFour, bool kRing>
__global__ void __launch_bounds__(kThreads, 2)
quantize_append_bulk_kernel(Layout y, uint8_t* pool, int n_blocks, int layer, int n_agents, int max_blocks,
                            const int32_t* __restrict__ tables, const int32_t* __restrict__ pos,
                            const int32_t* __restrict__ new_offs, const uint16_t* k_new, const uint16_t* v_new,
                            int32_t* flags, int units) {
  __shared__ ChunkUnit s_unit[kThreads / 32];
  extern __shared__ __align__(16) uint8_t stage_all[];  // one chunk per warp
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sub = warp % kWpc;                           // this warp of the unit
  const int gw = (blockIdx.x * (kThreads / 32) + warp) / kWpc;
  const int u = gw / y.Hkv, hk = gw - u * y.Hkv;
  if (u >= units) return;
  find_chunk_unit(u, n_agents, max_blocks, n_blocks, tables, pos, new_offs, flags, gw == 0 && sub == 0, &s_unit[warp]);
  __syncwarp();
  const ChunkUnit un = s_unit[warp];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (un.agent < 0) return;
  auto unit_sync = [&]() {
    if (kWpc == 1) __syncwarp(); else asm volatile("bar.sync %0, %1;" ::"r"(1 + warp / kWpc), "n"(32 * kWpc) : "memory");
  };

  const int s = lane & 7, gq0 = lane >> 3;             // position slot inside an octet, group inside a pass
  const int c0 = un.chunk << 5;                          // first cache position of the chunk
  const int lo = max(un.p, c0), hi = min(un.p + un.n, c0 + 32);
  const int o_first = (lo - c0) >> 3, o_last = (hi - 1 - c0) >> 3;
  // The chunk is put together in shared memory and leaves as whole 16-byte pieces (the words of a token are scattered
  // over the chunk: stored one by one they would reach L2 as a million and a half partial sectors per phase).  A
  // chunk that this phase fills only in part starts from its present bytes; this warp is its only writer.
  uint8_t* gchunk = head_block(pool, y, layer, un.block, hk) + (size_t)(un.chunk & 7) * y.chunk_bytes;
  uint8_t* chunk = stage_all + (size_t)(warp / kWpc) * y.chunk_bytes;
  const int n16 = y.chunk_bytes / 16;
  const int n_groups = y.G + (y.alias ? 0 : y.Gv);
  const int n_items = ((o_last - o_first + 1) * n_groups + 3) >> 2;
  constexpr float kMagic = 12582912.0f;                  // 1.5 * 2^23: q + kMagic holds q rounded to nearest even in its low bits
  constexpr uint32_t kMagicSum = 0x4B400000u * (1u + 16u + 256u);           // what eight of them add to a word (e > 2: shifted out)

  // Item t: the (octet, group) pairs 4 t .. 4 t + 3 of the chunk, groups fastest, K before V; lanes 8 i .. 8 i + 7 have pair 4 t + i.  (A
  // pass of four groups per octet left three quarters of every second item of the five groups at 192 / 128 without work, and of every
  // third of the latent cache's nine.)  The 32 rows of 128 bytes (pair, position) come by asynchronous copies, a position at a time --
  // the lanes of a copy then cover whole lines, where a lane that loads its own row asks for a piece of 32 lines --, while the item
  // before is quantized; 16-byte piece j of a row of position s lies at j ^ s, so that neither the copies nor the reads of a row
  // per lane conflict.  Rows that do not exist are zeros.
  uint8_t* const ring = stage_all + (size_t)(kThreads / 32 / kWpc) * y.chunk_bytes + (size_t)warp * kItemBytes;
  const float per_group = __fdividef(1.f, (float)n_groups);
  struct Pair { int o, gq; bool has; };
  auto pair_of = [&](int t) {                            // at most 4 x 24 pairs: the float quotient is exact
    if (kFour) return Pair{o_first + t, gq0, true};
    const int v = 4 * t + gq0, oo = (int)(((float)v + 0.5f) * per_group);
    return Pair{o_first + oo, v - oo * n_groups, o_first + oo <= o_last};
  };
  auto copy_item = [&](int t) {
    const Pair pr = pair_of(t);
    const int first = max(lo, c0 + 8 * pr.o), cnt = min(hi, c0 + 8 * pr.o + 8) - first, k0 = first & 7;
    const int gq = pr.gq;
    const bool is_v = gq >= y.G, has = pr.has;
    const uint16_t* const rows = is_v ? v_new + 64 * (gq - y.G) : k_new + 64 * gq;
    const size_t width = is_v ? y.Dv : y.D;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(ring + gq0 * 128);
    const size_t row0 = (size_t)(un.r0 + (first - un.p)) * y.Hkv + hk;
#pragma unroll
    for (int k = 0; k < 8; ++k) {                        // position k, piece s of this lane's group
      const bool real = has && k >= k0 && k < k0 + cnt;
      const uint16_t* src = real ? rows + (row0 + (size_t)(k - k0) * y.Hkv) * width + 8 * s : k_new;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + (uint32_t)(k * 512 + ((s ^ k) << 4))), "l"(src), "r"(real ? 16 : 0)
                   : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto load_item = [&](int t, uint4 (&raw)[8]) {
    const Pair pr = pair_of(t);
    const int first = max(lo, c0 + 8 * pr.o), cnt = min(hi, c0 + 8 * pr.o + 8) - first, i = s - (first & 7);
    const bool is_v = pr.gq >= y.G, real = pr.has && i >= 0 && i < cnt;
    const size_t row = (size_t)(un.r0 + (first - un.p) + i) * y.Hkv + hk;
    const uint4* const src = reinterpret_cast<const uint4*>(is_v ? v_new + row * y.Dv + 64 * (pr.gq - y.G) : k_new + row * y.D + 64 * pr.gq);
#pragma unroll
    for (int j = 0; j < 8; ++j) raw[j] = real ? __ldca(src + j) : make_uint4(0u, 0u, 0u, 0u);
  };
  uint4 raw[8];
  // On its way while the chunk's present bytes are fetched (behind them: 3 x 300 tokens at 8 KV heads 6.3 us a launch, now 5.8; 5 x 64 on
  // 1003 cached ones 6.1, now 5.8; and the registers did not suffice by three words)
  if (kRing && sub < n_items) copy_item(sub);
  if (lo != c0 || hi != c0 + 32) {
    for (int q = lane + 32 * sub; q < n16; q += 32 * kWpc) reinterpret_cast<uint4*>(chunk)[q] = reinterpret_cast<const uint4*>(gchunk)[q];
    unit_sync();
  }
  if (!kRing && sub < n_items) load_item(sub, raw);
  for (int t = sub; t < n_items; t += kWpc) {
    uint4 nxt[kRing ? 1 : 8];
    if constexpr (kRing) {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncwarp();
#pragma unroll
      for (int j = 0; j < 8; ++j) raw[j] = *reinterpret_cast<const uint4*>(ring + s * 512 + gq0 * 128 + ((j ^ s) << 4));
      __syncwarp();                                      // the whole warp has its rows: the next item's may come
      if (t + kWpc < n_items) copy_item(t + kWpc);
    } else if (t + kWpc < n_items) {
      load_item(t + kWpc, nxt);
    }
    const Pair pr = pair_of(t);
    const int o = pr.o, gq = pr.gq;
    const int first = max(lo, c0 + 8 * o), cnt = min(hi, c0 + 8 * o + 8) - first;
    const int k0 = first & 7;
    const int i = s - k0;                                // this lane's token of the octet
    const bool tok = i >= 0 && i < cnt;
    const int tau = 8 * o + s;                           // chunk token of this lane's position
    const uint32_t nib_mask = cnt == 8 ? 0xFFFFFFFFu : (((1u << (4 * cnt)) - 1u) << (4 * k0));
    const bool has = pr.has;
    const bool is_v = has && gq >= y.G;
    const int gi = is_v ? gq - y.G : gq;
    const bool active = has && tok;
    // minimum and maximum of the 64 elements on packed bf16 (values are exact, so this is the binary32 result)
    __nv_bfloat162 mn2 = *reinterpret_cast<const __nv_bfloat162*>(&raw[0].x), mx2 = mn2;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t wv[4] = {raw[j].x, raw[j].y, raw[j].z, raw[j].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162*>(&wv[e]);
        mn2 = __hmin2(mn2, v);
        mx2 = __hmax2(mx2, v);
      }
    }
    const uint32_t mnb = *reinterpret_cast<const uint32_t*>(&mn2), mxb = *reinterpret_cast<const uint32_t*>(&mx2);
    const float mn = fminf(__uint_as_float(mnb << 16), __uint_as_float(mnb & 0xffff0000u));
    const float mx = fmaxf(__uint_as_float(mxb << 16), __uint_as_float(mxb & 0xffff0000u));
    const GroupScale gs = group_scale(mn, mx, y.sb_bf16 != 0);
    uint32_t cw[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) cw[j] = 0u;
    if (gs.sf != 0.0f) {
      const float inv = __frcp_rn(gs.sf);
      const uint64_t nb2 = pair64(-gs.bf, -gs.bf), inv2 = pair64(inv, inv), ns2 = pair64(-gs.sf, -gs.sf), up2 = pair64(kMagic, kMagic);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint32_t wv[4] = {raw[j].x, raw[j].y, raw[j].z, raw[j].w};
        // quantize_code, two elements at a time; the quotient is at most 15 + a few ulps by construction of the scale, hence
        // no clamp
        uint32_t m[8];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const uint64_t t = add2(pair64(__uint_as_float(wv[e] << 16), __uint_as_float(wv[e] & 0xffff0000u)), nb2);
          const uint64_t q = mul2(t, inv2);
          const float2 r = unpair64(add2(fma2(fma2(ns2, q, t), inv2, q), up2));
          m[2 * e] = __float_as_uint(r.x); m[2 * e + 1] = __float_as_uint(r.y);
        }
        // (m0 + 16 m1) + 256 (m2 + 16 m3) + ...: sums of the low bits, the rest being known
        const uint32_t w01 = m[1] * 16u + m[0], w23 = m[3] * 16u + m[2], w45 = m[5] * 16u + m[4], w67 = m[7] * 16u + m[6];
        cw[j] = (w67 * 256u + w45) * 65536u + (w23 * 256u + w01) - kMagicSum;
      }
      if (inv > 3.0e38f) {
#pragma unroll
        for (int j = 0; j < 8; ++j) cw[j] = divided_word(raw[j], gs, inv);
      }
    }
    const uint32_t sb = gs.hs | (gs.hb << 16);
    if (active && !is_v) {
      // words w = 8 gi + 4 i2 + t sit in 16-byte pieces of four (group, half) words: this lane's pair is 8 bytes
      uint32_t* kc = reinterpret_cast<uint32_t*>(chunk + y.off_kc);
#pragma unroll
      for (int w = 0; w < 4; ++w)
        *reinterpret_cast<uint2*>(kc + k_word_offset(tau, 8 * gi + w, y.G)) = make_uint2(cw[w], cw[4 + w]);
      reinterpret_cast<uint32_t*>(chunk + y.off_ksb)[sb_offset(tau, gi, y.G)] = sb;
    }
    if (kFour ? !y.alias : __any_sync(0xffffffffu, is_v)) {             // not K groups only
      if (active && is_v) reinterpret_cast<uint32_t*>(chunk + y.off_vsb)[sb_offset(tau, gi, y.Gv)] = sb;
      // 8 x 8 transposition of words between the eight lanes of a group: afterwards lane s holds, in cw[w], word s
      // (elements 8s .. 8s+7 of the group) of position w
#pragma unroll
      for (int b = 4; b > 0; b >>= 1) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (j & b) continue;
          const uint32_t send = (s & b) ? cw[j] : cw[j | b];
          const uint32_t recv = __shfl_xor_sync(0xffffffffu, send, b);
          if (s & b) cw[j] = recv; else cw[j | b] = recv;
        }
      }
      transpose_nibbles_8x8_regs(cw);                    // cw[e]: element 8s + e of the group, nibble w = position w
      if (is_v) {
        uint32_t* vc = reinterpret_cast<uint32_t*>(chunk + y.off_vc);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          uint32_t* at = vc + v_word_offset(o, 64 * gi + 8 * s + e);
          *at = nib_mask == 0xFFFFFFFFu ? cw[e] : ((*at & ~nib_mask) | (cw[e] & nib_mask));
        }
      }
    }
    if constexpr (!kRing) {
#pragma unroll
      for (int j = 0; j < 8; ++j) raw[j] = nxt[j];
    }
  }
  unit_sync();
  for (int q = lane + 32 * sub; q < n16; q += 32 * kWpc) reinterpret_cast<uint4*>(gchunk)[q] = reinterpret_cast<const uint4*>(chunk)[q];
}

constexpr size_t kBulkSmem = 112 * 1024;                 // two CTAs per SM
size_t bulk_smem(const Layout& y, int wpc, bool ring = true) {
  return (size_t)(kThreads / 32 / wpc) * y.chunk_bytes + (ring ? (size_t)(kThreads / 32) * kItemBytes : 0);
}

template <int kWpc, bool kFour, bool kRing = true>
cudaError_t launch_bulk(const Layout& y, uint8_t* pool, int n_blocks, int layer, const q4kv_batch& b, const int32_t* pos,
                        const int32_t* new_offs, int chunk_units, const void* k_new, const void* v_new, int32_t* flags,
                        cudaStream_t st) {
  const long long warps = (long long)chunk_units * y.Hkv * kWpc;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((warps + kThreads / 32 - 1) / (kThreads / 32)));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = bulk_smem(y, kWpc, kRing);
  cfg.stream = st;
  static bool configured[64] = {};     // the attribute is per function and device: set it once for each
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    e = cudaFuncSetAttribute(quantize_append_bulk_kernel<kWpc, kFour, kRing>, cudaFuncAttributeMaxDynamicSharedMemorySize, kBulkSmem);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, quantize_append_bulk_kernel<kWpc, kFour, kRing>, y, pool, n_blocks, layer, b.n_agents, b.max_blocks,
                            b.block_tables, pos, new_offs, (const uint16_t*)k_new, (const uint16_t*)v_new, flags, chunk_units);
}

cudaError_t launch_octets(const Layout& y, uint8_t* pool, int n_blocks, int layer, const q4kv_batch& b, const int32_t* pos,
                          const int32_t* new_offs, int units, const void* k_new, const void* v_new, int32_t* flags,
                          cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(units, y.Hkv);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = y.alias ? 0 : (size_t)8 * y.Dv;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, quantize_append_kernel, y, pool, n_blocks, layer, b.n_agents, b.max_blocks,
                            b.block_tables, pos, new_offs, k_new, v_new, flags);
}

}  // namespace

cudaError_t launch_quantize_append(const Layout& y, void* pool, int n_blocks, int layer, const q4kv_batch& b,
                                   const int32_t* pos, const int32_t* new_offs, int total_new,
                                   const void* k_new, const void* v_new, int32_t* flags, cudaStream_t st) {
  if (total_new <= 0 || b.n_agents <= 0) return cudaSuccess;
  // >= sum over agents of ceil((pos%8+n)/8): n tokens touch at most n octets, and at most n / 8 + 2
  const int units = std::min(total_new, total_new / 8 + 2 * b.n_agents);
  if (total_new >= 8 * b.n_agents && (size_t)(kThreads / 32) * y.chunk_bytes <= kBulkSmem) {
    // a phase of many tokens per agent: one warp per (32-token chunk, KV head)
    const int chunk_units = total_new / 32 + 2 * b.n_agents;   // >= sum over agents of the chunks their new range touches
    // four warps per unit while one warp each would leave half of the resident warps (sixteen per SM) without work
    const long long all_units = (long long)chunk_units * y.Hkv;
    const bool four = all_units < 8ll * sm_count() || bulk_smem(y, 1) > kBulkSmem;
    // One unit or less for every two SMs, and not four groups a token: lanes load their own rows, which takes fewer steps and leaves
    // the next launch's CTAs their shared memory.  16 layers, us, through shared memory and without: latent cache 1 x 64 tokens (4 units)
    // 101.6 / 89.3, 4 x 500 (70) 120.6 / 118.4, 6 x 500 (105) 145.1 / 145.0, 6 x 1000 135.3 / 137.4; d = 256 1 x 44 (24) 104.2 / 99.9, 2 x 128
    // (96) 131.8 / 137.1; 192 / 128 2 x 64 (128) 109.2 / 112.0.  Before attention, four layers: d = 256, 44 tokens 81.3 / 75.7, 192 / 128, 56
    // tokens (48) 92.3 / 90.1.  Four groups a token (an item is an octet, a warp has one): 5 x 64 tokens 75.7 / 86.9, 2 x 100 79.5 / 84.6.
    const bool few = 2 * all_units <= sm_count();
    const auto launch = y.G + (y.alias ? 0 : y.Gv) == 4 ? (four ? launch_bulk<4, true> : launch_bulk<1, true>)
                        : few ? launch_bulk<4, false, false> : (four ? launch_bulk<4, false> : launch_bulk<1, false>);
    return launch(y, (uint8_t*)pool, n_blocks, layer, b, pos, new_offs, chunk_units, k_new, v_new, flags, st);
  }
  return launch_octets(y, (uint8_t*)pool, n_blocks, layer, b, pos, new_offs, units, k_new, v_new, flags, st);
}

}  // namespace q4kv
