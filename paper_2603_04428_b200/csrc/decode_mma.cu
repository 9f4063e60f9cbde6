// q4kv_decode_attention, tensor-core path for GQA shapes (d_qk = d_v in {128, 256}, or d_qk 192 with d_v 128): one
// query token per agent over its whole Q4 cache, read in place (Section 3.4 "Batched Quantized Inference": fused
// attention on the Q4 tensors; Section 3.6: GQA head mapping and sliding-window layers).
//
// The floor is HBM bandwidth; what a launch of a few MB per SM actually spends is latency (the first bytes, the merge of
// the partial results at its end) and instruction issue (about 450 warp instructions per 32-token chunk at d = 128).  So:
//   * Work = the list of 32-token chunks of all (agent, KV head) pairs inside their key range [lo, kv_len), cut into
//     contiguous ranges, one per CTA.  Where that costs few chunks (kWholeSlack) every pair is cut into equal parts of its
//     own and a CTA holds one part; otherwise the list is cut into equal ranges, so that ragged lengths balance by
//     construction, and a CTA may hold parts of several pairs ("segments").  A pair that lies inside one CTA is finished
//     there; otherwise every CTA that holds a piece writes a partial (acc, m, l) record and takes a ticket, and the CTA
//     that draws the pair's last ticket combines the records -- one launch, no waiting on other CTAs.
//   * Eight warps per CTA, two CTAs per SM, 128 registers: four warps per scheduler.  One warp's chunk is one dependent
//     chain (wait, products, maximum, exponentials, transposes, products), so the schedulers need that many to keep
//     busy; the earlier form with two (seven consumer warps of 255 registers and a planner warp) issued 0.45
//     instructions per scheduler and clock.  A second CTA also works through the first one's barriers and merges.
//   * The chunks of a CTA's range are dealt to its warps in turn, and every warp streams its own through its own slots
//     with one bulk asynchronous copy per chunk (a chunk is one contiguous byte range of the pool; two copies at
//     d = 256, keys and values, so that the key half is refilled while the values are in work).  Pool offsets are
//     looked up 32 chunks at a time, one per lane, before the warp needs them.  No two warps share a slot, so there
//     is nothing to hand over; warps meet only at the end of a segment.
//   * Arithmetic runs on the 4-bit codes, not on dequantized values.  With x^ = c*s + b and one
//     (s, b) per token and 64-element group,
//         q.k_t   = sum_g [ s_tg * (sum_{d in g} q_d c_td) + b_tg * (sum_{d in g} q_d) ]
//         (p.V)_d = sum_t (p_t s_tg(d)) c_td + sum_t p_t b_tg(d).
//     Both contractions are mma.sync m16n8k16 f16 with the code operand produced by masking the
//     packed word in place: a nibble in the low bits of a 16-bit lane IS the binary16 subnormal
//     c * 2^-24, and one nibble up it is 16c * 2^-24 -- the 16 is divided out of the other operand
//     (the matching query elements for q.K, the probabilities of odd key tiles for p.V).  The bf16
//     query is scaled per row by a power of two into binary16, so nothing is rounded before the
//     products, which are exact.  (The 8-bit float forms of mma.sync are not used: on this part
//     each costs two f16 tensor instructions plus conversions and adds.)
//   * In the score product the key codes are the A operand (16 tokens x 16 head-dim elements) and the query the B
//     operand, so a KV head's codes are unpacked once for all its query heads.  The probabilities times the token's
//     value scale enter the value product as a two-term binary16 split (accurate to ~2^-22), transposed across the warp
//     (movmatrix) into its B operand; the A operand is the token-packed value words.  Two forms by the eight columns of
//     the B operands: up to four query heads per KV head -- columns 4..7 repeat the heads in the score product and
//     carry the low halves of the split in the value product -- and, at d = 128, up to eight, the low halves in
//     products of their own.  More query heads per KV head are cut into equal sets (at most four heads wide, eight at
//     d = 128) that are attended like KV heads of their own and read the chunks again, from L2 for the most part.
// Measured per launch in a replayed step (before: the form with seven consumer warps and a planner): d = 128, 4 heads per
// KV head, 8 KV heads, agents x 4096 tokens: 1 agent 14.1 -> 8.9 us, 5 agents 17.5 -> 11.8 us (2.0 TB/s), 40 agents 72.9
// -> 49.8 us (3.8 TB/s); d = 256, 16 agents x 8192 tokens, 81.4 -> 72.1 us (4.2 TB/s); 8 query heads per KV head, 12 agents
// x 4096 tokens: 26 us with the append, 1.5 ms on the shape-agnostic kernel.
//   * The reference of a warp's online softmax is taken over the warp, and the accumulators are rescaled, only when one
//     vote says that some score outgrew it; it is then set kMargin above the maximum, so that it moves less often.
#include <climits>

#include "convert.cuh"
#include "q4kv_layout.cuh"
#include "quantize_core.cuh"
#include "tcgen05.cuh"

namespace q4kv {

namespace {

constexpr int kMaxGrid = 512;                          // upper bound on the grid (records are sized for it)
constexpr int kCtasPerSm = 2;
// warps per CTA: eight of 128 registers, or at d = 256, where the accumulators alone are 64, six of 168
__host__ __device__ constexpr int warps_of(int G) { return G == 4 ? 6 : 8; }
constexpr int kWholeSlack = 12;                        // see find_range
constexpr float kMargin = 0.35f;                       // see chunk_values
constexpr int kMaxRecords = 32;                        // a pair is cut over about this many CTAs at most (the merge reads them all)
constexpr uint32_t kSpinLimit = 1u << 22;              // bounded mbarrier waits (each try blocks a while in hardware)
constexpr uint32_t kMaskLo = 0x000F000Fu, kMaskHi = 0x00F000F0u;

// ---------------------------------------------------------------------------------------------
// PTX wrappers
// ---------------------------------------------------------------------------------------------

using tc::bulk_load, tc::mbar_arrive, tc::mbar_arrive_expect_tx, tc::mbar_init, tc::mbar_test_wait, tc::smem_u32;
// (without the suspension hint of the tcgen05 kernels' waits: every warp here waits for its own next bytes)
__device__ inline bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait: gives up after kSpinLimit tries or as soon as another warp has given up.
__device__ __noinline__ bool mbar_wait_long(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  for (uint32_t i = 0; i < kSpinLimit; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 63u) == 63u && *abort_flag) return false;
  }
  *abort_flag = 1;
  return false;
}
// Whole warp.  The usual case is that the bytes landed long ago (a blocking try costs more).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  if (__all_sync(0xffffffffu, mbar_test_wait(bar, parity))) return true;
  return __all_sync(0xffffffffu, mbar_wait_long(bar, parity, abort_flag));
}
__device__ inline void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ inline void prefetch_l2_bulk(const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
__device__ inline void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ inline void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ inline void mma_f16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// half2(lo = a, hi = b), both rounded toward zero
__device__ inline uint32_t f32x2_to_h2_rz(float a, float b) {
  uint32_t r;
  asm("cvt.rz.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(b), "f"(a));
  return r;
}

constexpr int kMaxLayersPerCall = 64;
struct DecodeParams {
  Layout y;
  const uint8_t* pool;
  int n_blocks, layer, n_agents, max_blocks, len_cap;
  // Several layers in one launch (the layer-batched entry): the work list runs over "virtual agents" v = li * n_real + a
  // (layer li of the call, real agent a).  q, out, lse, the new rows, the arrival counters and the partial records are
  // all indexed by v; lengths and block tables by a; the window and the pool layer by li.  n_agents = layer_count * n_real.
  int n_real, layer_count;
  int windows[kMaxLayersPerCall];   // sliding window of each layer of the call (0: none)
  const int32_t* tables;
  const int32_t* kv_lens;
  const uint16_t* q;          // bf16 [layer_count][A][Hq][D]
  float scale_log2;           // softmax_scale * log2(e)
  int Hkv, n_rep, sets;       // pairs are over sets of query heads: Hkv = y.Hkv * sets, n_rep = y.n_rep / sets
  int32_t* tickets;           // [A*Hkv], zero between calls
  float* partials;            // [A*Hkv + grid][n_rep][Dv + 4]
  void* out;
  int out_dtype;
  float* lse;
  int32_t* flags;
  const uint16_t* k_new;      // fused append: bf16 [A][Hkv][D] rows of the token at position kv_len - 1 (null: none)
  const uint16_t* v_new;
  const int32_t* q_offs;      // kSingles: see Params
};
// kSingles: the batch of a prefill call, in which this launch takes the agents with exactly one query (row q_offs[a]).  An
// instantiation of its own: the look-ups cost the others 1-4 % as a run-time branch.
template <bool kSinglesOnly>
struct Params : DecodeParams {
  static constexpr bool kSingles = kSinglesOnly;
};

// ---------------------------------------------------------------------------------------------
// Work list: chunks of all (agent, KV head) pairs, agent-major, then head, then chunk
// ---------------------------------------------------------------------------------------------
struct AgentRange { int n, lo, cf, nc; };   // keys [lo, n); chunks cf .. cf+nc-1

// len_cap: the host's bound on every length (at most max_blocks * 256); longer or negative lengths are rejected
template <class Par>
__device__ inline AgentRange agent_range(const Par& P, int a, bool& bad) {
  AgentRange r;
  const int li = P.layer_count > 1 ? a / P.n_real : 0;
  const int window = P.windows[li];
  r.n = P.kv_lens[a - li * P.n_real];
  bad = r.n < 0 || r.n > P.len_cap;
  if (Par::kSingles) {
    const bool one = P.q_offs[a + 1] - P.q_offs[a] == 1;
    bad = one && (bad || r.n < 1);
    if (!one) r.n = 0;
  }
  if (bad) r.n = 0;
  r.lo = window > 0 ? max(0, r.n - window) : 0;
  r.cf = r.lo >> 5;
  r.nc = r.n > r.lo ? ((r.n + 31) >> 5) - r.cf : 0;
  return r;
}

// Equal partition of U units over n CTAs (all quantities fit 31 bits; the host checks):
// the first U % n CTAs own U / n + 1 units, the others U / n.  Requires n <= U.
struct Partition {
  uint32_t U, n, q, r;
  __device__ void init(uint32_t U_, uint32_t n_) { U = U_; n = n_; q = U_ / n_; r = U_ - q * n_; }
  __device__ uint32_t begin(uint32_t c) const { return c * q + (c < r ? c : r); }
  __device__ int cta_of(uint32_t u) const {
    const uint32_t big = r * (q + 1);
    return u < big ? (int)(u / (q + 1)) : (int)(r + (u - big) / q);
  }
};

// Warp-cooperative: total number of units U, this CTA's range and the agent that contains its
// first unit.  One pass over the agents when there are at most 32 of them.
struct RangeStart {
  uint32_t U, u_begin, u_end, agent_start;
  int n_ctas, agent;
  bool any_bad;
  Partition part;
  int split, splits, pair;  // splits > 0: this CTA holds part `split` of the `splits` parts of head set `pair` of the agent,
  AgentRange r;             // whose range this is
};

// The agent that contains the CTA's first unit, among more than 32 of them (out of line: instruction fetches are what a
// launch starts with).
template <class Par>
__device__ __noinline__ void find_agent(const Par& P, RangeStart& rs) {
  const int lane = threadIdx.x & 31;
  uint32_t cum = 0;
#pragma unroll 1
  for (int base = 0; base < P.n_agents; base += 32) {
    const int a = base + lane;
    uint32_t cnt = 0;
    bool bad = false;
    if (a < P.n_agents) cnt = (uint32_t)(agent_range(P, a, bad).nc * P.Hkv);
    uint32_t inc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    const uint32_t tot = __shfl_sync(0xffffffffu, inc, 31);
    if (rs.u_begin < cum + tot) {
      const int l = __ffs(__ballot_sync(0xffffffffu, cum + inc > rs.u_begin)) - 1;
      rs.agent = base + l;
      rs.agent_start = cum + __shfl_sync(0xffffffffu, inc, l) - __shfl_sync(0xffffffffu, cnt, l);
      return;
    }
    cum += tot;
  }
}

// more_rounds: -1 for none, 0, 1, or 2 for 1 where the pairs are few (see below)
template <class Par>
__device__ inline RangeStart find_range(const Par& P, int cta, int grid, uint32_t nw, int more_rounds) {
  const int lane = threadIdx.x & 31;
  const int n_agents = P.n_agents, Hkv = P.Hkv;
  RangeStart rs;
  rs.any_bad = false;
  rs.agent = -1;
  rs.agent_start = 0;
  uint32_t cum = 0, cnt0 = 0;
  rs.r.n = 0; rs.r.lo = 0; rs.r.cf = 0; rs.r.nc = 0;
#pragma unroll 1
  for (int base = 0; base < n_agents; base += 32) {
    const int a = base + lane;
    uint32_t cnt = 0;
    bool bad = false;
    if (a < n_agents) { rs.r = agent_range(P, a, bad); cnt = (uint32_t)(rs.r.nc * Hkv); }
    rs.any_bad |= __any_sync(0xffffffffu, bad);
    cum += __reduce_add_sync(0xffffffffu, cnt);
    cnt0 = cnt;
  }
  rs.U = cum;
  // at least a chunk for every warp of a CTA, and not more CTAs on a pair than the merge takes quickly
  const uint32_t most = min((uint32_t)grid, (uint32_t)(n_agents * Hkv) * (uint32_t)kMaxRecords);
  rs.n_ctas = (int)min(most, (cum + nw - 1) / nw);
  rs.u_begin = rs.u_end = 0;
  rs.part.U = 0; rs.part.n = 1; rs.part.q = 0; rs.part.r = 0;
  rs.splits = 0; rs.split = 0; rs.pair = 0;
  if (cum == 0) return rs;
  if (n_agents <= 32) {
    // Cut every pair into equal parts of at most `size` chunks if that takes at most kWholeSlack chunks per CTA more than
    // an equal division of the list: a CTA then holds one segment, and the end of a segment (barriers, combination, the
    // next query: about two rounds of chunks) comes once.  Lane l tries size + l.
    // Measured with a slack of 0 / 6 / 12 / 24 / 31 chunks, us a launch: 8 KV heads at d = 128, 5 agents x 4096 tokens
    // 14.4 / 11.8 / 11.8 / 11.8 / 11.8; 13 agents x 1024..16384 23.6 / 23.6 / 21.0 / 21.0 / 21.0; 13 x 4096 23.7 / 23.7 / 23.7 /
    // 24.1 / 24.1; 32 x 4096 41.4 / 41.4 / 41.4 / 38.4 / 38.4; d = 256, 10 x 1024..16384 39.3 / 39.3 / 35.8 / 35.9 / 35.8.
    const int nc = lane < n_agents ? rs.r.nc : 0;
    // (No integer divisions: they and their like were 1.2 us of every CTA's start, which the late ones of a launch pay.  The
    // quotients of floats that size0 starts from may be off by one; every CTA finds the same.)
    const int nc_max = __reduce_max_sync(0xffffffffu, nc);
    const int size0 = max(max((int)nw, (int)ceilf(__fdividef((float)cum, (float)most))), (nc_max + kMaxRecords - 1) / kMaxRecords);
    const int size = size0 + lane;
    const float inv = __fdividef(1.f, (float)size);
    auto parts_of = [](int n, int sz, float rcp) {       // ceil(n / sz)
      int q = (int)((float)n * rcp);
      q += q * sz < n;
      q -= (q - 1) * sz >= n;
      return q;
    };
    int total = 0;
#pragma unroll 4
    for (int a = 0; a < n_agents; ++a) total += parts_of(__shfl_sync(0xffffffffu, nc, a), size, inv);
    const unsigned fits = __ballot_sync(0xffffffffu, total * Hkv <= (int)most && lane <= kWholeSlack);
    // A pair whole in one CTA needs no records and no ticket (2 us).  That is worth a round of chunks, one per warp, where the pairs are
    // few, and a seventh of the rounds where there are many.  Measured, us a launch, cut and whole: eight heads, 16 x 700 tokens
    // 15.0 / 15.9; d = 256, one x 350 9.0 / 9.9, 20 agents in a window of 1024 27.0 / 26.2.  Up to four heads at d = 128 stay cut all
    // the same: terms of p * s below 2^-24 are cut off against the reference of all the chunks that a warp adds up, and twice the
    // chunks lose more.  Error against 64 bits (relative, outlier channels), cut and whole, 8 KV heads: one agent x 480 tokens 1.44e-4 /
    // 1.95e-4 (6.5 / 5.8 us), 32 x 4096 8.5e-4 / 10.6e-4 (39.4 / 35.9 us); d = 256, 20 in a window 3.13e-4 / 3.13e-4.
    const int l = fits ? __ffs(fits) - 1 : 0, pairs = n_agents * Hkv;
    const int rounds = (size0 + l + (int)nw - 1) / (int)nw;
    const int extra = more_rounds < 0 ? 0 : (rounds * 37 >> 8) + (more_rounds == 1 || 4 * pairs <= (int)most ? min(more_rounds, 1) : 0);
    const bool uncut = pairs <= (int)most && (nc_max + (int)nw - 1) / (int)nw <= rounds + extra;
    if (fits || uncut) {
      const int best = uncut ? nc_max : size0 + l;
      rs.n_ctas = uncut ? pairs : __shfl_sync(0xffffffffu, total, l) * Hkv;
      if (cta >= rs.n_ctas) return rs;
      const int m = uncut ? (lane < n_agents ? 1 : 0) : parts_of(nc, best, __shfl_sync(0xffffffffu, inv, l));
      int inc = m * Hkv;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
      }
      const int a = __ffs(__ballot_sync(0xffffffffu, inc > cta)) - 1;
      rs.agent = a;
      rs.splits = __shfl_sync(0xffffffffu, m, a);
      const int at = cta - (__shfl_sync(0xffffffffu, inc, a) - rs.splits * Hkv), n = __shfl_sync(0xffffffffu, nc, a);
      const float per = __fdividef(1.f, (float)rs.splits);
      auto quotient = [&](int x) {                       // CTAs and a pair's chunks; below 2^20 the float quotient is off by one at most
        if (x >= 1 << 20) return x / rs.splits;
        int q = (int)((float)x * per);
        q -= q * rs.splits > x;
        return q + ((q + 1) * rs.splits <= x);
      };
      rs.pair = quotient(at);
      rs.split = at - rs.pair * rs.splits;
      rs.agent_start = 0;                                // units count from the pair's first chunk here
      rs.r.n = __shfl_sync(0xffffffffu, rs.r.n, a); rs.r.lo = __shfl_sync(0xffffffffu, rs.r.lo, a);
      rs.r.cf = __shfl_sync(0xffffffffu, rs.r.cf, a); rs.r.nc = n;
      const int each = quotient(n), more = n - each * rs.splits;         // the first `more` parts hold a chunk more
      rs.u_begin = (uint32_t)(rs.split * each + min(rs.split, more));
      rs.u_end = (uint32_t)(rs.u_begin + each + (rs.split < more ? 1 : 0));
      return rs;
    }
  }
  if (cta >= rs.n_ctas) return rs;
  rs.part.init(cum, (uint32_t)rs.n_ctas);
  rs.u_begin = rs.part.begin(cta);
  rs.u_end = rs.part.begin(cta + 1);
  const uint32_t want = rs.u_begin;
  if (n_agents <= 32) {
    uint32_t inc0 = cnt0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, inc0, o);
      if (lane >= o) inc0 += v;
    }
    const unsigned bal = __ballot_sync(0xffffffffu, inc0 > want);
    const int l = __ffs(bal) - 1;
    rs.agent = l;
    rs.agent_start = __shfl_sync(0xffffffffu, inc0, l) - __shfl_sync(0xffffffffu, cnt0, l);
    return rs;
  }
  find_agent(P, rs);
  return rs;
}

// One segment: the part of pair (agent a, head set hk) inside this CTA's unit range.
struct Segment {
  int a, hk, c0, c1;      // (virtual) agent, head set, logical chunk indices [c0, c1) of the agent
  int ar, li;             // real agent (lengths, block table) and layer of the call (pool layer)
  int n, lo;              // key range of the agent
  int cf, nc;             // the pair's whole chunk range
  int k0;                 // running chunk counter of the CTA at c0
  int first, last;        // CTAs that hold the pair's first and last chunk
};

// The one segment of a CTA that holds a part of one pair.
template <class Par>
__device__ inline void whole_segment(const Par& P, const RangeStart& rs, Segment& s) {
  s.li = P.layer_count > 1 ? rs.agent / P.n_real : 0; s.ar = rs.agent - s.li * P.n_real;
  s.a = rs.agent; s.hk = rs.pair; s.c0 = rs.r.cf + (int)rs.u_begin; s.c1 = rs.r.cf + (int)rs.u_end;
  s.n = rs.r.n; s.lo = rs.r.lo; s.cf = rs.r.cf; s.nc = rs.r.nc; s.k0 = 0;
  s.first = (int)blockIdx.x - rs.split;
  s.last = s.first + rs.splits - 1;
}

struct Walker {
  int n_agents, Hkv;
  uint32_t u, u_end;
  int k, a, hk, c;
  AgentRange r;

  template <class Par>
  __device__ __forceinline__ void init(const Par& P_, const RangeStart& rs) {
    n_agents = P_.n_agents; Hkv = P_.Hkv;
    u = rs.u_begin; u_end = rs.u_end; k = 0;
    a = rs.agent; hk = 0; c = 0;
    r.n = 0; r.lo = 0; r.cf = 0; r.nc = 0;
    if (u < u_end && a >= 0) {
      bool bad;
      r = agent_range(P_, a, bad);
      {
        const uint32_t rem = u - rs.agent_start;
        hk = (int)(rem / (uint32_t)r.nc);
        c = r.cf + (int)(rem - (uint32_t)hk * (uint32_t)r.nc);
      }
    }
  }
  template <class Par>
  __device__ __forceinline__ bool next(const Par& P, const RangeStart& rs, Segment& s) {
    if (u >= u_end || a < 0) { s.a = -1; return false; }
    const int pair_end = r.cf + r.nc;
    const uint32_t left = u_end - u;
    const int c1 = (uint32_t)(pair_end - c) <= left ? pair_end : c + (int)left;
    s.li = P.layer_count > 1 ? a / P.n_real : 0; s.ar = a - s.li * P.n_real;
    s.a = a; s.hk = hk; s.c0 = c; s.c1 = c1; s.n = r.n; s.lo = r.lo; s.cf = r.cf; s.nc = r.nc; s.k0 = k;
    const int cnt = c1 - c;
    s.first = s.last = 0;
    if (cnt != r.nc) {
      const uint32_t pair_u0 = u - (uint32_t)(c - r.cf);
      s.first = rs.part.cta_of(pair_u0);
      s.last = rs.part.cta_of(pair_u0 + (uint32_t)r.nc - 1u);
    }
    u += (uint32_t)cnt; k += cnt;
    if (c1 == pair_end) {
      ++hk;
      if (hk == Hkv) {
        hk = 0;
        bool bad;
        do {
          ++a;
          if (a >= n_agents) { a = -1; break; }
          r = agent_range(P, a, bad);
        } while (r.nc == 0);
      }
      if (a >= 0) c = r.cf;
    } else {
      c = c1;
    }
    return true;
  }
};

// ---------------------------------------------------------------------------------------------
// The kernel
// ---------------------------------------------------------------------------------------------
// The kernel is instantiated by the number of key groups G: 2 and 4 are the symmetric shapes (d_qk = d_v = 64 G), 3 is
// the asymmetric per-head MLA cache of Section 3.6 (d_qk 192, d_v 128); by the head columns H (4 or 8); and by the type
// of the scales and biases.
__host__ __device__ constexpr int kRecStride(int Dv) { return Dv + 4; }      // acc[Dv], m, l, pad: 16-byte multiples
__host__ __device__ constexpr int value_groups(int G) { return G == 3 ? 2 : G; }
constexpr uint32_t kOffBad = 0xFFFFFFFFu;   // pool offset of a chunk whose block id is outside the pool

template <int G, int H>
struct Smem {
  static constexpr int D = 64 * G, Gv = value_groups(G), Dv = 64 * Gv;
  static constexpr int kKeyBytes = 32 * (D / 2 + 4 * G), kValBytes = 32 * (Dv / 2 + 4 * Gv);
  static constexpr int kChunkBytes = kKeyBytes + kValBytes;
  static constexpr int NW = warps_of(G);
  // Slots of a warp.  Two whole chunks (147 KB per SM in flight: twice what HBM latency asks for); at d = 256 two key
  // halves and one value half, each with a barrier of its own (166 KB per SM).
  static constexpr bool kHalves = G == 4;
  static constexpr int kSlots = 2, kValSlots = kHalves ? 1 : 2;
  static constexpr int kWarpRing = kHalves ? kSlots * kKeyBytes + kValSlots * kValBytes : kSlots * kChunkBytes;
  static constexpr int kDepUnits = H * Dv / 128;
  alignas(128) uint8_t ring[NW][kWarpRing];
  alignas(16) float4 dep[NW][kDepUnits][32];            // accumulators of every warp, bias sums added (see deposit)
  float dep_m[NW][H], dep_l[NW][H];
  alignas(16) uint4 qfrag[2 * G][32];                   // [key word of a lane][lane = column * 4 + tid] = B registers
  float qsum[H][G];                                     // sum of the query over each group, in units of the score products
  float kappa[H];                                       // score products -> log2 units
  alignas(8) uint64_t full[NW][kSlots], full_v[NW][kValSlots];   // full_v: only where halves are copied
  RangeStart range;                                     // the CTA's range, for walks that start over
  Walker walker;                                        // runs two segments ahead
  uint32_t new_words[8 * (G + Gv)], new_sb[G + Gv];     // the quantized new row of the segment: K groups, then V groups
  Segment seg[3];                                       // segments s, s + 1, s + 2 at s % 3; a < 0: none
  int fin[2][4];                                        // the CTA's first and last segment: pair, first CTA, last CTA, row
  int fin_last[2];                                      // this CTA drew the pair's last ticket
  int abort_flag;
};

// Online-softmax state of one warp for one segment.  A lane owns two score columns (2 tid, 2 tid + 1 of eight) and, of
// every 32-token chunk, the four tokens 4 g .. 4 g + 3; l and the bias sums are per column, partial over the lane's
// tokens; the reference maximum m is common to the lanes of a column.
template <int G>
struct WarpState {
  static constexpr int Gv = value_groups(G);
  float m[2], l[2], bias[2][Gv];
  float o[4 * Gv][4];
  int head_room;                                         // H = 8: see chunk_values
  uint32_t vlimit;
  __device__ void reset() {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      m[c] = -INFINITY; l[c] = 0.f;
#pragma unroll
      for (int i = 0; i < Gv; ++i) bias[c][i] = 0.f;
    }
#pragma unroll
    for (int i = 0; i < 4 * Gv; ++i) { o[i][0] = 0.f; o[i][1] = 0.f; o[i][2] = 0.f; o[i][3] = 0.f; }
    head_room = 40;
    vlimit = 0u;
  }
};

// One warp stages one query row (column h) as binary16 in B-fragment order, scaled by a power of two so that nothing is
// rounded, plus the per-group sums of the query and the factor that undoes the scaling.  Key word w = 8*gi + 4*i2 + t of
// a token holds elements 8w..8w+7 and feeds two 16x8x16 products: (0,4 | 1,5) and (2,6 | 3,7), where the second pair of
// each meets codes in nibble 1 of their 16-bit lanes (a factor 16, divided out of the query here).  The uint4 of word
// p = 2*gi + i2 is {b0, b1} of the first product and {b0, b1} of the second, for the lane (column h, t).  The sign of
// the softmax scale goes into the query, so that the factor is positive.
template <int G, int H>
__device__ __forceinline__ void stage_query_row(uint4 (*qfrag)[32], float (*qsum)[G], float* kappa, const uint4 v, float scale_log2,
                                                int h, int lane) {
  constexpr int D = 64 * G;
  const int w = lane;
  const uint32_t u[4] = {v.x, v.y, v.z, v.w};          // lanes at or beyond D / 8 hold zeros
  float x[8];
#pragma unroll
  for (int i = 0; i < 4; ++i) { x[2 * i] = __uint_as_float(u[i] << 16); x[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u); }
  float mx = 0.f, sum = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) { mx = fmaxf(mx, fabsf(x[i])); sum += x[i]; }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);   // 8 words per group
  int ex = (int)((__float_as_uint(mx) >> 23) & 255u) - 127;
  if (mx == 0.f) ex = 0;
  ex = min(max(ex, -100), 100);
  float sf = __uint_as_float((uint32_t)(127 + 11 - ex) << 23);                 // 2048 <= max |q| * sf < 4096
  const float kap = fabsf(scale_log2) * __uint_as_float((uint32_t)(127 + 13 + ex) << 23);   // 2^24 / sf
  if (scale_log2 < 0.f) sf = -sf;
  if (scale_log2 == 0.f) sf = 0.f;
  const float sl = sf * 0.0625f;
  if (w < D / 8) {
    const uint4 f = make_uint4(f32x2_to_h2(x[0] * sf, x[4] * sf), f32x2_to_h2(x[1] * sl, x[5] * sl),
                               f32x2_to_h2(x[2] * sf, x[6] * sf), f32x2_to_h2(x[3] * sl, x[7] * sl));
    const int gi = w >> 3, i2 = (w >> 2) & 1, t = w & 3;
    qfrag[2 * gi + i2][h * 4 + t] = f;
    if (H == 4) qfrag[2 * gi + i2][(h + 4) * 4 + t] = f;                       // columns 4..7 repeat the heads
    if ((w & 7) == 0) qsum[h][gi] = sum * sf * 5.9604644775390625e-8f;         // 2^-24: the codes enter as c * 2^-24
    if (w == 0) kappa[h] = kap > 0.f ? kap : 1.f;
  }
}

// The fused append (one new token per agent).  The warp that holds the chunk of an agent's newest position writes the new row's
// words into it once it has landed -- in shared memory for this launch, in the pool for the following ones.  Every chunk is held
// by exactly one warp of the grid, so nobody else reads or writes these words during the launch.
// The value codes are token-packed: one nibble of each of the row's d_v words is replaced.
template <int G, int H>
__device__ __noinline__ void patch_new_row(const Smem<G, H>& sm, uint8_t* keys, uint8_t* values, uint8_t* gchunk, int tau, int lane) {
  constexpr int D = 64 * G, Gv = value_groups(G), Dv = 64 * Gv;
  constexpr uint32_t off_ksb = 32 * (D / 2), key_bytes = off_ksb + 128 * G, off_vsb = 32 * (Dv / 2);
  auto put = [&](uint8_t* half, uint32_t base, uint32_t at, uint32_t v) {
    *reinterpret_cast<uint32_t*>(half + at) = v;
    *reinterpret_cast<uint32_t*>(gchunk + base + at) = v;
  };
  if (lane < 8 * G) put(keys, 0u, 4u * k_word_offset(tau, lane, G), sm.new_words[lane]);
  if (lane < G) put(keys, 0u, off_ksb + 4u * sb_offset(tau, lane, G), sm.new_sb[lane]);
  if (lane < Gv) put(values, key_bytes, off_vsb + 4u * sb_offset(tau, lane, Gv), sm.new_sb[G + lane]);
  const int shift = 4 * (tau & 7);
#pragma unroll 1
  for (int d = lane; d < Dv; d += 32) {
    const uint32_t code = (sm.new_words[8 * G + (d >> 3)] >> (4 * (d & 7))) & 15u;
    const uint32_t at = 4u * v_word_offset(tau >> 3, d);
    put(values, key_bytes, at, (*reinterpret_cast<const uint32_t*>(values + at) & ~(15u << shift)) | (code << shift));
  }
}
// A chunk that sticks out of the key range: the slots outside may hold anything, their value scales and biases become
// zero in shared memory (their scores are masked), so that the common path need not look.
template <int G>
__device__ __noinline__ void clear_outside(uint8_t* vsb, int pos0, int key_lo, int key_n, int lane) {
  constexpr int Gv = value_groups(G);
  const int pos = pos0 + lane;
  if (pos >= key_lo && pos < key_n) return;
#pragma unroll
  for (int gi = 0; gi < Gv; ++gi) reinterpret_cast<uint32_t*>(vsb)[sb_offset(lane, gi, Gv)] = 0u;
}

// Transpose of an 8 x 8 matrix of 16-bit elements held one row per lane group (lane l: row l / 4, columns 2 * (l % 4)
// and + 1): afterwards lane l holds row l / 4 of the transposed matrix.
__device__ inline uint32_t transpose_8x8_b16(uint32_t a) {
  uint32_t d;
  asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
  return d;
}

// Scores of one 32-token chunk: sc[i][c] of token 4g + i for column 2 tid + c, times kappa in log2 units.
// The key codes are the A operand (16 tokens x 16 head-dim elements per product: lane (g, tid) holds the words of the
// tokens 4g + i, i = 0..3, so products pair the token rows (0, 1) and (2, 3)), the query the B operand.  A group's
// integer dot products meet the token's scale, and its bias the group's query sum, as soon as the group is done.
template <int G, bool kBf>
__device__ __forceinline__ void chunk_scores(const uint8_t* chunk, int g, int tid, const uint4* qb, const float* qs0,
                                             const float* qs1, float (&sc)[4][2]) {
  constexpr int D = 64 * G;
  constexpr int kPairs = 2;                 // token-row pairs in work together (registers)
  const uint4* kc4 = reinterpret_cast<const uint4*>(chunk);
  const uint8_t* ksb = chunk + 32 * (D / 2);
#pragma unroll
  for (int half = 0; half < (G + 1) / 2; ++half) {       // groups 2*half, 2*half+1: a 16-byte piece per token row
    const bool odd = (G & 1) && half == G / 2;           // the last group of an odd count: an 8-byte piece per token row
#pragma unroll
    for (int pr0 = 0; pr0 < 2; pr0 += kPairs) {
      float acc[kPairs][2][4];                           // [token-row pair][group]
#pragma unroll
      for (int pr = 0; pr < kPairs; ++pr)
#pragma unroll
        for (int gi = 0; gi < 2; ++gi) { acc[pr][gi][0] = 0.f; acc[pr][gi][1] = 0.f; acc[pr][gi][2] = 0.f; acc[pr][gi][3] = 0.f; }
      uint4 kw[2 * kPairs];
#pragma unroll
      for (int i = 0; i < 2 * kPairs; ++i) {
        if (odd) {
          const uint2 t = reinterpret_cast<const uint2*>(chunk)[((2 * pr0 + i) * 64 * G + (G / 2) * 128) / 2 + g * 4 + tid];
          kw[i] = make_uint4(t.x, t.y, 0u, 0u);
        } else {
          kw[i] = kc4[(2 * pr0 + i) * 16 * G + half * 32 + g * 4 + tid];
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {                      // word p = 4*half + j: group 2*half + j/2
        if (odd && j >= 2) break;
        const uint4 b = qb[(4 * half + j) * 32];
#pragma unroll
        for (int pr = 0; pr < kPairs; ++pr) {
          const uint4 &k0 = kw[2 * pr], &k1 = kw[2 * pr + 1];
          const uint32_t w0 = j == 0 ? k0.x : j == 1 ? k0.y : j == 2 ? k0.z : k0.w;
          const uint32_t w1 = j == 0 ? k1.x : j == 1 ? k1.y : j == 2 ? k1.z : k1.w;
          const uint32_t h0 = w0 >> 8, h1 = w1 >> 8;
          float (&a)[4] = acc[pr][j >> 1];
          mma_f16(a, w0 & kMaskLo, w1 & kMaskLo, w0 & kMaskHi, w1 & kMaskHi, b.x, b.y);
          mma_f16(a, h0 & kMaskLo, h1 & kMaskLo, h0 & kMaskHi, h1 & kMaskHi, b.z, b.w);
        }
      }
#pragma unroll
      for (int i = 2 * pr0; i < 2 * (pr0 + kPairs); ++i) {
        const uint8_t* at = ksb + (i * 8 + g) * 4 * G + 8 * half;
        uint2 v;
        if (odd) v = make_uint2(*reinterpret_cast<const uint32_t*>(at), 0u);
        else if (G & 1) v = make_uint2(*reinterpret_cast<const uint32_t*>(at), *reinterpret_cast<const uint32_t*>(at + 4));
        else v = *reinterpret_cast<const uint2*>(at);
        const float2 f0 = sb_to_f2<kBf>(v.x), f1 = sb_to_f2<kBf>(v.y);
        const float (&a)[2][4] = acc[(i >> 1) - pr0];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          float t = a[0][2 * (i & 1) + c] * f0.x;
          if (half > 0) t += sc[i][c];
          t = fmaf((c == 0 ? qs0 : qs1)[2 * half], f0.y, t);
          if (!odd) {
            t = fmaf(a[1][2 * (i & 1) + c], f1.x, t);
            t = fmaf((c == 0 ? qs0 : qs1)[2 * half + 1], f1.y, t);
          }
          sc[i][c] = t;
        }
      }
    }
  }
}

// Softmax step and value product of the chunk.  vc: its value half (codes, then scale/bias pairs).
//   The probabilities, multiplied by the token's value scale, are packed two columns to a register and transposed across
//   the warp into the B operand of the value product, whose A operand is the token-packed value words.
template <int G, int H, bool kBf>
__device__ __forceinline__ void chunk_values(const uint8_t* vhalf, bool edge, int pos0, int key_lo, int key_n, int g, int tid,
                                             const float (&kap)[2], uint32_t split_mask, float margin, float (&sc)[4][2],
                                             WarpState<G>& st) {
  constexpr int Gv = value_groups(G), Dv = 64 * Gv;
  const uint4* vc4 = reinterpret_cast<const uint4*>(vhalf);
  const uint8_t* vsb = vhalf + 32 * (Dv / 2);
  if (edge) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int pos = pos0 + 4 * g + i;
      if (pos < key_lo || pos >= key_n) { sc[i][0] = -INFINITY; sc[i][1] = -INFINITY; }
    }
  }
  // H = 4: probabilities stay at most 1, so p*s stays inside binary16 for every scale.  H = 8: the reference leaves the
  // probabilities as many binary orders above 1 as the value scales seen so far allow (p*s below 2^15), because the low
  // half of the split loses what falls below 2^-24 and the odd token rows (p/16 against 16c) lose sixteen times as much.
  float cm[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) cm[c] = fmaxf(fmaxf(sc[0][c], sc[1][c]), fmaxf(sc[2][c], sc[3][c])) * kap[c];
  bool grow;
  uint32_t vmax = 0u;                                    // H = 8: the largest value scale of the lane's tokens (bit pattern)
  if (H == 8) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int gp = 0; gp < Gv / 2; ++gp) {
        const uint2 v = *reinterpret_cast<const uint2*>(vsb + (i * 8 + g) * 4 * Gv + 8 * gp);
        vmax = __vmaxu2(vmax, __vmaxu2(v.x, v.y));
      }
    vmax &= 0xFFFFu;
    const float top = (float)st.head_room + 1.f;
    grow = cm[0] > st.m[0] + top || cm[1] > st.m[1] + top || vmax > st.vlimit;
  } else {
    grow = cm[0] > st.m[0] || cm[1] > st.m[1];
  }
  if (__any_sync(0xffffffffu, grow)) {
    int room = 0, old_room = 0;
    if (H == 8) {
      // scales below 2^e leave 14 - e binary orders for the probabilities
      vmax = __reduce_max_sync(0xffffffffu, vmax);
      if (vmax > 0x7FFFu) vmax = 0x7FFFu;                // a negative scale: no room
      const int e = kBf ? (int)(vmax >> 7) - 126 : (int)(vmax >> 10) - 14;
      old_room = st.head_room;
      room = min(st.head_room, 14 - max(e, -26));
      st.head_room = room;
      st.vlimit = max(st.vlimit, vmax | (kBf ? 0x7Fu : 0x3FFu));
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      float x = cm[c];
      x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 4));
      x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 8));
      x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 16));
      if (H == 8) x = fmaxf(st.m[c] + (float)old_room, x) - (float)room;
      else x = x > st.m[c] ? x + margin : st.m[c];
      const float f = fast_exp2(st.m[c] - x);            // m = -inf: 0
      st.m[c] = x;
      st.l[c] *= f;
#pragma unroll
      for (int gi = 0; gi < Gv; ++gi) st.bias[c][gi] *= f;
#pragma unroll
      for (int mt = 0; mt < Dv / 16; ++mt) { st.o[mt][c] *= f; st.o[mt][2 + c] *= f; }
    }
  }
  float p[4][2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
#pragma unroll
    for (int i = 0; i < 4; ++i) p[i][c] = fast_exp2(fmaf(sc[i][c], kap[c], -st.m[c]));
    st.l[c] += (p[0][c] + p[1][c]) + (p[2][c] + p[3][c]);
  }
#pragma unroll
  for (int gp = 0; gp < Gv / 2; ++gp) {
    uint2 sbw[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) sbw[i] = *reinterpret_cast<const uint2*>(vsb + (i * 8 + g) * 4 * Gv + 8 * gp);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int gi = 2 * gp + e;
      // p * s_v as a two-term binary16 pair, transposed: bh[i] = half2(tokens 8 tid + i, 8 tid + 4 + i) of column g
      uint32_t bh[4], bl[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 f = sb_to_f2<kBf>(e == 0 ? sbw[i].x : sbw[i].y);
        const float vs = (i & 1) ? f.x * 0.0625f : f.x;  // odd token rows: their value codes carry a factor 16
        const float x0 = p[i][0] * vs, x1 = p[i][1] * vs;
        st.bias[0][gi] = fmaf(p[i][0], f.y, st.bias[0][gi]);
        st.bias[1][gi] = fmaf(p[i][1], f.y, st.bias[1][gi]);
        if (H == 4) {
          // columns 0..3: trunc16(x); columns 4..7: trunc16(x - trunc11bits(x)) -- the binary16 conversion truncates
          const float r0 = x0 - __uint_as_float(__float_as_uint(x0) & split_mask);
          const float r1 = x1 - __uint_as_float(__float_as_uint(x1) & split_mask);
          bh[i] = transpose_8x8_b16(f32x2_to_h2_rz(r0, r1));
        } else {
          const float r0 = x0 - __uint_as_float(__float_as_uint(x0) & 0xFFFFE000u);
          const float r1 = x1 - __uint_as_float(__float_as_uint(x1) & 0xFFFFE000u);
          bh[i] = transpose_8x8_b16(f32x2_to_h2_rz(x0, x1));
          bl[i] = transpose_8x8_b16(f32x2_to_h2_rz(r0, r1));
        }
      }
      // P.V on the codes: 16 value rows x 8 columns x 32 tokens per accumulator tile
#pragma unroll
      for (int q4 = 2 * gi; q4 < 2 * gi + 2; ++q4) {
        const uint4 w4 = vc4[(q4 * 8 + g) * 4 + tid];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          const uint32_t x = t == 0 ? w4.x : w4.z, y = t == 0 ? w4.y : w4.w, xh = x >> 8, yh = y >> 8;
          float (&o)[4] = st.o[2 * q4 + t];
          if (H == 4) {
            mma_f16(o, x & kMaskLo, y & kMaskLo, x & kMaskHi, y & kMaskHi, bh[0], bh[1]);
            mma_f16(o, xh & kMaskLo, yh & kMaskLo, xh & kMaskHi, yh & kMaskHi, bh[2], bh[3]);
          } else {
            // the small terms first, and the chunk's sum joins the running one outside: the tensor cores truncate
            float a[4] = {0.f, 0.f, 0.f, 0.f};
            mma_f16(a, x & kMaskLo, y & kMaskLo, x & kMaskHi, y & kMaskHi, bl[0], bl[1]);
            mma_f16(a, xh & kMaskLo, yh & kMaskLo, xh & kMaskHi, yh & kMaskHi, bl[2], bl[3]);
            mma_f16(a, x & kMaskLo, y & kMaskLo, x & kMaskHi, y & kMaskHi, bh[0], bh[1]);
            mma_f16(a, xh & kMaskLo, yh & kMaskLo, xh & kMaskHi, yh & kMaskHi, bh[2], bh[3]);
            o[0] += a[0]; o[1] += a[1]; o[2] += a[2]; o[3] += a[3];
          }
        }
      }
    }
  }
}

__device__ inline void store_out(const DecodeParams& P, size_t index, float v) {
  if (P.out_dtype == Q4KV_OUT_BF16) reinterpret_cast<__nv_bfloat16*>(P.out)[index] = __float2bfloat16_rn(v);
  else reinterpret_cast<float*>(P.out)[index] = v;
}
__device__ __forceinline__ void store_four(const DecodeParams& P, size_t index, const float (&x)[4], float mul) {
  if (P.out_dtype == Q4KV_OUT_BF16) {
    const __nv_bfloat162 lo = __floats2bfloat162_rn(x[0] * mul, x[1] * mul), hi = __floats2bfloat162_rn(x[2] * mul, x[3] * mul);
    *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(P.out) + index) =
        make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
  } else {
    *reinterpret_cast<float4*>(reinterpret_cast<float*>(P.out) + index) = make_float4(x[0] * mul, x[1] * mul, x[2] * mul, x[3] * mul);
  }
}

// Leave this warp's state of a segment in its deposit, in fragment order (16 bytes per lane and unit): the accumulators
// with the bias sums added, and m, l per head.
//   H = 4: columns 4..7 (lanes tid 2, 3) hold the low-part products of heads 0..3; a pair of lanes exchanges the halves it
//   does not keep.  Unit u of lane (g, tid) is value rows 32 u + g + 8 * (tid / 2) (+ 16) of heads 2 * (tid % 2) (+ 1):
//   {row, head} {row, head + 1} {row + 16, head} {row + 16, head + 1}.
//   H = 8: unit u is value rows 16 u + g (+ 8) of heads 2 tid (+ 1): {row, head} {row, head + 1} {row + 8, ..} {row + 8, ..}.
template <int G, int H>
__device__ __forceinline__ void deposit(Smem<G, H>& sm, int warp, int lane, WarpState<G>& st, bool bad) {
  constexpr int Gv = value_groups(G);
  const int g = lane >> 2, tid = lane & 3;
  float bias[2][Gv];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    float l = st.l[c];                                   // over the lane's tokens -> over the chunk's (lanes of equal tid)
    l += __shfl_xor_sync(0xffffffffu, l, 4);
    l += __shfl_xor_sync(0xffffffffu, l, 8);
    l += __shfl_xor_sync(0xffffffffu, l, 16);
#pragma unroll
    for (int gi = 0; gi < Gv; ++gi) {
      float bb = st.bias[c][gi];
      bb += __shfl_xor_sync(0xffffffffu, bb, 4);
      bb += __shfl_xor_sync(0xffffffffu, bb, 8);
      bb += __shfl_xor_sync(0xffffffffu, bb, 16);
      bias[c][gi] = bb;
    }
    if (g == 0 && (H == 8 || tid < 2)) {
      sm.dep_m[warp][2 * tid + c] = st.m[c];
      sm.dep_l[warp][2 * tid + c] = bad ? -1.f : l;
    }
  }
  constexpr float k24 = 16777216.f;
#pragma unroll
  for (int u = 0; u < Smem<G, H>::kDepUnits; ++u) {
    float4 v;
    if (H == 4) {
      const bool up = tid >= 2;
      float x[2][2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float (&o)[4] = st.o[(2 * u + e) & (4 * Gv - 1)];
        x[e][0] = (up ? o[2] : o[0]) + __shfl_xor_sync(0xffffffffu, up ? o[0] : o[2], 2);
        x[e][1] = (up ? o[3] : o[1]) + __shfl_xor_sync(0xffffffffu, up ? o[1] : o[3], 2);
      }
      const float b0 = bias[0][u >> 1], b1 = bias[1][u >> 1];
      v = make_float4(fmaf(x[0][0], k24, b0), fmaf(x[0][1], k24, b1), fmaf(x[1][0], k24, b0), fmaf(x[1][1], k24, b1));
    } else {
      const float (&o)[4] = st.o[u & (4 * Gv - 1)];
      const float b0 = bias[0][(u >> 2) & (Gv - 1)], b1 = bias[1][(u >> 2) & (Gv - 1)];
      v = make_float4(fmaf(o[0], k24, b0), fmaf(o[1], k24, b1), fmaf(o[2], k24, b0), fmaf(o[3], k24, b1));
    }
    sm.dep[warp][u][lane] = v;
  }
}

// Combine the eight warps' deposits of a segment: unit `unit` (one warp each).  A pair that lies wholly inside this CTA is
// normalised and written out, otherwise the combination becomes this CTA's partial record.
template <int G, int H, class Par>
__device__ __forceinline__ void combine_deposits(const Smem<G, H>& sm, const Par& P, const Segment& seg, int cta, int unit,
                                                 int lane) {
  constexpr int Dv = Smem<G, H>::Dv, NW = Smem<G, H>::NW;
  const int g = lane >> 2, tid = lane & 3, n_rep = P.n_rep;
  const bool whole = seg.c1 - seg.c0 == seg.nc;
  // (m, l) of (warp, head): H = 4: lane 4 * warp + head; H = 8: two per lane, warps lane / 8 and lane / 8 + 4
  constexpr int kPer = (NW * H + 31) / 32;
  float e[kPer], M, L = 0.f;
  bool bad = false;
  {
    float m[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) m[k] = 32 * k + lane < NW * H ? (&sm.dep_m[0][0])[32 * k + lane] : -INFINITY;
    M = m[0];
#pragma unroll
    for (int k = 1; k < kPer; ++k) M = fmaxf(M, m[k]);
#pragma unroll
    for (int o = H; o < 32; o <<= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const float l = 32 * k + lane < NW * H ? (&sm.dep_l[0][0])[32 * k + lane] : 0.f;
      e[k] = m[k] == -INFINITY ? 0.f : fast_exp2(m[k] - M);
      L = fmaf(e[k], l, L);
      bad |= l < 0.f;
    }
#pragma unroll
    for (int o = H; o < 32; o <<= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
    bad = __any_sync(0xffffffffu, bad);
    if (bad) L = 0.f;
  }
  const int h0 = 2 * (tid & (H / 2 - 1));                // this lane's heads h0, h0 + 1
  float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    const float e0 = __shfl_sync(0xffffffffu, e[w * H / 32], (w * H & 31) + h0);
    const float e1 = __shfl_sync(0xffffffffu, e[w * H / 32], (w * H & 31) + h0 + 1);
    if (e0 != 0.f || e1 != 0.f) {                        // an empty deposit holds stale bytes
      const float4 x = sm.dep[w][unit][lane];
      a[0] = fmaf(e0, x.x, a[0]); a[1] = fmaf(e1, x.y, a[1]);
      a[2] = fmaf(e0, x.z, a[2]); a[3] = fmaf(e1, x.w, a[3]);
    }
  }
  const float L0 = __shfl_sync(0xffffffffu, L, h0), L1 = __shfl_sync(0xffffffffu, L, h0 + 1);
  const int d = H == 4 ? 32 * unit + g + 8 * (tid >> 1) : 16 * unit + g, step = H == 4 ? 16 : 8;
  const size_t row0 = (size_t)(Par::kSingles ? P.q_offs[seg.a] : seg.a) * P.y.Hq + (size_t)seg.hk * n_rep;
  if (whole) {
    const float i0 = L0 > 0.f ? 1.f / L0 : 0.f, i1 = L1 > 0.f ? 1.f / L1 : 0.f;
    if (h0 < n_rep) { store_out(P, (row0 + h0) * Dv + d, a[0] * i0); store_out(P, (row0 + h0) * Dv + d + step, a[2] * i0); }
    if (h0 + 1 < n_rep) { store_out(P, (row0 + h0 + 1) * Dv + d, a[1] * i1); store_out(P, (row0 + h0 + 1) * Dv + d + step, a[3] * i1); }
    if (unit == 0 && lane < n_rep && P.lse) P.lse[row0 + lane] = L > 0.f ? (M + log2f(L)) / kLog2e : -INFINITY;
  } else {
    float* rec = P.partials + (size_t)(seg.a * P.Hkv + seg.hk + cta) * n_rep * kRecStride(Dv);
    float* r0 = rec + h0 * kRecStride(Dv) + d;
    if (h0 < n_rep) { r0[0] = a[0]; r0[step] = a[2]; }
    if (h0 + 1 < n_rep) { r0[kRecStride(Dv)] = a[1]; r0[kRecStride(Dv) + step] = a[3]; }
    if (unit == 0 && lane < n_rep)
      *reinterpret_cast<float2*>(rec + lane * kRecStride(Dv) + Dv) = make_float2(M, bad ? -1.f : L);
  }
}

// Combination of the records of one pair for one head and 128 output elements, by one warp (lane: four elements).  The
// records sit in L2, a microsecond away: a batch of loads is in flight together with the (m, l) pairs.
__device__ __forceinline__ void combine_records(const DecodeParams& P, const float* base, size_t rstride, int R, int Dv, int d,
                                                size_t row, int lane) {
  constexpr int RB = 8;
  float M = -INFINITY, L = 0.f, acc[4] = {0.f, 0.f, 0.f, 0.f};
  bool bad = false;
#pragma unroll 1
  for (int r0 = 0; r0 < R; r0 += 32) {
    const int n = min(32, R - r0);
    const float2 ml = lane < n ? __ldcg(reinterpret_cast<const float2*>(base + (size_t)(r0 + lane) * rstride + Dv))
                               : make_float2(-INFINITY, 0.f);
    float e = 0.f;
#pragma unroll 1
    for (int b = 0; b < n; b += RB) {
      float4 x[RB];
#pragma unroll
      for (int i = 0; i < RB; ++i)
        x[i] = __ldcg(reinterpret_cast<const float4*>(base + (size_t)(r0 + min(b + i, n - 1)) * rstride + d));
      if (b == 0) {
        float Mn = ml.x;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) Mn = fmaxf(Mn, __shfl_xor_sync(0xffffffffu, Mn, o));
        Mn = fmaxf(M, Mn);
        const float f = Mn == -INFINITY ? 0.f : fast_exp2(M - Mn);       // M = -inf: 0
        e = ml.x == -INFINITY ? 0.f : fast_exp2(ml.x - Mn);
        bad |= __any_sync(0xffffffffu, ml.y < 0.f);
        float s = e * ml.y;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        L = L * f + s;
        M = Mn;
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k] *= f;
      }
#pragma unroll
      for (int i = 0; i < RB; ++i) {
        const float w = __shfl_sync(0xffffffffu, e, (b + i) & 31);       // past the last record: 0, or not added
        if (b + i < n) {
          acc[0] = fmaf(w, x[i].x, acc[0]); acc[1] = fmaf(w, x[i].y, acc[1]);
          acc[2] = fmaf(w, x[i].z, acc[2]); acc[3] = fmaf(w, x[i].w, acc[3]);
        }
      }
    }
  }
  if (bad) L = 0.f;
  store_four(P, row * Dv + d, acc, L > 0.f ? 1.f / L : 0.f);
  if (d == 0 && P.lse) P.lse[row] = L > 0.f ? (M + log2f(L)) / kLog2e : -INFINITY;
}

// Agents first, first + step, ... without any key (kv_len == 0 or a rejected length): zeros, lse = -inf.
template <class Par>
__device__ __forceinline__ void clear_empty_agents(const Par& P, int first, int step, int Dv, int lane) {
#pragma unroll 1
  for (int a = first; a < P.n_agents; a += step) {
    bool bad_len;
    if (agent_range(P, a, bad_len).nc > 0 || (Par::kSingles && P.q_offs[a + 1] - P.q_offs[a] != 1)) continue;
    const size_t row = Par::kSingles ? P.q_offs[a] : a;
#pragma unroll 1
    for (int i = lane; i < P.y.Hq * Dv; i += 32) store_out(P, row * P.y.Hq * Dv + i, 0.f);
#pragma unroll 1
    for (int i = lane; i < P.y.Hq && P.lse; i += 32) P.lse[row * P.y.Hq + i] = -INFINITY;
  }
}

// Pool offsets (16-byte units inside the layers of the call) of the warp's chunks 32 b .. 32 b + 31, one per lane: a walk
// of the CTA's segments from the start, out of line (a warp needs it once per 32 chunks).
__device__ __forceinline__ uint32_t chunk_offset(const DecodeParams& P, const Segment& s, int c, uint32_t chunk_bytes) {
  const int blk = P.tables[(size_t)s.ar * P.max_blocks + (c >> 3)];
  if (blk < 0 || blk >= P.n_blocks) { raise_flag(P.flags, Q4KV_FLAG_BAD_BLOCK); return kOffBad; }
  return (uint32_t)(((uint64_t)s.li * P.y.layer_bytes + (uint64_t)blk * P.y.block_bytes +
                     (uint64_t)(P.sets == 1 ? s.hk : s.hk / P.sets) * P.y.head_block_bytes + (uint64_t)(c & 7) * chunk_bytes) >> 4);
}
template <class Par>
__device__ __noinline__ uint32_t batch_offsets(const Par& P, const RangeStart& rs, int nw, int warp, int b, uint32_t chunk_bytes) {
  Segment s;
  uint32_t off = kOffBad;
  const int my_k = warp + nw * (32 * b + (int)(threadIdx.x & 31)), end = min((int)(rs.u_end - rs.u_begin), nw * 32 * (b + 1));
  if (rs.splits > 0) {
    whole_segment(P, rs, s);
    if (my_k < s.c1 - s.c0) off = chunk_offset(P, s, s.c0 + my_k, chunk_bytes);
    return off;
  }
  Walker wk;
  wk.init(P, rs);
  while (wk.next(P, rs, s)) {
    const int k1 = s.k0 + (s.c1 - s.c0);
    if (my_k >= s.k0 && my_k < k1) off = chunk_offset(P, s, s.c0 + (my_k - s.k0), chunk_bytes);
    if (k1 >= end) break;
  }
  return off;
}

template <int G, int H, bool kBf, bool kSingles>
__global__ void __launch_bounds__(warps_of(G) * 32, kCtasPerSm) decode_mma_kernel(const __grid_constant__ Params<kSingles> P) {
  using S = Smem<G, H>;
  constexpr int NW = S::NW, D = S::D, Gv = S::Gv, Dv = S::Dv, kSlots = S::kSlots, kValSlots = S::kValSlots;
  constexpr bool kHalves = S::kHalves;
  extern __shared__ __align__(128) uint8_t smem_raw[];
  S& sm = *reinterpret_cast<S*>(smem_raw);

  const Layout& y = P.y;
  const int warp = (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int cta = blockIdx.x;
  const int n_rep = P.n_rep;

  grid_launch_dependents();
  if (kSingles) {                                        // a prefill batch need not hold an agent with one query
    bool any = false;
    for (int a = threadIdx.x; a < P.n_agents; a += NW * 32) any |= P.q_offs[a + 1] - P.q_offs[a] == 1;
    if (!__syncthreads_or(any)) {
      grid_dependency_wait();                            // or this grid could complete before the one it follows
      return;
    }
  }
  // ---- this CTA's unit range and its first two segments: one warp, the others set up shared memory (lengths and block
  // tables are inputs that no kernel writes) ----
  if (warp == 0) {
    const RangeStart rs = find_range(P, cta, gridDim.x, NW, G == 4 ? 0 : H == 8 ? 2 : G == 3 ? 1 : -1);
    if (lane == 0) {
      if (rs.any_bad && cta == 0) raise_flag(P.flags, Q4KV_FLAG_BAD_LENGTH);
      sm.range = rs;
      if (rs.splits > 0) {
        whole_segment(P, rs, sm.seg[0]);
        sm.seg[1].a = -1; sm.seg[1].c0 = 0; sm.seg[1].c1 = 0; sm.seg[1].k0 = 0;
      } else {
        sm.walker.init(P, rs);
        sm.walker.next(P, rs, sm.seg[0]);
        sm.walker.next(P, rs, sm.seg[1]);
      }
    }
  } else {
    // columns of query heads that do not exist are never staged: they stay zero (factor 1)
    for (int i = threadIdx.x - 32; i < 2 * G * 32; i += (NW - 1) * 32) (&sm.qfrag[0][0])[i] = make_uint4(0u, 0u, 0u, 0u);
    if (warp == NW - 1) {
      for (int i = lane; i < H * G; i += 32) (&sm.qsum[0][0])[i] = 0.f;
      if (lane < H) sm.kappa[lane] = 1.f;
    }
    if (warp == NW - 2) {
      for (int i = lane; i < NW * kSlots; i += 32) mbar_init(&sm.full[0][0] + i, 1);
      for (int i = lane; i < NW * kValSlots; i += 32) mbar_init(&sm.full_v[0][0] + i, 1);
      if (lane == 0) { sm.abort_flag = 0; sm.fin[0][0] = -1; sm.fin[1][0] = -1; }
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
  }
  __syncthreads();
  const int n_chunks = (int)(sm.range.u_end - sm.range.u_begin);
  const uint8_t* layer_base = P.pool + (uint64_t)P.layer * y.layer_bytes;
  uint32_t off = kOffBad;                                // pool offset of the warp's chunk number `lane` (of 32 at a time)
  {
    const int k = warp + NW * lane;
    const Segment &s0 = sm.seg[0], &s1 = sm.seg[1];
    if (k < n_chunks) {
      const int n0 = s0.c1 - s0.c0;
      if (k < n0) off = chunk_offset(P, s0, s0.c0 + k, S::kChunkBytes);
      else if (k < n0 + (s1.c1 - s1.c0)) off = chunk_offset(P, s1, s1.c0 + k - n0, S::kChunkBytes);
    }
    if (sm.range.splits == 0 && n_chunks > s0.c1 - s0.c0 && n_chunks > s1.k0 + (s1.c1 - s1.c0)) off = batch_offsets(P, sm.range, NW, warp, 0, S::kChunkBytes);
  }
  uint8_t* const ring = sm.ring[warp];
  auto issue_keys = [&](int slot, uint32_t off) {        // the whole chunk unless it is copied in halves
    uint64_t* bar = &sm.full[warp][slot];
    constexpr uint32_t bytes = kHalves ? S::kKeyBytes : S::kChunkBytes;
    if (off == kOffBad) { mbar_arrive(bar); return; }
    mbar_arrive_expect_tx(bar, bytes);
    bulk_load(ring + slot * bytes, layer_base + (uint64_t)off * 16u, bytes, bar);
  };
  auto issue_values = [&](int slot, uint32_t off) {
    uint64_t* bar = &sm.full_v[warp][slot];
    if (off == kOffBad) { mbar_arrive(bar); return; }
    mbar_arrive_expect_tx(bar, S::kValBytes);
    bulk_load(ring + kSlots * S::kKeyBytes + slot * S::kValBytes, layer_base + (uint64_t)off * 16u + S::kKeyBytes, S::kValBytes, bar);
  };

  const int my_chunks = n_chunks > warp ? (n_chunks - warp + NW - 1) / NW : 0;
  const int g = lane >> 2, tid = lane & 3;
  // This warp's row of a segment's query.  The CTA that holds the newest position's chunk quantizes that token's K and V rows
  // (Section 3.2 quantizer, the arithmetic of the append kernel) when it stages the query: a warp per 64-element group, two
  // elements per lane, by the warps behind the query's (from 4 on), so that neither waits for the other.  (One warp doing all of
  // it, eight elements per lane, was 3.5 us on the critical path of every launch: 500 instructions that come from far away.)
  constexpr int kNewWarps = NW - 4, kNewRounds = (G + Gv + kNewWarps - 1) / kNewWarps;
  auto query_row = [&](const Segment& s) { return P.q + ((size_t)(kSingles ? P.q_offs[s.a] : s.a) * y.Hq + (size_t)s.hk * n_rep + warp) * D + 8 * lane; };
  auto new_pair = [&](const Segment& s, int grp) {
    const size_t head = (size_t)s.a * y.Hkv + s.hk;
    return (grp < G ? P.k_new + head * D + 64 * grp : P.v_new + head * Dv + 64 * (grp - G)) + 2 * lane;
  };
  // the segment's last chunk holds the agent's newest position, and the token is appended by this launch
  auto has_tail = [&](const Segment& s) { return P.k_new != nullptr && s.c1 == s.cf + s.nc; };
  uint4 qv = make_uint4(0u, 0u, 0u, 0u);                 // the next segment's query row and new-row groups, on their way
  uint32_t nv[kNewRounds];
  auto fetch_rows = [&](const Segment& s) {
    if (warp < n_rep && lane < D / 8) qv = *reinterpret_cast<const uint4*>(query_row(s));
    if (warp >= 4 && has_tail(s)) {
#pragma unroll
      for (int r = 0; r < kNewRounds; ++r) {
        const int grp = warp - 4 + kNewWarps * r;
        if (grp < G + Gv) nv[r] = *reinterpret_cast<const uint32_t*>(new_pair(s, grp));
      }
    }
  };
  // While the preceding kernel drains, ask L2 for the first chunks and rows.  A prefetch returns nothing to the kernel, and
  // L2 is where the preceding kernel's writes land, so what is read after the wait is current whatever it still writes.
  if (n_chunks > 0) {
    if (lane < 3 && lane < my_chunks && off != kOffBad) prefetch_l2_bulk(layer_base + (uint64_t)off * 16u, S::kChunkBytes);
    if (warp < n_rep && lane < D / 8 && (lane & 7) == 0) prefetch_l2(query_row(sm.seg[0]));
    if (warp >= 4 && has_tail(sm.seg[0]) && lane == 0)
      for (int grp = warp - 4; grp < G + Gv; grp += kNewWarps) prefetch_l2(new_pair(sm.seg[0], grp));
  }
  // Everything written here (outputs, records, tickets) may still be in use by the preceding kernels of the stream until
  // they have completed, and they may have written the pool, the queries and the new rows.
  grid_dependency_wait();
  if (n_chunks > 0) fetch_rows(sm.seg[0]);               // before the bulk copies, or the rows queue behind them
  if (lane < kSlots && lane < my_chunks) {
    issue_keys(lane, off);
    if (kHalves && lane < kValSlots) issue_values(lane, off);
  }

  if (cta * NW + warp < P.n_agents) clear_empty_agents(P, cta * NW + warp, gridDim.x * NW, Dv, lane);
  if (n_chunks == 0) return;                             // uniform over the CTA

  const int hcol[2] = {(2 * tid) & (H - 1), (2 * tid + 1) & (H - 1)};   // this lane's two score columns
  const uint32_t split_mask = tid >= 2 ? 0xFFFFE000u : 0u;
  const float margin = my_chunks > 1 ? kMargin : 0.f;
  bool aborted = false;
  uint32_t cur = __shfl_sync(0xffffffffu, off, 0), nxt = __shfl_sync(0xffffffffu, off, 1);   // offsets of the chunks in the two slots
  int i = 0;                                             // this warp's chunk counter: chunk k = warp + NW * i of the CTA
  const uint4* qb = &sm.qfrag[0][lane];
  for (int si = 0;; ++si) {
    const Segment& seg = sm.seg[si % 3];
    const int k0 = seg.k0, c0 = seg.c0, c1 = seg.c1, k1 = k0 + (c1 - c0);
    const int key_lo = seg.lo, key_n = seg.n;
    const bool newest = has_tail(seg);
    const bool tail = newest && (k1 - 1) % NW == warp;                  // this warp holds the chunk of the newest position
    if (warp < n_rep) stage_query_row<G, H>(sm.qfrag, sm.qsum, sm.kappa, qv, P.scale_log2, warp, lane);
    if (warp >= 4 && newest) {
#pragma unroll
      for (int r = 0; r < kNewRounds; ++r)
        if (warp - 4 + kNewWarps * r < G + Gv)
          quantize_row_group(nv[r], kBf, lane, sm.new_words + 8 * (warp - 4 + kNewWarps * r), sm.new_sb + warp - 4 + kNewWarps * r);
    }
    __syncthreads();
    const float* const qs0 = sm.qsum[hcol[0]];
    const float* const qs1 = sm.qsum[hcol[1]];
    const float kap[2] = {sm.kappa[hcol[0]], sm.kappa[hcol[1]]};
    WarpState<G> st;
    st.reset();
    bool poisoned = false;
    bool have = false;
#pragma unroll 1
    for (int k = warp + NW * i; k < k1; k += NW, ++i) {
      const int slot = i % kSlots;
      const uint32_t parity = (uint32_t)(i / kSlots) & 1u;
      const int j = i + kSlots;                          // the chunk this slot takes next
      const bool refill = j < my_chunks && !aborted;
      uint32_t noff = kOffBad;
      if (refill) {
        if ((j & 31) == 0) off = batch_offsets(P, sm.range, NW, warp, j >> 5, S::kChunkBytes);
        noff = __shfl_sync(0xffffffffu, off, j & 31);
      }
      const bool bad = cur == kOffBad;
      uint8_t* const chunk = ring + slot * (kHalves ? S::kKeyBytes : S::kChunkBytes);
      uint8_t* const vhalf = kHalves ? ring + kSlots * S::kKeyBytes : chunk + S::kKeyBytes;
      static_assert(!kHalves || kValSlots == 1, "");
      const bool patch = tail && k == k1 - 1;
      bool ok = mbar_wait(&sm.full[warp][slot], parity, &sm.abort_flag);
      if (kHalves && patch && ok) ok = mbar_wait(&sm.full_v[warp][0], (uint32_t)i & 1u, &sm.abort_flag);
      if (!ok) {
        // giving up: the copies this warp has in flight land (or are waited for long enough) before it goes on
        sm.abort_flag = 1;
        aborted = true;
        for (int s = 0; s < kSlots; ++s) {
          const int last = i + (s - slot + kSlots) % kSlots;
          if (last < my_chunks)
            for (uint32_t t = 0; t < 4096u && !mbar_try_wait(&sm.full[warp][s], (uint32_t)(last / kSlots) & 1u); ++t) {}
        }
        if (kHalves)
          for (uint32_t t = 0; t < 4096u && !mbar_try_wait(&sm.full_v[warp][0], (uint32_t)i & 1u); ++t) {}
        i = my_chunks;                                   // nothing is issued or read any more
        break;
      }
      const int pos0 = (c0 + (k - k0)) * 32;
      const bool edge = pos0 < key_lo || pos0 + 32 > key_n;
      if (bad) {
        poisoned = true;
      } else if (patch) {
        patch_new_row<G, H>(sm, chunk, vhalf, const_cast<uint8_t*>(layer_base) + (uint64_t)cur * 16u,
                            (key_n - 1) & 31, lane);
        __syncwarp();
      }
      float sc[4][2];
      if (!bad) chunk_scores<G, kBf>(chunk, g, tid, qb, qs0, qs1, sc);
      if (kHalves) {
        __syncwarp();
        if (refill && lane == 0) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the warp's reads and patches of the slot come first
          issue_keys(slot, noff);
        }
        if (!mbar_wait(&sm.full_v[warp][0], (uint32_t)i & 1u, &sm.abort_flag)) { sm.abort_flag = 1; poisoned = true; }
        __syncwarp();
      }
      if (!bad) {
        if (edge) {
          clear_outside<G>(vhalf + 32 * (Dv / 2), pos0, key_lo, key_n, lane);
          __syncwarp();
        }
        have = true;
        chunk_values<G, H, kBf>(vhalf, edge, pos0, key_lo, key_n, g, tid, kap, split_mask, margin, sc, st);
      }
      __syncwarp();
      if (kHalves) {
        if (i + 1 < my_chunks && lane == 0) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          issue_values(0, nxt);
        }
      } else if (refill && lane == 0) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        issue_keys(slot, noff);
      }
      cur = nxt;
      nxt = noff;
    }

    // ---- end of the segment: deposit, combine ----
    const bool more = sm.seg[(si + 1) % 3].a >= 0;
    if (more) fetch_rows(sm.seg[(si + 1) % 3]);
    if (have) {
      deposit<G, H>(sm, warp, lane, st, poisoned || aborted);
    } else if (lane < H) {
      sm.dep_m[warp][lane] = -INFINITY;
      sm.dep_l[warp][lane] = (poisoned || aborted) ? -1.f : 0.f;
    }
    __syncthreads();
    for (int unit = warp; unit < S::kDepUnits; unit += NW) combine_deposits<G, H>(sm, P, seg, cta, unit, lane);
    if (warp == NW - 1 && lane == 0) {
      if (seg.c1 - c0 != seg.nc) {                       // only the first and the last segment can be parts of a pair
        int* f = sm.fin[k0 == 0 ? 0 : 1];
        f[0] = seg.a * P.Hkv + seg.hk; f[1] = seg.first; f[2] = seg.last; f[3] = (kSingles ? P.q_offs[seg.a] : seg.a) * y.Hq + seg.hk * n_rep;
      }
      if (more) sm.walker.next(P, sm.range, sm.seg[(si + 2) % 3]);       // never where the CTA holds one segment
    }
    if (!more) break;
    __syncthreads();
  }
  if (aborted && lane == 0) raise_flag(P.flags, Q4KV_FLAG_INTERNAL);

  // ---- tickets: all CTAs end at about the same time, so the first segment's is drawn here too, beside the last one's.
  // The CTA's record stores are ordered before the atomic by the barrier, other CTAs' record loads after it by the second:
  // one acquire-release atomic takes the place of a fence on either side. ----
  __syncthreads();
  if (lane == 0 && warp % (NW / 2) == 0) {
    const int x = warp / (NW / 2);
    int last = 0;
    if (sm.fin[x][0] >= 0) {
      int old;
      asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(old) : "l"(&P.tickets[sm.fin[x][0]]) : "memory");
      last = old == sm.fin[x][2] - sm.fin[x][1];
      if (last) P.tickets[sm.fin[x][0]] = 0;             // ready for the next call
    }
    sm.fin_last[x] = last;
  }
  __syncthreads();
  const bool both = (sm.fin_last[0] & sm.fin_last[1]) != 0;
#pragma unroll 1
  for (int x = 0; x < 2; ++x) {
    if (!sm.fin_last[x]) continue;
    // one warp per head and 128 elements: all warps when one pair is to be combined, half of them each when there are two
    const int first = both ? NW / 2 * x : 0, count = both ? NW / 2 : NW;
    if (warp < first || warp >= first + count) continue;
    const size_t rstride = (size_t)n_rep * kRecStride(Dv);
    for (int t = warp - first; t < n_rep * (Dv / 128); t += count) {
      const int h = t / (Dv / 128), d = (t % (Dv / 128)) * 128 + 4 * lane;
      combine_records(P, P.partials + (size_t)(sm.fin[x][0] + sm.fin[x][1]) * rstride + (size_t)h * kRecStride(Dv), rstride,
                      sm.fin[x][2] - sm.fin[x][1] + 1, Dv, d, (size_t)sm.fin[x][3] + h, lane);
    }
  }
}

template <int G, int H, bool kBf, bool kSingles>
cudaError_t launch_g(const DecodeParams& P_, int grid, cudaStream_t st) {
  static bool configured[64] = {};     // the attributes are per function and device: set them once for each
  constexpr size_t smem = sizeof(Smem<G, H>);
  static_assert(smem <= 227 * 1024 / kCtasPerSm - 1024, "two CTAs per SM");
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    e = cudaFuncSetAttribute(decode_mma_kernel<G, H, kBf, kSingles>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(decode_mma_kernel<G, H, kBf, kSingles>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(warps_of(G) * 32);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  Params<kSingles> P;
  static_cast<DecodeParams&>(P) = P_;
  return cudaLaunchKernelEx(&cfg, decode_mma_kernel<G, H, kBf, kSingles>, P);
}
template <int G, int H>
cudaError_t launch_gh(const DecodeParams& P, int grid, cudaStream_t st) {
  if (P.q_offs) return P.y.sb_bf16 ? launch_g<G, H, true, true>(P, grid, st) : launch_g<G, H, false, true>(P, grid, st);
  return P.y.sb_bf16 ? launch_g<G, H, true, false>(P, grid, st) : launch_g<G, H, false, false>(P, grid, st);
}

// Sets of query heads a KV head's heads are cut into: the kernel's columns take four of them, or eight at d = 128
int head_sets(const Layout& y) {
  const int most = y.D == 128 ? 8 : 4;
  int sets = (y.n_rep + most - 1) / most;
  while (y.n_rep % sets) ++sets;
  return sets;
}

}  // namespace

// Number of SMs of the current device, looked up once per device.
int sm_count() {
  static int cached[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { (void)cudaGetLastError(); return 148; }
  if (cached[dev] == 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) { (void)cudaGetLastError(); n = 148; }
    cached[dev] = n < kMaxGrid ? n : kMaxGrid;
  }
  return cached[dev];
}

bool decode_mma_supported(const Layout& y) {
  return !y.alias && ((y.D == y.Dv && (y.D == 128 || y.D == 256)) || (y.D == 192 && y.Dv == 128));
}

// the kernel counts work units in 32 bits and keeps one arrival counter per (layer of the call, agent, head set) in
// the workspace header; chunk offsets inside the call's layers are kept in 16-byte units in 32 bits
bool decode_mma_fits(const Layout& y, int n_agents, int max_blocks, int layer_count) {
  const long long v = (long long)n_agents * layer_count * head_sets(y);
  return layer_count >= 1 && layer_count <= kMaxLayersPerCall && v * y.Hkv * (max_blocks * 8ll) < (1ll << 30) &&
         v * y.Hkv <= kMaxTicketPairs && (unsigned long long)layer_count * y.layer_bytes < (1ull << 36);
}

int decode_mma_tickets(const Layout& y, int n_agents) { return n_agents * y.Hkv * head_sets(y); }

// bytes behind the workspace header: one record per (layer, agent, head set) and per CTA of the largest grid
size_t decode_mma_workspace_bytes(const Layout& y, int n_agents, int layer_count) {
  const int sets = head_sets(y);
  const size_t pairs = (size_t)n_agents * layer_count * y.Hkv * sets;
  return (pairs + kMaxGrid) * (y.n_rep / sets) * kRecStride(y.Dv) * sizeof(float);
}

// layer_count == 1: `windows` points at the one window.  Otherwise q, out, lse and the new rows hold layer_count
// consecutive per-layer arrays and the launch covers layers layer .. layer + layer_count - 1.
cudaError_t launch_decode_mma(const Layout& y, const void* pool, int n_blocks, int layer, const q4kv_batch& b,
                              const int32_t* kv_lens, int max_kv_len, const int32_t* windows, int layer_count,
                              const void* q, float scale, void* out, int out_dtype, float* lse, void* ws, int32_t* flags,
                              cudaStream_t st, const void* k_new, const void* v_new, const int32_t* q_offs, int32_t* tickets) {
  if (b.n_agents <= 0 || layer_count <= 0) return cudaSuccess;
  DecodeParams P;
  P.y = y; P.pool = (const uint8_t*)pool; P.n_blocks = n_blocks; P.layer = layer; P.n_agents = b.n_agents * layer_count;
  P.n_real = b.n_agents; P.layer_count = layer_count;
  P.sets = head_sets(y); P.Hkv = y.Hkv * P.sets; P.n_rep = y.n_rep / P.sets;
  long long wanted = 0;
  for (int i = 0; i < kMaxLayersPerCall; ++i) {
    P.windows[i] = i < layer_count ? windows[i] : 0;
    if (i < layer_count) {
      const int span = (windows[i] > 0 && windows[i] + 32 < max_kv_len) ? windows[i] + 32 : max_kv_len;
      const int chunks = (span + 31) / 32, nw = warps_of(y.G);
      wanted += (long long)b.n_agents * P.Hkv * ((chunks + nw - 1) / nw);       // a chunk per warp, and no CTA with two pairs
    }
  }
  P.max_blocks = b.max_blocks; P.len_cap = max_kv_len; P.tables = b.block_tables; P.kv_lens = kv_lens;
  P.q = (const uint16_t*)q; P.scale_log2 = scale * kLog2e;
  P.tickets = tickets ? tickets : (int32_t*)ws; P.partials = (float*)((uint8_t*)ws + kWorkspaceHeaderBytes);
  P.out = out; P.out_dtype = out_dtype; P.lse = lse; P.flags = flags;
  P.k_new = (const uint16_t*)k_new; P.v_new = (const uint16_t*)v_new;
  P.q_offs = q_offs;
  // No more CTAs than can be of use: one that finds nothing to do costs the next launch a microsecond, because its CTAs come in as
  // this one's leave.  No fewer than pairs, which one CTA would take in turn: a launch on contexts of 30 tokens took 25.5 us with
  // a CTA per eight chunks, 4.3 with one per pair, on 100 tokens 7.2 and 4.3, at d = 256 13.8 and 6.7.
  // Every pair is rounded up at the longest length, the only one known here: 16 KV heads of 837, 1088 and 227 tokens take 7.36 us with
  // 240 CTAs and 7.31 with 204, but three of 1088 7.54 and 8.01, a round more for every pair.
  // Two CTAs per SM for small batches too.  One, so that the next launch's CTAs sit beside this one's: us a launch with one and with two,
  // 8 KV heads: 2 x 4096 9.8 / 9.2, 6 x 1500 9.4 / 8.8, 8 x 1000 9.8 / 8.6, 10 x 1000 12.0 / 9.6, 5 x 1100 9.1 / 7.9, 3 x 4096 11.1 / 10.4;
  // the other way round 16 agents x 300..700, 9.3 / 9.7.  It also doubles the chunks that a warp adds up, and the tensor cores truncate
  // their sums: against 64 bits, one agent x 4264 at 16 KV heads was off by 5.2e-4 instead of 4.1e-4.
  const long long slots = sm_count() * kCtasPerSm < kMaxGrid ? sm_count() * kCtasPerSm : kMaxGrid;
  const int grid = (int)(wanted < slots ? (wanted < 1 ? 1 : wanted) : slots);
  if (y.G == 2) return P.n_rep > 4 ? launch_gh<2, 8>(P, grid, st) : launch_gh<2, 4>(P, grid, st);
  return y.G == 3 ? launch_gh<3, 4>(P, grid, st) : launch_gh<4, 4>(P, grid, st);
}

}  // namespace q4kv
