// q4kv_prefill_attention on the MLA-latent cache in absorbed form (V aliasing K, d_qk 576, d_v 512): the queries of a new
// phase over the cached latents plus the causal new tokens, read from the Q4 cache in place (Sections 3.4, 3.5, 3.6).
//
// A dense contraction (1088 multiply-adds per query head and key), so it runs on the fifth-generation tensor cores.  Every
// key is key and value of all the heads, which decides the shape:
//   * A 128-row tile (128 / n_rep consecutive queries x the n_rep heads) has a 512-column accumulator, which is all of the
//     tensor memory.  So two CTAs share a tile: both take the scores over all 576 dims, each accumulates 256 of the 512 value
//     dims (832 instead of 544 multiply-adds per head, key and CTA: the price of not exchanging scores between SMs).
//     Tensor memory: O 256 columns, S 2 x 64, and the first 256 dims of the queries as packed binary16 (128); the other 320
//     dims of the queries are 80 KB of shared memory.
//   * Keys are walked 64 at a time.  Eight "dequantize" warps load a block's codes straight into registers, one block
//     ahead (the raw bytes would not fit beside the tiles, and each is used once), and write the binary16 tile K^ [64
//     keys][576 dims] (72 KB, two stages): x^ = c * s + b in one binary16 fma per pair of codes, one rounding per value.
//     The tile is the K-major B operand of the score product and, read the other way (MN-major), the B operand of the value
//     product: values are never written.  A packed word is one 16-byte row of a core matrix, elements in the order
//     0,4,1,5,2,6,3,7; the queries are stored in that order and the output columns are put back in place at the end.
//   * One thread issues the MMAs: S_b = Q K^T (M 128, N 64: 16 instructions with the queries in tensor memory at 33 clocks, 20
//     with them in shared memory at 55) and O += P_b V^ (M 128, N 256: 4 at 129): 2140 clocks of tensor pipe per block.
//     A CTA's value product reads 256 of a block's 576 dims; the other 320 can be overwritten as soon as the block's scores
//     are complete, and the next scores can start on them.  So a stage has two parts: part A (the 320), part B (the 256).
//     Score and value products are issued as their inputs become ready, not in a fixed order: a value product that waited
//     for the next scores would hold the K^ stage that the block after them needs (6200 clocks per block that way).
//   * Four softmax warps, one thread per score row: mask, online softmax with a lazily updated reference maximum (rescaling
//     only when the row maximum has grown by more than 2^8), P_b as packed binary16 over S_b.  Nothing is exchanged between
//     threads, so a row's softmax waits for nothing but its scores.
//   * With few tiles the keys of a tile are cut over several CTAs as well (plan_prefill_splits); these leave (acc, m, l)
//     records that merge_prefill_kernel combines.
// Measured on 3 agents x (250 .. 512 queries on 2000 .. 4000 keys), 16 heads (102 GFLOP): 36 ms on the shape-agnostic kernel,
// 0.196 ms here = 519 TFLOP/s back to back (0.203 with a thread loading and storing its own row); 3650 clocks per block, of which the dequantize warps are busy 2600 -- they, the softmax and the
// products share the shared-memory bandwidth (256 KB per block: 2000 clocks) and the issue slots.
// All hand-offs are mbarriers; every wait is bounded and a wait that runs out raises Q4KV_FLAG_INTERNAL, drains the tensor
// pipe and frees the tensor memory before the CTA returns.
#include <type_traits>

#include "prefill_common.cuh"

namespace q4kv {

namespace {

using namespace tc;
using namespace prefill;

constexpr int kSoftmaxWarps = 4, kDequantWarps = 8;
constexpr int kMmaWarp = kSoftmaxWarps + kDequantWarps;
constexpr int kThreads = (kMmaWarp + 1) * 32;            // 416: four warps on one scheduler at most, 128 registers
constexpr int kStages = 2;
constexpr int kG = 9, kD = 576, kDv = 512, kDvCta = 256;
constexpr int kQTmem = 256, kQSmem = kD - kQTmem;        // query dims in tensor memory and in shared memory
constexpr int kSboK = (kD / 8) * 128, kSboQ = (kQSmem / 8) * 128;
constexpr int kChunkBytes = 32 * (kD / 2 + 4 * kG);      // [Kc 9216 | Ksb 1152]
constexpr uint32_t kColO = 0, kColS = 256, kColQ = 384;

struct MlaPrefillParams {
  Layout y;
  const uint8_t* pool;
  int n_blocks, layer, n_agents, max_blocks;
  const int32_t* tables;
  const int32_t* kv_lens;
  const int32_t* q_offs;
  int window;
  const uint16_t* q;          // bf16 [total_q][Hq][576]
  float scale_log2;
  void* out;
  int out_dtype;
  float* lse;
  int32_t* flags;
  int n_splits;
  float* records;             // n_splits > 1: [total_q][Hq][n_splits][kRecord]
  CodeMasks masks;
};

struct MlaSmem {
  alignas(128) uint8_t khat[kStages][64 * kD * 2];       // [key][dim]: (n%8)*16 + (n/8)*kSboK + (k/8)*128
  alignas(128) uint8_t qs[128 * kQSmem * 2];             // [row][dim - 256]: (m%8)*16 + (m/8)*kSboQ + (k/8)*128
  alignas(8) uint64_t a_full[kStages], b_full[kStages], a_free[kStages], b_free[kStages], s_full[2], p_full[2], o_done, o_last, q_ready, drain;
  uint32_t tmem_base;
  int abort_flag, poisoned;
};

template <bool kBf>
__global__ void __launch_bounds__(kThreads, 1) prefill_mla_kernel(const __grid_constant__ MlaPrefillParams P) {
  extern __shared__ __align__(128) uint8_t smem_raw[];
  MlaSmem& sm = *reinterpret_cast<MlaSmem*>(smem_raw);

  const Layout& y = P.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_rep = y.n_rep;
  // grid: x = (tile, value half), y = (KV head, split), z = agent
  const int qt = blockIdx.x >> 1, hv = blockIdx.x & 1, hk = blockIdx.y / P.n_splits, split = blockIdx.y % P.n_splits, a = blockIdx.z;
  const int tile_q = 128 / n_rep;                        // queries of the CTA's 128-row tile

  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // ---- this CTA's queries and key range (inputs no kernel writes) ----
  const int q0 = P.q_offs[a], q_len = P.q_offs[a + 1] - q0;
  const int kv_len = P.kv_lens[a];
  const int i_min = qt * tile_q;
  if (i_min >= q_len) return;                            // uniform: nothing allocated, no barrier passed
  const bool bad_len = kv_len < 0 || kv_len > P.max_blocks * kBlockTokens || q_len > kv_len;
  const int i_max = min(q_len, i_min + tile_q) - 1;
  const int prefix = kv_len - q_len;                     // query i sits at position prefix + i
  const int W = P.window;
  const int c_end = bad_len ? 0 : (prefix + i_max) / 32 + 1;
  const int c_begin = (bad_len || W == 0) ? 0 : max(0, prefix + i_min - W + 1) >> 5;
  const int all0 = c_begin >> 1, n_all = max(0, ((c_end + 1) >> 1) - all0);
  const int it0 = all0 + n_all * split / P.n_splits;     // 64-key blocks it0 .. it0 + n_iter - 1
  const int n_iter = all0 + n_all * (split + 1) / P.n_splits - it0;

  if (threadIdx.x == 0) {
    if (bad_len) raise_flag(P.flags, Q4KV_FLAG_BAD_LENGTH);
    for (int s = 0; s < kStages; ++s) { 
      mbar_init(&sm.a_full[s], kDequantWarps); mbar_init(&sm.b_full[s], kDequantWarps);
      mbar_init(&sm.a_free[s], 1); mbar_init(&sm.b_free[s], 1);
    }
    for (int b = 0; b < 2; ++b) { mbar_init(&sm.s_full[b], 1); mbar_init(&sm.p_full[b], kSoftmaxWarps * 32); }
    mbar_init(&sm.o_done, 1);
    mbar_init(&sm.o_last, 1);
    mbar_init(&sm.q_ready, kSoftmaxWarps * 32);
    mbar_init(&sm.drain, 1);
    sm.abort_flag = 0; sm.poisoned = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  if (warp == kMmaWarp) { tmem_alloc(&sm.tmem_base, 512); tmem_relinquish(); }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tb = sm.tmem_base;
  if (warp == kSoftmaxWarps) ask_for_blocks(P, a, hk, it0, min(n_iter, 2), kChunkBytes);
  if (warp < kSoftmaxWarps && !bad_len) {
    const int h = (int)threadIdx.x / tile_q, i = i_min + (int)threadIdx.x % tile_q;
    if (i < q_len && h < n_rep) ask_for_row<kD>(P.q + ((size_t)(q0 + i) * y.Hq + (size_t)hk * n_rep + h) * kD);
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");     // the new tokens were appended by the preceding kernel
  volatile int* abort_flag = &sm.abort_flag;

  if (warp >= kSoftmaxWarps && warp < kMmaWarp) {
    // =============================== dequantize warps ==========================================
    // Thread (chunk c1 of the block, token tau = 4 kg + ki, kt): the words 4 p + kt, p = 0..17, of its token (four 16-byte
    // pieces and an 8-byte one) and the token's nine (scale, bias) pairs.  A lane group of eight holds the eight tokens of
    // a core matrix at one kt: its stores fill a 128-byte line, its loads are two pieces of each of four lines.
    const int x = threadIdx.x - kSoftmaxWarps * 32;      // 0..255
    const int c1 = x >> 7, kt = (x >> 3) & 3, ki = x & 3, kg = 2 * ((x >> 5) & 3) + ((x >> 2) & 1);
    const int ktau = 4 * kg + ki;
    const int read16 = ki * (256 * kG) + kg * 64 + kt * 16, read8 = ki * (256 * kG) + 2048 + kg * 32 + kt * 8;
    const int read_sb = 1024 * kG + (((ktau & 3) * 4 + (ktau >> 3)) * 2 + ((ktau >> 2) & 1)) * (4 * kG);
    const int n = c1 * 32 + ktau;
    const int write = (n & 7) * 16 + (n >> 3) * kSboK + kt * 128;         // + p * 512
    uint4 w16[4];
    uint2 w8;
    uint32_t sb[kG];
    // this thread's part of a block, piece by piece; nullptr (no pool block, or a token past the end): zeros
    auto locate = [&](int j) {
      const int c = 2 * (it0 + j) + c1;
      const int blk = __ldg(&P.tables[(size_t)a * P.max_blocks + (c >> 3)]);
      const bool bad = blk < 0 || blk >= P.n_blocks;
      if (bad && lane == 0) { sm.poisoned = 1; raise_flag(P.flags, Q4KV_FLAG_BAD_BLOCK); }
      if (bad || c * 32 + ktau >= kv_len) return (const uint8_t*)nullptr;
      return head_block(P.pool, y, P.layer, blk, hk) + (size_t)(c & 7) * kChunkBytes;
    };
    auto fetch16 = [&](const uint8_t* chunk, int i) {
      w16[i] = chunk ? __ldcg(reinterpret_cast<const uint4*>(chunk + read16 + 512 * i)) : make_uint4(0u, 0u, 0u, 0u);
    };
    auto fetch8 = [&](const uint8_t* chunk) { w8 = chunk ? __ldcg(reinterpret_cast<const uint2*>(chunk + read8)) : make_uint2(0u, 0u); };
    auto fetch_sb = [&](const uint8_t* chunk, int i) {
      // through L1 (a line holds several tokens' pairs), but not as read-only data: the append before writes them while this runs
      sb[i] = chunk ? *reinterpret_cast<const uint32_t*>(chunk + read_sb + 4 * i) : 0u;
    };
    const uint8_t* next = nullptr;
    if (n_iter > 0) {
      next = locate(0);
#pragma unroll
      for (int i = 0; i < 4; ++i) fetch16(next, i);
      fetch8(next);
#pragma unroll
      for (int i = 0; i < kG; ++i) fetch_sb(next, i);
      next = n_iter > 1 ? locate(1) : nullptr;
    }
    // Word p of a token belongs to part B if it is one of the CTA's value dims (words 8 hv .. 8 hv + 7), else to part A.
    auto run = [&](auto half) {
      constexpr int kHv = decltype(half)::value;
      for (int j = 0; j < n_iter; ++j) {
        const int s = j % kStages;
        uint8_t* dst = sm.khat[s] + write;
        bool overflow = false;
        // a register that has been used takes the next block's bytes at once, so that the loads are spread over the block
        const uint8_t* const chunk = next;
        auto word = [&](int p) {
          if (kBf && (p & 1) == 0) sb[p >> 1] = bf16_pair_to_h2(sb[p >> 1], overflow);
          const uint4& v = w16[(p >> 2) & 3];
          const uint32_t w = p >= 16 ? (p == 16 ? w8.x : w8.y) : (p & 3) == 0 ? v.x : (p & 3) == 1 ? v.y : (p & 3) == 2 ? v.z : v.w;
          const uint32_t sp = __byte_perm(sb[p >> 1], sb[p >> 1], 0x1010), bp = __byte_perm(sb[p >> 1], sb[p >> 1], 0x3232);
          *reinterpret_cast<uint4*>(dst + p * 512) = dequant8(w, sp, bp, sp, bp, sp, bp, sp, bp, P.masks);
          if (p & 1) fetch_sb(chunk, p >> 1);
          if (p < 16 && (p & 3) == 3) fetch16(chunk, p >> 2);
          if (p == 17) fetch8(chunk);
        };
        if (j >= kStages && !mbar_wait(&sm.a_free[s], (uint32_t)(j / kStages - 1), abort_flag)) break;
#pragma unroll
        for (int p = 0; p < 18; ++p)
          if (p / 8 != kHv) word(p);
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.a_full[s]);
        if (j >= kStages && !mbar_wait(&sm.b_free[s], (uint32_t)(j / kStages - 1), abort_flag)) break;
#pragma unroll
        for (int p = 8 * kHv; p < 8 * kHv + 8; ++p) word(p);
        if (kBf && overflow) raise_flag(P.flags, Q4KV_FLAG_SB_RANGE);
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.b_full[s]);
        next = j + 2 < n_iter ? locate(j + 2) : nullptr;
      }
    };
    if (hv == 0) run(std::integral_constant<int, 0>()); else run(std::integral_constant<int, 1>());
  } else if (warp == kMmaWarp) {
    // =============================== MMA issue ==================================================
    // The whole warp runs this code, and one elected lane (always the same) issues: one election for a whole product
    // (an election per MMA made the issue of a block 20 % longer than its execution).
    if (n_iter > 0) {
      constexpr uint32_t kIdescS = idesc_f16(128, 64), kIdescO = idesc_f16(128, kDvCta, 0, 1);
      const uint64_t qd = smem_desc(smem_u32(sm.qs), 128, kSboQ);
      // part A or B of S_b = Q K^T: the 16-dim steps outside / inside the CTA's value dims
      auto issue_qk = [&](int b, int s, auto half, auto part_b) {
        constexpr int kHv = decltype(half)::value;
        constexpr bool kB = decltype(part_b)::value;
        constexpr int kFirst = kHv == 0 ? 16 : 0;        // of part A
        const uint64_t kd = smem_desc(smem_u32(sm.khat[s]), 128, kSboK);
        if (elect_one()) {
#pragma unroll
          for (int k = 0; k < kD / 16; ++k) {
            if ((k / 16 == kHv) != kB) continue;
            const uint32_t accumulate = !kB && k == kFirst ? 0u : 1u;
            if (k < kQTmem / 16)
              mma_f16_ts(tb + kColS + 64 * b, tb + kColQ + 8 * k, kd + 16 * k, kIdescS, accumulate);
            else
              mma_f16_ss(tb + kColS + 64 * b, qd + 16 * (k - kQTmem / 16), kd + 16 * k, kIdescS, accumulate);
          }
          if (kB) { commit(&sm.s_full[b]); commit(&sm.a_free[s]); }
        }
        __syncwarp();
      };
      auto issue_pv = [&](int b, int s, bool first, bool last) {    // O (+)= P_b V^; afterwards the stage is free
        const uint64_t vd = smem_desc(smem_u32(sm.khat[s]) + hv * (kDvCta / 8) * 128, kSboK, 128);
        if (elect_one()) {
#pragma unroll
          for (int k = 0; k < 4; ++k)
            mma_f16_ts(tb + kColO, tb + kColS + 64 * b + 8 * k, vd + (2 * kSboK / 16) * k, kIdescO, (!first || k > 0) ? 1u : 0u);
          commit(&sm.o_done);
          if (last) commit(&sm.o_last);
          commit(&sm.b_free[s]);
        }
        __syncwarp();
      };
      bool ok = __all_sync(0xffffffffu, mbar_wait(&sm.q_ready, 0, abort_flag));
      int na = 0, nb = 0, np = 0;                        // blocks whose scores (parts A, B) / values have been issued
      uint32_t idle = 0;
      auto run = [&](auto half) {
        while (ok && np < n_iter) {
          if (np < nb && __all_sync(0xffffffffu, mbar_test_wait(&sm.p_full[np & 1], (uint32_t)(np >> 1) & 1u))) {
            fence_after_sync();
            issue_pv(np & 1, np % kStages, np == 0, np + 1 == n_iter);
            ++np;
            idle = 0;
          }
          // part A of block na: its keys are there, and the probabilities that its buffer held have been used
          if (na < n_iter && na < np + 2 && __all_sync(0xffffffffu, mbar_test_wait(&sm.a_full[na % kStages], (uint32_t)(na / kStages) & 1u))) {
            fence_after_sync();
            issue_qk(na & 1, na % kStages, half, std::false_type());
            ++na;
            idle = 0;
          }
          if (nb < na && __all_sync(0xffffffffu, mbar_test_wait(&sm.b_full[nb % kStages], (uint32_t)(nb / kStages) & 1u))) {
            fence_after_sync();
            issue_qk(nb & 1, nb % kStages, half, std::true_type());
            ++nb;
            idle = 0;
          }
          if (++idle > 64) {
            __nanosleep(64);
            ok = __all_sync(0xffffffffu, idle < (1u << 25) && !*abort_flag);
            if (!ok) *abort_flag = 1;
          }
        }
      };
      if (hv == 0) run(std::integral_constant<int, 0>()); else run(std::integral_constant<int, 1>());
    }
  } else if (warp < kSoftmaxWarps) {
    // =============================== softmax warps: one thread per score row ===================
    const int row = warp * 32 + lane;                    // tensor-memory lane
    const uint32_t lane_addr = tb + ((uint32_t)(warp * 32) << 16);
    const int h = row / tile_q, i = i_min + row % tile_q;
    const bool mine = i < q_len && h < n_rep;            // a row of the output
    const int pq = prefix + i;                           // this row's position
    const size_t row_index = (size_t)(q0 + i) * y.Hq + (size_t)hk * n_rep + h;
    float kappa = 0.f;                                   // score in log2 units = S * kappa
    {
      // ---- stage the warp's query rows: bf16 -> binary16 times a power of two per row; pieces of eight dims 0..31 go to tensor
      //      memory, 32..71 to shared memory.  The lanes share the rows' lines (see load_rows), eight rows at a time: 18 loads a
      //      lane in flight are enough, and unrolled over all rows it spills (the launches of few tiles then take 33 us for 30).  Of
      //      the shared-memory part only the maximum is wanted in this pass, so its registers are free before the others are used
      //      (all 18 kept: 24 bytes spilled; 3 x (3000 + 400) tokens, two layers, 704.4 -> 697.2 us).  The warp's part of the
      //      shared-memory tile is the buffer on the way to tensor memory. ----
      uint8_t* const buf = sm.qs + 4 * warp * kSboQ;     // 16 KB of the warp's 20: [quarter of the tensor-memory part][32 rows x 128 bytes]
      const float per = __fdividef(1.f, (float)tile_q);
      auto row_at = [&](int r) -> const uint16_t* {      // the query in row r of the tile, this lane's first piece of it
        const int h = (int)(((float)r + 0.5f) * per), i = i_min + r - h * tile_q;   // r < 128: exact
        return i < q_len && h < n_rep && !bad_len ? P.q + ((size_t)(q0 + i) * y.Hq + (size_t)hk * n_rep + h) * kD + 8 * (lane >> 3) : nullptr;
      };
      float sf_own = 0.f;
#pragma unroll 1
      for (int g = 0; g < 4; ++g) {
        const uint16_t* row_g = row_at(warp * 32 + 8 * g + (lane & 7));
        uint4 v[kQTmem / 32];
        float mx = 0.f;
        {
          uint4 rest[kQSmem / 32];
#pragma unroll
          for (int k = 0; k < kQSmem / 32; ++k) rest[k] = piece_of(row_g, kQTmem / 8 + 4 * k);
#pragma unroll
          for (int k = 0; k < kQTmem / 32; ++k) v[k] = piece_of(row_g, 4 * k);
#pragma unroll
          for (int k = 0; k < kQSmem / 32; ++k) mx = fmaxf(mx, max_abs8(rest[k]));
        }
#pragma unroll
        for (int k = 0; k < kQTmem / 32; ++k) mx = fmaxf(mx, max_abs8(v[k]));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
        int ex = (int)((__float_as_uint(mx) >> 23) & 255u) - 127;
        if (mx == 0.f) ex = 0;
        ex = min(max(ex, -100), 100);
        const float sf = __uint_as_float((uint32_t)(127 + 8 - ex) << 23);      // 256 <= max |q| * sf < 512
        if ((lane >> 3) == g) {
          sf_own = sf;
          kappa = P.scale_log2 * __uint_as_float((uint32_t)(127 - 8 + ex) << 23);
        }
#pragma unroll
        for (int k = 0; k < kQTmem / 32; ++k)            // pieces 4 k + lane / 8: half of a 128-byte row's
          *reinterpret_cast<uint4*>(buf + (k >> 1) * kRowsBytes + piece_at(8 * g + (lane & 7), 4 * (k & 1) + (lane >> 3))) = query8(v[k], sf);
      }
      __syncwarp();
#pragma unroll 1
      for (int c = 0; c < kQTmem / 64; ++c) {            // 32 columns (64 dims) at a time
        uint32_t qa[32];
#pragma unroll
        for (int p = 0; p < 8; ++p) *reinterpret_cast<uint4*>(qa + 4 * p) = *reinterpret_cast<const uint4*>(buf + c * kRowsBytes + piece_at(lane, p));
        tmem_st32(lane_addr + kColQ + 32 * c, qa);
      }
      __syncwarp();                                      // the buffer has been read: the shared-memory part takes its place
#pragma unroll 1
      for (int g = 0; g < 4; g += 2) {
        uint4 v[2][kQSmem / 32];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const uint16_t* row_g = row_at(warp * 32 + 8 * (g + e) + (lane & 7));
#pragma unroll
          for (int k = 0; k < kQSmem / 32; ++k) v[e][k] = piece_of(row_g, kQTmem / 8 + 4 * k);
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int r = warp * 32 + 8 * (g + e) + (lane & 7);
          const float sf = __shfl_sync(0xffffffffu, sf_own, 8 * (g + e) + (lane & 7));
#pragma unroll
          for (int k = 0; k < kQSmem / 32; ++k)
            *reinterpret_cast<uint4*>(sm.qs + (r & 7) * 16 + (r >> 3) * kSboQ + (4 * k + (lane >> 3)) * 128) = query8(v[e][k], sf);
        }
      }
      wait_st();
      fence_async_smem();
      fence_before_sync();
      mbar_arrive(&sm.q_ready);
    }
    float m_ref = -INFINITY, l = 0.f;                    // p = 2^(s - m_ref); m_ref trails the true maximum by at most kLazy
    for (int j = 0; j < n_iter; ++j) {
      const int b = j & 1;
      if (!mbar_wait(&sm.s_full[b], (uint32_t)(j >> 1), abort_flag)) break;
      fence_after_sync();
      __syncwarp();
      uint32_t sr[64];
      tmem_ld32(lane_addr + kColS + 64 * b, sr);
      tmem_ld32(lane_addr + kColS + 64 * b + 32, sr + 32);
      wait_ld32(sr);
      wait_ld32(sr + 32);
      const int pos0 = (it0 + j) * 64;
      // column c is key pos0 + c; causal and window masks on edge blocks only
      if (pos0 + 63 > pq || (W > 0 && pos0 <= pq - W)) {
#pragma unroll
        for (int c = 0; c < 64; ++c)
          if (pos0 + c > pq || (W > 0 && pos0 + c <= pq - W)) sr[c] = 0xff800000u;   // -inf
      }
      float cm4[4] = {__uint_as_float(sr[0]), __uint_as_float(sr[1]), __uint_as_float(sr[2]), __uint_as_float(sr[3])};
#pragma unroll
      for (int c = 4; c < 64; ++c) cm4[c & 3] = fmaxf(cm4[c & 3], __uint_as_float(sr[c]));
      float cm = fmaxf(fmaxf(cm4[0], cm4[1]), fmaxf(cm4[2], cm4[3]));
      if (cm != -INFINITY) cm *= kappa;                  // kappa > 0
      const float m_new = fmaxf(m_ref, cm);
      const bool grow = m_new > m_ref + kLazy || (m_ref == -INFINITY && m_new != -INFINITY);
      if (__any_sync(0xffffffffu, grow)) {
        if (j > 0) {
          // rescale the accumulator row: the previous block's value product must have landed
          if (!mbar_wait(&sm.o_done, (uint32_t)(j - 1), abort_flag)) break;
          fence_after_sync();
          __syncwarp();
          const float f = grow ? fast_exp2(m_ref - m_new) : 1.f;           // m_ref = -inf: 0
#pragma unroll 1
          for (int part = 0; part < kDvCta / 16; ++part) {
            uint32_t orow[16];
            tmem_ld16(lane_addr + kColO + 16 * part, orow);
            wait_ld16(orow);
#pragma unroll
            for (int c = 0; c < 16; ++c) orow[c] = __float_as_uint(__uint_as_float(orow[c]) * f);
            tmem_st16(lane_addr + kColO + 16 * part, orow);
          }
          if (grow) l *= f;
        }
        if (grow) m_ref = m_new;
      }
      const float neg_m = m_ref == -INFINITY ? 0.f : -m_ref;
      float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
      uint32_t pr[32];
#pragma unroll
      for (int c = 0; c < 32; c += 2) {
        const float p0 = fast_exp2(fmaf(__uint_as_float(sr[2 * c]), kappa, neg_m));
        const float p1 = fast_exp2(fmaf(__uint_as_float(sr[2 * c + 1]), kappa, neg_m));
        const float p2 = fast_exp2(fmaf(__uint_as_float(sr[2 * c + 2]), kappa, neg_m));
        const float p3 = fast_exp2(fmaf(__uint_as_float(sr[2 * c + 3]), kappa, neg_m));
        s0 += p0; s1 += p1; s2 += p2; s3 += p3;
        pr[c] = f32x2_to_h2(p0, p1);
        pr[c + 1] = f32x2_to_h2(p2, p3);
      }
      l += (s0 + s1) + (s2 + s3);
      tmem_st32(lane_addr + kColS + 64 * b, pr);         // P_b overlays the first 32 columns of S_b
      wait_st();
      fence_before_sync();
      mbar_arrive(&sm.p_full[b]);
    }
    // ---- normalise and write the row, or leave it as a record ----
    bool ok = !*abort_flag;
    // (the last two value products may both be under way, and a wait on o_done could not tell which phase it sees)
    if (ok && n_iter > 0) ok = mbar_wait(&sm.o_last, 0, abort_flag);
    ok = __all_sync(0xffffffffu, ok);                    // the loads below are warp-wide
    if (ok) fence_after_sync();
    const bool bad = !ok || sm.poisoned != 0;
    const bool zero = bad || n_iter == 0 || l <= 0.f;
    const bool final = P.n_splits == 1;
    const float inv = zero ? 0.f : final ? 1.f / l : 1.f;
    // (the queries are not needed any more: every product that read them is complete)
    uint8_t* const buf = sm.qs + 4 * warp * kSboQ;
    const size_t at = final ? row_index * kDv : (row_index * P.n_splits + split) * prefill_record(kDv);
    const RowsOut to = rows_out(at + kDvCta * hv, mine, final && P.out_dtype == Q4KV_OUT_BF16);
#pragma unroll 1
    for (int part = 0; part < kDvCta / 32; ++part) {
      uint32_t orow[32];
      if (ok && n_iter > 0) {
        tmem_ld32(lane_addr + kColO + 32 * part, orow);
        wait_ld32(orow);
      }
      float x[32];                                       // slot j of every eight columns is value dim elem_of(j)
#pragma unroll
      for (int c = 0; c < 32; ++c) x[c] = zero ? 0.f : __uint_as_float(orow[(c & ~7) + slot_of(c & 7)]) * inv;
      store_rows(buf, x, to, final ? P.out : P.records, 32 * part);
    }
    if (hv == 0 && mine) {
      if (!final) *reinterpret_cast<float2*>(P.records + at + kDv) = make_float2(zero ? -INFINITY : m_ref, bad ? -1.f : zero ? 0.f : l);
      else if (P.lse) P.lse[row_index] = zero ? -INFINITY : (m_ref + log2f(l)) / kLog2e;
    }
  }

  // ---- teardown: nothing may be in flight in the tensor pipe when the columns are given back ----
  fence_before_sync();
  __syncthreads();
  if (warp == kMmaWarp) {
    if (sm.abort_flag) {
      if (elect_one()) {                                 // the lane that issued the MMAs
        commit(&sm.drain);
        for (uint32_t k = 0; k < kSpinLimit && !mbar_try_wait(&sm.drain, 0); ++k) {}
        raise_flag(P.flags, Q4KV_FLAG_INTERNAL);
      }
      __syncwarp();
    }
    fence_after_sync();
    tmem_dealloc(tb, 512);
  }
}

}  // namespace

bool prefill_mla_supported(const Layout& y) { return y.alias && y.D == kD && y.Dv == kDv && y.n_rep <= 128; }

cudaError_t launch_prefill_mla(const Layout& y, const void* pool, int n_blocks, int layer, const q4kv_batch& b,
                               const int32_t* kv_lens, const int32_t* q_offs, int total_q, int max_q_len, int max_kv_len,
                               int window, const void* q, float scale, void* out, int out_dtype, float* lse, void* ws,
                               size_t ws_bytes, int32_t* flags, cudaStream_t st) {
  if (b.n_agents <= 0 || max_q_len <= 0) return cudaSuccess;
  MlaPrefillParams P;
  P.y = y; P.pool = (const uint8_t*)pool; P.n_blocks = n_blocks; P.layer = layer; P.n_agents = b.n_agents;
  P.max_blocks = b.max_blocks; P.tables = b.block_tables; P.kv_lens = kv_lens; P.q_offs = q_offs; P.window = window;
  P.q = (const uint16_t*)q; P.scale_log2 = scale * kLog2e; P.out = out; P.out_dtype = out_dtype; P.lse = lse; P.flags = flags;
  const int tile_q = 128 / y.n_rep;
  P.n_splits = plan_prefill_splits(y, tile_q, 2, b.n_agents, total_q, max_q_len, max_kv_len, window, ws_bytes);
  P.records = (float*)ws;
  static bool configured[64][2] = {};
  const int bf = y.sb_bf16 ? 1 : 0;
  void (*kernel)(const MlaPrefillParams) = bf ? prefill_mla_kernel<true> : prefill_mla_kernel<false>;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64 || !configured[dev][bf]) {
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MlaSmem));
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) configured[dev][bf] = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * ((max_q_len + tile_q - 1) / tile_q), y.Hkv * P.n_splits, b.n_agents);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = sizeof(MlaSmem);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, kernel, P);
  if (e != cudaSuccess || P.n_splits == 1) return e;
  return launch_merge_prefill(y, total_q, P.n_splits, P.records, out, out_dtype, lse, st);
}

}  // namespace q4kv
