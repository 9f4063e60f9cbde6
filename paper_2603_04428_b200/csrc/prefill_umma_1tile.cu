// q4kv_prefill_attention, tcgen05 path with one query tile per CTA, for the head shapes whose
// accumulator leaves no room for two: d_qk = d_v = 256 (the sliding-window model of Section 3.6) and
// d_qk 192 / d_v 128 (the per-head MLA cache of Section 3.6).  The
// queries of a new phase over the cached Q4 prefix plus the causal new tokens, read from the Q4
// cache in place (Sections 3.4 "chunked prefill" and 3.5 "cross-phase context injection").
//
// The d = 128 kernel's structure with one 128-row tile per CTA: at d = 256 a tile's accumulator
// alone is 256 of the 512 tensor-memory columns, and at 192 / 128 the queries of two tiles would not
// fit beside the accumulators.  What the second tile gave there -- its MMAs run while the first
// tile's softmax does -- comes here from two score buffers:
//   * A CTA owns 128 score rows (128 / n_rep consecutive queries x the n_rep heads of one KV head)
//     and walks the keys 64 at a time (two 32-token chunks, one bulk copy).
//   * Eight "dequantize" warps turn each raw block into binary16 tiles K^ [64 keys][d_qk] and
//     V^ [d_v][64 keys] in shared memory (two or three stages each), in the core-matrix order a K-major
//     tcgen05 operand wants: x^ = c * s + b in one binary16 fma per pair of codes, each value rounded
//     once to 11 significant bits.  A packed word becomes one 16-byte row of a core matrix; the order
//     of the eight elements inside a row (0,4,1,5,2,6,3,7) is absorbed by storing the queries, and
//     the key rows, in the same order.
//   * One thread issues the MMAs: S_b = Q K^T (M 128, N 64, K d_qk: d_qk / 16 instructions) into score
//     buffer b = block % 2, with Q resident in tensor memory as packed binary16 (each bf16 row scaled
//     by a power of two, so nothing is rounded), and O += P_b V^ (M 128, N d_v, K 64: 4 instructions)
//     with P_b read from tensor memory too, where it overlays S_b.  The scores of block j + 1 are
//     issued before the probabilities of block j exist, so the tensor pipe works through the softmax.
//     Tensor memory: O d_v columns, S 2 x 64, Q d_qk / 2.
//   * Eight softmax warps, two threads per score row (each takes 32 of the 64 scores and half of the accumulator columns):
//     mask, online softmax with a lazily updated reference maximum, P_b as packed binary16 over the half of S_b that the
//     thread has read.  The two warps of a row meet once per block at a barrier that carries the vote whether the reference
//     has to move; maxima are exchanged only then.
//   * One warp streams the raw blocks through a three-slot ring with bulk asynchronous copies.
// All hand-offs are mbarriers; every wait is bounded and a wait that runs out raises
// Q4KV_FLAG_INTERNAL, drains the tensor pipe and frees the tensor memory before the CTA returns.
//
// Bound by the dequantize warps' chain per block (2650 clocks per 64 keys; the two products take 1250, and with the tiles left
// as they are a block takes 2100).  With one barrier for all eight softmax warps, maxima exchanged in every block and 96
// registers for every warp (the d = 256 form spilled) it took 3400.  8 agents x (4096 + 512) tokens, 16 query heads, d = 256:
// 508 -> 382 us (575 -> 765 TFLOP/s) in a run of seconds, 363 us in one of a few launches; 192 / 128: 350 -> 282 (648), 281.
// With the output stored a line at a time (store_rows): 371 (788) and 354; 192 / 128: 275 (665) and 278.
#include "prefill_common.cuh"

namespace q4kv {

namespace {

using namespace tc;
using namespace prefill;

constexpr int kSoftmaxWarps = 8, kDequantWarps = 8;
constexpr int kMmaWarp = kSoftmaxWarps + kDequantWarps, kLoadWarp = kMmaWarp + 1;
constexpr int kThreads = (kMmaWarp + 4) * 32;            // 640: five warpgroups (the last: MMA, load, two that only bfloat16 caches need)
constexpr int kRegsSoftmax = 144, kRegsOther = 64;       // of the 96 each thread is launched with
static_assert(kSoftmaxWarps * 32 * kRegsSoftmax + (kThreads - kSoftmaxWarps * 32) * kRegsOther <= kThreads * 96, "");
constexpr int kStages = 2;                               // K^ tiles in flight
constexpr int kRawSlots = 3;                             // raw 64-key blocks in flight
constexpr uint32_t kColO = 0, kColS = 256, kColQ = 384;  // tensor-memory columns (d_v <= 256, 2 x 64, d_qk / 2 <= 128)
// G, Gv: groups of 64 along the key and value head dims
template <int G, int Gv>
struct Shape {
  static constexpr int D = 64 * G, Dv = 64 * Gv;
  static constexpr int kOffKsb = 16 * D, kOffVc = kOffKsb + 128 * G, kOffVsb = kOffVc + 16 * Dv;
  static constexpr int kChunkBytes = kOffVsb + 128 * Gv; // [Kc | Ksb | Vc | Vsb]: 9216 at 256 / 256, 5760 at 192 / 128
  static constexpr int kRawBytes = 2 * kChunkBytes;
  static constexpr int kTileK = 64 * D * 2, kTileV = Dv * 64 * 2;   // binary16 tiles
  // V^ tiles in flight.  The dequantize warps' value tile of a block waits for a value product and delays the next key tile; a
  // third stage takes that wait out at 192 / 128 (335 -> 326 us); at 256 / 256 it costs more than it gives (399 -> 408).
  static constexpr int kStagesV = G == 4 ? 2 : 3;
  static constexpr int kSboK = (D / 8) * 128;            // bytes between 8-key groups of K^
};

struct UmmaParams {
  Layout y;
  const uint8_t* pool;
  int n_blocks, layer, n_agents, max_blocks;
  const int32_t* tables;
  const int32_t* kv_lens;
  const int32_t* q_offs;
  int window;
  const uint16_t* q;          // bf16 [total_q][Hq][d_qk]
  float scale_log2;
  void* out;
  int out_dtype;
  float* lse;
  int32_t* flags;
  PrefillExtra x;
  CodeMasks masks;
};

template <int G, int Gv>
struct UmmaSmem {
  using Sh = Shape<G, Gv>;
  alignas(128) uint8_t khat[kStages][Sh::kTileK];        // [key 64][dim d_qk]: (n%8)*16 + (n/8)*kSboK + (k/8)*128
  alignas(128) uint8_t vhat[Sh::kStagesV][Sh::kTileV];   // [dim d_v][key 64]: (n%8)*16 + (n/8)*1024 + (k/8)*128
  alignas(128) uint8_t raw[kRawSlots][Sh::kRawBytes];
  alignas(8) uint64_t raw_full[kRawSlots], raw_free[kRawSlots], sb_done[kRawSlots];
  uint64_t k_full[kStages], v_full[Sh::kStagesV], k_free[kStages], v_free[Sh::kStagesV];
  uint64_t s_full[2], p_full[2], o_done, o_last, q_ready, drain;
  uint32_t tmem_base;
  int bad[kRawSlots];
  float xchg[2][2][128];                                 // [parity][column half][row]: maxima / sums of the two threads of a row
  int spoiled;
  int abort_flag, poisoned;
};

template <int G, int Gv, bool kBf>
__global__ void __launch_bounds__(kThreads, 1) prefill_umma_1tile_kernel(const __grid_constant__ UmmaParams P) {
  using Sh = Shape<G, Gv>;
  constexpr int kD = Sh::D, kDv = Sh::Dv, kChunkBytes = Sh::kChunkBytes, kRawBytes = Sh::kRawBytes;
  constexpr int kOffKsb = Sh::kOffKsb, kOffVc = Sh::kOffVc, kOffVsb = Sh::kOffVsb;
  extern __shared__ __align__(128) uint8_t smem_raw[];
  UmmaSmem<G, Gv>& sm = *reinterpret_cast<UmmaSmem<G, Gv>*>(smem_raw);

  const Layout& y = P.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int qt = blockIdx.x, hk = blockIdx.y / P.x.n_splits, split = blockIdx.y % P.x.n_splits, a = blockIdx.z;
  const int n_rep = y.n_rep;
  const int tile_q = 128 / n_rep;                        // queries of the CTA's 128-row tile

  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // ---- this CTA's queries and key range (inputs no kernel writes) ----
  const int q0 = P.q_offs[a], q_len = P.q_offs[a + 1] - q0;
  const int kv_len = P.kv_lens[a];
  const int i_min = qt * tile_q;
  if (P.x.tickets && qt == 0 && blockIdx.y == 0 && a == 0) clear_tickets(P.x);
  if (i_min >= q_len || (P.x.tickets && q_len == 1)) return;   // uniform: nothing allocated, no barrier passed
  const bool bad_len = kv_len < 0 || kv_len > P.max_blocks * kBlockTokens || q_len > kv_len;
  const int i_max = min(q_len, i_min + tile_q) - 1;
  const int prefix = kv_len - q_len;                     // query i sits at position prefix + i
  const int W = P.window;
  const int c_end = bad_len ? 0 : (prefix + i_max) / 32 + 1;
  const int c_begin = (bad_len || W == 0) ? 0 : max(0, prefix + i_min - W + 1) >> 5;
  const int all0 = c_begin >> 1, n_all = max(0, ((c_end + 1) >> 1) - all0);
  const int it0 = all0 + n_all * split / P.x.n_splits;   // 64-key blocks it0 .. it0 + n_iter - 1
  const int n_iter = all0 + n_all * (split + 1) / P.x.n_splits - it0;

  if (threadIdx.x == 0) {
    if (bad_len) raise_flag(P.flags, Q4KV_FLAG_BAD_LENGTH);
    for (int s = 0; s < kRawSlots; ++s) { mbar_init(&sm.raw_full[s], 1); mbar_init(&sm.raw_free[s], kDequantWarps); mbar_init(&sm.sb_done[s], 2); sm.bad[s] = 0; }
    for (int s = 0; s < kStages; ++s) { mbar_init(&sm.k_full[s], kDequantWarps); mbar_init(&sm.k_free[s], 1); }
    for (int s = 0; s < Sh::kStagesV; ++s) { mbar_init(&sm.v_full[s], kDequantWarps); mbar_init(&sm.v_free[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&sm.s_full[b], 1); mbar_init(&sm.p_full[b], kSoftmaxWarps * 32); }
    mbar_init(&sm.o_done, 1);
    mbar_init(&sm.o_last, 1);
    mbar_init(&sm.q_ready, kSoftmaxWarps * 32);
    sm.spoiled = 0;
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
  if (warp < kSoftmaxWarps / 2 && !bad_len) {
    const int h = (int)threadIdx.x / tile_q, i = i_min + (int)threadIdx.x % tile_q;
    if (i < q_len && h < n_rep) ask_for_row<kD>(P.q + ((size_t)(q0 + i) * y.Hq + (size_t)hk * n_rep + h) * kD);
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");     // the new tokens were appended by the preceding kernel
  volatile int* abort_flag = &sm.abort_flag;

  if (warp >= kMmaWarp) {
    fewer_registers<kRegsOther>();
    if (warp == kLoadWarp) {
      // =============================== raw block loader ==========================================
      if (lane == 0) {
        int issued = 0;
        for (int j = 0; j < n_iter; ++j) {
          const int r = j % kRawSlots;
          if (j >= kRawSlots && !mbar_wait(&sm.raw_free[r], (uint32_t)(j / kRawSlots - 1), abort_flag)) break;
          const int c = 2 * (it0 + j);
          const int blk = P.tables[(size_t)a * P.max_blocks + (c >> 3)];
          if (blk < 0 || blk >= P.n_blocks) {
            sm.bad[r] = 1;
            sm.poisoned = 1;
            raise_flag(P.flags, Q4KV_FLAG_BAD_BLOCK);
            mbar_arrive(&sm.raw_full[r]);
          } else {
            sm.bad[r] = 0;
            mbar_arrive_expect_tx(&sm.raw_full[r], kRawBytes);
            bulk_load(sm.raw[r], head_block(P.pool, y, P.layer, blk, hk) + (size_t)(c & 7) * kChunkBytes, kRawBytes,
                      &sm.raw_full[r]);
          }
          issued = j + 1;
        }
        // a CTA that is giving up still lets its own copies land before shared memory is released
        if (*abort_flag) {
          for (int j = max(0, issued - kRawSlots); j < issued; ++j) {
            const int r = j % kRawSlots;
            for (uint32_t i = 0; i < kSpinLimit && !mbar_try_wait(&sm.raw_full[r], (uint32_t)(j / kRawSlots) & 1u); ++i) {}
          }
        }
      }
    } else if (warp == kMmaWarp) {
      // =============================== MMA issue ==================================================
      // The whole warp runs this code; one elected lane (always the same) issues the MMAs and the commits.
      if (n_iter > 0) {
        constexpr uint32_t kIdescS = idesc_f16(128, 64), kIdescO = idesc_f16(128, kDv);
        // one election for a whole product: an election per MMA costs more issue time than the MMA takes
        auto issue_qk = [&](int b, int s) {                // S_b = Q K^T; afterwards the K^ stage is free
          const uint64_t kd = smem_desc(smem_u32(sm.khat[s]), 128, Sh::kSboK);
          if (elect_one()) {
  #pragma unroll
            for (int k = 0; k < kD / 16; ++k) mma_f16_ts(tb + kColS + 64 * b, tb + kColQ + 8 * k, kd + 16 * k, kIdescS, k > 0);
            commit(&sm.s_full[b]);
            commit(&sm.k_free[s]);
          }
          __syncwarp();
        };
        auto issue_pv = [&](int b, int s, bool first, bool last) {    // O (+)= P_b V^; afterwards the V^ stage is free
          const uint64_t vd = smem_desc(smem_u32(sm.vhat[s]), 128, 1024);
          if (elect_one()) {
  #pragma unroll
            for (int k = 0; k < 4; ++k)
              mma_f16_ts(tb + kColO, tb + kColS + 64 * b + 32 * (k >> 1) + 8 * (k & 1), vd + 16 * k, kIdescO, (!first || k > 0) ? 1u : 0u);
            commit(&sm.o_done);
            if (last) commit(&sm.o_last);
            commit(&sm.v_free[s]);
          }
          __syncwarp();
        };
        bool ok = mbar_wait(&sm.q_ready, 0, abort_flag) && mbar_wait(&sm.k_full[0], 0, abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (ok) {
          fence_after_sync();
          issue_qk(0, 0);
          if (n_iter > 1) {
            ok = __all_sync(0xffffffffu, mbar_wait(&sm.k_full[1], 0, abort_flag));
            if (ok) {
              fence_after_sync();
              issue_qk(1, 1);
            }
          }
        }
        for (int j = 0; ok && j < n_iter; ++j) {
          const int b = j & 1, s = j % kStages, sv = j % Sh::kStagesV;
          ok = mbar_wait(&sm.p_full[b], (uint32_t)(j >> 1), abort_flag) && mbar_wait(&sm.v_full[sv], (uint32_t)(j / Sh::kStagesV), abort_flag);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          fence_after_sync();
          issue_pv(b, sv, j == 0, j + 1 == n_iter);
          if (j + 2 < n_iter) {                            // the scores of block j + 2 replace P_b once the product above has read it
            ok = __all_sync(0xffffffffu, mbar_wait(&sm.k_full[s], (uint32_t)((j + 2) / kStages), abort_flag));
            if (!ok) break;
            fence_after_sync();
            issue_qk(b, s);
          }
        }
      }
    } else if (kBf) {
      // =============================== bfloat16 scales and biases ================================
      // They become binary16 in place (the tiles are binary16), by a warp for each chunk of a block, ahead of the dequantize warps
      // (one wait fewer in their chain: 8 x (4096 + 512) tokens 423 -> 366 us, 192 / 128 351 -> 275).  Only tokens below the agent's
      // length count for the range report (bytes past the end are whatever was there).
      const int ci = warp - (kLoadWarp + 1);
      const int tau = 8 * ((lane >> 1) & 3) + 4 * (lane & 1) + (lane >> 3);      // row (i * 4 + tid) * 2 + e: token 8 tid + 4 e + i
      for (int j = 0; j < n_iter; ++j) {
        const int r = j % kRawSlots;
        if (!mbar_wait(&sm.raw_full[r], (uint32_t)(j / kRawSlots), abort_flag)) break;
        uint32_t* k = reinterpret_cast<uint32_t*>(sm.raw[r] + ci * kChunkBytes + kOffKsb) + G * lane;
        uint32_t* v = reinterpret_cast<uint32_t*>(sm.raw[r] + ci * kChunkBytes + kOffVsb) + Gv * lane;
        bool over = false;
#pragma unroll
        for (int g = 0; g < G; ++g) k[g] = bf16_pair_to_h2(k[g], over);
#pragma unroll
        for (int g = 0; g < Gv; ++g) v[g] = bf16_pair_to_h2(v[g], over);
        if (over && !sm.bad[r] && (it0 + j) * 64 + ci * 32 + tau < kv_len) raise_flag(P.flags, Q4KV_FLAG_SB_RANGE);
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.sb_done[r]);
      }
    }
  } else if (warp >= kSoftmaxWarps) {
    fewer_registers<kRegsOther>();
    // =============================== dequantize warps ==========================================
    // 256 threads.  At 256 / 256 a thread takes one of the two 16-byte key pieces of a token row (kj) and one value
    // piece, in both chunks of the block; at 192 / 128 a token row is a 16-byte and an 8-byte key piece and there are
    // half as many value pieces, and a thread works on one chunk of the block (c1).
    const int x = threadIdx.x - kSoftmaxWarps * 32;      // 0..255
    const int x7 = x & 127, c1 = x >> 7;
    // K: token tau = 4 kg + ki of a chunk, piece kt of its lane group.  The eight lanes of a shared-memory phase read
    // eight different 16-byte columns and write eight different rows.
    const int ki = x & 3, kg = 2 * ((x >> 3) & 3) + ((x >> 2) & 1), kt = (ki + (x7 >> 5)) & 3, kj = G == 4 ? c1 : 0;
    const int ktau = 4 * kg + ki;
    const int k_read = ki * (256 * G) + kj * 512 + kg * 64 + kt * 16;       // 16-byte piece: words 16 kj + kt + 4 m, m = 0..3
    const int k_read2 = ki * (256 * G) + 512 + kg * 32 + kt * 8;            // G = 3: the 8-byte piece, words 16 + kt, 20 + kt
    const int k_tok = ((ktau & 3) * 4 + (ktau >> 3)) * 2 + ((ktau >> 2) & 1);   // the token's place among the (scale, bias) rows
    const int k_sb = kOffKsb + (k_tok * G + 2 * kj) * 4;
    const int k_row = 8 * (ktau >> 3) + slot_of(ktau & 7);       // row of the token inside its chunk's 32 rows
    // V: one 16-byte piece (dims 32 vq + 8 k + vr, k = 0..3) of token octet vo per chunk.
    const int vr = x & 7, vq = ((x >> 3) & 3) + (Gv == 4 ? 4 * c1 : 0), vo = ((vr >> 1) + (x7 >> 5)) & 3;
    const int v_read = kOffVc + ((vq * 8 + vr) * 4 + vo) * 16;
    const int v_sb = kOffVsb + (vo * 2 * Gv + (vq >> 1)) * 4;    // + (i * 8 + e) * Gv * 4: token 8 vo + 4 e + i, group vq / 2
    constexpr int kChunksPerThread = G == 4 ? 2 : 1;
    for (int j = 0; j < n_iter; ++j) {
      const int s = j % kStages, sv = j % Sh::kStagesV, r = j % kRawSlots;
      if (!mbar_wait(kBf ? &sm.sb_done[r] : &sm.raw_full[r], (uint32_t)(j / kRawSlots), abort_flag)) break;
      const bool bad = sm.bad[r] != 0;
      const int pos_base = (it0 + j) * 64;
      uint4 kws[kChunksPerThread], vws[kChunksPerThread];    // the codes, read while the stages are not yet free
#pragma unroll
      for (int cc = 0; cc < kChunksPerThread; ++cc) {
        const uint8_t* chunk = sm.raw[r] + (G == 4 ? cc : c1) * kChunkBytes;
        kws[cc] = *reinterpret_cast<const uint4*>(chunk + k_read); vws[cc] = *reinterpret_cast<const uint4*>(chunk + v_read);
      }
      if (j >= kStages && !mbar_wait(&sm.k_free[s], (uint32_t)(j / kStages - 1), abort_flag)) break;
#pragma unroll
      for (int cc = 0; cc < kChunksPerThread; ++cc) {
        const int ci = G == 4 ? cc : c1;
        const uint8_t* chunk = sm.raw[r] + ci * kChunkBytes;
        const bool dead = bad || pos_base + ci * 32 + ktau >= kv_len;      // stale bytes past the end
        const int n = ci * 32 + k_row;
        uint8_t* dst = sm.khat[s] + (n & 7) * 16 + (n >> 3) * Sh::kSboK + (16 * kj + kt) * 128;
        const uint4 kw = kws[cc];
        uint32_t e0 = *reinterpret_cast<const uint32_t*>(chunk + k_sb);       // (scale, bias) of groups 2 kj and 2 kj + 1
        uint32_t e1 = *reinterpret_cast<const uint32_t*>(chunk + k_sb + 4);
        if (dead) { e0 = 0u; e1 = 0u; }
        const uint32_t s0 = __byte_perm(e0, e0, 0x1010), b0 = __byte_perm(e0, e0, 0x3232);
        const uint32_t s1 = __byte_perm(e1, e1, 0x1010), b1 = __byte_perm(e1, e1, 0x3232);
        *reinterpret_cast<uint4*>(dst + 0 * 512) = dequant8(kw.x, s0, b0, s0, b0, s0, b0, s0, b0, P.masks);
        *reinterpret_cast<uint4*>(dst + 1 * 512) = dequant8(kw.y, s0, b0, s0, b0, s0, b0, s0, b0, P.masks);
        *reinterpret_cast<uint4*>(dst + 2 * 512) = dequant8(kw.z, s1, b1, s1, b1, s1, b1, s1, b1, P.masks);
        *reinterpret_cast<uint4*>(dst + 3 * 512) = dequant8(kw.w, s1, b1, s1, b1, s1, b1, s1, b1, P.masks);
        if (G == 3) {
          const uint2 kw2 = *reinterpret_cast<const uint2*>(chunk + k_read2);
          uint32_t e2 = *reinterpret_cast<const uint32_t*>(chunk + k_sb + 8);  // group 2
          if (dead) e2 = 0u;
          const uint32_t s2 = __byte_perm(e2, e2, 0x1010), b2 = __byte_perm(e2, e2, 0x3232);
          *reinterpret_cast<uint4*>(dst + 4 * 512) = dequant8(kw2.x, s2, b2, s2, b2, s2, b2, s2, b2, P.masks);
          *reinterpret_cast<uint4*>(dst + 5 * 512) = dequant8(kw2.y, s2, b2, s2, b2, s2, b2, s2, b2, P.masks);
        }
      }
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.k_full[s]);
      if (j >= Sh::kStagesV && !mbar_wait(&sm.v_free[sv], (uint32_t)(j / Sh::kStagesV - 1), abort_flag)) break;
#pragma unroll
      for (int cc = 0; cc < kChunksPerThread; ++cc) {
        const int ci = G == 4 ? cc : c1;
        const uint8_t* chunk = sm.raw[r] + ci * kChunkBytes;
        const uint4 vw = vws[cc];
        uint32_t sp[4], bp[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          uint32_t e0 = *reinterpret_cast<const uint32_t*>(chunk + v_sb + i * 32 * Gv);
          uint32_t e1 = *reinterpret_cast<const uint32_t*>(chunk + v_sb + i * 32 * Gv + 4 * Gv);
          const int pos = pos_base + ci * 32 + 8 * vo + i;
          if (bad || pos >= kv_len) e0 = 0u;
          if (bad || pos + 4 >= kv_len) e1 = 0u;
          sp[i] = __byte_perm(e0, e1, 0x5410);                             // scales of tokens i and i + 4
          bp[i] = __byte_perm(e0, e1, 0x7632);                             // biases
        }
        uint8_t* dst = sm.vhat[sv] + vr * 16 + (4 * vq) * 1024 + (ci * 4 + vo) * 128;
        *reinterpret_cast<uint4*>(dst + 0 * 1024) = dequant8(vw.x, sp[0], bp[0], sp[1], bp[1], sp[2], bp[2], sp[3], bp[3], P.masks);
        *reinterpret_cast<uint4*>(dst + 1 * 1024) = dequant8(vw.y, sp[0], bp[0], sp[1], bp[1], sp[2], bp[2], sp[3], bp[3], P.masks);
        *reinterpret_cast<uint4*>(dst + 2 * 1024) = dequant8(vw.z, sp[0], bp[0], sp[1], bp[1], sp[2], bp[2], sp[3], bp[3], P.masks);
        *reinterpret_cast<uint4*>(dst + 3 * 1024) = dequant8(vw.w, sp[0], bp[0], sp[1], bp[1], sp[2], bp[2], sp[3], bp[3], P.masks);
      }
      fence_async_smem();
      __syncwarp();
      if (lane == 0) { mbar_arrive(&sm.v_full[sv]); mbar_arrive(&sm.raw_free[r]); }
    }
  } else {
    more_registers<kRegsSoftmax>();
    // =============================== softmax warps: two threads per score row ===================
    // Warp w: column half = w / 4, tensor-memory lanes 32 (w % 4) ...  The warps w and w + 4 share their rows: they meet at a
    // named barrier once per block, which tells both whether a row's maximum has outgrown its reference (or a wait has run
    // out: they leave the loop together); only then are maxima exchanged through shared memory, and at the end the sums.
    const int half = (warp >> 2) & 1;
    const int row = (warp & 3) * 32 + lane;              // tensor-memory lane
    const uint32_t lane_addr = tb + ((uint32_t)((warp & 3) * 32) << 16);
    const int h = row / tile_q, i = i_min + row % tile_q;
    const bool mine = i < q_len && h < n_rep;            // (128 need not be a multiple of n_rep: the last rows are idle)
    const bool valid = mine && !bad_len;
    const int pq = prefix + i;                           // this row's position
    auto tile_barrier = [&]() { asm volatile("bar.sync 1, 256;" ::: "memory"); };
    auto pair_any = [&](bool p) {                        // of the 64 threads of the rows' two warps
      uint32_t any;
      asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\tbar.red.or.pred p, %2, 64, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                   : "=r"(any) : "r"((uint32_t)p), "r"(2 + (warp & 3)) : "memory");
      return any != 0u;
    };
    float kappa;                                         // score in log2 units = S * kappa
    {
      // ---- stage this thread's half of the query row: bf16 -> binary16 times a power of two, element order
      //      (0,4,1,5,2,6,3,7) inside every eight ----
      constexpr int kQWords = kD / 4;                    // packed binary16 words of this thread's half row: 64 or 48
      const uint16_t* qrow = P.q + ((size_t)(q0 + (valid ? i : 0)) * y.Hq + (size_t)hk * n_rep + h) * kD + (kD / 2) * half;
      uint32_t qa[kQWords];
      float mx = 0.f;
      if (valid) {
#pragma unroll
        for (int w = 0; w < kQWords / 4; ++w) {
          const uint4 v = *reinterpret_cast<const uint4*>(qrow + 8 * w);
          qa[4 * w] = v.x; qa[4 * w + 1] = v.y; qa[4 * w + 2] = v.z; qa[4 * w + 3] = v.w;
          mx = fmaxf(mx, fmaxf(fmaxf(fabsf(__uint_as_float(v.x << 16)), fabsf(__uint_as_float(v.x & 0xffff0000u))),
                               fmaxf(fabsf(__uint_as_float(v.y << 16)), fabsf(__uint_as_float(v.y & 0xffff0000u)))));
          mx = fmaxf(mx, fmaxf(fmaxf(fabsf(__uint_as_float(v.z << 16)), fabsf(__uint_as_float(v.z & 0xffff0000u))),
                               fmaxf(fabsf(__uint_as_float(v.w << 16)), fabsf(__uint_as_float(v.w & 0xffff0000u)))));
        }
      } else {
#pragma unroll
        for (int w = 0; w < kQWords; ++w) qa[w] = 0u;
      }
      sm.xchg[1][half][row] = mx;                        // slot 1: block 0 of the loop below writes slot 0
      tile_barrier();
      mx = fmaxf(mx, sm.xchg[1][half ^ 1][row]);
      int ex = (int)((__float_as_uint(mx) >> 23) & 255u) - 127;
      if (mx == 0.f) ex = 0;
      ex = min(max(ex, -100), 100);
      const float sf = __uint_as_float((uint32_t)(127 + 8 - ex) << 23);      // 256 <= max |q| * sf < 512
      kappa = P.scale_log2 * __uint_as_float((uint32_t)(127 - 8 + ex) << 23);
#pragma unroll
      for (int w = 0; w < kQWords / 4; ++w) {
        // elements 8w..8w+7 arrive as bf16 pairs (0,1) (2,3) (4,5) (6,7); columns hold (0,4) (1,5) (2,6) (3,7)
        const uint32_t u01 = qa[4 * w], u23 = qa[4 * w + 1], u45 = qa[4 * w + 2], u67 = qa[4 * w + 3];
        const float x0 = __uint_as_float(u01 << 16) * sf, x1 = __uint_as_float(u01 & 0xffff0000u) * sf;
        const float x2 = __uint_as_float(u23 << 16) * sf, x3 = __uint_as_float(u23 & 0xffff0000u) * sf;
        const float x4 = __uint_as_float(u45 << 16) * sf, x5 = __uint_as_float(u45 & 0xffff0000u) * sf;
        const float x6 = __uint_as_float(u67 << 16) * sf, x7 = __uint_as_float(u67 & 0xffff0000u) * sf;
        qa[4 * w] = f32x2_to_h2(x0, x4); qa[4 * w + 1] = f32x2_to_h2(x1, x5);
        qa[4 * w + 2] = f32x2_to_h2(x2, x6); qa[4 * w + 3] = f32x2_to_h2(x3, x7);
      }
      // 32-column stores start at multiples of 32 columns, 16-column stores at multiples of 16
      if (kQWords == 64) {
        tmem_st32(lane_addr + kColQ + 64 * half, qa);
        tmem_st32(lane_addr + kColQ + 64 * half + 32, qa + 32);
      } else if (half == 0) {
        tmem_st32(lane_addr + kColQ, qa);
        tmem_st16(lane_addr + kColQ + 32, qa + 32);
      } else {
        tmem_st16(lane_addr + kColQ + 48, qa);
        tmem_st32(lane_addr + kColQ + 64, qa + 16);
      }
      wait_st();
      fence_before_sync();
      mbar_arrive(&sm.q_ready);
    }
    float m_ref = -INFINITY, l = 0.f;                    // p = 2^(s - m_ref); m_ref trails the true maximum by at most kLazy
    for (int j = 0; j < n_iter; ++j) {
      const int b = j & 1;
      const bool quit = !mbar_wait(&sm.s_full[b], (uint32_t)(j >> 1), abort_flag);   // raises the give-up flag; both warps leave below
      fence_after_sync();
      uint32_t sr[32];
      tmem_ld32(lane_addr + kColS + 64 * b + 32 * half, sr);
      wait_ld32(sr);
      const int pos0 = (it0 + j) * 64 + 32 * half;
      // column c of this half is key pos0 + (c & ~7) + elem_of(c & 7); causal and window masks on edge blocks only
      if (pos0 + 31 > pq || (W > 0 && pos0 <= pq - W)) {
#pragma unroll
        for (int c = 0; c < 32; ++c) {
          const int pos = pos0 + (c & ~7) + elem_of(c & 7);
          if (pos > pq || (W > 0 && pos <= pq - W)) sr[c] = 0xff800000u;   // -inf
        }
      }
      // Probabilities against the current reference, and the block maximum beside them (independent instruction
      // streams); only when some row's maximum has outgrown its reference is the reference moved, the accumulator
      // rescaled and the probabilities taken again.  The scores stay in registers meanwhile.
      float sum = 0.f;
      uint32_t pr[16];
      const uint64_t kk = pair64(kappa, kappa);
      auto probabilities = [&](float neg_m) {
        const uint64_t nn = pair64(neg_m, neg_m);
        uint64_t sum0 = 0u, sum1 = 0u;                   // (+0, +0)
#pragma unroll
        for (int c = 0; c < 16; c += 2) {
          const float2 u = unpair64(fma2(pair64(__uint_as_float(sr[2 * c]), __uint_as_float(sr[2 * c + 1])), kk, nn));
          const float2 v = unpair64(fma2(pair64(__uint_as_float(sr[2 * c + 2]), __uint_as_float(sr[2 * c + 3])), kk, nn));
          const float p0 = fast_exp2(u.x), p1 = fast_exp2(u.y), p2 = fast_exp2(v.x), p3 = fast_exp2(v.y);
          sum0 = add2(sum0, pair64(p0, p1)); sum1 = add2(sum1, pair64(p2, p3));
          pr[c] = f32x2_to_h2(p0, p1);
          pr[c + 1] = f32x2_to_h2(p2, p3);
        }
        const float2 s01 = unpair64(sum0), s23 = unpair64(sum1);
        sum = (s01.x + s01.y) + (s23.x + s23.y);
      };
      probabilities(m_ref == -INFINITY ? 0.f : -m_ref);
      float cm4[4] = {__uint_as_float(sr[0]), __uint_as_float(sr[1]), __uint_as_float(sr[2]), __uint_as_float(sr[3])};
#pragma unroll
      for (int c = 4; c < 32; ++c) cm4[c & 3] = fmaxf(cm4[c & 3], __uint_as_float(sr[c]));
      float cm = fmaxf(fmaxf(cm4[0], cm4[1]), fmaxf(cm4[2], cm4[3]));
      // P_b overlays the half of S_b that this thread has read: 16 columns from column 32 half on
      tmem_st16(lane_addr + kColS + 64 * b + 32 * half, pr);
      const float cs = cm == -INFINITY ? cm : cm * kappa;                  // kappa > 0
      if (pair_any(quit || cs > m_ref + kLazy || (m_ref == -INFINITY && cs != -INFINITY))) {
        sm.xchg[j & 1][half][row] = cs;
        if (pair_any(quit)) break;
        const float m_new = fmaxf(m_ref, fmaxf(cs, sm.xchg[j & 1][half ^ 1][row]));
        const bool grow = m_new > m_ref + kLazy || (m_ref == -INFINITY && m_new != -INFINITY);
        if (j > 0) {
          // rescale this thread's half of the accumulator row: the previous block's value product must have landed
          mbar_wait(&sm.o_done, (uint32_t)(j - 1), abort_flag);
          fence_after_sync();
          const float f = grow ? fast_exp2(m_ref - m_new) : 1.f;           // m_ref = -inf: 0
#pragma unroll 1
          for (int part = 0; part < kDv / 64; ++part) {
            uint32_t orow[32];
            tmem_ld32(lane_addr + kColO + (kDv / 2) * half + 32 * part, orow);
            wait_ld32(orow);
#pragma unroll
            for (int c = 0; c < 32; ++c) orow[c] = __float_as_uint(__uint_as_float(orow[c]) * f);
            tmem_st32(lane_addr + kColO + (kDv / 2) * half + 32 * part, orow);
          }
          if (grow) l *= f;
        }
        if (grow) m_ref = m_new;
        probabilities(m_ref == -INFINITY ? 0.f : -m_ref);
        wait_st();
        tmem_st16(lane_addr + kColS + 64 * b + 32 * half, pr);
      }
      l += sum;
      wait_st();
      fence_before_sync();
      mbar_arrive(&sm.p_full[b]);
    }
    // ---- normalise and write this thread's half of the row ----
    bool ok = !*abort_flag;
    // (the last two value products may both be under way, and a wait on o_done could not tell which phase it sees)
    if (ok && n_iter > 0) ok = mbar_wait(&sm.o_last, 0, abort_flag);
    const int slot = n_iter & 1;                         // not the slot the last block used
    sm.xchg[slot][half][row] = l;
    if (!ok) sm.spoiled = 1;                             // anyone who gave up spoils the tile
    tile_barrier();
    ok = sm.spoiled == 0;                                // uniform over the tile: the loads below are warp-wide
    l += sm.xchg[slot][half ^ 1][row];
    if (ok) fence_after_sync();
    const bool bad = !ok || sm.poisoned != 0;
    const bool zero = bad || n_iter == 0 || l <= 0.f;
    const bool final = P.x.n_splits == 1;                // else the row is left as a record
    const float inv = zero ? 0.f : final ? 1.f / l : 1.f;
    const size_t row_index = (size_t)(q0 + i) * y.Hq + (size_t)hk * n_rep + h;
    const size_t at = final ? row_index * kDv : (row_index * P.x.n_splits + split) * prefill_record(kDv);
    uint8_t* const buf = &sm.khat[0][0] + warp * kRowsBytes;   // the products with the keys are done
    const RowsOut to = rows_out(at + (kDv / 2) * half, mine, final && P.out_dtype == Q4KV_OUT_BF16);
#pragma unroll 1
    for (int part = 0; part < kDv / 64; ++part) {
      uint32_t orow[32];
      if (ok && n_iter > 0) {
        tmem_ld32(lane_addr + kColO + (kDv / 2) * half + 32 * part, orow);
        wait_ld32(orow);
      }
      float x[32];
#pragma unroll
      for (int c = 0; c < 32; ++c) x[c] = zero ? 0.f : __uint_as_float(orow[c]) * inv;
      store_rows(buf, x, to, final ? P.out : P.x.records, 32 * part);
    }
    if (half == 0 && mine) {
      if (!final) *reinterpret_cast<float2*>(P.x.records + at + kDv) = make_float2(zero ? -INFINITY : m_ref, bad ? -1.f : zero ? 0.f : l);
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

bool prefill_umma_1tile_supported(const Layout& y) {
  const bool shape = (y.D == 256 && y.Dv == 256) || (y.D == 192 && y.Dv == 128);
  return !y.alias && shape && y.n_rep <= 128;
}

namespace {
template <int G, int Gv, bool kBf>
cudaError_t launch_shape(const UmmaParams& P, int max_q_len, cudaStream_t st) {
  static bool configured[64] = {};
  const size_t smem = sizeof(UmmaSmem<G, Gv>);
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    e = cudaFuncSetAttribute(prefill_umma_1tile_kernel<G, Gv, kBf>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  const int cta_q = 128 / P.y.n_rep;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((max_q_len + cta_q - 1) / cta_q, P.y.Hkv * P.x.n_splits, P.n_agents);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, prefill_umma_1tile_kernel<G, Gv, kBf>, P);
}
}  // namespace

cudaError_t launch_prefill_umma_1tile(const Layout& y, const void* pool, int n_blocks, int layer, const q4kv_batch& b,
                                      const int32_t* kv_lens, const int32_t* q_offs, int max_q_len, int window,
                                      const void* q, float scale, void* out, int out_dtype, float* lse, int32_t* flags,
                                      cudaStream_t st, const PrefillExtra& x) {
  if (b.n_agents <= 0 || max_q_len <= 0) return cudaSuccess;
  UmmaParams P;
  P.y = y; P.pool = (const uint8_t*)pool; P.n_blocks = n_blocks; P.layer = layer; P.n_agents = b.n_agents;
  P.max_blocks = b.max_blocks; P.tables = b.block_tables; P.kv_lens = kv_lens; P.q_offs = q_offs; P.window = window;
  P.q = (const uint16_t*)q; P.scale_log2 = scale * kLog2e; P.out = out; P.out_dtype = out_dtype; P.lse = lse; P.flags = flags;
  P.x = x;
  if (y.D == 256) return y.sb_bf16 ? launch_shape<4, 4, true>(P, max_q_len, st) : launch_shape<4, 4, false>(P, max_q_len, st);
  return y.sb_bf16 ? launch_shape<3, 2, true>(P, max_q_len, st) : launch_shape<3, 2, false>(P, max_q_len, st);
}

}  // namespace q4kv
