// q4kv_prefill_attention, tcgen05 path (d_qk = d_v = 128): the
// queries of a new phase over the cached Q4 prefix plus the causal new tokens, read from the Q4
// cache in place (Sections 3.4 "chunked prefill" and 3.5 "cross-phase context injection"; GQA and
// sliding windows: Section 3.6).
//
// Prefill is a dense contraction, so it runs on the fifth-generation tensor cores, and the 4-bit
// cache is expanded exactly once per CTA and key block, not once per query row:
//   * A CTA owns 256 score rows = two tiles of 128 rows (128 / n_rep consecutive queries x the n_rep heads of one KV head)
//     and walks the keys 128 at a time.  Per such step the tensor pipe is needed for 2100 clocks, the exponential unit for
//     2050, shared memory for 2300 (operands 1570, tiles written 510, raw blocks 150) and the issue slots for 1700, so what
//     matters is that all of them work at once: few, long hand-offs.  (Steps of 64 keys with the queries in tensor memory and
//     two threads per row, which exchanged their maxima, took 2 x 3000 clocks.)  Measured on 8 agents x (8192 + 1024 tokens),
//     32 / 8 heads: 4150 clocks per step; 1112 us per launch = 1051 TFLOP/s in a run of a few launches, 1240 us = 943 TFLOP/s in a
//     run of seconds, under the power cap (1156 and 1298 us before the lanes shared the rows' lines at both ends of a tile).
//     Before that, 5000 clocks, 1240 and 1357 us: the issuing warp was the bottleneck, with eight
//     waits a step of which each cost 140 to 350 clocks although its phase was over; it has five now (see there), and a reference
//     that moves by the sum of the probabilities instead of their maximum takes 70 of 230 instructions per 64 keys out of the
//     softmax.  What is left is the chain of a tile's step: scores 250 clocks after their product, exponentials 2 x 1100, value
//     and score products 1200.  Measured without gain: four softmax warps per row pair (16 in all), score buffers of 64 keys
//     issued two blocks ahead, an issuing warp per tile (the tiles fall into step: 1399 us), scores fetched ahead (1196 for
//     1188), the maximum before the exponentials (1351), 1/16, 1/8 or 1/4 of the exponentials as a polynomial on the FMA pipe
//     (1169, 1182, 1222 for 1168), the issuing warp's group first in the CTA (1188 for 1169).
//   * Eight "dequantize" warps turn each raw 64-key block into binary16 tiles K^ [64 keys][128 dims] and V^ [128 dims][64
//     keys] in shared memory (four of each), in the core-matrix order a K-major tcgen05 operand wants: x^ = c * s + b in one
//     binary16 fma per pair of codes (the code is made a binary16 integer by or-ing the masked nibble into the mantissa of
//     1024 or 64 and subtracting), i.e. each value is rounded once, to 11 significant bits.  A packed word becomes one 16-byte
//     row of a core matrix; the order of the eight elements inside a row (0,4,1,5,2,6,3,7) is absorbed by storing the queries,
//     and the key rows, in the same order.
//   * One thread issues the MMAs: S_t = Q_t K^T (M 128, N 128, K 128) with Q_t in shared memory as binary16 (each bf16 query
//     row scaled by a power of two, so nothing is rounded), and O_t += P_t V^ (M 128, N 128, K 128) with P_t read from tensor
//     memory.  The f32 accumulators fill the tensor memory (O 2 x 128, S 2 x 128); P_t overlays S_t.  At
//     N = 128 a product whose A operand is in shared memory runs at the full rate (66 clocks per instruction).
//   * Eight softmax warps, one thread per score row (a tensor-memory lane): mask, online softmax with a lazily updated
//     reference (see kSumLimit), P_t as packed binary16, in halves of 64 keys, so that the first half's value product runs
//     under the second half's exponentials.  The two tiles alternate, so one tile's softmax overlaps the other tile's MMAs.
//   * One warp streams the raw blocks through a small ring with bulk asynchronous copies.
// All hand-offs are mbarriers; every wait is bounded and a wait that runs out raises
// Q4KV_FLAG_INTERNAL, drains the tensor pipe and frees the tensor memory before the CTA returns.
#include "prefill_common.cuh"

namespace q4kv {

namespace {

using namespace tc;
using namespace prefill;

constexpr int kSoftmaxWarps = 8, kDequantWarps = 8;
constexpr int kLastGroup = kSoftmaxWarps + kDequantWarps, kLoadWarp = kLastGroup, kMmaWarp = kLastGroup + 3;
constexpr int kThreads = (kLastGroup + 4) * 32;            // 640: five warpgroups (the last: MMA, load, two that only bfloat16 caches need), ...
// ... launched with 96 registers per thread; the softmax warpgroups take 144, the others keep 64 (61440 in all)
constexpr int kRegsSoftmax = 144, kRegsOther = 64;
static_assert(kSoftmaxWarps * 32 * kRegsSoftmax + (kThreads - kSoftmaxWarps * 32) * kRegsOther <= kThreads * 96, "");
constexpr int kStages = 4;                               // K^ / V^ tiles of 64 keys in flight: two steps
constexpr int kRawSlots = 3;                             // raw 64-key blocks in flight
constexpr int kChunkBytes = 4608;                        // d = 128: [Kc 2048 | Ksb 256 | Vc 2048 | Vsb 256]
constexpr int kRawBytes = 2 * kChunkBytes;
constexpr int kTileBytes = 64 * 128 * 2;                 // one binary16 tile
// The reference of a row's exponentials moves when its probabilities of 64 keys add up to more than this (they are positive, so
// none is above it, far below binary16's 65504).  The sum is needed anyway, a maximum beside it was 64 comparisons of a warp's
// 230 instructions: 1233 -> 1188 us on the launch named above.
constexpr float kSumLimit = 4096.f;
constexpr uint32_t kColO = 0, kColS = 256;               // tensor-memory columns (+128 t; P inside S)

struct UmmaParams {
  Layout y;
  const uint8_t* pool;
  int n_blocks, layer, n_agents, max_blocks;
  const int32_t* tables;
  const int32_t* kv_lens;
  const int32_t* q_offs;
  int window;
  const uint16_t* q;          // bf16 [total_q][Hq][128]
  float scale_log2;
  void* out;
  int out_dtype;
  float* lse;
  int32_t* flags;
  PrefillExtra x;
  CodeMasks masks;
};

struct UmmaSmem {
  alignas(128) uint8_t qs[2][128 * 128 * 2];             // [row][dim]: (m%8)*16 + (m/8)*2048 + (k/8)*128
  alignas(128) uint8_t khat[kStages][kTileBytes];        // [key 64][dim 128]: (n%8)*16 + (n/8)*2048 + (k/8)*128
  alignas(128) uint8_t vhat[kStages][kTileBytes];        // [dim 128][key 64]: (n%8)*16 + (n/8)*1024 + (k/8)*128
  alignas(128) uint8_t raw[kRawSlots][kRawBytes];
  alignas(8) uint64_t raw_full[kRawSlots], raw_free[kRawSlots], sb_done[kRawSlots];
  uint64_t k_full[kStages], v_full[kStages], k_free[kStages / 2], v_free[kStages / 2];   // free: a step's two tiles
  uint64_t s_full[2], p_full[2][2], o_half[2], o_done[2], q_ready, drain;    // p_full: [tile][half of the step]
  uint32_t tmem_base;
  int bad[kRawSlots];
  int abort_flag, poisoned;
};

template <bool kBf>
__global__ void __launch_bounds__(kThreads, 1) prefill_umma_kernel(const __grid_constant__ UmmaParams P) {
  extern __shared__ __align__(128) uint8_t smem_raw[];
  UmmaSmem& sm = *reinterpret_cast<UmmaSmem*>(smem_raw);

  const Layout& y = P.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int qt = blockIdx.x, hk = blockIdx.y / P.x.n_splits, split = blockIdx.y % P.x.n_splits, a = blockIdx.z;
  const int n_rep = y.n_rep;
  const int tile_q = 128 / n_rep;                        // queries per 128-row tile

  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // ---- this CTA's queries and key range (inputs no kernel writes) ----
  const int q0 = P.q_offs[a], q_len = P.q_offs[a + 1] - q0;
  const int kv_len = P.kv_lens[a];
  const int i_min = qt * 2 * tile_q;
  if (P.x.tickets && qt == 0 && blockIdx.y == 0 && a == 0) clear_tickets(P.x);
  if (i_min >= q_len || (P.x.tickets && q_len == 1)) return;   // uniform: nothing allocated, no barrier passed
  const bool bad_len = kv_len < 0 || kv_len > P.max_blocks * kBlockTokens || q_len > kv_len;
  const int i_max = min(q_len, i_min + 2 * tile_q) - 1;
  const int prefix = kv_len - q_len;                     // query i sits at position prefix + i
  const int W = P.window;
  const int c_end = bad_len ? 0 : (prefix + i_max) / 32 + 1;
  const int c_begin = (bad_len || W == 0) ? 0 : max(0, prefix + i_min - W + 1) >> 5;
  // steps of 128 keys (the last one may reach past the end, inside its pool block: zeros)
  const int all0 = c_begin >> 2, n_all = max(0, ((c_end + 3) >> 2) - all0);
  const int st0 = all0 + n_all * split / P.x.n_splits;   // steps st0 .. st0 + n_step - 1
  const int n_step = all0 + n_all * (split + 1) / P.x.n_splits - st0;
  const int it0 = 2 * st0, n_iter = 2 * n_step;          // 64-key blocks

  if (threadIdx.x == 0) {
    if (bad_len) raise_flag(P.flags, Q4KV_FLAG_BAD_LENGTH);
    for (int s = 0; s < kRawSlots; ++s) { mbar_init(&sm.raw_full[s], 1); mbar_init(&sm.raw_free[s], kDequantWarps); mbar_init(&sm.sb_done[s], 2); sm.bad[s] = 0; }
    for (int s = 0; s < kStages; ++s) { mbar_init(&sm.k_full[s], kDequantWarps); mbar_init(&sm.v_full[s], kDequantWarps); }
    for (int s = 0; s < kStages / 2; ++s) { mbar_init(&sm.k_free[s], 1); mbar_init(&sm.v_free[s], 1); }
    for (int t = 0; t < 2; ++t) {
      mbar_init(&sm.s_full[t], 1); mbar_init(&sm.o_half[t], 1); mbar_init(&sm.o_done[t], 1);
      mbar_init(&sm.p_full[t][0], 4); mbar_init(&sm.p_full[t][1], 4);
    }
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
  asm volatile("griddepcontrol.wait;" ::: "memory");     // the new tokens were appended by the preceding kernel
  volatile int* abort_flag = &sm.abort_flag;

  if (warp >= kLastGroup) {
    fewer_registers<kRegsOther>();
    if (warp == kLoadWarp) {
    // =============================== raw block loader ==========================================
    if (lane == 0) {
      int issued = 0;
      for (int j = 0; j < n_iter; ++j) {
        const int r = j % kRawSlots;
        if (j >= kRawSlots && !mbar_doze(&sm.raw_free[r], (uint32_t)(j / kRawSlots - 1), abort_flag)) break;
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
    if (n_step > 0) {
      constexpr uint32_t kIdesc = idesc_f16(128, 128);
      const uint64_t qd0 = smem_desc(smem_u32(sm.qs[0]), 128, 2048), kd0 = smem_desc(smem_u32(sm.khat[0]), 128, 2048);
      const uint64_t vd0 = smem_desc(smem_u32(sm.vhat[0]), 128, 1024);
      // one election for a whole product: an election per MMA costs more issue time than the MMA takes
      auto issue_qk = [&](int t, int s) {                // S_t = Q_t K^T over the tiles 2 s, 2 s + 1
        const uint64_t qd = qd0 + (uint64_t)(t * (sizeof(sm.qs[0]) >> 4)), kd = kd0 + (uint64_t)(s * (2 * kTileBytes >> 4));
        if (elect_one()) {
#pragma unroll                                           // rolled, every MMA waits for its own operand arithmetic: 2x slower
          for (int k = 0; k < 8; ++k) mma_f16_ss(tb + kColS + 128 * t, qd + 16 * k, kd + 16 * k, kIdesc, k > 0);
          commit(&sm.s_full[t]);
          if (t == 1) commit(&sm.k_free[s]);             // both tiles' products have been issued
        }
        __syncwarp();
      };
      auto issue_pv = [&](int t, int s, int half, bool first) {    // O_t (+)= P_t V^ over half of the step's keys
        const uint64_t vd = vd0 + (uint64_t)((2 * s + half) * (kTileBytes >> 4));
        if (elect_one()) {
#pragma unroll
          for (int k = 0; k < 4; ++k)
            mma_f16_ts(tb + kColO + 128 * t, tb + kColS + 128 * t + 64 * half + 8 * k, vd + 16 * k, kIdesc, (!first || k > 0) ? 1u : 0u);
          commit(half == 0 ? &sm.o_half[t] : &sm.o_done[t]);
          if (t == 1 && half == 1) commit(&sm.v_free[s]);
        }
        __syncwarp();
      };
      auto wait = [&](uint64_t* bar, int use) {
        const bool ok = mbar_spin(bar, (uint32_t)use, abort_flag);
        if (ok) fence_after_sync();
        return ok;
      };
      // A wait costs 150 to 300 clocks here even when its phase is over, and the tensor pipe idles meanwhile, so as few as can be:
      // a dequantize warp arrives for its tiles in the order K0 V0 K1 V1 of a step's two blocks, so the second key tile of a step
      // implies the first value tile of the step and everything of the step before it.
      auto keys_of = [&](int j) { return wait(&sm.k_full[2 * (j & 1) + 1], j >> 1); };
      bool ok = wait(&sm.q_ready, 0) && keys_of(0);
      if (ok) {
        issue_qk(0, 0);
        issue_qk(1, 0);
      }
      for (int j = 0; ok && j < n_step; ++j) {
        const int s = j & 1;
#pragma unroll 1
        for (int t = 0; t < 2; ++t) {
          ok = wait(&sm.p_full[t][0], j);
          if (!ok) break;
          issue_pv(t, s, 0, j == 0);
          if (t == 0) ok = j + 1 < n_step ? keys_of(j + 1) : wait(&sm.v_full[2 * s + 1], j >> 1);
          ok = ok && wait(&sm.p_full[t][1], j);
          if (!ok) break;
          issue_pv(t, s, 1, false);
          if (j + 1 < n_step) issue_qk(t, s ^ 1);
        }
      }
    }
    } else if (kBf) {
    // =============================== bfloat16 scales and biases ==================================
    // They become binary16 in place (the tiles are binary16), by a warp for each chunk of a block, ahead of the dequantize warps (which
    // did it themselves, behind a barrier of their own, one more wait in their chain: 1350 us on 8 x (8192 + 1024) tokens, 1227 this way).
    // Only tokens below the agent's length count for the range report (bytes past the end are whatever was there).
    const int ci = warp - (kLoadWarp + 1);
    const int tau = 8 * ((lane >> 1) & 3) + 4 * (lane & 1) + (lane >> 3);        // row (i * 4 + tid) * 2 + e: token 8 tid + 4 e + i
    for (int j = 0; j < n_iter; ++j) {
      const int r = j % kRawSlots;
      if (!mbar_wait(&sm.raw_full[r], (uint32_t)(j / kRawSlots), abort_flag)) break;
      uint2* at = reinterpret_cast<uint2*>(sm.raw[r] + ci * kChunkBytes + 2048) + lane;      // both groups of the row's token: Ksb, Vsb
      uint2 k = at[0], v = at[(4352 - 2048) / 8];
      bool over = false;
      k.x = bf16_pair_to_h2(k.x, over); k.y = bf16_pair_to_h2(k.y, over);
      v.x = bf16_pair_to_h2(v.x, over); v.y = bf16_pair_to_h2(v.y, over);
      at[0] = k;
      at[(4352 - 2048) / 8] = v;
      if (over && !sm.bad[r] && (it0 + j) * 64 + ci * 32 + tau < kv_len) raise_flag(P.flags, Q4KV_FLAG_SB_RANGE);
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.sb_done[r]);
    }
    }
  } else if (warp >= kSoftmaxWarps) {
    fewer_registers<kRegsOther>();
    // =============================== dequantize warps ==========================================
    const int x = threadIdx.x - kSoftmaxWarps * 32, ci = x >> 7, x7 = x & 127;     // ci: the thread's chunk of the block
    // K: one 16-byte piece (words w = 4j + kt, j = 0..3) of token tau = 4 kg + ki.  The eight lanes
    // of a shared-memory phase read eight different 16-byte columns and write eight different rows.
    const int ki = x & 3, kg = 2 * ((x >> 3) & 3) + ((x >> 2) & 1), kt = (ki + (x7 >> 5)) & 3;
    const int ktau = 4 * kg + ki;
    const int k_read = ci * kChunkBytes + (ki * 32 + kg * 4 + kt) * 16;
    const int k_sb = ci * kChunkBytes + 2048 + (((ktau & 3) * 4 + (ktau >> 3)) * 2 + ((ktau >> 2) & 1)) * 8;
    const int k_row = ci * 32 + 8 * (ktau >> 3) + slot_of(ktau & 7);      // row of the token in the tile
    const int k_write = (k_row & 7) * 16 + (k_row >> 3) * 2048 + kt * 128;
    // V: one 16-byte piece (dims 32 vq + 8 k + vr, k = 0..3) of token octet vo.
    const int vr = x & 7, vq = (x >> 3) & 3, vo = ((vr >> 1) + (x7 >> 5)) & 3;
    const int v_read = ci * kChunkBytes + 2304 + ((vq * 8 + vr) * 4 + vo) * 16;
    const int v_sb = ci * kChunkBytes + 4352 + (vo * 2 * 2 + (vq >> 1)) * 4;        // + i * 64 + e * 8: token 8 vo + 4 e + i, group vq / 2
    const int v_write = vr * 16 + (4 * vq) * 1024 + (ci * 4 + vo) * 128;
    for (int j = 0; j < n_iter; ++j) {
      const int s = j % kStages, r = j % kRawSlots;
      if (j >= kStages && !mbar_doze(&sm.k_free[s >> 1], (uint32_t)(j / kStages - 1), abort_flag)) break;
      if (!mbar_doze(kBf ? &sm.sb_done[r] : &sm.raw_full[r], (uint32_t)(j / kRawSlots), abort_flag)) break;
      const bool bad = sm.bad[r] != 0;
      const int pos_base = (it0 + j) * 64 + ci * 32;
      const uint8_t* raw = sm.raw[r];
      {
        const uint4 kw = *reinterpret_cast<const uint4*>(raw + k_read);
        uint2 sb = *reinterpret_cast<const uint2*>(raw + k_sb);            // (scale, bias) of groups 0 and 1
        if (bad || pos_base + ktau >= kv_len) sb = make_uint2(0u, 0u);     // stale bytes past the end
        const uint32_t s0 = __byte_perm(sb.x, sb.x, 0x1010), b0 = __byte_perm(sb.x, sb.x, 0x3232);
        const uint32_t s1 = __byte_perm(sb.y, sb.y, 0x1010), b1 = __byte_perm(sb.y, sb.y, 0x3232);
        uint8_t* dst = sm.khat[s] + k_write;
        *reinterpret_cast<uint4*>(dst + 0 * 512) = dequant8(kw.x, s0, b0, s0, b0, s0, b0, s0, b0, P.masks);
        *reinterpret_cast<uint4*>(dst + 1 * 512) = dequant8(kw.y, s0, b0, s0, b0, s0, b0, s0, b0, P.masks);
        *reinterpret_cast<uint4*>(dst + 2 * 512) = dequant8(kw.z, s1, b1, s1, b1, s1, b1, s1, b1, P.masks);
        *reinterpret_cast<uint4*>(dst + 3 * 512) = dequant8(kw.w, s1, b1, s1, b1, s1, b1, s1, b1, P.masks);
      }
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.k_full[s]);
      if (j >= kStages && !mbar_doze(&sm.v_free[s >> 1], (uint32_t)(j / kStages - 1), abort_flag)) break;
      {
        const uint4 vw = *reinterpret_cast<const uint4*>(raw + v_read);
        uint32_t sp[4], bp[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          uint32_t e0 = *reinterpret_cast<const uint32_t*>(raw + v_sb + i * 64);
          uint32_t e1 = *reinterpret_cast<const uint32_t*>(raw + v_sb + i * 64 + 8);
          const int pos = pos_base + 8 * vo + i;
          if (bad || pos >= kv_len) e0 = 0u;
          if (bad || pos + 4 >= kv_len) e1 = 0u;
          sp[i] = __byte_perm(e0, e1, 0x5410);                             // scales of tokens i and i + 4
          bp[i] = __byte_perm(e0, e1, 0x7632);                             // biases
        }
        uint8_t* dst = sm.vhat[s] + v_write;
        *reinterpret_cast<uint4*>(dst + 0 * 1024) = dequant8(vw.x, sp[0], bp[0], sp[1], bp[1], sp[2], bp[2], sp[3], bp[3], P.masks);
        *reinterpret_cast<uint4*>(dst + 1 * 1024) = dequant8(vw.y, sp[0], bp[0], sp[1], bp[1], sp[2], bp[2], sp[3], bp[3], P.masks);
        *reinterpret_cast<uint4*>(dst + 2 * 1024) = dequant8(vw.z, sp[0], bp[0], sp[1], bp[1], sp[2], bp[2], sp[3], bp[3], P.masks);
        *reinterpret_cast<uint4*>(dst + 3 * 1024) = dequant8(vw.w, sp[0], bp[0], sp[1], bp[1], sp[2], bp[2], sp[3], bp[3], P.masks);
      }
      fence_async_smem();
      __syncwarp();
      if (lane == 0) { mbar_arrive(&sm.v_full[s]); mbar_arrive(&sm.raw_free[r]); }
    }
  } else {
    more_registers<kRegsSoftmax>();
    // =============================== softmax warps: one thread per score row ===================
    const int t = warp >> 2;
    const int row = (warp & 3) * 32 + lane;              // tensor-memory lane
    const uint32_t lane_addr = tb + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t s_addr = lane_addr + kColS + 128 * t, o_addr = lane_addr + kColO + 128 * t;
    float kappa = 0.f;                                   // score in log2 units = S * kappa
    {
      // ---- stage the warp's query rows: bf16 -> binary16 times a power of two per row.  Lane l takes the pieces l / 8, + 4, + 8, + 12 of
      //      row 8 g + l % 8 (see load_rows; the rows go to shared memory here, so nothing has to change hands) ----
      const RowsIn in = rows_in(P.q, (warp & 3) * 32, tile_q, i_min + t * tile_q, q0, q_len, y.Hq, hk * n_rep, n_rep, 128, bad_len);
      uint4 v[16];                                       // [piece / 4][g]
      load_rows<16>(in, v);
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        const int r = (warp & 3) * 32 + 8 * g + (lane & 7);
        float mx = fmaxf(fmaxf(max_abs8(v[g]), max_abs8(v[4 + g])), fmaxf(max_abs8(v[8 + g]), max_abs8(v[12 + g])));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
        int ex = (int)((__float_as_uint(mx) >> 23) & 255u) - 127;
        if (mx == 0.f) ex = 0;
        ex = min(max(ex, -100), 100);
        const float sf = __uint_as_float((uint32_t)(127 + 8 - ex) << 23);      // 256 <= max |q| * sf < 512
        if ((lane >> 3) == g) kappa = P.scale_log2 * __uint_as_float((uint32_t)(127 - 8 + ex) << 23);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          *reinterpret_cast<uint4*>(sm.qs[t] + (r & 7) * 16 + (r >> 3) * 2048 + (4 * k + (lane >> 3)) * 128) = query8(v[4 * k + g], sf);
      }
      fence_async_smem();
      mbar_arrive(&sm.q_ready);
    }
    const int h = row / tile_q, i = i_min + t * tile_q + row % tile_q;
    const bool mine = i < q_len && h < n_rep;            // (128 need not be a multiple of n_rep: the last rows are idle)
    const int pq = prefix + i;                           // this row's position
    const size_t row_index = (size_t)(q0 + i) * y.Hq + (size_t)hk * n_rep + h;
    float m_ref = -INFINITY, l = 0.f;                    // p = 2^(s - m_ref); m_ref trails the true maximum by at most 2^12
    for (int j = 0; j < n_step; ++j) {
      // one warp of the tile polls and the others sleep at a barrier: polling takes issue slots from the other tile's warps
      // (6 % of the kernel's time, like the sleeping waits of the dequantize warps)
      if ((warp & 3) == 1 + t) mbar_spin(&sm.s_full[t], (uint32_t)j, abort_flag);
      asm volatile("bar.sync %0, 128;" ::"r"(1 + t) : "memory");
      fence_after_sync();
      const int pos0 = (st0 + j) * 128;
      const bool edge = pos0 + 127 > pq || (W > 0 && pos0 <= pq - W);
      // column c of x is key pos0 + c0 + (c & ~7) + elem_of(c & 7); causal and window masks on edge steps only
      auto mask = [&](uint32_t* x, int c0) {
        const int last = pq - (pos0 + c0), first = W > 0 ? last - W + 1 : -1000;     // columns [first, last] count
#pragma unroll
        for (int c = 0; c < 32; ++c) {
          const int k = (c & ~7) + elem_of(c & 7);
          if (k > last || k < first) x[c] = 0xff800000u;   // -inf
        }
      };
      auto maximum = [&](const uint32_t* x) {
        float m0 = __uint_as_float(x[0]), m1 = __uint_as_float(x[1]);
#pragma unroll
        for (int c = 2; c < 30; c += 4) {
          m0 = fmaxf(m0, fmaxf(__uint_as_float(x[c]), __uint_as_float(x[c + 1])));
          m1 = fmaxf(m1, fmaxf(__uint_as_float(x[c + 2]), __uint_as_float(x[c + 3])));
        }
        return fmaxf(fmaxf(m0, __uint_as_float(x[30])), fmaxf(m1, __uint_as_float(x[31])));
      };
#pragma unroll 1
      for (int half = 0; half < 2; ++half) {             // 64 keys at a time: the first half's value product starts meanwhile
        const uint32_t half_addr = s_addr + 64 * half;
        const uint64_t kk = pair64(kappa, kappa);
        float neg_m = m_ref == -INFINITY ? 0.f : -m_ref;
        uint64_t nn = pair64(neg_m, neg_m);
        uint32_t pr[32];
        uint64_t sum0 = 0ull, sum1 = 0ull;
        auto probabilities = [&](const uint32_t* x, uint32_t* p) {
#pragma unroll
          for (int c = 0; c < 16; c += 2) {
            const float2 a = unpair64(fma2(pair64(__uint_as_float(x[2 * c]), __uint_as_float(x[2 * c + 1])), kk, nn));
            const float2 b = unpair64(fma2(pair64(__uint_as_float(x[2 * c + 2]), __uint_as_float(x[2 * c + 3])), kk, nn));
            const float a0 = fast_exp2(a.x), a1 = fast_exp2(a.y), b0 = fast_exp2(b.x), b1 = fast_exp2(b.y);
            sum0 = add2(sum0, pair64(a0, a1));
            sum1 = add2(sum1, pair64(b0, b1));
            p[c] = f32x2_to_h2(a0, a1);
            p[c + 1] = f32x2_to_h2(b0, b1);
          }
        };
        // P overlays the half's first 32 columns of S, each part stored as soon as it is there (1168 -> 1156 us); the scores stay
        // in registers until the half is final
        uint32_t xa[32], xb[32];
        tmem_ld32(half_addr, xa);
        wait_ld32(xa);
        tmem_ld32(half_addr + 32, xb);
        if (edge) mask(xa, 64 * half);
        probabilities(xa, pr);
        wait_ld32(xb);
        tmem_st16(half_addr, pr);
        if (edge) mask(xb, 64 * half + 32);
        probabilities(xb, pr + 16);
        tmem_st16(half_addr + 16, pr + 16);
        float2 u = unpair64(add2(sum0, sum1));
        float s_half = u.x + u.y;
        const bool outgrown = !(s_half <= kSumLimit) || m_ref == -INFINITY;
        if (__any_sync(0xffffffffu, outgrown)) {         // rare: a row's reference may have to move
          float cm = fmaxf(maximum(xa), maximum(xb));
          if (cm != -INFINITY) cm *= kappa;              // kappa > 0
          const float m_new = fmaxf(m_ref, cm);
          const bool grow = outgrown && m_new > m_ref;
          // (no row's moves where the rows without a reference have no key here either: a window's or a part's first steps)
          if (__any_sync(0xffffffffu, grow)) {
            if (j + half > 0) {
              // rescale the accumulator row once the value products issued so far have landed (those of earlier steps have:
              // the scores were issued behind them)
              if (half == 1 && !__all_sync(0xffffffffu, mbar_wait(&sm.o_half[t], (uint32_t)j, abort_flag))) break;
              fence_after_sync();
              const float f = grow ? fast_exp2(m_ref - m_new) : 1.f;       // m_ref = -inf: 0
#pragma unroll 1
              for (int part = 0; part < 8; ++part) {
                uint32_t orow[16];
                tmem_ld16(o_addr + 16 * part, orow);
                wait_ld16(orow);
#pragma unroll
                for (int c = 0; c < 16; ++c) orow[c] = __float_as_uint(__uint_as_float(orow[c]) * f);
                tmem_st16(o_addr + 16 * part, orow);
              }
              if (grow) l *= f;
            }
            if (grow) m_ref = m_new;
            neg_m = m_ref == -INFINITY ? 0.f : -m_ref;
            nn = pair64(neg_m, neg_m);
            sum0 = sum1 = 0ull;
            probabilities(xa, pr);
            probabilities(xb, pr + 16);
            wait_st();                                   // the stores above go to the same columns, and only this orders two stores
            tmem_st32(half_addr, pr);
            u = unpair64(add2(sum0, sum1));
            s_half = u.x + u.y;
          }
        }
        l += s_half;
        wait_st();
        fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.p_full[t][half]);
      }
    }
    // ---- normalise and write the row, or leave it as a record ----
    bool ok = !*abort_flag;
    if (ok && n_step > 0) ok = mbar_wait(&sm.o_done[t], (uint32_t)(n_step - 1), abort_flag);
    ok = __all_sync(0xffffffffu, ok);                    // the loads below are warp-wide
    if (ok) fence_after_sync();
    const bool bad = !ok || sm.poisoned != 0;
    const bool zero = bad || n_step == 0 || l <= 0.f;
    const bool final = P.x.n_splits == 1;                // else the row is left as a record
    const float inv = zero ? 0.f : final ? 1.f / l : 1.f;
    // the warp's own query rows, which no product needs any more (another warp's may still be on their way here where the CTA has no keys)
    uint8_t* const buf = sm.qs[t] + (warp & 3) * 4 * 2048;
    static_assert(kRowsBytes <= 4 * 2048, "");
    const size_t at = final ? row_index * 128 : (row_index * P.x.n_splits + split) * prefill_record(128);
    const RowsOut to = rows_out(at, mine, final && P.out_dtype == Q4KV_OUT_BF16);
#pragma unroll 1
    for (int part = 0; part < 4; ++part) {
      uint32_t orow[32];
      if (ok && n_step > 0) {
        tmem_ld32(o_addr + 32 * part, orow);
        wait_ld32(orow);
      }
      float x[32];
#pragma unroll
      for (int c = 0; c < 32; ++c) x[c] = zero ? 0.f : __uint_as_float(orow[c]) * inv;
      store_rows(buf, x, to, final ? P.out : P.x.records, 32 * part);
    }
    if (mine) {
      if (!final) *reinterpret_cast<float2*>(P.x.records + at + 128) = make_float2(zero ? -INFINITY : m_ref, bad ? -1.f : zero ? 0.f : l);
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

bool prefill_umma_supported(const Layout& y) {
  return !y.alias && y.D == 128 && y.Dv == 128 && y.n_rep <= 128;
}

cudaError_t launch_prefill_umma(const Layout& y, const void* pool, int n_blocks, int layer, const q4kv_batch& b,
                                const int32_t* kv_lens, const int32_t* q_offs, int max_q_len, int window, const void* q,
                                float scale, void* out, int out_dtype, float* lse, int32_t* flags, cudaStream_t st,
                                const PrefillExtra& x) {
  if (b.n_agents <= 0 || max_q_len <= 0) return cudaSuccess;
  UmmaParams P;
  P.y = y; P.pool = (const uint8_t*)pool; P.n_blocks = n_blocks; P.layer = layer; P.n_agents = b.n_agents;
  P.max_blocks = b.max_blocks; P.tables = b.block_tables; P.kv_lens = kv_lens; P.q_offs = q_offs; P.window = window;
  P.q = (const uint16_t*)q; P.scale_log2 = scale * kLog2e; P.out = out; P.out_dtype = out_dtype; P.lse = lse; P.flags = flags;
  P.x = x;
  static bool configured[64][2] = {};
  const size_t smem = sizeof(UmmaSmem);
  const int bf = y.sb_bf16 ? 1 : 0;
  void (*kernel)(const UmmaParams) = bf ? prefill_umma_kernel<true> : prefill_umma_kernel<false>;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64 || !configured[dev][bf]) {
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) configured[dev][bf] = true;
  }
  const int cta_q = 2 * (128 / y.n_rep);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((max_q_len + cta_q - 1) / cta_q, y.Hkv * x.n_splits, b.n_agents);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P);
}

}  // namespace q4kv
