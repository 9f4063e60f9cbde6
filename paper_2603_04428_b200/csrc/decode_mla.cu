// q4kv_decode_attention for the MLA-latent cache (d_qk = 576 = 512 latent + 64 rope, d_v = 512, V
// aliases the first 512 dims of K, one shared KV head, up to 16 query heads): one query token per
// agent in absorbed form over the Q4 latent cache, read in place (Section 3.4 "Batched Quantized
// Inference"; the MLA cache of Section 3.6).
//
// Every key serves all 16 heads and is both key and value: its words are expanded once, used as tensor-core operands for the
// scores from the registers that expanded them, and stored once as binary16 for the value product.
//   * Work is split along the keys: CTA (split, agent) walks its share of the agent's keys 64 at a time (two 32-token chunks =
//     one bulk copy of 20736 bytes into a three-slot ring, issued three blocks ahead by one thread), leaves an (acc, m, l)
//     record per head, and a second kernel combines the records of an agent.
//   * Scores: the two warps of a pair own two key octets and half of the words each.  A lane expands a word of its key
//     (x^ = c * s + b, one binary16 fma per pair of codes, rounded once); the four pairs of elements are the B fragments of
//     two mma.sync m16n8k16 whose A operand, the queries (staged once as binary16 scaled by a power of two per head), has its
//     columns in the same order and stays in registers.  The pair's halves meet through 4 KB of shared memory.
//   * Values: the same registers are stored as one 16-byte row per (key, word), two stages deep; warp w owns dims 64w..64w+63:
//     O[16 heads][64 dims] += P V^ by 32 mma.sync, with V^ read through ldmatrix.trans and P through a 2 KB shared tile.  The
//     value product of a block is interleaved with the expansion and the scores of the next one.  (A tcgen05 version of this
//     kernel was measured at 40 us per call: with only 16 heads every tensor-memory MMA is tiny, and one whose A operand comes
//     from shared memory costs 55 to 110 clocks whatever its N.)
//   * Softmax with a lazily moved reference maximum per head, shared by the CTA: a block whose scores exceed it by more than
//     2^8 triggers an exact per-head maximum (shuffles + shared memory), a rescale of the register accumulators and the
//     probabilities anew; otherwise a block costs four exponentials per thread.  Row sums stay per-thread until the end.
// One CTA-wide barrier per block, and one per pair of warps; the raw blocks arrive on mbarriers with bounded waits
// (Q4KV_FLAG_INTERNAL when one runs out; the 256 threads then leave together).
//
// What bounds it: 2800 clocks per block, of which 2050 are the expansion with both products (the tensor instructions of a
// scheduler's two warps alone take 1150), 250 the softmax, 500 the barrier and the wait for the block; and per launch about
// 5 us of prologue, first block, record and merge.  Eight warps because the queries' fragments, the accumulators and two
// words in flight need the registers: sixteen warps of 128 registers (four per group of octets) took 22.1 us where this
// took 20.2 (4 agents x 16384 tokens with the merge; 18.3 with the present merge), two groups of four warps with separate
// chunks 20.9.  The first form, with an expanded key tile read through ldmatrix for the scores and
// three barriers per block, took 21.3 (23.8 with bfloat16 scales, now 19.9); 32 agents x 8192 tokens 110 us, now 60.
#include <algorithm>

#include "convert.cuh"
#include "q4kv_layout.cuh"
#include "quantize_core.cuh"
#include "tcgen05.cuh"

namespace q4kv {

namespace {

using namespace tc;   // mbarrier and bulk-copy wrappers

constexpr int kD = 576, kDv = 512, kHeads = 16;
constexpr int kComputeWarps = 8;
constexpr int kThreads = kComputeWarps * 32;            // 256
constexpr int kChunkBytes = 32 * (kD / 2 + 4 * (kD / 64));   // 10368: [Kc 9216 | Ksb 1152]
constexpr int kRawBytes = 2 * kChunkBytes;               // one 64-key block
constexpr int kOctetBytes = (kDv / 8) * 128;             // 8192: one key octet of the value tile
constexpr int kTileBytes = 8 * kOctetBytes;              // 65536
constexpr int kGroupStride = (kD / 8) * 128;             // 9216: bytes between 8-row groups of a [rows][576] tile
constexpr int kStages = 2, kRawSlots = 3;
constexpr float kLazy = 8.f;

using MlaParams = MlaDecodeParams;

struct MlaSmem {
  // [key octet = warp][word of 8 dims][8 keys x 16 bytes]; key k of the octet sits in slot k ^ 2 * (word % 4)
  alignas(128) uint8_t vhat[kStages][kTileBytes];
  alignas(128) uint8_t raw[kRawSlots][kRawBytes];
  alignas(128) uint8_t qtile[kHeads * kD * 2];           // [head 16][dim 576], same form
  alignas(128) uint8_t ptile[2][kHeads * 64 * 2];         // [head 16][key 64]: (h%8)*16 + (h/8)*1024 + (key/8)*128
  float kappa[kHeads];                                   // score in log2 units = S * kappa[head]
  float wmax[8][kHeads];                                 // per key octet
  float wsum[8][kHeads];
  float4 exch[kComputeWarps][32];                        // half scores on their way to the other warp of a pair
  alignas(8) uint64_t raw_full[kRawSlots];
  int bad[kRawSlots];
  int abort_flag, poisoned;
  uint32_t masks[2];
  uint32_t new_words[kD / 8], new_sb[kD / 64];           // the new token's codes and (scale, bias) pairs (update-and-fetch)
};

__device__ inline void compute_barrier() { asm volatile("bar.sync 1, 256;" ::: "memory"); }   // all eight warps
// the same, and whether the predicate holds for any of the threads
__device__ inline bool compute_any(bool p) {
  uint32_t any;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\tbar.red.or.pred p, 1, 256, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(any) : "r"((uint32_t)p) : "memory");
  return any != 0u;
}
__device__ inline uint4 lds128(uint32_t at) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(at));
  return v;
}
__device__ inline uint32_t lds32(uint32_t at) {
  uint32_t v;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(at));
  return v;
}
__device__ inline void sts128(uint32_t at, uint4 v) {
  asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(at), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ inline uint2 lds64(uint32_t at) {
  uint2 v;
  asm volatile("ld.shared.v2.b32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(at));
  return v;
}
__device__ inline void pair_barrier(int op) { asm volatile("bar.sync %0, 64;" ::"r"(2 + op) : "memory"); }
// (the two loads below carry no memory clobber: they stay between the barriers, which are volatile and do)
// four 8x8 b16 matrices; lane l supplies the address of row l % 8 of matrix l / 8; register i <- matrix i,
// thread (g, t) of the warp receiving the elements (row g, columns 2t, 2t+1)
__device__ inline void ldmatrix_x4(uint32_t (&r)[4], uint32_t smem_addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_addr));
}
// the same with every matrix transposed: thread (g, t) receives the elements (rows 2t, 2t+1, column g)
__device__ inline void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t smem_addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_addr));
}
__device__ inline void mma_f16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <bool kBf>
__global__ void __launch_bounds__(kThreads, 1) decode_mla_kernel(const __grid_constant__ MlaParams P) {
  extern __shared__ __align__(128) uint8_t smem_raw[];
  MlaSmem& sm = *reinterpret_cast<MlaSmem*>(smem_raw);

  const Layout& y = P.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int split = blockIdx.x, a = blockIdx.y;
  const int n_rep = y.Hq;                                // one KV head

  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // ---- this CTA's share of the agent's keys (inputs no kernel writes) ----
  int n = P.kv_lens[a];
  const bool bad_len = n < 0 || n > P.len_cap;       // the host's bound on every length: the key shares cover that many keys
  if (bad_len) n = 0;
  const int lo = P.window > 0 ? max(0, n - P.window) : 0;
  const int b_lo = lo >> 6, b_hi = (n + 63) >> 6;        // 64-key blocks of the attended range
  const int b0 = min(b_hi, b_lo + split * P.blocks_per_split);
  const int n_iter = min(b_hi, b0 + P.blocks_per_split) - b0;
  float* rec = P.records + ((size_t)a * P.n_splits + split) * kHeads * kDv;
  float2* rec_ml = mla_record_pairs(P.records, P.n_agents, P.n_splits) + (size_t)a * kHeads * P.n_splits + split;   // + head * n_splits
  if (n_iter <= 0) {
    // nothing to attend in this share: an empty record (the preceding kernels may still be reading the records)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (threadIdx.x < kHeads) rec_ml[threadIdx.x * P.n_splits] = make_float2(-INFINITY, 0.f);
    if (bad_len && split == 0 && threadIdx.x == 0) raise_flag(P.flags, Q4KV_FLAG_BAD_LENGTH);
    return;
  }

  if (threadIdx.x == 0) {
    for (int s = 0; s < kRawSlots; ++s) { mbar_init(&sm.raw_full[s], 1); sm.bad[s] = 0; }
    sm.abort_flag = 0; sm.poisoned = 0;
    sm.masks[0] = 0x000F000Fu; sm.masks[1] = 0x00F000F0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  __syncthreads();
  // While the preceding kernel drains, L2 is asked for the first raw blocks (block tables are inputs) and the agent's query rows (a
  // prefetch returns nothing to the kernel, so it may precede the wait, and L2 is where the preceding kernels' writes land).
  if (threadIdx.x < kRawSlots && threadIdx.x < n_iter) {
    const int c = 2 * (b0 + (int)threadIdx.x), blk = P.tables[(size_t)a * P.max_blocks + (c >> 3)];
    if (blk >= 0 && blk < P.n_blocks)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(head_block(P.pool, y, P.layer, blk, 0) + (size_t)(c & 7) * kChunkBytes),
                   "r"((uint32_t)kRawBytes) : "memory");
  }
  {
    const int lines = n_rep * kD * 2 / 128;                // 128-byte lines of the agent's n_rep query rows
    const uint16_t* qrows = P.q + (size_t)a * y.Hq * kD;
    for (int i = threadIdx.x; i < lines; i += kThreads) asm volatile("prefetch.global.L2 [%0];" ::"l"(qrows + i * 64));
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");     // the new token was appended by the preceding kernel
  volatile int* abort_flag = &sm.abort_flag;

  // Raw 64-key blocks: one bulk copy each into a three-slot ring, issued by thread 0 -- blocks 0 to 2 here, block
  // j + 3 once every warp has left block j's raw bytes (the block's CTA-wide barrier).
  auto block_of = [&](int j) { return P.tables[(size_t)a * P.max_blocks + ((2 * (b0 + j)) >> 3)]; };
  auto issue_block = [&](int j, int blk) {
    const int r = j % kRawSlots;
    const int c = 2 * (b0 + j);
    if (blk < 0 || blk >= P.n_blocks) {
      sm.bad[r] = 1;
      sm.poisoned = 1;
      raise_flag(P.flags, Q4KV_FLAG_BAD_BLOCK);
      mbar_arrive(&sm.raw_full[r]);
    } else {
      sm.bad[r] = 0;
      mbar_arrive_expect_tx(&sm.raw_full[r], kRawBytes);
      bulk_load(sm.raw[r], head_block(P.pool, y, P.layer, blk, 0) + (size_t)(c & 7) * kChunkBytes, kRawBytes, &sm.raw_full[r]);
    }
  };
  int issued = 0;                                        // thread 0: blocks whose copy has been issued
  if (threadIdx.x == 0) {
    issue_block(0, block_of(0));
    issued = min(n_iter, kRawSlots);
    for (int j = 1; j < issued; ++j) issue_block(j, block_of(j));
  }

  // Update-and-fetch: the CTA whose share ends with the agent's last block quantizes the row of position n - 1
  // (a warp per group, while the first copies are in flight; one warp for all of it was 3.4 us on this CTA's path) and, once
  // that block has landed, patches it in shared memory and stores the same words to the pool.  No other CTA reads that block.
  const bool has_new = P.k_new != nullptr && b0 + n_iter == b_hi;
  if (has_new) {
    for (int grp = warp; grp < kD / 64; grp += kComputeWarps)
      quantize_row_group(*reinterpret_cast<const uint32_t*>(P.k_new + (size_t)a * kD + 64 * grp + 2 * lane), kBf, lane, sm.new_words + 8 * grp,
                         sm.new_sb + grp);
  }

  // =============================== compute warps ================================================
  const int tq = threadIdx.x;                            // 0..255
  const int g = lane >> 2, tid = lane & 3;               // fragment coordinates
  {
    // ---- stage the queries: bf16 -> binary16 times a power of two per head, element order (0,4,1,5,2,6,3,7) ----
    const int h = tq >> 4, sub = tq & 15;                // sixteen consecutive lanes share a head; words sub, sub + 16, ...
    const bool live = h < n_rep;
    const uint16_t* qrow = P.q + ((size_t)a * y.Hq + (live ? h : 0)) * kD;
    uint4 v[5];
    float mx = 0.f;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const int w = sub + 16 * k;
      v[k] = (live && w < kD / 8) ? *reinterpret_cast<const uint4*>(qrow + 8 * w) : make_uint4(0u, 0u, 0u, 0u);
      const uint32_t u[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
#pragma unroll
      for (int e = 0; e < 4; ++e)
        mx = fmaxf(mx, fmaxf(fabsf(__uint_as_float(u[e] << 16)), fabsf(__uint_as_float(u[e] & 0xffff0000u))));
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    int ex = (int)((__float_as_uint(mx) >> 23) & 255u) - 127;
    if (mx == 0.f) ex = 0;
    ex = min(max(ex, -100), 100);
    const float sf = __uint_as_float((uint32_t)(127 + 8 - ex) << 23);        // 256 <= max |q| * sf < 512
    if (sub == 0) sm.kappa[h] = P.scale_log2 * __uint_as_float((uint32_t)(127 - 8 + ex) << 23);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const int w = sub + 16 * k;
      if (w >= kD / 8) continue;
      const uint32_t u01 = v[k].x, u23 = v[k].y, u45 = v[k].z, u67 = v[k].w;
      const float x0 = __uint_as_float(u01 << 16) * sf, x1 = __uint_as_float(u01 & 0xffff0000u) * sf;
      const float x2 = __uint_as_float(u23 << 16) * sf, x3 = __uint_as_float(u23 & 0xffff0000u) * sf;
      const float x4 = __uint_as_float(u45 << 16) * sf, x5 = __uint_as_float(u45 & 0xffff0000u) * sf;
      const float x6 = __uint_as_float(u67 << 16) * sf, x7 = __uint_as_float(u67 & 0xffff0000u) * sf;
      *reinterpret_cast<uint4*>(sm.qtile + ((h & 7) ^ (2 * (w & 3))) * 16 + (h >> 3) * kGroupStride + w * 128) =
          make_uint4(f32x2_to_h2(x0, x4), f32x2_to_h2(x1, x5), f32x2_to_h2(x2, x6), f32x2_to_h2(x3, x7));
    }
  }
  compute_barrier();                                     // queries and kappa are complete

  // Dequantize and score coordinates: the warps h = 0, 1 of pair op own the key octets 2 op and 2 op + 1 -- octet e is key
  // tile e % 4 of chunk e / 4, the tokens 4 g + e % 4.  Lane (g, tid) of warp h takes the words 4 p + tid of token g of both
  // octets for p = 8 h + i, i < 8 (two 16-byte pieces each), and of its own octet, 2 op + h, for p = 16 and 17 (an 8-byte
  // one): eighteen words, which are the score product's B fragments once they are expanded.
  const int op = warp & 3, hh = warp >> 2;               // the warps of a pair share a scheduler
  const int ci = op >> 1, tile0 = 2 * (op & 1) + hh;     // own octet; the other one is tile0 ^ 1
  const int oct = 4 * ci + tile0;
  const uint32_t raw0 = smem_u32(sm.raw[0]) + ci * kChunkBytes;
  const uint32_t rd_a = raw0 + (tile0 * 144 + hh * 64 + lane) * 16, rd_b = raw0 + ((tile0 ^ 1) * 144 + hh * 64 + lane) * 16;
  const uint32_t rd8 = raw0 + (tile0 * 576 + 512) * 4 + lane * 8;
  auto sb_row = [&](int t) { return raw0 + 9216 + (((t * 4 + (g >> 1)) * 2 + (g & 1)) * 9) * 4; };
  const uint32_t sb_a = sb_row(tile0) + 16 * hh, sb_b = sb_row(tile0 ^ 1) + 16 * hh;    // + 4 (i / 2)
  const uint32_t sb_8 = sb_row(tile0) + 32;
  const uint32_t wr = smem_u32(sm.vhat[0]) + oct * kOctetBytes + (32 * hh + tid) * 128 + (g ^ (2 * tid)) * 16;   // + 512 i
  const int wr_b = (oct & 1) ? -kOctetBytes : kOctetBytes;

  // from memory, so that the compiler does not know them: (w & mask) | magic is one instruction with one immediate
  const CodeMasks masks = {sm.masks[0], sm.masks[1]};

  // ldmatrix lane addresses (lane l: matrix l / 8, row l % 8)
  const int lm = lane >> 3, lr = lane & 7;
  const uint32_t p_lane = smem_u32(sm.ptile[0]) + lr * 16 + (lm & 1) * 1024 + (lm >> 1) * 128;        // + 256 per k-step
  // values: key octets 2 ks + lm % 2, words 8 warp + 2 cc + lm / 2; from an even to an odd cc the slot's bit 2 flips
  const uint32_t v_lane = smem_u32(sm.vhat[0]) + (lm & 1) * kOctetBytes + (8 * warp + (lm >> 1)) * 128 + (lr ^ (2 * (lm >> 1))) * 16;
  const int v_step = 256 + ((lr & 4) ? -64 : 64);

  // The queries never change: the A fragments that meet this warp's words (20 k-steps x 4 registers) live in registers for
  // the whole launch.  A k-step's 16 columns are elements 0, 4 | 1, 5 (or 2, 6 | 3, 7) of the four words 4 p + tid, so that
  // what a lane has expanded from its own word is its B fragment.
  uint32_t qa[20][4];
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    const int w = 4 * (i < 8 ? 8 * hh + i : 8 + i) + tid;                   // of heads g and g + 8
    const uint4 q0 = *reinterpret_cast<const uint4*>(sm.qtile + (g ^ (2 * tid)) * 16 + w * 128);
    const uint4 q1 = *reinterpret_cast<const uint4*>(sm.qtile + kGroupStride + (g ^ (2 * tid)) * 16 + w * 128);
    qa[2 * i][0] = q0.x; qa[2 * i][1] = q1.x; qa[2 * i][2] = q0.y; qa[2 * i][3] = q1.y;
    qa[2 * i + 1][0] = q0.z; qa[2 * i + 1][1] = q1.z; qa[2 * i + 1][2] = q0.w; qa[2 * i + 1][3] = q1.w;
  }
  const float kap[2] = {sm.kappa[g], sm.kappa[g + 8]};
  float m_ref[2] = {-INFINITY, -INFINITY}, l_part[2] = {0.f, 0.f};          // heads g and g + 8
  float o[8][4];                                         // [word 8 warp + c][head g: slots 2 tid, 2 tid + 1 | head g + 8: same]
#pragma unroll
  for (int c = 0; c < 8; ++c) { o[c][0] = 0.f; o[c][1] = 0.f; o[c][2] = 0.f; o[c][3] = 0.f; }

  // Units of the value product, u = 4 ks + cc: 16 keys (k-step ks) x 16 dims (words 2 cc, 2 cc + 1 of this warp's eight)
  auto load_values = [&](uint32_t (&bv)[4], uint32_t v_tile, int u) {
    ldmatrix_x4_trans(bv, v_tile + (u >> 2) * 2 * kOctetBytes + ((u >> 1) & 1) * 512 + ((u & 1) ? v_step : 0));
  };
  auto values = [&](int u, const uint32_t (&pa)[4], const uint32_t (&bv)[4]) {
    mma_f16(o[2 * (u & 3)], pa, bv[0], bv[1]);
    mma_f16(o[2 * (u & 3) + 1], pa, bv[2], bv[3]);
  };

  bool stopped = false;
  for (int j = 0; j < n_iter; ++j) {
    const int r = j % kRawSlots;
    int next_blk = 0;
    if (tq == 0 && j + kRawSlots < n_iter) next_blk = block_of(j + kRawSlots);
    mbar_wait(&sm.raw_full[r], (uint32_t)(j / kRawSlots), abort_flag);     // a wait that runs out raises the give-up flag
    if (has_new && j == n_iter - 1) {
      // words 0..71 and the nine (scale, bias) pairs of position n - 1, one per thread
      if (sm.bad[r] == 0 && tq < kD / 8 + kD / 64) {
        const int tau_n = (n - 1) & 31, c = 2 * (b0 + j);
        const uint32_t at = (uint32_t)(((n - 1) >> 5) & 1) * kChunkBytes +
                            (tq < kD / 8 ? y.off_kc + 4u * k_word_offset(tau_n, tq, kD / 64)
                                         : y.off_ksb + 4u * sb_offset(tau_n, tq - kD / 8, kD / 64));
        const uint32_t val = tq < kD / 8 ? sm.new_words[tq] : sm.new_sb[tq - kD / 8];
        *reinterpret_cast<uint32_t*>(sm.raw[r] + at) = val;
        const int blk = P.tables[(size_t)a * P.max_blocks + (c >> 3)];      // checked when the copy was issued
        // the caller of the update-and-fetch entry owns the pool for writing
        uint8_t* dst = const_cast<uint8_t*>(head_block(P.pool, y, P.layer, blk, 0)) + (size_t)(c & 7) * kChunkBytes + at;
        *reinterpret_cast<uint32_t*>(dst) = val;
      }
      compute_barrier();
    }
    // ---- expand this warp's share of eight keys; scores from the registers, the value part to shared memory; meanwhile the
    //      value product of the block before (its probabilities are complete since the barrier at the end of its turn) ----
    float sc[4];
    {
      const uint32_t at = r * kRawBytes, dst = wr + (j & 1) * kTileBytes;
      const uint32_t p_prev = p_lane + ((j - 1) & 1) * (kHeads * 64 * 2), v_prev = v_lane + ((j - 1) & 1) * kTileBytes;
      const int live = sm.bad[r] != 0 ? 0 : n - ((b0 + j) * 64 + ci * 32 + 4 * g);   // tokens from 4 g on; stale bytes past the end
      bool overflow = false;
      uint32_t sb[9];                                    // [own octet's four groups, the other one's, the own one's last]
      uint4 k4[2] = {lds128(rd_a + at), lds128(rd_b + at)};
#pragma unroll
      for (int i = 0; i < 4; ++i) { sb[i] = lds32(sb_a + at + 4 * i); sb[4 + i] = lds32(sb_b + at + 4 * i); }
      sb[8] = lds32(sb_8 + at);
      const uint2 k8 = lds64(rd8 + at);
      uint32_t pa[2][4], bv[2][4];
      ldmatrix_x4(pa[0], p_prev);
      load_values(bv[0], v_prev, 0);
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        if (live <= (i >= 4 && i < 8 ? tile0 ^ 1 : tile0)) sb[i] = 0u;
        if (kBf) sb[i] = bf16_pair_to_h2(sb[i], overflow);
      }
      auto expand = [&](uint32_t w, uint32_t pair) {
        return dequant8(w, __byte_perm(pair, pair, 0x1010), __byte_perm(pair, pair, 0x3232), masks);
      };
      float acc[2][4];                                   // [own octet, the other one]
#pragma unroll
      for (int i = 0; i < 2; ++i) { acc[i][0] = 0.f; acc[i][1] = 0.f; acc[i][2] = 0.f; acc[i][3] = 0.f; }
      uint4 next[2] = {};
#pragma unroll
      for (int u = 0; u < 16; ++u) {                     // one word's expansion and scores, one unit of the value product
        const int i = u >> 1, l = u & 1;
        if (u == 4) { next[0] = lds128(rd_a + at + 512); next[1] = lds128(rd_b + at + 512); }
        if (u == 8) { k4[0] = next[0]; k4[1] = next[1]; }
        if ((u & 3) == 2 && u < 14) ldmatrix_x4(pa[((u >> 2) + 1) & 1], p_prev + ((u >> 2) + 1) * 256);
        if (u < 15) load_values(bv[(u + 1) & 1], v_prev, u + 1);
        const uint4 x = expand((i & 3) == 0 ? k4[l].x : (i & 3) == 1 ? k4[l].y : (i & 3) == 2 ? k4[l].z : k4[l].w, sb[4 * l + (i >> 1)]);
        values(u, pa[(u >> 2) & 1], bv[u & 1]);
        sts128(dst + (l ? wr_b : 0) + i * 512, x);
        mma_f16(acc[l], qa[2 * i], x.x, x.y);
        mma_f16(acc[l], qa[2 * i + 1], x.z, x.w);
      }
      // the halves of the words meet: each warp takes its own octet
      sm.exch[warp ^ 4][lane] = make_float4(acc[1][0], acc[1][1], acc[1][2], acc[1][3]);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const uint4 x = expand(i ? k8.y : k8.x, sb[8]);
        mma_f16(acc[0], qa[16 + 2 * i], x.x, x.y);
        mma_f16(acc[0], qa[17 + 2 * i], x.z, x.w);
      }
      if (j == 0) {                                      // there was no block before: what was summed is no product
#pragma unroll
        for (int c = 0; c < 8; ++c) { o[c][0] = 0.f; o[c][1] = 0.f; o[c][2] = 0.f; o[c][3] = 0.f; }
      }
      if (kBf && overflow && sm.bad[r] == 0) raise_flag(P.flags, Q4KV_FLAG_SB_RANGE);
      pair_barrier(op);
      const float4 e = sm.exch[warp][lane];
      sc[0] = acc[0][0] + e.x; sc[1] = acc[0][1] + e.y; sc[2] = acc[0][2] + e.z; sc[3] = acc[0][3] + e.w;
    }
    // this thread: heads g (sc[0], sc[1]) and g + 8 (sc[2], sc[3]), keys 2 tid and 2 tid + 1 of the own octet
    const int pos = (b0 + j) * 64 + ci * 32 + 8 * tid + tile0;
    const bool v0 = pos >= lo && pos < n, v1 = pos + 4 >= lo && pos + 4 < n;
    sc[0] = v0 ? sc[0] * kap[0] : -INFINITY; sc[1] = v1 ? sc[1] * kap[0] : -INFINITY;
    sc[2] = v0 ? sc[2] * kap[1] : -INFINITY; sc[3] = v1 ? sc[3] * kap[1] : -INFINITY;
    const float mx0 = fmaxf(sc[0], sc[1]), mx1 = fmaxf(sc[2], sc[3]);
    const bool grow = mx0 > m_ref[0] + kLazy || (m_ref[0] == -INFINITY && mx0 != -INFINITY) ||
                      mx1 > m_ref[1] + kLazy || (m_ref[1] == -INFINITY && mx1 != -INFINITY);
    // ---- probabilities relative to the references so far (a head without any key yet: reference -inf and p = 0) ----
    float p[4];
    uint32_t* pt = reinterpret_cast<uint32_t*>(sm.ptile[j & 1] + g * 16 + oct * 128 + 4 * tid);
    auto probabilities = [&]() {
      p[0] = v0 ? fast_exp2(sc[0] - m_ref[0]) : 0.f; p[1] = v1 ? fast_exp2(sc[1] - m_ref[0]) : 0.f;
      p[2] = v0 ? fast_exp2(sc[2] - m_ref[1]) : 0.f; p[3] = v1 ? fast_exp2(sc[3] - m_ref[1]) : 0.f;
      pt[0] = f32x2_to_h2(p[0], p[1]);
      pt[256] = f32x2_to_h2(p[2], p[3]);
    };
    probabilities();
    // The block's only barrier: the probabilities of all 64 keys and their value tile are in place; nobody reads the raw
    // slot, or the tile and the probabilities of the block before, any more; growth (or a wait that ran out) is agreed.
    if (compute_any(grow || *abort_flag != 0)) {
      // ---- exact per-head maxima of the block, new references, rescale of what has been accumulated, probabilities anew ----
      float w0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1)), w1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1));
      w0 = fmaxf(w0, __shfl_xor_sync(0xffffffffu, w0, 2)); w1 = fmaxf(w1, __shfl_xor_sync(0xffffffffu, w1, 2));
      if (tid == 0) { sm.wmax[oct][g] = w0; sm.wmax[oct][g + 8] = w1; }
      if (compute_any(*abort_flag != 0)) { stopped = true; break; }        // all leave in the same block
      float f[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        float m_new = m_ref[e];
#pragma unroll
        for (int w = 0; w < 8; ++w) m_new = fmaxf(m_new, sm.wmax[w][g + 8 * e]);
        f[e] = m_new == -INFINITY ? 1.f : fast_exp2(m_ref[e] - m_new);     // m_ref = -inf: 0
        l_part[e] *= f[e];
        m_ref[e] = m_new;
      }
#pragma unroll
      for (int c = 0; c < 8; ++c) { o[c][0] *= f[0]; o[c][1] *= f[0]; o[c][2] *= f[1]; o[c][3] *= f[1]; }
      probabilities();
      compute_barrier();
    }
    l_part[0] += p[0] + p[1]; l_part[1] += p[2] + p[3];
    if (tq == 0 && j + kRawSlots < n_iter) { issue_block(j + kRawSlots, next_blk); issued = j + kRawSlots + 1; }
  }
  if (!stopped) {                                        // the last block's value product
    const uint32_t p_last = p_lane + ((n_iter - 1) & 1) * (kHeads * 64 * 2), v_last = v_lane + ((n_iter - 1) & 1) * kTileBytes;
    uint32_t pa[4], bv[2][4];
    load_values(bv[0], v_last, 0);
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      if ((u & 3) == 0) ldmatrix_x4(pa, p_last + (u >> 2) * 256);
      if (u < 15) load_values(bv[(u + 1) & 1], v_last, u + 1);
      values(u, pa, bv[u & 1]);
    }
  }

  // ---- this share's record: acc[16][512] (unnormalised, relative to m), m, l ----
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    float lh = l_part[e];
    lh += __shfl_xor_sync(0xffffffffu, lh, 1);
    lh += __shfl_xor_sync(0xffffffffu, lh, 2);
    if (tid == 0) sm.wsum[oct][g + 8 * e] = lh;
  }
  compute_barrier();
  const bool spoiled = stopped || sm.poisoned != 0;
  if (stopped && tq == 0) {
    // giving up: let the copies that may still be in flight land before shared memory is released
    for (int jj = max(0, issued - kRawSlots); jj < issued; ++jj)
      for (uint32_t i = 0; i < 64 && !mbar_try_wait(&sm.raw_full[jj % kRawSlots], (uint32_t)(jj / kRawSlots) & 1u); ++i) {}
    raise_flag(P.flags, Q4KV_FLAG_INTERNAL);
  }
  // Slots 2 tid and 2 tid + 1 of a word's row are its elements tid and tid + 4: even and odd lanes exchange one of the two, so
  // that an even lane stores the elements tid and tid + 1, an odd one tid + 3 and tid + 4 (whole sectors of eight floats).
  const int d_lane = 8 * 8 * warp + ((tid & 1) ? tid + 3 : tid);
#pragma unroll
  for (int c = 0; c < 8; ++c) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float got = __shfl_xor_sync(0xffffffffu, (tid & 1) ? o[c][2 * e] : o[c][2 * e + 1], 1);
      float2 v = (tid & 1) ? make_float2(got, o[c][2 * e + 1]) : make_float2(o[c][2 * e], got);
      if (spoiled) v = make_float2(0.f, 0.f);
      *reinterpret_cast<float2*>(rec + (g + 8 * e) * kDv + d_lane + 8 * c) = v;
    }
  }
  if (warp == 0 && tid == 0) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int h = g + 8 * e;
      float lsum = 0.f;
#pragma unroll
      for (int w = 0; w < kComputeWarps; ++w) lsum += sm.wsum[w][h];
      rec_ml[h * P.n_splits] = make_float2(spoiled ? -INFINITY : m_ref[e], spoiled ? -1.f : lsum);         // negative: poisoned
    }
  }
}

// grid: (16 heads, n_agents, 128 / kLanes slices of the value dims), 512 threads; combines the records of one (agent, head)
// for 4 kLanes output dims.  The records sit in L2 a microsecond away, so nothing here is a chain of dependent loads: the
// 512 / kLanes groups of threads each take every so-many-th split, with its m, while every warp fetches all (m, l) pairs for
// itself -- one round trip --, works out the maximum and the sum without the others, and the groups' sums meet in registers
// (groups of one warp) and shared memory, at the kernel's only barrier.  (With the weights agreed on by the block, behind four
// barriers, and the pairs beside the records, 32 KB apart: 4 agents x 16384 tokens 19.2 us for kernel and merge, now 18.3;
// 3 x 700 10.8, now 8.7.  Every warp for itself with the pairs beside the records: 20.0.)  How narrow the slices are depends on the count of
// splits: with four of them sixteen groups would leave most threads idle (and make four times the CTAs), with 148 each group
// would walk nine.
// The pointers carry no __restrict__: the records are written by the preceding kernel while this one is already resident, and
// read-only loads are not defined for such data.
constexpr int kMergeThreads = 512, kMaxSplits = 512;
template <int kLanes>
__global__ void __launch_bounds__(kMergeThreads) merge_mla_kernel(int Hq, int n_splits, const float* records, void* out, int out_dtype,
                                                                  float* lse) {
  constexpr int kGroups = kMergeThreads / kLanes;
  constexpr int kRows = kLanes < 32 ? kMergeThreads / 32 : kGroups;         // sums that meet in shared memory
  __shared__ float4 s_acc[kRows - 1][kLanes];
  const int h = blockIdx.x, a = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");     // the records come from the preceding kernel
  if (h >= Hq) return;
  const float* rec = records + ((size_t)a * n_splits * kHeads + h) * kDv;
  const float2* pairs = mla_record_pairs(const_cast<float*>(records), gridDim.y, n_splits) + ((size_t)a * kHeads + h) * n_splits;
  const size_t step = (size_t)kHeads * kDv;              // between the splits of one head
  // The loads of the first kGroups * kPre splits are issued before anything is known (an empty split's data is whatever an
  // earlier call left there; it is dropped below).
  constexpr int kPre = 4;
  const int grp = tid / kLanes, gl = tid % kLanes, d = 4 * (kLanes * blockIdx.z + gl);   // 4 consecutive dims per thread
  auto fetch = [&](int sp) { return *reinterpret_cast<const float4*>(rec + sp * step + d); };
  float4 pre[kPre];
  float pre_m[kPre];
#pragma unroll
  for (int u = 0; u < kPre; ++u) {
    const int sp = grp + kGroups * u;
    pre[u] = make_float4(0.f, 0.f, 0.f, 0.f);
    pre_m[u] = -INFINITY;
    if (sp < n_splits) { pre[u] = fetch(sp); pre_m[u] = pairs[sp].x; }
  }
  float M = -INFINITY, L = 0.f;
  bool bad = false;
  for (int base = 0; base < n_splits; base += 64) {      // two pairs per lane at a time
    float2 ml[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int sp = base + 32 * k + lane;
      ml[k] = sp < n_splits ? pairs[sp] : make_float2(-INFINITY, 0.f);
    }
    float m = fmaxf(ml[0].x, ml[1].x);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    m = fmaxf(m, M);
    float s = (ml[0].x == -INFINITY ? 0.f : fast_exp2(ml[0].x - m) * ml[0].y) + (ml[1].x == -INFINITY ? 0.f : fast_exp2(ml[1].x - m) * ml[1].y);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    L = (M == -INFINITY ? 0.f : L * fast_exp2(M - m)) + s;
    M = m;
    bad |= ml[0].y < 0.f || ml[1].y < 0.f;
  }
  if (__any_sync(0xffffffffu, bad)) L = 0.f;             // a poisoned split zeroes the row
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  auto add = [&](float m, const float4& v) {
    const float w = fast_exp2(m - M);
    if (!(w > 0.f)) return;                              // an empty split's record holds no data; no weight (NaN) where M is infinite
    acc.x = fmaf(w, v.x, acc.x); acc.y = fmaf(w, v.y, acc.y); acc.z = fmaf(w, v.z, acc.z); acc.w = fmaf(w, v.w, acc.w);
  };
#pragma unroll
  for (int u = 0; u < kPre; ++u) add(pre_m[u], pre[u]);
  for (int sp = grp + kGroups * kPre; sp < n_splits; sp += kGroups) add(pairs[sp].x, fetch(sp));
  if (kLanes < 32) {
#pragma unroll
    for (int o = kLanes; o < 32; o *= 2) {
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o); acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
      acc.z += __shfl_xor_sync(0xffffffffu, acc.z, o); acc.w += __shfl_xor_sync(0xffffffffu, acc.w, o);
    }
  }
  const int row = kLanes < 32 ? warp : grp;
  if (row > 0 && (kLanes >= 32 || lane < kLanes)) s_acc[row - 1][gl] = acc;
  __syncthreads();
  if (tid >= kLanes) return;
  const float inv = L > 0.f ? 1.f / L : 0.f;
#pragma unroll
  for (int g = 0; g < kRows - 1; ++g) { const float4 o = s_acc[g][gl]; acc.x += o.x; acc.y += o.y; acc.z += o.z; acc.w += o.w; }
  acc.x *= inv; acc.y *= inv; acc.z *= inv; acc.w *= inv;
  const size_t out_index = ((size_t)a * Hq + h) * kDv;
  if (out_dtype == Q4KV_OUT_BF16) {
    const __nv_bfloat162 b0 = __floats2bfloat162_rn(acc.x, acc.y), b1 = __floats2bfloat162_rn(acc.z, acc.w);
    uint2 v;
    v.x = *reinterpret_cast<const uint32_t*>(&b0);
    v.y = *reinterpret_cast<const uint32_t*>(&b1);
    *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(out) + out_index + d) = v;
  } else {
    *reinterpret_cast<float4*>(reinterpret_cast<float*>(out) + out_index + d) = acc;
  }
  if (tid == 0 && blockIdx.z == 0 && lse) lse[(size_t)a * Hq + h] = L > 0.f ? (M + log2f(L)) / kLog2e : -INFINITY;
}

struct MlaPlan { int n_splits, blocks_per_split; };
MlaPlan plan_mla(int n_agents, int max_kv_len, int window) {
  const int span = (window > 0 && window + 64 < max_kv_len) ? window + 64 : max_kv_len;
  const int blocks = (span + 63) / 64 + 1;               // a window may straddle one more 64-key block
  // One CTA per SM, in as few waves as the count of agents allows: rounding the shares of an agent up puts up to n_agents - 1
  // CTAs into a second wave, which pays only where the shares get that much shorter.  A wave costs its blocks and about
  // four more for its prologue and its record.
  const int sms = sm_count(), up = (sms + n_agents - 1) / n_agents, down = sms / n_agents;
  auto cost = [&](int n) { return ((long long)n * n_agents + sms - 1) / sms * ((blocks + n - 1) / n + 4); };
  int n_splits = down > 0 && cost(down) <= cost(up) ? down : up;
  if (n_splits > blocks) n_splits = blocks;
  if (n_splits > kMaxSplits) n_splits = kMaxSplits;
  MlaPlan p;
  p.blocks_per_split = (blocks + n_splits - 1) / n_splits;
  p.n_splits = (blocks + p.blocks_per_split - 1) / p.blocks_per_split;
  return p;
}

}  // namespace

bool decode_mla_supported(const Layout& y) {
  return y.alias && y.D == kD && y.Dv == kDv && y.Hkv == 1 && y.Hq <= kHeads;
}

size_t decode_mla_workspace_bytes(const Layout& y, int n_agents, int max_kv_len) {
  (void)y;
  // the split count depends on the window through the span: room for the most that any span gets
  const int blocks = (max_kv_len + 63) / 64 + 1, most = (sm_count() + n_agents - 1) / n_agents;
  return (size_t)n_agents * std::min(std::min(blocks, most), kMaxSplits) * kHeads * (kDv + 2) * sizeof(float);
}

cudaError_t launch_decode_mla(const Layout& y, const void* pool, int n_blocks, int layer, const q4kv_batch& b,
                              const int32_t* kv_lens, int max_kv_len, int window, const void* q, float scale, void* out,
                              int out_dtype, float* lse, void* ws, int32_t* flags, cudaStream_t st, const void* k_new,
                              bool on_codes) {
  if (b.n_agents <= 0) return cudaSuccess;
  const MlaPlan plan = plan_mla(b.n_agents, max_kv_len, window);
  MlaParams P;
  P.y = y; P.pool = (const uint8_t*)pool; P.n_blocks = n_blocks; P.layer = layer; P.n_agents = b.n_agents;
  P.max_blocks = b.max_blocks; P.tables = b.block_tables; P.kv_lens = kv_lens; P.len_cap = max_kv_len; P.window = window;
  P.q = (const uint16_t*)q; P.k_new = (const uint16_t*)k_new; P.scale_log2 = scale * kLog2e; P.n_splits = plan.n_splits;
  P.blocks_per_split = plan.blocks_per_split; P.records = (float*)ws; P.flags = flags;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaError_t e;
  if (on_codes) {
    e = launch_mla_codes_kernel(P, st);
  } else {
    static bool configured[64][2] = {};
    const size_t smem = sizeof(MlaSmem);
    const int bf = y.sb_bf16 ? 1 : 0;
    void (*kernel)(const MlaParams) = bf ? decode_mla_kernel<true> : decode_mla_kernel<false>;
    int dev = 0;
    e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !configured[dev][bf]) {
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      if (dev >= 0 && dev < 64) configured[dev][bf] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(plan.n_splits, b.n_agents);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kernel, P);
  }
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t mcfg = {};
  // 4, 8, 16 or 32 groups of threads share the splits, so that a thread's loads are few and all in flight together, but no more
  // CTAs than needed.  Measured, merge and kernel, on 128 / 64 / 32 / 16 lanes: 4 splits x 32 agents 58.9 / 61.3 / 64.0 / 74.0 us,
  // 9 x 16 19.7 / 20.7 / 22.2 / 27.2, 14 x 10 23.1 / 23.6 / 24.4 / 27.7, 18 x 8 20.5 / 19.6 / 20.7 / 23.1, 24 x 6 25.2 / 24.6 / 25.0 / 27.1,
  // 37 x 4 20.2 / 19.1 / 18.8 / 19.5, 49 x 3 18.1 / 17.4 / 16.9 / 17.5, 74 x 2 16.4 / 16.4 / 15.9 / 14.9, 148 x 1 26.1 / 23.0 / 22.0 / 20.0.
  const int lanes = plan.n_splits <= 14 ? 128 : plan.n_splits <= 30 ? 64 : plan.n_splits <= 64 ? 32 : 16;
  void (*merge)(int, int, const float*, void*, int, float*) =
      lanes == 128 ? merge_mla_kernel<128> : lanes == 64 ? merge_mla_kernel<64> : lanes == 32 ? merge_mla_kernel<32> : merge_mla_kernel<16>;
  mcfg.gridDim = dim3(kHeads, b.n_agents, kDv / 4 / lanes);
  mcfg.blockDim = dim3(kMergeThreads);
  mcfg.stream = st;
  mcfg.attrs = attr;
  mcfg.numAttrs = 1;
  return cudaLaunchKernelEx(&mcfg, merge, (int)y.Hq, plan.n_splits, (const float*)ws, out, out_dtype, lse);
}

}  // namespace q4kv
