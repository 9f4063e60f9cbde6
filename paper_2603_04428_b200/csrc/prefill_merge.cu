// Launches of the tcgen05 prefill kernels that cut the keys of a query tile over several CTAs: how many parts, and the
// combination of the (acc, m, l) records they leave.
#include "prefill_common.cuh"

namespace q4kv {

namespace {

using namespace prefill;

// One warp per (query row, head); with q_offs, the rows of agents with a single query are the decode kernel's and are left
// alone (no part of theirs was written).  Weights of the parts, then the weighted sum, 128 output elements at a time.  Bound by
// the latency of the records in L2; the parts of a row are in flight together.
__global__ void __launch_bounds__(128)
merge_prefill_kernel(int rows, int Hq, int Dv, int n_splits, const float* records, void* out, int out_dtype, float* lse,
                     const int32_t* __restrict__ q_offs, int n_agents) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int lane = threadIdx.x & 31;
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  bool single = false;
  if (q_offs)
    for (int a = lane; a < n_agents; a += 32) single |= q_offs[a] == row / Hq && q_offs[a + 1] == row / Hq + 1;
  single = __any_sync(0xffffffffu, single);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (row >= rows || single) return;
  const int stride = prefill_record(Dv);
  const float* rec = records + (size_t)row * n_splits * stride;
  const float2 ml = lane < n_splits ? __ldcg(reinterpret_cast<const float2*>(rec + (size_t)lane * stride + Dv)) : make_float2(-INFINITY, 0.f);
  float M = ml.x;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
  const float e = ml.x == -INFINITY ? 0.f : fast_exp2(ml.x - M);
  float L = e * ml.y;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
  if (__any_sync(0xffffffffu, ml.y < 0.f)) L = 0.f;
  const float inv = L > 0.f ? 1.f / L : 0.f;
  for (int d = 4 * lane; d < Dv; d += 128) {
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int s = 0; s < n_splits; ++s) {
      const float w = __shfl_sync(0xffffffffu, e, s);
      const float4 v = __ldcg(reinterpret_cast<const float4*>(rec + (size_t)s * stride + d));
      if (w != 0.f) { a.x = fmaf(w, v.x, a.x); a.y = fmaf(w, v.y, a.y); a.z = fmaf(w, v.z, a.z); a.w = fmaf(w, v.w, a.w); }
    }
    if (out_dtype == Q4KV_OUT_BF16) {
      const __nv_bfloat162 lo = __floats2bfloat162_rn(a.x * inv, a.y * inv), hi = __floats2bfloat162_rn(a.z * inv, a.w * inv);
      *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(out) + (size_t)row * Dv + d) =
          make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
    } else {
      *reinterpret_cast<float4*>(reinterpret_cast<float*>(out) + (size_t)row * Dv + d) = make_float4(a.x * inv, a.y * inv, a.z * inv, a.w * inv);
    }
  }
  if (lane == 0 && lse) lse[row] = L > 0.f ? (M + log2f(L)) / kLog2e : -INFINITY;
}

}  // namespace

// Parts the keys of every query tile are cut into.  tile_q: queries per CTA tile; per_tile: CTAs that share a tile.  The
// number of CTAs is estimated (lengths are on the device) from the rows and agents that the launch takes; with singles, the
// agents with one query are not its own: of n_agents agents with total_q queries and at most max_q_len each, at least
// (total_q - n_agents) / (max_q_len - 1) bring more than one, and every other agent takes one row away.  A launch
// of c CTAs in s parts takes about ceil(c s / SMs) / s of a whole tile's time plus a fixed cost per part (start-up and
// records: about four 64-key blocks), so few tiles on long contexts are cut, many tiles or short contexts are not.
// (Eight layers of two chunks of 512 beside ten single queries, 32 / 8 heads, up to 6000 keys, a workspace with room: 1255 us with
// the single queries counted in -- three parts, 52 MB of records and a merge launch a layer -- and 815 as one wave of whole tiles.)
int plan_prefill_splits(const Layout& y, int tile_q, int per_tile, int n_agents, int total_q, int max_q_len, int max_kv_len,
                        int window, size_t ws_bytes, bool singles) {
  const long long sms = sm_count();
  const int full = singles ? max(1, (total_q - n_agents + max_q_len - 2) / (max_q_len - 1))
                           : (total_q + max_q_len - 1) / max_q_len;          // agents it takes at least
  const int rows = singles ? max(full, total_q - (n_agents - full)) : total_q;
  const long long ctas = ((long long)rows / tile_q + full) * y.Hkv * per_tile;
  const int span = window > 0 && window + tile_q < max_kv_len ? window + tile_q : max_kv_len;
  const double blocks = (span + 63) / 64;
  int best = 1;
  double best_time = (double)((ctas + sms - 1) / sms) * (blocks + 4.0);
  for (int s = 2; s <= kMaxPrefillSplits && s * 4 <= blocks; ++s) {
    if (prefill_record_bytes(y, total_q, s) > ws_bytes) break;
    const double t = (double)((ctas * s + sms - 1) / sms) * (blocks / s + 4.0) + 4.0;
    if (t < 0.95 * best_time) { best = s; best_time = t; }
  }
  return best;
}

cudaError_t launch_merge_prefill(const Layout& y, int total_q, int n_splits, const float* records, void* out, int out_dtype,
                                 float* lse, cudaStream_t st, const int32_t* q_offs, int n_agents) {
  cudaLaunchConfig_t cfg = {};
  const int rows = total_q * y.Hq;
  cfg.gridDim = dim3((rows + 3) / 4);
  cfg.blockDim = dim3(128);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, merge_prefill_kernel, rows, y.Hq, y.Dv, n_splits, records, out, out_dtype, lse, q_offs, n_agents);
}

}  // namespace q4kv
