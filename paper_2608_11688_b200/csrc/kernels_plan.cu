// ffn_plan_kernel: the execution sets of a batched step (B > 1), the (expert, token) pair list sorted by expert for the
// tensor-core grouped GEMM, and the rest of that kernel's preparation.
#include <cooperative_groups.h>

#include "apex_internal.hpp"
#include "ptx.cuh"
#include "token_plan.cuh"

namespace cg = cooperative_groups;

namespace apex {

// Clusters of ceil(B / 32) CTAs (at most 8) of 32 warps.  The first cluster plans.  Phase A: a warp per token (planning
// a token costs a warp 2-3 us of dependent latency, so eight tokens per warp on one SM were 16 us at B = 256); its
// execution mask and gates go into the leader CTA's shared memory through distributed shared memory.  Phase B, leader
// CTA only: warp w owns experts w and w+32 and gathers the tokens that execute them with ballots, so the pair list is
// sorted by (expert, token).  Shared-expert pairs (expert id N) follow.
// The other clusters zero y and round h' to bf16 (the rows the GEMM gathers by token), so no kernel of its own does that.
// Nothing here waits for the host link: the sets the host needs leave from the GEMM kernel (a system-scope fence at
// this kernel's end was 2 us on the path of everything behind it).
constexpr int kPlanMaxCtas = APEX_MAX_BATCH / 32;
static_assert(kPlanMaxCtas <= 8, "one token per warp needs a cluster of at most 8 CTAs");

__global__ void __launch_bounds__(1024) ffn_plan_kernel(const FfnParams p) {
  cg::cluster_group cluster = cg::this_cluster();
  const unsigned crank = cluster.block_rank();
  __shared__ unsigned long long s_exec[APEX_MAX_BATCH], s_kr[APEX_MAX_BATCH];
  __shared__ float s_pgate[APEX_MAX_BATCH][APEX_MAX_TOPK];  // gate of the j-th executed expert of each token
  __shared__ float s_sgate[APEX_MAX_BATCH];                 // weight of the shared expert for each token (gated variant)
  __shared__ int s_count[APEX_MAX_EXPERTS + 1];
  __shared__ int s_off[APEX_MAX_EXPERTS + 2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
  const int N = p.N, k = p.k, B = p.B;
  SPAN_BEGIN();
  pdl_wait();               // the gate's outputs are complete, and nobody reads the previous step's plan any more
  pdl_launch_dependents();
  if (blockIdx.x >= cluster.num_blocks()) {  // helpers
    const size_t n8 = (size_t)B * p.d / 8, stride = (size_t)(gridDim.x - cluster.num_blocks()) * blockDim.x;
    float4* y4 = reinterpret_cast<float4*>(p.y);
    const float4* h4 = reinterpret_cast<const float4*>(p.hpost);
    auto pack = [](float a, float b) {
      const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
      return *reinterpret_cast<const uint32_t*>(&v);
    };
    for (size_t i = (size_t)(blockIdx.x - cluster.num_blocks()) * blockDim.x + threadIdx.x; i < n8; i += stride) {
      const float4 a = __ldg(h4 + 2 * i), b = __ldg(h4 + 2 * i + 1);
      // in the order in which the GEMM's converters leave the weights (kernels_ffn_tc.cu)
      uint4 o;
      if (p.fmt == 2) o = make_uint4(pack(a.x, b.x), pack(a.y, b.y), pack(a.z, b.z), pack(a.w, b.w));
      else if (p.fmt == 1) o = make_uint4(pack(a.x, a.z), pack(a.y, a.w), pack(b.x, b.z), pack(b.y, b.w));
      else o = make_uint4(pack(a.x, a.y), pack(a.z, a.w), pack(b.x, b.y), pack(b.z, b.w));
      reinterpret_cast<uint4*>(p.xb)[i] = o;
      if (!p.accumulate) y4[2 * i] = y4[2 * i + 1] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    return;
  }
  // the leader's copies of the per-token results
  unsigned long long* l_exec = cluster.map_shared_rank(&s_exec[0], 0);
  unsigned long long* l_kr = cluster.map_shared_rank(&s_kr[0], 0);
  float* l_pgate = cluster.map_shared_rank(&s_pgate[0][0], 0);
  float* l_sgate = cluster.map_shared_rank(&s_sgate[0], 0);
  if (crank == 0)
    for (int i = threadIdx.x; i < kTcSyncWords; i += (int)blockDim.x) p.tc_sync[i] = 0u;
  const int b = (int)crank * nwarp + warp;
  if (b < B) {
    const TokenLoads tl = load_token(p.idx + (size_t)b * k, p.z_r + (size_t)b * N, p.alpha + (size_t)b * N, N, k, p.mode, lane);
    const TokenPlan tp = plan_token(tl, p.mode, p.norm_topk, p.snap.resident_mask, lane);
    if (lane == 0) {
      l_exec[b] = tp.exec_mask;
      l_kr[b] = tp.kr_mask;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int e = lane + 32 * h;
      if ((tp.exec_mask >> e) & 1) {
        const int pos = __popcll(tp.exec_mask & ((1ull << e) - 1ull));
        const float g = h ? tp.g1 : tp.g0;
        if (pos < APEX_MAX_TOPK) l_pgate[b * APEX_MAX_TOPK + pos] = g;
        if (p.post_exec && p.exec_idx) p.exec_idx[(size_t)b * k + pos] = e;
        if (p.post_exec && p.exec_gate) p.exec_gate[(size_t)b * k + pos] = g;
      }
    }
    if (p.run_shared && p.shared_gate) {
      const float sg = shared_gate_weight(p.shared_gate, p.hpost + (size_t)b * p.d, p.d, lane);
      if (lane == 0) l_sgate[b] = sg;
    }
    if (p.post_exec && lane == 0 && p.stats) {
      const int subst = __popcll(tp.exec_mask & ~tp.kr_mask), hits = __popcll(tp.kr_mask & p.snap.resident_mask);
      if (subst) atomicAdd(&p.stats->substitutions, (unsigned long long)subst);
      if (hits) atomicAdd(&p.stats->hits_R, (unsigned long long)hits);
    }
  }
  cluster.sync();  // every token's mask and gates are in the leader's shared memory
  if (crank != 0) return;
  // ---- phase B, counts: warp w counts the tokens of experts w and w + 32
  for (int e = warp; e < N; e += nwarp) {
    int c = 0;
    if ((p.run_mask >> e) & 1)
      for (int b0 = 0; b0 < B; b0 += 32) {
        const int t = b0 + lane;
        c += __popc(__ballot_sync(0xffffffffu, t < B && ((s_exec[t] >> e) & 1)));
      }
    if (lane == 0) s_count[e] = c;
  }
  __syncthreads();
  if (warp == 0) {
    // exclusive prefix over the experts (lane owns experts lane and lane + 32), then the group table: one group per
    // executed expert, then the shared expert
    const int c0 = lane < N ? s_count[lane] : 0, c1 = lane + 32 < N ? s_count[lane + 32] : 0;
    int i0 = c0, i1 = c1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u0 = __shfl_up_sync(0xffffffffu, i0, o), u1 = __shfl_up_sync(0xffffffffu, i1, o);
      if (lane >= o) {
        i0 += u0;
        i1 += u1;
      }
    }
    const int tot0 = __shfl_sync(0xffffffffu, i0, 31), acc = tot0 + __shfl_sync(0xffffffffu, i1, 31);
    const int off0 = i0 - c0, off1 = tot0 + i1 - c1;
    if (lane < N) s_off[lane] = off0;
    if (lane + 32 < N) s_off[lane + 32] = off1;
    const unsigned g0m = __ballot_sync(0xffffffffu, c0 > 0), g1m = __ballot_sync(0xffffffffu, c1 > 0);
    const int ng_routed = __popc(g0m) + __popc(g1m);
    if (c0 > 0) {
      const int gi = __popc(g0m & ((1u << lane) - 1u));
      p.grp[4 + 3 * gi] = lane;
      p.grp[5 + 3 * gi] = off0;
      p.grp[6 + 3 * gi] = c0;
    }
    if (c1 > 0) {
      const int gi = __popc(g0m) + __popc(g1m & ((1u << lane) - 1u));
      p.grp[4 + 3 * gi] = lane + 32;
      p.grp[5 + 3 * gi] = off1;
      p.grp[6 + 3 * gi] = c1;
    }
    if (lane == 0) {
      s_off[N] = acc;  // routed pairs
      p.grp[0] = ng_routed;
      if (p.run_shared) {
        p.grp[4 + 3 * ng_routed] = N;
        p.grp[5 + 3 * ng_routed] = acc;
        p.grp[6 + 3 * ng_routed] = B;
      }
      p.grp[1] = ng_routed + (p.run_shared ? 1 : 0);
    }
  } else if (warp == 1) {  // unions over the tokens
    unsigned long long kr = 0ull, ex = 0ull;
    for (int t = lane; t < B; t += 32) {
      kr |= s_kr[t];
      ex |= s_exec[t];
    }
    const unsigned kl = __reduce_or_sync(0xffffffffu, (unsigned)kr), kh = __reduce_or_sync(0xffffffffu, (unsigned)(kr >> 32));
    const unsigned el = __reduce_or_sync(0xffffffffu, (unsigned)ex), eh = __reduce_or_sync(0xffffffffu, (unsigned)(ex >> 32));
    if (lane == 0) {
      p.plan_masks[0] = ((unsigned long long)kh << 32) | kl;
      p.plan_masks[1] = ((unsigned long long)eh << 32) | el;
    }
  }
  __syncthreads();
  // ---- phase B, placement: token b of expert e goes to s_off[e] + (number of earlier tokens of e)
  for (int e = warp; e < N; e += nwarp) {
    if (s_count[e] == 0) continue;
    int o = s_off[e];
    for (int b0 = 0; b0 < B; b0 += 32) {
      const int t = b0 + lane;
      const bool has = t < B && ((s_exec[t] >> e) & 1);
      const unsigned m = __ballot_sync(0xffffffffu, has);
      if (has) {
        const int at = o + __popc(m & ((1u << lane) - 1u));
        p.pair_tok[at] = t;
        p.pair_gate[at] = s_pgate[t][__popcll(s_exec[t] & ((1ull << e) - 1ull))];
      }
      o += __popc(m);
    }
  }
  if (p.run_shared) {
    const int base = s_off[N];
    for (int t = threadIdx.x; t < B; t += blockDim.x) {
      p.pair_tok[base + t] = t;
      p.pair_gate[base + t] = p.shared_gate ? s_sgate[t] : 1.f;
    }
  }
  SPAN_END(6);
}

cudaError_t launch_ffn_plan(const FfnParams& p, int n_sm, cudaStream_t s) {
  int n_cta = (p.B + 31) / 32;
  n_cta = n_cta < 1 ? 1 : (n_cta > kPlanMaxCtas ? kPlanMaxCtas : n_cta);
  // helpers: eight values per thread while the GPU has SMs for it
  int helpers = ((int)((size_t)p.B * p.d / 8 + 1023) / 1024 + n_cta - 1) / n_cta;
  const int most = n_sm / n_cta - 1;
  helpers = helpers > most ? most : helpers;
  helpers = helpers < 1 ? 1 : helpers;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_cta * (1 + helpers), 1, 1);
  cfg.blockDim = dim3(1024, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = n_cta;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, ffn_plan_kernel, p);
}

}  // namespace apex
