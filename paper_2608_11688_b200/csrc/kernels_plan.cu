// ffn_plan_kernel: the execution sets of a batched step (B > 1) and the (expert, token) pair list sorted by expert, for the
// per-pair streaming kernel.  (The grouped GEMM derives its plan itself.)
//
// A cluster of ceil(B / 32) CTAs (at most 8) of 32 warps.  Phase A: every warp of the cluster plans one token (planning
// a token costs a warp 2-3 us of dependent latency, so eight tokens per warp on one SM were 16 us at B = 256) and puts
// its masks and gates into the leader CTA's shared memory through distributed shared memory.  Phase B, leader
// CTA only: warp w owns experts w and w+32 and gathers the tokens that execute them with ballots, so the pair list is
// sorted by (expert, token).  Shared-expert pairs (expert id N) follow.
#include <cooperative_groups.h>

#include "apex_internal.hpp"
#include "ptx.cuh"
#include "token_plan.cuh"

namespace cg = cooperative_groups;

namespace apex {

constexpr int kPlanWarps = 32;
static_assert(APEX_MAX_BATCH <= 8 * kPlanWarps, "one token per warp needs a cluster of at most 8 CTAs");

__global__ void __launch_bounds__(kPlanWarps * 32) ffn_plan_kernel(const FfnParams p) {
  SPAN_BEGIN();
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ unsigned long long s_kr[APEX_MAX_BATCH], s_exec[APEX_MAX_BATCH];
  __shared__ float s_pgate[APEX_MAX_BATCH][APEX_MAX_TOPK];  // gate of the j-th executed expert of each token
  __shared__ float s_sgate[APEX_MAX_BATCH];                 // weight of the shared expert for each token (gated variant)
  __shared__ int s_count[APEX_MAX_EXPERTS], s_off[APEX_MAX_EXPERTS + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int N = p.N, k = p.k, B = p.B;
  const int b = (int)cluster.block_rank() * kPlanWarps + warp;  // this warp's token
  if (b < B) {
    // the leader's copies of the per-token results
    unsigned long long *l_kr = cluster.map_shared_rank(&s_kr[0], 0), *l_exec = cluster.map_shared_rank(&s_exec[0], 0);
    float *l_pgate = cluster.map_shared_rank(&s_pgate[0][0], 0), *l_sgate = cluster.map_shared_rank(&s_sgate[0], 0);
    const TokenLoads tl = load_token(p.idx + (size_t)b * k, p.z_r + (size_t)b * N, p.alpha + (size_t)b * N, N, k, p.mode, lane);
    const TokenPlan tp = plan_token(tl, p.mode, p.norm_topk, p.snap.resident_mask, lane);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int e = lane + 32 * h;
      if (!((tp.exec_mask >> e) & 1)) continue;
      const int pos = __popcll(tp.exec_mask & ((1ull << e) - 1ull));
      if (pos < APEX_MAX_TOPK) l_pgate[b * APEX_MAX_TOPK + pos] = h ? tp.g1 : tp.g0;
    }
    if (lane == 0) {
      l_kr[b] = tp.kr_mask;
      l_exec[b] = tp.exec_mask;
    }
    if (p.run_shared && p.shared_gate) {
      const float sg = shared_gate_weight(p.shared_gate, p.hpost + (size_t)b * p.d, p.d, lane);
      if (lane == 0) l_sgate[b] = sg;
    }
    if (p.post_exec) {
      store_token_plan(tp, lane, k, p.exec_idx ? p.exec_idx + (size_t)b * k : nullptr, p.exec_gate ? p.exec_gate + (size_t)b * k : nullptr, nullptr);
      if (lane == 0 && p.stats) {
        const int subst = __popcll(tp.exec_mask & ~tp.kr_mask), hits = __popcll(tp.kr_mask & p.snap.resident_mask);
        if (subst) atomicAdd(&p.stats->substitutions, (unsigned long long)subst);
        if (hits) atomicAdd(&p.stats->hits_R, (unsigned long long)hits);
      }
    }
  }
  cluster.sync();  // every token's masks and gates are in the leader's shared memory
  if (cluster.block_rank() != 0) return;
  if (p.post_exec && warp == kPlanWarps - 1) {
    // the unions for the host: one 16-byte store each, with the sequence number
    unsigned u[4] = {0u, 0u, 0u, 0u};
    for (int t = lane; t < B; t += 32) {
      u[0] |= (unsigned)s_kr[t];
      u[1] |= (unsigned)(s_kr[t] >> 32);
      u[2] |= (unsigned)s_exec[t];
      u[3] |= (unsigned)(s_exec[t] >> 32);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) u[j] = __reduce_or_sync(0xffffffffu, u[j]);
    if (lane < 2)
      asm volatile("st.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p.mbox_rec + 4 * lane), "r"(lane ? u[2] : u[0]), "r"(lane ? u[3] : u[1]), "r"(p.seq_value), "r"(0u)
                   : "memory");
  }
  // ---- counts: warp w counts the tokens of experts w and w + 32
  for (int e = warp; e < N; e += kPlanWarps) {
    int c = 0;
    if ((p.run_mask >> e) & 1)
      for (int t0 = 0; t0 < B; t0 += 32) {
        const int t = t0 + lane;
        c += __popc(__ballot_sync(0xffffffffu, t < B && ((s_exec[t] >> e) & 1)));
      }
    if (lane == 0) s_count[e] = c;
  }
  __syncthreads();
  if (warp == 0) {
    // exclusive prefix over the experts (lane owns experts lane and lane + 32)
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
    const int tot0 = __shfl_sync(0xffffffffu, i0, 31), all = tot0 + __shfl_sync(0xffffffffu, i1, 31);
    if (lane < N) s_off[lane] = i0 - c0;
    if (lane + 32 < N) s_off[lane + 32] = tot0 + i1 - c1;
    if (lane == 0) {
      s_off[N] = all;
      p.n_pairs[0] = all + (p.run_shared ? B : 0);
    }
  }
  __syncthreads();
  // ---- placement: token t of expert e goes to s_off[e] + (number of earlier tokens of e)
  for (int e = warp; e < N; e += kPlanWarps) {
    if (s_count[e] == 0) continue;
    int o = s_off[e];
    for (int t0 = 0; t0 < B; t0 += 32) {
      const int t = t0 + lane;
      const bool has = t < B && ((s_exec[t] >> e) & 1);
      const unsigned m = __ballot_sync(0xffffffffu, has);
      if (has) {
        const int at = o + __popc(m & ((1u << lane) - 1u));
        p.pair_tok[at] = t;
        p.pair_expert[at] = e;
        p.pair_gate[at] = s_pgate[t][__popcll(s_exec[t] & ((1ull << e) - 1ull))];
      }
      o += __popc(m);
    }
  }
  if (p.run_shared) {
    for (int t = threadIdx.x; t < B; t += blockDim.x) {
      p.pair_tok[s_off[N] + t] = t;
      p.pair_expert[s_off[N] + t] = N;
      p.pair_gate[s_off[N] + t] = p.shared_gate ? s_sgate[t] : 1.f;
    }
  }
  SPAN_END(6);
}

cudaError_t launch_ffn_plan(const FfnParams& p, cudaStream_t s) {
  const int n_cta = (p.B + kPlanWarps - 1) / kPlanWarps;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_cta, 1, 1);
  cfg.blockDim = dim3(kPlanWarps * 32, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = n_cta;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, ffn_plan_kernel, p);
}

}  // namespace apex
