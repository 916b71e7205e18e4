// Device code shared by the router kernels and the persistent decode kernel: the fixed-order warp reductions, the
// budget selection of one token (Eq. (8), (9), (1)) and the per-token epilogue of a router (softmax, ranking, top-k,
// metrics of Eq. (2), (3)).
#ifndef APEX_ROUTER_COMMON_CUH
#define APEX_ROUTER_COMMON_CUH

#include "apex_internal.hpp"

#ifndef RTL
#define RTL(i) do { } while (0)
#endif

namespace apex {

__device__ __forceinline__ float warp_sum_tree(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {  // (as fmaxf: a NaN is passed over)
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ int warp_max_int(int v) { return __reduce_max_sync(0xffffffffu, v); }

// One cluster per token.  CTA r of the cluster owns experts r*wpc .. r*wpc+wpc-1, one warp per
// expert; the logits are gathered in the leader CTA's shared memory through distributed shared
// memory, and the leader's first warp does softmax, ranking, top-k and (for the gate) the
// per-step metrics of Eq. (2)-(3).
// Budget selection for one token by one warp (Eq. (8), (9) in the logit domain; Eq. (1)).
// Lane l holds positions l and l+32 of the ranked list E: pj = expert at that position, x = its
// prefetch probability (so x is the prefetch distribution in descending order).
//   s = w.x   (lane partial: position l then l+32 with fused multiply-adds, then the xor tree)
//   delta_hat = first delta with theta_delta - s >= logit(tau), capped to C - k
//   K_p = first k + delta_hat experts of E
// The budget itself (uniform over the warp): returns delta_hat after the cap, *uncapped receives it before.
// w0, w1: w at positions lane, lane + 32; th0, th1: theta at lane, lane + 32 (anything where there is none).
__device__ __forceinline__ int select_budget_vals(float w0, float w1, float th0, float th1, float t_tau, int force, int N, int k,
                                                  int C, int lane, float x0, float x1, int* uncapped) {
  float part = 0.f;
  if (lane < N) part = fmaf(w0, x0, part);
  if (lane + 32 < N) part = fmaf(w1, x1, part);
  const float sdot = warp_sum_tree(part);
  const int nth = N - k + 1;
  const bool pass0 = lane < nth && (th0 - sdot >= t_tau);
  const bool pass1 = lane + 32 < nth && (th1 - sdot >= t_tau);
  const unsigned m0 = __ballot_sync(0xffffffffu, pass0), m1 = __ballot_sync(0xffffffffu, pass1);
  int d_hat = m0 ? (__ffs(m0) - 1) : (m1 ? 32 + __ffs(m1) - 1 : N - k);
  if (force == 1) d_hat = 0;
  if (force == 2) d_hat = N - k;
  *uncapped = d_hat;
  return min(d_hat, C - k);
}
// The parameters of the confidence model a lane needs, loaded ahead of the token's logits
struct SelectVals {
  float w0 = 0.f, w1 = 0.f, th0 = 0.f, th1 = 0.f;
};
__device__ __forceinline__ SelectVals load_select_vals(const SelectParams& p, int lane) {
  const int nth = p.N - p.k + 1;
  SelectVals v;
  if (lane < p.N) v.w0 = __ldg(p.w + lane);
  if (lane + 32 < p.N) v.w1 = __ldg(p.w + lane + 32);
  if (lane < nth) v.th0 = __ldg(p.theta + lane);
  if (lane + 32 < nth) v.th1 = __ldg(p.theta + lane + 32);
  return v;
}

__device__ __forceinline__ void select_token(const SelectParams& p, const SelectVals& v, int b, int lane, int pj0, int pj1, float x0, float x1) {
  const int N = p.N, k = p.k, C = p.C;
  int uncapped;
  const int d_hat = select_budget_vals(v.w0, v.w1, v.th0, v.th1, p.t_tau, p.force, N, k, C, lane, x0, x1, &uncapped);
  const int ncand = k + d_hat;
  const bool in0 = lane < ncand, in1 = lane + 32 < ncand;
  // the candidate set as a 64-bit mask
  unsigned lo = 0, hi = 0;
  if (in0) { if (pj0 < 32) lo |= 1u << pj0; else hi |= 1u << (pj0 - 32); }
  if (in1) { if (pj1 < 32) lo |= 1u << pj1; else hi |= 1u << (pj1 - 32); }
  lo = __reduce_or_sync(0xffffffffu, lo);
  hi = __reduce_or_sync(0xffffffffu, hi);
  // The host needs only the sets, a record per token: mask, count and sequence number travel in ONE aligned 16-byte store,
  // so no system-scope fence and no counter over the batch sits on the kernel's path.  (The ranked list below is
  // advisory for the host at B = 1: it is used for the issue order only if it matches the mask.)
  if (lane == 0)
    asm volatile("st.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p.mbox_rec + 4 * b), "r"(lo), "r"(hi), "r"((unsigned)ncand), "r"(p.seq_value)
                 : "memory");
  // candidates in rank order, padded with -1
  if (lane < C) {
    const int e = in0 ? pj0 : -1;
    p.cand_out[(size_t)b * C + lane] = e;
    if (p.B == 1) p.mbox_cand[lane] = e;
  }
  if (lane + 32 < C) {
    const int e = in1 ? pj1 : -1;
    p.cand_out[(size_t)b * C + lane + 32] = e;
    if (p.B == 1) p.mbox_cand[lane + 32] = e;
  }
  if (lane == 0) {
    p.ncand_out[b] = ncand;
    p.ncand_keep[b] = ncand;
    if (p.stats) {
      atomicAdd(&p.stats->tokens, 1ull);
      atomicAdd(&p.stats->sum_delta_hat, (unsigned long long)d_hat);
      atomicAdd(&p.stats->sum_ncand, (unsigned long long)ncand);
      atomicAdd(&p.stats->capped, (unsigned long long)(uncapped > d_hat ? 1 : 0));
      atomicAdd(&p.stats->near_full, (unsigned long long)(2 * ncand > N ? 1 : 0));
    }
  }
}


// Softmax, ranking, top-k and the per-token outputs of one token by one warp (lanes own experts lane and lane+32),
// from the token's N logits in shared memory; then either the budget selection (prefetch router, fused launch) or
// the metrics of Eq. (2), (3) against the prefetch stage (gate).  qs, pis, posp: this warp's scratch, 64 entries each.
// Softmax over the N logits in shared memory and the rank of this lane's two experts (e0 = lane, e1 = lane + 32):
// rank = number of experts ordered before it by (value descending, index ascending).
struct RankedLogits {
  float z0, z1;  // logits (most negative float where the lane has no expert)
  float q0, q1;  // softmax
  int r0, r1;    // ranks
};
// the two halves of softmax_and_rank, for callers that need the ranks before the probabilities
// (zs: 16-byte aligned)
__device__ __forceinline__ void rank_lane_logits(const float* zs, int N, int lane, RankedLogits* R) {
  const int e0 = lane, e1 = lane + 32;
  const float NEG = -3.402823466e38f;
  R->z0 = e0 < N ? zs[e0] : NEG;
  R->z1 = e1 < N ? zs[e1] : NEG;
  // The larger ones alone first, two instructions per comparison.  Without ties the ranks of the N experts add up to N (N - 1) / 2;
  // a tie (or a NaN) leaves a pair out, and then the order of the indices is looked at too.  With that in every comparison, and
  // the maximum by shuffles, barrier, ranking and softmax of 60 experts took 4 000 to 5 000 cycles of a router, 3 000 to 3 600 so; a token
  // of 32 layers (d = 1536, N = 40) 658 us and 652.
  int r0 = 0, r1 = 0;
  auto count = [&](float zf) {
    r0 += zf > R->z0 ? 1 : 0;
    r1 += zf > R->z1 ? 1 : 0;
  };
  int f = 0;
#pragma unroll 4
  for (; f + 4 <= N; f += 4) {
    const float4 v = *reinterpret_cast<const float4*>(zs + f);
    count(v.x);
    count(v.y);
    count(v.z);
    count(v.w);
  }
  for (; f < N; ++f) count(zs[f]);
  const int all = __reduce_add_sync(0xffffffffu, (e0 < N ? r0 : 0) + (e1 < N ? r1 : 0));
  if (all != N * (N - 1) / 2) {
    r0 = r1 = 0;
    for (f = 0; f < N; ++f) {
      const float zf = zs[f];
      r0 += (zf > R->z0 || (zf == R->z0 && f < e0)) ? 1 : 0;
      r1 += (zf > R->z1 || (zf == R->z1 && f < e1)) ? 1 : 0;
    }
  }
  R->r0 = r0;
  R->r1 = r1;
}
__device__ __forceinline__ void softmax_lane_logits(int N, int lane, RankedLogits* R) {
  const int e0 = lane, e1 = lane + 32;
  const float m = warp_max(fmaxf(R->z0, R->z1));
  const float x0 = e0 < N ? expf(R->z0 - m) : 0.f;
  const float x1 = e1 < N ? expf(R->z1 - m) : 0.f;
  const float sum = warp_sum_tree(x0 + x1);
  R->q0 = x0 / sum;
  R->q1 = x1 / sum;
}
__device__ __forceinline__ RankedLogits softmax_and_rank(const float* zs, int N, int lane) {
  RankedLogits R;
  rank_lane_logits(zs, N, lane, &R);
  softmax_lane_logits(N, lane, &R);
  return R;
}

// What the epilogue of a token reads from memory besides the logits, asked for before they are there: the confidence
// model (fused selection), or the prefetch stage's ranking and budget (gate).
struct EpilogueVals {
  SelectVals sel;
  int pred0 = -1, pred1 = -1, ncand = 0;
};
__device__ __forceinline__ void load_prediction(const RouterParams& p, int b, int lane, EpilogueVals* v) {  // after the dependency wait
  if (!p.pi_pred || b >= p.B) return;
  const size_t row = (size_t)b * p.N;
  if (lane < p.N) v->pred0 = __ldg(p.pi_pred + row + lane);
  if (lane + 32 < p.N) v->pred1 = __ldg(p.pi_pred + row + lane + 32);
  v->ncand = __ldg(p.ncand_pred + b);
}

__device__ __forceinline__ void router_epilogue(const RouterParams& p, const EpilogueVals& v, int b, int lane, const float* zs, float* qs,
                                                int* pis, int* posp) {
  const int N = p.N, k = p.k;
  const int e0 = lane, e1 = lane + 32;
  const RankedLogits R = softmax_and_rank(zs, N, lane);
  const float z0 = R.z0, z1 = R.z1, q0 = R.q0, q1 = R.q1;
  const int r0 = R.r0, r1 = R.r1;
  auto outputs = [&]() {
    const size_t row = (size_t)b * N;
    if (e0 < N) {
      p.z_out[row + e0] = z0;
      p.q_out[row + e0] = q0;
      if (p.pi_out) p.pi_out[row + r0] = e0;
      if (p.topk_out && r0 < k) p.topk_out[(size_t)b * k + r0] = e0;
    }
    if (e1 < N) {
      p.z_out[row + e1] = z1;
      p.q_out[row + e1] = q1;
      if (p.pi_out) p.pi_out[row + r1] = e1;
      if (p.topk_out && r1 < k) p.topk_out[(size_t)b * k + r1] = e1;
    }
  };
  RTL(4);
  if (p.fuse_select) {
    // prefetch router and budget selection in one launch: the ranked list goes through shared memory
    if (e0 < N) { qs[e0] = q0; pis[r0] = e0; }
    if (e1 < N) { qs[e1] = q1; pis[r1] = e1; }
    __syncwarp();
    const int pj0 = lane < N ? pis[lane] : -1, pj1 = lane + 32 < N ? pis[lane + 32] : -1;
    const float x0 = pj0 >= 0 ? qs[pj0] : 0.f, x1 = pj1 >= 0 ? qs[pj1] : 0.f;
    select_token(p.sel, v.sel, b, lane, pj0, pj1, x0, x1);
    outputs();
    RTL(5);
    return;
  }
  if (p.mbox_rec) {  // the host waits for the routed set: first of all
    const unsigned lo = __ballot_sync(0xffffffffu, e0 < N && r0 < k), hi = __ballot_sync(0xffffffffu, e1 < N && r1 < k);
    if (lane == 0)
      asm volatile("st.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p.mbox_rec), "r"(lo), "r"(hi), "r"(p.seq_value), "r"(0u) : "memory");
  }
  outputs();
  if (!p.topk_out || !p.stats) return;

  // ---- gate epilogue: metrics of this token against the prefetch stage (Eq. (2), (3))
  const bool in0 = e0 < N && r0 < k, in1 = e1 < N && r1 < k;
  {
    int dstar = 0, hitsP = 0, have_pred = 0;
    if (p.pi_pred) {
      have_pred = 1;
      if (e0 < N) posp[v.pred0] = e0;  // position of expert pi[j] in E is j
      if (e1 < N) posp[v.pred1] = e1;
      __syncwarp();
      const int nc = v.ncand;
      const int pos0 = in0 ? posp[e0] : -1, pos1 = in1 ? posp[e1] : -1;
      dstar = warp_max_int(max(pos0, pos1)) + 1 - k;
      hitsP = __popc(__ballot_sync(0xffffffffu, in0 && pos0 < nc)) + __popc(__ballot_sync(0xffffffffu, in1 && pos1 < nc));
    }
    if (lane == 0) {
      atomicAdd(&p.stats->routed, (unsigned long long)k);
      if (have_pred) {
        atomicAdd(&p.stats->sum_delta_star, (unsigned long long)dstar);
        atomicAdd(&p.stats->hits_P, (unsigned long long)hitsP);
        atomicAdd(&p.stats->covered, (unsigned long long)(hitsP == k ? 1 : 0));
      }
    }
  }
  RTL(5);
}

}  // namespace apex

#endif  // APEX_ROUTER_COMMON_CUH
