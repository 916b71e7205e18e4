// The token kernel (see kernels_decode.cu: all L layer-steps of one token in one cooperative launch, the steps and their
// dependences as there) for rows that are worked on in tiles by all warps of a CTA (ffn_tiles.cuh).
//
// A CTA has eight worker warps and a group of four, of which three have something to do:
//   planner  owns the shared-memory ring and everything that decides what goes through it: waits for the other CTAs' counters, streams the
//            CTA's share of the attention stand-in, derives the routed and the execution set from the ranks the workers have
//            counted, confirms the slot table, waits for ready flags and demand copies, and requests the expert rows
//   gates    probabilities and gates of the executed experts, while the first rows are on their way
//   clerk    (in one CTA, the poster) candidate set of the prefetch router, the outputs, counters and records for the host
// The workers take the router logits and the tiles, and nothing else: with every warp planning for itself and requesting its own
// rows, a tile's chain was 2 400 cycles instead of 2 100, the first request came 1 us later, and the kernel's state did not
// fit its registers.  The group of four gives registers to the workers (setmaxnreg); without that 400 bytes were spilled, and
// d = 1536 took 754 us per token (32 layers, 8 of 40 experts of 512 rows) instead of 658.  With it none, or up to 20 bytes (bf16 d = 2048,
// e4m3 from d = 1536 on, e2m1 d = 1536).
//
// Ring: NT tiles of kRows rows, used in order by stand-in pieces and by row tiles alike; `full` completes with a tile's bytes,
// `empty` when the eight workers have read it (the planner stands in for them where it consumed a stand-in piece).
//
// What bounds it: HBM while stand-in and rows stream (two thirds of the layer at d = 1536), the chain between them otherwise.  us
// per token, all experts resident, against the row-per-warp kernel: d = 1536 as above 677 -> 658; 8 layers of 4 experts:
// d = 256, I = 7000 323 -> 171; d = 512, I = 1500 and a shared expert of 500 134 -> 112; d = 768, I = 3000 212 -> 162; d = 1024,
// I = 2500 208 -> 175; d = 2048, I = 3000 and 700 322 -> 318.  At d = 256 a copy per row is what is left: the copy engine takes one
// every 85 cycles.
// Quantised stores, 8 layers of 4 experts, against the row-per-warp kernel: e4m3 d = 512, I = 6000 314 -> 163; d = 1024, I = 2500
// 203 -> 153; d = 1536, I = 1500 195 -> 160; d = 2048, I = 2500 294 -> 224 (61.6 MB of rows per layer, and 42 of the stand-in: 16 us of its 28
// are bytes); e2m1, the same sizes, 316 -> 175, 202 -> 147, 194 -> 166, 299 -> 224: the conversions of the codes.
#include <cuda_bf16.h>

#include "apex_internal.hpp"
#include "decode_common.cuh"
#include "ffn_tiles.cuh"
#include "ptx.cuh"
#include "router_common.cuh"
#include "token_plan.cuh"

namespace apex {

namespace {

constexpr int kPlanner = kDecWarps, kClerk = kDecWarps + 1, kGates = kDecWarps + 2;  // warp indices; the last of their warpgroup leaves at once
constexpr int kTileThreads = kDecThreads + 128;
// Registers: 384 threads start with 168 each; the four warps of the planner's group give up what the workers take
constexpr int kPlanRegs = 104, kWorkRegs = 200;
static_assert(kPlanRegs * 128 + kWorkRegs * kDecThreads <= 168 * kTileThreads, "the split is served from the block's own registers");

// Rows of a tile: enough for the chain of a tile (some 1 200 cycles) to be worth it, and three tiles in the ring at least where a
// row allows it.  Quantised rows: two 8-row blocks make one MMA of the down projection, so 16 rows even where the ring holds two tiles
// (e4m3 d = 2048, I = 2500: 224 us against 235 with eight rows); with 32 e2m1 d = 1024 takes 171 us instead of 182, d = 1536 213 instead of 193.
__host__ __device__ constexpr int tile_blocks(int fmt, int d) {
  return fmt_entry_bytes(fmt, d) <= 1700u ? 4 : fmt_entry_bytes(fmt, d) <= (fmt == kFmtBf16 ? 3200u : 6400u) ? 2 : 1;
}
// (the kernel's static variables: 3 KB and the exchange of a tile, twice; a d = 1536 bf16 ring of three tiles fills the rest)
__host__ __device__ constexpr int tile_ring(int fmt, int d) {
  const int n = (kDecSmemTotal - 3328 - 8 * tile_blocks(fmt, d) * (2 * kPartStride * 4 + (fmt == kFmtBf16 ? 0 : kTileWarps * 6)) - 4 * d) / (int)(tile_stride(fmt_entry_bytes(fmt, d)) * 8 * tile_blocks(fmt, d));
  return n > 8 ? 8 : n;
}

// Row weights: 16 per CTA; with the prefetch stage running 14 for the CTAs of the first cluster, which take its logits too
__device__ __forceinline__ unsigned tile_weight_prefix(int cta, bool prefetching) {
  return 16u * cta - (prefetching ? 2u * min(cta, kDecCluster) : 0u);
}
// ---- waits.  What happens when one is not met at once stands out of line: inlined at every wait it was half of the kernel's
// 190 KB of code, and a layer's path, which runs through most of it, waited for instructions.
struct Limits {
  int* abort;                // this CTA has given up, or has learnt that another one did
  unsigned int* abort_all;   // device word: somebody gave up
  volatile uint32_t* status;
  long long wait_ns;
};
__device__ __forceinline__ bool stop_requested(const Limits& h) {
  if (*(volatile int*)h.abort) return true;
  if (ld_volatile_u32(h.abort_all)) {
    atomicExch(h.abort, 1);
    return true;
  }
  return false;
}
__device__ __forceinline__ void give_up(const Limits h) {  // a wait ran out: tell the CTA, the other CTAs and the host
  atomicExch(h.abort, 1);
  atomicExch(h.abort_all, 1u);
  *h.status = 1u;
}
// whole warp: bounded wait on a shared-memory barrier that also leaves when anybody has given up
__device__ __forceinline__ bool warp_wait_on(uint64_t* bar, uint32_t parity, const Limits h) {
  bool met = false;
  const unsigned long long t0 = globaltimer_ns();
  for (uint32_t it = 1; !met; ++it) {
    met = mbar_try_wait(bar, parity);
    if (!met && (it & 127u) == 0u && (stop_requested(h) || (long long)(globaltimer_ns() - t0) > h.wait_ns)) break;
  }
  met = __all_sync(0xffffffffu, met);
  if (!met && (threadIdx.x & 31) == 0 && !stop_requested(h)) give_up(h);
  return met;
}
// What a warp waits for in memory: how a word is read, and when it will do
enum PollKind { kPollCount, kPollSeq64, kPollSeqGpu, kPollSeqSys, kPollTag, kPollGen };
__device__ __forceinline__ bool poll_met(PollKind kind, const void* at, unsigned long long want) {
  if (kind == kPollCount) return ld_acquire_gpu_u64(static_cast<const unsigned long long*>(at)) >= want;
  if (kind == kPollSeq64) return ld_acquire_gpu_u64(static_cast<const unsigned long long*>(at)) == want;
  if (kind == kPollSeqGpu) return ld_acquire_gpu_u32(static_cast<const uint32_t*>(at)) == (uint32_t)want;
  const uint32_t v = ld_acquire_sys(static_cast<const uint32_t*>(at));
  if (kind == kPollSeqSys) return v == (uint32_t)want;
  if (kind == kPollTag) return (v >> 8) == (uint32_t)want;
  return (int32_t)(v - (uint32_t)want) >= 0;  // kPollGen
}
// whole warp, lane 0 polls: nanoseconds waited, or -1
__device__ __forceinline__ long long warp_poll_on(PollKind kind, const void* at, unsigned long long want, int pause_ns, const Limits h) {
  long long r = 0;
  if ((threadIdx.x & 31) == 0) {
    const unsigned long long t0 = globaltimer_ns();
    for (uint32_t it = 1;; ++it) {
      __nanosleep(pause_ns);
      if (poll_met(kind, at, want)) break;
      if ((it & 7u) == 0u && (stop_requested(h) || (long long)(globaltimer_ns() - t0) > h.wait_ns)) {
        r = -1;
        break;
      }
    }
    if (r == 0) r = (long long)(globaltimer_ns() - t0);
    else if (!stop_requested(h)) give_up(h);
  }
  return __shfl_sync(0xffffffffu, r, 0);
}
// one lane of a converged warp
__device__ __forceinline__ bool elect_one() {
  uint32_t r;
  asm volatile("{\n.reg .pred e;\nelect.sync _|e, 0xffffffff;\nselp.u32 %0, 1, 0, e;\n}" : "=r"(r));
  return r != 0;
}
__device__ __forceinline__ void workers_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(kDecThreads) : "memory"); }

}  // namespace

template <int NCH, int FMT>
__global__ void __launch_bounds__(kTileThreads, 1) decode_tiles_kernel(const DecodeParams p) {
  constexpr int d = NCH * 256;
  constexpr uint32_t entry_bytes = fmt_entry_bytes(FMT, d), stride = tile_stride(entry_bytes);
  constexpr int R = tile_blocks(FMT, d), kRows = 8 * R, NT = tile_ring(FMT, d);
  constexpr uint32_t tile_bytes = kRows * stride;
  constexpr int NV = d / 128;                  // float4 per lane of a router row
  constexpr int SLICE4 = d / 4 / kDecCluster;  // float4 columns of y a CTA adds for its cluster
  static_assert(NT >= 2, "ring too small");
  static_assert(SLICE4 >= 1 && SLICE4 <= kDecThreads, "one thread per float4 of the cluster slice");
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ uint64_t s_full[NT], s_empty[NT];
  __shared__ uint64_t s_xbar[2];     // logits of the prefetch router / of the gate have arrived from the whole cluster
  __shared__ uint64_t s_cbar[2];     // the planner has seen: the previous layer's y complete / the stand-in complete
  __shared__ uint64_t s_rbar;        // every worker has added its share of the gate's rank counts
  __shared__ uint64_t s_hbar;        // every worker has taken its h': the ring may be filled
  __shared__ uint64_t s_gbar[2];     // the gates of the layer's rows are there (of their repetition)
  __shared__ unsigned long long s_run[2];  // per pass: execution set
  __shared__ uint64_t s_plan;        // the layer's tiles are known
  __shared__ uint64_t s_verdict;     // ... and whether they were requested from the right slot table
  __shared__ unsigned s_rank[APEX_MAX_EXPERTS / 4];  // rank of each expert's gate logit, four 8-bit counts to a word (zero between layers)
  __shared__ __align__(16) float s_zp[APEX_MAX_EXPERTS];
  __shared__ __align__(16) float s_zr[APEX_MAX_EXPERTS];
  __shared__ float s_q[APEX_MAX_EXPERTS];            // clerk: prefetch probabilities by expert
  __shared__ int s_pi[APEX_MAX_EXPERTS];             // ... expert by rank
  __shared__ int s_posp[APEX_MAX_EXPERTS];           // ... position of each expert in the prefetch ranking
  __shared__ float s_gate[APEX_MAX_EXPERTS + 1];     // gates of the executed experts, of the shared one
  __shared__ uint8_t s_exp[NT * kRows];              // expert of each row in the ring (N: the shared one)
  __shared__ int s_use[2], s_rows[2];                // per pass: ring use of the first tile, rows
  __shared__ int s_again;                            // the rows are to be repeated with the published table
  __shared__ int s_abort;
  __shared__ int s_stop[2];                          // a worker has given up
  __shared__ __align__(16) float s_part[2][kRows * kPartStride];  // the warps' shares of a tile's dot products
  __shared__ __align__(16) __half s_planes[FMT == kFmtBf16 ? 1 : kTileWarps][FMT == kFmtBf16 ? 2 : 3 * kRows];  // a worker's planes of a tile's gated intermediate
  float4* part4 = reinterpret_cast<float4*>(smem + (size_t)NT * tile_bytes);  // this CTA's partial y (behind the ring)

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int N = p.N, k = p.k, I = p.I, L = p.L;
  const int G = gridDim.x, cta = blockIdx.x;
  const uint32_t crank = cluster_ctarank();
  const bool poster = cta == kDecCluster - 1;  // the CTA that writes global outputs, counters and the host's records

  SPAN_BEGIN();
  if (tid == 0) {
    s_abort = 0;
    s_stop[0] = s_stop[1] = 0;
    for (int i = 0; i < NT; ++i) {
      mbar_init(&s_full[i], 1);
      mbar_init(&s_empty[i], kDecWarps);
    }
    mbar_init(&s_xbar[0], 1);
    mbar_init(&s_xbar[1], 1);
    mbar_init(&s_cbar[0], 1);
    mbar_init(&s_cbar[1], 1);
    mbar_init(&s_rbar, kDecWarps);
    mbar_init(&s_hbar, kDecWarps);
    mbar_init(&s_gbar[0], 1);
    mbar_init(&s_gbar[1], 1);
    mbar_init(&s_plan, 1);
    mbar_init(&s_verdict, 1);
  }
  if (tid < APEX_MAX_EXPERTS / 4) s_rank[tid] = 0u;
  if (p.zero_y) {
    // y of all layers, a slice per CTA.  Nobody adds to it before the first layer's cluster barrier, which follows the count
    // of the stand-in by every CTA, and a CTA counts itself in behind the barrier below.
    float4* y4 = reinterpret_cast<float4*>(p.y);
    for (int i = cta * kTileThreads + tid; i < L * (d / 4); i += G * kTileThreads) y4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  __syncthreads();
  cluster_barrier();  // nobody sends into a CTA whose barriers are not initialised yet

  // the router row a worker owns in every layer (CTA r of the cluster: experts 8r .. 8r+7)
  const int my_e = (int)crank * kDecWarps + warp;
  const bool has_wr = warp < kDecWarps && my_e < N;
  const bool has_wp = p.prefetching && has_wr && cta < kDecCluster;  // (the first cluster computes the prefetch router)

  // attention stand-in: the CTA's bytes, in pieces of up to a tile
  const size_t attn_bytes = p.run_attn ? p.attn_bytes : 0;
  const size_t attn_per = ((attn_bytes + G - 1) / G + 127) / 128 * 128;
  const size_t attn_lo = attn_per * cta < attn_bytes ? attn_per * cta : attn_bytes;
  const size_t attn_n = attn_lo + attn_per < attn_bytes ? attn_per : attn_bytes - attn_lo;
  constexpr uint32_t piece_bytes = tile_bytes / 128 * 128;
  const int n_pieces = (int)((attn_n + piece_bytes - 1) / piece_bytes);

  // Row range of this CTA for the usual row space (k executed experts and the shared expert): the same in every layer
  const int std_total = k * I + ((p.shared_w && p.I_shared > 0) ? p.I_shared : 0);
  const unsigned pre_lo = tile_weight_prefix(cta, p.prefetching != 0), pre_hi = tile_weight_prefix(cta + 1, p.prefetching != 0);
  const unsigned pre_all = tile_weight_prefix(G, p.prefetching != 0);
  const int std_lo = (int)((unsigned long long)std_total * pre_lo / pre_all);
  const int std_n = (int)((unsigned long long)std_total * pre_hi / pre_all) - std_lo;
  const int std_pidx = std_lo < k * I ? std_lo / I : k;  // place of its first row
  const int std_i = std_lo - std_pidx * I;

  bool ok = true;  // false once a wait of this warp ran out
  unsigned long long waited = 0;
  uint32_t use = 0;       // planner: ring uses so far
  uint32_t piece = 0;     // planner: ring use of the next piece of the stand-in to land
  int n_ahead = 0;        // planner: stand-in pieces of the next layer already requested

  const Limits lim{&s_abort, p.abort_flag, p.mbox_status, p.wait_limit_ns};
  // warp-uniform: has a thread of this CTA given up (or learnt that another CTA did)?
  auto cta_stopped = [&]() -> bool { return __any_sync(0xffffffffu, *(volatile int*)&s_abort != 0); };
  // whole warp; `ok` tells whether it was met
  auto warp_wait = [&](uint64_t* bar, uint32_t parity) -> bool {
    if (!__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) ok = ok && warp_wait_on(bar, parity, lim);
    return ok;
  };
  auto warp_poll = [&](PollKind kind, const void* at, unsigned long long want, int pause_ns) -> bool {
    if (!__all_sync(0xffffffffu, lane != 0 || poll_met(kind, at, want))) {
      const long long ns = warp_poll_on(kind, at, want, pause_ns, lim);
      if (ns < 0) ok = false;
      else if (kind != kPollCount && kind != kPollSeq64) waited += (unsigned long long)ns;
    }
    __syncwarp();
    return ok;
  };
  auto wait_count = [&](const unsigned long long* ctr) -> bool { return warp_poll(kPollCount, ctr, p.bar_target, 20); };

  if (warp >= kDecWarps) {
    // ============================================================ planner and clerk
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kPlanRegs));
    if (warp > kGates || (warp == kClerk && !poster)) return;
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");  // (for the first layer's wait)
    const bool planner = warp == kPlanner, clerk = warp == kClerk;
    // ---- planner: the ring
    auto acquire = [&]() -> int {  // the next slot, free (-1: given up)
      const int s = (int)(use % NT);
      if (!warp_wait(&s_empty[s], ((use / NT) & 1u) ^ 1u)) return -1;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the slot has been read by threads
      return s;
    };
    auto request_piece = [&](int layer, int i) {  // piece i of the stand-in of `layer`, an eighth per lane
      const int s = acquire();
      if (s < 0) return;
      const size_t off = (size_t)i * piece_bytes;
      const uint32_t n = attn_n - off < piece_bytes ? (uint32_t)(attn_n - off) : piece_bytes;
      const uint32_t part = ((n + 7) / 8 + 15) / 16 * 16, lo = part * lane;
      if (lane == 0) mbar_expect_tx(&s_full[s], n);
      __syncwarp();
      if (lane < 8 && lo < n)
        bulk_g2s(smem + (size_t)s * tile_bytes + lo, p.attn + (size_t)(layer % p.attn_layers) * p.attn_bytes + attn_lo + off + lo, n - lo < part ? n - lo : part, &s_full[s]);
      ++use;
    };
    auto land_pieces = [&](uint32_t upto) {  // the stand-in's pieces, in order: landed, their slots free
      for (; ok && piece != upto; ++piece) {
        const int s = (int)(piece % NT);
        if (warp_wait(&s_full[s], (piece / NT) & 1u) && lane < kDecWarps) mbar_arrive(&s_empty[s]);
      }
    };
    auto request_pieces = [&](int layer, int from, int upto) {
      for (int i = from; i < upto && ok; ++i) {
        if (use - piece == NT) land_pieces(piece + 1);
        if (ok) request_piece(layer, i);
      }
    };
    for (int l = 0; l < L; ++l) {
      __syncwarp();
      const bool running = ok && !cta_stopped();  // per warp: skip the work, keep the barriers
      int ncand_p = 0;  // clerk: k + delta_hat
      DTL(0);
      const uint32_t lpar = (uint32_t)(l & 1);
      const float* hpl = p.hpost + (size_t)l * d;
      const unsigned long long* bar_prev_ffn = l > 0 ? p.bar + 2 * (l - 1) : nullptr;
      unsigned long long* bar_attn = p.bar + 2 * l + 1;
      if (planner) {
        // ================= planner
        // The stand-in is this layer's attention block: its window opens when the previous layer's y is complete.  (With
        // standin_ahead its bytes were requested earlier, while the previous layer was still finishing: the window then
        // overlaps that layer's tail -- including any wait for its experts -- which is not what Eq. (12) describes.)
        auto pass_previous = [&]() {
          if (!running || !ok || !bar_prev_ffn) return;
          if (wait_count(bar_prev_ffn) && lane == 0) mbar_arrive(&s_cbar[0]);
          DTL(15);
        };
        if (!p.standin_ahead) pass_previous();
        if (running && ok && p.run_attn) {
          if (n_ahead == 0) piece = use;
          request_pieces(l, n_ahead, n_pieces);
          land_pieces(use);
          DTL(3);
          // (nothing but the zeroes of y, before the first layer, is published by this count: the others need no fence, 0.5 us)
          if (ok && lane == 0) {
            if (l == 0) red_release_gpu_u64(bar_attn, 1ull);
            else red_relaxed_gpu_u64(bar_attn, 1ull);
          }
        }
        n_ahead = 0;
        if (p.standin_ahead) pass_previous();
        if (running && ok && p.run_attn && wait_count(bar_attn) && lane == 0) mbar_arrive(&s_cbar[1]);
      } else if (clerk) {
        float cw0 = 0.f, cw1 = 0.f, cth0 = 0.f, cth1 = 0.f;  // confidence model of this layer
        if (p.prefetching) {
          const float* wl = p.w + (size_t)l * N;
          const float* thl = p.theta + (size_t)l * (N - k + 1);
          if (lane < N) cw0 = __ldg(wl + lane);
          if (lane + 32 < N) cw1 = __ldg(wl + lane + 32);
          if (lane < N - k + 1) cth0 = __ldg(thl + lane);
          if (lane + 32 < N - k + 1) cth1 = __ldg(thl + lane + 32);
        }
        // softmax, ranking, budget, candidate set, as soon as the prefetch logits are complete
        if (p.prefetching && running && warp_wait(&s_xbar[0], lpar)) {
          const RankedLogits Rp = softmax_and_rank(s_zp, N, lane);
          const int e0 = lane, e1 = lane + 32;
          if (e0 < N) { s_q[e0] = Rp.q0; s_pi[Rp.r0] = e0; s_posp[e0] = Rp.r0; }
          if (e1 < N) { s_q[e1] = Rp.q1; s_pi[Rp.r1] = e1; s_posp[e1] = Rp.r1; }
          __syncwarp();
          const int pj0 = lane < N ? s_pi[lane] : -1, pj1 = lane + 32 < N ? s_pi[lane + 32] : -1;
          const float x0 = pj0 >= 0 ? s_q[pj0] : 0.f, x1 = pj1 >= 0 ? s_q[pj1] : 0.f;
          // the budget and the candidate mask, first of all for every other CTA (device memory) ...
          int uncapped;
          const int d_hat = select_budget_vals(cw0, cw1, cth0, cth1, p.t_tau, p.force, N, k, p.C, lane, x0, x1, &uncapped);
          ncand_p = k + d_hat;
          unsigned lo = 0, hi = 0;
          if (lane < ncand_p) { if (pj0 < 32) lo |= 1u << pj0; else hi |= 1u << (pj0 - 32); }
          if (lane + 32 < ncand_p) { if (pj1 < 32) lo |= 1u << pj1; else hi |= 1u << (pj1 - 32); }
          lo = __reduce_or_sync(0xffffffffu, lo);
          hi = __reduce_or_sync(0xffffffffu, hi);
          if (lane == 0) {
            p.cand_rec[2 * l] = ((unsigned long long)hi << 32) | lo;
            asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p.cand_rec + 2 * l + 1), "l"((unsigned long long)p.seq) : "memory");
          }
          DTL(2);
          // ... then the outputs of S1-S3, the counters and the record the host plans the copies from (one 16-byte store
          // to mapped memory; kept behind the release above, which would otherwise have to wait for it)
          if (e0 < N) { p.zp_out[e0] = Rp.z0; p.qp_out[e0] = Rp.q0; p.pi_out[Rp.r0] = e0; }
          if (e1 < N) { p.zp_out[e1] = Rp.z1; p.qp_out[e1] = Rp.q1; p.pi_out[Rp.r1] = e1; }
          SelectParams sp;
          sp.w = p.w + (size_t)l * N;
          sp.theta = p.theta + (size_t)l * (N - k + 1);
          sp.cand_out = p.cand_dev;
          sp.ncand_out = p.ncand_dev;
          sp.ncand_keep = p.ncand_keep;
          sp.mbox_cand = p.mbox[l].cand;
          sp.mbox_rec = p.mbox[l].sel_rec;
          sp.seq_value = p.seq;
          sp.stats = p.stats + l;
          sp.t_tau = p.t_tau;
          sp.force = p.force;
          sp.N = N; sp.k = k; sp.C = p.C; sp.B = 1;
          SelectVals sv;
          sv.w0 = cw0; sv.w1 = cw1; sv.th0 = cth0; sv.th1 = cth1;
          select_token(sp, sv, 0, lane, pj0, pj1, x0, x1);
          DTL(10);
        }
      }
      if (warp == kGates) {
        // ---- probabilities and gates of the executed experts, while the planner requests their rows
        if (running && warp_wait(&s_xbar[1], lpar)) {
          const int e0 = lane, e1 = lane + 32;
          const float NEG = -3.402823466e38f;
          RankedLogits Rg;
          Rg.z0 = e0 < N ? s_zr[e0] : NEG;
          Rg.z1 = e1 < N ? s_zr[e1] : NEG;
          softmax_lane_logits(N, lane, &Rg);
          if (p.shared_w && p.I_shared > 0) {  // the shared expert: weight 1, or its gate's value
            const float* wsg = p.shared_gate ? p.shared_gate[l] : nullptr;
            const float w = wsg ? shared_gate_weight(wsg, hpl, d, lane) : 1.f;
            if (lane == 0) s_gate[APEX_MAX_EXPERTS] = w;
          }
          for (int pass = 0; pass < 2; ++pass) {
            if (!warp_wait(pass == 0 ? &s_plan : &s_verdict, lpar) || (pass == 1 && !s_again)) break;
            float g0, g1;
            exec_gates(s_run[pass], e0 < N ? Rg.q0 : 0.f, e1 < N ? Rg.q1 : 0.f, p.norm_topk, lane, &g0, &g1);
            s_gate[e0] = g0;
            s_gate[e1] = g1;
            __syncwarp();
            if (lane == 0) mbar_arrive(&s_gbar[pass]);
          }
        }
      } else
      // ---- the plan: by the planner, which requests the rows, and by the clerk, which tells the host
      if (running && ok && !cta_stopped()) {
        // Slot table of this layer as it stood at launch, and the ready flags of its slots (none of this comes from earlier work of
        // this kernel: asked for while the ranks are waited for); lanes own experts lane and lane + 32.  Declared here and not
        // at the start of the layer: held across the logits these registers were spilled there.
        const SlotSnapshot* tab = p.tab + l;
        const uint32_t* slot_ready = p.slot_ready + (size_t)l * p.C;
        int sl0 = -1, sl1 = -1;
        uint32_t need0 = 0u, need1 = 0u, f0 = 0u, f1 = 0u;
        unsigned long long resident = 0ull;
        auto take_flags = [&]() {
          f0 = sl0 >= 0 ? ld_relaxed_sys(slot_ready + sl0) : 0u;
          f1 = sl1 >= 0 ? ld_relaxed_sys(slot_ready + sl1) : 0u;
        };
        if (lane < N) { sl0 = tab->expert_slot[lane]; need0 = tab->need_gen[lane]; }
        if (lane + 32 < N) { sl1 = tab->expert_slot[lane + 32]; need1 = tab->need_gen[lane + 32]; }
        resident = tab->resident_mask;
        take_flags();
        unsigned long long kr_mask = 0ull, run = 0ull, ready_mask = 0ull;
        RankedLogits Rg;
        Rg.z0 = Rg.z1 = Rg.q0 = Rg.q1 = 0.f;
        Rg.r0 = Rg.r1 = 0;
        // Which slot table?  The one the kernel was launched with is this step's table unless the host changes it, which it
        // does only if a candidate of this step is not resident (it then publishes the new table).  Whether that is so is
        // known once the poster's candidate mask has arrived -- a few microseconds after the gate on the hit path.  Where
        // the host expects no change for this layer (opt[l]: the layer's previous step copied nothing) the rows are requested from
        // the launch-time table at once; in the rare case that the table did change, what they gave is dropped and the layer's
        // rows are repeated with the published table.  Nothing is waited for (flag or demand copy) on an unconfirmed table.
        bool verified = !p.prefetching;  // the table at hand is known to be this step's
        bool changed = false;            // ... and it is not the launch-time table
        const bool optimistic = p.prefetching && p.cache_reuse && p.opt[l] != 0;
        const unsigned long long* cand_seq = p.cand_rec + 2 * l + 1;
        // whole warp: wait for the candidate mask, take this step's table (false: a wait ran out)
        auto confirm_table = [&]() -> bool {
          if (verified) return true;
          if (!warp_poll(kPollSeq64, cand_seq, (unsigned long long)p.seq, 40)) return false;
          (void)ld_acquire_gpu_u64(cand_seq);  // every lane: its read of the mask comes after the sequence word
          const unsigned long long cand = *(volatile const unsigned long long*)(p.cand_rec + 2 * l);
          verified = true;
          if (p.cache_reuse && (cand & ~resident) == 0ull) return true;  // every candidate was resident: nothing changes
          // The host publishes the new table in mapped host memory.  ONE warp of the grid reads it there and passes it on
          // through device memory: a poll of host memory is a read over the host link, and a hundred warps polling would
          // take the link away from the very copies they are waiting for.
          const DecodeHostSnap* hs = p.snap + l;
          DecodeHostSnap* ds_ = p.snap_dev + l;
          if (cta == 0 && planner) {
            if (!warp_poll(kPollSeqSys, &hs->seq, p.seq, 400)) return false;
            const volatile SlotSnapshot* vt = &hs->tab;
            if (lane < N) { ds_->tab.expert_slot[lane] = vt->expert_slot[lane]; ds_->tab.need_gen[lane] = vt->need_gen[lane]; }
            if (lane + 32 < N) { ds_->tab.expert_slot[lane + 32] = vt->expert_slot[lane + 32]; ds_->tab.need_gen[lane + 32] = vt->need_gen[lane + 32]; }
            if (lane == 0) ds_->tab.resident_mask = vt->resident_mask;
            __threadfence();
            __syncwarp();
            if (lane == 0) asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(&ds_->seq), "r"(p.seq) : "memory");
          }
          if (!warp_poll(kPollSeqGpu, &ds_->seq, p.seq, 200)) return false;
          (void)ld_acquire_gpu_u32(&ds_->seq);  // every lane: its reads of the table come after the sequence word
          const volatile SlotSnapshot* vt = &ds_->tab;
          sl0 = lane < N ? vt->expert_slot[lane] : -1;
          sl1 = lane + 32 < N ? vt->expert_slot[lane + 32] : -1;
          need0 = lane < N ? vt->need_gen[lane] : 0u;
          need1 = lane + 32 < N ? vt->need_gen[lane + 32] : 0u;
          resident = vt->resident_mask;
          take_flags();
          changed = true;
          return true;
        };
        // ranks (counted by the workers) -> K_r
        auto take_ranks = [&]() -> bool {
          if (!warp_wait(&s_rbar, lpar)) return false;
          const int e0 = lane, e1 = lane + 32;
          const float NEG = -3.402823466e38f;
          Rg.z0 = e0 < N ? s_zr[e0] : NEG;
          Rg.z1 = e1 < N ? s_zr[e1] : NEG;
          Rg.r0 = e0 < N ? (int)((s_rank[e0 >> 2] >> (8 * (e0 & 3))) & 0xffu) : N;
          Rg.r1 = e1 < N ? (int)((s_rank[e1 >> 2] >> (8 * (e1 & 3))) & 0xffu) : N;
          kr_mask = ((unsigned long long)__ballot_sync(0xffffffffu, e1 < N && Rg.r1 < k) << 32) | __ballot_sync(0xffffffffu, e0 < N && Rg.r0 < k);
          return true;
        };
        auto derive_sets = [&]() {  // from the current table: which slots are ready, which experts are executed
          const bool r0 = sl0 >= 0 && (int32_t)(f0 - need0) >= 0, r1 = sl1 >= 0 && (int32_t)(f1 - need1) >= 0;
          ready_mask = ((unsigned long long)__ballot_sync(0xffffffffu, r1) << 32) | __ballot_sync(0xffffffffu, r0);
          run = exec_set(kr_mask, p.mode, resident, Rg.z0, Rg.z1, lane);
        };
        if (take_ranks()) {
        if (!planner && lane == 0) {  // K_r does not depend on the table: the host gets it at once
          asm volatile("st.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p.mbox[l].kr_rec), "r"((uint32_t)kr_mask),
                       "r"((uint32_t)(kr_mask >> 32)), "r"(p.seq), "r"(0u)
                       : "memory");
          if (p.mode == APEX_MODE_EXACT)  // ... and in this mode neither does the execution set
            asm volatile("st.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p.mbox[l].exec_rec), "r"((uint32_t)kr_mask),
                         "r"((uint32_t)(kr_mask >> 32)), "r"(p.seq), "r"(0u)
                         : "memory");
        }
        bool confirm = !verified && !(planner && optimistic);
        for (int pass = 0;;) {
          if (confirm && !confirm_table()) break;
          if (pass == 1) {  // the rows have been requested from the launch-time table: does it hold?
            if (lane == 0) {
              s_again = changed ? 1 : 0;
              if (!changed) mbar_arrive(&s_verdict);
            }
            if (!changed) break;
          }
          derive_sets();
          if (planner && !verified && (run & ~ready_mask) != 0ull) {  // something to wait for: only on the confirmed table
            confirm = true;
            continue;
          }
          if (!planner) {
            const int e0 = lane, e1 = lane + 32;
            softmax_lane_logits(N, lane, &Rg);
            const size_t zo = (size_t)l * p.zr_stride;
            if (e0 < N) { p.zr_out[zo + e0] = Rg.z0; p.alpha_out[zo + e0] = Rg.q0; if (Rg.r0 < k) p.idx_out[(size_t)l * p.idx_stride + Rg.r0] = e0; }
            if (e1 < N) { p.zr_out[zo + e1] = Rg.z1; p.alpha_out[zo + e1] = Rg.q1; if (Rg.r1 < k) p.idx_out[(size_t)l * p.idx_stride + Rg.r1] = e1; }
            const bool in0 = e0 < N && Rg.r0 < k, in1 = e1 < N && Rg.r1 < k;
            int dstar = 0, hitsP = 0;
            if (p.prefetching) {
              const int pos0 = in0 ? s_posp[e0] : -1, pos1 = in1 ? s_posp[e1] : -1;
              dstar = warp_max_int(max(pos0, pos1)) + 1 - k;
              hitsP = __popc(__ballot_sync(0xffffffffu, in0 && pos0 < ncand_p)) + __popc(__ballot_sync(0xffffffffu, in1 && pos1 < ncand_p));
            }
            if (lane == 0) {
              if (p.mode != APEX_MODE_EXACT)
                asm volatile("st.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p.mbox[l].exec_rec), "r"((uint32_t)run), "r"((uint32_t)(run >> 32)),
                             "r"(p.seq), "r"(0u)
                             : "memory");
              DevStats* st = p.stats + l;
              atomicAdd(&st->routed, (unsigned long long)k);
              if (p.prefetching) {
                atomicAdd(&st->sum_delta_star, (unsigned long long)dstar);
                atomicAdd(&st->hits_P, (unsigned long long)hitsP);
                atomicAdd(&st->covered, (unsigned long long)(hitsP == k ? 1 : 0));
              }
              const int ns = __popcll(run & ~kr_mask);
              if (ns) atomicAdd(&st->substitutions, (unsigned long long)ns);
              atomicAdd(&st->hits_R, (unsigned long long)__popcll(kr_mask & resident));
            }
            break;
          }
          // row space of the expert FFN: executed experts in ascending index, then the shared expert
          const uint8_t* shared_w = (p.shared_w && p.I_shared > 0) ? p.shared_w[l] : nullptr;
          const uint8_t* cache_l = p.cache + (size_t)l * p.C * p.slot_stride;
          const int n_routed = __popcll(run);
          const int total = n_routed * I + (shared_w ? p.I_shared : 0);
          int lo = std_lo, n = std_n, pidx = std_pidx, i = std_i;
          if (total != std_total) {  // fewer experts executed than k: the range is worked out for this row count
            lo = (int)((unsigned long long)total * pre_lo / pre_all);
            n = (int)((unsigned long long)total * pre_hi / pre_all) - lo;
            pidx = min(lo / I, n_routed);
            i = lo - pidx * I;
          }
          const int pos_e = lane < n_routed ? nth_set_bit64(run, lane) : -1;
          const int tiles = (n + kRows - 1) / kRows;
          DTL(6);
          if (lane == 0) {
            s_use[pass] = (int)use;
            s_rows[pass] = n;
            s_run[pass] = run;
            mbar_arrive(pass == 0 ? &s_plan : &s_verdict);
          }
          if (pass == 0 && !warp_wait(&s_hbar, lpar)) break;
          const bool all_ready = (run & ~ready_mask) == 0ull;
          bool fresh = true;
          int e = N;                      // expert of the tile's first row
          const uint8_t* base = nullptr;  // its rows
          for (int q = 0; q < tiles && ok; ++q) {
            const int here = n - q * kRows < kRows ? n - q * kRows : kRows;
            for (; pidx < n_routed && i >= I; i -= I, ++pidx) fresh = true;
            if (fresh) {
              fresh = false;
              e = pidx < n_routed ? __shfl_sync(0xffffffffu, pos_e, pidx & 31) : N;
              const int slot = __shfl_sync(0xffffffffu, e < 32 ? sl0 : sl1, e & 31);
              base = e < N ? cache_l + (size_t)slot * p.slot_stride : shared_w;
            }
            const int s = (int)(use % NT);
            if (all_ready && (e == N || i + here <= I)) {
              // the usual case: rows that follow one another.  Issued by one elected lane from warp-uniform registers: as a copy per
              // lane the eight were 650 cycles of a tile
              if (acquire() < 0) break;
              const uint8_t* src = base + (size_t)i * entry_bytes;
              uint8_t* dst = smem + (size_t)s * tile_bytes;
              if (lane < kRows) s_exp[s * kRows + lane] = (uint8_t)e;
              __syncwarp();
              if (elect_one()) {
                mbar_expect_tx(&s_full[s], here * entry_bytes);
#pragma unroll
                for (int r = 0; r < kRows; ++r)
                  if (r < here) bulk_g2s(dst + r * stride, src + (size_t)r * entry_bytes, entry_bytes, &s_full[s]);
              }
              __syncwarp();
            } else {
              // rows of several experts, or experts to be waited for: a row per lane
              int li = i + lane, lp = pidx;
              while (__any_sync(0xffffffffu, lane < here && lp < n_routed && li >= I)) {
                const bool over = lp < n_routed && li >= I;
                li -= over ? I : 0;
                lp += over ? 1 : 0;
              }
              const int at_e = __shfl_sync(0xffffffffu, pos_e, lp & 31);
              const int le = lp < n_routed ? at_e : N;
              const bool in = lane < here && le < N;
              const unsigned long long wanted = ((unsigned long long)__reduce_or_sync(0xffffffffu, in && le >= 32 ? 1u << (le - 32) : 0u) << 32) |
                                                __reduce_or_sync(0xffffffffu, in && le < 32 ? 1u << le : 0u);
              for (unsigned long long rest = wanted & ~ready_mask; rest && ok; rest &= rest - 1) {
                const int w = __ffsll((long long)rest) - 1;
                int slot = __shfl_sync(0xffffffffu, w < 32 ? sl0 : sl1, w & 31);
                const uint32_t need = __shfl_sync(0xffffffffu, w < 32 ? need0 : need1, w & 31);
                // not resident when the table was taken: the host fetches it on demand and publishes (tag, slot)
                // after the copy -- asynchronous miss correction inside the launch (exact mode only)
                const bool missing = slot < 0;
                const uint32_t* word = missing ? p.demand + (size_t)l * N + w : slot_ready + slot;
                if (!warp_poll(missing ? kPollTag : kPollGen, word, missing ? p.demand_tag : need, 64)) break;
                if (missing) {
                  slot = __shfl_sync(0xffffffffu, (int)(ld_acquire_sys(word) & 0xffu), 0);
                  if (slot >= p.C) {  // a published slot outside the cache: refuse
                    if (lane == 0) give_up(lim);
                    ok = false;
                    break;
                  }
                  if (lane == (w & 31)) (w < 32 ? sl0 : sl1) = slot;
                }
                ready_mask |= 1ull << w;
                asm volatile("fence.proxy.async;" ::: "memory");
              }
              if (!ok || acquire() < 0) break;
              const int slot0 = __shfl_sync(0xffffffffu, sl0, le & 31), slot1 = __shfl_sync(0xffffffffu, sl1, le & 31);
              const uint8_t* row = (le < N ? cache_l + (size_t)(le < 32 ? slot0 : slot1) * p.slot_stride : shared_w) + (size_t)li * entry_bytes;
              if (lane < here) s_exp[s * kRows + lane] = (uint8_t)le;
              __syncwarp();
              if (lane == 0) mbar_expect_tx(&s_full[s], here * entry_bytes);
              __syncwarp();
              if (lane < here) bulk_g2s(smem + (size_t)s * tile_bytes + lane * stride, row, entry_bytes, &s_full[s]);
              fresh = true;  // (slots may have been filled in)
            }
            ++use;
            i += kRows;
          }
          if (!ok || pass == 1) break;
          if (verified) {
            if (lane == 0) {
              s_again = 0;
              mbar_arrive(&s_verdict);
            }
            break;
          }
          pass = 1;
          confirm = true;
        }
        }
        if (!planner) waited = 0;  // (the planners count)
      }
      if (planner) {
        if (lane == 0 && waited) atomicAdd(&p.stats[l].stall_ns, waited * (unsigned long long)p.n_sm / (unsigned long long)G);  // the host divides by the SM count
        waited = 0;
        if (p.standin_ahead && ok && l + 1 < L && !cta_stopped()) {
          piece = use;
          n_ahead = n_pieces < NT ? n_pieces : NT;
          request_pieces(l + 1, 0, n_ahead);
        }
      }
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // (the barriers of the layer's end, see the workers)
      cluster_barrier();
      asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    }
    // nothing may be in flight into this CTA's shared memory when it leaves
    for (uint32_t t = use > NT ? use - NT : 0u; t != use; ++t) mbar_wait(&s_full[t % NT], (t / NT) & 1u, nullptr, p.wait_limit_ns);
  } else {
    // ============================================================ workers
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kWorkRegs));
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");  // (for the first layer's wait)
    // ---- workers: a barrier at which all of them learn that one has given up.  A word per parity: what a warp raises for the next
    // barrier, past this one, is not taken for this one's.
    uint32_t votes = 0;
    bool halted = false;
    auto halt = [&](bool failed) -> bool {
      if (failed && lane == 0) *(volatile int*)&s_stop[votes & 1u] = 1;
      workers_barrier();
      halted = __any_sync(0xffffffffu, *(volatile int*)&s_stop[votes & 1u] != 0);
      ++votes;
      return halted;
    };
    // Router rows (a worker's, one of W_p and one of W_r per layer): up to d = 1024 in registers from the start of the layer,
    // wider ones prefetched into L2 there and read when the dot product is taken (two rows of d = 1536 held from the start of the
    // layer cost the rows more than the loads cost the logits, 19.3 against 17.2 us per layer in the row-per-warp kernel; two of
    // d = 2048 spilled); the gate's row of d = 1536 comes into registers right before the wait for the attention window (+ 3 %).
    constexpr int NVRP = NV <= 8 ? NV : 1;   // prefetch-router row
    constexpr int NVRR = NV <= 12 ? NV : 1;  // gate row
    constexpr bool WR_LATE = NV > 8 && NV <= 12;
    auto load_row = [&](const float* __restrict__ W_row, auto& wr) {
      constexpr int NVR = (int)(sizeof(wr) / sizeof(float4));
      constexpr bool ROW_REGS = NVR > 1 || NV == 1;
      if (!ROW_REGS) return;
      const float4* rp = reinterpret_cast<const float4*>(W_row);
  #pragma unroll
      for (int i = 0; i < NVR; ++i)  // volatile: keep the loads here, ahead of the waits
        asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(wr[i].x), "=f"(wr[i].y), "=f"(wr[i].z), "=f"(wr[i].w) : "l"(rp + i * 32 + lane));
    };
    // dot product of the row with x (reduction order of router_kernel), plus bias; sent to CTAs [rank_lo, rank_hi) of the cluster
    auto row_logit = [&](const float* __restrict__ W_row, const auto& wr, bool held, const float* __restrict__ x, float bias, float* zs,
                         uint64_t* xbar, int rank_lo, int rank_hi) {
      constexpr int NVR = (int)(sizeof(wr) / sizeof(float4));
      constexpr bool ROW_REGS = NVR > 1 || NV == 1;
      const float4* __restrict__ xv = reinterpret_cast<const float4*>(x);
      const float4* __restrict__ rp = reinterpret_cast<const float4*>(W_row);
      float acc = 0.f;
      if (ROW_REGS && held) {
        float4 xr[NVR];
  #pragma unroll
        for (int i = 0; i < NVR; ++i) xr[i] = __ldg(xv + i * 32 + lane);
  #pragma unroll
        for (int i = 0; i < NVR; ++i) {
          acc = fmaf(wr[i].x, xr[i].x, acc);
          acc = fmaf(wr[i].y, xr[i].y, acc);
          acc = fmaf(wr[i].z, xr[i].z, acc);
          acc = fmaf(wr[i].w, xr[i].w, acc);
        }
      } else {
  #pragma unroll 8
        for (int i = 0; i < NV; ++i) {
          const float4 wv = __ldg(rp + i * 32 + lane);
          const float4 v = __ldg(xv + i * 32 + lane);
          acc = fmaf(wv.x, v.x, acc);
          acc = fmaf(wv.y, v.y, acc);
          acc = fmaf(wv.z, v.z, acc);
          acc = fmaf(wv.w, v.w, acc);
        }
      }
      acc = warp_sum_tree(acc);
      const float z = acc + bias;
      if (lane >= rank_lo && lane < rank_hi) st_async_remote(&zs[my_e], xbar, (uint32_t)lane, z);
    };
    auto prefetch_l2 = [&](const void* ptr) { asm volatile("prefetch.global.L2 [%0];" ::"l"(ptr)); };
    uint32_t repeats = 0;  // layers whose rows were repeated so far
    RowTiles<d, FMT> rt;
    for (int l = 0; l < L; ++l) {
      __syncwarp();
      const bool running = ok && !cta_stopped();  // per warp: skip the work, keep the barriers
      DTL(0);
      const uint32_t lpar = (uint32_t)(l & 1);
      const float* hl = p.h + (size_t)l * d;
      const float* hpl = p.hpost + (size_t)l * d;
      const unsigned long long* bar_prev_ffn = l > 0 ? p.bar + 2 * (l - 1) : nullptr;
      unsigned long long* bar_ffn = p.bar + 2 * l;
      bool rows_kept = false;  // this CTA's sums are to be added to y
      if (tid == 0 && !*(volatile int*)&s_abort) {  // arm this layer's exchange barriers: N logits of 4 bytes each
        if (p.prefetching && poster) mbar_expect_tx(&s_xbar[0], (uint32_t)N * 4u);
        mbar_expect_tx(&s_xbar[1], (uint32_t)N * 4u);
      }
      // parameters of this layer this warp will need: fetched now, used after the waits
      float bias_p = 0.f, bias_r = 0.f;
      float4 wp_row[NVRP], wr_row[NVRR];
      const float* Wp_row = p.W_p + ((size_t)l * N + (has_wr ? my_e : 0)) * d;
      const float* Wr_row = p.W_r + ((size_t)l * N + (has_wr ? my_e : 0)) * d;
      if (has_wp) load_row(Wp_row, wp_row);
      if (has_wr && !has_wp && !WR_LATE) load_row(Wr_row, wr_row);  // (a warp with both rows fetches W_r after its W_p dot product)
      if (has_wr) {
        if (has_wp) bias_p = __ldg(p.b_p + (size_t)l * N + my_e);
        bias_r = __ldg(p.b_r + (size_t)l * N + my_e);
        // x of the two dot products: brought into L2 ahead of time (in a model the previous layer has just written it there)
        if ((lane & 7) == 0) {
#pragma unroll
          for (int i = 0; i < NV; ++i) {
            if (has_wp) prefetch_l2(reinterpret_cast<const float4*>(hl) + i * 32 + lane);
            prefetch_l2(reinterpret_cast<const float4*>(hpl) + i * 32 + lane);
            // ... and so are the router rows that are not held in registers
            if (NVRP == 1 && NV > 1 && has_wp) prefetch_l2(reinterpret_cast<const float4*>(Wp_row) + i * 32 + lane);
            if (NVRR == 1 && NV > 1) prefetch_l2(reinterpret_cast<const float4*>(Wr_row) + i * 32 + lane);
          }
        }
      }
      // prefetch router first of all: the sooner the candidate set is out, the more of the window the copies can use
      if (has_wp && running && (!bar_prev_ffn || warp_wait(&s_cbar[0], (uint32_t)((l - 1) & 1)))) {
        row_logit(Wp_row, wp_row, true, hl, bias_p, s_zp, &s_xbar[0], kDecCluster - 1, kDecCluster);  // to the poster only
        DTL(1);
        if (!WR_LATE) load_row(Wr_row, wr_row);
      }
      // exact gate: this warp's logit, once the whole stand-in has been streamed (a real attention block would only then
      // have produced h') and the previous layer's y is complete
      if (has_wr && ok && !cta_stopped()) {
        // (a wide gate row comes into registers only now, from L2: its latency passes while the counters are waited for)
        if (WR_LATE && p.run_attn) load_row(Wr_row, wr_row);  // (without a window to wait for, the row is read with x)
        bool go = true;
        if (p.run_attn) go = warp_wait(&s_cbar[1], lpar);
        else if (bar_prev_ffn && !has_wp) go = warp_wait(&s_cbar[0], (uint32_t)((l - 1) & 1));
        if (go) {
          DTL(14);
          row_logit(Wr_row, wr_row, !WR_LATE || p.run_attn != 0, hpl, bias_r, s_zr, &s_xbar[1], 0, kDecCluster);
          DTL(4);
        }
      }
      typename RowTiles<d, FMT>::Raw h_raw;  // this lane's share of h' for the expert rows
      RowTiles<d, FMT>::ask_h(h_raw, hpl, warp, lane);
      if (ok && !cta_stopped() && warp_wait(&s_xbar[1], lpar)) {
        DTL(5);
        // Ranks by counting, the count shared by the CTA's warps: warp w compares every logit with the logits of experts
        // w, w + 8, ... only and adds its counts up in shared memory.
        const int e0 = lane, e1 = lane + 32;
        const float NEG = -3.402823466e38f;
        const float z0 = e0 < N ? s_zr[e0] : NEG, z1 = e1 < N ? s_zr[e1] : NEG;
        int c0 = 0, c1 = 0;
        for (int f = warp; f < N; f += kDecWarps) {
          const float zf = s_zr[f];
          c0 += (zf > z0 || (zf == z0 && f < e0)) ? 1 : 0;
          c1 += (zf > z1 || (zf == z1 && f < e1)) ? 1 : 0;
        }
        // (counts stay below N <= 64: no carry between the bytes of a word)
        if (e0 < N && c0) atomicAdd(s_rank + (e0 >> 2), (unsigned)c0 << (8 * (e0 & 3)));
        if (e1 < N && c1) atomicAdd(s_rank + (e1 >> 2), (unsigned)c1 << (8 * (e1 & 3)));
        __syncwarp();
        if (lane == 0) mbar_arrive(&s_rbar);
        // h' goes to the MMA's operand layout through the ring, which is empty: the stand-in has landed (the logits of this cluster
        // were behind its count), and the planner asks for rows only when every worker has arrived below
        rt.take_h(h_raw, smem, warp, lane);
        __syncwarp();
        if (lane == 0) mbar_arrive(&s_hbar);
      }
      // ---- the expert rows
      if (!halted) {
        bool met = ok && warp_wait(&s_plan, lpar) && warp_wait(&s_gbar[0], lpar);
        for (int pass = 0; pass < 2 && !halt(!met); ++pass) {
          rt.clear();
          const int n = s_rows[pass], tiles = (n + kRows - 1) / kRows;
          uint32_t s = (uint32_t)s_use[pass] % NT, par = ((uint32_t)s_use[pass] / NT) & 1u;
          const int row = lane & (kRows - 1);
          for (int q = 0; q < tiles; ++q) {
            const int here = n - q * kRows < kRows ? n - q * kRows : kRows;
            const uint32_t tile = smem_u32(smem) + s * tile_bytes;
            float* part = s_part[q & 1];
            const bool landed = warp_wait(&s_full[s], par);
            if (q == 0 && pass == 0) DTL(7);
            float2* share = reinterpret_cast<float2*>(part + (lane >> 2) * kPartStride + 2 * warp);
            constexpr int kShare8 = 8 * kPartStride / 2;  // (eight rows on)
            [[maybe_unused]] typename RowTiles<d, FMT>::template Scales<kRows> scales;
            if (landed) {
              bool fp32 = false;  // the planes do not hold all of h' or of the gate and up rows
              if constexpr (FMT != kFmtBf16) {
                scales = rt.template scales_of<kRows>(tile, stride, warp, lane, here);
                fp32 = rt.template needs_fp32<kRows>(tile, stride, warp, lane, here);
              }
#pragma unroll
              for (int r = 0; r < R; ++r) {
                float g, u;
                if constexpr (FMT == kFmtBf16) rt.gate_up(tile + (lane & 7) * stride + r * 8 * stride, warp, lane, g, u);
                else rt.gate_up(tile + r * 8 * stride, stride, warp, lane, g, u);
                if ((lane & 3) == 0) share[r * kShare8] = make_float2(g, u);
              }
              if constexpr (FMT != kFmtBf16) {
                if (fp32) {
#pragma unroll 1
                  for (int r = 0; r < R; ++r) {
                    const float2 gu = rt.gate_up_fp32(smem + s * tile_bytes + r * 8 * stride, stride, warp, lane, hpl);
                    if ((lane & 3) == 0) share[r * kShare8] = gu;
                  }
                }
              }
            }
            // (behind the last tile's barrier everybody knows whether the rows are to be repeated)
            const bool last = pass == 0 && q + 1 == tiles;
            if (halt(!landed || (last && !warp_wait(&s_verdict, lpar)))) break;
            const int e = row < here ? (int)s_exp[s * kRows + row] : N;
            const float gate = s_gate[e < N ? e : APEX_MAX_EXPERTS];
            float g, u;
            sum_shares(part, row, g, u);
            if constexpr (FMT == kFmtBf16) {
              float a = gate * g * __frcp_rn(1.f + expf(-g)) * u;
              a = row < here ? a : 0.f;
#pragma unroll
              for (int r = 0; r < R; ++r) {
                const int k0 = r * 8 + 2 * (lane & 3);
                const float a0 = __shfl_sync(0xffffffffu, a, k0), a1 = __shfl_sync(0xffffffffu, a, k0 + 1);
                rt.down(tile + ((lane & 7) + r * 8) * stride, warp, lane, a0, a1, here - k0, here == kRows);
              }
            } else {
              float a = rt.gated(smem + s * tile_bytes + row * stride, gate, g, u);
              a = row < here ? a : 0.f;
              uint32_t b[R];
              int reach;
              const float unit = rt.template take_a<kRows>(a, s_planes[warp], lane, b, reach);
              rt.template down<kRows>(smem + s * tile_bytes, tile, stride, warp, lane, b, unit, here, a, reach, scales);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&s_empty[s]);
            if (++s == NT) {
              s = 0;
              par ^= 1u;
            }
          }
          if (pass == 0 && tiles == 0 && !halted) halt(!warp_wait(&s_verdict, lpar));
          if (halted) break;
          rows_kept = true;
          if (pass == 1 || !s_again) break;
          met = warp_wait(&s_gbar[1], repeats++ & 1u);
        }
        if (halted) rows_kept = false;
      }
      DTL(8);
    // ------------------------------------------------------------ y: workers -> cluster -> memory; count the CTA in
    // (a tile's warps have their own columns of y: nothing to add up inside the CTA)
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // the peers have read the sums of the layer before
    if (!rows_kept) rt.clear();
    rt.store(reinterpret_cast<float*>(part4), warp, lane);
    DTL(11);
    cluster_barrier();  // every CTA's partial y is complete
    DTL(12);
    if (tid < APEX_MAX_EXPERTS / 4) s_rank[tid] = 0u;  // (read by now; the next layer adds to zeros)
    if (tid < SLICE4) {
      // CTA r of the cluster adds columns [r * d/8, (r+1) * d/8) of the cluster's eight partial vectors to y
      const int col4 = (int)crank * SLICE4 + tid;
      float4 sacc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (uint32_t r = 0; r < (uint32_t)kDecCluster; ++r) {
        uint32_t ra;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(smem_u32(part4 + col4)), "r"(r));
        float4 v;
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(ra) : "memory");
        sacc.x += v.x; sacc.y += v.y; sacc.z += v.z; sacc.w += v.w;
      }
      atomicAdd(reinterpret_cast<float4*>(p.y + (size_t)l * d) + col4, sacc);
    }
    workers_barrier();
    DTL(13);
    // This CTA's part of y[l] is in memory: first of all, as everybody's next layer waits for it.  The barrier behind it says that
    // the peers' partial sums have been read and publishes nothing (a release there took 0.5 us of the count's way).
    if (tid == 0) red_release_gpu_u64(bar_ffn, 1ull);
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    DTL(9);
  }

  }
  if (lane == 0 && !ok) atomicAdd(&p.stats[0].timeouts, 1ull);
  if (tid == 0 && *(volatile int*)&s_abort) __threadfence_system();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  cluster_barrier();  // nobody leaves while a peer may still send into (or read from) its shared memory
  SPAN_END(10);
}

// ---------------------------------------------------------------- host side
namespace {

template <int NCH, int FMT>
cudaError_t launch_tiles_t(const DecodeParams& p, int n_clusters, cudaStream_t s, int* max_clusters_out) {
  constexpr int d = NCH * 256;
  const size_t smem = (size_t)tile_ring(FMT, d) * tile_blocks(FMT, d) * 8 * tile_stride(fmt_entry_bytes(FMT, d)) + (size_t)d * sizeof(float);  // ring, then the CTA's partial y
  static bool configured[kMaxDevices] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  if (!configured[dev]) {
    e = cudaFuncSetAttribute(decode_tiles_kernel<NCH, FMT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    configured[dev] = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kTileThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kDecCluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeCooperative;  // all CTAs resident together: they wait for one another
  attr[1].val.cooperative = 1;
  cfg.attrs = attr;
  if (max_clusters_out) {
    cfg.gridDim = dim3(kDecCluster, 1, 1);
    cfg.numAttrs = 1;
    int n = 0;
    e = cudaOccupancyMaxActiveClusters(&n, decode_tiles_kernel<NCH, FMT>, &cfg);
    *max_clusters_out = e == cudaSuccess ? n : 0;
    return e;
  }
  cfg.gridDim = dim3(kDecCluster * n_clusters, 1, 1);
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, decode_tiles_kernel<NCH, FMT>, p);
}

template <int FMT>
cudaError_t launch_quantised(const DecodeParams& p, int n_clusters, cudaStream_t s, int* max_clusters_out) {
  switch (p.d) {
    case 512: return launch_tiles_t<2, FMT>(p, n_clusters, s, max_clusters_out);
    case 1024: return launch_tiles_t<4, FMT>(p, n_clusters, s, max_clusters_out);
    case 1536: return launch_tiles_t<6, FMT>(p, n_clusters, s, max_clusters_out);
    case 2048: return launch_tiles_t<8, FMT>(p, n_clusters, s, max_clusters_out);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

bool decode_in_tiles(int d) { return d <= 2048; }

cudaError_t launch_decode_tiles(const DecodeParams& p, int n_clusters, cudaStream_t s, int* max_clusters_out) {
  if (p.fmt == kFmtE4m3) return launch_quantised<kFmtE4m3>(p, n_clusters, s, max_clusters_out);
  if (p.fmt == kFmtMxfp4) return launch_quantised<kFmtMxfp4>(p, n_clusters, s, max_clusters_out);
  switch (p.d) {
    case 256: return launch_tiles_t<1, kFmtBf16>(p, n_clusters, s, max_clusters_out);
    case 512: return launch_tiles_t<2, kFmtBf16>(p, n_clusters, s, max_clusters_out);
    case 768: return launch_tiles_t<3, kFmtBf16>(p, n_clusters, s, max_clusters_out);
    case 1024: return launch_tiles_t<4, kFmtBf16>(p, n_clusters, s, max_clusters_out);
    case 1536: return launch_tiles_t<6, kFmtBf16>(p, n_clusters, s, max_clusters_out);
    case 2048: return launch_tiles_t<8, kFmtBf16>(p, n_clusters, s, max_clusters_out);
  }
  return cudaErrorInvalidValue;
}

}  // namespace apex
