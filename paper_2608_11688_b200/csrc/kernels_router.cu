// Router kernels: the prefetch router and the exact gate share one GEMV + softmax + ranking kernel
// (Sec. IV-D: the prefetch router mirrors the original router), plus the budget selection of
// Eq. (8)-(9) and the stand-in attention stream that provides the hiding window of Eq. (12).
//
// Reduction order (fixed, so results are reproducible run to run): a dot product of length d is
// split over the 32 lanes of one warp; lane l accumulates float4 columns l, l+32, l+64, ... in
// ascending order with fused multiply-adds (x, y, z, w of each float4 in that order), then the 32
// partial sums are combined by a 5-step xor-shuffle tree (offsets 16, 8, 4, 2, 1).
#include <cooperative_groups.h>

#include <mutex>

#include "apex_internal.hpp"
#include "ptx.cuh"

namespace apex {
#ifdef APEX_TIMELINE
__device__ long long g_router_tl[16];
#define RTL(i) do { if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) g_router_tl[i] = clock64(); } while (0)
extern "C" int apex_debug_read_router_tl(long long* host) { return (int)cudaMemcpyFromSymbol(host, g_router_tl, sizeof(long long) * 16); }
#else
#define RTL(i) do { } while (0)
#endif
}  // namespace apex

#include "router_common.cuh"

namespace cg = cooperative_groups;

namespace apex {

constexpr int kRouterMaxVec = 32;  // float4 per lane of one weight row: d <= 4096


__global__ void __launch_bounds__(256) router_kernel(const RouterParams p) {
  SPAN_BEGIN();
  cg::cluster_group cluster = cg::this_cluster();
  const unsigned crank = cluster.block_rank();
  const int b = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __shared__ __align__(16) float zs[APEX_MAX_EXPERTS];
  __shared__ float qs[APEX_MAX_EXPERTS];
  __shared__ int pis[APEX_MAX_EXPERTS];
  __shared__ int posp[APEX_MAX_EXPERTS];
  __shared__ float4 xs[kRouterMaxVec * 32];

  // The router weights are parameters, not results of the preceding kernel: this warp's row is
  // loaded into registers before the dependency wait, so its DRAM latency hides behind that kernel.
  const int e = (int)crank * p.warps_per_cta + warp;
  const bool active = warp < p.warps_per_cta && e < p.N;
  const int nv = p.d >> 2;
  float4 wreg[kRouterMaxVec];
  float bias_e = 0.f;
  if (active) {
    const float4* __restrict__ Wrow = reinterpret_cast<const float4*>(p.W + (size_t)e * p.d);
#pragma unroll
    for (int i = 0; i < kRouterMaxVec; ++i) {
      const int c = i * 32 + lane;
      if (c < nv) wreg[i] = __ldg(Wrow + c);
    }
    if (p.bias) bias_e = __ldg(p.bias + e);
  }
  EpilogueVals ev;
  if (p.fuse_select && crank == 0 && warp == 0) ev.sel = load_select_vals(p.sel, lane);
  RTL(0);
  pdl_wait();               // everything queued before this kernel is complete: x may be read
  pdl_launch_dependents();  // the next kernel may begin its own prologue
  RTL(1);
  if (crank == 0 && warp == 0) load_prediction(p, b, lane, &ev);

  // x is staged in shared memory by the whole CTA in one round of loads
  {
    const float4* __restrict__ xv = reinterpret_cast<const float4*>(p.x + (size_t)b * p.d);
    for (int c = threadIdx.x; c < nv; c += blockDim.x) xs[c] = __ldg(xv + c);
  }
  __syncthreads();
  if (active) {
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < kRouterMaxVec; ++i) {
      const int c = i * 32 + lane;
      if (c < nv) {
        const float4 x = xs[c];
        acc = fmaf(wreg[i].x, x.x, acc);
        acc = fmaf(wreg[i].y, x.y, acc);
        acc = fmaf(wreg[i].z, x.z, acc);
        acc = fmaf(wreg[i].w, x.w, acc);
      }
    }
    acc = warp_sum_tree(acc);
    if (lane == 0) {
      const float z = acc + bias_e;
      float* dst = cluster.map_shared_rank(zs, 0);
      dst[e] = z;
    }
  }
  RTL(2);
  cluster.sync();
  RTL(3);
  if (crank != 0 || warp != 0) return;

  // ---- leader warp
  router_epilogue(p, ev, b, lane, zs, qs, pis, posp);
  SPAN_END((p.fuse_select || !p.topk_out || !p.stats) ? 1 : 4);
}

// Streams the bytes of an attention block once, through shared memory by bulk copies: four threads keep a 16 KB copy
// each in flight (64 KB per SM, 9.5 MB on the GPU against the 8 MB that latency times bandwidth asks for).  Few
// registers and 64 KB, so a router's CTAs fit beside it; as 512-thread CTAs with loads in registers it took 12 to 17 us for the
// 42 MB of d = 2048, and no router fitted beside two of them.
constexpr int kAttnChunk = 16 * 1024, kAttnWarps = 4;

// one of kAttnWarps warps of CTA `cta` of `ctas`; buf: its kAttnChunk bytes
__device__ __forceinline__ void attn_stream(const AttnParams& p, uint8_t* buf, uint64_t* bar, int warp, int lane, int cta, int ctas) {
  if (lane != 0) return;
  uint32_t parity = 0;
  const size_t stride = (size_t)ctas * kAttnWarps * kAttnChunk;
  for (size_t off = ((size_t)warp * ctas + cta) * kAttnChunk; off < p.bytes; off += stride, parity ^= 1u) {
    const uint32_t n = p.bytes - off < (size_t)kAttnChunk ? (uint32_t)(p.bytes - off) : (uint32_t)kAttnChunk;
    mbar_expect_tx(bar, n);
    bulk_g2s(buf, p.buf + off, n, bar);
    if (!mbar_wait(bar, parity, nullptr, 2000000000ll)) {  // (bounded like every wait; a copy of this GPU's own memory)
      *(volatile unsigned*)p.status = 1u;
      break;
    }
  }
}

// The same for a batch (B > 1): a cluster takes TT tokens, its CTA r the experts r * wpc .. r * wpc + wpc - 1 (wpc <= 8).
// Rows of W and of x come into shared memory by bulk copies in chunks of 512 or 1024 columns, two buffers (the W rows are
// parameters and are asked for before the dependency wait).  A warp takes a tile of tokens x experts with its lanes along
// the columns: per (token, expert) every lane runs the multiply-add chain of router_kernel and the lanes are added by the
// same xor tree -- halving the set of values a lane keeps at every level, which pairs the same partial sums -- so the
// logits have the same bits.  Each token's logits go to one CTA of the cluster, whose warps finish the tokens.
//
// Bound by latency: two rounds of loads, 16 multiply-adds per lane, token and expert at d = 2048, one cluster barrier, a
// serial epilogue.  As one token per pass over register-held rows it took 29 us at B = 256, N = 60, d = 2048.
// columns per chunk: with 512 two of the largest CTAs share an SM (a GPU holds 15 clusters of eight CTAs, one to an SM, and
// 16 are needed at B = 256: the last one ran behind the others)
// (The gate and the prefetch stage share a kernel on purpose: with one of its own each, for chunks of 1 024 columns at eight tokens,
// the second came upon cold instructions and a layer took 2 to 3 us more.)
__host__ __device__ constexpr int router_chunk(int tt) { return tt >= 8 ? 512 : 1024; }
__host__ __device__ constexpr int router_smem(int tt) { return 2 * (tt + 8) * router_chunk(tt) * (int)sizeof(float); }
static_assert(router_smem(1) >= kAttnWarps * kAttnChunk && router_smem(8) >= kAttnWarps * kAttnChunk, "a CTA of the stand-in runs in a router CTA's shared memory");
constexpr int kRouterWarps = 8;

__host__ __device__ constexpr int router_tile_tok(int tt) { return tt < 4 ? tt : 4; }
__host__ __device__ constexpr int router_tile_exp(int tt) { return tt <= 4 ? 1 : tt / 4; }

// What a token gets whose logits could not be computed: nothing that looks like a routing.  No record goes to the host, which
// stops waiting for it when it sees the status.
__device__ __forceinline__ void router_failed(const RouterParams& p, int b, int lane) {
  for (int e = lane; e < p.N; e += 32) {
    p.z_out[(size_t)b * p.N + e] = p.q_out[(size_t)b * p.N + e] = __int_as_float(0x7fffffff);
    if (p.pi_out) p.pi_out[(size_t)b * p.N + e] = e;  // (the gate indexes with it)
  }
  if (p.topk_out)
    for (int j = lane; j < p.k; j += 32) p.topk_out[(size_t)b * p.k + j] = -1;
  if (p.fuse_select) {
    for (int j = lane; j < p.C; j += 32) p.sel.cand_out[(size_t)b * p.C + j] = -1;
    if (lane == 0) p.sel.ncand_out[b] = p.sel.ncand_keep[b] = 0;
  }
}

template <int TT>
__global__ void __launch_bounds__(kRouterWarps * 32, 2) router_batched_kernel(const RouterParams p) {
  SPAN_BEGIN();
  cg::cluster_group cluster = cg::this_cluster();
  const unsigned crank = cluster.block_rank(), csize = cluster.num_blocks();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int CH = router_chunk(TT);
  constexpr int NT = router_tile_tok(TT), NX = router_tile_exp(TT);
  __shared__ __align__(16) float zs[TT][APEX_MAX_EXPERTS];   // tokens finished here (at most all of them)
  __shared__ float qs[kRouterWarps][APEX_MAX_EXPERTS];
  __shared__ int pis[kRouterWarps][APEX_MAX_EXPERTS];
  __shared__ int posp[kRouterWarps][APEX_MAX_EXPERTS];
  __shared__ uint64_t s_bar[2];
  __shared__ uint64_t s_attn[kAttnWarps];
  __shared__ int s_bad;                         // a wait of a CTA of the cluster ran out
  extern __shared__ __align__(128) float tiles[];  // [2][TT + 8][CH]: x rows, W rows
  const int b0 = blockIdx.y * TT, nt = min(TT, p.B - b0);
  const int e0 = (int)crank * p.warps_per_cta, ne = max(0, min(p.warps_per_cta, p.N - e0));
  const int n_chunks = (p.d + CH - 1) / CH;
  const int groups = (p.B + TT - 1) / TT;  // of tokens
  if ((int)blockIdx.y >= groups) {  // the attention block's bytes, beside the routers
    if (warp >= kAttnWarps) return;
    if (lane == 0) {
      mbar_init(&s_attn[warp], 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    pdl_wait();
    pdl_launch_dependents();
    attn_stream(p.attn, reinterpret_cast<uint8_t*>(tiles) + warp * kAttnChunk, &s_attn[warp], warp, lane, ((int)blockIdx.y - groups) * (int)csize + (int)crank,
                ((int)gridDim.y - groups) * (int)csize);
    SPAN_END_OF(3, groups);
    return;
  }
  if (threadIdx.x == 0) {
    s_bad = 0;
    mbar_init(&s_bar[0], 2);
    mbar_init(&s_bar[1], 2);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  auto chunk_bytes = [&](int c) { return (uint32_t)(min(CH, p.d - c * CH) * 4); };
  auto load_w = [&](int c) {  // warp 0
    if (lane == 0) mbar_expect_tx(&s_bar[c & 1], ne * chunk_bytes(c) + (p.starve && c == 0 && blockIdx.x == 0 && blockIdx.y == 0 ? 16u : 0u));
    __syncwarp();
    if (lane < ne) bulk_g2s(tiles + ((c & 1) * (TT + 8) + TT + lane) * CH, p.W + (size_t)(e0 + lane) * p.d + c * CH, chunk_bytes(c), &s_bar[c & 1]);
  };
  auto load_x = [&](int c) {
    if (lane == 0) mbar_expect_tx(&s_bar[c & 1], nt * chunk_bytes(c));
    __syncwarp();
    if (lane < nt) bulk_g2s(tiles + ((c & 1) * (TT + 8) + lane) * CH, p.x + (size_t)(b0 + lane) * p.d + c * CH, chunk_bytes(c), &s_bar[c & 1]);
  };
  if (warp == 0)
    for (int c = 0; c < 2 && c < n_chunks; ++c) load_w(c);
  const int te = warp * (int)csize + (int)crank;  // the token this warp finishes
  EpilogueVals ev;
  if (p.fuse_select && te < nt) ev.sel = load_select_vals(p.sel, lane);
  RTL(0);
  pdl_wait();
  pdl_launch_dependents();
  RTL(1);
  if (te < nt) load_prediction(p, b0 + te, lane, &ev);
  if (warp == 0)
    for (int c = 0; c < 2 && c < n_chunks; ++c) load_x(c);
  // this warp's tile: tokens t0 .. t0 + NT - 1, experts x0 .. x0 + NX - 1 of the CTA
  constexpr int TILES_T = TT / NT;
  const int t0 = (warp % TILES_T) * NT, x0 = (warp / TILES_T) * NX;
  const bool active = x0 < ne && t0 < nt;
  float acc[NT * NX];
#pragma unroll
  for (int v = 0; v < NT * NX; ++v) acc[v] = 0.f;
  // A wait that runs out (the GPU held for the length of the limit, say) does not end the loop, which has barriers: the cluster's
  // flag is set, which ends its other waits, and the tokens are marked below
  int loaded = min(2, n_chunks);  // chunks asked for (warp 0)
  for (int c = 0; c < n_chunks; ++c) {
    if (!mbar_wait(&s_bar[c & 1], (c >> 1) & 1, &s_bad, p.wait_limit_ns)) {
      for (unsigned r = 0; r < csize; ++r) *(volatile int*)cluster.map_shared_rank(&s_bad, r) = 1;
    }
    if (active) {
      const int nv = min(CH, p.d - c * CH) >> 2;
      const float4* xt = reinterpret_cast<const float4*>(tiles + ((c & 1) * (TT + 8) + t0) * CH) + lane;
      const float4* wt = reinterpret_cast<const float4*>(tiles + ((c & 1) * (TT + 8) + TT + x0) * CH) + lane;
      auto step = [&](int i) {
        float4 xv[NT];
#pragma unroll
        for (int t = 0; t < NT; ++t) xv[t] = xt[t * (CH / 4) + i];
#pragma unroll
        for (int x = 0; x < NX; ++x) {
          const float4 wv = wt[x * (CH / 4) + i];
#pragma unroll
          for (int t = 0; t < NT; ++t) {
            float a = acc[x * NT + t];
            a = fmaf(wv.x, xv[t].x, a);
            a = fmaf(wv.y, xv[t].y, a);
            a = fmaf(wv.z, xv[t].z, a);
            a = fmaf(wv.w, xv[t].w, a);
            acc[x * NT + t] = a;
          }
        }
      };
      int i = 0;
#pragma unroll 2
      for (; i + 32 <= nv; i += 32) step(i);
      if (i + lane < nv) step(i);  // (a remainder of columns: some lanes)
    }
    if (c + 2 < n_chunks) {
      __syncthreads();  // everybody has read this buffer
      if (warp == 0 && !__shfl_sync(0xffffffffu, *(volatile int*)&s_bad, 0)) {  // (a buffer whose copies are still out is not filled again)
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        load_w(c + 2);
        load_x(c + 2);
        loaded = c + 3;
      }
    }
  }
  RTL(2);
  // The xor tree over the lanes.  While more than one value is left, a lane keeps the half of the values its bit selects
  // and hands the other half to its partner.
  int idx = 0;  // index of the value this lane ends up with
  {
    int n = NT * NX;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      if (n > 1) {
        n >>= 1;
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int v = 0; v < NT * NX / 2; ++v) {
          if (v < n) {
            const float give = up ? acc[v] : acc[v + n], keep = up ? acc[v + n] : acc[v];
            acc[v] = keep + __shfl_xor_sync(0xffffffffu, give, o);
          }
        }
        idx = idx * 2 + (up ? 1 : 0);
      } else {
        acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
      }
    }
  }
  constexpr int DUP = 32 / (NT * NX);  // lanes that end up with the same value
  if (active && (lane & (DUP - 1)) == 0) {
    const int x = x0 + idx / NT, t = t0 + idx % NT;
    if (x < ne && t < nt) {
      const float z = acc[0] + (p.bias ? __ldg(p.bias + e0 + x) : 0.f);
      float* dst = cluster.map_shared_rank(&zs[0][0], t % csize);
      dst[(t / csize) * APEX_MAX_EXPERTS + e0 + x] = z;
    }
  }
  RTL(3);
  cluster.sync();
  RTL(4);
  if (s_bad) {
    if (warp == 0) {  // what is still on its way into this CTA's shared memory (bounded)
      for (int c = max(0, loaded - 2); c < loaded; ++c) mbar_wait(&s_bar[c & 1], (c >> 1) & 1, nullptr, p.wait_limit_ns);
      if (lane == 0 && p.status) *p.status = 1u;
    }
    for (int t = te; t < nt; t += kRouterWarps * (int)csize) router_failed(p, b0 + t, lane);
    return;
  }
  if (te < nt) router_epilogue(p, ev, b0 + te, lane, zs[warp], qs[warp], pis[warp], posp[warp]);
  for (int t = te + kRouterWarps * (int)csize; t < nt; t += kRouterWarps * (int)csize) {  // (a cluster of one CTA: more tokens than warps)
    __syncwarp();
    load_prediction(p, b0 + t, lane, &ev);
    router_epilogue(p, ev, b0 + t, lane, zs[t / csize], qs[warp], pis[warp], posp[warp]);
  }
  RTL(6);
  SPAN_END((p.fuse_select || !p.topk_out || !p.stats) ? 1 : 4);
}

// Clusters that stream the attention block beside the routers: a CTA per SM (64 KB in flight each), fewer where it is short.  All of
// them are resident with the routers', two CTAs to an SM, as long as clusters of eight are no more than kMaxClusters8.
constexpr int kMaxClusters8 = 31;
int attn_clusters(const AttnParams& a, int csize, int groups) {
  const size_t ctas = (a.bytes + kAttnWarps * kAttnChunk - 1) / (kAttnWarps * kAttnChunk);
  if (ctas == 0) return 0;
  const int n = ctas < (size_t)a.n_sm ? ((int)ctas + csize - 1) / csize : a.n_sm / csize;
  return csize < 8 || n + groups <= kMaxClusters8 ? n : kMaxClusters8 - groups;
}

template <int TT>
cudaError_t launch_router_batched(const RouterParams& p, cudaLaunchConfig_t& cfg, int csize) {
  constexpr int smem = router_smem(TT);
  static bool configured[kMaxDevices];
  static std::mutex setup_mutex;  // contexts of several host threads (and the context-free gate) share this set-up
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  {
    std::lock_guard<std::mutex> lock(setup_mutex);
    if (!configured[dev]) {
      if ((e = cudaFuncSetAttribute(router_batched_kernel<TT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess) return e;
      configured[dev] = true;
    }
  }
  prefer_max_shared<router_batched_kernel<TT>>();
  const int groups = (p.B + TT - 1) / TT;
  cfg.gridDim = dim3(csize, groups + attn_clusters(p.attn, csize, groups), 1);
  cfg.dynamicSmemBytes = smem;
  return cudaLaunchKernelEx(&cfg, router_batched_kernel<TT>, p);
}

cudaError_t launch_router(const RouterParams& p, cudaStream_t s) {
  // cluster size: power of two, up to 8 CTAs of up to 8 warps
  int csize = 1;
  while (csize < 8 && csize * 8 < p.N) csize <<= 1;
  RouterParams q = p;
  q.warps_per_cta = (p.N + csize - 1) / csize;
  if (q.wait_limit_ns <= 0) q.wait_limit_ns = 2000000000ll;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(csize, p.B, 1);
  cfg.blockDim = dim3(256, 1, 1);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = csize;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  if (p.B == 1) {
    prefer_max_shared<router_kernel>();
    return cudaLaunchKernelEx(&cfg, router_kernel, q);
  }
  // Tokens per cluster: as few as let all clusters run at once (15 of eight CTAs; 128 CTAs of smaller ones), since a cluster's time
  // grows with its tokens; at most 16
  const int clusters = csize < 8 ? 128 / csize : 15;
  if (p.B <= clusters) return launch_router_batched<1>(q, cfg, csize);
  if (p.B <= 2 * clusters) return launch_router_batched<2>(q, cfg, csize);
  if (p.B <= 4 * clusters) return launch_router_batched<4>(q, cfg, csize);
  if (p.B <= 8 * clusters) return launch_router_batched<8>(q, cfg, csize);
  return launch_router_batched<16>(q, cfg, csize);
}

// One warp per token: x_j = q_p[pi[j]] (the prefetch distribution in descending order),
// s = w.x, delta_hat = first delta with theta_delta - s >= logit(tau)  (Eq. (8), (9) in the logit
// domain), capped to C - k; K_p = first k + delta_hat experts of E (Eq. (1)).
__global__ void __launch_bounds__(128) select_kernel(const SelectParams p) {
  SPAN_BEGIN();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.x * (blockDim.x >> 5) + warp;
  const SelectVals sv = load_select_vals(p, lane);
  pdl_wait();
  pdl_launch_dependents();
  if (b >= p.B) return;
  const int N = p.N;
  const size_t row = (size_t)b * N;
  int pj0 = -1, pj1 = -1;
  float x0 = 0.f, x1 = 0.f;
  if (lane < N) {
    pj0 = __ldg(p.pi + row + lane);
    x0 = __ldg(p.q + row + pj0);
  }
  if (lane + 32 < N) {
    pj1 = __ldg(p.pi + row + lane + 32);
    x1 = __ldg(p.q + row + pj1);
  }
  select_token(p, sv, b, lane, pj0, pj1, x0, x1);
  SPAN_END(2);
}

cudaError_t launch_select(const SelectParams& p, cudaStream_t s) {
  prefer_max_shared<select_kernel>();
  const int wpb = 4;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((p.B + wpb - 1) / wpb, 1, 1);
  cfg.blockDim = dim3(wpb * 32, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, select_kernel, p);
}

__global__ void __launch_bounds__(kAttnWarps * 32) attention_standin_kernel(const AttnParams p) {
  SPAN_BEGIN();
  extern __shared__ __align__(128) uint8_t attn_smem[];
  __shared__ uint64_t s_bar[kAttnWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    mbar_init(&s_bar[warp], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (p.wait_first) pdl_wait();
  pdl_launch_dependents();
  attn_stream(p, attn_smem + warp * kAttnChunk, &s_bar[warp], warp, lane, blockIdx.x, gridDim.x);
  // Streamed beside the preceding kernel: wait for it now, so that whoever waits for this kernel has, as
  // always, everything before it on the stream complete.
  if (!p.wait_first) pdl_wait();
  SPAN_END(3);
}

cudaError_t launch_attention(const AttnParams& p, int n_sm, cudaStream_t s) {
  static std::atomic<bool> configured[kMaxDevices];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  if (!configured[dev].load(std::memory_order_acquire)) {
    if ((e = cudaFuncSetAttribute(attention_standin_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kAttnWarps * kAttnChunk)) != cudaSuccess) return e;
    configured[dev].store(true, std::memory_order_release);
  }
  prefer_max_shared<attention_standin_kernel>();
  cudaLaunchConfig_t cfg = {};
  const size_t chunks = (p.bytes + kAttnChunk - 1) / kAttnChunk;
  cfg.gridDim = dim3((unsigned)(chunks < (size_t)n_sm ? chunks : (size_t)n_sm), 1, 1);
  cfg.blockDim = dim3(kAttnWarps * 32, 1, 1);
  cfg.dynamicSmemBytes = kAttnWarps * kAttnChunk;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, attention_standin_kernel, p);
}

}  // namespace apex
