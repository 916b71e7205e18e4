// apex_distill_router: trains the prefetch router q_p = softmax(W_p h + b_p) to match the frozen router's
// distribution q_r on a calibration set (Sec. IV-C, Eq. (10)): minimise the mean over tokens of
// KL(q_r || q_p) by full-batch Adam (0.9 / 0.999 / 1e-8) in fp64 with a fixed iteration count.
//
// Both passes of an iteration are fp64 contractions over H (T x d), so both run on the fp64 tensor path
// (mma.sync m8n8k4, 37 TFLOP/s measured, the same peak as fp64 FMAs but with a quarter of the operand fetches):
//
//   distill_fwd_kernel   a CTA owns 8 W tokens: their N logits (M = tokens, N = experts, K = d), softmax,
//                        G[t][e] = (q_p - q_r) / T  (d loss / d logits) and the CTA's sum of G for the bias
//   distill_bwd_kernel   a CTA owns 64 columns and a segment of the tokens: its part of
//                        d loss / d W[e][j] = sum_t G[t][e] h[t][j]   (M = experts, N = columns, K = tokens)
//   distill_step_kernel  a thread per parameter: the segments' parts in order, Adam
//
// Four producer warps bring the operands in (asynchronous 16-byte copies into a four-stage ring, counted on mbarriers),
// so the MMA warps never meet at a CTA barrier and keep the tensor pipe busy while they drift (one barrier per K tile
// with everybody copying left it idle 45 % of the time).  H stays fp32 in shared memory and is widened in registers,
// each value by one warp only.  Every sum has a fixed order (K slices of a CTA, segments, token tiles are added by
// index), so the result is reproducible bit for bit.
// The floor is the 4 T N d flops of an iteration at 37 TFLOP/s: 54 us at T = 8192, N = 40, d = 1536.  A warp per token
// re-reading W and a thread per column re-reading G took 795 us there; this form
// takes 78 us (about 34 for each pass, the rest step and launches).
#include <cmath>
#include <cstdio>
#include <vector>

#include "apex_internal.hpp"
#include "ptx.cuh"
#include "workspace.hpp"

namespace {

constexpr int kProducers = 128;    // threads of the four producer warps (the first of a CTA)
constexpr int kFwdWarps = 28;      // MMA warps of the forward pass: seven on each scheduler
constexpr int kFwdThreads = kProducers + kFwdWarps * 32;
constexpr int kBwdWarps = 16;      // ... of the backward pass: four groups of 16 columns, four K slices
constexpr int kBwdThreads = kProducers + kBwdWarps * 32;
constexpr int kKd = 64;         // columns of H and W per pipeline stage (forward)
constexpr int kTokTile = 64;    // tokens per pipeline stage (backward)
constexpr int kCols = 64;       // columns per CTA (backward)
constexpr int kStages = 4;
constexpr int kMaxSeg = 37;     // token segments (backward)
constexpr int kFewSeg = 12;     // (a shorter unrolled sum in the step kernel)
// Row strides in shared memory: fragment loads touch 8 rows x 4 columns (or the transpose) at once; with these strides
// the words of one access fall into different banks.
constexpr int kLdH = kKd + 4, kLdW = kKd + 4, kLdHb = kCols + 8;
constexpr long long kWaitLimitNs = 2000000000ll;  // bound of the ring's waits (they depend on nothing outside the CTA)

// K slices of a forward CTA: warps per eight tokens, a power of two (a stage has 16 K steps)
__host__ __device__ constexpr int fwd_slices(int tok_warps) {
  return tok_warps == 1 ? 16 : tok_warps <= 3 ? 8 : tok_warps <= 7 ? 4 : 2;
}

struct DistillParams {
  const float* H;    // [T][d]
  const float* Qr;   // [T][N]
  double* W;         // [8 NE][ldw], rows >= N and columns >= d are zero
  double* b;         // [8 NE]
  double* m;         // Adam moments: [8 NE][ldw], then the bias's [8 NE]
  double* v;
  double* G;         // [T][8 NE]
  double* gb;        // [forward CTAs][8 NE]: sums of G over a CTA's tokens
  double* partial;   // [column tiles][segments][8 NE][kCols]
  int T, N, d, ldw;
  int tok_warps;     // forward: tokens per CTA / 8, 1 to 8
  int n_fwd, n_tiles, n_seg, seg_len;
  int* status;       // 1: a wait of a ring ran out
  int starve;        // test hook: the first forward CTA's ring expects an arrival that never comes
  double lr, c1, c2;  // step size; bias corrections 1 - 0.9^it, 1 - 0.999^it
};

__device__ __forceinline__ void dmma(double (&c)[2], double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(c[0]), "+d"(c[1]) : "d"(a), "d"(b));
}
// bytes of the chunk that exist are copied, the rest of it is zero
__device__ __forceinline__ void cp16(void* dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(apex::smem_u32(dst)), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp4(void* dst, const void* src, bool valid) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(apex::smem_u32(dst)), "l"(src), "r"(valid ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_arrive(uint64_t* bar) {  // this thread's copies so far count on the barrier when they land
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(apex::smem_u32(bar)) : "memory");
}

// A producer thread's part of `rows` x 64 floats of H from (row0, col0) into a tile with row stride ld; beyond rows_end
// and d: zero.  VEC: 16-byte copies (d a multiple of 4 and H 16-byte aligned), else word by word.
template <bool VEC>
__device__ __forceinline__ void load_h(float* dst, int ld, const DistillParams& p, int row0, int rows, int rows_end, int col0) {
  const int pt = threadIdx.x;
  if (VEC) {
    const int c = (pt & 15) * 4;
    const float* src = p.H + (size_t)(row0 + (pt >> 4)) * p.d + col0 + c;
    const bool col_ok = col0 + c < p.d;
#pragma unroll 4
    for (int r = pt >> 4; r < rows; r += kProducers / 16, src += (size_t)(kProducers / 16) * p.d) {
      const bool ok = col_ok && row0 + r < rows_end;
      cp16(dst + r * ld + c, ok ? src : p.H, ok);
    }
  } else {
    for (int i = pt; i < rows * 64; i += kProducers) {
      const int r = i >> 6, c = i & 63;
      const bool ok = row0 + r < rows_end && col0 + c < p.d;
      cp4(dst + r * ld + c, ok ? p.H + (size_t)(row0 + r) * p.d + col0 + c : p.H, ok);
    }
  }
}

__host__ __device__ constexpr size_t fwd_stage_bytes(int ne, int toks) { return (size_t)toks * kLdH * 4 + (size_t)8 * ne * kLdW * 8; }
__host__ __device__ constexpr size_t bwd_stage_bytes(int ne) { return (size_t)kTokTile * (8 * ne + 4) * 8 + (size_t)kTokTile * kLdHb * 4; }
constexpr size_t fwd_smem_bytes(int ne, int tok_warps) {
  // the pipeline, later reused for the K slices' partial logits
  const size_t ring = kStages * fwd_stage_bytes(ne, 8 * tok_warps);
  const size_t red = (size_t)(fwd_slices(tok_warps) + 1) * 8 * tok_warps * 8 * ne * 8;
  return ring > red ? ring : red;
}
constexpr size_t bwd_smem_bytes(int ne) {
  const size_t ring = kStages * bwd_stage_bytes(ne), red = (size_t)4 * 8 * ne * kCols * 8;
  return ring > red ? ring : red;
}

// (a whole line: the dynamic shared memory behind it starts on one; 16 bytes off, an iteration took 1.5 us of 84 more)
struct alignas(128) Ring {
  uint64_t full[kStages], empty[kStages];
  int dead;  // a wait ran out: nobody waits any more; the host does not use the result
};
__device__ __forceinline__ void ring_init(Ring* r, int mma_warps, int extra = 0) {
  if (threadIdx.x == 0) {
    r->dead = 0;
    for (int s = 0; s < kStages; ++s) {
      apex::mbar_init(&r->full[s], kProducers + extra);
      apex::mbar_init(&r->empty[s], mma_warps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
}

// A wait that runs out ends the others of the CTA; the loops go on over whatever the stages hold (a warp must not leave them
// lane by lane: its MMAs are the whole warp's)
__device__ __forceinline__ void ring_wait(Ring* r, uint64_t* bar, uint32_t parity, int* status) {
  if (apex::mbar_wait(bar, parity, &r->dead, kWaitLimitNs)) return;
  *(volatile int*)&r->dead = 1;
  *(volatile int*)status = 1;
}
// the ring is reused behind the loops: a producer's copies must have landed, also where nobody waited for them any more
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <int NE, bool VEC>
__global__ void __launch_bounds__(kFwdThreads, 1) distill_fwd_kernel(const DistillParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Ring ring;
  const int tid = threadIdx.x, lane = tid & 31;
  const int TW = p.tok_warps, toks = 8 * TW, KS = fwd_slices(TW);
  const int t0 = blockIdx.x * toks;
  const int n_kt = (p.d + kKd - 1) / kKd;
  const size_t stage = fwd_stage_bytes(NE, toks);
  ring_init(&ring, TW * KS, p.starve && blockIdx.x == 0 ? 1 : 0);
  const int mw = (tid - kProducers) >> 5;                // MMA warp
  const int tw = mw % TW, kslice = mw / TW;              // its eight tokens and its share of a stage's K steps
  const int fr = lane >> 2, fc = lane & 3;
  double acc[NE][2];
#pragma unroll
  for (int j = 0; j < NE; ++j) acc[j][0] = acc[j][1] = 0.0;
  if (tid < kProducers) {
    for (int kt = 0; kt < n_kt; ++kt) {
      const int s = kt % kStages;
      if (kt >= kStages) ring_wait(&ring, &ring.empty[s], (kt / kStages - 1) & 1, p.status);
      float* th = reinterpret_cast<float*>(smem + s * stage);
      double* tw_ = reinterpret_cast<double*>(smem + s * stage + (size_t)toks * kLdH * 4);
      load_h<VEC>(th, kLdH, p, t0, toks, p.T, kt * kKd);
      if (kt == 0) {  // H is an input of the whole call; W is what the previous kernel wrote
        apex::pdl_wait();
        apex::pdl_launch_dependents();
      }
      const double* src = p.W + (size_t)(tid >> 5) * p.ldw + kt * kKd + lane * 2;  // ldw is a multiple of kKd
#pragma unroll 4
      for (int r = tid >> 5; r < 8 * NE; r += kProducers / 32, src += (size_t)(kProducers / 32) * p.ldw)
        cp16(tw_ + r * kLdW + lane * 2, src, true);
      cp_arrive(&ring.full[s]);
    }
    cp_wait_all();
  } else if (kslice < KS) {
    for (int kt = 0; kt < n_kt; ++kt) {
      const int s = kt % kStages;
      ring_wait(&ring, &ring.full[s], (kt / kStages) & 1, p.status);
      const float* hp = reinterpret_cast<const float*>(smem + s * stage) + (tw * 8 + fr) * kLdH + fc;
      const double* wp = reinterpret_cast<const double*>(smem + s * stage + (size_t)toks * kLdH * 4) + fr * kLdW + fc;
#pragma unroll 4
      for (int ks = kslice; ks < kKd / 4; ks += KS) {
        const double a = (double)hp[ks * 4];
#pragma unroll
        for (int j = 0; j < NE; ++j) dmma(acc[j], a, wp[j * 8 * kLdW + ks * 4]);
      }
      __syncwarp();
      if (lane == 0) apex::mbar_arrive(&ring.empty[s]);
    }
  }
  apex::pdl_wait();  // (the bias, read below, comes from the previous kernel as well)
  __syncthreads();
  // logits: the K slices' partial sums in order, plus the bias
  double* z = reinterpret_cast<double*>(smem);                                // [KS][toks][8 NE]
  double* zs = z + (size_t)KS * toks * 8 * NE;                                // [toks][8 NE]
  if (tid >= kProducers && kslice < KS) {
#pragma unroll
    for (int j = 0; j < NE; ++j) {
      double* dst = z + ((size_t)kslice * toks + tw * 8 + fr) * (8 * NE) + j * 8 + fc * 2;
      dst[0] = acc[j][0];
      dst[1] = acc[j][1];
    }
  }
  __syncthreads();
  // softmax: eight lanes per token, each with experts q, q + 8, ...
  const double inv_T = 1.0 / (double)p.T;
  if (tid < 8 * toks) {  // (whole warps: toks is a multiple of 8)
    const int tl = tid >> 3, q = tid & 7;
    const bool on = t0 + tl < p.T;
    double x[NE], mx = -INFINITY;
#pragma unroll
    for (int j = 0; j < NE; ++j) {
      const int e = j * 8 + q;
      x[j] = -INFINITY;
      if (on && e < p.N) {
        double s = z[(size_t)tl * (8 * NE) + e];
        for (int k = 1; k < KS; ++k) s += z[((size_t)k * toks + tl) * (8 * NE) + e];
        x[j] = s + p.b[e];
      }
      mx = fmax(mx, x[j]);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    double sum = 0.0;
#pragma unroll
    for (int j = 0; j < NE; ++j) {
      x[j] = (on && j * 8 + q < p.N) ? exp(x[j] - mx) : 0.0;
      sum += x[j];
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const double inv = on ? 1.0 / sum : 0.0;
#pragma unroll
    for (int j = 0; j < NE; ++j) {
      const int e = j * 8 + q;
      const double g = (on && e < p.N) ? (x[j] * inv - (double)p.Qr[(size_t)(t0 + tl) * p.N + e]) * inv_T : 0.0;
      if (on) p.G[(size_t)(t0 + tl) * (8 * NE) + e] = g;
      zs[tl * (8 * NE) + e] = g;
    }
  }
  __syncthreads();
  // the bias's gradient: sums over the CTA's tokens, eight at a time, then the groups in order
  double* gs = z;  // [TW][8 NE] (the partial logits are no longer needed)
  for (int i = tid; i < TW * 8 * NE; i += kFwdThreads) {
    const int g = i / (8 * NE), e = i - g * 8 * NE;
    double s = 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u) s += zs[(g * 8 + u) * (8 * NE) + e];
    gs[i] = s;
  }
  __syncthreads();
  if (tid < 8 * NE) {
    double s = 0.0;
    for (int g = 0; g < TW; ++g) s += gs[g * 8 * NE + tid];
    p.gb[(size_t)blockIdx.x * (8 * NE) + tid] = s;
  }
}

__device__ __forceinline__ void adam(const DistillParams& p, double* w, double* mm, double* vv, double g) {
  const double m = 0.9 * *mm + 0.1 * g;
  const double v = 0.999 * *vv + 0.001 * g * g;
  *mm = m;
  *vv = v;
  *w = *w - p.lr * (m / p.c1) / (sqrt(v / p.c2) + 1e-8);
}

// grid: column tiles x segments
template <int NE, bool VEC>
__global__ void __launch_bounds__(kBwdThreads, 1) distill_bwd_kernel(const DistillParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Ring ring;
  const int tid = threadIdx.x, lane = tid & 31;
  constexpr int LDG = 8 * NE + 4;
  const int tile = blockIdx.x / p.n_seg, seg = blockIdx.x - tile * p.n_seg;
  const int col0 = tile * kCols;
  const int t_lo = min(p.T, seg * p.seg_len), t_hi = min(p.T, t_lo + p.seg_len);
  const int n_kt = (t_hi - t_lo + kTokTile - 1) / kTokTile;
  constexpr size_t stage = bwd_stage_bytes(NE);
  ring_init(&ring, kBwdWarps);
  const int mw = (tid - kProducers) >> 5, cg = mw & 3, kslice = mw >> 2;  // MMA warp: 16 columns, every fourth K step
  const int fr = lane >> 2, fc = lane & 3;
  double acc[NE][2][2];
#pragma unroll
  for (int j = 0; j < NE; ++j) acc[j][0][0] = acc[j][0][1] = acc[j][1][0] = acc[j][1][1] = 0.0;
  if (tid < kProducers) {
    for (int kt = 0; kt < n_kt; ++kt) {
      const int s = kt % kStages, t0 = t_lo + kt * kTokTile;
      if (kt >= kStages) ring_wait(&ring, &ring.empty[s], (kt / kStages - 1) & 1, p.status);
      double* tg = reinterpret_cast<double*>(smem + s * stage);
      load_h<VEC>(reinterpret_cast<float*>(smem + s * stage + (size_t)kTokTile * LDG * 8), kLdHb, p, t0, kTokTile, t_hi, col0);
      if (kt == 0) {
        apex::pdl_wait();
        apex::pdl_launch_dependents();
      }
      const double* src = p.G + (size_t)t0 * (8 * NE);
#pragma unroll 4
      for (int i = tid; i < kTokTile * 4 * NE; i += kProducers) {
        const int r = i / (4 * NE), c = (i - r * (4 * NE)) * 2;
        const bool ok = t0 + r < t_hi;
        cp16(tg + r * LDG + c, ok ? src + i * 2 : p.G, ok);
      }
      cp_arrive(&ring.full[s]);
    }
    cp_wait_all();
  } else {
    for (int kt = 0; kt < n_kt; ++kt) {
      const int s = kt % kStages;
      ring_wait(&ring, &ring.full[s], (kt / kStages) & 1, p.status);
      const double* gp = reinterpret_cast<const double*>(smem + s * stage) + fc * LDG + fr;                                  // A: experts x tokens
      const float* hp = reinterpret_cast<const float*>(smem + s * stage + (size_t)kTokTile * LDG * 8) + fc * kLdHb + cg * 16 + fr;  // B: tokens x columns
#pragma unroll
      for (int ks = kslice; ks < kTokTile / 4; ks += 4) {
        const double b0 = (double)hp[ks * 4 * kLdHb], b1 = (double)hp[ks * 4 * kLdHb + 8];
#pragma unroll
        for (int j = 0; j < NE; ++j) {
          const double a = gp[ks * 4 * LDG + j * 8];
          dmma(acc[j][0], a, b0);
          dmma(acc[j][1], a, b1);
        }
      }
      __syncwarp();
      if (lane == 0) apex::mbar_arrive(&ring.empty[s]);
    }
  }
  apex::pdl_wait();  // (an empty segment's CTA, too, writes its part only after the previous step has read the old ones)
  __syncthreads();
  double* red = reinterpret_cast<double*>(smem);  // [4 K slices][8 NE][kCols]
  if (tid >= kProducers) {
#pragma unroll
    for (int j = 0; j < NE; ++j)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        double* dst = red + ((size_t)kslice * 8 * NE + j * 8 + fr) * kCols + cg * 16 + h * 8 + fc * 2;
        dst[0] = acc[j][h][0];
        dst[1] = acc[j][h][1];
      }
  }
  __syncthreads();
  constexpr int n = 8 * NE * kCols;
  double* part = p.partial + ((size_t)tile * p.n_seg + seg) * n;
  for (int i = tid; i < n; i += kBwdThreads) part[i] = ((red[i] + red[n + i]) + red[2 * n + i]) + red[3 * n + i];
}

constexpr int kStepThreads = 256;
// CTAs 0 .. grid-2: a thread per weight, in the order of the parts (column tile, expert, column); the last CTA: the bias
__global__ void __launch_bounds__(kStepThreads) distill_step_kernel(const DistillParams p, int rows) {
  __shared__ double part_b[kStepThreads];
  apex::pdl_wait();
  apex::pdl_launch_dependents();
  const size_t n_w = (size_t)rows * p.ldw;
  if (blockIdx.x == gridDim.x - 1) {
    const int per = kStepThreads / rows, e = threadIdx.x % rows, q = threadIdx.x / rows;  // `per` interleaved partial sums per expert
    if (q < per) {
      double s = 0.0;
#pragma unroll 4
      for (int c = q; c < p.n_fwd; c += per) s += p.gb[(size_t)c * rows + e];
      part_b[q * rows + e] = s;
    }
    __syncthreads();
    if (threadIdx.x < p.N) {
      double s = 0.0;
      for (int i = 0; i < per; ++i) s += part_b[i * rows + threadIdx.x];
      adam(p, p.b + threadIdx.x, p.m + n_w + threadIdx.x, p.v + n_w + threadIdx.x, s);
    }
    return;
  }
  const int n = rows * kCols;
  const int i = blockIdx.x * kStepThreads + threadIdx.x, tile = i / n, r = i - tile * n;
  const int e = r / kCols, j = tile * kCols + (r & (kCols - 1));
  if (tile >= p.n_tiles || e >= p.N || j >= p.d) return;
  const double* part = p.partial + (size_t)tile * p.n_seg * n + r;
  double g = 0.0;
  // in order; all loads in flight together (in turns of twelve 2 us more at 32 segments)
  if (p.n_seg <= kFewSeg) {
#pragma unroll
    for (int s = 0; s < kFewSeg; ++s)
      if (s < p.n_seg) g += part[(size_t)s * n];
  } else {
#pragma unroll
    for (int s = 0; s < kMaxSeg; ++s)
      if (s < p.n_seg) g += part[(size_t)s * n];
  }
  const size_t at = (size_t)e * p.ldw + j;
  adam(p, p.W + at, p.m + at, p.v + at, g);
}

// fp32 <-> fp64 copies of the parameters ([N][d] and [N] on the outside)
__global__ void distill_unpack_kernel(const float* in, DistillParams p) {
  const size_t n = (size_t)p.N * p.d;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n + p.N; i += (size_t)gridDim.x * blockDim.x) {
    if (i < n) p.W[i / p.d * p.ldw + i % p.d] = (double)in[i];
    else p.b[i - n] = (double)in[i];
  }
}
__global__ void distill_pack_kernel(float* out, DistillParams p) {
  const size_t n = (size_t)p.N * p.d;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n + p.N; i += (size_t)gridDim.x * blockDim.x)
    out[i] = i < n ? (float)p.W[i / p.d * p.ldw + i % p.d] : (float)p.b[i - n];
}

template <int NE, bool VEC>
cudaError_t run_iterations(DistillParams p, int iters, cudaStream_t cs) {
  const size_t smem_f = fwd_smem_bytes(NE, p.tok_warps), smem_b = bwd_smem_bytes(NE);
  cudaError_t e = cudaFuncSetAttribute(distill_fwd_kernel<NE, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_f);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(distill_bwd_kernel<NE, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_b);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = cs;
  const int n_step = (int)(((size_t)p.n_tiles * 8 * NE * kCols + kStepThreads - 1) / kStepThreads) + 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  for (int it = 1; it <= iters && e == cudaSuccess; ++it) {
    p.c1 = 1.0 - std::pow(0.9, (double)it);
    p.c2 = 1.0 - std::pow(0.999, (double)it);
    cfg.gridDim = dim3(p.n_fwd, 1, 1);
    cfg.blockDim = dim3(kFwdThreads, 1, 1);
    cfg.dynamicSmemBytes = smem_f;
    e = cudaLaunchKernelEx(&cfg, distill_fwd_kernel<NE, VEC>, p);
    cfg.gridDim = dim3(p.n_tiles * p.n_seg, 1, 1);
    cfg.blockDim = dim3(kBwdThreads, 1, 1);
    cfg.dynamicSmemBytes = smem_b;
    if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, distill_bwd_kernel<NE, VEC>, p);
    cfg.gridDim = dim3(n_step, 1, 1);
    cfg.blockDim = dim3(kStepThreads, 1, 1);
    cfg.dynamicSmemBytes = 0;
    if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, distill_step_kernel, p, 8 * NE);
    p.starve = 0;
  }
  return e;
}

template <bool VEC>
cudaError_t run_iterations(const DistillParams& p, int ne, int iters, cudaStream_t cs) {
  switch (ne) {
    case 1: return run_iterations<1, VEC>(p, iters, cs);
    case 2: return run_iterations<2, VEC>(p, iters, cs);
    case 3: return run_iterations<3, VEC>(p, iters, cs);
    case 4: return run_iterations<4, VEC>(p, iters, cs);
    case 5: return run_iterations<5, VEC>(p, iters, cs);
    case 6: return run_iterations<6, VEC>(p, iters, cs);
    case 7: return run_iterations<7, VEC>(p, iters, cs);
    default: return run_iterations<8, VEC>(p, iters, cs);
  }
}

thread_local bool starve_next = false;  // armed test hook

void say(char* err, size_t err_len, const char* msg) {
  if (err && err_len) snprintf(err, err_len, "%s", msg);
}

}  // namespace

extern "C" int apex_test_starve_distill(void) {
  starve_next = true;
  return APEX_OK;
}

extern "C" int apex_distill_router(const float* H_dev, const float* Qr_dev, int T, int N, int d, int iters, double lr,
                                   float* W_host, float* b_host, void* stream, char* err, size_t err_len) {
  say(err, err_len, "");
  if (!H_dev || !Qr_dev || !W_host || !b_host || T < 1 || N < 1 || N > APEX_MAX_EXPERTS || d < 1 || iters < 1 || !(lr > 0.0)) {
    say(err, err_len, "apex_distill_router: bad argument (N <= 64, T, d, iters >= 1, lr > 0, no null pointer)");
    return APEX_EINVAL;
  }
  cudaStream_t cs = (cudaStream_t)stream;
  int n_sm = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  const int ne = (N + 7) / 8, rows = 8 * ne;
  DistillParams p{};
  p.H = H_dev; p.Qr = Qr_dev; p.T = T; p.N = N; p.d = d; p.lr = lr;
  p.starve = starve_next ? 1 : 0;
  starve_next = false;
  p.ldw = (d + kKd - 1) / kKd * kKd;
  // Forward: 8 W tokens per CTA, W the smallest that needs one round of the SMs, 8 at most (W = 7, 28 MMA warps, seven per
  // scheduler, fills 147 of 148 SMs at T = 8192, where 8 fills 128).  With W from 1, 2, 4, 7 and 8 alone, T = 5800 took 7, 104 CTAs,
  // where 5 fills 145: 75.6 us per iteration against 65.9 (d = 1536, N = 30).
  const int want = (T + 8 * n_sm - 1) / (8 * n_sm);
  p.tok_warps = want < 8 ? want : 8;
  p.n_fwd = (T + 8 * p.tok_warps - 1) / (8 * p.tok_warps);
  // Backward: column tiles times segments within one round of the SMs.  A segment is whole pipeline stages of tokens (a token
  // more than a stage costs a stage), and there are at most kMaxSeg of them (the step kernel adds them up): the SMs per column tile of d = 256.
  // With twelve at most, T = 8192, N = 40, d = 256 ran on 48 CTAs, now on 128 (32 segments of four stages).
  p.n_tiles = (d + kCols - 1) / kCols;
  p.n_seg = n_sm / p.n_tiles;
  const int stages = (T + kTokTile - 1) / kTokTile;
  p.n_seg = p.n_seg < 1 ? 1 : (p.n_seg > kMaxSeg ? kMaxSeg : p.n_seg);
  const int per_seg = (stages + p.n_seg - 1) / p.n_seg;
  p.n_seg = (stages + per_seg - 1) / per_seg;
  p.seg_len = per_seg * kTokTile;
  const size_t n_w = (size_t)rows * p.ldw, n_io = (size_t)N * d + N;
  // zeroed: parameters and moments; not zeroed: G, partial sums, the fp32 parameters
  const size_t zeroed = ((3 * (n_w + rows) + 1) * sizeof(double) + 255) / 256 * 256;  // (and the status word; G behind it keeps whole lines)
  const size_t n_rest = (size_t)T * rows + (size_t)p.n_fwd * rows + (size_t)p.n_tiles * p.n_seg * rows * kCols;
  uint8_t* buf = nullptr;
  cudaError_t e = apex::workspace_alloc(reinterpret_cast<void**>(&buf), zeroed + n_rest * sizeof(double) + n_io * sizeof(float), cs);
  if (e != cudaSuccess) {
    say(err, err_len, cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? APEX_ENOMEM : APEX_ECUDA;
  }
  p.W = reinterpret_cast<double*>(buf); p.b = p.W + n_w;
  p.m = p.b + rows; p.v = p.m + n_w + rows;
  p.status = reinterpret_cast<int*>(p.v + n_w + rows);
  p.G = reinterpret_cast<double*>(buf + zeroed);
  p.gb = p.G + (size_t)T * rows;
  p.partial = p.gb + (size_t)p.n_fwd * rows;
  float* io = reinterpret_cast<float*>(p.partial + (size_t)p.n_tiles * p.n_seg * rows * kCols);
  std::vector<float> host(n_io);
  for (size_t i = 0; i < (size_t)N * d; ++i) host[i] = W_host[i];
  for (int i = 0; i < N; ++i) host[(size_t)N * d + i] = b_host[i];
  const bool vec = d % 4 == 0 && ((uintptr_t)H_dev & 15) == 0;
  e = cudaMemsetAsync(buf, 0, zeroed, cs);
  if (e == cudaSuccess) e = cudaMemcpyAsync(io, host.data(), n_io * sizeof(float), cudaMemcpyHostToDevice, cs);
  if (e == cudaSuccess) {
    distill_unpack_kernel<<<n_sm, 256, 0, cs>>>(io, p);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = vec ? run_iterations<true>(p, ne, iters, cs) : run_iterations<false>(p, ne, iters, cs);
  if (e == cudaSuccess) {
    distill_pack_kernel<<<n_sm, 256, 0, cs>>>(io, p);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(host.data(), io, n_io * sizeof(float), cudaMemcpyDeviceToHost, cs);
  int status = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&status, p.status, sizeof(int), cudaMemcpyDeviceToHost, cs);
  apex::workspace_free(buf, cs);                     // (in front of the synchronisation, at which the pool lets go of what it need not keep)
  const cudaError_t e2 = cudaStreamSynchronize(cs);  // also after an error
  if (e == cudaSuccess) e = e2;
  if (e == cudaSuccess && status == 0) {
    for (size_t i = 0; i < (size_t)N * d; ++i) W_host[i] = host[i];
    for (int i = 0; i < N; ++i) b_host[i] = host[(size_t)N * d + i];
  }
  if (e != cudaSuccess) {
    say(err, err_len, cudaGetErrorString(e));
    return APEX_ECUDA;
  }
  if (status != 0) {
    say(err, err_len, "apex_distill_router: a device-side wait ran out");
    return APEX_ECUDA;
  }
  return APEX_OK;
}
