// apex_fit_cdf: fits the ordinal-logistic confidence model p_delta(x) = sigmoid(theta_delta - w.x)
// (Eq. (8)) on a calibration set by the cumulative binary cross-entropy of Eq. (11), on the GPU.
//
//   loss(w, theta) = -(1/T) sum_t sum_delta [ y log p + (1 - y) log(1 - p) ],  y = [delta >= delta*_t]
//
// theta is kept non-decreasing by the parametrisation theta_delta = t0 + sum_{i <= delta} softplus(u_i).
// Full-batch Adam (beta 0.9 / 0.999, eps 1e-8) in fp64 with a fixed iteration count, started from
// w = 0 and the logit of the empirical distribution of delta*; every reduction runs in a fixed order,
// so two runs give the same bits.
//
// ONE kernel runs all iterations: an iteration is a few hundred fp64 operations deep and only a few thousand tokens
// wide, so it is bound by latency, and two launches with a serial thread in each took 46 us of it (T = 8192, N = 40).
// Clusters of eight CTAs, 64 tokens per CTA as long as the GPU has room (the calibration set then stays in shared
// memory), every CTA with its own copy of the parameters:
//   - eight lanes per token: s = w.x, the token's d loss / d z for every threshold.  sigmoid(theta - s) is taken as
//     1 / (1 + e^s e^-theta): one exponential per token and one per threshold instead of one per pair, and reciprocals
//     by Newton-Raphson, which interleave (a division is a call);
//   - a thread per parameter and quarter of the tokens adds up and sends its sum to the CTA of the cluster that owns the
//     parameter (st.async: value and arrival in one message); a warp there adds the 32 contributions, the CTA exchanges
//     its sums with the same CTA of the other clusters (blocks of 16-byte records {sum, iteration} in global memory: data
//     and flag travel together, so there is no grid barrier; a warp polls one cluster's block, two lines a poll) and
//     sends the totals to the eight CTAs of its cluster;
//   - every CTA takes the same Adam step; theta is rebuilt by warp scans.
// T = 8192, N = 40: 5.2 us per iteration (10 000 cycles: 4 000 the exchange, 2 900 the tokens, 2 200 the step), 3.5 us for
// one cluster; 46 us before.
#include <cooperative_groups.h>

#include <cmath>
#include <cstdio>
#include <vector>

#include "apex_internal.hpp"
#include "ptx.cuh"
#include "workspace.hpp"

namespace cg = cooperative_groups;

namespace {

constexpr int kThreads = 512;
constexpr int kTokPass = kThreads / 8;  // tokens per pass: eight lanes each
constexpr int kCluster = 8;
constexpr int kMaxParams = 2 * APEX_MAX_EXPERTS;  // w [N], then t0 and u_1 .. u_{nth-1}: N + (N - k + 1) <= 2 N
constexpr int kOwned = kMaxParams / kCluster;     // parameters a CTA adds up for its cluster: 16 r .. 16 r + 15, one per warp
constexpr int kMaxClusters = 16;        // 8192 tokens in one pass; more tokens are walked in passes
constexpr int kLdG = kTokPass + 1;      // row stride of the per-threshold gradients (threads of a warp read different rows)
constexpr double kExpRange = 300.0;     // |s| and |theta| up to here: e^s, e^-theta and their product stay finite
constexpr long long kWaitLimitNs = 2000000000ll;

struct FitParams {
  const double* X;       // [T][N]
  const int32_t* dstar;  // [T]
  const double* init;    // [N + nth]: w | t0 | u
  const double* theta0;  // [nth]
  double* out;           // [N + nth]: fitted w | theta
  ulonglong2* rec;       // [2][kCluster][kMaxClusters][kOwned]: {a cluster's sum of d loss / d parameter, iteration}; zero at launch
  int* status;           // 1: a wait ran out
  int T, N, nth, iters, tok_per_cta;
  double lr;
};

// Row stride of the cached tokens for up to 8 NM experts: a multiple of 8 that is not one of 16, so that the eight lanes of
// a token and of its neighbour read different banks
__host__ __device__ constexpr int fit_ldx(int nm) { return nm % 2 ? 8 * nm : 8 * nm + 8; }

__device__ __forceinline__ double shfl_xor_add(double v, int o) { return v + __shfl_xor_sync(0xffffffffu, v, o); }
// 1 / d for 1e-300 < d < 1e300: the hardware's coarse reciprocal and two Newton-Raphson steps (error squared each time)
__device__ __forceinline__ double reciprocal(double d) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
  r = fma(r, fma(-d, r, 1.0), r);
  return fma(r, fma(-d, r, 1.0), r);
}
// value into CTA `rank`'s copy of *dst; the 8 bytes count on its copy of *bar
__device__ __forceinline__ void send(double* dst, uint64_t* bar, uint32_t rank, double v) {
  uint32_t ra, rb;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(apex::smem_u32(dst)), "r"(rank));
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(apex::smem_u32(bar)), "r"(rank));
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(ra), "l"(__double_as_longlong(v)), "r"(rb)
               : "memory");
}
// a record is written and read whole (one 128-bit access)
__device__ __forceinline__ void put_record(ulonglong2* at, double v, unsigned long long it) {
  asm volatile("{\n.reg .b128 t;\nmov.b128 t, {%1, %2};\nst.relaxed.gpu.global.b128 [%0], t;\n}" ::"l"(at), "l"(__double_as_longlong(v)), "l"(it) : "memory");
}
__device__ __forceinline__ ulonglong2 get_record(const ulonglong2* at) {
  ulonglong2 r;
  asm volatile("{\n.reg .b128 t;\nld.relaxed.gpu.global.b128 t, [%2];\nmov.b128 {%0, %1}, t;\n}" : "=l"(r.x), "=l"(r.y) : "l"(at) : "memory");
  return r;
}

// NM = ceil(N / 8): experts (and thresholds) per lane of a token's octet.  CACHED: the CTA's tokens are in shared memory.
template <int NM, bool CACHED>
__global__ void __launch_bounds__(kThreads, 2) cdf_fit_kernel(const FitParams p) {
  extern __shared__ __align__(16) double s_x[];         // CACHED: [tok_per_cta, a multiple of kTokPass][LDX], then dstar
  constexpr int LDX = fit_ldx(NM);
  __shared__ double s_w[APEX_MAX_EXPERTS], s_theta[APEX_MAX_EXPERTS], s_etheta[APEX_MAX_EXPERTS];
  __shared__ double s_g[APEX_MAX_EXPERTS * kLdG];       // d loss / d z, by threshold and token of the pass
  __shared__ __align__(16) double s_gsum[kTokPass];
  __shared__ double s_in[2][kOwned][32];                // contributions to the parameters this CTA owns: [4 quarters of 8 CTAs]
  __shared__ double s_tot[2][kMaxParams];               // sums over all tokens
  __shared__ double s_own[kOwned], s_clu[kMaxClusters][kOwned + 1];  // this cluster's sums; all clusters'
  __shared__ double s_sp[APEX_MAX_EXPERTS];
  __shared__ uint64_t s_bar_in, s_bar_tot;
  __shared__ int s_wide[2];                             // a threshold left the range of the factored exponentials
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, crank = (int)cluster.block_rank();
  const int n_clusters = gridDim.x / kCluster, my_cluster = blockIdx.x / kCluster;
  const int N = p.N, nth = p.nth, P = N + nth;
  const int t_lo = min(p.T, (int)blockIdx.x * p.tok_per_cta), n_cta = min(p.T, t_lo + p.tok_per_cta) - t_lo;
  const int n_owned = min(kOwned, max(0, P - crank * kOwned));
  int32_t* s_ds = reinterpret_cast<int32_t*>(s_x + (size_t)p.tok_per_cta * LDX);
  if (tid == 0) {
    apex::mbar_init(&s_bar_in, 1);
    apex::mbar_init(&s_bar_tot, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (CACHED) {
    for (int i = tid; i < p.tok_per_cta * LDX; i += kThreads) s_x[i] = 0.0;
    __syncthreads();
    for (int i = tid; i < n_cta * N; i += kThreads) s_x[i / N * LDX + i % N] = p.X[(size_t)t_lo * N + i];
    for (int i = tid; i < n_cta; i += kThreads) s_ds[i] = p.dstar[t_lo + i];
  }
  const double* xg = p.X + (size_t)t_lo * N;
  const int32_t* dsg = p.dstar + t_lo;
  // Parameters and moments live in threads 0 .. 63 (t0, u_1 ..: warps 0 and 1) and 64 .. 127 (w); a copy in every CTA
  const bool has_u = tid < nth, has_w = tid >= 64 && tid - 64 < N;
  double par = has_u ? p.init[N + tid] : (has_w ? p.init[tid - 64] : 0.0), mom = 0.0, var = 0.0;
  double sig = 1.0;  // d softplus(u) / d u; 1 for t0 and w
  if (has_u && tid > 0) {
    const double e = exp(-fabs(par));
    sig = (par >= 0.0 ? 1.0 : e) * reciprocal(1.0 + e);
  }
  if (tid >= 64 && tid < 128) s_w[tid - 64] = has_w ? par : 0.0;
  if (tid < 64) {
    const double th = has_u ? p.theta0[tid] : 0.0;
    s_theta[tid] = th;
    s_etheta[tid] = exp(-th);
    const bool far = __any_sync(0xffffffffu, !(fabs(th) <= kExpRange));
    if (lane == 0) s_wide[warp] = far;
  }
  double b1 = 1.0, b2 = 1.0;  // 0.9^it, 0.999^it
  const double inv_T = 1.0 / (double)p.T;
  bool dead = false;          // a wait of this thread ran out: it goes on without waiting
  auto gave_up = [&]() {
    dead = true;
    *(volatile int*)p.status = 1;
  };
  cluster.sync();  // barriers are initialised, parameters in place
  for (int it = 1; it <= p.iters; ++it) {
    const int buf = it & 1;
    const uint32_t parity = (uint32_t)((it - 1) & 1);
    if (tid == 0) {
      if (n_owned > 0) apex::mbar_expect_tx(&s_bar_in, (uint32_t)n_owned * 32u * 8u);
      apex::mbar_expect_tx(&s_bar_tot, (uint32_t)P * 8u);
    }
    const int par_i = tid & (kMaxParams - 1), quarter = tid / kMaxParams;
    double acc = 0.0;
    const bool wide = (s_wide[0] | s_wide[1]) != 0;
    for (int base = 0; base < n_cta; base += kTokPass) {
      const int n_tok = min(kTokPass, n_cta - base);
      {
        const int tl = tid >> 3, q = tid & 7;
        const bool on = tl < n_tok;
        double s0 = 0.0, s1 = 0.0;  // (experts beyond N have weight 0)
#pragma unroll
        for (int m = 0; m < NM; ++m) {
          const double x = CACHED ? s_x[(base + tl) * LDX + q + 8 * m] : xg[(size_t)(base + (on ? tl : 0)) * N + min(q + 8 * m, N - 1)];
          if (m & 1) s1 = fma(x, s_w[q + 8 * m], s1);
          else s0 = fma(x, s_w[q + 8 * m], s0);
        }
        double s = s0 + s1;
        s = shfl_xor_add(s, 1);
        s = shfl_xor_add(s, 2);
        s = shfl_xor_add(s, 4);
        const int ds = on ? (CACHED ? s_ds[base + tl] : dsg[base + tl]) : 0;
        double gsum = 0.0;
        if (!wide && fabs(s) <= kExpRange) {
          const double es = exp(s);
          double g[NM];
#pragma unroll
          for (int m = 0; m < NM; ++m) g[m] = reciprocal(fma(es, s_etheta[q + 8 * m], 1.0));  // (thresholds beyond the last: unused)
#pragma unroll
          for (int m = 0; m < NM; ++m) {
            const int dl = q + 8 * m;
            const double v = on && dl < nth ? (g[m] - (dl >= ds ? 1.0 : 0.0)) * inv_T : 0.0;  // d loss / d z
            s_g[dl * kLdG + tl] = v;
            gsum += v;
          }
        } else {
          for (int dl = q; dl < nth; dl += 8) {
            const double v = on ? (1.0 / (1.0 + exp(s - s_theta[dl])) - (dl >= ds ? 1.0 : 0.0)) * inv_T : 0.0;
            s_g[dl * kLdG + tl] = v;
            gsum += v;
          }
        }
        __syncwarp();
        gsum = shfl_xor_add(gsum, 1);
        gsum = shfl_xor_add(gsum, 2);
        gsum = shfl_xor_add(gsum, 4);
        if (q == 0) s_gsum[tl] = gsum;
      }
      __syncthreads();
      const int u_lo = quarter * (kTokPass / 4);
      double a[4] = {0.0, 0.0, 0.0, 0.0};
      if (par_i < N) {  // z = theta - w.x: d z / d w_i = -x_i  (tokens beyond the last have gsum = 0)
#pragma unroll
        for (int u = 0; u < kTokPass / 4; u += 2) {
          const double2 gs = *reinterpret_cast<const double2*>(s_gsum + u_lo + u);
          const double x0 = CACHED ? s_x[(base + u_lo + u) * LDX + par_i] : xg[(size_t)(base + min(u_lo + u, n_tok - 1)) * N + par_i];
          const double x1 = CACHED ? s_x[(base + u_lo + u + 1) * LDX + par_i] : xg[(size_t)(base + min(u_lo + u + 1, n_tok - 1)) * N + par_i];
          a[u & 3] = fma(-gs.x, x0, a[u & 3]);
          a[(u + 1) & 3] = fma(-gs.y, x1, a[(u + 1) & 3]);
        }
      } else if (par_i < P) {
        const double* g = s_g + (par_i - N) * kLdG + u_lo;
#pragma unroll
        for (int u = 0; u < kTokPass / 4; ++u) a[u & 3] += g[u];
      }
      acc += (a[0] + a[1]) + (a[2] + a[3]);
      if (base + kTokPass < n_cta) __syncthreads();  // (the pass's scratch is rewritten by the next)
    }
    if (par_i < P) send(&s_in[buf][par_i % kOwned][crank * 4 + quarter], &s_bar_in, (uint32_t)(par_i / kOwned), acc);
    b1 *= 0.9;
    b2 *= 0.999;
    const double ic1 = 1.0 / (1.0 - b1), ic2 = 1.0 / (1.0 - b2);
    // owner: a warp adds a parameter's 32 contributions, then the clusters' sums, and sends the total to its cluster
    if (n_owned > 0) {
      double v = 0.0;
      if (warp < n_owned) {
        if (!dead && !apex::mbar_wait(&s_bar_in, parity, nullptr, kWaitLimitNs)) gave_up();
        __syncwarp();
        v = s_in[buf][warp][lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = shfl_xor_add(v, o);
      }
      if (n_clusters > 1) {
        if (lane == 0 && warp < kOwned) s_own[warp] = v;
        __syncthreads();
        if (warp < n_clusters) {  // warp c: cluster c's block of records
          ulonglong2* rec = p.rec + (((size_t)buf * kCluster + crank) * kMaxClusters + warp) * kOwned + lane;
          if (warp == my_cluster) {
            if (lane < kOwned) {
              put_record(rec, s_own[lane], (unsigned long long)it);
              s_clu[warp][lane] = s_own[lane];
            }
          } else if (lane < kOwned) {
            ulonglong2 r = get_record(rec);
            if (r.y != (unsigned long long)it && !dead) {
              const unsigned long long t0 = apex::globaltimer_ns();
              for (uint32_t n = 1; r.y != (unsigned long long)it; ++n) {
                if ((n & 63u) == 0u && ((long long)(apex::globaltimer_ns() - t0) > kWaitLimitNs || *(volatile int*)p.status)) {
                  gave_up();
                  break;
                }
                r = get_record(rec);
              }
            }
            s_clu[warp][lane] = __longlong_as_double((long long)r.x);
          }
        }
        __syncthreads();
        v = warp < kOwned && lane < n_clusters ? s_clu[lane][warp] : 0.0;
#pragma unroll
        for (int o = kMaxClusters / 2; o > 0; o >>= 1) v = shfl_xor_add(v, o);
      }
      if (warp < n_owned && lane < kCluster) send(&s_tot[buf][crank * kOwned + warp], &s_bar_tot, (uint32_t)lane, v);
    }
    if (tid < 2 * APEX_MAX_EXPERTS && !dead && !apex::mbar_wait(&s_bar_tot, parity, nullptr, kWaitLimitNs)) gave_up();
    __syncwarp();
    // theta_j = t0 + sum_{i <= j} softplus(u_i):  d / d t0 = sum_j g_theta[j],  d / d u_j = sigmoid(u_j) sum_{m >= j} g_theta[m]
    if (tid < 64) {
      double lo = lane < nth ? s_tot[buf][N + lane] : 0.0, hi = lane + 32 < nth ? s_tot[buf][N + lane + 32] : 0.0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {  // suffix sums, by both warps
        const double a = __shfl_down_sync(0xffffffffu, lo, o), b = __shfl_down_sync(0xffffffffu, hi, o);
        if (lane + o < 32) {
          lo += a;
          hi += b;
        }
      }
      lo += __shfl_sync(0xffffffffu, hi, 0);
      const double g = (warp == 0 ? lo : hi) * sig;
      mom = 0.9 * mom + 0.1 * g;
      var = 0.999 * var + 0.001 * g * g;
      if (has_u) par = par - p.lr * (mom * ic1) * reciprocal(sqrt(var * ic2) + 1e-8);
      double sp = par;  // t0 leads the prefix sums
      if (tid > 0) {
        const double e = exp(-fabs(par));
        sp = fmax(par, 0.0) + log1p(e);
        sig = (par >= 0.0 ? 1.0 : e) * reciprocal(1.0 + e);
      }
      s_sp[tid] = sp;
      asm volatile("bar.sync 1, 64;" ::: "memory");
      lo = lane < nth ? s_sp[lane] : 0.0;
      hi = lane + 32 < nth ? s_sp[lane + 32] : 0.0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {  // theta: prefix sums
        const double a = __shfl_up_sync(0xffffffffu, lo, o), b = __shfl_up_sync(0xffffffffu, hi, o);
        if (lane >= o) {
          lo += a;
          hi += b;
        }
      }
      hi += __shfl_sync(0xffffffffu, lo, 31);
      const double th = warp == 0 ? lo : hi;
      s_theta[tid] = th;
      s_etheta[tid] = exp(-th);
      const bool far = __any_sync(0xffffffffu, has_u && !(fabs(th) <= kExpRange));
      if (lane == 0) s_wide[warp] = far;
    } else if (has_w) {
      const double g = s_tot[buf][tid - 64];
      mom = 0.9 * mom + 0.1 * g;
      var = 0.999 * var + 0.001 * g * g;
      par = par - p.lr * (mom * ic1) * reciprocal(sqrt(var * ic2) + 1e-8);
      s_w[tid - 64] = par;
    }
    __syncthreads();
  }
  if (blockIdx.x == 0) {
    if (has_w) p.out[tid - 64] = par;
    if (has_u) p.out[N + tid] = s_theta[tid];
  }
  cluster.sync();  // nobody leaves while a peer may still send into its shared memory
}

typedef void (*FitKernel)(const FitParams);
template <bool CACHED>
FitKernel fit_kernel(int nm) {
  switch (nm) {
    case 1: return cdf_fit_kernel<1, CACHED>;
    case 2: return cdf_fit_kernel<2, CACHED>;
    case 3: return cdf_fit_kernel<3, CACHED>;
    case 4: return cdf_fit_kernel<4, CACHED>;
    case 5: return cdf_fit_kernel<5, CACHED>;
    case 6: return cdf_fit_kernel<6, CACHED>;
    case 7: return cdf_fit_kernel<7, CACHED>;
    default: return cdf_fit_kernel<8, CACHED>;
  }
}

void say(char* err, size_t err_len, const char* msg) {
  if (err && err_len) snprintf(err, err_len, "%s", msg);
}

}  // namespace

extern "C" int apex_fit_cdf(const double* X_dev, const int32_t* dstar_dev, int T, int N, int k, int iters, double lr,
                            float* w_host, float* theta_host, void* stream, char* err, size_t err_len) {
  say(err, err_len, "");
  if (!X_dev || !dstar_dev || !w_host || !theta_host || T < 1 || N < 1 || N > APEX_MAX_EXPERTS || k < 1 || k > N || iters < 1 ||
      !(lr > 0.0)) {
    say(err, err_len, "apex_fit_cdf: bad argument (N <= 64, 1 <= k <= N, T >= 1, iters >= 1, lr > 0)");
    return APEX_EINVAL;
  }
  cudaStream_t cs = (cudaStream_t)stream;
  const int nth = N - k + 1, P = N + nth;
  // start: w = 0, theta = logit of the empirical distribution of delta*, increments at least 1e-3
  std::vector<int32_t> ds(T);
  cudaError_t e = cudaMemcpyAsync(ds.data(), dstar_dev, sizeof(int32_t) * T, cudaMemcpyDeviceToHost, cs);
  if (e == cudaSuccess) e = cudaStreamSynchronize(cs);
  if (e != cudaSuccess) {
    say(err, err_len, cudaGetErrorString(e));
    return APEX_ECUDA;
  }
  std::vector<double> init(P, 0.0), th0(nth);
  std::vector<long long> at_most(nth, 0);  // tokens with delta* <= j
  for (int t = 0; t < T; ++t)
    if (ds[t] < nth) ++at_most[ds[t] > 0 ? ds[t] : 0];
  for (int j = 1; j < nth; ++j) at_most[j] += at_most[j - 1];
  for (int j = 0; j < nth; ++j) {
    const long long c = at_most[j];
    double f = (double)c / (double)T;
    f = f < 1e-3 ? 1e-3 : (f > 1.0 - 1e-3 ? 1.0 - 1e-3 : f);
    th0[j] = std::log(f / (1.0 - f));
  }
  init[N] = th0[0];
  for (int j = 1; j < nth; ++j) {
    const double inc = th0[j] - th0[j - 1] > 1e-3 ? th0[j] - th0[j - 1] : 1e-3;
    init[N + j] = std::log(std::expm1(inc));  // inverse softplus
  }
  std::vector<double> theta_init(nth);
  theta_init[0] = init[N];
  double csum = 0.0;
  for (int j = 1; j < nth; ++j) {
    const double u = init[N + j];
    csum += std::fmax(u, 0.0) + std::log1p(std::exp(-std::fabs(u)));
    theta_init[j] = init[N] + csum;
  }

  FitParams p{};
  p.X = X_dev; p.dstar = dstar_dev;
  p.T = T; p.N = N; p.nth = nth; p.lr = lr; p.iters = iters;
  double* buf = nullptr;
  int rc = APEX_OK;
  auto fail = [&](cudaError_t ce) {
    say(err, err_len, cudaGetErrorString(ce));
    rc = ce == cudaErrorMemoryAllocation ? APEX_ENOMEM : APEX_ECUDA;
  };
  do {
    // Clusters: 64 tokens per CTA while the GPU holds them all at once (they wait for one another: cooperative launch)
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.stream = cs;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kCluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeCooperative;
    attr[1].val.cooperative = 1;
    cfg.attrs = attr;
    int clusters = (T + kTokPass * kCluster - 1) / (kTokPass * kCluster);
    clusters = clusters > kMaxClusters ? kMaxClusters : clusters;
    constexpr size_t cache_limit = 64 * 1024;  // (and 46 KB of static shared memory: two CTAs to an SM, so 16 clusters fit)
    const int nm = (N + 7) / 8;
    FitKernel kernel = nullptr;
    for (;; --clusters) {
      const int per = (T + clusters * kCluster - 1) / (clusters * kCluster);
      p.tok_per_cta = (per + kTokPass - 1) / kTokPass * kTokPass;
      const size_t want = (size_t)p.tok_per_cta * (fit_ldx(nm) * sizeof(double) + sizeof(int32_t));
      kernel = want <= cache_limit ? fit_kernel<true>(nm) : fit_kernel<false>(nm);
      cfg.dynamicSmemBytes = want <= cache_limit ? want : 0;
      cfg.gridDim = dim3(kCluster, 1, 1);
      cfg.numAttrs = 1;
      int fit = 0;
      if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cache_limit)) != cudaSuccess) break;
      if ((e = cudaOccupancyMaxActiveClusters(&fit, kernel, &cfg)) != cudaSuccess) break;
      if (clusters <= fit || clusters == 1) break;
    }
    if (e != cudaSuccess) { fail(e); break; }
    cfg.gridDim = dim3(kCluster * clusters, 1, 1);
    cfg.numAttrs = 2;
    const size_t n_rec = 2 * (size_t)kMaxClusters * kMaxParams;
    if ((e = apex::workspace_alloc(reinterpret_cast<void**>(&buf), n_rec * sizeof(ulonglong2) + (2 + 2 * (size_t)P + nth) * sizeof(double), cs)) != cudaSuccess) { fail(e); break; }
    p.rec = reinterpret_cast<ulonglong2*>(buf);
    double* rest = reinterpret_cast<double*>(p.rec + n_rec);
    p.status = reinterpret_cast<int*>(rest);
    double* init_dev = rest + 2;
    p.init = init_dev; p.theta0 = init_dev + P; p.out = init_dev + P + nth;
    init.insert(init.end(), theta_init.begin(), theta_init.end());
    if ((e = cudaMemsetAsync(buf, 0, n_rec * sizeof(ulonglong2) + sizeof(double), cs)) != cudaSuccess) { fail(e); break; }
    if ((e = cudaMemcpyAsync(init_dev, init.data(), sizeof(double) * (P + nth), cudaMemcpyHostToDevice, cs)) != cudaSuccess) { fail(e); break; }
    if ((e = cudaLaunchKernelEx(&cfg, kernel, p)) != cudaSuccess) { fail(e); break; }
    std::vector<double> out(P);  // w | theta
    if ((e = cudaMemcpyAsync(out.data(), p.out, sizeof(double) * P, cudaMemcpyDeviceToHost, cs)) != cudaSuccess) { fail(e); break; }
    int status = 0;
    if ((e = cudaMemcpyAsync(&status, p.status, sizeof(int), cudaMemcpyDeviceToHost, cs)) != cudaSuccess) { fail(e); break; }
    apex::workspace_free(buf, cs);  // (in front of the synchronisation, at which the pool lets go of what it need not keep)
    buf = nullptr;
    if ((e = cudaStreamSynchronize(cs)) != cudaSuccess) { fail(e); break; }
    if (status != 0) {
      say(err, err_len, "apex_fit_cdf: a device-side wait ran out");
      rc = APEX_ECUDA;
      break;
    }
    for (int j = 0; j < N; ++j) w_host[j] = (float)out[j];
    float run = -INFINITY;
    for (int j = 0; j < nth; ++j) {  // fp32 rounding must not break the order
      const float t = (float)out[N + j];
      run = t > run ? t : run;
      theta_host[j] = run;
    }
  } while (false);
  if (buf) {
    apex::workspace_free(buf, cs);
    cudaStreamSynchronize(cs);
  }
  return rc;
}
