// Device helpers of the two kernels that run all layers of a token (kernels_decode.cu, kernels_decode_tiles.cu).
#ifndef APEX_DECODE_COMMON_CUH
#define APEX_DECODE_COMMON_CUH

#include "apex_internal.hpp"
#include "ptx.cuh"

namespace apex {

constexpr int kDecSmemTotal = 227 * 1024;  // shared memory of a CTA

#ifdef APEX_TIMELINE
// per CTA and layer (the warp that writes last wins): 0 layer start, 1 W_p logit sent, 2 candidate mask out (poster),
// 3 own attention share landed, 4 W_r logit sent, 5 gate logits complete, 6 plan done, 7 first expert row landed, 8 last
// row consumed, 9 layer counted in, 10 candidate record posted (poster), 11 warps' partial y in shared memory, 12 cluster's
// partial y complete, 13 y added, 14 both counters passed (W_r), 15 previous layer's counter passed (W_p)
extern __device__ unsigned long long g_dec_tl[160][64][16];
#define DTL(i) do { if (lane == 0 && blockIdx.x < 160 && l < 64) g_dec_tl[blockIdx.x][l][(i)] = globaltimer_ns(); } while (0)
#else
#define DTL(i) do { } while (0)
#endif

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// one 32-bit value into the shared memory of CTA `rank` of this cluster; the receiver's mbarrier counts its 4 bytes
__device__ __forceinline__ void st_async_remote(void* local_dst, uint64_t* local_bar, uint32_t rank, float value) {
  uint32_t ra, rb;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(smem_u32(local_dst)), "r"(rank));
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(smem_u32(local_bar)), "r"(rank));
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(ra), "r"(__float_as_uint(value)),
               "r"(rb)
               : "memory");
}
__device__ __forceinline__ void red_release_gpu_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void red_relaxed_gpu_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint32_t ld_acquire_gpu_u32(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned ld_volatile_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.volatile.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

}  // namespace apex

#endif  // APEX_DECODE_COMMON_CUH
