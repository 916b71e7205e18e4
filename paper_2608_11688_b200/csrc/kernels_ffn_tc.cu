// Batched expert FFN on the 5th-generation tensor cores (tcgen05 + TMEM), for decode steps with many
// tokens (Sec. V-B: several concurrent requests are decoded as one batch).
//
// With B tokens per step an expert serves several tokens, so its weights should be read once and
// applied to all of them: a grouped GEMM, one group per executed expert (plus the shared expert).
// The step is still HBM-bound (a few tens of flop per weight byte at most), so the kernel is
// organised around streaming the weights once; the tensor cores only keep arithmetic off the
// critical path.  "Swap-AB": the weight rows are the MMA's M dimension, the group's tokens are N (16..128),
// so a small token count does not waste a 128-row tile.
//
//   gate/up    G, U [128 x n] = W_gate/up[128 rows of I x d] . X^T       accumulators in TMEM; the rows of X (h' in bf16)
//              a = g_pair * silu(G) * U  (fp32) is kept as TWO bf16        are gathered by token index by the TMA loads
//              planes, a_hi = bf16(a) and a_lo = bf16(a - a_hi), so feeding it back to the tensor cores loses 2^-17,
//              not 2^-9                                                    -> global scratch (L2)
//   down       D [256 cols of d x 2n] = downT[K x 256]^T . [a_hi ; a_lo]^T  (downT is MN-major, two M = 128 halves; both
//              y[token][col] += D[:, j] + D[:, n + j]      fp32 atomics       planes in one MMA: N = 2n)
//
// Every CTA first derives the step's plan (execution sets, tokens per expert, pair list) from the gate's outputs.
// ONE persistent kernel runs both projections: the units of both projections form one list, gate/up first, and the CTAs take
// tickets.  A down unit needs its group's intermediate, so its activations are loaded once the group's gate/up units have
// been counted in (its weights, which wait for nothing, are already on their way); the tickets are handed out in list
// order, so whatever a unit waits for is already running somewhere and no co-residency is assumed.  As two kernels the
// step lost a partial round of units at the end of each (748 units of 1 MB on 148 SMs: 5.05 rounds) and a pipeline
// refill in between; with the plan and gather kernels in front 256 us against 200 at B = 256 (60 experts of 17 MB and a shared
// one of 69 MB: 1.11 GB), 124 against 93 at B = 8.
//
// A pipeline stage is 64 K values of two 128-row weight tiles (gate and up | the two column halves of downT: 32 KB) and
// of the group's activations.  Roles: a warp loads weights and takes the tickets, a warp loads activations, a thread
// issues MMAs, four warps run the epilogue out of TMEM.  Accumulators are double-buffered in TMEM (2 x 256 columns), so
// the epilogue of one unit overlaps the MMAs of the next.  An MMA with M = 128, K = 16 takes 47 cycles up to N = 48 and
// 67 at N = 128 (measured), eight per stage, against 1400 cycles of an SM's share of HBM per 32 KB: the streaming bounds
// the bf16 step at every batch size.  Every wait is bounded.
//
// Operands reach shared memory through TMA tensor maps with the 128-byte swizzle and are consumed
// by tcgen05.mma through shared-memory descriptors (K-major for gate, up, X, A; MN-major for downT).
//
// Quantised stores (e4m3 codes with a scale per row vector, e2m1 codes with a power-of-two scale per 32
// elements) take the same path with one more role: the weights arrive as raw code bytes in a ring of their own, in tiles
// of 128 bytes per row (two or four stages' worth; boxes of one stage, 64 or 32 bytes wide, had the TMA requests of
// short rows and eight-fold re-read scale bytes as the pace), and sixteen converter warps expand them to bf16 in
// the swizzled operand layout the MMA descriptors expect.  Both code sets are exact in bf16 (3 and 1 mantissa bits), and
// so is an e2m1 value times its power-of-two scale, so the tensor cores see the dequantised weights exactly; the
// per-vector fp32 scales of an e4m3 row are not exact in bf16 and are applied in fp32 instead: gate and up scales to the
// accumulators, the down scale folded into the intermediate before it is split into its two bf16 planes.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>

#include "apex_internal.hpp"
#include "ptx.cuh"
#include "token_plan.cuh"

namespace apex {

namespace {

constexpr int kWWarp = 0;      // weight loads, tickets
constexpr int kBWarp = 1;      // activation loads
constexpr int kMmaWarp = 2;    // MMA issue, TMEM owner
constexpr int kEpiWarp0 = 3;   // four epilogue warps
constexpr int kCvWarp0 = 7;    // sixteen converter warps (quantised stores only): four per scheduler hide the latency of shared memory and ALU
constexpr int kCvThreads = 512;
__host__ __device__ constexpr int tc_threads(int qf) { return kCvWarp0 * 32 + (qf ? kCvThreads : 0); }
// Gate/up units of kRowsSmall rows: a stage takes tc_wide(QF) K tiles (8 KB of operand each), which on the quantised stores
// is a whole raw tile.
constexpr int kRowsSmall = 32;
constexpr int kHandBytes = 2 * 16 * 32 * 4;  // their epilogue: up values handed from one warp to another, two batches of 16 columns
__host__ __device__ constexpr int tc_wide(int qf) { return qf == 1 ? 2 : 4; }
constexpr int kKTile = 64;           // K values per stage (128 bytes of bf16: one swizzle span)
constexpr int kABytes = 2 * 128 * 128;  // the two weight tiles of a stage
constexpr int kMaxStages = 8, kMaxRaw = 4;
constexpr int kARowsPerLoad = 16;    // rows per box of the intermediate, and of X where the tokens follow one another: the granularity of N
constexpr int kUnitRing = 4;         // unit descriptors between the ticket taker and the other roles
// quantised stores: stages fed by one raw tile, and its bytes (codes, e2m1 block scales)
__host__ __device__ constexpr int tc_sub(int qf) { return qf == 2 ? 4 : qf == 1 ? 2 : 1; }
__host__ __device__ constexpr int tc_raw_bytes(int qf) { return qf == 2 ? 32768 + 4096 : qf == 1 ? 32768 : 0; }
// K tiles per down unit, at most: small enough for an even end of the launch, large enough that a unit's epilogue and
// ticket stay small beside it
constexpr int kDownTiles = 16, kDownTilesQ = 8;  // bf16 | quantised

__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, int c3, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(smem_u32(dst)),
      "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int c0, int c1, uint64_t* bar) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(smem_u32(dst)),
               "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1)
               : "memory");
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, uint64_t* bar) {
  asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(smem_u32(dst)),
               "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2)
               : "memory");
}
// four rows of a [rows][cols] map (box one row high), 64 columns each, to four consecutive 128-byte rows
__device__ __forceinline__ void tma_gather4(void* dst, const CUtensorMap* map, int c0, int r0, int r1, int r2, int r3, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];" ::"r"(
          smem_u32(dst)),
      "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(r0), "r"(r1), "r"(r2), "r"(r3)
      : "memory");
}
// Expanding codes to bf16.  A code's exponent and mantissa bits, placed at the top of a bf16's mantissa and the bottom of
// its exponent field, read as the code's value times 2^(code bias - 127), subnormal codes included (they become bf16
// subnormals, which the multiply does not flush); a multiply by a power of two puts the exponent right and is exact.
// The integer pipe (16 lanes per scheduler and cycle) is the converters' bound, so the fields are masked there and moved by
// multiply-adds, which run beside it (by kernel parameters: multiplications by constants the compiler knows would be
// turned back into shifts): two masks per pair of codes instead of five integer operations.  A pair is made of
// the codes that lie 16 bits apart in their word, so the values come out in the order 0 2 1 3 (e4m3: within four) and
// 0 4 1 5 2 6 3 7 (e2m1: within eight): the activations a gate/up tile meets are stored in that order, and for a
// down tile, whose codes run along the output columns, the epilogue undoes it.
__host__ __device__ constexpr int tc_column_of(int qf, int j) {  // value at position j
  return qf == 2 ? (j & ~7) | ((j & 1) << 2) | ((j >> 1) & 3) : qf == 1 ? (j & ~3) | ((j & 1) << 1) | ((j >> 1) & 1) : j;
}
__device__ __forceinline__ uint32_t mul_bf16x2(uint32_t a, uint32_t b) {
  uint32_t o;
  asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(o) : "r"(a), "r"(b));
  return o;
}
// (c & sign) * up_s + (c & rest) * up_r: fields that do not meet
__device__ __forceinline__ uint32_t place(uint32_t c, uint32_t sign, uint32_t up_s, uint32_t rest, uint32_t up_r) {
  const uint32_t o = (c & sign) * up_s + (c & rest) * up_r;
  return o;
}
// four e4m3 codes (s eeee mmm, bias 7) -> bf16 pairs (0, 2), (1, 3)
__device__ __forceinline__ void e4m3x4_to_bf16(const TcShifts& k, uint32_t c, uint32_t& o0, uint32_t& o1) {
  const uint32_t e = 0x7B807B80u;  // 2^120, twice
  o0 = mul_bf16x2(place(c, 0x00800080u, k.up8, 0x007f007fu, k.up4), e);
  o1 = mul_bf16x2(place(c >> 8, 0x00800080u, k.up8, 0x007f007fu, k.up4), e);
}
// the block scale 2^(sb - 127) of e2m1 codes times 2^126, twice; for scales above 2 (never produced for weights of ordinary
// size) that exceeds bf16: half the exponent, to be applied twice
__device__ __forceinline__ uint32_t e2m1_scale(uint32_t sb, uint32_t& again) {
  uint32_t m = sb ? (sb + 126u) << 7 : 0u;
  again = 0x3F803F80u;
  if (sb > 128u) {
    m = 253u << 7;  // 2^126
    again = sb << 7;
    again |= again << 16;
  }
  return m | (m << 16);
}
// eight e2m1 codes (s ee m, bias 1; the even element in the low nibble of its byte) -> bf16 pairs (0, 4), (1, 5), (2, 6), (3, 7)
template <bool TWICE>
__device__ __forceinline__ uint4 e2m1x8_to_bf16(const TcShifts& k, uint32_t c, uint32_t m, uint32_t again) {
  const uint32_t c2 = c >> 8;
  uint4 o;
  o.x = mul_bf16x2(place(c, 0x00080008u, k.up12, 0x00070007u, k.up6), m);
  o.y = mul_bf16x2(place(c, 0x00800080u, k.up8, 0x00700070u, k.up2), m);
  o.z = mul_bf16x2(place(c2, 0x00080008u, k.up12, 0x00070007u, k.up6), m);
  o.w = mul_bf16x2(place(c2, 0x00800080u, k.up8, 0x00700070u, k.up2), m);
  if (TWICE) {
    o.x = mul_bf16x2(o.x, again);
    o.y = mul_bf16x2(o.y, again);
    o.z = mul_bf16x2(o.z, again);
    o.w = mul_bf16x2(o.w, again);
  }
  return o;
}
// the 32 codes of one block
__device__ __forceinline__ void e2m1x32_to_bf16(const TcShifts& k, const uint4& v, uint32_t sb, uint4 (&o)[4]) {
  uint32_t again;
  const uint32_t m = e2m1_scale(sb, again);
  if (__any_sync(0xffffffffu, sb > 128u)) {
    o[0] = e2m1x8_to_bf16<true>(k, v.x, m, again);
    o[1] = e2m1x8_to_bf16<true>(k, v.y, m, again);
    o[2] = e2m1x8_to_bf16<true>(k, v.z, m, again);
    o[3] = e2m1x8_to_bf16<true>(k, v.w, m, again);
  } else {
    o[0] = e2m1x8_to_bf16<false>(k, v.x, m, again);
    o[1] = e2m1x8_to_bf16<false>(k, v.y, m, again);
    o[2] = e2m1x8_to_bf16<false>(k, v.z, m, again);
    o[3] = e2m1x8_to_bf16<false>(k, v.w, m, again);
  }
}
// shared-memory matrix descriptor, 128-byte swizzle (layout type 2), version 1
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
// instruction descriptor: bf16 x bf16 -> fp32, M x N, optional MN-major A
__device__ __forceinline__ uint32_t umma_idesc(int M, int N, int a_mn_major) {
  uint32_t d = 0;
  d |= 1u << 4;    // D fp32
  d |= 1u << 7;    // A bf16
  d |= 1u << 10;   // B bf16
  d |= (uint32_t)a_mn_major << 15;
  d |= (uint32_t)(N >> 3) << 17;
  d |= (uint32_t)(M >> 4) << 24;
  return d;
}
__device__ __forceinline__ void umma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem_d),
               "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
               : "memory");
}
// A from TMEM (lane = row, a 32-bit column holds two consecutive K values)
__device__ __forceinline__ void umma_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(tmem_d),
               "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
               : "memory");
}
// One lane of a converged warp.  MMAs are issued under this predicate in warp-uniform code, so descriptors stay in uniform
// registers; issued from `if (lane == 0)` an MMA cost 47 cycles of moves whatever its size, and three times that beside
// busy converter warps.
__device__ __forceinline__ bool elect_one() {
  uint32_t r;
  asm volatile("{\n.reg .pred e;\nelect.sync _|e, 0xffffffff;\nselp.u32 %0, 1, 0, e;\n}" : "=r"(r));
  return r != 0;
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15};" ::"r"(r[0]), "r"(r[1]),
      "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]),
      "r"(r[14]), "r"(r[15]), "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

#ifdef APEX_TIMELINE
// per CTA and unit: 0 ticket taken, 1 first weights landed (MMA thread), 2 MMAs issued, 3 accumulators complete, 4 epilogue done
__device__ unsigned long long g_tc_tl[148][64][8];
#define TCTL(u, i) do { if ((u) < 64u && blockIdx.x < 148) g_tc_tl[blockIdx.x][(u)][(i)] = globaltimer_ns(); } while (0)
#else
#define TCTL(u, i) do { } while (0)
#endif

// weight maps, by projection (boxes differ in height) and store (slots, shared expert)
struct TcWeightMaps {
  CUtensorMap codes[2][2], scales[2][2];
};
// One unit of work: the (part of a) group, the M block and the K-tile range of one of the projections (phase 1: gate/up,
// 2: down; 0: the list is at its end).
struct GroupDesc {
  int expert, pair_off, n_tok;
};
struct UnitDesc {
  int phase, group, expert, pair_off, n_tok, blk, kt_begin, kt_end;
};
// TMEM.  bf16 stores: two accumulator buffers of 256 columns.  Quantised stores: two of 128 columns, which a unit with more
// than 64 (gate/up) or 32 (down) tokens takes together, and above them the gate/up weight tiles of the operand stages
// (64 columns each).  The MMA thread and the epilogue walk the units with the same bookkeeping.
__host__ __device__ constexpr uint32_t tc_acc_cols(int qf) { return qf ? 128u : 256u; }
constexpr uint32_t kTmemA = 256;
// Position in a ring: slot, and the parity of its current round (a "full" barrier is waited for with it, an "empty" barrier
// with the other, which passes at once in the first round).  Counters, not divisions by the run-time depth: those were a
// third of the converters' instructions.
struct RingPos {
  uint32_t s = 0, parity = 0;
  __device__ __forceinline__ void next(uint32_t depth) {
    if (++s == depth) {
      s = 0;
      parity ^= 1u;
    }
  }
};
struct AccBuffers {
  uint32_t next = 0, uses[2] = {0, 0};  // buffer of the next unit that needs one; units that have used each
};
template <int QF>
__device__ __forceinline__ bool unit_is_wide(const UnitDesc& ud) { return QF != 0 && ud.n_tok > (ud.phase == 1 ? 64 : 32); }

}  // namespace

// tm_w: weights of the slots and of the shared expert.  bf16: boxes of 64 columns x 64 rows; quantised: the raw row
// bytes, boxes of 128 bytes x 128 rows, and the same bytes in boxes of 16 bytes x 128 rows (e2m1 block scales); for gate/up
// units of fewer rows, boxes of that many.
// tm_x, tm_xc: h' in bf16, boxes of one row (gathered) and of kARowsPerLoad.  tm_act: the intermediate, plane a_lo below plane a_hi.
template <int QF>
__global__ void __launch_bounds__(tc_threads(QF), 1)
ffn_tc_kernel(const __grid_constant__ TcWeightMaps tm_w, const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_xc,
              const __grid_constant__ CUtensorMap tm_act, const TcParams p) {
  SPAN_BEGIN();
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  constexpr int SUB = tc_sub(QF);
  constexpr int RAW_BYTES = tc_raw_bytes(QF), WIDE = tc_wide(QF);
  const int STAGE_BYTES = p.stage_bytes, NS = p.nstage, NR = p.nraw;
  uint8_t* raw_ring = smem + (size_t)NS * STAGE_BYTES;
  __shared__ uint64_t full[kMaxStages], empty[kMaxStages], rawfull[kMaxRaw], rawempty[kMaxRaw], tmem_full[2], tmem_empty[2];
  __shared__ uint64_t unit_full[kUnitRing], unit_empty[kUnitRing];
  __shared__ UnitDesc s_unit[kUnitRing];
  __shared__ uint32_t tmem_base_s;
  __shared__ int s_abort;
  __shared__ uint2 s_end[3 + (QF ? kCvThreads / 32 : 0)];  // slot and parity at which each role that walks a ring has stopped: weights, activations, MMA, converters
  __shared__ int s_u[2][APEX_MAX_EXPERTS + 1], s_units[2];  // per projection: units before each group's in list order; all units
  __shared__ GroupDesc s_grp[APEX_MAX_EXPERTS + 1];         // executed experts, then the shared one
  constexpr int kTokWords = APEX_MAX_BATCH / 32;
  __shared__ unsigned s_mask[APEX_MAX_EXPERTS][kTokWords];  // tokens of each expert
  __shared__ short s_off[APEX_MAX_EXPERTS][kTokWords];
  __shared__ float s_inv[APEX_MAX_BATCH];                // what its gates are divided by
  __shared__ unsigned long long s_union[2];              // of the routed sets, of the execution sets
  __shared__ uint8_t s_tok[APEX_MAX_BATCH * (APEX_MAX_TOPK + 1)];  // token of each pair

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int N = p.f.N, d = p.f.d;

  if (tid == 0) {
    s_abort = 0;
    s_union[0] = s_union[1] = 0ull;
    for (int s = 0; s < kMaxStages; ++s) {
      mbar_init(&full[s], QF ? 1 + kCvThreads / 32 : 2);  // the activations' bytes, and the weights' (bytes, or the converter warps)
      mbar_init(&empty[s], 1);
    }
    for (int r = 0; r < kMaxRaw; ++r) {
      mbar_init(&rawfull[r], 1);
      mbar_init(&rawempty[r], kCvThreads / 32);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tmem_full[b], 1);
      mbar_init(&tmem_empty[b], 128);
    }
    for (int u = 0; u < kUnitRing; ++u) {
      mbar_init(&unit_full[u], 1);
      mbar_init(&unit_empty[u], 6 + (QF ? kCvThreads / 32 : 0));  // every warp that reads the descriptor
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int ph = 0; ph < 2; ++ph) {
      for (int st = 0; st <= (p.f.run_shared ? 1 : 0); ++st) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_w.codes[ph][st]) : "memory");
        if (QF == 2) asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_w.scales[ph][st]) : "memory");
      }
    }
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_x) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_act) : "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // Slot-ready flags of all resident experts in one round of loads (neither the flags nor the snapshot come from the
  // preceding kernel): the weight warp then skips the per-unit check, a system-scope load and a proxy fence on its path
  // at every unit boundary, for every expert already seen ready here.
  unsigned long long ready_mask = 0;
  if (warp == kWWarp) {
    bool r0 = false, r1 = false;
    const int e0 = lane, e1 = lane + 32;
    if (e0 < N) {
      const int sl = p.f.snap.expert_slot[e0];
      if (sl >= 0) r0 = (int32_t)(ld_acquire_sys(p.f.slot_ready + sl) - p.f.snap.need_gen[e0]) >= 0;
    }
    if (e1 < N) {
      const int sl = p.f.snap.expert_slot[e1];
      if (sl >= 0) r1 = (int32_t)(ld_acquire_sys(p.f.slot_ready + sl) - p.f.snap.need_gen[e1]) >= 0;
    }
    ready_mask = ((unsigned long long)__ballot_sync(0xffffffffu, r1) << 32) | __ballot_sync(0xffffffffu, r0);
    __syncwarp();  // (every lane's acquires, before the loads of whichever lane)
    asm volatile("fence.proxy.async.global;" ::: "memory");  // the tensor-map loads below read what the flags cover
  }
  tc_fence_before();
  __syncthreads();  // barriers initialised, TMEM allocated
  tc_fence_after();
  // everything above (barriers, TMEM, tensor-map prefetch, flags) is independent of the preceding kernel
  pdl_wait();
  pdl_launch_dependents();

  bool ok = true;
  auto give_up = [&]() {  // a wait ran out: tell the CTA, the other CTAs and the host
    atomicExch(&s_abort, 1);
    atomicExch(p.sync + kTcAbort, 1u);
    *p.f.mbox_status = 1u;
    if (p.f.stats) atomicAdd(&p.f.stats->timeouts, 1ull);
  };
  // ---- The step's plan, by every CTA for itself: all of them need it, and as a kernel of its own (one cluster, then the
  // boundary) it was 4 to 16 us before the first weight was asked for.  The weight warp meanwhile takes the first
  // tickets: a token each, whose h' it rounds to bf16 for the gathers and whose row of y it zeroes.
  const int B = p.f.B, k = p.f.k;
  int ticket = 0;
  auto unit_list_barrier = [&]() { asm volatile("bar.sync 4, %0;" ::"r"((int)blockDim.x) : "memory"); };
  if (warp == kWWarp) {
    ticket = lane == 0 ? (int)atomicAdd(p.sync + kTcTicket, 1u) : 0;
    for (;;) {
      const int t = __shfl_sync(0xffffffffu, ticket, 0);
      if (t >= B) break;
      if (lane == 0) ticket = (int)atomicAdd(p.sync + kTcTicket, 1u);
      const float4* h4 = reinterpret_cast<const float4*>(p.f.hpost + (size_t)t * d);
      float4* y4 = reinterpret_cast<float4*>(p.f.y + (size_t)t * d);
      uint4* x4 = reinterpret_cast<uint4*>(p.xb + (size_t)t * d);
      auto pack = [](float a, float b) {
        const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
        return *reinterpret_cast<const uint32_t*>(&v);
      };
#pragma unroll 4
      for (int i = lane; i < d / 8; i += 32) {
        const float4 a = __ldg(h4 + 2 * i), b = __ldg(h4 + 2 * i + 1);
        // in the order in which the converters leave the weights
        x4[i] = QF == 2   ? make_uint4(pack(a.x, b.x), pack(a.y, b.y), pack(a.z, b.z), pack(a.w, b.w))
                : QF == 1 ? make_uint4(pack(a.x, a.z), pack(a.y, a.w), pack(b.x, b.z), pack(b.y, b.w))
                          : make_uint4(pack(a.x, a.y), pack(a.z, a.w), pack(b.x, b.y), pack(b.z, b.w));
        if (!p.f.accumulate) y4[2 * i] = y4[2 * i + 1] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
      if (p.f.run_shared && p.f.shared_gate) {
        const float sg = shared_gate_weight(p.f.shared_gate, p.f.hpost + (size_t)t * d, d, lane);
        if (lane == 0) p.sgate[t] = sg;
      }
      __syncwarp();
      if (lane == 0) asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p.sync + kTcRows), "r"(1u) : "memory");
    }
    unit_list_barrier();
  } else {
    const int pt = tid - 32, pn = (int)blockDim.x - 32, pwarp = warp - 1, pwarps = pn / 32;
    auto plan_barrier = [&]() { asm volatile("bar.sync 3, %0;" ::"r"(pn) : "memory"); };  // everybody but the weight warp
    // a thread per token: K_r, the execution set (S6), the sum of its gates
    unsigned long long kr_all = 0ull, ex_all = 0ull;
    for (int w = pwarp; w * 32 < B; w += pwarps) {
      const int t = w * 32 + lane;
      const bool on = t < B;
      int id[APEX_MAX_TOPK];
      float al[APEX_MAX_TOPK];
#pragma unroll
      for (int j = 0; j < APEX_MAX_TOPK; ++j) id[j] = on && j < k ? __ldg(p.f.idx + (size_t)t * k + j) : -1;
#pragma unroll
      for (int j = 0; j < APEX_MAX_TOPK; ++j) al[j] = id[j] >= 0 ? __ldg(p.f.alpha + (size_t)t * N + id[j]) : 0.f;
      unsigned long long kr = 0ull;
      float den = 0.f;  // sum of the executed experts' weights
#pragma unroll
      for (int j = 0; j < APEX_MAX_TOPK; ++j) {
        if (id[j] >= 0) kr |= 1ull << id[j];
        den += al[j];
      }
      unsigned long long ex = kr;
      const unsigned long long resident = p.f.snap.resident_mask;
      if (on && p.f.mode == APEX_MODE_STALL_FREE && (kr & ~resident)) {
        // Algorithm 1: the |M| best remaining resident experts by router weight, i.e. by (logit descending, index ascending)
        ex = kr & resident;
        unsigned long long cand = resident & ~kr;
        const float* z = p.f.z_r + (size_t)t * N;
        for (int miss = __popcll(kr & ~resident); miss > 0 && cand; --miss) {
          int best = -1;
          float zb = 0.f;
          for (unsigned long long rest = cand; rest; rest &= rest - 1) {
            const int e = __ffsll((long long)rest) - 1;
            const float ze = __ldg(z + e);
            if (best < 0 || ze > zb) {
              best = e;
              zb = ze;
            }
          }
          ex |= 1ull << best;
          cand &= ~(1ull << best);
        }
        den = 0.f;
        for (unsigned long long rest = ex; rest; rest &= rest - 1) den += __ldg(p.f.alpha + (size_t)t * N + __ffsll((long long)rest) - 1);
      }
      if (!p.f.norm_topk) den = 1.f;
      if (on) s_inv[t] = den;
      kr_all |= kr;
      ex_all |= ex;
      // the transpose: lane e (and e + 32) keeps the tokens of its two experts as a 32-bit word
      const unsigned long long rx = on ? ex & p.f.run_mask : 0ull;
      unsigned m0 = 0u, m1 = 0u;
#pragma unroll
      for (int e = 0; e < 32; ++e) {
        const unsigned a = __ballot_sync(0xffffffffu, (rx >> e) & 1), b = __ballot_sync(0xffffffffu, (rx >> (e + 32)) & 1);
        if (lane == e) {
          m0 = a;
          m1 = b;
        }
      }
      s_mask[lane][w] = m0;
      s_mask[lane + 32][w] = m1;
      if (on && blockIdx.x == 0 && p.f.post_exec) {
        int pos = 0;
        for (unsigned long long rest = ex; rest; rest &= rest - 1, ++pos) {
          const int e = __ffsll((long long)rest) - 1;
          if (p.f.exec_idx) p.f.exec_idx[(size_t)t * k + pos] = e;
          if (p.f.exec_gate) p.f.exec_gate[(size_t)t * k + pos] = __ldg(p.f.alpha + (size_t)t * N + e) / den;
        }
        if (p.f.stats) {
          const int subst = __popcll(ex & ~kr), hits = __popcll(kr & resident);
          if (subst) atomicAdd(&p.f.stats->substitutions, (unsigned long long)subst);
          if (hits) atomicAdd(&p.f.stats->hits_R, (unsigned long long)hits);
        }
      }
    }
    if (blockIdx.x == 0 && p.f.post_exec) {
      atomicOr(&s_union[0], kr_all);
      atomicOr(&s_union[1], ex_all);
    }
    plan_barrier();
    if (tid == 32 && blockIdx.x == 0 && p.f.post_exec) {
      // the unions for the host: one 16-byte store each, with the sequence number
      const unsigned long long kr = s_union[0], ex = s_union[1];
      asm volatile("st.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p.f.mbox_rec), "r"((uint32_t)kr), "r"((uint32_t)(kr >> 32)), "r"(p.f.seq_value), "r"(0u) : "memory");
      asm volatile("st.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p.f.mbox_rec + 4), "r"((uint32_t)ex), "r"((uint32_t)(ex >> 32)), "r"(p.f.seq_value), "r"(0u) : "memory");
    }
    if (pwarp == 0) {
      // exclusive prefix over the experts (lane owns experts lane and lane + 32), then the groups
      int c0 = 0, c1 = 0, units_after[2][2], units_all[2];
      for (int w = 0; w * 32 < B; ++w) {
        c0 += __popc(s_mask[lane][w]);
        c1 += __popc(s_mask[lane + 32][w]);
      }
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
      const int off0 = i0 - c0, off1 = tot0 + i1 - c1;
      for (int w = 0, a = off0, b = off1; w * 32 < B; ++w) {  // first pair of each expert and 32 tokens
        s_off[lane][w] = (short)a;
        s_off[lane + 32][w] = (short)b;
        a += __popc(s_mask[lane][w]);
        b += __popc(s_mask[lane + 32][w]);
      }
      // Unit list: both projections take the groups from the end of the table -- the shared expert (the widest token tiles,
      // the longest epilogues) first, so that its epilogues overlap later units.  A group of n tokens is cut into parts;
      // parts fastest, so the CTAs that share a weight block run at the same time and the second reader hits L2.  The K of
      // a down unit is cut into equal chunks of at most kDownTiles tiles (partial sums meet in y).  s_u[q][g]: the units of
      // the groups after g; the units of group g end at s_u[q][g - 1].
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int per = q == 0 ? p.geo[0].blocks1 : (d >> 8) * p.geo[0].kch, round = (1 << (q == 0 ? p.shift1 : p.shift2)) - 1;
        const int sh = q == 0 ? p.shift1 : p.shift2;
        const int a = per * ((c0 + round) >> sh), b = per * ((c1 + round) >> sh);
        int va = a, vb = b;  // suffix sums over the experts
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int u0 = __shfl_down_sync(0xffffffffu, va, o), u1 = __shfl_down_sync(0xffffffffu, vb, o);
          if (lane + o < 32) {
            va += u0;
            vb += u1;
          }
        }
        const int tb = __shfl_sync(0xffffffffu, vb, 0);
        const int sh_units = p.f.run_shared ? (q == 0 ? p.geo[1].blocks1 : (d >> 8) * p.geo[1].kch) * ((B + round) >> sh) : 0;
        units_after[q][0] = sh_units + tb + va - a;
        units_after[q][1] = sh_units + vb - b;
        units_all[q] = sh_units + tb + __shfl_sync(0xffffffffu, va, 0);
      }
      const unsigned g0m = __ballot_sync(0xffffffffu, c0 > 0), g1m = __ballot_sync(0xffffffffu, c1 > 0);
      const int n_routed = __popc(g0m) + __popc(g1m);
      auto put = [&](int g, int expert, int off, int n, int u1, int u2) {
        s_grp[g] = GroupDesc{expert, off, n};
        s_u[0][g] = u1;
        s_u[1][g] = u2;
      };
      if (c0 > 0) put(__popc(g0m & ((1u << lane) - 1u)), lane, off0, c0, units_after[0][0], units_after[1][0]);
      if (c1 > 0) put(__popc(g0m) + __popc(g1m & ((1u << lane) - 1u)), lane + 32, off1, c1, units_after[0][1], units_after[1][1]);
      if (lane == 0) {
        if (p.f.run_shared) put(n_routed, N, all, B, 0, 0);
        s_units[0] = units_all[0];
        s_units[1] = units_all[1];
      }
    }
    unit_list_barrier();  // the ticket taker may go on
    // the pair list, sorted by (expert, token)
    for (int e = pt >> 3; e < N; e += pn >> 3) {
      const int w = pt & 7;
      if (w * 32 >= B) continue;
      int o = s_off[e][w];
      for (unsigned m = s_mask[e][w]; m; m &= m - 1) s_tok[o++] = (uint8_t)(w * 32 + __ffs((int)m) - 1);
    }
    if (p.f.run_shared && pt < 32) {
      int at = 0;  // the shared expert's pairs follow all others
      for (int w = 0; w * 32 < B; ++w) at += __popc(s_mask[lane][w]) + __popc(s_mask[lane + 32][w]);
      at = (int)__reduce_add_sync(0xffffffffu, (unsigned)at);
      for (int t = lane; t < B; t += 32) s_tok[at + t] = (uint8_t)t;
    }
    plan_barrier();
  }
  const uint32_t tmem_base = tmem_base_s;
  const int n1 = s_units[0], n2 = s_units[1];

  // a count that other CTAs raise (one thread; bounded)
  auto wait_count = [&](const unsigned* ctr, unsigned want) -> bool {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
    if (v >= want) return true;
    const unsigned long long t0 = globaltimer_ns();
    for (uint32_t n_poll = 1; v < want; ++n_poll) {
      if ((n_poll & 31u) == 0u && (*(volatile int*)&s_abort || *(volatile unsigned*)(p.sync + kTcAbort) ||
                                   (long long)(globaltimer_ns() - t0) > p.f.wait_limit_ns))
        return false;
      __nanosleep(40);
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
    }
    return true;
  };
  // the descriptor of this role's n-th unit; phase 0 at the end of the list and after an abort
  auto next_unit = [&](uint32_t n) -> UnitDesc {
    UnitDesc ud = {};
    const uint32_t s = n % kUnitRing;
    if (__all_sync(0xffffffffu, mbar_wait(&unit_full[s], (n / kUnitRing) & 1, &s_abort, p.f.wait_limit_ns))) {
      ud = s_unit[s];
      __syncwarp();
      if (lane == 0) mbar_arrive(&unit_empty[s]);
    }
    return ud;
  };

  if (warp == kWWarp) {
    // ================= tickets and weight loads.  One elected lane issues the loads of a stage, from warp-uniform registers: issued
    // by lanes under a condition on the lane number the loop took 800 cycles per stage, the pace of a launch of few units.
    RingPos rp;  // over the stages (bf16) or the raw tiles (quantised)
    // The next ticket is taken a ring's depth before the end of a unit: the answer is there when the unit's last load has
    // been issued (taken only then, it left the ring empty for 1.5 us per unit), and no unit waits long for its CTA.
    const int ahead = (QF ? NR : NS) * SUB;
    // (lane 0 holds one from the rows above)
    for (uint32_t n = 0; ok; ++n) {
      const int t = __shfl_sync(0xffffffffu, ticket, 0) - B;
      bool taken = false;
      UnitDesc ud = {};
      if (t < n1 + n2) {
        const bool down = t >= n1;
        const int u = down ? t - n1 : t;
        const int* su = s_u[down ? 1 : 0];
        // the group: the first one (in table order) whose units begin at or before u.  Entries fall along the table
        const unsigned m0 = __ballot_sync(0xffffffffu, su[lane] <= u), m1 = __ballot_sync(0xffffffffu, su[lane + 32] <= u);
        const int g = m0 ? __ffs((int)m0) - 1 : m1 ? 31 + __ffs((int)m1) : 64;
        const GroupDesc gr = s_grp[g];
        const int sh = down ? p.shift2 : p.shift1, nmax = down ? p.nmax2 : p.nmax1;
        const int parts = (gr.n_tok + (1 << sh) - 1) >> sh;  // (at most four)
        const uint32_t parts_inv = parts == 2 ? 0x80000000u : parts == 3 ? 0x55555556u : 0x40000000u;
        const int rest = u - su[g];
        const int local = parts == 1 ? rest : (int)__umulhi((uint32_t)rest, parts_inv), part = rest - local * parts;
        const TcGeometry& geo = p.geo[gr.expert >= N ? 1 : 0];
        ud.phase = down ? 2 : 1;
        ud.group = g;
        ud.expert = gr.expert;
        ud.pair_off = gr.pair_off + part * nmax;
        ud.n_tok = min(gr.n_tok - part * nmax, nmax);
        if (down) {
          ud.blk = geo.kch == 1 ? local : (int)__umulhi((uint32_t)local, geo.kch_inv);
          ud.kt_begin = (local - ud.blk * geo.kch) * geo.chunk;
          ud.kt_end = min(ud.kt_begin + geo.chunk, geo.tiles);
        } else {
          ud.blk = local;
          ud.kt_end = d / kKTile;
        }
      }
      if (lane == 0) {
        const uint32_t s = n % kUnitRing;
        if (n >= kUnitRing && !mbar_wait(&unit_empty[s], (n / kUnitRing - 1) & 1, &s_abort, p.f.wait_limit_ns)) ok = false;
        s_unit[s] = ud;
        mbar_arrive(&unit_full[s]);
        TCTL(n, 0);
      }
      ok = __all_sync(0xffffffffu, ok);
      if (ud.phase == 0 || !ok) break;
      const bool shared = ud.expert >= N;
      int slot = 0;
      if (!shared) {
        slot = p.f.snap.expert_slot[ud.expert];
        if (slot < 0) ok = false;
        if (ok && !((ready_mask >> ud.expert) & 1ull)) {
          if (lane == 0) {
            const uint32_t need = p.f.snap.need_gen[ud.expert];
            const uint32_t* flag = p.f.slot_ready + slot;
            const unsigned long long t0 = globaltimer_ns();
            for (uint32_t n_poll = 1; (int32_t)(ld_acquire_sys(flag) - need) < 0; ++n_poll) {
              if ((long long)(globaltimer_ns() - t0) > p.f.wait_limit_ns || ((n_poll & 7u) == 0u && *(volatile unsigned*)(p.sync + kTcAbort))) {
                ok = false;
                break;
              }
              __nanosleep(64);
            }
            if (p.f.stats) atomicAdd(&p.f.stats->stall_ns, globaltimer_ns() - t0);
          }
          ready_mask |= 1ull << ud.expert;
          __syncwarp();  // lane 0's acquire, before the loads of whichever lane
          asm volatile("fence.proxy.async.global;" ::: "memory");
        }
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        slot += p.layer_slot0;  // the tensor map covers the slots of all layers
      }
      // (shuffles: the compiler keeps what comes out of them in uniform registers)
      const int phase = __shfl_sync(0xffffffffu, ud.phase, 0), blk = __shfl_sync(0xffffffffu, ud.blk, 0), usl = __shfl_sync(0xffffffffu, slot, 0);
      const int kt_begin = __shfl_sync(0xffffffffu, ud.kt_begin, 0), kt_end = __shfl_sync(0xffffffffu, ud.kt_end, 0);
      const int store = __shfl_sync(0xffffffffu, shared ? 1 : 0, 0);
      const CUtensorMap* wmap = &tm_w.codes[phase - 1][store];
      const CUtensorMap* smap = &tm_w.scales[phase - 1][store];
      const int rows1 = p.rows1;
      const bool small = phase == 1 && rows1 == kRowsSmall;
      const uint32_t tile_bytes = QF == 0 ? kABytes : small ? RAW_BYTES / 128 * kRowsSmall : RAW_BYTES;
      const int step = QF == 0 && small ? WIDE : SUB;
      for (int kt = kt_begin; kt < kt_end; kt += step, rp.next(QF ? NR : NS)) {
        uint64_t* bar = QF ? &rawfull[rp.s] : &full[rp.s];
        uint8_t* dst = QF ? raw_ring + rp.s * RAW_BYTES : smem + rp.s * STAGE_BYTES;
        ok = __all_sync(0xffffffffu, mbar_wait(QF ? &rawempty[rp.s] : &empty[rp.s], rp.parity ^ 1, &s_abort, p.f.wait_limit_ns));
        if (!ok) break;
        if (!taken && kt + ahead >= kt_end) {
          taken = true;
          if (lane == 0) ticket = (int)atomicAdd(p.sync + kTcTicket, 1u);
        }
        if (elect_one()) {
          mbar_expect_tx(bar, tile_bytes);
          if (QF == 0) {
            if (phase == 2) {
#pragma unroll
              for (int i = 0; i < 4; ++i) tma_load_4d(dst + i * 8192, wmap, blk * 256 + i * 64, 2, kt * kKTile, usl, bar);  // downT, 64 columns each
            } else if (!small) {
#pragma unroll
              for (int i = 0; i < 4; ++i) tma_load_4d(dst + i * 8192, wmap, kt * kKTile, i >> 1, blk * 128 + (i & 1) * 64, usl, bar);  // gate | up, two row halves each
            } else {
#pragma unroll
              for (int i = 0; i < 2 * WIDE; ++i) tma_load_4d(dst + i * (kRowsSmall * 128), wmap, (kt + (i >> 1)) * kKTile, i & 1, blk * kRowsSmall, usl, bar);  // per K tile: gate, up
            }
          } else if (QF == 1) {  // row: gate | up | downT codes (d bytes each), then the scales
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              if (phase == 1) tma_load_3d(dst + i * 16384, wmap, i * d + kt * kKTile, blk * rows1, usl, bar);
              else tma_load_3d(dst + i * 16384, wmap, 2 * d + blk * 256 + i * 128, kt * kKTile, usl, bar);
            }
          } else {  // row: gate | up | downT codes (d/2 bytes each), then their scale bytes (d/32 each)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              if (phase == 1) {
                tma_load_3d(dst + i * 16384, wmap, i * (d / 2) + kt * (kKTile / 2), blk * rows1, usl, bar);
                tma_load_3d(dst + 32768 + i * 2048, smap, 3 * (d / 2) + i * (d / 32) + ((kt * 2) & ~15), blk * rows1, usl, bar);
              } else {
                tma_load_3d(dst + i * 16384, wmap, d + blk * 128, kt * kKTile + i * 128, usl, bar);
                tma_load_3d(dst + 32768 + i * 2048, smap, 3 * (d / 2) + 2 * (d / 32) + ((blk * 8) & ~15), kt * kKTile + i * 128, usl, bar);
              }
            }
          }
        }
        __syncwarp();
      }
    }
    if (!ok && lane == 0) give_up();
    if (lane == 0) s_end[0] = make_uint2(rp.s, rp.parity);
  } else if (warp == kBWarp) {
    // ================= activation loads: rows of X gathered by token index, or the group's rows of a_hi and a_lo
    RingPos rp;
    for (uint32_t n = 0; ok; ++n) {
      const UnitDesc ud = next_unit(n);
      if (ud.phase == 0) break;
      const int n_pad = (ud.n_tok + 15) & ~15;
      const bool gather = ud.phase == 1 && ud.expert < N;
      const int n_loads = gather ? (ud.n_tok + 3) / 4 : n_pad / kARowsPerLoad;
      // load number and K tile of the stage this lane issues, where it takes a lane each
      const bool small = ud.phase == 1 && p.rows1 == kRowsSmall;
      const int li = small ? lane % n_loads : lane, kj = small ? lane / n_loads : 0;
      int tok[4] = {0, 0, 0, 0};
      if (ud.phase == 1) {  // load j: rows 4 j .. 4 j + 3 (past the last token: any row, the result is not used)
#pragma unroll
        for (int i = 0; i < 4; ++i) tok[i] = s_tok[ud.pair_off + min(4 * li + i, ud.n_tok - 1)];
      }
      // what is loaded must be complete: the rows of X (once), or every gate/up unit of the group
      if (ud.phase == 2 || n == 0) {
        if (lane == 0) {
          const unsigned want = ud.phase == 1 ? (unsigned)B : (unsigned)(p.geo[ud.expert >= N ? 1 : 0].blocks1 * ((s_grp[ud.group].n_tok + (1 << p.shift1) - 1) >> p.shift1));
          if (!wait_count(p.sync + (ud.phase == 1 ? kTcRows : kTcDone + ud.group), want)) ok = false;
        }
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        // The bulk loads below read what other CTAs' threads have stored, and any lane may issue one: lane 0's acquire reaches
        // the others through the warp barrier (a vote or shuffle orders no memory), and each lane's fence its own loads
        // (of global memory only: over all state spaces a warp's fence took 0.4 us more per layer of a small step)
        __syncwarp();
        asm volatile("fence.proxy.async.global;" ::: "memory");
      }
      // The shared expert runs all tokens in order: plain boxes (32 gathers per stage were its pace, 1.3 us at 128 tokens)
      const int tiles = __shfl_sync(0xffffffffu, small ? WIDE : 1, 0);   // K tiles of a stage
      const uint32_t bytes = (uint32_t)tiles * (gather ? n_loads * 512u : (uint32_t)(ud.phase * n_pad * 128));
      const int phase = __shfl_sync(0xffffffffu, ud.phase, 0), loads = __shfl_sync(0xffffffffu, n_loads, 0), pads = __shfl_sync(0xffffffffu, n_pad, 0);
      const int kt_begin = __shfl_sync(0xffffffffu, ud.kt_begin, 0), kt_end = __shfl_sync(0xffffffffu, ud.kt_end, 0);
      const int row0 = __shfl_sync(0xffffffffu, phase == 2 ? ud.pair_off : tok[0], 0);  // (the shared expert's tokens follow one another)
      const bool few = loads <= 2;  // one elected lane issues them; otherwise a lane each
      int t0[4], t1[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        t0[i] = __shfl_sync(0xffffffffu, tok[i], 0);
        t1[i] = __shfl_sync(0xffffffffu, tok[i], 1);
      }
      for (int kt = kt_begin; kt < kt_end; kt += tiles, rp.next(NS)) {
        const uint32_t s = rp.s;
        ok = __all_sync(0xffffffffu, mbar_wait(&empty[s], rp.parity ^ 1, &s_abort, p.f.wait_limit_ns));
        if (!ok) break;
        uint8_t* dst = smem + s * STAGE_BYTES + kABytes;
        if (few) {
          if (elect_one()) {
            mbar_expect_tx(&full[s], bytes);
            if (phase == 2) {
              tma_load_2d(dst, &tm_act, kt * kKTile, row0, &full[s]);
              tma_load_2d(dst + pads * 128, &tm_act, kt * kKTile, p.act_rows + row0, &full[s]);
              if (loads == 2) {
                tma_load_2d(dst + kARowsPerLoad * 128, &tm_act, kt * kKTile, row0 + kARowsPerLoad, &full[s]);
                tma_load_2d(dst + (pads + kARowsPerLoad) * 128, &tm_act, kt * kKTile, p.act_rows + row0 + kARowsPerLoad, &full[s]);
              }
            } else if (gather) {
              for (int j = 0; j < tiles; ++j) {
                tma_gather4(dst + j * pads * 128, &tm_x, (kt + j) * kKTile, t0[0], t0[1], t0[2], t0[3], &full[s]);
                if (loads == 2) tma_gather4(dst + j * pads * 128 + 512, &tm_x, (kt + j) * kKTile, t1[0], t1[1], t1[2], t1[3], &full[s]);
              }
            } else {
              for (int j = 0; j < tiles; ++j) {
                tma_load_2d(dst + j * pads * 128, &tm_xc, (kt + j) * kKTile, row0, &full[s]);
                if (loads == 2) tma_load_2d(dst + (j * pads + kARowsPerLoad) * 128, &tm_xc, (kt + j) * kKTile, row0 + kARowsPerLoad, &full[s]);
              }
            }
          }
        } else {
          if (lane == 0) mbar_expect_tx(&full[s], bytes);
          __syncwarp();
          if (phase == 1 && !gather) {
            if (lane < tiles * loads) tma_load_2d(dst + (kj * pads + li * kARowsPerLoad) * 128, &tm_xc, (kt + kj) * kKTile, row0 + li * kARowsPerLoad, &full[s]);
          } else if (phase == 1) {
            if (lane < tiles * loads) tma_gather4(dst + kj * pads * 128 + li * 512, &tm_x, (kt + kj) * kKTile, tok[0], tok[1], tok[2], tok[3], &full[s]);
          } else if (lane < 2 * loads) {  // (at most 64 tokens: 4 boxes per plane)
            const int pl = lane >= loads ? 1 : 0, r = lane - pl * loads;
            tma_load_2d(dst + (pl * pads + r * kARowsPerLoad) * 128, &tm_act, kt * kKTile, pl * p.act_rows + row0 + r * kARowsPerLoad, &full[s]);
          }
        }
        __syncwarp();
      }
    }
    if (!ok && lane == 0) give_up();
    if (lane == 0) s_end[1] = make_uint2(rp.s, rp.parity);
  } else if (warp == kMmaWarp) {
    // ================= MMA issuer: the whole warp walks the stages, one elected lane issues
    RingPos rp;
    AccBuffers acc;
    const uint64_t desc_a1 = umma_desc(smem_u32(smem), 16, 1024), desc_a2 = umma_desc(smem_u32(smem), 64 * 128, 1024);
    const uint64_t desc_b = umma_desc(smem_u32(smem) + kABytes, 16, 1024);
    const uint32_t tbase = __shfl_sync(0xffffffffu, tmem_base, 0);
    for (uint32_t n = 0; ok; ++n) {
      const UnitDesc ud = next_unit(n);
      // (shuffles: the compiler keeps what comes out of them in uniform registers)
      const int phase = __shfl_sync(0xffffffffu, ud.phase, 0), n_tok = __shfl_sync(0xffffffffu, ud.n_tok, 0);
      if (phase == 0) break;
      const int kt_begin = __shfl_sync(0xffffffffu, ud.kt_begin, 0), kt_end = __shfl_sync(0xffffffffu, ud.kt_end, 0);
      // this unit's MMAs run while the epilogue warps still read the previous unit's accumulators
      const bool wide = unit_is_wide<QF>(ud);
      const uint32_t b0 = wide ? 0u : acc.next, b1 = wide ? 1u : acc.next;
      for (uint32_t b = b0; b <= b1; ++b)
        if (acc.uses[b]++ > 0) ok = ok && mbar_wait(&tmem_empty[b], acc.uses[b] & 1, &s_abort, p.f.wait_limit_ns);
      if (!wide) acc.next ^= 1u;
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const bool down = phase == 2;
      const int n_pad = (n_tok + 15) & ~15;
      const uint32_t tacc = tbase + b0 * tc_acc_cols(QF);
      const uint32_t second = QF != 0 && !wide ? 64u : 128u;   // columns of U | of the upper 128 output columns
      const uint32_t idesc = umma_idesc(128, down ? 2 * n_pad : n_pad, down ? 1 : 0);
      const uint64_t desc_a = down ? desc_a2 : desc_a1;
      const uint64_t a_step = down ? 128 : 2;   // per 16 K values: 16 rows of 128 bytes (MN-major) | 32 bytes of a row
      const bool small = !down && p.rows1 == kRowsSmall;
      const int tiles = small ? WIDE : 1;
      for (int kt = kt_begin; kt < kt_end; kt += tiles, rp.next(NS)) {
        const uint32_t s = rp.s;
        ok = __all_sync(0xffffffffu, mbar_wait(&full[s], rp.parity, &s_abort, p.f.wait_limit_ns));
        if (!ok) break;
        if (lane == 0 && kt == kt_begin) TCTL(n, 1);
        tc_fence_after();
        // descriptors differ from the stage-0, k-step-0 ones only in the start-address field (address >> 4, the low
        // 14 bits; the sums below stay inside the CTA's shared memory, so nothing carries into the next field)
        const uint64_t soff = (uint64_t)(s * (uint32_t)STAGE_BYTES >> 4);
        const uint64_t da = desc_a + soff, db = desc_b + soff;
        if (elect_one()) {
          if (small) {
            // Gate and up rows in one MMA (TMEM lanes 0 .. 31 and 32 .. 63); M = 128 all the same: the rows past the 64 are
            // whatever lies behind them (inside the stage: 8 KB of activations at least), and nobody reads theirs of the result.
#pragma unroll
            for (int j = 0; j < WIDE; ++j) {
              const uint64_t daj = da + (uint64_t)(j * (2 * kRowsSmall * 128 / 16)), dbj = db + (uint64_t)(j * n_pad * (128 / 16));
#pragma unroll
              for (int ks = 0; ks < kKTile / 16; ++ks) {
                const uint32_t a = (kt > kt_begin || j > 0 || ks > 0) ? 1u : 0u;
                umma(tacc, daj + (uint64_t)(ks * 2), dbj + (uint64_t)(ks * 2), idesc, a);
              }
            }
          } else if (QF != 0 && !down) {
            const uint32_t ta = tbase + kTmemA + s * 64u;  // gate, then up: 32 columns each
#pragma unroll
            for (int ks = 0; ks < kKTile / 16; ++ks) {
              const uint32_t a = (kt > kt_begin || ks > 0) ? 1u : 0u;
              umma_ts(tacc, ta + ks * 8, db + (uint64_t)(ks * 2), idesc, a);                 // G
              umma_ts(tacc + second, ta + 32 + ks * 8, db + (uint64_t)(ks * 2), idesc, a);   // U
            }
          } else {
#pragma unroll
            for (int ks = 0; ks < kKTile / 16; ++ks) {
              const uint32_t a = (kt > kt_begin || ks > 0) ? 1u : 0u;
              umma(tacc, da + a_step * ks, db + (uint64_t)(ks * 2), idesc, a);                                     // G | columns 0 .. 127
              umma(tacc + second, da + (uint64_t)(128 * 128 / 16) + a_step * ks, db + (uint64_t)(ks * 2), idesc, a);  // U | columns 128 .. 255
            }
          }
          umma_commit(&empty[s]);  // the stage is free once these MMAs have read it
          if (kt + tiles >= kt_end) {
            umma_commit(&tmem_full[b0]);
            if (wide) umma_commit(&tmem_full[1]);
          }
        }
        __syncwarp();
      }
      if (lane == 0) TCTL(n, 2);
    }
    if (!ok && lane == 0) atomicExch(&s_abort, 1);
    if (lane == 0) s_end[2] = make_uint2(rp.s, rp.parity);
  } else if (QF != 0 && warp >= kCvWarp0) {
    // ================= converters: the codes of a raw tile -> bf16 operand tiles of its SUB stages.  Gate and up go to
    // TMEM (lane = row, as the codes lie): a shared-memory tile is written once and read by its MMAs once at 128 bytes per
    // cycle, 500 cycles of a stage, and an MMA with A in TMEM takes N / 2 cycles where one from shared memory takes 40 at
    // least.  downT, whose rows are K, goes to shared memory in the 128-byte-swizzled layout (a tile row is 128 bytes = 64
    // values; its 16-byte chunk j sits at chunk j ^ (row mod 8)).  The raw tile has the same swizzle.  A lane owns a row, so
    // the eight lanes of an access phase touch eight different chunks.
    const int ct = tid - kCvWarp0 * 32;
    RingPos rp, rr;  // stages, raw tiles
    for (uint32_t n = 0; ok; ++n) {
      const UnitDesc ud = next_unit(n);
      if (ud.phase == 0) break;
      if (ud.phase == 1 && p.rows1 == kRowsSmall) {
        // 32 rows of gate and up: all of the raw tile into one stage's shared memory (K-major, a K tile's gate rows, then
        // its up rows).  Through TMEM, whose lanes are rows, the four warps of one scheduler would do all of it.
        for (int kt = ud.kt_begin; kt < ud.kt_end; kt += SUB, rr.next(NR)) {
          const uint32_t r = rr.s;
          ok = __all_sync(0xffffffffu, mbar_wait(&rawfull[r], rr.parity, &s_abort, p.f.wait_limit_ns));
          if (!ok) break;
          const uint8_t* raw = raw_ring + r * RAW_BYTES;
          const uint32_t s = rp.s;
          ok = __all_sync(0xffffffffu, mbar_wait(&empty[s], rp.parity ^ 1, &s_abort, p.f.wait_limit_ns));
          if (!ok) break;
          tc_fence_after();
          const int cw = ct >> 5, t = cw & 1, x = lane & 7;
          const uint8_t* src = raw + t * 16384 + lane * 128;
          uint8_t* dst = smem + s * STAGE_BYTES + t * (kRowsSmall * 128) + lane * 128;
          if (QF == 1) {  // warp: gate | up, 16-value quarter, K tile
            const int q = (cw >> 1) & 3, j = cw >> 3;
            const uint4 v = *reinterpret_cast<const uint4*>(src + (((4 * j + q) ^ x) << 4));
            uint4 o0, o1;
            e4m3x4_to_bf16(p.shifts, v.x, o0.x, o0.y);
            e4m3x4_to_bf16(p.shifts, v.y, o0.z, o0.w);
            e4m3x4_to_bf16(p.shifts, v.z, o1.x, o1.y);
            e4m3x4_to_bf16(p.shifts, v.w, o1.z, o1.w);
            dst += j * (2 * kRowsSmall * 128);
            *reinterpret_cast<uint4*>(dst + (((2 * q) ^ x) << 4)) = o0;
            *reinterpret_cast<uint4*>(dst + (((2 * q + 1) ^ x) << 4)) = o1;
          } else {  // warp: gate | up, 32-value half (one scale block), K tile
            const int h = (cw >> 1) & 1, j = cw >> 2;
            const uint4 v = *reinterpret_cast<const uint4*>(src + (((2 * j + h) ^ x) << 4));
            uint4 o[4];
            e2m1x32_to_bf16(p.shifts, v, raw[32768 + t * 2048 + lane * 16 + ((kt * 2) & 15) + 2 * j + h], o);
            dst += j * (2 * kRowsSmall * 128);
#pragma unroll
            for (int i = 0; i < 4; ++i) *reinterpret_cast<uint4*>(dst + (((4 * h + i) ^ x) << 4)) = o[i];
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(&full[s]);
            mbar_arrive(&rawempty[r]);
          }
          rp.next(NS);
        }
        continue;
      }
      for (int kt = ud.kt_begin; kt < ud.kt_end && ok; kt += SUB, rr.next(NR)) {
        const uint32_t r = rr.s;
        ok = __all_sync(0xffffffffu, mbar_wait(&rawfull[r], rr.parity, &s_abort, p.f.wait_limit_ns));
        if (!ok) break;
        const uint8_t* raw = raw_ring + r * RAW_BYTES;
        // gate/up: tile (gate, up), row and 32-value half of the stage; down: K row of the stage and group of 32 columns
        // (a warp reaches the TMEM lanes of its quarter only: warp mod 4)
        const int t1 = (ct >> 7) & 1, row1 = (warp & 3) * 32 + lane, hf = ct >> 8, kk = ct & 63, og = ct >> 6;
        uint2 sc1 = make_uint2(0u, 0u);
        if (QF == 2 && ud.phase == 1) sc1 = *reinterpret_cast<const uint2*>(raw + 32768 + t1 * 2048 + row1 * 16 + ((kt * 2) & 15));
#pragma unroll
        for (int sub = 0; sub < SUB; ++sub) {
          if (kt + sub >= ud.kt_end) break;
          const uint32_t s = rp.s;
          ok = __all_sync(0xffffffffu, mbar_wait(&empty[s], rp.parity ^ 1, &s_abort, p.f.wait_limit_ns));
          if (!ok) break;
          tc_fence_after();  // (the MMAs that read this stage's tiles before have completed)
          uint8_t* st = smem + s * STAGE_BYTES;
          if (ud.phase == 1) {
            const uint8_t* src = raw + t1 * 16384 + row1 * 128;
            const int x = row1 & 7;
            uint4 o[4];
            if (QF == 1) {
#pragma unroll
              for (int cc = 0; cc < 2; ++cc) {
                const uint4 v = *reinterpret_cast<const uint4*>(src + (((4 * sub + 2 * hf + cc) ^ x) << 4));
                e4m3x4_to_bf16(p.shifts, v.x, o[2 * cc].x, o[2 * cc].y);
                e4m3x4_to_bf16(p.shifts, v.y, o[2 * cc].z, o[2 * cc].w);
                e4m3x4_to_bf16(p.shifts, v.z, o[2 * cc + 1].x, o[2 * cc + 1].y);
                e4m3x4_to_bf16(p.shifts, v.w, o[2 * cc + 1].z, o[2 * cc + 1].w);
              }
            } else {
              const uint4 v = *reinterpret_cast<const uint4*>(src + (((2 * sub + hf) ^ x) << 4));  // 32 codes: one scale block
              e2m1x32_to_bf16(p.shifts, v, ((sub < 2 ? sc1.x : sc1.y) >> (8 * (2 * (sub & 1) + hf))) & 0xffu, o);
            }
            tmem_st16(tmem_base + kTmemA + s * 64u + t1 * 32 + hf * 16 + ((uint32_t)((warp & 3) * 32) << 16), reinterpret_cast<const uint32_t*>(o));
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            tc_fence_before();
          } else {
            const int x = kk & 7;
            uint8_t* dst = st + (og >> 1) * (64 * 128) + kk * 128;
            if (QF == 1) {
              const uint8_t* src = raw + (og >> 2) * 16384 + (sub * 64 + kk) * 128;
#pragma unroll
              for (int cc = 0; cc < 2; ++cc) {
                const int c = (og & 1) * 2 + cc;
                const uint4 v = *reinterpret_cast<const uint4*>(src + (((((og >> 1) & 1) * 4 + c) ^ x) << 4));
                uint4 o0, o1;
                e4m3x4_to_bf16(p.shifts, v.x, o0.x, o0.y);
                e4m3x4_to_bf16(p.shifts, v.y, o0.z, o0.w);
                e4m3x4_to_bf16(p.shifts, v.z, o1.x, o1.y);
                e4m3x4_to_bf16(p.shifts, v.w, o1.z, o1.w);
                *reinterpret_cast<uint4*>(dst + (((2 * c) ^ x) << 4)) = o0;
                *reinterpret_cast<uint4*>(dst + (((2 * c + 1) ^ x) << 4)) = o1;
              }
            } else {
              const uint8_t* src = raw + (sub * 64 + kk) * 128;
              const uint4 v = *reinterpret_cast<const uint4*>(src + ((og ^ x) << 4));
              const int c = og & 1;
              uint4 o[4];
              e2m1x32_to_bf16(p.shifts, v, raw[32768 + (sub * 64 + kk) * 16 + ((ud.blk * 8) & 15) + og], o);
#pragma unroll
              for (int j = 0; j < 4; ++j) *reinterpret_cast<uint4*>(dst + (((4 * c + j) ^ x) << 4)) = o[j];
            }
          }
          if (ud.phase == 2) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the MMAs read these tiles through the async proxy
          __syncwarp();
          if (lane == 0) mbar_arrive(&full[s]);
          rp.next(NS);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&rawempty[r]);
      }
    }
    if (!ok && lane == 0) atomicExch(&s_abort, 1);
    if (lane == 0) s_end[3 + warp - kCvWarp0] = make_uint2(rp.s, rp.parity);
  } else {
    // ================= epilogue: warp w owns TMEM lanes 32*(w%4) .. +31
    const int quad = warp & 3;
    const int row = quad * 32 + lane;  // row of the 128-row tile
    AccBuffers acc;
    // (behind the rings)
    float* s_up = reinterpret_cast<float*>(raw_ring + (size_t)NR * RAW_BYTES);
    uint32_t handed = 0;     // batches of accumulator columns passed between the two warps
    bool rows_seen = false;  // every row of y has been zeroed (and the shared expert's gates are there)
    for (uint32_t n = 0;; ++n) {
      const UnitDesc ud = next_unit(n);
      if (ud.phase == 0) break;
      if (!rows_seen) {
        if (!__shfl_sync(0xffffffffu, lane == 0 ? (wait_count(p.sync + kTcRows, (unsigned)B) ? 1 : 0) : 0, 0)) {
          if (lane == 0) give_up();
          break;
        }
        __syncwarp();  // lane 0's acquire, before every lane's additions into y
        rows_seen = true;
      }
      const bool shared = ud.expert >= N;
      const bool wide = unit_is_wide<QF>(ud);
      const uint32_t b0 = wide ? 0u : acc.next, b1 = wide ? 1u : acc.next;
      // the pairs' weights, sixteen at a time, asked for before the wait and then one batch ahead
      auto load_gates = [&](int c0) {
        const int c = c0 + (lane & 15);
        if (ud.phase != 1 || c >= ud.n_tok) return 0.f;
        const int t = s_tok[ud.pair_off + c];
        if (shared) return p.f.shared_gate ? __ldcg(p.sgate + t) : 1.f;
        return __ldg(p.f.alpha + (size_t)t * N + ud.expert) / s_inv[t];
      };
      float gates_next = load_gates(0);
      bool landed = true;
      for (uint32_t b = b0; b <= b1; ++b) landed = landed && mbar_wait(&tmem_full[b], acc.uses[b]++ & 1, &s_abort, p.f.wait_limit_ns);
      if (!wide) acc.next ^= 1u;
      if (!__all_sync(0xffffffffu, landed)) break;
      auto release = [&]() {
        tc_fence_before();
        for (uint32_t b = b0; b <= b1; ++b) mbar_arrive(&tmem_empty[b]);
      };
      const uint32_t second = QF != 0 && !wide ? 64u : 128u;
      tc_fence_after();
      if (warp == kEpiWarp0 && lane == 0) TCTL(n, 3);
      const uint32_t tacc = tmem_base + b0 * tc_acc_cols(QF) + ((uint32_t)(quad * 32) << 16);
      if (ud.phase == 1) {
        const int i = ud.blk * p.rows1 + row;
        const bool row_ok = row < p.rows1;
        float sg = 1.f, su = 1.f, sd = 1.f;
        if (QF == 1 && row_ok) {  // the row's three fp32 scales follow its 3 d code bytes
          const uint8_t* wb = shared ? p.f.shared_w : p.f.cache + (size_t)p.f.snap.expert_slot[ud.expert] * p.f.slot_stride;
          const float* sc = reinterpret_cast<const float*>(wb + (size_t)i * (3u * d + 16u) + 3u * d);
          sg = __ldg(sc);
          su = __ldg(sc + 1);
          sd = __ldg(sc + 2);
        }
        const bool small = p.rows1 == kRowsSmall;
        // (32 rows: the up half of the accumulator is the second warp's; it passes its values on, two batches in turn)
        for (int c0 = 0; c0 < ud.n_tok && !(small && quad > 0); c0 += 16) {
          uint32_t a[16], b2[16];
          tmem_ld16(tacc + (uint32_t)c0, a);
          if (small) {
            const float* up = s_up + (handed++ & 1u) * 512 + lane;
            asm volatile("bar.sync 2, 64;" ::: "memory");
#pragma unroll
            for (int j = 0; j < 16; ++j) b2[j] = __float_as_uint(up[j * 32]);
          } else {
            tmem_ld16(tacc + second + (uint32_t)c0, b2);
          }
          const float gates = gates_next;
          gates_next = load_gates(c0 + 16);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          __nv_bfloat16* dst = p.act + (size_t)(ud.pair_off + c0) * p.act_stride + i;
          // (eight independent chains at a time; columns past the last token are not stored)
#pragma unroll
          for (int j0 = 0; j0 < 16; j0 += 8) {
            if (c0 + j0 >= ud.n_tok) break;
            float v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float gq = sg * __uint_as_float(a[j0 + j]), uq = su * __uint_as_float(b2[j0 + j]);
              v[j] = __shfl_sync(0xffffffffu, gates, j0 + j) * (gq / (1.f + expf(-gq))) * uq * sd;
            }
            if (row_ok) {
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                if (c0 + j0 + j < ud.n_tok) {
                  const __nv_bfloat16 hi = __float2bfloat16(v[j]);
                  dst[(size_t)(j0 + j) * p.act_stride] = hi;
                  dst[(size_t)(j0 + j) * p.act_stride + p.act_plane] = __float2bfloat16(v[j] - __bfloat162float(hi));
                }
              }
            }
          }
        }
        if (small && quad == 1) {
          for (int c0 = 0; c0 < ud.n_tok; c0 += 16) {
            uint32_t u[16];
            tmem_ld16(tacc + (uint32_t)c0, u);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            float* up = s_up + (handed++ & 1u) * 512 + lane;
#pragma unroll
            for (int j = 0; j < 16; ++j) up[j * 32] = __uint_as_float(u[j]);
            asm volatile("bar.sync 2, 64;" ::: "memory");
          }
        }
        release();
        // count the unit in: the stores of the four warps, ordered before another CTA's bulk loads of the intermediate
        // (the proxy fence stands on the reading side, behind the acquire)
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (warp == kEpiWarp0 && lane == 0)
          asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p.sync + kTcDone + ud.group), "r"(1u) : "memory");
      } else {
        const int n_pad = (ud.n_tok + 15) & ~15;
        for (int half = 0; half < 2; ++half) {
          float* ycol = p.f.y + ud.blk * 256 + half * 128 + tc_column_of(QF, row);
          for (int c0 = 0; c0 < ud.n_tok; c0 += 16) {
            uint32_t a[16], b2[16];
            tmem_ld16(tacc + half * second + (uint32_t)c0, a);
            tmem_ld16(tacc + half * second + (uint32_t)(n_pad + c0), b2);   // the a_lo half of the product
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int j = 0; j < 16; ++j)
              if (c0 + j < ud.n_tok) atomicAdd(ycol + (size_t)s_tok[ud.pair_off + c0 + j] * d, __uint_as_float(a[j]) + __uint_as_float(b2[j]));
          }
        }
        release();
      }
      if (warp == kEpiWarp0 && lane == 0) TCTL(n, 4);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (*(volatile int*)&s_abort) {
    // Copies into this CTA's shared memory and MMAs may still be under way: waited for (bounded), a ring slot per lane.  A role
    // is never a round ahead of another on a slot, so where some have arrived in the barrier's current phase (the one whose
    // parity has not completed) and others have not, the missing arrivals are made up for and the phase ends with its bytes.
    if (warp == 0) {
      auto last = [&](int role, uint32_t s) { return s < s_end[role].x ? s_end[role].y : s_end[role].y ^ 1u; };  // (1 before any: complete)
      if (lane < NS) {
        const uint32_t s = (uint32_t)lane, q = mbar_try_wait(&full[s], 0) ? 1u : 0u;
        int in = 0, missing = 0;
        auto arrived = [&](int role) { last(role, s) == q ? ++in : ++missing; };
        arrived(1);
        if (QF == 0) arrived(0);
        for (int cw = 0; QF != 0 && cw < kCvThreads / 32; ++cw) arrived(3 + cw);
        if (in > 0) {
          for (; missing > 0; --missing) mbar_arrive(&full[s]);
          mbar_wait(&full[s], q, nullptr, p.f.wait_limit_ns);
        }
        mbar_wait(&empty[s], last(2, s), nullptr, p.f.wait_limit_ns);
      } else if (QF != 0 && lane >= 16 && lane < 16 + NR) {
        mbar_wait(&rawfull[lane - 16], last(0, (uint32_t)lane - 16u), nullptr, p.f.wait_limit_ns);
      }
    }
    __syncthreads();
  }
  if (tid == 0) {  // the last CTA leaves the counters zero for the next launch (which waits for this one)
    __threadfence();
    if (atomicAdd(p.sync + kTcExits, 1u) == gridDim.x - 1) {
      for (int i = 0; i < kTcSyncWords; ++i) p.sync[i] = 0u;
      __threadfence();
    }
  }
  if (warp == kMmaWarp) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
  SPAN_END(8);
}

#ifdef APEX_TIMELINE
extern "C" int apex_debug_read_tc_timeline(unsigned long long* host) {
  return (int)cudaMemcpyFromSymbol(host, g_tc_tl, sizeof(g_tc_tl));
}
#endif

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qr) == cudaSuccess && qr == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
    cudaGetLastError();
  }
  return fn;
}

static bool encode(void* out, CUtensorMapDataType type, int rank, const void* base, const cuuint64_t* dims, const cuuint64_t* strides,
                   const cuuint32_t* box, CUtensorMapSwizzle swizzle) {
  EncodeTiledFn fn = encode_fn();
  const cuuint32_t es[4] = {1, 1, 1, 1};
  return fn && fn(reinterpret_cast<CUtensorMap*>(out), type, rank, const_cast<void*>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Row-major bf16 matrix [rows][cols] with row stride `stride_elems`; boxes of 64 columns and `box_rows` rows.
static bool rows_map(void* out, const void* base, int cols, size_t rows, size_t stride_elems, int box_rows) {
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows}, strides[1] = {(cuuint64_t)stride_elems * 2};
  const cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
  return encode(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B);
}

// Batches run here where I and I_shared are multiples of the 128-row tile.  This path rounds h' to bf16 and carries the
// intermediate to 2^-17; the streaming kernel, which takes all other sizes a (expert, token) pair at a time, keeps both in
// fp32, and so do its batches: relative error of y at d = 512 2e-7 .. 3e-7 there against 2e-3 here for h' with 24 bits
// (for bf16-representable h' 2e-6 to 3e-6 here).
bool tc_shape_supported(int I, int I_shared) { return I % 128 == 0 && I_shared % 128 == 0; }

bool tc_make_activation_maps(TcMaps* m, const void* xb, int d, int max_batch, const void* act, size_t act_rows, int act_stride) {
  return rows_map(m->x, xb, d, max_batch, d, 1) && rows_map(m->xc, xb, d, max_batch, d, kARowsPerLoad) && rows_map(m->act, act, act_stride, 2 * act_rows, act_stride, kARowsPerLoad);
}

// The weight maps of one store (the slots of all layers, or one shared expert): n_slots consecutive slots of I rows.
bool tc_make_store_maps(int fmt, unsigned char (*weights)[128], unsigned char (*scales)[128], const void* base, int d, int I, size_t n_slots, size_t slot_bytes) {
  const cuuint32_t rows[2] = {fmt == 0 ? 64u : 128u, (cuuint32_t)kRowsSmall};
  if (fmt == 0) {  // [I][3][d] bf16
    const cuuint64_t dims[4] = {(cuuint64_t)d, 3, (cuuint64_t)I, (cuuint64_t)n_slots};
    const cuuint64_t strides[3] = {(cuuint64_t)d * 2, (cuuint64_t)d * 6, (cuuint64_t)slot_bytes};
    for (int i = 0; i < 2; ++i) {
      const cuuint32_t box[4] = {64, 1, rows[i], 1};
      if (!encode(weights[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, base, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B)) return false;
    }
    return true;
  }
  const size_t rb = ffn_row_bytes(fmt, d);  // raw bytes [I][row bytes]
  const cuuint64_t dims[3] = {(cuuint64_t)rb, (cuuint64_t)I, (cuuint64_t)n_slots};
  const cuuint64_t strides[2] = {(cuuint64_t)rb, (cuuint64_t)slot_bytes};
  for (int i = 0; i < 2; ++i) {
    const cuuint32_t box[3] = {128, rows[i], 1}, sbox[3] = {16, rows[i], 1};
    if (!encode(weights[i], CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, base, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !encode(scales[i], CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, base, dims, strides, sbox, CU_TENSOR_MAP_SWIZZLE_NONE))
      return false;
  }
  return true;
}

namespace {
constexpr int kTcSmemBudget = 215 * 1024;  // rings of a CTA, 1 KB of alignment included

template <int QF>
cudaError_t launch_tc(const TcParams& p, const TcMaps& m, cudaLaunchConfig_t& cfg) {
  static bool configured[kMaxDevices] = {};  // the attribute is per device
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= kMaxDevices || !configured[dev]) {
    cudaError_t e = cudaFuncSetAttribute(ffn_tc_kernel<QF>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcSmemBudget);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < kMaxDevices) configured[dev] = true;
  }
  TcWeightMaps w;
  const int v1 = p.rows1 == kRowsSmall ? 1 : 0;
  for (int ph = 0; ph < 2; ++ph) {
    const int v = ph ? 0 : v1;
    memcpy(&w.codes[ph][0], m.w[v], 128);
    memcpy(&w.codes[ph][1], p.f.shared_w ? m.ws[v] : m.w[v], 128);
    // the 16-byte-box maps are used for the e2m1 store only; the others pass the weight maps again
    memcpy(&w.scales[ph][0], QF == 2 ? m.sc[v] : m.w[v], 128);
    memcpy(&w.scales[ph][1], QF == 2 ? (p.f.shared_w ? m.ssc[v] : m.sc[v]) : m.w[v], 128);
  }
  cfg.blockDim = dim3(tc_threads(QF), 1, 1);
  return cudaLaunchKernelEx(&cfg, ffn_tc_kernel<QF>, w, *reinterpret_cast<const CUtensorMap*>(m.x), *reinterpret_cast<const CUtensorMap*>(m.xc),
                            *reinterpret_cast<const CUtensorMap*>(m.act), p);
}
}  // namespace

cudaError_t launch_ffn_tc(const TcParams& p_in, const TcMaps& m, int n_sm, cudaStream_t s) {
  TcParams p = p_in;
  p.shifts = TcShifts{1u << 2, 1u << 4, 1u << 6, 1u << 8, 1u << 12};
  const int qf = p.f.fmt;
  // Tokens per unit: up to 128 (gate/up), 64 (down: both planes of the intermediate share an MMA).  Small batches leave
  // the activations' share of a stage small and get deeper rings.
  const int b16 = (p.f.B + 15) & ~15;
  p.nmax1 = b16 < 128 ? b16 : 128;
  p.nmax2 = b16 < 64 ? b16 : 64;
  p.shift1 = p.f.B <= p.nmax1 ? 20 : 7;  // (more tokens than a unit takes: the unit takes 128 or 64)
  p.shift2 = p.f.B <= p.nmax2 ? 20 : 6;
  // Rows of I per gate/up unit: 32 where that gives every CTA two units at most, were all experts executed that B tokens
  // can ask for.  A unit is a chain over all of d, so with fewer units than CTAs the launch takes as long as one unit does,
  // and what a stage costs is the loops of its roles, 800 cycles whatever it holds: at d = 4096, I = 256 a step of
  // two tokens was 79 us per layer (bf16) and 99 (e2m1) with 128 rows and one K tile per stage, 65 and 77 so.  Two rounds of
  // 32 rows are half of one of 128: 256 units in six layers of d = 1024, B = 16 251 us (bf16) against 243, of d = 2048, B = 30 409
  // against 387 (e2m1).  With more units 128 rows, which read the activations a quarter as often: at 512 units d = 1024, B = 32 takes 308 us,
  // 325 with 32 rows.  (More than 128 rows of X in a stage of several K tiles would leave no room for a ring.)
  const int experts = p.f.N < p.f.B * p.f.k ? p.f.N : p.f.B * p.f.k;
  const int small_units = experts * (p.f.I / kRowsSmall) + (p.f.run_shared ? p.f.I_shared / kRowsSmall : 0);
  const bool small = small_units <= 2 * n_sm && p.nmax1 * tc_wide(qf) <= 128;
  p.rows1 = small ? kRowsSmall : 128;
  // Chunks of K per down unit: more where the units would leave half of the CTAs without one, or any of them on the quantised
  // stores, whose stages take longer (d = 2048, I = 512, B = 30, e2m1 381 -> 358 us; d = 512, I = 1024, B = 12, e4m3 257 -> 238; d = 4096, B = 8,
  // e2m1 345 -> 329; a chunk keeps four tiles, and with many
  // tokens its epilogue, one atomic per token and column, costs more than the idle CTAs).  64 units -> 128, six layers: d = 1024, I = 512,
  // B = 16 243 -> 234 us (bf16), 285 -> 255 (e4m3); at B = 100 297 -> 309; 128 units -> 256, d = 4096, B = 8 429 -> 441.
  const int most = qf ? kDownTilesQ : kDownTiles;
  auto chunks = [&](int rows) { return (rows / kKTile + most - 1) / most; };
  const int down_units = (p.f.d >> 8) * (experts * chunks(p.f.I) + (p.f.run_shared ? chunks(p.f.I_shared) : 0));
  int split = 1;
  while (p.f.B <= 32 && (qf ? 1 : 2) * split * down_units <= n_sm) split *= 2;
  for (int q = 0; q < 2; ++q) {
    TcGeometry& g = p.geo[q];
    const int rows = q ? p.f.I_shared : p.f.I, sub = tc_sub(qf);
    g.blocks1 = rows / p.rows1;
    g.tiles = rows / kKTile;
    if (!g.tiles) continue;
    const int fewest = chunks(rows), finest = g.tiles / 4 > fewest ? g.tiles / 4 : fewest;
    const int n = fewest * split < finest ? fewest * split : finest;
    g.chunk = ((g.tiles + n - 1) / n + sub - 1) / sub * sub;  // whole raw tiles
    g.kch = (g.tiles + g.chunk - 1) / g.chunk;
    g.kch_inv = g.kch > 1 ? (uint32_t)((0x100000000ull + g.kch - 1) / g.kch) : 0u;
  }
  const int b1 = p.nmax1 * (small ? tc_wide(qf) : 1);
  const int b_bytes = b1 * 128 > 2 * p.nmax2 * 128 ? b1 * 128 : 2 * p.nmax2 * 128;
  p.stage_bytes = kABytes + ((b_bytes + 1023) & ~1023);
  const int behind = small ? kHandBytes : 0;
  const int budget = kTcSmemBudget - 1024 - behind;
  if (qf == 0) {
    p.nraw = 0;
    p.nstage = budget / p.stage_bytes < kMaxStages ? budget / p.stage_bytes : kMaxStages;
  } else {  // two operand stages; the raw ring, which covers the HBM latency, gets the rest
    p.nstage = 2;
    const int left = (budget - p.nstage * p.stage_bytes) / tc_raw_bytes(qf);
    p.nraw = left < kMaxRaw ? left : kMaxRaw;
  }
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // the prologue overlaps the preceding kernel's tail
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3(n_sm, 1, 1);
  // Each CTA allocates all 512 TMEM columns, so two CTAs must never share an SM (the second would sit in
  // tcgen05.alloc until the first has finished): the rings take more than half an SM's shared memory in any case.
  cfg.dynamicSmemBytes = (size_t)p.nstage * p.stage_bytes + (size_t)p.nraw * tc_raw_bytes(qf) + 1024 + behind;
  return qf == 1 ? launch_tc<1>(p, m, cfg) : qf == 2 ? launch_tc<2>(p, m, cfg) : launch_tc<0>(p, m, cfg);
}

}  // namespace apex
