// Expert rows on the tensor cores, eight rows at a time, for one token.
//
// The row-per-warp way (ffn_rows.cuh) unpacks every weight into an fp32 register and pays a shuffle reduction, an exponential
// and the latency of both per row: 1 260 cycles of a warp, whatever the row's length.  Here the eight warps of a CTA work on
// the same rows, each on d / 8 of the columns, with mma.sync, whose operands ldmatrix takes from shared memory as they lie there:
//
//   gate, up    [8 gate rows | 8 up rows] x d/8 columns times h' (m16n8k16): the warp's share of the sixteen dot products
//   exchange    the shares meet in shared memory (one barrier per tile), a_i = g * silu(gate_i) * up_i
//   down        downT^T (16 columns x 8 rows, through ldmatrix.trans) times a (m16n8k8): y of the warp's own columns stays
//               in registers over all rows of the CTA, so the warps' results need no reduction
//
// (tcgen05 would want 128 rows of one expert and its operands in TMEM: a token's rows of a layer are 34 per SM.)  Nothing is rounded on
// the way in: h' and a are cut into three bf16 values whose sum they are (8 + 8 + 8 bits), which occupy three of the MMA's eight
// columns; products of bf16 values are exact in fp32.  Error of y against 64 bits 1.5e-7 to 4e-7, as with fp32 products (of which
// 1.5e-7 come from the gates).
//
// A tile's rows lie a multiple of 128 bytes plus 16 apart (tile_stride), so the eight rows an ldmatrix phase reads fall into
// different banks.
#ifndef APEX_FFN_TILES_CUH
#define APEX_FFN_TILES_CUH

#include "ffn_rows.cuh"
#include "ptx.cuh"

namespace apex {

constexpr int kTileWarps = 8;       // warps that share a tile's columns
constexpr int kPartStride = 20;     // floats per row of the exchange: eight warps' (gate, up), and four more against bank conflicts

// bytes between the rows of a tile in shared memory
__host__ __device__ constexpr uint32_t tile_stride(uint32_t entry_bytes) { return (entry_bytes + 111u) / 128u * 128u + 16u; }

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4_t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
// D = A B: every product starts from zero and is added up in fp32 outside.  Chained through the MMA's accumulator the sums
// lose up to twice as much (y of d = 2048, I = 1408 against 64 bits: 3.7e-7, 1.8e-7 so), as the tensor cores cut what they
// align to the accumulator.
__device__ __forceinline__ void mma_bf16_k16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ void mma_bf16_k8(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5}, {%6}, {%7, %7, %7, %7};"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
      : "r"(a0), "r"(a1), "r"(b0), "f"(0.f));
}

// x as three bf16 values (the upper halves): x = p[0] + p[1] + p[2], each the leading eight bits of what the ones before it leave
// (cut, not rounded: a rounded leading plane could overflow).  An infinity or a NaN is p[0] alone.
struct Planes {
  uint32_t p[3];
};
__device__ __forceinline__ Planes bf16_planes(float x) {
  const uint32_t b = __float_as_uint(x);
  const uint32_t quiet = fabsf(x) <= __uint_as_float(0x7f800000u) ? 0u : 0x00400000u;   // (a NaN stays one when its low bits go)
  const uint32_t finite = fabsf(x) <= 3.402823466e38f ? 0xffff0000u : 0u;
  const float r1 = x - __uint_as_float(b & 0xffff0000u);
  const float r2 = r1 - __uint_as_float(__float_as_uint(r1) & 0xffff0000u);
  return Planes{{(b | quiet) & 0xffff0000u, __float_as_uint(r1) & finite, __float_as_uint(r2) & finite}};
}
// Plane j of two values, packed; planes 3 to 7 are zero.  Selected by masks: as conditions on j, which differs between the
// lanes, the three cases became branches, 500 cycles of a tile.
__device__ __forceinline__ uint32_t bf16_plane_pair(float lo, float hi, int j) {
  const uint32_t m0 = j == 0 ? ~0u : 0u, m1 = j == 1 ? ~0u : 0u, m2 = j == 2 ? ~0u : 0u;
  const Planes a = bf16_planes(lo), b = bf16_planes(hi);
  return (__byte_perm(a.p[0], b.p[0], 0x7632) & m0) | (__byte_perm(a.p[1], b.p[1], 0x7632) & m1) | (__byte_perm(a.p[2], b.p[2], 0x7632) & m2);
}

// The three planes' results of one row or column, which lie in two neighbouring lanes (columns 0, 1 | 2, 3 of the MMA): their
// sum, valid in the lanes of columns 0 and 1.  What is not finite in the leading plane is the result (the products of the zero
// planes with an infinite weight are not).
__device__ __forceinline__ float join_planes(float c0, float c1) {
  const float third = __shfl_down_sync(0xffffffffu, c0, 1);
  return fabsf(c0) <= 3.402823466e38f ? c0 + (c1 + third) : c0;
}

// One warp's share (columns warp * d/8 ...) of a CTA's rows.
template <int D, int FMT>
struct RowTiles;

template <int D>
struct RowTiles<D, kFmtBf16> {
  static constexpr int KW = D / 128;  // 16-column steps
  static_assert(D % 256 == 0, "two steps of 16 columns per warp at least");
  uint32_t hb[KW][2];  // h', B operand of the gate and up products
  float y[KW][4];      // accumulators of the down projection

  // h' in two steps: a lane asks for every 32nd of its warp's columns, cuts them into planes and passes them on to the lanes
  // whose operands they are, through 3 (d / 4 + 16) bytes of shared memory per warp.  (A lane that cut all its operands itself
  // did so eight times as often, 1 us of every layer at d = 1536.)
  struct Raw {
    float v[D / 256];
  };
  __device__ __forceinline__ static void ask_h(Raw& raw, const float* __restrict__ h, int warp, int lane) {
#pragma unroll
    for (int i = 0; i < D / 256; ++i) asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(raw.v[i]) : "l"(h + warp * (D / 8) + i * 32 + lane));
  }
  __device__ __forceinline__ void take_h(const Raw& raw, uint8_t* scratch, int warp, int lane) {
    constexpr int PLANE = D / 4 + 16;  // bytes
    uint8_t* mine = scratch + warp * (3 * PLANE);
#pragma unroll
    for (int i = 0; i < D / 256; ++i) {
      const Planes x = bf16_planes(raw.v[i]);
      uint16_t* at = reinterpret_cast<uint16_t*>(mine) + i * 32 + lane;
      at[0] = (uint16_t)(x.p[0] >> 16);
      at[PLANE / 2] = (uint16_t)(x.p[1] >> 16);
      at[PLANE] = (uint16_t)(x.p[2] >> 16);
    }
    __syncwarp();
    const int plane = lane >> 2;
    const uint32_t* src = reinterpret_cast<const uint32_t*>(mine + (plane < 3 ? plane : 0) * PLANE) + (lane & 3);
#pragma unroll
    for (int s = 0; s < KW; ++s) {
      hb[s][0] = plane < 3 ? src[s * 8] : 0u;
      hb[s][1] = plane < 3 ? src[s * 8 + 4] : 0u;
    }
  }
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int s = 0; s < KW; ++s) y[s][0] = y[s][1] = y[s][2] = y[s][3] = 0.f;
  }
  // Shares of the dot products of the tile's rows; row: shared-memory address of tile row lane mod 8.  (g, u) of row lane / 4
  // in the lanes with lane mod 4 = 0.
  __device__ __forceinline__ void gate_up(uint32_t row, int warp, int lane, float& g, float& u) const {
    // matrices: gate rows, up rows, columns 0 .. 7 of the step, then both of columns 8 .. 15
    const uint32_t at = row + ((lane >> 3) & 1) * (2 * D) + (lane >> 4) * 16 + warp * (D / 4);
    float sum[4] = {};
#pragma unroll
    for (int s = 0; s < KW; ++s) {
      uint32_t a[4];
      float c[4];
      ldsm4(a, at + s * 32);
      mma_bf16_k16(c, a, hb[s][0], hb[s][1]);
#pragma unroll
      for (int i = 0; i < 4; ++i) sum[i] += c[i];
    }
    g = join_planes(sum[0], sum[1]);
    u = join_planes(sum[2], sum[3]);
  }
  // y += downT^T a, eight rows; a0, a1: the gated intermediate of rows 2 (lane mod 4) and the next, zero past the tile's last row;
  // left: rows the tile has from the lane's first one on (the shared memory of the others may hold anything)
  __device__ __forceinline__ void down(uint32_t row, int warp, int lane, float a0, float a1, int left, bool full) {
    const uint32_t b = bf16_plane_pair(a0, a1, lane >> 2);
    const uint32_t at = row + 4 * D + (lane >> 3) * 16 + warp * (D / 4);
    const uint32_t keep = left >= 2 ? 0xffffffffu : left == 1 ? 0xffffu : 0u;
#pragma unroll
    for (int s = 0; s < KW; s += 2) {
      uint32_t m[4];
      float c[2][4];
      ldsm4_t(m, at + s * 32);
      if (!full) {
#pragma unroll
        for (int i = 0; i < 4; ++i) m[i] &= keep;
      }
      mma_bf16_k8(c[0], m[0], m[1], b);
      mma_bf16_k8(c[1], m[2], m[3], b);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        y[s][i] += c[0][i];
        y[s + 1][i] += c[1][i];
      }
    }
  }
  // the warp's columns of y
  __device__ __forceinline__ void store(float* dst, int warp, int lane) const {
#pragma unroll
    for (int s = 0; s < KW; ++s) {
      const float lo = join_planes(y[s][0], y[s][1]), hi = join_planes(y[s][2], y[s][3]);
      if ((lane & 3) == 0) {
        float* at = dst + warp * (D / 8) + s * 16 + (lane >> 2);
        at[0] = lo;
        at[8] = hi;
      }
    }
  }
};

// The exchange of one tile: the sums of the eight warps' shares of a row.
__device__ __forceinline__ void sum_shares(const float* part, int row, float& g, float& u) {
  const float4* src = reinterpret_cast<const float4*>(part + row * kPartStride);
  const float4 v0 = src[0], v1 = src[1], v2 = src[2], v3 = src[3];
  g = ((v0.x + v0.z) + (v1.x + v1.z)) + ((v2.x + v2.z) + (v3.x + v3.z));
  u = ((v0.y + v0.w) + (v1.y + v1.w)) + ((v2.y + v2.w) + (v3.y + v3.w));
}

}  // namespace apex

#endif  // APEX_FFN_TILES_CUH
