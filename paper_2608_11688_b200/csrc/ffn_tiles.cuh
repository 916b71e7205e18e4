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
// Quantised rows go the same way as fp16 (QuantTiles below).
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
  template <int ROWS>
  struct Scales {};  // (see the e2m1 rows)
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

// ---- quantised rows: the codes become fp16 values, which hold both code sets exactly, two by one conversion.  What bounds them is
// issue slots: a conversion is 1.7 cycles of a scheduler, a k16 MMA 16 (the e4m3 MMA of sm_100a, k32, takes 30 and no conversions, the
// same; as bf16 a pair of codes would cost five integer operations).
__device__ __forceinline__ void mma_f16_k16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}
// the lower and the upper two of four e4m3 codes
__device__ __forceinline__ void e4m3x4_to_f16(uint32_t v, uint32_t& lo, uint32_t& hi) {
  asm("{\n.reg .b16 l, h;\nmov.b32 {l, h}, %2;\ncvt.rn.f16x2.e4m3x2 %0, l;\ncvt.rn.f16x2.e4m3x2 %1, h;\n}" : "=r"(lo), "=r"(hi) : "r"(v));
}
// four e2m1 codes, two to a byte
__device__ __forceinline__ void e2m1x4_to_f16(uint16_t v, uint32_t& lo, uint32_t& hi) {
  asm("{\n.reg .b8 l, h;\nmov.b16 {l, h}, %2;\ncvt.rn.f16x2.e2m1x2 %0, l;\ncvt.rn.f16x2.e2m1x2 %1, h;\n}" : "=r"(lo), "=r"(hi) : "h"(v));
}
// eight of them; for whole words (a zero-extended half word gave zeroes for all four in down_rows_fp32, nvcc 12.9)
__device__ __forceinline__ void e2m1x8_to_f16(uint32_t v, uint32_t (&o)[4]) {
  asm("{\n.reg .b8 b0, b1, b2, b3;\nmov.b32 {b0, b1, b2, b3}, %4;\ncvt.rn.f16x2.e2m1x2 %0, b0;\ncvt.rn.f16x2.e2m1x2 %1, b1;\n"
      "cvt.rn.f16x2.e2m1x2 %2, b2;\ncvt.rn.f16x2.e2m1x2 %3, b3;\n}"
      : "=r"(o[0]), "=r"(o[1]), "=r"(o[2]), "=r"(o[3])
      : "r"(v));
}

// Activations beside them are cut into fp16 planes, three times eleven bits.  fp16's exponents do not reach far, so the values of a
// group (a warp's columns of h', a tile's a) share a power of two that puts the largest between 2^14 and 2^15:
//   x * up = p[0] + 2^-11 p[1] + 2^-22 p[2]
// to the last bit of x where the group spans no more than 36 binades; a group that spans more is worked on in fp32.
struct PlaneScale {
  float up, down;  // the power of two and its inverse
};
__device__ __forceinline__ PlaneScale plane_scale(uint32_t largest) {  // bits of the largest magnitude
  const int f = min(268 - (int)(largest >> 23), 253);                  // (numbers below 2^-112 keep what 2^126 leaves them)
  return PlaneScale{__uint_as_float((uint32_t)f << 23), __uint_as_float((uint32_t)(254 - f) << 23)};
}
__device__ __forceinline__ void f16_planes(float x, float up, __half (&p)[3]) {
  const float s = x * up;
  p[0] = __float2half_rn(s);
  const float r1 = fabsf(s) < 65536.f ? (s - __half2float(p[0])) * 2048.f : 0.f;  // (an infinity or a NaN is p[0] alone)
  p[1] = __float2half_rn(r1);
  p[2] = __float2half_rn((r1 - __half2float(p[1])) * 2048.f);
}
// as join_planes; times the inverse of `up` the value
__device__ __forceinline__ float join_f16_planes(float c0, float c1) {
  const float third = __shfl_down_sync(0xffffffffu, c0, 1);
  return fabsf(c0) <= 3.402823466e38f ? fmaf(fmaf(third, 0x1p-11f, c1), 0x1p-11f, c0) : c0;
}

// How many binades below the group's largest value its smallest one may still sink (by an fp16 factor, say) before a plane drops
// bits: a value 36 binades down keeps its 24.  Negative: it does not, or the largest is so far from 1 that what the
// planes' scales are multiplied by leaves fp32's exponents.
__device__ __forceinline__ int plane_reach(uint32_t largest, uint32_t smallest) {  // bits of the magnitudes; smallest: of those above zero
  const int top = (int)(largest >> 23);
  return largest == 0u ? 36 : top < 77 || top > 187 ? -1 : 36 - (top - (int)(smallest >> 23));
}

// What the planes do not hold is worked on in fp32, a weight at a time, by the two functions below.  Out of line: they are hardly
// ever run.
// Four columns of a 32-column block of 16 rows' downT times a.  at: the lane's codes of the first row's block (scale: its scale byte,
// e2m1); a: of row lane mod 16 or 32; of the rows row0 .. row0 + 15 those below `here` exist.  The sums of the columns this lane group
// has in the accumulators, in the lanes of plane 0 (zero in the others).
template <int FMT>
__device__ __noinline__ float4 down_rows_fp32(const uint8_t* at, const uint8_t* scale, uint32_t stride, float a, int row0, int here) {
  const int lane = threadIdx.x & 31;
  float s[4] = {};
#pragma unroll 1
  for (int i = 0; i < 4; ++i) {
    const int r = row0 + 4 * i + (lane & 3);
    float ar = __shfl_sync(0xffffffffu, a, r);
    if (r < here) {
      uint32_t w[2];
      const uint16_t* codes = reinterpret_cast<const uint16_t*>(at + r * stride);
      if (FMT == kFmtE4m3) {
        e4m3x4_to_f16(codes[0] | (uint32_t)codes[8] << 16, w[0], w[1]);  // (two columns of each of two 16-column steps)
      } else {
        e2m1x4_to_f16(codes[0], w[0], w[1]);
        ar *= __uint_as_float((uint32_t)scale[r * stride] << 23);
      }
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[j]));
        s[2 * j] = fmaf(ar, f.x, s[2 * j]);
        s[2 * j + 1] = fmaf(ar, f.y, s[2 * j + 1]);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    s[j] += __shfl_xor_sync(0xffffffffu, s[j], 1);
    s[j] += __shfl_xor_sync(0xffffffffu, s[j], 2);
    if (lane & 3) s[j] = 0.f;
  }
  return make_float4(s[0], s[1], s[2], s[3]);
}

// The warp's shares of eight rows' gate and up dot products (before the e4m3 scales), in all lanes of row lane / 4.  row: the warp's
// gate codes of that row, vec_bytes before the up codes; scales: of its gate blocks, scale_bytes before the up ones (e2m1); h: the warp's columns.
template <int FMT>
__device__ __noinline__ float2 gate_up_rows_fp32(const uint8_t* row, uint32_t vec_bytes, const uint8_t* scales, uint32_t scale_bytes, const float* __restrict__ h, int blocks) {
  const int t = threadIdx.x & 3;
  float g = 0.f, u = 0.f;
#pragma unroll 1
  for (int b = 0; b < blocks; ++b) {  // eight columns of every 32
    float gw[8], uw[8], hh[8];
    load8<FMT>(row, b * 4 + t, gw);
    load8<FMT>(row + vec_bytes, b * 4 + t, uw);
    const float4 h0 = __ldg(reinterpret_cast<const float4*>(h) + (b * 4 + t) * 2), h1 = __ldg(reinterpret_cast<const float4*>(h) + (b * 4 + t) * 2 + 1);
    hh[0] = h0.x; hh[1] = h0.y; hh[2] = h0.z; hh[3] = h0.w; hh[4] = h1.x; hh[5] = h1.y; hh[6] = h1.z; hh[7] = h1.w;
    float pg = 0.f, pu = 0.f;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      pg = fmaf(gw[m], hh[m], pg);
      pu = fmaf(uw[m], hh[m], pu);
    }
    g = fmaf(FMT == kFmtMxfp4 ? block_scale(scales, b * 4) : 1.f, pg, g);
    u = fmaf(FMT == kFmtMxfp4 ? block_scale(scales + scale_bytes, b * 4) : 1.f, pu, u);
  }
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
    g += __shfl_xor_sync(0xffffffffu, g, o);
    u += __shfl_xor_sync(0xffffffffu, u, o);
  }
  return make_float2(g, u);
}

// What the two quantised formats share: h' and a as fp16 planes.  K order of a step: an 8x8 matrix of ldmatrix gives a lane 4
// consecutive bytes of a row, hence codes that follow one another, while the MMA wants columns 2t, 2t+1, 2t+8, 2t+9 in lane t:
// h' is handed out in the order the codes arrive in, a sum does not mind.
template <int D, int FMT>
struct QuantTiles {
  static constexpr int KW = D / 128;  // 16-column steps
  static constexpr int KB = D / 256;  // 32-column blocks
  static_assert(D % 512 == 0, "whole loads of four matrices");
  uint32_t hb[KW][2];  // h', B operand of the gate and up products
  float y[KW][4];      // accumulators of the down projection
  float h_down;        // inverse of the power of two that the warp's h' was multiplied by
  bool h_wide;         // the warp's h' are not all held: rows times h' in fp32

  struct Raw {
    float v[D / 256];
  };
  __device__ __forceinline__ static void ask_h(Raw& raw, const float* __restrict__ h, int warp, int lane) {
#pragma unroll
    for (int i = 0; i < D / 256; ++i) asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(raw.v[i]) : "l"(h + warp * (D / 8) + i * 32 + lane));
  }
  // (through 3 (d / 4 + 16) bytes of shared memory per warp)
  __device__ __forceinline__ void take_h(const Raw& raw, uint8_t* scratch, int warp, int lane) {
    constexpr int PLANE = D / 4 + 16;  // bytes
    uint8_t* mine = scratch + warp * (3 * PLANE);
    uint32_t largest = 0u, smallest = 0xffffffffu;
#pragma unroll
    for (int i = 0; i < D / 256; ++i) {
      const uint32_t bits = __float_as_uint(raw.v[i]) & 0x7fffffffu;
      largest = max(largest, bits);
      smallest = min(smallest, bits == 0u ? 0xffffffffu : bits);
    }
    largest = __reduce_max_sync(0xffffffffu, largest);
    h_wide = plane_reach(largest, __reduce_min_sync(0xffffffffu, smallest)) < 0;
    const PlaneScale sc = plane_scale(largest);
    h_down = sc.down;
#pragma unroll
    for (int i = 0; i < D / 256; ++i) {
      __half x[3];
      f16_planes(raw.v[i], sc.up, x);
      __half* at = reinterpret_cast<__half*>(mine) + i * 32 + lane;
      at[0] = x[0];
      at[PLANE / 2] = x[1];
      at[PLANE] = x[2];
    }
    __syncwarp();
    const int plane = lane >> 2;
    const uint8_t* src = mine + (plane < 3 ? plane : 0) * PLANE;
#pragma unroll
    for (int s = 0; s < KW; s += 2) {
      // e4m3: step s has columns 16 s + 4 t .. + 3; e2m1: steps s and s + 1 have columns 16 s + 8 t .. + 3 and .. + 7
      uint2 v0, v1;
      if (FMT == kFmtE4m3) {
        v0 = *reinterpret_cast<const uint2*>(src + s * 32 + (lane & 3) * 8);
        v1 = *reinterpret_cast<const uint2*>(src + s * 32 + 32 + (lane & 3) * 8);
      } else {
        const uint4 v = *reinterpret_cast<const uint4*>(src + s * 32 + (lane & 3) * 16);
        v0 = make_uint2(v.x, v.y);
        v1 = make_uint2(v.z, v.w);
      }
      hb[s][0] = plane < 3 ? v0.x : 0u;
      hb[s][1] = plane < 3 ? v0.y : 0u;
      hb[s + 1][0] = plane < 3 ? v1.x : 0u;
      hb[s + 1][1] = plane < 3 ? v1.y : 0u;
    }
  }
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int s = 0; s < KW; ++s) y[s][0] = y[s][1] = y[s][2] = y[s][3] = 0.f;
  }
  // The gated intermediate of ROWS rows (lane's row: lane mod ROWS) as the B operands of their 8-row blocks, and the inverse of
  // their power of two; planes: the warp's scratch, 3 ROWS fp16 values; reach: see plane_reach.
  template <int ROWS>
  __device__ __forceinline__ static float take_a(float a, __half* planes, int lane, uint32_t (&b)[ROWS / 8], int& reach) {
    const uint32_t bits = __float_as_uint(a) & 0x7fffffffu;
    const uint32_t largest = __reduce_max_sync(0xffffffffu, bits);
    reach = plane_reach(largest, __reduce_min_sync(0xffffffffu, bits == 0u ? 0xffffffffu : bits));
    const PlaneScale sc = plane_scale(largest);
    __half x[3];
    f16_planes(a, sc.up, x);
    __syncwarp();  // (the tile before has been read)
    if (lane < ROWS) {
      planes[lane] = x[0];
      planes[ROWS + lane] = x[1];
      planes[2 * ROWS + lane] = x[2];
    }
    __syncwarp();
    const int plane = lane >> 2;
    const uint32_t* src = reinterpret_cast<const uint32_t*>(planes + (plane < 3 ? plane : 0) * ROWS) + (lane & 3);
#pragma unroll
    for (int r = 0; r < ROWS / 8; ++r) b[r] = plane < 3 ? src[r * 4] : 0u;
    return sc.down;
  }
};

template <int D>
struct RowTiles<D, kFmtE4m3> : QuantTiles<D, kFmtE4m3> {
  using Base = QuantTiles<D, kFmtE4m3>;
  using Base::KW;
  using Base::hb;
  using Base::y;
  template <int ROWS>
  struct Scales {};  // (see the e2m1 rows)
  template <int ROWS>
  __device__ __forceinline__ static Scales<ROWS> scales_of(uint32_t, uint32_t, int, int, int) { return Scales<ROWS>{}; }
  template <int ROWS>
  __device__ __forceinline__ bool needs_fp32(uint32_t, uint32_t, int, int, int) const { return Base::h_wide; }
  // the same of eight rows in fp32; rows: their generic address, h: h' in global memory
  __device__ __forceinline__ float2 gate_up_fp32(const uint8_t* rows, uint32_t stride, int warp, int lane, const float* __restrict__ h) const {
    return gate_up_rows_fp32<kFmtE4m3>(rows + (lane >> 2) * stride + warp * (D / 8), D, nullptr, 0u, h + warp * (D / 8), D / 256);
  }
  // shares of the dot products of rows' codes; see the bf16 rows.  tile: the eight rows' shared-memory address
  __device__ __forceinline__ void gate_up(uint32_t tile, uint32_t stride, int warp, int lane, float& g, float& u) const {
    // matrices: gate rows, up rows, columns 0 .. 15 of the step, then both of the next step
    const uint32_t at = tile + (lane & 7) * stride + ((lane >> 3) & 1) * D + (lane >> 4) * 16 + warp * (D / 8);
    float sum[4] = {};
#pragma unroll
    for (int s = 0; s < KW; s += 2) {
      uint32_t v[4];
      ldsm4(v, at + s * 16);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        uint32_t g0, g1, u0, u1;
        float c[4];
        e4m3x4_to_f16(v[2 * j], g0, g1);
        e4m3x4_to_f16(v[2 * j + 1], u0, u1);
        mma_f16_k16(c, g0, u0, g1, u1, hb[s + j][0], hb[s + j][1]);
#pragma unroll
        for (int i = 0; i < 4; ++i) sum[i] += c[i];
      }
    }
    g = join_f16_planes(sum[0], sum[1]) * Base::h_down;
    u = join_f16_planes(sum[2], sum[3]) * Base::h_down;
  }
  // a from the summed shares of a row: its scales are at the end of the row
  __device__ __forceinline__ static float gated(const uint8_t* row, float gate, float g, float u) {
    const float4 sc = *reinterpret_cast<const float4*>(row + 3 * D);
    g *= sc.x;
    return gate * g * __frcp_rn(1.f + expf(-g)) * (u * sc.y) * sc.z;
  }
  // y += downT^T a of ROWS rows, of which `here` exist
  template <int ROWS>
  __device__ __forceinline__ void down(const uint8_t* rows, uint32_t tile, uint32_t stride, int warp, int lane, const uint32_t (&b)[ROWS / 8], float unit, int here, float a_row,
                                       int reach, const Scales<ROWS>&) {
    static_assert(ROWS % 16 == 0, "two 8-row blocks to an MMA");
    if (reach < 0) {
#pragma unroll 1
      for (int r = 0; r < ROWS; r += 16) {
#pragma unroll
        for (int s = 0; s < KW; s += 2) {
          const float4 v = down_rows_fp32<kFmtE4m3>(rows + 2 * D + warp * (D / 8) + s * 16 + (lane >> 2) * 2, nullptr, stride, a_row, r, here);
          y[s][0] += v.x;
          y[s][2] += v.y;
          y[s + 1][0] += v.z;
          y[s + 1][2] += v.w;
        }
      }
      return;
    }
    // matrices: 8-row blocks 0 and 1 of a step, both of the next one
    const uint32_t at = tile + ((lane & 7) + ((lane >> 3) & 1) * 8) * stride + 2 * D + warp * (D / 8) + (lane >> 4) * 16;
#pragma unroll
    for (int r = 0; r < ROWS / 8; r += 2) {
      uint32_t keep[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int left = here - (r + i) * 8 - 2 * (lane & 3);
        keep[i] = left >= 2 ? 0xffffffffu : left == 1 ? 0xffffu : 0u;
      }
#pragma unroll
      for (int s = 0; s < KW; s += 2) {
        uint32_t v[4];
        ldsm4_t(v, at + r * 8 * stride + s * 16);
        if (here != ROWS) {  // (what lies behind the rows may be a NaN's code)
#pragma unroll
          for (int i = 0; i < 4; ++i) v[i] &= keep[i & 1];
        }
        // a register: columns 2g, 2g+1 of row 2t, then of row 2t+1.  As MMA rows: g column 2g, g + 8 column 2g+1
        uint32_t a[4][2];
#pragma unroll
        for (int i = 0; i < 4; ++i) e4m3x4_to_f16(__byte_perm(v[i], 0u, 0x3120), a[i][0], a[i][1]);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          float c[4];
          mma_f16_k16(c, a[2 * j][0], a[2 * j][1], a[2 * j + 1][0], a[2 * j + 1][1], b[r], b[r + 1]);
#pragma unroll
          for (int i = 0; i < 4; ++i) y[s + j][i] = fmaf(c[i], unit, y[s + j][i]);
        }
      }
    }
  }
  __device__ __forceinline__ void store(float* dst, int warp, int lane) const {
#pragma unroll
    for (int s = 0; s < KW; ++s) {
      const float lo = join_f16_planes(y[s][0], y[s][1]), hi = join_f16_planes(y[s][2], y[s][3]);
      if ((lane & 3) == 0) *reinterpret_cast<float2*>(dst + warp * (D / 8) + s * 16 + (lane >> 2) * 2) = make_float2(lo, hi);
    }
  }
};

template <int D>
struct RowTiles<D, kFmtMxfp4> : QuantTiles<D, kFmtMxfp4> {
  using Base = QuantTiles<D, kFmtMxfp4>;
  using Base::hb;
  using Base::KB;
  using Base::y;
  static constexpr int SW = (KB + 3) / 4;  // words of scales of a warp's blocks
  // scales (biased exponents) of the warp's blocks of a vector
  __device__ __forceinline__ static void load_scales(uint32_t at, uint32_t (&sc)[SW]) {
    if (KB == 8) {
      asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(sc[0]), "=r"(sc[SW - 1]) : "r"(at) : "memory");
    } else if (KB == 4) {
      asm volatile("ld.shared.u32 %0, [%1];" : "=r"(sc[0]) : "r"(at) : "memory");
    } else {
#pragma unroll
      for (int i = 0; i < KB; i += 2) {
        uint16_t v;
        asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(at + i) : "memory");
        if ((i & 2) == 0) sc[i / 4] = v;
        else sc[i / 4] |= (uint32_t)v << 16;
      }
    }
  }
  __device__ __forceinline__ static uint32_t byte_of(const uint32_t (&sc)[SW], int i) { return __byte_perm(sc[i / 4], 0u, 0x4440 | (i & 3)); }

  // Is anything in the tile's gate or up rows beyond the planes?  Scales between 2^-63 and 2^64 (and zero) leave the planes' sums inside fp32's
  // exponents.  A lane looks at the scales of a row (of 16: at the gate's or the up row's).
  template <int ROWS>
  __device__ __forceinline__ bool needs_fp32(uint32_t tile, uint32_t stride, int warp, int lane, int here) const {
    const int row = lane & (ROWS - 1);
    const uint32_t at = tile + row * stride + 3 * (D / 2) + warp * KB;
    uint32_t bits = 0u, sc[SW];
    auto look = [&]() {
#pragma unroll
      for (int i = 0; i < SW; ++i) {
        const uint32_t w = sc[i], some = ((w & 0x3f3f3f3fu) + 0x3f3f3f3fu) << 1;  // bit 7 of a byte: its lower six bits are not zero; of w << 1: its bit 6
        bits |= (some & ~(w | w << 1)) | (w & w << 1);
      }
    };
    load_scales(at + (ROWS == 32 ? 0 : (lane >> 4) * (D / 32)), sc);
    look();
    if (ROWS == 32) {
      load_scales(at + D / 32, sc);
      look();
    }
    return __any_sync(0xffffffffu, Base::h_wide || (row < here && (bits & 0x80808080u) != 0u));
  }
  __device__ __forceinline__ float2 gate_up_fp32(const uint8_t* rows, uint32_t stride, int warp, int lane, const float* __restrict__ h) const {
    const uint8_t* row = rows + (lane >> 2) * stride;
    return gate_up_rows_fp32<kFmtMxfp4>(row + warp * (D / 16), D / 2, row + 3 * (D / 2) + warp * KB, D / 32, h + warp * (D / 8), KB);
  }
  __device__ __forceinline__ void gate_up(uint32_t tile, uint32_t stride, int warp, int lane, float& g, float& u) const {
    // matrices: gate rows, up rows of a block, then both of the next block
    const uint32_t at = tile + (lane & 7) * stride + ((lane >> 3) & 1) * (D / 2) + (lane >> 4) * 16 + warp * (D / 16);
    const uint32_t scales = tile + (lane >> 2) * stride + 3 * (D / 2) + warp * KB;
    uint32_t sg[SW], su[SW];
    load_scales(scales, sg);
    load_scales(scales + D / 32, su);
    float sum[4] = {};
#pragma unroll
    for (int b = 0; b < KB; b += 2) {
      uint32_t v[4];
      ldsm4(v, at + b * 16);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        uint32_t gw[4], uw[4];
        float c0[4], c1[4];
        e2m1x8_to_f16(v[2 * j], gw);
        e2m1x8_to_f16(v[2 * j + 1], uw);
        const int s = 2 * (b + j);
        mma_f16_k16(c0, gw[0], uw[0], gw[1], uw[1], hb[s][0], hb[s][1]);
        mma_f16_k16(c1, gw[2], uw[2], gw[3], uw[3], hb[s + 1][0], hb[s + 1][1]);
        const float fg = __uint_as_float(byte_of(sg, b + j) << 23), fu = __uint_as_float(byte_of(su, b + j) << 23);
        sum[0] = fmaf(c0[0] + c1[0], fg, sum[0]);
        sum[1] = fmaf(c0[1] + c1[1], fg, sum[1]);
        sum[2] = fmaf(c0[2] + c1[2], fu, sum[2]);
        sum[3] = fmaf(c0[3] + c1[3], fu, sum[3]);
      }
    }
    g = join_f16_planes(sum[0], sum[1]) * Base::h_down;
    u = join_f16_planes(sum[2], sum[3]) * Base::h_down;
  }
  __device__ __forceinline__ static float gated(const uint8_t*, float gate, float g, float u) { return gate * g * __frcp_rn(1.f + expf(-g)) * u; }
  // y += downT^T a.  A block's scale differs from row to row, along the sum, so it goes to the B operand: the row's planes times
  // 2^(scale - largest scale of the block in the 16 rows of an MMA); the largest scale is applied to the result.  A plane's last bit is
  // 2^4 at the top of the reach and 2^-24 is fp16's, so nothing is cut where the smallest a lies with the smallest scale 28 binades
  // below the largest of both.  A tile whose scales (or a) span more, in any block, is taken in fp32: a row that sinks below the
  // largest scale times the largest a, which no row need have together, may be all there is of a column.
  template <int ROWS>
  struct Scales {
    uint32_t e[ROWS / 8], top[ROWS / 16];  // lane 4 b + t, block b: the factors of rows 2t, 2t+1 of each 8-row block; the largest scales
    int span;                              // binades between the scales of a block, at most (any lane's)
  };
  // What does not depend on a: looked at in front of the exchange's barrier.  With the tests behind it, a branch for every eight rows, d = 512
  // took 209 us (8 layers of 4 experts of 6000 rows), d = 2048 247 (2500 rows); 182 and 236 so, 175 and 221 without tests.
  template <int ROWS>
  __device__ __forceinline__ static Scales<ROWS> scales_of(uint32_t tile, uint32_t stride, int warp, int lane, int here) {
    static_assert(ROWS % 16 == 0, "two 8-row blocks to an MMA");
    Scales<ROWS> f;
    // a lane works out its block and passes the factors on (every lane for itself and all blocks: 60 instructions per block instead of 5)
    const uint32_t scales = tile + 2 * (lane & 3) * stride + 3 * (D / 2) + 2 * (D / 32) + warp * KB + min(lane >> 2, KB - 1);
    uint32_t span = 0u;
#pragma unroll
    for (int r = 0; r < ROWS / 8; r += 2) {
      uint32_t sc[4], top = 0u;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int row = (r + (i >> 1)) * 8 + (i & 1);
        asm volatile("ld.shared.u8 %0, [%1];" : "=r"(sc[i]) : "r"(scales + row * stride) : "memory");
        sc[i] = row + 2 * (lane & 3) < here ? sc[i] : 0u;
        top = max(top, sc[i]);
      }
      top = max(top, __shfl_xor_sync(0xffffffffu, top, 1));
      top = max(top, __shfl_xor_sync(0xffffffffu, top, 2));
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        // 2^-k in fp16, a subnormal from 15 on, zero from 25 on; a scale of zero is zero
        const uint32_t k = top - sc[i];
        const uint32_t v = sc[i] == 0u ? 0u : k < 15u ? (15u - k) << 10 : 0x400u >> min(k - 14u, 31u);
        if (i & 1) f.e[r + (i >> 1)] |= v << 16;
        else f.e[r + (i >> 1)] = v;
        span = max(span, sc[i] == 0u ? 0u : sc[i] - 64u > 127u ? 255u : k);
      }
      f.top[r / 2] = top;
    }
    f.span = (int)__reduce_max_sync(0xffffffffu, span);
    return f;
  }
  template <int ROWS>
  __device__ __forceinline__ void down(const uint8_t* rows, uint32_t tile, uint32_t stride, int warp, int lane, const uint32_t (&b)[ROWS / 8], float unit, int here, float a_row,
                                       int reach, const Scales<ROWS>& sc) {
    if (sc.span > reach - 8) {
      const uint8_t* codes = rows + D + warp * (D / 16) + (lane >> 2) * 2;
#pragma unroll 1
      for (int r = 0; r < ROWS; r += 16) {
#pragma unroll
        for (int blk = 0; blk < KB; ++blk) {
          const float4 v = down_rows_fp32<kFmtMxfp4>(codes + blk * 16, rows + 3 * (D / 2) + 2 * (D / 32) + warp * KB + blk, stride, a_row, r, here);
          y[2 * blk][0] += v.x;
          y[2 * blk][2] += v.y;
          y[2 * blk + 1][0] += v.z;
          y[2 * blk + 1][2] += v.w;
        }
      }
      return;
    }
    const uint32_t at = tile + ((lane & 7) + ((lane >> 3) & 1) * 8) * stride + D + warp * (D / 16) + (lane >> 4) * 16;
#pragma unroll
    for (int r = 0; r < ROWS / 8; r += 2) {
      const float back = __uint_as_float(sc.top[r / 2] << 23) * unit;
#pragma unroll
      for (int b0 = 0; b0 < KB; b0 += 2) {  // blocks
        uint32_t v[4];
        ldsm4_t(v, at + r * 8 * stride + b0 * 16);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int blk = b0 + j;
          uint32_t bs[2], a[2][4];
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const uint32_t es = __shfl_sync(0xffffffffu, sc.e[r + i], blk * 4 + (lane & 3));
            const __half2 t = __hmul2(*reinterpret_cast<const __half2*>(&b[r + i]), *reinterpret_cast<const __half2*>(&es));
            bs[i] = *reinterpret_cast<const uint32_t*>(&t);
            // a register: columns 4g .. 4g+3 of row 2t, then of row 2t+1, a nibble each: brought together by column
            const uint32_t m = __byte_perm(v[2 * j + i], 0u, 0x3120);
            const uint32_t swap = (m ^ (m >> 4)) & 0x00f000f0u;
            e2m1x8_to_f16(m ^ swap ^ (swap << 4), a[i]);
          }
          const float f = __shfl_sync(0xffffffffu, back, blk * 4);
#pragma unroll
          for (int t = 0; t < 2; ++t) {  // columns 4g and 4g+1, then 4g+2 and 4g+3
            float c[4];
            mma_f16_k16(c, a[0][2 * t], a[0][2 * t + 1], a[1][2 * t], a[1][2 * t + 1], bs[0], bs[1]);
#pragma unroll
            for (int i = 0; i < 4; ++i) y[2 * blk + t][i] = fmaf(c[i], f, y[2 * blk + t][i]);
          }
        }
      }
    }
  }
  __device__ __forceinline__ void store(float* dst, int warp, int lane) const {
#pragma unroll
    for (int b = 0; b < KB; ++b) {
      float4 v;
      v.x = join_f16_planes(y[2 * b][0], y[2 * b][1]);
      v.y = join_f16_planes(y[2 * b][2], y[2 * b][3]);
      v.z = join_f16_planes(y[2 * b + 1][0], y[2 * b + 1][1]);
      v.w = join_f16_planes(y[2 * b + 1][2], y[2 * b + 1][3]);
      if ((lane & 3) == 0) *reinterpret_cast<float4*>(dst + warp * (D / 8) + b * 32 + (lane >> 2) * 4) = v;
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
