// What the two translation units of the INT8 linear layer's GEMMs share: tile extents, the conversion of INT8 codes to the bf16
// operand, the store of an accumulator.
#pragma once

#include "qg_common.cuh"
#include "sm100_ptx.cuh"
#include "tensor_map.cuh"

namespace qg {
namespace linear {

using namespace ptx;

constexpr int kBK = 64;        // K extent of a pipeline stage
constexpr int kTileM = 128;    // accumulator rows (TMEM lanes)
constexpr int kTileN = 256;    // accumulator columns; a multiple of the quantization group along n
constexpr int kSlab = 64 * kBK * 2;   // one 64-wide MN-major slab of a stage: 64 K rows of 128 bytes

enum : int { kForward = 0, kInputGrad = 1, kWeightGrad = 2 };

__device__ __forceinline__ void raise_expired(int32_t* status) {
  if (status) atomicOr(status, QG_DEV_WAIT_EXPIRED);
}

// Sixteen INT8 codes (one 16-byte word) -> sixteen bfloat16 of (q - z) * s, as two 16-byte words.
// bias = 2^23 + 128 + z: the code byte with its sign bit flipped is q + 128, placed in the low mantissa
// byte of 2^23 it reads as the float 2^23 + 128 + q, and subtracting bias leaves q - z exactly; one
// binary32 multiplication and one rounding to bfloat16 follow, the same two roundings as the definition.
__device__ __forceinline__ void dequant16(const uint4 codes, float bias, float s, uint4& lo, uint4& hi) {
  const uint32_t w[4] = {codes.x ^ 0x80808080u, codes.y ^ 0x80808080u, codes.z ^ 0x80808080u, codes.w ^ 0x80808080u};
  const float2 nb = make_float2(-bias, -bias), s2 = make_float2(s, s);
  uint32_t out[8];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 a = make_float2(__uint_as_float(__byte_perm(w[i], 0x4B000000u, 0x7440)),
                                 __uint_as_float(__byte_perm(w[i], 0x4B000000u, 0x7441)));
    const float2 b = make_float2(__uint_as_float(__byte_perm(w[i], 0x4B000000u, 0x7442)),
                                 __uint_as_float(__byte_perm(w[i], 0x4B000000u, 0x7443)));
    const float2 va = mul2(add2(a, nb), s2), vb = mul2(add2(b, nb), s2);
    __nv_bfloat162 pa = __floats2bfloat162_rn(va.x, va.y), pb = __floats2bfloat162_rn(vb.x, vb.y);
    out[2 * i] = *reinterpret_cast<uint32_t*>(&pa);
    out[2 * i + 1] = *reinterpret_cast<uint32_t*>(&pb);
  }
  lo = make_uint4(out[0], out[1], out[2], out[3]);
  hi = make_uint4(out[4], out[5], out[6], out[7]);
}

// Four lanes 4 g .. 4 g + 3 hold a row of four 16-byte pieces each; afterwards lane 4 g + j holds piece j of all four rows, so
// that they store 64 contiguous bytes of one row together.  (A row per lane is 32 half-filled sectors per instruction: input
// gradient 8192 x 2048 x 5461 160 -> 147 us, forward 4690 x 4254 x 128 38 -> 27.)
__device__ __forceinline__ void quad_transpose(uint4 (&p)[4], int lane) {
#pragma unroll
  for (int bit = 1; bit <= 2; bit <<= 1) {
    const bool up = lane & bit;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (c & bit) continue;
      uint4 &lo = p[c], &hi = p[c | bit];
      const uint4 out = up ? lo : hi;
      const uint4 in = make_uint4(__shfl_xor_sync(0xFFFFFFFFu, out.x, bit), __shfl_xor_sync(0xFFFFFFFFu, out.y, bit),
                                  __shfl_xor_sync(0xFFFFFFFFu, out.z, bit), __shfl_xor_sync(0xFFFFFFFFu, out.w, bit));
      if (up) lo = in; else hi = in;
    }
  }
}

// Thirty-two fp32 columns of an accumulator row per lane (32 rows of a warp from row0 on, columns from col0 on) leave as bfloat16.
__device__ __forceinline__ void store_piece(uint16_t* D, int64_t ldd, int rows, int cols, int row0, int col0, int lane, const uint32_t (&v)[32]) {
  uint4 pk[4];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    __nv_bfloat162 h2 = __floats2bfloat162_rn(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
    reinterpret_cast<uint32_t*>(pk)[i] = *reinterpret_cast<uint32_t*>(&h2);
  }
  quad_transpose(pk, lane);                    // pk[i]: columns 8 (lane % 4) .. + 7 of row 4 (lane / 4) + i
  const int col = col0 + 8 * (lane & 3);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = row0 + (lane & ~3) + i;
    uint16_t* d = D + (int64_t)row * ldd + col;
    if (row < rows && col + 8 <= cols) {
      *reinterpret_cast<uint4*>(d) = pk[i];
    } else if (row < rows && col < cols) {
      const uint32_t u[4] = {pk[i].x, pk[i].y, pk[i].z, pk[i].w};
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (col + e < cols) d[e] = (uint16_t)((e & 1) ? (u[e >> 1] >> 16) : (u[e >> 1] & 0xFFFFu));
    }
  }
}

// linear_single.cu: the forward product and the weight gradient by single CTAs
int launch_single(int mode, const uint16_t* act, int64_t ld_act, const uint16_t* act2, int64_t ld_act2, const qg_qtensor* W, int64_t T, int64_t m,
                  int64_t n, uint16_t* D, int64_t ldd, int32_t* status, cudaStream_t st);

}  // namespace linear
}  // namespace qg
