// The forward product of the INT8 linear layer (App. A) for a handful of activations: Y (T x m) = X (T x n) W~^T with
// T <= kSkinnyTokens, as when a model that is being trained is sampled from.
//
// Bound: the weight's bytes.  The product is a stream over W, so nothing is staged: every warp loads INT8 codes straight
// into registers, 16 bytes per lane, dequantizes them there to the A fragments of mma.sync.m16n8k16 (W~ = bf16((q - z) * s),
// the same two roundings as everywhere) and multiplies them with X fragments that come through L1.  The order of K inside
// an MMA is free as long as both operands share it: lane t of a quad takes columns 16 t .. 16 t + 15 of every 64, so both
// operands are loaded in 16-byte pieces and no lane ever exchanges anything.  A CTA owns 16 rows of W; its warps take the
// quantization groups of those rows in turn, and their partial sums meet in shared memory.
//
// Measured, kernel alone, T = 8, against the tcgen05 kernel (128 x 256 tiles, one CTA per 128 rows of W, a serial chain of
// K blocks): 11008 x 4096 47.9 -> 13.1 us (45 MB: 3.4 TB/s), 4096 x 11008 83 -> 15.9, 2048 x 5461 43 -> 7.1, 768 x 768
// 10.4 -> 2.5; at T = 16 33 -> 21.7 and 82 -> 20.2.  Eight-row tiles (X as the A operand), 32-row tiles, a ring of codes in
// shared memory by cp.async and register prefetch of the next group were all slower at 11008 x 4096.
#include <cuda_bf16.h>

#include "qg_common.cuh"
#include "sm100_ptx.cuh"

namespace qg {

namespace {

using ptx::add2;
using ptx::mul2;

struct SkinnyArgs {
  const uint16_t* X;
  int64_t ldx;
  const int8_t* codes;
  int64_t ldw;
  const float* scales;
  const float* zeros;
  uint16_t* Y;
  int64_t ldy;
  int32_t T, m, n, ngroups;
};

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Four INT8 codes -> four bfloat16 of (q - z) * s, two per word; nbias = -(2^23 + 128 + z): the code byte with its sign bit
// flipped, dropped into the mantissa of 2^23, is the float 2^23 + 128 + q.
__device__ __forceinline__ void dequant4(uint32_t w, float2 nbias, float2 s, uint32_t& lo, uint32_t& hi) {
  w ^= 0x80808080u;
  const float2 a = make_float2(__uint_as_float(__byte_perm(w, 0x4B000000u, 0x7440)), __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7441)));
  const float2 b = make_float2(__uint_as_float(__byte_perm(w, 0x4B000000u, 0x7442)), __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7443)));
  const float2 va = mul2(add2(a, nbias), s), vb = mul2(add2(b, nbias), s);
  const __nv_bfloat162 pa = __floats2bfloat162_rn(va.x, va.y), pb = __floats2bfloat162_rn(vb.x, vb.y);
  lo = *reinterpret_cast<const uint32_t*>(&pa);
  hi = *reinterpret_cast<const uint32_t*>(&pb);
}

// NT: tiles of 8 activations, WARPS: warps that share the groups of sixteen rows
template <int NT, int WARPS>
__global__ void __launch_bounds__(WARPS * 32)
int8_linear_skinny_kernel(const SkinnyArgs a) {
  __shared__ float sums[WARPS][16][NT * 8 + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int row0 = blockIdx.x * 16;
  float acc[NT][4] = {};
  const int8_t* wrow[2];
  const float *srow[2], *zrow[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {                   // rows past the matrix read its last one; their sums are not stored
    const int64_t row = min(row0 + 8 * h + g, a.m - 1);
    wrow[h] = a.codes + row * a.ldw + 16 * t;
    srow[h] = a.scales + row * a.ngroups;
    zrow[h] = a.zeros + row * a.ngroups;
  }
  const uint16_t* xrow[NT];
  bool live[NT];
#pragma unroll
  for (int c = 0; c < NT; ++c) {
    live[c] = 8 * c + g < a.T;
    xrow[c] = a.X + (int64_t)min(8 * c + g, a.T - 1) * a.ldx + 16 * t;
  }
  for (int grp = warp; grp < a.ngroups; grp += WARPS) {
    const int k0 = grp * kGroup;
    uint4 w[2][4];
    float2 s[2], nb[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
      for (int b = 0; b < 4; ++b) {               // a 16-byte piece lies inside the row's pitch or past it as a whole
        const int k = k0 + 64 * b;
        w[h][b] = k + 16 * t < a.n ? __ldcs(reinterpret_cast<const uint4*>(wrow[h] + k)) : make_uint4(0u, 0u, 0u, 0u);
      }
      const float sc = __ldg(srow[h] + grp), z = __ldg(zrow[h] + grp);
      s[h] = make_float2(sc, sc);
      nb[h] = make_float2(-(8388736.0f + z), -(8388736.0f + z));
    }
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int k = k0 + 64 * b;
      uint32_t x[NT][8];
#pragma unroll
      for (int c = 0; c < NT; ++c) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int kk = k + 16 * t + 8 * h;
          const uint4 v = live[c] && kk < a.n ? __ldg(reinterpret_cast<const uint4*>(xrow[c] + k + 8 * h)) : make_uint4(0u, 0u, 0u, 0u);
          x[c][4 * h] = v.x; x[c][4 * h + 1] = v.y; x[c][4 * h + 2] = v.z; x[c][4 * h + 3] = v.w;
          if (kk + 8 > a.n)                       // what lies past the row may be anything
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              if (kk + 2 * i >= a.n) x[c][4 * h + i] = 0u;
              else if (kk + 2 * i + 1 >= a.n) x[c][4 * h + i] &= 0xFFFFu;
            }
        }
      }
      const uint32_t wl[4] = {w[0][b].x, w[0][b].y, w[0][b].z, w[0][b].w}, wh[4] = {w[1][b].x, w[1][b].y, w[1][b].z, w[1][b].w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        uint32_t f[4];
        dequant4(wl[i], nb[0], s[0], f[0], f[2]);
        dequant4(wh[i], nb[1], s[1], f[1], f[3]);
#pragma unroll
        for (int c = 0; c < NT; ++c) mma_bf16(acc[c], f, x[c][2 * i], x[c][2 * i + 1]);
      }
    }
  }
#pragma unroll
  for (int c = 0; c < NT; ++c)
#pragma unroll
    for (int e = 0; e < 4; ++e) sums[warp][8 * (e >> 1) + g][8 * c + 2 * t + (e & 1)] = acc[c][e];
  __syncthreads();
  for (int i = threadIdx.x; i < 16 * NT * 8; i += WARPS * 32) {
    const int row = i % 16, tok = i / 16;
    float v = 0.f;
#pragma unroll
    for (int k = 0; k < WARPS; ++k) v += sums[k][row][tok];
    if (tok < a.T && row0 + row < a.m) a.Y[(int64_t)tok * a.ldy + row0 + row] = float_to_bf16_bits(v);
  }
}

template <int NT, int WARPS>
int launch(const SkinnyArgs& a, cudaStream_t st) {
  int8_linear_skinny_kernel<NT, WARPS><<<(unsigned)ceil_div(a.m, 16), WARPS * 32, 0, st>>>(a);
  QG_LAUNCH_CHECK();
  return QG_OK;
}

}  // namespace

// Warps per CTA: no more than there are groups (four groups: 11008 x 512 takes 4.0 us with four warps, 5.8 with eight), and
// sixteen where the rows alone give less than a CTA per SM and there are groups for them (2048 x 5461: 7.1 us against 8.0).
int launch_int8_linear_skinny(const uint16_t* X, int64_t ldx, const qg_qtensor* W, int64_t T, uint16_t* Y, int64_t ldy, cudaStream_t st) {
  const SkinnyArgs a{X, ldx, (const int8_t*)W->codes, W->ld, W->scales, W->zeros, Y, ldy, (int32_t)T, (int32_t)W->rows,
                     (int32_t)W->cols, (int32_t)ceil_div(W->cols, kGroup)};
  const int warps = a.ngroups <= 4 ? 4 : ceil_div(a.m, 16) <= sm_count() && a.ngroups >= 16 ? 16 : 8;
  if (T <= 8) return warps == 4 ? launch<1, 4>(a, st) : warps == 8 ? launch<1, 8>(a, st) : launch<1, 16>(a, st);
  return warps == 4 ? launch<2, 4>(a, st) : warps == 8 ? launch<2, 8>(a, st) : launch<2, 16>(a, st);
}

}  // namespace qg
