// Stream kernels of the block-wise quantizer (Sec. 3.1, Sec. 3.3) and of the similarity
// statistic between adjacent projection matrices (Sec. 3.2).  All are HBM-bound.
#include "qg_common.cuh"

namespace qg {

// Both quantizer streams work in runs of kRunGroups groups (512 columns) of a row, one warp each.  A lane takes four
// consecutive columns out of every 128, so that every load and store of a warp is contiguous, and has the loads of its
// whole run in flight before it uses the first.  Measured on 4096 x 11008 at 8 bits, against eight consecutive columns
// per lane (two loads 32 bytes apart, scalar stores of the dequantized values) and one group per warp:
// quantize 57 -> 52 us, dequantize 150 -> 33 us, both together 225 -> 86 us (450 MB: 5.3 TB/s of 6.55 measured).
constexpr int kRunGroups = 2, kRunPieces = kRunGroups * 2, kStreamWarps = 8;

// Row and run of this warp; false past the end.
__device__ __forceinline__ bool stream_unit(int64_t rows, int runs, int64_t& row, int& run) {
  const int64_t u = (int64_t)blockIdx.x * kStreamWarps + (threadIdx.x >> 5), total = rows * runs;
  if (u >= total) return false;
  if (total <= 0xFFFFFFFFll) {                      // the short division
    row = (uint32_t)u / (uint32_t)runs;
    run = (int)((uint32_t)u - (uint32_t)row * (uint32_t)runs);
  } else {
    row = u / runs;
    run = (int)(u - row * runs);
  }
  return true;
}

__device__ __forceinline__ float redux_min(float v) {
  float r;
  asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ float redux_max(float v) {
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}

// ------------------------------------------------------------------------ quantize (RTN)
template <int BITS>
__global__ void __launch_bounds__(kStreamWarps * 32)
quantize_rtn_kernel(const float* __restrict__ src, int64_t ld_src, int64_t rows, int64_t cols,
                    uint8_t* __restrict__ codes, int64_t ld_code_bytes,
                    float* __restrict__ scales, float* __restrict__ zeros, int ngroups) {
  const int lane = threadIdx.x & 31;
  int64_t row;
  int run;
  if (!stream_unit(rows, (ngroups + kRunGroups - 1) / kRunGroups, row, run)) return;      // whole warps leave together
  const int64_t c0 = (int64_t)run * kRunGroups * kGroup + lane * 4;
  const float* p = src + row * ld_src + c0;
  float v[kRunPieces][4];
  int nv[kRunPieces];                               // valid columns of each piece
#pragma unroll
  for (int i = 0; i < kRunPieces; ++i) {
    nv[i] = (int)max((int64_t)0, min((int64_t)4, cols - (c0 + 128 * i)));
    if (nv[i] == 4) {
      const float4 a = __ldcs(reinterpret_cast<const float4*>(p + 128 * i));
      v[i][0] = a.x; v[i][1] = a.y; v[i][2] = a.z; v[i][3] = a.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) v[i][e] = (e < nv[i]) ? __ldg(p + 128 * i + e) : 0.0f;
    }
  }
#pragma unroll
  for (int h = 0; h < kRunGroups; ++h) {
    const int g = run * kRunGroups + h;
    if (g >= ngroups) break;
    float mn = INFINITY, mx = -INFINITY;
#pragma unroll
    for (int i = 2 * h; i < 2 * h + 2; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (e < nv[i]) { mn = fminf(mn, v[i][e]); mx = fmaxf(mx, v[i][e]); }
    mn = redux_min(mn);
    mx = redux_max(mx);
    const GroupParams gp = group_params<BITS>(mn, mx);
    // rint(t) + z as integers: adding 1.5 * 2^23 rounds t to the nearest integer, ties to even, and leaves it in the low
    // mantissa bits; exact while |t| < 2^22, i.e. for all of a group whose zero point is below 2^20 and whose scale comes from
    // its extent.  Where it does not (an infinity, an extent past binary32's largest) t may be anything: above 2^22 the sum
    // only grows and the code is the largest; below -2^21, and for a NaN, it is the smallest, as fmaxf makes it here and there.
    const bool small = fabsf(gp.z) < 0x1p20f;
    const int iz = small ? (int)gp.z - 0x4B400000 : 0;
    if (lane == 0) {
      scales[row * ngroups + g] = gp.s;
      zeros[row * ngroups + g] = gp.z;
    }
#pragma unroll
    for (int i = 2 * h; i < 2 * h + 2; ++i) {
      if (nv[i] == 0) continue;
      constexpr int kPerByte = 8 / BITS, kOffset = BITS == 8 ? 0 : 1 << (BITS - 1);
      uint32_t w = 0;                               // unused positions hold code 0, as stored
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        int q;
        if (small) {
          q = __float_as_int(__fadd_rn(fmaxf(__fmul_rn(v[i][e], gp.inv), -0x1p21f), 12582912.0f)) + iz;
          q = min(max(q, -(1 << (BITS - 1))), (1 << (BITS - 1)) - 1);
        } else {
          q = (int)rtn_code<BITS>(v[i][e], gp);
        }
        if (e >= nv[i]) q = 0;
        w |= ((uint32_t)(q + kOffset) & ((1u << BITS) - 1u)) << (BITS * e);
      }
      uint8_t* out = codes + row * ld_code_bytes + (c0 + 128 * i) / kPerByte;
      if (nv[i] == 4) {
        if (BITS == 8) *reinterpret_cast<uint32_t*>(out) = w;
        else if (BITS == 4) *reinterpret_cast<uint16_t*>(out) = (uint16_t)w;
        else *out = (uint8_t)w;
      } else {
        for (int e = 0; e < (nv[i] + kPerByte - 1) / kPerByte; ++e) out[e] = (uint8_t)((w >> (8 * e)) & 0xFF);
      }
    }
  }
}

int launch_quantize_rtn(int bits, const float* src, int64_t rows, int64_t cols, int64_t ld_src,
                        const qg_qtensor* dst, cudaStream_t st) {
  const int ngroups = (int)ceil_div(cols, kGroup);
  const int64_t blocks = ceil_div(rows * ceil_div(ngroups, kRunGroups), kStreamWarps);
  if (blocks > 0x7FFFFFFFll) return QG_UNSUPPORTED_SHAPE;
  auto kern = bits == 8 ? quantize_rtn_kernel<8> : bits == 4 ? quantize_rtn_kernel<4> : quantize_rtn_kernel<2>;
  kern<<<(unsigned)blocks, kStreamWarps * 32, 0, st>>>(src, ld_src, rows, cols, (uint8_t*)dst->codes, dst->ld * bits / 8,
                                                       dst->scales, dst->zeros, ngroups);
  QG_LAUNCH_CHECK();
  return QG_OK;
}

// ------------------------------------------------------------------------ dequantize
template <int BITS>
__global__ void __launch_bounds__(kStreamWarps * 32)
dequantize_kernel(const uint8_t* __restrict__ codes, int64_t ld_code_bytes, const float* __restrict__ scales,
                  const float* __restrict__ zeros, int64_t rows, int64_t cols, int ngroups, float* __restrict__ dst, int64_t ld_dst) {
  const int lane = threadIdx.x & 31;
  int64_t row;
  int run;
  if (!stream_unit(rows, (ngroups + kRunGroups - 1) / kRunGroups, row, run)) return;
  constexpr int kPerByte = 8 / BITS, kOffset = BITS == 8 ? 0 : 1 << (BITS - 1);
  const int64_t c0 = (int64_t)run * kRunGroups * kGroup + lane * 4;
  const uint8_t* p = codes + row * ld_code_bytes + c0 / kPerByte;
  float* out = dst + row * ld_dst + c0;
  uint32_t w[kRunPieces];
  int nv[kRunPieces];
#pragma unroll
  for (int i = 0; i < kRunPieces; ++i) {
    nv[i] = (int)max((int64_t)0, min((int64_t)4, cols - (c0 + 128 * i)));
    const uint8_t* pi = p + 128 * i / kPerByte;
    w[i] = 0;
    if (nv[i] == 4) {
      if (BITS == 8) w[i] = __ldcs(reinterpret_cast<const uint32_t*>(pi));
      else if (BITS == 4) w[i] = __ldcs(reinterpret_cast<const uint16_t*>(pi));
      else w[i] = *pi;
    } else {
      for (int e = 0; e < (nv[i] + kPerByte - 1) / kPerByte; ++e) w[i] |= (uint32_t)pi[e] << (8 * e);
    }
  }
  float s[kRunGroups], z[kRunGroups];
#pragma unroll
  for (int h = 0; h < kRunGroups; ++h) {
    const int g = min(run * kRunGroups + h, ngroups - 1);
    s[h] = __ldg(scales + row * ngroups + g);
    z[h] = __ldg(zeros + row * ngroups + g);
  }
#pragma unroll
  for (int i = 0; i < kRunPieces; ++i) {
    float v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const uint32_t bits = (w[i] >> (BITS * e)) & ((1u << BITS) - 1u);
      const int q = BITS == 8 ? (int)(int8_t)bits : (int)bits - kOffset;
      v[e] = __fmul_rn(__fsub_rn((float)q, z[i / 2]), s[i / 2]);
    }
    if (nv[i] == 4) {
      *reinterpret_cast<float4*>(out + 128 * i) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (e < nv[i]) out[128 * i + e] = v[e];
    }
  }
}

int launch_dequantize(const qg_qtensor* src, float* dst, int64_t ld_dst, cudaStream_t st) {
  const int ngroups = (int)ceil_div(src->cols, kGroup);
  const int64_t blocks = ceil_div(src->rows * ceil_div(ngroups, kRunGroups), kStreamWarps);
  if (blocks > 0x7FFFFFFFll) return QG_UNSUPPORTED_SHAPE;
  auto kern = src->bits == 8 ? dequantize_kernel<8> : src->bits == 4 ? dequantize_kernel<4> : dequantize_kernel<2>;
  kern<<<(unsigned)blocks, kStreamWarps * 32, 0, st>>>((const uint8_t*)src->codes, src->ld * src->bits / 8, src->scales, src->zeros,
                                                       src->rows, src->cols, ngroups, dst, ld_dst);
  QG_LAUNCH_CHECK();
  return QG_OK;
}

// ------------------------------------------------------------------------ similarity (Sec. 3.2)
// Stage 1: each block takes kSimRows rows and all leading c columns (thread t: columns 8t..8t+7),
// accumulates the column dot products <a_j, b_j> over its rows and the two squared norms, and
// writes them to partial[block][...].  Stage 2 (one block) adds the partials in a fixed order,
// takes |.| per column and reduces with warp shuffles.  Deterministic: no atomics.
constexpr int kSimRows = 32;

__device__ __forceinline__ void load_p8(const qg_qtensor& T, int64_t row, int64_t c0, int ngroups, int nvalid,
                                        float v[8]) {
  const int g = (int)(c0 / kGroup);
  const float s = __ldg(T.scales + row * ngroups + g), z = __ldg(T.zeros + row * ngroups + g);
  float q[8];
  load_codes8(T, row, c0, nvalid, q);
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = (i < nvalid) ? __fmul_rn(__fsub_rn(q[i], z), s) : 0.0f;
}

__global__ void __launch_bounds__(256)
similarity_partial_kernel(qg_qtensor A, qg_qtensor B, int c, int c_pad, float* __restrict__ partial) {
  const int ngroups = (int)((A.cols + kGroup - 1) / kGroup);
  const int64_t row0 = (int64_t)blockIdx.x * kSimRows;
  const int64_t row1 = min(A.rows, row0 + kSimRows);
  float* out = partial + (int64_t)blockIdx.x * (c_pad + 2);
  float na = 0.f, nb = 0.f;
  for (int c0 = threadIdx.x * 8; c0 < c_pad; c0 += blockDim.x * 8) {
    const int nvalid = max(0, min(8, c - c0));
    float dot[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (nvalid > 0) {
      for (int64_t row = row0; row < row1; ++row) {
        float a[8], b[8];
        load_p8(A, row, c0, ngroups, nvalid, a);
        load_p8(B, row, c0, ngroups, nvalid, b);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          dot[i] = fmaf(a[i], b[i], dot[i]);
          na = fmaf(a[i], a[i], na);
          nb = fmaf(b[i], b[i], nb);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) out[c0 + i] = dot[i];
  }
  __shared__ float s_na[8], s_nb[8];
  na = warp_sum(na);
  nb = warp_sum(nb);
  if ((threadIdx.x & 31) == 0) { s_na[threadIdx.x >> 5] = na; s_nb[threadIdx.x >> 5] = nb; }
  __syncthreads();
  if (threadIdx.x == 0) {
    float ta = 0.f, tb = 0.f;
    for (int w = 0; w < 8; ++w) { ta += s_na[w]; tb += s_nb[w]; }
    out[c_pad] = ta;
    out[c_pad + 1] = tb;
  }
}

__global__ void __launch_bounds__(1024)
similarity_final_kernel(const float* __restrict__ partial, int nblocks, int c, int c_pad, float* __restrict__ sim) {
  double num = 0.0, na = 0.0, nb = 0.0;
  for (int j = threadIdx.x; j < c; j += blockDim.x) {
    double d = 0.0;
    for (int b = 0; b < nblocks; ++b) d += (double)partial[(int64_t)b * (c_pad + 2) + j];
    num += fabs(d);
  }
  for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
    na += (double)partial[(int64_t)b * (c_pad + 2) + c_pad];
    nb += (double)partial[(int64_t)b * (c_pad + 2) + c_pad + 1];
  }
  __shared__ double s[3][32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    num += __shfl_xor_sync(0xFFFFFFFFu, num, o);
    na += __shfl_xor_sync(0xFFFFFFFFu, na, o);
    nb += __shfl_xor_sync(0xFFFFFFFFu, nb, o);
  }
  if ((threadIdx.x & 31) == 0) {
    s[0][threadIdx.x >> 5] = num; s[1][threadIdx.x >> 5] = na; s[2][threadIdx.x >> 5] = nb;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double tn = 0, ta = 0, tb = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { tn += s[0][w]; ta += s[1][w]; tb += s[2][w]; }
    const double den = sqrt(ta) * sqrt(tb);
    *sim = den > 0.0 ? (float)(tn / den) : 0.0f;
  }
}

size_t similarity_workspace_bytes(int64_t rows, int64_t cols) {
  const int64_t nblocks = ceil_div(rows, kSimRows);
  return (size_t)(nblocks * (round_up(cols, 8) + 2)) * sizeof(float);
}

int launch_similarity(const qg_qtensor* A, const qg_qtensor* B, int32_t c, float* sim_dev, void* ws,
                      cudaStream_t st) {
  const int nblocks = (int)ceil_div(A->rows, kSimRows);
  const int c_pad = (int)round_up(c, 8);
  similarity_partial_kernel<<<nblocks, 256, 0, st>>>(*A, *B, c, c_pad, (float*)ws);
  QG_LAUNCH_CHECK();
  similarity_final_kernel<<<1, 1024, 0, st>>>((const float*)ws, nblocks, c, c_pad, sim_dev);
  QG_LAUNCH_CHECK();
  return QG_OK;
}

}  // namespace qg

// ------------------------------------------------------------------------ similarity without a caller workspace
// The scratch of the two similarity kernels lives in this fixed device array instead of memory the
// caller allocates.  Every device that loads the library carries these 2 MiB until the process exits.
namespace {
constexpr size_t kStaticSimilarityBytes = 2u << 20;
static __device__ __align__(256) unsigned char g_similarity_scratch[kStaticSimilarityBytes];
constexpr int kMaxDevices = 64;
void* g_similarity_scratch_ptr[kMaxDevices] = {};   // device address of the array, per device ordinal
}  // namespace

extern "C" QG_API size_t qgalore_subspace_similarity_static_max_bytes(void) { return kStaticSimilarityBytes; }

extern "C" QG_API int qgalore_subspace_similarity_static(const qg_qtensor* A, const qg_qtensor* B, int32_t sim_cols,
                                                         float* sim_dev, void* stream) {
  using namespace qg;
  if (!sim_dev) return QG_INVALID_ARGUMENT;
  // exactly the rules of qgalore_subspace_similarity: what that entry point refuses, this one refuses too
  int rc = check_projection_qtensor(A);
  if (rc != QG_OK) return rc;
  rc = check_projection_qtensor(B);
  if (rc != QG_OK) return rc;
  if (A->rows != B->rows || A->cols != B->cols) return QG_INVALID_ARGUMENT;
  if (!aligned4(sim_dev)) return QG_MISALIGNED;
  if (A->cols > 16384) return QG_UNSUPPORTED_SHAPE;
  // the shape must fit the fixed array: report it as a workspace that cannot be made larger
  if (similarity_workspace_bytes(A->rows, A->cols) > kStaticSimilarityBytes) return QG_WORKSPACE_TOO_SMALL;
  int dev = 0;
  QG_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return QG_UNSUPPORTED_SHAPE;
  if (!g_similarity_scratch_ptr[dev]) {
    // In host code the array's name is only a handle; the kernels need its address on the current device.
    void* p = nullptr;
    QG_CUDA_TRY(cudaGetSymbolAddress(&p, g_similarity_scratch));
    g_similarity_scratch_ptr[dev] = p;
  }
  const int32_t c = (sim_cols <= 0 || sim_cols > A->cols) ? (int32_t)A->cols : sim_cols;
  // the first kernel overwrites every scratch word the second one reads, so nothing has to be cleared
  return launch_similarity(A, B, c, sim_dev, g_similarity_scratch_ptr[dev], (cudaStream_t)stream);
}
