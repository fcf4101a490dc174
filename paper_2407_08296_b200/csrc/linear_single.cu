// The forward product and the weight gradient of the INT8 linear layer (App. A) by single CTAs: one persistent CTA per SM, tiles of 128 x
// 256.  linear_tc.cu, whose CTA pairs move fewer bytes per multiplication, takes the products that are long enough; a pair costs
// some 3 to 4 us more from launch to end (cluster launch and barriers, the second CTA's operand by way of a relay), which is what
// a product of a few hundred columns takes altogether.  Every barrier wait is bounded; a wait that runs out raises
// QG_DEV_WAIT_EXPIRED and the role stops.
#include <cstring>

#include "linear_common.cuh"

namespace qg {
namespace linear {

namespace {

struct SingleArgs {
  CUtensorMap mapA;            // bf16: X of the forward product (K-major, the MMA's B operand); dY of the weight gradient (chunked)
  CUtensorMap mapB;            // INT8 codes of W (2-D, bytes); X of the weight gradient (chunked)
  const float* scales;         // of W: [w_rows][ngroups]
  const float* zeros;
  int32_t ngroups, w_rows;
  uint16_t* D;                 // bf16 output, row-major
  int64_t ldd;
  int32_t rows, cols, K;       // accumulator extents (forward: rows of W x rows of X) and contraction length
  int32_t mblocks, nblocks;
};

// ----------------------------------------------------------------------------------------------------------
// Forward: the converted weight handed to the MMA through TENSOR memory.  The product is computed transposed,
// Y^T = W~ X^T: the accumulator's 128 rows are rows of W, its 256 columns are rows of X (tokens); operand A is a
// 128 x 64 tile of W~ that a converter thread per row writes with one tcgen05.st (64 bf16 = 32 packed registers),
// operand B is a K-major tile of X by TMA.  A K block takes about 0.5 us: the MMA's load of A from tensor memory does
// not overlap.  Tensor memory: columns 0..255 the accumulator, 256..383 its copy rounded to bfloat16, 384..511 four A
// stages of 32 columns: there is no room for a second accumulator, so the epilogue first parks the rounded
// accumulator in the copy (fast: tensor memory to registers and back), releases the accumulator to the MMA, and
// writes the copy out beside the next tile's main loop.
// Warp roles: 0 TMA producer (X tiles and codes), 1 MMA issuer and tensor-memory owner, 4-7 and 12-15 two
// converter groups that take alternate K blocks (a warp reaches the lane quarter warp % 4), 8-11 epilogue.
struct FwdSmem {
  static constexpr int kBBytes = kTileN * kBK * 2;             // 32 KB of X
  static constexpr int kStages = 5;
  static constexpr int kRawBytes = kTileM * kBK;               // 8 KB of codes
  static constexpr int kRawStages = 4;
  static constexpr int kAStages = 4, kACols = kBK / 2;         // tensor-memory stages of A, 32 columns each
  static constexpr int kCopyCol = kTileN;                      // tensor-memory columns of the accumulator's bf16 copy
  static constexpr int kACol0 = kCopyCol + kTileN / 2;         // ... and of the first A stage
  static_assert(kACol0 + kAStages * kACols <= 512, "tensor memory columns");
  // per epilogue warp: a 32 x 32 bf16 block on its way to being stored transposed (rows of 64 bytes)
  static constexpr int kTransRow = 64, kTransBytes = 32 * kTransRow;
  static constexpr int kTransOffset = kStages * kBBytes + kRawStages * kRawBytes;
  static constexpr int kBarOffset = kTransOffset + 4 * kTransBytes;
  static constexpr int kBytes = kBarOffset + 512 + 1024;
  static constexpr int kThreads = 512;
};

__global__ void __launch_bounds__(FwdSmem::kThreads, 1)
linear_forward_kernel(const __grid_constant__ SingleArgs a, int32_t* __restrict__ status) {
  using S = FwdSmem;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* b_base = smem;
  uint8_t* raw_base = smem + S::kStages * S::kBBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S::kBarOffset);
  uint64_t* b_full = bars;
  uint64_t* b_empty = b_full + S::kStages;
  uint64_t* raw_full = b_empty + S::kStages;
  uint64_t* raw_empty = raw_full + S::kRawStages;
  uint64_t* a_full = raw_empty + S::kRawStages;
  uint64_t* a_empty = a_full + S::kAStages;
  uint64_t* acc_full = a_empty + S::kAStages;
  uint64_t* acc_empty = acc_full + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < S::kStages; ++i) { mbar_init(&b_full[i], 1); mbar_init(&b_empty[i], 1); }
    for (int i = 0; i < S::kRawStages; ++i) { mbar_init(&raw_full[i], 1); mbar_init(&raw_empty[i], 4); }
    for (int i = 0; i < S::kAStages; ++i) { mbar_init(&a_full[i], 4); mbar_init(&a_empty[i], 1); }
    mbar_init(acc_full, 1);
    mbar_init(acc_empty, 4);
    fence_mbar_init();
    fence_proxy_async_smem();
  }
  if (warp == 1) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  const uint32_t tmem_a = tmem_base + S::kACol0;

  // here a.rows / a.mblocks count rows of W (the accumulator's rows), a.cols / a.nblocks rows of X (its columns);
  // consecutive tiles (concurrent CTAs) share the block of X
  const int total = a.mblocks * a.nblocks;
  const int kblocks = (a.K + kBK - 1) / kBK;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer: X tile and codes
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int t = blockIdx.x; ok && t < total; t += gridDim.x) {
        const int m0 = (t % a.mblocks) * kTileM, n0 = (t / a.mblocks) * kTileN;
        for (int kb = 0; kb < kblocks; ++kb, ++it) {
          const int rs = it % S::kRawStages, s = it % S::kStages;
          if (!mbar_wait(&raw_empty[rs], ((it / S::kRawStages) & 1) ^ 1)) { ok = false; break; }
          mbar_arrive_expect_tx(&raw_full[rs], S::kRawBytes);
          tma_load_2d(raw_base + rs * S::kRawBytes, &a.mapB, &raw_full[rs], kb * kBK, m0);
          if (!mbar_wait(&b_empty[s], ((it / S::kStages) & 1) ^ 1)) { ok = false; break; }
          mbar_arrive_expect_tx(&b_full[s], S::kBBytes);
          tma_load_2d(b_base + s * S::kBBytes, &a.mapA, &b_full[s], kb * kBK, n0);
        }
      }
      ok = ok && mbar_drain<S::kStages>(b_empty, it) && mbar_drain<S::kAStages>(a_empty, it);
      if (!ok) raise_expired(status);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      constexpr uint32_t idesc = umma_idesc_bf16(kTileM, kTileN, false, false);
      const uint64_t desc_b0 = umma_smem_desc_sw128(smem_u32(b_base), 16, 1024);
      uint32_t it = 0, tcount = 0;
      bool ok = true;
      for (int t = blockIdx.x; ok && t < total; t += gridDim.x, ++tcount) {
        if (!mbar_wait(acc_empty, (tcount & 1) ^ 1)) { ok = false; break; }
        tc_fence_after_sync();
        for (int kb = 0; kb < kblocks; ++kb, ++it) {
          const int s = it % S::kStages, as = it % S::kAStages;
          if (!mbar_wait(&b_full[s], (it / S::kStages) & 1) || !mbar_wait(&a_full[as], (it / S::kAStages) & 1)) { ok = false; break; }
          tc_fence_after_sync();
          const uint64_t db = desc_b0 + (uint64_t)((s * S::kBBytes) >> 4);
#pragma unroll
          for (int k = 0; k < kBK / 16; ++k)
            umma_bf16_tmem_a(tmem_base, tmem_a + as * S::kACols + k * 8, db + k * (32 >> 4), idesc, (kb | k) != 0);
          umma_commit(&b_empty[s]);
          umma_commit(&a_empty[as]);
        }
        if (ok) umma_commit(acc_full);
      }
      if (!ok) raise_expired(status);
    }
  } else if (warp >= 8 && warp < 12) {
    // ------------------------------------------------------------------ epilogue: row i of the tile is row m0 + i of W,
    // column c is row n0 + c of X.  A thread holds one row of the tile; each 32 x 32 block goes through shared
    // memory so that four lanes together store the 64 contiguous bytes it holds of one row of Y (2-byte stores,
    // 256 per thread and tile, took longer than the main loop of a short K; 16-byte stores to 32 different rows
    // per instruction flooded L2 with half-sector writes)
    const int q = warp & 3;
    uint8_t* trans = smem + S::kTransOffset + q * S::kTransBytes;
    uint32_t tcount = 0;
    bool ok = true;
    for (int t = blockIdx.x; ok && t < total; t += gridDim.x, ++tcount) {
      const int m0 = (t % a.mblocks) * kTileM, n0 = (t / a.mblocks) * kTileN;
      ok = mbar_wait_warp(acc_full, tcount & 1);
      if (!ok) break;
      tc_fence_after_sync();
      const uint32_t tacc = tmem_base + ((uint32_t)(q * 32) << 16), tcopy = tacc + S::kCopyCol;
      // Phase 1: the accumulator is rounded to bfloat16 and parked in 128 spare columns of tensor memory, 32
      // columns at a time with the next load in flight; then the MMA may start the next tile.
      {
        uint32_t va[32], vb[32];
        auto park = [&](int c, const uint32_t* v) {
          uint32_t pk[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
            pk[i] = *reinterpret_cast<uint32_t*>(&h);
          }
          tmem_st_32x16(tcopy + 16 * c, pk);
        };
        tmem_ld_32x32(tacc, va);
#pragma unroll 1
        for (int c = 0; c < kTileN / 32; c += 2) {
          tmem_ld_wait();
          tmem_ld_32x32(tacc + 32 * (c + 1), vb);
          park(c, va);
          tmem_ld_wait();
          if (c + 2 < kTileN / 32) tmem_ld_32x32(tacc + 32 * (c + 2), va);
          park(c + 1, vb);
        }
        tmem_st_wait();
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty);
      }
      // Phase 2, beside the next tile's main loop: the copy leaves through shared memory, transposed.
      auto emit = [&](int c, const uint32_t* pk) {
#pragma unroll
        for (int i = 0; i < 16; ++i) {                   // block[j][lane] = D[lane][j], columns 2i and 2i + 1 in pk[i]
          *reinterpret_cast<uint16_t*>(trans + (2 * i) * S::kTransRow + lane * 2) = (uint16_t)(pk[i] & 0xFFFFu);
          *reinterpret_cast<uint16_t*>(trans + (2 * i + 1) * S::kTransRow + lane * 2) = (uint16_t)(pk[i] >> 16);
        }
        __syncwarp();
        const int piece = lane & 3, w0 = m0 + q * 32 + 8 * piece;   // this lane's 8 values of a row of Y start at w0
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int j = (lane >> 2) + 8 * i, tok = n0 + 32 * c + j;
          if (tok < a.cols) {
            const uint4 val = *reinterpret_cast<const uint4*>(trans + j * S::kTransRow + 16 * piece);
            uint16_t* y = a.D + (int64_t)tok * a.ldd + w0;
            if (w0 + 8 <= a.rows) {
              *reinterpret_cast<uint4*>(y) = val;
            } else {
              const uint32_t w[4] = {val.x, val.y, val.z, val.w};
#pragma unroll
              for (int e = 0; e < 8; ++e)
                if (w0 + e < a.rows) y[e] = (uint16_t)((e & 1) ? (w[e >> 1] >> 16) : (w[e >> 1] & 0xFFFFu));
            }
          }
        }
        __syncwarp();
      };
      uint32_t pa[16], pb[16];
      tmem_ld_32x16(tcopy, pa);
#pragma unroll 1
      for (int c = 0; c < kTileN / 32; c += 2) {
        tmem_ld_wait();
        tmem_ld_32x16(tcopy + 16 * (c + 1), pb);
        emit(c, pa);
        tmem_ld_wait();
        if (c + 2 < kTileN / 32) tmem_ld_32x16(tcopy + 16 * (c + 2), pa);
        emit(c + 1, pb);
      }
    }
    if (!ok && lane == 0) raise_expired(status);
  } else if ((warp >= 4 && warp < 8) || warp >= 12) {
    // ------------------------------------------------------------------ converters: codes -> bf16 rows of A in tensor memory
    const int grp = warp >= 12 ? 1 : 0, q = warp & 3;
    const int row = q * 32 + lane;                       // row of the tile = lane of tensor memory
    uint32_t it = 0;
    bool ok = true;
    for (int t = blockIdx.x; ok && t < total; t += gridDim.x) {
      const int wr = (t % a.mblocks) * kTileM + row;
      const bool valid = wr < a.w_rows;
      for (int kb = 0; kb < kblocks; ++kb, ++it) {
        if ((int)(it & 1) != grp) continue;
        const int64_t idx = (int64_t)wr * a.ngroups + (kb >> 2);
        const float sc = valid ? __ldg(a.scales + idx) : 0.f;
        const float bias = 8388736.0f + (valid ? __ldg(a.zeros + idx) : 0.f);      // 2^23 + 128 + z
        const int rs = it % S::kRawStages, as = it % S::kAStages;
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(&raw_full[rs], (it / S::kRawStages) & 1) && mbar_wait(&a_empty[as], ((it / S::kAStages) & 1) ^ 1));
        if (!ok) break;
        tc_fence_after_sync();
        // codes: [128 rows][64 bytes], 16-byte piece c of row r stored at c ^ ((r >> 1) & 3)
        const uint8_t* rrow = raw_base + rs * S::kRawBytes + row * 64;
        uint32_t packed[32];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const uint4 codes = *reinterpret_cast<const uint4*>(rrow + ((c ^ ((row >> 1) & 3)) << 4));
          uint4 lo, hi;
          dequant16(codes, bias, sc, lo, hi);
          packed[8 * c + 0] = lo.x; packed[8 * c + 1] = lo.y; packed[8 * c + 2] = lo.z; packed[8 * c + 3] = lo.w;
          packed[8 * c + 4] = hi.x; packed[8 * c + 5] = hi.y; packed[8 * c + 6] = hi.z; packed[8 * c + 7] = hi.w;
        }
        tmem_st_32x32(tmem_a + ((uint32_t)(q * 32) << 16) + as * S::kACols, packed);
        tmem_st_wait();
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) { mbar_arrive(&a_full[as]); mbar_arrive(&raw_empty[rs]); }
      }
    }
    if (!ok && lane == 0) raise_expired(status);
  }

  __syncwarp();                                        // also the warps of which one lane had a role
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, 512);
  }
}

// ----------------------------------------------------------------------------------------------------------
// Weight gradient: G = dY^T X, both operands by TMA in MN-major form; two accumulators, so that the epilogue of a
// tile overlaps the main loop of the next.  Warp roles: 0 TMA producer, 1 MMA issuer and tensor-memory owner, 4-7
// epilogue.
struct GradSmem {
  static constexpr int kABytes = kTileM * kBK * 2, kBBytes = kTileN * kBK * 2;
  static constexpr int kStageBytes = kABytes + kBBytes;        // 48 KB
  static constexpr int kStages = 4;
  static constexpr int kBarOffset = kStages * kStageBytes;
  static constexpr int kBytes = kBarOffset + 256 + 1024;       // barriers + slack for 1024-byte alignment
  static constexpr int kThreads = 8 * 32;
};

__global__ void __launch_bounds__(GradSmem::kThreads, 1)
linear_weight_grad_kernel(const __grid_constant__ SingleArgs a, int32_t* __restrict__ status) {
  using S = GradSmem;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + S::kBarOffset);
  uint64_t* empty = full + S::kStages;
  uint64_t* acc_full = empty + S::kStages;
  uint64_t* acc_empty = acc_full + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < S::kStages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], 4); }
    fence_mbar_init();
    fence_proxy_async_smem();
  }
  if (warp == 1) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  // consecutive tiles (concurrent CTAs) share the columns of X
  const int total = a.mblocks * a.nblocks, kblocks = (a.K + kBK - 1) / kBK;

  if (warp == 0) {
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int t = blockIdx.x; ok && t < total; t += gridDim.x) {
        const int m0 = (t % a.mblocks) * kTileM, n0 = (t / a.mblocks) * kTileN;
        for (int kb = 0; kb < kblocks; ++kb, ++it) {
          const int s = it % S::kStages;
          if (!mbar_wait(&empty[s], ((it / S::kStages) & 1) ^ 1)) { ok = false; break; }
          uint8_t* sA = smem + s * S::kStageBytes;
          mbar_arrive_expect_tx(&full[s], S::kStageBytes);
          tma_load_3d(sA, &a.mapA, &full[s], 0, kb * kBK, m0 / 64);
          tma_load_3d(sA + S::kABytes, &a.mapB, &full[s], 0, kb * kBK, n0 / 64);
        }
      }
      ok = ok && mbar_drain<S::kStages>(empty, it);
      if (!ok) raise_expired(status);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = umma_idesc_bf16(kTileM, kTileN, true, true);
      const uint64_t desc_a0 = umma_smem_desc_sw128(smem_u32(smem), kSlab, 1024);
      const uint64_t desc_b0 = umma_smem_desc_sw128(smem_u32(smem) + S::kABytes, kSlab, 1024);
      uint32_t it = 0, tcount = 0;
      bool ok = true;
      for (int t = blockIdx.x; ok && t < total; t += gridDim.x, ++tcount) {
        const uint32_t ab = tcount & 1;
        if (!mbar_wait(&acc_empty[ab], ((tcount >> 1) & 1) ^ 1)) { ok = false; break; }
        tc_fence_after_sync();
        for (int kb = 0; kb < kblocks; ++kb, ++it) {
          const int s = it % S::kStages;
          if (!mbar_wait(&full[s], (it / S::kStages) & 1)) { ok = false; break; }
          tc_fence_after_sync();
          const uint64_t off = (uint64_t)((s * S::kStageBytes) >> 4);
#pragma unroll
          for (int k = 0; k < kBK / 16; ++k)
            umma_bf16(tmem_base + ab * kTileN, desc_a0 + off + k * (2048 >> 4), desc_b0 + off + k * (2048 >> 4), idesc, (kb | k) != 0);
          umma_commit(&empty[s]);
        }
        if (ok) umma_commit(&acc_full[ab]);
      }
      if (!ok) raise_expired(status);
    }
  } else if (warp >= 4) {
    const int q = warp & 3;
    uint32_t tcount = 0;
    bool ok = true;
    for (int t = blockIdx.x; ok && t < total; t += gridDim.x, ++tcount) {
      const int m0 = (t % a.mblocks) * kTileM, n0 = (t / a.mblocks) * kTileN;
      const uint32_t ab = tcount & 1;
      ok = mbar_wait_warp(&acc_full[ab], (tcount >> 1) & 1);
      if (!ok) break;
      tc_fence_after_sync();
#pragma unroll 1
      for (int c = 0; c < kTileN / 32; ++c) {
        uint32_t v[32];
        tmem_ld_32x32(tmem_base + ((uint32_t)(q * 32) << 16) + ab * kTileN + 32 * c, v);
        tmem_ld_wait();
        if (c == kTileN / 32 - 1) {                    // every read of this accumulator has landed
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_empty[ab]);
        }
        if (n0 + 32 * c < a.cols) store_piece(a.D, a.ldd, a.rows, a.cols, m0 + q * 32, n0 + 32 * c, lane, v);
        __syncwarp();                                  // the next loads from tensor memory are the whole warp's
      }
    }
    if (!ok && lane == 0) raise_expired(status);
  }
  __syncwarp();                                        // also the warps of which one lane had a role
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, 512);
  }
}

// Opts a kernel into its shared memory, once per device, and launches it on as many SMs as there are tiles for.
template <auto KERN, int THREADS, int SMEM>
int launch_persistent(const SingleArgs& a, int32_t* status, cudaStream_t st) {
  static int sms[64] = {};                            // 0: not asked yet
  int dev = 0;
  QG_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return QG_UNSUPPORTED_SHAPE;
  if (!sms[dev]) {
    int n = 0;
    QG_CUDA_TRY(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev));
    QG_CUDA_TRY(cudaFuncSetAttribute(KERN, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM));
    sms[dev] = n;
  }
  const int total = a.mblocks * a.nblocks;
  KERN<<<total < sms[dev] ? total : sms[dev], THREADS, SMEM, st>>>(a, status);
  QG_LAUNCH_CHECK();
  return QG_OK;
}

}  // namespace

int launch_single(int mode, const uint16_t* act, int64_t ld_act, const uint16_t* act2, int64_t ld_act2, const qg_qtensor* W, int64_t T, int64_t m,
                  int64_t n, uint16_t* D, int64_t ldd, int32_t* status, cudaStream_t st) {
  SingleArgs a;
  memset(&a, 0, sizeof(a));
  a.D = D;
  a.ldd = ldd;
  bool ok = true;
  if (mode == kWeightGrad) {
    // act = dY (T x m), act2 = X (T x n); both enter as 64-wide column slabs, K = T runs down the rows
    ok &= make_map_chunked(&a.mapA, act, T, (m + 63) / 64, ld_act, kBK, 2);
    ok &= make_map_chunked(&a.mapB, act2, T, (n + 63) / 64, ld_act2, kBK, 4);
    a.rows = (int32_t)m; a.cols = (int32_t)n; a.K = (int32_t)T;
  } else {
    // the product is computed transposed: rows of the accumulator are rows of W, its columns rows of X
    a.scales = W->scales;
    a.zeros = W->zeros;
    a.ngroups = (int32_t)((n + kGroup - 1) / kGroup);
    a.w_rows = (int32_t)m;
    ok &= make_map(&a.mapA, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, act, n, T, ld_act, kBK, kTileN, CU_TENSOR_MAP_SWIZZLE_128B);
    ok &= make_map(&a.mapB, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, W->codes, n, m, W->ld, kBK, kTileM, CU_TENSOR_MAP_SWIZZLE_64B);
    a.rows = (int32_t)m; a.cols = (int32_t)T; a.K = (int32_t)n;
  }
  if (!ok) return QG_CUDA_ERROR;
  a.mblocks = (a.rows + kTileM - 1) / kTileM;
  a.nblocks = (a.cols + kTileN - 1) / kTileN;
  return mode == kWeightGrad ? launch_persistent<linear_weight_grad_kernel, GradSmem::kThreads, GradSmem::kBytes>(a, status, st)
                             : launch_persistent<linear_forward_kernel, FwdSmem::kThreads, FwdSmem::kBytes>(a, status, st);
}

}  // namespace linear
}  // namespace qg
