// The INT8 linear layer of App. A as tcgen05 GEMMs that take the INT8 weight as it is stored:
//
//   forward          Y   = X W~^T       (T x m)    A = X    K-major,   B = W~    K-major         (K = n)
//   input gradient   dX  = dY W~        (T x n)    A = dY   K-major,   B = W~    MN-major        (K = m)
//   weight gradient  G   = dY^T X       (m x n)    A = dY^T MN-major,  B = X     MN-major        (K = T)
//
// with W~ = bf16((q - z) * s), the weight dequantized in binary32 per group of 256 (Sec. 3.1) and rounded once
// to the activations' type.  W~ never exists in global memory: the INT8 codes of a tile arrive in shared memory
// by TMA and converter warps dequantize them straight into the 128-byte-swizzled layout that the MMA reads.
// The accumulator (fp32, tensor memory) leaves as bfloat16.  The weight gradient has no quantized operand: both
// tiles come by TMA in MN-major form, and its output is the matrix G the optimizer step reads.
//
// Persistent CTA PAIRS, one CTA per SM, tiles of 512 or 256 rows x 256 columns: each CTA brings half the rows of A and
// converts (or brings) half the columns of B, and one thread of the pair issues MMAs over both (cta_group::2).  Warp roles:
// 0 TMA producer (A, and B of the weight gradient), 1 MMA issuer and tensor-memory owner, 2 TMA producer of the INT8 tiles,
// 4-7 epilogue, from 8 on converters; 3 and the last two (of the second CTA) relay its converters' arrivals to the issuer.
//
// What bounds it: shared memory's 128 bytes per clock against the MMA, then power.  Per K block of 64 and 256 rows a CTA's
// MMAs take 512 clocks.  A 256-row tile's traffic (A, half of B, codes, each written once and read once) is 80 KB, 640
// clocks, with a converted operand and 64 KB, 512 clocks, without; a 512-row tile uses B twice: 64 KB and 56 KB per 256 rows,
// and half the conversions.  (Single CTAs with tiles of 128 or 256 rows: 96 to 128 KB.)  A 256-row tile leaves tensor memory
// room for a second accumulator, so that its epilogue overlaps the next tile.  The tensor pipe is busy 69 to 82 % of the active
// clocks with a converted operand (8192 rows), 90 % without.  Time by single CTAs -> by pairs, T x m x n: forward 8192 x 2048 x 5461
// 175 -> 144 us, 3001 x 11008 x 4096 240 -> 209; input gradient 210 -> 150, 365 -> 203; weight gradient 155 -> 132, 217 -> 194.
// Short products stay with single CTAs (linear_single.cu; see single_pays).
// Every barrier wait is bounded; a wait that runs out raises QG_DEV_WAIT_EXPIRED and the role stops.
#include <algorithm>
#include <atomic>
#include <cstring>

#include "launch.cuh"
#include "linear_common.cuh"

namespace qg {

using namespace linear;

namespace {

struct LinArgs {
  CUtensorMap mapA;            // bf16 activations: K-major 2-D (X of the forward product, dY of the input gradient) or
                               // chunked 3-D (dY of the weight gradient)
  CUtensorMap mapB;            // INT8 codes of W (2-D, bytes) or, for the weight gradient, X chunked 3-D
  const float* scales;         // of W: [w_rows][ngroups]
  const float* zeros;
  int32_t ngroups, w_rows;
  uint16_t* D;                 // bf16 output, row-major
  int64_t ldd;
  int32_t rows, cols, K;       // accumulator extents and contraction length
  int32_t mblocks, nblocks;
  int32_t tile0, tile_end;     // the tiles of this launch
  int32_t split;               // 1: persistent pairs walk the tiles; else one cluster of `split` pairs per tile, see Walk
};

// The tiles and K blocks of a CTA pair.  A launch is either persistent (pairs walk whole tiles) or split: the pairs of a
// cluster take one tile together, each a run of its K blocks, and add up their accumulators through distributed shared
// memory.
struct Walk {
  int first, end, stride, kb0, kb1;
  uint32_t half, leader, part;   // this CTA's rows of the tile (0 or 1), its pair's first CTA, its pair among the tile's
  __device__ explicit Walk(const LinArgs& a) {
    const int kblocks = (a.K + kBK - 1) / kBK;
    const uint32_t rank = cluster_ctarank();
    half = rank & 1; leader = rank & ~1u; part = rank >> 1;
    first = a.tile0 + (int)blockIdx.x / (2 * a.split);
    if (a.split == 1) {
      end = a.tile_end; stride = (int)gridDim.x / 2;
      kb0 = 0; kb1 = kblocks;
    } else {
      end = first + 1; stride = 1;
      kb0 = (int)((int64_t)kblocks * part / a.split); kb1 = (int)((int64_t)kblocks * (part + 1) / a.split);
    }
  }
};

// The K blocks of a pair's tiles one after the other, for warps that take them in turn.
struct BlockWalk {
  const Walk& w;
  int t, kb;
  __device__ BlockWalk(const Walk& walk, int skip) : w(walk), t(walk.first), kb(walk.kb0) { advance(skip); }
  __device__ bool valid() const { return t < w.end; }
  __device__ void advance(int n) {
    kb += n;
    while (kb >= w.kb1 && t < w.end) { kb -= w.kb1 - w.kb0; t += w.stride; }
  }
};

// Sum over the pairs of a cluster of one 128 x 256 accumulator.  `cta_sums` (128 KB of this CTA's shared memory): piece c of
// 32 columns is eight planes of four columns, each 16 bytes per row, so that a warp's accesses are contiguous (with each
// row's 128 bytes together, remote reads took eight times as long: 22 us for the accumulators of seven CTAs).
constexpr int kSumPiece = kTileM * 128;
__device__ __forceinline__ void dump_piece(uint8_t* cta_sums, int c, int row, const uint32_t (&v)[32]) {
  uint8_t* p = cta_sums + c * kSumPiece + row * 16;
#pragma unroll
  for (int u = 0; u < 8; ++u) *reinterpret_cast<uint4*>(p + u * (kTileM * 16)) = make_uint4(v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
}
// Columns 16 j .. 16 j + 15 of a row, summed over the CTAs half, half + 2, .. of the cluster in order, as bfloat16 pairs;
// eight loads on their way at a time.
__device__ __forceinline__ void sum_columns16(const uint8_t* cta_sums, int j, int row, uint32_t half, int pairs, uint32_t (&pk)[8]) {
  float acc[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) acc[i] = 0.f;
  const uint32_t p = smem_u32(cta_sums + (j >> 1) * kSumPiece + (j & 1) * 4 * (kTileM * 16) + row * 16);
#pragma unroll 1
  for (int r = 0; r < pairs; r += 2) {
    float4 x[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (r + h < pairs) {
        const uint32_t q = mapa_u32(p, half + 2 * (uint32_t)(r + h));
#pragma unroll
        for (int u = 0; u < 4; ++u)
          asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x[h][u].x), "=f"(x[h][u].y), "=f"(x[h][u].z), "=f"(x[h][u].w) : "r"(q + u * (kTileM * 16)) : "memory");
      }
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (r + h < pairs)
#pragma unroll
        for (int u = 0; u < 4; ++u) { acc[4 * u] += x[h][u].x; acc[4 * u + 1] += x[h][u].y; acc[4 * u + 2] += x[h][u].z; acc[4 * u + 3] += x[h][u].w; }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    __nv_bfloat162 h = __floats2bfloat162_rn(acc[2 * i], acc[2 * i + 1]);
    pk[i] = *reinterpret_cast<uint32_t*>(&h);
  }
}

template <int MODE, int MT>                                    // MT: 256-row blocks per tile
struct LinSmem {
  static constexpr bool kConvert = MODE != kWeightGrad;
  static constexpr int kABytes = MT * kTileM * kBK * 2;       // 16 KB per row block: this CTA's 128 rows of each
  static constexpr int kBBytes = kTileN / 2 * kBK * 2;         // 16 KB: its half of the columns
  static constexpr int kStageBytes = kABytes + kBBytes;
  static constexpr int kStages = MT == 2 ? 4 : kConvert ? 5 : 6;
  static constexpr int kRawBytes = kTileN / 2 * kBK;           // its half of an INT8 tile: 8 KB
  static constexpr int kRawStages = 4;
  static constexpr int kBarOffset = kStages * kStageBytes + (kConvert ? kRawStages * kRawBytes : 0);
  static constexpr int kBytes = kBarOffset + 256 + 1024;       // barriers + slack for 1024-byte alignment
  static constexpr int kGroups = MODE == kWeightGrad ? 2 : 3;   // of four converter warps (of no use but for the sums of a split tile
                                                               // where nothing is converted)
  static constexpr int kEpiWarps = 4, kConvWarps = 4 * kGroups;
  static constexpr int kRelays = kConvert ? 3 : 0;             // warp 3 and those past the converters
  static constexpr int kThreads = (4 + kEpiWarps + kConvWarps + (kConvert ? kRelays - 1 : 0)) * 32;
  static_assert(kBytes <= 227 * 1024, "shared memory budget");
  static_assert(kBytes > kHalfOfSharedMemory, "see launch_overlapping");
};

// A load that stays where it is written (the compiler moves others down to their first use).
__device__ __forceinline__ float ld_early(const float* p) {
  float v;
  asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}

template <int MODE, int MT>
__global__ void __launch_bounds__(LinSmem<MODE, MT>::kThreads, 1)
int8_linear_kernel(const __grid_constant__ LinArgs a, int32_t* __restrict__ status) {
  using S = LinSmem<MODE, MT>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* stage_base = smem;
  uint8_t* raw_base = smem + S::kStages * S::kStageBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S::kBarOffset);
  uint64_t* full = bars;
  uint64_t* empty = full + S::kStages;
  uint64_t* raw_full = empty + S::kStages;
  uint64_t* raw_empty = raw_full + 4;
  uint64_t* acc_full = raw_empty + 4;
  uint64_t* acc_empty = acc_full + 2;
  uint64_t* converted = acc_empty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(converted + S::kStages);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < S::kStages; ++i) {
      mbar_init(&full[i], S::kConvert ? 1 + 4 + 1 : 1);    // the leader's TMA producer, a group of its converter warps, the peer's relay
      mbar_init(&empty[i], 1);
      mbar_init(&converted[i], 4);
    }
    for (int i = 0; i < S::kRawStages; ++i) { mbar_init(&raw_full[i], 1); mbar_init(&raw_empty[i], 4); }
    for (int i = 0; i < 2; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], 2 * S::kEpiWarps); }
    fence_mbar_init();
    fence_proxy_async_smem();
  }
  if (warp == 1) { tmem_alloc_pair(tmem_slot, 512); tmem_relinquish_pair(); }
  tc_fence_before_sync();
  __syncthreads();
  cluster_sync_all();                              // the other CTAs' barriers exist before anything signals them
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  // Whole rounds are an ordinary launch, so everything before them is complete; the shared tiles behind them let nobody begin.
  if (a.split == 1) grid_launch_dependents();

  // tile t -> (m block, n block): consecutive tiles (concurrent pairs) share the n block, i.e. the same
  // columns of B, which for two of the three products is the weight.  `full` and `acc_empty` are the leader's.
  const Walk wk(a);

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer of A (and bf16 B)
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int t = wk.first; ok && t < wk.end; t += wk.stride) {
        const int m0 = (t % a.mblocks) * (MT * 2 * kTileM) + (int)wk.half * kTileM, n0 = (t / a.mblocks) * kTileN;
        for (int kb = wk.kb0; kb < wk.kb1; ++kb, ++it) {
          const int s = it % S::kStages;
          if (!mbar_wait(&empty[s], ((it / S::kStages) & 1) ^ 1)) { ok = false; break; }
          uint8_t* sA = stage_base + s * S::kStageBytes;
          if (wk.half == 0) mbar_arrive_expect_tx(&full[s], 2 * (MODE == kWeightGrad ? S::kStageBytes : S::kABytes));
          const uint32_t lead_full = mapa_u32(smem_u32(&full[s]), wk.leader);
          if (MODE == kWeightGrad) {
#pragma unroll
            for (int h = 0; h < MT; ++h)
              tma_load_3d_pair(sA + h * (S::kABytes / MT), &a.mapA, lead_full, 0, kb * kBK, (m0 + h * 2 * kTileM) / 64);
            tma_load_3d_pair(sA + S::kABytes, &a.mapB, lead_full, 0, kb * kBK, n0 / 64 + 2 * (int)wk.half);
          } else {
#pragma unroll
            for (int h = 0; h < MT; ++h)                             // rows past the matrix read as zero
              tma_load_2d_pair(sA + h * (S::kABytes / MT), &a.mapA, lead_full, kb * kBK, m0 + h * 2 * kTileM);
          }
        }
      }
      ok = ok && mbar_drain<S::kStages>(empty, it);
      if (!ok) raise_expired(status);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    if (lane == 0 && wk.half == 0) {
      constexpr uint32_t idesc = umma_idesc_bf16(2 * kTileM, kTileN, MODE == kWeightGrad, MODE != kForward);
      // K-major: rows of 128 bytes, 8-row groups 1024 bytes apart, 16 K indices = 32 bytes along the row.
      // MN-major: 64-wide slabs of kSlab bytes, 8 K indices = 1024 bytes, 16 K indices = 2048 bytes.
      const uint64_t desc_a0 = MODE == kWeightGrad ? umma_smem_desc_sw128(smem_u32(stage_base), kSlab, 1024)
                                                   : umma_smem_desc_sw128(smem_u32(stage_base), 16, 1024);
      const uint64_t desc_b0 = MODE == kForward ? umma_smem_desc_sw128(smem_u32(stage_base) + S::kABytes, 16, 1024)
                                                : umma_smem_desc_sw128(smem_u32(stage_base) + S::kABytes, kSlab, 1024);
      constexpr uint64_t astep = MODE == kWeightGrad ? (2048 >> 4) : (32 >> 4);
      constexpr uint64_t bstep = MODE == kForward ? (32 >> 4) : (2048 >> 4);
      uint32_t it = 0, tcount = 0;
      bool ok = true;
      for (int t = wk.first; ok && t < wk.end; t += wk.stride, ++tcount) {
        // one row block per tile: two accumulators take alternate tiles; two: the tile has both, each handed over by itself
        const uint32_t ab = MT == 1 ? (tcount & 1) : 0u, use = MT == 1 ? (tcount >> 1) : tcount;
        if (!mbar_wait_cluster(&acc_empty[ab], (use & 1) ^ 1)) { ok = false; break; }
        tc_fence_after_sync();
        const uint32_t d_tmem = tmem_base + ab * kTileN;
        for (int kb = wk.kb0; kb < wk.kb1; ++kb, ++it) {
          const int s = it % S::kStages;
          if (!(S::kConvert ? mbar_wait_cluster(&full[s], (it / S::kStages) & 1) : mbar_wait(&full[s], (it / S::kStages) & 1))) { ok = false; break; }
          tc_fence_after_sync();
          const uint64_t da = desc_a0 + (uint64_t)((s * S::kStageBytes) >> 4);
          const uint64_t db = desc_b0 + (uint64_t)((s * S::kStageBytes) >> 4);
#pragma unroll
          for (int h = 0; h < MT; ++h) {
            if (h == 1 && kb == wk.kb0) {
              if (!mbar_wait_cluster(&acc_empty[1], (use & 1) ^ 1)) { ok = false; break; }
              tc_fence_after_sync();
            }
#pragma unroll
            for (int k = 0; k < kBK / 16; ++k)
              umma_bf16_pair(d_tmem + h * kTileN, da + (uint64_t)((h * (S::kABytes / MT)) >> 4) + k * astep, db + k * bstep, idesc,
                             (kb != wk.kb0) || (k != 0));
          }
          if (!ok) break;
          umma_commit_pair(&empty[s], wk.leader);
        }
        if (ok) umma_commit_pair(&acc_full[ab], wk.leader);
      }
      if (!ok) raise_expired(status);
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------------ TMA producer of the INT8 tiles
    if (S::kConvert && lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int t = wk.first; ok && t < wk.end; t += wk.stride) {
        const int n0 = (t / a.mblocks) * kTileN + (int)wk.half * (kTileN / 2);
        for (int kb = wk.kb0; kb < wk.kb1; ++kb, ++it) {
          const int rs = it % S::kRawStages;
          if (!mbar_wait(&raw_empty[rs], ((it / S::kRawStages) & 1) ^ 1)) { ok = false; break; }
          mbar_arrive_expect_tx(&raw_full[rs], S::kRawBytes);
          // input gradient: 64 rows of W (the tile's K) x 128 bytes along n (this CTA's half of its N), no swizzle;
          // forward: 128 rows of W (its half of the tile's N) x 64 bytes along n (the tile's K), 64-byte swizzle
          if (MODE == kForward) tma_load_2d(raw_base + rs * S::kRawBytes, &a.mapB, &raw_full[rs], kb * kBK, n0);
          else tma_load_2d(raw_base + rs * S::kRawBytes, &a.mapB, &raw_full[rs], n0, kb * kBK);
        }
      }
      if (!ok) raise_expired(status);
    }
  } else if (warp == 3 || warp >= 4 + S::kEpiWarps + S::kConvWarps) {
    // ------------------------------------------------------------------ relays: the second CTA's converted operand -> the issuer
    // An arrival that orders a converter's stores for the other CTA's issuer has to release at cluster scope, which takes some 600
    // clocks or more (a converter also waits for its loads of the next scales then).  So the converters arrive at CTA scope on a
    // barrier of their own CTA, and threads that have nothing else to do pass their arrivals on: they release what they have
    // acquired.  One such thread would be the limit, three take the K blocks in turn.  Forward 8192 x 2048 x 5461 / input gradient
    // 3001 x 11008 x 4096: the converters at cluster scope 159 / 216 us, one relay 179 / 249, three 145 / 204.
    const int relay = warp == 3 ? 0 : warp - (4 + S::kEpiWarps + S::kConvWarps) + 1;
    if (S::kConvert && wk.half == 1 && lane == 0) {
      uint32_t it = relay;
      bool ok = true;
      for (BlockWalk bw(wk, relay); ok && bw.valid(); bw.advance(S::kRelays), it += S::kRelays) {
        const int s = it % S::kStages;
        ok = mbar_wait(&converted[s], (it / S::kStages) & 1);
        if (ok) mbar_arrive_cluster(mapa_u32(smem_u32(&full[s]), wk.leader));
      }
      if (!ok) raise_expired(status);
    }
  } else if (warp >= 4 && warp < 4 + S::kEpiWarps) {
    // ------------------------------------------------------------------ epilogue: fp32 accumulator -> bf16
    const int q = warp & 3;
    uint32_t tcount = 0;
    bool ok = true;
    for (int t = wk.first; ok && t < wk.end; t += wk.stride, ++tcount) {
      const int m0 = (t % a.mblocks) * (MT * 2 * kTileM) + (int)wk.half * kTileM, n0 = (t / a.mblocks) * kTileN;
      const uint32_t ab = MT == 1 ? (tcount & 1) : 0u, use = MT == 1 ? (tcount >> 1) : tcount;
      ok = mbar_wait_warp(&acc_full[ab], use & 1);
      if (!ok) break;
      tc_fence_after_sync();
      if (a.split > 1) break;                          // see the end of the kernel
#pragma unroll 1
      for (int cc = 0; cc < MT * (kTileN / 32); ++cc) {
        const int h = cc / (kTileN / 32), c = cc % (kTileN / 32);      // row block, 32-column piece
        const uint32_t tacc = tmem_base + ((uint32_t)(q * 32) << 16) + (ab + h) * kTileN;
        uint32_t v[32];
        tmem_ld_32x32(tacc + 32 * c, v);
        tmem_ld_wait();
        if (c == kTileN / 32 - 1) {                    // every read of this tile's accumulator has landed
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) {
            if (wk.half == 0) mbar_arrive(&acc_empty[ab + h]);
            else mbar_arrive_cluster(mapa_u32(smem_u32(&acc_empty[ab + h]), wk.leader));
          }
        }
        if (n0 + 32 * c < a.cols) store_piece(a.D, a.ldd, a.rows, a.cols, m0 + h * 2 * kTileM + q * 32, n0 + 32 * c, lane, v);
        __syncwarp();                                  // the next loads from tensor memory are the whole warp's
      }
    }
    if (!ok && lane == 0) raise_expired(status);
  } else if (S::kConvert && warp >= 8) {   // (up to the relays above)
    // ------------------------------------------------------------------ converters: INT8 tile -> bf16 operand
    // Groups of four warps take K blocks in turn, so that the chain of one block (wait, load, convert, store, fence, arrive:
    // 900 to 1600 clocks) overlaps those of the next: with two groups the input gradient 3001 x 11008 x 4096 took a quarter
    // longer; four are no better.  The scales are loaded a block ahead.
    const int grp = (warp - 8) >> 2, lt = threadIdx.x & 127;
    uint32_t it = grp;
    bool ok = true;
    constexpr int kRows = MODE == kForward ? 1 : 2;      // rows of W a thread converts
    float next_sc[kRows], next_z[kRows];
    auto fetch = [&](const BlockWalk& b) {
      // forward: row n0 + 128 half + lt of W, scale of group kb / 4; input gradient: rows 64 kb + lt / 4 and + 32, group n0 / 256
      const int nb = b.t / a.mblocks;
#pragma unroll
      for (int h = 0; h < kRows; ++h) {
        const int wr = MODE == kForward ? nb * kTileN + (int)wk.half * (kTileN / 2) + lt : b.kb * kBK + (lt >> 2) + 32 * h;
        const int64_t idx = (int64_t)wr * a.ngroups + (MODE == kForward ? b.kb / (kGroup / kBK) : nb * (kTileN / kGroup));
        const bool valid = b.valid() && wr < a.w_rows;
        next_sc[h] = valid ? ld_early(a.scales + idx) : 0.f;
        next_z[h] = valid ? ld_early(a.zeros + idx) : 0.f;
      }
    };
    BlockWalk bw(wk, grp);
    fetch(bw);
    for (; ok && bw.valid(); it += S::kGroups) {
      {
        float sc[kRows], bias[kRows];
#pragma unroll
        for (int h = 0; h < kRows; ++h) { sc[h] = next_sc[h]; bias[h] = 8388736.0f + next_z[h]; }     // 2^23 + 128 + z
        bw.advance(S::kGroups);
        fetch(bw);
        const int rs = it % S::kRawStages, s = it % S::kStages;
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(&raw_full[rs], (it / S::kRawStages) & 1) && mbar_wait(&empty[s], ((it / S::kStages) & 1) ^ 1));
        if (!ok) break;
        const uint8_t* raw = raw_base + rs * S::kRawBytes;
        uint8_t* sB = stage_base + s * S::kStageBytes + S::kABytes;
        if (MODE == kForward) {
          // raw: [128 rows][64 bytes], 16-byte piece c of row r at c ^ ((r >> 1) & 3); operand (K-major): [128 rows][128 bytes],
          // piece j of row r at j ^ (r & 7)
          const uint8_t* rrow = raw + lt * 64;
          uint8_t* orow = sB + lt * 128;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const uint4 codes = *reinterpret_cast<const uint4*>(rrow + ((c ^ ((lt >> 1) & 3)) << 4));
            uint4 lo, hi;
            dequant16(codes, bias[0], sc[0], lo, hi);
            *reinterpret_cast<uint4*>(orow + (((2 * c) ^ (lt & 7)) << 4)) = lo;
            *reinterpret_cast<uint4*>(orow + (((2 * c + 1) ^ (lt & 7)) << 4)) = hi;
          }
        } else {
#pragma unroll
          for (int h = 0; h < kRows; ++h) {
            // raw: [64 rows][128 bytes]; operand (MN-major): slab i holds columns 64 i .. 64 i + 63 as
            // [64 K rows][128 bytes], 16-byte piece j of row k stored at j ^ (k & 7)
            const int k = (lt >> 2) + 32 * h, q4 = lt & 3;
            const uint8_t* rrow = raw + k * 128 + q4 * 16;
            uint8_t* orow = sB + k * 128;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const uint4 codes = *reinterpret_cast<const uint4*>(rrow + i * 64);
              uint4 lo, hi;
              dequant16(codes, bias[h], sc[h], lo, hi);
              *reinterpret_cast<uint4*>(orow + i * kSlab + (((2 * q4) ^ (k & 7)) << 4)) = lo;
              *reinterpret_cast<uint4*>(orow + i * kSlab + (((2 * q4 + 1) ^ (k & 7)) << 4)) = hi;
            }
          }
        }
        fence_proxy_async_smem();                      // the MMA reads these stores through the async proxy
        __syncwarp();
        if (lane == 0) { mbar_arrive(&raw_empty[rs]); mbar_arrive(wk.half == 0 ? &full[s] : &converted[s]); }
      }
    }
    if (!ok && lane == 0) raise_expired(status);
  }

  __syncwarp();                                        // also the warps of which one lane had a role
  if (a.split > 1) {
    // Every MMA of the tile is complete, so the operand stages are free: they hold the sums on their way.  The
    // epilogue warps and the converters add up and store, sixteen columns at a time, whatever share of the tile this CTA has.  The cluster barriers
    // count warps: only stores are under a condition of the lane, and every warp joins before each of them.
    const int q = warp & 3, row = q * 32 + lane;
    const int m0 = (wk.first % a.mblocks) * (MT * 2 * kTileM) + (int)wk.half * kTileM, n0 = (wk.first / a.mblocks) * kTileN;
#pragma unroll 1
    for (int h = 0; h < MT; ++h) {
      const bool some = m0 + h * 2 * kTileM < a.rows;
      if (some && warp >= 4 && warp < 4 + S::kEpiWarps) {
#pragma unroll 1
        for (int c = 0; c < kTileN / 32 && n0 + 32 * c < a.cols; ++c) {
          uint32_t v[32];
          tmem_ld_32x32(tmem_base + ((uint32_t)(q * 32) << 16) + h * kTileN + 32 * c, v);
          tmem_ld_wait();
          dump_piece(stage_base, c, row, v);
        }
      }
      __syncwarp();
      cluster_sync_all();
      if (some && warp >= 4 && warp < 4 + S::kEpiWarps + S::kConvWarps) {
#pragma unroll 1
        for (int j = (int)wk.part + a.split * ((warp - 4) >> 2); j < kTileN / 16 && n0 + 16 * j < a.cols; j += a.split * (1 + S::kGroups)) {
          uint32_t pk[8];
          sum_columns16(stage_base, j, row, wk.half, a.split, pk);
          const int gr = m0 + h * 2 * kTileM + row, col = n0 + 16 * j;
          uint16_t* d = a.D + (int64_t)gr * a.ldd + col;
          if (gr < a.rows && col + 16 <= a.cols) {
            *reinterpret_cast<uint4*>(d) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            *reinterpret_cast<uint4*>(d + 8) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
          } else if (gr < a.rows) {
#pragma unroll
            for (int i = 0; i < 16; ++i)
              if (col + i < a.cols) d[i] = (uint16_t)((i & 1) ? (pk[i >> 1] >> 16) : (pk[i >> 1] & 0xFFFFu));
          }
        }
      }
      __syncwarp();
      if (h + 1 < MT) cluster_sync_all();          // nobody refills its sums before all have read them
    }
    grid_dependency_wait();                            // the launch before this one, which it may have overtaken
  }
  tc_fence_before_sync();
  __syncthreads();
  cluster_sync_all();                              // nobody leaves while another may still signal it or read its sums
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc_pair(tmem_base, 512);
  }
  __syncwarp();
  cluster_sync_all();                              // nor while its peer still gives tensor memory back: see tmem_dealloc_pair
}

constexpr int kDevices = 64, kMaxSplit = 4;

// Clusters of `split` CTA pairs of a kernel that are resident at once, asked once per device.
template <auto KERN, int THREADS, int SMEM>
int resident_clusters(int split, int dev) {
  static std::atomic<int> known[kDevices][kMaxSplit + 1];
  int v = known[dev][split].load(std::memory_order_relaxed);
  if (v != 0) return v - 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(2 * split * 64));
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = SMEM;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = (unsigned)(2 * split); attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, KERN, &cfg) != cudaSuccess) { (void)cudaGetLastError(); n = 0; }
  known[dev][split].store(n + 1, std::memory_order_relaxed);
  return n;
}

// CTA pairs that share a tile of the last, unfilled round (`tiles` of them for `pairs` pairs): as many as keep every tile's
// cluster resident, each with at least four K blocks.  1 (the round as it is) where that saves fewer than `saves` K blocks:
// adding up the accumulators takes 4 to 8 us, a K block 0.27 (weight gradient) to 0.5 us.  Measured, a pair to each tile and
// shared, 256 rows: forward 310 x 1159 x 5993 52 -> 30 us, 512 x 2048 x 5461 61 -> 36, 64 x 4096 x 4096 38 -> 24; input gradient 64 x 4096
// x 4096 38 -> 24, 18 x 1137 x 163 18 -> 16; weight gradient 2000 x 600 x 900 24 -> 20.
template <auto KERN, int THREADS, int SMEM>
int choose_split(int tiles, int kblocks, int pairs, int saves, int dev) {
  int split = tiles > 0 ? pairs / tiles : 1;
  split = std::min(std::min(split, kMaxSplit), kblocks / 4);
  while (split > 1 && resident_clusters<KERN, THREADS, SMEM>(split, dev) < tiles) --split;
  return split > 1 && kblocks - (kblocks + split - 1) / split >= saves ? split : 1;
}

// How a kernel takes a product: whole rounds of one tile per pair by persistent CTAs, and the remainder, where that pays, by a
// second launch of clusters.
struct Rounds {
  int mblocks, pairs, whole, rest, split;
  double time;                 // estimate, in K blocks of the kernel with one row block per tile
};

template <int MODE, int MT>
int plan_rounds(const LinArgs& a, int dev, Rounds& r) {
  using S = LinSmem<MODE, MT>;
  constexpr auto kern = int8_linear_kernel<MODE, MT>;
  static bool smem_set[kDevices] = {};               // opted into its shared memory, per device
  if (!smem_set[dev]) {
    QG_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, S::kBytes));
    smem_set[dev] = true;
  }
  r.pairs = resident_clusters<kern, S::kThreads, S::kBytes>(1, dev);
  if (r.pairs < 1) return QG_CUDA_ERROR;
  const int rows = MT * 2 * kTileM, kblocks = (a.K + kBK - 1) / kBK;
  r.mblocks = (a.rows + rows - 1) / rows;
  const int total = r.mblocks * a.nblocks;
  r.rest = total % r.pairs;
  r.split = choose_split<kern, S::kThreads, S::kBytes>(r.rest, kblocks, r.pairs, MODE == kWeightGrad ? 16 : 8, dev);
  r.whole = total - r.rest;
  // A K block of a 512-row tile takes 1.9 of a 256-row tile's time without a converted operand and 1.57 with one, as fitted to
  // products of few rounds; where 512 rows are taken for their rounds it is less (16384 x 4096 x 4096 forward 652 us for 14
  // rounds, 437 for 7).  Its epilogue, which nothing overlaps, and the sums of a split tile count as 6 and 12 blocks per 256
  // rows.  So small products keep 256 rows (512 x 2048 x 5461 forward 36 us against 46, 2000 x 600 x 900 22 against 30), and weight
  // gradients but for a few (904 x 6535 x 4003 42 against 53).
  const double block = MT == 1 ? 1.0 : MODE == kWeightGrad ? 1.9 : 1.57, tile = MT == 1 ? 0 : 6, sums = r.split > 1 ? MT * 12 : 0;
  r.time = (r.whole / r.pairs) * (kblocks * block + tile) + (r.rest ? (kblocks + r.split - 1) / r.split * block + tile + sums : 0);
  if (r.split == 1) { r.whole = total; r.rest = 0; }
  return QG_OK;
}

// The second launch may begin while the first drains (programmatic dependent launch): it shares no data with it, and waits
// for its completion only at its own end.
template <int MODE, int MT>
int launch_rounds(LinArgs a, const Rounds& r, int32_t* status, cudaStream_t st) {
  using S = LinSmem<MODE, MT>;
  a.mblocks = r.mblocks;
  auto launch = [&](int tile0, int tile_end, int split, int clusters, bool overlap) -> int {
    a.tile0 = tile0; a.tile_end = tile_end; a.split = split;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(clusters * 2 * split));
    cfg.blockDim = dim3(S::kThreads);
    cfg.dynamicSmemBytes = S::kBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[2]{};
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)(2 * split); attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap ? 2 : 1;
    QG_CUDA_TRY(cudaLaunchKernelEx(&cfg, int8_linear_kernel<MODE, MT>, a, status));
    count_launch();
    return QG_OK;
  };
  if (r.whole > 0) {
    const int rc = launch(0, r.whole, 1, std::min(r.whole, r.pairs), false);
    if (rc != QG_OK) return rc;
  }
  return r.rest > 0 ? launch(r.whole, r.whole + r.rest, r.split, r.rest, r.whole > 0) : QG_OK;
}

// Whether single CTAs (linear_single.cu) take the forward product or the weight gradient in less time than the pairs' plan `r`.  Both
// in microseconds, fitted to 107 products of 17 .. 8192 tokens and 163 .. 11008 rows and columns, device time: what a launch
// takes from begin to end, K blocks, what a further round adds, and a second launch that has to wait for whole clusters of free SMs.
// The pairs have to be the faster by more than the fit is off by.  Pairs and single CTAs, T x m x n: forward 256 x 512 x 512 14.4
// and 12.3, 1024 x 1024 x 1024 16.5 and 16.4, 256 x 2048 x 2048 18.5 and 22.6, 8192 x 4096 x 512 57 and 49, 8192 x 2048 x 2048 71 and 84;
// weight gradient 256 x 1024 x 1024 10.3 and 8.2, 1024 x 2048 x 2048 14.5 and 12.4, 4096 x 512 x 512 18.5 and 24.8, 8192 x 768 x 2048 34
// and 52.  (The input gradient by single CTAs was slower throughout.)
template <int MODE>
bool single_pays(const LinArgs& a, const Rounds& r, int mt) {
  const double kb = (a.K + kBK - 1) / kBK;
  const int across = MODE == kForward ? a.cols : a.rows, along = MODE == kForward ? a.rows : a.cols;   // forward is computed transposed
  const int64_t tiles = (int64_t)((across + kTileM - 1) / kTileM) * ((along + kTileN - 1) / kTileN);
  if (tiles > (int64_t)1 << 30) return false;                        // the tile index is an int
  const double more = (double)((tiles - 1) / (2 * r.pairs)), pairs_more = (r.whole + r.pairs - 1) / r.pairs - 1.0;
  const bool two_launches = r.whole > 0 && r.rest > 0;
  if (MODE == kForward) {
    const double single = 8.5 + 0.43 * kb + more * std::max(0.48 * kb + 2.0, 4.0);
    const double pairs = 11.7 + (mt == 1 ? 0.33 * r.time + 3.0 * std::max(pairs_more, 0.0) : 0.45 * r.time) + (two_launches ? 9.0 : 0.0);
    return pairs >= 0.96 * single;
  }
  const double single = 8.0 + 0.27 * kb * (more + 1.0) + 1.6 * more;
  const double pairs = 10.0 + 0.27 * r.time + std::max(pairs_more, 0.0) * std::max(2.4 - 0.27 * kb, 0.0) + (two_launches ? 8.0 : 0.0);
  return pairs >= 0.94 * single;
}

// One or two row blocks per tile, or single CTAs (`by_single_ctas` launches them), whichever is estimated to take less time.
// `operands` fills in what the pairs read from.
template <int MODE, class Operands, class Single>
int launch_product(const LinArgs& a, int32_t* status, cudaStream_t st, Operands operands, Single by_single_ctas) {
  int dev = 0;
  QG_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kDevices) return QG_UNSUPPORTED_SHAPE;
  Rounds one, two;
  int rc = plan_rounds<MODE, 1>(a, dev, one);
  if (rc == QG_OK) rc = plan_rounds<MODE, 2>(a, dev, two);
  if (rc != QG_OK) return rc;
  const bool tall = two.time < one.time;
  if (MODE != kInputGrad && single_pays<MODE>(a, tall ? two : one, tall ? 2 : 1)) return by_single_ctas();
  if (!operands()) return QG_CUDA_ERROR;
  return tall ? launch_rounds<MODE, 2>(a, two, status, st) : launch_rounds<MODE, 1>(a, one, status, st);
}

}  // namespace

int launch_int8_linear(int mode, const uint16_t* act, int64_t ld_act, const uint16_t* act2, int64_t ld_act2,
                       const qg_qtensor* W, int64_t T, int64_t m, int64_t n, uint16_t* D, int64_t ldd,
                       int32_t* status, cudaStream_t st) {
  if (mode == kForward && T <= kSkinnyTokens) return launch_int8_linear_skinny(act, ld_act, W, T, D, ldd, st);
  LinArgs a;
  memset(&a, 0, sizeof(a));
  a.D = D;
  a.ldd = ldd;
  a.rows = (int32_t)(mode == kWeightGrad ? m : T);
  a.cols = (int32_t)(mode == kForward ? m : n);
  a.K = (int32_t)(mode == kForward ? n : mode == kInputGrad ? m : T);
  a.nblocks = (a.cols + kTileN - 1) / kTileN;
  if ((int64_t)((a.rows + 2 * kTileM - 1) / (2 * kTileM)) * a.nblocks > (int64_t)1 << 30) return QG_UNSUPPORTED_SHAPE;   // the tile index is an int
  const auto operands = [&] {
    if (mode == kWeightGrad)
      // act = dY (T x m), act2 = X (T x n); both enter as 64-wide column slabs, K = T runs down the rows
      return make_map_chunked(&a.mapA, act, T, (m + 63) / 64, ld_act, kBK, 2) && make_map_chunked(&a.mapB, act2, T, (n + 63) / 64, ld_act2, kBK, 2);
    a.scales = W->scales;
    a.zeros = W->zeros;
    a.ngroups = (int32_t)((n + kGroup - 1) / kGroup);
    a.w_rows = (int32_t)m;
    // act = X (T x n) or dY (T x m)
    return make_map(&a.mapA, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, act, a.K, T, ld_act, kBK, kTileM, CU_TENSOR_MAP_SWIZZLE_128B) &&
           (mode == kForward ? make_map(&a.mapB, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, W->codes, n, m, W->ld, kBK, kTileN / 2, CU_TENSOR_MAP_SWIZZLE_64B)
                             : make_map(&a.mapB, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, W->codes, n, m, W->ld, kTileN / 2, kBK, CU_TENSOR_MAP_SWIZZLE_NONE));
  };
  const auto single = [&] { return launch_single(mode, act, ld_act, act2, ld_act2, W, T, m, n, D, ldd, status, st); };
  if (mode == kForward) return launch_product<kForward>(a, status, st, operands, single);
  if (mode == kInputGrad) return launch_product<kInputGrad>(a, status, st, operands, single);
  return launch_product<kWeightGrad>(a, status, st, operands, single);
}

}  // namespace qg
