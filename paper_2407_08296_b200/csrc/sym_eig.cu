// Leading eigenvectors of symmetric matrices, several of one size at a time, for the subspace refresh (Sec. 3.5).
//
//   1. Householder reduction to tridiagonal form, A = H T H^T, H = H_0 H_1 ... (binary32)
//   2. the r largest eigenvalues of T by multisection on Sturm counts (binary64)
//   3. their eigenvectors by one twisted factorisation of T - lambda each (binary64)
//   4. X = H Z (binary32)
//
// The reduction is a chain of N dependent steps whatever runs it, so it is laid out for the shortest step: the matrix
// stays on the SMs (columns dealt out to the CTAs, in registers and shared memory), one pass over it per step applies the
// previous rank-2 update and multiplies by the new Householder vector, and ONE exchange through L2 per step carries what
// every CTA needs of the others.  That exchange has no barrier: every value travels in a 64-bit word of its own together with
// the step's number, and the reader polls the word itself.
#include <algorithm>
#include <cmath>
#include <mutex>

#include "refresh_common.cuh"
#include "sm100_ptx.cuh"

namespace qg {

namespace {

using ptx::fma2;
using ptx::mul2;

// ------------------------------------------------------------------------------------------ 1. tridiagonal form
// Column j of a matrix belongs to CTA j mod C of its C; row and column indices below the step are dead, so a cyclic deal
// keeps the CTAs level to the end.  Both triangles are kept: column j then yields (A v)_j by itself, with no sum over
// CTAs, and element k + 1 of column j is element j of the next pivot column, so the owner of column j publishes both
// values the next step wants at index j.  Of step k (v, tau: the Householder vector of step k - 1, its update pending):
//     P_j = (A v)_j, R_j = A_kj                      received for j >= k
//     w = tau P - kappa v, kappa = tau^2 (P . v) / 2
//     x = R - w - v w_k = (R - tau P) + v mu          (column k with the pending update; mu = 2 kappa - tau P_k, v_k = 1)
//     d_k = x_k;  v', tau', e_k annihilate x below k + 1
//     A <- A - v w^T - w v^T,  P' = A v'              one pass over the columns j > k
//     publish P'_j and A_{k+1, j}
// What bounds a step is latency: the trip through L2, two CTA barriers and the reductions.  |x|^2 is therefore taken
// from sums over R - tau P and v that are reduced together with P . v (one barrier less); where the two terms of x
// cancel the sum is taken again over x itself.
// A thread keeps rows tid + THREADS q of every column, the last columns in registers, those before in shared memory and,
// past that, in global memory (L2): the row's v, w, v' are then registers too, and the pass reads nothing but two
// scalars per column.
constexpr uint32_t kPollLimit = 1u << 20;
constexpr int kTriSmem = 225 * 1024;

// Two values of a step, each with the step's number beside it in ONE 8-byte element: an access of the memory model covers an
// element, so a reader that sees the number has the value.
struct __align__(16) Tagged {
  uint64_t a, b;               // (tag << 32) | bits of the value
};
__device__ __forceinline__ Tagged ld_tagged(const Tagged* p) {
  Tagged v;
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(v.a), "=l"(v.b) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_tagged(Tagged* p, float a, float b, uint32_t tag) {
  const uint64_t high = (uint64_t)tag << 32;
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(high | __float_as_uint(a)), "l"(high | __float_as_uint(b)) : "memory");
}
__device__ __forceinline__ uint32_t tag_of(uint64_t x) { return (uint32_t)(x >> 32); }
__device__ __forceinline__ float value_of(uint64_t x) { return __uint_as_float((uint32_t)x); }

struct TriArgs {
  Ptrs<float> A, V, tau, d, e;
  Ptrs<Tagged> xchg;
  int N, Np, C;
  int in_smem;               // columns per CTA that shared memory holds
};

__device__ __forceinline__ float2 both(float x) { return make_float2(x, x); }
// Sums of several values over the lanes of a warp, by halving the values and the lanes together.
__device__ __forceinline__ float halve(float lo, float hi, int bit, int lane) {
  const bool up = lane & bit;
  return (up ? hi : lo) + __shfl_xor_sync(0xFFFFFFFFu, up ? lo : hi, bit);
}
// lane 8 i: the sum of value i
__device__ __forceinline__ float warp_sums4(const float (&v)[4], int lane) {
  const float a = halve(v[0], v[2], 16, lane), b = halve(v[1], v[3], 16, lane);
  float s = halve(a, b, 8, lane);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
  return s;
}
// lane 4 i: the sum of value i
__device__ __forceinline__ float warp_sums8(const float2 (&v)[4], int lane) {
  const float a = halve(v[0].x, v[2].x, 16, lane), b = halve(v[0].y, v[2].y, 16, lane);
  const float c = halve(v[1].x, v[3].x, 16, lane), d = halve(v[1].y, v[3].y, 16, lane);
  const float e = halve(a, c, 8, lane), f = halve(b, d, 8, lane);
  float s = halve(e, f, 4, lane);
  s += __shfl_xor_sync(0xFFFFFFFFu, s, 2);
  s += __shfl_xor_sync(0xFFFFFFFFu, s, 1);
  return s;
}

template <int NQ, int THREADS, int RC>         // rows per thread (N <= NQ * THREADS), columns in registers
__global__ void __launch_bounds__(THREADS, 1)
tridiagonal_kernel(const __grid_constant__ TriArgs a, int32_t* __restrict__ status) {
  constexpr int WARPS = THREADS / 32;
  extern __shared__ __align__(16) float tri_smem[];
  __shared__ __align__(16) float4 red1[16];
  __shared__ float red_x[WARPS];
  __shared__ float s_pk, s_a1, s_v1;
  __shared__ int s_fail;
  const int N = a.N, Np = a.Np, C = a.C;
  const int mat = blockIdx.x / C, cta = blockIdx.x % C;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float* const A = a.A.p[mat];
  float* const Vg = a.V.p[mat];
  Tagged* const xchg = a.xchg.p[mat];
  const int ncols = (N - cta + C - 1) / C;     // this CTA's columns: cta + l C, l = 0 .. ncols - 1
  const int nr = min(ncols, RC), ns = min(ncols - nr, a.in_smem), ng = ncols - nr - ns;   // registers, shared, global (these retire first)
  const int nc8 = ((N + C - 1) / C + 8) & ~7;  // pitch of the per-column arrays: groups of eight may reach past the end
  float* const colP = tri_smem;                // P_j and v_j of this CTA's columns
  float* const colV = colP + 2 * nc8;          // (twice the room: a group starts anywhere)
  float* const pivot = colV + 2 * nc8;         // A_{k+1, j}
  float* const part = pivot + 2 * nc8;         // [warp][column] partial sums of P'_j
  float4* const scols = reinterpret_cast<float4*>(part + WARPS * 2 * nc8);   // [group of four columns][Np]

  float2 ar[NQ][RC / 2];
  float v[NQ], w[NQ], vn[NQ], r[NQ];
  int slot[NQ];                                // the row's own column, if it is this CTA's, else -1
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int j = tid + q * THREADS;
    v[q] = w[q] = 0.f;
    r[q] = j < N ? Vg[(int64_t)(N - 1) * Np + j] : 0.f;   // row 0 as eig_scale_kernel put it aside
    slot[q] = j < N && j % C == cta ? j / C : -1;
#pragma unroll
    for (int c = 0; c < RC; c += 2) {
      const int l = ng + ns + c;
      ar[q][c / 2].x = (l < ncols && j < Np) ? A[(int64_t)(cta + l * C) * Np + j] : 0.f;
      ar[q][c / 2].y = (l + 1 < ncols && j < Np) ? A[(int64_t)(cta + (l + 1) * C) * Np + j] : 0.f;
    }
  }
  for (int l = 0; l < ns; l += 4)
    for (int i = tid; i < Np; i += THREADS) {
      float x[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) x[c] = l + c < ns ? A[(int64_t)(cta + (ng + l + c) * C) * Np + i] : 0.f;
      scols[(l >> 2) * Np + i] = make_float4(x[0], x[1], x[2], x[3]);
    }
  for (int i = tid; i < 6 * nc8; i += THREADS) tri_smem[i] = 0.f;
  if (tid < 16) red1[tid] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (tid == 0) { s_fail = 0; s_pk = 0.f; }
  __syncthreads();

  // A CTA works while it owns a column beyond the step's, i.e. while it has something to publish: whoever has received a
  // step's values then knows that everybody who will ever read the step before has done so, and may overwrite them (the
  // exchange is double buffered by the step's parity).  The owner of column k + 1 records what step k yields.
  const int last = cta + (ncols - 1) * C;
  float tau = 0.f;
  for (int k = 0; k < N && (last > k || last == N - 1); ++k) {
    const bool writer = k == N - 1 || cta == (k + 1) % C;
    // ---- receive; sums over P . v, and over a = R - tau P and v below row k + 1
    float sums[4] = {0.f, 0.f, 0.f, 0.f};
    bool ok = true;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int j = tid + q * THREADS;
      // The whole warp stays in the loop, so that what follows is executed once and not by parts of it, and reaches the barrier
      // together.  Row after row: with all of a thread's words asked for at once the polls hold up the words themselves (2048 x
      // 5461: 9.4 ms as it is, 14.3 at once); a lane that waits alone for the rest of its warp adds a trip (10.3).
      const bool wanted = k > 0 && j >= k && j < N;
      const Tagged* const in = xchg + (k & 1) * Np + j;
      Tagged got{0, 0};
      bool here = !wanted;
      for (uint32_t polls = 0; polls < kPollLimit && !__all_sync(0xFFFFFFFFu, here); ++polls)
        if (!here) {
          got = ld_tagged(in);
          here = tag_of(got.a) == (uint32_t)k && tag_of(got.b) == (uint32_t)k;
        }
      ok = ok && here;
      float p = 0.f;
      if (j >= k && j < N) {
        if (wanted) {
          p = value_of(got.a);
          r[q] = value_of(got.b);
        }
        if (j == k) s_pk = p;
      } else {
        r[q] = 0.f;
      }
      if (slot[q] >= 0) { colP[slot[q]] = p; colV[slot[q]] = v[q]; }
      w[q] = p;
      r[q] = fmaf(-tau, p, r[q]);
      if (j == k + 1) { s_a1 = r[q]; s_v1 = v[q]; }
      sums[0] = fmaf(p, v[q], sums[0]);
      if (j > k + 1) {
        sums[1] = fmaf(r[q], r[q], sums[1]);
        sums[2] = fmaf(r[q], v[q], sums[2]);
        sums[3] = fmaf(v[q], v[q], sums[3]);
      }
    }
    if (!ok) s_fail = 1;
    {
      const float s = warp_sums4(sums, lane);
      if ((lane & 7) == 0) reinterpret_cast<float*>(&red1[warp])[lane >> 3] = s;
    }
    __syncthreads();
    if (s_fail) {                              // somebody's values never came: every CTA runs into the same limit
      if (tid == 0 && status) atomicOr(status, QG_DEV_WAIT_EXPIRED);
      return;
    }
    float s_pv, s_aa, s_av, s_vv;
    {
      const float4 t = red1[lane & 15];
      const float e = halve(t.x, t.z, 8, lane), f = halve(t.y, t.w, 8, lane);
      float s = halve(e, f, 4, lane);
      s += __shfl_xor_sync(0xFFFFFFFFu, s, 2);
      s += __shfl_xor_sync(0xFFFFFFFFu, s, 1);
      s_pv = __shfl_sync(0xFFFFFFFFu, s, 0);
      s_aa = __shfl_sync(0xFFFFFFFFu, s, 4);
      s_av = __shfl_sync(0xFFFFFFFFu, s, 8);
      s_vv = __shfl_sync(0xFFFFFFFFu, s, 12);
    }
    const float kappa = 0.5f * tau * tau * s_pv, mu = fmaf(-tau, s_pk, 2.f * kappa);
    const float alpha = fmaf(mu, s_v1, s_a1);
    float sig = fmaf(mu, fmaf(mu, s_vv, 2.f * s_av), s_aa);
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int j = tid + q * THREADS;
      w[q] = fmaf(tau, w[q], -kappa * v[q]);
      r[q] = fmaf(mu, v[q], r[q]);             // x
      if (j == k && writer) a.d.p[mat][k] = r[q];
    }
    if (k == N - 1) break;
    if (!(sig >= 0.25f * s_aa)) {              // the same in every thread of every CTA
      sig = 0.f;
#pragma unroll
      for (int q = 0; q < NQ; ++q)
        if (tid + q * THREADS > k + 1) sig = fmaf(r[q], r[q], sig);
      sig = warp_sum(sig);
      if (lane == 0) red_x[warp] = sig;
      __syncthreads();
      sig = 0.f;
      for (int i = 0; i < WARPS; ++i) sig += red_x[i];
    }
    const float tau_old = tau;
    float beta = alpha, scl = 0.f;
    tau = 0.f;
    if (sig > 1e-36f) {
      // correctly rounded, not the approximate forms: tau and scl have to be those of one reflector to the last bits
      beta = -copysignf(sqrtf(fmaf(alpha, alpha, sig)), alpha);
      tau = (beta - alpha) / beta;
      scl = 1.f / (alpha - beta);
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int j = tid + q * THREADS;
      vn[q] = j > k + 1 ? r[q] * scl : (j == k + 1 ? 1.f : 0.f);
      if (writer && j < Np) Vg[(int64_t)k * Np + j] = vn[q];
    }
    if (writer && tid == 0) { a.tau.p[mat][k] = tau; a.e.p[mat][k] = beta; }

    // ---- the pass, eight columns at a time
    const int k1 = k + 1, qk = k1 / THREADS;
    const bool pivot_thread = tid == k1 % THREADS;
    const float2 tau2 = both(tau_old), kap2 = both(-kappa);
    auto scalars = [&](int l, float2 (&wj)[4], float2 (&vj)[4]) {      // w_j, v_j of columns l .. l + 7
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        vj[c] = make_float2(colV[l + 2 * c], colV[l + 2 * c + 1]);
        wj[c] = fma2(tau2, make_float2(colP[l + 2 * c], colP[l + 2 * c + 1]), mul2(kap2, vj[c]));
      }
    };
    auto partial = [&](int l, const float2 (&acc)[4]) {
      const float s = warp_sums8(acc, lane);
      if ((lane & 3) == 0) part[warp * 2 * nc8 + l + (lane >> 2)] = s;
    };
    // columns in memory, four to a load (get(l, row), put(l, row, x): columns l .. l + 3), the next row's on its way
    auto memory_columns = [&](int l0, int l1, auto get, auto put) {
      const int q0 = k1 / THREADS;
      for (int l = l0; l < l1; l += 4) {
        if (cta + min(l + 3, l1 - 1) * C <= k) continue;               // all of them retired
        float2 wj[2], vj[2], acc[2] = {};
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          vj[c] = make_float2(colV[l + 2 * c], colV[l + 2 * c + 1]);
          wj[c] = fma2(tau2, make_float2(colP[l + 2 * c], colP[l + 2 * c + 1]), mul2(kap2, vj[c]));
        }
        float4 next = make_float4(0.f, 0.f, 0.f, 0.f);
        if (tid + q0 * THREADS < Np) next = get(l, tid + q0 * THREADS);
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          const int row = tid + q * THREADS;
          if (q * THREADS + THREADS - 1 <= k || row >= Np) continue;
          float2 lo = make_float2(next.x, next.y), hi = make_float2(next.z, next.w);
          if (q + 1 < NQ && row + THREADS < Np) next = get(l, row + THREADS);
          const float2 nv = both(-v[q]), nw = both(-w[q]), n2 = both(vn[q]);
          lo = fma2(nw, vj[0], fma2(nv, wj[0], lo));
          hi = fma2(nw, vj[1], fma2(nv, wj[1], hi));
          put(l, row, make_float4(lo.x, lo.y, hi.x, hi.y));
          acc[0] = fma2(lo, n2, acc[0]);
          acc[1] = fma2(hi, n2, acc[1]);
          if (pivot_thread && q == qk) { pivot[l] = lo.x; pivot[l + 1] = lo.y; pivot[l + 2] = hi.x; pivot[l + 3] = hi.y; }
        }
        const float sums[4] = {acc[0].x, acc[0].y, acc[1].x, acc[1].y};
        const float s = warp_sums4(sums, lane);
        if ((lane & 7) == 0 && l + (lane >> 3) < l1) part[warp * 2 * nc8 + l + (lane >> 3)] = s;
      }
    };
    if (ng > 0) {
      auto at = [&](int l, int row) -> float& { return A[(int64_t)(cta + min(l, ng - 1) * C) * Np + row]; };
      memory_columns(0, ng, [&](int l, int row) { return make_float4(at(l, row), at(l + 1, row), at(l + 2, row), at(l + 3, row)); },
                     [&](int l, int row, const float4& x) {
                       at(l, row) = x.x;
                       if (l + 1 < ng) at(l + 1, row) = x.y;
                       if (l + 2 < ng) at(l + 2, row) = x.z;
                       if (l + 3 < ng) at(l + 3, row) = x.w;
                     });
    }
    if (ns > 0) {
      auto at = [&](int l, int row) -> float4& { return scols[((l - ng) >> 2) * Np + row]; };
      memory_columns(ng, ng + ns, at, [&](int l, int row, const float4& x) { at(l, row) = x; });
    }
#pragma unroll
    for (int g = 0; g < RC / 8; ++g) {
      const int l = ng + ns + 8 * g;
      if (l < ncols && cta + min(l + 7, ncols - 1) * C > k) {
        float2 wj[4], vj[4], acc[4] = {};
        scalars(l, wj, vj);
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          if (q * THREADS + THREADS - 1 <= k) continue;
          const float2 nv = both(-v[q]), nw = both(-w[q]), n2 = both(vn[q]);
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            float2& x = ar[q][4 * g + c];
            x = fma2(nw, vj[c], fma2(nv, wj[c], x));
            acc[c] = fma2(x, n2, acc[c]);
            if (pivot_thread && q == qk) { pivot[l + 2 * c] = x.x; pivot[l + 2 * c + 1] = x.y; }
          }
        }
        partial(l, acc);
      }
    }
    __syncthreads();
    // ---- publish
    for (int l = tid; l < ncols; l += THREADS) {
      const int j = cta + l * C;
      if (j <= k) continue;
      float s = 0.f;
#pragma unroll
      for (int i = 0; i < WARPS; ++i) s += part[i * 2 * nc8 + l];
      st_tagged(xchg + (k1 & 1) * Np + j, s, pivot[l], (uint32_t)k1);
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < NQ; ++q) v[q] = vn[q];
  }
}

// The power of two that brings the largest diagonal element of a positive semi-definite A into [1, 2), so that squares
// in the reduction neither over- nor underflow.
__global__ void __launch_bounds__(256)
eig_scale_factor_kernel(const Ptrs<const float> Ab, int N, int Np, const Ptrs<float> scaleb) {
  const float* A = Ab.p[blockIdx.x];
  __shared__ float red[8];
  float top = 0.f;
  for (int i = threadIdx.x; i < N; i += 256) top = fmaxf(top, fabsf(A[(int64_t)i * Np + i]));
  top = warp_max(top);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = top;
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int i = 0; i < 8; ++i) top = fmaxf(top, red[i]);
  const int ex = (int)(__float_as_uint(top) >> 23) - 127;
  scaleb.p[blockIdx.x][0] = !(top >= FLT_MIN) || !isfinite(top) ? 1.f : ex >= 127 ? 0x1p-126f : __uint_as_float((uint32_t)(127 - ex) << 23);
}

// Applies it, zeroes the padding columns, and puts row 0 aside (in the last row of V, which holds no Householder vector):
// every CTA of the reduction starts from it, while their owners already write the columns.
__global__ void __launch_bounds__(256)
eig_scale_kernel(const Ptrs<float> Ab, int N, int Np, const Ptrs<const float> scaleb, const Ptrs<float> Vb) {
  const float s = scaleb.p[blockIdx.y][0];
  float* row = Ab.p[blockIdx.y] + (int64_t)blockIdx.x * Np;
  float* aside = blockIdx.x == 0 ? Vb.p[blockIdx.y] + (int64_t)(N - 1) * Np : nullptr;
  for (int i = threadIdx.x; i < Np; i += 256) {
    const float x = i < N ? row[i] * s : 0.f;
    row[i] = x;
    if (aside) aside[i] = x;
  }
}

// ------------------------------------------------------------------------------------------ 2. eigenvalues
// One warp per eigenvalue, 32 trial points per round.  The number of eigenvalues below x is the number of sign changes of
// p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2}; the chain per row is one fused multiply-add, and both terms are scaled
// back by a power of two every eight rows.  e^2 is kept above a floor, so that two consecutive p never vanish.
constexpr int kSturmWarps = 8;

// The diagonal as steps 2 and 3 see it: each element raised by its own part of 2^-30 of the largest (A is scaled so that
// that is between 1 and 2), a sixtieth of a unit in the last place.  Eigenvalues that coincide, as those of zero rows do,
// come apart by it and have orthogonal vectors.
__device__ __forceinline__ double diagonal(const float* d, int i) { return (double)d[i] + 0x1p-62 * (double)(uint32_t)(2654435769u * (uint32_t)i); }
constexpr double kE2Floor = 1e-36;

__device__ __forceinline__ int sturm_count(const double2* __restrict__ t, int N, double x) {
  double p0 = 1.0, p1 = t[0].x - x;
  int cnt = __double2hiint(p1) < 0 ? 1 : 0;
  int i = 1;
  for (; i + 8 <= N; i += 8) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const double2 te = t[i + u];                 // (d_i, e_{i-1}^2)
      const double p2 = fma(te.x - x, p1, -(te.y * p0));
      cnt += (uint32_t)(__double2hiint(p2) ^ __double2hiint(p1)) >> 31;
      p0 = p1;
      p1 = p2;
    }
    const int h = max(__double2hiint(p0) & 0x7FF00000, __double2hiint(p1) & 0x7FF00000);
    const double sc = __hiloint2double(min(max(0x7FE00000 - h, 0x00100000), 0x7FD00000), 0);   // 2^-exponent of the larger
    p0 *= sc;
    p1 *= sc;
  }
  for (; i < N; ++i) {
    const double2 te = t[i];
    const double p2 = fma(te.x - x, p1, -(te.y * p0));
    cnt += (uint32_t)(__double2hiint(p2) ^ __double2hiint(p1)) >> 31;
    p0 = p1;
    p1 = p2;
  }
  return cnt;
}

__global__ void __launch_bounds__(kSturmWarps * 32)
eigenvalue_kernel(const Ptrs<const float> db, const Ptrs<const float> eb, int N, int r, const Ptrs<double> lamb) {
  extern __shared__ __align__(16) double2 sturm_smem[];
  __shared__ double bound[kSturmWarps];
  const float* d = db.p[blockIdx.y];
  const float* e = eb.p[blockIdx.y];
  double b = 0.0;                                // every |eigenvalue| <= max |d_i| + |e_{i-1}| + |e_i|
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    const double di = diagonal(d, i), el = i > 0 ? (double)e[i - 1] : 0.0, er = i + 1 < N ? (double)e[i] : 0.0;
    sturm_smem[i] = make_double2(di, fmax(el * el, kE2Floor));
    b = fmax(b, fabs(di) + fabs(el) + fabs(er));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) b = fmax(b, __shfl_xor_sync(0xFFFFFFFFu, b, o));
  if ((threadIdx.x & 31) == 0) bound[threadIdx.x >> 5] = b;
  __syncthreads();
  for (int i = 0; i < kSturmWarps; ++i) b = fmax(b, bound[i]);
  const int lane = threadIdx.x & 31, j = blockIdx.x * kSturmWarps + (threadIdx.x >> 5);
  if (j >= r) return;
  const int below = N - 1 - j;                   // eigenvalues smaller than the j-th largest
  double lo = -1.001 * b - 1e-30, hi = 1.001 * b + 1e-30;
  for (int round = 0; round < 16 && hi - lo > 2.3e-16 * b; ++round) {
    const double h = (hi - lo) * (1.0 / 33.0), x = fma(h, (double)(lane + 1), lo);
    const uint32_t mask = __ballot_sync(0xFFFFFFFFu, sturm_count(sturm_smem, N, x) <= below);
    const int n = __popc(mask);                  // the trial points at or below it
    hi = n < 32 ? fma(h, (double)(n + 1), lo) : hi;
    lo = n > 0 ? fma(h, (double)n, lo) : lo;
  }
  if (lane == 0) lamb.p[blockIdx.y][j] = 0.5 * (lo + hi);
}

// Whether binary32 resolved the vectors: A and its reduction carry an error of some units in the last place of the largest
// eigenvalue, and neighbours in the bulk of a gradient's spectrum lie about lambda / N apart.  Below this bound the subspace
// can be off by more than 1e-2 rad (768 rows: lambda_r / lambda_1 = 3e-6 gave 3.5e-2).  `wanted`: of the vectors computed, those the
// caller asked for.
__global__ void resolved_kernel(const Ptrs<const double> lamb, int N, int wanted, int32_t* __restrict__ status) {
  const double* lam = lamb.p[blockIdx.x];
  if (!(lam[wanted - 1] >= 0.1 * N * 0x1p-24 * lam[0]) && status) atomicOr(status, QG_DEV_BAD_FACTOR);
}

// ------------------------------------------------------------------------------------------ 3. eigenvectors of T
// T - lambda = L D+ L^T from the top and U D- U^T from the bottom; where gamma_i = D+_i + D-_i - (d_i - lambda) is smallest
// the two factorisations are joined, and the vector follows outward from that row by products of multipliers alone, without
// cancellation.  Bound: the chain of binary64 divisions, so a pair of threads takes an eigenvalue, one from each end (warp 0
// and warp 1 of a CTA): 768 rows, 256 vectors 320 -> 208 us.
constexpr double kPivotFloor = 1e-280;
__device__ __forceinline__ double guarded(double q) { return fabs(q) < kPivotFloor ? copysign(kPivotFloor, q) : q; }

__global__ void __launch_bounds__(64)
tridiagonal_vectors_kernel(const Ptrs<const float> db, const Ptrs<const float> eb, int N, int t0, int count, int r, const Ptrs<const double> lamb,
                           const Ptrs<double> plusb, const Ptrs<double> minusb, const Ptrs<float> Zb, const Ptrs<double> invb) {
  extern __shared__ double vec_smem[];
  __shared__ double s_best[2][32], s_sum[32];
  __shared__ int s_at[2][32];
  double* d = vec_smem;
  float* e = reinterpret_cast<float*>(vec_smem + N);
  const int mat = blockIdx.y, lane = threadIdx.x & 31, side = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < N; i += 64) {
    d[i] = diagonal(db.p[mat], i);
    e[i] = i + 1 < N ? eb.p[mat][i] : 0.f;
  }
  __syncthreads();
  const int t = blockIdx.x * 32 + lane;             // of the vectors t0 .. t0 + count - 1 (of r), whose pivots have pitch count
  const bool live = t < count;
  const double lam = live ? lamb.p[mat][t0 + t] : 0.0;
  double* plus = plusb.p[mat] + min(t, count - 1);  // D+_i, D-_i
  double* minus = minusb.p[mat] + min(t, count - 1);
  if (live && side == 0) {
    double q = guarded(d[0] - lam);
    plus[0] = q;
#pragma unroll 4
    for (int i = 1; i < N; ++i) {
      const double ei = e[i - 1];
      q = guarded((d[i] - lam) - ei * (ei / q));
      plus[(int64_t)i * count] = q;
    }
  } else if (live) {
    double q = guarded(d[N - 1] - lam);
    minus[(int64_t)(N - 1) * count] = q;
#pragma unroll 4
    for (int i = N - 2; i >= 0; --i) {
      const double ei = e[i];
      q = guarded((d[i] - lam) - ei * (ei / q));
      minus[(int64_t)i * count] = q;
    }
  }
  __syncthreads();
  // the row with the smallest gamma: each thread looks through half of them (loads in batches: they come from L2)
  constexpr int kBatch = 16;
  {
    double best = 1e300;
    int at = 0;
    const int i0 = side * (N / 2), i1 = side ? N : N / 2;
    if (live)
      for (int b = i0; b < i1; b += kBatch) {
        double p[kBatch], m[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
          const int64_t i = min(b + u, N - 1);
          p[u] = plus[i * count];
          m[u] = minus[i * count];
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
          if (b + u >= i1) break;
          const double gamma = fabs(p[u] + (m[u] - (d[b + u] - lam)));
          if (gamma < best) { best = gamma; at = b + u; }
        }
      }
    s_best[side][lane] = best;
    s_at[side][lane] = at;
  }
  __syncthreads();
  const int twist = s_best[1][lane] < s_best[0][lane] ? s_at[1][lane] : s_at[0][lane];
  float* Z = Zb.p[mat] + t0 + min(t, count - 1);
  double z = 1.0, sum = 0.0;
  if (live && side == 0) {                          // z_i = -(e_i / D+_i) z_{i+1} above the twist
    for (int b = twist - 1; b >= 0; b -= kBatch) {
      double l[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) { const int64_t i = max(b - u, 0); l[u] = plus[i * count]; }
#pragma unroll
      for (int u = 0; u < kBatch; ++u) l[u] = (double)e[max(b - u, 0)] / l[u];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        if (b - u < 0) break;
        z *= -l[u];
        sum = fma(z, z, sum);
        Z[(int64_t)(b - u) * r] = (float)z;
      }
    }
    Z[(int64_t)twist * r] = 1.f;
    s_sum[lane] = sum + 1.0;
  } else if (live) {                                // z_i = -(e_{i-1} / D-_i) z_{i-1} below
    for (int b = twist + 1; b < N; b += kBatch) {
      double l[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) { const int64_t i = min(b + u, N - 1); l[u] = minus[i * count]; }
#pragma unroll
      for (int u = 0; u < kBatch; ++u) l[u] = (double)e[min(b + u, N - 1) - 1] / l[u];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        if (b + u >= N) break;
        z *= -l[u];
        sum = fma(z, z, sum);
        Z[(int64_t)(b + u) * r] = (float)z;
      }
    }
  }
  __syncthreads();
  if (live && side == 1) invb.p[mat][t0 + t] = 1.0 / sqrt(s_sum[lane] + sum);
}

// ------------------------------------------------------------------------------------------ 4. X = H Z
// A warp keeps VW vectors in registers (lane: rows 128 c + 4 lane .. + 3) and runs through all Householder vectors, the
// last first; the CTA's warps share them from a ring in shared memory that is filled several pairs ahead.  Bound: the chain of
// dot product and update.  So the reflectors are applied two at a time, with one reduction for both,
//     s_k = v_k . x,  s_{k-1} = v_{k-1} . x - tau_k s_k (v_{k-1} . v_k),  x <- x - tau_k s_k v_k - tau_{k-1} s_{k-1} v_{k-1},
// and few vectors are spread over many CTAs of two warps.
// 768 rows, 256 vectors 605 -> 228 us; 2048 rows, eight times 512 vectors 4180 -> 2665.
constexpr int back_stages(int nch) { return nch <= 16 ? 6 : 4; }   // pairs of reflectors in the ring

// `bytes` (a multiple of 16) consecutive bytes to shared memory by the copy engine.
__device__ __forceinline__ void bulk_load(void* smem_dst, const void* gsrc, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(ptx::smem_u32(smem_dst)), "l"(gsrc),
               "r"(bytes), "r"(ptx::smem_u32(bar))
               : "memory");
}

// cross_k = v_k . v_{k-1} for k = N - 1, N - 3, ... (v_{N-1} counts as zero): a warp each
__global__ void __launch_bounds__(128)
reflector_pairs_kernel(const Ptrs<const float> Vb, int N, int Np, const Ptrs<float> crossb) {
  const int k = N - 1 - 2 * (int)(blockIdx.x * 4 + (threadIdx.x >> 5)), lane = threadIdx.x & 31;
  if (k < 1) return;
  const float* v = Vb.p[blockIdx.y] + (int64_t)k * Np;
  float s = 0.f;
  if (k < N - 1)
    for (int i = (k + 1) / 4 * 4 + 4 * lane; i < Np; i += 128) {
      const float4 x = *reinterpret_cast<const float4*>(v + i), y = *reinterpret_cast<const float4*>(v - Np + i);
      s = fmaf(x.x, y.x, fmaf(x.y, y.y, fmaf(x.z, y.z, fmaf(x.w, y.w, s))));
    }
  s = warp_sum(s);
  if (lane == 0) crossb.p[blockIdx.y][k] = s;
}

template <int NCH, int VW, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, 1)
back_transform_kernel(const Ptrs<const float> Vb, const Ptrs<const float> taub, const Ptrs<const float> crossb, int N, int Np, int r,
                      const Ptrs<float> Zb, const Ptrs<const double> invb, int32_t* __restrict__ status) {
  extern __shared__ __align__(16) float back_smem[];
  constexpr int kBackStages = back_stages(NCH);
  __shared__ __align__(8) uint64_t landed[kBackStages];
  constexpr int kW = WARPS * VW, kThreads = WARPS * 32;   // vectors and threads of this CTA
  // chunks are taken in groups, so that their loads overlap; a group that begins above the reflector's first row meets zeros
  constexpr int kGrp = NCH % 4 == 0 ? 4 : 3, kPitch = NCH * 128;
  float* ring = back_smem;                          // [kBackStages][2][kPitch]
  float* tile = ring + 2 * kBackStages * kPitch;    // [128][kW + 1]
  float* taus = tile + 128 * (kW + 1);              // [N]
  float* cross = taus + N;                          // [N]
  const int mat = blockIdx.y, t0 = blockIdx.x * kW;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const float* V = Vb.p[mat];
  float* Z = Zb.p[mat];
  const int chunks = Np / 128;
  for (int i = tid; i < N; i += kThreads) {
    taus[i] = i + 1 < N ? taub.p[mat][i] : 0.f;
    cross[i] = crossb.p[mat][i];
  }

  for (int i = tid; i < 2 * kBackStages * kPitch; i += kThreads) ring[i] = 0.f;   // what lies past Np stays zero
  if (tid == 0) {
    for (int i = 0; i < kBackStages; ++i) ptx::mbar_init(&landed[i], 1);
    ptx::fence_mbar_init();
  }
  ptx::fence_proxy_async_smem();                    // these stores come before the copies that go over most of the ring
  auto fetch = [&](int step) {                      // one thread: reflectors k = N - 1 - 2 step and k - 1, rows k .. on in whole groups
    const int k = N - 1 - 2 * step;
    if (tid != 0 || k < 0) return;
    uint64_t* bar = &landed[step % kBackStages];
    float* dst = ring + (step % kBackStages) * 2 * kPitch;
    const float* src = V + (int64_t)k * Np;
    const int i = k / (128 * kGrp) * (128 * kGrp);
    const uint32_t bytes = (uint32_t)(Np - i) * 4u;
    ptx::fence_proxy_async_smem();
    ptx::mbar_arrive_expect_tx(bar, k > 0 ? 2 * bytes : bytes);
    bulk_load(dst + i, src + i, bytes, bar);
    if (k > 0) bulk_load(dst + kPitch + i, src - Np + i, bytes, bar);
  };
  __syncthreads();
  for (int s = 0; s < kBackStages - 1; ++s) fetch(s);

  float inv[VW];
#pragma unroll
  for (int u = 0; u < VW; ++u) { const int t = t0 + warp * VW + u; inv[u] = t < r ? (float)invb.p[mat][t] : 0.f; }
  float4 x[VW][NCH];
#pragma unroll
  for (int ch = 0; ch < NCH; ++ch) {
    if (ch < chunks) {
      __syncthreads();
      for (int i = tid; i < 128 * kW; i += kThreads) {
        const int row = i / kW, col = i % kW;
        tile[row * (kW + 1) + col] = (ch * 128 + row < N && t0 + col < r) ? Z[(int64_t)(ch * 128 + row) * r + t0 + col] : 0.f;
      }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < VW; ++u) {
        const float* p = tile + lane * 4 * (kW + 1) + warp * VW + u;
        x[u][ch] = make_float4(p[0] * inv[u], p[kW + 1] * inv[u], p[2 * (kW + 1)] * inv[u], p[3 * (kW + 1)] * inv[u]);
      }
    } else {
#pragma unroll
      for (int u = 0; u < VW; ++u) x[u][ch] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  int step = 0;
  for (int k = N - 1; k >= 0; k -= 2, ++step) {
    __syncthreads();                                // everybody is done with the slot refilled now
    fetch(step + kBackStages - 1);
    if (!ptx::mbar_wait(&landed[step % kBackStages], (step / kBackStages) & 1)) {   // (the copies in flight end by themselves)
      if (status) atomicOr(status, QG_DEV_WAIT_EXPIRED);
    }
    const float* va = ring + (step % kBackStages) * 2 * kPitch + lane * 4;   // v_k (tau = 0 stands for v_{N-1}), v_{k-1}
    const float* vb = va + kPitch;
    const bool two = k > 0;
    const int g0 = k / (128 * kGrp);
    const float ta = taus[k], tb = two ? taus[k - 1] : 0.f, cr = two ? cross[k] : 0.f;
    float sa[VW], sb[VW];
#pragma unroll
    for (int u = 0; u < VW; ++u) sa[u] = sb[u] = 0.f;
#pragma unroll
    for (int g = 0; g < NCH / kGrp; ++g) {
      if (g < g0) continue;
      float4 a4[kGrp], b4[kGrp];
#pragma unroll
      for (int c = 0; c < kGrp; ++c) {
        a4[c] = *reinterpret_cast<const float4*>(va + (g * kGrp + c) * 128);
        b4[c] = two ? *reinterpret_cast<const float4*>(vb + (g * kGrp + c) * 128) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int c = 0; c < kGrp; ++c) {
        const int ch = g * kGrp + c;
#pragma unroll
        for (int u = 0; u < VW; ++u) {
          sa[u] = fmaf(a4[c].x, x[u][ch].x, fmaf(a4[c].y, x[u][ch].y, fmaf(a4[c].z, x[u][ch].z, fmaf(a4[c].w, x[u][ch].w, sa[u]))));
          sb[u] = fmaf(b4[c].x, x[u][ch].x, fmaf(b4[c].y, x[u][ch].y, fmaf(b4[c].z, x[u][ch].z, fmaf(b4[c].w, x[u][ch].w, sb[u]))));
        }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int u = 0; u < VW; ++u) {
        sa[u] += __shfl_xor_sync(0xFFFFFFFFu, sa[u], o);
        sb[u] += __shfl_xor_sync(0xFFFFFFFFu, sb[u], o);
      }
#pragma unroll
    for (int u = 0; u < VW; ++u) {
      sa[u] *= -ta;
      sb[u] = -tb * fmaf(cr, sa[u], sb[u]);
    }
#pragma unroll
    for (int g = 0; g < NCH / kGrp; ++g) {
      if (g < g0) continue;
      float4 a4[kGrp], b4[kGrp];
#pragma unroll
      for (int c = 0; c < kGrp; ++c) {
        a4[c] = *reinterpret_cast<const float4*>(va + (g * kGrp + c) * 128);
        b4[c] = two ? *reinterpret_cast<const float4*>(vb + (g * kGrp + c) * 128) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int c = 0; c < kGrp; ++c) {
        const int ch = g * kGrp + c;
#pragma unroll
        for (int u = 0; u < VW; ++u) {
          x[u][ch].x = fmaf(sa[u], a4[c].x, fmaf(sb[u], b4[c].x, x[u][ch].x));
          x[u][ch].y = fmaf(sa[u], a4[c].y, fmaf(sb[u], b4[c].y, x[u][ch].y));
          x[u][ch].z = fmaf(sa[u], a4[c].z, fmaf(sb[u], b4[c].z, x[u][ch].z));
          x[u][ch].w = fmaf(sa[u], a4[c].w, fmaf(sb[u], b4[c].w, x[u][ch].w));
        }
      }
    }
  }
#pragma unroll
  for (int ch = 0; ch < NCH; ++ch) {
    if (ch < chunks) {
      __syncthreads();
#pragma unroll
      for (int u = 0; u < VW; ++u) {
        float* p = tile + lane * 4 * (kW + 1) + warp * VW + u;
        p[0] = x[u][ch].x; p[kW + 1] = x[u][ch].y; p[2 * (kW + 1)] = x[u][ch].z; p[3 * (kW + 1)] = x[u][ch].w;
      }
      __syncthreads();
      for (int i = tid; i < 128 * kW; i += kThreads) {
        const int row = i / kW, col = i % kW;
        if (ch * 128 + row < N && t0 + col < r) Z[(int64_t)(ch * 128 + row) * r + t0 + col] = tile[row * (kW + 1) + col];
      }
    }
  }
}

// ------------------------------------------------------------------------------------------ host side
constexpr int kDevices = 64;
std::mutex g_coop_mutex;
cudaEvent_t g_coop_done[kDevices] = {};        // completion of the last cooperative launch, per device ordinal

// Opts a kernel instance into its dynamic shared memory, once per device and instance.
template <class K>
int opt_in(K kernel, int bytes, bool* done) {
  int dev = 0;
  QG_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kDevices) return QG_UNSUPPORTED_SHAPE;
  if (done[dev]) return QG_OK;
  QG_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  done[dev] = true;
  return QG_OK;
}

template <int NQ, int THREADS, int RC>
int launch_tridiagonal(TriArgs a, int nb, int32_t* status, cudaStream_t st) {
  static bool done[kDevices] = {};
  auto kern = tridiagonal_kernel<NQ, THREADS, RC>;
  const int rc = opt_in(kern, kTriSmem, done);
  if (rc != QG_OK) return rc;
  void* args[] = {&a, &status};
  return launch_cooperative((const void*)kern, (unsigned)(a.C * nb), THREADS, args, (size_t)kTriSmem, st);
}

template <int NCH, int VW, int WARPS>
int launch_back(const Ptrs<const float>& V, const Ptrs<const float>& tau, const Ptrs<const float>& cross, int nb, int64_t N, int64_t Np, int64_t r, const Ptrs<float>& Z,
                const Ptrs<const double>& inv, int32_t* status, cudaStream_t st) {
  constexpr int kBackStages = back_stages(NCH);
  static bool done[kDevices] = {};
  auto kern = back_transform_kernel<NCH, VW, WARPS>;
  const int rc = opt_in(kern, ((2 * kBackStages + 2) * NCH * 128 + 128 * (WARPS * VW + 1)) * 4, done);
  if (rc != QG_OK) return rc;
  const size_t smem = (size_t)(2 * kBackStages * NCH * 128 + 128 * (WARPS * VW + 1) + 2 * N) * 4;
  kern<<<dim3((unsigned)ceil_div(r, WARPS * VW), (unsigned)nb), WARPS * 32, smem, st>>>(V, tau, cross, (int)N, (int)Np, (int)r, Z, inv, status);
  QG_LAUNCH_CHECK();
  return QG_OK;
}

}  // namespace

int launch_cooperative(const void* kern, unsigned grid, unsigned block, void** args, size_t smem, cudaStream_t st) {
  std::lock_guard<std::mutex> lock(g_coop_mutex);
  int dev = 0;
  QG_CUDA_TRY(cudaGetDevice(&dev));
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  QG_CUDA_TRY(cudaStreamIsCapturing(st, &cap));
  const bool chain = cap == cudaStreamCaptureStatusNone && dev >= 0 && dev < kDevices;
  if (chain) {
    if (!g_coop_done[dev]) QG_CUDA_TRY(cudaEventCreateWithFlags(&g_coop_done[dev], cudaEventDisableTiming));
    else QG_CUDA_TRY(cudaStreamWaitEvent(st, g_coop_done[dev], 0));
  }
  QG_CUDA_TRY(cudaLaunchCooperativeKernel(kern, dim3(grid), dim3(block), args, smem, st));
  count_launch();
  if (chain) QG_CUDA_TRY(cudaEventRecord(g_coop_done[dev], st));
  return QG_OK;
}

// The vectors of a launch of step 3: as many as have their D+ where A was; half of that for large matrices, whose scratch matters
// (a refresh asks for a quarter of the vectors there are as a rule, so that either is one launch).
static int64_t vectors_at_once(int64_t N, int64_t r) { return std::min(r, eig_pitch(N) / (N <= 2048 ? 2 : 4)); }

size_t carve_eig(void* base, int64_t N, int64_t r, EigBuffers* out) {
  size_t off = 0;
  auto take = [&](size_t bytes) { void* p = base ? (char*)base + off : nullptr; off += (size_t)round_up((int64_t)bytes, 256); return p; };
  const int64_t Np = eig_pitch(N);
  EigBuffers w{};
  w.A = (float*)take((size_t)(N * Np * 4));
  w.V = (float*)take((size_t)(N * Np * 4));
  w.tau = (float*)take((size_t)(N * 4));
  w.d = (float*)take((size_t)(N * 4));
  w.e = (float*)take((size_t)(N * 4));
  w.cross = (float*)take((size_t)(N * 4));
  w.scale = (float*)take(4);
  w.lam = (double*)take((size_t)(r * 8));
  w.inv = (double*)take((size_t)(r * 8));
  w.minus = (double*)take((size_t)(N * vectors_at_once(N, r) * 8));
  w.plus = (double*)w.A;                            // done with when the pivots come
  w.Z = (float*)take((size_t)(N * r * 4));
  w.xchg = (uint4*)take((size_t)(2 * Np * 16));
  if (out) *out = w;
  return off;
}

int launch_sym_eig(const EigBuffers* w, int nb, int64_t N, int64_t r, int64_t wanted, int32_t* status, cudaStream_t st) {
  if (N < 2 || N > kEigMax || r < 1 || r > N || wanted < 1 || wanted > r || nb < 1 || nb > kMaxBatch) return QG_UNSUPPORTED_SHAPE;
  const int64_t Np = eig_pitch(N);
  Ptrs<float> A{}, V{}, tau{}, d{}, e{}, Z{}, scale{}, cross{};
  Ptrs<const float> Ac{}, Vc{}, tauc{}, dc{}, ec{}, scalec{}, crossc{};
  Ptrs<double> lam{}, inv{}, plus{}, minus{};
  Ptrs<const double> lamc{}, invc{};
  Ptrs<Tagged> xchg{};
  for (int i = 0; i < nb; ++i) {
    Ac.p[i] = A.p[i] = w[i].A; Vc.p[i] = V.p[i] = w[i].V; tauc.p[i] = tau.p[i] = w[i].tau;
    dc.p[i] = d.p[i] = w[i].d; ec.p[i] = e.p[i] = w[i].e; Z.p[i] = w[i].Z; scalec.p[i] = scale.p[i] = w[i].scale; crossc.p[i] = cross.p[i] = w[i].cross;
    lamc.p[i] = lam.p[i] = w[i].lam; invc.p[i] = inv.p[i] = w[i].inv; plus.p[i] = w[i].plus; minus.p[i] = w[i].minus; xchg.p[i] = (Tagged*)w[i].xchg;
    QG_CUDA_TRY(cudaMemsetAsync(w[i].xchg, 0, (size_t)(2 * Np * 16), st));   // no tag of an earlier call
  }
  eig_scale_factor_kernel<<<nb, 256, 0, st>>>(Ac, (int)N, (int)Np, scale);
  QG_LAUNCH_CHECK();
  eig_scale_kernel<<<dim3((unsigned)N, (unsigned)nb), 256, 0, st>>>(A, (int)N, (int)Np, scalec, V);
  QG_LAUNCH_CHECK();

  // Matrices reduced together share the SMs; as many as stay (all but a fifth of their columns, the first to retire) in
  // registers and shared memory.
  const int sms = sm_count();
  // Threads: as few rows without a column's element as may be, every warp repeats the step's scalars and reductions (768 rows:
  // 3.0 ms with 512 threads, 2.8 with 384).  Columns in registers: the loop should stay in the instruction cache, so only 16
  // where a CTA has no more (768 rows 2.9 -> 2.7 ms against 40).
  using Launch = int (*)(TriArgs, int, int32_t*, cudaStream_t);
  struct Shape { int threads, columns; Launch few, many; };                // columns in registers: 16 if that is all, or `columns`
  const Shape f = Np <= 256    ? Shape{256, 32, launch_tridiagonal<1, 256, 16>, launch_tridiagonal<1, 256, 32>}
                  : Np <= 512  ? Shape{256, 32, launch_tridiagonal<2, 256, 16>, launch_tridiagonal<2, 256, 32>}
                  : Np <= 768  ? Shape{384, 32, launch_tridiagonal<2, 384, 16>, launch_tridiagonal<2, 384, 32>}
                  : Np <= 1024 ? Shape{512, 32, launch_tridiagonal<2, 512, 16>, launch_tridiagonal<2, 512, 32>}
                  : Np <= 1536 ? Shape{384, 16, launch_tridiagonal<4, 384, 16>, launch_tridiagonal<4, 384, 16>}
                  : Np <= 2048 ? Shape{512, 16, launch_tridiagonal<4, 512, 16>, launch_tridiagonal<4, 512, 16>}
                  : Np <= 3072 ? Shape{384, 8, launch_tridiagonal<8, 384, 8>, launch_tridiagonal<8, 384, 8>}
                               : Shape{512, 8, launch_tridiagonal<8, 512, 8>, launch_tridiagonal<8, 512, 8>};
  // (a matrix alone: 128 CTAs are faster than 148 although more of its columns spill, 4096 rows 64 -> 57 ms, 2500 25 -> 22)
  auto ctas = [&](int cnt) { return std::max<int64_t>(1, std::min<int64_t>(cnt == 1 ? std::min(sms, 128) : sms / cnt, ceil_div(N, 16))); };
  auto in_smem = [&](int64_t C) { return std::max<int64_t>(0, (kTriSmem / 4 - (6 + f.threads / 16) * (ceil_div(N, C) + 8)) / Np) & ~3ll; };
  int together = nb;
  while (together > 1 && ctas(together) * (f.columns + in_smem(ctas(together))) * 5 < N * 4) --together;
  for (int first = 0; first < nb; first += together) {
    const int cnt = std::min(together, nb - first);
    TriArgs a{};
    for (int i = 0; i < cnt; ++i) {
      a.A.p[i] = A.p[first + i]; a.V.p[i] = V.p[first + i]; a.tau.p[i] = tau.p[first + i];
      a.d.p[i] = d.p[first + i]; a.e.p[i] = e.p[first + i]; a.xchg.p[i] = xchg.p[first + i];
    }
    a.N = (int)N; a.Np = (int)Np;
    a.C = (int)ctas(cnt);
    a.in_smem = (int)in_smem(a.C);
    const int rc = (ceil_div(N, a.C) <= 16 ? f.few : f.many)(a, cnt, status, st);
    if (rc != QG_OK) return rc;
  }
  {
    static bool done[kDevices] = {};
    const int rc = opt_in(eigenvalue_kernel, (int)kEigMax * 16, done);
    if (rc != QG_OK) return rc;
    eigenvalue_kernel<<<dim3((unsigned)ceil_div(r, kSturmWarps), (unsigned)nb), kSturmWarps * 32, (size_t)N * 16, st>>>(dc, ec, (int)N, (int)r, lam);
    QG_LAUNCH_CHECK();
  }
  resolved_kernel<<<nb, 1, 0, st>>>(lamc, (int)N, (int)wanted, status);
  QG_LAUNCH_CHECK();
  {
    static bool done[kDevices] = {};
    const int rc = opt_in(tridiagonal_vectors_kernel, (int)kEigMax * 12, done);
    if (rc != QG_OK) return rc;
  }
  const int64_t at_once = vectors_at_once(N, r);
  for (int64_t t0 = 0; t0 < r; t0 += at_once) {
    const int64_t count = std::min(at_once, r - t0);
    tridiagonal_vectors_kernel<<<dim3((unsigned)ceil_div(count, 32), (unsigned)nb), 64, (size_t)N * 12, st>>>(dc, ec, (int)N, (int)t0, (int)count, (int)r, lamc, plus, minus,
                                                                                                             Z, inv);
    QG_LAUNCH_CHECK();
  }
  reflector_pairs_kernel<<<dim3((unsigned)ceil_div(N, 8), (unsigned)nb), 128, 0, st>>>(Vc, (int)N, (int)Np, cross);
  QG_LAUNCH_CHECK();
  const bool few = nb * r <= 4 * sms;                // a CTA of two warps per SM
  if (Np <= 512) return few ? launch_back<4, 1, 2>(Vc, tauc, crossc, nb, N, Np, r, Z, invc, status, st) : launch_back<4, 2, 8>(Vc, tauc, crossc, nb, N, Np, r, Z, invc, status, st);
  if (Np <= 768) return few ? launch_back<6, 1, 2>(Vc, tauc, crossc, nb, N, Np, r, Z, invc, status, st) : launch_back<6, 2, 8>(Vc, tauc, crossc, nb, N, Np, r, Z, invc, status, st);
  if (Np <= 1024) return few ? launch_back<8, 1, 2>(Vc, tauc, crossc, nb, N, Np, r, Z, invc, status, st) : launch_back<8, 2, 8>(Vc, tauc, crossc, nb, N, Np, r, Z, invc, status, st);
  if (Np <= 2048) return few ? launch_back<16, 1, 4>(Vc, tauc, crossc, nb, N, Np, r, Z, invc, status, st) : launch_back<16, 2, 8>(Vc, tauc, crossc, nb, N, Np, r, Z, invc, status, st);
  return launch_back<32, 1, 8>(Vc, tauc, crossc, nb, N, Np, r, Z, invc, status, st);
}

}  // namespace qg
