// Sketch-and-precondition least squares: LSQR (Paige and Saunders, ACM TOMS 1982) on A with the
// right preconditioner R^{-1}, where S A = Q R is the FP64 QR of the sketch from sk_solve (paper
// Sec. 5.1 forms S A and its QR; the discussion names sketch-and-precondition as the use of that R
// as a preconditioner). The preconditioned operator M = A R^{-1} has singular values within the
// sketch's distortion of 1, so LSQR needs few iterations, and it converges to the least-squares
// solution of A itself: the rounding rule of the sketch only changes the preconditioner.
//
// Everything of an iteration runs on the GPU, in two launches. The products with A run on the FP32
// pipe with about twice FP32 precision (exact products and compensated sums, df_acc2); the step and
// the recurrence are FP64:
//   lsqr_pass_kernel  u <- A p - c u, ||u||^2 and z <- A^T u in ONE pass over A: the entry u_i needs
//                     only row i of A, and so does its contribution to z, so a row is read once
//   lsqr_step_kernel  the n-vector part: v = R^{-T} z / beta - beta v, alpha, the plane rotation,
//                     y and w updates, p = R^{-1} v        (one cluster of 8 CTAs; n <= 512)
// The step applies R^{-1} as an explicit triangular matrix, formed once per solve
// (lsqr_invert_kernel): a triangular solve is a chain of n dependent steps with a CTA barrier in each
// (451 us a step at n = 128), two matrix-vector products are n^2/2 independent FMAs each. LSQR then
// runs on A W, W = fl(R^{-1}), and x = x0 + W y, so W's rounding only perturbs the preconditioner.
// u is kept unnormalized (its scale is folded into the next step), the iterate is x = x0 + W y with
// x0 the sketch-and-solve solution.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "sk_device.cuh"
#include "sk_internal.h"

namespace sk {

namespace {

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Products of A's FP32 entries with an FP64 vector y = yh + yl (two floats) accumulated in about
// twice FP32 precision on the FP32 pipe: the product a * yh is split exactly into p + e (FMA), the
// running sum takes p through TwoSum (Knuth), and the error terms e + a * yl and the TwoSum errors are
// summed in a second float (cascaded summation, Ogita, Rump and Oishi, SIAM J. Sci. Comput. 2005).
// Explicit round-to-nearest intrinsics keep the compiler from fusing the error-free steps. Two columns
// at a time, with packed FP32 operations (each half is rounded as the scalar operation is; x - y is
// fma(y, -1, x)): half the instructions of the scalar form, the same arithmetic.
__device__ __forceinline__ void df_acc2(float2 a, float2 yh, float2 yl, float2& s, float2& c) {
  const float2 m1 = make_float2(-1.f, -1.f);
  const float2 p = __fmul2_rn(a, yh);
  const float2 e = __ffma2_rn(a, yh, __fmul2_rn(p, m1));
  const float2 t = __fadd2_rn(s, p);
  const float2 bb = __ffma2_rn(s, m1, t);
  const float2 s1 = __ffma2_rn(__ffma2_rn(bb, m1, t), m1, s);
  const float2 err = __fadd2_rn(s1, __ffma2_rn(bb, m1, p));
  s = t;
  c = __fadd2_rn(c, __fadd2_rn(err, __ffma2_rn(a, yl, e)));
}

__device__ __forceinline__ void split_df(double x, float& hi, float& lo) {
  hi = __double2float_rn(x);
  lo = __double2float_rn(x - (double)hi);
}

// (s, c) += (s2, c2) of float pairs whose second parts are small: TwoSum of the leading parts.
__device__ __forceinline__ void df_add(float& s, float& c, float s2, float c2) {
  const float t = __fadd_rn(s, s2);
  const float bb = __fsub_rn(t, s);
  const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(s2, bb));
  s = t;
  c = __fadd_rn(__fadd_rn(c, c2), err);
}

// c = (hi + lo) * scale with hi of magnitude 1/2 to 1 and scale a power of two (2^-120 to 2^120): lo keeps its
// bits whatever c's exponent, where the second float of c itself would be subnormal from about 1e-31 down.
__device__ __forceinline__ void split_scaled(double c, float& hi, float& lo, float& scale) {
  // (exponent and power of two by their bits: frexp and ldexp cost a pass 2 us of FP64 operations)
  const int e = (int)(((unsigned)__double2hiint(c) >> 20) & 0x7FFu) - 1022;
  const int es = max(-120, min(120, e));
  split_df(c * __hiloint2double((1023 - es) << 20, 0), hi, lo);
  scale = __uint_as_float((uint32_t)(es + 127) << 23);
}

constexpr int kPassThreads = 256;
constexpr int kPassCols = 16;  // columns per lane
constexpr int kPassDepth = 4;  // row groups in flight per warp, one of them being used

// One slot of the pass's ring: every thread copies its own part of a row (and the row's u or b) into its
// own places and reads them back, so the ring needs no barrier.
struct PassStage {
  float4 a[kPassCols / 4][kPassThreads];
  float uh[kPassThreads], ul[kPassThreads];
};

// Asynchronous copies of 16 and 4 bytes into shared memory; zeros if !ok (nothing is read then).
__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(ok ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(ok ? 4 : 0)
               : "memory");
}

// One pass over A: u_i <- A_i . p + c u_i with c = sc[kLsqrC] (or b_i - A_i . p when `b` is given),
// sc[kLsqrBeta2] += sum of u_i^2, z += A^T u (z zero before the launch). LPR lanes share a row, 16
// columns each (16 LPR >= n), 32 / LPR rows per warp at a time; the row stays in registers between
// its dot product and its contribution to z. p is in shared memory as (hi, lo) floats; u is kept as
// (hi, lo) floats (uh = first m, ul = next m floats of the u buffer).
//
// Bounds: the bytes of A (once) and, close behind, the FP32 pipe: df_acc2 is 12 operations, twice
// per pair of elements. The partial dot products are combined over the LPR lanes and c u is added in float pairs:
// on this GPU an FP64 operation takes a warp 16 cycles of the SM's FP64 pipe, and here it would be
// repeated by the LPR lanes of a row. That is no less exact than a lane's row-long float-pair sum followed by an
// FP64 combination: x off by 1.3e-16 at 2^18 x 128 (7.6e-16 with the latter), 5.8e-16 at 65536 x 512 (1.2e-14),
// 1.3e-13 at 2^18 x 100 with column scales from 1 to 1e-3 (2.4e-13). Rows arrive through a per-thread cp.async ring: with the next row
// prefetched into registers only, 336 us, the loads' latency exposed. The FP64 sum of u^2 takes one lane per row: the lanes of a row
// keep the u of LPR successive rows, then all 32 add theirs. Measured on GB300 at 2^21 x 128: 303 us
// against 327 us (A p) + 295 us (A^T u) in two passes.
template <int LPR, bool VEC>
__global__ void __launch_bounds__(kPassThreads, 2) lsqr_pass_kernel(const LsqrLaunch L, const float* b) {
  constexpr int kCols = kPassCols * LPR;  // padded columns
  constexpr int kRows = 32 / LPR;         // rows per warp and step
  extern __shared__ __align__(16) PassStage ring[];
  __shared__ __align__(16) float ph[kCols], pl[kCols];
  __shared__ double zs[kCols];
  __shared__ double sqs[kPassThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int li = lane & (LPR - 1), rsub = lane / LPR;
  const int64_t n = L.n, m = L.m, lda = L.lda;
  for (int j = tid; j < kCols; j += kPassThreads) {
    float h = 0.f, l = 0.f;
    if (j < n) split_df(L.p[j], h, l);
    ph[j] = h;
    pl[j] = l;
    zs[j] = 0.0;
  }
  __syncthreads();
  float ch = 0.f, cl = 0.f, cscale = 1.f;
  if (!b) split_scaled(L.sc[kLsqrC], ch, cl, cscale);
  float* uh = reinterpret_cast<float*>(L.u);
  float* ul = uh + m;
  // Column of this lane's element q: whole float4 chunks (VEC) or single floats, interleaved over the
  // lanes of the row.
  auto col = [&](int q) { return VEC ? 4 * (li + LPR * (q >> 2)) + (q & 3) : li + LPR * q; };
  // Start the copies of this lane's part of row `row` into its part of a ring slot (zeros past the last
  // row or column); one commit group per call.
  auto fetch = [&](int64_t row, int slot) {
    PassStage& S = ring[slot];
    const bool live = row < m;
    const float* ar = L.A + (live ? row : 0) * lda;
#pragma unroll
    for (int q = 0; q < kPassCols; q += VEC ? 4 : 1) {
      const bool ok = live && col(q) < n;
      if constexpr (VEC) cp_async16(&S.a[q >> 2][tid], ok ? ar + col(q) : L.A, ok);
      else cp_async4(reinterpret_cast<float*>(&S.a[q >> 2][tid]) + (q & 3), ok ? ar + col(q) : L.A, ok);
    }
    cp_async4(&S.uh[tid], live ? (b ? b : uh) + row : L.A, live);
    cp_async4(&S.ul[tid], live && !b ? ul + row : L.A, live && !b);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float2 zh[kPassCols / 2], zl[kPassCols / 2];
#pragma unroll
  for (int q = 0; q < kPassCols / 2; ++q) zh[q] = zl[q] = make_float2(0.f, 0.f);
  double sq = 0.0;
  float kh = 0.f, kl = 0.f;  // the u this lane keeps for the FP64 sum of squares
  int it = 0;
  const int64_t step = (int64_t)gridDim.x * (kPassThreads / 32) * kRows;
  int64_t row = ((int64_t)blockIdx.x * (kPassThreads / 32) + warp) * kRows + rsub;
#pragma unroll
  for (int i = 0; i < kPassDepth - 1; ++i) fetch(row + i * step, i);
  // (the warp's rows start together: the loop runs while its first row exists)
  for (; row - rsub < m; row += step, ++it) {
    // the slot refilled here was read in the previous iteration, by this thread only
    fetch(row + (kPassDepth - 1) * step, (it + kPassDepth - 1) % kPassDepth);
    asm volatile("cp.async.wait_group %0;" ::"n"(kPassDepth - 1) : "memory");
    const PassStage& S = ring[it % kPassDepth];
    float a[kPassCols];
#pragma unroll
    for (int q = 0; q < kPassCols; q += 4) {
      const float4 v = S.a[q >> 2][tid];
      a[q] = v.x;
      a[q + 1] = v.y;
      a[q + 2] = v.z;
      a[q + 3] = v.w;
    }
    const float oh = cscale * S.uh[tid], ol = cscale * S.ul[tid];  // (exact; cscale is 1 where these are b)
    const bool live = row < m;
    float2 s2 = make_float2(0.f, 0.f), c2 = make_float2(0.f, 0.f);
    if constexpr (VEC) {
#pragma unroll
      for (int q = 0; q < kPassCols; q += 4) {
        const float4 h = *reinterpret_cast<const float4*>(ph + col(q));
        const float4 l = *reinterpret_cast<const float4*>(pl + col(q));
        df_acc2(make_float2(a[q], a[q + 1]), make_float2(h.x, h.y), make_float2(l.x, l.y), s2, c2);
        df_acc2(make_float2(a[q + 2], a[q + 3]), make_float2(h.z, h.w), make_float2(l.z, l.w), s2, c2);
      }
    } else {
#pragma unroll
      for (int q = 0; q < kPassCols; q += 2)
        df_acc2(make_float2(a[q], a[q + 1]), make_float2(ph[col(q)], ph[col(q + 1)]),
                make_float2(pl[col(q)], pl[col(q + 1)]), s2, c2);
    }
    float s = s2.x, c = c2.x;
    df_add(s, c, s2.y, c2.y);
#pragma unroll
    for (int o = LPR / 2; o > 0; o >>= 1) {
      const float so = __shfl_xor_sync(0xffffffffu, s, o), co = __shfl_xor_sync(0xffffffffu, c, o);
      df_add(s, c, so, co);
    }
    if (b) {
      s = -s;
      c = -c;
      df_add(s, c, oh, 0.f);
    } else {
      const float t = __fmul_rn(ch, oh);
      const float e = __fmaf_rn(ch, ol, __fmaf_rn(cl, oh, __fmaf_rn(ch, oh, -t)));
      df_add(s, c, t, e);
    }
    const float h = __fadd_rn(s, c);
    const float l = __fsub_rn(c, __fsub_rn(h, s));
    if (live && li == 0) {
      uh[row] = h;
      ul[row] = l;
    }
#pragma unroll
    for (int q = 0; q < kPassCols / 2; ++q)
      df_acc2(make_float2(a[2 * q], a[2 * q + 1]), make_float2(h, h), make_float2(l, l), zh[q], zl[q]);
    if ((it & (LPR - 1)) == li) {
      kh = live ? h : 0.f;
      kl = live ? l : 0.f;
    }
    if ((it & (LPR - 1)) == LPR - 1) {
      const double u = (double)kh + (double)kl;
      sq = fma(u, u, sq);
      kh = kl = 0.f;
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  {
    const double u = (double)kh + (double)kl;
    sq = fma(u, u, sq);
  }
  sq = warp_sum_d(sq);
  if (lane == 0) sqs[warp] = sq;
#pragma unroll
  for (int q = 0; q < kPassCols; ++q) {
    const float2 z2 = zh[q / 2], l2 = zl[q / 2];
    double t = (q & 1) ? (double)z2.y + (double)l2.y : (double)z2.x + (double)l2.x;
#pragma unroll
    for (int o = LPR; o < 32; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (rsub == 0 && t != 0.0) atomicAdd(zs + col(q), t);
  }
  __syncthreads();
  for (int j = threadIdx.x; j < n; j += kPassThreads)
    if (zs[j] != 0.0) atomicAdd(L.z + j, zs[j]);
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kPassThreads / 32; ++w) t += sqs[w];
    if (t != 0.0) atomicAdd(L.sc + kLsqrBeta2, t);
  }
}

// W = R^{-1}, one warp per row i of W: w R = e_i, solved from column i on. The row stays in registers
// (lane l holds columns l, l + 32, ...: NB of them); column l's value is final when it is broadcast,
// and row l of R then takes it out of the columns to its right. Row l + 1 of R is loaded meanwhile:
// the chain of a step is one shuffle, one product and one FMA. X (n x (n+1) doubles) receives W and its
// transpose side by side: row r holds W^T[r][0..r] in columns 0..r and W[r][r..n-1] in columns
// r+1..n, so both products of the step read rows.
template <int NB>
__global__ void __launch_bounds__(128) lsqr_invert_kernel(const LsqrLaunch L) {
  __shared__ double rinv[kLsqrMaxN];
  const int n = (int)L.n;
  const int64_t ldx = n + 1;
  const int lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < n; i += blockDim.x) rinv[i] = 1.0 / L.R[i * L.ldr + i];
  __syncthreads();
  const int i = blockIdx.x * 4 + (threadIdx.x >> 5);
  if (i >= n) return;
  double acc[NB], nx[NB];
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const int j = lane + 32 * q;
    acc[q] = 0.0;
    nx[q] = (j > i && j < n) ? L.R[i * L.ldr + j] : 0.0;
  }
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    for (int l = max(i, 32 * q); l < min(n, 32 * q + 32); ++l) {
      double r[NB];
#pragma unroll
      for (int t = q; t < NB; ++t) {
        const int j = lane + 32 * t;
        r[t] = nx[t];
        nx[t] = (j > l + 1 && j < n) ? L.R[(l + 1) * L.ldr + j] : 0.0;
      }
      const double w = (l == i ? 1.0 : __shfl_sync(0xffffffffu, acc[q], l & 31)) * rinv[l];
#pragma unroll
      for (int t = q; t < NB; ++t) acc[t] = fma(-w, r[t], acc[t]);
      if (lane == (l & 31)) acc[q] = w;
    }
  }
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const int j = lane + 32 * q;
    if (j < i || j >= n) continue;
    L.X[i * ldx + j + 1] = acc[q];
    L.X[j * ldx + i] = acc[q];
  }
}

constexpr int kStepCtas = 8;  // CTAs of the step's cluster
constexpr int kStepThreads = 256;

__device__ __forceinline__ void cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Sum over the lanes of w[l] x[l], l in [l0, l1): one warp, all lanes get it.
__device__ __forceinline__ double warp_dot(const double* w, const double* x, int l0, int l1, int lane) {
  double t = 0.0;
  for (int l = l0 + lane; l < l1; l += 32) t = fma(__ldg(w + l), x[l], t);
  return warp_sum_d(t);
}

// The n-vector part of an LSQR iteration (first: the initialization from r0 = b - A x0). One cluster;
// row r of the two products with W belongs to CTA r mod 8, a warp per row: spread over 8 SMs the
// 2 n^2/2 FP64 FMAs take 0.5 us (n = 128) to 8 us (n = 512) at 2 per SM and cycle. The CTAs exchange
// q through L.p in global memory, ordered by the cluster barriers.
// Measured on GB300 at n = 128: 14 us a step against 451 us for the two triangular solves on one CTA.
__global__ void __cluster_dims__(kStepCtas, 1, 1) __launch_bounds__(kStepThreads)
    lsqr_step_kernel(const LsqrLaunch L, int first) {
  __shared__ double sh[kLsqrMaxN];
  __shared__ double part[kStepThreads / 32];
  __shared__ double scal[4];  // beta, alpha, phi / rho, -theta / rho
  const int n = (int)L.n;
  const int64_t ldx = n + 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rank = blockIdx.x;
  double* sc = L.sc;
  // (CTA 0 writes the scalars after the last cluster barrier; every CTA reads them before it)
  if (__ldcg(sc + kLsqrDone) != 0.0) return;
  // FP64 division and square root are long sequences on a pipe of 2 lanes per cycle: one thread forms
  // the scalars.
  double beta = 0.0, rho = 1.0, cs = 0.0, sn = 0.0, phibar = 0.0;
  if (threadIdx.x == 0) {
    beta = sqrt(__ldcg(sc + kLsqrBeta2));
    scal[0] = beta;
  }
  __syncthreads();
  // q = W^T (A^T u_stored) / beta = M^T u (u normalized), less beta v
  const double bt = scal[0];
  for (int j = threadIdx.x; j < n; j += kStepThreads) sh[j] = (bt > 0.0) ? __ldcg(L.z + j) / bt : 0.0;
  __syncthreads();
  for (int j = rank + kStepCtas * warp; j < n; j += kStepCtas * (kStepThreads / 32)) {
    double q = warp_dot(L.X + j * ldx, sh, 0, j + 1, lane);
    if (!first) q = fma(-bt, L.v[j], q);
    if (lane == 0) __stcg(L.p + j, q);
  }
  if (threadIdx.x == 0 && !first) {  // the plane rotation, while the other warps finish q
    const double rhobar = sc[kLsqrRhobar];
    phibar = sc[kLsqrPhibar];
    rho = hypot(rhobar, beta);
    cs = rhobar / rho;
    sn = beta / rho;
  }
  cluster_sync();
  // ||q|| (every CTA, in the same order)
  double s = 0.0;
  for (int j = threadIdx.x; j < n; j += kStepThreads) {
    const double q = __ldcg(L.p + j);
    sh[j] = q;
    s = fma(q, q, s);
  }
  s = warp_sum_d(s);
  if (lane == 0) part[warp] = s;
  __syncthreads();
  double alpha = 0.0;
  if (threadIdx.x == 0) {
    for (int w = 0; w < kStepThreads / 32; ++w) alpha += part[w];
    alpha = sqrt(alpha);
    scal[1] = alpha;
    scal[2] = cs * phibar / rho;
    scal[3] = -sn * alpha / rho;
  }
  __syncthreads();
  const double al = scal[1], t1 = scal[2], t2 = scal[3];
  for (int j = threadIdx.x; j < n; j += kStepThreads) {
    const double v = (al > 0.0) ? sh[j] / al : 0.0;
    sh[j] = v;
    if (j % kStepCtas != rank) continue;
    L.v[j] = v;
    if (first) {
      L.w[j] = v;
      L.y[j] = 0.0;
    } else {
      const double wj = L.w[j];
      L.y[j] = fma(t1, wj, L.y[j]);
      L.w[j] = fma(t2, wj, v);
    }
  }
  cluster_sync();  // every CTA has read q and the scalars
  // next A p: p = W v
  for (int i = rank + kStepCtas * warp; i < n; i += kStepCtas * (kStepThreads / 32)) {
    const double p = warp_dot(L.X + i * ldx + 1, sh, i, n, lane);
    if (lane == 0) {
      __stcg(L.p + i, p);
      __stcg(L.z + i, 0.0);
    }
  }
  if (rank != 0 || threadIdx.x != 0) return;
  if (first) {
    sc[kLsqrPhibar] = beta;
    sc[kLsqrRhobar] = alpha;
    sc[kLsqrAnorm2] = alpha * alpha;
    sc[kLsqrBnorm] = beta;
    sc[kLsqrRnorm] = beta;
    sc[kLsqrArnorm] = alpha * beta;
  } else {
    sc[kLsqrRhobar] = -cs * alpha;
    sc[kLsqrPhibar] = sn * phibar;
    sc[kLsqrAnorm2] += alpha * alpha + beta * beta;
    sc[kLsqrRnorm] = sn * phibar;
    sc[kLsqrArnorm] = sn * phibar * alpha * fabs(cs);
    sc[kLsqrIters] += 1.0;
  }
  // the scale of the stored u: u_next = A p - (alpha / beta) u_stored
  sc[kLsqrC] = (beta > 0.0) ? -alpha / beta : 0.0;
  sc[kLsqrAlpha] = alpha;
  sc[kLsqrBeta2] = 0.0;
  if (alpha == 0.0 || beta == 0.0) sc[kLsqrDone] = 1.0;
}

// x = x0 + W y (FP64), one warp per row.
__global__ void __launch_bounds__(256) lsqr_finish_kernel(const LsqrLaunch L) {
  __shared__ double sh[kLsqrMaxN];
  const int n = (int)L.n;
  for (int j = threadIdx.x; j < n; j += blockDim.x) sh[j] = L.y[j];
  __syncthreads();
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= n) return;
  const double t = warp_dot(L.X + (int64_t)i * (n + 1) + 1, sh, i, n, threadIdx.x & 31);
  if ((threadIdx.x & 31) == 0) L.x[i] = L.x0[i] + t;
}

// p = x0 (as the vector the residual kernel multiplies), from the FP32 sketch-and-solve solution.
__global__ void lsqr_start_kernel(const LsqrLaunch L, const float* x0f) {
  for (int64_t j = threadIdx.x; j < L.n; j += blockDim.x) {
    L.x0[j] = (double)x0f[j];
    L.p[j] = (double)x0f[j];
    L.z[j] = 0.0;
  }
  if (threadIdx.x == 0)
    for (int q = 0; q < kLsqrScalars; ++q) L.sc[q] = 0.0;
}

// The fused pass with the fewest lanes per row that cover n columns, two CTAs per SM (its register
// budget), fewer when the rows run out.
template <int LPR>
cudaError_t launch_pass_lpr(const LsqrLaunch& L, const float* b, int sms, cudaStream_t st) {
  const bool vec = (L.n & 3) == 0 && (L.lda & 3) == 0 && (reinterpret_cast<uintptr_t>(L.A) & 15u) == 0;
  const int64_t rows_cta = (kPassThreads / 32) * (32 / LPR);
  const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((L.m + rows_cta - 1) / rows_cta, 2 * (int64_t)sms));
  auto kern = vec ? lsqr_pass_kernel<LPR, true> : lsqr_pass_kernel<LPR, false>;
  const int smem = kPassDepth * (int)sizeof(PassStage);
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  kern<<<grid, kPassThreads, smem, st>>>(L, b);
  return cudaSuccess;
}

cudaError_t launch_pass(const LsqrLaunch& L, const float* b, int sms, cudaStream_t st) {
  if (L.n <= 16) return launch_pass_lpr<1>(L, b, sms, st);
  if (L.n <= 32) return launch_pass_lpr<2>(L, b, sms, st);
  if (L.n <= 64) return launch_pass_lpr<4>(L, b, sms, st);
  if (L.n <= 128) return launch_pass_lpr<8>(L, b, sms, st);
  if (L.n <= 256) return launch_pass_lpr<16>(L, b, sms, st);
  return launch_pass_lpr<32>(L, b, sms, st);
}

void launch_invert(const LsqrLaunch& L, cudaStream_t st) {
  const unsigned grid = (unsigned)((L.n + 3) / 4);
  if (L.n <= 32) lsqr_invert_kernel<1><<<grid, 128, 0, st>>>(L);
  else if (L.n <= 64) lsqr_invert_kernel<2><<<grid, 128, 0, st>>>(L);
  else if (L.n <= 128) lsqr_invert_kernel<4><<<grid, 128, 0, st>>>(L);
  else if (L.n <= 256) lsqr_invert_kernel<8><<<grid, 128, 0, st>>>(L);
  else lsqr_invert_kernel<16><<<grid, 128, 0, st>>>(L);
}

}  // namespace

cudaError_t lsqr_start(const LsqrLaunch& L, const float* b, const float* x0f, int sms, cudaStream_t st,
                       int32_t* launches) {
  lsqr_start_kernel<<<1, 512, 0, st>>>(L, x0f);
  launch_invert(L, st);
  // u = b - A x0, ||u||^2, z = A^T u
  const cudaError_t e = launch_pass(L, b, sms, st);
  if (e != cudaSuccess) return e;
  lsqr_step_kernel<<<kStepCtas, kStepThreads, 0, st>>>(L, 1);
  if (launches) *launches += 4;
  return cudaGetLastError();
}

cudaError_t lsqr_iterate(const LsqrLaunch& L, int sms, cudaStream_t st, int32_t* launches) {
  // u <- A p + c u with c = -alpha / beta, written by the previous step kernel; z = A^T u
  const cudaError_t e = launch_pass(L, nullptr, sms, st);
  if (e != cudaSuccess) return e;
  lsqr_step_kernel<<<kStepCtas, kStepThreads, 0, st>>>(L, 0);
  if (launches) *launches += 2;
  return cudaGetLastError();
}

cudaError_t lsqr_finish(const LsqrLaunch& L, cudaStream_t st, int32_t* launches) {
  lsqr_finish_kernel<<<(unsigned)((L.n + 7) / 8), 256, 0, st>>>(L);
  if (launches) *launches += 1;
  return cudaGetLastError();
}

}  // namespace sk
