// FP64 back end of sketch-and-solve least squares (paper Sec. 5.1: minimize ||SA x - Sb||_2 through
// a reduced QR of SA and a triangular solve). The paper factors in FP32; here the factorization,
// Q^T Sb and the back substitution run in FP64.
//
// One cooperative launch factors W = [SA | Sb] (d x (n+1)) by Householder reflections, NB columns (a
// panel) at a time. The rows are dealt to the CTAs in turn (row r to CTA r mod grid, one CTA per SM at
// most); each CTA keeps its rows of W in shared memory for the whole factorization. A sketch too tall
// for the GPU's shared memory is factored as a tree (TSQR): groups of rows are factored by separate
// launches, their n x (n+1) factors [R_g | c_g] are stacked in FP64 and factored again, until one
// launch holds the whole stack. Dropping each group's last row (its residual norm) only removes a
// constant from ||W x~||, so the minimizer is unchanged.
//
// Why panels. A reflector needs x^T x and x^T W[:, c] over all rows: formed column by column that is
// one grid-wide reduction and barrier per column, and the barrier, the loads behind it and the FP64
// square root and division cost 7 to 11 us a column, several times the arithmetic. A panel needs two
// reductions:
//   1. the Gram matrix of its columns. Reflections keep inner products, so with the Gram matrix and
//      the panel's top NB rows every CTA can run the panel's reflectors through by itself: after
//      reflector i, G_ab loses R_ia R_ib (row i leaves the active rows), and the norms and products of
//      the next column are at hand (panel_factor). Every CTA then applies the reflectors to its own
//      rows of the panel, which leaves the Householder vectors V in their place.
//   2. V^T [W | V] over the trailing columns and the panel itself. With L_ia = tau_a v_i^T v_a (i > a)
//      and U = V diag(tau) L^{-1}, the product of the panel's reflectors takes W to W - U (V^T W).
// The downdated G_ii loses digits if column i nearly depends on the panel's earlier columns: its relative
// error grows by what it was over what is left of it. Where less than kPanelCut is left, the panel ends
// before column i, and the next one starts there from a Gram matrix formed anew: a panel's first column
// is always exact, and the worst case is one column per panel. All CTAs decide alike, from the same sums.
// The cut at 1/16 (four bits of a squared norm, two of R's diagonal) keeps kappa about as near the exact one
// as one reduction per column did: 12 monomials in 128 columns (kappa 1700) 2e-14 off, 2.6e-14 then, 3.6e-12
// with the cut at 1/1024; 64 columns with singular values from 1 to 1e-6 2.8e-12, 8e-13 and 1.4e-11.
// Gaussian columns, and autoregressive ones up to a correlation of 0.96, are not cut; at 0.999 1024 x 64
// takes 301 us, the monomials in 64 columns 368 us, instead of 275 (474 column by column).
// Every grid synchronization waits at most about two seconds: on expiry the kernel sets
// kStatusTimeout in the status word and all CTAs leave at the next check, so a stalled launch cannot
// hang the GPU.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "sk_device.cuh"
#include "sk_internal.h"

namespace sk {

namespace {

// Columns of W = [SA | Sb] the kernel handles (n + 1 <= kQRMaxCols).
constexpr int kQRMaxCols = 1032;
constexpr int kQRThreads = 256;

// A grid barrier gives up after about two seconds of waiting (in SM clock cycles at ~2 GHz).
constexpr long long kBarrierCycles = 4000000000ll;

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Grid synchronization for a co-resident (cooperative) grid with monotonic arrival counters (zero at
// launch and never reset): every CTA's thread 0 adds 1 with release semantics, after a CTA barrier,
// to counter b mod kBarCounters (128 bytes apart), then polls them with acquire loads until their sum
// reaches `target` (= grid size x synchronization number). The CTA's writes before the call are
// visible to every CTA after it. Gives up after `limit` SM clock cycles. Returns false if this CTA, or
// any CTA before it, gave up waiting.
// One counter: spreading the arrivals over 8 counters was measured slower on GB300 (QR at n = 1024,
// d = 2048: 12.7 -> 14.6 ms), the polls of 8 counters costing more than the queued arrivals.
constexpr int kBarCounters = 1;
constexpr int kBarStride = 32;  // unsigned words between counters

__device__ bool grid_arrive_wait(unsigned* bar, unsigned target, unsigned* status, long long limit) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned* mine = bar + (blockIdx.x % kBarCounters) * kBarStride;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(mine) : "memory");
    const long long t0 = clock64();
    unsigned polls = 0;
    while (true) {
      unsigned sum = 0;
#pragma unroll
      for (int q = 0; q < kBarCounters; ++q) sum += ld_acquire_u32(bar + q * kBarStride);
      if (sum >= target) break;
      // the clock is read on the first poll (so that a limit of a few cycles takes effect at once)
      // and every 256 polls after it
      if ((++polls & 255u) == 1u || (polls & 255u) == 0u) {
        if (clock64() - t0 > limit) {
          atomicOr(status, kStatusTimeout);
          break;
        }
        // Another CTA already gave up: stop waiting.
        if (*(volatile unsigned*)status & kStatusTimeout) break;
      }
      if (polls > 512) __nanosleep(32);
    }
    ok = (*(volatile unsigned*)status & kStatusTimeout) == 0;
  }
  __syncthreads();
  return ok != 0;
}

// Columns per panel at most (the kernel's NB: 16, or fewer where the scratch of a narrow sketch holds
// less), and the part of a column's squared norm that has to be left after the panel's earlier columns.
constexpr double kPanelCut = 1.0 / 16.0;

// Scratch of one launch, in doubles: two Gram matrices (NB x NB), the panel's top rows (NB x NB), two
// buffers of reduced products (NB x (n+1)). The pairs alternate between panels, so that one is cleared
// while the other is in use.
constexpr int64_t panel_scratch(int64_t nb, int64_t n) { return 3 * nb * nb + 2 * nb * (n + 1); }

struct QRArgs {
  SolveLaunch L;
  int32_t rpc;     // rows per CTA
  int32_t shares_R;  // 1: the scratch overlaps L.R, which may be written only when all have read it
};

template <typename T>
__device__ __forceinline__ double load_val(const void* p, int64_t idx) {
  if constexpr (std::is_same<T, double>::value) return reinterpret_cast<const double*>(p)[idx];
  else if constexpr (std::is_same<T, __half>::value) return (double)__half2float(reinterpret_cast<const __half*>(p)[idx]);
  else if constexpr (std::is_same<T, __nv_bfloat16>::value)
    return (double)__bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p)[idx]);
  else return (double)reinterpret_cast<const float*>(p)[idx];
}

// One panel's reflectors from its Gram matrix and top rows (one warp; NB <= 16). Lane c < NB holds column
// c of the top rows, lane NB + c column c of the Gram matrix (further lanes repeat those). Writes the
// panel's w_ic = v_i^T W_c (c > i), R's rows, tau_i and v_i's entry on row i, and returns the panel's
// width: `wmax` columns, fewer if one is cut off. (Not inlined: its 16 doubles a lane then take no registers
// from the other phases. 1024 x 64 with 128 registers a thread 279 -> 275 us; 4096 x 1024 11450 -> 11290.)
template <int NB>
__device__ __noinline__ int panel_factor(const double* G, const double* top, int wmax, double* wsm, double* rsm, double* taus,
                            double* v0s) {
  const int lane = threadIdx.x & 31;
  const int c = lane % NB;
  const bool gram = lane >= NB;
  double x[NB];
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const int lo = min(q, c), hi = max(q, c);
    x[q] = (hi >= wmax) ? 0.0 : (gram ? __ldcg(G + lo * NB + hi) : __ldcg(top + q * NB + c));
  }
  const double full = (c < wmax) ? __ldcg(G + c * NB + c) : 0.0;  // norms before the panel's first reflector
  int width = 0;
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    if (width < i || i >= wmax) continue;
    const double norm2 = __shfl_sync(0xffffffffu, x[i], NB + i);
    const double x0 = __shfl_sync(0xffffffffu, x[i], i);
    const double t_ic = __shfl_sync(0xffffffffu, x[i], c);
    const double g_ic = __shfl_sync(0xffffffffu, x[i], NB + c);
    if (i > 0 && !(norm2 > kPanelCut * __shfl_sync(0xffffffffu, full, i))) continue;
    // alpha = -sign(x0) ||x||, v_i = x0 - alpha, tau = 2 / v^T v
    const double alpha = -copysign(sqrt(norm2), x0);
    const double v0 = x0 - alpha;
    const double vtv = (norm2 - x0 * x0) + v0 * v0;
    const double tau = (vtv > 0.0) ? 2.0 / vtv : 0.0;
    const double w = g_ic - alpha * t_ic;
    const double r = t_ic - tau * v0 * w;
    if (lane < NB) {
      wsm[i * NB + c] = w;
      rsm[i * NB + c] = (c == i) ? alpha : r;
    }
    if (lane == 0) {
      taus[i] = tau;
      v0s[i] = v0;
    }
    // top rows: t_qc -= (tau w_c) t_qi; Gram: G_qc -= R_ic R_iq
    const double f = (c > i) ? (gram ? -r : -(tau * w)) : 0.0;
#pragma unroll
    for (int q = i + 1; q < NB; ++q) {
      const double m = __shfl_sync(0xffffffffu, gram ? r : x[q], gram ? NB + q : i);
      if (c > i) x[q] = fma(m, f, x[q]);
    }
    width = i + 1;
  }
  return width;
}

// x = R^{-1} c, kappa and the singularity check (one CTA; rhs: n doubles of shared memory). Blocks of 32
// unknowns from the bottom: one warp solves the block, a row of it per lane, then every thread takes the
// block's unknowns out of the rows above. (Unknown by unknown, two CTA barriers, a division and a load
// in each, this was about a microsecond per unknown.)
__device__ void back_substitute(const SolveLaunch& L, double* rhs) {
  __shared__ double xs[32];
  __shared__ double red[2][kQRThreads / 32];
  const int n = (int)L.n;
  const int64_t ldr = n + 1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double rmax = 0.0, rmin = __longlong_as_double(0x7ff0000000000000ll);
  for (int l = tid; l < n; l += kQRThreads) {
    rhs[l] = __ldcg(L.R + l * ldr + n);
    const double r = fabs(__ldcg(L.R + l * ldr + l));
    rmax = fmax(rmax, r);
    rmin = fmin(rmin, r);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    rmax = fmax(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
    rmin = fmin(rmin, __shfl_xor_sync(0xffffffffu, rmin, o));
  }
  if (lane == 0) {
    red[0][warp] = rmax;
    red[1][warp] = rmin;
  }
  __syncthreads();
  for (int w = 0; w < kQRThreads / 32; ++w) {
    rmax = fmax(rmax, red[0][w]);
    rmin = fmin(rmin, red[1][w]);
  }
  const bool singular = rmin == 0.0;
  for (int b0 = (n - 1) / 32 * 32; b0 >= 0; b0 -= 32) {
    const int nb = min(32, n - b0);
    if (warp == 0) {
      double r[32];
#pragma unroll
      for (int c = 0; c < 32; ++c) r[c] = (c >= lane && c < nb) ? __ldcg(L.R + (b0 + lane) * ldr + b0 + c) : 0.0;
      double diag = 1.0;
#pragma unroll
      for (int c = 0; c < 32; ++c)
        if (c == lane && c < nb) diag = r[c];
      const double inv = (diag != 0.0) ? 1.0 / diag : 0.0;
      double t = (lane < nb) ? rhs[b0 + lane] : 0.0;
#pragma unroll
      for (int c = 31; c >= 0; --c) {
        const double x = __shfl_sync(0xffffffffu, t * inv, c);
        if (c < nb && lane < c) t = fma(-r[c], x, t);
        if (lane == c) t = x;
      }
      xs[lane] = t;
      if (lane < nb) L.x[b0 + lane] = singular ? __int_as_float(0x7fc00000) : (float)t;
    }
    __syncthreads();
    for (int l = tid; l < b0; l += kQRThreads) {
      const double* rr = L.R + l * ldr + b0;
      double t0 = rhs[l], t1 = 0.0;
      for (int c = 0; c + 1 < nb; c += 2) {
        t0 = fma(-rr[c], xs[c], t0);
        t1 = fma(-rr[c + 1], xs[c + 1], t1);
      }
      if (nb & 1) t0 = fma(-rr[nb - 1], xs[nb - 1], t0);
      rhs[l] = t0 + t1;
    }
    __syncthreads();
  }
  if (tid == 0) {
    if (singular) atomicOr(L.status, kStatusNumeric);
    // (fmax and fmin drop NaN: with nothing but NaN on the diagonal rmax is still 0 and rmin infinite)
    const double inf = __longlong_as_double(0x7ff0000000000000ll);
    *L.kappa = (rmin > 0.0 && rmin <= rmax && rmax < inf) ? rmax / rmin : inf;
  }
}

// CTAS: CTAs that an SM's registers are to have room for. A wide sketch takes most of an SM's shared memory per
// CTA, and its CTAs all the registers they can use. A narrow one has to leave room: its cooperative launch
// starts when every CTA has a place, and a CTA with 255 registers a thread has none beside another request's
// kernel. A service's saturated stream of requests (n up to 256; m from 2^14 to 2^24, or to 2^20 rows) then
// makes 363 / 1290 solves a second, with 128 registers 382 / 1550, with 80 390 / 1610 (384 / 1360 with the
// kernel that took one reduction per column and 64 registers). A QR alone: 1024 x 64 275 -> 279 us.
template <typename T, int NB, int CTAS>
__global__ void __launch_bounds__(kQRThreads, CTAS) qr64_kernel(const QRArgs a) {
  const long long wait = a.L.wait_cycles > 0 ? a.L.wait_cycles : kBarrierCycles;
  extern __shared__ __align__(16) double Wl[];  // rpc x (n+1) rows of W (row-major)
  __shared__ double wsm[NB * NB], rsm[NB * NB], lsm[NB * NB], taus[NB], v0s[NB];
  __shared__ int width_sh;
  const SolveLaunch& L = a.L;
  const int n = (int)L.n, ldw = n + 1;
  const int b = blockIdx.x, P = (int)gridDim.x;
  const int tid = threadIdx.x;
  const int nown = (L.d > b) ? (int)((L.d - b + P - 1) / P) : 0;  // local row rl is row b + rl * P
  double* const top = L.part + 2 * NB * NB;
  const int s_size = NB * ldw;
  // Load own rows of [SA | Sb] as FP64.
  for (int64_t e = tid; e < (int64_t)nown * ldw; e += kQRThreads) {
    const int64_t rl = e / ldw, c = e - rl * ldw;
    const int64_t r = b + rl * P;
    Wl[e] = (c < n) ? load_val<T>(L.SA, r * L.lda_sa + c) : load_val<T>(L.Sb, r * L.sb_stride);
  }
  // This thread's entry (pa <= pb) of the Gram matrix, and its share of the rows.
  constexpr int kPairs = NB * (NB + 1) / 2;
  constexpr int kPairGroups = kQRThreads / kPairs;
  int pa = 0, pb = tid % kPairs;
  while (pb >= NB - pa) pb -= NB - pa++;
  pb += pa;
  const int pg = tid / kPairs;
  unsigned syncs = 0;
  int p = 0;
  for (int j = 0; j < n; p ^= 1) {
    __syncthreads();  // W is up to date
    double* const Gm = L.part + p * (NB * NB);                             // this panel's buffers, and
    double* const Sm = top + NB * NB + p * s_size;                         // the next one's
    double* const Gnext = L.part + (p ^ 1) * (NB * NB);
    double* const Snext = top + NB * NB + (p ^ 1) * s_size;
    const int wmax = min(NB, n - j);
    const int rl0 = (j > b) ? (j - b + P - 1) / P : 0;  // first local row with r >= j
    // 1. Gram matrix of the panel's columns over the rows >= j; the owners publish the top rows.
    if (pg < kPairGroups && pb < wmax) {
      double s0 = 0.0, s1 = 0.0;
      int rl = rl0 + pg;
      for (; rl + kPairGroups < nown; rl += 2 * kPairGroups) {
        const double* r0 = Wl + (int64_t)rl * ldw + j;
        const double* r1 = r0 + (int64_t)kPairGroups * ldw;
        s0 = fma(r0[pa], r0[pb], s0);
        s1 = fma(r1[pa], r1[pb], s1);
      }
      if (rl < nown) s0 = fma(Wl[(int64_t)rl * ldw + j + pa], Wl[(int64_t)rl * ldw + j + pb], s0);
      s0 += s1;
      if (s0 != 0.0) atomicAdd(Gm + pa * NB + pb, s0);
    }
    if (tid < NB * NB) {
      const int i = tid / NB, c = tid % NB, r = j + i;
      if (i < wmax && c < wmax && r % P == b) __stcg(top + tid, Wl[(int64_t)(r / P) * ldw + j + c]);
    }
    if (!grid_arrive_wait(L.bar, P * ++syncs, L.status, wait)) return;
    if (tid < 32) {
      const int w = panel_factor<NB>(Gm, top, wmax, wsm, rsm, taus, v0s);
      if (tid == 0) width_sh = w;
    } else {
      // Clear the other pair of buffers for the next panel: all CTAs have read them before this barrier
      // (products) or the one before (Gram matrix), and add to them after the next one.
      if (b == 0 && tid - 32 < NB * NB) __stcg(Gnext + tid - 32, 0.0);
      if (b == 0 && NB * NB > kQRThreads - 32 && tid - 32 + kQRThreads - 32 < NB * NB)
        __stcg(Gnext + tid - 32 + kQRThreads - 32, 0.0);
      for (int x = b * (kQRThreads - 32) + tid - 32; x < NB * ldw; x += P * (kQRThreads - 32)) __stcg(Snext + x, 0.0);
    }
    __syncthreads();
    const int w = width_sh;
    // The reflectors applied to this CTA's rows of the panel; V takes the rows' place.
#pragma unroll 1
    for (int rl = rl0 + tid; rl < nown; rl += kQRThreads) {
      double* wr = Wl + (int64_t)rl * ldw + j;
      const int i0 = b + rl * P - j;  // row i0 of the panel's top rows (none if >= w)
      double x[NB];
#pragma unroll
      for (int q = 0; q < NB; ++q) x[q] = (q < w) ? wr[q] : 0.0;
#pragma unroll
      for (int i = 0; i < NB; ++i) {
        if (i >= w) continue;
        const double v = (i < i0) ? x[i] : (i == i0 ? v0s[i] : 0.0);
        const double f = -(taus[i] * v);
#pragma unroll
        for (int q = i + 1; q < NB; ++q)
          if (q < w) x[q] = fma(f, wsm[i * NB + q], x[q]);
        wr[i] = v;
      }
    }
    __syncthreads();
    // 2. V^T [V | W]: column j + cc, rows dealt to groups of threads when there are few columns.
    {
      const int cols = n + 1 - j;
      const int groups = max(1, kQRThreads / cols);
#pragma unroll 1
      for (int x = tid; x < groups * cols; x += kQRThreads) {
        const int g = x / cols, cc = x - g * cols;
        double s[NB];
#pragma unroll
        for (int i = 0; i < NB; ++i) s[i] = 0.0;
#pragma unroll 2
        for (int rl = rl0 + g; rl < nown; rl += groups) {
          const double* wr = Wl + (int64_t)rl * ldw + j;
          const double wv = wr[cc];
#pragma unroll
          for (int i = 0; i < NB; ++i)
            if (i < w) s[i] = fma(wr[i], wv, s[i]);
        }
        // v_i^T v_cc (i > cc) goes to columns 0..w-1, which no trailing column uses
        double* dst = Sm + (cc < w ? cc : j + cc);
#pragma unroll
        for (int i = 0; i < NB; ++i)
          if (i < w && (cc >= w || i > cc) && s[i] != 0.0) atomicAdd(dst + (int64_t)i * ldw, s[i]);
      }
    }
    if (!grid_arrive_wait(L.bar, P * ++syncs, L.status, wait)) return;
    if (tid < NB * NB) {
      const int i = tid / NB, q = tid % NB;
      lsm[tid] = (q < i && i < w) ? taus[q] * __ldcg(Sm + (int64_t)i * ldw + q) : 0.0;
    }
    __syncthreads();
    // U = V diag(tau) L^{-1}, row by row, in V's place.
#pragma unroll 1
    for (int rl = rl0 + tid; rl < nown; rl += kQRThreads) {
      double* wr = Wl + (int64_t)rl * ldw + j;
      double u[NB];
#pragma unroll
      for (int i = 0; i < NB; ++i) u[i] = (i < w) ? taus[i] * wr[i] : 0.0;
#pragma unroll
      for (int i = NB - 1; i >= 0; --i) {
        if (i >= w) continue;
#pragma unroll
        for (int q = 0; q < i; ++q) u[q] = fma(-u[i], lsm[i * NB + q], u[q]);
        wr[i] = u[i];
      }
    }
    __syncthreads();
    // W -= U (V^T W) on the trailing columns.
    {
      const int cols = n + 1 - j - w;
      const int groups = max(1, kQRThreads / cols);
#pragma unroll 1
      for (int x = tid; x < groups * cols; x += kQRThreads) {
        const int g = x / cols, c = j + w + x - g * cols;
        double s[NB];
#pragma unroll
        for (int i = 0; i < NB; ++i) s[i] = (i < w) ? __ldcg(Sm + (int64_t)i * ldw + c) : 0.0;
#pragma unroll 2
        for (int rl = rl0 + g; rl < nown; rl += groups) {
          double* wr = Wl + (int64_t)rl * ldw;
          double t0 = wr[c], t1 = 0.0;
#pragma unroll
          for (int i = 0; i < NB; i += 2) {
            if (i < w) t0 = fma(-wr[j + i], s[i], t0);
            if (i + 1 < w) t1 = fma(-wr[j + i + 1], s[i + 1], t1);
          }
          wr[c] = t0 + t1;
        }
      }
    }
    __syncthreads();
    // The panel's own part of R's rows, where U was.
    if (tid < NB * NB) {
      const int i = tid / NB, q = tid % NB, r = j + i;
      if (i < w && q >= i && q < w && r % P == b) Wl[(int64_t)(r / P) * ldw + j + q] = rsm[tid];
    }
    j += w;
  }
  __syncthreads();
  // R's rows (zero below the diagonal in a group of a tree level, whose whole output [R | c] is).
  if (a.shares_R && !grid_arrive_wait(L.bar, P * ++syncs, L.status, wait)) return;
  for (int rl = 0; rl < nown && b + rl * P < n; ++rl) {
    const int r = b + rl * P;
    for (int c = tid; c <= n; c += kQRThreads)
      if (c >= r || !L.solve_x) L.R[(int64_t)r * ldw + c] = (c >= r) ? Wl[(int64_t)rl * ldw + c] : 0.0;
  }
  if (!L.solve_x) return;
  if (!grid_arrive_wait(L.bar, P * ++syncs, L.status, wait)) return;
  if (b == 0) back_substitute(L, Wl);
}

// Dynamic shared memory a QR CTA may use: the opt-in limit less 10 KB for the static arrays (7 KB) and a margin.
// (Rows are counted with n + 3 doubles below, two more than they take: the split into groups and CTAs that the
// solvers' results were measured with.)
size_t solve_smem_budget(size_t smem_optin) {
  const size_t fixed = sizeof(double) * (kQRMaxCols + 4) + 2048;
  return smem_optin > fixed ? smem_optin - fixed : 0;
}

}  // namespace

size_t solve_bar_bytes() { return sizeof(unsigned) * kBarCounters * kBarStride; }

int64_t solve_rows_cap(int64_t n, int32_t sms, size_t smem_optin) {
  if (n < 1 || n + 1 > kQRMaxCols) return 0;
  return (int64_t)sms * (int64_t)(solve_smem_budget(smem_optin) / ((size_t)(n + 3) * 8));
}

int32_t solve_ctas(int64_t d, int64_t n, int32_t sms, size_t smem_optin) {
  if (n < 1 || d < n || n + 1 > kQRMaxCols) return 0;
  const size_t budget = solve_smem_budget(smem_optin);
  int64_t ncta = std::min<int64_t>(sms, std::max<int64_t>(1, (d + 7) / 8));
  for (; ncta <= sms; ++ncta) {
    const int64_t rpc = (d + ncta - 1) / ncta;
    if ((size_t)rpc * (size_t)(n + 3) * 8 <= budget) return (int32_t)ncta;
  }
  return 0;
}

// The kernel for an element type and panel width.
template <int NB, int CTAS>
static const void* qr_kernel(const SolveLaunch& L) {
  if (L.src_fp64) return (const void*)qr64_kernel<double, NB, CTAS>;
  if (L.rule == kFP32) return (const void*)qr64_kernel<float, NB, CTAS>;
  if (L.rule == kBF16) return (const void*)qr64_kernel<__nv_bfloat16, NB, CTAS>;
  return (const void*)qr64_kernel<__half, NB, CTAS>;
}

cudaError_t launch_solve(const SolveLaunch& L, cudaStream_t st, int32_t* launches) {
  QRArgs a;
  a.L = L;
  a.rpc = (int32_t)((L.d + L.ncta - 1) / L.ncta);
  // The widest panel whose buffers the scratch holds: 16 columns from n = 29 on, 8 from n = 14, else 4
  // (48 + 8 (n + 1) doubles, which the 256-byte granularity of the regions covers from n = 1 on).
  const int nb = panel_scratch(16, L.n) <= L.part_doubles ? 16 : panel_scratch(8, L.n) <= L.part_doubles ? 8 : 4;
  const int64_t need = panel_scratch(nb, L.n);
  if (need > L.part_doubles) return cudaErrorInvalidValue;
  a.shares_R = need > L.part_own ? 1 : 0;
  cudaError_t e = cudaMemsetAsync(L.part, 0, sizeof(double) * (size_t)need, st);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(L.bar, 0, solve_bar_bytes(), st);
  if (e != cudaSuccess) return e;
  const size_t smem = std::max<size_t>((size_t)a.rpc * (size_t)(L.n + 1) * 8, (size_t)L.n * 8);
  void* args[] = {(void*)&a};
  const bool alone = 2 * smem > 200 * 1024;  // no second CTA of this size on an SM
  const void* kern = nb == 16 ? (alone ? qr_kernel<16, 1>(L) : qr_kernel<16, 3>(L))
                     : nb == 8 ? qr_kernel<8, 2>(L)  // (128 registers hold these without spilling)
                               : qr_kernel<4, 2>(L);
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = cudaLaunchCooperativeKernel(kern, dim3((unsigned)L.ncta), dim3(kQRThreads), args, smem, st);
  if (launches) *launches += 1;
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace sk
