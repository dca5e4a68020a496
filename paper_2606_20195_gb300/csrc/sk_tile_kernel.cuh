// The chunked tile kernel (fast path of the single-matrix sketch), templated on the rounding rule
// and the element type of A. Paper Sec. 4.1 (SparseStack scatter) and Sec. 4.2 (FP16 variants).
#pragma once

#include "sk_tile.cuh"

namespace sk {

// ------------------------------------------------------------------ tile kernel

// Wait until every CTA of a co-resident (cooperative) grid has arrived. Writes before the call are visible to
// every CTA after it. bar[0] counts arrivals, bar[1] departures and, from bit 16 on, those of CTAs that gave up,
// after `limit` SM clock cycles (false is returned then, and the status word says so). The last CTA to depart,
// when all have arrived and added what they had to add, clears both words and, if one gave up, the `totals`
// floats at `P` too: whatever happened, the next launch finds them at zero. (A grid has fewer than 2^16 CTAs,
// being resident at once. A word of its own for those that gave up cost the last CTA a microsecond.)
__device__ __forceinline__ bool tile_grid_barrier(unsigned* bar, unsigned* status, long long limit, float* P,
                                                  int64_t totals) {
  __shared__ int ok, clean;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 0;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    const long long t0 = clock64();
    while (clock64() - t0 < limit) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if (v >= gridDim.x) {
        ok = 1;
        break;
      }
    }
    if (!ok && status) atomicOr(status, kStatusTimeout);
    clean = 0;
    const unsigned left = atomicAdd(bar + 1, ok ? 1u : 0x10001u);
    if ((left & 0xFFFFu) == gridDim.x - 1) {
      bar[0] = 0u;
      bar[1] = 0u;
      clean = !ok || (left >> 16) != 0u;
    }
  }
  __syncthreads();
  if (clean) {
    __threadfence();
    for (int64_t i = threadIdx.x; i < totals; i += blockDim.x) __stcg(P + i, 0.f);
  }
  return ok != 0;
}

// One CTA per SM (or per work item), work items in a grid-stride loop: scatter, then flush into Y or
// into the chunk totals. TA is the element type of A; the FP32 instantiations live in sk_kernels.cu,
// the 16-bit ones in sk_kernels_a16.cu (compiled in parallel).
template <int RULE, typename TA, bool FINISH>
__global__ void __launch_bounds__(1024) tile_kernel(const TileGrid P, const __grid_constant__ CUtensorMap tmap) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ int abort_flag;
  float* acc = reinterpret_cast<float*>(smem_raw);
  const int warp = threadIdx.x >> 5;
  const int nwarps = blockDim.x >> 5;
  const int RBh = 32 / (int)P.D.kp;
  const SmemPlan SL = smem_plan(P.acc_floats, nwarps, ring_slot_bytes(RBh * P.D.mb, 1 << P.D.log2NC), P.depth);
  uint32_t* wbuf = reinterpret_cast<uint32_t*>(smem_raw + SL.wbuf_off) + warp * kWordsPerWarp;
  WarpRing ring = make_ring(smem_raw, SL, warp);
  for (int x = threadIdx.x; x < P.acc_floats; x += blockDim.x) acc[x] = 0.f;
  if (threadIdx.x == 0) abort_flag = 0;
  __syncthreads();
  TileDesc D = P.D;
  D.tmap = P.use_tma ? (const void*)&tmap : nullptr;
  const int64_t dn = (int64_t)D.B * D.k * D.n;
  for (int64_t w = blockIdx.x; w < P.items; w += gridDim.x) {
    const int32_t g = (int32_t)(w % P.ncg);
    int64_t rest = w / P.ncg;
    const int32_t bg = (int32_t)(rest % P.nbg);
    rest /= P.nbg;
    const int32_t sl = (int32_t)(rest % P.slices);
    const int64_t tl = rest / P.slices;
    const int64_t t = P.t_first + tl;
    const int64_t c0 = max(t * P.R, P.row_begin);
    const int64_t c1 = min((t + 1) * P.R, P.row_end);
    const int64_t r0 = c0 + (c1 - c0) * sl / P.slices;
    const int64_t r1 = c0 + (c1 - c0) * (sl + 1) / P.slices;
    const int32_t j0 = bg * D.kb;
    const int32_t kbe = min(D.kb, (int32_t)D.k - j0);
    if (!tile_scatter_typed<TA>(D, r0, r1, g, j0, kbe, acc, wbuf, ring, warp, nwarps)) {
      abort_flag = 1;
      if (P.status) atomicOr(P.status, kStatusTimeout);
    }
    __syncthreads();
    if (abort_flag) break;
    if (P.slices == 1) {
      tile_flush<RULE>(D, t, g, j0, kbe, acc);
    } else {
      // slice partials into the chunk totals; the end of this kernel (FINISH) or chunk_finish_kernel after
      // it adds them into Y
      tile_flush_partial(D, g, j0, kbe, acc, P.P + tl * dn);
    }
    __syncthreads();
  }
  // One-launch form for sketches too small for a second one: once every CTA's partials are in, the grid
  // finishes the chunk totals itself and writes all of Y. At 16384 x 16, d = 256, k = 4, FP32 the separate
  // finish and the zeroing of Y took 7 of 20 us. An instantiation of its own, as this code costs the scatter
  // loops of the other one 7 to 15 % (131072 x 65, d = 2080: 182 -> 201 us at k = 8, 79 -> 92 at k = 1).
  if constexpr (FINISH) {
    if (!tile_grid_barrier(P.bar, P.status, P.wait_cycles, P.P, P.chunks * dn)) return;
    const int64_t nq = (D.n + 3) >> 2, quads = (int64_t)D.B * D.k * nq;
    for (int64_t f = (int64_t)threadIdx.x * gridDim.x + blockIdx.x; f < quads; f += (int64_t)gridDim.x * blockDim.x) {
      const int64_t r = f / nq;
      finish_quad<RULE, 4, true>(D, (uint32_t)r, 4 * (f - r * nq), P.P, P.t_first, P.chunks, dn);
    }
  }
}

using TileKernelFn = void (*)(const TileGrid, const CUtensorMap);

// The tile kernel for a rule and a 16-bit element type of A (kAF16, kABF16), from sk_kernels_a16.cu.
TileKernelFn tile_kernel_a16(int32_t rule, int32_t a_type, bool finish);

}  // namespace sk
