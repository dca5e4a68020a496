// Gather kernel: the chunked sketch by output rows. Each output row of a work item has one owner, which
// fetches the rows of A that S sends to it straight from global memory.
//
// Paper Sec. 4.1 (every element of A is added, with its sign, into its k target rows, Listing 1) with the
// chunked FP32 pre-combine of the other kernels: a work item's sums are added into the per-chunk totals P,
// and the chunk finish scales, rounds (Sec. 4.2) and adds them into Y in chunk order.
//
// Why. The tile kernel adds every element by a shared-memory reduction, for which this GPU has no FP32
// instruction (a compare-and-swap loop): 2^22 x 64 at k = 1 took 516 us, where reading A takes 158. The
// register kernel stages all rows of a box for every group of 1024 output rows, which is cheap where most of
// them have a target in the group (k >= 2 with blocks of up to 512 rows) and wasteful elsewhere. Here a group
// hashes all rows, which costs no memory traffic, and reads only those with a target in it: k reads of A over
// all groups, of which L2 serves the repeats.
//
// Work item: rows [r0, r1) of chunk t (all of it or a slice), 64 columns and up to 512 output rows. Half-warp
// h of the CTA owns the rows h, h + 64, ... of the group; their sums (FP32, 256 bytes each) lie in shared
// memory, where only their owner touches them, so adding is a plain load, FMA and store. The rows come in
// boxes:
//   1. hash: all threads evaluate the box's SplitMix64 outputs (the same generator as every other kernel); a
//      counter per half-warp hands out a slot in its list of (row of the box, output row, sign) entries;
//   2. fetch: every half-warp walks its list, eight rows at a time: eight loads of 256 bytes in flight, then
//      eight additions. One list per half-warp and not per output row: no padding to the longest of many short
//      lists, and a warp waits only for the longer of two.
// Lists and counters are double-buffered: in the phase between two barriers half of the warps hash the next
// box before they fetch and half after, so that hashing and memory latency overlap.
// What bounds it: at k = 1 the loads in flight (at most 128 KB a CTA, and half of its warps hash meanwhile; 4.1
// TB/s at 2^22 x 64), at k = 4 the L1 data path
// (k |A| through it) and the sums' shared-memory traffic. Boxes of about 64 entries per half-warp: with 32 the
// barrier waits for the longest list (k = 4, 7 slices: 616 us against 544), with 96 the lists take the shared memory that
// the L1 cache needs for rows in flight (614 us).
// Measured at 2^22 x 64, d = 4096 (before: tile kernel): k = 1 516 -> 264 us, k = 2 618 -> 369, k = 4 759 -> 582;
// 2^19 x 1024, d = 4096, k = 4 1659 -> 1487; 50001 x 33 (unaligned rows), d = 1056, k = 4 55 -> 39 us (175 before short slices).
#include <algorithm>
#include <cmath>
#include <cstring>

#include "sk_internal.h"
#include "sk_tile.cuh"

namespace sk {

namespace {

constexpr int kGatThreads = 1024;
constexpr int kGatHalves = kGatThreads / 16;       // half-warps: each reads rows of 64 columns
constexpr int kGatSlots = 8;                       // output rows per half-warp (3 bits of an entry)
constexpr int kGatTargets = kGatHalves * kGatSlots;  // output rows per work item at most
constexpr int kGatCols = 64;                       // columns per work item
constexpr int kGatMaxBox = 32768;                  // rows per box: an entry has 15 bits for the row
constexpr double kGatFill = 64.0;                  // entries of a half-warp per box, about
constexpr int kGatAhead = 8;                       // rows a half-warp loads together

struct GatGrid {
  TileDesc D;
  int64_t row_begin, row_end;  // global rows processed
  int64_t R;                   // chunk rows
  int64_t t_first;             // first chunk index
  int64_t items;               // chunks * slices * ncg * ntg
  int32_t ncg, ntg, slices;
  int32_t tgs;                 // output rows per target group
  int32_t box;                 // rows per box (a multiple of kGatThreads)
  int32_t cap;                 // list entries per half-warp and box (a multiple of kGatAhead)
  float* P;                    // per-chunk FP32 totals, chunk-major, d x n each (zero on entry)
};

struct GatItem {
  int64_t r0, r1;                 // global rows
  int32_t tr0, ntr;               // first output row of the group, output rows in it
  int32_t jlo, jhi, plo, np;      // blocks that reach the group, and their 64-bit stream outputs
  int32_t nbox, xcol;             // boxes, first column
  uint64_t z0;                    // SplitMix64 state of row r0's first stream output for the group
  float* P;                       // chunk totals at (tr0, xcol)
};

__device__ __forceinline__ GatItem gat_item(const GatGrid& G, int64_t w) {
  GatItem I;
  const int32_t tg = (int32_t)(w % G.ntg);
  int64_t rest = w / G.ntg;
  const int32_t g = (int32_t)(rest % G.ncg);
  rest /= G.ncg;
  const int32_t sl = (int32_t)(rest % G.slices);
  const int64_t tl = rest / G.slices;
  const int64_t t = G.t_first + tl;
  const int64_t c0 = max(t * G.R, G.row_begin);
  const int64_t c1 = min((t + 1) * G.R, G.row_end);
  I.r0 = c0 + (c1 - c0) * sl / G.slices;
  I.r1 = c0 + (c1 - c0) * (sl + 1) / G.slices;
  const int64_t B = G.D.B, d = B * G.D.k;
  I.tr0 = tg * G.tgs;
  I.ntr = (int32_t)min((int64_t)G.tgs, d - I.tr0);
  I.jlo = (int32_t)(I.tr0 / B);
  I.jhi = (int32_t)((I.tr0 + I.ntr - 1) / B);
  I.plo = I.jlo >> 1;
  I.np = (I.jhi >> 1) - I.plo + 1;
  I.nbox = (int32_t)((I.r1 - I.r0 + G.box - 1) / G.box);
  I.xcol = g * kGatCols;
  I.z0 = G.D.seed + ((uint64_t)I.r0 * G.D.kp + (uint32_t)I.plo + 1ull) * kSplitMixGamma;
  I.P = G.P + tl * (d * G.D.n) + (int64_t)I.tr0 * G.D.n + I.xcol;
  return I;
}

// FP32 vector reduction of four columns (`left` of them inside the matrix) into the chunk totals.
__device__ __forceinline__ void gat_red_quad(float* p, int64_t n, int32_t left, float4 v) {
  if ((n & 3) == 0 && left >= 4) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
  } else {
    atomicAdd(p, v.x);
    if (left > 1) atomicAdd(p + 1, v.y);
    if (left > 2) atomicAdd(p + 2, v.z);
    if (left > 3) atomicAdd(p + 3, v.w);
  }
}

// Step 1 for box b of the item: the box's rows into the half-warps' lists. A list holds its mean number of
// entries and five standard deviations; this thread adds a row that finds it full into the chunk totals.
template <typename TA>
__device__ __forceinline__ void gat_hash(const GatGrid& G, const GatItem& I, int32_t b, uint32_t* cnt, uint32_t* tab) {
  const int64_t rb0 = I.r0 + (int64_t)b * G.box;
  const int32_t left = (int32_t)min((int64_t)G.box, I.r1 - rb0);
  const uint32_t B = G.D.B;
  const uint64_t step = G.D.kp * kSplitMixGamma;
  for (int32_t pr = 0; pr < I.np; ++pr) {
    uint64_t z = I.z0 + (uint64_t)((uint32_t)(b * G.box) + threadIdx.x) * step + (uint64_t)pr * kSplitMixGamma;
    const int32_t jp = 2 * (I.plo + pr);
#pragma unroll 2
    for (int32_t i = (int32_t)threadIdx.x; i < left; i += kGatThreads, z += kGatThreads * step) {
      const uint64_t h = splitmix_finalize(z);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        if (jp + e < I.jlo || jp + e > I.jhi) continue;
        const uint32_t wd = e ? (uint32_t)h : (uint32_t)(h >> 32);
        const uint32_t tgt = (uint32_t)((jp + e) * (int32_t)B + (int32_t)word_to_slot(wd, B) - I.tr0);
        if (tgt >= (uint32_t)I.ntr) continue;
        const uint32_t hw = tgt % kGatHalves, s = tgt / kGatHalves;
        const uint32_t pos = atomicAdd(cnt + hw, 1u);
        if (pos < (uint32_t)G.cap) {
          tab[hw * G.cap + pos] = (uint32_t)i | (s << 16) | (wd << 31);
        } else {
          const TA* a = static_cast<const TA*>(G.D.A) + (rb0 + i - G.D.row_base) * G.D.lda + I.xcol;
          const int32_t nc = (int32_t)min((int64_t)kGatCols, G.D.n - I.xcol);
          float* p = I.P + (int64_t)tgt * G.D.n;
          for (int32_t c = 0; c < nc; ++c) atomicAdd(p + c, (wd & 1u) ? -ld_a(a + c) : ld_a(a + c));
        }
      }
    }
  }
}

// This lane's four columns of a row, as FP32: four adjacent ones by one load (VEC: rows and columns come in
// aligned quads), or every 16th of those inside the matrix. Rows are not kept in L1: no other half-warp of the
// CTA reads them but by chance.
template <typename TA, bool VEC>
__device__ __forceinline__ float4 gat_load(const TA* p, int32_t left) {
  if constexpr (VEC && sizeof(TA) == 4) {
    float4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p));
    return v;
  } else if constexpr (VEC) {
    uint32_t a, b;
    asm volatile("ld.global.nc.L1::no_allocate.v2.b32 {%0, %1}, [%2];" : "=r"(a), "=r"(b) : "l"(p));
    if constexpr (std::is_same<TA, __half>::value) {
      const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&a));
      const float2 g = __half22float2(*reinterpret_cast<const __half2*>(&b));
      return make_float4(f.x, f.y, g.x, g.y);
    } else {
      return make_float4(__uint_as_float(a << 16), __uint_as_float(a & 0xFFFF0000u), __uint_as_float(b << 16),
                         __uint_as_float(b & 0xFFFF0000u));
    }
  } else {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (left > 0) v.x = ld_a(p);
    if (left > 16) v.y = ld_a(p + 16);
    if (left > 32) v.z = ld_a(p + 32);
    if (left > 48) v.w = ld_a(p + 48);
    return v;
  }
}

template <typename TA, bool VEC>
__global__ void __launch_bounds__(kGatThreads, 1) gather_kernel(const GatGrid G) {
  extern __shared__ __align__(16) unsigned char sm[];
  float* acc = reinterpret_cast<float*>(sm);                                     // [tgs][kGatCols]
  uint32_t* cnt = reinterpret_cast<uint32_t*>(acc + (size_t)G.tgs * kGatCols);   // [2][kGatHalves]
  uint32_t* tab = cnt + 2 * kGatHalves;                                          // [2][kGatHalves][cap]
  const int32_t tid = (int32_t)threadIdx.x;
  const int32_t hw = tid >> 4;
  const int32_t c0 = VEC ? (tid & 15) * 4 : (tid & 15);  // this lane's first column; the others follow, or every 16th
  for (int i = tid; i < 2 * kGatHalves; i += kGatThreads) cnt[i] = 0u;
  for (int i = tid; i < G.tgs * kGatCols; i += kGatThreads) acc[i] = 0.f;
  float* my = acc + hw * kGatCols + c0;  // output row hw of the group; slot s is 64 rows further each
  uint32_t sq = 0;
  for (int64_t w = blockIdx.x; w < G.items; w += gridDim.x) {
    const GatItem I = gat_item(G, w);
    const int32_t left = (int32_t)min((int64_t)kGatCols, G.D.n - I.xcol) - c0;  // columns from this lane's first
    const int64_t row_bytes = G.D.lda * (int64_t)sizeof(TA);
    __syncthreads();
    gat_hash<TA>(G, I, 0, cnt + (sq & 1u) * kGatHalves, tab + (sq & 1u) * kGatHalves * G.cap);
    __syncthreads();
    for (int32_t b = 0; b < I.nbox; ++b, ++sq) {
      const uint32_t cur = sq & 1u, nxt = cur ^ 1u;
      const bool first = (tid >> 5) & 1;
      if (first && b + 1 < I.nbox) gat_hash<TA>(G, I, b + 1, cnt + nxt * kGatHalves, tab + nxt * kGatHalves * G.cap);
      const char* base = static_cast<const char*>(G.D.A) + (I.r0 + (int64_t)b * G.box - G.D.row_base) * row_bytes +
                         (int64_t)(I.xcol + c0) * sizeof(TA);
      const int32_t c = (int32_t)min(cnt[cur * kGatHalves + hw], (uint32_t)G.cap);
      const int32_t cm = max(c, __shfl_xor_sync(0xffffffffu, c, 16));
      const uint4* lp = reinterpret_cast<const uint4*>(tab + (cur * kGatHalves + hw) * G.cap);
#pragma unroll 1
      for (int32_t i = 0; i < cm; i += kGatAhead, lp += kGatAhead / 4) {
        uint32_t e[kGatAhead];
        float4 v[kGatAhead];
#pragma unroll
        for (int q = 0; q < kGatAhead; q += 4) {
          const uint4 x = lp[q / 4];
          e[q] = x.x, e[q + 1] = x.y, e[q + 2] = x.z, e[q + 3] = x.w;
        }
#pragma unroll
        for (int q = 0; q < kGatAhead; ++q)
          if (i + q < c && left > 0)
            v[q] = gat_load<TA, VEC>(reinterpret_cast<const TA*>(base + (uint64_t)(e[q] & 0x7FFFu) * (uint32_t)row_bytes), left);
#pragma unroll
        for (int q = 0; q < kGatAhead; ++q) {
          if (i + q < c && left > 0) {
            const float sg = __uint_as_float((e[q] & 0x80000000u) | 0x3F800000u);
            float* a = my + ((e[q] >> 16) & 7u) * (kGatHalves * kGatCols);
            if constexpr (VEC) {
              float4 s = *reinterpret_cast<float4*>(a);
              s.x = fmaf(v[q].x, sg, s.x), s.y = fmaf(v[q].y, sg, s.y);
              s.z = fmaf(v[q].z, sg, s.z), s.w = fmaf(v[q].w, sg, s.w);
              *reinterpret_cast<float4*>(a) = s;
            } else {
              a[0] = fmaf(v[q].x, sg, a[0]);
              if (left > 16) a[16] = fmaf(v[q].y, sg, a[16]);
              if (left > 32) a[32] = fmaf(v[q].z, sg, a[32]);
              if (left > 48) a[48] = fmaf(v[q].w, sg, a[48]);
            }
          }
        }
      }
      __syncwarp();
      if ((tid & 15) == 0) cnt[cur * kGatHalves + hw] = 0u;
      if (!first && b + 1 < I.nbox) gat_hash<TA>(G, I, b + 1, cnt + nxt * kGatHalves, tab + nxt * kGatHalves * G.cap);
      __syncthreads();
    }
    // The item's sums into the chunk totals, and zero again (each half-warp its own output rows).
    for (int32_t t = hw; t < I.ntr; t += kGatHalves) {
      float4* a = reinterpret_cast<float4*>(acc + t * kGatCols) + (tid & 15);
      const float4 v = *a;
      *a = make_float4(0.f, 0.f, 0.f, 0.f);
      const int32_t cq = (tid & 15) * 4;
      const int32_t lq = (int32_t)min((int64_t)kGatCols, G.D.n - I.xcol) - cq;
      if (lq > 0 && (v.x != 0.f || v.y != 0.f || v.z != 0.f || v.w != 0.f))
        gat_red_quad(I.P + (int64_t)t * G.D.n + cq, G.D.n, lq, v);
    }
  }
}

}  // namespace

// Output rows per target group: the d rows split evenly over the groups, in whole slots.
int32_t gat_targets(int64_t d) {
  const int64_t ntg = (d + kGatTargets - 1) / kGatTargets;
  return (int32_t)(((d + ntg - 1) / ntg + kGatHalves - 1) / kGatHalves * kGatHalves);
}

int32_t gat_cols() { return kGatCols; }

// Rows per box, list capacity (cap_fixed > 0: imposed) and shared-memory bytes for items of `rows` rows.
static void gat_box(int64_t d, int64_t B, int64_t rows, int32_t cap_fixed, int32_t* box, int32_t* cap, size_t* smem) {
  const int32_t tgs = gat_targets(d);
  const int32_t slots = tgs / kGatHalves;
  int64_t bx = (int64_t)std::ceil(kGatFill * (double)B / slots / kGatThreads) * kGatThreads;
  bx = std::min<int64_t>(std::max<int64_t>(bx, kGatThreads), kGatMaxBox);
  *box = (int32_t)std::min<int64_t>(bx, (rows + kGatThreads - 1) / kGatThreads * kGatThreads);
  const double lam = (double)*box / (double)B * slots;
  const int64_t c = cap_fixed > 0 ? cap_fixed : (int64_t)std::ceil(lam + 5.0 * std::sqrt(lam) + 4.0);
  *cap = (int32_t)((c + kGatAhead - 1) / kGatAhead * kGatAhead);
  *smem = (size_t)tgs * kGatCols * 4 + 2 * kGatHalves * 4 + 2 * (size_t)kGatHalves * *cap * 4;
}

size_t gat_smem_bytes(int64_t d, int64_t B, int64_t rows) {
  int32_t box, cap;
  size_t smem;
  gat_box(d, B, rows, 0, &box, &cap, &smem);
  return smem;
}

cudaError_t launch_gather(const TileLaunch& L, cudaStream_t st, int32_t* launches) {
  if (!L.P) return cudaErrorInvalidValue;
  GatGrid G;
  memset(&G, 0, sizeof(G));
  const int64_t B = L.d / L.k;
  G.D.A = L.A;
  G.D.Y = L.Y;
  G.D.lda = L.lda;
  G.D.n = L.n;
  G.D.row_base = L.row_begin;
  G.D.seed = L.seed;
  G.D.scale = L.scale;
  G.D.B = (uint32_t)B;
  G.D.k = (uint32_t)L.k;
  G.D.kp = (uint32_t)((L.k + 1) / 2);
  G.D.kb = L.k;
  G.D.S = 1;
  G.D.col_off = L.col_off;
  G.D.a_type = L.a_type;
  G.row_begin = L.row_begin;
  G.row_end = L.row_end;
  G.R = L.R;
  G.t_first = L.row_begin / L.R;
  const int64_t chunks = (L.row_end - 1) / L.R - G.t_first + 1;
  G.ncg = (int32_t)((L.n + kGatCols - 1) / kGatCols);
  G.tgs = gat_targets(L.d);
  G.ntg = (int32_t)((L.d + G.tgs - 1) / G.tgs);
  G.slices = std::max(1, L.slices);
  G.items = chunks * G.slices * G.ncg * G.ntg;
  G.P = L.P;
  const int64_t rows = (std::min<int64_t>(L.R, L.row_end - L.row_begin) + G.slices - 1) / G.slices;
  size_t smem = 0;
  gat_box(L.d, B, rows, L.reg_cap, &G.box, &G.cap, &smem);
  const bool vec = (reinterpret_cast<uintptr_t>(L.A) & 15u) == 0 && L.lda % 4 == 0 && L.n % 4 == 0;
  void (*kern)(const GatGrid) =
      L.a_type == kAF32   ? (vec ? gather_kernel<float, true> : gather_kernel<float, false>)
      : L.a_type == kAF16 ? (vec ? gather_kernel<__half, true> : gather_kernel<__half, false>)
                          : (vec ? gather_kernel<__nv_bfloat16, true> : gather_kernel<__nv_bfloat16, false>);
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(L.grid > 0 ? L.grid : sms, G.items));
  kern<<<(unsigned)grid, kGatThreads, smem, st>>>(G);
  if (launches) *launches += 1;
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (L.no_finish) return cudaSuccess;
  return launch_chunk_finish(G.D, L.rule, G.P, G.t_first, chunks, st, launches);
}

}  // namespace sk
