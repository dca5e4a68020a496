// C ABI of libsk: plan objects, argument validation, kernel dispatch, the host-buffer pipeline
// and the sketch-and-solve driver. Declarations and contracts: include/sk.h.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>

#include "../../include/sk.h"
#include "sk_hostutil.h"
#include "sk_internal.h"
#include "sk_tile.cuh"

namespace sk {

namespace {
thread_local char g_err[512] = {0};
}

sk_status set_error(sk_status code, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
  return code;
}

void clear_error() { g_err[0] = 0; }

const char* last_error_message() { return g_err; }

}  // namespace sk

using namespace sk;

namespace sk {
sk_status noalloc_read_status(unsigned* out);  // sk_noalloc.cu
size_t noalloc_P_bytes();                      // chunk-total bytes its static array holds
}

struct sk_plan_s {
  int64_t d = 0, m = 0, B = 0;
  int32_t k = 0, rule = 0;
  uint64_t seed = 0;
  float scale = 1.f;
  // parameters
  int64_t R = 0;
  int32_t mode = SK_MODE_ATOMIC;
  int64_t row_offset = 0;
  int32_t kernel = SK_KERNEL_AUTO;
  int32_t tile_cols = 0;
  int32_t threads = 0;
  int64_t solve_group_rows = 0;  // rows per QR group of sk_solve (0: as many as shared memory holds)
  int32_t list_cap = 0;          // register kernel: list entries per output row and box (0: automatic)
  int64_t scratch_limit = 0;     // bound on the plan's device scratch in bytes (0: none)
  int64_t solve_wait_cycles = 0; // bound on each grid-barrier wait of the QR kernel (0: default)
  int64_t sketch_wait_cycles = 0;  // and of one-launch sketches
  int64_t last_launches = 0, last_R = 0;
  int32_t last_kernel = 0;  // kernel of the last sketch: 1 tile, 2 literal, 3 owner, 4 global, 5 deterministic, 6 register, 7 gather
  bool last_noalloc = false;  // the last sketch was an sk_apply_noalloc call (status in the static array)
  // device scratch
  float* det_P = nullptr;
  size_t det_P_bytes = 0;
  unsigned* dstatus = nullptr;  // sticky device status word of the sketch kernels
  float* tileP = nullptr;       // two-level chunk totals (zero between launches)
  double* lsqr = nullptr;       // sk_solve_precond: u (m), 8 n-vectors, scalars, x0 (n floats)
  size_t lsqr_bytes = 0;
  size_t tileP_bytes = 0;
  // for sketches that could do without chunk totals: the words of the one-launch form's grid barrier, then the
  // totals (all zero between launches). The words stay at one place whatever n and d: totals may end as -0,
  // which is zero as a number and not as a counter.
  unsigned* fastP = nullptr;
  size_t fastP_bytes = 0;
  cudaEvent_t fast_done = nullptr;     // behind the last call that used fastP,
  unsigned long long fast_stream = 0;  // and the id of its stream (ids, unlike handles, are not used again)
  void* solve_buf = nullptr;
  size_t solve_bytes = 0;
  size_t solve_status_off = 0, solve_kappa_off = 0;
  // host-pipeline staging
  float* stage[2] = {nullptr, nullptr};
  size_t stage_bytes = 0;
  void* ydev = nullptr;
  size_t ydev_bytes = 0;
  cudaStream_t copy_stream = nullptr;
  cudaEvent_t ev_copied[2] = {nullptr, nullptr};
  cudaEvent_t ev_used[2] = {nullptr, nullptr};
};

namespace {

constexpr int32_t kMaxK = 64;
constexpr int64_t kMaxN = 65535;
constexpr int32_t kMaxSolveN = 1024;

sk_status cuda_fail(cudaError_t e, const char* what) {
  return set_error(SK_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

struct DevInfo {
  int sms = 0, optin = 0;
};

sk_status dev_info(DevInfo* di) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  cudaDeviceGetAttribute(&di->sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&di->optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  return SK_OK;
}

size_t elem_size(int32_t rule) { return rule == SK_FP32 ? 4 : 2; }

// Device scratch the plan holds, in bytes.
size_t plan_scratch_bytes(const sk_plan_s* p) {
  return p->det_P_bytes + (p->dstatus ? sizeof(unsigned) : 0) + p->tileP_bytes + p->fastP_bytes + p->lsqr_bytes + p->solve_bytes +
         2 * p->stage_bytes + p->ydev_bytes;
}

// Give back the chunk totals that the plan's sketches can do without (cudaFree waits for their users).
bool drop_fast(sk_plan_s* p) {
  if (!p->fastP) return false;
  cudaFree(p->fastP);
  p->fastP = nullptr;
  p->fastP_bytes = 0;
  return true;
}

// Whether `bytes` more of scratch in place of `cur` fit the plan's limit, if need be after giving back the
// totals that its sketches can do without.
bool fits_limit(sk_plan_s* p, size_t cur, size_t bytes) {
  if (p->scratch_limit <= 0) return true;
  const size_t limit = (size_t)p->scratch_limit, others = plan_scratch_bytes(p) - cur + bytes;
  if (others <= limit) return true;
  return others - p->fastP_bytes <= limit && drop_fast(p);
}

// Replace one plan buffer (*ptr of *cur bytes) by a new one of `bytes`: checked against the plan's
// scratch limit first, so a refused call leaves the plan's buffers as they were and enqueues nothing;
// SK_ERR_OOM also when cudaMalloc fails.
template <typename T>
sk_status plan_grow(sk_plan_s* p, T** ptr, size_t* cur, size_t bytes, const char* what) {
  if (!fits_limit(p, *cur, bytes))
    return set_error(SK_ERR_OOM, "%s (%zu bytes) would take the plan's scratch above its limit of %lld bytes", what,
                     bytes, (long long)p->scratch_limit);
  if (*ptr) cudaFree(*ptr);
  *ptr = nullptr;
  *cur = 0;
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(ptr), bytes);
  if (e != cudaSuccess && drop_fast(p)) e = cudaMalloc(reinterpret_cast<void**>(ptr), bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return set_error(SK_ERR_OOM, "%s (%zu bytes)", what, bytes);
  }
  *cur = bytes;
  return SK_OK;
}

// Tile-kernel configuration for a plan and a column count.
struct TileCfg {
  int32_t NC = 0, kb = 0, threads = 0, grid = 0, slices = 1, depth = 1, mb = 1;
  int32_t long_slices = 1;  // slices without fill_slices: for callers short of chunk-total scratch
  int64_t R = 0;
  bool serial = false;
  bool lr = false;
  bool own = false;
  bool vec = false;
  bool glob = false;
  bool reg = false, gat = false;
  bool other = false;  // chosen for speed: another kernel, which may need no chunk totals, runs where these cannot be had
  int32_t reg_nsub = 0, reg_cap = 0;
  bool tile_alone() const { return !glob && !reg && !gat && !own; }
};

// Default chunk length: at most 8 chunks per matrix (each output then receives at most 8 rounded
// contributions) and at least 4096 rows per chunk; a multiple of 32.
int64_t default_chunk_rows(int64_t m) {
  int64_t R = std::max<int64_t>(4096, (m + 7) / 8);
  return ((R + 31) / 32) * 32;
}

// Whether A (device pointer, row stride lda, es-byte elements) can be staged through TMA: a
// 16-byte-aligned base and a row stride that is a multiple of 16 bytes.
bool tma_layout_ok(const void* A, int64_t lda, int64_t es = 4) {
  return (reinterpret_cast<uintptr_t>(A) & 15u) == 0 && (lda * es) % 16 == 0;
}

// Split each chunk into slices: at least about 4 work items per resident CTA, slices at least
// max(4096, 2d) rows long so the partial flushes (d x NC floats each) stay small, and, among the
// slice counts up to 4x that minimum, the one whose work items fill the last round of CTAs best
// (the items of one launch are of equal size, so a last round of 120 items on 152 CTAs idles 21 % of
// the GPU for a whole item).
int32_t choose_slices(const sk_plan_s* p, int64_t rows, int64_t R, int64_t ncg, int64_t nbg, int32_t cps,
                      const DevInfo& di) {
  const int64_t first = ((p->row_offset % R) + R) % R;  // offset of the first row inside its chunk
  const int64_t chunks = (first + rows + R - 1) / R;
  const int64_t G = (int64_t)di.sms * std::max(cps, 1);
  const int64_t per = std::max<int64_t>(1, chunks * ncg * nbg);
  const int64_t s_lo = std::max<int64_t>(1, (4 * G + per - 1) / per);
  const int64_t min_rows = std::max<int64_t>(4096, 2 * p->d);
  const int64_t s_max = std::min<int64_t>(std::max<int64_t>(1, std::min(R, rows) / min_rows), 4096);
  int64_t best = std::min(s_lo, s_max);
  double best_waste = 1e30;
  for (int64_t sl = std::min(s_lo, s_max); sl <= std::min(4 * s_lo, s_max); ++sl) {
    const int64_t items = per * sl;
    const double waste = (double)((items + G - 1) / G * G) / (double)items;
    if (waste < best_waste - 0.005) {
      best_waste = waste;
      best = sl;
    }
  }
  return (int32_t)best;
}

// More slices per chunk where `slices` of them give fewer work items than the GPU holds CTAs: as many as
// fit in one round of CTAs, of at least 64 rows each. Below that size an item costs its CTA's start and its
// flush of d x NC floats, and its rows hardly count; a 153rd item would cost a second round. Where one
// slice needs no chunk totals (`finishes` false), only from three slices on, which pay for adding them up
// (two were 2 us slower at 5000 x 256, d = 4096, k = 4), and with n % 4 != 0, where every float of a flush is
// an atomic of its own, only while an item's rows make as many additions (8192 x 130, d = 4160, k = 1, four
// slices: 45 us, not 36). Measured, all slices at least 4096 rows / filled up
// (and, but for the register kernel, one launch that finishes the chunk totals itself): 16384 x 16,
// d = 256, k = 4 (4 items / 152): 42 / 14.5 us; 50001 x 33, d = 1056, k = 4 (16 / 144): 175 / 55;
// 65536 x 64, d = 1024, k = 4 (32 / 144, register kernel): 47 / 28; 8192 x 64, d = 8192, k = 4: 43 / 28.
// Where half of the CTAs make slices of up to 320 rows, half it is: alone such a call is as fast, and two run side
// by side (30 plans on 30 streams, us a call: 16384 x 16 11.5 -> 6.2, one slice a chunk 7.0; 3000 x 12, d = 4096,
// k = 2 14.9 -> 7.9 and 6.7). Larger ones lose beside others part of what they gain alone: 65536 x 64 48 -> 29
// alone, 8.5 -> 13.3 beside 29 others; 60000 x 20, d = 320, k = 8 201 -> 27 and 12 -> 25.
int32_t fill_slices(const sk_plan_s* p, int64_t n, int64_t rows, int64_t R, int64_t ncg, int64_t nbg, int32_t cps,
                    const DevInfo& di, int32_t slices, bool finishes) {
  const int64_t first = ((p->row_offset % R) + R) % R;
  const int64_t per = (first + rows + R - 1) / R * ncg * nbg;
  const int64_t chunk = std::min(R, rows);
  int64_t fit = std::min((int64_t)di.sms * std::max(cps, 1) / per, std::max<int64_t>(1, chunk / 64));
  const int64_t half = (int64_t)di.sms * std::max(cps, 1) / (2 * per);
  if (half >= 3 && chunk <= 320 * half) fit = std::min(fit, half);
  if (n % 4 != 0) fit = std::min(fit, chunk * p->k / p->d);
  if (fit <= slices || (!finishes && slices == 1 && fit < 3)) return slices;
  return (int32_t)fit;
}

// Whether the chunks of `rows` rows are long enough for a kernel whose chunk totals another form would do
// without: the default chunk length always (at most 8 chunks, one more with a row offset, of at least 4096
// rows); shorter ones the caller has set while the totals are no larger than A in FP32, and many of them while
// a quarter of it. So what a plan may hold for speed is bounded by A or by 9 d n floats. Chunks shorter than
// that cost their totals' traffic and a work item's start for few rows each: gather kernel, 50001 x 33,
// d = 1056, FP32, R = 6256 / 2112 / 528: 39 / 60 / 106 us, tile kernel without totals 124 / 57 / 59; register
// kernel, bfloat16, 2^20 x 64, d = 1024, k = 4, R = 2^17 / 4096 / 1024: 112 / 199 / 558 us, tile 220 / 234 / 353.
bool chunks_pay_totals(const sk_plan_s* p, int64_t rows, int64_t R) {
  const int64_t chunks = (p->row_offset % R + rows + R - 1) / R;
  if (chunks > 9) return chunks <= rows / (4 * p->d);
  return chunks == 1 || R >= 4096 || chunks * p->d <= rows;
}

// Owner-kernel configuration (atomic mode, SK_KERNEL_OWNER): blocks per item kb = 2 when two blocks
// of 32-column lines fit in shared memory, else 1; false if the kernel does not apply.
bool choose_own(const sk_plan_s* p, int64_t n, int64_t rows, const DevInfo& di, bool tma_ok, TileCfg* cfg) {
  if (p->mode != SK_MODE_ATOMIC || !tma_ok || n < 32 || rows >= ((int64_t)1 << 31)) return false;
  if (p->kernel != SK_KERNEL_OWNER) return false;
  const size_t optin = (size_t)std::min(di.optin, 232448) - 1024;
  int32_t kb = 0;
  if (p->k >= 2 && own_smem_bytes(p->B, 2) <= optin) kb = 2;
  else if (own_smem_bytes(p->B, 1) <= optin) kb = 1;
  if (kb == 0) return false;
  const int64_t R = p->R > 0 ? p->R : default_chunk_rows(p->m);
  const int32_t cps = own_ctas_per_sm(p->rule, own_smem_bytes(p->B, kb));
  if (cps < 1) return false;
  const int64_t ncg = (n + 31) / 32;
  const int64_t nbg = (p->k + kb - 1) / kb;
  cfg->NC = 32;
  cfg->kb = kb;
  cfg->threads = own_threads();
  cfg->grid = 0;
  cfg->R = R;
  cfg->slices = cfg->long_slices = choose_slices(p, rows, R, ncg, nbg, cps, di);
  cfg->depth = 1;
  cfg->mb = 1;
  cfg->serial = false;
  cfg->lr = false;
  cfg->own = true;
  cfg->vec = false;
  return true;
}

// Global-accumulator configuration: chunk totals in device memory (any block height).
void choose_global(const sk_plan_s* p, TileCfg* cfg) {
  *cfg = TileCfg();
  cfg->NC = 4;
  cfg->kb = p->k;
  cfg->threads = 256;
  cfg->R = p->R > 0 ? p->R : default_chunk_rows(p->m);
  cfg->slices = 1;
  cfg->glob = true;
}

// Register-kernel configuration (atomic mode, A staged through TMA): the staged box and list
// capacity for the plan's block height, the default chunk length and the slice count. AUTO takes it
// for k >= 2, n >= 32 and blocks of at most 512 rows (not n >= 256 with k = 2, which goes to the
// global kernel), where it is faster than the tile kernel
// (measured at 2^22 x 64: d = 4096, k = 8: 1060 vs 818 GB/s; d = 1024, k = 8: 1520 vs 798; taller blocks, as
// d = 4096 with k = 4 or 2, are the gather kernel's: 582 and 369 us, tile kernel 759 and 618, this one 791 and 741;
// bfloat16 A: d = 4096, k = 8: 732 vs 1332 us; d = 1024, k = 4: 287 vs 735; 2^21 x 40, d = 320, k = 4:
// 162 vs 356; 20000 x 128, d = 2048, k = 4: 26 vs 34; 2^18 x 1024, d = 2048, k = 4: 546 vs 917).
bool choose_reg(const sk_plan_s* p, int64_t n, int64_t rows, const DevInfo& di, bool tma_ok, int32_t a_type,
                TileCfg* cfg) {
  if (p->mode != SK_MODE_ATOMIC || !tma_ok || rows >= ((int64_t)1 << 31)) return false;
  if (p->kernel == SK_KERNEL_AUTO) {
    if (p->tile_cols != 0 || p->threads != 0 || p->k < 2 || n < 32 || p->B > 512) return false;
    if (n >= 256 && p->k <= 2) return false;  // the global kernel's case (wide rows, few nonzeros)
  } else if (p->kernel != SK_KERNEL_REGISTER || a_type != SK_A_FP32) {
    return false;
  }
  const size_t optin = (size_t)std::min(di.optin, 232448) - 1024;
  const int64_t R = p->R > 0 ? p->R : default_chunk_rows(p->m);
  if (a_type != SK_A_FP32 && !chunks_pay_totals(p, rows, R)) return false;
  int32_t nsub = 0, cap = 0;
  if (!reg_choose_box(p->d, p->B, a_type, optin, p->list_cap, &nsub, &cap)) return false;
  const int64_t ncg = (n + reg_cols(a_type) - 1) / reg_cols(a_type);
  const int64_t ntg = (p->d + reg_targets(a_type) - 1) / reg_targets(a_type);
  *cfg = TileCfg();
  cfg->NC = 32;
  cfg->kb = p->k;
  cfg->threads = reg_threads(a_type);
  cfg->R = R;
  cfg->long_slices = choose_slices(p, rows, R, ncg, ntg, 1, di);
  cfg->slices = fill_slices(p, n, rows, R, ncg, ntg, 1, di, cfg->long_slices, true);
  cfg->reg = true;
  cfg->other = p->kernel == SK_KERNEL_AUTO && a_type != SK_A_FP32;
  cfg->reg_nsub = nsub;
  cfg->reg_cap = cap;
  return true;
}

// Where AUTO takes the gather kernel: where it was the faster one of 16500 shapes (n from 17 to 4097, d up to 65536,
// k = 1, 2, 3, 4, 8, 2^13 to 2^22 rows, default chunk length; over the 14500 inside the line 1.8 times as fast as
// the kernel taken otherwise in the mean, 0.9 or less at 16). Every group of 512 output rows and every 64 columns
// hash all rows again, so the cost grows with d n, and the rows have to pay for it. In brackets the time of the
// other kernel over the gather kernel's beyond the line.
// - Aligned rows, n < 256, from 65536 rows on (8192 with d >= 4096, n >= 64): k = 1 from 24 columns on, d up to
//   8192; k = 2 below the register kernel's 32 columns (24 use 3/8 of the lanes: 0.73 at 2^22 rows, d = 4096);
//   blocks too tall for that kernel, B > 512, while k reads of a row waste few lanes, or FP32 and d from 8192 to
//   12288 (d = 14336: 0.7 to 0.9 below 2^20 rows). Not below 110000 rows with 129 to 159 columns (0.74 to 0.9) or
//   k = 4 and more than 96 columns (0.82 to 0.94), both at d from 4096 to 8191; k = 4, d < 4096, n > 192: 0.77.
// - FP32, n >= 256, from 131072 rows on: k <= 2 with n <= 512 and d <= 2048 (d = 2 n at 131072 rows: 0.81), k = 3 or 4
//   with B in (512, 1024]; elsewhere the global kernel stays ahead.
// - FP32 rows that TMA cannot read: d <= 8448 or a 128th of the rows (0.5 to 0.8 above); from 32768 rows on,
//   with k >= 2, n < 256 and d from 512 to 4224 from 8192. k = 8 not with 40 % of the last 64 columns' lanes idle;
//   k <= 2 later: an even n, for which the other kernel adds pairs (0.72 to 0.9 before), and k = 1 with few
//   columns and output rows (0.84) or with n >= 256, where the global kernel makes few reductions (0.7 to 0.9).
bool gather_wins(const sk_plan_s* p, int64_t n, int64_t rows, bool tma_ok, int32_t a_type) {
  const int64_t k = p->k, d = p->d, B = p->B, lanes = (n + 63) / 64 * 64;
  const bool f32 = a_type == SK_A_FP32;
  if (rows >= ((int64_t)1 << 31) || rows < 8192 || B < 64 || k > 8 || n < 16) return false;
  if (!tma_ok) {
    if (!f32 || n < 17 || (k > 4 && 5 * n < 3 * lanes) || (d > 8448 && (k == 1 || rows < 128 * d))) return false;
    if (n > 4100 || (n > 1024 && d > (k < 3 ? 2048 : 4096))) return false;
    if (rows < 32768) return k >= 2 && n < 256 && d >= 512 && d <= 4224;
    if (k == 2) {
      if (n >= 256 && n < 384) return rows >= std::min<int64_t>(131072, std::max<int64_t>(50000, 128 * d));
      return n % 2 != 0 || rows >= 50000;
    }
    if (k > 2 || d <= 128) return true;
    if (n >= 512) return d <= 2048 || rows >= 32 * d;
    if (n >= 256) return rows >= std::max<int64_t>(131072, 32 * d);
    if (n % 2 == 0) return rows >= (d <= 2048 ? 65000 : 110000);
    return rows >= 50000 || d >= 1024 || n >= 160;
  }
  if (n % 4 != 0 || (rows < 65536 && (d < 4096 || n < 64))) return false;
  if (n < 256) {
    const bool mid = d >= 4096 && d < 8192;
    if (n > 128 && n < 160 && mid && rows <= 110000) return false;
    if (k == 4 && rows >= 24000 && rows < 110000 && ((n > 96 && mid) || (n > 192 && d < 4096 && rows < 80000))) return false;
    if (k == 1) return (n >= 24 || rows >= (1 << 20)) && d <= 8192;
    if (n < 32) return k == 2 && n >= 24 && d <= 8192 && (rows <= (1 << 20) || d <= (n < 28 ? 512 : 4096));
    if (B <= 512 || n < 48) return false;
    if (k * lanes <= 5 * n) return d <= 8192;
    return f32 && d >= 8192 && d < 16384 && (d <= 12288 || (n <= 64 && rows >= (1 << 20)));
  }
  if (!f32 || rows < 131072) return false;
  if (k <= 2) return n <= 512 && d <= 2048 && (d <= n || (d <= 2 * n && rows >= (1 << 18)) || rows >= (1 << 20));
  return k <= 4 && n <= 2048 && B > 512 && B <= 1024;
}

// Gather-kernel configuration. The slices are the ones for which the rounds of work items end first, an item
// taking (measured at 2^22 x 64, d = 4096) 0.53 ns for each of its rows' hashes, 3.6 ns for each row it
// fetches and 9 us to start and flush: k = 1, 2 / 7 / 14 slices 250 / 254 / 288 us, k = 4 611 / 544 / 565.
// Few slices make long FP32 sums: of an output's N = chunk / B additions a slice makes N / s one after another,
// and the chunk total s. The squared error grows with N / s + s, least at s = sqrt(N); slices that make it more
// than 3 % larger than that are not taken (2^21 x 128, d = 4096, k = 4: tile kernel with 19 slices 1.25e-7,
// here with 25 % allowed 1.34e-7).
bool choose_gather(const sk_plan_s* p, int64_t n, int64_t rows, const DevInfo& di, bool tma_ok, int32_t a_type,
                   TileCfg* cfg) {
  const int64_t R = p->R > 0 ? p->R : default_chunk_rows(p->m);
  if (p->mode != SK_MODE_ATOMIC || p->kernel != SK_KERNEL_AUTO || p->tile_cols != 0 || p->threads != 0 ||
      !gather_wins(p, n, rows, tma_ok, a_type) ||
      !chunks_pay_totals(p, rows, R) ||
      gat_smem_bytes(p->d, p->B, rows) > (size_t)std::min(di.optin, 232448) - 1024)
    return false;
  const int64_t ncg = (n + gat_cols() - 1) / gat_cols();
  const int64_t tgs = gat_targets(p->d), ntg = (p->d + tgs - 1) / tgs;
  const int64_t first = ((p->row_offset % R) + R) % R;
  const int64_t chunks = (first + rows + R - 1) / R;
  const double row_ns = 0.53 + 3.6 * (double)std::min<int64_t>(tgs, p->d) / (double)p->B;
  const int64_t chunk = std::min(R, rows);
  const double adds = (double)chunk / (double)p->B, adds_max = std::max(4.0, 2.06 * std::sqrt(adds));
  const int64_t most = std::min<int64_t>(1024, std::max<int64_t>(1, chunk / 64));
  int64_t best = std::min(most, std::max<int64_t>(1, (int64_t)std::sqrt(adds)));
  double best_ns = 1e300;
  for (int64_t sl = 1; sl <= std::min<int64_t>(most, 256); ++sl) {
    if (adds / (double)sl + (double)sl > adds_max) continue;
    const double rounds = (double)((chunks * sl * ncg * ntg + di.sms - 1) / di.sms);
    const double ns = rounds * ((double)chunk / (double)sl * row_ns + 9000.0);
    if (ns < best_ns) best_ns = ns, best = sl;
  }
  *cfg = TileCfg();
  cfg->NC = 32;
  cfg->kb = p->k;
  cfg->R = R;
  cfg->slices = cfg->long_slices = (int32_t)best;
  cfg->reg_cap = p->list_cap;
  cfg->gat = cfg->other = true;
  return true;
}

sk_status choose_tile(const sk_plan_s* p, int64_t n, int64_t rows, const DevInfo& di, TileCfg* cfg,
                      bool tma_ok = false, int32_t a_type = SK_A_FP32, bool scratch = true) {
  if (scratch && choose_gather(p, n, rows, di, tma_ok, a_type, cfg)) return SK_OK;
  if (choose_reg(p, n, rows, di, tma_ok, a_type, cfg) && (scratch || !cfg->other)) return SK_OK;
  *cfg = TileCfg();
  if (p->kernel == SK_KERNEL_REGISTER)
    return set_error(SK_ERR_UNSUPPORTED,
                     "register kernel: needs atomic mode, FP32 A, A 16-byte aligned with lda %% 4 == 0 and fewer "
                     "than 2^31 rows");
  if (p->kernel == SK_KERNEL_GLOBAL) {
    if (p->mode != SK_MODE_ATOMIC) return set_error(SK_ERR_UNSUPPORTED, "the global kernel runs in atomic mode only");
    choose_global(p, cfg);
    return SK_OK;
  }
  if (choose_own(p, n, rows, di, tma_ok, cfg)) return SK_OK;
  if (p->kernel == SK_KERNEL_OWNER)
    return set_error(SK_ERR_UNSUPPORTED,
                     "owner kernel: needs atomic mode, n >= 32, A 16-byte aligned with lda %% 4 == 0 and "
                     "2 x %lld x 128 bytes of shared memory",
                     (long long)p->B);
  const bool serial = (p->mode == SK_MODE_SERIAL_TILE);
  if (n == 1 && !serial && p->tile_cols <= 4) {
    // A single column: the vector path (one thread per row, accumulator lines of one quad).
    const int32_t threads = p->threads > 0 ? p->threads : 1024;
    int32_t kb = 0;
    for (int32_t kbt = p->k; kbt >= 1; --kbt) {
      const int64_t fl = tile_acc_floats((uint32_t)p->B, kbt, tile_slots(4, kbt), 4);
      if (tile_smem_bytes(p->B, kbt, 4, threads, p->k, 1) <= (size_t)std::min(di.optin, 232448) - 1024 && fl < (1 << 29)) {
        kb = kbt;
        break;
      }
    }
    if (kb > 0) {
      const int64_t R = p->R > 0 ? p->R : default_chunk_rows(p->m);
      const int64_t nbg = (p->k + kb - 1) / kb;
      const int32_t cps = tile_ctas_per_sm(p->rule, threads, tile_smem_bytes(p->B, kb, 4, threads, p->k, 1));
      cfg->NC = 4;
      cfg->kb = kb;
      cfg->threads = threads;
      cfg->grid = 0;
      cfg->R = R;
      cfg->long_slices = choose_slices(p, rows, R, 1, nbg, cps, di);
      cfg->slices = fill_slices(p, n, rows, R, 1, nbg, cps, di, cfg->long_slices, false);
      cfg->depth = 1;
      cfg->mb = 1;
      cfg->serial = false;
      cfg->lr = false;
      cfg->own = false;
      cfg->vec = true;
      return SK_OK;
    }
  }
  const int32_t threads = serial ? 32 : (p->threads > 0 ? p->threads : 1024);
  const int32_t nwarps = threads / 32;
  const int32_t RB = 32 / ((p->k + 1) / 2);
  const size_t optin = (size_t)std::min(di.optin, 232448) - 1024;
  // Fits: accumulator + target words + a ring of at least one slot per warp.
  auto fits = [&](int32_t c, int32_t kbt) {
    const int64_t fl = tile_acc_floats((uint32_t)p->B, kbt, tile_slots(c, kbt), c);
    return tile_smem_bytes(p->B, kbt, c, threads, p->k, 1) <= optin && fl < (1 << 29);
  };
  const int32_t widths[4] = {32, 16, 8, 4};
  int32_t NC = 0, kb = 0;
  for (int32_t c : widths) {
    if (p->tile_cols > 0 && c != p->tile_cols) continue;
    if (!serial && c > 4 && (c / 2 >= n || c * RB > 256)) continue;
    // Serial (verification) mode needs the lane groups of a pass to hit distinct blocks.
    if (serial && (32 / c > p->k || p->k % (32 / c) != 0)) continue;
    if (fits(c, p->k)) {
      NC = c;
      kb = p->k;
      break;
    }
  }
  if (NC == 0 && !serial) {
    NC = p->tile_cols > 0 ? p->tile_cols : 4;
    for (int32_t kbt = p->k; kbt >= 1; --kbt) {
      if (fits(NC, kbt)) {
        kb = kbt;
        break;
      }
    }
  }
  if (NC == 0 || kb == 0) {
    // A block too tall for the on-chip accumulator: chunk totals in device memory instead.
    if (!serial && p->kernel == SK_KERNEL_AUTO) {
      choose_global(p, cfg);
      return SK_OK;
    }
    return set_error(SK_ERR_UNSUPPORTED,
                     "tile kernel: a block of %lld rows does not fit in shared memory with the requested width",
                     (long long)p->B);
  }
  // Where the tile kernel would need several block groups (the target-word scatter, 5-7x slower
  // than the global kernel at n = 1024 and d >= 16384), or only 4-column items for a wide matrix
  // (each row's hash evaluated n/4 times), AUTO takes the global-accumulator kernel. So it does for
  // wide matrices at k <= 2: there the tile kernel's cost is the per-item overhead (hash and staging
  // per column group for only k * NC updates per row) while the global kernel's k n / 4 L2
  // reductions per row are few (measured at n = 256 / 1024, d/n = 2: k = 1 1809 -> 3100 and
  // 2035 -> 3745 GB/s, k = 2 1559 -> 2504 and 1810 -> 2686 GB/s; at k = 4 the two are within 3 %).
  if (!serial && p->kernel == SK_KERNEL_AUTO && p->tile_cols == 0 &&
      (kb < p->k || (NC <= 4 && n >= 256) || (p->k <= 2 && n >= 256))) {
    choose_global(p, cfg);
    return SK_OK;
  }
  // One block group (outside serial mode): every work item takes the lane-row path, with several
  // hash rounds per TMA box (boxes of up to 1 KiB).
  const bool lr = !serial && kb == p->k;
  int32_t mb = 1;
  if (lr) mb = std::max(1, std::min(8, 1024 / (RB * NC * 4)));
  while (mb > 1 && tile_smem_bytes(p->B, kb, NC, threads, p->k, 1, mb) > optin) mb /= 2;
  int32_t depth = 1;
  while (depth < kMaxRingDepth && tile_smem_bytes(p->B, kb, NC, threads, p->k, depth + 1, mb) <= optin) ++depth;
  int64_t R = p->R > 0 ? p->R : default_chunk_rows(p->m);
  int32_t slices = 1, long_slices = 1;
  if (!serial) {
    const int64_t ncg = (n + NC - 1) / NC;
    const int64_t nbg = (p->k + kb - 1) / kb;
    const int32_t cps = tile_ctas_per_sm(p->rule, threads, tile_smem_bytes(p->B, kb, NC, threads, p->k, depth, mb));
    long_slices = choose_slices(p, rows, R, ncg, nbg, cps, di);
    slices = fill_slices(p, n, rows, R, ncg, nbg, cps, di, long_slices, false);
  }
  cfg->NC = NC;
  cfg->kb = kb;
  cfg->threads = threads;
  cfg->grid = serial ? 1 : 0;
  cfg->R = R;
  cfg->slices = slices;
  cfg->long_slices = long_slices;
  cfg->depth = depth;
  cfg->mb = mb;
  cfg->lr = lr;
  cfg->own = false;
  cfg->vec = false;
  cfg->serial = serial;
  return SK_OK;
}

sk_status validate_apply(const sk_plan_s* p, const void* A, int64_t lda, int64_t n, const void* Y,
                         uintptr_t a_align = 4) {
  if (!p) return set_error(SK_ERR_INVALID_ARG, "plan is NULL");
  if (!A) return set_error(SK_ERR_INVALID_ARG, "A is NULL");
  if (!Y) return set_error(SK_ERR_INVALID_ARG, "Y is NULL");
  if (n < 1 || n > kMaxN) return set_error(SK_ERR_INVALID_ARG, "n=%lld outside [1, %lld]", (long long)n, (long long)kMaxN);
  if (lda < n) return set_error(SK_ERR_INVALID_ARG, "lda=%lld < n=%lld", (long long)lda, (long long)n);
  if ((reinterpret_cast<uintptr_t>(A) & (a_align - 1)) != 0)
    return set_error(SK_ERR_INVALID_ARG, "A must be %d-byte aligned", (int)a_align);
  if ((reinterpret_cast<uintptr_t>(Y) & 3u) != 0) return set_error(SK_ERR_INVALID_ARG, "Y must be 4-byte aligned");
  if (p->m > (int64_t)1 << 40 || lda > ((int64_t)1 << 40) / std::max<int64_t>(p->m, 1))
    return set_error(SK_ERR_UNSUPPORTED, "A larger than 2^40 elements");
  return SK_OK;
}

bool capturing(cudaStream_t st) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) return cudaGetLastError(), true;
  return cap != cudaStreamCaptureStatusNone;
}

// Chunk-total bytes of a sketch with chunk length R.
size_t totals_bytes(const sk_plan_s* p, int64_t n, int64_t row_begin, int64_t row_end, int64_t R) {
  return sizeof(float) * (size_t)(((row_end - 1) / R - row_begin / R + 1) * p->d * n);
}

// Whether a buffer of the plan (`cur` bytes now) holds `need` bytes or may be grown to: within the scratch
// limit, and not while the stream is being captured.
bool can_hold(const sk_plan_s* p, size_t cur, size_t need, cudaStream_t st) {
  if (cur >= need) return true;
  if (p->scratch_limit > 0 && plan_scratch_bytes(p) - cur + need > (size_t)p->scratch_limit) return false;
  return !capturing(st);
}

// For the calls inside its scope, another stream's capture in global mode is no error (this thread's stream is
// not the captured one): the allocations and queries made for optional scratch must not end it.
struct RelaxedCapture {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

// A buffer of chunk totals of the plan with room for `need` bytes, zero where it is new. False where the memory
// is not to be had: no error yet, as the caller may have a form that needs less.
template <typename T>
bool grow_totals(sk_plan_s* p, T** ptr, size_t* cur, size_t need, cudaStream_t st) {
  if (*cur >= need) return true;
  if (plan_grow(p, ptr, cur, need, "chunk-total scratch") != SK_OK) return clear_error(), false;
  if (cudaMemsetAsync(*ptr, 0, need, st) == cudaSuccess) return true;
  cudaFree(*ptr);  // (not zero: must not be taken for totals by a later call)
  *ptr = nullptr;
  *cur = 0;
  return cudaGetLastError(), false;
}

// The `need` bytes of chunk totals in p->fastP, for a sketch that can do without any; null where they are not to
// be had. Not in a stream capture, even with the buffer in place: the graph would hold its address,
// which a later call that needs a larger one frees. And not while a call on another stream may still be using
// them: without totals a sketch touches only its own A and Y, so one thread may issue several with one plan on
// several streams. The caller launches on st next and then calls leave_fast.
float* take_fast(sk_plan_s* p, size_t need, cudaStream_t st) {
  need += sizeof(unsigned) * kBarrierWords;
  if (capturing(st) || !can_hold(p, p->fastP_bytes, need, st)) return nullptr;
  unsigned long long id = 0;
  if (cudaStreamGetId(st, &id) != cudaSuccess) return cudaGetLastError(), nullptr;
  RelaxedCapture relaxed;
  if (!p->fast_done) {
    if (cudaEventCreateWithFlags(&p->fast_done, cudaEventDisableTiming) != cudaSuccess) return cudaGetLastError(), nullptr;
  } else if (id != p->fast_stream && cudaEventQuery(p->fast_done) != cudaSuccess) {
    return cudaGetLastError(), nullptr;
  }
  p->fast_stream = id;
  if (!grow_totals(p, &p->fastP, &p->fastP_bytes, need, st)) return nullptr;
  return reinterpret_cast<float*>(p->fastP + kBarrierWords);
}

// The call's launches on st that use p->fastP are enqueued.
sk_status leave_fast(sk_plan_s* p, cudaStream_t st) {
  cudaError_t e = cudaEventRecord(p->fast_done, st);
  return e == cudaSuccess ? SK_OK : cuda_fail(e, "chunk-total scratch");
}

// Enqueue Y = S * A for rows [row_begin, row_begin + rows) (A row 0 = row_begin) with chunk rows R.
// Y must already be zero, or zero_y set: then Y is zeroed on the stream once the plan's scratch is in
// place (a call refused for lack of scratch leaves Y untouched). a_type: element type of A
// (SK_A_FP32, SK_A_FP16, SK_A_BF16).
sk_status enqueue_sketch(sk_plan_s* p, const void* A, int64_t lda, int64_t n, int64_t row_begin, int64_t rows, void* Y,
                         int64_t R_fixed, cudaStream_t st, int32_t* launches, int64_t* R_used, int64_t col_off = 0,
                         int32_t a_type = SK_A_FP32, bool zero_y = false) {
  p->last_noalloc = false;
  DevInfo di;
  sk_status s = dev_info(&di);
  if (s != SK_OK) return s;
  const int64_t row_end = row_begin + rows;
  const bool literal = (p->kernel == SK_KERNEL_LITERAL);
  if (p->mode == SK_MODE_DETERMINISTIC) {
    int64_t R = R_fixed > 0 ? R_fixed : p->R;
    if (R <= 0) {
      TileCfg cfg;
      s = choose_tile(p, n, p->m, di, &cfg);
      if (s != SK_OK) return s;
      R = literal ? 1 : cfg.R;
    }
    const size_t need = sizeof(float) * (size_t)(p->d * n);
    if (p->det_P_bytes < need) {
      s = plan_grow(p, &p->det_P, &p->det_P_bytes, need, "deterministic-mode scratch");
      if (s != SK_OK) return s;
    }
    if (zero_y) {
      cudaError_t ez = cudaMemsetAsync(Y, 0, elem_size(p->rule) * (size_t)(p->d * n), st);
      if (ez != cudaSuccess) return cuda_fail(ez, "zeroing Y");
    }
    DetLaunch L;
    L.A = A;
    L.a_type = a_type;
    L.Y = Y;
    L.P = p->det_P;
    L.lda = lda;
    L.n = n;
    L.row_begin = row_begin;
    L.row_end = row_end;
    L.d = p->d;
    L.k = p->k;
    L.rule = p->rule;
    L.seed = p->seed;
    L.scale = p->scale;
    L.R = R;
    L.col_off = col_off;
    cudaError_t e = launch_det(L, st, launches);
    if (e != cudaSuccess) return cuda_fail(e, "deterministic kernel launch");
    p->last_kernel = 5;
    if (R_used) *R_used = R;
    return SK_OK;
  }
  if (literal) {
    if (p->R > 1 || R_fixed > 1) return set_error(SK_ERR_INVALID_ARG, "the literal kernel implements chunk rows R = 1 only");
    if (zero_y) {
      cudaError_t ez = cudaMemsetAsync(Y, 0, elem_size(p->rule) * (size_t)(p->d * n), st);
      if (ez != cudaSuccess) return cuda_fail(ez, "zeroing Y");
    }
    LiteralLaunch L;
    L.A = A;
    L.a_type = a_type;
    L.Y = Y;
    L.lda = lda;
    L.n = n;
    L.row_begin = row_begin;
    L.row_end = row_end;
    L.d = p->d;
    L.k = p->k;
    L.rule = p->rule;
    L.seed = p->seed;
    L.scale = p->scale;
    L.col_off = col_off;
    cudaError_t e = launch_literal(L, st, launches);
    if (e != cudaSuccess) return cuda_fail(e, "literal kernel launch");
    p->last_kernel = SK_KERNEL_LITERAL;
    if (R_used) *R_used = 1;
    return SK_OK;
  }
  TileCfg cfg;
  const bool tma_ok = tma_layout_ok(A, lda, a_type == SK_A_FP32 ? 4 : 2);
  s = choose_tile(p, n, rows, di, &cfg, tma_ok, a_type);
  if (s != SK_OK) return s;
  if (cfg.own && a_type != SK_A_FP32) return set_error(SK_ERR_UNSUPPORTED, "the owner kernel reads FP32 A only");
  if (R_fixed > 0) cfg.R = R_fixed;
  if (!p->dstatus) {
    size_t cur = 0;
    s = plan_grow(p, &p->dstatus, &cur, sizeof(unsigned), "status word");
    if (s != SK_OK) return s;
    cudaError_t ez = cudaMemsetAsync(p->dstatus, 0, sizeof(unsigned), st);
    if (ez != cudaSuccess) return cuda_fail(ez, "zeroing status word");
  }
  // Chunk totals of a sketch that another kernel, or one slice per chunk, makes without any: taken if they can
  // be had, else that form runs. (Sketches that need totals either way keep them in p->tileP.)
  float* fast = nullptr;
  if (cfg.other) {
    TileCfg alt;
    s = choose_tile(p, n, rows, di, &alt, tma_ok, a_type, false);
    if (s != SK_OK) return s;
    if (R_fixed > 0) alt.R = R_fixed;
    bool ok;
    if (alt.tile_alone() && alt.long_slices == 1) {
      alt.slices = 1;
      fast = take_fast(p, totals_bytes(p, n, row_begin, row_end, cfg.R), st);
      ok = fast != nullptr;
    } else {
      const size_t need = totals_bytes(p, n, row_begin, row_end, cfg.R);
      ok = can_hold(p, p->tileP_bytes, need, st) && grow_totals(p, &p->tileP, &p->tileP_bytes, need, st);
    }
    if (!ok) cfg = alt;
  } else if (cfg.tile_alone() && cfg.slices > 1 && cfg.long_slices == 1) {
    fast = take_fast(p, totals_bytes(p, n, row_begin, row_end, cfg.R), st);
    if (!fast) cfg.slices = 1;
  }
  TileLaunch L;
  L.A = A;
  L.a_type = a_type;
  L.Y = Y;
  L.lda = lda;
  L.n = n;
  L.row_begin = row_begin;
  L.row_end = row_end;
  L.d = p->d;
  L.k = p->k;
  L.rule = p->rule;
  L.seed = p->seed;
  L.scale = p->scale;
  L.R = cfg.R;
  L.NC = cfg.NC;
  L.kb = cfg.kb;
  L.threads = cfg.threads;
  L.grid = cfg.grid;
  L.slices = cfg.slices;
  L.depth = cfg.depth;
  L.mb = cfg.mb;
  L.lr = cfg.lr ? 1 : 0;
  L.own = cfg.own ? 1 : 0;
  L.vec = cfg.vec ? 1 : 0;
  L.glob = cfg.glob ? 1 : 0;
  L.reg = cfg.reg ? 1 : 0;
  L.gat = cfg.gat ? 1 : 0;
  L.reg_nsub = cfg.reg_nsub;
  L.reg_cap = cfg.reg_cap;
  L.col_off = col_off;
  L.allow_tma = cfg.vec ? 0 : 1;
  L.status = p->dstatus;
  L.P = fast;
  if (fast) {
    // The short slices finish in the same launch if Y is this call's alone (not one that other calls add to).
    if (zero_y && cfg.tile_alone()) L.bar = p->fastP;
    L.wait_cycles = p->sketch_wait_cycles;
  } else if (cfg.slices > 1 || cfg.glob || cfg.reg || cfg.gat) {
    const size_t needP = sizeof(float) * (size_t)launch_P_floats(L);
    if (p->tileP_bytes < needP) {
      s = plan_grow(p, &p->tileP, &p->tileP_bytes, needP, "chunk-total scratch");
      if (s != SK_OK) return s;
      cudaError_t ez = cudaMemsetAsync(p->tileP, 0, needP, st);
      if (ez != cudaSuccess) return cuda_fail(ez, "zeroing chunk totals");
    }
    L.P = p->tileP;
  }
  if (zero_y && !L.bar) {
    cudaError_t ez = cudaMemsetAsync(Y, 0, elem_size(p->rule) * (size_t)(p->d * n), st);
    if (ez != cudaSuccess) return cuda_fail(ez, "zeroing Y");
  }
  cudaError_t e = launch_tile(L, st, launches);
  if (fast) {
    s = leave_fast(p, st);
    if (e == cudaSuccess && s != SK_OK) return s;
  }
  if (e != cudaSuccess)
    return cuda_fail(e, cfg.gat   ? "gather kernel launch"
                        : cfg.glob  ? "global kernel launch"
                        : cfg.reg ? "register kernel launch"
                        : cfg.own ? "owner kernel launch"
                                  : "tile kernel launch");
  p->last_kernel = cfg.gat ? SK_KERNEL_GATHER : cfg.glob ? SK_KERNEL_GLOBAL : cfg.reg ? SK_KERNEL_REGISTER : cfg.own ? SK_KERNEL_OWNER : SK_KERNEL_TILE;
  if (R_used) *R_used = cfg.R;
  return SK_OK;
}

}  // namespace

extern "C" {

int32_t sk_version(void) { return 10000; }

const char* sk_last_error(void) { return last_error_message(); }

sk_status sk_plan_create(int64_t d, int64_t m, int32_t k, int32_t rule, uint64_t seed, sk_plan* out) {
  clear_error();
  if (!out) return set_error(SK_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  if (k < 1 || k > kMaxK) return set_error(SK_ERR_INVALID_ARG, "k=%d outside [1, %d]", k, kMaxK);
  if (d < 1 || d % k != 0) return set_error(SK_ERR_INVALID_ARG, "d=%lld must be a positive multiple of k=%d", (long long)d, k);
  if (d > 0x7fffffffLL) return set_error(SK_ERR_UNSUPPORTED, "d=%lld above 2^31-1", (long long)d);
  if (m < 1) return set_error(SK_ERR_INVALID_ARG, "m=%lld must be >= 1", (long long)m);
  if (m > ((int64_t)1 << 56)) return set_error(SK_ERR_UNSUPPORTED, "m=%lld too large", (long long)m);
  if (rule < SK_FP32 || rule > SK_BF16_RN) return set_error(SK_ERR_INVALID_ARG, "unknown rule %d", rule);
  sk_plan_s* p = new (std::nothrow) sk_plan_s();
  if (!p) return set_error(SK_ERR_OOM, "host allocation failed");
  p->d = d;
  p->m = m;
  p->k = k;
  p->B = d / k;
  p->rule = rule;
  p->seed = seed;
  p->scale = (float)(1.0 / std::sqrt((double)k));
  *out = p;
  return SK_OK;
}

sk_status sk_plan_set(sk_plan p, int32_t key, int64_t v) {
  clear_error();
  if (!p) return set_error(SK_ERR_INVALID_ARG, "plan is NULL");
  switch (key) {
    case SK_PARAM_CHUNK_ROWS:
      if (v < 0) return set_error(SK_ERR_INVALID_ARG, "chunk rows must be >= 0");
      p->R = v;
      return SK_OK;
    case SK_PARAM_MODE:
      if (v < 0 || v > 2) return set_error(SK_ERR_INVALID_ARG, "mode must be 0 (atomic), 1 (deterministic) or 2 (serial tile)");
      p->mode = (int32_t)v;
      return SK_OK;
    case SK_PARAM_ROW_OFFSET:
      if (v < 0) return set_error(SK_ERR_INVALID_ARG, "row offset must be >= 0");
      p->row_offset = v;
      return SK_OK;
    case SK_PARAM_KERNEL:
      if (v < SK_KERNEL_AUTO || (v > SK_KERNEL_GLOBAL && v != SK_KERNEL_REGISTER))
        return set_error(SK_ERR_INVALID_ARG, "unknown kernel %lld", (long long)v);
      p->kernel = (int32_t)v;
      return SK_OK;
    case SK_PARAM_TILE_COLS:
      if (v != 0 && v != 4 && v != 8 && v != 16 && v != 32)
        return set_error(SK_ERR_INVALID_ARG, "tile cols must be 0, 4, 8, 16 or 32");
      p->tile_cols = (int32_t)v;
      return SK_OK;
    case SK_PARAM_THREADS:
      if (v != 0 && (v < 128 || v > 1024 || v % 32 != 0))
        return set_error(SK_ERR_INVALID_ARG, "threads must be 0 or a multiple of 32 in [128, 1024]");
      p->threads = (int32_t)v;
      return SK_OK;
    case SK_PARAM_SOLVE_GROUP_ROWS:
      if (v < 0) return set_error(SK_ERR_INVALID_ARG, "solve group rows must be >= 0");
      p->solve_group_rows = v;
      return SK_OK;
    case SK_PARAM_LIST_CAP:
      if (v < 0 || v > 64) return set_error(SK_ERR_INVALID_ARG, "list capacity must be in [0, 64]");
      p->list_cap = (int32_t)v;
      return SK_OK;
    case SK_PARAM_ROWS:
      if (v < 1) return set_error(SK_ERR_INVALID_ARG, "rows must be >= 1");
      if (v > ((int64_t)1 << 56)) return set_error(SK_ERR_UNSUPPORTED, "rows=%lld too large", (long long)v);
      p->m = v;
      return SK_OK;
    case SK_PARAM_SCRATCH_LIMIT:
      if (v < 0) return set_error(SK_ERR_INVALID_ARG, "scratch limit must be >= 0");
      p->scratch_limit = v;
      return SK_OK;
    case SK_PARAM_SOLVE_WAIT_CYCLES:
      if (v < 0) return set_error(SK_ERR_INVALID_ARG, "solve wait cycles must be >= 0");
      p->solve_wait_cycles = v;
      return SK_OK;
    case SK_PARAM_SKETCH_WAIT_CYCLES:
      if (v < 0) return set_error(SK_ERR_INVALID_ARG, "sketch wait cycles must be >= 0");
      p->sketch_wait_cycles = v;
      return SK_OK;
    default:
      return set_error(SK_ERR_INVALID_ARG, "unknown or read-only key %d", key);
  }
}

sk_status sk_plan_get(sk_plan p, int32_t key, int64_t* v) {
  clear_error();
  if (!p || !v) return set_error(SK_ERR_INVALID_ARG, "NULL argument");
  switch (key) {
    case SK_PARAM_CHUNK_ROWS: *v = p->R; return SK_OK;
    case SK_PARAM_MODE: *v = p->mode; return SK_OK;
    case SK_PARAM_ROW_OFFSET: *v = p->row_offset; return SK_OK;
    case SK_PARAM_KERNEL: *v = p->kernel; return SK_OK;
    case SK_PARAM_TILE_COLS: *v = p->tile_cols; return SK_OK;
    case SK_PARAM_THREADS: *v = p->threads; return SK_OK;
    case SK_PARAM_SOLVE_GROUP_ROWS: *v = p->solve_group_rows; return SK_OK;
    case SK_PARAM_LIST_CAP: *v = p->list_cap; return SK_OK;
    case SK_PARAM_SCRATCH_LIMIT: *v = p->scratch_limit; return SK_OK;
    case SK_PARAM_ROWS: *v = p->m; return SK_OK;
    case SK_PARAM_SOLVE_WAIT_CYCLES: *v = p->solve_wait_cycles; return SK_OK;
    case SK_PARAM_SKETCH_WAIT_CYCLES: *v = p->sketch_wait_cycles; return SK_OK;
    case SK_PARAM_SCRATCH_BYTES: *v = (int64_t)plan_scratch_bytes(p); return SK_OK;
    case SK_PARAM_LAST_LAUNCHES: *v = p->last_launches; return SK_OK;
    case SK_PARAM_LAST_CHUNK_ROWS: *v = p->last_R; return SK_OK;
    case SK_PARAM_LAST_KERNEL: *v = p->last_kernel; return SK_OK;
    case SK_PARAM_DEVICE_STATUS: {
      *v = 0;
      if (!p->dstatus && !p->last_noalloc) return SK_OK;
      cudaError_t e = cudaDeviceSynchronize();
      if (e != cudaSuccess) return cuda_fail(e, "device status");
      unsigned w = 0;
      if (p->dstatus) {
        e = cudaMemcpy(&w, p->dstatus, sizeof(unsigned), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) return cuda_fail(e, "device status");
      }
      if (p->last_noalloc) {
        unsigned wn = 0;
        sk_status s = noalloc_read_status(&wn);
        if (s != SK_OK) return s;
        w |= wn;
      }
      *v = (int64_t)w;
      return SK_OK;
    }
    default: return set_error(SK_ERR_INVALID_ARG, "unknown key %d", key);
  }
}

sk_status sk_apply(sk_plan p, const float* A, int64_t lda, int64_t n, void* Y, void* stream) {
  clear_error();
  sk_status s = validate_apply(p, A, lda, n, Y);
  if (s != SK_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  int32_t launches = 0;
  int64_t R_used = 0;
  s = enqueue_sketch(p, A, lda, n, p->row_offset, p->m, Y, 0, st, &launches, &R_used, 0, SK_A_FP32, true);
  p->last_launches = launches;
  p->last_R = R_used;
  return s;
}

sk_status sk_apply_typed(sk_plan p, const void* A, int32_t a_type, int64_t lda, int64_t n, void* Y, void* stream) {
  clear_error();
  if (a_type != SK_A_FP32 && a_type != SK_A_FP16 && a_type != SK_A_BF16)
    return set_error(SK_ERR_INVALID_ARG, "unknown element type %d of A", a_type);
  sk_status s = validate_apply(p, A, lda, n, Y, a_type == SK_A_FP32 ? 4 : 2);
  if (s != SK_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  int32_t launches = 0;
  int64_t R_used = 0;
  s = enqueue_sketch(p, A, lda, n, p->row_offset, p->m, Y, 0, st, &launches, &R_used, 0, a_type, true);
  p->last_launches = launches;
  p->last_R = R_used;
  return s;
}

sk_status sk_apply_host(sk_plan p, const float* A_host, int64_t lda, int64_t n, void* Y_host, void* stream) {
  clear_error();
  sk_status s = validate_apply(p, A_host, lda, n, Y_host);
  if (s != SK_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  DevInfo di;
  s = dev_info(&di);
  if (s != SK_OK) return s;
  // Chunk rows of the whole matrix, so that the tiles reproduce sk_apply's chunks exactly.
  int64_t R = p->R;
  if (p->kernel == SK_KERNEL_LITERAL) R = 1;
  if (R <= 0) {
    TileCfg cfg;
    s = choose_tile(p, n, p->m, di, &cfg);
    if (s != SK_OK) return s;
    R = cfg.R;
  }
  // Tiles of whole chunks, about 128 MiB each.
  const int64_t row_bytes = lda * 4;
  const int64_t target_rows = std::max<int64_t>(1, ((int64_t)128 << 20) / row_bytes);
  int64_t tile_rows;
  if (R >= target_rows) {
    tile_rows = R;
  } else {
    tile_rows = (target_rows / R) * R;
  }
  // The first chunk may be partial when the row offset is not a multiple of R: align tiles to the
  // global chunk grid.
  tile_rows = std::min(tile_rows, p->m + (p->row_offset % R));
  const size_t tile_bytes = (size_t)tile_rows * (size_t)row_bytes;
  const size_t ybytes = elem_size(p->rule) * (size_t)(p->d * n);
  if (p->stage_bytes < tile_bytes) {
    // both staging tiles at once against the limit (plan_grow counts stage_bytes twice)
    if (!fits_limit(p, 2 * p->stage_bytes, 2 * tile_bytes))
      return set_error(SK_ERR_OOM, "host pipeline staging (2 x %zu bytes) would take the plan's scratch above its limit",
                       tile_bytes);
    for (int b = 0; b < 2; ++b) {
      if (p->stage[b]) cudaFree(p->stage[b]);
      p->stage[b] = nullptr;
    }
    p->stage_bytes = 0;
    for (int b = 0; b < 2; ++b) {
      if (cudaMalloc(&p->stage[b], tile_bytes) != cudaSuccess &&
          (!drop_fast(p) || cudaMalloc(&p->stage[b], tile_bytes) != cudaSuccess)) {
        cudaGetLastError();
        return set_error(SK_ERR_OOM, "host pipeline staging (%zu bytes)", tile_bytes);
      }
    }
    p->stage_bytes = tile_bytes;
  }
  if (p->ydev_bytes < ybytes) {
    s = plan_grow(p, &p->ydev, &p->ydev_bytes, ybytes, "host pipeline Y buffer");
    if (s != SK_OK) return s;
  }
  if (!p->copy_stream) {
    if (cudaStreamCreateWithFlags(&p->copy_stream, cudaStreamNonBlocking) != cudaSuccess)
      return cuda_fail(cudaGetLastError(), "copy stream");
    for (int b = 0; b < 2; ++b) {
      cudaEventCreateWithFlags(&p->ev_copied[b], cudaEventDisableTiming);
      cudaEventCreateWithFlags(&p->ev_used[b], cudaEventDisableTiming);
    }
  }
  int32_t launches = 0;
  cudaError_t e = cudaMemsetAsync(p->ydev, 0, ybytes, st);
  if (e != cudaSuccess) return cuda_fail(e, "zeroing Y");
  // Buffers start free: mark both as used-and-finished on the compute stream.
  for (int b = 0; b < 2; ++b) cudaEventRecord(p->ev_used[b], st);
  int64_t done = 0;
  int which = 0;
  const int64_t g0 = p->row_offset;
  while (done < p->m) {
    // Tile boundaries on the global chunk grid.
    const int64_t gstart = g0 + done;
    const int64_t chunk_start = (gstart / R) * R;
    int64_t gend = chunk_start + tile_rows;
    if (gend <= gstart) gend = gstart + R;
    gend = std::min(gend, g0 + p->m);
    const int64_t rows = gend - gstart;
    float* buf = p->stage[which];
    e = cudaStreamWaitEvent(p->copy_stream, p->ev_used[which], 0);
    if (e != cudaSuccess) return cuda_fail(e, "pipeline wait");
    if (lda == n) {
      e = cudaMemcpyAsync(buf, A_host + done * lda, (size_t)rows * n * 4, cudaMemcpyHostToDevice, p->copy_stream);
    } else {
      e = cudaMemcpy2DAsync(buf, (size_t)lda * 4, A_host + done * lda, (size_t)lda * 4, (size_t)n * 4, (size_t)rows,
                            cudaMemcpyHostToDevice, p->copy_stream);
    }
    if (e != cudaSuccess) return cuda_fail(e, "host to device copy");
    cudaEventRecord(p->ev_copied[which], p->copy_stream);
    cudaStreamWaitEvent(st, p->ev_copied[which], 0);
    s = enqueue_sketch(p, buf, lda, n, gstart, rows, p->ydev, R, st, &launches, nullptr);
    if (s != SK_OK) return s;
    cudaEventRecord(p->ev_used[which], st);
    done += rows;
    which ^= 1;
  }
  e = cudaMemcpyAsync(Y_host, p->ydev, ybytes, cudaMemcpyDeviceToHost, st);
  if (e != cudaSuccess) return cuda_fail(e, "device to host copy");
  e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail(e, "sk_apply_host");
  p->last_launches = launches;
  p->last_R = R;
  return SK_OK;
}

sk_status sk_materialize_S(sk_plan p, int64_t i0, int64_t cnt, int32_t* rows, int8_t* signs, void* stream) {
  clear_error();
  if (!p || !rows || !signs) return set_error(SK_ERR_INVALID_ARG, "NULL argument");
  if (i0 < 0 || cnt < 0) return set_error(SK_ERR_INVALID_ARG, "negative range");
  if (cnt == 0) return SK_OK;
  cudaError_t e = launch_pattern(p->d, p->k, p->seed, i0, cnt, rows, signs, (cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_fail(e, "pattern kernel launch");
  return SK_OK;
}

// Solve scratch layout (bytes, each region 256-byte aligned):
//   Y_A (d*n elements), Y_b (d elements), part (n + n*(n+1) doubles: the QR's reduction buffers, then
//   LSQR's R^-1), R (n*(n+1) doubles), tail (n doubles more for the reduction buffers, which may use R's
//   region too), bar (grid-barrier counters), status (1 word), kappa (1 double).
namespace {
struct SolveLayout {
  size_t ya, yb, part, R, tail, bar, status, kappa, stack[2], total;
};
size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }
// stack_groups: groups of the first tree level (0: the sketch is factored by one launch).
SolveLayout solve_layout(int64_t d, int64_t n, int32_t rule, int64_t stack_groups) {
  SolveLayout L;
  size_t off = 0;
  const size_t es = elem_size(rule);
  L.ya = off; off = al256(off + es * (size_t)(d * n));
  L.yb = off; off = al256(off + es * (size_t)d);
  L.part = off; off = al256(off + 8 * (size_t)(n + n * (n + 1)));
  L.R = off; off = al256(off + 8 * (size_t)(n * (n + 1)));
  L.tail = off; off = al256(off + 8 * (size_t)n);
  L.bar = off; off = al256(off + solve_bar_bytes());
  L.status = off; off = al256(off + 4);
  L.kappa = off; off = al256(off + 8);
  for (int i = 0; i < 2; ++i) {
    L.stack[i] = off;
    off = al256(off + 8 * (size_t)(stack_groups * n * (n + 1)));
  }
  L.total = off;
  return L;
}

// Rows per group of the QR tree for a d x (n+1) sketch: the whole sketch if it fits one launch,
// else a cap of at least 2n rows (each level then shrinks the stack at least by half). 0: unsupported.
int64_t solve_group_cap(const sk_plan_s* p, int64_t n, const DevInfo& di) {
  const int64_t cap_auto = solve_rows_cap(n, di.sms, (size_t)di.optin);
  if (cap_auto < n) return 0;
  int64_t cap = cap_auto;
  if (p->solve_group_rows > 0) cap = std::min(cap, std::max(p->solve_group_rows, 2 * n));
  if (p->d > cap && cap < 2 * n) return 0;
  return cap;
}

// QR back end of sketch-and-solve (paper Sec. 5.3: QR of the sketch SA, then R x = (Q^T Sb)[:n]):
// x from the sketch columns SA (d x n, row stride lda_sa) and Sb (d values, stride sb_stride) in the
// plan's element type, in FP64; tree levels (groups of at most `cap` rows factored, their [R | c]
// factors stacked and factored again) when the sketch is taller than one QR launch holds.
sk_status solve_backend(sk_plan_s* p, const void* SA, int64_t lda_sa, const void* Sb, int64_t sb_stride, int64_t n,
                        float* x, cudaStream_t st, const DevInfo& di, int64_t cap, const SolveLayout& Lo,
                        int32_t* launches) {
  char* base = (char*)p->solve_buf;
  SolveLaunch L;
  L.wait_cycles = p->solve_wait_cycles;
  L.SA = SA;
  L.Sb = Sb;
  L.lda_sa = lda_sa;
  L.sb_stride = sb_stride;
  L.rule = p->rule;
  L.src_fp64 = 0;
  L.n = n;
  // The QR's reduction buffers may spread over the R region behind `part` (R is written at the end).
  L.part = (double*)(base + Lo.part);
  L.part_doubles = (int64_t)(Lo.bar - Lo.part) / 8;
  L.part_own = (int64_t)(Lo.R - Lo.part) / 8;
  L.bar = (unsigned*)(base + Lo.bar);
  L.status = (unsigned*)(base + Lo.status);
  L.kappa = (double*)(base + Lo.kappa);
  L.x = x;
  // Tree levels: factor groups of at most `cap` rows, stack their [R | c] factors, repeat.
  int64_t rows = p->d;
  int level = 0;
  while (rows > cap) {
    const int64_t g = (rows + cap - 1) / cap;
    double* dst = (double*)(base + Lo.stack[level & 1]);
    const size_t es_src = L.src_fp64 ? sizeof(double) : elem_size(p->rule);
    for (int64_t gi = 0; gi < g; ++gi) {
      const int64_t r0 = gi * rows / g, r1 = (gi + 1) * rows / g;
      SolveLaunch G = L;
      G.SA = (const char*)L.SA + es_src * (size_t)(r0 * L.lda_sa);
      G.Sb = (const char*)L.Sb + es_src * (size_t)(r0 * L.sb_stride);
      G.d = r1 - r0;
      G.R = dst + gi * n * (n + 1);
      G.solve_x = 0;
      G.ncta = solve_ctas(G.d, n, di.sms, (size_t)di.optin);
      if (G.ncta < 1) return set_error(SK_ERR_UNSUPPORTED, "QR group of %lld rows does not fit", (long long)G.d);
      cudaError_t e = launch_solve(G, st, launches);
      if (e != cudaSuccess) return cuda_fail(e, "QR group launch");
    }
    L.SA = dst;
    L.Sb = dst + n;
    L.lda_sa = n + 1;
    L.sb_stride = n + 1;
    L.src_fp64 = 1;
    rows = g * n;
    ++level;
  }
  L.d = rows;
  L.R = (double*)(base + Lo.R);
  L.solve_x = 1;
  L.ncta = solve_ctas(rows, n, di.sms, (size_t)di.optin);
  if (L.ncta < 1) return set_error(SK_ERR_UNSUPPORTED, "FP64 QR of a %lld x %lld matrix does not fit", (long long)rows, (long long)(n + 1));
  cudaError_t e = launch_solve(L, st, launches);
  if (e != cudaSuccess) return cuda_fail(e, "QR launch");
  return SK_OK;
}

}  // namespace

sk_status sk_solve(sk_plan p, const float* A, int64_t lda, int64_t n, const float* b, float* x, void* stream) {
  clear_error();
  sk_status s = validate_apply(p, A, lda, n, x);
  if (s != SK_OK) return s;
  if (!b) return set_error(SK_ERR_INVALID_ARG, "b is NULL");
  if (n > p->d) return set_error(SK_ERR_INVALID_ARG, "sketch-and-solve needs n=%lld <= d=%lld", (long long)n, (long long)p->d);
  if (n > kMaxSolveN) return set_error(SK_ERR_UNSUPPORTED, "sketch-and-solve supports n <= %d", kMaxSolveN);
  DevInfo di;
  s = dev_info(&di);
  if (s != SK_OK) return s;
  const int64_t cap = solve_group_cap(p, n, di);
  if (cap < 1)
    return set_error(SK_ERR_UNSUPPORTED, "FP64 QR of a %lld x %lld sketch: too many columns for shared memory",
                     (long long)p->d, (long long)(n + 1));
  const int64_t groups1 = (p->d > cap) ? (p->d + cap - 1) / cap : 0;
  const SolveLayout Lo = solve_layout(p->d, n, p->rule, groups1);
  if (p->solve_bytes < Lo.total) {
    s = plan_grow(p, &p->solve_buf, &p->solve_bytes, Lo.total, "sketch-and-solve scratch");
    if (s != SK_OK) return s;
    // On the call's stream: a memset on the legacy default stream is not ordered with a non-blocking
    // caller stream and could land after this call's kernels have written the scratch.
    cudaError_t ez = cudaMemsetAsync(p->solve_buf, 0, Lo.total, (cudaStream_t)stream);
    if (ez != cudaSuccess) return cuda_fail(ez, "zeroing sketch-and-solve scratch");
  }
  p->solve_status_off = Lo.status;
  p->solve_kappa_off = Lo.kappa;
  char* base = (char*)p->solve_buf;
  cudaStream_t st = (cudaStream_t)stream;
  int32_t launches = 0;
  const size_t es = elem_size(p->rule);
  cudaError_t e = cudaMemsetAsync(base + Lo.ya, 0, Lo.part - Lo.ya, st);  // Y_A and Y_b
  if (e != cudaSuccess) return cuda_fail(e, "zeroing sketches");
  e = cudaMemsetAsync(base + Lo.status, 0, 4, st);
  if (e != cudaSuccess) return cuda_fail(e, "zeroing status");
  (void)es;
  int64_t R_used = 0;
  s = enqueue_sketch(p, A, lda, n, p->row_offset, p->m, base + Lo.ya, 0, st, &launches, &R_used);
  if (s != SK_OK) return s;
  // Sb is column n of [A | b]: the same chunks, and the rounding bits of global column n.
  s = enqueue_sketch(p, b, 1, 1, p->row_offset, p->m, base + Lo.yb, R_used, st, &launches, nullptr, n);
  if (s != SK_OK) return s;
  s = solve_backend(p, base + Lo.ya, n, base + Lo.yb, 1, n, x, st, di, cap, Lo, &launches);
  if (s != SK_OK) return s;
  p->last_launches = launches;
  p->last_R = R_used;
  return SK_OK;
}

sk_status sk_solve_sketched(sk_plan p, const void* SAb, int64_t ld, int64_t n, float* x, void* stream) {
  clear_error();
  if (!p) return set_error(SK_ERR_INVALID_ARG, "plan is NULL");
  if (!SAb || !x) return set_error(SK_ERR_INVALID_ARG, "NULL sketch or x");
  if (n < 1 || ld < n + 1) return set_error(SK_ERR_INVALID_ARG, "need n >= 1 and ld >= n + 1 (n=%lld ld=%lld)",
                                            (long long)n, (long long)ld);
  if (n > p->d) return set_error(SK_ERR_INVALID_ARG, "sketch-and-solve needs n=%lld <= d=%lld", (long long)n, (long long)p->d);
  if (n > kMaxSolveN) return set_error(SK_ERR_UNSUPPORTED, "sketch-and-solve supports n <= %d", kMaxSolveN);
  const size_t es = elem_size(p->rule);
  if ((reinterpret_cast<uintptr_t>(SAb) % es) != 0) return set_error(SK_ERR_INVALID_ARG, "sketch not aligned to its elements");
  DevInfo di;
  sk_status s = dev_info(&di);
  if (s != SK_OK) return s;
  const int64_t cap = solve_group_cap(p, n, di);
  if (cap < 1)
    return set_error(SK_ERR_UNSUPPORTED, "FP64 QR of a %lld x %lld sketch: too many columns for shared memory",
                     (long long)p->d, (long long)(n + 1));
  const int64_t groups1 = (p->d > cap) ? (p->d + cap - 1) / cap : 0;
  const SolveLayout Lo = solve_layout(p->d, n, p->rule, groups1);
  if (p->solve_bytes < Lo.total) {
    s = plan_grow(p, &p->solve_buf, &p->solve_bytes, Lo.total, "sketch-and-solve scratch");
    if (s != SK_OK) return s;
    // On the call's stream: a memset on the legacy default stream is not ordered with a non-blocking
    // caller stream and could land after this call's kernels have written the scratch.
    cudaError_t ez = cudaMemsetAsync(p->solve_buf, 0, Lo.total, (cudaStream_t)stream);
    if (ez != cudaSuccess) return cuda_fail(ez, "zeroing sketch-and-solve scratch");
  }
  p->solve_status_off = Lo.status;
  p->solve_kappa_off = Lo.kappa;
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e = cudaMemsetAsync((char*)p->solve_buf + Lo.status, 0, 4, st);
  if (e != cudaSuccess) return cuda_fail(e, "zeroing status");
  int32_t launches = 0;
  const char* sa = static_cast<const char*>(SAb);
  s = solve_backend(p, sa, ld, sa + es * (size_t)n, ld, n, x, st, di, cap, Lo, &launches);
  if (s != SK_OK) return s;
  p->last_launches = launches;
  return SK_OK;
}

sk_status sk_solve_precond(sk_plan p, const float* A, int64_t lda, int64_t n, const float* b, double* x,
                           int32_t max_iters, double tol, int32_t* iters_out, void* stream) {
  clear_error();
  if (!p) return set_error(SK_ERR_INVALID_ARG, "plan is NULL");
  if (!x) return set_error(SK_ERR_INVALID_ARG, "x is NULL");
  if (n > kLsqrMaxN) return set_error(SK_ERR_UNSUPPORTED, "sketch-and-precondition supports n <= %d", kLsqrMaxN);
  if (max_iters <= 0) max_iters = 100;
  if (!(tol > 0.0)) tol = 1e-10;
  cudaStream_t st = (cudaStream_t)stream;
  // Scratch: u (m doubles), v w y p z x0 (6 n-vectors), scalars, the FP32 sketch-and-solve x0.
  const int64_t m = p->m;
  const size_t nv = (size_t)((n + 31) / 32 * 32);
  const size_t need = sizeof(double) * ((size_t)m + 6 * nv + kLsqrScalars) + sizeof(float) * nv;
  if (p->lsqr_bytes < need) {
    sk_status sg = plan_grow(p, &p->lsqr, &p->lsqr_bytes, need, "sketch-and-precondition scratch");
    if (sg != SK_OK) return sg;
  }
  double* base = p->lsqr;
  float* x0f = reinterpret_cast<float*>(base + m + 6 * nv + kLsqrScalars);
  sk_status s = sk_solve(p, A, lda, n, b, x0f, stream);
  if (s != SK_OK) return s;
  const int64_t solve_launches = p->last_launches;
  s = sk_solve_status(p, nullptr, stream);
  if (s != SK_OK) return s;
  DevInfo di;
  s = dev_info(&di);
  if (s != SK_OK) return s;
  LsqrLaunch L;
  L.A = A;
  L.lda = lda;
  L.m = m;
  L.n = n;
  const SolveLayout Lo = solve_layout(p->d, n, p->rule, 0);  // the offset of R does not depend on the tree
  L.R = reinterpret_cast<const double*>((char*)p->solve_buf + Lo.R);
  L.ldr = n + 1;
  L.X = reinterpret_cast<double*>((char*)p->solve_buf + Lo.part) + n;
  L.u = base;
  L.v = base + m;
  L.w = L.v + nv;
  L.y = L.w + nv;
  L.p = L.y + nv;
  L.z = L.p + nv;
  L.x0 = L.z + nv;
  L.sc = L.x0 + nv;
  L.x = x;
  int32_t launches = (int32_t)solve_launches;
  cudaError_t e = lsqr_start(L, b, x0f, di.sms, st, &launches);
  if (e != cudaSuccess) return cuda_fail(e, "LSQR start");
  double sc[kLsqrScalars];
  int32_t it = 0;
  while (it < max_iters) {
    e = lsqr_iterate(L, di.sms, st, &launches);
    if (e != cudaSuccess) return cuda_fail(e, "LSQR iteration");
    ++it;
    if (it % 4 != 0 && it != max_iters) continue;
    e = cudaMemcpyAsync(sc, L.sc, sizeof(sc), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "LSQR convergence test");
    if (sc[kLsqrDone] != 0.0) break;
    const double anorm = sqrt(sc[kLsqrAnorm2]);
    const double rnorm = sc[kLsqrRnorm], arnorm = sc[kLsqrArnorm];
    if (!std::isfinite(rnorm) || !std::isfinite(arnorm))
      return set_error(SK_ERR_NUMERIC, "LSQR produced a non-finite residual estimate");
    if (rnorm <= tol * sc[kLsqrBnorm] || arnorm <= tol * anorm * rnorm) break;
  }
  e = lsqr_finish(L, st, &launches);
  if (e != cudaSuccess) return cuda_fail(e, "LSQR finish");
  e = cudaMemcpyAsync(sc, L.sc, sizeof(sc), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail(e, "LSQR result");
  if (iters_out) *iters_out = (int32_t)sc[kLsqrIters];
  p->last_launches = launches;
  return SK_OK;
}

sk_status sk_apply_partials(sk_plan p, const float* A, int64_t lda, int64_t n, float* P, int64_t t0, int64_t nchunks,
                            void* stream) {
  clear_error();
  sk_status s = validate_apply(p, A, lda, n, P);
  if (s != SK_OK) return s;
  if ((reinterpret_cast<uintptr_t>(P) & 15u) != 0) return set_error(SK_ERR_INVALID_ARG, "P must be 16-byte aligned");
  if (p->mode != SK_MODE_ATOMIC || p->kernel == SK_KERNEL_LITERAL)
    return set_error(SK_ERR_UNSUPPORTED, "sk_apply_partials runs in atomic mode with a chunked kernel");
  const int64_t R = p->R;
  if (R <= 0)
    return set_error(SK_ERR_INVALID_ARG,
                     "sk_apply_partials needs SK_PARAM_CHUNK_ROWS set (the same on every shard of the matrix)");
  const int64_t tf = p->row_offset / R, tl = (p->row_offset + p->m - 1) / R;
  if (t0 < 0 || nchunks < 1 || tf < t0 || tl >= t0 + nchunks)
    return set_error(SK_ERR_INVALID_ARG, "the plan's chunks [%lld, %lld] are not inside P's chunks [%lld, %lld)",
                     (long long)tf, (long long)tl, (long long)t0, (long long)(t0 + nchunks));
  DevInfo di;
  s = dev_info(&di);
  if (s != SK_OK) return s;
  TileCfg cfg;
  s = choose_tile(p, n, p->m, di, &cfg, tma_layout_ok(A, lda));
  if (s != SK_OK) return s;
  if (cfg.glob) {
    // The global kernel finishes its passes as it goes; partials take the tile kernel instead.
    sk_plan_s tmp = *p;
    tmp.kernel = SK_KERNEL_TILE;
    s = choose_tile(&tmp, n, p->m, di, &cfg, tma_layout_ok(A, lda));
    if (s != SK_OK) return s;
  }
  cfg.R = R;
  if (!cfg.reg && !cfg.gat && cfg.slices < 2) cfg.slices = 2;  // work items flush into the chunk totals
  if (!p->dstatus) {
    size_t cur = 0;
    s = plan_grow(p, &p->dstatus, &cur, sizeof(unsigned), "status word");
    if (s != SK_OK) return s;
  }
  cudaStream_t st = (cudaStream_t)stream;
  if (cudaMemsetAsync(p->dstatus, 0, sizeof(unsigned), st) != cudaSuccess) return cuda_fail(cudaGetLastError(), "zeroing status");
  TileLaunch L;
  L.A = A;
  L.a_type = SK_A_FP32;
  L.Y = nullptr;
  L.lda = lda;
  L.n = n;
  L.row_begin = p->row_offset;
  L.row_end = p->row_offset + p->m;
  L.d = p->d;
  L.k = p->k;
  L.rule = p->rule;
  L.seed = p->seed;
  L.scale = p->scale;
  L.R = R;
  L.NC = cfg.NC;
  L.kb = cfg.kb;
  L.threads = cfg.threads;
  L.grid = cfg.grid;
  L.slices = cfg.slices;
  L.depth = cfg.depth;
  L.mb = cfg.mb;
  L.lr = cfg.lr ? 1 : 0;
  L.own = cfg.own ? 1 : 0;
  L.vec = cfg.vec ? 1 : 0;
  L.glob = 0;
  L.reg = cfg.reg ? 1 : 0;
  L.gat = cfg.gat ? 1 : 0;
  L.reg_nsub = cfg.reg_nsub;
  L.reg_cap = cfg.reg_cap;
  L.col_off = 0;
  L.allow_tma = cfg.vec ? 0 : 1;
  L.status = p->dstatus;
  L.P = P + (tf - t0) * p->d * n;
  L.no_finish = 1;
  int32_t launches = 0;
  cudaError_t e = launch_tile(L, st, &launches);
  if (e != cudaSuccess) return cuda_fail(e, "sketch kernel launch (partials)");
  p->last_noalloc = false;
  p->last_launches = launches;
  p->last_R = R;
  p->last_kernel = cfg.gat ? SK_KERNEL_GATHER : cfg.reg ? SK_KERNEL_REGISTER : cfg.own ? SK_KERNEL_OWNER : SK_KERNEL_TILE;
  return SK_OK;
}

sk_status sk_finish_partials(sk_plan p, float* P, int64_t t0, int64_t nchunks, int64_t n, void* Y, void* stream) {
  clear_error();
  if (!p) return set_error(SK_ERR_INVALID_ARG, "plan is NULL");
  if (!P || !Y) return set_error(SK_ERR_INVALID_ARG, "P and Y must not be NULL");
  if (n < 1 || n > kMaxN) return set_error(SK_ERR_INVALID_ARG, "n=%lld outside [1, %lld]", (long long)n, (long long)kMaxN);
  if (t0 < 0 || nchunks < 1) return set_error(SK_ERR_INVALID_ARG, "need t0 >= 0 and nchunks >= 1");
  if ((reinterpret_cast<uintptr_t>(P) & 15u) != 0) return set_error(SK_ERR_INVALID_ARG, "P must be 16-byte aligned");
  if ((reinterpret_cast<uintptr_t>(Y) & 3u) != 0) return set_error(SK_ERR_INVALID_ARG, "Y must be 4-byte aligned");
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e = cudaMemsetAsync(Y, 0, elem_size(p->rule) * (size_t)(p->d * n), st);
  if (e != cudaSuccess) return cuda_fail(e, "zeroing Y");
  TileDesc D;
  memset(&D, 0, sizeof(D));
  D.Y = Y;
  D.n = n;
  D.seed = p->seed;
  D.scale = p->scale;
  D.B = (uint32_t)p->B;
  D.k = (uint32_t)p->k;
  D.kp = (uint32_t)((p->k + 1) / 2);
  D.col_off = 0;
  D.ldy = 0;
  int32_t launches = 0;
  e = launch_chunk_finish(D, p->rule, P, t0, nchunks, st, &launches);
  if (e != cudaSuccess) return cuda_fail(e, "chunk-finish launch");
  p->last_launches = launches;
  return SK_OK;
}

sk_status sk_solve_status(sk_plan p, double* kappa, void* stream) {
  clear_error();
  if (!p) return set_error(SK_ERR_INVALID_ARG, "plan is NULL");
  if (!p->solve_buf) return set_error(SK_ERR_INVALID_ARG, "no sk_solve has run on this plan");
  cudaStream_t st = (cudaStream_t)stream;
  // One copy of the status word and kappa (adjacent in the scratch layout), ordered on the caller's
  // stream: a copy on the legacy default stream would also wait for unrelated work queued there.
  unsigned status = 0;
  double kap = 0.0;
  const size_t lo = std::min(p->solve_status_off, p->solve_kappa_off);
  const size_t hi = std::max(p->solve_status_off + 4, p->solve_kappa_off + 8);
  unsigned char words[1024];
  cudaError_t e;
  if (hi - lo <= sizeof(words)) {
    e = cudaMemcpyAsync(words, (char*)p->solve_buf + lo, hi - lo, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "reading solve status");
    memcpy(&status, words + (p->solve_status_off - lo), 4);
    memcpy(&kap, words + (p->solve_kappa_off - lo), 8);
  } else {
    e = cudaMemcpyAsync(&status, (char*)p->solve_buf + p->solve_status_off, 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&kap, (char*)p->solve_buf + p->solve_kappa_off, 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "reading solve status");
  }
  if (kappa) *kappa = kap;
  if (status & 1u) return set_error(SK_ERR_TIMEOUT, "a grid barrier of the QR kernel timed out");
  if (status & 2u) return set_error(SK_ERR_NUMERIC, "SA is rank deficient (zero pivot in the QR)");
  return SK_OK;
}

void sk_destroy(sk_plan p) {
  if (!p) return;
  cudaDeviceSynchronize();
  if (p->det_P) cudaFree(p->det_P);
  if (p->dstatus) cudaFree(p->dstatus);
  if (p->tileP) cudaFree(p->tileP);
  if (p->fastP) cudaFree(p->fastP);
  if (p->fast_done) cudaEventDestroy(p->fast_done);
  if (p->lsqr) cudaFree(p->lsqr);
  if (p->solve_buf) cudaFree(p->solve_buf);
  for (int b = 0; b < 2; ++b) {
    if (p->stage[b]) cudaFree(p->stage[b]);
    if (p->ev_copied[b]) cudaEventDestroy(p->ev_copied[b]);
    if (p->ev_used[b]) cudaEventDestroy(p->ev_used[b]);
  }
  if (p->ydev) cudaFree(p->ydev);
  if (p->copy_stream) cudaStreamDestroy(p->copy_stream);
  delete p;
}

}  // extern "C"

namespace sk {

// Tile-kernel launch description for sk_apply_noalloc (sk_noalloc.cu): the same configuration
// sk_apply's atomic tile path chooses, with no scratch attached. Allocates nothing.
// `one_launch`: the caller is to attach the words of a grid barrier (TileLaunch::bar) behind the totals.
sk_status noalloc_tile_launch(const sk_plan_s* p, const float* A, int64_t lda, int64_t n, void* Y, TileLaunch* L,
                              bool* one_launch) {
  *one_launch = false;
  sk_status s = validate_apply(p, A, lda, n, Y);
  if (s != SK_OK) return s;
  if (p->mode != SK_MODE_ATOMIC || p->kernel == SK_KERNEL_LITERAL)
    return set_error(SK_ERR_UNSUPPORTED, "sk_apply_noalloc runs the atomic-mode tile kernel only");
  DevInfo di;
  s = dev_info(&di);
  if (s != SK_OK) return s;
  TileCfg cfg;
  s = choose_tile(p, n, p->m, di, &cfg, tma_layout_ok(A, lda));
  if (s != SK_OK) return s;
  const int64_t chunks = (p->row_offset + p->m - 1) / cfg.R - p->row_offset / cfg.R + 1;
  if (cfg.other && sizeof(float) * (size_t)(chunks * p->d * n) > noalloc_P_bytes()) {
    s = choose_tile(p, n, p->m, di, &cfg, tma_layout_ok(A, lda), SK_A_FP32, false);
    if (s != SK_OK) return s;
  }
  L->A = A;
  L->Y = Y;
  L->lda = lda;
  L->n = n;
  L->row_begin = p->row_offset;
  L->row_end = p->row_offset + p->m;
  L->d = p->d;
  L->k = p->k;
  L->rule = p->rule;
  L->seed = p->seed;
  L->scale = p->scale;
  L->R = cfg.R;
  L->NC = cfg.NC;
  L->kb = cfg.kb;
  L->threads = cfg.threads;
  L->grid = cfg.grid;
  L->slices = cfg.slices;
  // One slice per chunk needs no chunk totals: taken where they would not fit in the static array.
  if (cfg.slices > 1 && cfg.long_slices == 1 && !cfg.glob && !cfg.reg && !cfg.gat) {
    *one_launch = sizeof(float) * (size_t)(launch_P_floats(*L) + kBarrierWords) <= noalloc_P_bytes();
    if (!*one_launch) L->slices = 1;
  }
  L->depth = cfg.depth;
  L->mb = cfg.mb;
  L->lr = cfg.lr ? 1 : 0;
  L->own = cfg.own ? 1 : 0;
  L->vec = cfg.vec ? 1 : 0;
  L->glob = cfg.glob ? 1 : 0;
  L->reg = cfg.reg ? 1 : 0;
  L->gat = cfg.gat ? 1 : 0;
  L->reg_nsub = cfg.reg_nsub;
  L->reg_cap = cfg.reg_cap;
  L->col_off = 0;
  L->allow_tma = 1;
  L->status = nullptr;
  L->P = nullptr;
  return SK_OK;
}

size_t noalloc_elem_size(const sk_plan_s* p) { return elem_size(p->rule); }

void noalloc_record(sk_plan_s* p, int64_t launches, int64_t R, int32_t kernel) {
  p->last_launches = launches;
  p->last_R = R;
  p->last_kernel = kernel;
  p->last_noalloc = true;
}

}  // namespace sk
