// c2f_kernels.cu -- the GB300 kernels of the fire-growth path.
//
//   k_cell_prep / k_hour_prep   hoisted per-cell and per-hour FBP terms
//   k_ros_table   (K1)  per (cell, hour): FBP HROS/BROS/LB, Eqs. (1)-(4), the 8
//                       axis rates as 2^32 fixed-point per-period increments
//   k_ignite      (K2)  Step 1 of Alg. 1: ignition cell per replica
//   k_frontier    (K3)  Step 2 of Alg. 1 for whole replicas: send / receive /
//                       burn-out in windows of fire periods, one warp per replica
//   k_burn_prob   (K4)  burn-probability counts over replicas
//   k_compare_hours / k_compare_final   scar comparison metrics of Sec. 4.1
// plus landscape set-up (burnable bit plane and list) and result export.
//
// Frontier semantics (Sec. 3.1, 3.4, A5; Alg. 1):
//   - a cell ignited in period t advances each open axis from period t+1 by
//     its per-period increment while the neighbour on that axis is Available
//     at the start of the period; when the progress reaches the axis length
//     (the centre-to-centre distance) a message is sent and the axis closes;
//   - a messaged Available cell ignites in that period if HROS * f exceeds
//     the threshold (f: the perturbation of the receiver for the hour);
//   - at the end of a period a burning cell with no Available neighbour, or
//     (delta > 0) with HROS * f < delta, becomes Burned;
//   - the work count adds the number of burning cells at the start of each
//     period.
// The increment of an axis is constant within a weather hour, so within an
// hour the period at which an axis reaches its neighbour's centre is an
// integer function of the progress at the start of the hour; the kernel
// stores that crossing period (as an offset in the hour) instead of adding
// the increment every period, and only visits periods at which something
// happens, several of them at a time.  All progress arithmetic is int64, so the
// crossing periods are the ones the period-by-period loop produces.
#include <cstdint>
#include <mutex>
#include <type_traits>

#include "c2f_fbp.cuh"

namespace c2f {

// host: fill the per-device constant tables (math coefficients, fuel table)
cudaError_t upload_constants() {
  MathConstants mc;
  make_math_constants(&mc);
  FuelCoef ft[F_NCODES];
  make_fuel_table(ft);
  cudaError_t e = cudaMemcpyToSymbol(g_mc, &mc, sizeof mc);
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_fuel, ft, sizeof ft);
  if (e == cudaSuccess) {
    k_math_tables<<<1, 256>>>();
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  return e;
}

// once per device and process, for every entry point that launches kernels
cudaError_t init_device_constants(int device) {
  static std::once_flag once[64];
  static cudaError_t err[64];
  if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
  std::call_once(once[device], [device] { err[device] = upload_constants(); });
  return err[device];
}

// axis k = 0..7 at 45 k degrees counter-clockwise from east: (row, col) offsets
// E (0,+1), NE (-1,+1), N (-1,0), NW (-1,-1), W (0,-1), SW (+1,-1), S (+1,0), SE (+1,+1),
// kept as offset + 1 in the nibbles of one immediate: lanes index them with
// different k, which a __constant__ table would serve one address at a time
__device__ __forceinline__ int axis_dr(int k) { return (int)((0x22210001u >> (4 * k)) & 0xFu) - 1; }
__device__ __forceinline__ int axis_dc(int k) { return (int)((0x21000122u >> (4 * k)) & 0xFu) - 1; }

// bit 0 of each byte of x, gathered into bits 0..3 (byte 0 -> bit 0)
__device__ __forceinline__ uint32_t byte_lsbs(uint32_t x) {
  return (((x & 0x01010101u) * 0x00204081u) >> 21) & 0xFu;
}

// ------------------------------------------------------------------ set-up
// burnable plane (bit per cell, rows padded to 32-bit words) and per-word counts
__global__ void k_burnable_plane(const uint8_t *__restrict__ fuel, const uint8_t *__restrict__ unb,
                                 int32_t rows, int32_t cols, int32_t wpr, uint32_t *plane,
                                 int32_t *word_count) {
  const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= (int64_t)rows * wpr) return;
  const int32_t row = (int32_t)(w / wpr), cw = (int32_t)(w % wpr);
  uint32_t bits = 0;
  for (int b = 0; b < 32; ++b) {
    const int32_t col = cw * 32 + b;
    if (col >= cols) break;
    const int64_t cell = (int64_t)row * cols + col;
    const bool ok = fuel[cell] != 0 && !(unb && unb[cell]);
    bits |= (ok ? 1u : 0u) << b;
  }
  plane[w] = bits;
  word_count[w] = __popc(bits);
}

// exclusive scan of the per-word counts, one block (set-up only)
__global__ void k_scan_counts(const int32_t *__restrict__ cnt, int64_t n, int32_t *offs,
                              int32_t *total) {
  __shared__ int32_t s_part[1024];
  const int t = threadIdx.x, T = blockDim.x;
  const int64_t per = (n + T - 1) / T;
  const int64_t b = per * t, e = (b + per < n) ? b + per : n;
  int32_t acc = 0;
  for (int64_t i = b; i < e; ++i) acc += cnt[i];
  s_part[t] = acc;
  __syncthreads();
  if (t == 0) {
    int32_t run = 0;
    for (int i = 0; i < T; ++i) { const int32_t v = s_part[i]; s_part[i] = run; run += v; }
    *total = run;
  }
  __syncthreads();
  int32_t run = s_part[t];
  for (int64_t i = b; i < e; ++i) { offs[i] = run; run += cnt[i]; }
}

__global__ void k_burnable_list(const uint32_t *__restrict__ plane, const int32_t *__restrict__ offs,
                                int32_t rows, int32_t cols, int32_t wpr, int32_t *list) {
  const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= (int64_t)rows * wpr) return;
  const int32_t row = (int32_t)(w / wpr), cw = (int32_t)(w % wpr);
  uint32_t bits = plane[w];
  int32_t o = offs[w];
  while (bits) {
    const int b = __ffs(bits) - 1;
    bits &= bits - 1;
    list[o++] = row * cols + cw * 32 + b;
  }
}

// ------------------------------------------------------------------ K1 prep
__global__ void k_cell_prep(const float *__restrict__ slope, const float *__restrict__ aspect,
                            int64_t n, CellPrep *out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  CellPrep cp;
  cell_prep(slope ? (double)slope[i] : 0.0, aspect ? (double)aspect[i] : 0.0, &cp);
  out[i] = cp;
}

// 16 threads per hour, one per fuel code: weather-only terms
__global__ void k_hour_prep(const double *__restrict__ weather, int32_t hours, double o1_curing,
                            HourPrep *out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int h = min(t >> 4, hours - 1);   // the last block's spare threads repeat the last hour
  const double *w = weather + (size_t)h * 4;
  hour_prep(t & 15, w[0], w[1], w[2], w[3], curing_factor(o1_curing), &out[h]);
}

// ------------------------------------------------------------------ K1

// Cells grouped by (fuel code, slope > 0) so that the lanes of a warp take the
// same branches of the FBP code (set-up, once per landscape): a per-bucket
// count, an exclusive scan, then a scatter; the order inside a bucket is
// immaterial because every cell writes its own table row.
__device__ __forceinline__ int order_bucket(const uint8_t *fuel, const float *slope,
                                            const uint32_t *burnable, int32_t cols, int32_t wpr,
                                            int64_t cell) {
  const int32_t row = (int32_t)(cell / cols), col = (int32_t)(cell % cols);
  const bool burn = (burnable[(int64_t)row * wpr + (col >> 5)] >> (col & 31)) & 1u;
  if (!burn) return 0;
  const bool sloped = slope && slope[cell] > 0.0f;
  return 2 * (int)fuel[cell] + (sloped ? 1 : 0);
}

__global__ void k_order_count(const uint8_t *fuel, const float *slope, const uint32_t *burnable,
                              int32_t rows, int32_t cols, int32_t wpr, int32_t *counts) {
  __shared__ int32_t h[kOrderBuckets];
  if (threadIdx.x < kOrderBuckets) h[threadIdx.x] = 0;
  __syncthreads();
  const int64_t cell = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (cell < (int64_t)rows * cols)
    atomicAdd(&h[order_bucket(fuel, slope, burnable, cols, wpr, cell)], 1);
  __syncthreads();
  if (threadIdx.x < kOrderBuckets && h[threadIdx.x]) atomicAdd(&counts[threadIdx.x], h[threadIdx.x]);
}

__global__ void k_order_scan(int32_t *counts_to_cursor) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    int32_t run = 0;
    for (int b = 0; b < kOrderBuckets; ++b) {
      const int32_t c = counts_to_cursor[b];
      counts_to_cursor[b] = run;
      run += c;
    }
  }
}

__global__ void k_order_scatter(const uint8_t *fuel, const float *slope, const uint32_t *burnable,
                                int32_t rows, int32_t cols, int32_t wpr, int32_t *cursor,
                                int32_t *order) {
  __shared__ int32_t h[kOrderBuckets], base[kOrderBuckets];
  if (threadIdx.x < kOrderBuckets) h[threadIdx.x] = 0;
  __syncthreads();
  const int64_t cell = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int b = -1, local = 0;
  if (cell < (int64_t)rows * cols) {
    b = order_bucket(fuel, slope, burnable, cols, wpr, cell);
    local = atomicAdd(&h[b], 1);
  }
  __syncthreads();
  if (threadIdx.x < kOrderBuckets && h[threadIdx.x]) base[threadIdx.x] = atomicAdd(&cursor[threadIdx.x], h[threadIdx.x]);
  __syncthreads();
  if (b >= 0) order[base[b] + local] = (int32_t)cell;
}

// the 8 axis rates and HROS of one burnable cell at one hour
// (const_ros > 0: the deterministic test rates -- all 8 axes at const_ros, or,
// with const_bros > 0 or const_lb > 1, the ellipse of HROS = const_ros,
// BROS = const_bros (0: const_ros), LB = const_lb headed along the hour's wind)
template <bool INTS>
__device__ __forceinline__ void row_rates(int fuel, const float *slope, int64_t cell,
                                          const CellPrep &cp, const HourPrep &hp, double pcf,
                                          double const_ros, double const_bros, double const_lb,
                                          int ellipse_mode, AxisRates *o) {
  if (pos(const_ros)) {
    if (pos(const_bros) || gt_c(const_lb, 1.0)) {
      ellipse_axes<INTS>(const_ros, pos(const_bros) ? const_bros : const_ros, gt_c(const_lb, 1.0) ? const_lb : 1.0,
                   hp.sin_w, hp.cos_w, ellipse_mode, o);
      return;
    }
    o->hros = const_ros;
    o->paired = false;
#pragma unroll
    for (int k = 0; k < 8; ++k) o->ros[k] = const_ros;
    return;
  }
  fbp_row<INTS>(fuel, slope ? (double)slope[cell] : 0.0, cp, hp, pcf, ellipse_mode, o);
}

// a table row: the 8 per-period increments B_k = fixed(ros_k * dt * 2^32) in one
// 64-byte line (four 16-byte stores), HROS beside it in its own array
__device__ __forceinline__ void row_store(int64_t *row, double *hros_at, const AxisRates &o, double dt2p32) {
  const PeriodScale fixed(dt2p32);
  int64_t v[8];
  if (o.paired) {
    const int64_t back = fixed(o.back);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int64_t ahead = fixed(o.ros[j]);
      const bool behind = (o.behind >> j) & 1u;
      v[j] = behind ? back : ahead;
      v[j + 4] = behind ? ahead : back;
    }
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = fixed(o.ros[k]);
  }
  longlong2 *dst = reinterpret_cast<longlong2 *>(row);
#pragma unroll
  for (int k = 0; k < 8; k += 2) dst[k / 2] = make_longlong2(v[k], v[k + 1]);
  *hros_at = o.hros;
}

// nanoseconds of the GPU's global timer
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// one launch-trace record (c2f_trace); records past the capacity are counted, not written
__device__ __forceinline__ void trace_record(const TraceArgs &tr, uint32_t kind, uint32_t aux, long long tag,
                                             unsigned long long t0, unsigned long long t1) {
  const unsigned long long i = atomicAdd(tr.cursor, 1ull);
  if (i < (unsigned long long)tr.cap) {
    uint32_t smid;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
    unsigned long long *p = tr.rec + 4 * i;
    p[0] = (unsigned long long)kind | ((unsigned long long)smid << 8) | ((unsigned long long)aux << 32);
    p[1] = (unsigned long long)tag;
    p[2] = t0;
    p[3] = t1;
  }
}

__global__ void __launch_bounds__(128) k_ros_table(RosTableArgs a) {
  const int64_t n = (int64_t)a.rows * a.cols;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool traced = a.trace.rec != nullptr && threadIdx.x == 0;   // thread 0 stands for its CTA
  const unsigned long long t_start = traced ? global_ns() : 0ull;
  if (t >= n) return;
  const int64_t cell = a.order ? (int64_t)a.order[t] : t;
  const int h = a.hour0 + blockIdx.y;
  const int32_t row = (int32_t)(cell / a.cols), col = (int32_t)(cell % a.cols);
  const bool burn = (a.burnable[(int64_t)row * a.wpr + (col >> 5)] >> (col & 31)) & 1u;
  const size_t idx = (size_t)h * n + cell;
  AxisRates o;
  if (burn) {
    row_rates<true>(a.fuel[cell], a.slope, cell, a.cell[cell], a.hour[h], a.pcf, a.const_ros, a.const_bros, a.const_lb,
              a.ellipse_mode, &o);
    if (a.base) row_store(a.base + idx * 8, a.hros + idx, o, a.dt2p32);
  } else if (a.base) {
    longlong2 *dst = reinterpret_cast<longlong2 *>(a.base + idx * 8);
#pragma unroll
    for (int k = 0; k < 4; ++k) dst[k] = make_longlong2(0, 0);
    a.hros[idx] = 0.0;
  }
  if (a.ros8) {
#pragma unroll
    for (int k = 0; k < 8; ++k) a.ros8[(size_t)cell * 8 + k] = burn ? o.of(k) : 0.0;
  }
  if (traced) trace_record(a.trace, kTraceTable, (uint32_t)h, a.trace.tag, t_start, global_ns());
}

// ------------------------------------------------------------------ K2
__global__ void k_ignite(const SimJob *jobs, int32_t job) {
  const SimJob &J = jobs[job];
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= J.n_replicas) return;
  int32_t ic = J.ignition_cell;
  if (J.ignition_mode == 1) {
    const U4 x = philox4x32_10(U4{(uint32_t)r, 0u, 0u, 1u}, (uint32_t)J.seed,
                               (uint32_t)(J.seed >> 32));
    const uint64_t idx = ((uint64_t)x.x * (uint64_t)(uint32_t)J.n_burnable) >> 32;
    ic = J.burnable_list[idx];
  }
  J.ign_cell[r] = ic;
  if (J.n_scen > 1) {   // Sec. 3.1 (3): the first s with x0 < T_s, x0 from counter (r, 0, 0, 2)
    const U4 x = philox4x32_10(U4{(uint32_t)r, 0u, 0u, 2u}, (uint32_t)J.seed,
                               (uint32_t)(J.seed >> 32));
    int32_t s = 0;
    while (s < J.n_scen - 1 && (uint64_t)x.x >= J.scen_thr[s]) ++s;
    J.scen[r] = s;
  }
}

// ------------------------------------------------------------------ K3
// the least byte (16-bit minima: bytewise ones are emulated on this GPU)
__device__ __forceinline__ uint32_t min_byte8(uint64_t v) {
  const uint32_t lo = (uint32_t)v, hi = (uint32_t)(v >> 32), m8 = 0x00FF00FFu;
  const uint32_t m = __vminu2(__vminu2(lo & m8, (lo >> 8) & m8), __vminu2(hi & m8, (hi >> 8) & m8));
  return min(m & 0xFFFFu, m >> 16);
}

// The number of periods n <= nmax <= 60 after which an axis with rem > 0 to go
// reaches its neighbour's centre at inc a period (the smallest n >= 1 with
// n * inc >= rem), or 0 if it takes more; rem and inc are below 2^(31 + shift).
// A binary32 estimate of the quotient from the top bits, never more than its
// ceiling (inc is rounded up), then one exact int64 step; it falls short by two
// or more only when inc has few top bits, i.e. for the last few units of a
// nearly finished axis.
__device__ __forceinline__ int32_t periods_to_cross(int64_t rem, int64_t inc, int32_t nmax, int shift) {
  const bool in_time = inc > 0 && inc * nmax >= rem;
  const float a = (float)(uint32_t)((uint64_t)rem >> shift), b = (float)((uint32_t)((uint64_t)inc >> shift) + 1u);
  int32_t n = in_time ? (int32_t)__fdividef(a, b) : 0;
  int64_t left = rem - (int64_t)((uint64_t)(uint32_t)n * (uint64_t)inc);
  n += left > 0 ? 1 : 0;
  left -= inc;
  while (in_time && left > 0) { ++n; left -= inc; }
  return in_time ? n : 0;
}

// The frontier's two binary64 tests are kept out of line: inlined, the
// compiler issues their FP64 instructions (predicated off) in every round and
// set-up pass even when no threshold or delta is set, and each of them waits
// for the FP64 pipe, which a table build running beside the frontier keeps
// busy.  Called only when a threshold (receive) or a delta (burn-out) is set.

// receive test of a messaged Available cell (Sec. 3.1): HROS * f > threshold
__device__ __noinline__ bool receive_ok(const SimJob &J, int32_t r, int64_t j, int32_t h, int64_t n) {
  if (J.thr < 0.0) return true;
  const double hr = __ldcg(J.hros + (size_t)h * n + j);
  if (J.thr == 0.0) {
    if (hr > 1e-200) return true;   // f >= exp(-5.9) for sigma <= 1, so HROS * f > 0
    if (!(hr > 0.0)) return false;
  }
  const float f = noise_factor(J.seed, (uint32_t)r, (uint32_t)j, (uint32_t)h, J.sigma);
  return __dmul_rn(hr, (double)f) > J.thr;
}

// A5 (i): the cell's HROS * f this hour is below delta
__device__ __noinline__ bool below_delta(const double *hrosh, int64_t cell, float f, double delta) {
  return __dmul_rn(__ldcg(hrosh + cell), (double)f) < delta;
}

__device__ __forceinline__ int64_t find_job(const int64_t *begin, int32_t n, int64_t item) {
  int32_t lo = 0, hi = n - 1;
  while (lo < hi) {
    const int32_t mid = (lo + hi + 1) >> 1;
    if (begin[mid] <= item) lo = mid; else hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ uint32_t warp_min(uint32_t v) {
  return __reduce_min_sync(0xffffffffu, v);   // one warp-wide reduction instruction
}

__device__ __forceinline__ uint32_t rc_pack(int32_t r, int32_t c) {
  return ((uint32_t)r << 16) | (uint32_t)c;
}

// a table row into L2 ahead of its use
__device__ __forceinline__ void prefetch_l2(const void *p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// chunk state, read at device scope from L2.  A relaxed load suffices: a warp
// reads a chunk's rows (with L2 loads, __ldcg) only after a branch on the
// state it loaded has resolved, and the computing warp made its rows visible
// device-wide (__threadfence) before it set the state.  An acquire load would
// also invalidate the SM's L1 on every check.
__device__ __forceinline__ uint32_t ld_state(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// waits for a table chunk that another warp is computing give up after
// FrontierArgs::wait_limit polls (this many when it is 0: about a second);
// the replica then stops with status 4 (a bounded wait ran out)
constexpr uint32_t kChunkSpinLimit = 1u << 23;

// On-demand table rows: the rows at hour h of the 32 cells of bit-plane word w
// (one lane per cell, all 32 lanes of the warp), then the chunk's state goes
// to done once every lane's stores are visible device-wide.
__device__ __forceinline__ void table_chunk(const SimJob &J, int32_t h, int32_t w) {
  const int lane = threadIdx.x & 31;
  const int32_t row = w / J.wpr, cw = w - row * J.wpr;
  const int32_t col = cw * 32 + lane;
  if (col < J.cols && ((__ldg(&J.burnable[w]) >> lane) & 1u)) {
    const int64_t n = (int64_t)J.rows * J.cols;
    const int64_t cell = (int64_t)row * J.cols + col;
    AxisRates o;
    row_rates<false>(__ldg(&J.fuel[cell]), J.slope, cell, J.cell[cell], J.hour[h], J.pcf, J.const_ros, J.const_bros,
              J.const_lb, J.ellipse_mode, &o);
    const size_t idx = (size_t)h * n + cell;
    row_store(J.base + idx * 8, J.hros + idx, o, J.dt2p32);
  }
  __threadfence();
  __syncwarp();
  if (lane == 0) atomicExch(J.chunk_state + (size_t)h * J.rows * J.wpr + w, 2u);
  __syncwarp();
}

// A SIZE x SIZE block of an Available plane from (r, c) on, row by row of SIZE
// bits, that crosses the window's or the grid's edges or lies outside the
// window (sav: the window from row r0, word w0 on, or nullptr; cells outside
// the grid are 0).  Out of line: a warp's path through the frontier is long,
// and with several warps on a scheduler a fifth of its time went into
// instruction fetches.
template <int SIZE>
__device__ __noinline__ uint32_t block_at_edge(const uint32_t *sav, const uint32_t *gav, int32_t r0, int32_t w0,
                                               int32_t rows, int32_t wpr, int32_t r, int32_t c) {
  const int32_t wl = c >> 5, wh = (c + SIZE - 1) >> 5;
  const bool lo_in = sav != nullptr && (uint32_t)(wl - w0) < (uint32_t)kWinWords;
  const bool hi_in = sav != nullptr && (uint32_t)(wh - w0) < (uint32_t)kWinWords;
  uint32_t lo[SIZE], hi[SIZE];
#pragma unroll
  for (int d = 0; d < SIZE; ++d) {
    const int32_t rr = r + d;
    const bool grid = rr >= 0 && rr < rows, win = (uint32_t)(rr - r0) < (uint32_t)kWinRows;
    lo[d] = hi[d] = 0u;
    if (grid && wl >= 0) lo[d] = win && lo_in ? sav[(rr - r0) * kWinWords + (wl - w0)] : gav[rr * wpr + wl];
    if (grid && wh < wpr) hi[d] = win && hi_in ? sav[(rr - r0) * kWinWords + (wh - w0)] : gav[rr * wpr + wh];
  }
  uint32_t v = 0u;
#pragma unroll
  for (int d = 0; d < SIZE; ++d)
    v |= (__funnelshift_r(lo[d], hi[d], (uint32_t)c & 31u) & ((1u << SIZE) - 1u)) << (d * SIZE);
  return v;
}

// The replica's Available bit plane, and with A5 (i) on a plane of the cells
// that burned out by it.  With WIN, a window of kWinRows x (32 kWinWords)
// cells of the Available plane around the ignition cell lives in shared
// memory and the rest of the grid in global memory; without it, all in global
// memory.  In global memory the plane holds only the rows [g0, g1) that the
// fire can reach, or look at, by the end of the hour (reach()); the others are
// the burnable plane's.  (Copying all of it at the start cost a replica of a
// 4096 x 4096 landscape 2.7 of its 8.3 ms.)  A cell burned out by A5 (ii) needs no bit of its own: it is one
// that ignited and has no Available neighbour.
template <bool WIN>
struct Planes {
  uint32_t *sav;         // shared-memory window
  uint32_t *gav, *gbr;   // full planes, global memory
  const uint32_t *burnable;
  int32_t r0, w0, rows, wpr, g0, g1;
  __device__ __forceinline__ bool in_win(int32_t r, int32_t w) const {
    if constexpr (WIN) return (uint32_t)(r - r0) < (uint32_t)kWinRows && (uint32_t)(w - w0) < (uint32_t)kWinWords;
    else return false;
  }
  // copies [i, end) of the burnable plane into the global Available plane
  // (one warp, eight loads in flight)
  __device__ __forceinline__ void fill(int32_t i, int32_t end, int lane) const {
    for (i += lane; i + 7 * 32 < end; i += 8 * 32) {
      uint32_t v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = __ldg(&burnable[i + 32 * j]);
#pragma unroll
      for (int j = 0; j < 8; ++j) gav[i + 32 * j] = v[j];
    }
    for (; i < end; i += 32) gav[i] = __ldg(&burnable[i]);
  }
  // makes the global rows hold those of rows [ra, rb], columns [ca, cb] and
  // `far` around them, unless all of that lies in the window (whole warp)
  __device__ __forceinline__ void reach(int32_t ra, int32_t rb, int32_t ca, int32_t cb, int32_t far, int lane) {
    ra = max(ra - far, 0);
    rb = min(rb + far + 1, rows);
    if constexpr (WIN) {
      if (ra >= r0 && rb <= r0 + kWinRows && max(ca - far, 0) >> 5 >= w0 && min((cb + far) >> 5, wpr - 1) < w0 + kWinWords)
        return;   // all in the window
    }
    if (g0 == g1) g0 = g1 = ra;   // none yet
    if (ra < g0) {
      fill(ra * wpr, g0 * wpr, lane);
      g0 = ra;
    }
    if (rb > g1) {
      fill(g1 * wpr, rb * wpr, lane);
      g1 = rb;
    }
    __syncwarp();
  }
  // ignition: clears the Available bit
  __device__ __forceinline__ void take(int32_t r, int32_t c) const {
    const uint32_t bit = 1u << (c & 31);
    const int32_t w = c >> 5;
    if (in_win(r, w)) atomicAnd(sav + (r - r0) * kWinWords + (w - w0), ~bit);
    else atomicAnd(gav + r * wpr + w, ~bit);
  }
  // the (2 D + 1) x (2 D + 1) block of Available bits around (r, c), one row
  // per element, bit j = column c - D + j; cells outside the grid are 0.  The
  // common case lies in the window (without one: away from the grid's edges): a
  // row comes out of two adjacent words by one funnel shift (bits past the last
  // column and rows past the last one are 0 there)
  template <int D>
  __device__ __forceinline__ void block(int32_t r, int32_t c, uint32_t b[2 * D + 1]) const {
    constexpr uint32_t mask = (1u << (2 * D + 1)) - 1u;
    const uint32_t sh = (uint32_t)(c - D) & 31u;
    const int32_t wl = (c - D) >> 5, wh = (c + D) >> 5;
    const uint32_t *p;
    int32_t step;
    bool inside;
    if constexpr (WIN) {
      inside = (uint32_t)(r - D - r0) < (uint32_t)(kWinRows - 2 * D) && wl >= w0 && wh < w0 + kWinWords;
      p = sav + (r - D - r0) * kWinWords - w0;
      step = kWinWords;
    } else {
      inside = r >= D && r + D < rows && wl >= 0 && wh < wpr;
      p = gav + (r - D) * wpr;
      step = wpr;
    }
    if (inside) {
#pragma unroll
      for (int d = 0; d < 2 * D + 1; ++d) b[d] = __funnelshift_r(p[d * step + wl], p[d * step + wh], sh) & mask;
    } else {
      const uint32_t v = block_at_edge<2 * D + 1>(WIN ? sav : nullptr, gav, WIN ? r0 : 0, WIN ? w0 : 0, rows, wpr, r - D, c - D);
#pragma unroll
      for (int d = 0; d < 2 * D + 1; ++d) b[d] = (v >> (d * (2 * D + 1))) & mask;
    }
  }
  // A5 (i): has (r, c) burned out by it / the first to mark it so
  __device__ __forceinline__ bool burned(int32_t r, int32_t c) const { return (gbr[r * wpr + (c >> 5)] >> (c & 31)) & 1u; }
  __device__ __forceinline__ bool burn(int32_t r, int32_t c) const {
    const uint32_t bit = 1u << (c & 31);
    return (atomicOr(gbr + r * wpr + (c >> 5), bit) & bit) == 0;
  }
};

// three 3-bit rows around a cell (bit j = column c - 1 + j) as the 8 axes' mask, bit k = axis k
__device__ __forceinline__ uint32_t axes_of_rows(uint32_t up, uint32_t mid, uint32_t dn) {
  return ((mid >> 2) & 1u) | ((__brev(up) >> 28) & 0xEu) | ((mid & 1u) << 4) | ((dn & 7u) << 5);
}

// The bytes of an entry's crossing offsets: 0..sph-1 the offset in the hour
// at which that axis reaches its neighbour's centre, kOpen an open axis with
// no crossing this hour, kNone a closed axis (message sent, or the neighbour
// was not Available when the axis was set up)
constexpr uint32_t kOpen = 0xFEu;

// the open axes of an entry (bytes that are not kNone) as an 8-bit mask
__device__ __forceinline__ uint32_t open_axes(uint64_t c8) {
  // a byte is below 64, 0xFE or 0xFF: closed iff bits 7 and 0 are both set
  const uint32_t lo = (uint32_t)c8, hi = (uint32_t)(c8 >> 32);
  return ~(byte_lsbs((lo >> 7) & lo) | (byte_lsbs((hi >> 7) & hi) << 4)) & 0xFFu;
}

// the bytes of x below e (e <= 60), as the top bits of the bytes: an offset is
// below 64, so (byte | 0x80) - e borrows from no neighbour and keeps its top
// bit unless the byte is an offset below e
__device__ __forceinline__ uint32_t msb_below(uint32_t x, uint32_t e) {
  return ~((x | 0x80808080u) - e * 0x01010101u) & 0x80808080u;
}

// the axes of an entry that cross before offset e, as an 8-bit mask
__device__ __forceinline__ uint32_t bytes_below(uint64_t c8, uint32_t e) {
  return byte_lsbs(msb_below((uint32_t)c8, e) >> 7) | (byte_lsbs(msb_below((uint32_t)(c8 >> 32), e) >> 7) << 4);
}

// a 4-bit mask as bytes: 0xFF where the bit is set
__device__ __forceinline__ uint32_t bytes_of(uint32_t m) { return ((m & 0xFu) * 0x00204081u & 0x01010101u) * 0xFFu; }

// entries that a window is made long enough for (of the 64 it can hold, by the
// density of crossings in the last window): about 0.7 crossings an entry lead
// to Available cells, and a window handles 32
constexpr int32_t kWindowFill = 44;

// 16 bytes of global memory into shared memory, asynchronously, through L2
// only (a lazy table's rows may have been written by another SM)
__device__ __forceinline__ void copy_async16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
               ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Chunks of on-demand table rows that a frontier warp hands to its CTA's
// helper warps: n chunks of hour h of job *job (n < 0: no more will come).
struct ChunkWork {
  const SimJob *job;
  int32_t h, n, chunk[32];
};
__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
// a helper warp (wib = 1 .. helpers): waits at barrier 1 for chunks, computes
// every (helpers + 1)-th of them from its own number on, meets at barrier 2
template <int HELPERS>
__device__ __forceinline__ void help_with_chunks(const ChunkWork *work) {
  constexpr int kThreads = 32 * (HELPERS + 1);
  for (;;) {
    bar_sync(1, kThreads);
    const int32_t n = work->n;
    if (n < 0) return;
    for (int32_t i = threadIdx.x >> 5; i < n; i += HELPERS + 1) table_chunk(*work->job, work->h, work->chunk[i]);
    bar_sync(2, kThreads);
  }
}

// One warp per replica; replicas come from a work list of (simulation,
// replica) items that every warp pulls from.  There is no CTA barrier: the
// warp's counters stay in registers, appends to the burning list are placed
// by ballot + popc, and phases are ordered with __syncwarp.  Per replica: an
// Available plane (burnable, not harvested, not yet ignited); with WIN its
// window around the ignition cell and the burning-list arrays sit in shared
// memory.  The scar plane (burnable and no longer Available) is written at
// the end.
//
// Within an hour every axis crosses at a known offset.  The warp advances by
// windows of consecutive periods [o1, E): no cell that ignites in a window
// sends before the window's end, so all its crossings are known at its start
// and are handled at once.  o1 is the lowest bit of a 64-bit calendar mask of
// the offsets at which some entry crosses; E is found as the window is worked
// out:
//   A1  the entries whose earliest crossing lies in [o1, o1 + width), by a
//       scan of one byte per entry, four to a word, 32 words at a time;
//   A2  their crossings in the window towards Available cells, one per lane,
//   A3  ranked by offset; a cell reached several times ignites at the first;
//   C1  lane i takes the i-th cell to ignite: table row into shared memory
//       (asynchronously), perturbation;
//   C2  one open axis of the new cells per lane: the offset at which it sends,
//       or its progress to the end of the hour;
//   C3  E = the earliest of these offsets (at most o1 + width); the cells that
//       ignite before E are taken and listed (the others stay Available and
//       their crossings open); cells with no Available neighbour left burn
//       out at the last ignition next to them;
//   C4  the crossings before E are closed.
// Every window is at least one period long (a cell sends after the period in
// which it ignites).  width follows the density of crossings and what the last
// window reached.
//
// What bounds it: a replica is one dependent chain, so with few replicas a
// warp's instruction count times some five cycles an instruction, and with a
// dozen warps on an SM the instruction fetches of the long path (hence loops
// and out-of-line edges rather than unrolled code).  One period at a time, a
// replica of the 512 x 512 landscape (24 h) issued some 980 instructions in each
// of its 1,090 visited periods, most of them in passes that few lanes had work
// for; a window holds 5 to 6 periods there, 25 entries, 18 crossings and 15 new
// cells.  1,000 replicas: 4.42 ms one period at a time, 2.02 to 2.29 ms now;
// 64 replicas 1.96 ms.  Where a period takes dozens of windows (uniform fuel at a
// constant rate: rings of hundreds of cells), scanning the list from its start
// and compacting it before every window would grow with its square: 4 replicas,
// 1500 x 1500 at 60 m/min for 24 h: 3.63 s so, 0.66 s with scan0 and room below
// (one period at a time: 1.32 s); 2,000 replicas, 200 x 200 at 99: 113, 29 (81) ms.
//
// HELPERS warps of the CTA beside the frontier's own only compute on-demand
// table rows (with WPC = 1; `work` in shared memory).
template <int WPC, bool WIN, bool LAZY, bool PROF, int HELPERS = 0>
__device__ __forceinline__ void frontier_warp(const FrontierArgs &A, ChunkWork *work = nullptr) {
  extern __shared__ __align__(16) uint32_t s_dyn[];
  __shared__ SimJob s_job[WPC];
  constexpr uint32_t FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int k = lane & 7, grp = lane >> 3;   // four cells at a time: lane k of group grp looks at axis k
  const uint32_t lt = (1u << lane) - 1u;
  const size_t slot = (size_t)blockIdx.x * WPC + wib;
  const int32_t cap = A.cap;
  // compact the list within an hour once it holds more than this many entries
  const int32_t compact_at = (A.compact_at > 0 && A.compact_at < cap) ? A.compact_at : cap - cap / 4;
  const uint32_t wait_limit = A.wait_limit ? A.wait_limit : kChunkSpinLimit;
  uint32_t *my = s_dyn + (size_t)wib * A.smem_warp_words;   // [Available window][lists]
  uint32_t *erc;     // row << 16 | col
  uint8_t *ecofs;    // 8 crossing-offset bytes per entry
  uint8_t *enx;      // the entry's earliest crossing (the least of its 8 bytes)
  Planes<WIN> pl;
  pl.gav = A.avail_scratch + slot * (size_t)A.pw_max;
  pl.gbr = A.brn_scratch + slot * (size_t)A.pw_max;
  if constexpr (WIN) {
    pl.sav = my;
    uint32_t *ls = my + kWinRows * kWinWords;
    ecofs = reinterpret_cast<uint8_t *>(ls);
    erc = ls + 2 * (size_t)cap;
    enx = reinterpret_cast<uint8_t *>(ls + 3 * (size_t)cap);
  } else {
    pl.sav = nullptr;
    erc = reinterpret_cast<uint32_t *>(A.ent_cell) + slot * cap;
    ecofs = A.ent_cofs + slot * (size_t)cap * 8;
    enx = A.ent_next + slot * (size_t)((cap + 3) & ~3);
  }
  int64_t *eP = A.ent_P + slot * (size_t)cap * 8;
  __shared__ __align__(16) int64_t s_rows[WPC][32 * 8];   // table rows of 32 cells
  __shared__ __align__(16) int64_t s_prg[WPC][32 * 8];    // hour boundary: their progress
  __shared__ int32_t s_qent[WPC][64];                     // hour boundary: kept entries
  __shared__ uint8_t s_qam[WPC][64];                      // and their open axes
  __shared__ int32_t s_went[WPC][64];                     // a window's entries
  __shared__ uint8_t s_wleft[WPC][64];                    // and their crossings that found no lane
  __shared__ uint32_t s_buf[WPC][32];                     // crossings, new cells, burn-outs
  __shared__ uint8_t s_off[WPC][32];                      // the new cells' offsets
  __shared__ uint8_t s_items[WPC][256];                   // cell (lane) | axis << 5 items of 32 cells
  __shared__ uint32_t s_dbits[WPC][LAZY ? kWinRows * kWinWords / 32 : 1];   // chunks known done this hour
  __shared__ int32_t s_claim[WPC][LAZY ? 32 : 1];
  __shared__ long long s_prof[WPC][PROF ? kProfCounters : 1];
  int64_t *rowbuf = s_rows[wib], *prgbuf = s_prg[wib];
  int32_t *qent = s_qent[wib];
  uint8_t *qam = s_qam[wib];
  uint32_t *buf = s_buf[wib];
  uint8_t *ibuf = s_items[wib];
  int32_t *went = s_went[wib];
  uint8_t *wleft = s_wleft[wib];
  uint8_t *obuf = s_off[wib];
  uint32_t *dbits = s_dbits[wib];
  int32_t *claim = HELPERS > 0 ? work->chunk : s_claim[wib];
  SimJob &J = s_job[wib];

  for (;;) {
    long long item = -1;
    int32_t jidx = 0;
    if (lane == 0) {
      const unsigned long long i = atomicAdd(A.counter, 1ull);
      if ((int64_t)i < A.n_items) {
        item = A.item_list ? A.item_list[i] : (long long)i;
        jidx = (int32_t)find_job(A.item_begin, A.n_jobs, item);
        J = A.jobs[jidx];
        if (J.n_scen > 1) {   // this replica's scenario: its stacked table
          const int64_t s = J.scen[item - A.item_begin[jidx]];
          const int64_t n = (int64_t)J.rows * J.cols;
          J.base += s * J.scen_hours * n * 8;
          J.hros += s * J.scen_hours * n;
          J.hour += s * J.prep_hours;
          if (J.chunk_state) J.chunk_state += s * J.scen_hours * J.rows * J.wpr;
        }
      }
    }
    item = __shfl_sync(FULL, item, 0);
    jidx = __shfl_sync(FULL, jidx, 0);
    __syncwarp();
    if (item < 0) return;
    const unsigned long long t_start = A.trace.rec ? global_ns() : 0ull;
    const int32_t r = (int32_t)(item - A.item_begin[jidx]);
    const int32_t rows = J.rows, cols = J.cols, wpr = J.wpr;
    const int64_t n = (int64_t)rows * cols;
    const int32_t pw = rows * wpr;
    const int32_t sph = J.sph, H = J.hours;
    // A5 general condition (1): burning hours per day, drawn per replica
    int32_t bhours = 24;
    if (J.burn_max > 0) {
      const U4 x = philox4x32_10(U4{(uint32_t)r, 0u, 0u, 3u}, (uint32_t)J.seed, (uint32_t)(J.seed >> 32));
      bhours = J.burn_min + (int32_t)(((uint64_t)x.x * (uint64_t)(J.burn_max - J.burn_min + 1)) >> 32);
    }
    const bool lazy = LAZY && J.chunk_state != nullptr;
    const double delta = J.delta;
    const bool use_delta = delta > 0.0;   // A5 (i) burn-out on
    int32_t width = 4;   // of the next window, in periods
    const uint64_t seed = J.seed;
    const float sigma = J.sigma;
    const uint32_t *burnable = J.burnable;
    int32_t *istep = J.ign_step ? J.ign_step + (size_t)r * n : nullptr;
    const int len_shift = max(0, 33 - __clzll(J.d_diag));   // lengths >> len_shift fit 31 bits
    const int32_t ic = J.ign_cell[r];
    // an ignition cell outside the grid or not burnable (possible only for
    // ignition cells a caller passes in): status 3, nothing else is written
    if ((uint32_t)ic >= (uint32_t)n ||
        !((__ldg(&burnable[(ic / cols) * wpr + ((ic % cols) >> 5)]) >> ((ic % cols) & 31)) & 1u)) {
      if (lane == 0) J.status[r] = 3;
      __syncwarp();
      continue;
    }
    const int32_t ir = ic / cols, icc = ic - ir * cols;
    // window of the done-chunk bitmap, centred on the ignition cell like the plane's
    const int32_t dr0 = min(max(ir - kWinRows / 2, 0), max(rows - kWinRows, 0));
    const int32_t dw0 = min(max((icc >> 5) - kWinWords / 2, 0), max(wpr - kWinWords, 0));
    pl.rows = rows;
    pl.wpr = wpr;
    pl.burnable = burnable;
    pl.g0 = pl.g1 = 0;
    if constexpr (WIN) {   // window centred on the ignition cell, clamped to the grid
      pl.r0 = min(max(ir - kWinRows / 2, 0), max(rows - kWinRows, 0));
      pl.w0 = min(max((icc >> 5) - kWinWords / 2, 0), max(wpr - kWinWords, 0));
#pragma unroll 8
      for (int32_t i = lane; i < kWinRows * kWinWords; i += 32) {
        const int32_t rr = pl.r0 + i / kWinWords, ww = pl.w0 + i % kWinWords;
        pl.sav[i] = (rr < rows && ww < wpr) ? __ldg(&burnable[rr * wpr + ww]) : 0u;
      }
    }
    pl.reach(ir, ir, icc, icc, 2, lane);
    if (use_delta)
      for (int32_t i = lane; i < pw; i += 32) pl.gbr[i] = 0u;
    __syncwarp();

    // per-replica profile (J.prof, off unless the caller asked for it; the
    // layout of c2f_get_replica_profile), kept in shared memory by lane 0 so
    // that it costs no registers
    const bool prof = PROF && J.prof != nullptr;   // compiled out of the production kernels
    long long pc_t = 0;
    long long *pq = s_prof[wib];
    if (prof && lane == 0) {
#pragma unroll
      for (int i = 0; i < kProfCounters; ++i) pq[i] = 0;
      pq[0] = clock64();
    }

    // Step 1 of Alg. 1: the ignition cell burns from period 0.  Work: a cell
    // counts in the periods after its ignition up to its burn-out (or the
    // end), so W = sum of burn-out periods - ignition periods, less the
    // dormant hours.
    int32_t live = 1, nign = 1, cnt = 1, status = 0;
    long long W = 0;
    {
      if (lane == 0) {
        pl.take(ir, icc);
        if (istep) istep[ic] = 0;
      }
      __syncwarp();
      uint32_t b[3];
      pl.template block<1>(ir, icc, b);
      const uint32_t am = axes_of_rows(b[0], b[1], b[2]);
      if (lane < 8) {
        eP[lane] = 0;
        ecofs[lane] = (uint8_t)(((am >> lane) & 1u) ? kOpen : kNone);
      }
      if (lane == 0) erc[0] = rc_pack(ir, icc);
      if (am == 0) {   // no Available neighbour: Burned at the end of period 1
        live = 0;
        W = (H * sph >= 1) ? 1 : 0;
      }
      __syncwarp();
    }

    // On-demand table rows (lazy tables): before a row of hour h is read, the
    // chunk holding it must be done.  A chunk is looked up in the bitmap of
    // chunks known done this hour, else in chunk_state: claimed when empty (the
    // warp computes its claims at once, all lanes on one chunk), waited for
    // when another warp is computing it -- that warp is running and never
    // waits while it holds a claim.
    auto ensure = [&](int32_t h, bool valid, int32_t cr, int32_t cc) {
      if (status != 0) return;   // the replica has stopped: no more claims or waits
      uint32_t *sth = J.chunk_state + (size_t)h * pw;
      const int32_t wr = cr, wc = cc >> 5;
      const int32_t w = wr * wpr + wc;
      const bool inwin = wr >= dr0 && wr < dr0 + kWinRows && wc >= dw0 && wc < dw0 + kWinWords;
      const int32_t bi = inwin ? (wr - dr0) * kWinWords + (wc - dw0) : 0;
      bool need = false, mine = false;
      if (valid && !(inwin && ((dbits[bi >> 5] >> (bi & 31)) & 1u))) {
        uint32_t st = ld_state(sth + w);
        if (st == 0u) {
          st = atomicCAS(sth + w, 0u, 1u);
          mine = st == 0u;
        }
        need = !mine && st < 2u;
        if (st >= 2u && inwin) atomicOr(&dbits[bi >> 5], 1u << (bi & 31));
      }
      const uint32_t mb = __ballot_sync(FULL, mine);
      if (mine) claim[__popc(mb & lt)] = w;
      __syncwarp();
      const int nm = __popc(mb);
      if constexpr (HELPERS > 0) {
        if (nm > 1) {
          if (lane == 0) {
            work->job = &J;
            work->h = h;
            work->n = nm;
          }
          __syncwarp();
          bar_sync(1, 32 * (HELPERS + 1));
          for (int i = 0; i < nm; i += HELPERS + 1) table_chunk(J, h, claim[i]);
          bar_sync(2, 32 * (HELPERS + 1));
        } else if (nm == 1) {
          table_chunk(J, h, claim[0]);
        }
      } else {
        for (int i = 0; i < nm; ++i) table_chunk(J, h, claim[i]);
      }
      if (mine && inwin) atomicOr(&dbits[bi >> 5], 1u << (bi & 31));
      if (need) {
        uint32_t polls = 0;
        bool gave_up = false;
        while (ld_state(sth + w) < 2u) {
          if (++polls > wait_limit) { status = 4; gave_up = true; break; }
          __nanosleep(128);
        }
        if (!gave_up && inwin) atomicOr(&dbits[bi >> 5], 1u << (bi & 31));
      }
      __syncwarp();
      status = (int32_t)__reduce_max_sync(FULL, (uint32_t)status);   // the warp's worst status
    };

    // the calendar bit of offset nx (0 when it is not a crossing of this hour)
    auto cal_bit = [&](uint32_t nx) -> uint64_t { return nx < (uint32_t)sph ? 1ull << nx : 0ull; };
    auto cal_or = [&](uint64_t bits) -> uint64_t {   // OR of the lanes' calendar bits
      return ((uint64_t)__reduce_or_sync(FULL, (uint32_t)(bits >> 32)) << 32) |
             (uint64_t)__reduce_or_sync(FULL, (uint32_t)bits);
    };
    // the scan of A1 reads enx by words: the bytes that share the list's last
    // word with it hold no crossing
    auto end_list = [&](int32_t count) {
      if ((count & 3) != 0 && lane < 4 - (count & 3)) enx[count + lane] = kNone;
    };

    // drop burned-out cells and cells with no open axis from the burning list
    // (order kept) when it nears its capacity within an hour; the calendar
    // keeps its bits (an offset whose entries are gone is an empty window)
    auto compact = [&](int32_t &count) {
      int32_t out = 0;
      for (int32_t b0 = 0; b0 < count; b0 += 32) {
        const int32_t e = b0 + lane;
        bool keep = false;
        uint32_t rc = 0;
        uint64_t c8 = ~0ull;
        uint8_t nx = 0;
        int64_t P[8];
        if (e < count) {
          rc = erc[e];
          c8 = *reinterpret_cast<const uint64_t *>(ecofs + (size_t)e * 8);
          nx = enx[e];
          const uint32_t m = open_axes(c8);
          const int32_t cr = (int32_t)(rc >> 16), cc = (int32_t)(rc & 0xFFFFu);
          if (use_delta) {
            keep = m != 0u && !pl.burned(cr, cc);
          } else if (m != 0u) {
            uint32_t b[3];
            pl.template block<1>(cr, cc, b);
            keep = (m & axes_of_rows(b[0], b[1], b[2])) != 0u;
          }
          if (keep) {
#pragma unroll
            for (int q = 0; q < 8; ++q) P[q] = eP[(size_t)e * 8 + q];
          }
        }
        const uint32_t bal = __ballot_sync(FULL, keep);
        const int32_t pos = out + __popc(bal & lt);
        __syncwarp();
        if (keep) {
          erc[pos] = rc;
          *reinterpret_cast<uint64_t *>(ecofs + (size_t)pos * 8) = c8;
          enx[pos] = nx;
#pragma unroll
          for (int q = 0; q < 8; ++q) eP[(size_t)pos * 8 + q] = P[q];
        }
        out += __popc(bal);
        __syncwarp();
      }
      count = out;
      end_list(count);
      __syncwarp();
    };

    for (int32_t h = 0; h < H && live > 0 && status == 0; ++h) {
      const int32_t s0 = h * sph + 1;   // the hour's first period
      if (h % 24 >= bhours) {   // a dormant hour: nothing moves, no work is counted
        W -= (long long)live * sph;
        continue;
      }
      const int64_t *baseh = J.base + (size_t)h * n * 8;
      const double *hrosh = J.hros + (size_t)h * n;
      // receive tests can be skipped when the threshold is 0 and every HROS of
      // the hour is positive (then HROS * f > 0), or when the threshold is < 0
      const bool gate_free = J.recv_gate <= 1 || (J.recv_gate == 2 && J.hour && J.hour[h].pos);
      int32_t dying = 0;   // cells Burned at the end of the hour's first period (A5 (i))
      if (lazy) {
        for (int32_t i = lane; i < kWinRows * kWinWords / 32; i += 32) dbits[i] = 0u;
        __syncwarp();
      }
      uint64_t cal = 0;   // offsets of this hour at which some entry crosses

      if (prof && lane == 0) pc_t = clock64();
      // ---- hour boundary.  (B1) drop burned-out cells and cells with no way
      // left (order kept): one lane per listed cell, the kept ones queued up to
      // 32; (B2) lane i takes the i-th of them: table row and progress into
      // shared memory (asynchronously), the perturbation for this hour; (B3)
      // one open axis per lane: the crossing period of this hour, or the
      // progress carried to the next; (B4) the entry at its new place.
      {
        int32_t out = 0, queued = 0, b0 = 0;
        int32_t ra = 0x7fffffff, rb = 0, ca = 0x7fffffff, cb = 0;   // the kept cells' rows and columns
        while (b0 < cnt || queued > 0) {
          if (b0 < cnt && queued < 32) {
            const int32_t e = b0 + lane;
            bool keep = false;
            uint32_t am = 0u;   // open axes toward Available cells
            int32_t cr = 0, cc = 0;
            if (e < cnt) {
              const uint32_t rc = erc[e];
              const uint32_t m = open_axes(*reinterpret_cast<const uint64_t *>(ecofs + (size_t)e * 8));
              cr = (int32_t)(rc >> 16);
              cc = (int32_t)(rc & 0xFFFFu);
              uint32_t b[3];
              pl.template block<1>(cr, cc, b);
              am = m & axes_of_rows(b[0], b[1], b[2]);
              // with A5 (i) a cell with no way left may still die before its neighbours are gone
              keep = use_delta ? m != 0u && (b[0] | b[1] | b[2]) != 0u && !pl.burned(cr, cc) : am != 0u;
            }
            const uint32_t bal = __ballot_sync(FULL, keep);
            if (keep) {
              const int32_t at = queued + __popc(bal & lt);
              qent[at] = e;
              qam[at] = (uint8_t)am;
              ra = min(ra, cr); rb = max(rb, cr);
              ca = min(ca, cc); cb = max(cb, cc);
            }
            queued += __popc(bal);
            b0 += 32;
            __syncwarp();
            continue;
          }
          const int32_t m = min(queued, 32);
          const bool act = lane < m;
          uint32_t rc = 0u, am = 0u;
          float f = 1.0f;
          bool dies = false;
          if (act) {
            rc = erc[qent[lane]];
            am = qam[lane];
          }
          const int32_t cr = (int32_t)(rc >> 16), cc = (int32_t)(rc & 0xFFFFu);
          const int64_t cell = (int64_t)cr * cols + cc;
          if (lazy) ensure(h, act, cr, cc);   // this hour's row of the cell
          if (act) {
            const int64_t *row = baseh + cell * 8, *pp = eP + (size_t)qent[lane] * 8;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              copy_async16(rowbuf + lane * 8 + 2 * j, row + 2 * j);
              copy_async16(prgbuf + lane * 8 + 2 * j, pp + 2 * j);
            }
            // the cell's row of the next hour into L2, for the next boundary
            if (!LAZY && h + 1 < H) prefetch_l2(row + n * 8);
            f = noise_factor(seed, (uint32_t)r, (uint32_t)cell, (uint32_t)h, sigma);
            // A5 (i): a cell whose HROS * f is below delta still sends in the
            // first period of the hour and is Burned after it
            if (use_delta) dies = below_delta(hrosh, cell, f, delta);
          }
          copy_async_wait();
          __syncwarp();
          // every entry of the batch has been read: its new places (never past
          // its old ones) can be written
          if (act) *reinterpret_cast<uint64_t *>(ecofs + (size_t)(out + lane) * 8) = ~0ull;
          int32_t ni = 0;
          for (int32_t i0 = 0; i0 < m; i0 += 4) {   // lane k of each 8-lane group looks at axis k of an entry
            const uint32_t ai = __shfl_sync(FULL, am, (i0 + grp) & 31);   // 0 past the last entry
            const bool open = (ai >> k) & 1u;
            const uint32_t bal = __ballot_sync(FULL, open);
            if (open) ibuf[ni + __popc(bal & lt)] = (uint8_t)((i0 + grp) | (k << 5));
            ni += __popc(bal);
          }
          __syncwarp();
#pragma unroll 1
          for (int32_t t0 = 0; t0 < ni; t0 += 32) {
            const bool item = t0 + lane < ni;
            const uint32_t c = item ? ibuf[t0 + lane] : 0u;
            const int i = (int)(c & 31u), q = (int)(c >> 5);
            const float fi = __shfl_sync(FULL, f, i);
            const int64_t dq = (q & 1) ? J.d_diag : J.d_orth;
            const int64_t inc = apply_noise(rowbuf[i * 8 + q], noise_fixed(fi), dq);
            const int64_t P = prgbuf[i * 8 + q];
            const int32_t n1 = item ? periods_to_cross(dq - P, inc, sph, len_shift) : 0;
            if (item) {
              ecofs[(size_t)(out + i) * 8 + q] = (uint8_t)(n1 ? (uint32_t)n1 - 1u : kOpen);
              if (!n1) eP[(size_t)(out + i) * 8 + q] = P + inc * sph;
            }
          }
          __syncwarp();
          uint64_t bit = 0;
          bool burns = false;
          if (act) {
            uint64_t c8 = *reinterpret_cast<const uint64_t *>(ecofs + (size_t)(out + lane) * 8);
            if (dies) {
              for (int q = 0; q < 8; ++q)
                if ((c8 >> (8 * q)) & 0xFFull) c8 |= 0xFFull << (8 * q);
              *reinterpret_cast<uint64_t *>(ecofs + (size_t)(out + lane) * 8) = c8;
              burns = pl.burn(cr, cc);
            }
            const uint32_t nx = min_byte8(c8);
            erc[out + lane] = rc;
            enx[out + lane] = (uint8_t)nx;
            bit = cal_bit(nx);
          }
          cal |= cal_or(bit);
          if (use_delta) dying += __popc(__ballot_sync(FULL, burns));
          out += m;
          queued -= m;
          const int32_t qe = lane < queued ? qent[32 + lane] : 0;   // at most 31 are left
          const uint8_t qa = lane < queued ? qam[32 + lane] : 0;
          __syncwarp();
          if (lane < queued) {
            qent[lane] = qe;
            qam[lane] = qa;
          }
          __syncwarp();
        }
        cnt = out;
        end_list(cnt);
        // a fire advances by at most one cell a period and looks two cells ahead
        if (cnt > 0)
          pl.reach((int32_t)__reduce_min_sync(FULL, (uint32_t)ra), (int32_t)__reduce_max_sync(FULL, (uint32_t)rb),
                   (int32_t)__reduce_min_sync(FULL, (uint32_t)ca), (int32_t)__reduce_max_sync(FULL, (uint32_t)cb), sph + 2, lane);
        __syncwarp();
      }
      if (prof && lane == 0) pq[1] += clock64() - pc_t;
      if (status) break;
      live -= dying;
      W += (long long)dying * s0;

      // ---- the periods of this hour at which some axis reaches a centre
      // scan0: where A1 starts.  Not 0 only with width 1, when this period has
      // been begun: no entry before it crosses in it any more
      int32_t scan0 = 0;
      int32_t room = compact_at;   // compact above this many entries
      while (cal != 0ull) {
        const int32_t o1 = __ffsll((long long)cal) - 1;
        if (prof && lane == 0) { pc_t = clock64(); pq[7] = max(pq[7], (long long)cnt); }
        // keep room for new cells.  Again only when half of the room that a
        // compaction left is used up: a dense period has dozens of windows, and
        // a list of mostly live entries would be compacted before each
        // Not in an hour's first period with the threshold: cells that burn out
        // at the boundary still send in it
        if (cnt > room && (o1 > 0 || !use_delta)) {
          compact(cnt);
          scan0 = 0;
          room = max(compact_at, cnt + (cap - cnt) / 2);
          if (prof && lane == 0) pq[9] += 1;
        }
        const int32_t Ew = min(o1 + width, sph);   // the window is [o1, Ew), shortened below
        // (A1) the entries that cross in the window, up to 64
        int32_t got = 0;
        bool full = false;
        int32_t g0 = scan0;
        for (; g0 < cnt && !full; g0 += 1024) {
          uint32_t w = 0;   // bit 8 b + 7 - j: byte b of this lane's j-th word crosses
#pragma unroll 2
          for (int j = 0; j < 8; ++j) {
            const int32_t e0 = g0 + (j * 32 + lane) * 4;
            if (g0 + j * 128 >= cnt) break;
            if (e0 < cnt) w |= msb_below(*reinterpret_cast<const uint32_t *>(enx + e0), (uint32_t)Ew) >> j;
          }
          const uint32_t nw = (uint32_t)__popc(w);   // places by the lanes' counts, a ballot per bit
          int32_t pos = got;
#pragma unroll
          for (int j = 0; j < 6; ++j) {
            const uint32_t bal = __ballot_sync(FULL, (nw >> j) & 1u);
            pos += __popc(bal & lt) << j;
            got += __popc(bal) << j;
          }
          for (; w != 0u && pos < 64; ++pos) {
            const int32_t b = 31 - __clz((int)w);
            w ^= 1u << b;
            went[pos] = g0 + ((7 - (b & 7)) * 32 + lane) * 4 + (b >> 3);
          }
          full = got > 64;
        }
        __syncwarp();
        if (full && width > 1) {   // more than 64: a shorter window
          width = max(1, min(width - 1, width * kWindowFill / got));
          continue;
        }
        got = min(got, 64);
        if (prof && lane == 0) pq[8] += clock64() - pc_t;
        if (got == 0) { cal &= ~(1ull << o1); scan0 = 0; continue; }   // its entries were dropped by a compaction
        // (A2) their crossings in the window towards Available cells, up to
        // 32: target cell into buf, offset into obuf
        bool broken = false, more = false;   // more: more than 32 crossings
        int32_t np = 0;
#pragma unroll 1
        for (int32_t i0 = 0; i0 < got; i0 += 32) {
          uint32_t rc = 0u, left = 0u;
          uint64_t x8 = ~0ull;
          if (i0 + lane < got) {
            const int32_t e = went[i0 + lane];
            x8 = *reinterpret_cast<const uint64_t *>(ecofs + (size_t)e * 8);
            rc = erc[e];
            left = bytes_below(x8, (uint32_t)Ew);
            broken |= left == 0u;
            uint32_t b[3];
            pl.template block<1>((int32_t)(rc >> 16), (int32_t)(rc & 0xFFFFu), b);
            left &= axes_of_rows(b[0], b[1], b[2]);
          }
          while (np < 32) {
            const uint32_t bal = __ballot_sync(FULL, left != 0u);
            if (bal == 0u) break;
            const int32_t pos = np + __popc(bal & lt);
            if (left && pos < 32) {
              const int q = __ffs(left) - 1;
              left &= left - 1u;
              buf[pos] = rc + (uint32_t)(axis_dr(q) * 65536 + axis_dc(q));
              obuf[pos] = (uint8_t)__byte_perm((uint32_t)x8, (uint32_t)(x8 >> 32), (uint32_t)q);
            }
            np += __popc(bal);
          }
          more |= __any_sync(FULL, left != 0u) != 0;
          wleft[i0 + lane] = (uint8_t)left;
        }
        // every gathered entry closes an axis, or the hour would not end; cannot happen
        if (__any_sync(FULL, broken)) { status = 2; break; }
        __syncwarp();
        if (more && width > 1) {
          width = max(1, min(width - 1, width * 3 / 4));
          continue;
        }
        np = min(np, 32);
        // (A3) in the order of their offsets (rank by the offset's bits), one crossing per lane
        uint32_t trc = lane < np ? buf[lane] : 0u, toff = lane < np ? obuf[lane] : (uint32_t)o1;
        if (width > 1) {
          const uint32_t v = toff - (uint32_t)o1;
          uint32_t eq = np >= 32 ? FULL : (1u << np) - 1u;
          int32_t pos = 0;
#pragma unroll (WIN ? 5 : 1)
          for (int j = 4; j >= 0; --j) {
            const uint32_t bal = __ballot_sync(FULL, (v >> j) & 1u);
            if ((v >> j) & 1u) {
              pos += __popc(eq & ~bal);
              eq &= bal;
            } else {
              eq &= ~bal;
            }
          }
          pos += __popc(eq & lt);
          __syncwarp();
          if (lane < np) {
            buf[pos] = trc;
            obuf[pos] = (uint8_t)toff;
          }
          __syncwarp();
          if (lane < np) {
            trc = buf[lane];
            toff = obuf[lane];
          }
        }
        const int32_t tr = (int32_t)(trc >> 16), tc = (int32_t)(trc & 0xFFFFu);
        bool hit = lane < np;
        if (lazy && !gate_free) {   // the receivers' HROS
          ensure(h, hit, tr, tc);
          if (status) break;
        }
        if (!gate_free && hit) hit = receive_ok(J, r, (int64_t)tr * cols + tc, h, n);   // else consumed
        // a cell reached by several crossings ignites at the first of them (row
        // 65535 does not exist, so the idle lanes' keys are no cell)
        const uint32_t peers = __match_any_sync(FULL, hit ? trc : (0xFFFF0000u | (uint32_t)lane));
        const bool won = hit && (peers & lt) == 0u;
        const uint32_t wins = __ballot_sync(FULL, won);
        const int32_t nc = __popc(wins);
        if (won) {
          buf[__popc(wins & lt)] = trc;
          obuf[__popc(wins & lt)] = (uint8_t)toff;
        }
        __syncwarp();
        if (prof && lane == 0) {
          const long long t1 = clock64();
          pq[2] += t1 - pc_t;
          pc_t = t1;
          pq[10] += got > 32 ? 2 : 1;
        }
        if (cnt + nc > cap) { status = 1; break; }
        // (C1) lane i holds the i-th cell that ignites
        const bool act = lane < nc;
        const uint32_t nrc = act ? buf[lane] : 0u, no = act ? obuf[lane] : 0u;
        const int32_t nr = (int32_t)(nrc >> 16), ncol = (int32_t)(nrc & 0xFFFFu);
        const int64_t ncell = (int64_t)nr * cols + ncol;
        if (lazy) {   // this hour's rows of the new cells
          ensure(h, act, nr, ncol);
          if (status) break;
        }
        float f = 1.0f;
        uint32_t nam = 0u;   // its axes towards Available cells | offset << 8
        uint32_t fuel_lo[3] = {0u, 0u, 0u}, fuel_hi[3] = {0u, 0u, 0u};   // the burnable plane around it
        bool dies = false;
        if (act) {
          const int64_t *row = baseh + ncell * 8;
#pragma unroll
          for (int j = 0; j < 4; ++j) copy_async16(rowbuf + lane * 8 + 2 * j, row + 2 * j);
          uint32_t b[3];
          pl.template block<1>(nr, ncol, b);
          nam = axes_of_rows(b[0], b[1], b[2]) | (no << 8);
          const int32_t wl = (ncol - 1) >> 5, wh = (ncol + 1) >> 5;
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const int32_t rr = nr - 1 + d;
            const bool in = rr >= 0 && rr < rows;
            fuel_lo[d] = in && wl >= 0 ? __ldg(&burnable[rr * wpr + wl]) : 0u;
            fuel_hi[d] = in && wh < wpr ? __ldg(&burnable[rr * wpr + wh]) : 0u;
          }
          f = noise_factor(seed, (uint32_t)r, (uint32_t)ncell, (uint32_t)h, sigma);
          if (use_delta && below_delta(hrosh, ncell, f, delta)) { dies = true; nam &= ~0xFFu; }   // A5 (i)
        }
        copy_async_wait();
        __syncwarp();
        // (C2) one open axis per lane: first crossings, progress to the end of
        // the hour.  One round at a time: with two in flight (more code) 4,000
        // replicas took 5.99 instead of 5.38 ms and 64 no less, for the
        // instruction fetches
        if (act) *reinterpret_cast<uint64_t *>(ecofs + (size_t)(cnt + lane) * 8) = ~0ull;
        int32_t ni = 0;
        for (int32_t b0 = 0; b0 < nc; b0 += 4) {   // lane k of each 8-lane group looks at axis k of a cell
          const uint32_t am = __shfl_sync(FULL, nam, (b0 + grp) & 31);   // 0 past the last cell
          const bool open = (am >> k) & 1u;
          const uint32_t bal = __ballot_sync(FULL, open);
          if (open) ibuf[ni + __popc(bal & lt)] = (uint8_t)((b0 + grp) | (k << 5));
          ni += __popc(bal);
        }
        __syncwarp();
#pragma unroll 1
        for (int32_t t0 = 0; t0 < ni; t0 += 32) {
          const bool item = t0 + lane < ni;
          const uint32_t c = item ? ibuf[t0 + lane] : 0u;
          const int i = (int)(c & 31u), q = (int)(c >> 5);
          const uint32_t oa = __shfl_sync(FULL, nam, i);
          const float fi = __shfl_sync(FULL, f, i);
          const int64_t dq = (q & 1) ? J.d_diag : J.d_orth;
          const int32_t o = (int32_t)(oa >> 8), nmax = sph - 1 - o;   // nmax: periods left in the hour
          const int64_t inc = apply_noise(rowbuf[i * 8 + q], noise_fixed(fi), dq);
          const int32_t n1 = periods_to_cross(dq, inc, nmax, len_shift);
          if (item) {
            ecofs[(size_t)(cnt + i) * 8 + q] = (uint8_t)(n1 ? o + n1 : (int32_t)kOpen);
            eP[(size_t)(cnt + i) * 8 + q] = inc * nmax;   // read only while the axis is open
          }
        }
        __syncwarp();
        // (C3) the window's end, and the cells that ignite before it: taken and listed
        uint64_t c8 = ~0ull;
        if (act) c8 = *reinterpret_cast<const uint64_t *>(ecofs + (size_t)(cnt + lane) * 8);
        const int32_t E = (int32_t)min((uint32_t)Ew, warp_min(min_byte8(c8)));
        const bool commit = act && (int32_t)no < E;
        const int32_t done = __popc(__ballot_sync(FULL, commit));
        uint64_t bits = 0;      // calendar bits this lane sets
        uint32_t out = 0;       // cells this lane turned Burned: count << 16 | sum of their offsets
        if (commit) pl.take(nr, ncol);
        __syncwarp();
        uint32_t gone = 0u;     // burnable cells of the block around it with no Available cell around them
        if (commit) {
          uint32_t b[5];
          pl.template block<2>(nr, ncol, b);
          const uint32_t am = axes_of_rows((b[1] >> 1) & 7u, (b[2] >> 1) & 7u, (b[3] >> 1) & 7u);
          c8 |= ((uint64_t)bytes_of(~am >> 4) << 32) | bytes_of(~am);   // the axes that are still open
          const uint32_t nx = min_byte8(c8);
          erc[cnt + lane] = nrc;
          *reinterpret_cast<uint64_t *>(ecofs + (size_t)(cnt + lane) * 8) = c8;
          enx[cnt + lane] = (uint8_t)nx;
          if (istep) istep[ncell] = s0 + (int32_t)no;
          bits = cal_bit(nx);
          if (dies && pl.burn(nr, ncol)) out = (1u << 16) + no;
          const uint32_t v0 = b[0] | b[1] | b[2], v1 = b[1] | b[2] | b[3], v2 = b[2] | b[3] | b[4];
          gone = ~((v0 | (v0 >> 1) | (v0 >> 2)) & 7u | (((v1 | (v1 >> 1) | (v1 >> 2)) & 7u) << 3) |
                   (((v2 | (v2 >> 1) | (v2 >> 2)) & 7u) << 6));
          uint32_t fuel9 = 0u;
#pragma unroll
          for (int d = 0; d < 3; ++d)
            fuel9 |= (__funnelshift_r(fuel_lo[d], fuel_hi[d], (uint32_t)(ncol - 1) & 31u) & 7u) << (3 * d);
          gone &= fuel9;
        }
        // A5 (ii): the ignited cells among them have burned out in this window
        // (a cell next to an ignition of the window had an Available neighbour
        // before it), at the last ignition next to them, unless A5 (i) had
        // them burn out earlier
        if (__any_sync(FULL, gone != 0u)) {
          // the last cells' first: places counted from the highest lane
          const uint32_t ng = (uint32_t)__popc(gone);
          int32_t at = 0, total = 0;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const uint32_t bal = __ballot_sync(FULL, (ng >> j) & 1u);
            at += __popc(bal & ~lt & ~(1u << lane)) << j;
            total += __popc(bal) << j;
          }
          for (int32_t t0 = 0; t0 < total; t0 += 32) {
            while (gone != 0u && at < t0 + 32) {
              const uint32_t p = (uint32_t)(__ffs(gone) - 1);
              gone &= gone - 1u;
              buf[at - t0] = (uint32_t)lane | (p << 5);
              ++at;
            }
            __syncwarp();
            const bool valid = t0 + lane < total;
            const uint32_t c = valid ? buf[lane] : 0u;
            const uint32_t crc = __shfl_sync(FULL, nrc, (int)(c & 31u));
            const uint32_t co = __shfl_sync(FULL, no, (int)(c & 31u));
            const int32_t p = (int32_t)(c >> 5), pr3 = (p * 11) >> 5;   // p / 3
            const int32_t xr = (int32_t)(crc >> 16) + pr3 - 1, xc = (int32_t)(crc & 0xFFFFu) + p - 3 * pr3 - 1;
            const uint32_t key = valid ? rc_pack(xr, xc) : (0xFFFF0000u | (uint32_t)lane);
            bool first = (__match_any_sync(FULL, key) & lt) == 0u;
            if (total > 32) {   // nor in an earlier round (rowbuf is free by now)
              uint32_t *keys = reinterpret_cast<uint32_t *>(rowbuf);
              for (int32_t j = 0; j < t0; ++j) first = first && keys[j] != key;
              __syncwarp();
              keys[t0 + lane] = key;
            }
            if (valid && first && (!use_delta || pl.burn(xr, xc))) out += (1u << 16) + co;
            __syncwarp();
          }
        }
        // (C4) the crossings before E are closed
        if (!full) cal &= ~((1ull << E) - 1ull);   // E <= 60
        uint64_t seen = 0;      // profile: periods at which a crossing was processed, entries with one
        int32_t crossed = 0;
        uint32_t rest = full ? (uint32_t)(g0 - 1024) : 0xFFFFFFFFu;   // the first entry that may still cross before E
#pragma unroll 1
        for (int32_t i0 = 0; i0 < got; i0 += 32) {
          bool closed = false;
          if (i0 + lane < got) {
            const int32_t e = went[i0 + lane];
            uint64_t *at = reinterpret_cast<uint64_t *>(ecofs + (size_t)e * 8);
            const uint32_t x0 = (uint32_t)*at, x1 = (uint32_t)(*at >> 32);
            uint32_t lo = msb_below(x0, (uint32_t)E), hi = msb_below(x1, (uint32_t)E);
            if (more) {   // crossings that found no lane stay open
              lo &= ~bytes_of(wleft[i0 + lane]);
              hi &= ~bytes_of(wleft[i0 + lane] >> 4);
            }
            closed = (lo | hi) != 0u;
            if (closed) {
              const uint64_t v = ((uint64_t)(x1 | (hi >> 7) * 0xFFu) << 32) | (x0 | (lo >> 7) * 0xFFu);
              const uint32_t nx = min_byte8(v);
              *at = v;
              enx[e] = (uint8_t)nx;
              bits |= cal_bit(nx);
              if ((int32_t)nx < E) rest = min(rest, (uint32_t)e);
            } else if (more) {
              bits |= 1ull << o1;
              rest = min(rest, (uint32_t)e);
            }
            if (PROF && closed)
              for (int j = 0; j < 8; ++j) {
                const uint32_t u = ((j < 4 ? x0 : x1) >> (8 * (j & 3))) & 0xFFu;
                if ((int32_t)u < E) seen |= 1ull << u;
              }
          }
          if (PROF) crossed += __popc(__ballot_sync(FULL, closed));
        }
        cal |= cal_or(bits);
        const uint32_t ob = __reduce_add_sync(FULL, out);
        const int32_t on = (int32_t)__reduce_add_sync(FULL, commit ? no : 0u);
        const int32_t burned = (int32_t)(ob >> 16);
        W += (long long)(burned - done) * s0 + ((int32_t)(ob & 0xFFFFu) - on);
        if (PROF) {
          seen = cal_or(seen);
          if (prof && lane == 0) {
            pq[3] += clock64() - pc_t;
            if (!full && !more) pq[4] += __popcll(seen);
            pq[5] += crossed;
            pq[6] += done;
            pq[11] += (done + 3) / 4;
          }
        }
        nign += done;
        live += done - burned;
        cnt += done;
        end_list(cnt);
        // the next window: as long as should fill it, a little longer than what this one reached
        width = min(max(1, (Ew - o1) * kWindowFill / got), E < Ew ? E - o1 + 2 : 32);
        width = min(width, 32);
        if (scan0 > 0) width = 1;   // the end of a long period says nothing of the next one's density
        scan0 = 0;
        if (full || more) {         // one period, not done yet: on from its first entry that is left
          rest = __reduce_min_sync(FULL, rest);
          if (rest != 0xFFFFFFFFu) {
            scan0 = (int32_t)(rest & ~1023u);
            width = 1;
          }
        }
        __syncwarp();
        if (live == 0) break;
      }
    }
    W += (long long)live * (long long)H * sph;
    {   // scar plane: burnable cells that are no longer Available
      uint32_t *dst = J.ign_plane + (size_t)r * pw;
      auto scar = [&](int32_t i) -> uint32_t {
        const int32_t rr = i / wpr, ww = i - rr * wpr;
        if (pl.in_win(rr, ww)) return __ldg(&burnable[i]) & ~pl.sav[(rr - pl.r0) * kWinWords + (ww - pl.w0)];
        return rr >= pl.g0 && rr < pl.g1 ? __ldg(&burnable[i]) & ~pl.gav[i] : 0u;
      };
      // only the rows of the window and of the global plane hold ignited cells
      int32_t ra = pl.g0, rb = pl.g1;
      if constexpr (WIN) {
        ra = pl.g0 == pl.g1 ? pl.r0 : min(pl.r0, pl.g0);
        rb = pl.g0 == pl.g1 ? min(pl.r0 + kWinRows, rows) : max(min(pl.r0 + kWinRows, rows), pl.g1);
      }
      const int32_t ia = ra * wpr, ib = rb * wpr;
      for (int32_t i = lane; i < ia; i += 32) dst[i] = 0u;
      for (int32_t i = ib + lane; i < pw; i += 32) dst[i] = 0u;
      int32_t i = ia + lane;
      for (; i + 3 * 32 < ib; i += 4 * 32) {   // four words in flight
        uint32_t v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = scar(i + 32 * j);
#pragma unroll
        for (int j = 0; j < 4; ++j) dst[i + 32 * j] = v[j];
      }
      for (; i < ib; i += 32) dst[i] = scar(i);
    }
    if (lane == 0) {
      if (A.trace.rec) trace_record(A.trace, kTraceReplica, (uint32_t)r, J.trace_tag, t_start, global_ns());
      J.work[r] = W;
      J.n_ignited[r] = nign;
      J.status[r] = status;
      if (prof) {
        long long *q = J.prof + (size_t)r * kProfCounters;
        q[0] = clock64() - pq[0];
#pragma unroll
        for (int i = 1; i < kProfCounters; ++i) q[i] = pq[i];
      }
    }
    __syncwarp();
  }
}

// Variants: warps per CTA (1, 2, 4); planes windowed and lists in shared
// memory (w), or everything in global memory (g); l: tables filled on demand;
// p: the per-replica profile counters compiled in (one-warp CTAs; the
// production kernels leave that code out, which makes them about 4 % faster).
// Register budgets: one-warp CTAs with windows sized so that 11 fit on an SM
// (their shared memory allows no more, and fewer registers would spill), those
// with global lists so that 13 fit (48 waiting requests: 46.1 ms at 11, 43.6 at
// 13, 43.6 at 16); two-warp CTAs so that 5 fit
__global__ void __launch_bounds__(32, 13) k_frontier_g1(FrontierArgs A) { frontier_warp<1, false, false, false>(A); }
__global__ void __launch_bounds__(64, 5) k_frontier_g2(FrontierArgs A) { frontier_warp<2, false, false, false>(A); }
__global__ void __launch_bounds__(128) k_frontier_g4(FrontierArgs A) { frontier_warp<4, false, false, false>(A); }
__global__ void __launch_bounds__(32, 11) k_frontier_w1(FrontierArgs A) { frontier_warp<1, true, false, false>(A); }
__global__ void __launch_bounds__(64, 5) k_frontier_w2(FrontierArgs A) { frontier_warp<2, true, false, false>(A); }
__global__ void __launch_bounds__(128) k_frontier_w4(FrontierArgs A) { frontier_warp<4, true, false, false>(A); }
__global__ void __launch_bounds__(32, 11) k_frontier_pg1(FrontierArgs A) { frontier_warp<1, false, false, true>(A); }
__global__ void __launch_bounds__(32, 11) k_frontier_pw1(FrontierArgs A) { frontier_warp<1, true, false, true>(A); }
// on-demand table rows: one warp per CTA; the FBP code inlined into the
// frontier needs the whole register budget of a one-warp CTA
__global__ void __launch_bounds__(32, 1) k_frontier_lg1(FrontierArgs A) { frontier_warp<1, false, true, false>(A); }
__global__ void __launch_bounds__(32, 1) k_frontier_lw1(FrontierArgs A) { frontier_warp<1, true, true, false>(A); }
// the same with seven helper warps, for launches that leave SMs to spare: a
// single warp computes 32 rows at the FP64 unit's latency (few fires on
// 4096 x 4096, 8 replicas: three quarters of their time)
constexpr int kHelpers = 7;
template <bool WIN>
__device__ __forceinline__ void frontier_helped(const FrontierArgs &A) {
  __shared__ ChunkWork work;
  if (threadIdx.x >= 32) {
    help_with_chunks<kHelpers>(&work);
    return;
  }
  frontier_warp<1, WIN, true, false, kHelpers>(A, &work);
  if (threadIdx.x == 0) work.n = -1;
  __syncwarp();
  bar_sync(1, 32 * (kHelpers + 1));
}
__global__ void __launch_bounds__(32 * (kHelpers + 1), 1) k_frontier_lg1h(FrontierArgs A) { frontier_helped<false>(A); }
__global__ void __launch_bounds__(32 * (kHelpers + 1), 1) k_frontier_lw1h(FrontierArgs A) { frontier_helped<true>(A); }
__global__ void __launch_bounds__(32, 1) k_frontier_plg1(FrontierArgs A) { frontier_warp<1, false, true, true>(A); }
__global__ void __launch_bounds__(32, 1) k_frontier_plw1(FrontierArgs A) { frontier_warp<1, true, true, true>(A); }

// ------------------------------------------------------------------ K4
// counts[c] = sum over replicas of the scar bit of c.  Each thread owns one
// 32-cell word and adds the replicas' words into a bit-sliced (vertical)
// counter: plane i holds bit i of the 32 per-cell counts.
// With scen, only the replicas whose drawn weather scenario is `want` count.
__global__ void k_burn_prob(const uint32_t *__restrict__ planes, int32_t R, int32_t rows,
                            int32_t cols, int32_t wpr, int32_t r_chunk, uint32_t *counts,
                            int32_t accumulate, const int32_t *__restrict__ scen, int32_t want) {
  const int64_t pw = (int64_t)rows * wpr;
  const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= pw) return;
  const int32_t r0 = blockIdx.y * r_chunk;
  const int32_t r1 = min(R, r0 + r_chunk);
  uint32_t c[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) c[i] = 0;
  for (int32_t r = r0; r < r1; ++r) {
    if (scen && __ldg(&scen[r]) != want) continue;
    uint32_t carry = __ldg(&planes[(size_t)r * pw + w]);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const uint32_t t = c[i] & carry;
      c[i] ^= carry;
      carry = t;
    }
  }
  const int32_t row = (int32_t)(w / wpr), cw = (int32_t)(w % wpr);
  for (int b = 0; b < 32; ++b) {
    const int32_t col = cw * 32 + b;
    if (col >= cols) break;
    uint32_t v = 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) v |= ((c[i] >> b) & 1u) << i;
    const int64_t cell = (int64_t)row * cols + col;
    if (accumulate) { if (v) atomicAdd(&counts[cell], v); }
    else counts[cell] = v;
  }
}

// ignition steps -> one byte per (replica, cell): ignited by period smax
__global__ void k_scar_at_step(const int32_t *__restrict__ ign_step, int64_t total, int32_t smax,
                               uint8_t *out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  const int32_t s = ign_step[i];
  out[i] = (s >= 0 && s <= smax) ? 1 : 0;
}

// scar bits -> one byte per (replica, cell)
__global__ void k_scar_bytes(const uint32_t *__restrict__ planes, int32_t R, int32_t rows,
                             int32_t cols, int32_t wpr, uint8_t *out) {
  const int64_t n = (int64_t)rows * cols;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n * R) return;
  const int64_t r = i / n, cell = i % n;
  const int32_t row = (int32_t)(cell / cols), col = (int32_t)(cell % cols);
  out[i] = (planes[(size_t)r * rows * wpr + (size_t)row * wpr + (col >> 5)] >> (col & 31)) & 1u;
}

// ------------------------------------------------------------------ calibration
// FP64 fused multiply-add throughput of the device: eight independent chains
// per thread, enough warps to cover the pipe's latency; the roofline peak of
// the table kernel, which is FP64-bound.
__global__ void k_dfma_peak(double *out, int32_t iters) {
  const double m = 0.999999999, c = 1e-12;
  double a[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) a[j] = 1.0 + 1e-3 * (threadIdx.x + j);
  for (int32_t i = 0; i < iters; ++i) {
#pragma unroll
    for (int j = 0; j < 8; ++j) a[j] = __fma_rn(a[j], m, c);
  }
  double t = 0.0;
#pragma unroll
  for (int j = 0; j < 8; ++j) t += a[j];
  if (t == 12345.678) out[blockIdx.x] = t;   // never true; keeps the chains alive
}

// ------------------------------------------------------------------ scar comparison
// Sec. 4.1 compares two runs' scars X^t, Y^t (0-1 grids, 1 = ignited by the
// end of weather hour t) by MSE, SSIM and, for the final scars, ||X - Y||.
// For 0-1 grids all three are functions of a = |X|, b = |Y|, c = |X and Y|
// and N: sum |X - Y|^2 = a + b - 2c; the means are a/N, b/N; the 1/(N-1)
// variances a(N-a)/(N(N-1)), b(N-b)/(N(N-1)); the covariance
// (cN - ab)/(N(N-1)).  SSIM takes Wang et al.'s C1 = 0.01^2, C2 = 0.03^2
// (dynamic range 1) and sigma_X^2 + sigma_Y^2 + C2 in its denominator.
constexpr double kSsimC1 = 0.0001;   // (0.01 * 1)^2
constexpr double kSsimC2 = 0.0009;   // (0.03 * 1)^2

__device__ inline void scar_metrics(double a, double b, double c, double n, double *mse,
                                    double *ssim) {
  *mse = (a + b - 2.0 * c) / n;
  const double mx = a / n, my = b / n;
  const double nn1 = n * (n - 1.0);
  const double vx = a * (n - a) / nn1, vy = b * (n - b) / nn1;
  const double cxy = (c * n - a * b) / nn1;
  *ssim = ((2.0 * mx * my + kSsimC1) * (2.0 * cxy + kSsimC2)) /
          ((mx * mx + my * my + kSsimC1) * (vx + vy + kSsimC2));
}

// weather hour in which ignition step s falls (step 0 = the ignition, hour 0);
// -1 for a cell that never ignites
__device__ __forceinline__ int32_t ign_hour(int32_t s, int32_t sph) {
  return s < 0 ? -1 : (s == 0 ? 0 : (s - 1) / sph);
}

__device__ __forceinline__ void count_cell(int32_t sx, int32_t sy, int32_t sph, int32_t H,
                                           uint32_t *hist) {
  const int32_t hx = ign_hour(sx, sph), hy = ign_hour(sy, sph);
  if (hx >= 0 && hx < H) atomicAdd(&hist[hx], 1u);
  if (hy >= 0 && hy < H) atomicAdd(&hist[H + hy], 1u);
  if (hx >= 0 && hy >= 0 && max(hx, hy) < H) atomicAdd(&hist[2 * H + max(hx, hy)], 1u);
}

__device__ __forceinline__ void count_cells4(const int4 &a, const int4 &b, int32_t sph, int32_t H,
                                             uint32_t *hist) {
  // four cells that neither run ignites (the common case) cost one test
  if ((a.x & a.y & a.z & a.w & b.x & b.y & b.z & b.w) < 0) return;
  count_cell(a.x, b.x, sph, H, hist);
  count_cell(a.y, b.y, sph, H, hist);
  count_cell(a.z, b.z, sph, H, hist);
  count_cell(a.w, b.w, sph, H, hist);
}

// One CTA per replica: histograms of the ignition hours of X, of Y and of the
// later of the two (cells both runs ignite), then prefix sums over hours give
// a, b, c of every hour's scars; one pass over the two ignition-step arrays,
// streamed with 16-byte loads (when the rows are aligned), four per array in
// flight per thread.  HBM-bound, given enough threads in flight: CTAs of 128 to
// 1,024 threads, as many as keep every replica of the launch resident at once
// (500 pairs of 512 x 512: 287 us with 128 threads, 186 us, 5.6 TB/s, with 512;
// 100 pairs 252 and, with 1,024, 60 us; a cluster of CTAs a replica was slower
// than 128 threads).  Dynamic shared memory: 3 H counters.  The final scars are
// the scars of the last hour, so ||X - Y|| comes from the same counts.
__global__ void __launch_bounds__(1024) k_compare_hours(const int32_t *__restrict__ step_x,
                                                       const int32_t *__restrict__ step_y, int64_t n,
                                                       int32_t sph, int32_t H, double *mse, double *ssim,
                                                       double *dnorm) {
  extern __shared__ uint32_t hist[];
  const int32_t r = blockIdx.x;
  for (int32_t i = threadIdx.x; i < 3 * H; i += blockDim.x) hist[i] = 0u;
  __syncthreads();
  const int32_t *x = step_x + (size_t)r * n;
  const int32_t *y = step_y + (size_t)r * n;
  if ((n & 3) == 0 && ((reinterpret_cast<uintptr_t>(step_x) | reinterpret_cast<uintptr_t>(step_y)) & 15u) == 0) {
    const int4 *x4 = reinterpret_cast<const int4 *>(x);
    const int4 *y4 = reinterpret_cast<const int4 *>(y);
    const int64_t n4 = n / 4, bd = blockDim.x;
    int64_t i = threadIdx.x;
    for (; i + 3 * bd < n4; i += 4 * bd) {
      int4 a[4], b[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        a[u] = __ldcs(x4 + i + u * bd);
        b[u] = __ldcs(y4 + i + u * bd);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) count_cells4(a[u], b[u], sph, H, hist);
    }
    for (; i < n4; i += bd) count_cells4(__ldcs(x4 + i), __ldcs(y4 + i), sph, H, hist);
  } else {
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) count_cell(__ldcs(x + i), __ldcs(y + i), sph, H, hist);
  }
  __syncthreads();
  if (threadIdx.x < 3) {   // counts of scars at hour t: inclusive prefix sums
    uint32_t *h = hist + threadIdx.x * H;
    uint32_t acc = 0u;
    for (int32_t t = 0; t < H; ++t) { acc += h[t]; h[t] = acc; }
  }
  __syncthreads();
  for (int32_t t = threadIdx.x; t < H; t += blockDim.x) {
    double m, q;
    scar_metrics((double)hist[t], (double)hist[H + t], (double)hist[2 * H + t], (double)n, &m, &q);
    if (mse) mse[(size_t)r * H + t] = m;
    if (ssim) ssim[(size_t)r * H + t] = q;
  }
  if (dnorm && threadIdx.x == 0)   // |X xor Y| = a + b - 2c, exact in binary64
    dnorm[r] = sqrt((double)hist[H - 1] + (double)hist[2 * H - 1] - 2.0 * (double)hist[3 * H - 1]);
}

// ||X - Y|| of the final scars from the bit planes: one CTA per replica
// (256 threads), popcounts of X, Y and X and Y over the replica's words.
__global__ void k_compare_final(const uint32_t *__restrict__ px, const uint32_t *__restrict__ py,
                                int64_t pw, double *dnorm) {
  __shared__ unsigned long long part[8];
  const int32_t r = blockIdx.x;
  const uint32_t *x = px + (size_t)r * pw;
  const uint32_t *y = py + (size_t)r * pw;
  unsigned long long d = 0;   // sum |X - Y|^2 = |X xor Y|
  for (int64_t i = threadIdx.x; i < pw; i += blockDim.x) d += (unsigned)__popc(__ldcs(x + i) ^ __ldcs(y + i));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = d;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long t = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += part[w];
    dnorm[r] = sqrt((double)t);
  }
}

}  // namespace c2f
