// step_f64.cu -- the plain FP64 form of ion_step (ION_F64_PLAIN): FP64 data
// and arithmetic everywhere.  It is bound by GB300's FP64 pipe (2 lanes per
// clock and SM: one FP64 instruction costs the issue time of ~64 FP32 ones),
// not by memory, so its design is about needing few FP64 instructions and
// keeping that pipe's lanes busy:
//   * the rates by table (fp64_math.cuh), the series by boundary flows
//     (taylor_flow_f64), every choice and comparison on FP32 copies or bits;
//   * a persistent grid of warps draws groups of 32 cells from a counter in
//     the workspace header;
//   * cold cells (every window rate below the field at which the FP64 series
//     would take a term) are finished where they are found: N and the
//     freed electrons are left as they are, only the window rule runs;
//   * the others are sorted into per-warp queues by window width and by an
//     FP32 estimate of their largest W dt (Taylor by the number of its
//     terms, Bateman form), and each queue is worked off 32 cells at a time,
//     so that the FP64 arithmetic runs in full warps whose lanes take the
//     same path at exactly their width (in as many terms as that needs: kThrFlow);
//     at the end the warps of a block put their leftovers together;
//   * a grid too small to fill those queues runs one cell per lane
//     (ion_step_f64_direct), on as many SMs as it has warps.
#include <cstdint>
#include <mutex>

#include "ion_cell.cuh"
#include "ion_step.cuh"

namespace ion {

namespace {

constexpr int kWarps = 8;
constexpr int kThreads = 32 * kWarps;
// widths 2..6 x forms {Taylor of at most 3, 6, 18 terms, Bateman}
constexpr int kWidths = ION_MAX_WINDOW - 1;
constexpr int kForms = 4;
constexpr int kClasses = kForms * kWidths;
// a queue holds at most 31 cells left over plus one group's 32
constexpr int kQueueCap = 64;
constexpr int kRunF64 = 4;  // groups drawn per counter update

struct F64Smem {
  StagedF64 tab;
  StagedF32 tab32;  // for the FP32 estimate of the rates
  uint32_t queue[kWarps][kClasses][kQueueCap];
  int count[kWarps][kClasses];
};

// The form class of an FP32 estimate of the largest W dt (2 W dt below
// kThrF64[R] takes at most R terms at any width; above 0.49 the cell most likely takes
// the Bateman form: its own FP64 rates decide).
__device__ __forceinline__ int form_class(float lmax) {
  const float x = 2.0f * lmax;
  return x > 0.98f ? 3 : (x > kThrF64[6]) + (x > kThrF64[3]);
}

// One cell of exactly W states; returns |change of sum_k N_k|
// (ION_CONSERVATION_CHECK).
template <int W>
__device__ __forceinline__ double f64_cell(const JobIO& J, const Policy& pol,
                                           const StagedF64& tab, int c, double E, int lo) {
  double* __restrict__ p = static_cast<double*>(J.N) + (int64_t)lo * J.ld + c;
  double v[W], lam[W];
#pragma unroll
  for (int r = 0; r < W; ++r) v[r] = __ldcs(p + (int64_t)r * J.ld);
  const FieldF64 f = field_f64(E);
  float lmax = 0.0f;
#pragma unroll
  for (int r = 0; r < W - 1; ++r) {
    lam[r] = pol.zero_dt ? 0.0 : rate_dt_f64<kTopStep>(tab, lo + r, f);
    lmax = fmaxf(lmax, f32_of_f64(lam[r]));
  }
  lam[W - 1] = 0.0;
  lmax *= 1.0f + 0x1p-22f;  // an upper bound of the largest rate
  const bool check = (pol.flags & ION_CONSERVATION_CHECK) != 0;
  ExactSum<double> acc;
  if (check) {
#pragma unroll
    for (int r = 0; r < W; ++r) acc.add(-v[r]);
  }
  const double dne =
      lmax <= DDParams<double>::prop_max
          ? taylor_flow_f64<W>(v, lam, flow_terms<W>(2.0f * lmax))
          : dd_update<double, W>(v, lam, W);
  if (check) {
#pragma unroll
    for (int r = 0; r < W; ++r) acc.add(v[r]);
  }
#pragma unroll
  for (int r = 0; r < W; ++r) __stcs(p + (int64_t)r * J.ld, v[r]);
  const double* __restrict__ G = static_cast<const double*>(J.n_gas);
  __stcs(static_cast<double*>(J.dne) + c, G ? dne * G[c] : dne);
  const int hi = lo + W - 1;
  int nlo = lo, nhi = hi;
  window_after_step<double, W>(J, pol, v, W, nlo, nhi);
  if (nlo != lo || nhi != hi) {
    J.lo[c] = (uint8_t)nlo;
    J.hi[c] = (uint8_t)nhi;
  }
  return check ? fabs(acc.value()) : 0.0;
}

// A cell of w states (2 <= w <= ION_MAX_WINDOW; w uniform over the active
// lanes); the bits of its change of sum_k N_k.
__device__ __forceinline__ uint32_t f64_cell_of(int w, const JobIO& J, const Policy& pol,
                                                const StagedF64& tab, int c, double E, int lo) {
  double d;
  if (w == 2)
    d = f64_cell<2>(J, pol, tab, c, E, lo);
  else if (w == 3)
    d = f64_cell<3>(J, pol, tab, c, E, lo);
  else if (w == 4)
    d = f64_cell<4>(J, pol, tab, c, E, lo);
  else if (w == 5)
    d = f64_cell<5>(J, pol, tab, c, E, lo);
  else
    d = f64_cell<6>(J, pol, tab, c, E, lo);
  return abs_bits(d);
}

// A cell that keeps its populations: no electron is freed (a single state
// has nowhere to go; a cold window's series would take no term), and only the
// window rule runs.
__device__ __forceinline__ void f64_still_cell(const JobIO& J, const Policy& pol, int c, int lo,
                                               int hi) {
  static_cast<double*>(J.dne)[c] = 0.0;
  if ((pol.flags & ION_NO_WINDOW_UPDATE) != 0 || hi == lo || hi >= J.Z) return;
  const double* p = static_cast<const double*>(J.N) + (int64_t)lo * J.ld + c;
  if (p[0] < pol.eps) {
    double v[ION_MAX_WINDOW];
#pragma unroll
    for (int r = 0; r < ION_MAX_WINDOW; ++r) v[r] = r < hi - lo ? p[(int64_t)r * J.ld] : 0.0;
    int nl = lo, nh = hi;
    slide_window<double, ION_MAX_WINDOW>(v, hi - lo + 1, J.Z, pol.eps, nl, nh);
    J.lo[c] = (uint8_t)nl;
    J.hi[c] = (uint8_t)nh;
  }
}

// FP32 estimate of the window's largest W dt.
__device__ __forceinline__ float estimate_f32(const StagedF32& tab, const Policy& pol, double E,
                                              int lo, int w) {
  const FieldF32 f = field_f32(f32_of_f64(E));
  float lmax = 0.0f;
  if (!pol.zero_dt)
    for (int r = 0; r < w - 1; ++r) lmax = fmaxf(lmax, rate_dt_f32(tab, lo + r, f));
  return lmax;
}

// 33.5M nitrogen cells: 1,787 us (5,573 with library functions, four FP64
// instructions per slot and term, choices by FP64 comparisons and widths rounded up to
// 2, 4, 6; 20 + 16 w bytes per cell take 381 us).
__global__ void __launch_bounds__(kThreads, 2)
    ion_step_f64_kernel(const __grid_constant__ JobIO J, const __grid_constant__ Policy pol,
                        uint32_t* hdr) {
  __shared__ F64Smem sm;
  __shared__ float ecold[ION_MAX_Z + ION_MAX_WINDOW];
  stage_f64(J.tab, pol.log2dt, &sm.tab);
  stage_f32(J.tab, pol.log2dt, &sm.tab32);
  if (threadIdx.x < 32) stage_cold(J.tab, pol.log2dt, kColdLog2F64, ecold, threadIdx.x);
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  if (lane < kClasses) sm.count[wib][lane] = 0;
  __syncthreads();
  cudaGridDependencySynchronize();  // the header is zero
  uint32_t(*queue)[kQueueCap] = sm.queue[wib];
  int* count = sm.count[wib];
  const unsigned below = (1u << lane) - 1u;
  const int ngroups = (J.ncells + 31) / 32;
  int g = 0, left = 0;
  uint32_t cmax = 0;
  // works off cell c of class cls
  auto work = [&](int c, int cls) {
    cmax = max(cmax, f64_cell_of(2 + cls % kWidths, J, pol, sm.tab, c,
                                 static_cast<const double*>(J.E)[c], J.lo[c]));
  };
  for (;;) {
    if (left == 0) {
      int b = 0;
      if (lane == 0) b = (int)atomicAdd(&hdr[kHdrChunk], (unsigned)kRunF64);
      g = __shfl_sync(kFull, b, 0);
      left = kRunF64;
    }
    if (g >= ngroups) break;  // groups come in increasing order: no more
    const int c = g * 32 + lane;
    ++g;
    --left;
    int cls = -1;
    if (c < J.ncells) {
      const double Ec = static_cast<const double*>(J.E)[c];
      const int lo = J.lo[c], hi = J.hi[c], w = hi - lo + 1;
      if (!window_ok(lo, hi, J.Z)) {
        atomicAdd(&hdr[kHdrInvalid], 1u);
      } else if (w == 1 || (!pol.adaptive && fabsf(f32_of_f64(Ec)) < ecold[lo])) {
        // Cold: |E| (in FP32, within the margin of ecold) below the field at
        // which the largest window rate reaches 2^kColdLog2F64, 2 W dt <=
        // kThrF64[0].  (The adaptive policy goes the full way.)
        f64_still_cell(J, pol, c, lo, hi);
      } else {
        cls = form_class(estimate_f32(sm.tab32, pol, Ec, lo, w)) * kWidths + (w - 2);
      }
    }
    // append to the class queues; work off every queue holding a full warp
    unsigned todo = __ballot_sync(kFull, cls >= 0);
    while (todo) {
      const int q = __shfl_sync(kFull, cls, __ffs(todo) - 1);
      const unsigned m = __ballot_sync(kFull, cls == q);
      todo &= ~m;
      const int n0 = count[q];
      if (cls == q) queue[q][n0 + __popc(m & below)] = (uint32_t)c;
      int n = n0 + __popc(m);
      __syncwarp();
      if (n >= 32) {
        n -= 32;
        work((int)queue[q][n + lane], q);
        __syncwarp();
      }
      if (lane == 0) count[q] = n;
      __syncwarp();
    }
  }
  // what is left in the queues: the block's warps put theirs together, so
  // that the last, partly filled batches are one per class and block
  __syncthreads();
  int turn = 0;
#pragma unroll 1
  for (int q = 0; q < kClasses; ++q) {
    int total = 0;
    for (int w = 0; w < kWarps; ++w) total += sm.count[w][q];
#pragma unroll 1
    for (int b = 0; b < total; b += 32, ++turn) {
      if (turn % kWarps != wib || b + lane >= total) continue;
      int i = b + lane, w = 0;
      while (i >= sm.count[w][q]) i -= sm.count[w++][q];
      work((int)sm.queue[w][q][i], q);
    }
  }
  __syncwarp();
  if (pol.flags & ION_CONSERVATION_CHECK) warp_max_into(&hdr[kHdrCons], cmax);
}

// One cell per lane, for grids of at most kDirectGroups warps per SM: the
// queues cost a batch per class and block at the end, and save nothing until
// they fill.  Direct against queued, us a step in a graph, nitrogen (Kr-like) cells: 16,384
// 21.6 against 34.2 (33.5, 93.3); 80,000 32.4 against 36.5 (68.6, 141); 120,000 35.9 against
// 36.8 (97.8, 161); 160,000 44.7 against 39.0 (115, 183); 320,000 71.7 against 48.8 (209,
// 235): the line lies between the two gases' crossings, where what the one loses is small
// against what the other gains.  Bound by latency: an FP64 instruction holds its scheduler
// 64 cycles whatever its lanes, and a warp with Taylor and Bateman lanes runs
// both.  A warp runs its lanes' widths one after another (cells
// side by side mostly share theirs); a cell whose FP32 estimate is far below
// the first term's threshold keeps its populations.
constexpr int kDirectThreads = 64;
constexpr int kDirectGroups = 32;

__global__ void __launch_bounds__(kDirectThreads)
    ion_step_f64_direct(const __grid_constant__ JobIO J, const __grid_constant__ Policy pol,
                        uint32_t* hdr) {
  __shared__ StagedF64 tab;
  __shared__ StagedF32 tab32;
  const int c = blockIdx.x * kDirectThreads + threadIdx.x;
  const bool on = c < J.ncells;
  // the cell's inputs travel while the table is staged
  const double E = on ? static_cast<const double*>(J.E)[c] : 0.0;
  const int lo = on ? J.lo[c] : 0, hi = on ? J.hi[c] : 0;
  stage_f64(J.tab, pol.log2dt, &tab);
  stage_f32(J.tab, pol.log2dt, &tab32);
  __syncthreads();
  cudaGridDependencySynchronize();  // the header is zero
  const bool ok = window_ok(lo, hi, J.Z);
  if (on && !ok) atomicAdd(&hdr[kHdrInvalid], 1u);
  int w = on && ok ? hi - lo + 1 : 0;
  if (w == 1 || (w > 1 && !pol.adaptive && estimate_f32(tab32, pol, E, lo, w) < 0x1p-59f)) {
    f64_still_cell(J, pol, c, lo, hi);
    w = 0;
  }
  uint32_t cmax = 0;
  unsigned todo = __ballot_sync(kFull, w > 0);
  while (todo) {
    const int W = __shfl_sync(kFull, w, __ffs(todo) - 1);
    if (w == W) cmax = f64_cell_of(W, J, pol, tab, c, E, lo);
    todo &= ~__ballot_sync(kFull, w == W);
  }
  if (pol.flags & ION_CONSERVATION_CHECK) warp_max_into(&hdr[kHdrCons], cmax);
}

std::mutex g_mu;
constexpr int kMaxDevices = 64;
int g_fit[kMaxDevices] = {};  // resident blocks per SM, per device (0: not yet)

}  // namespace

cudaError_t launch_step_f64(const JobIO& job, const Policy& pol, uint32_t* hdr, bool first,
                            bool dependent, cudaStream_t s) {
  dependent = dependent && first;
  if (job.ncells == 0) return cudaSuccess;
  int dev = 0, fit = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
    return e;
  const int64_t groups = ((int64_t)job.ncells + 31) / 32;
  if (groups <= (int64_t)kDirectGroups * sms) {
    const unsigned blocks = (job.ncells + kDirectThreads - 1) / kDirectThreads;
    return launch_after(dependent, ion_step_f64_direct, blocks, kDirectThreads, 0, s, job, pol,
                        hdr);
  }
  {
    std::lock_guard<std::mutex> lock(g_mu);
    const bool cache = dev >= 0 && dev < kMaxDevices;
    if (cache) fit = g_fit[dev];
    if (fit < 1) {
      if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, ion_step_f64_kernel,
                                                             kThreads, 0)) != cudaSuccess)
        return e;
      fit = fit < 1 ? 1 : fit;
      if (cache) g_fit[dev] = fit;
    }
  }
  // the group counter starts at 0 for every job (the caller has cleared the
  // header for the first)
  if (!first &&
      (e = cudaMemsetAsync(hdr + kHdrChunk, 0, sizeof(uint32_t), s)) != cudaSuccess)
    return e;
  const int64_t need = (groups + kWarps - 1) / kWarps;
  const int64_t cap = (int64_t)fit * sms;
  const int blocks = (int)(need < cap ? need : cap);
  return launch_after(dependent, ion_step_f64_kernel, blocks, kThreads, 0, s, job, pol, hdr);
}

}  // namespace ion
