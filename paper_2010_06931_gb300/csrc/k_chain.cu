// Time-ordered chain of each scan's A-scans (the temporal regulariser's pairs,
// Ploner et al., Sec. 2.1): the previous and next A-scan in acquisition order
// (by time, then by index) and the weight dt_min / dt of each pair.
//
// A raster scan's times increase along its rows or along its columns, and then
// the order needs no sort: one kernel tests both orders and takes the smallest
// positive time step of each, the next writes the chain of the order that
// holds.  Times in neither order are sorted by the caller on the host.
// Differences, quotients and the order are those of the host's float64
// arithmetic, so both give the same chain.  300 x 300 A-scans, 3 levels, both
// scans: 7.3 ms of host sorts -> about 60 us.
#include "common.cuh"

namespace octmc {
namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ int64_t at_row(int64_t m, int, int) { return m; }
__device__ __forceinline__ int64_t at_col(int64_t m, int w, int h) { return (m % h) * w + m / h; }

// Position m and m + 1 of one order: whether A-scan a comes before b, and the step.
__device__ __forceinline__ void step_of(const double* __restrict__ t, int64_t a, int64_t b, bool* bad,
                                        unsigned long long* dt) {
  const double ta = t[a], tb = t[b];
  if (!(ta < tb || (ta == tb && a < b))) *bad = true;
  const double s = tb - ta;
  if (s > 0.0) *dt = min(*dt, (unsigned long long)__double_as_longlong(s));  // positive: ordered as integers
}

__global__ void __launch_bounds__(kThreads) chain_scan_kernel(const double* __restrict__ t, int w, int h,
                                                              ChainInfo* info) {
  const int64_t n = (int64_t)w * h;
  bool bad_r = false, bad_c = false, nonfin = false;
  unsigned long long dr = 0x7ff0000000000000ull, dc = dr;
  for (int64_t m = (int64_t)blockIdx.x * kThreads + threadIdx.x; m < n; m += (int64_t)gridDim.x * kThreads) {
    if (!isfinite(t[m])) nonfin = true;
    if (m + 1 < n) {
      step_of(t, at_row(m, w, h), at_row(m + 1, w, h), &bad_r, &dr);
      step_of(t, at_col(m, w, h), at_col(m + 1, w, h), &bad_c, &dc);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    dr = min(dr, __shfl_xor_sync(0xffffffffu, dr, o));
    dc = min(dc, __shfl_xor_sync(0xffffffffu, dc, o));
  }
  const bool any_r = __any_sync(0xffffffffu, bad_r), any_c = __any_sync(0xffffffffu, bad_c),
             any_n = __any_sync(0xffffffffu, nonfin);
  if ((threadIdx.x & 31) == 0) {
    if (any_r) atomicOr(&info->row_bad, 1u);
    if (any_c) atomicOr(&info->col_bad, 1u);
    if (any_n) atomicOr(&info->nonfinite, 1u);
    atomicMin(&info->row_dt, dr);
    atomicMin(&info->col_dt, dc);
  }
}

__global__ void __launch_bounds__(kThreads) chain_write_kernel(const double* __restrict__ t, int w, int h,
                                                               const ChainInfo* __restrict__ info, int* prev, int* next,
                                                               float* wprev, float* wnext) {
  const bool row = !info->row_bad;
  if (!row && info->col_bad) return;  // neither order: sorted on the host
  const int64_t n = (int64_t)w * h;
  const double dtmin = __longlong_as_double((long long)(row ? info->row_dt : info->col_dt));
  auto at = [&](int64_t m) { return row ? at_row(m, w, h) : at_col(m, w, h); };
  for (int64_t m = (int64_t)blockIdx.x * kThreads + threadIdx.x; m < n; m += (int64_t)gridDim.x * kThreads) {
    const int64_t a = at(m);
    if (m == 0) {
      prev[a] = -1;
      wprev[a] = 0.f;
    }
    if (m + 1 == n) {
      next[a] = -1;
      wnext[a] = 0.f;
    } else {
      const int64_t b = at(m + 1);
      const float om = (float)(isinf(dtmin) ? 1.0 : dtmin / fmax(t[b] - t[a], dtmin));
      next[a] = (int)b;
      wnext[a] = om;
      prev[b] = (int)a;
      wprev[b] = om;
    }
  }
}

// 2 x 2 mean of the sampling times, odd sizes repeat the edge.
__global__ void __launch_bounds__(kThreads) time_down_kernel(const double* __restrict__ t, int w, int h,
                                                             double* __restrict__ out) {
  const int w2 = (w + 1) / 2, h2 = (h + 1) / 2;
  const int64_t n = (int64_t)w2 * h2;
  for (int64_t e = (int64_t)blockIdx.x * kThreads + threadIdx.x; e < n; e += (int64_t)gridDim.x * kThreads) {
    const int i = (int)(e % w2), j = (int)(e / w2);
    const int i1 = min(2 * i + 1, w - 1), j1 = min(2 * j + 1, h - 1);
    out[e] = (t[(int64_t)2 * j * w + 2 * i] + t[(int64_t)2 * j * w + i1] + t[(int64_t)j1 * w + 2 * i] +
              t[(int64_t)j1 * w + i1]) /
             4.0;
  }
}

inline unsigned grid_for(int64_t n) {
  int64_t b = (n + kThreads - 1) / kThreads;
  return (unsigned)(b < 1 ? 1 : (b > 8 * 152 ? 8 * 152 : b));
}

}  // namespace

cudaError_t launch_chain_scan(const double* t, int w, int h, ChainInfo* info, cudaStream_t s) {
  chain_scan_kernel<<<grid_for((int64_t)w * h), kThreads, 0, s>>>(t, w, h, info);
  return cudaGetLastError();
}

cudaError_t launch_chain_write(const double* t, int w, int h, const ChainInfo* info, int* prev, int* next, float* wprev,
                               float* wnext, cudaStream_t s) {
  chain_write_kernel<<<grid_for((int64_t)w * h), kThreads, 0, s>>>(t, w, h, info, prev, next, wprev, wnext);
  return cudaGetLastError();
}

cudaError_t launch_time_down(const double* t, int w, int h, double* out, cudaStream_t s) {
  time_down_kernel<<<grid_for((int64_t)((w + 1) / 2) * ((h + 1) / 2)), kThreads, 0, s>>>(t, w, h, out);
  return cudaGetLastError();
}

}  // namespace octmc
