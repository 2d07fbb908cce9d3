// Vector kernels of the on-device L-BFGS (Ploner et al. Sec. 2.1:
// "gradient-based L-BFGS solver"): dot products of the history with probe
// vectors, the direction as a linear combination, pair differences and axpy.
//
// Everything is float64: the history pairs, the products with them (FMAs
// on doubles) and their sums.  Each thread sums a strided share of the
// elements, warps reduce with a fixed butterfly and blocks with fixed
// trees, so every result is deterministic.
#include <algorithm>

#include "common.cuh"

namespace octmc {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kHistChunk = 6;          // history vectors per block row
constexpr int kVals = 2 * kHistChunk + 2;  // sums per block row: h . q0, h . q1, then q0 . q0, q1 . q1

__device__ bool last_block_2d(unsigned* counter) {
  __shared__ bool is_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned t = atomicAdd(counter, 1u);
    is_last = (t == gridDim.x * gridDim.y - 1);
  }
  __syncthreads();
  if (is_last) __threadfence();
  return is_last;
}

__device__ __forceinline__ unsigned long long abs_bits(double v) {
  return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}

// grid (G, rows): block (bx, r) takes history vectors r*6 .. r*6+5 over
// a contiguous share of the n elements; row 0 also takes
// q0.q0, q1.q1 and max|q1| (the maximum on the bit patterns: exact, and NaN
// wins).  Compiled for the probes that are given (kQ0, kQ1): bound by the
// float64 pipe (0.50 T FMA/s measured), so the products with an absent probe
// are left out.  16 vectors and one probe of 540000 elements: 86 -> 48 us
// with two blocks per SM; three, so that the three rows of 16 vectors are all
// resident, take another 13 us (whole direction 99.7 -> 86.5 us; two rows of 8
// or 10 vectors at two blocks per SM: 89.8, 86.9 us).
// partials layout: [output][G].
template <bool kQ0, bool kQ1>
__global__ void __launch_bounds__(kThreads, 3) hist_dots_kernel(const HistDots D, int64_t n, double* partials,
                                                                unsigned* counter, double* out) {
  __shared__ double sm[32 * kWarps];
  __shared__ unsigned long long smx[kWarps];
  const int G = gridDim.x;
  const int k0 = blockIdx.y * kHistChunk;
  const int kn = min(kHistChunk, D.K - k0);  // <= 0 only in row 0 of an empty history
  const bool first = blockIdx.y == 0;
  const double* h[kHistChunk];
#pragma unroll
  for (int k = 0; k < kHistChunk; k++) h[k] = (k < kn) ? D.h[k0 + k] : nullptr;
  // v[2 k] = h_k . q0, v[2 k + 1] = h_k . q1, then q0 . q0, q1 . q1
  static_assert(kVals <= 32, "one reduce-scatter");
  double v[32];
#pragma unroll
  for (int k = 0; k < 32; k++) v[k] = 0.0;
  unsigned long long mx = 0ull;
  const int64_t share = ((n + G - 1) / G + 31) / 32 * 32;
  const int64_t e0 = min(n, (int64_t)blockIdx.x * share), e1 = min(n, e0 + share);
  for (int64_t e = e0 + threadIdx.x; e < e1; e += kThreads) {
    const double p0 = kQ0 ? __ldg(D.q0 + e) : 0.0;
    const double p1 = kQ1 ? __ldg(D.q1 + e) : 0.0;
#pragma unroll
    for (int k = 0; k < kHistChunk; k++) {
      if (k < kn) {
        const double hv = __ldg(h[k] + e);
        if (kQ0) v[2 * k] = fma(hv, p0, v[2 * k]);
        if (kQ1) v[2 * k + 1] = fma(hv, p1, v[2 * k + 1]);
      }
    }
    if (first) {
      if (kQ0) v[2 * kHistChunk] = fma(p0, p0, v[2 * kHistChunk]);
      if (kQ1) {
        v[2 * kHistChunk + 1] = fma(p1, p1, v[2 * kHistChunk + 1]);
        mx = max(mx, abs_bits(p1));
      }
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  sm[lane * kWarps + warp] = warp_reduce_scatter32(v, lane);
  if (kQ1 && first) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) smx[warp] = mx;
  }
  __syncthreads();
  const int t = threadIdx.x;
  int o = -1;
  if (t < 2 * max(kn, 0)) o = 2 * k0 + t;
  else if (first && t >= 2 * kHistChunk && t < kVals) o = 2 * D.K + (t - 2 * kHistChunk);
  if (o >= 0) {
    double s = 0.0;
    for (int w = 0; w < kWarps; w++) s += sm[t * kWarps + w];
    partials[(int64_t)o * G + blockIdx.x] = s;
  }
  if (first && t == kVals) {
    unsigned long long m = 0ull;
    if (kQ1)
      for (int w = 0; w < kWarps; w++) m = max(m, smx[w]);
    partials[(int64_t)(2 * D.K + 2) * G + blockIdx.x] = __longlong_as_double((long long)m);
  }
  if (last_block_2d(counter)) {
    // one warp per output: lanes take a fixed strided share of the blocks,
    // then a butterfly
    const int nout = hist_dots_outputs(D.K);
    for (int o = warp; o < nout; o += kWarps) {
      const bool is_max = (o == nout - 1);
      double s = 0.0;
      unsigned long long m = 0ull;
      for (int bx = lane; bx < G; bx += 32) {
        const double u = partials[(int64_t)o * G + bx];
        if (is_max) m = max(m, (unsigned long long)__double_as_longlong(u));
        else s += u;
      }
      if (is_max) {
#pragma unroll
        for (int x = 16; x > 0; x >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, x));
      } else {
        s = warp_sum(s);
      }
      if (lane == 0) out[o] = is_max ? __longlong_as_double((long long)m) : s;
    }
    __syncthreads();
    if (threadIdx.x == 0) *counter = 0u;
  }
}

// out = cg g + sum_k c_k h_k in float64, the terms added in a fixed order.
__global__ void __launch_bounds__(kThreads) hist_comb_kernel(const HistComb C, int64_t n, double* __restrict__ out) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    double s = 0.0;
#pragma unroll 8
    for (int k = 0; k < C.K; k++) s = fma(C.c[k], C.h[k][e], s);
    out[e] = fma(C.cg, C.g[e], s);
  }
}

__global__ void sub2_kernel(const double* __restrict__ x1, const double* __restrict__ x0,
                            const double* __restrict__ g1, const double* __restrict__ g0,
                            double* __restrict__ s, double* __restrict__ y, int64_t n) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    s[e] = x1[e] - x0[e];
    y[e] = g1[e] - g0[e];
  }
}

__global__ void axpy_kernel(const double* __restrict__ x, double a, const double* __restrict__ d,
                            double* __restrict__ out, int64_t n) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x)
    out[e] = fma(a, d[e], x[e]);
}

inline unsigned grid_for(int64_t n) {
  int64_t b = (n + kThreads - 1) / kThreads;
  if (b < 1) b = 1;
  if (b > 4 * 152) b = 4 * 152;
  return (unsigned)b;
}

}  // namespace

// Blocks per row: one per SM, fewer on short vectors.
int hist_dots_blocks(int64_t n) {
  const int64_t b = (n + kThreads - 1) / kThreads;
  return (int)(b < 1 ? 1 : std::min<int64_t>(b, device_sm_count()));
}

cudaError_t launch_hist_dots(const HistDots& hd, int64_t n, double* partials, unsigned* counter, double* out,
                             cudaStream_t s) {
  if (hd.K < 0 || hd.K > kMaxHist || (!hd.q0 && !hd.q1)) return cudaErrorInvalidValue;
  const int G = hist_dots_blocks(n);
  const int rows = hd.K > 0 ? (hd.K + kHistChunk - 1) / kHistChunk : 1;
  const dim3 g(G, rows);
  if (hd.q0 && hd.q1) hist_dots_kernel<true, true><<<g, kThreads, 0, s>>>(hd, n, partials, counter, out);
  else if (hd.q0) hist_dots_kernel<true, false><<<g, kThreads, 0, s>>>(hd, n, partials, counter, out);
  else hist_dots_kernel<false, true><<<g, kThreads, 0, s>>>(hd, n, partials, counter, out);
  return cudaGetLastError();
}

cudaError_t launch_hist_comb(const HistComb& hc, int64_t n, double* out, cudaStream_t s) {
  if (hc.K < 0 || hc.K > kMaxHist) return cudaErrorInvalidValue;
  hist_comb_kernel<<<grid_for(n), kThreads, 0, s>>>(hc, n, out);
  return cudaGetLastError();
}

cudaError_t launch_sub2(const double* x1, const double* x0, const double* g1, const double* g0,
                        double* s_out, double* y_out, int64_t n, cudaStream_t st) {
  sub2_kernel<<<grid_for(n), kThreads, 0, st>>>(x1, x0, g1, g0, s_out, y_out, n);
  return cudaGetLastError();
}

cudaError_t launch_axpy(const double* x, double a, const double* d, double* out, int64_t n,
                        cudaStream_t s) {
  axpy_kernel<<<grid_for(n), kThreads, 0, s>>>(x, a, d, out, n);
  return cudaGetLastError();
}

}  // namespace octmc
