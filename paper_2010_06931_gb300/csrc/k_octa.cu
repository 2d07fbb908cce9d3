// Angiography preprocessing of one scan (Ploner et al., Sec. 2.2 and 2.3):
// saccade validity of the B-scans and the en-face OCTA projection.
//
//   bscan_sum_kernel     per-B-scan sums (groups of 8 samples summed exactly in
//                        float, then float64, fixed tree per block): mean
//                        decorrelation of each B-scan, and the OCT sums for
//                        the OCT threshold
//   validity_kernel      mu, sigma of the B-scan means, the 3-sigma test and
//                        the +-2 B-scan dilation (one block, float64)
//   median3_kernel       3x3x3 median per voxel (edge replicated): the 27
//                        samples sorted along depth, y and x where outputs
//                        share them, 14 dropped on either side of the median,
//                        forgetful selection of the median of the 13 others
//   rank15_kernel        3rd smallest of 15 samples along x or y (edge
//                        replicated) from running 3 smallest of half windows
//   select_init_kernel   the ranks of the percentiles' order statistics
//   radix_hist_kernel /  exact order statistics of the filtered voxels of the
//   radix_pick_kernel    valid B-scans by 3 passes of 11-bit (last 10-bit)
//                        radix selection on order-preserving integer keys
//                        (integer histograms: deterministic)
//   finish_kernel        percentiles (linear interpolation), the mask cut
//                        and the OCT threshold (float64, one warp)
//   project_kernel       per A-scan (one warp): mean of the OCTA voxels whose
//                        filtered value is below the cut and whose OCT value
//                        is above the threshold
//   bscan_median_kernel  median of each B-scan's en-face values (bitonic sort
//                        in shared memory) subtracted from them
//   replace_kernel       invalid B-scans take the nearest valid one
//
// Volumes are float32 [h][w][d], depth contiguous.  B-scans of an X-fast
// scan (fast_axis 0) are the rows j, of a Y-fast scan the columns i.
#include <algorithm>
#include <cmath>
#include <new>

#include "common.cuh"

namespace octmc {
namespace {

constexpr int kT = 256;
constexpr int kRadixBins = 2048;
constexpr int kTargets = 4;  // order statistics: floor/ceil positions of two percentiles

struct Select {
  int any;            // some B-scan is valid
  int nvalid;
  unsigned long long kept;  // voxels in both masks
  // per target: rank (0-based) among the selected voxels, key prefix found so
  // far, and the value once known
  long long rank[kTargets];
  unsigned prefix[kTargets];
  float value[kTargets];
  double pos[2];      // q (n - 1) of the two percentiles
  double p[2];        // the percentiles
  double cut;         // p_lo + thresh (p_hi - p_lo)
  double t_oct;       // OCT threshold
  float cut_f;        // smallest float >= cut: x < cut  <=>  x < cut_f
  float toct_f;       // largest float <= t_oct: x > t_oct <=> x > toct_f
};

__device__ __forceinline__ int64_t ascan_of(int w, int fast_axis, int b, int f) {
  return fast_axis == 0 ? (int64_t)b * w + f : (int64_t)f * w + b;
}

// ---------------------------------------------------------------- sums
// Block b sums the voxels of B-scan b (nf columns of d samples).  vec: the
// columns are 16-byte aligned and d is a multiple of 4; each lane then takes 8
// samples at a time, summed exactly in float (exact_sum8), so 2 float64
// additions replace 8 and the sum's error is no larger.  Bound by HBM once
// they do: 300 x 300 x 512 117 -> 37 us.
constexpr int kSumThreads = 1024;
__global__ void __launch_bounds__(kSumThreads) bscan_sum_kernel(const float* __restrict__ vol, int w, int h, int d,
                                                                int fast_axis, bool vec, double* __restrict__ sums) {
  const int b = blockIdx.x;
  const int nf = fast_axis == 0 ? w : h;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // two independent chains per lane for the float64 latency
  double acc0 = 0.0, acc1 = 0.0;
  for (int f = warp; f < nf; f += kSumThreads / 32) {
    const float* col = vol + ascan_of(w, fast_axis, b, f) * d;
    if (vec) {
      const float4* c4 = reinterpret_cast<const float4*>(col);
      const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int g = lane; g < d / 4; g += 64) {
        const float4 u = c4[g], v = g + 32 < d / 4 ? c4[g + 32] : zero;
        const float x[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
        float s, e;
        if (exact_sum8(x, &s, &e)) {
          acc0 += widen_exact(s);
          acc1 += widen_exact(e);
        } else {
#pragma unroll
          for (int k = 0; k < 8; k += 2) {
            acc0 += widen_exact(x[k]);
            acc1 += widen_exact(x[k + 1]);
          }
        }
      }
    } else {
      int k = lane;
      for (; k + 32 < d; k += 64) {
        acc0 += widen_exact(col[k]);
        acc1 += widen_exact(col[k + 32]);
      }
      if (k < d) acc0 += widen_exact(col[k]);
    }
  }
  double acc = warp_sum(acc0 + acc1);
  __shared__ double sm[kSumThreads / 32];
  if (lane == 0) sm[warp] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < kSumThreads / 32; i++) t += sm[i];
    sums[b] = t;
  }
}

// One block: means, mu, sigma, saturation test, validity.
__global__ void __launch_bounds__(1024) validity_kernel(const double* sums, int nb, double per, float* __restrict__ v,
                                                        double* means) {
  __shared__ double sm[32];
  __shared__ double s_mu, s_sig;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  double a = 0.0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) a += sums[b] / per;
  a = warp_sum(a);
  if (lane == 0) sm[warp] = a;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < nw; i++) t += sm[i];
    s_mu = t / nb;
  }
  __syncthreads();
  const double mu = s_mu;
  double q = 0.0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    const double m = sums[b] / per;
    q += (m - mu) * (m - mu);
  }
  q = warp_sum(q);
  __syncthreads();
  if (lane == 0) sm[warp] = q;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < nw; i++) t += sm[i];
    s_sig = sqrt(t / nb);
  }
  __syncthreads();
  const double lim = mu + 3.0 * s_sig;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    bool ok = true;
    for (int o = -2; o <= 2; o++) {
      const int c = b + o;
      if (c >= 0 && c < nb && sums[c] / per > lim) ok = false;
    }
    v[b] = ok ? 1.0f : 0.0f;
  }
  __syncthreads();  // sums may be the means' own buffer
  if (means)
    for (int b = threadIdx.x; b < nb; b += blockDim.x) means[b] = sums[b] / per;
}

// ---------------------------------------------------------------- filters
__device__ __forceinline__ int clampn(int i, int n) { return i < 0 ? 0 : (i >= n ? n - 1 : i); }

__device__ __forceinline__ void cmpx(float& a, float& b) {  // a <- min, b <- max
  const float mn = fminf(a, b), mx = fmaxf(a, b);
  a = mn;
  b = mx;
}

// Forgetful selection of the median of N = W + M values: a[0..W-1] holds
// the first W, rest[0..M-1] the others (W = (N+1)/2 + 1).  Each step moves
// the minimum of the current window a[LO..W-1] to a[LO] and its maximum to
// a[W-1], forgets both (the window start advances, the next value replaces
// the maximum); three candidates remain and the median is their middle one.
template <int W, int M, int LO = 0>
__device__ __forceinline__ void forget_steps(float (&a)[W], const float (&rest)[M]) {
  if constexpr (LO < M) {
    cmpx(a[LO], a[W - 1]);
#pragma unroll
    for (int i = LO + 1; i < W - 1; i++) {
      cmpx(a[LO], a[i]);
      cmpx(a[i], a[W - 1]);
    }
    a[W - 1] = rest[LO];
    forget_steps<W, M, LO + 1>(a, rest);
  }
}

__device__ __forceinline__ float median3_of(float x, float y, float z) {
  return fmaxf(fminf(x, y), fminf(fmaxf(x, y), z));
}

__device__ __forceinline__ void sort3(float& a, float& b, float& c) {
  cmpx(a, b);
  cmpx(b, c);
  cmpx(a, b);
}
// a <= b <= c with one end not needed (5 instead of 6 minima and maxima)
__device__ __forceinline__ void upper2(float a, float& b, float& c) {  // b, c: the two larger
  cmpx(a, b);
  cmpx(b, c);
  b = fmaxf(a, b);
}
__device__ __forceinline__ void lower2(float& a, float& b, float c) {  // a, b: the two smaller
  cmpx(b, c);
  cmpx(a, b);
  b = fminf(b, c);
}

// The samples of one column i over the rows j-1..j+1 and depths k-1..k+1:
// sorted along depth into lows, mids and highs, and each of these along j.
struct Slab {
  float lo[3], mid[3], hi[3];
};

// The median of the 27 samples of three neighbouring slabs.  In the order of
// the 27 the 5 smallest lows and the 2 smallest mids lie at or below the median
// (each has at least 14 values at or above it), the 5 largest highs and the 2
// largest mids at or above it; 13 others remain -- the 4 largest lows, the
// middle 5 mids, the 4 smallest highs -- and the median is theirs.  Each class
// is a 3 x 3 matrix sorted along j; sorted along i too (both orders hold
// then), its extremes sit in known places: of 9 lows M[r][c], M[2][2], M[2][1]
// and M[1][2] are the 3 largest with the maximum of M[2][0], M[0][2], M[1][1]
// the fourth, and so on.
__device__ __forceinline__ float median27(const Slab& A, const Slab& B, const Slab& C) {
  // lows: l22 >= l21, l12, l4
  float l20 = A.lo[2], l21 = B.lo[2], l22 = C.lo[2];
  sort3(l20, l21, l22);
  float l11 = B.lo[1], l12 = C.lo[1];
  upper2(A.lo[1], l11, l12);
  const float l02 = fmaxf(fmaxf(A.lo[0], B.lo[0]), C.lo[0]);
  float l4 = fmaxf(fmaxf(l20, l02), l11);
  // highs: h00 <= h01, h10, h4
  float h00 = A.hi[0], h01 = B.hi[0], h02 = C.hi[0];
  sort3(h00, h01, h02);
  float h10 = A.hi[1], h11 = B.hi[1];
  lower2(h10, h11, C.hi[1]);
  const float h20 = fminf(fminf(A.hi[2], B.hi[2]), C.hi[2]);
  float h4 = fminf(fminf(h02, h20), h11);
  // mids: the middle 5
  float m01 = B.mid[0], m02 = C.mid[0];
  upper2(A.mid[0], m01, m02);
  float m10 = A.mid[1], m11 = B.mid[1], m12 = C.mid[1];
  sort3(m10, m11, m12);
  float m20 = A.mid[2], m21 = B.mid[2];
  lower2(m20, m21, C.mid[2]);
  const float ma = fmaxf(m01, m10), mb = fminf(m12, m21);
  // the first window: 4 lows and 4 highs.  Its minimum is among l21, l12, l4 and
  // h00 (l22 is the largest low, h00 the smallest high), its maximum among l22,
  // h01, h10 and h4: 6 exchanges instead of 13
  cmpx(l4, l21);
  cmpx(l4, l12);
  cmpx(l4, h00);
  cmpx(l22, h4);
  cmpx(h01, h4);
  cmpx(h10, h4);
  // l4 and h4 dropped; 6 + 1 in the window, 4 to come
  float a[7] = {l21, l12, h00, l22, h01, h10, ma};
  const float rest[4] = {mb, m02, m20, m11};
  forget_steps<7, 4>(a, rest);
  return median3_of(a[4], a[5], a[6]);
}

// The median of 27 samples some of which may be NaN: a minimum or maximum of a
// NaN and a number is the number, so which numbers take the NaNs' places
// depends on the order of the exchanges.  This order defines it: the 9 columns
// r[0..2] + o[0..2] sorted along depth, then the 13 values that median27 keeps
// by partial selection over the 9 lows, mids and highs.
__device__ __forceinline__ float median27_nan(const float* const r[3], const int64_t o[3], int km, int kp) {
  float lo[9], mid[9], hi[9];
#pragma unroll
  for (int c = 0; c < 9; c++) {
    const float* col = r[c / 3] + o[c % 3];
    lo[c] = __ldg(col + km);
    mid[c] = __ldg(col);
    hi[c] = __ldg(col + kp);
    sort3(lo[c], mid[c], hi[c]);
  }
#pragma unroll
  for (int e = 8; e >= 5; e--)  // the 4 largest lows
#pragma unroll
    for (int i = 0; i < e; i++) cmpx(lo[i], lo[e]);
#pragma unroll
  for (int b = 0; b <= 3; b++)  // the 4 smallest highs
#pragma unroll
    for (int i = b + 1; i < 9; i++) cmpx(hi[b], hi[i]);
#pragma unroll
  for (int q = 0; q < 2; q++) {  // the middle 5 mids
    cmpx(mid[q], mid[8 - q]);
#pragma unroll
    for (int i = q + 1; i < 8 - q; i++) {
      cmpx(mid[q], mid[i]);
      cmpx(mid[i], mid[8 - q]);
    }
  }
  float a[8] = {lo[5], lo[6], lo[7], lo[8], mid[2], mid[3], mid[4], mid[5]};
  const float rest[5] = {mid[6], hi[0], hi[1], hi[2], hi[3]};
  forget_steps<8, 5>(a, rest);
  return median3_of(a[5], a[6], a[7]);
}

constexpr int kSx = 32, kSy = 8;

// The medians of columns i0..i0+n-1 at (j, k) where a sample may be NaN.  Out
// of line: strips of numbers never come here.
__device__ __noinline__ void median_strip_nan(const float* __restrict__ in, int w, int h, int d, int i0, int n, int j,
                                              int k, float* __restrict__ out) {
  const int64_t row = (int64_t)w * d;
  const float* r[3] = {in + clampn(j - 1, h) * row + k, in + j * row + k, in + clampn(j + 1, h) * row + k};
  const int km = k > 0 ? -1 : 0, kp = k + 1 < d ? 1 : 0;
#pragma unroll 1
  for (int i = i0; i < i0 + n; i++) {
    const int64_t o[3] = {(int64_t)clampn(i - 1, w) * d, (int64_t)i * d, (int64_t)clampn(i + 1, w) * d};
    out[j * row + o[1] + k] = median27_nan(r, o, km, kp);
  }
}

// Block (32 depths, 8 strips), grid (depth chunks, groups of strips, rows): a
// thread walks kMedI consecutive columns i of one row, so each slab's 18
// exchanges are made once for three medians, which then take 64 more: 86 per
// voxel with the strips' ends (150 when every voxel sorted its own 27 samples).
// Bound by the minimum / maximum rate (62 lanes per clock and SM measured; the
// pipe is 90 % busy): 300 x 300 x 512 851 -> 454 us, with the sum that finds NaNs
// taken per strip (a test per window costs 32 us more).
constexpr int kMedI = 10;
__global__ void __launch_bounds__(kSx * kSy) median3_kernel(const float* __restrict__ in, int w, int h, int d,
                                                            float* __restrict__ out) {
  const int k = blockIdx.x * kSx + threadIdx.x;
  const int i0 = (blockIdx.y * kSy + threadIdx.y) * kMedI;
  const int j = blockIdx.z;
  if (k >= d || i0 >= w) return;
  const int64_t row = (int64_t)w * d;
  const float* r[3] = {in + clampn(j - 1, h) * row + k, in + j * row + k, in + clampn(j + 1, h) * row + k};
  const int km = k > 0 ? -1 : 0, kp = k + 1 < d ? 1 : 0;
  float sum = 0.f;  // of all samples: NaN if one of them is (or infinities of both signs are among them)
  auto slab = [&](int i, Slab& S) {
    const int64_t o = (int64_t)clampn(i, w) * d;
    float part = 0.f;
#pragma unroll
    for (int q = 0; q < 3; q++) {
      S.lo[q] = __ldg(r[q] + o + km);
      S.mid[q] = __ldg(r[q] + o);
      S.hi[q] = __ldg(r[q] + o + kp);
      part += S.lo[q] + S.mid[q] + S.hi[q];
      sort3(S.lo[q], S.mid[q], S.hi[q]);
    }
    sum += part;
    sort3(S.lo[0], S.lo[1], S.lo[2]);
    sort3(S.mid[0], S.mid[1], S.mid[2]);
    sort3(S.hi[0], S.hi[1], S.hi[2]);
  };
  Slab A, B, C;
  slab(i0 - 1, A);
  slab(i0, B);
  float* o = out + j * row + (int64_t)i0 * d + k;
  const int n = min(kMedI, w - i0);
  for (int q = 0; q < n; q++, o += d) {
    slab(i0 + q + 1, C);
    *o = median27(A, B, C);
    A = B;
    B = C;
  }
  if (sum != sum) median_strip_nan(in, w, h, d, i0, n, j, k, out);
}

// The 3 smallest of a running set, sorted.
struct Low3 {
  float a, b, c;
  __device__ __forceinline__ void add(float x) {
    const float t = fmaxf(a, x);
    a = fminf(a, x);
    const float u = fmaxf(b, t);
    b = fminf(b, t);
    c = fminf(c, u);
  }
};

// The outputs of one segment where a sample may be NaN: each window's samples
// in turn.  A NaN repeats the smallest sample before it in the window, so the
// split windows of rank15_kernel would give other values.
constexpr int kSeg = 15, kRad = 7;
__device__ __forceinline__ void rank_segment_nan(const float* c, int n, int64_t stride, int p0, float* o) {
#pragma unroll 1
  for (int u = 0; u < kSeg && p0 + u < n; u++) {
    Low3 s = {INFINITY, INFINITY, INFINITY};
#pragma unroll 1
    for (int t = -kRad; t <= kRad; t++) s.add(__ldg(c + clampn(p0 + u + t, n) * stride));
    o[u * stride] = s.c;
  }
}

// 3rd smallest of the 15 samples p-7..p+7 along an axis.  A thread makes the 15
// outputs of one segment at one depth: the windows split at the segment's
// centre into a part of the 15 samples before and a part of the 14 after it, whose 3
// smallest run along (5 minima / maxima per sample), and the 3rd smallest of
// the two triples is min(s3, p3, max(s1, p2), max(s2, p1)): 15 per output and 2
// loads instead of 75 and 15.  n, stride: length and stride of the axis; m,
// ostride: the other transverse axis.  Bound by the minimum / maximum rate (79 %
// busy; HBM 48 %): 300 x 300 x 512 86 us along either axis (381 and 488 us one
// window per thread; 100 us at the 70 registers it takes without the sum).
__global__ void __launch_bounds__(kSx * kSy) rank15_kernel(const float* __restrict__ in, int n, int64_t stride, int m,
                                                           int64_t ostride, int d, float* __restrict__ out) {
  const int k = blockIdx.x * kSx + threadIdx.x;
  if (k >= d) return;
  for (int other = blockIdx.z * kSy + threadIdx.y; other < m; other += gridDim.z * kSy)
    for (int seg = blockIdx.y; seg * kSeg < n; seg += gridDim.y) {
      const int p0 = seg * kSeg;
      const float* c = in + other * ostride + k;
      float* o = out + other * ostride + (int64_t)p0 * stride + k;
      float x[kSeg], sum = 0.f;  // sum: of all samples, as in median3_kernel
#pragma unroll
      for (int t = 0; t < kSeg; t++) {
        x[t] = __ldg(c + clampn(p0 - kRad + t, n) * stride);
        sum += x[t];
      }
      Low3 suf[kSeg];  // suf[t]: of x[t..14]
      suf[kSeg - 1] = {x[kSeg - 1], INFINITY, INFINITY};
#pragma unroll
      for (int t = kSeg - 2; t >= 0; t--) {
        suf[t] = suf[t + 1];
        suf[t].add(x[t]);
      }
      Low3 pre = {INFINITY, INFINITY, INFINITY};
#pragma unroll
      for (int u = 0; u < kSeg; u++) {
        if (p0 + u < n)
          o[u * stride] = fminf(fminf(suf[u].c, pre.c), fminf(fmaxf(suf[u].a, pre.b), fmaxf(suf[u].b, pre.a)));
        if (u + 1 < kSeg) {
          const float y = __ldg(c + clampn(p0 + kRad + 1 + u, n) * stride);
          sum += y;
          pre.add(y);
        }
      }
      if (sum != sum) rank_segment_nan(c, n, stride, p0, o);
    }
}

// ---------------------------------------------------------------- selection
__device__ __forceinline__ unsigned order_key(float x) {
  const unsigned u = __float_as_uint(x);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_value(unsigned k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// digit pass `pass` (0: bits 31..21, 1: 20..10, 2: 9..0)
__device__ __forceinline__ int digit_shift(int pass) { return pass == 0 ? 21 : (pass == 1 ? 10 : 0); }
__device__ __forceinline__ unsigned digit_mask(int pass) { return pass == 2 ? 0x3ffu : 0x7ffu; }

// Histogram of the current digit of the selected voxels whose higher digits
// equal each target's prefix.  hist [kTargets][kRadixBins]; targets with the
// same prefix share one count (U distinct prefixes, 1 in the first pass).
// Each thread takes runs of kRun consecutive voxels and counts equal
// consecutive digits in registers before one shared atomic per run of equal
// digits: the filtered volume is smooth along depth, so the few hot bins of the
// leading digit (sign and exponent) are not hammered.  Bound by issue; the
// prefix test is compiled for the number of distinct prefixes: 300 x 300 x 512
// 63 / 93 / 55 us for the three passes (131 / 147 / 116 us with the test of
// all four targets at every voxel).
constexpr int kRun = 16;
template <int U>
__device__ __forceinline__ void hist_runs(const float* __restrict__ vol, int w, unsigned d, int64_t n, int fast_axis,
                                          const float* __restrict__ v, bool any, int hs, int sft, unsigned msk,
                                          const unsigned* pre, unsigned (*sh)[kRadixBins]) {
  const int64_t nrun = (n + kRun - 1) / kRun;
  auto selected = [&](int64_t p) {
    if (!any) return true;
    return v[fast_axis == 0 ? (unsigned)(p / w) : (unsigned)(p % w)] != 0.0f;
  };
  unsigned pr[U];
#pragma unroll
  for (int u = 0; u < U; u++) pr[u] = pre[u];
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nrun; r += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = r * kRun;
    const int64_t p = n <= 0xffffffffll ? (int64_t)((unsigned)e / d) : e / d;
    const unsigned k = (unsigned)(e - p * d);
    unsigned cur[U], cnt[U];
#pragma unroll
    for (int u = 0; u < U; u++) cur[u] = cnt[u] = 0u;
    auto count = [&](float x) {
      const unsigned key = order_key(x);
      const unsigned dig = (key >> sft) & msk;
#pragma unroll
      for (int u = 0; u < U; u++) {
        if (hs < 32 && (key >> hs) != pr[u]) continue;
        if (dig != cur[u]) {
          if (cnt[u]) atomicAdd(&sh[u][cur[u]], cnt[u]);
          cur[u] = dig;
          cnt[u] = 0u;
        }
        cnt[u]++;
      }
    };
    if (k + kRun <= d && ((reinterpret_cast<uintptr_t>(vol + e) & 15u) == 0)) {  // within one A-scan
      if (!selected(p)) continue;
      float4 f[kRun / 4];
#pragma unroll
      for (int q = 0; q < kRun / 4; q++) f[q] = __ldg(reinterpret_cast<const float4*>(vol + e) + q);
#pragma unroll
      for (int q = 0; q < kRun / 4; q++) {
        count(f[q].x);
        count(f[q].y);
        count(f[q].z);
        count(f[q].w);
      }
    } else {
      int64_t pp = p;
      unsigned kk = k;
      bool s = selected(pp);
      for (int q = 0; q < kRun && e + q < n; q++) {
        if (s) count(__ldg(vol + e + q));
        if (++kk == d) {
          kk = 0;
          pp++;
          if (e + q + 1 < n) s = selected(pp);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; u++)
      if (cnt[u]) atomicAdd(&sh[u][cur[u]], cnt[u]);
  }
}

__global__ void __launch_bounds__(kT) radix_hist_kernel(const float* __restrict__ vol, int w, int h, int d,
                                                        int fast_axis, const float* __restrict__ v,
                                                        const Select* __restrict__ sel, int pass,
                                                        unsigned* __restrict__ hist) {
  __shared__ unsigned sh[kTargets][kRadixBins];
  for (int t = threadIdx.x; t < kTargets * kRadixBins; t += kT) (&sh[0][0])[t] = 0u;
  __syncthreads();
  const int sft = digit_shift(pass);
  const unsigned msk = digit_mask(pass);
  // the distinct prefixes and each target's slot among them
  unsigned pre[kTargets];
  int slot[kTargets], nu = 0;
#pragma unroll
  for (int t = 0; t < kTargets; t++) {
    const unsigned q = sel->prefix[t];
    int s = -1;
#pragma unroll
    for (int u = 0; u < kTargets; u++)
      if (u < nu && pre[u] == q) s = u;
    if (s < 0) {
      s = nu++;
#pragma unroll
      for (int u = 0; u < kTargets; u++)
        if (u == s) pre[u] = q;
    }
    slot[t] = s;
  }
  const int hs = sft + (pass == 2 ? 10 : 11);  // the bits above the digit start at hs
  const int64_t n = (int64_t)w * h * d;
  const bool any = sel->any != 0;
  switch (nu) {
    case 1: hist_runs<1>(vol, w, d, n, fast_axis, v, any, hs, sft, msk, pre, sh); break;
    case 2: hist_runs<2>(vol, w, d, n, fast_axis, v, any, hs, sft, msk, pre, sh); break;
    default: {
      unsigned p4[kTargets];
#pragma unroll
      for (int t = 0; t < kTargets; t++) p4[t] = t < nu ? pre[t] : pre[0];
      // slots past nu repeat slot 0's prefix: counted, never read
      hist_runs<kTargets>(vol, w, d, n, fast_axis, v, any, hs, sft, msk, p4, sh);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kTargets * kRadixBins; i += kT) {
    const int t = i / kRadixBins, bin = i % kRadixBins;
    const int st = t == 0 ? slot[0] : (t == 1 ? slot[1] : (t == 2 ? slot[2] : slot[3]));
    const unsigned c = sh[st][bin];
    if (c) atomicAdd(hist + i, c);
  }
}

// One block: the number of valid B-scans and from it the ranks of the order
// statistics the percentiles interpolate between.
__global__ void __launch_bounds__(1024) select_init_kernel(Select* sel, const float* __restrict__ v, int nb,
                                                           double per_bscan, double q_lo, double q_hi) {
  __shared__ int cnt;
  if (threadIdx.x == 0) cnt = 0;
  __syncthreads();
  int c = 0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) c += v[b] != 0.0f;
  atomicAdd(&cnt, c);
  __syncthreads();
  if (threadIdx.x != 0) return;
  const int any = cnt > 0;
  const long long nsel = (long long)(any ? cnt : nb) * (long long)per_bscan;
  sel->any = any;
  sel->nvalid = cnt;
  sel->kept = 0ull;
  for (int q = 0; q < 2; q++) {
    const double pos = __dmul_rn(q == 0 ? q_lo : q_hi, (double)(nsel - 1));
    const long long lo = (long long)floor(pos);
    sel->pos[q] = pos;
    sel->rank[2 * q] = lo;
    sel->rank[2 * q + 1] = lo + 1 < nsel ? lo + 1 : lo;
    sel->prefix[2 * q] = sel->prefix[2 * q + 1] = 0u;
  }
}

// One block of kRadixBins / 2 threads: for each target, the bin holding its
// rank (block-wide exclusive scan of the histogram, each thread owning two
// consecutive bins); prefix and rank are narrowed to that bin.  After the
// last pass the key is complete.  Clears the histograms for the next pass.
constexpr int kPickThreads = kRadixBins / 2;
__global__ void __launch_bounds__(kPickThreads) radix_pick_kernel(Select* sel, unsigned* hist, int pass) {
  __shared__ unsigned long long warp_tot[kPickThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned nbins = digit_mask(pass) + 1u;
  const int width = pass == 2 ? 10 : 11;
  for (int t = 0; t < kTargets; t++) {
    unsigned* hb = hist + t * kRadixBins;
    const unsigned c0 = 2 * tid < (int)nbins ? hb[2 * tid] : 0u;
    const unsigned c1 = 2 * tid + 1 < (int)nbins ? hb[2 * tid + 1] : 0u;
    // inclusive scan of the pair sums within the warp, then across warps
    unsigned long long x = (unsigned long long)c0 + c1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[warp] = x;
    __syncthreads();
    unsigned long long before = 0;
    for (int i = 0; i < warp; i++) before += warp_tot[i];
    const unsigned long long incl = before + x;
    const unsigned long long excl = incl - c0 - c1;
    const long long r = sel->rank[t];
    __syncthreads();  // every thread has read rank[t] and warp_tot before they change
    if ((long long)excl <= r && r < (long long)incl) {
      const bool first = r < (long long)(excl + c0);
      const unsigned bin = 2 * tid + (first ? 0u : 1u);
      sel->prefix[t] = (sel->prefix[t] << width) | bin;
      sel->rank[t] = r - (long long)(first ? excl : excl + c0);
      if (pass == 2) sel->value[t] = key_value(sel->prefix[t]);
    }
    __syncthreads();
  }
  for (int i = tid; i < kTargets * kRadixBins; i += kPickThreads) hist[i] = 0u;
}

// One warp.
__global__ void finish_kernel(Select* sel, const double* __restrict__ oct_sums, const float* __restrict__ v,
                              int nb, double per_bscan, double thresh, double t_oct_in) {
  double t = t_oct_in;
  if (isnan(t)) {
    const bool any = sel->any != 0;
    double s = 0.0;
    for (int b = threadIdx.x; b < nb; b += 32)
      if (!any || v[b] != 0.0f) s += oct_sums[b];
    s = warp_sum(s);
    t = s / ((double)(any ? sel->nvalid : nb) * per_bscan);
  }
  if (threadIdx.x != 0) return;
  for (int q = 0; q < 2; q++) {
    const double pos = sel->pos[q];
    const double lo = floor(pos);
    const double a = sel->value[2 * q], b = sel->value[2 * q + 1];
    sel->p[q] = a + (pos - lo) * (b - a);
  }
  sel->cut = sel->p[0] + thresh * (sel->p[1] - sel->p[0]);
  sel->t_oct = t;
  // float bounds that reproduce the double comparisons exactly
  float c = (float)sel->cut;  // round to nearest
  if ((double)c < sel->cut) c = nextafterf(c, INFINITY);
  else if ((double)nextafterf(c, -INFINITY) >= sel->cut) c = nextafterf(c, -INFINITY);
  sel->cut_f = c;
  float o = (float)t;
  if ((double)o > t) o = nextafterf(o, -INFINITY);
  sel->toct_f = o;
}

// ---------------------------------------------------------------- projection
// One warp per A-scan.  vec: d is a multiple of 4 and the volumes are 16-byte
// aligned.  Bound by HBM (three volumes read): 300 x 300 x 512 196 -> 80 us.
__global__ void __launch_bounds__(kT) project_kernel(const float* __restrict__ A, const float* __restrict__ S,
                                                     const float* __restrict__ F, int64_t nasc, int d, bool vec,
                                                     Select* __restrict__ sel, float* __restrict__ E) {
  const int lane = threadIdx.x & 31;
  const float cut = sel->cut_f, to = sel->toct_f;
  __shared__ unsigned block_kept;  // one global atomic per block
  if (threadIdx.x == 0) block_kept = 0u;
  __syncthreads();
  unsigned mine = 0u;
  for (int64_t p = (int64_t)blockIdx.x * (kT / 32) + (threadIdx.x >> 5); p < nasc;
       p += (int64_t)gridDim.x * (kT / 32)) {  // warp-uniform
    float s = 0.f;
    int c = 0;
    auto take = [&](float f, float o, float a) {
      if (f < cut && o > to) {
        s += a;
        c++;
      }
    };
    if (vec) {
      const float4 *f4 = reinterpret_cast<const float4*>(F + p * d), *s4 = reinterpret_cast<const float4*>(S + p * d),
                   *a4 = reinterpret_cast<const float4*>(A + p * d);
#pragma unroll 4
      for (int g = lane; g < d / 4; g += 32) {
        const float4 f = __ldg(f4 + g), o = __ldg(s4 + g), a = __ldg(a4 + g);
        take(f.x, o.x, a.x);
        take(f.y, o.y, a.y);
        take(f.z, o.z, a.z);
        take(f.w, o.w, a.w);
      }
    } else {
      for (int k = lane; k < d; k += 32) take(F[p * d + k], S[p * d + k], A[p * d + k]);
    }
    s = warp_sum(s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (lane == 0) {
      E[p] = c ? s / (float)c : 0.0f;
      mine += (unsigned)c;
    }
  }
  if (lane == 0 && mine) atomicAdd(&block_kept, mine);
  __syncthreads();
  if (threadIdx.x == 0 && block_kept) atomicAdd(&sel->kept, (unsigned long long)block_kept);
}

// One block per B-scan: bitonic sort of its en-face values in shared memory,
// median, subtraction.  nf <= kMaxFast.
constexpr int kMaxFast = 4096;
__global__ void __launch_bounds__(1024) bscan_median_kernel(float* __restrict__ E, int w, int h, int fast_axis) {
  __shared__ float s[kMaxFast];
  const int b = blockIdx.x;
  const int nf = fast_axis == 0 ? w : h;
  int np = 1;
  while (np < nf) np <<= 1;
  for (int f = threadIdx.x; f < np; f += blockDim.x) s[f] = f < nf ? E[ascan_of(w, fast_axis, b, f)] : INFINITY;
  __syncthreads();
  for (int size = 2; size <= np; size <<= 1)
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = threadIdx.x; i < np; i += blockDim.x) {
        const int jx = i ^ stride;
        if (jx > i) {
          const bool up = (i & size) == 0;
          const float x = s[i], y = s[jx];
          if ((x > y) == up) {
            s[i] = y;
            s[jx] = x;
          }
        }
      }
      __syncthreads();
    }
  const double med = (nf & 1) ? (double)s[nf / 2] : 0.5 * ((double)s[nf / 2 - 1] + (double)s[nf / 2]);
  __syncthreads();
  for (int f = threadIdx.x; f < nf; f += blockDim.x) {
    float* e = E + ascan_of(w, fast_axis, b, f);
    *e = (float)((double)*e - med);
  }
}

// Block per B-scan: an invalid B-scan takes the nearest valid one (lower index
// on a tie), if there is one; valid B-scans are only read.
__global__ void replace_kernel(float* E, int w, int h, int fast_axis, const float* __restrict__ v) {
  const int b = blockIdx.x;
  const int nb = fast_axis == 0 ? h : w, nf = fast_axis == 0 ? w : h;
  if (v[b] != 0.0f) return;
  int best = -1;
  for (int dist = 1; dist < nb && best < 0; dist++) {
    if (b - dist >= 0 && v[b - dist] != 0.0f) best = b - dist;
    else if (b + dist < nb && v[b + dist] != 0.0f) best = b + dist;
  }
  if (best < 0) return;
  for (int f = threadIdx.x; f < nf; f += blockDim.x) E[ascan_of(w, fast_axis, b, f)] = E[ascan_of(w, fast_axis, best, f)];
}

// One element (or A-scan) per thread (warp) up to the grid limit.
inline unsigned grid_for(int64_t n, int per = kT) {
  int64_t b = (n + per - 1) / per;
  if (b < 1) b = 1;
  if (b > 0x7fffffff) b = 0x7fffffff;
  return (unsigned)b;
}

struct CudaErr {
  cudaError_t e;
};
inline void ck(cudaError_t e) {
  if (e != cudaSuccess) throw CudaErr{e};
}

inline bool aligned16(const void* q) { return ((uintptr_t)q & 15u) == 0; }
inline size_t round256(size_t n) { return (n + 255) & ~size_t(255); }

// Scratch of one projection: two volumes (the median and the rank-filtered
// volume share one), the OCT sums, the selection state and its histograms.
struct EnfaceScratch {
  float *v0, *v1;
  double* osum;
  Select* sel;
  unsigned* hist;
  size_t bytes;
  EnfaceScratch(char* base, int64_t nvox, int nb) {
    size_t o = 0;
    auto take = [&](size_t n) {
      char* p = base + o;
      o += round256(n);
      return p;
    };
    v0 = reinterpret_cast<float*>(take(sizeof(float) * (size_t)nvox));
    v1 = reinterpret_cast<float*>(take(sizeof(float) * (size_t)nvox));
    osum = reinterpret_cast<double*>(take(sizeof(double) * nb));
    sel = reinterpret_cast<Select*>(take(sizeof(Select)));
    hist = reinterpret_cast<unsigned*>(take(sizeof(unsigned) * kTargets * kRadixBins));
    bytes = o;
  }
};

// Whether a projection takes scans of this size.
int enface_size(int w, int h, int d, int fast_axis) {
  if (w < 1 || h < 1 || d < 1 || (fast_axis != 0 && fast_axis != 1)) return OCTMC_ERR_INVALID_ARG;
  const int nf = fast_axis == 0 ? w : h;
  return nf > kMaxFast || h > 65535 || (w + 7) / 8 > 65535 ? OCTMC_ERR_UNSUPPORTED : OCTMC_OK;
}

int enface_check(const float* octa, const float* oct, int w, int h, int d, int fast_axis, const float* v, double q_lo,
                 double q_hi, double thresh, const float* enface) {
  const int size = enface_size(w, h, d, fast_axis);
  if (!octa || !oct || !v || !enface || size == OCTMC_ERR_INVALID_ARG) return OCTMC_ERR_INVALID_ARG;
  if (!(q_lo >= 0.0 && q_lo <= 1.0 && q_hi >= 0.0 && q_hi <= 1.0) || !std::isfinite(thresh))
    return OCTMC_ERR_INVALID_ARG;
  return size;
}

void rank15(const float* in, int w, int h, int d, int axis, float* out, cudaStream_t st) {
  const int n = axis == 0 ? w : h, m = axis == 0 ? h : w;
  const int64_t sx = d, sy = (int64_t)w * d;
  const dim3 g((unsigned)((d + kSx - 1) / kSx), (unsigned)std::min((n + kSeg - 1) / kSeg, 65535),
               (unsigned)std::min((m + kSy - 1) / kSy, 65535));
  rank15_kernel<<<g, dim3(kSx, kSy), 0, st>>>(in, n, axis == 0 ? sx : sy, m, axis == 0 ? sy : sx, d, out);
  ck(cudaGetLastError());
}

// The whole projection on `st`, without a host wait.
void enface_run(const float* octa, const float* oct, int w, int h, int d, int fast_axis, const float* v, double q_lo,
                double q_hi, double thresh, double t_oct, float* enface, float* filtered, const EnfaceScratch& X,
                cudaStream_t st) {
  const int nb = fast_axis == 0 ? h : w, nf = fast_axis == 0 ? w : h;
  const int64_t nvox = (int64_t)w * h * d, nasc = (int64_t)w * h;
  const double per = (double)nf * d;
  float* m3 = X.v0;
  float* r1 = X.v1;
  float* r2 = filtered ? filtered : X.v0;  // the median is read before it is written
  ck(cudaMemsetAsync(X.hist, 0, sizeof(unsigned) * kTargets * kRadixBins, st));
  select_init_kernel<<<1, 1024, 0, st>>>(X.sel, v, nb, per, q_lo, q_hi);
  ck(cudaGetLastError());
  const dim3 mg((unsigned)((d + kSx - 1) / kSx), (unsigned)((w + kSy * kMedI - 1) / (kSy * kMedI)), (unsigned)h);
  median3_kernel<<<mg, dim3(kSx, kSy), 0, st>>>(octa, w, h, d, m3);
  ck(cudaGetLastError());
  // fast axis first, then the slow axis
  rank15(m3, w, h, d, fast_axis, r1, st);
  rank15(r1, w, h, d, 1 - fast_axis, r2, st);
  // percentiles of the filtered voxels of the valid B-scans
  for (int pass = 0; pass < 3; pass++) {
    // streaming, no reuse: a resident-size grid, each block one shared histogram
    const unsigned hb = (unsigned)std::min<int64_t>((nvox / kRun + kT) / kT, 152 * 6);
    radix_hist_kernel<<<hb, kT, 0, st>>>(r2, w, h, d, fast_axis, v, X.sel, pass, X.hist);
    ck(cudaGetLastError());
    radix_pick_kernel<<<1, kPickThreads, 0, st>>>(X.sel, X.hist, pass);
    ck(cudaGetLastError());
  }
  // OCT threshold from the per-B-scan OCT sums, cut, projection
  if (std::isnan(t_oct)) {
    bscan_sum_kernel<<<nb, kSumThreads, 0, st>>>(oct, w, h, d, fast_axis, d % 4 == 0 && aligned16(oct), X.osum);
    ck(cudaGetLastError());
  }
  finish_kernel<<<1, 32, 0, st>>>(X.sel, X.osum, v, nb, per, thresh, t_oct);
  ck(cudaGetLastError());
  const bool vec = d % 4 == 0 && aligned16(octa) && aligned16(oct) && aligned16(r2);
  project_kernel<<<grid_for(nasc, kT / 32), kT, 0, st>>>(octa, oct, r2, nasc, d, vec, X.sel, enface);
  ck(cudaGetLastError());
  bscan_median_kernel<<<nb, 1024, 0, st>>>(enface, w, h, fast_axis);
  ck(cudaGetLastError());
  replace_kernel<<<nb, 256, 0, st>>>(enface, w, h, fast_axis, v);
  ck(cudaGetLastError());
}

int enface_with(char* ws, const float* octa, const float* oct, int w, int h, int d, int fast_axis, const float* v,
                double q_lo, double q_hi, double thresh, double t_oct, float* enface, float* filtered, double* info,
                cudaStream_t st) {
  try {
    const EnfaceScratch X(ws, (int64_t)w * h * d, fast_axis == 0 ? h : w);
    enface_run(octa, oct, w, h, d, fast_axis, v, q_lo, q_hi, thresh, t_oct, enface, filtered, X, st);
    if (info) {
      Select s1;
      ck(cudaMemcpyAsync(&s1, X.sel, sizeof(Select), cudaMemcpyDeviceToHost, st));
      ck(cudaStreamSynchronize(st));
      info[0] = s1.p[0];
      info[1] = s1.p[1];
      info[2] = s1.t_oct;
      info[3] = (double)s1.kept;
    }
  } catch (const CudaErr&) {
    cudaGetLastError();
    return OCTMC_ERR_CUDA;
  }
  return OCTMC_OK;
}

}  // namespace
}  // namespace octmc

using namespace octmc;

extern "C" int octmc_saccade_validity(const float* octa, int w, int h, int d, int fast_axis, float* v,
                                      double* means, void* stream) {
  if (!octa || !v || w < 1 || h < 1 || d < 1 || (fast_axis != 0 && fast_axis != 1)) return OCTMC_ERR_INVALID_ARG;
  const cudaStream_t st = (cudaStream_t)stream;
  const int nb = fast_axis == 0 ? h : w, nf = fast_axis == 0 ? w : h;
  double* sums = means;  // the means' buffer holds the sums first
  try {
    if (!means) ck(cudaMallocAsync(&sums, sizeof(double) * nb, st));
    bscan_sum_kernel<<<nb, kSumThreads, 0, st>>>(octa, w, h, d, fast_axis, d % 4 == 0 && aligned16(octa), sums);
    ck(cudaGetLastError());
    validity_kernel<<<1, 1024, 0, st>>>(sums, nb, (double)nf * d, v, means);
    ck(cudaGetLastError());
    if (!means) ck(cudaFreeAsync(sums, st));
    ck(cudaStreamSynchronize(st));
  } catch (const CudaErr&) {
    cudaGetLastError();
    return OCTMC_ERR_CUDA;
  }
  return OCTMC_OK;
}

extern "C" int64_t octmc_enface_workspace(int w, int h, int d, int fast_axis) {
  if (enface_size(w, h, d, fast_axis) != OCTMC_OK) return -1;
  return (int64_t)EnfaceScratch(nullptr, (int64_t)w * h * d, fast_axis == 0 ? h : w).bytes;
}

extern "C" int octmc_enface_ws(const float* octa, const float* oct, int w, int h, int d, int fast_axis, const float* v,
                               double q_lo, double q_hi, double thresh, double t_oct, float* enface, float* filtered,
                               double* info, void* workspace, int64_t workspace_bytes, void* stream) {
  const int rc = enface_check(octa, oct, w, h, d, fast_axis, v, q_lo, q_hi, thresh, enface);
  if (rc != OCTMC_OK) return rc;
  if (!workspace || ((uintptr_t)workspace & 255u) || workspace_bytes < octmc_enface_workspace(w, h, d, fast_axis))
    return OCTMC_ERR_INVALID_ARG;
  const cudaStream_t st = (cudaStream_t)stream;
  const int r = enface_with(static_cast<char*>(workspace), octa, oct, w, h, d, fast_axis, v, q_lo, q_hi, thresh, t_oct,
                            enface, filtered, info, st);
  if (cudaStreamSynchronize(st) != cudaSuccess && r == OCTMC_OK) return OCTMC_ERR_CUDA;
  return r;
}

extern "C" int octmc_enface(const float* octa, const float* oct, int w, int h, int d, int fast_axis, const float* v,
                            double q_lo, double q_hi, double thresh, double t_oct, float* enface, float* filtered,
                            double* info, void* stream) {
  const int rc = enface_check(octa, oct, w, h, d, fast_axis, v, q_lo, q_hi, thresh, enface);
  if (rc != OCTMC_OK) return rc;
  const cudaStream_t st = (cudaStream_t)stream;
  char* ws = nullptr;
  if (cudaMallocAsync(&ws, (size_t)octmc_enface_workspace(w, h, d, fast_axis), st) != cudaSuccess) {
    cudaGetLastError();
    return OCTMC_ERR_CUDA;
  }
  int r = enface_with(ws, octa, oct, w, h, d, fast_axis, v, q_lo, q_hi, thresh, t_oct, enface, filtered, info, st);
  cudaFreeAsync(ws, st);
  if (cudaStreamSynchronize(st) != cudaSuccess && r == OCTMC_OK) r = OCTMC_ERR_CUDA;
  return r;
}
