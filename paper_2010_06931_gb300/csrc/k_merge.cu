// Merging weights of the final resampling (Ploner et al., Sec. 2.1 last
// paragraphs, Sec. 2.5): per motion-corrected A-scan and scan, the sampling
// density (how many corrected A-scans sample the same input location), an
// exponentially decaying weight above the normal density, clipping and
// normalisation, and the validity-weighted en-face angiography merge.
//
// The density map is accumulated with 64-bit fixed-point integer atomics
// (weights in units of 2^-32), so its value does not depend on the order of
// the additions.
#include "common.cuh"
#include "sample.cuh"

namespace octmc {
namespace {

constexpr int kThreads = 256;
constexpr double kFix = 4294967296.0;  // 2^32

// Bilinear footprint of (u, v) = (i + dx, j + dy) clamped into the grid.
struct Foot {
  int x0, x1, y0, y1;
  float fx, fy;
};

__device__ __forceinline__ Foot footprint(const double* disp, int64_t n, int64_t p, int V, int i, int j, int w,
                                          int h) {
  Foot F;
  split_exact((unsigned long long)__double_as_longlong(disp[(int64_t)(3 * V + 0) * n + p]), i, 0, w - 1, &F.x0, &F.fx);
  split_exact((unsigned long long)__double_as_longlong(disp[(int64_t)(3 * V + 1) * n + p]), j, 0, h - 1, &F.y0, &F.fy);
  F.x1 = min(F.x0 + 1, w - 1);
  F.y1 = min(F.y0 + 1, h - 1);
  return F;
}

__global__ void splat_kernel(const double* __restrict__ disp, int w, int h, unsigned long long* counts) {
  const int64_t n = (int64_t)w * h;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < 2 * n; e += (int64_t)gridDim.x * blockDim.x) {
    const int V = (int)(e / n);
    const int64_t p = e % n;
    const Foot F = footprint(disp, n, p, V, (int)(p % w), (int)(p / w), w, h);
    unsigned long long* c = counts + V * n;
    atomicAdd(c + (int64_t)F.y0 * w + F.x0, (unsigned long long)((1.0f - F.fx) * (1.0f - F.fy) * (float)kFix));
    atomicAdd(c + (int64_t)F.y0 * w + F.x1, (unsigned long long)(F.fx * (1.0f - F.fy) * (float)kFix));
    atomicAdd(c + (int64_t)F.y1 * w + F.x0, (unsigned long long)((1.0f - F.fx) * F.fy * (float)kFix));
    atomicAdd(c + (int64_t)F.y1 * w + F.x1, (unsigned long long)(F.fx * F.fy * (float)kFix));
  }
}

__device__ __forceinline__ float count_value(unsigned long long c) {
  // integer part + fraction (2^-32 units), without float64 arithmetic
  return (float)(unsigned)(c >> 32) + (float)(unsigned)(c & 0xffffffffull) * 2.3283064365386963e-10f;
}

__global__ void weights_kernel(LevelDev L, const double* __restrict__ disp, float beta, float tau,
                               const unsigned long long* __restrict__ counts, float* weights, float* angio) {
  const int w = L.w, h = L.h;
  const int64_t n = (int64_t)w * h;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(p % w), j = (int)(p / w);
    float wt[2];
    for (int V = 0; V < 2; V++) {
      const Foot F = footprint(disp, n, p, V, i, j, w, h);
      const unsigned long long* c = counts + V * n;
      const float rho = (1.0f - F.fx) * (1.0f - F.fy) * count_value(c[(int64_t)F.y0 * w + F.x0]) +
                        F.fx * (1.0f - F.fy) * count_value(c[(int64_t)F.y0 * w + F.x1]) +
                        (1.0f - F.fx) * F.fy * count_value(c[(int64_t)F.y1 * w + F.x0]) +
                        F.fx * F.fy * count_value(c[(int64_t)F.y1 * w + F.x1]);
      wt[V] = expf(-beta * fmaxf(0.0f, rho - 1.0f));
    }
    float c0 = wt[0] >= tau ? wt[0] : 0.0f, c1 = wt[1] >= tau ? wt[1] : 0.0f;
    if (c0 == 0.0f && c1 == 0.0f) {
      if (wt[0] >= wt[1]) c0 = 1.0f;
      else c1 = 1.0f;
    }
    const float wx = c0 / (c0 + c1), wy = c1 / (c0 + c1);
    if (weights) {
      weights[p] = wx;
      weights[n + p] = wy;
    }
    if (angio && L.ax) {
      // resampled en-face images (Eq. 6 positions) and validity (Eq. 7)
      float a[2], va[2] = {1.0f, 1.0f};
      for (int V = 0; V < 2; V++) {
        int bx, by;
        float tx, ty, wxv[4], dwx[4], wyv[4], dwy[4];
        split_exact((unsigned long long)__double_as_longlong(disp[(int64_t)(3 * V + 0) * n + p]), i, -4, w + 3, &bx, &tx);
        split_exact((unsigned long long)__double_as_longlong(disp[(int64_t)(3 * V + 1) * n + p]), j, -4, h + 3, &by, &ty);
        keys_weights(tx, wxv, dwx);
        keys_weights(ty, wyv, dwy);
        const float* img = V == 0 ? L.ax : L.ay;
        float s = 0.0f;
        for (int b = 0; b < 4; b++)
          for (int q = 0; q < 4; q++)
            s = fmaf(wxv[q] * wyv[b], img[(int64_t)clampi(by - 1 + b, h) * w + clampi(bx - 1 + q, w)], s);
        a[V] = s;
        const float* vv = V == 0 ? L.vx : L.vy;
        if (vv) {
          float dv;
          if (V == 0) validity_hermite(vv, h, by, ty, &va[V], &dv);
          else validity_hermite(vv, w, bx, tx, &va[V], &dv);
        }
      }
      const float a0 = fmaxf(0.0f, c0 * va[0]), a1 = fmaxf(0.0f, c1 * va[1]);
      angio[p] = (a0 + a1 > 0.0f) ? (a0 * a[0] + a1 * a[1]) / (a0 + a1) : 0.0f;
    }
  }
}

constexpr int kWarpsPerBlock = 8;

struct ColVol {
  const void* base;    // the volume; addressed in groups of 4 samples
  unsigned roff[4];    // row offsets (in groups) of the 4 neighbour rows
  unsigned coff[4];    // column offsets (in groups) of the 4 neighbour columns
  float wx[4], wy[4], wz[4];
  int q, r;            // floor(dz) = 4 q + r, 0 <= r < 4
  int bx, by;          // floor of the transverse coordinates
};

// Coordinate split of the 6 displacement values of A-scan (i, j) by lanes
// 0..5 (lane = 3 V + c), broadcast to the warp: floor(u) and the float
// fraction for u = i + dx and u = j + dy clamped to [-4, n + 3] (beyond that
// every tap is an edge sample) and u = dz clamped to +-(d + 8) (all depth
// taps are then edge samples).  Integer arithmetic only (split_exact).
__device__ __forceinline__ void split_displacement(const double* disp, int64_t nasc, int64_t p, int i,
                                                   int j, const LevelDev& L, int lane, int base[6],
                                                   float frac[6]) {
  int b = 0;
  float t = 0.f;
  if (lane < 6) {
    const int c = lane % 3;
    const unsigned long long bits =
        (unsigned long long)__double_as_longlong(disp[(int64_t)lane * nasc + p]);
    if (c == 0) split_exact(bits, i, -4, L.w + 3, &b, &t);
    else if (c == 1) split_exact(bits, j, -4, L.h + 3, &b, &t);
    else split_exact(bits, 0, -L.d - 8, L.d + 8, &b, &t);
  }
#pragma unroll
  for (int c = 0; c < 6; c++) {
    base[c] = __shfl_sync(0xffffffffu, b, c);
    frac[c] = __shfl_sync(0xffffffffu, t, c);
  }
}

__device__ __forceinline__ void setup_col(ColVol& V, const void* vol, const LevelDev& L, const int base[3],
                                          const float frac[3]) {
  V.bx = base[0];
  V.by = base[1];
  const int kz0 = base[2];
  V.q = kz0 >> 2;  // arithmetic shift: floor division by 4
  V.r = kz0 & 3;
  float dw[4];  // the derivative weights are not used here
  keys_weights(frac[0], V.wx, dw);
  keys_weights(frac[1], V.wy, dw);
  keys_weights(frac[2], V.wz, dw);
  const unsigned nq = (unsigned)(L.dp >> 2);
#pragma unroll
  for (int a = 0; a < 4; a++) {
    V.roff[a] = (unsigned)clampi(V.by - 1 + a, L.h) * (unsigned)L.w * nq;
    V.coff[a] = (unsigned)clampi(V.bx - 1 + a, L.w) * nq;
  }
  V.base = vol;
}

// Four consecutive depth samples as two packed pairs (k, k+1), (k+2, k+3).
struct Q4 {
  float2 lo, hi;
};

__device__ __forceinline__ Q4 q4(const float4& v) { return {make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
__device__ __forceinline__ Q4 q4zero() { return {make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }

// acc += w * s on all four samples (w broadcast to both halves)
__device__ __forceinline__ void qfma(Q4& acc, float2 w, const Q4& s) {
  acc.lo = ffma2(w, s.lo, acc.lo);
  acc.hi = ffma2(w, s.hi, acc.hi);
}

__device__ __forceinline__ float4 f4(const Q4& q) { return make_float4(q.lo.x, q.lo.y, q.hi.x, q.hi.y); }

__device__ __forceinline__ float4 bcast(float v) { return make_float4(v, v, v, v); }

// Axial 4-tap filter for the lane's 4 outputs.  e[1..4] hold the lane's
// own input group, e[0] the last sample of lane-1's group, e[5..8] lane+1's
// group and e[9] the first sample of lane+2's.  Output o, tap c reads
// e[R + o + c], where R = floor(dz) mod 4.
template <int R>
__device__ __forceinline__ void axial_col(const float4& T, const float wz[4], float I[4]) {
  float e[10];
  e[1] = T.x; e[2] = T.y; e[3] = T.z; e[4] = T.w;
  if (R == 0) e[0] = __shfl_up_sync(kFull, T.w, 1);
  e[5] = __shfl_down_sync(kFull, T.x, 1);
  e[6] = __shfl_down_sync(kFull, T.y, 1);
  if (R >= 1) e[7] = __shfl_down_sync(kFull, T.z, 1);
  if (R >= 2) e[8] = __shfl_down_sync(kFull, T.w, 1);
  if (R == 3) e[9] = __shfl_down_sync(kFull, T.x, 2);
  // outputs in packed pairs (o, o + 1); each half adds its 4 taps in the
  // scalar order
#pragma unroll
  for (int o = 0; o < 4; o += 2) {
    float2 a = make_float2(0.f, 0.f);
#pragma unroll
    for (int c = 0; c < 4; c++)
      a = ffma2(make_float2(wz[c], wz[c]), make_float2(e[R + o + c], e[R + o + 1 + c]), a);
    I[o] = a.x; I[o + 1] = a.y;
  }
}

// Interpolated values of one volume at the lane's 4 outputs.  qk: first input
// depth of the lane's group (samples, may lie outside the volume); qc: index
// of that group's (clamped) samples in the volume.
template <typename S>
__device__ __forceinline__ void sample_col_group(const ColVol& V, int qk, unsigned qc, int dp, float I[4]) {
  // transverse 4 x 4 interpolation of the group, in packed pairs along depth
  // (same operations and order as scalar FMAs)
  Q4 Tq = q4zero();
#pragma unroll
  for (int b = 0; b < 4; b++) {
    Q4 U = q4zero();
#pragma unroll
    for (int a = 0; a < 4; a++) {
      const unsigned idx = V.roff[b] + V.coff[a] + qc;
      qfma(U, make_float2(V.wx[a], V.wx[a]), q4(load4<S>(V.base, idx)));
    }
    qfma(Tq, make_float2(V.wy[b], V.wy[b]), U);
  }
  float4 T = f4(Tq);
  // groups entirely before sample 0 / after the last sample hold the edge value
  if (qk < 0) T = bcast(T.x);
  else if (qk >= dp) T = bcast(T.w);
  switch (V.r) {
    case 0: axial_col<0>(T, V.wz, I); break;
    case 1: axial_col<1>(T, V.wz, I); break;
    case 2: axial_col<2>(T, V.wz, I); break;
    default: axial_col<3>(T, V.wz, I); break;
  }
}

// Interpolated values of one volume at the lane's 4 outputs of the depth
// block starting at kb.
template <typename S>
__device__ __forceinline__ void sample_col_block(const ColVol& V, int kb, int lane, int dp, float I[4]) {
  const int qk = kb + 4 * V.q + 4 * (lane - 1);  // first input depth of the lane's group
  const unsigned qc = (unsigned)(min(max(qk, 0), dp - 4) >> 2);
  sample_col_group<S>(V, qk, qc, dp, I);
}

// Motion-corrected resampling and merging of one A-scan (warp): both scans
// resampled along depth at the displaced positions, merged with the per-A-scan weights.
// Forward only, so it fits in 40 registers: 6 blocks (48 warps) per SM keep
// more loads in flight than the data kernel's 32 warps.  Bound by the L1 data
// pipe (87 % of its wavefronts: 160 column loads per A-scan at depth 512).  vec4: d % 4 == 0 and every
// output 16-byte aligned, so a lane's 4 outputs go out as one 128-bit store.
template <typename T>
__global__ void __launch_bounds__(kWarpsPerBlock * kWarp, 6)
resample_merge_kernel(const LevelDev L, const double* __restrict__ disp, const float* __restrict__ weights,
                      float* merged, float* cx, float* cy, bool vec4) {
  const int64_t nasc = (int64_t)L.w * L.h;
  const int64_t p = (int64_t)blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
  if (p >= nasc) return;
  const int lane = threadIdx.x & 31;
  const int i = (int)(p % L.w), j = (int)(p / L.w);
  int base[6];
  float frac[6];
  split_displacement(disp, nasc, p, i, j, L, lane, base, frac);
  ColVol VX, VY;
  setup_col(VX, L.sx, L, base, frac);
  setup_col(VY, L.sy, L, base + 3, frac + 3);
  const float wx = weights ? weights[p] : 0.5f, wy = weights ? weights[nasc + p] : 0.5f;
  for (int kb = 0; kb < L.d; kb += kOutPerIter) {
    float IX[4], IY[4];
    sample_col_block<T>(VX, kb, lane, L.dp, IX);
    sample_col_block<T>(VY, kb, lane, L.dp, IY);
    const int k0 = kb + 4 * (lane - 1);
    if (lane >= 1 && lane <= kOutLanes && k0 < L.d) {
      const int64_t e0 = p * L.d + k0;
      if (vec4) {  // k0 + 3 < d as d % 4 == 0
        if (merged)
          *reinterpret_cast<float4*>(merged + e0) =
              make_float4(fmaf(wx, IX[0], wy * IY[0]), fmaf(wx, IX[1], wy * IY[1]), fmaf(wx, IX[2], wy * IY[2]),
                          fmaf(wx, IX[3], wy * IY[3]));
        if (cx) *reinterpret_cast<float4*>(cx + e0) = make_float4(IX[0], IX[1], IX[2], IX[3]);
        if (cy) *reinterpret_cast<float4*>(cy + e0) = make_float4(IY[0], IY[1], IY[2], IY[3]);
      } else {
#pragma unroll
        for (int o = 0; o < 4; o++) {
          if (k0 + o < L.d) {
            if (merged) merged[e0 + o] = fmaf(wx, IX[o], wy * IY[o]);
            if (cx) cx[e0 + o] = IX[o];
            if (cy) cy[e0 + o] = IY[o];
          }
        }
      }
    }
  }
}

inline unsigned grid_for(int64_t n) {
  int64_t b = (n + kThreads - 1) / kThreads;
  if (b < 1) b = 1;
  if (b > 65535) b = 65535;
  return (unsigned)b;
}

}  // namespace

cudaError_t launch_resample_merge(const LevelDev& L, const double* disp, const float* weights, float* merged,
                                  float* cx, float* cy, cudaStream_t s) {
  const int64_t nasc = (int64_t)L.w * L.h;
  const int64_t blocks = (nasc + kWarpsPerBlock - 1) / kWarpsPerBlock;
  if (blocks <= 0) return cudaSuccess;
  auto a16 = [](const float* q) { return ((uintptr_t)q & 15u) == 0; };
  const bool vec4 = (L.d % 4 == 0) && a16(merged) && a16(cx) && a16(cy);
  const unsigned threads = kWarpsPerBlock * kWarp;
  if (L.dtype == OCTMC_BF16)
    resample_merge_kernel<__nv_bfloat16><<<(unsigned)blocks, threads, 0, s>>>(L, disp, weights, merged, cx, cy, vec4);
  else if (L.dtype == OCTMC_F16)
    resample_merge_kernel<__half><<<(unsigned)blocks, threads, 0, s>>>(L, disp, weights, merged, cx, cy, vec4);
  else
    resample_merge_kernel<float><<<(unsigned)blocks, threads, 0, s>>>(L, disp, weights, merged, cx, cy, vec4);
  return cudaGetLastError();
}

cudaError_t launch_merge_weights(const LevelDev& L, const double* disp, double beta, double tau,
                                 unsigned long long* counts, float* weights, float* angio, cudaStream_t s) {
  const int64_t n = (int64_t)L.w * L.h;
  cudaError_t e = cudaMemsetAsync(counts, 0, sizeof(unsigned long long) * 2 * n, s);
  if (e != cudaSuccess) return e;
  splat_kernel<<<grid_for(2 * n), kThreads, 0, s>>>(disp, L.w, L.h, counts);
  weights_kernel<<<grid_for(n), kThreads, 0, s>>>(L, disp, (float)beta, (float)tau, counts, weights, angio);
  return cudaGetLastError();
}

}  // namespace octmc
