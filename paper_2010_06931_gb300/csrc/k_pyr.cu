// Multi-resolution pyramid (factor 2, Ploner et al. Sec. 2.1; the validity
// is downsampled "in the same way", Sec. 2.2), displacement prolongation
// between levels, and depth padding of the device volumes.
//
// Box mean over 2 samples per axis; an odd size rounds up and the missing
// sample repeats the edge sample.  The 8 (4, 2) float samples are added in
// double (or with the same result, mean8), which is exact for float inputs of
// similar magnitude, and the mean is rounded once to float.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <string.h>

#include <algorithm>

#include "common.cuh"

namespace octmc {
namespace {

constexpr int kThreads = 256;

__global__ void pad_depth_kernel(float* vol, int64_t columns, int d, int dp) {
  const int padn = dp - d;
  const int64_t n = columns * padn;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t col = e / padn;
    const int k = d + (int)(e % padn);
    vol[col * dp + k] = vol[col * dp + d - 1];
  }
}

__device__ __forceinline__ float to_float(float v) { return v; }
__device__ __forceinline__ float to_float(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float to_float(__half v) { return __half2float(v); }

template <typename T>
__global__ void unpad_depth_kernel(const T* vol, int64_t columns, int d, int dp, float* out) {
  const int64_t n = columns * d;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t col = e / d;
    out[e] = to_float(vol[col * dp + (e % d)]);
  }
}

// float32 -> 16-bit storage type, round to nearest even.
__device__ __forceinline__ void store_as(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
__device__ __forceinline__ void store_as(__half* p, float v) { *p = __float2half_rn(v); }

// Four samples per thread (n4 groups: the padded depth is a multiple of 4): one
// 16-byte load, one 8-byte store.  237 x 301 x 468: 82 -> 36 us a volume.
template <typename T>
__global__ void __launch_bounds__(kThreads) convert_kernel(const float4* __restrict__ in, uint2* __restrict__ out,
                                                           int64_t n4) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n4;
       e += (int64_t)gridDim.x * blockDim.x) {
    const float4 f = in[e];
    T v[4];
    store_as(v, f.x);
    store_as(v + 1, f.y);
    store_as(v + 2, f.z);
    store_as(v + 3, f.w);
    uint2 u;
    memcpy(&u, v, 8);
    out[e] = u;
  }
}

// Mean of 8 samples: the sum added in double (in the order of x) or, with the
// same result, exactly in float (exact_sum8: the double sum needs 43 of 53
// bits there), rounded once to float.
__device__ __forceinline__ float mean8(const float x[8]) {
  float s, e;
  if (exact_sum8(x, &s, &e)) return __fmul_rn(__fadd_rn(s, e), 0.125f);
  double q = 0.0;
#pragma unroll
  for (int k = 0; k < 8; k += 2) q += (double)x[k] + (double)x[k + 1];
  return (float)(q * 0.125);
}

// Block (32, 8): 32 groups of 4 output depths along x, 8 columns i2 along y;
// blockIdx.y: strips of columns, blockIdx.z: j2 (both volumes: z >= h2 is the
// second).  A thread makes 4 consecutive outputs from two 16-byte loads of
// each of 4 columns; the input's depth pad repeats its last sample, so only
// the output's pad needs a clamp.  Bound by HBM; 300 x 300 x 512 to 150 x 150 x
// 256: 2 x 194 -> 70 us for both volumes (one output and 8 scalar loads per
// thread, all sums in double).
__global__ void __launch_bounds__(kThreads) pyr_volume_kernel(const float* __restrict__ inx, const float* __restrict__ iny,
                                                              int w, int h, int d, int dp, float* __restrict__ outx,
                                                              float* __restrict__ outy, int w2, int h2, int d2,
                                                              int dp2) {
  const int strips = (w2 + 7) / 8;
  for (int64_t z = blockIdx.z; z < (int64_t)2 * h2; z += gridDim.z)
  for (int ys = blockIdx.y; ys < strips; ys += gridDim.y) {
    const int i2 = ys * 8 + threadIdx.y;
    if (i2 >= w2) continue;
    const int jz = (int)z;
    const int j2 = jz < h2 ? jz : jz - h2;
    const float* in = jz < h2 ? inx : iny;
    float* out = jz < h2 ? outx : outy;
    const int ia = 2 * i2, ib = min(2 * i2 + 1, w - 1), ja = 2 * j2, jb = min(2 * j2 + 1, h - 1);
    const float* c[4] = {in + ((int64_t)ja * w + ia) * dp, in + ((int64_t)ja * w + ib) * dp,
                         in + ((int64_t)jb * w + ia) * dp, in + ((int64_t)jb * w + ib) * dp};
    float* o = out + ((int64_t)j2 * w2 + i2) * dp2;
    for (int g = blockIdx.x * 32 + threadIdx.x; 4 * g < dp2; g += gridDim.x * 32) {
      float r[4];
      if (4 * g + 4 <= d2 && 8 * g + 8 <= dp) {
        float4 v[4][2];
#pragma unroll
        for (int q = 0; q < 4; q++) {
          v[q][0] = __ldg(reinterpret_cast<const float4*>(c[q] + 8 * g));
          v[q][1] = __ldg(reinterpret_cast<const float4*>(c[q] + 8 * g + 4));
        }
#pragma unroll
        for (int k = 0; k < 4; k++) {
          float x[8];
#pragma unroll
          for (int q = 0; q < 4; q++) {
            const float4& f = v[q][k >> 1];
            x[2 * q] = (k & 1) ? f.z : f.x;
            x[2 * q + 1] = (k & 1) ? f.w : f.y;
          }
          r[k] = mean8(x);
        }
      } else {
#pragma unroll
        for (int k = 0; k < 4; k++) {
          const int k2 = min(4 * g + k, d2 - 1);  // depth pad repeats the last sample
          const int ka = 2 * k2, kb = min(2 * k2 + 1, d - 1);
          float x[8];
#pragma unroll
          for (int q = 0; q < 4; q++) {
            x[2 * q] = c[q][ka];
            x[2 * q + 1] = c[q][kb];
          }
          r[k] = mean8(x);
        }
      }
      *reinterpret_cast<float4*>(o + 4 * g) = make_float4(r[0], r[1], r[2], r[3]);
    }
  }
}

__global__ void pyr_image_kernel(const float* __restrict__ in, int w, int h, float* __restrict__ out) {
  const int w2 = (w + 1) / 2, h2 = (h + 1) / 2;
  const int64_t n = (int64_t)w2 * h2;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int i2 = (int)(e % w2), j2 = (int)(e / w2);
    const int i0 = 2 * i2, i1 = min(2 * i2 + 1, w - 1), j0 = 2 * j2, j1 = min(2 * j2 + 1, h - 1);
    const double s = (double)in[(int64_t)j0 * w + i0] + (double)in[(int64_t)j0 * w + i1] +
                     (double)in[(int64_t)j1 * w + i0] + (double)in[(int64_t)j1 * w + i1];
    out[e] = (float)(s * 0.25);
  }
}

__global__ void pyr_line_kernel(const float* __restrict__ in, int n, float* __restrict__ out) {
  const int n2 = (n + 1) / 2;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n2; e += gridDim.x * blockDim.x)
    out[e] = (float)(((double)in[2 * e] + (double)in[min(2 * e + 1, n - 1)]) * 0.5);
}

// Fine A-scan i sits at (i - 1/2)/2 on the coarse grid (box-filter centres);
// bilinear there with the coordinate clamped into the grid, value doubled
// because the pixel unit halves.
__global__ void prolong_kernel(const double* __restrict__ coarse, int wc, int hc,
                               double* __restrict__ fine, int wf, int hf) {
  const int64_t pf = (int64_t)wf * hf, pc = (int64_t)wc * hc;
  const int64_t n = 6 * pf;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int plane = (int)(e / pf);
    const int64_t q = e % pf;
    const int i = (int)(q % wf), j = (int)(q / wf);
    const double x = fmin(fmax(0.5 * i - 0.25, 0.0), (double)(wc - 1));
    const double y = fmin(fmax(0.5 * j - 0.25, 0.0), (double)(hc - 1));
    const int x0 = (int)x, y0 = (int)y;  // x, y >= 0: truncation is floor
    const int x1 = min(x0 + 1, wc - 1), y1 = min(y0 + 1, hc - 1);
    const double fx = x - x0, fy = y - y0;
    const double* c = coarse + plane * pc;
    const double top = c[(int64_t)y0 * wc + x0] + fx * (c[(int64_t)y0 * wc + x1] - c[(int64_t)y0 * wc + x0]);
    const double bot = c[(int64_t)y1 * wc + x0] + fx * (c[(int64_t)y1 * wc + x1] - c[(int64_t)y1 * wc + x0]);
    fine[e] = 2.0 * (top + fy * (bot - top));
  }
}

inline unsigned grid_for(int64_t n) {
  int64_t b = (n + kThreads - 1) / kThreads;
  if (b < 1) b = 1;
  if (b > 65535) b = 65535;
  return (unsigned)b;
}

}  // namespace

cudaError_t launch_pad_depth(float* vol, int64_t columns, int d, int dp, cudaStream_t s) {
  if (dp == d) return cudaSuccess;
  pad_depth_kernel<<<grid_for(columns * (dp - d)), kThreads, 0, s>>>(vol, columns, d, dp);
  return cudaGetLastError();
}

cudaError_t launch_unpad_depth(const void* vol, int dtype, int64_t columns, int d, int dp, float* out,
                               cudaStream_t s) {
  const unsigned g = grid_for(columns * d);
  if (dtype == OCTMC_BF16)
    unpad_depth_kernel<<<g, kThreads, 0, s>>>(static_cast<const __nv_bfloat16*>(vol), columns, d, dp, out);
  else if (dtype == OCTMC_F16)
    unpad_depth_kernel<<<g, kThreads, 0, s>>>(static_cast<const __half*>(vol), columns, d, dp, out);
  else
    unpad_depth_kernel<<<g, kThreads, 0, s>>>(static_cast<const float*>(vol), columns, d, dp, out);
  return cudaGetLastError();
}

cudaError_t launch_convert(const float* in, void* out, int dtype, int64_t n, cudaStream_t s) {
  const unsigned g = grid_for(n / 4);
  if (dtype == OCTMC_BF16)
    convert_kernel<__nv_bfloat16><<<g, kThreads, 0, s>>>(reinterpret_cast<const float4*>(in), static_cast<uint2*>(out), n / 4);
  else if (dtype == OCTMC_F16)
    convert_kernel<__half><<<g, kThreads, 0, s>>>(reinterpret_cast<const float4*>(in), static_cast<uint2*>(out), n / 4);
  else
    return cudaErrorInvalidValue;
  return cudaGetLastError();
}

cudaError_t launch_pyr_volume(const float* inx, const float* iny, int w, int h, int d, int dp, float* outx, float* outy,
                              int w2, int h2, int d2, int dp2, cudaStream_t s) {
  const dim3 b(32, 8), g((unsigned)std::min((dp2 / 4 + 31) / 32, 1024), (unsigned)std::min((w2 + 7) / 8, 65535),
                         (unsigned)std::min<int64_t>(2 * (int64_t)h2, 65535));
  pyr_volume_kernel<<<g, b, 0, s>>>(inx, iny, w, h, d, dp, outx, outy, w2, h2, d2, dp2);
  return cudaGetLastError();
}

cudaError_t launch_pyr_image(const float* in, int w, int h, float* out, cudaStream_t s) {
  pyr_image_kernel<<<grid_for((int64_t)((w + 1) / 2) * ((h + 1) / 2)), kThreads, 0, s>>>(in, w, h, out);
  return cudaGetLastError();
}

cudaError_t launch_pyr_line(const float* in, int n, float* out, cudaStream_t s) {
  pyr_line_kernel<<<grid_for((n + 1) / 2), kThreads, 0, s>>>(in, n, out);
  return cudaGetLastError();
}

cudaError_t launch_prolong(const double* coarse, int wc, int hc, double* fine, int wf, int hf,
                           cudaStream_t s) {
  prolong_kernel<<<grid_for(6LL * wf * hf), kThreads, 0, s>>>(coarse, wc, hc, fine, wf, hf);
  return cudaGetLastError();
}

}  // namespace octmc
