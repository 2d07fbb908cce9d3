// Data term of one output A-scan by one warp (Ploner et al., Eq. 2-8),
// shared by the data-term kernels and the persistent small-level solve:
// the two displaced Catmull-Rom resamplings, the loss and its depth sums,
// the per-A-scan angiography, validity and delta, and the eight outputs.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "common.cuh"
#include "sample.cuh"

namespace octmc {
namespace {

// Eq. 4 (or squared differences) of a residual and its derivative.  The
// pseudo-Huber loss is evaluated as (R^2/eps) / (1 + sqrt(1 + (R/eps)^2)): no
// cancellation near 0.  The square root's argument is at least 1 and the
// divisor between 1 and 2^65, so neither of their flush-to-zero approximations
// meets a subnormal, and they save its scaling.  The numerator R^2/eps can be
// subnormal: it is multiplied by the divisor's reciprocal without flushing.
__device__ __forceinline__ float rsqrt_ge1(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_ge1(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void loss_grad(float R, float inv_eps, bool ssd, float* Lv, float* dL) {
  if (ssd) {
    *Lv = R * R;
    *dL = 2.0f * R;
  } else {
    const float rr = R * inv_eps;
    const float qv = fmaf(rr, rr, 1.0f);
    const float is = rsqrt_ge1(qv);
    *dL = rr * is;
    *Lv = __fmul_rn(R * rr, rcp_ge1(fmaf(qv, is, 1.0f)));
  }
}

// Totals over the warp of 8 per-lane values: lane 4 v + x ends with the total
// of value v.  The lanes are paired as in a butterfly (16, 8, 4, 2, 1), but
// each of the first three stages keeps half of the values, so 9 shuffles do
// the work of 40; the sums are those of a butterfly per value.
__device__ __forceinline__ float warp_totals8(float v[8], int lane) {
#pragma unroll
  for (int n = 4; n >= 1; n >>= 1) {
    const bool up = (lane & (4 * n)) != 0;
#pragma unroll
    for (int k = 0; k < n; k++) {
      const float send = up ? v[k] : v[k + n];
      const float keep = up ? v[k + n] : v[k];
      v[k] = keep + __shfl_xor_sync(kFull, send, 4 * n);
    }
  }
  float t = v[0];
  t += __shfl_xor_sync(kFull, t, 2);
  t += __shfl_xor_sync(kFull, t, 1);
  return t;
}

// Adds one depth block to the sums acc: L, then the x, y, z sums of dL dI for X
// and for Y.  left: outputs inside the volume from the lane's first output on;
// those outside add nothing, whatever their lanes hold.
__device__ __forceinline__ void add_block(float acc[8], const float2 XZ[4], const float2 XG[4], const float2 YZ[4],
                                          const float2 YG[4], int left, float inv_eps, bool ssd) {
  auto add = [&](int o) {
    float Lv, dL;
    loss_grad(XZ[o].x - YZ[o].x, inv_eps, ssd, &Lv, &dL);
    acc[0] += Lv;
    float2 t = ffma2(both(dL), XG[o], make_float2(acc[1], acc[2]));
    acc[1] = t.x; acc[2] = t.y;
    acc[3] = fmaf(dL, XZ[o].y, acc[3]);
    t = ffma2(both(dL), YG[o], make_float2(acc[4], acc[5]));
    acc[4] = t.x; acc[5] = t.y;
    acc[6] = fmaf(dL, YZ[o].y, acc[6]);
  };
  if (left >= 4) {
#pragma unroll
    for (int o = 0; o < 4; o++) add(o);
  } else if (left > 0) {
    add(0);
    if (left > 1) add(1);
    if (left > 2) add(2);
  }
}

// The outputs of an A-scan from its depth sums: lane 4 v returns output v: v = 0
// the structural term, v = 1 + 3 V + c the gradient component c of scan V; lane
// 28 the angiographic term.
__device__ __forceinline__ float data_outputs(const DataArgs& A, const VolTab* tab, const Vol& VX, const Vol& VY,
                                              float acc[8], float inv_eps, bool ssd, int lane) {
  const LevelDev& L = A.L;
  // the loads of the epilogue together, before the sums: this lane's tap of the
  // en-face images (lanes 0..15 A^X, 16..31 A^Y) and, in lanes 0..3, the
  // validity nodes around the displaced positions.  (Issued ahead of the depth
  // loop they cost 11 us at 300 x 300 x 512 in spilled registers.)
  const bool isX = lane < 16;
  const int ta = lane & 3, tb = (lane >> 2) & 3;
  float tap = 0.f, node = 1.f;
  if (L.ax)
    tap = (isX ? L.ax : L.ay)[(int64_t)clampi((isX ? VX.by : VY.by) - 1 + tb, L.h) * L.w +
                              clampi((isX ? VX.bx : VY.bx) - 1 + ta, L.w)];
  if (lane < 2) {
    if (L.vx) node = L.vx[clampi(VX.by + lane, L.h)];
  } else if (lane < 4) {
    if (L.vy) node = L.vy[clampi(VY.bx + lane - 2, L.w)];
  }

  const float tot = warp_totals8(acc, lane);
  const float Lsum = __shfl_sync(kFull, tot, 0);

  // ---- per-A-scan scalars (Eq. 6-8), float, every lane
  // Eq. 7: X validity along y at j + dy^X, Y validity along x at i + dx^Y,
  // by the zero-tangent Hermite interpolant (no overshoot: 0 <= delta <= delta_0)
  float vtx, dvtx, vty, dvty;
  hermite01(__shfl_sync(kFull, node, 0), __shfl_sync(kFull, node, 1), VX.ts, &vtx, &dvtx);
  hermite01(__shfl_sync(kFull, node, 2), __shfl_sync(kFull, node, 3), VY.ts, &vty, &dvty);
  const float delta0 = (float)A.delta0;
  const float delta = delta0 * vtx * vty;  // Eq. 8
  const float d = (float)L.d;

  // Eq. 6: the 16 taps of either image, a butterfly within each half-warp
  float La = 0.f, dLa = 0.f, im = 0.f;
  const int v = lane >> 2;  // this lane's output
  if (L.ax) {
    const VolTab& S = tab[isX ? 0 : 1];
    const float wa = S.wx[ta].y, dwa = S.wx[ta].x, wb = S.wy[tb].x, dwb = S.wy[tb].y;
    float a = wa * wb * tap, ax = dwa * wb * tap, ay = wa * dwb * tap;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
      a += __shfl_xor_sync(kFull, a, o);
      ax += __shfl_xor_sync(kFull, ax, o);
      ay += __shfl_xor_sync(kFull, ay, o);
    }
    const float other = __shfl_xor_sync(kFull, a, 16);
    loss_grad(isX ? a - other : other - a, inv_eps, ssd, &La, &dLa);
    // the image derivative of gradient components x and y; outputs 1, 2 lie in
    // the lanes of A^X, 4, 5 in those of A^Y
    im = (v == 1 || v == 4) ? ax : ay;
  }

  const float eta = (float)(A.eta_dev ? *A.eta_dev : A.eta);
  const float cs = eta * (1.0f - delta);
  const float ca = delta * d / eta * dLa;
  const float ddelta = -eta * Lsum + d * La / eta;
  // scan Y enters the residuals with the opposite sign
  float out = v < 4 ? cs * tot : -cs * tot;
  if (v == 1 || v == 2) out = fmaf(ca, im, out);
  if (v == 4 || v == 5) out = fmaf(-cs, tot, -(ca * im));
  if (v == 2) out = fmaf(ddelta * delta0 * dvtx, vty, out);
  if (v == 4) out = fmaf(ddelta * delta0 * vtx, dvty, out);
  if (v == 0) out = (1.0f - delta) * Lsum;
  if (v == 7) out = delta * d * La;
  return out;
}

// The data-term computation of output A-scan p (i, j) by one warp from the
// volumes in global memory, with `tab` (2 entries) the warp's shared-memory
// table; the value of this lane's output (see data_outputs).
template <typename T>
__device__ __forceinline__ float data_value(const DataArgs& A, VolTab* tab, int64_t p, int i, int j, int lane) {
  const LevelDev& L = A.L;
  Vol VX, VY;
  setup_pair(VX, VY, tab, A.disp, (int64_t)L.w * L.h, p, i, j, L, lane);
  const Sampler WX(tab[0]), WY(tab[1]);
  const float inv_eps = 1.0f / A.eps_h;
  const bool ssd = (A.loss == OCTMC_LOSS_SSD);
  float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  // outputs inside the volume from this lane's first output on (none for the halo lanes)
  int left = (lane >= 1 && lane <= kOutLanes) ? L.d - 4 * (lane - 1) : 0;
  for (int kb = 0; kb < L.d; kb += kOutPerIter, left -= kOutPerIter) {
    float2 XZ[4], XG[4], YZ[4], YG[4];
    sample_block<T>(VX, WX, kb, lane, L.dp, XZ, XG);
    sample_block<T>(VY, WY, kb, lane, L.dp, YZ, YG);
    add_block(acc, XZ, XG, YZ, YG, left, inv_eps, ssd);
  }
  return data_outputs(A, tab, VX, VY, acc, inv_eps, ssd, lane);
}

// ---- fields without transverse displacement (the axial prealignment)
// At dx = dy = 0 the transverse weights are exactly (0, 1, 0, 0), so the
// interpolant is the A-scan's own column filtered along depth: one column per
// scan instead of 16, the same floats in the same order as data_value.  Only
// the axial gradient components (c = 2) are formed.
template <int R>
__device__ __forceinline__ void axial_z(const float T[4], const float2 wz[4], float2 Iz[4]) {
  float e[10];
#pragma unroll
  for (int k = 0; k < 4; k++) e[1 + k] = T[k];
  halo<R>(e);
#pragma unroll
  for (int o = 0; o < 4; o++) {
    float2 a = fmul2(wz[0], both(e[R + o]));
#pragma unroll
    for (int c = 1; c < 4; c++) a = ffma2(wz[c], both(e[R + o + c]), a);
    Iz[o] = a;
  }
}

__device__ __forceinline__ void column_filter(float4 f, int qk, int dp, int r, const float2 wz[4], float2 Iz[4]) {
  // groups entirely before sample 0 / after the last sample hold the edge value
  if (__any_sync(kFull, (unsigned)qk >= (unsigned)dp)) {
    if (qk < 0) f.y = f.z = f.w = f.x;
    else if (qk >= dp) f.x = f.y = f.z = f.w;
  }
  const float T[4] = {f.x, f.y, f.z, f.w};
  switch (r) {
    case 0: axial_z<0>(T, wz, Iz); break;
    case 1: axial_z<1>(T, wz, Iz); break;
    case 2: axial_z<2>(T, wz, Iz); break;
    default: axial_z<3>(T, wz, Iz); break;
  }
}

template <typename T>
__device__ __forceinline__ void data_column(const DataArgs& A, int64_t p, int i, int j, int lane) {
  const LevelDev& L = A.L;
  const int64_t nasc = (int64_t)L.w * L.h;
  int b = 0;
  float t = 0.f;
  if (lane < 2)  // lane = scan
    split_exact((unsigned long long)__double_as_longlong(A.disp[(int64_t)(3 * lane + 2) * nasc + p]), 0, -L.d - 8,
                L.d + 8, &b, &t);
  const int zx = __shfl_sync(kFull, b, 0), zy = __shfl_sync(kFull, b, 1);
  float2 wx[4], wy[4];  // axial weights of scan X, scan Y
  {
    float w[4], dw[4];
    keys_weights(__shfl_sync(kFull, t, 0), w, dw);
#pragma unroll
    for (int a = 0; a < 4; a++) wx[a] = make_float2(w[a], dw[a]);
    keys_weights(__shfl_sync(kFull, t, 1), w, dw);
#pragma unroll
    for (int a = 0; a < 4; a++) wy[a] = make_float2(w[a], dw[a]);
  }
  const unsigned col = (unsigned)p * (unsigned)(L.dp >> 2);
  const float inv_eps = 1.0f / A.eps_h;
  const bool ssd = (A.loss == OCTMC_LOSS_SSD);
  int left = (lane >= 1 && lane <= kOutLanes) ? L.d - 4 * (lane - 1) : 0;
  // first input depth of the lane's group, as in sample_block
  int qx = 4 * (zx >> 2) + 4 * (lane - 1), qy = 4 * (zy >> 2) + 4 * (lane - 1);
  auto load = [&](const void* vol, int qk) { return load4<T>(vol, col + (unsigned)(min(max(qk, 0), L.dp - 4) >> 2)); };
  float4 fx = load(L.sx, qx), fy = load(L.sy, qy);
  float Ls = 0.f, gx = 0.f, gy = 0.f;
  for (int kb = 0; kb < L.d; kb += kOutPerIter, left -= kOutPerIter) {
    // the next depth block's loads are in flight while this one is computed
    float4 nx, ny;
    const bool more = kb + kOutPerIter < L.d;
    if (more) {
      nx = load(L.sx, qx + kOutPerIter);
      ny = load(L.sy, qy + kOutPerIter);
    }
    float2 X[4], Y[4];
    column_filter(fx, qx, L.dp, zx & 3, wx, X);
    column_filter(fy, qy, L.dp, zy & 3, wy, Y);
    auto add = [&](int o) {
      float Lv, dL;
      loss_grad(X[o].x - Y[o].x, inv_eps, ssd, &Lv, &dL);
      Ls += Lv;
      gx = fmaf(dL, X[o].y, gx);
      gy = fmaf(dL, Y[o].y, gy);
    };
    if (left >= 4) {
#pragma unroll
      for (int o = 0; o < 4; o++) add(o);
    } else if (left > 0) {
      add(0);
      if (left > 1) add(1);
      if (left > 2) add(2);
    }
    if (more) {
      fx = nx;
      fy = ny;
    }
    qx += kOutPerIter;
    qy += kOutPerIter;
  }
  Ls = warp_sum(Ls);
  gx = warp_sum(gx);
  gy = warp_sum(gy);
  if (lane > 2) return;
  // validity and angiography at the A-scan itself (Eq. 6-8)
  float delta = (float)A.delta0;
  if (L.vx) delta *= L.vx[j];
  if (L.vy) delta *= L.vy[i];
  float La = 0.f, dLa = 0.f;
  if (L.ax) loss_grad(L.ax[p] - L.ay[p], inv_eps, ssd, &La, &dLa);
  const float eta = (float)(A.eta_dev ? *A.eta_dev : A.eta);
  const float cs = eta * (1.0f - delta);
  if (lane == 0) A.str_out[p] = (1.0f - delta) * Ls;
  else if (lane == 1) A.ang_out[p] = delta * (float)L.d * La;
  if (A.grad && lane >= 1) A.grad[(lane == 1 ? 2 : 5) * nasc + p] = lane == 1 ? cs * gx : -cs * gy;
}

// This lane's output of A-scan p written out.
__device__ __forceinline__ void data_store(const DataArgs& A, int64_t p, float out, int lane) {
  const int64_t nasc = (int64_t)A.L.w * A.L.h;
  const int v = lane >> 2;
  if (lane & 3) return;
  if (v == 0) A.str_out[p] = out;
  else if (v == 7) A.ang_out[p] = out;
  else if (A.grad) A.grad[(int64_t)(v - 1) * nasc + p] = out;
}

// Output A-scan p = (i, j) by one warp: data_value written out.
template <typename T>
__device__ __forceinline__ void data_ascan(const DataArgs& A, VolTab* tab, int64_t p, int i, int j, int lane) {
  data_store(A, p, data_value<T>(A, tab, p, i, j, lane), lane);
}

}  // namespace
}  // namespace octmc
