// Displaced Catmull-Rom sampling of one A-scan by one warp, with its
// derivatives (Ploner et al., Eq. 2): coordinate split and interpolation
// tables, the lane-parallel transverse 4x4 interpolation of aligned groups of
// 4 input samples and the 4-tap axial filter with its halo shuffles.
//
// Depth is processed in blocks of 116 outputs; lane L (1..29) owns outputs
// kb + 4(L-1) .. +3, loads one aligned group of 4 input samples from each of
// the 16 transverse neighbour columns with one 128-bit load per column
// (coalesced along depth across the warp), and gets the neighbouring input
// depths the axial filter needs from the adjacent lanes by shuffles.  Lanes
// 0, 30 and 31 only supply those halo values.
//
// The packed multiply-add (fma.rn.f32x2: two lanes, one issue slot, two FMA
// pipe cycles) takes a scalar broadcast to both halves at no cost but needs
// its pairs in aligned registers.  So the pairs here are (value, derivative):
// the weights come as pairs, each sample is broadcast, and the results of one
// stage are the pairs of the next; pairing neighbouring depths instead costs
// moves in the axial filter, whose taps start at odd offsets (462.4 M against
// 370.3 M warp instructions per launch at 300 x 300 x 512, both with the weights
// read from shared memory; 322.2 M with them in uniform registers, see Sampler).
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "common.cuh"

namespace octmc {
namespace {

constexpr int kOutLanes = 29;
constexpr int kOutPerIter = 4 * kOutLanes;
constexpr unsigned kFull = 0xffffffffu;

// Sampling of one volume at one A-scan: the offsets of the 4 x 4 neighbour
// columns and the interpolation weights, in shared memory (one table per warp
// and volume; every lane reads the same address).
struct alignas(16) VolTab {
  float2 wx[4];     // x weights as (derivative, value)
  float2 wz[4];     // z weights as (value, derivative)
  float2 wy[4];     // y weights as (value, derivative)
  unsigned off[8];  // offsets (in groups of 4 samples) of the 4 neighbour rows, then columns
};

struct Vol {
  const void* base;    // the volume; addressed in groups of 4 samples
  int q, r;            // floor(dz) = 4 q + r, 0 <= r < 4
  int bx, by;          // floor of the transverse coordinates
  float ts;            // the fraction along the scan's slow axis (y for X, x for Y), Eq. 7
};

// Coordinate split of the 6 displacement values of A-scan (i, j) by lanes
// 0..5 (lane = 3 V + c): floor(u) and the float fraction for u = i + dx and
// u = j + dy clamped to [-4, n + 3] (beyond that every tap is an edge sample)
// and u = dz clamped to +-(d + 8) (all depth taps are then edge samples).
// Integer arithmetic only (split_exact).  The lane then evaluates the 4
// weights of its component into the table, once per A-scan.  Returns, in lanes
// 0..15, the clamped index of a neighbour row or column: lanes 0..7 volume X,
// 8..15 volume Y; 4 rows, then 4 columns.
__device__ __forceinline__ int split_pair(Vol& VX, Vol& VY, VolTab* tab, const double* disp, int64_t nasc, int64_t p,
                                          int i, int j, const LevelDev& L, int lane) {
  int b = 0;
  float t = 0.f;
  const int c = lane < 3 ? lane : lane - 3;
  if (lane < 6) {
    const unsigned long long bits =
        (unsigned long long)__double_as_longlong(disp[(int64_t)lane * nasc + p]);
    const int off = c == 0 ? i : (c == 1 ? j : 0);
    const int lo = c == 2 ? -L.d - 8 : -4;
    const int hi = c == 0 ? L.w + 3 : (c == 1 ? L.h + 3 : L.d + 8);
    split_exact(bits, off, lo, hi, &b, &t);
    float w[4], dw[4];
    keys_weights(t, w, dw);
    VolTab& W = tab[lane < 3 ? 0 : 1];
    float2* dst = c == 0 ? W.wx : (c == 1 ? W.wy : W.wz);
#pragma unroll
    for (int a = 0; a < 4; a++) dst[a] = c == 0 ? make_float2(dw[a], w[a]) : make_float2(w[a], dw[a]);
  }
  VX.bx = __shfl_sync(kFull, b, 0);
  VX.by = __shfl_sync(kFull, b, 1);
  const int zx = __shfl_sync(kFull, b, 2);
  VY.bx = __shfl_sync(kFull, b, 3);
  VY.by = __shfl_sync(kFull, b, 4);
  const int zy = __shfl_sync(kFull, b, 5);
  VX.ts = __shfl_sync(kFull, t, 1);
  VY.ts = __shfl_sync(kFull, t, 3);
  VX.q = zx >> 2;  // arithmetic shift: floor division by 4
  VX.r = zx & 3;
  VY.q = zy >> 2;
  VY.r = zy & 3;
  VX.base = L.sx;
  VY.base = L.sy;
  const bool isY = lane >= 8;
  const int a = (lane & 3) - 1;
  return (lane & 4) ? clampi((isY ? VY.bx : VX.bx) + a, L.w) : clampi((isY ? VY.by : VX.by) + a, L.h);
}

// The same with the table's offsets into the volumes in global memory.
__device__ __forceinline__ void setup_pair(Vol& VX, Vol& VY, VolTab* tab, const double* disp, int64_t nasc, int64_t p,
                                           int i, int j, const LevelDev& L, int lane) {
  const int n = split_pair(VX, VY, tab, disp, nasc, p, i, j, L, lane);
  const unsigned nq = (unsigned)(L.dp >> 2);
  if (lane < 16) tab[lane >> 3].off[lane & 7] = (unsigned)n * ((lane & 4) ? nq : (unsigned)L.w * nq);
  __syncwarp();
}

// Four consecutive samples (one aligned group) widened to float: float32
// storage is one 16-byte load, bfloat16/float16 one 8-byte load.
template <typename T>
__device__ __forceinline__ float4 load4(const void* base, unsigned idx);
template <>
__device__ __forceinline__ float4 load4<float>(const void* base, unsigned idx) {
  return __ldg(reinterpret_cast<const float4*>(base) + idx);
}
template <>
__device__ __forceinline__ float4 load4<__nv_bfloat16>(const void* base, unsigned idx) {
  const uint2 u = __ldg(reinterpret_cast<const uint2*>(base) + idx);
  return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u),
                     __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
}
template <>
__device__ __forceinline__ float4 load4<__half>(const void* base, unsigned idx) {
  const uint2 u = __ldg(reinterpret_cast<const uint2*>(base) + idx);
  const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
  const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
  return make_float4(a.x, a.y, b.x, b.y);
}

// ---------------------------------------------------------------- packed float pairs
// Two float lanes per instruction (fma.rn.f32x2): each half is rounded like
// fmaf, so packed and scalar code give bitwise equal results; the packed
// form halves the issue slots of the interpolation's multiply-adds.
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
      "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}

__device__ __forceinline__ float2 fmul2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "mul.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 both(float s) { return make_float2(s, s); }

// Axial 4-tap filter of NQ quantities for the lane's 4 outputs: the lane's
// group of each is e[1..4], e[0] the last sample of lane - 1's group, e[5..8]
// lane + 1's group and e[9] the first sample of lane + 2's.  Output o, tap c
// reads e[R + o + c], where R = floor(dz) mod 4.
template <int R>
__device__ __forceinline__ void halo(float e[10]) {
  if (R == 0) e[0] = __shfl_up_sync(kFull, e[4], 1);
  e[5] = __shfl_down_sync(kFull, e[1], 1);
  e[6] = __shfl_down_sync(kFull, e[2], 1);
  if (R >= 1) e[7] = __shfl_down_sync(kFull, e[3], 1);
  if (R >= 2) e[8] = __shfl_down_sync(kFull, e[4], 1);
  if (R == 3) e[9] = __shfl_down_sync(kFull, e[1], 2);
}

template <int R>
__device__ __forceinline__ void axial(const float T[4], const float2 Txy[4], const float2 wz[4], float2 Iz[4],
                                      float2 Ixy[4]) {
  float e[10], ex[10], ey[10];
#pragma unroll
  for (int k = 0; k < 4; k++) {
    e[1 + k] = T[k];
    ex[1 + k] = Txy[k].x;
    ey[1 + k] = Txy[k].y;
  }
  halo<R>(e);
  halo<R>(ex);
  halo<R>(ey);
#pragma unroll
  for (int o = 0; o < 4; o++) {
    float2 a = fmul2(wz[0], both(e[R + o]));
    float2 g = fmul2(both(wz[0].x), make_float2(ex[R + o], ey[R + o]));
#pragma unroll
    for (int c = 1; c < 4; c++) {
      a = ffma2(wz[c], both(e[R + o + c]), a);
      g = ffma2(both(wz[c].x), make_float2(ex[R + o + c], ey[R + o + c]), g);
    }
    Iz[o] = a;
    Ixy[o] = g;
  }
}

// The table's weights and offsets as warp-uniform values.  A warp reduction
// delivers its result in a uniform register, which the packed multiply-add
// takes as an operand, so the 48 weights and 16 offsets of an A-scan hardly need
// the vector registers that limit the warps per SM: 64 registers hold all of
// them with about 110 bytes spilled.  Read from shared memory in every depth
// block instead (72 registers) they cost the L1 data pipe, the kernel's bound:
// 300 x 300 x 512, float32 466 -> 420 us, bfloat16 446 -> 395 us; 237 x 301 x
// 465, float16 358 -> 332 us.
struct Sampler {
  float2 wx[4], wy[4], wz[4];
  unsigned roff[4], coff[4];
  static __device__ __forceinline__ unsigned uniform(unsigned v) { return __reduce_or_sync(kFull, v); }
  static __device__ __forceinline__ float2 uniform(float2 v) {
    return make_float2(__uint_as_float(uniform(__float_as_uint(v.x))), __uint_as_float(uniform(__float_as_uint(v.y))));
  }
  __device__ __forceinline__ explicit Sampler(const VolTab& T) {
#pragma unroll
    for (int a = 0; a < 4; a++) {
      wx[a] = uniform(T.wx[a]);
      wy[a] = uniform(T.wy[a]);
      wz[a] = uniform(T.wz[a]);
      roff[a] = uniform(T.off[a]);
      coff[a] = uniform(T.off[4 + a]);
    }
  }
};

// (I, dI/dz) and (dI/dx, dI/dy) of one volume at the lane's 4 outputs.  qk:
// first input depth of the lane's group (samples, may lie outside the
// volume); load(b, a): the group's (clamped) samples in neighbour row b, column
// a.
template <typename Load>
__device__ __forceinline__ void sample_group(const Sampler& W, int r, int qk, int dp, Load&& load, float2 Iz[4],
                                             float2 Ixy[4]) {
  float T[4];
  float2 Txy[4];
#pragma unroll
  for (int b = 0; b < 4; b++) {
    float2 U[4];  // (d/dx, value) of row b
#pragma unroll
    for (int a = 0; a < 4; a++) {
      const float4 f = load(b, a);
      const float s[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
      for (int k = 0; k < 4; k++) U[k] = a == 0 ? fmul2(W.wx[0], both(s[k])) : ffma2(W.wx[a], both(s[k]), U[k]);
    }
#pragma unroll
    for (int k = 0; k < 4; k++) {
      Txy[k] = b == 0 ? fmul2(W.wy[0], U[k]) : ffma2(W.wy[b], U[k], Txy[k]);
      T[k] = b == 0 ? W.wy[0].x * U[k].y : fmaf(W.wy[b].x, U[k].y, T[k]);
    }
  }
  // groups entirely before sample 0 / after the last sample hold the edge value
  if (__any_sync(kFull, (unsigned)qk >= (unsigned)dp)) {
    if (qk < 0) {
#pragma unroll
      for (int k = 1; k < 4; k++) { T[k] = T[0]; Txy[k] = Txy[0]; }
    } else if (qk >= dp) {
#pragma unroll
      for (int k = 0; k < 3; k++) { T[k] = T[3]; Txy[k] = Txy[3]; }
    }
  }
  switch (r) {
    case 0: axial<0>(T, Txy, W.wz, Iz, Ixy); break;
    case 1: axial<1>(T, Txy, W.wz, Iz, Ixy); break;
    case 2: axial<2>(T, Txy, W.wz, Iz, Ixy); break;
    default: axial<3>(T, Txy, W.wz, Iz, Ixy); break;
  }
}

// The same at the lane's 4 outputs of the depth block starting at kb, from the
// volume in global memory.
template <typename S>
__device__ __forceinline__ void sample_block(const Vol& V, const Sampler& W, int kb, int lane, int dp, float2 Iz[4],
                                             float2 Ixy[4]) {
  const int qk = kb + 4 * V.q + 4 * (lane - 1);  // first input depth of the lane's group
  const unsigned qc = (unsigned)(min(max(qk, 0), dp - 4) >> 2);
  sample_group(W, V.r, qk, dp, [&](int b, int a) { return load4<S>(V.base, W.roff[b] + W.coff[a] + qc); }, Iz, Ixy);
}

}  // namespace
}  // namespace octmc
