// History update and compact-form L-BFGS algebra of the device-resident
// level solve (Ploner et al., Sec. 2.1; Byrd, Nocedal & Schnabel compact
// representation), shared by the products kernel and the persistent
// small-level kernel.  Each block that runs it works on its own copy of the
// SolveState.
#pragma once
#include <math.h>
#include <stddef.h>

#include "common.cuh"

namespace octmc {
namespace {

// ---- history update, after the products are known: S the working copy of the
// state, SY and YY the products of the stored pairs (by buffer id).  Every
// thread of the block; barriers around it are the caller's.
__device__ void history_update(SolveState* S, double* SY, double* YY) {
  const double* r = S->dots;
  const int K = 2 * S->ncand, k = S->k, nb = S->spare, tid = threadIdx.x;
  bool stored = false;
  if (S->mode == kModeAccept) {
    // the new pair is the last candidate
    const double s_y = r[2 * (2 * k)], y_y = r[2 * K];
    stored = s_y > 1e-12 * y_y && isfinite(s_y) && isfinite(y_y);
    if (stored) {
      if (tid < k) {
        const int b = S->order[tid];
        SY[b * (kMaxM + 1) + nb] = r[2 * (2 * tid)];
        const double v = r[2 * (2 * tid + 1)];
        YY[b * (kMaxM + 1) + nb] = v;
        YY[nb * (kMaxM + 1) + b] = v;
      } else if (tid == k) {
        SY[nb * (kMaxM + 1) + nb] = s_y;
        YY[nb * (kMaxM + 1) + nb] = y_y;
      }
    }
  }
  if (tid < S->ncand) {
    const int b = S->cand[tid];
    S->sg[b] = r[2 * (2 * tid) + 1];
    S->yg[b] = r[2 * (2 * tid + 1) + 1];
  }
  __syncthreads();  // order, k and spare are read above, changed below
  if (tid == 0) {
    S->gg = r[2 * K + 1];
    if (stored) {
      int kk = k;
      if (kk == S->m) {
        for (int t = 0; t + 1 < kk; t++) S->order[t] = S->order[t + 1];
        kk--;
      }
      S->order[kk++] = nb;
      S->k = kk;
      // the spare buffer: the first id not in the history
      unsigned long long used = 0ull;
      for (int t = 0; t < kk; t++) used |= 1ull << S->order[t];
      S->spare = __ffsll((long long)~used) - 1;
    }
  }
}

// Block-wide copy of the solver state, 16 bytes per load, all of a thread's
// loads issued before its stores.
template <int kBlock, size_t kBytes>
__device__ __forceinline__ void copy_state(void* dst, const void* src) {
  constexpr int kWords = (int)(kBytes / 16);
  constexpr int kPer = (kWords + kBlock - 1) / kBlock;
  const int4* s4 = reinterpret_cast<const int4*>(src);
  int4* d4 = reinterpret_cast<int4*>(dst);
  int4 buf[kPer];
#pragma unroll
  for (int i = 0; i < kPer; i++) {
    const int w = threadIdx.x + i * kBlock;
    if (w < kWords) buf[i] = s4[w];
  }
#pragma unroll
  for (int i = 0; i < kPer; i++) {
    const int w = threadIdx.x + i * kBlock;
    if (w < kWords) d4[w] = buf[i];
  }
}
constexpr size_t kStateHead = offsetof(SolveState, SY);  // without the products of the stored pairs
static_assert(sizeof(SolveState) % 16 == 0 && kStateHead % 16 == 0, "solver state is copied in 16-byte words");

// After the products: history update and the compact-form
// (Byrd, Nocedal & Schnabel) direction dir = -H g with H0 = gamma I, gamma
// from the newest pair, as coefficients of g and the history vectors; g . dir
// follows from the products (no extra pass).  Run by every thread of one
// block: the k x k blocks of S'Y and Y'Y are staged in shared memory, then one
// warp holds one pair per lane (k <= 32).  Every sum keeps the order of the
// serial recursion -- a solve's iterates depend on its last bits -- so
// u = R^{-1} a stays a chain of k (k - 1) / 2 multiply-adds (its operands come
// ahead of it by shuffles), while the rows of w and of R^{-T} w run in
// parallel.
struct Algebra {
  double R[kMaxM][kMaxM + 1];   // R_ij = s_i . y_j
  double YY[kMaxM][kMaxM + 1];  // y_i . y_j
  double a[kMaxM], b[kMaxM], u[kMaxM], top[kMaxM];
};

__device__ void after_products(SolveState* S, double* SY, double* YY, Algebra& A) {
  history_update(S, SY, YY);
  __syncthreads();
  const int k = S->k;
  for (int t = threadIdx.x; t < k * k; t += blockDim.x) {
    const int i = t / k, j = t % k, e = S->order[i] * (kMaxM + 1) + S->order[j];
    A.R[i][j] = SY[e];
    A.YY[i][j] = YY[e];
  }
  __syncthreads();
  if (threadIdx.x >= 32) return;
  const int lane = threadIdx.x;
  constexpr unsigned kAll = 0xffffffffu;
  double gamma = 0.0;
  if (k > 0) {
    const bool in = lane < k;
    const int buf = in ? S->order[lane] : 0;
    const double a = in ? S->sg[buf] : 0.0, b = in ? S->yg[buf] : 0.0;
    // the divisions (long float64 sequences) off the serial solves below
    const double rd = in ? 1.0 / A.R[lane][lane] : 0.0;
    gamma = A.R[k - 1][k - 1] / A.YY[k - 1][k - 1];
    double u = 0.0;
    for (int i = k - 1; i >= 0; i--) {  // u = R^{-1} a (R upper triangular), every lane the same chain
      double s = __shfl_sync(kAll, a, i);
#pragma unroll 4
      for (int j = i + 1; j < k; j++) s = fma(-A.R[i][j], __shfl_sync(kAll, u, j), s);
      s *= __shfl_sync(kAll, rd, i);
      if (lane == i) u = s;
    }
    double s = in ? A.R[lane][lane] * u : 0.0;  // w = (D + gamma Y'Y) u - gamma b
    for (int j = 0; j < k; j++) {
      const double uj = __shfl_sync(kAll, u, j);
      if (in) s = fma(gamma * A.YY[lane][j], uj, s);
    }
    s = fma(-gamma, b, s);
    double top = 0.0;
    for (int i = 0; i < k; i++) {  // top = R^{-T} w: row i subtracts its terms as they become known
      const double ti = __shfl_sync(kAll, s * rd, i);
      if (lane == i) top = ti;
      if (lane > i && in) s = fma(-A.R[i][lane], ti, s);
    }
    if (in) {
      A.a[lane] = a;
      A.b[lane] = b;
      A.u[lane] = u;
      A.top[lane] = top;
      S->hid[2 * lane] = 2 * buf;
      S->coef[2 * lane] = -top;
      S->hid[2 * lane + 1] = 2 * buf + 1;
      S->coef[2 * lane + 1] = gamma * u;
    }
  }
  __syncwarp();
  if (lane != 0) return;
  double gd;
  if (k > 0) {
    S->cg = -gamma;
    S->nc = 2 * k;
    gd = -gamma * S->gg;
    for (int i = 0; i < k; i++) gd += -A.top[i] * A.a[i] + gamma * A.u[i] * A.b[i];
    if (!(gd < 0.0)) {  // not a descent direction: drop the history, -g
      S->k = 0;
      S->cg = -1.0;
      S->nc = 0;
      gd = -S->gg;
    }
  } else {
    S->cg = -1.0;
    S->nc = 0;
    gd = -S->gg;
  }
  S->dg0 = gd;
  S->a = (S->k == 0) ? 1.0 / sqrt(S->gg) : 1.0;
  S->lo = 0.0;
  S->hi = INFINITY;
  S->have_lo = 0;
  S->ls = 0;
  S->mode = kModeTrial;
}

}  // namespace
}  // namespace octmc
