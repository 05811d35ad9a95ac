// Arithmetic of the inner ADMM (Appendix D) shared by the iteration's kernels
// and the gradient's: FP32 operations written with their rounding, and the
// register-resident tridiagonal solve.
#ifndef OPF_TRI_H_
#define OPF_TRI_H_

#include <cuda_runtime.h>

namespace opfk {

constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float radd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float rsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float rdiv(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }

// x / q by the rounded reciprocal rq = 1 / q and one residual correction, in
// three dependent operations: the division's result, correctly rounded, while
// q, x and the quotient are normal numbers with room for the residual (|q| <=
// 2^126, |x| >= 2^-100 or 0).  rq is within half an ulp of 1 / q and q0 within
// 1.5 ulp of x / q, the residual is exact, so the sum rounds wrongly only if
// x / q lies within 1.5 * 2^-24 ulp of a rounding boundary: |x 2^k - M q| <= 3
// for a boundary M and significands x, q < 2^24.  All pairs with |...| <= 16
// round as the division does (8e8 of them, enumerated; the test samples them).
// Smaller x: within one ulp.  An infinite q, x or quotient gives NaN.
__device__ __forceinline__ float qdiv(float x, float q, float rq) {
  const float q0 = rmul(x, rq);
  return rfma(rfma(-q0, q, x), rq, q0);
}

// The tridiagonal system of a device, as the solves of its inner iterations
// read it (element i = lane C + j, valid while i < n): pivots q, their
// reciprocals rq, a = -off / q, and the multipliers of the two warp scans.  A
// scan composes the lanes' affine maps x -> A x + B; the A of a lane at each
// scan step depends on the pivots alone, so it is formed once per device and
// the scans of the ten inner iterations move only B: one shuffle and one FMA
// per step in place of two shuffles, an FMA and a product, and no division
// sequence in the chain.  Bound: latency (the chain of dependent shuffles).
template <int C>
struct TriFac {
  float q[C], rq[C], a[C], f[5], b[5];
  // q set (1 from element n on); off_neg = -off
  __device__ __forceinline__ void init(float off_neg, int n, int lane) {
#pragma unroll
    for (int j = 0; j < C; ++j) {
      rq[j] = __frcp_rn(q[j]);
      a[j] = lane * C + j < n ? qdiv(off_neg, q[j], rq[j]) : 0.f;
    }
    init_scans(n, lane);
  }
  // q and a set (1 and 0 from element n on)
  __device__ __forceinline__ void init(int n, int lane) {
#pragma unroll
    for (int j = 0; j < C; ++j) rq[j] = __frcp_rn(q[j]);
    init_scans(n, lane);
  }
  __device__ __forceinline__ void init_scans(int n, int lane) {
    const int i0 = lane * C;
    float Af = 1.f, Ab = 1.f;
#pragma unroll
    for (int j = 0; j < C; ++j) Af = rmul((i0 + j == 0) ? 0.f : a[j], Af);
#pragma unroll
    for (int j = C - 1; j >= 0; --j) Ab = rmul((i0 + j == n - 1) ? 0.f : a[j], Ab);
#pragma unroll
    for (int l = 0; l < 5; ++l) {
      const int d = 1 << l;
      f[l] = Af;
      b[l] = Ab;
      const float Pf = __shfl_up_sync(FULL, Af, d), Pb = __shfl_down_sync(FULL, Ab, d);
      if (lane >= d) Af = rmul(Af, Pf);
      if (lane + d < 32) Ab = rmul(Ab, Pb);
    }
  }
};

// x := M^-1 x on a chunk held in registers: first-order recurrences (forward
// y_i = a_i y_{i-1} + r_i / q_i, then backward) composed over each lane's
// chunk, then across the warp by shuffle scans.  Elements from n on take part
// with x = 0, pivot 1 and a = 0 (and stay 0), so no lane branches.
template <int C>
__device__ __forceinline__ void warp_tri_solve_r(const TriFac<C> &m, float (&x)[C], int n, int lane) {
  const int i0 = lane * C;
  float r[C];
  float Bc = 0.f;
#pragma unroll
  for (int j = 0; j < C; ++j) {
    r[j] = qdiv(x[j], m.q[j], m.rq[j]);
    Bc = rfma((i0 + j == 0) ? 0.f : m.a[j], Bc, r[j]);
  }
#pragma unroll
  for (int l = 0; l < 5; ++l) {
    const float Bp = __shfl_up_sync(FULL, Bc, 1 << l);
    if (lane >= (1 << l)) Bc = rfma(m.f[l], Bp, Bc);
  }
  float prev = __shfl_up_sync(FULL, Bc, 1);
  if (lane == 0) prev = 0.f;
#pragma unroll
  for (int j = 0; j < C; ++j) {
    prev = rfma((i0 + j == 0) ? 0.f : m.a[j], prev, r[j]);
    x[j] = prev;
  }
  Bc = 0.f;
#pragma unroll
  for (int j = C - 1; j >= 0; --j) Bc = rfma((i0 + j == n - 1) ? 0.f : m.a[j], Bc, x[j]);
#pragma unroll
  for (int l = 0; l < 5; ++l) {
    const float Bp = __shfl_down_sync(FULL, Bc, 1 << l);
    if (lane + (1 << l) < 32) Bc = rfma(m.b[l], Bp, Bc);
  }
  float nxt = __shfl_down_sync(FULL, Bc, 1);
  if (lane == 31) nxt = 0.f;
#pragma unroll
  for (int j = C - 1; j >= 0; --j) {
    nxt = rfma((i0 + j == n - 1) ? 0.f : m.a[j], nxt, x[j]);
    x[j] = nxt;
  }
}

}  // namespace opfk

#endif  // OPF_TRI_H_
