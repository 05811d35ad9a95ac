// Proximal message passing for contingency-constrained DC OPF -- sm_103a kernels.
//
// One iteration of the message-passing form of ADMM (Section 3.2) is three
// phases replayed from CUDA graphs; each kernel reads the iteration's scalars
// (penalty factors, buffer parity, whether residuals are read) from the
// device, so the same graph serves every iteration:
//   dev    step 2: avg_k(pbar + u) from the stored pbar + u at every node with
//          devices (a node's K+1 rows are one run), the closed-form prox with
//          weight (K+1) rho_p of its generators/loads, and one warp per
//          ramp-limited generator, battery or HVDC link: the inner ADMM of
//          Appendix D (lanes over time steps, tridiagonal x-updates by
//          warp-wide scans) or the link's closed form.  Where the line pass is
//          long enough to hide the devices this is three kernels: xs (averages
//          and closed forms), dev (the inner ADMM alone), dsum (the node sums
//          of device powers and their Welford change state);
//   line   step 1, one thread per (line, contingency, 4 time steps): the line
//          prox from the previous iterate at both ends (second stream, beside
//          the devices), the deferred v update, over-relaxed blends;
//   node   step 3: pbar, theta_bar, u += pbar as register sums over the node's
//          terminals in CSR order (no atomics).  One kernel holds two passes:
//          the one without residuals, and, where they are read (stopping test,
//          adaptation, end of a call), one that also forms their partial sums
//          (one-pass Welford sums).  The CTA that ends last reduces them in
//          FP64 in a fixed order, decides the stopping test and the adaptive
//          penalty (Section 3.5) and advances the counter.
// Small instances without inner-ADMM devices run the three phases on one CTA,
// many iterations per launch (small_kernel).
//
// Splitting the phases lets each kernel run at its own register budget.
// There is no spin-wait on the device: ordering comes from kernel boundaries
// and graph edges.  Every kernel body also serves a batch of independent
// instances: the batch entry points take the instances' parameters and a
// CTA schedule, so one launch per phase covers all instances (devices that
// solve in shared memory have one of their own), and the node phase's CTAs are
// dealt out on the device over the instances that still run.
//
// Memory layout (line- and node-major), numbering and the deferred v
// update: opf_internal.h.
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "opf_internal.h"
#include "opf_tri.h"

namespace opfk {

constexpr int WARPS = BLOCK / 32;
constexpr int ST_NONFINITE = 5;  // opf_status value set on the device
constexpr int NODE_VW = 4;       // time steps per node item
constexpr int NODE_CTAS = 4;     // resident CTAs per SM the node kernel is compiled for (64 registers)
// A node pass of few items is latency alone, and a variant with the registers
// to request all loads of an item together (two CTAs per SM) is faster.  Items
// of four steps: while that variant's CTAs are one wave, half of the node
// grid's threads (us per iteration, 30 buses 9.0 -> 8.6, 900 buses T = 24, 76k
// items, 16.9 -> 16.4; with a second wave, 500 buses T = 168, 105k, 35.1 ->
// 36.5).  Items of one step, whose loads are shorter: measured, up to this many
// (301 buses T = 31 14.4 -> 13.8, 5k buses T = 1, 105k, 15.5 -> 14.9).
constexpr long long NODE_LAT_ITEMS1 = 1 << 17;
constexpr int NODE_RX_CTAS = 3;  // ... its over-relaxed variant (80 registers)
constexpr int NODE_RES_NB = 1;   // line terminals gathered together where residuals are formed ...
constexpr int NODE_LEAN_NB = 2;  // ... and where they are not
constexpr int LINE_IPT = 4;      // line items per thread (CTA-sized blocks of items; all of a batch's instances)
constexpr long long LINE_SHORT = 1 << 20;   // ... one, up to this many items
constexpr int DEVB = 128;        // threads per CTA of the device kernel (its inner-ADMM warps spread over more SMs)
constexpr int DEV_WARPS = DEVB / 32;
constexpr int CLOSED_LANES4 = 2, CLOSED_LANES1 = 8;   // lanes per closed-form item: the classes of ksum2 / ksum8
// microseconds of a small instance's iteration on one CTA: base, per round of
// items, and the limit (opfk_plan)
constexpr double SMALL_BASE = 2.7, SMALL_LINE = 0.8, SMALL_CLOSED = 0.45, SMALL_NODE = 1.2, SMALL_LIMIT = 8.0;
// Without inner-ADMM devices: the line pass (microseconds, estimated) from
// which averages and device sums as kernels of their own are hidden beside it
// (opfk_plan).
constexpr double HIDE_US = 16.0;
constexpr int REG_C = 8;           // largest chunk of the register-resident inner ADMM ...
constexpr int REG_T = 32 * REG_C - 1;   // ... its longest horizon (T + 1 <= 32 C)
constexpr int BATCH_C = 4;         // the same in batches, whose kernels hold every chunk up to theirs
constexpr int BATCH_REG_T = 32 * BATCH_C - 1;

// shared floats per warp of the shared-memory inner ADMM: 3 (T+1) for the
// work arrays and one device's (lam, beta)
__host__ __device__ inline int warp_smem_floats(int T) { return (T + 1) * (3 + 2 * SG_N); }
// warps of a CTA with `bytes` of shared memory that can each hold a device
__host__ __device__ inline int smem_warps(int T, size_t bytes) {
  int nw = DEV_WARPS;
  while (nw > 1 && nw * (size_t)warp_smem_floats(T) * sizeof(float) > bytes) nw /= 2;
  return nw;
}

// warps' worth of work of the inner kernels: a device each, a link one per 32 steps
__host__ __device__ inline int inner_units(const Params &p) { return p.n_stor + p.n_ramp + p.n_hvdc * ((p.T + 31) >> 5); }

// register chunk of the inner ADMM at horizon T: a battery's T + 1 elements
// over 32 lanes (1 .. REG_C); 0 beyond longest (the shared-memory path)
__host__ __device__ inline int inner_chunk(int T, int longest = REG_T) { return T <= longest ? (T + 32) >> 5 : 0; }

// ---------------------------------------------------------------------------
// The inner ADMM (Appendix D) writes every product, sum and quotient with its
// rounding (__fmul_rn, __fadd_rn, __fmaf_rn, ...), which the compiler may not
// contract or reorder: its shared-memory and register forms, and each kernel
// that inlines them (one instance, a batch), compute the same bits.
// ---------------------------------------------------------------------------
// one projected dual step of an inequality row (Appendix D): lam += al - nb,
// beta = nb = min(al + lam, 0)
__device__ __forceinline__ void ineq_step(float al, float &lam, float &bet) {
  const float nb = fminf(radd(al, lam), 0.f);
  lam = radd(lam, rsub(al, nb));
  bet = nb;
}

// ---------------------------------------------------------------------------
// tridiagonal systems with constant off-diagonal `off` and diagonal d_end at
// both ends, d_mid inside (every x-update of Appendix D reduces to one).
// Factor: pivots q_i = d_i - off^2 / q_{i-1} (Thomas); the solve divides by
// the pivots (correctly rounded) rather than multiplying by rounded
// reciprocals, which would bias every solve of a device the same way.
// ---------------------------------------------------------------------------
__device__ void tri_factor(float *q, int n, float d_end, float d_mid, float off) {
  float prev = 0.f;
  for (int i = 0; i < n; ++i) {
    const float d = (i == 0 || i == n - 1) ? d_end : d_mid;
    const float qi = (i == 0) ? d : rsub(d, rmul(off, rdiv(off, prev)));
    q[i] = qi;
    prev = qi;
  }
}

// What the solves read of a factored system, [3][n]: the pivots q, then (by
// the whole warp) their reciprocals and a_i = -off / q_i.
__device__ __forceinline__ void tri_tables(float *m, int n, float off, int lane) {
  __syncwarp();
  for (int i = lane; i < n; i += 32) {
    const float q = m[i], rq = __frcp_rn(q);
    m[n + i] = rq;
    m[2 * n + i] = qdiv(-off, q, rq);
  }
  __syncwarp();
}

// Solve in place (buf: right-hand side in, solution out; shared memory), with
// m the tables above.  Forward  y_i = a_i y_{i-1} + r_i / q_i  and backward
// x_i = a_i x_{i+1} + y_i are first-order linear recurrences; each lane
// composes the affine maps of a contiguous chunk, a 5-step shuffle scan
// composes the chunks across the warp, then each lane applies the prefix to
// its chunk.  The chunks are serial chains (32 elements at T = 1000), so what
// they read comes from the tables, without a division on the way: 30 buses,
// T = 1000, 1060 -> 1005 us per iteration.
__device__ void warp_tri_solve(const float *__restrict__ m, float *buf, int n, int lane) {
  const float *q = m, *rq = m + n, *a = m + 2 * n;
  const int cs = (n + 31) >> 5;
  const int i0 = min(lane * cs, n), i1 = min(i0 + cs, n);
  // forward (r_i = buf_i / q_i is kept in buf for the second pass)
  float Ac = 1.f, Bc = 0.f;
#pragma unroll 4
  for (int i = i0; i < i1; ++i) {
    const float ri = qdiv(buf[i], q[i], rq[i]);
    const float Ai = (i == 0) ? 0.f : a[i];
    buf[i] = ri;
    Bc = rfma(Ai, Bc, ri);
    Ac = rmul(Ai, Ac);
  }
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const float Ap = __shfl_up_sync(FULL, Ac, d);
    const float Bp = __shfl_up_sync(FULL, Bc, d);
    if (lane >= d) {
      Bc = rfma(Ac, Bp, Bc);
      Ac = rmul(Ac, Ap);
    }
  }
  float prev = __shfl_up_sync(FULL, Bc, 1);
  if (lane == 0) prev = 0.f;
#pragma unroll 4
  for (int i = i0; i < i1; ++i) {
    prev = rfma((i == 0) ? 0.f : a[i], prev, buf[i]);
    buf[i] = prev;
  }
  __syncwarp();
  // backward
  Ac = 1.f;
  Bc = 0.f;
#pragma unroll 4
  for (int i = i1 - 1; i >= i0; --i) {
    const float Ci = (i == n - 1) ? 0.f : a[i];
    Bc = rfma(Ci, Bc, buf[i]);
    Ac = rmul(Ci, Ac);
  }
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const float Ap = __shfl_down_sync(FULL, Ac, d);
    const float Bp = __shfl_down_sync(FULL, Bc, d);
    if (lane + d < 32) {
      Bc = rfma(Ac, Bp, Bc);
      Ac = rmul(Ac, Ap);
    }
  }
  float nxt = __shfl_down_sync(FULL, Bc, 1);
  if (lane == 31) nxt = 0.f;
#pragma unroll 4
  for (int i = i1 - 1; i >= i0; --i) {
    nxt = rfma((i == n - 1) ? 0.f : a[i], nxt, buf[i]);
    buf[i] = nxt;
  }
  __syncwarp();
}

// ---------------------------------------------------------------------------
// VW consecutive time steps per thread (4 -> 128-bit accesses when T % 4 == 0)
// ---------------------------------------------------------------------------
template <int VW>
struct FV {
  float v[VW];
};

template <int VW>
__device__ __forceinline__ FV<VW> ldv(const float *p) {
  FV<VW> r;
  if constexpr (VW == 4) {
    const float4 t = *reinterpret_cast<const float4 *>(p);
    r.v[0] = t.x; r.v[1] = t.y; r.v[2] = t.z; r.v[3] = t.w;
  } else if constexpr (VW == 2) {
    const float2 t = *reinterpret_cast<const float2 *>(p);
    r.v[0] = t.x; r.v[1] = t.y;
  } else {
    r.v[0] = *p;
  }
  return r;
}

// streaming load (read once per iteration: evict first)
template <int VW>
__device__ __forceinline__ FV<VW> ldv_cs(const float *p) {
  FV<VW> r;
  if constexpr (VW == 4) {
    const float4 t = __ldcs(reinterpret_cast<const float4 *>(p));
    r.v[0] = t.x; r.v[1] = t.y; r.v[2] = t.z; r.v[3] = t.w;
  } else if constexpr (VW == 2) {
    const float2 t = __ldcs(reinterpret_cast<const float2 *>(p));
    r.v[0] = t.x; r.v[1] = t.y;
  } else {
    r.v[0] = __ldcs(p);
  }
  return r;
}

template <int VW>
__device__ __forceinline__ void stv(float *p, const FV<VW> &r) {
  if constexpr (VW == 4) {
    *reinterpret_cast<float4 *>(p) = make_float4(r.v[0], r.v[1], r.v[2], r.v[3]);
  } else if constexpr (VW == 2) {
    *reinterpret_cast<float2 *>(p) = make_float2(r.v[0], r.v[1]);
  } else {
    *p = r.v[0];
  }
}

// streaming store (not read again in this iteration: evict first)
template <int VW>
__device__ __forceinline__ void stv_cs(float *p, const FV<VW> &r) {
  if constexpr (VW == 4) {
    __stcs(reinterpret_cast<float4 *>(p), make_float4(r.v[0], r.v[1], r.v[2], r.v[3]));
  } else if constexpr (VW == 2) {
    __stcs(reinterpret_cast<float2 *>(p), make_float2(r.v[0], r.v[1]));
  } else {
    __stcs(p, r.v[0]);
  }
}

// x / c given r = 1/c rounded to nearest: one FMA correction step gives the
// correctly rounded quotient for these well-scaled operands (a plain x * r
// would carry the rounding bias of r into every node average, iteration
// after iteration).
__device__ __forceinline__ float div_rn(float x, float c, float r) {
  const float q = x * r;
  return fmaf(fmaf(-q, c, x), r, q);
}

__device__ __forceinline__ void prefetch_l1(const void *a) { asm volatile("prefetch.global.L1 [%0];" ::"l"(a)); }

// the current iteration's scalars (the same two loads in every thread)
__device__ __forceinline__ Iter load_iter(const Params &p) {
  union {
    Iter r;
    int4 v[2];
  } x;
  static_assert(sizeof(Iter) == 32, "Iter is loaded as two int4");
  const int4 *s = reinterpret_cast<const int4 *>(&p.sc->cur);
  x.v[0] = s[0];
  x.v[1] = s[1];
  return x.r;
}

// Sums over contingencies k of a node array (o: its offset of k = 0; rows T
// floats apart).  The order of each sum is fixed, so that every form of the
// device averages (one thread here, a group of lanes in closed_body) agrees
// bit for bit: ksum2 adds two partial sums, over even and odd k; ksum8 eight,
// over k mod 8 while whole groups of eight last, the rest going to the first.
template <int VW>
__device__ __forceinline__ FV<VW> ksum2(const float *a, size_t o, int T, int Kp) {
  FV<VW> c[2];
#pragma unroll
  for (int e = 0; e < VW; ++e) c[0].v[e] = c[1].v[e] = 0.f;
  const float *r = a + o;
  int k = 0;
  constexpr int U = VW == 1 ? 8 : VW == 2 ? 4 : 2;   // 16 values in flight
#pragma unroll U
  for (; k + 2 <= Kp; k += 2, r += 2 * (size_t)T) {
    const FV<VW> x = ldv<VW>(r), y = ldv<VW>(r + T);
#pragma unroll
    for (int e = 0; e < VW; ++e) {
      c[0].v[e] += x.v[e];
      c[1].v[e] += y.v[e];
    }
  }
  FV<VW> s;
#pragma unroll
  for (int e = 0; e < VW; ++e) s.v[e] = 0.f;
  if (k < Kp) s = ldv<VW>(r);
#pragma unroll
  for (int e = 0; e < VW; ++e) s.v[e] = (c[0].v[e] + s.v[e]) + c[1].v[e];
  return s;
}

__device__ __forceinline__ float ksum8(const float *a, size_t o, int T, int Kp) {
  float c[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) c[j] = 0.f;
  const float *r = a + o;
  int k = 0;
#pragma unroll 1
  for (; k + 8 <= Kp; k += 8, r += 8 * (size_t)T) {
#pragma unroll
    for (int j = 0; j < 8; ++j) c[j] += r[j * (size_t)T];
  }
  float x[7];   // the rest together in flight
#pragma unroll
  for (int j = 0; j < 7; ++j) x[j] = k + j < Kp ? r[j * (size_t)T] : 0.f;
#pragma unroll
  for (int j = 0; j < 7; ++j)
    if (k + j < Kp) c[0] += x[j];
  return ((c[0] + c[1]) + (c[2] + c[3])) + ((c[4] + c[5]) + (c[6] + c[7]));
}

// avg_k(pbar + s u) = (sum_k PU + (s - 1) sum_k u) / (K+1) from the two sums
// (Section 3.2 step 2)
__device__ __forceinline__ float avg_of(const Params &p, float sm1, float sp, float sq) {
  const float kpf = (float)p.Kp_glob;
  return div_rn(fmaf(sm1, sq, sp), kpf, __frcp_rn(kpf));
}

// the average at node n, steps t0 .. t0 + VW - 1; u is read only while a
// penalty rescale s != 1 is pending.  Horizons of whole 4-step blocks sum in
// the order of ksum2, others (one step at a time) in that of ksum8.
template <int VW>
__device__ __forceinline__ FV<VW> node_avg(const Params &p, const Iter &q, int n, int t0) {
  const size_t o = (size_t)n * p.Kp * p.T + t0;   // a node's K+1 rows are contiguous
  const float sm1 = q.fsu - 1.f;
  FV<VW> sp, sq;
#pragma unroll
  for (int e = 0; e < VW; ++e) sq.v[e] = 0.f;
  if (VW > 1 || p.T % 4 == 0) {
    sp = ksum2<VW>(p.PU[q.old], o, p.T, p.Kp);
    if (sm1 != 0.f) sq = ksum2<VW>(p.U[q.old], o, p.T, p.Kp);
  } else {
    sp.v[0] = ksum8(p.PU[q.old], o, p.T, p.Kp);
    if (sm1 != 0.f) sq.v[0] = ksum8(p.U[q.old], o, p.T, p.Kp);
  }
#pragma unroll
  for (int e = 0; e < VW; ++e) sp.v[e] = avg_of(p, sm1, sp.v[e], sq.v[e]);
  return sp;
}

// Over-relaxation (Section 3.6) in the form kept on the device: the stored
// schedules are the relaxed P = alpha p + (1 - alpha) P_prev, whose node
// averages are the copies' complements (z = P - avg_n P, xi = avg_n Theta);
// alpha = 1 returns p exactly.
__device__ __forceinline__ float relaxed(float alpha, float pnew, float pold) {
  return rfma(alpha, pnew, rmul(rsub(1.f, alpha), pold));
}

// X[t] = p_d[t] - avg_k(pbar + u) at the device's node n, t in [0, T), by one
// warp (Section 3.2 step 2 input).  avg: the warp forms the average itself;
// else xs_kernel left it in XS.
__device__ __forceinline__ void device_x(const Params &p, const Iter &q, int n, const float *pd, float *X, int lane,
                                         bool avg) {
  const int T = p.T;
  const float *xs = p.XS + (size_t)n * T;
  for (int t = lane; t < T; t += 32) X[t] = rsub(pd[t], avg ? node_avg<1>(p, q, n, t).v[0] : __ldcg(xs + t));
  __syncwarp();
}

// the averages of a lane's C consecutive steps from t0 (0 beyond T)
template <int C>
__device__ __forceinline__ void lane_avg(const Params &p, const Iter &q, int n, int t0, float (&xs)[C], bool avg) {
  const int T = p.T;
  if constexpr (C == 2 || C == 4) {
    if (avg && T % 4 == 0) {   // the lane's rows as one 64- or 128-bit load
      if (t0 < T) {
        const FV<C> a = node_avg<C>(p, q, n, t0);
#pragma unroll
        for (int j = 0; j < C; ++j) xs[j] = a.v[j];
      }
      return;
    }
  }
#pragma unroll
  for (int j = 0; j < C; ++j) {
    xs[j] = 0.f;
    if (t0 + j < T) xs[j] = avg ? node_avg<1>(p, q, n, t0 + j).v[0] : __ldcg(p.XS + (size_t)n * T + t0 + j);
  }
}

// The warp's inner-ADMM state (lam, beta) lives in shared memory during the
// inner iterations when it fits (lam_sh != nullptr), else in global memory.
__device__ __forceinline__ void stage_in(float *&lam, float *&bet, float *lam_sh, int n, int lane) {
  if (!lam_sh) return;
  float *bsh = lam_sh + n;
  int i = lane;
  for (; i + 7 * 32 < n; i += 8 * 32) {   // 16 values in flight
    float x[8], y[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      x[q] = lam[i + 32 * q];
      y[q] = bet[i + 32 * q];
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      lam_sh[i + 32 * q] = x[q];
      bsh[i + 32 * q] = y[q];
    }
  }
  for (; i < n; i += 32) {
    lam_sh[i] = lam[i];
    bsh[i] = bet[i];
  }
  __syncwarp();
  lam = lam_sh;
  bet = bsh;
}

__device__ __forceinline__ void stage_out(float *lam_g, float *bet_g, const float *lam_sh, int n, int lane) {
  if (!lam_sh) return;
  __syncwarp();
  for (int i = lane; i < n; i += 32) {
    lam_g[i] = lam_sh[i];
    bet_g[i] = lam_sh[n + i];
  }
}

// ---------------------------------------------------------------------------
// Appendix D inner ADMM, ramp-limited generator (one warp, lanes over t).
// Rows: p_t <= pmax_t, -p_t <= -pmin_t, p_{t+1} - p_t <= R, p_t - p_{t+1} <= R.
// x-update matrix (2a + rho + 2 omega) I + 2 omega D'D is tridiagonal.
// ---------------------------------------------------------------------------
__device__ void ramp_prox(const Params &p, int r, float *sm, float *state_sh, int lane, bool avg) {
  const Iter q = load_iter(p);
  if (q.flags & ITF_SKIP) return;
  const int T = p.T;
  const float rho = q.rho_dev;
  const int d = p.ramp_ids[r];
  const int n = p.dev_node[d];
  const float a = p.dev_a[d], b = p.dev_b[d], R = p.ramp_R[r];
  const float om = rho, om2 = rmul(2.f, om);
  float *const lam_g = p.ramp_lam + (size_t)r * RG_N * T;
  float *const bet_g = p.ramp_beta + (size_t)r * RG_N * T;
  float *lam = lam_g, *bet = bet_g;
  stage_in(lam, bet, state_sh, RG_N * T, lane);
  float *mf = p.ramp_q + (size_t)r * 3 * T;
  const float *lo = p.dev_lo + (size_t)d * T;
  const float *hi = p.dev_hi + (size_t)d * T;
  float *pd = p.PD + (size_t)d * T;
  float *X = sm, *W = sm + (T + 1), *Z = sm + 2 * (T + 1);

  // keep the unscaled inner duals omega * lam when omega changes; refactor
  // (2a + rho + 2 omega) I + 2 omega D'D
  const float rho_old = p.ramp_rho[r];
  if (rho_old != rho) {
    const float ls = (rho_old == 0.f) ? 1.f : rdiv(fabsf(rho_old), rho);
    for (int t = lane; t < RG_N * T; t += 32) lam[t] = rmul(lam[t], ls);
    if (lane == 0) {
      const float base = radd(rmul(2.f, a), rho);
      tri_factor(mf, T, radd(base, rmul(4.f, om)), radd(base, rmul(6.f, om)), -om2);
      p.ramp_rho[r] = rho;
    }
    tri_tables(mf, T, -om2, lane);
  } else if (mf[T] == 0.f) {   // no_tables
    tri_tables(mf, T, -om2, lane);
  }
  device_x(p, q, n, pd, X, lane, avg);   // p_d - avg_k(pbar + u)
  for (int itn = 0; itn < p.inner_iters; ++itn) {
    for (int t = lane; t < T - 1; t += 32)
      W[t] = rsub(rsub(bet[RG_RU * T + t], lam[RG_RU * T + t]), rsub(bet[RG_RD * T + t], lam[RG_RD * T + t]));
    __syncwarp();
    for (int t = lane; t < T; t += 32) {
      float atr = rsub(rsub(radd(hi[t], bet[RG_UP * T + t]), lam[RG_UP * T + t]),
                       rsub(radd(-lo[t], bet[RG_LO * T + t]), lam[RG_LO * T + t]));
      if (t >= 1) atr = radd(atr, W[t - 1]);
      if (t <= T - 2) atr = rsub(atr, W[t]);
      Z[t] = rfma(om, atr, rfma(rho, X[t], -b));
    }
    __syncwarp();
    warp_tri_solve(mf, Z, T, lane);
    for (int t = lane; t < T; t += 32) {
      const float pt = Z[t];
      ineq_step(rsub(pt, hi[t]), lam[RG_UP * T + t], bet[RG_UP * T + t]);
      ineq_step(rsub(lo[t], pt), lam[RG_LO * T + t], bet[RG_LO * T + t]);
      if (t < T - 1) {
        const float pn = Z[t + 1];
        ineq_step(rsub(rsub(pn, pt), R), lam[RG_RU * T + t], bet[RG_RU * T + t]);
        ineq_step(rsub(rsub(pt, pn), R), lam[RG_RD * T + t], bet[RG_RD * T + t]);
      }
    }
    __syncwarp();
  }
  stage_out(lam_g, bet_g, state_sh, RG_N * T, lane);
  for (int t = lane; t < T; t += 32) {
    const float pn = relaxed(p.alpha, Z[t], pd[t]);
    p.DPD[(size_t)d * T + t] = rsub(pn, pd[t]);
    pd[t] = pn;
  }
  __syncwarp();
}

// ---------------------------------------------------------------------------
// HVDC link (a warp per link and 32 time steps, lanes over t: each step's
// averages are a chain of loads, and one warp walking a long horizon was the
// whole phase: 100 buses, K = 4, us per iteration, T = 1000 51.7 -> 15.7,
// T = 2048 118 -> 24.7, T = 300 28.3 -> 14.5, T = 168 18.5 -> 12.6): with x_i = p_i - avg_k(pbar + u) at
// terminal i, p2 = clip((x2 - x1) / 2, -u, u) and p1 = -p2 (the minimiser
// of the two squared distances over p1 + p2 = 0, clipped to the limit)
// ---------------------------------------------------------------------------
__device__ void hvdc_prox(const Params &p, int unit, int lane, bool avg) {
  const Iter q = load_iter(p);
  if (q.flags & ITF_SKIP) return;
  const int T = p.T, nt = (T + 31) >> 5, h = unit / nt, t = (unit - h * nt) * 32 + lane;
  const int d1 = p.hvdc0 + 2 * h, d2 = d1 + 1;
  const float u = p.hvdc_u[h];
  const int m1 = p.dev_node[d1], m2 = p.dev_node[d2];
  const float *xs1 = p.XS + (size_t)m1 * T, *xs2 = p.XS + (size_t)m2 * T;
  float *pd1 = p.PD + (size_t)d1 * T, *pd2 = p.PD + (size_t)d2 * T;
  if (t < T) {
    const float q1 = pd1[t], q2 = pd2[t];
    const float x1 = q1 - (avg ? node_avg<1>(p, q, m1, t).v[0] : __ldcg(xs1 + t));
    const float x2 = q2 - (avg ? node_avg<1>(p, q, m2, t).v[0] : __ldcg(xs2 + t));
    const float f = fminf(fmaxf(0.5f * (x2 - x1), -u), u);
    const float r1 = relaxed(p.alpha, -f, q1), r2 = relaxed(p.alpha, f, q2);
    p.DPD[(size_t)d1 * T + t] = r1 - q1;
    p.DPD[(size_t)d2 * T + t] = r2 - q2;
    pd1[t] = r1;
    pd2[t] = r2;
  }
}

// ---------------------------------------------------------------------------
// Appendix D inner ADMM, battery (one warp, lanes over t).  Variables
// (p, c, delta, s), rows as in opf.h.  The x-update eliminates p_t, then
// (c_t, delta_t) per step (a 2x2 Schur complement), leaving a tridiagonal
// system of size T + 1 in the state of charge s.
// ---------------------------------------------------------------------------
__device__ void stor_prox(const Params &p, int sidx, float *sm, float *state_sh, int lane, bool avg) {
  const Iter it = load_iter(p);
  if (it.flags & ITF_SKIP) return;
  const int T = p.T, Tp = T + 1;
  const float rho = it.rho_dev;
  const int d = p.stor_ids[sidx];
  const int n = p.dev_node[d];
  const float eta = p.stor_eff[sidx], Pm = p.stor_P[sidx], Em = rmul(p.stor_dur[sidx], Pm);
  const float q = p.stor_cost[sidx];
  const float om = rho, om2 = rmul(2.f, om);
  float *const lam_g = p.stor_lam + (size_t)sidx * SG_N * Tp;
  float *const bet_g = p.stor_beta + (size_t)sidx * SG_N * Tp;
  float *lam = lam_g, *bet = bet_g;
  stage_in(lam, bet, state_sh, SG_N * Tp, lane);
  float *mf = p.stor_q + (size_t)sidx * 3 * Tp;
  float *pd = p.PD + (size_t)d * T;
  float *dl_out = p.stor_delta + (size_t)sidx * T;
  float *X = sm, *TAU = sm + Tp, *S = sm + 2 * Tp;

  // 2x2 block of (c, delta) after eliminating p; constants of the reduction
  const float kap = rdiv(rmul(rho, om), radd(rho, om));
  const float h00 = radd(radd(kap, om2), rmul(rmul(om, eta), eta));
  const float h01 = rsub(-kap, rmul(om, eta)), h11 = radd(kap, rmul(3.f, om));
  const float det = rsub(rmul(h00, h11), rmul(h01, h01));
  const float i00 = rdiv(h11, det), i01 = rdiv(-h01, det), i11 = rdiv(h00, det);
  const float f1c = rmul(om, eta), f1d = -om;
  const float w0 = radd(rmul(i00, f1c), rmul(i01, f1d)), w1 = radd(rmul(i01, f1c), rmul(i11, f1d));
  const float gam = rsub(om, radd(rmul(f1c, w0), rmul(f1d, w1)));
  const float rpo = radd(rho, om), rrpo = __frcp_rn(rpo), rgam = __frcp_rn(gam);

  const float rho_old = p.stor_rho[sidx];
  if (rho_old != rho) {
    const float ls = (rho_old == 0.f) ? 1.f : rdiv(fabsf(rho_old), rho);
    for (int t = lane; t < SG_N * Tp; t += 32) lam[t] = rmul(lam[t], ls);
    if (lane == 0) {
      tri_factor(mf, Tp, radd(gam, rmul(3.f, om)), radd(rmul(2.f, gam), om2), -gam);
      p.stor_rho[sidx] = rho;
    }
    tri_tables(mf, Tp, -gam, lane);
  } else if (mf[Tp] == 0.f) {   // no_tables
    tri_tables(mf, Tp, -gam, lane);
  }
  device_x(p, it, n, pd, X, lane, avg);   // p_d - avg_k(pbar + u)
#define LAM(g, t) lam[(g) * Tp + (t)]
#define BET(g, t) bet[(g) * Tp + (t)]
  for (int itn = 0; itn < p.inner_iters; ++itn) {
    for (int t = lane; t < T; t += 32) {
      const float r1 = -LAM(SG_E1, t), r2 = -LAM(SG_E2, t);
      const float mc = rmul(0.5f, rsub(rsub(radd(Pm, BET(SG_CU, t)), LAM(SG_CU, t)), rsub(BET(SG_CL, t), LAM(SG_CL, t))));
      const float md = rmul(0.5f, rsub(rsub(radd(Pm, BET(SG_DU, t)), LAM(SG_DU, t)), rsub(BET(SG_DL, t), LAM(SG_DL, t))));
      const float e1 = rsub(r1, X[t]);
      const float f0c = rfma(kap, e1, rmul(om2, mc));
      const float f0d = rfma(om2, md, rsub(rmul(-kap, e1), q));
      TAU[t] = radd(r2, qdiv(rfma(w0, f0c, rmul(w1, f0d)), gam, rgam));
    }
    __syncwarp();
    for (int j = lane; j < Tp; j += 32) {
      const float ms = rmul(0.5f, rsub(rsub(radd(Em, BET(SG_SU, j)), LAM(SG_SU, j)), rsub(BET(SG_SL, j), LAM(SG_SL, j))));
      float rhs = rmul(om2, ms);
      if (j >= 1) rhs = rfma(gam, TAU[j - 1], rhs);
      if (j <= T - 1) rhs = rfma(-gam, TAU[j], rhs);
      if (j == 0) rhs = rfma(-om, LAM(SG_E3, 0), rhs);
      if (j == T) rhs = rfma(-om, LAM(SG_E3, 1), rhs);
      S[j] = rhs;
    }
    __syncwarp();
    warp_tri_solve(mf, S, Tp, lane);
    for (int t = lane; t < T; t += 32) {
      const float r1 = -LAM(SG_E1, t), r2 = -LAM(SG_E2, t);
      const float mc = rmul(0.5f, rsub(rsub(radd(Pm, BET(SG_CU, t)), LAM(SG_CU, t)), rsub(BET(SG_CL, t), LAM(SG_CL, t))));
      const float md = rmul(0.5f, rsub(rsub(radd(Pm, BET(SG_DU, t)), LAM(SG_DU, t)), rsub(BET(SG_DL, t), LAM(SG_DL, t))));
      const float e1 = rsub(r1, X[t]);
      const float f0c = rfma(kap, e1, rmul(om2, mc));
      const float f0d = rfma(om2, md, rsub(rmul(-kap, e1), q));
      const float s0 = S[t], s1 = S[t + 1];
      const float ds = rsub(s1, s0);
      const float g = rsub(ds, r2);
      const float fc = rfma(g, f1c, f0c), fd = rfma(g, f1d, f0d);
      const float c = rfma(i00, fc, rmul(i01, fd));
      const float dl = rfma(i01, fc, rmul(i11, fd));
      const float pt = qdiv(rfma(om, radd(rsub(r1, c), dl), rmul(rho, X[t])), rpo, rrpo);
      TAU[t] = pt;  // TAU is consumed; keep p_t for the end
      dl_out[t] = dl;
      LAM(SG_E1, t) = radd(LAM(SG_E1, t), rsub(radd(pt, c), dl));   // equality rows: beta = 0
      LAM(SG_E2, t) = radd(LAM(SG_E2, t), radd(rfma(-eta, c, ds), dl));
      ineq_step(rsub(c, Pm), LAM(SG_CU, t), BET(SG_CU, t));
      ineq_step(-c, LAM(SG_CL, t), BET(SG_CL, t));
      ineq_step(rsub(dl, Pm), LAM(SG_DU, t), BET(SG_DU, t));
      ineq_step(-dl, LAM(SG_DL, t), BET(SG_DL, t));
    }
    for (int j = lane; j < Tp; j += 32) {
      const float sj = S[j];
      if (j == 0) LAM(SG_E3, 0) = radd(LAM(SG_E3, 0), sj);
      if (j == T) LAM(SG_E3, 1) = radd(LAM(SG_E3, 1), sj);
      ineq_step(rsub(sj, Em), LAM(SG_SU, j), BET(SG_SU, j));
      ineq_step(-sj, LAM(SG_SL, j), BET(SG_SL, j));
    }
    __syncwarp();
  }
#undef LAM
#undef BET
  stage_out(lam_g, bet_g, state_sh, SG_N * Tp, lane);
  for (int t = lane; t < T; t += 32) {
    const float pn = relaxed(p.alpha, TAU[t], pd[t]);
    p.DPD[(size_t)d * T + t] = rsub(pn, pd[t]);
    pd[t] = pn;
  }
  __syncwarp();
}

// ---------------------------------------------------------------------------
// The same inner ADMM with the device's state in registers, for horizons of
// at most REG_T steps: lane l holds the C = ceil(n / 32) consecutive
// elements l C .. l C + C - 1 of each vector (the solve's chunks), so the
// inner iterations touch no memory; neighbours across a chunk boundary come
// by one shuffle.  Every product, sum and quotient is written with its
// rounding (__fmul_rn, __fadd_rn, __fmaf_rn, ...), which the compiler may
// not contract or reorder, so each kernel that inlines this path (one
// instance, a batch) computes the same bits.
// ---------------------------------------------------------------------------

// Pivots written without the tables that the shared-memory form reads beside
// them (a batch solves devices beyond BATCH_REG_T steps that way): the first
// reciprocal, never 0 otherwise, says so, and that form makes them when it
// comes to the device.  (Writing them here too cost a week of 500 buses 0.4 %.)
template <int C>
__device__ __forceinline__ void no_tables(float *mf, int n) {
  if (32 * C > BATCH_REG_T) mf[n] = 0.f;
}

// Lanes beyond the horizon run along (right-hand side 0, nothing of theirs is
// stored or read by others), which spares the inner iterations a branch per
// element.
// The state that does not depend on the iteration's scalars is requested
// first, with them; the contingency rows of the node and the box follow when
// the device's record arrives, so the ten inner iterations wait for two rounds
// of loads.
template <int C>
__device__ void ramp_prox_r(const Params &p, int r, int lane, bool avg) {
  const int T = p.T, t0 = lane * C;
  const int2 ids = p.irec[p.n_stor + r];           // device, node
  const float4 par = p.ipar[p.n_stor + r];         // a, b, ramp limit
  float *const lam_g = p.ramp_lam + (size_t)r * RG_N * T;
  float *const bet_g = p.ramp_beta + (size_t)r * RG_N * T;
  float *mf = p.ramp_q + (size_t)r * 3 * T;
  const float rho_old = p.ramp_rho[r];
  float lam[RG_N][C], bet[RG_N][C], hi[C], lo[C], X[C], pd[C], Z[C];
  TriFac<C> tf;
#pragma unroll
  for (int j = 0; j < C; ++j) {
    const int t = t0 + j;
    const bool in = t < T;
#pragma unroll
    for (int g = 0; g < RG_N; ++g) {
      lam[g][j] = in ? lam_g[g * T + t] : 0.f;
      bet[g][j] = in ? bet_g[g * T + t] : 0.f;
    }
    tf.q[j] = in ? mf[t] : 1.f;
    Z[j] = 0.f;
  }
  const Iter q = load_iter(p);
  if (q.flags & ITF_SKIP) return;
  const int d = ids.x, n = ids.y;
  const float a = par.x, b = par.y, R = par.z;
  const float rho = q.rho_dev, om = rho, om2 = rmul(2.f, om);
#pragma unroll
  for (int j = 0; j < C; ++j) {
    const int t = t0 + j;
    const bool in = t < T;
    hi[j] = in ? p.dev_hi[(size_t)d * T + t] : 0.f;
    lo[j] = in ? p.dev_lo[(size_t)d * T + t] : 0.f;
    pd[j] = in ? p.PD[(size_t)d * T + t] : 0.f;
  }
  lane_avg<C>(p, q, n, t0, X, avg);
  // keep the unscaled inner duals omega * lam when omega changes; refactor
  // (2a + rho + 2 omega) I + 2 omega D'D
  if (rho_old != rho) {
    const float ls = (rho_old == 0.f) ? 1.f : rdiv(fabsf(rho_old), rho);
    if (lane == 0) {
      const float base = radd(rmul(2.f, a), rho);
      tri_factor(mf, T, radd(base, rmul(4.f, om)), radd(base, rmul(6.f, om)), -om2);
      no_tables<C>(mf, T);
      p.ramp_rho[r] = rho;
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < C; ++j) {
#pragma unroll
      for (int g = 0; g < RG_N; ++g) lam[g][j] = rmul(lam[g][j], ls);
      tf.q[j] = t0 + j < T ? mf[t0 + j] : 1.f;
    }
  }
#pragma unroll
  for (int j = 0; j < C; ++j) X[j] = t0 + j < T ? rsub(pd[j], X[j]) : 0.f;   // p_d - avg_k(pbar + u)
  tf.init(om2, T, lane);   // off = -2 omega
  for (int itn = 0; itn < p.inner_iters; ++itn) {
    float W[C];
#pragma unroll
    for (int j = 0; j < C; ++j)
      W[j] = rsub(rsub(bet[RG_RU][j], lam[RG_RU][j]), rsub(bet[RG_RD][j], lam[RG_RD][j]));
    const float wprev = __shfl_up_sync(FULL, W[C - 1], 1);
#pragma unroll
    for (int j = 0; j < C; ++j) {
      const int t = t0 + j;
      float atr = rsub(rsub(radd(hi[j], bet[RG_UP][j]), lam[RG_UP][j]),
                       rsub(radd(-lo[j], bet[RG_LO][j]), lam[RG_LO][j]));
      if (t >= 1) atr = radd(atr, (j == 0) ? wprev : W[j - 1]);
      if (t <= T - 2) atr = rsub(atr, W[j]);
      Z[j] = t < T ? rfma(om, atr, rfma(rho, X[j], -b)) : 0.f;
    }
    warp_tri_solve_r<C>(tf, Z, T, lane);
    const float znext = __shfl_down_sync(FULL, Z[0], 1);
#pragma unroll
    for (int j = 0; j < C; ++j) {
      const float pt = Z[j];
      ineq_step(rsub(pt, hi[j]), lam[RG_UP][j], bet[RG_UP][j]);
      ineq_step(rsub(lo[j], pt), lam[RG_LO][j], bet[RG_LO][j]);
      if (t0 + j < T - 1) {
        const float pn = (j == C - 1) ? znext : Z[j + 1];
        ineq_step(rsub(rsub(pn, pt), R), lam[RG_RU][j], bet[RG_RU][j]);
        ineq_step(rsub(rsub(pt, pn), R), lam[RG_RD][j], bet[RG_RD][j]);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < C; ++j) {
    const int t = t0 + j;
    if (t < T) {
#pragma unroll
      for (int g = 0; g < RG_N; ++g) {
        lam_g[g * T + t] = lam[g][j];
        bet_g[g * T + t] = bet[g][j];
      }
      const float pn = relaxed(p.alpha, Z[j], pd[j]);
      p.DPD[(size_t)d * T + t] = rsub(pn, pd[j]);
      p.PD[(size_t)d * T + t] = pn;
    }
  }
}

template <int C>
__device__ void stor_prox_r(const Params &p, int sidx, int lane, bool avg) {
  const int T = p.T, Tp = T + 1, t0 = lane * C;
  const int2 ids = p.irec[sidx];                   // device, node
  const float4 par = p.ipar[sidx];                 // efficiency, power, duration, cost
  float *const lam_g = p.stor_lam + (size_t)sidx * SG_N * Tp;
  float *const bet_g = p.stor_beta + (size_t)sidx * SG_N * Tp;
  float *mf = p.stor_q + (size_t)sidx * 3 * Tp;
  const float rho_old = p.stor_rho[sidx];
  // element e = t0 + j: step t = e of (p, c, delta) while e < T, state of
  // charge s_e while e < T + 1
  float lE1[C], lE2[C], lCU[C], lCL[C], lDU[C], lDL[C], lSU[C], lSL[C];
  float bCU[C], bCL[C], bDU[C], bDL[C], bSU[C], bSL[C];
  float X[C], pd[C], S[C], TAU[C], DL[C];
  TriFac<C> tf;
  float e3a = lam_g[SG_E3 * Tp], e3b = lam_g[SG_E3 * Tp + 1];   // s_0 and s_T rows
#define LD_L(arr, g) arr[j] = in ? lam_g[(g) * Tp + e] : 0.f
#define LD_B(arr, g) arr[j] = in ? bet_g[(g) * Tp + e] : 0.f
#pragma unroll
  for (int j = 0; j < C; ++j) {
    const int e = t0 + j;
    const bool in = e < Tp;
    LD_L(lE1, SG_E1); LD_L(lE2, SG_E2); LD_L(lCU, SG_CU); LD_L(lCL, SG_CL);
    LD_L(lDU, SG_DU); LD_L(lDL, SG_DL); LD_L(lSU, SG_SU); LD_L(lSL, SG_SL);
    LD_B(bCU, SG_CU); LD_B(bCL, SG_CL); LD_B(bDU, SG_DU); LD_B(bDL, SG_DL);
    LD_B(bSU, SG_SU); LD_B(bSL, SG_SL);
    tf.q[j] = in ? mf[e] : 1.f;
    S[j] = TAU[j] = DL[j] = 0.f;
  }
#undef LD_L
#undef LD_B
  const Iter it = load_iter(p);
  if (it.flags & ITF_SKIP) return;
  const int d = ids.x, n = ids.y;
#pragma unroll
  for (int j = 0; j < C; ++j) pd[j] = t0 + j < T ? p.PD[(size_t)d * T + t0 + j] : 0.f;
  lane_avg<C>(p, it, n, t0, X, avg);
  const float rho = it.rho_dev;
  const float eta = par.x, Pm = par.y, Em = rmul(par.z, Pm);
  const float q = par.w;
  const float om = rho, om2 = rmul(2.f, om);

  // 2x2 block of (c, delta) after eliminating p; constants of the reduction
  const float kap = rdiv(rmul(rho, om), radd(rho, om));
  const float h00 = radd(radd(kap, om2), rmul(rmul(om, eta), eta));
  const float h01 = rsub(-kap, rmul(om, eta)), h11 = radd(kap, rmul(3.f, om));
  const float det = rsub(rmul(h00, h11), rmul(h01, h01));
  const float i00 = rdiv(h11, det), i01 = rdiv(-h01, det), i11 = rdiv(h00, det);
  const float f1c = rmul(om, eta), f1d = -om;
  const float w0 = radd(rmul(i00, f1c), rmul(i01, f1d)), w1 = radd(rmul(i01, f1c), rmul(i11, f1d));
  const float gam = rsub(om, radd(rmul(f1c, w0), rmul(f1d, w1)));
  const float rpo = radd(rho, om), rrpo = __frcp_rn(rpo), rgam = __frcp_rn(gam);

  if (rho_old != rho) {
    const float ls = (rho_old == 0.f) ? 1.f : rdiv(fabsf(rho_old), rho);
    if (lane == 0) {
      tri_factor(mf, Tp, radd(gam, rmul(3.f, om)), radd(rmul(2.f, gam), om2), -gam);
      no_tables<C>(mf, Tp);
      p.stor_rho[sidx] = rho;
    }
    __syncwarp();
    e3a = rmul(e3a, ls);
    e3b = rmul(e3b, ls);
#pragma unroll
    for (int j = 0; j < C; ++j) {
      lE1[j] = rmul(lE1[j], ls); lE2[j] = rmul(lE2[j], ls);
      lCU[j] = rmul(lCU[j], ls); lCL[j] = rmul(lCL[j], ls);
      lDU[j] = rmul(lDU[j], ls); lDL[j] = rmul(lDL[j], ls);
      lSU[j] = rmul(lSU[j], ls); lSL[j] = rmul(lSL[j], ls);
      tf.q[j] = t0 + j < Tp ? mf[t0 + j] : 1.f;
    }
  }
#pragma unroll
  for (int j = 0; j < C; ++j) X[j] = t0 + j < T ? rsub(pd[j], X[j]) : 0.f;   // p_d - avg_k(pbar + u)
  tf.init(gam, Tp, lane);   // off = -gam
  for (int itn = 0; itn < p.inner_iters; ++itn) {
    float f0c[C], f0d[C];
#pragma unroll
    for (int j = 0; j < C; ++j) {
      const float r1 = -lE1[j], r2 = -lE2[j];
      const float mc = rmul(0.5f, rsub(rsub(radd(Pm, bCU[j]), lCU[j]), rsub(bCL[j], lCL[j])));
      const float md = rmul(0.5f, rsub(rsub(radd(Pm, bDU[j]), lDU[j]), rsub(bDL[j], lDL[j])));
      const float e1 = rsub(r1, X[j]);
      f0c[j] = rfma(kap, e1, rmul(om2, mc));
      f0d[j] = rfma(om2, md, rsub(rmul(-kap, e1), q));
      TAU[j] = radd(r2, qdiv(rfma(w0, f0c[j], rmul(w1, f0d[j])), gam, rgam));
    }
    const float tprev = __shfl_up_sync(FULL, TAU[C - 1], 1);
#pragma unroll
    for (int j = 0; j < C; ++j) {
      const int e = t0 + j;
      const float ms = rmul(0.5f, rsub(rsub(radd(Em, bSU[j]), lSU[j]), rsub(bSL[j], lSL[j])));
      float rhs = rmul(om2, ms);
      if (e >= 1) rhs = rfma(gam, (j == 0) ? tprev : TAU[j - 1], rhs);
      if (e <= T - 1) rhs = rfma(-gam, TAU[j], rhs);
      if (e == 0) rhs = rfma(-om, e3a, rhs);
      if (e == T) rhs = rfma(-om, e3b, rhs);
      S[j] = e < Tp ? rhs : 0.f;
    }
    warp_tri_solve_r<C>(tf, S, Tp, lane);
    const float snext = __shfl_down_sync(FULL, S[0], 1);
#pragma unroll
    for (int j = 0; j < C; ++j) {
      const float r1 = -lE1[j], r2 = -lE2[j];
      const float s0 = S[j], s1 = (j == C - 1) ? snext : S[j + 1];
      const float ds = rsub(s1, s0);
      const float g = rsub(ds, r2);
      const float fc = rfma(g, f1c, f0c[j]), fd = rfma(g, f1d, f0d[j]);
      const float c = rfma(i00, fc, rmul(i01, fd));
      const float dl = rfma(i01, fc, rmul(i11, fd));
      const float pt = qdiv(rfma(om, radd(rsub(r1, c), dl), rmul(rho, X[j])), rpo, rrpo);
      TAU[j] = pt;   // TAU is consumed; keep p_t for the end
      DL[j] = dl;
      lE1[j] = radd(lE1[j], rsub(radd(pt, c), dl));   // equality rows: beta = 0
      lE2[j] = radd(lE2[j], radd(rfma(-eta, c, ds), dl));
      ineq_step(rsub(c, Pm), lCU[j], bCU[j]);
      ineq_step(-c, lCL[j], bCL[j]);
      ineq_step(rsub(dl, Pm), lDU[j], bDU[j]);
      ineq_step(-dl, lDL[j], bDL[j]);
    }
#pragma unroll
    for (int j = 0; j < C; ++j) {
      const int e = t0 + j;
      const float sj = S[j];
      if (e == 0) e3a = radd(e3a, sj);
      if (e == T) e3b = radd(e3b, sj);
      ineq_step(rsub(sj, Em), lSU[j], bSU[j]);
      ineq_step(-sj, lSL[j], bSL[j]);
    }
  }
#define ST_L(arr, g) lam_g[(g) * Tp + e] = arr[j]
#define ST_B(arr, g) bet_g[(g) * Tp + e] = arr[j]
#pragma unroll
  for (int j = 0; j < C; ++j) {
    const int e = t0 + j;
    if (e < T) {
      ST_L(lE1, SG_E1); ST_L(lE2, SG_E2); ST_L(lCU, SG_CU); ST_L(lCL, SG_CL);
      ST_L(lDU, SG_DU); ST_L(lDL, SG_DL);
      ST_B(bCU, SG_CU); ST_B(bCL, SG_CL); ST_B(bDU, SG_DU); ST_B(bDL, SG_DL);
      const float pn = relaxed(p.alpha, TAU[j], pd[j]);
      p.DPD[(size_t)d * T + e] = rsub(pn, pd[j]);
      p.PD[(size_t)d * T + e] = pn;
      p.stor_delta[(size_t)sidx * T + e] = DL[j];
    }
    if (e < Tp) {
      ST_L(lSU, SG_SU); ST_L(lSL, SG_SL);
      ST_B(bSU, SG_SU); ST_B(bSL, SG_SL);
      if (e == 0) lam_g[SG_E3 * Tp] = e3a;
      if (e == T) lam_g[SG_E3 * Tp + 1] = e3b;
    }
  }
#undef ST_L
#undef ST_B
}

// one-pass sum of squared deviations from the mean (Welford)
template <int VW>
struct Welf {
  float n;
  float mean[VW], m2[VW];
  __device__ __forceinline__ void reset() {
    n = 0.f;
#pragma unroll
    for (int e = 0; e < VW; ++e) { mean[e] = 0.f; m2[e] = 0.f; }
  }
  __device__ __forceinline__ void add(const float *x) {
    n += 1.f;
    const float r = __frcp_rn(n);
#pragma unroll
    for (int e = 0; e < VW; ++e) {
      const float d = x[e] - mean[e];
      mean[e] = fmaf(d, r, mean[e]);
      m2[e] = fmaf(d, x[e] - mean[e], m2[e]);
    }
  }
};

// the mean alone (the same bits as Welf's)
template <int VW>
struct WelfMean {
  float n;
  float mean[VW];
  __device__ __forceinline__ void reset() {
    n = 0.f;
#pragma unroll
    for (int e = 0; e < VW; ++e) mean[e] = 0.f;
  }
  __device__ __forceinline__ void add(const float *x) {
    n += 1.f;
    const float r = __frcp_rn(n);
#pragma unroll
    for (int e = 0; e < VW; ++e) mean[e] = fmaf(x[e] - mean[e], r, mean[e]);
  }
};

// one-pass sums of two series over a node's terminals (Welford with the
// co-moment): means, centred second moments and sum (x - mean_x)(y - mean_y)
template <int VW>
struct Welf2 {
  float n;
  float mx[VW], my[VW], m2x[VW], m2y[VW], cxy[VW];
  __device__ __forceinline__ void reset() {
    n = 0.f;
#pragma unroll
    for (int e = 0; e < VW; ++e) { mx[e] = my[e] = m2x[e] = m2y[e] = cxy[e] = 0.f; }
  }
  __device__ __forceinline__ void add(const float *x, const float *y) {
    n += 1.f;
    const float r = __frcp_rn(n);
#pragma unroll
    for (int e = 0; e < VW; ++e) {
      const float dx = x[e] - mx[e], dy = y[e] - my[e];
      mx[e] = fmaf(dx, r, mx[e]);
      my[e] = fmaf(dy, r, my[e]);
      m2x[e] = fmaf(dx, x[e] - mx[e], m2x[e]);
      m2y[e] = fmaf(dy, y[e] - my[e], m2y[e]);
      cxy[e] = fmaf(dx, y[e] - my[e], cxy[e]);
    }
  }
};

// Index (a, b, c) of a row-major [.][B][C] item space, advanced by a fixed
// stride with carries instead of 64-bit divisions per item.
struct Idx3 {
  int a, b, c;
  __device__ __forceinline__ void set(unsigned x, int B, int C) {
    c = (int)(x % (unsigned)C);
    const unsigned q = x / (unsigned)C;
    b = (int)(q % (unsigned)B);
    a = (int)(q / (unsigned)B);
  }
  __device__ __forceinline__ void step(const Idx3 &d, int B, int C) {
    c += d.c;
    if (c >= C) { c -= C; ++b; }
    b += d.b;
    if (b >= B) { b -= B; ++a; }
    a += d.a;
  }
};

// ---------------------------------------------------------------------------
// line prox item (Section 3.2 step 1, Section 2.1 f^ac, Section 4.2): one
// (contingency k, line l, VW time steps).  x = p~ - u and y = theta_bar - v at
// both terminals from the previous iterate; the deferred phase-dual update
// v += theta - theta_bar of the previous iteration is applied on the way.
// ---------------------------------------------------------------------------
template <int VW>
__device__ __forceinline__ void line_item(const Params &p, int old, int nw, int k, int l, int toff, float frp,
                                          float frt, float fsu, float fsv, bool v_fresh) {
  // offsets of the line and its end nodes' rows: lidx / nidx
  const int n1 = p.line_n1[l], n2 = p.line_n2[l];
  const bool act = p.out_line[k] != l;
  const size_t ol = lidx(p, k, l, toff);
  const size_t o1 = nidx(p, k, n1, toff), o2 = nidx(p, k, n2, toff);
  // p stays cached: the node sums read its old value again
  FV<VW> P = ldv<VW>(p.P[old] + ol), M = ldv_cs<VW>(p.MID[old] + ol);
  FV<VW> V1 = ldv_cs<VW>(p.V1[old] + ol), V2 = ldv_cs<VW>(p.V2[old] + ol);
  // pbar + s u at both ends from PU = pbar + u; u itself only while a
  // penalty rescale s != 1 is pending (an adaptation iteration)
  const FV<VW> B1 = ldv<VW>(p.PU[old] + o1), B2 = ldv<VW>(p.PU[old] + o2);
  FV<VW> U1, U2;
  const bool rescale = fsu != 1.f;
  if (rescale) {
    U1 = ldv<VW>(p.U[old] + o1);
    U2 = ldv<VW>(p.U[old] + o2);
  }
  const FV<VW> G1 = ldv<VW>(p.THBAR[old] + o1), G2 = ldv<VW>(p.THBAR[old] + o2);
  float tb = 1.f, den = 1.f, ulim = 0.f;
  if (act) {
    const float bb = p.line_b[l];
    ulim = p.line_u[l];
    tb = 2.f * bb;
    den = 2.f * frp + frt / (tb * bb);   // 2 rho_p + rho_theta / (2 b^2), Section 4.2 (reading of the garbled print)
  }
  const float rden = __frcp_rn(den), rtb = __frcp_rn(tb);
  const float al = p.alpha, oma = 1.f - p.alpha;
#pragma unroll
  for (int e = 0; e < VW; ++e) {
    // the previous prox's terminal values (stored as p and the mean angle;
    // relaxed values when alpha != 1, Section 3.6)
    const float po = act ? P.v[e] : 0.f;
    const float ho = act ? div_rn(P.v[e], tb, rtb) : P.v[e];
    const float a1 = M.v[e] + ho, a2 = M.v[e] - ho;
    const float w1 = rescale ? fmaf(fsu - 1.f, U1.v[e], B1.v[e]) : B1.v[e];   // pbar + s u
    const float w2 = rescale ? fmaf(fsu - 1.f, U2.v[e], B2.v[e]) : B2.v[e];
    const float x1 = -po - w1;                              // p~ - u at terminal 1 (z - u relaxed)
    const float x2 = po - w2;                               // p~ - u at terminal 2
    const float r1 = a1 - G1.v[e], r2 = a2 - G2.v[e];       // theta - theta_bar (Theta - xi relaxed)
    const float v1 = v_fresh ? fsv * V1.v[e] : fsv * (V1.v[e] + r1);
    const float v2 = v_fresh ? fsv * V2.v[e] : fsv * (V2.v[e] + r2);
    const float y1 = G1.v[e] - v1, y2 = G2.v[e] - v2;       // theta_bar - v
    const float mo = M.v[e], sto = P.v[e];
    M.v[e] = fmaf(al, 0.5f * (y1 + y2), oma * mo);
    if (act) {
      const float num = frp * (x2 - x1) + div_rn(frt * (y1 - y2), tb, rtb);
      P.v[e] = fminf(fmaxf(div_rn(num, den, rden), -ulim), ulim);   // theta_{1,2} = mid +- p / (2b)
    } else {
      P.v[e] = 0.5f * (y1 - y2);   // outaged line: p = 0, the terminals decouple, theta = y
    }
    P.v[e] = fmaf(al, P.v[e], oma * sto);
    // v' = v - (Theta - xi) is what the next pass completes:
    // v'_new = v + alpha theta~_new - (Theta_new - xi_new) = v - (1 - alpha) (Theta - xi)
    V1.v[e] = fmaf(-oma, r1, v1);
    V2.v[e] = fmaf(-oma, r2, v2);
  }
  // p and the mean angle are read back by the node sums; v is not
  stv<VW>(p.P[nw] + ol, P);
  stv<VW>(p.MID[nw] + ol, M);
  stv_cs<VW>(p.V1[nw] + ol, V1);
  stv_cs<VW>(p.V2[nw] + ol, V2);
}

// ---------------------------------------------------------------------------
// node item (Section 3.2 step 3, Eq. average-op, Section 3.3): one
// (contingency k, node n, VW time steps).  Sums the node's terminals in CSR
// order (no atomics), forms pbar, theta_bar, u += pbar, and the residual
// partial sums: ||pbar||^2, ||theta~||^2 and ||p~ - p~_prev||^2 by one-pass
// Welford sums over the terminals, ||theta_bar - theta_bar_prev||^2.  The
// terminal codes come four at a time so that a node's row loads issue
// together.
// ---------------------------------------------------------------------------
// RES false: the iteration's residuals are not read, so the node sums skip the
// inputs only they need (old p and theta_bar rows, the device Welford state)
// and their accumulation; the relaxed variant still needs the mean change of p
// (its u update), so it reads the old p rows and keeps that mean alone.
// NB: line terminals gathered together.  LAT (with ILD): the first two
// devices' powers are requested with the first line rows.
// ILD: the pass sums the node's device powers (and the Welford state of their
// changes) itself; else dsum_kernel has left them in DSP, DSM and DSQ.
template <int VW, bool RELAX, bool RES, int NB, bool ILD, bool LAT>
__device__ __forceinline__ void node_item(const Params &p, int old, int nw, int k, int n, int toff, float fsu,
                                          float *acc) {
  const int T = p.T;
  constexpr bool dp = RES || RELAX;   // the change of p is read
  // level 1: the node record, the node's old rows and its device sums
  const int4 r0 = p.nrec[3 * n], r1 = p.nrec[3 * n + 1], r2 = p.nrec[3 * n + 2];
  const float cp = __int_as_float(r0.x), ct = __int_as_float(r0.y);
  const float rcp = __int_as_float(r0.z), rct = __int_as_float(r0.w);
  const size_t on = nidx(p, k, n, toff), os = (size_t)n * T + toff;
  const FV<VW> uo = ldv_cs<VW>(p.U[old] + on);
  FV<VW> go;
  if constexpr (RES) go = ldv_cs<VW>(p.THBAR[old] + on);
  // device terminals first: the sum and the Welford state after them, the
  // same in every contingency, in the order of dcsr_idx
  FV<VW> sp, st;
  Welf<VW> wdp, wth;
  Welf2<VW> wrx;   // RELAX: (Theta_new, Theta_new - Theta_old) over the line terminals
  WelfMean<VW> wm; // RELAX without residuals: the mean change of p
  if constexpr (RELAX && RES) wrx.reset();
  if constexpr (!ILD) {
    sp = ldv<VW>(p.DSP + os);
    if constexpr (RELAX && !RES) {
      const FV<VW> m = ldv<VW>(p.DSM + os);
      wm.n = (float)r2.z;
#pragma unroll
      for (int e = 0; e < VW; ++e) wm.mean[e] = m.v[e];
    }
    if constexpr (RES) {
      const FV<VW> m = ldv<VW>(p.DSM + os), q = ldv<VW>(p.DSQ + os);
      wdp.n = (float)r2.z;
#pragma unroll
      for (int e = 0; e < VW; ++e) { wdp.mean[e] = m.v[e]; wdp.m2[e] = q.v[e]; }
    }
  }
  FV<VW> pd0, pd1, dd0, dd1;
  int4 dv = make_int4(0, 0, 0, 0);
  if constexpr (ILD) {
#pragma unroll
    for (int e = 0; e < VW; ++e) sp.v[e] = 0.f;
    if constexpr (RES) wdp.reset();
    if constexpr (RELAX && !RES) wm.reset();
    if constexpr (LAT) {
      dv = p.ndev4[n];
      if (r2.z > 0) {
        pd0 = ldv<VW>(p.PD + (size_t)dv.x * T + toff);
        if constexpr (dp) dd0 = ldv<VW>(p.DPD + (size_t)dv.x * T + toff);
      }
      if (r2.z > 1) {
        pd1 = ldv<VW>(p.PD + (size_t)dv.y * T + toff);
        if constexpr (dp) dd1 = ldv<VW>(p.DPD + (size_t)dv.y * T + toff);
      }
    } else {
      for (int j = r2.w; j < r2.w + r2.z; ++j) {
        const size_t od = (size_t)p.dcsr_idx[j] * T + toff;
        const FV<VW> pd = ldv<VW>(p.PD + od);
#pragma unroll
        for (int e = 0; e < VW; ++e) sp.v[e] += pd.v[e];
        if constexpr (RES) wdp.add(ldv<VW>(p.DPD + od).v);
        else if constexpr (RELAX) wm.add(ldv<VW>(p.DPD + od).v);
      }
    }
  }
  bool first = ILD && LAT;
  wth.reset();
#pragma unroll
  for (int e = 0; e < VW; ++e) st.v[e] = 0.f;
  // level 2: the rows of the line terminals, four at a time; a terminal's
  // angle is mid +- p / (2b) (mid +- the stored value on the outaged line)
  const size_t kb = (size_t)k * T + toff, lrow = (size_t)p.Kp * T;   // line l's row of k: l * lrow + kb
  const int lout = p.out_line[k];
  int4 c4 = r1;
  for (int j = r2.x - 4;;) {
#pragma unroll 1
    for (int half = 0; half < 4; half += NB) {
    // the next NB codes; the rest move up (an indexed array of the four would
    // live in local memory)
    const int code[4] = {c4.x, c4.y, c4.z, c4.w};
    c4 = NB == 1 ? make_int4(code[1], code[2], code[3], 0) : make_int4(code[2], code[3], 0, 0);
    static_assert(NB == 1 || NB == 2 || NB == 4, "codes taken together");
    FV<VW> pn[NB], po[NB], mq[NB], mo[RELAX && RES ? NB : 1];
    float bq[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      if (code[q] >= 0) {
        const int l = code[q] >> 1;
        const size_t ol = (size_t)l * lrow + kb;
        pn[q] = ldv<VW>(p.P[nw] + ol);
        if constexpr (dp) po[q] = ldv<VW>(p.P[old] + ol);   // kept in L2 for the line's other end
        mq[q] = ldv<VW>(p.MID[nw] + ol);
        if constexpr (RELAX && RES) mo[q] = ldv<VW>(p.MID[old] + ol);
        bq[q] = p.line_b[l];
      }
    }
    if (first) {   // the device terminals, with the line rows in flight
      first = false;
      for (int i = 0; i < r2.z; ++i) {
        const int d = i == 2 ? dv.z : i == 3 ? dv.w : i < 2 ? 0 : p.dcsr_idx[r2.w + i];
        const size_t od = (size_t)d * T + toff;
        const FV<VW> pd = i == 0 ? pd0 : i == 1 ? pd1 : ldv<VW>(p.PD + od);
#pragma unroll
        for (int e = 0; e < VW; ++e) sp.v[e] += pd.v[e];
        if constexpr (dp) {
          const FV<VW> dd = i == 0 ? dd0 : i == 1 ? dd1 : ldv<VW>(p.DPD + od);
          if constexpr (RES) wdp.add(dd.v);
          else wm.add(dd.v);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      if (code[q] >= 0) {
        const bool t2 = code[q] & 1, act = (code[q] >> 1) != lout;
        const float tb = 2.f * bq[q], rtb = __frcp_rn(tb);
        float dpo[VW], th[VW], dth[VW];
#pragma unroll
        for (int e = 0; e < VW; ++e) {
          const float pv = act ? pn[q].v[e] : 0.f, pov = (act && dp) ? po[q].v[e] : 0.f;
          const float h = act ? div_rn(pn[q].v[e], tb, rtb) : pn[q].v[e];
          th[e] = t2 ? mq[q].v[e] - h : mq[q].v[e] + h;
          sp.v[e] += t2 ? pv : -pv;
          st.v[e] += th[e];
          dpo[e] = t2 ? pv - pov : pov - pv;
          if constexpr (RELAX && RES) {
            const float ho = act ? div_rn(po[q].v[e], tb, rtb) : po[q].v[e];
            dth[e] = th[e] - (t2 ? mo[q].v[e] - ho : mo[q].v[e] + ho);
          }
        }
        if constexpr (RES) {
          wdp.add(dpo);
          if constexpr (RELAX) wrx.add(th, dth);
          else wth.add(th);
        } else if constexpr (RELAX) {
          wm.add(dpo);
        }
      }
    }
    }
    j += 4;
    if (j >= r2.y) break;
    c4 = *reinterpret_cast<const int4 *>(p.tcode + j);   // terminals beyond the first four
  }
  FV<VW> pb, tbar, un;
#pragma unroll
  for (int e = 0; e < VW; ++e) {
    pb.v[e] = div_rn(sp.v[e], cp, rcp);                      // Eq. (average-op)
    tbar.v[e] = ct > 0.f ? div_rn(st.v[e], ct, rct) : 0.f;
    if constexpr (!RES) {
      if constexpr (RELAX) {
        const float a = p.alpha;
        un.v[e] = fsu * uo.v[e] + fmaf(a, pb.v[e], (1.f - a) * wm.mean[e]);
      } else {
        un.v[e] = fsu * uo.v[e] + pb.v[e];                   // u += pbar
      }
      continue;
    }
    const float dt = tbar.v[e] - go.v[e];
    if constexpr (RELAX) {
      // stored values are relaxed: pb = Q = avg_n P, tbar = xi.  The actual
      // iterate is P + c dP with c = (1 - alpha) / alpha, so
      //   u += alpha pbar_actual = alpha Q + (1 - alpha) dQ,
      //   ||p - z||^2 = c^2 sum (dP - dQ)^2 + |n| (Q + c dQ)^2,
      //   ||theta - xi||^2 = sum (Theta - xi + c dTheta)^2 by the co-moment
      const float a = p.alpha, c = (1.f - a) / a, dq = wdp.mean[e];
      un.v[e] = fsu * uo.v[e] + fmaf(a, pb.v[e], (1.f - a) * dq);
      const float qc = fmaf(c, dq, pb.v[e]);
      acc[SL_PP] += fmaf(c * c, wdp.m2[e], cp * qc * qc);
      acc[SL_PT] += wrx.m2x[e] + c * (2.f * wrx.cxy[e] + c * fmaf(wrx.n * wrx.my[e], wrx.my[e], wrx.m2y[e]));
    } else {
      un.v[e] = fsu * uo.v[e] + pb.v[e];                     // u += pbar
      acc[SL_PP] += cp * pb.v[e] * pb.v[e];
      acc[SL_PT] += wth.m2[e];
    }
    acc[SL_DP] += wdp.m2[e];
    acc[SL_DT] += ct * dt * dt;
    if (!isfinite(un.v[e]) || !isfinite(tbar.v[e])) acc[SL_NF] += 1.f;
  }
  // the new node rows are read in the next iteration only
  stv_cs<VW>(p.U[nw] + on, un);
  FV<VW> pu;
#pragma unroll
  for (int e = 0; e < VW; ++e) pu.v[e] = pb.v[e] + un.v[e];
  stv_cs<VW>(p.PU[nw] + on, pu);
  stv_cs<VW>(p.THBAR[nw] + on, tbar);
}

// closed-form prox of device d at VW time steps, given the average there
// (Section 4.2, weight (K+1) rho_p)
template <int VW>
__device__ __forceinline__ void closed_prox(const Params &p, const Iter &q, int d, int t0, const FV<VW> &xs) {
  const size_t od = (size_t)d * p.T + t0;
  const float den = 2.f * p.dev_a[d] + q.rho_dev, rden = __frcp_rn(den), bd = p.dev_b[d];
  const FV<VW> pd = ldv<VW>(p.PD + od), lo = ldv<VW>(p.dev_lo + od), hi = ldv<VW>(p.dev_hi + od);
  FV<VW> pn, dp;
#pragma unroll
  for (int e = 0; e < VW; ++e) {
    const float x = pd.v[e] - xs.v[e];                 // p_d - avg_k(pbar + u)
    pn.v[e] = relaxed(p.alpha, fminf(fmaxf(div_rn(q.rho_dev * x - bd, den, rden), lo.v[e]), hi.v[e]), pd.v[e]);
    dp.v[e] = pn.v[e] - pd.v[e];
  }
  stv<VW>(p.DPD + od, dp);
  stv<VW>(p.PD + od, pn);
}

// ---------------------------------------------------------------------------
// xs: avg_k(pbar + u) at each node with devices, one (node, VW time steps)
// item per thread; the node's closed-form devices are updated on the spot
// (Section 4.2), nodes with inner-ADMM devices keep the average in XS
// ---------------------------------------------------------------------------
template <int VW>
__device__ __forceinline__ void xs_body(const Params &p, unsigned bid, unsigned nblk) {
  const Iter q = load_iter(p);
  if (q.flags & ITF_SKIP) return;
  const int T = p.T, TV = p.T / VW;
  const unsigned n_xv = (unsigned)p.n_dnode * (unsigned)TV;
  for (unsigned item = bid * BLOCK + threadIdx.x; item < n_xv; item += nblk * BLOCK) {
    const int ci = (int)(item / (unsigned)TV), t0 = (int)(item % (unsigned)TV) * VW, n = p.dnode_ids[ci];
    const size_t on = (size_t)n * T + t0;
    FV<VW> xs;
    if (p.slice) {
      // a contingency slice: the sums over every slice's k, exchanged
      const float kpf = (float)p.Kp_glob, rkp = __frcp_rn(kpf), sm1 = q.fsu - 1.f;
      const double *esp = p.xsum + (size_t)ci * T + t0, *esq = p.xsum + (size_t)(p.n_dnode + ci) * T + t0;
#pragma unroll
      for (int e = 0; e < VW; ++e) xs.v[e] = div_rn(fmaf(sm1, (float)esq[e], (float)esp[e]), kpf, rkp);
    } else {
      xs = node_avg<VW>(p, q, n, t0);
    }
    if (p.dnode_keep[ci]) stv<VW>(p.XS + on, xs);
    for (int j = p.dnode_ptr[ci]; j < p.dnode_ptr[ci + 1]; ++j) closed_prox<VW>(p, q, p.dnode_dev[j], t0, xs);
  }
}

// ---------------------------------------------------------------------------
// closed: the closed-form devices of the nodes that have some, a group of
// lanes per (node, VW time steps): each lane sums one class of contingencies
// (the order of ksum2 at VW = 4, of ksum8 at VW = 1), then they share the
// node's devices.  With one thread per item the row loads, a few in flight at
// a time, were most of the 5 us that this phase took in front of the inner
// ADMM at 2k buses.
// ---------------------------------------------------------------------------
// the group's sums over k (every lane returns the total)
template <int VW, int G>
__device__ __forceinline__ FV<VW> group_ksum(const float *r, int T, int Kp, int c, unsigned gmask) {
  FV<VW> s;
#pragma unroll
  for (int e = 0; e < VW; ++e) s.v[e] = 0.f;
  const int whole = G == 8 ? (Kp & ~7) : Kp;
#pragma unroll 4
  for (int k = c; k < whole; k += G) {
    const FV<VW> x = ldv<VW>(r + (size_t)k * T);
#pragma unroll
    for (int e = 0; e < VW; ++e) s.v[e] += x.v[e];
  }
  if (G == 8 && c == 0) {
    for (int k = whole; k < Kp; ++k) {
      const FV<VW> x = ldv<VW>(r + (size_t)k * T);
#pragma unroll
      for (int e = 0; e < VW; ++e) s.v[e] += x.v[e];
    }
  }
#pragma unroll
  for (int m = 1; m < G; m <<= 1)
#pragma unroll
    for (int e = 0; e < VW; ++e) s.v[e] += __shfl_xor_sync(gmask, s.v[e], m);
  return s;
}

template <int VW>
__device__ __forceinline__ void closed_body(const Params &p, const Iter &q, unsigned bid, unsigned nblk) {
  constexpr int G = VW == 4 ? CLOSED_LANES4 : CLOSED_LANES1;
  if (q.flags & ITF_SKIP) return;
  const int T = p.T, TV = T / VW, Kp = p.Kp, c = threadIdx.x & (G - 1);
  const unsigned gmask = ((1u << G) - 1u) << ((threadIdx.x & 31) & ~(G - 1));
  const float sm1 = q.fsu - 1.f;
  const unsigned n = (unsigned)p.n_cnode * (unsigned)TV, step = (nblk * blockDim.x) / G;
  for (unsigned item = (bid * blockDim.x + threadIdx.x) / G; item < n; item += step) {
    const int t0 = (int)(item % (unsigned)TV) * VW;
    const int4 r = p.crec[item / (unsigned)TV];   // node, its first and one past its last entry of dnode_dev
    const int d0 = r.y + c < r.z ? p.dnode_dev[r.y + c] : -1;
    const size_t o = (size_t)r.x * Kp * T + t0;
    FV<VW> xs = group_ksum<VW, G>(p.PU[q.old] + o, T, Kp, c, gmask), sq;
#pragma unroll
    for (int e = 0; e < VW; ++e) sq.v[e] = 0.f;
    if (sm1 != 0.f) sq = group_ksum<VW, G>(p.U[q.old] + o, T, Kp, c, gmask);
#pragma unroll
    for (int e = 0; e < VW; ++e) xs.v[e] = avg_of(p, sm1, xs.v[e], sq.v[e]);
    if (d0 >= 0) closed_prox<VW>(p, q, d0, t0, xs);
    for (int j = r.y + c + G; j < r.z; j += G) closed_prox<VW>(p, q, p.dnode_dev[j], t0, xs);
  }
}

// the register path at the device's own chunk (cs, cr <= C; ONLY: cs = C and
// cr is C or C - 1, as for one instance)
template <int C, bool ONLY>
__device__ __forceinline__ void stor_r(const Params &p, int sidx, int lane, int cs, bool avg) {
  if constexpr (C > 1 && !ONLY) {
    if (cs < C) {
      stor_r<C - 1, false>(p, sidx, lane, cs, avg);
      return;
    }
  }
  stor_prox_r<C>(p, sidx, lane, avg);
}

template <int C, bool ONLY>
__device__ __forceinline__ void ramp_r(const Params &p, int r, int lane, int cr, bool avg) {
  if constexpr (C > 1) {
    if (cr < C) {
      if constexpr (ONLY) ramp_prox_r<C - 1>(p, r, lane, avg);
      else ramp_r<C - 1, false>(p, r, lane, cr, avg);
      return;
    }
  }
  ramp_prox_r<C>(p, r, lane, avg);
}

// ---------------------------------------------------------------------------
// inner: one warp per battery, then per ramp-limited generator (Appendix D),
// then per HVDC link and 32 steps.  C > 0: the register path, for horizons of at most
// REG_T steps (ONLY: chunks of C, else of at most C, by the instance's horizon);
// C = 0: the shared-memory path.  avg: each warp forms its node's average over
// contingencies (else it is in XS).  nw: the CTA's warps that take devices.  The
// shared-memory path holds the device's state there through the ten inner
// iterations; in global memory each row's read, step and write is a round trip
// to L2, or L1 while it holds them (30 buses, T = 1000: 1005 -> 352 us per
// iteration; 40 buses, T = 300: 103 -> 108).
// ---------------------------------------------------------------------------
template <int C, bool ONLY>
__device__ __forceinline__ void inner_body(const Params &p, unsigned bid, unsigned nblk, float *smem, bool avg, int nw) {
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  if (wib >= nw) return;
  const int T = p.T, n_inner = inner_units(p);
  float *wsm = C == 0 ? smem + (size_t)wib * warp_smem_floats(T) : nullptr;
  float *state_sh = C == 0 ? wsm + 3 * (T + 1) : nullptr;
  const int cs = (T + 32) >> 5, cr = (T + 31) >> 5;   // chunks of T + 1 and T elements
  for (int w = bid * nw + wib; w < n_inner; w += nblk * nw) {
    if (w < p.n_stor) {
      if constexpr (C > 0) stor_r<C, ONLY>(p, w, lane, cs, avg);
      else stor_prox(p, w, wsm, state_sh, lane, avg);
    } else if (w < p.n_stor + p.n_ramp) {
      if constexpr (C > 0) ramp_r<C, ONLY>(p, w - p.n_stor, lane, cr, avg);
      else ramp_prox(p, w - p.n_stor, wsm, state_sh, lane, avg);
    } else {
      hvdc_prox(p, w - p.n_stor - p.n_ramp, lane, avg);
    }
  }
}

// ---------------------------------------------------------------------------
// dsum: per (node, VW time steps), the sum of the node's device powers and
// the Welford state of their changes, in device order (the node sums of
// every contingency start from it)
// ---------------------------------------------------------------------------
template <int VW>
__device__ __forceinline__ void dsum_body(const Params &p, unsigned bid, unsigned nblk) {
  const Iter q = load_iter(p);
  if (q.flags & ITF_SKIP) return;
  const int T = p.T, TV = T / VW;
  const unsigned n_items = (unsigned)p.N * (unsigned)TV;
  for (unsigned item = bid * BLOCK + threadIdx.x; item < n_items; item += nblk * BLOCK) {
    const int n = (int)(item / (unsigned)TV), t0 = (int)(item % (unsigned)TV) * VW;
    FV<VW> sp;
    Welf<VW> w;
    w.reset();
#pragma unroll
    for (int e = 0; e < VW; ++e) sp.v[e] = 0.f;
    for (int j = p.dcsr_ptr[n]; j < p.dcsr_ptr[n + 1]; ++j) {
      const size_t od = (size_t)p.dcsr_idx[j] * T + t0;
      const FV<VW> pd = ldv<VW>(p.PD + od), dpd = ldv<VW>(p.DPD + od);
#pragma unroll
      for (int e = 0; e < VW; ++e) sp.v[e] += pd.v[e];
      w.add(dpd.v);
    }
    FV<VW> m, q2;
#pragma unroll
    for (int e = 0; e < VW; ++e) { m.v[e] = w.mean[e]; q2.v[e] = w.m2[e]; }
    const size_t os = (size_t)n * T + t0;
    stv<VW>(p.DSP + os, sp);
    stv<VW>(p.DSM + os, m);
    stv<VW>(p.DSQ + os, q2);
  }
}

// ---------------------------------------------------------------------------
// line: step 1 for every (contingency, line, VW time steps)
// ---------------------------------------------------------------------------
template <int VW>
__device__ __forceinline__ void line_body(const Params &p, unsigned bid, int ipt) {
  const int L = p.L, TV = p.T / VW;
  const unsigned n = (unsigned)p.Kp * (unsigned)L * (unsigned)TV;
  // each CTA takes ipt consecutive blocks of BLOCK items, so CTAs are
  // short-lived and the device kernels' CTAs find room beside them
  const unsigned base = bid * (unsigned)(BLOCK * ipt) + threadIdx.x;
  // items (line, contingency, step block): a line's K+1 rows are contiguous
  const int Kp = p.Kp;
  Idx3 ix, dx;
  ix.set(base, Kp, TV);
  dx.set(BLOCK, Kp, TV);
  if (base < n) {   // static: requested beside the scalars
    prefetch_l1(p.line_n1 + ix.a);
    prefetch_l1(p.line_n2 + ix.a);
    prefetch_l1(p.line_b + ix.a);
    prefetch_l1(p.line_u + ix.a);
  }
  const Iter q = load_iter(p);
  if (q.flags & ITF_SKIP) return;
#pragma unroll 1
  for (int j = 0; j < ipt; ++j, ix.step(dx, Kp, TV)) {
    if (base + (unsigned)(j * BLOCK) < n)
      line_item<VW>(p, q.old, q.old ^ 1, ix.b, ix.a, ix.c * VW, q.frp, q.frt, q.fsu, q.fsv, q.flags & ITF_VFRESH);
  }
}

// ---------------------------------------------------------------------------
// decide: residuals (Section 3.3) from the node kernel's n_part CTA partials
// in FP64 and a fixed order, the stopping test of Eq. (converge) and the
// adaptive penalty (Section 3.5); advances the iteration counter.
// ---------------------------------------------------------------------------
// the node kernel's n_part CTA partial sums reduced in FP64 and a fixed
// order; thread 0 returns true with the totals (written by other CTAs of the
// same launch: read past L1)
__device__ __forceinline__ bool reduce_partials(const Params &p, int n_part, double tot[NSLOT],
                                                double (*red)[NSLOT]) {
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) tot[s] = 0.0;
  for (int b = threadIdx.x; b < n_part; b += BLOCK) {
#pragma unroll
    for (int s = 0; s < NSLOT; ++s) tot[s] += __ldcg(p.partials + (size_t)b * NSLOT + s);
  }
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) {
    double v = tot[s];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) red[wib][s] = v;
  }
  __syncthreads();
  if (threadIdx.x != 0) return false;
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) {
    double v = 0.0;
    for (int w = 0; w < WARPS; ++w) v += red[w][s];
    tot[s] = v;
  }
  return true;
}

// the scalars of the iteration after q, which formed no residuals
__device__ __forceinline__ Iter next_iter(Iter q) {
  q.fsu = q.fsv = 1.f;
  q.old ^= 1;
  q.left -= 1;
  q.flags = q.left == 0 ? ITF_RES : 0;
  return q;
}

// An iteration whose residuals nobody reads (a non-finite value is caught at
// the next one that forms them): one thread advances the counter with stores
// alone.  Reading the scalars back and forming the next iteration's from them
// (FP64 conversions, 64-bit remainders) at the end of every iteration took
// about 3 us.
__device__ __forceinline__ void advance(const Params &p) {
  union {
    Iter r;
    int4 v[2];
  } x;
  x.r = next_iter(load_iter(p));
  int4 *d = reinterpret_cast<int4 *>(&p.sc->cur);
  d[0] = x.v[0];
  d[1] = x.v[1];
  atomicAdd(reinterpret_cast<unsigned long long *>(&p.sc->it), 1ull);
  p.sc->su = 1.0;
  p.sc->sv = 1.0;
  p.sc->v_fresh = 0;
}

// (dirty: told of a stop)
__device__ __forceinline__ void decide_body(const Params &p, int n_part, double (*red)[NSLOT], int *dirty = nullptr) {
  double tot[NSLOT];
  if (p.slice) {
    // a contingency slice: the residual sums of every slice, exchanged
    if (threadIdx.x != 0) return;
#pragma unroll
    for (int s = 0; s < NSLOT; ++s) tot[s] = p.xsum[(size_t)2 * p.n_dnode * p.T + s];
  } else {
    if (!reduce_partials(p, n_part, tot, red)) return;
  }
  DevScalars sc = *p.sc;
  const long long itn = sc.it + 1;
  const bool check_now = p.eps > 0 && p.check_every > 0 && (itn % p.check_every) == 0;
  const double rho_p = sc.rho_p, rho_th = sc.rho_th;
  int flags = 0;
  const double r_pp = sqrt(fmax(tot[SL_PP], 0.0));
  const double r_pt = sqrt(fmax(tot[SL_PT], 0.0));
  const double r_dp = rho_p * sqrt(fmax(tot[SL_DP], 0.0));
  const double r_dt = rho_th * sqrt(fmax(tot[SL_DT], 0.0));
  const double rp = sqrt(r_pp * r_pp + r_pt * r_pt);
  const double rd = sqrt(r_dp * r_dp + r_dt * r_dt);
  double nrp = rho_p, nrt = rho_th;
  if (!isfinite(rp) || !isfinite(rd) || tot[SL_NF] != 0.0) {
    sc.status = ST_NONFINITE;
    sc.stop = 1;
    flags |= HF_NONFINITE;
  } else {
    const double m = fmax(rp, rd);
    if (check_now && m <= p.tol) {
      sc.converged = 1;
      sc.stop = 1;
      flags |= HF_CONVERGED;
    } else if (check_now && p.stall_window > 0) {
      // stall rule (include/opf.h, opf_options): progress is a fall of the
      // best m by 1 %; without it for stall_window iterations, fix adapting
      // penalties, else stop with a stall
      if (m < 0.99 * sc.stall_ref) {
        sc.stall_ref = m;
        sc.stall_it = itn;
      } else if (itn - sc.stall_it >= p.stall_window) {
        if (adapting(p, sc, itn)) {
          sc.frozen_at = itn;
          sc.stall_ref = m;
          sc.stall_it = itn;
          flags |= HF_FROZEN;
        } else {
          sc.stalled = 1;
          sc.stop = 1;
          flags |= HF_STALLED;
        }
      }
    }
    if (adapt_at(p, sc, itn)) {   // Section 3.5 (strict comparisons, FP64)
      if (r_pp > p.mu * r_dp) nrp = rho_p * p.gamma;
      else if (r_dp > p.mu * r_pp) nrp = rho_p / p.gamma;
      if (r_pt > p.mu * r_dt) nrt = rho_th * p.gamma;
      else if (r_dt > p.mu * r_pt) nrt = rho_th / p.gamma;
      if (nrp != rho_p || nrt != rho_th) flags |= HF_ADAPTED;
    }
  }
  if (p.hist_cap > 0) {   // residual history ring (opf_history)
    double *row = p.hist + (size_t)(sc.hist_n % p.hist_cap) * HIST_COLS;
    row[0] = (double)itn;
    row[1] = rp;
    row[2] = rd;
    row[3] = r_pp;
    row[4] = r_pt;
    row[5] = r_dp;
    row[6] = r_dt;
    row[7] = rho_p;
    row[8] = rho_th;
    row[9] = (double)flags;
    sc.hist_n += 1;
  }
  sc.res[0] = rp; sc.res[1] = rd; sc.res[2] = r_pp; sc.res[3] = r_pt; sc.res[4] = r_dp; sc.res[5] = r_dt;
  sc.su = rho_p / nrp;   // pending rescale of u and v (Section 3.5), applied on their next read
  sc.sv = rho_th / nrt;
  sc.rho_p = nrp;
  sc.rho_th = nrt;
  sc.it = itn;
  sc.v_fresh = 0;
  set_iter(p, sc);
  *p.sc = sc;
  if (dirty && (sc.cur.flags & ITF_SKIP)) *dirty = 1;
}

// the CTA's residual partial sums, FP32 per thread and FP64 across warps, as
// partial number `part`
__device__ __forceinline__ void write_partials(const Params &p, unsigned part, const float (&acc)[NSLOT],
                                               double (*red)[NSLOT]) {
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) {
    float v = acc[s];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) red[wib][s] = (double)v;
  }
  __syncthreads();
  if (threadIdx.x < NSLOT) {
    double v = 0.0;
    for (int w = 0; w < WARPS; ++w) v += red[w][threadIdx.x];
    p.partials[(size_t)part * NSLOT + threadIdx.x] = v;
  }
}

// The warp's FP32 sums of acc, in the order of write_partials (every pair that
// its shuffles add meets here): at each step a lane keeps half of its sums and
// hands the others over, 8 shuffles for the five sums instead of 25.
__device__ __forceinline__ void warp_sums(const float (&acc)[NSLOT], float *out) {
  static_assert(NSLOT == 5, "the halves below");
  const int lane = threadIdx.x & 31;
  const bool h = lane & 16, b = lane & 8, c = lane & 4;
  auto give = [](float v, int o) { return __shfl_xor_sync(FULL, v, o); };
  // sums 0 1 2 to the lower half, 3 4 to the upper
  float x0 = (h ? acc[3] : acc[0]) + give(h ? acc[0] : acc[3], 16);
  float x1 = (h ? acc[4] : acc[1]) + give(h ? acc[1] : acc[4], 16);
  float x2 = acc[2] + give(acc[2], 16);   // (unused in the upper half)
  // the first two to the lower quarters, the third to the upper
  float y0 = (b ? x2 : x0) + give(b ? x0 : x2, 8);
  float y1 = x1 + give(x1, 8);            // (unused in the upper quarters)
  float z = (c ? y1 : y0) + give(c ? y0 : y1, 4);
  z += give(z, 2);
  z += give(z, 1);
  // lanes 0, 4, 8, 16, 20 hold sums 0, 1, 2, 3, 4
  const int slot = (h ? 3 : 0) + (b ? 2 : 0) + (c ? 1 : 0);
  if ((lane & 3) == 0 && !(b && c) && slot < NSLOT) out[slot] = z;
}

// the node kernel's shared memory
struct NodeMem {
  double red[WARPS][NSLOT];
  int last;
};
// The pass with residuals of a batch's instance.  Its partial sums are always
// those of its own grid (p.node_grid, one per CTA there), so that the residuals
// do not depend on how many CTAs the instance has here: each CTA forms several.
// A warp leaves its sums of each in p.wsums and goes on; one barrier later the
// CTA adds them up by partial sum (a barrier for each cost 64 mixed instances 24
// us per step, though one iteration in ten forms them; one for every eight, in
// shared memory, 40 instances of T = 7 and 31 0.9 us).  Out of line: inlined, it took registers
// from the pass without residuals (16 mixed instances 1.1 us per step).
template <int VW, bool RELAX>
__device__ __noinline__ void node_units(const Params &p, unsigned bid, unsigned nblk) {
  const int TV = p.T / VW, Kp = p.Kp;
  const unsigned n = (unsigned)Kp * (unsigned)p.N * (unsigned)TV;
  const unsigned parts = (unsigned)p.node_grid, ustride = parts * BLOCK;
  const Iter q = load_iter(p);
  Idx3 ix, dx;
  dx.set(ustride, Kp, TV);
  for (unsigned u = bid; u < parts; u += nblk) {
    float acc[NSLOT] = {0.f, 0.f, 0.f, 0.f, 0.f};
    unsigned item = u * BLOCK + threadIdx.x;
    ix.set(item, Kp, TV);
    for (; item < n; item += ustride, ix.step(dx, Kp, TV))
      node_item<VW, RELAX, true, NODE_RES_NB, true, false>(p, q.old, q.old ^ 1, ix.b, ix.a, ix.c * VW, q.fsu, acc);
    warp_sums(acc, p.wsums + ((size_t)u * WARPS + (threadIdx.x >> 5)) * NSLOT);
  }
  __syncthreads();
  const unsigned units = (parts - bid + nblk - 1) / nblk;   // bid < nblk <= parts
  for (unsigned x = threadIdx.x; x < units * NSLOT; x += BLOCK) {   // as write_partials
    const unsigned u = bid + x / NSLOT * nblk, s = x % NSLOT;
    const float *f = p.wsums + (size_t)u * WARPS * NSLOT + s;
    double v = 0.0;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) v += (double)f[w * NSLOT];
    p.partials[(size_t)u * NSLOT + s] = v;
  }
}

// ---------------------------------------------------------------------------
// node: step 3 for every (contingency, node, VW time steps); where the
// residuals are read, the CTA's partial sums (FP32 per thread, FP64 across
// warps); then the last CTA to finish takes the decisions and advances the
// iteration (a slice's decisions wait for the exchange: opf_slice_finish).
// One launch serves both kinds of iteration and the decisions: as three
// kernels (a residual-free pass, a general one and the decisions, each
// returning at once when not due) an iteration of 2k buses spent about 5 of
// its 36 us on their launches.  At 64 registers (four CTAs per SM, what the
// residual-free pass wants) the general pass gathers one terminal at a time.
// ---------------------------------------------------------------------------
// UNITS (batches): an instance's CTAs are fewer than its residual partial sums
// (node_units).
template <int VW, bool RELAX, bool ILD, bool LAT = false, bool UNITS = false>
__device__ __forceinline__ void node_body(const Params &p, unsigned bid, unsigned nblk, NodeMem &mem,
                                          int *dirty = nullptr) {
  double(*red)[NSLOT] = mem.red;
  const int N = p.N, TV = p.T / VW, Kp = p.Kp;
  const unsigned n = (unsigned)Kp * (unsigned)N * (unsigned)TV;
  const unsigned stride = nblk * BLOCK;
  unsigned item = bid * BLOCK + threadIdx.x;
  // items (node, contingency, step block): a node's K+1 rows are contiguous,
  // and so are the K+1 rows of each line it gathers
  Idx3 ix, dx;
  ix.set(item, Kp, TV);
  dx.set(stride, Kp, TV);
  if (item < n) prefetch_l1(p.nrec + 3 * ix.a);   // static: requested beside the scalars
  const Iter q = load_iter(p);
  if (q.flags & ITF_SKIP) return;
  const bool res = q.flags & ITF_RES;
  float acc[NSLOT] = {0.f, 0.f, 0.f, 0.f, 0.f};
  if constexpr (UNITS) {
    if (res) node_units<VW, RELAX>(p, bid, nblk);
  }
  if (!UNITS && res) {
    for (; item < n; item += stride, ix.step(dx, Kp, TV))
      node_item<VW, RELAX, true, LAT ? 4 : NODE_RES_NB, ILD, LAT>(p, q.old, q.old ^ 1, ix.b, ix.a, ix.c * VW, q.fsu, acc);
  } else if (!res) {
    for (; item < n; item += stride, ix.step(dx, Kp, TV))
      node_item<VW, RELAX, false, LAT ? 4 : NODE_LEAN_NB, ILD, LAT>(p, q.old, q.old ^ 1, ix.b, ix.a, ix.c * VW, q.fsu, acc);
  }
  if (res && !UNITS) write_partials(p, bid, acc, red);
  if (p.slice) return;
  // the count is taken after every thread of the CTA has read the scalars and
  // (res) its partial sums are written; the last CTA alone goes on
  __syncthreads();
  if (threadIdx.x == 0) {
    if (res) __threadfence();
    const bool last = atomicAdd(p.done, 1u) == nblk - 1;
    mem.last = last;
    if (last) {
      *p.done = 0;
      if (!res) advance(p);
    }
  }
  if (!res) return;
  __syncthreads();
  if (!mem.last) return;
  __threadfence();
  decide_body(p, UNITS ? p.node_grid : (int)nblk, red, dirty);
}

// ---------------------------------------------------------------------------
// kernel entry points: one instance (parameters in the constant bank), or a
// batch of instances (each CTA looks up its instance, its block index within
// the instance and the instance's block count in a schedule, and works on a
// shared-memory copy of that instance's parameters)
// ---------------------------------------------------------------------------
template <int VW>
__global__ void __launch_bounds__(BLOCK) xs_kernel(Params p) { xs_body<VW>(p, blockIdx.x, gridDim.x); }

// Every device of an iteration in one launch (step 2): the first inner_blocks
// CTAs take the inner-ADMM devices and links, the others the closed-form
// ones.  Each forms its node's average itself, so nothing runs in front of
// the inner ADMM, the longest chain of the phase; nodes with several
// inner-ADMM devices form it once per device.  Where the averages and the
// closed-form devices are a kernel of their own (avg false), only the first
// part is launched.
template <int C>
__global__ void __launch_bounds__(DEVB) dev_kernel(Params p, int inner_blocks, bool avg, int nw) {
  extern __shared__ float smem[];
  if ((int)blockIdx.x < inner_blocks) inner_body<C, true>(p, blockIdx.x, inner_blocks, smem, avg, nw);
  else if (p.T % 4 == 0) closed_body<4>(p, load_iter(p), blockIdx.x - inner_blocks, gridDim.x - inner_blocks);
  else closed_body<1>(p, load_iter(p), blockIdx.x - inner_blocks, gridDim.x - inner_blocks);
}

template <int VW>
__global__ void __launch_bounds__(BLOCK) dsum_kernel(Params p) { dsum_body<VW>(p, blockIdx.x, gridDim.x); }

template <int VW>
__global__ void __launch_bounds__(BLOCK, 4) line_kernel(Params p, int ipt) {
  line_body<VW>(p, blockIdx.x, ipt);
}

// The over-relaxed variant reads one more row per terminal and carries the mean
// change of p: three CTAs per SM at 80 registers (1k buses, T = 48, K = 20,
// alpha = 1.5, us per iteration: two 28.6, three 26.9, four 28.3; 39.8 when
// every iteration carried the residual sums).  ILD: device sums in the pass.
template <int VW, bool RELAX, bool ILD, bool LAT>
__global__ void __launch_bounds__(BLOCK, LAT ? 2 : RELAX ? NODE_RX_CTAS : NODE_CTAS) node_kernel(Params p) {
  __shared__ NodeMem mem;
  node_body<VW, RELAX, ILD, LAT>(p, blockIdx.x, gridDim.x, mem);
}

// ---------------------------------------------------------------------------
// A small instance on one CTA: n iterations in one launch, their phases apart
// by CTA barriers instead of kernel boundaries (a microsecond each, and the
// scalars and static rows come back through L2 every time).  The items, their
// arithmetic and the residuals' partial sums (one per 256 node items) are
// those of the kernels above.  30 buses, T = 1, K = 5: 8.35 -> 5.1 us per
// iteration; what is left are rows that other threads wrote, read through L2.
// Which instances: opfk_plan.
// ---------------------------------------------------------------------------
template <int VW, bool RELAX>
__device__ __forceinline__ int small_iteration(const Params &p, const Iter &q, double (*red)[NSLOT]) {
  const int T = p.T, TV = T / VW, Kp = p.Kp;
  closed_body<VW>(p, q, 0, 1);
  const unsigned nl = (unsigned)Kp * (unsigned)p.L * (unsigned)TV, nn = (unsigned)Kp * (unsigned)p.N * (unsigned)TV;
  Idx3 ix;
  for (unsigned i = threadIdx.x; i < nl; i += BLOCK) {
    ix.set(i, Kp, TV);
    line_item<VW>(p, q.old, q.old ^ 1, ix.b, ix.a, ix.c * VW, q.frp, q.frt, q.fsu, q.fsv, q.flags & ITF_VFRESH);
  }
  __syncthreads();
  const bool res = q.flags & ITF_RES;
  unsigned part = 0;
  for (unsigned base = 0; base < nn; base += BLOCK, ++part) {
    const unsigned i = base + threadIdx.x;
    float acc[NSLOT] = {0.f, 0.f, 0.f, 0.f, 0.f};
    if (i < nn) {
      ix.set(i, Kp, TV);
      if (res) node_item<VW, RELAX, true, 4, true, true>(p, q.old, q.old ^ 1, ix.b, ix.a, ix.c * VW, q.fsu, acc);
      else node_item<VW, RELAX, false, 4, true, true>(p, q.old, q.old ^ 1, ix.b, ix.a, ix.c * VW, q.fsu, acc);
    }
    if (res) {
      write_partials(p, part, acc, red);
      __syncthreads();   // red is used again
    }
  }
  return (int)part;
}

template <bool RELAX>
__global__ void __launch_bounds__(BLOCK) small_kernel(Params p, int n) {
  __shared__ double red[WARPS][NSLOT];
  Iter q = load_iter(p);   // every thread's own copy, stored where residuals are formed and at the end
  int ahead = 0;           // iterations run since it was last stored
  auto store = [&]() {
    if (threadIdx.x == 0 && ahead) {
      DevScalars sc = *p.sc;
      sc.it += ahead;
      sc.su = sc.sv = 1.0;
      sc.v_fresh = 0;
      sc.cur = q;
      *p.sc = sc;
    }
    ahead = 0;
  };
  for (int i = 0; i < n && !(q.flags & ITF_SKIP); ++i) {
    const bool res = q.flags & ITF_RES;
    const int parts = p.T % 4 == 0 ? small_iteration<4, RELAX>(p, q, red) : small_iteration<1, RELAX>(p, q, red);
    if (res) {
      store();
      decide_body(p, parts, red);
      __syncthreads();
      q = load_iter(p);
    } else {
      q = next_iter(q);
      ++ahead;
      __syncthreads();
    }
  }
  store();
}

// a slice's decisions, from the exchanged sums
__global__ void __launch_bounds__(BLOCK) decide_kernel(Params p) {
  __shared__ double red[WARPS][NSLOT];
  const Iter q = load_iter(p);
  if (q.flags & ITF_SKIP) return;
  if (q.flags & ITF_RES) decide_body(p, 0, red);
  else if (threadIdx.x == 0) advance(p);
}

// A contingency slice's contributions to the exchange (after its node
// sums): sum over its k of pbar + u at every node with devices, the same of
// u on adaptation iterations (whose decision may rescale u before the next
// device prox reads it), and its residual partial sums on iterations that
// form residuals.  A stopped context (and `prime`, before the first
// iteration) contributes the sums of its current state, so that the
// caller's exchange always sums fresh contributions of every slice.
__global__ void __launch_bounds__(BLOCK) slice_sums_kernel(Params p, int prime) {
  __shared__ double red[WARPS][NSLOT];
  __shared__ int s_buf, s_with_u, s_res;
  if (threadIdx.x == 0) {
    const DevScalars sc = *p.sc;
    const long long itn = sc.it + 1;
    const bool stopped = sc.status != 0 || sc.stop != 0;
    const bool current = prime || stopped;
    const int old = (int)(sc.it & 1);
    s_buf = current ? old : old ^ 1;
    s_with_u = current || adapt_at(p, sc, itn);
    s_res = !current && res_at(p, sc, itn);
  }
  __syncthreads();
  const int T = p.T, Kp = p.Kp;
  const size_t KT = (size_t)Kp * T;
  const float *W = p.PU[s_buf], *U = p.U[s_buf];
  const bool with_u = s_with_u != 0;
  double *esp = p.xsum, *esq = p.xsum + (size_t)p.n_dnode * T;
  for (long long i = (long long)blockIdx.x * BLOCK + threadIdx.x; i < (long long)p.n_dnode * T;
       i += (long long)gridDim.x * BLOCK) {
    const int ci = (int)(i / T), t = (int)(i % T);
    const size_t o = (size_t)p.dnode_ids[ci] * KT + t;
    esp[i] = (double)ksum8(W, o, T, Kp);
    esq[i] = with_u ? (double)ksum8(U, o, T, Kp) : 0.0;
  }
  if (blockIdx.x == 0) {
    double tot[NSLOT];
    double *tail = p.xsum + (size_t)2 * p.n_dnode * T;
    if (s_res) {
      if (reduce_partials(p, p.node_grid, tot, red))
        for (int s = 0; s < NSLOT; ++s) tail[s] = tot[s];
    } else if (threadIdx.x < NSLOT) {
      tail[threadIdx.x] = 0.0;
    }
  }
}

// the instance of this CTA, from its schedule entry e: its parameters copied
// to shared memory, and (block, blocks) within the instance
__device__ __forceinline__ const Params &batch_params(const Params *ps, const int4 e, Params &sp,
                                                      unsigned &bid, unsigned &nblk) {
  static_assert(sizeof(Params) % 4 == 0, "Params is copied as 32-bit words");
  const int *src = reinterpret_cast<const int *>(ps + e.x);
  int *dst = reinterpret_cast<int *>(&sp);
  for (int i = threadIdx.x; i < (int)(sizeof(Params) / 4); i += blockDim.x) dst[i] = src[i];
  __syncthreads();
  bid = (unsigned)e.y;
  nblk = (unsigned)e.z;
  return sp;
}

// The node kernel's CTAs shared out over the running instances, by the device
// kernel's first CTA in front of its devices, in the iterations that follow the
// start of a call or an instance's stop: floor(slots x items / all running
// items) CTAs each, at least one and at most its grid.  64 mixed instances, us
// per step as given: all running 721 with a grid of its own for each (in
// seven launches), 570 with shares that stay when others stop, 576 with these;
// the last one running, the others compacted away, 34 to 90, 92 to 142 and 16
// to 67; four running 106, 177 and 65.
// (mem: the CTA's shared memory for an instance's parameters, not in use yet.
// More would change the kernel's share of L1, which the concurrent line kernel's
// CTAs cannot follow: with arrays of its own 16 mixed instances took 3 us more
// per step.)
struct DealMem {
  static constexpr int N = 64;   // instances at a time
  unsigned long long sum[DEV_WARPS];
  int m[N], inst[N];
};
__device__ void deal_nodes(const Params *ps, const NodeDeal &d, DealMem &mem) {
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  auto runs = [&](const NodeShare &s) { return !(ps[s.inst].sc->cur.flags & ITF_SKIP); };
  unsigned long long sum = 0;
  for (int i = tid; i < d.n; i += DEVB) {
    const NodeShare s = d.share[i];
    if (runs(s)) sum += s.items;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(FULL, sum, o);
  if (lane == 0) mem.sum[w] = sum;
  __syncthreads();
  sum = 0;
#pragma unroll
  for (int i = 0; i < DEV_WARPS; ++i) sum += mem.sum[i];
  int at = 0;   // entries written
  for (int i0 = 0; i0 < d.n; i0 += DealMem::N) {
    const int i = i0 + tid;
    if (tid < DealMem::N && i < d.n) {
      const NodeShare s = d.share[i];
      mem.m[tid] = runs(s) ? min(s.grid, max(1, (int)((unsigned long long)d.slots * s.items / sum))) : 0;
      mem.inst[tid] = s.inst;
    }
    __syncthreads();
    for (int j = 0; j < DealMem::N && i0 + j < d.n; ++j) {
      const int mj = mem.m[j];
      for (int r = tid; r < mj; r += DEVB) d.slot[at + r] = make_int4(mem.inst[j], r, mj, 0);
      at += mj;
    }
    __syncthreads();
  }
  for (int b = at + tid; b < d.cap; b += DEVB) d.slot[b] = make_int4(-1, 0, 0, 0);
  if (tid == 0) *d.dirty = 0;
}

// The devices of every instance: the first inner_blocks CTAs of the schedule
// take links and inner-ADMM devices of up to BATCH_REG_T steps, the others
// closed-form ones.  C: the largest register chunk of the batch's instances.
// Registers are held to 80, 128, 128 and 168: left to the compiler, C = 1 took
// 93 and five CTAs per SM instead of six (40 instances of T = 7 and 31 60.0
// against 57.0 us per step, 256 of T = 1 and 24 57.3 against 55.9).
template <int C>
__global__ void __launch_bounds__(DEVB, C == 1 ? 6 : C == 4 ? 3 : 4) dev_kernel_b(
    const Params *ps, const int4 *sched, int inner_blocks, int blocks, NodeDeal deal) {
  __shared__ Params sp;
  if (blockIdx.x == 0) {
    static_assert(sizeof(DealMem) <= sizeof(Params) && alignof(DealMem) <= alignof(Params), "shared by turns");
    if (*deal.dirty) deal_nodes(ps, deal, *reinterpret_cast<DealMem *>(&sp));
    if (blocks == 0) return;   // no device in any instance
  }
  unsigned bid, nblk;
  const Params &p = batch_params(ps, sched[blockIdx.x], sp, bid, nblk);
  if ((int)blockIdx.x < inner_blocks) inner_body<C, false>(p, bid, nblk, nullptr, true, DEV_WARPS);
  else if (p.T % 4 == 0) closed_body<4>(p, load_iter(p), bid, nblk);
  else closed_body<1>(p, load_iter(p), bid, nblk);
}

// The inner-ADMM devices of the instances beyond BATCH_REG_T steps, staged in
// shared memory, on a stream of their own: their chains are the longest of the
// phase, and the other devices' CTAs are not held to the room that they leave
// (one launch for all, unstaged: 15 instances of T = 24 with one of T = 1000
// took 771 us per step, now 340; 16 instances of T = 168 165 -> 138).
__global__ void __launch_bounds__(DEVB) smem_kernel_b(const Params *ps, const int4 *sched, unsigned bytes) {
  extern __shared__ float smem[];
  __shared__ Params sp;
  unsigned bid, nblk;
  const Params &p = batch_params(ps, sched[blockIdx.x], sp, bid, nblk);
  inner_body<0, true>(p, bid, nblk, smem, true, smem_warps(p.T, bytes));
}

// the lines of every instance: the first n4 CTAs of the schedule take those
// whose horizon is whole 4-step blocks, the others the rest
__global__ void __launch_bounds__(BLOCK, 4) line_kernel_b(const Params *ps, const int4 *sched, int n4) {
  __shared__ Params sp;
  unsigned bid, nblk;
  const Params &p = batch_params(ps, sched[blockIdx.x], sp, bid, nblk);
  if ((int)blockIdx.x < n4) line_body<4>(p, bid, LINE_IPT);
  else line_body<1>(p, bid, LINE_IPT);
}

template <bool RELAX>
__global__ void __launch_bounds__(BLOCK, RELAX ? NODE_RX_CTAS : NODE_CTAS) node_kernel_b(
    const Params *ps, const int4 *slot, int *dirty) {
  __shared__ Params sp;
  __shared__ NodeMem mem;
  const int4 e = slot[blockIdx.x];   // dealt out by deal_nodes
  if (e.x < 0) return;
  unsigned bid, nblk;
  const Params &p = batch_params(ps, e, sp, bid, nblk);
  if (p.T % NODE_VW == 0) node_body<NODE_VW, RELAX, true, false, true>(p, bid, nblk, mem, dirty);
  else node_body<1, RELAX, true, false, true>(p, bid, nblk, mem, dirty);
}

// A line's terminal values from its stored (p, mid) at contingency k:
// p2 (0 on the outaged line) and theta_{1,2} = mid +- h, h = p / (2b) on an
// active line and the stored value itself on the outaged line.
// the actual iterate from two relaxed ones: (P - (1 - alpha) P_prev) / alpha
__device__ __forceinline__ float actual(float alpha, float cur, float prev) {
  return (cur - (1.f - alpha) * prev) / alpha;
}

__device__ __forceinline__ void line_terminals(const Params &p, int cur, int k, int l, size_t i, float &p2,
                                               float &th1, float &th2) {
  const float ps = p.P[cur][i], m = p.MID[cur][i];
  float h = ps;
  p2 = 0.f;
  if (p.out_line[k] != l) {
    const float tb = 2.f * p.line_b[l];
    h = div_rn(ps, tb, __frcp_rn(tb));
    p2 = ps;
  }
  th1 = m + h;
  th2 = m - h;
}

// ---------------------------------------------------------------------------
// import / export between internal and caller numbering
// ---------------------------------------------------------------------------
__global__ void import_kernel(Params p, int cur, const float *pl, const float *a1, const float *a2,
                              const float *v1, const float *v2, const float *u) {
  const int T = p.T, L = p.L, N = p.N;
  const long long nl = (long long)p.Kp * L * T, nn = (long long)p.Kp * N * T;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nl + nn;
       i += (long long)gridDim.x * blockDim.x) {
    if (i < nl) {
      const int k = (int)(i / ((long long)L * T));
      const long long rem = i - (long long)k * L * T;
      const int l = (int)(rem / T), t = (int)(rem % T);
      const size_t src = ((size_t)k * L + p.line_perm[l]) * T + t, dst = lidx(p, k, l, t);
      // stored as p and the mean angle; the outaged line keeps its half
      // angle difference in p's place (its p is 0)
      const float x1 = a1 ? a1[src] : 0.f, x2 = a2 ? a2[src] : 0.f;
      const bool act = p.out_line[k] != l;
      p.P[cur][dst] = act ? (pl ? pl[src] : 0.f) : 0.5f * (x1 - x2);
      p.MID[cur][dst] = 0.5f * (x1 + x2);
      p.V1[cur][dst] = v1 ? v1[src] : 0.f;
      p.V2[cur][dst] = v2 ? v2[src] : 0.f;
    } else {
      const long long j = i - nl;
      const int k = (int)(j / ((long long)N * T));
      const long long rem = j - (long long)k * N * T;
      const int n = (int)(rem / T), t = (int)(rem % T);
      p.U[cur][nidx(p, k, n, t)] = u ? u[((size_t)k * N + p.node_perm[n]) * T + t] : 0.f;
    }
  }
}

// Entry i of the exported inner-ADMM state (opf_get_info's layout: per
// ramp-limited generator, then per battery, lambda then beta over the
// constraint rows): its place in the device arrays, nullptr for a battery's
// equality rows' beta (always 0).
__device__ __forceinline__ float *inner_slot(const Params &p, long long i) {
  const int T = p.T, Tp = T + 1, mr = 4 * T - 2, ms = 8 * T + 4;
  const long long nr = (long long)p.n_ramp * 2 * mr;
  if (i < nr) {
    const int r = (int)(i / (2 * mr));
    int x = (int)(i - (long long)r * 2 * mr);
    float *a = x < mr ? p.ramp_lam : p.ramp_beta;
    if (x >= mr) x -= mr;
    // rows p <= pmax, -p <= -pmin (T each), ramp up, ramp down (T - 1 each)
    const int g = x < 2 * T ? x / T : RG_RU + (x - 2 * T) / (T - 1);
    const int t = x < 2 * T ? x % T : (x - 2 * T) % (T - 1);
    return a + ((size_t)r * RG_N + g) * T + t;
  }
  i -= nr;
  const int b = (int)(i / (2 * ms));
  int x = (int)(i - (long long)b * 2 * ms);
  const bool beta = x >= ms;
  if (beta) x -= ms;
  float *a = (beta ? p.stor_beta : p.stor_lam) + (size_t)b * SG_N * Tp;
  if (x < 2 * T + 2) {   // p + c - delta = 0, soc dynamics (T each), s_1 = 0, s_{T+1} = 0
    if (beta) return nullptr;
    return x < 2 * T ? a + (x / T) * Tp + x % T : a + SG_E3 * Tp + (x - 2 * T);
  }
  x -= 2 * T + 2;        // limits of c and delta (T each), of s (T + 1 each)
  return x < 4 * T ? a + (SG_CU + x / T) * Tp + x % T : a + (SG_SU + (x - 4 * T) / Tp) * Tp + (x - 4 * T) % Tp;
}

__global__ void inner_export_kernel(Params p, float *out, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float *s = inner_slot(p, i);
    out[i] = s ? *s : 0.f;
  }
}

// the arrays were zeroed; rho: the penalty the duals are scaled for, negative
// so that the factors are rebuilt on first use
__global__ void inner_import_kernel(Params p, const float *in, long long n, float rho) {
  const long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (long long i = i0; i < n; i += (long long)gridDim.x * blockDim.x) {
    float *s = inner_slot(p, i);
    if (s) *s = in[i];
  }
  for (long long i = i0; i < (long long)p.n_ramp + p.n_stor; i += (long long)gridDim.x * blockDim.x)
    (i < p.n_ramp ? p.ramp_rho[i] : p.stor_rho[i - p.n_ramp]) = rho;
}

// A starting state from node rows in the caller's numbering, rows[(t N + n)
// stride + 0] = price / price_scale and [+ 1] = node angle: u_k = -price /
// (rho_p (K+1)) in every contingency (prices are -rho_p sum_k u_k), every
// line terminal at its node's angle, line power b (theta1 - theta2) clipped
// to the limit (0 on the outaged line of a contingency, whose terminals keep
// their angles), v = 0.  The same construction as a host-built state
// imported through import_kernel.
__global__ void start_from_nodes_kernel(Params p, int cur, const float *rows, int stride, float price_scale,
                                        float u_scale) {
  const int T = p.T, L = p.L, N = p.N;
  const long long nl = (long long)p.Kp * L * T, nn = (long long)p.Kp * N * T;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nl + nn;
       i += (long long)gridDim.x * blockDim.x) {
    if (i < nl) {
      const int k = (int)(i / ((long long)L * T));
      const long long rem = i - (long long)k * L * T;
      const int l = (int)(rem / T), t = (int)(rem % T);
      const float x1 = rows[((size_t)t * N + p.node_perm[p.line_n1[l]]) * stride + 1];
      const float x2 = rows[((size_t)t * N + p.node_perm[p.line_n2[l]]) * stride + 1];
      const bool act = p.out_line[k] != l;
      const float u = p.line_u[l];
      const size_t dst = lidx(p, k, l, t);
      p.P[cur][dst] = act ? fminf(fmaxf(p.line_b[l] * (x1 - x2), -u), u) : 0.5f * (x1 - x2);
      p.MID[cur][dst] = 0.5f * (x1 + x2);
      p.V1[cur][dst] = 0.f;
      p.V2[cur][dst] = 0.f;
    } else {
      const long long j = i - nl;
      const int k = (int)(j / ((long long)N * T));
      const long long rem = j - (long long)k * N * T;
      const int n = (int)(rem / T), t = (int)(rem % T);
      const float price = rows[((size_t)t * N + p.node_perm[n]) * stride] * price_scale;
      p.U[cur][nidx(p, k, n, t)] = -price * u_scale;
    }
  }
}

// node averages from the stored terminal values (after import)
__global__ void node_average_kernel(Params p, int cur) {
  const int T = p.T, N = p.N;
  for (long long item = (long long)blockIdx.x * blockDim.x + threadIdx.x; item < (long long)N * T;
       item += (long long)gridDim.x * blockDim.x) {
    const int n = (int)(item / T), t = (int)(item % T);
    float devsum = 0.f;
    for (int j = p.dcsr_ptr[n]; j < p.dcsr_ptr[n + 1]; ++j) devsum += p.PD[(size_t)p.dcsr_idx[j] * T + t];
    for (int k = 0; k < p.Kp; ++k) {
      float sp = devsum, st = 0.f;
      for (int j = p.lcsr_ptr[n]; j < p.lcsr_ptr[n + 1]; ++j) {
        const int code = p.lcsr[j].x;
        const size_t ol = lidx(p, k, code >> 1, t);
        float p2, th1, th2;
        line_terminals(p, cur, k, code >> 1, ol, p2, th1, th2);
        sp += (code & 1) ? p2 : -p2;
        st += (code & 1) ? th2 : th1;
      }
      const size_t on = nidx(p, k, n, t);
      const float pb = sp / p.cnt_p[n];
      p.PU[cur][on] = pb + p.U[cur][on];   // u was imported before
      p.THBAR[cur][on] = p.cnt_th[n] > 0.f ? st / p.cnt_th[n] : 0.f;
    }
  }
}

// v projected onto v_bar = 0 per node and contingency (Appendix C)
__global__ void project_v_kernel(Params p, int cur) {
  const int T = p.T, N = p.N;
  for (long long item = (long long)blockIdx.x * blockDim.x + threadIdx.x;
       item < (long long)p.Kp * N * T; item += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(item / ((long long)N * T));
    const long long rem = item - (long long)k * N * T;
    const int n = (int)(rem / T), t = (int)(rem % T);
    const int l0 = p.lcsr_ptr[n], l1 = p.lcsr_ptr[n + 1];
    if (l1 == l0) continue;
    float s = 0.f;
    for (int j = l0; j < l1; ++j) {
      const int code = p.lcsr[j].x;
      const size_t ol = lidx(p, k, code >> 1, t);
      s += (code & 1) ? p.V2[cur][ol] : p.V1[cur][ol];
    }
    const float m = s / p.cnt_th[n];
    for (int j = l0; j < l1; ++j) {
      const int code = p.lcsr[j].x;
      const size_t ol = lidx(p, k, code >> 1, t);
      if (code & 1) p.V2[cur][ol] -= m; else p.V1[cur][ol] -= m;
    }
  }
}

// lines to caller numbering; v = sv (V + theta - theta_bar) unless fresh
__global__ void export_lines_kernel(Params p, int cur, float *pl, float *a1, float *a2, float *v1,
                                    float *v2) {
  const DevScalars sc = *p.sc;
  const float sv = (float)sc.sv;
  const int T = p.T, L = p.L;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < (long long)p.Kp * L * T;
       i += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(i / ((long long)L * T));
    const long long rem = i - (long long)k * L * T;
    const int l = (int)(rem / T), t = (int)(rem % T);
    const size_t dst = ((size_t)k * L + p.line_perm[l]) * T + t, li = lidx(p, k, l, t);
    float p2, th1, th2;
    line_terminals(p, cur, k, l, li, p2, th1, th2);
    if (v1 || v2) {
      float x = p.V1[cur][li], y = p.V2[cur][li];
      if (!sc.v_fresh) {
        x += th1 - p.THBAR[cur][nidx(p, k, p.line_n1[l], t)];
        y += th2 - p.THBAR[cur][nidx(p, k, p.line_n2[l], t)];
      }
      if (v1) v1[dst] = sv * x;
      if (v2) v2[dst] = sv * y;
    }
    if (p.alpha != 1.f && !sc.v_fresh) {
      // over-relaxed: the buffers hold P = alpha p + (1 - alpha) P_prev
      float q2, q1a, q2a;
      line_terminals(p, cur ^ 1, k, l, li, q2, q1a, q2a);
      p2 = actual(p.alpha, p2, q2);
      th1 = actual(p.alpha, th1, q1a);
      th2 = actual(p.alpha, th2, q2a);
    }
    if (pl) pl[dst] = p2;
    if (a1) a1[dst] = th1;
    if (a2) a2[dst] = th2;
  }
}

// nodes to caller numbering: u (pending rescale applied), theta_bar, and the
// prices -rho_p sum_k u_k
__global__ void export_nodes_kernel(Params p, int cur, float *u, float *theta, float *price) {
  const DevScalars sc = *p.sc;
  const int T = p.T, N = p.N;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < (long long)N * T;
       i += (long long)gridDim.x * blockDim.x) {
    const int n = (int)(i / T), t = (int)(i % T);
    const size_t ext = (size_t)p.node_perm[n] * T + t;
    double s = 0.0;
    for (int k = 0; k < p.Kp; ++k) {
      const size_t o = nidx(p, k, n, t);
      const float uu = p.U[cur][o];
      if (u) u[(size_t)k * N * T + ext] = (float)(sc.su * uu);
      if (theta)
        theta[(size_t)k * N * T + ext] = (p.alpha != 1.f && !sc.v_fresh)
                                             ? actual(p.alpha, p.THBAR[cur][o], p.THBAR[cur ^ 1][o])
                                             : p.THBAR[cur][o];
      s += uu;
    }
    if (price) price[ext] = (float)(-sc.rho_p * sc.su * s);
  }
}

// device powers in caller order: the actual iterate (relaxed state undone)
__global__ void export_pdev_kernel(Params p, float *out) {
  const DevScalars sc = *p.sc;
  const bool rx = p.alpha != 1.f && !sc.v_fresh;
  const float c = (1.f - p.alpha) / p.alpha;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < (long long)p.S * p.T;
       i += (long long)gridDim.x * blockDim.x)
    out[i] = rx ? fmaf(c, p.DPD[i], p.PD[i]) : p.PD[i];
}

__global__ void begin_kernel(Params p, long long n, int clear_stop) {
  DevScalars sc = *p.sc;
  if (clear_stop) {
    sc.stop = 0;
    if (sc.stalled) {   // a new call after a stall restarts the stall window
      sc.stalled = 0;
      sc.stall_ref = HUGE_VAL;
      sc.stall_it = sc.it;
    }
  }
  sc.it_last = sc.it + n;
  set_iter(p, sc);
  *p.sc = sc;
}

__global__ void begin_batch_kernel(const Params *ps, int n_inst, long long n, int *dirty) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) *dirty = 1;   // instances may have been reset since the last call
  if (i >= n_inst) return;
  DevScalars sc = *ps[i].sc;
  sc.it_last = sc.it + n;
  set_iter(ps[i], sc);
  *ps[i].sc = sc;
}

__global__ void set_scalars_kernel(DevScalars *d, DevScalars sc) { *d = sc; }

__global__ void set_rho_kernel(Params p, double rho) {
  DevScalars s = *p.sc;
  s.su *= s.rho_p / rho;
  s.sv *= s.rho_th / rho;
  s.rho_p = rho;
  s.rho_th = rho;
  set_iter(p, s);
  *p.sc = s;
}

static size_t inner_smem(int T, int warps) { return (size_t)warps * warp_smem_floats(T) * sizeof(float); }

}  // namespace opfk

using namespace opfk;

// blocks of a grid-stride kernel: resident CTAs per SM times the SM count
template <class F>
static int resident_grid(F fn, size_t smem) {
  int dev = 0, sms = 0, nb = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return -1;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, BLOCK, smem) != cudaSuccess || nb < 1) return -1;
  return nb * sms;
}

// shared memory a CTA may take on this device
static size_t max_smem() {
  int dev = 0, m = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&m, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
    return 0;
  return (size_t)m;
}

// let a device kernel take it (the limit is the function's, not a context's:
// always the same value, so that no context lowers another's)
template <class F>
static bool allow_smem(F fn, size_t smem) {
  cudaFuncAttributes a;
  if (cudaFuncGetAttributes(&a, fn) != cudaSuccess) return false;
  if (a.sharedSizeBytes + smem <= 48 * 1024) return true;   // static and dynamic together
  const size_t m = max_smem();
  if (a.sharedSizeBytes + smem > m) return false;
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(m - a.sharedSizeBytes)) ==
         cudaSuccess;
}

int opfk_plan(const Params &p, IterPlan *plan) {
  const bool v4 = (p.T % 4 == 0), v2 = (p.T % 2 == 0);
  // the inner ADMM in registers up to REG_T steps, else in shared memory
  const int ic = inner_chunk(p.T);
  const bool vn = (p.T % NODE_VW == 0);
  const int gn = vn ? resident_grid(node_kernel<NODE_VW, false, false, false>, 0) : resident_grid(node_kernel<1, false, false, false>, 0);
  const int gx = v4 ? resident_grid(xs_kernel<4>, 0) : resident_grid(xs_kernel<1>, 0);
  const int gd = v2 ? resident_grid(dsum_kernel<2>, 0) : resident_grid(dsum_kernel<1>, 0);
  if (gn < 1 || gx < 1 || gd < 1) return -1;
  const long long tvl = p.T / (v4 ? 4 : 1), tvn = p.T / (vn ? NODE_VW : 1);
  const long long nl = (long long)p.Kp * p.L * tvl, nn = (long long)p.Kp * p.N * tvn;
  const long long nx = (long long)p.n_dnode * tvl;
  const int n_inner = inner_units(p);
  plan->line_ipt = nl <= LINE_SHORT ? 1 : LINE_IPT;
  plan->line_grid = (int)((nl + (long long)BLOCK * plan->line_ipt - 1) / ((long long)BLOCK * plan->line_ipt));
  plan->node_grid = (int)std::min<long long>(gn, (nn + BLOCK - 1) / BLOCK);
  plan->inner_c = ic;
  // One device kernel beside the line kernel, or three (averages, inner ADMM,
  // device sums)?  The inner ADMM is latency-bound, one warp per device.  When
  // the line pass is long enough to hide it, few CTAs walking the devices in
  // several rounds leave the line kernel more of the GPU, and the averages and
  // sums, formed once per node, are hidden as well.  Otherwise the devices are
  // the critical path: one launch, every device at once, averages formed where
  // they are used, device sums in the node pass.  The estimates: the line pass
  // moves about 32 bytes per (line, contingency, step) at 6.5 TB/s; a round of
  // devices takes about 5 + 0.08 T microseconds from registers, 0.45 T in
  // shared memory.  At 10k buses, T = 96, K = 50 (3,000 devices), ms per
  // iteration by warps of the inner kernel: 3,000 0.706, 608 0.706, 304 0.698,
  // 200 0.696, 152 0.704, 96 0.851: the fewest whose rounds fit in half the
  // line pass; device sums in the node pass 0.701 against 0.697.  At 2k buses,
  // T = 24, K = 20: three device kernels 31.7 us per iteration, one 25.2.
  const double line_us = (double)p.Kp * p.L * p.T * 32.0 / 6.5e6;
  // warps per CTA: the shared-memory path as many as its staged states leave
  // room for (no shared memory where no device needs it: every CTA of the
  // device kernel would take it, the closed-form ones too, and run one or two
  // to an SM)
  const bool admm = p.n_stor + p.n_ramp > 0;
  const int nw = !ic && admm ? smem_warps(p.T, max_smem()) : DEV_WARPS;
  plan->inner_warps = nw;
  const int one_round = (n_inner + nw - 1) / nw;
  const double round_us = ic ? 5.0 + 0.08 * p.T : 0.45 * p.T;
  const int max_rounds = (int)std::floor((ic ? 0.5 : 0.7) * line_us / round_us);
  const size_t ism = ic || !admm ? 0 : inner_smem(p.T, nw);
  if (!allow_smem(dev_kernel<0>, ism)) return -1;
  plan->inner_smem = ism;
  // Without inner-ADMM devices the chain is averages and closed forms alone,
  // which a line pass of HIDE_US hides (us per iteration with one device
  // kernel / with averages and sums apart, by the line pass's estimate: 2k
  // buses T = 24 K = 20 7.9 us 21.1 / 24.5, 5k T = 24 K = 10 10.4 us 27.7 /
  // 27.7, 3k T = 25 K = 20 12.4 us 64.3 / 56.8, 1k T = 96 K = 20 with three
  // links 15.9 us 39.3 / 42.0, 2k T = 96 K = 10 16.6 us 43.1 / 39.3, 2k T = 252
  // K = 4 19.8 us 59.1 / 49.5).
  plan->fused = !p.slice && (admm ? max_rounds < 2 : line_us < HIDE_US);
  plan->node_lat = plan->fused && nn <= (vn ? (long long)gn * BLOCK / 2 : NODE_LAT_ITEMS1);
  // A small instance without inner-ADMM devices runs on one CTA (small_kernel)
  // where its rounds of 256 line, closed-form and node items are estimated to
  // take less than the kernels' 8.3 us: 30 buses, T = 1, K = 5 8.35 -> 5.1 us,
  // 100 buses, K = 0 8.2 -> 5.9, 20 buses, T = 24, K = 2 8.5 -> 6.6; beyond
  // the limit 60 buses, K = 5 8.3 against 8.0, 100 buses, K = 10 8.6 against 14.6.
  const long long nc = (long long)p.n_cnode * tvl * (v4 ? CLOSED_LANES4 : CLOSED_LANES1);
  auto rounds = [](long long items) { return (double)((items + BLOCK - 1) / BLOCK); };
  plan->small = plan->fused && n_inner == 0 &&
                SMALL_BASE + SMALL_LINE * rounds(nl) + SMALL_CLOSED * rounds(nc) + SMALL_NODE * rounds(nn) <= SMALL_LIMIT;
  plan->xs_grid = plan->dsum_grid = plan->dev_closed = 0;
  plan->dev_inner = one_round;
  if (plan->fused) {
    plan->dev_closed = (int)std::min<long long>(
        4096, ((long long)p.n_cnode * tvl * (v4 ? CLOSED_LANES4 : CLOSED_LANES1) + DEVB - 1) / DEVB);
    return 0;
  }
  if (max_rounds >= 2) plan->dev_inner = (one_round + max_rounds - 1) / max_rounds;
  plan->xs_grid = (int)std::min<long long>(gx, (nx + BLOCK - 1) / BLOCK);
  const long long nd = (long long)p.N * (p.T / (v2 ? 2 : 1));
  plan->dsum_grid = (int)std::min<long long>(gd, (nd + BLOCK - 1) / BLOCK);
  return 0;
}

static int aux_grid(long long work);

static int iteration_enqueue(const Params &p, const IterPlan &plan, void *main_stream, void *aux_stream,
                             void *ev_fork, void *ev_join, bool slice) {
  cudaStream_t sm = (cudaStream_t)main_stream, sa = (cudaStream_t)aux_stream;
  const bool v4 = (p.T % 4 == 0), v2 = (p.T % 2 == 0);
  // The line proxes (aux stream) read only the previous iterate; the node
  // sums (main stream) follow them and the device kernels.
  if (cudaEventRecord((cudaEvent_t)ev_fork, sm) != cudaSuccess) return -1;
  if (cudaStreamWaitEvent(sa, (cudaEvent_t)ev_fork, 0) != cudaSuccess) return -1;
  if (!plan.fused && plan.xs_grid > 0) {
    if (v4) xs_kernel<4><<<plan.xs_grid, BLOCK, 0, sm>>>(p);
    else xs_kernel<1><<<plan.xs_grid, BLOCK, 0, sm>>>(p);
  }
  const int ni = plan.dev_inner, nd = ni + plan.dev_closed;
  const bool avg = plan.fused;
  if (nd > 0) {
#define DEV_LAUNCH(C) case C: dev_kernel<C><<<nd, DEVB, plan.inner_smem, sm>>>(p, ni, avg, plan.inner_warps); break
    static_assert(REG_C == 8, "the chunks launched below");
    switch (plan.inner_c) {
      DEV_LAUNCH(0); DEV_LAUNCH(1); DEV_LAUNCH(2); DEV_LAUNCH(3); DEV_LAUNCH(4);
      DEV_LAUNCH(5); DEV_LAUNCH(6); DEV_LAUNCH(7); DEV_LAUNCH(8);
    }
#undef DEV_LAUNCH
  }
  if (!plan.fused) {
    if (v2) dsum_kernel<2><<<plan.dsum_grid, BLOCK, 0, sm>>>(p);
    else dsum_kernel<1><<<plan.dsum_grid, BLOCK, 0, sm>>>(p);
  }
  if (plan.line_grid > 0) {
    if (v4) line_kernel<4><<<plan.line_grid, BLOCK, 0, sa>>>(p, plan.line_ipt);
    else line_kernel<1><<<plan.line_grid, BLOCK, 0, sa>>>(p, plan.line_ipt);
  }
  if (cudaEventRecord((cudaEvent_t)ev_join, sa) != cudaSuccess) return -1;
  if (cudaStreamWaitEvent(sm, (cudaEvent_t)ev_join, 0) != cudaSuccess) return -1;
  const bool vn = p.T % NODE_VW == 0, rx = p.alpha != 1.f;
  const int g = plan.node_grid;
#define NODE_LAUNCH(RX, ILD, LAT)                                          \
  if (vn) node_kernel<NODE_VW, RX, ILD, LAT><<<g, BLOCK, 0, sm>>>(p);      \
  else node_kernel<1, RX, ILD, LAT><<<g, BLOCK, 0, sm>>>(p)
  if (plan.node_lat) {
    if (rx) { NODE_LAUNCH(true, true, true); }
    else { NODE_LAUNCH(false, true, true); }
  } else if (rx && plan.fused) { NODE_LAUNCH(true, true, false); }
  else if (rx) { NODE_LAUNCH(true, false, false); }
  else if (plan.fused) { NODE_LAUNCH(false, true, false); }
  else { NODE_LAUNCH(false, false, false); }
#undef NODE_LAUNCH
  if (slice) slice_sums_kernel<<<aux_grid((long long)p.n_dnode * p.T), BLOCK, 0, sm>>>(p, 0);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int opfk_iteration_enqueue(const Params &p, const IterPlan &plan, void *main_stream, void *aux_stream,
                           void *ev_fork, void *ev_join) {
  return iteration_enqueue(p, plan, main_stream, aux_stream, ev_fork, ev_join, false);
}

int opfk_slice_local_enqueue(const Params &p, const IterPlan &plan, void *main_stream, void *aux_stream,
                             void *ev_fork, void *ev_join) {
  return iteration_enqueue(p, plan, main_stream, aux_stream, ev_fork, ev_join, true);
}

int opfk_small_launch(const Params &p, int n, void *stream) {
  cudaStream_t s = (cudaStream_t)stream;
  const bool rx = p.alpha != 1.f;
  if (rx) small_kernel<true><<<1, BLOCK, 0, s>>>(p, n);
  else small_kernel<false><<<1, BLOCK, 0, s>>>(p, n);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int opfk_slice_finish_enqueue(const Params &p, void *stream) {
  decide_kernel<<<1, BLOCK, 0, (cudaStream_t)stream>>>(p);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int opfk_slice_prime_launch(const Params &p, void *stream) {
  slice_sums_kernel<<<aux_grid((long long)p.n_dnode * p.T), BLOCK, 0, (cudaStream_t)stream>>>(p, 1);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int opfk_batch_plan(const Params *hp, const IterPlan *plans, int n, const BatchLayout &lay, int *sched_out,
                    long long sched_cap, long long *sched_len, NodeShare *share, BatchPlan *bp) {
  long long len = 0;
  cudaFuncAttributes fa;
  if (cudaFuncGetAttributes(&fa, smem_kernel_b) != cudaSuccess) return -1;
  const size_t smem_max = max_smem() - fa.sharedSizeBytes;
  size_t ism = 0;
  int ic_max = 1;
  auto put = [&](int inst, long long b, long long blocks) -> bool {
    if (sched_out) {
      if (len >= sched_cap) return false;
      int *e = sched_out + 4 * len;
      e[0] = inst;
      e[1] = (int)b;
      e[2] = (int)blocks;
      e[3] = 0;
    }
    ++len;
    return true;
  };
  const int div = std::max(1, lay.div);
  std::vector<long long> nb(n);
  for (int kind = 0; kind < BK_COUNT; ++kind) {
    bp->offset[kind] = (int)len;
    long long most = 0;
    for (int j = 0; j < n; ++j) {
      const int i = lay.order ? lay.order[j] : j;
      const Params &p = hp[i];
      const bool v4 = (p.T % 4 == 0);
      const long long tv4 = p.T / (v4 ? 4 : 1);
      const int n_inner = inner_units(p);
      long long blocks = 0;
      switch (kind) {
        case BK_SMEM: case BK_INNER:
          // by the form that the instance's horizon takes (links alone need none)
          if ((kind == BK_SMEM) == (p.T > BATCH_REG_T && p.n_stor + p.n_ramp > 0)) {
            const int nw = kind == BK_SMEM ? smem_warps(p.T, smem_max) : DEV_WARPS;
            blocks = (n_inner + nw - 1) / nw;
            if (kind == BK_SMEM) ism = std::max(ism, inner_smem(p.T, nw));
            else if (p.n_stor + p.n_ramp > 0) ic_max = std::max(ic_max, inner_chunk(p.T));
          }
          break;
        case BK_CLOSED:
          blocks = ((long long)p.n_cnode * tv4 * (v4 ? CLOSED_LANES4 : CLOSED_LANES1) + DEVB - 1) / DEVB;
          break;
        case BK_LINE4: case BK_LINE1:
          if ((kind == BK_LINE4) == v4 && p.L > 0)
            blocks = ((long long)p.Kp * p.L * tv4 + (long long)BLOCK * LINE_IPT - 1) / ((long long)BLOCK * LINE_IPT);
          break;
      }
      // the devices take any block count: `div` puts more work in each CTA
      if (blocks > 0 && (kind == BK_SMEM || kind == BK_INNER || kind == BK_CLOSED))
        blocks = (blocks + div - 1) / div;
      nb[j] = blocks;
      most = std::max(most, blocks);
    }
    // instances in `order`, each instance's CTAs together or dealt round-robin
    if (lay.interleave) {
      for (long long r = 0; r < most; ++r)
        for (int j = 0; j < n; ++j)
          if (r < nb[j] && !put(lay.order ? lay.order[j] : j, r, nb[j])) return -1;
    } else {
      for (int j = 0; j < n; ++j)
        for (long long r = 0; r < nb[j]; ++r)
          if (!put(lay.order ? lay.order[j] : j, r, nb[j])) return -1;
    }
    bp->count[kind] = (int)(len - bp->offset[kind]);
  }
  bp->inner_c = ic_max;
  bp->inner_smem = ism;
  bp->relax = (n > 0 && hp[0].alpha != 1.f) ? 1 : 0;
  for (int i = 0; i < n; ++i)
    if ((hp[i].alpha != 1.f) != (bp->relax != 0)) return -2;   // one node kernel for every instance
  bp->deal = NodeDeal{};
  bp->deal.n = n;
  bp->deal.slots = bp->relax ? resident_grid(node_kernel_b<true>, 0) : resident_grid(node_kernel_b<false>, 0);
  if (bp->deal.slots < 1) return -1;
  // the shares round down and are at least one each, at most the grid
  long long grids = 0;
  for (int j = 0; j < n; ++j) {
    const int i = lay.order ? lay.order[j] : j;
    const Params &p = hp[i];
    const int tv = p.T % NODE_VW == 0 ? p.T / NODE_VW : p.T;
    if (share) share[j] = NodeShare{i, (unsigned)p.Kp * (unsigned)p.N * (unsigned)tv, plans[i].node_grid, 0};
    grids += plans[i].node_grid;
  }
  bp->deal.cap = (int)std::min<long long>(grids, (long long)bp->deal.slots + n);
  if (!allow_smem(smem_kernel_b, ism)) return -1;
  *sched_len = len;
  return 0;
}

int opfk_batch_enqueue(const Params *d_params, const int *d_sched, const BatchPlan &bp, const Lanes &on) {
  cudaStream_t sm = (cudaStream_t)on.main, sa = (cudaStream_t)on.aux, sd = (cudaStream_t)on.dev;
  if (bp.deal.n == 0) return 0;
  const int4 *sched = reinterpret_cast<const int4 *>(d_sched);
  auto at = [&](int kind) { return sched + bp.offset[kind]; };
  if (cudaEventRecord((cudaEvent_t)on.ev_fork, sm) != cudaSuccess) return -1;
  if (cudaStreamWaitEvent(sa, (cudaEvent_t)on.ev_fork, 0) != cudaSuccess) return -1;
  // the devices first, the longest chains ahead: a graph's first iteration
  // starts its kernels in this order, and line CTAs that fill the GPU hold up
  // the device chain (16 instances of T = 128, calls of 9 steps: 172 -> 140 us
  // per step)
  const int ns = bp.count[BK_SMEM];
  if (ns) {
    if (cudaStreamWaitEvent(sd, (cudaEvent_t)on.ev_fork, 0) != cudaSuccess) return -1;
    smem_kernel_b<<<ns, DEVB, bp.inner_smem, sd>>>(d_params, at(BK_SMEM), (unsigned)bp.inner_smem);
    if (cudaEventRecord((cudaEvent_t)on.ev_dev, sd) != cudaSuccess) return -1;
  }
  static_assert(BK_CLOSED == BK_INNER + 1, "one launch over both parts of the schedule");
  const int ni = bp.count[BK_INNER], nd = ni + bp.count[BK_CLOSED], gd = std::max(nd, 1);
  const int4 *si = at(BK_INNER);
  switch (bp.inner_c) {
    case 1: dev_kernel_b<1><<<gd, DEVB, 0, sm>>>(d_params, si, ni, nd, bp.deal); break;
    case 2: dev_kernel_b<2><<<gd, DEVB, 0, sm>>>(d_params, si, ni, nd, bp.deal); break;
    case 3: dev_kernel_b<3><<<gd, DEVB, 0, sm>>>(d_params, si, ni, nd, bp.deal); break;
    default: dev_kernel_b<4><<<gd, DEVB, 0, sm>>>(d_params, si, ni, nd, bp.deal); break;
  }
  static_assert(BATCH_C == 4, "the chunks launched above");
  static_assert(BK_LINE1 == BK_LINE4 + 1, "one launch over both widths' schedules");
  const int l4 = bp.count[BK_LINE4], nl = l4 + bp.count[BK_LINE1];
  if (nl) line_kernel_b<<<nl, BLOCK, 0, sa>>>(d_params, at(BK_LINE4), l4);
  if (cudaEventRecord((cudaEvent_t)on.ev_join, sa) != cudaSuccess) return -1;
  if (cudaStreamWaitEvent(sm, (cudaEvent_t)on.ev_join, 0) != cudaSuccess) return -1;
  if (ns && cudaStreamWaitEvent(sm, (cudaEvent_t)on.ev_dev, 0) != cudaSuccess) return -1;
  if (bp.relax) node_kernel_b<true><<<bp.deal.cap, BLOCK, 0, sm>>>(d_params, bp.deal.slot, bp.deal.dirty);
  else node_kernel_b<false><<<bp.deal.cap, BLOCK, 0, sm>>>(d_params, bp.deal.slot, bp.deal.dirty);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

static int aux_grid(long long work) {
  long long g = (work + 255) / 256;
  if (g > 4096) g = 4096;
  if (g < 1) g = 1;
  return (int)g;
}

int opfk_import_launch(const Params &p, int cur, const float *pl, const float *a1, const float *a2,
                       const float *v1, const float *v2, const float *u, void *stream) {
  const long long work = (long long)p.Kp * (p.L + p.N) * p.T;
  import_kernel<<<aux_grid(work), 256, 0, (cudaStream_t)stream>>>(p, cur, pl, a1, a2, v1, v2, u);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int opfk_start_from_nodes_launch(const Params &p, int cur, const float *rows, int stride, float price_scale,
                                 float u_scale, void *stream) {
  start_from_nodes_kernel<<<aux_grid((long long)p.Kp * (p.L + p.N) * p.T), 256, 0, (cudaStream_t)stream>>>(
      p, cur, rows, stride, price_scale, u_scale);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int opfk_inner_export_launch(const Params &p, float *out, long long n, void *stream) {
  inner_export_kernel<<<aux_grid(n), 256, 0, (cudaStream_t)stream>>>(p, out, n);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int opfk_inner_import_launch(const Params &p, const float *in, long long n, float rho, void *stream) {
  inner_import_kernel<<<aux_grid(n), 256, 0, (cudaStream_t)stream>>>(p, in, n, rho);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int opfk_node_average_launch(const Params &p, int cur, void *stream) {
  node_average_kernel<<<aux_grid((long long)p.N * p.T), 256, 0, (cudaStream_t)stream>>>(p, cur);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int opfk_project_v_launch(const Params &p, int cur, void *stream) {
  project_v_kernel<<<aux_grid((long long)p.Kp * p.N * p.T), 256, 0, (cudaStream_t)stream>>>(p, cur);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int opfk_export_lines_launch(const Params &p, int cur, float *pl, float *a1, float *a2, float *v1,
                             float *v2, void *stream) {
  export_lines_kernel<<<aux_grid((long long)p.Kp * p.L * p.T), 256, 0, (cudaStream_t)stream>>>(
      p, cur, pl, a1, a2, v1, v2);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int opfk_begin_launch(const Params &p, long long n, int clear_stop, void *stream) {
  begin_kernel<<<1, 1, 0, (cudaStream_t)stream>>>(p, n, clear_stop);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int opfk_begin_batch_launch(const Params *d_params, const BatchPlan &bp, int n_inst, long long n, void *stream) {
  begin_batch_kernel<<<(n_inst + 255) / 256, 256, 0, (cudaStream_t)stream>>>(d_params, n_inst, n, bp.deal.dirty);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int opfk_export_pdev_launch(const Params &p, float *out, void *stream) {
  export_pdev_kernel<<<aux_grid((long long)p.S * p.T), 256, 0, (cudaStream_t)stream>>>(p, out);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int opfk_export_nodes_launch(const Params &p, int cur, float *u, float *theta, float *price,
                             void *stream) {
  export_nodes_kernel<<<aux_grid((long long)p.N * p.T), 256, 0, (cudaStream_t)stream>>>(p, cur, u, theta,
                                                                                         price);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int opfk_set_scalars_launch(const Params &p, const DevScalars &sc, void *stream) {
  set_scalars_kernel<<<1, 1, 0, (cudaStream_t)stream>>>(p.sc, sc);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int opfk_set_rho_launch(const Params &p, double rho, void *stream) {
  set_rho_kernel<<<1, 1, 0, (cudaStream_t)stream>>>(p, rho);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}
