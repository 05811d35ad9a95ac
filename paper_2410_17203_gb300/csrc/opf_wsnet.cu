// Learned warm-start network (include/opf_wsnet.h): forward pass, backward
// pass and Adam for a three-layer message-passing network over the bus graph.
// The paper has no counterpart; the network only proposes a starting point
// for the message-passing iteration.
//
// Layout: activations are row-major [R][64] with rows r = t * N + n.  A layer
// is one kernel: persistent CTAs hold the layer's bfloat16 weights in shared
// memory and walk tiles of 64 rows; the neighbour average (a CSR
// gather) is formed tile by tile where it is used, in the forward pass from
// the layer's input, in the backward pass, transposed, from the previous
// layer's product.  Every output is summed over k in order in FP32.  Weight
// gradients are partial sums over fixed row ranges, each over its rows in
// order, reduced in a fixed order, so results are deterministic.  The relu
// mask is the sign of the kept output.
//
// A training pass over 48,000 rows (2k buses, T = 24) moves about 0.35 GB and
// does 7.3 GFLOP outside the tensor cores (the FP32 activations keep their
// precision), 0.1 ms of the FP32 pipes.  Its layer kernels are bound by neither
// pipes nor memory: they issue in half of their cycles (12 warps per SM), the
// rest waits for the gather of a tile's rows, which does not overlap its
// products, and 750 tiles on 608 CTAs leave the second round mostly empty.  As
// fifty launches (averages, layers, relu masks and each weight gradient apart)
// a pass took 0.97 ms, as sixteen (weight gradients beside the chain of layers)
// 0.37 ms.  Device memory: about 4.2 KB per row (fifteen arrays of 64 floats,
// and per 256 rows a partial sum of every parameter).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "opf_internal.h"
#include "opf_wsnet.h"

namespace {

constexpr int HID = OPF_WSNET_HIDDEN;
constexpr int NOUT = OPF_WSNET_OUT;
constexpr int NMP = 3;         // message-passing layers
constexpr int TB = 256;        // threads per CTA of the element-wise kernels
constexpr int LB = 128;        // threads per CTA of the layer kernels
constexpr int TR = 64;         // rows per tile of the layer kernels
constexpr int RT = 8;          // ... and of a thread's block there (RT rows x 4 columns)
constexpr int AS = HID + 4;    // row stride of a tile in shared memory (16-byte rows on shifting banks)
constexpr int GRAD_ROWS = 256; // rows per partial sum of the weight gradients
constexpr int GB = 64;         // threads per CTA of the weight-gradient kernel
constexpr int GK = 32;         // weight rows (k) per CTA there
constexpr int GS = 32;         // activation rows staged together there

// Neighbours of a node: the first four (-1 = none) and their weights, the
// rest at ptr[n] + 4 .. ptr[n + 1] of the CSR arrays.
struct Graph {
  const int *ptr, *nbr;
  const float *w;      // A's weights, or A^T's
  const int4 *nbr4;
  const float4 *w4;
  int N;
};

__device__ __forceinline__ float4 fma4(float a, const float4 &x, const float4 &s) {
  return make_float4(fmaf(a, x.x, s.x), fmaf(a, x.y, s.y), fmaf(a, x.z, s.z), fmaf(a, x.w, s.w));
}

// sum_j w[j] in[t, nbr[j]][4 c4 ..] over row r's neighbours, in CSR order;
// the first four rows are requested together
__device__ __forceinline__ float4 gather4(const Graph &g, const float *__restrict__ in, int r, int c4) {
  const int t = r / g.N, n = r - t * g.N;
  const int4 nb = g.nbr4[n];
  const float4 w = g.w4[n];
  const float *base = in + (size_t)t * g.N * HID + 4 * c4;
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  auto row = [&](int j) { return *reinterpret_cast<const float4 *>(base + (size_t)j * HID); };
  const float4 x0 = nb.x >= 0 ? row(nb.x) : z, x1 = nb.y >= 0 ? row(nb.y) : z;
  const float4 x2 = nb.z >= 0 ? row(nb.z) : z, x3 = nb.w >= 0 ? row(nb.w) : z;
  float4 s = z;
  if (nb.x >= 0) s = fma4(w.x, x0, s);
  if (nb.y >= 0) s = fma4(w.y, x1, s);
  if (nb.z >= 0) s = fma4(w.z, x2, s);
  if (nb.w >= 0) {
    s = fma4(w.w, x3, s);
    for (int j = g.ptr[n] + 4; j < g.ptr[n + 1]; ++j) s = fma4(g.w[j], row(g.nbr[j]), s);
  }
  return s;
}

// a layer's bfloat16 weights [64][64] into shared memory, ws[k][j] = W[k][j],
// or W[j][k] with TRANS
// (16-byte reads, all of a thread's in flight: a CTA walks few tiles, so this
// is on its path)
template <bool TRANS>
__device__ __forceinline__ void stage_weights(__nv_bfloat16 *ws, const __nv_bfloat16 *__restrict__ W) {
  constexpr int NQ = HID * HID / 8 / LB;
  uint4 v[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) v[q] = reinterpret_cast<const uint4 *>(W)[threadIdx.x + q * LB];
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int i = threadIdx.x + q * LB;
    if constexpr (!TRANS) {
      reinterpret_cast<uint4 *>(ws)[i] = v[q];
    } else {
      const int j = i / (HID / 8), k = 8 * (i % (HID / 8));
      const unsigned x[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
      for (int e = 0; e < 8; ++e)
        reinterpret_cast<unsigned short *>(ws)[(k + e) * HID + j] = (unsigned short)(x[e >> 1] >> (16 * (e & 1)));
    }
  }
}

// four bfloat16 weights as FP32 (their bits are the upper half of the float's)
__device__ __forceinline__ float4 weights4(const __nv_bfloat16 *p) {
  const uint2 v = *reinterpret_cast<const uint2 *>(p);
  return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                     __uint_as_float(v.y & 0xffff0000u));
}

// acc[i][c] += sum_k at[RT ty + i][k] ws[k][4 tx + c], k in order.  Within the
// products shared memory is the limit, not the FP32 pipes: rows are read four k at a time
// (one 16-byte read serves 16 lanes), weights as bfloat16 (a warp's 16 columns
// groups are one 128-byte wavefront), and eight rows share a weight, so that
// four k are 12 wavefronts for 128 products per lane (FP32 weights and 4 x 4
// blocks: 24).  A layer of 48,000 rows takes 37 us, 10 of them products; the
// rest is the gather of its tiles and the last, partly filled round of tiles.
__device__ __forceinline__ void tile_mma(float (&acc)[RT][4], const float *__restrict__ at,
                                         const __nv_bfloat16 *__restrict__ ws, int tx, int ty) {
#pragma unroll 2
  for (int k = 0; k < HID; k += 4) {
    float a[RT][4];
#pragma unroll
    for (int i = 0; i < RT; ++i) {
      const float4 v = *reinterpret_cast<const float4 *>(at + (RT * ty + i) * AS + k);
      a[i][0] = v.x; a[i][1] = v.y; a[i][2] = v.z; a[i][3] = v.w;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 w = weights4(ws + (k + q) * HID + 4 * tx);
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        acc[i][0] = fmaf(a[i][q], w.x, acc[i][0]);
        acc[i][1] = fmaf(a[i][q], w.y, acc[i][1]);
        acc[i][2] = fmaf(a[i][q], w.z, acc[i][2]);
        acc[i][3] = fmaf(a[i][q], w.w, acc[i][3]);
      }
    }
  }
}

template <int M>
__device__ __forceinline__ void zero_acc(float (&acc)[M][4]) {
#pragma unroll
  for (int i = 0; i < M; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[i][c] = 0.f;
}

__device__ __forceinline__ float4 relu4(const float4 &v) {
  return make_float4(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f), fmaxf(v.z, 0.f), fmaxf(v.w, 0.f));
}

// H0 = relu(X W0 + b0), X [R][K], K <= 64
__global__ void __launch_bounds__(LB) input_kernel(const float *__restrict__ x, const __nv_bfloat16 *__restrict__ W,
                                                   const float *__restrict__ bias, float *__restrict__ out, int R,
                                                   int K) {
  __shared__ __align__(16) float at[TR * AS];
  __shared__ __align__(16) __nv_bfloat16 ws[HID * HID];
  for (int i = threadIdx.x; i < K * HID; i += LB) ws[i] = W[i];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const float4 b4 = *reinterpret_cast<const float4 *>(bias + 4 * tx);
  for (int r0 = blockIdx.x * TR; r0 < R; r0 += gridDim.x * TR) {
    const int nr = min(TR, R - r0);
    __syncthreads();
    for (int i = threadIdx.x; i < TR * K; i += LB) {   // a tile's rows are one run
      const int rr = i / K;
      at[rr * AS + i - rr * K] = rr < nr ? x[(size_t)r0 * K + i] : 0.f;
    }
    __syncthreads();
    float acc[RT][4];
    zero_acc(acc);
    for (int k = 0; k < K; ++k) {
      const float4 w = weights4(ws + k * HID + 4 * tx);
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        const float a = at[(RT * ty + i) * AS + k];
        acc[i][0] = fmaf(a, w.x, acc[i][0]);
        acc[i][1] = fmaf(a, w.y, acc[i][1]);
        acc[i][2] = fmaf(a, w.z, acc[i][2]);
        acc[i][3] = fmaf(a, w.w, acc[i][3]);
      }
    }
#pragma unroll
    for (int i = 0; i < RT; ++i) {
      const int rr = RT * ty + i;
      if (rr >= nr) break;
      *reinterpret_cast<float4 *>(out + (size_t)(r0 + rr) * HID + 4 * tx) =
          relu4(make_float4(acc[i][0] + b4.x, acc[i][1] + b4.y, acc[i][2] + b4.z, acc[i][3] + b4.w));
    }
  }
}

// One message-passing layer: M = A H (kept where m is not NULL), H' = relu(H
// Ws + M Wn + b).  LAST: also Y = H' Wo + bo; H' is kept where out is not NULL.
// Dynamic shared memory: LAYER_SMEM.
constexpr size_t LAYER_SMEM = 2 * HID * HID * sizeof(__nv_bfloat16) + 2 * TR * AS * sizeof(float);
template <bool LAST>
__global__ void __launch_bounds__(LB, 512 / LB) layer_kernel(Graph g, const float *__restrict__ h,
                                                      const __nv_bfloat16 *__restrict__ Ws,
                                                      const __nv_bfloat16 *__restrict__ Wn,
                                                      const float *__restrict__ bias, float *__restrict__ m,
                                                      float *__restrict__ out, const __nv_bfloat16 *__restrict__ Wo,
                                                      const float *__restrict__ bo, float *__restrict__ y, int R) {
  extern __shared__ __align__(16) float sm[];
  __shared__ float wo[LAST ? HID * NOUT : 1];
  float *at = sm, *am = at + TR * AS;
  __nv_bfloat16 *ws = reinterpret_cast<__nv_bfloat16 *>(am + TR * AS), *wn = ws + HID * HID;
  stage_weights<false>(ws, Ws);
  stage_weights<false>(wn, Wn);
  if constexpr (LAST)
    for (int i = threadIdx.x; i < HID * NOUT; i += LB) wo[i] = __bfloat162float(Wo[i]);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const float4 b4 = *reinterpret_cast<const float4 *>(bias + 4 * tx), z = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int r0 = blockIdx.x * TR; r0 < R; r0 += gridDim.x * TR) {
    __syncthreads();
#pragma unroll 2
    for (int q = 0; q < TR / (LB / 16); ++q) {   // 16 threads a row
      const int rr = ty + (LB / 16) * q, r = r0 + rr;
      const bool in = r < R;
      const size_t o = (size_t)r * HID + 4 * tx;
      const float4 v = in ? *reinterpret_cast<const float4 *>(h + o) : z;
      const float4 a = in ? gather4(g, h, r, tx) : z;
      *reinterpret_cast<float4 *>(at + rr * AS + 4 * tx) = v;
      *reinterpret_cast<float4 *>(am + rr * AS + 4 * tx) = a;
      if (m && in) *reinterpret_cast<float4 *>(m + o) = a;
    }
    __syncthreads();
    float acc[RT][4];
    zero_acc(acc);
    tile_mma(acc, at, ws, tx, ty);
    tile_mma(acc, am, wn, tx, ty);
    if constexpr (LAST) __syncthreads();   // at takes the output rows
#pragma unroll
    for (int i = 0; i < RT; ++i) {
      const int rr = RT * ty + i, r = r0 + rr;
      const float4 v = relu4(make_float4(acc[i][0] + b4.x, acc[i][1] + b4.y, acc[i][2] + b4.z, acc[i][3] + b4.w));
      if (out && r < R) *reinterpret_cast<float4 *>(out + (size_t)r * HID + 4 * tx) = v;
      if constexpr (LAST) *reinterpret_cast<float4 *>(at + rr * AS + 4 * tx) = v;
    }
    if constexpr (LAST) {
      __syncthreads();
      static_assert(LB == TR * NOUT, "a thread per output of the tile");
      const int rr = threadIdx.x / NOUT, j = threadIdx.x % NOUT, r = r0 + rr;
      if (r < R) {
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < HID; k += 4) {
          const float4 v = *reinterpret_cast<const float4 *>(at + rr * AS + k);
          s = fmaf(v.x, wo[k * NOUT + j], s);
          s = fmaf(v.y, wo[(k + 1) * NOUT + j], s);
          s = fmaf(v.z, wo[(k + 2) * NOUT + j], s);
          s = fmaf(v.w, wo[(k + 3) * NOUT + j], s);
        }
        y[(size_t)r * NOUT + j] = s + bo[j];
      }
    }
  }
}

// One layer backwards: the adjoint of its output H' -- dY Wo^T (FIRST), else
// dS + A^T dM of the layer above -- masked where H' > 0 into dZ, and, unless
// dm is NULL (the input layer), dM = dZ Wn^T and dS = dZ Ws^T for the layer
// below.  Dynamic shared memory: BACK_SMEM.
constexpr size_t BACK_SMEM = 2 * HID * HID * sizeof(__nv_bfloat16) + TR * AS * sizeof(float);
template <bool FIRST>
__global__ void __launch_bounds__(LB, 512 / LB) back_kernel(Graph g, const float *__restrict__ dy,
                                                     const __nv_bfloat16 *__restrict__ Wo,
                                                     const float *__restrict__ ds_up, const float *__restrict__ dm_up,
                                                     const float *__restrict__ h, const __nv_bfloat16 *__restrict__ Ws,
                                                     const __nv_bfloat16 *__restrict__ Wn, float *__restrict__ dz,
                                                     float *__restrict__ dm, float *__restrict__ ds, int R) {
  extern __shared__ __align__(16) float sm[];
  float *at = sm;
  __nv_bfloat16 *ws = reinterpret_cast<__nv_bfloat16 *>(at + TR * AS), *wn = ws + HID * HID;
  if (dm) {
    stage_weights<true>(ws, Ws);
    stage_weights<true>(wn, Wn);
  }
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  float wo[4][NOUT];
  if constexpr (FIRST) {
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int j = 0; j < NOUT; ++j) wo[c][j] = __bfloat162float(Wo[(4 * tx + c) * NOUT + j]);
  }
  for (int r0 = blockIdx.x * TR; r0 < R; r0 += gridDim.x * TR) {
    __syncthreads();
#pragma unroll 2
    for (int q = 0; q < TR / (LB / 16); ++q) {
      const int rr = ty + (LB / 16) * q, r = r0 + rr;
      const size_t o = (size_t)r * HID + 4 * tx;
      float4 d = z;
      if (r < R) {
        const float4 hv = *reinterpret_cast<const float4 *>(h + o);
        if constexpr (FIRST) {
          const float2 e = *reinterpret_cast<const float2 *>(dy + (size_t)r * NOUT);
          d = make_float4(fmaf(e.y, wo[0][1], e.x * wo[0][0]), fmaf(e.y, wo[1][1], e.x * wo[1][0]),
                          fmaf(e.y, wo[2][1], e.x * wo[2][0]), fmaf(e.y, wo[3][1], e.x * wo[3][0]));
        } else {
          const float4 sv = *reinterpret_cast<const float4 *>(ds_up + o), a = gather4(g, dm_up, r, tx);
          d = make_float4(sv.x + a.x, sv.y + a.y, sv.z + a.z, sv.w + a.w);
        }
        if (!(hv.x > 0.f)) d.x = 0.f;
        if (!(hv.y > 0.f)) d.y = 0.f;
        if (!(hv.z > 0.f)) d.z = 0.f;
        if (!(hv.w > 0.f)) d.w = 0.f;
        *reinterpret_cast<float4 *>(dz + o) = d;
      }
      if (dm) *reinterpret_cast<float4 *>(at + rr * AS + 4 * tx) = d;
    }
    if (!dm) continue;
    __syncthreads();
    float acc[RT][4];
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
      zero_acc(acc);
      tile_mma(acc, at, pass ? ws : wn, tx, ty);
      float *o = pass ? ds : dm;
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        const int r = r0 + RT * ty + i;
        if (r < R)
          *reinterpret_cast<float4 *>(o + (size_t)r * HID + 4 * tx) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
      }
    }
  }
}

// Partial weight gradients over rows GRAD_ROWS blockIdx.x ..: part[k][j] =
// sum over the rows in order of a[r][k] g[r][j], a [R][K] and g [R][64].
// blockIdx.y: up to two such products over the same g (a0 into column p0 of
// the partial's parameter vector, then a1 into p1), GK values of k each; the
// first also sums g itself (pb, the bias).  VEC: a's rows are 64 floats on
// 16-byte boundaries (the network's own arrays; the caller's features need
// not be), and the next rows are requested before the current ones are used.
// A thread keeps an 8 x 4 block in registers (32 products per three 16-byte
// shared-memory reads); splitting k over CTAs fills the SMs (one CTA per row
// range left the second wave nearly empty: 32 us a product, now 26 for two).
template <bool VEC>
__global__ void __launch_bounds__(GB) wgrad_kernel(const float *__restrict__ a0, const float *__restrict__ a1,
                                                   const float *__restrict__ g, float *__restrict__ part, int R, int K,
                                                   long long C, long long p0, long long p1, long long pb) {
  __shared__ __align__(16) float at[GS * GK], gt[GS * HID];
  constexpr int NG = GS * HID / 4 / GB, NA = GS * GK / 4 / GB, AQ = GK / 4;
  const int nk = (K + GK - 1) / GK, second = blockIdx.y >= nk, k0 = (blockIdx.y - (second ? nk : 0)) * GK;
  const float *a = second ? a1 : a0;
  float *out = part + (size_t)blockIdx.x * C;
  const int r0 = blockIdx.x * GRAD_ROWS, r1 = min(R, r0 + GRAD_ROWS);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;   // j = 4 tx .., k = k0 + 8 ty ..
  const bool bias = blockIdx.y == 0 && ty == 0;
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  float acc[RT][4], ab[4] = {0.f, 0.f, 0.f, 0.f};
  zero_acc(acc);
  float4 vg[NG], va[NA];
  auto load = [&](int rb) {   // rows rb .. rb + GS - 1 (0 beyond r1)
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      const int i = threadIdx.x + q * GB, r = rb + i / (HID / 4);
      vg[q] = r < r1 ? *reinterpret_cast<const float4 *>(g + (size_t)r * HID + 4 * (i % (HID / 4))) : z;
    }
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int i = threadIdx.x + q * GB, r = rb + i / AQ, k = k0 + 4 * (i % AQ);
      if constexpr (VEC) {
        va[q] = r < r1 ? *reinterpret_cast<const float4 *>(a + (size_t)r * HID + k) : z;
      } else {
        const float *x = a + (size_t)r * K + k;
        va[q] = make_float4(r < r1 && k < K ? x[0] : 0.f, r < r1 && k + 1 < K ? x[1] : 0.f,
                            r < r1 && k + 2 < K ? x[2] : 0.f, r < r1 && k + 3 < K ? x[3] : 0.f);
      }
    }
  };
  load(r0);
  for (int rb = r0; rb < r1; rb += GS) {
    const int nr = min(GS, r1 - rb);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NG; ++q) reinterpret_cast<float4 *>(gt)[threadIdx.x + q * GB] = vg[q];
#pragma unroll
    for (int q = 0; q < NA; ++q) reinterpret_cast<float4 *>(at)[threadIdx.x + q * GB] = va[q];
    __syncthreads();
    if (rb + GS < r1) load(rb + GS);
#pragma unroll 4
    for (int rr = 0; rr < nr; ++rr) {
      const float4 x = *reinterpret_cast<const float4 *>(at + rr * GK + RT * ty);
      const float4 y = *reinterpret_cast<const float4 *>(at + rr * GK + RT * ty + 4);
      const float4 g4 = *reinterpret_cast<const float4 *>(gt + rr * HID + 4 * tx);
      const float av[RT] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w}, gv[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
      for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[i][c] = fmaf(av[i], gv[c], acc[i][c]);
      if (bias)
#pragma unroll
        for (int c = 0; c < 4; ++c) ab[c] += gv[c];
    }
  }
  float *w = out + (second ? p1 : p0);
#pragma unroll
  for (int i = 0; i < RT; ++i) {
    const int k = k0 + RT * ty + i;
    if (k >= K) break;
#pragma unroll
    for (int c = 0; c < 4; ++c) w[(size_t)k * HID + 4 * tx + c] = acc[i][c];
  }
  if (bias)
#pragma unroll
    for (int c = 0; c < 4; ++c) out[pb + 4 * tx + c] = ab[c];
}

// the same for the output layer: dWo = H^T dY [64][2] and dbo
constexpr int OB = HID * NOUT;
__global__ void __launch_bounds__(OB) wgrad_out_kernel(const float *__restrict__ h, const float *__restrict__ dy,
                                                       float *__restrict__ part, int R, long long C, long long pw,
                                                       long long pb) {
  __shared__ __align__(16) float ht[2 * GS * HID], gt[2 * GS * NOUT];
  constexpr int ST = 2 * GS;
  const int r0 = blockIdx.x * GRAD_ROWS, r1 = min(R, r0 + GRAD_ROWS);
  const int k = threadIdx.x / NOUT, j = threadIdx.x % NOUT;
  float s = 0.f, b = 0.f;
  for (int rb = r0; rb < r1; rb += ST) {
    const int nr = min(ST, r1 - rb);
    __syncthreads();
    float4 v[ST * HID / 4 / OB];
#pragma unroll
    for (int q = 0; q < ST * HID / 4 / OB; ++q) {   // all requested together
      const int i = threadIdx.x + q * OB;
      if (i < nr * (HID / 4)) v[q] = reinterpret_cast<const float4 *>(h + (size_t)rb * HID)[i];
    }
    static_assert(ST * NOUT == OB, "one value of dY per thread");
    if (threadIdx.x < nr * NOUT) gt[threadIdx.x] = dy[(size_t)rb * NOUT + threadIdx.x];
#pragma unroll
    for (int q = 0; q < ST * HID / 4 / OB; ++q) {
      const int i = threadIdx.x + q * OB;
      if (i < nr * (HID / 4)) reinterpret_cast<float4 *>(ht)[i] = v[q];
    }
    __syncthreads();
#pragma unroll 8
    for (int rr = 0; rr < nr; ++rr) {
      const float gv = gt[rr * NOUT + j];
      s = fmaf(ht[rr * HID + k], gv, s);
      b += gv;
    }
  }
  float *out = part + (size_t)blockIdx.x * C;
  out[pw + k * NOUT + j] = s;
  if (k == 0) out[pb + j] = b;
}

// The partial sums reduced in order, grad[o] = sum over c of part[c][o], and
// with ADAM the step on the FP32 parameters and their bfloat16 copy
constexpr int GC = 48;
template <bool ADAM>
__global__ void __launch_bounds__(GB) grad_kernel(const float *__restrict__ part, float *__restrict__ grad, int n_part,
                                                  long long n, float *p, float *m, float *v, __nv_bfloat16 *pb,
                                                  float lr, float bc1, float bc2) {
  const long long i = (long long)blockIdx.x * GB + threadIdx.x;
  if (i >= n) return;
  float s = 0.f;
  for (int c0 = 0; c0 < n_part; c0 += GC) {   // GC values in flight, added in order
    float x[GC];
#pragma unroll
    for (int q = 0; q < GC; ++q) x[q] = c0 + q < n_part ? part[(size_t)(c0 + q) * n + i] : 0.f;
#pragma unroll
    for (int q = 0; q < GC; ++q)
      if (c0 + q < n_part) s += x[q];
  }
  grad[i] = s;
  if constexpr (ADAM) {
    const float mi = 0.9f * m[i] + 0.1f * s;
    const float vi = 0.999f * v[i] + 0.001f * s * s;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / bc1) / (sqrtf(vi / bc2) + 1e-8f);
    p[i] = pi;
    pb[i] = __float2bfloat16_rn(pi);
  }
}

// dY = 2 scale (Y - Y*) / R; per-CTA partial loss sums (FP64)
__global__ void __launch_bounds__(TB) loss_kernel(const float *__restrict__ y, const float *__restrict__ yt,
                                                  float *__restrict__ dy, double *__restrict__ lpart, int R,
                                                  float c0, float c1) {
  __shared__ double red[TB];
  double s = 0.0;
  const size_t n = (size_t)R * NOUT;
  for (size_t i = (size_t)blockIdx.x * TB + threadIdx.x; i < n; i += (size_t)gridDim.x * TB) {
    const float c = (i & 1) ? c1 : c0;
    const float d = y[i] - yt[i];
    dy[i] = 2.f * c * d / (float)R;
    s += (double)c * d * d;
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = TB / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) lpart[blockIdx.x] = red[0];
}

__global__ void __launch_bounds__(TB) to_bf16_kernel(const float *__restrict__ p, __nv_bfloat16 *pb, long long n) {
  for (long long i = (long long)blockIdx.x * TB + threadIdx.x; i < n; i += (long long)gridDim.x * TB)
    pb[i] = __float2bfloat16_rn(p[i]);
}

int grid_for(size_t work) { return (int)std::min<size_t>((work + TB - 1) / TB, 4096); }

}  // namespace

struct opf_wsnet {
  int N = 0, T = 0, F = 0, R = 0;
  cudaStream_t stream = nullptr;
  // the weight gradients run here, each beside the layers below it
  cudaStream_t aux = nullptr;
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
  long long C = 0;  // parameters
  long long oW0 = 0, ob0 = 0, oWs[NMP] = {}, oWn[NMP] = {}, ob[NMP] = {}, oWo = 0, obo = 0;
  int step = 0;
  // device memory
  int *ptr = nullptr, *nbr = nullptr;
  float *wA = nullptr, *wAT = nullptr;
  float *P = nullptr, *G = nullptr, *Mo = nullptr, *Vo = nullptr;
  __nv_bfloat16 *Pb = nullptr;
  int4 *nbr4 = nullptr;
  float4 *wA4 = nullptr, *wAT4 = nullptr;
  float *H0 = nullptr, *M[NMP] = {}, *H[NMP] = {}, *Y = nullptr;
  // dM and dS of a layer, read at the neighbours by the layer below: two of each
  float *dY = nullptr, *dZ[NMP + 1] = {}, *dM[2] = {}, *dS[2] = {}, *part = nullptr;
  double *lpart = nullptr;
  int n_lpart = 0, n_gpart = 0;
  int g_in = 0, g_layer = 0, g_back = 0;   // persistent CTAs of the layer kernels
  std::vector<void *> allocs;
};

namespace {

opf_status wfail(opf_status s, const char *msg) { return (opf_status)opf_record_error((int)s, msg); }

#define WCK(call)                                                        \
  do {                                                                   \
    cudaError_t e_ = (call);                                             \
    if (e_ != cudaSuccess) return wfail(OPF_ECUDA, cudaGetErrorString(e_)); \
  } while (0)

template <class T>
cudaError_t walloc(opf_wsnet *w, T **p, size_t n) {
  const cudaError_t e = cudaMalloc(reinterpret_cast<void **>(p), std::max<size_t>(n, 1) * sizeof(T));
  if (e == cudaSuccess) w->allocs.push_back(*p);
  return e;
}

void wfree(opf_wsnet *w) {
  for (void *p : w->allocs) cudaFree(p);
  w->allocs.clear();
  for (cudaEvent_t ev : {w->ev_fork, w->ev_join})
    if (ev) cudaEventDestroy(ev);
  if (w->aux) cudaStreamDestroy(w->aux);
  w->ev_fork = w->ev_join = nullptr;
  w->aux = nullptr;
}

// He-uniform weights from a counter-based generator (splitmix64), zero biases
void he_init(std::vector<float> &p, const opf_wsnet *w, uint64_t seed) {
  uint64_t x = seed;
  auto next = [&]() {
    x += 0x9E3779B97F4A7C15ull;
    uint64_t z = x;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return (double)(z >> 11) * (1.0 / 9007199254740992.0);
  };
  std::fill(p.begin(), p.end(), 0.f);
  auto fill = [&](long long off, int fan_in, long long n) {
    const double lim = std::sqrt(6.0 / fan_in);
    for (long long i = 0; i < n; ++i) p[off + i] = (float)((2.0 * next() - 1.0) * lim);
  };
  fill(w->oW0, w->F, (long long)w->F * HID);
  for (int l = 0; l < NMP; ++l) {
    fill(w->oWs[l], HID, HID * HID);
    fill(w->oWn[l], HID, HID * HID);
  }
  fill(w->oWo, HID, HID * NOUT);
}

Graph graph(const opf_wsnet *w, bool transposed) {
  return Graph{w->ptr, w->nbr, transposed ? w->wAT : w->wA, w->nbr4, transposed ? w->wAT4 : w->wA4, w->N};
}

// Y (into y); keep: the activations the backward pass reads
void forward(opf_wsnet *w, const float *x, float *y, bool keep) {
  const Graph g = graph(w, false);
  input_kernel<<<w->g_in, LB, 0, w->stream>>>(x, w->Pb + w->oW0, w->P + w->ob0, w->H0, w->R, w->F);
  const float *h = w->H0;
  for (int l = 0; l < NMP; ++l) {
    const bool last = l == NMP - 1;
    const __nv_bfloat16 *Ws = w->Pb + w->oWs[l], *Wn = w->Pb + w->oWn[l];
    const float *b = w->P + w->ob[l];
    float *m = keep ? w->M[l] : nullptr;
    if (last)
      layer_kernel<true><<<w->g_layer, LB, LAYER_SMEM, w->stream>>>(g, h, Ws, Wn, b, m, keep ? w->H[l] : nullptr,
                                                                     w->Pb + w->oWo, w->P + w->obo, y, w->R);
    else
      layer_kernel<false><<<w->g_layer, LB, LAYER_SMEM, w->stream>>>(g, h, Ws, Wn, b, m, w->H[l], nullptr, nullptr,
                                                                      nullptr, w->R);
    h = w->H[l];
  }
}

// Loss partials and the partial weight gradients (grad_kernel finishes them).
// A weight gradient waits only for its layer's dZ: they run on the second
// stream beside the chain of layers (a row range's 256 rows one after another
// are latency, 18 us a launch however few the rows).
cudaError_t backward(opf_wsnet *w, const float *x, const float *yt, const float scale[2]) {
  const int R = w->R;
  const Graph g = graph(w, true);
  auto fork = [&]() {
    const cudaError_t e = cudaEventRecord(w->ev_fork, w->stream);
    return e == cudaSuccess ? cudaStreamWaitEvent(w->aux, w->ev_fork, 0) : e;
  };
  loss_kernel<<<w->n_lpart, TB, 0, w->stream>>>(w->Y, yt, w->dY, w->lpart, R, scale[0], scale[1]);
  cudaError_t e = fork();
  if (e != cudaSuccess) return e;
  wgrad_out_kernel<<<w->n_gpart, OB, 0, w->aux>>>(w->H[NMP - 1], w->dY, w->part, R, w->C, w->oWo, w->obo);
  for (int l = NMP - 1; l >= 0; --l) {   // layer l's dZ is dZ[l + 1]
    const int i = l & 1, up = i ^ 1;
    const __nv_bfloat16 *Ws = w->Pb + w->oWs[l], *Wn = w->Pb + w->oWn[l];
    if (l == NMP - 1)
      back_kernel<true><<<w->g_back, LB, BACK_SMEM, w->stream>>>(g, w->dY, w->Pb + w->oWo, nullptr, nullptr, w->H[l], Ws,
                                                                  Wn, w->dZ[l + 1], w->dM[i], w->dS[i], R);
    else
      back_kernel<false><<<w->g_back, LB, BACK_SMEM, w->stream>>>(g, nullptr, nullptr, w->dS[up], w->dM[up], w->H[l], Ws,
                                                                   Wn, w->dZ[l + 1], w->dM[i], w->dS[i], R);
    if ((e = fork()) != cudaSuccess) return e;
    const dim3 grid(w->n_gpart, 2 * HID / GK);
    wgrad_kernel<true><<<grid, GB, 0, w->aux>>>(l == 0 ? w->H0 : w->H[l - 1], w->M[l], w->dZ[l + 1], w->part, R, HID, w->C,
                                                w->oWs[l], w->oWn[l], w->ob[l]);
  }
  back_kernel<false><<<w->g_back, LB, BACK_SMEM, w->stream>>>(g, nullptr, nullptr, w->dS[0], w->dM[0], w->H0, nullptr,
                                                               nullptr, w->dZ[0], nullptr, nullptr, R);
  const dim3 grid(w->n_gpart, (w->F + GK - 1) / GK);
  wgrad_kernel<false><<<grid, GB, 0, w->stream>>>(x, nullptr, w->dZ[0], w->part, R, w->F, w->C, w->oW0, 0, w->ob0);
  e = cudaEventRecord(w->ev_join, w->aux);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(w->stream, w->ev_join, 0);
  return e == cudaSuccess ? cudaGetLastError() : e;
}

// persistent CTAs of a layer kernel: what is resident, or one per tile
template <class Fn>
cudaError_t layer_grid(Fn fn, size_t smem, int R, int *grid) {
  int dev = 0, sms = 0, nb = 0;
  cudaError_t e = smem > 48 * 1024 ? cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                                   : cudaSuccess;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, LB, smem);
  *grid = std::max(1, std::min((R + TR - 1) / TR, std::max(nb, 1) * sms));
  return e;
}

opf_status read_loss(opf_wsnet *w, double *loss) {
  std::vector<double> lp(w->n_lpart);
  WCK(cudaMemcpyAsync(lp.data(), w->lpart, lp.size() * sizeof(double), cudaMemcpyDeviceToHost, w->stream));
  WCK(cudaStreamSynchronize(w->stream));
  double s = 0.0;
  for (double x : lp) s += x;
  *loss = s / w->R;
  return OPF_OK;
}

}  // namespace

extern "C" {

int64_t opf_wsnet_param_count(int32_t F) {
  return (int64_t)F * HID + HID + NMP * (2 * HID * HID + HID) + HID * NOUT + NOUT;
}

opf_status opf_wsnet_create(int32_t n_nodes, int32_t n_lines, const int32_t *line_from, const int32_t *line_to,
                            const double *line_b, int32_t T, int32_t F, const float *params, uint64_t seed,
                            void *cuda_stream, opf_wsnet **out) {
  if (!out) return wfail(OPF_EINVAL, "out is NULL");
  *out = nullptr;
  if (n_nodes < 1 || n_lines < 0 || T < 1 || F < 1 || F > HID)
    return wfail(OPF_EINVAL, "wsnet: need n_nodes >= 1, n_lines >= 0, T >= 1, 1 <= n_features <= 64");
  if ((long long)n_nodes * T * HID >= (1LL << 31)) return wfail(OPF_EINVAL, "wsnet: too many rows");
  if (n_lines > 0 && (!line_from || !line_to || !line_b)) return wfail(OPF_EINVAL, "wsnet: NULL line array");
  std::vector<double> bsum(n_nodes, 0.0);
  for (int l = 0; l < n_lines; ++l) {
    const int f = line_from[l], t = line_to[l];
    if (f < 0 || f >= n_nodes || t < 0 || t >= n_nodes || f == t || !(line_b[l] > 0) || !std::isfinite(line_b[l]))
      return wfail(OPF_EINVAL, "wsnet: bad line (node id, self loop or susceptance)");
    bsum[f] += line_b[l];
    bsum[t] += line_b[l];
  }
  // neighbour lists by node: weight of A (this end) and of A^T (other end)
  std::vector<int> ptr(n_nodes + 1, 0), nbr(2 * (size_t)n_lines);
  std::vector<float> wa(2 * (size_t)n_lines), wat(2 * (size_t)n_lines);
  for (int l = 0; l < n_lines; ++l) {
    ++ptr[line_from[l] + 1];
    ++ptr[line_to[l] + 1];
  }
  for (int n = 0; n < n_nodes; ++n) ptr[n + 1] += ptr[n];
  std::vector<int> fillp(ptr.begin(), ptr.end() - 1);
  for (int l = 0; l < n_lines; ++l) {
    const int f = line_from[l], t = line_to[l];
    const double wf = line_b[l] / bsum[f], wt = line_b[l] / bsum[t];
    int j = fillp[f]++;
    nbr[j] = t;
    wa[j] = (float)wf;
    wat[j] = (float)wt;
    j = fillp[t]++;
    nbr[j] = f;
    wa[j] = (float)wt;
    wat[j] = (float)wf;
  }
  auto *w = new (std::nothrow) opf_wsnet();
  if (!w) return wfail(OPF_ENOMEM, "host allocation failed");
  w->N = n_nodes;
  w->T = T;
  w->F = F;
  w->R = n_nodes * T;
  w->stream = (cudaStream_t)cuda_stream;
  w->C = opf_wsnet_param_count(F);
  long long o = 0;
  w->oW0 = o; o += (long long)F * HID;
  w->ob0 = o; o += HID;
  for (int l = 0; l < NMP; ++l) {
    w->oWs[l] = o; o += HID * HID;
    w->oWn[l] = o; o += HID * HID;
    w->ob[l] = o; o += HID;
  }
  w->oWo = o; o += HID * NOUT;
  w->obo = o; o += NOUT;
  w->n_lpart = 256;
  w->n_gpart = (w->R + GRAD_ROWS - 1) / GRAD_ROWS;
  const size_t RH = (size_t)w->R * HID;
  cudaError_t e = cudaSuccess;
  auto A = [&](auto **p, size_t n) {
    if (e == cudaSuccess) e = walloc(w, p, n);
  };
  A(&w->ptr, n_nodes + 1);
  A(&w->nbr, nbr.size());
  A(&w->wA, wa.size());
  A(&w->wAT, wat.size());
  A(&w->P, w->C);
  A(&w->G, w->C);
  A(&w->Mo, w->C);
  A(&w->Vo, w->C);
  A(&w->Pb, w->C);
  A(&w->nbr4, n_nodes);
  A(&w->wA4, n_nodes);
  A(&w->wAT4, n_nodes);
  A(&w->H0, RH);
  for (int l = 0; l < NMP; ++l) {
    A(&w->M[l], RH);
    A(&w->H[l], RH);
  }
  A(&w->Y, (size_t)w->R * NOUT);
  A(&w->dY, (size_t)w->R * NOUT);
  for (int l = 0; l <= NMP; ++l) A(&w->dZ[l], RH);
  for (int i = 0; i < 2; ++i) {
    A(&w->dM[i], RH);
    A(&w->dS[i], RH);
  }
  A(&w->part, (size_t)w->n_gpart * w->C);
  A(&w->lpart, w->n_lpart);
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&w->aux, cudaStreamNonBlocking);
  for (cudaEvent_t *ev : {&w->ev_fork, &w->ev_join})
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming);
  int g2 = 0;
  if (e == cudaSuccess) e = layer_grid(input_kernel, 0, w->R, &w->g_in);
  if (e == cudaSuccess) e = layer_grid(layer_kernel<false>, LAYER_SMEM, w->R, &w->g_layer);
  if (e == cudaSuccess) e = layer_grid(layer_kernel<true>, LAYER_SMEM, w->R, &g2);
  w->g_layer = std::min(w->g_layer, g2);
  if (e == cudaSuccess) e = layer_grid(back_kernel<false>, BACK_SMEM, w->R, &w->g_back);
  if (e == cudaSuccess) e = layer_grid(back_kernel<true>, BACK_SMEM, w->R, &g2);
  w->g_back = std::min(w->g_back, g2);
  std::vector<int4> nbr4(n_nodes);
  std::vector<float4> wa4(n_nodes), wat4(n_nodes);
  for (int n = 0; n < n_nodes; ++n) {
    int nb[4] = {-1, -1, -1, -1};
    float u[4] = {0.f, 0.f, 0.f, 0.f}, v[4] = {0.f, 0.f, 0.f, 0.f};
    for (int j = ptr[n], q = 0; j < ptr[n + 1] && q < 4; ++j, ++q) {
      nb[q] = nbr[j];
      u[q] = wa[j];
      v[q] = wat[j];
    }
    nbr4[n] = make_int4(nb[0], nb[1], nb[2], nb[3]);
    wa4[n] = make_float4(u[0], u[1], u[2], u[3]);
    wat4[n] = make_float4(v[0], v[1], v[2], v[3]);
  }
  if (e == cudaSuccess) e = cudaMemcpy(w->nbr4, nbr4.data(), n_nodes * sizeof(int4), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(w->wA4, wa4.data(), n_nodes * sizeof(float4), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(w->wAT4, wat4.data(), n_nodes * sizeof(float4), cudaMemcpyHostToDevice);
  std::vector<float> p0(w->C);
  if (params) std::memcpy(p0.data(), params, w->C * sizeof(float));
  else he_init(p0, w, seed);
  if (e == cudaSuccess) e = cudaMemcpy(w->ptr, ptr.data(), ptr.size() * sizeof(int), cudaMemcpyHostToDevice);
  if (e == cudaSuccess && n_lines > 0) {
    e = cudaMemcpy(w->nbr, nbr.data(), nbr.size() * sizeof(int), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(w->wA, wa.data(), wa.size() * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(w->wAT, wat.data(), wat.size() * sizeof(float), cudaMemcpyHostToDevice);
  }
  if (e == cudaSuccess) e = cudaMemcpy(w->P, p0.data(), w->C * sizeof(float), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(w->Mo, 0, w->C * sizeof(float));
  if (e == cudaSuccess) e = cudaMemset(w->Vo, 0, w->C * sizeof(float));
  if (e == cudaSuccess) {
    to_bf16_kernel<<<grid_for(w->C), TB>>>(w->P, w->Pb, w->C);
    e = cudaDeviceSynchronize();
  }
  if (e != cudaSuccess) {
    const opf_status s = e == cudaErrorMemoryAllocation ? wfail(OPF_ENOMEM, "wsnet: device allocation failed")
                                                        : wfail(OPF_ECUDA, cudaGetErrorString(e));
    wfree(w);
    delete w;
    return s;
  }
  *out = w;
  return OPF_OK;
}

opf_status opf_wsnet_get_params(opf_wsnet *w, float *params) {
  if (!w || !params) return wfail(OPF_EINVAL, "NULL argument");
  WCK(cudaMemcpyAsync(params, w->P, w->C * sizeof(float), cudaMemcpyDeviceToHost, w->stream));
  WCK(cudaStreamSynchronize(w->stream));
  return OPF_OK;
}

opf_status opf_wsnet_set_params(opf_wsnet *w, const float *params) {
  if (!w || !params) return wfail(OPF_EINVAL, "NULL argument");
  WCK(cudaMemcpyAsync(w->P, params, w->C * sizeof(float), cudaMemcpyHostToDevice, w->stream));
  to_bf16_kernel<<<grid_for(w->C), TB, 0, w->stream>>>(w->P, w->Pb, w->C);
  WCK(cudaGetLastError());
  WCK(cudaStreamSynchronize(w->stream));
  return OPF_OK;
}

opf_status opf_wsnet_forward(opf_wsnet *w, const float *x, float *y) {
  if (!w || !x || !y) return wfail(OPF_EINVAL, "NULL argument");
  forward(w, x, y, false);
  WCK(cudaGetLastError());
  return OPF_OK;
}

opf_status opf_wsnet_gradient(opf_wsnet *w, const float *x, const float *yt, const float scale[2], double *loss,
                              float *grad) {
  if (!w || !x || !yt || !scale) return wfail(OPF_EINVAL, "NULL argument");
  forward(w, x, w->Y, true);
  WCK(backward(w, x, yt, scale));
  grad_kernel<false><<<(int)((w->C + GB - 1) / GB), GB, 0, w->stream>>>(w->part, w->G, w->n_gpart, w->C, nullptr, nullptr,
                                                                       nullptr, nullptr, 0.f, 1.f, 1.f);
  WCK(cudaGetLastError());
  if (grad) WCK(cudaMemcpyAsync(grad, w->G, w->C * sizeof(float), cudaMemcpyDeviceToHost, w->stream));
  if (loss) return read_loss(w, loss);
  WCK(cudaStreamSynchronize(w->stream));
  return OPF_OK;
}

opf_status opf_wsnet_train_step(opf_wsnet *w, const float *x, const float *yt, const float scale[2], float lr,
                                double *loss) {
  if (!w || !x || !yt || !scale) return wfail(OPF_EINVAL, "NULL argument");
  if (!(lr > 0.f) || !std::isfinite(lr)) return wfail(OPF_EINVAL, "wsnet: learning rate must be > 0");
  forward(w, x, w->Y, true);
  WCK(backward(w, x, yt, scale));
  ++w->step;
  const float bc1 = 1.f - std::pow(0.9f, (float)w->step), bc2 = 1.f - std::pow(0.999f, (float)w->step);
  grad_kernel<true><<<(int)((w->C + GB - 1) / GB), GB, 0, w->stream>>>(w->part, w->G, w->n_gpart, w->C, w->P, w->Mo, w->Vo,
                                                                      w->Pb, lr, bc1, bc2);
  WCK(cudaGetLastError());
  if (loss) return read_loss(w, loss);
  return OPF_OK;
}

void opf_wsnet_destroy(opf_wsnet *w) {
  if (!w) return;
  cudaStreamSynchronize(w->stream);
  cudaStreamSynchronize(w->aux);
  wfree(w);
  delete w;
}

}  // extern "C"
