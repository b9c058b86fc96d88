// Adjoint (backward) kernels of the reconstruction and of the degradation,
// and the MAP energy of Sec. 4 (Eq. 5, 8, 9): with the neighbour IDs and
// weights held fixed,
//   E(R) = || D B x - y ||^2 + lambda * sum_{4-neighbour patches p,q} ||P_p - P_q||^2_overlap,
//   x = overlap average of the patches P_n = mu_n + sum_m w_nm R[nbr_nm].
// All reductions are deterministic (fixed order, no atomics on values).
#include <math.h>

#include <algorithm>

#include "device_common.cuh"
#include "zoom_internal.h"

namespace {

// P[n][p] = mu_n + sum_m w_nm R[nbr_nm][p], rows of ph2pad values; one thread
// per 4 pixels of a patch (the residual rows are padded alike).
__global__ void __launch_bounds__(256) k_patches(const int32_t* __restrict__ nbr, const float* __restrict__ wgt,
                                                 const float* __restrict__ mu, const float4* __restrict__ hr_res,
                                                 int row4, int K, int64_t nq, float4* __restrict__ P) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nq * row4) return;
  const int64_t n = t / row4;
  const int p = (int)(t - n * row4);
  const float m0 = mu[n];
  float4 v = make_float4(m0, m0, m0, m0);
#pragma unroll 4
  for (int m = 0; m < K; ++m) {
    const float wm = wgt[n * K + m];
    const float4 r = __ldg(hr_res + (int64_t)nbr[n * K + m] * row4 + p);
    v.x = fmaf(wm, r.x, v.x);
    v.y = fmaf(wm, r.y, v.y);
    v.z = fmaf(wm, r.z, v.z);
    v.w = fmaf(wm, r.w, v.w);
  }
  P[t] = v;
}

// 1-D weights of the blur + s-box decimation (see the forward kernels).
struct Wts {
  int n;
  float w[8];
};

// y = D B x (- sub): FP32, separable, clamped.
__global__ void k_degrade(const float* __restrict__ x, int H, int W, int h, int w, int s, Wts wt,
                          const float* __restrict__ sub, float* __restrict__ y) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= h || j >= w) return;
  float acc = 0.f;
  for (int a = 0; a < wt.n; ++a) {
    const int r = zoom_clampi(s * i + a - 1, 0, H - 1);
    float row = 0.f;
    for (int b = 0; b < wt.n; ++b) row = fmaf(wt.w[b], x[(int64_t)r * W + zoom_clampi(s * j + b - 1, 0, W - 1)], row);
    acc = fmaf(wt.w[a], row, acc);
  }
  y[(int64_t)i * w + j] = sub ? acc - sub[(int64_t)i * w + j] : acc;
}

// Weight of HR position X in the window of LR position j: one of the window's
// weights inside, the sum of those that the clamp brings to an edge there.
__device__ __forceinline__ float window_weight(int X, int N, int s, int j, const Wts& wt) {
  if (X > 0 && X < N - 1) {
    const int b = X - s * j + 1;
    return b >= 0 && b < wt.n ? wt.w[b] : 0.f;
  }
  float v = 0.f;
  for (int b = 0; b < wt.n; ++b)
    if (zoom_clampi(s * j + b - 1, 0, N - 1) == X) v += wt.w[b];
  return v;
}

// g = alpha * B^T D^T r in gather form: HR pixel (Y, X) collects, from every
// LR pixel (i, j) whose window reads it (through the clamp), the weights
// W_a(i -> Y) W_b(j -> X) times r(i, j).
__global__ void k_degrade_adjoint(const float* __restrict__ r, int h, int w, int H, int W, int s, Wts wt,
                                  float alpha, float* __restrict__ g) {
  const int X = blockIdx.x * blockDim.x + threadIdx.x;
  const int Y = blockIdx.y * blockDim.y + threadIdx.y;
  if (X >= W || Y >= H) return;
  // LR rows whose window [s*i - 1, s*i + s] (clamped) contains Y
  const int i0 = max(0, (Y - s) / s - 1), i1 = min(h - 1, (Y + 1) / s + 1);
  const int j0 = max(0, (X - s) / s - 1), j1 = min(w - 1, (X + 1) / s + 1);
  float acc = 0.f;
  for (int i = i0; i <= i1; ++i) {
    const float wy = window_weight(Y, H, s, i, wt);
    if (wy == 0.f) continue;
    float row = 0.f;
    for (int j = j0; j <= j1; ++j) row = fmaf(window_weight(X, W, s, j, wt), r[(int64_t)i * w + j], row);
    acc = fmaf(wy, row, acc);
  }
  g[(int64_t)Y * W + X] = alpha * acc;
}

// The patch pixel p = (a, b): a, b and a / s, b / s, a byte each (PH <= 20).
__device__ __forceinline__ uint32_t pixel_code(int p, int PH, int s) {
  const int a = p / PH, b = p - a * PH;
  return (uint32_t)a | ((uint32_t)b << 8) | ((uint32_t)(a / s) << 16) | ((uint32_t)(b / s) << 24);
}
constexpr int kMaxPatchPixels = 400;   // (s P)^2 at s = 4, P = 5

// dE/dP[n][p] = gx(Y, X) / n_cov(Y, X) + lambda * 2 * sum over the 4 LR-grid
// neighbour patches q overlapping pixel p of (P_n - P_q) at that pixel.  A
// warp per patch, lanes over its pixels, rows of ph2pad values (the padding
// is written 0).  Bound by the rows written; with a thread per value, which
// divided for its patch, pixel and counts, 119,691 patches of 15 x 15 took
// 214 us, 87 us so.
__global__ void __launch_bounds__(256) k_patch_grad(const float* __restrict__ gx, const float* __restrict__ P,
                                                    int h, int w, int s, int Pp, int ph2pad, float lambda,
                                                    float* __restrict__ gP) {
  __shared__ uint32_t s_px[kMaxPatchPixels];
  const int PH = s * Pp, ph2 = PH * PH;
  const int nh = h - Pp + 1, nw = w - Pp + 1, W = s * w;
  for (int p = threadIdx.x; p < ph2; p += blockDim.x) s_px[p] = pixel_code(p, PH, s);
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t nq = (int64_t)nh * nw, nwarp = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t n = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); n < nq; n += nwarp) {
    const int i = (int)(n / nw), j = (int)(n - (int64_t)i * nw);
    const float* g0 = gx + (int64_t)(s * i) * W + s * j;
    for (int p = lane; p < ph2pad; p += 32) {
      float g = 0.f;
      if (p < ph2) {
        const uint32_t c = s_px[p];
        const int a = c & 255, b = (c >> 8) & 255, as = (c >> 16) & 255, bs = c >> 24;
        // patches covering HR row Y = s i + a: min(Y / s, nh - 1) down to
        // (Y - PH) / s + 1 (0 where Y < PH); Y / s = i + a / s
        const int ci = min(i + as, nh - 1) - max(0, i + as - Pp + 1) + 1;
        const int cj = min(j + bs, nw - 1) - max(0, j + bs - Pp + 1) + 1;
        g = g0[a * W + b] / (float)(ci * cj);
        if (lambda != 0.f) {   // P is read only for the prior term
          const float* pn = P + n * ph2pad;
          const float pv = pn[p];
          float pr = 0.f;
          if (j + 1 < nw && b >= s) pr += pv - pn[ph2pad + p - s];
          if (j > 0 && b < PH - s) pr += pv - pn[p + s - ph2pad];
          if (i + 1 < nh && a >= s) pr += pv - pn[(int64_t)nw * ph2pad + p - s * PH];
          if (i > 0 && a < PH - s) pr += pv - pn[p + s * PH - (int64_t)nw * ph2pad];
          g = fmaf(2.f * lambda, pr, g);
        }
      }
      gP[n * ph2pad + p] = g;
    }
  }
}

// acc += sum over the uses [u0, u1) of w[u] * gP[u / K], 4 pixels a lane and V
// such groups: the uses' numbers and weights are read 32 at a time, and the
// rows of U uses are in flight together, added in order.
template <int V, int U>
__device__ __forceinline__ void add_uses(int u0, int u1, const int32_t* __restrict__ sorted_use,
                                         const float* __restrict__ wgt, const float4* __restrict__ gP, int K,
                                         int row4, int lane, float4 (&acc)[V]) {
  for (int ub = u0; ub < u1; ub += 32) {
    const int use = ub + lane < u1 ? sorted_use[ub + lane] : 0;
    const float wu = ub + lane < u1 ? wgt[use] : 0.f;
    const int row = use / K;
    const int n = min(32, u1 - ub);
    for (int t0 = 0; t0 < n; t0 += U) {
      float4 x[U][V];
#pragma unroll
      for (int t = 0; t < U; ++t) {
        const float4* g = gP + (int64_t)__shfl_sync(0xffffffffu, row, t0 + t) * row4;
#pragma unroll
        for (int v = 0; v < V; ++v)
          if (t0 + t < n && v * 32 + lane < row4) x[t][v] = __ldg(g + v * 32 + lane);
      }
#pragma unroll
      for (int t = 0; t < U; ++t) {
        const float wt = __shfl_sync(0xffffffffu, wu, t0 + t);
        if (t0 + t < n) {
#pragma unroll
          for (int v = 0; v < V; ++v) {
            if (v * 32 + lane < row4) {
              acc[v].x = fmaf(wt, x[t][v].x, acc[v].x);
              acc[v].y = fmaf(wt, x[t][v].y, acc[v].y);
              acc[v].z = fmaf(wt, x[t][v].z, acc[v].z);
              acc[v].w = fmaf(wt, x[t][v].w, acc[v].w);
            }
          }
        }
      }
    }
  }
}

template <int V>
__device__ __forceinline__ void store_grad(float* out, int ph2, int lane, int v, float4 a) {
  const int p = 4 * (v * 32 + lane);
  if (p < ph2) out[p] = a.x;
  if (p + 1 < ph2) out[p + 1] = a.y;
  if (p + 2 < ph2) out[p + 2] = a.z;
  if (p + 3 < ph2) out[p + 3] = a.w;
}

// grad_R[id][p] = sum over the uses u of entry id (sorted, ascending) of
// w[u] * gP[u / K][p].  A warp per used entry; entries with more than kDgLong
// uses (flat patches are near thousands of queries) are listed for
// k_dict_grad_long: a block each, a sixteenth of the uses per warp, the warps'
// sums added in order.  Bound by the rows read, K times each; with a block per
// entry and one use after the other 119,691 patches of 15 x 15 with K = 8
// took 340 us and 63,504 of 10 x 10 129 us, the longest entries most of it:
// 202 and 80 us so.
constexpr int kDgWarps = 16;

template <int V>
__global__ void __launch_bounds__(128) k_dict_grad(const int32_t* __restrict__ sorted_use,
                                                   const int32_t* __restrict__ offs,
                                                   const uint64_t* __restrict__ ukeys,
                                                   const int32_t* __restrict__ nuniq,
                                                   const float* __restrict__ wgt, const float4* __restrict__ gP,
                                                   int K, int row4, int ph2, int out_stride,
                                                   float* __restrict__ grad, int32_t* __restrict__ long_list) {
  const int seg = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (seg >= *nuniq) return;   // warp-uniform
  const int u0 = offs[seg], u1 = offs[seg + 1];
  if (u1 - u0 > kDgLong) {
    if (lane == 0) long_list[1 + atomicAdd(long_list, 1)] = seg;
    return;
  }
  float4 acc[V];
#pragma unroll
  for (int v = 0; v < V; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
  add_uses<V, 4 / V>(u0, u1, sorted_use, wgt, gP, K, row4, lane, acc);
  float* out = grad + (int64_t)ukeys[seg] * out_stride;
#pragma unroll
  for (int v = 0; v < V; ++v) store_grad<V>(out, ph2, lane, v, acc[v]);
}

template <int V>
__global__ void __launch_bounds__(kDgWarps * 32) k_dict_grad_long(
    const int32_t* __restrict__ sorted_use, const int32_t* __restrict__ offs, const uint64_t* __restrict__ ukeys,
    const float* __restrict__ wgt, const float4* __restrict__ gP, int K, int row4, int ph2, int out_stride,
    float* __restrict__ grad, const int32_t* __restrict__ long_list) {
  __shared__ float4 s_part[kDgWarps][V * 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int count = long_list[0];
  for (int k = blockIdx.x; k < count; k += gridDim.x) {
    const int seg = long_list[1 + k];
    const int b0 = offs[seg], n = offs[seg + 1] - b0;
    float4 acc[V];
#pragma unroll
    for (int v = 0; v < V; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    add_uses<V, 8 / V>(b0 + (int)((int64_t)n * warp / kDgWarps), b0 + (int)((int64_t)n * (warp + 1) / kDgWarps),
                       sorted_use, wgt, gP, K, row4, lane, acc);
#pragma unroll
    for (int v = 0; v < V; ++v) s_part[warp][v * 32 + lane] = acc[v];
    __syncthreads();
    if (warp < V) {
      float4 a = s_part[0][warp * 32 + lane];
      for (int j = 1; j < kDgWarps; ++j) {
        const float4 x = s_part[j][warp * 32 + lane];
        a.x += x.x;
        a.y += x.y;
        a.z += x.z;
        a.w += x.w;
      }
      store_grad<V>(grad + (int64_t)ukeys[seg] * out_stride, ph2, lane, warp, a);
    }
    __syncthreads();   // the sums have been read
  }
}

// grad_mu[n] = sum_p OA^T(g)[n][p] (the patch mean enters every pixel).
__global__ void k_mu_grad(const float* __restrict__ gP, int64_t nq, int ph2, int ph2pad, float* __restrict__ gmu) {
  const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nq) return;
  float acc = 0.f;
  for (int p = 0; p < ph2; ++p) acc += gP[n * ph2pad + p];
  gmu[n] = acc;
}

// per-block partial sums (in FP64) of r^2 over n values
__global__ void k_sumsq_partials(const float* __restrict__ r, int64_t n, double* __restrict__ part) {
  __shared__ double sh[256];
  double acc = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    acc += (double)r[i] * (double)r[i];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// per-block partial sums of the overlap prior: each (patch, pixel) adds the
// squared difference to its right and down neighbours where they overlap, in
// FP64 throughout.  Bound by the GPU's few FP64 units (63,504 patches of 10 x
// 10: 114 us; 81 us with sixteen values at a time in pairs of floats, which
// loses bits and FP64's range).
__global__ void k_prior_partials(const float* __restrict__ P, int h, int w, int s, int Pp, int ph2pad,
                                 double* __restrict__ part) {
  __shared__ double sh[256];
  __shared__ uint32_t s_px[kMaxPatchPixels];
  const int PH = s * Pp, ph2 = PH * PH;
  const int nh = h - Pp + 1, nw = w - Pp + 1;
  for (int p = threadIdx.x; p < ph2; p += blockDim.x) s_px[p] = pixel_code(p, PH, s);
  __syncthreads();
  const int64_t total = (int64_t)nh * nw * ph2, step = (int64_t)gridDim.x * blockDim.x;
  // (n, p) and (i, j) of the running value, advanced by the step's whole
  // patches and pixels
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int64_t n = t / ph2;
  int p = (int)(t - n * ph2);
  const int64_t dn = step / ph2;
  const int dp = (int)(step - dn * ph2);
  int i = (int)(n / nw), j = (int)(n - (int64_t)i * nw);
  const int di = (int)(dn / nw), dj = (int)(dn - (int64_t)di * nw);
  double acc = 0.0;
#pragma unroll 4
  for (; t < total; t += step) {
    const uint32_t c = s_px[p];
    const int a = c & 255, b = (c >> 8) & 255;
    const float* pn = P + n * ph2pad;
    const double pv = (double)pn[p];
    if (j + 1 < nw && b >= s) {
      const double d = pv - (double)pn[ph2pad + p - s];
      acc += d * d;
    }
    if (i + 1 < nh && a >= s) {
      const double d = pv - (double)pn[(int64_t)nw * ph2pad + p - s * PH];
      acc += d * d;
    }
    n += dn;
    p += dp;
    i += di;
    j += dj;
    if (p >= ph2) {
      p -= ph2;
      ++n;
      ++j;
    }
    if (j >= nw) {
      j -= nw;
      ++i;
    }
  }
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// dist[n][m] = |q_n - c_{nbr[n][m]}|^2 (FP32 difference form)
template <int D>
__global__ void k_nbr_dist(const float* __restrict__ qfeat, int dpad, int64_t nq, const float* __restrict__ dfeat,
                           const int32_t* __restrict__ nbr, int K, float* __restrict__ dist) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nq * K) return;
  const int64_t n = t / K;
  const int64_t id = nbr[t];
  float dd = 0.f;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    const float df = qfeat[n * dpad + i] - dfeat[id * dpad + i];
    dd = fmaf(df, df, dd);
  }
  dist[t] = dd;
}

Wts degrade_wts(int s, double sigma) {
  Wts wt;
  double e = exp(-1.0 / (2.0 * sigma * sigma));
  double t[3] = {e / (1.0 + 2.0 * e), 1.0 / (1.0 + 2.0 * e), e / (1.0 + 2.0 * e)};
  double acc[8] = {0};
  for (int b = 0; b < s; ++b)
    for (int u = 0; u < 3; ++u) acc[b + u] += t[u] / s;
  wt.n = s + 2;
  for (int a = 0; a < 8; ++a) wt.w[a] = (float)acc[a];
  return wt;
}

}  // namespace

cudaError_t launch_patches(const int32_t* nbr, const float* wgt, const float* mu, const float* hr_res,
                           int ph2pad, int K, int64_t nq, float* P, cudaStream_t st) {
  const int64_t tot = nq * (ph2pad / 4);
  k_patches<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(nbr, wgt, mu, (const float4*)hr_res, ph2pad / 4, K, nq,
                                                           (float4*)P);
  return cudaGetLastError();
}

cudaError_t launch_degrade(const float* x, int H, int W, int s, double sigma, const float* sub, float* y,
                           cudaStream_t st) {
  const int h = H / s, w = W / s;
  dim3 blk(32, 8), grd((w + 31) / 32, (h + 7) / 8);
  k_degrade<<<grd, blk, 0, st>>>(x, H, W, h, w, s, degrade_wts(s, sigma), sub, y);
  return cudaGetLastError();
}

cudaError_t launch_degrade_adjoint(const float* r, int h, int w, int H, int W, int s, double sigma,
                                   float alpha, float* g, cudaStream_t st) {
  dim3 blk(32, 8), grd((W + 31) / 32, (H + 7) / 8);
  k_degrade_adjoint<<<grd, blk, 0, st>>>(r, h, w, H, W, s, degrade_wts(s, sigma), alpha, g);
  return cudaGetLastError();
}

cudaError_t launch_patch_grad(const float* gx, const float* P, int h, int w, int s, int Pp, int ph2pad,
                              float lambda, float* gP, cudaStream_t st) {
  if (s * Pp * s * Pp > kMaxPatchPixels) return cudaErrorInvalidValue;
  const int64_t nq = (int64_t)(h - Pp + 1) * (w - Pp + 1);
  const int64_t blocks = std::min<int64_t>((nq + 7) / 8, 8192);
  k_patch_grad<<<(unsigned)blocks, 256, 0, st>>>(gx, P, h, w, s, Pp, ph2pad, lambda, gP);
  return cudaGetLastError();
}

cudaError_t launch_dict_grad(const int32_t* sorted_use, const int32_t* offs, const uint64_t* ukeys,
                             const int32_t* nuniq, int64_t max_segments, const float* wgt, const float* gP,
                             int K, int ph2, int ph2pad, int out_stride, float* grad, int32_t* long_list, cudaStream_t st) {
  if (max_segments <= 0) return cudaSuccess;
  const unsigned blocks = (unsigned)((max_segments + 3) / 4);
  const int row4 = ph2pad / 4;
  const float4* g4 = (const float4*)gP;
  cudaError_t e = cudaMemsetAsync(long_list, 0, sizeof(int32_t), st);
  if (e != cudaSuccess) return e;
#define ZOOM_DG(V)                                                                                               \
  do {                                                                                                           \
    k_dict_grad<V><<<blocks, 128, 0, st>>>(sorted_use, offs, ukeys, nuniq, wgt, g4, K, row4, ph2, out_stride, grad, \
                                           long_list);                                                           \
    k_dict_grad_long<V><<<304, kDgWarps * 32, 0, st>>>(sorted_use, offs, ukeys, wgt, g4, K, row4, ph2, out_stride, \
                                                       grad, long_list);                                         \
  } while (0)
  if (row4 <= 32) ZOOM_DG(1);
  else if (row4 <= 64) ZOOM_DG(2);
  else if (row4 <= 128) ZOOM_DG(4);
  else return cudaErrorInvalidValue;
#undef ZOOM_DG
  return cudaGetLastError();
}

cudaError_t launch_mu_grad(const float* gP, int64_t nq, int ph2, int ph2pad, float* gmu, cudaStream_t st) {
  k_mu_grad<<<(unsigned)((nq + 127) / 128), 128, 0, st>>>(gP, nq, ph2, ph2pad, gmu);
  return cudaGetLastError();
}

cudaError_t launch_energy_partials(const float* r, int64_t n_r, const float* P, int h, int w, int s, int Pp,
                                   int ph2pad, double* part, int nblocks, cudaStream_t st) {
  if (s * Pp * s * Pp > kMaxPatchPixels) return cudaErrorInvalidValue;
  k_sumsq_partials<<<nblocks, 256, 0, st>>>(r, n_r, part);
  k_prior_partials<<<nblocks, 256, 0, st>>>(P, h, w, s, Pp, ph2pad, part + nblocks);
  return cudaGetLastError();
}

cudaError_t launch_nbr_dist(const float* qfeat, int dpad, int d, int64_t nq, const float* dfeat,
                            const int32_t* nbr, int K, float* dist, cudaStream_t st) {
  const int64_t tot = nq * K;
  const unsigned blocks = (unsigned)((tot + 127) / 128);
  if (d == 9) k_nbr_dist<9><<<blocks, 128, 0, st>>>(qfeat, dpad, nq, dfeat, nbr, K, dist);
  else if (d == 25) k_nbr_dist<25><<<blocks, 128, 0, st>>>(qfeat, dpad, nq, dfeat, nbr, K, dist);
  else if (d == 18) k_nbr_dist<18><<<blocks, 128, 0, st>>>(qfeat, dpad, nq, dfeat, nbr, K, dist);
  else if (d == 50) k_nbr_dist<50><<<blocks, 128, 0, st>>>(qfeat, dpad, nq, dfeat, nbr, K, dist);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}
