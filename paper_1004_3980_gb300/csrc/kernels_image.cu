// HR image steps: blend + overlap average (Eq. 14; averaging of overlaps)
// and the error back-projection with the approximate cross-bilateral filter
// (Sec. 4, Eq. 6-7; Sec. 4.3, Eq. 15-17).
#include <math.h>

#include <algorithm>

#include "device_common.cuh"
#include "zoom_internal.h"

namespace {

// Overlap average in one pass: each HR pixel sums, over the patches covering
// it, the patch's blended value mu_n + sum_m w_nm R[nbr_nm] at its offset,
// patch rows i ascending, then columns j, and divides by the number of
// covering patches.  No atomics.
//
// A block takes the s HR rows of one LR row and the columns of kOvTile LR
// columns.  Of a patch that touches it the block needs s whole rows, which
// are one run of s PH values of every neighbour's residual row: the runs are
// read in order and blended into shared memory, patch row by patch row (two
// buffers), and the pixels add them up from there.  Every blended value is
// used by one pixel, so nothing is computed twice but the P - 1 patches
// beside the tile.  Bound by the neighbours' rows from L2: with each pixel
// fetching its own values, scattered, 119,691 patches of 15 x 15 and K = 8
// took 307 us, 210 us so.  K = 0: hr_res holds
// the blended patches themselves, row n for patch n.
constexpr int kOvTile = 32;
constexpr int kOvThreads = 256;

__global__ void __launch_bounds__(kOvThreads) k_overlap_add(const int32_t* __restrict__ nbr,
                                                            const float* __restrict__ wgt,
                                                            const float* __restrict__ mu,
                                                            const float* __restrict__ hr_res, int64_t stride,
                                                            int K, int h, int w, int s, int P, int row0,
                                                            float* __restrict__ hr) {
  const int PH = s * P, nh = h - P + 1, nw = w - P + 1, W = s * w, run = s * PH;
  const int I = row0 + blockIdx.y, J0 = blockIdx.x * kOvTile;
  const int jb = max(0, J0 - P + 1), je = min(nw, J0 + kOvTile), np = je - jb;   // patches [jb, je) of a row
  const int i_lo = max(0, I - P + 1), i_hi = min(I, nh - 1), ni = i_hi - i_lo + 1;
  extern __shared__ float s_ov[];
  float* s_w = s_ov + 2 * (kOvTile + P - 1) * run;                 // [ni][np][K]
  int32_t* s_n = (int32_t*)(s_w + P * (kOvTile + P - 1) * K);      // [ni][np][K]
  const int tid = threadIdx.x;
  for (int e = tid; e < ni * np * K; e += kOvThreads) {
    const int i = e / (np * K), r = e - i * (np * K);
    const int64_t g = ((int64_t)(i_lo + i) * nw + jb) * K + r;
    s_n[e] = nbr[g];
    s_w[e] = wgt[g];
  }
  // this thread's pixels of the s x (s kOvTile) tile: at most two
  const int tw = s * kOvTile, npx = s * tw;
  float acc[2] = {0.f, 0.f};
  int src[2], nj[2];   // first value in a buffer, covering patch columns
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    const int px = tid + t * kOvThreads;
    const int ar = px / tw, X = s * J0 + (px - ar * tw);
    const int j_hi = min(X / s, nw - 1), j_lo = X >= PH ? (X - PH) / s + 1 : 0;
    nj[t] = px < npx && X < W ? j_hi - j_lo + 1 : 0;
    src[t] = ar * PH + X + (j_lo - jb) * run - s * j_lo;
  }
  const float inv = 1.f / (float)run;   // (e + 0.5) / run is far enough from whole numbers
  __syncthreads();
  for (int i = 0; i < ni; ++i) {
    float* buf = s_ov + (i & 1) * (kOvTile + P - 1) * run;
    const int off0 = s * (I - (i_lo + i)) * PH;
    const int64_t n0 = (int64_t)(i_lo + i) * nw + jb;
    for (int e = tid; e < np * run; e += kOvThreads) {
      const int q = (int)(((float)e + 0.5f) * inv), o = e - q * run;
      if (K == 0) {   // the patches as they are
        buf[e] = __ldg(hr_res + (n0 + q) * stride + off0 + o);
        continue;
      }
      const int32_t* nb = s_n + (i * np + q) * K;
      const float* wq = s_w + (i * np + q) * K;
      const float* col = hr_res + off0 + o;
      float v = mu[n0 + q];
      for (int m0 = 0; m0 < K; m0 += 8) {
        float r[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) r[u] = m0 + u < K ? __ldg(col + nb[m0 + u] * stride) : 0.f;
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (m0 + u < K) v = fmaf(wq[m0 + u], r[u], v);
      }
      buf[e] = v;
    }
    __syncthreads();   // (the other buffer's readers are past it: one barrier a round)
#pragma unroll
    for (int t = 0; t < 2; ++t)
      for (int j = 0; j < nj[t]; ++j) acc[t] += buf[src[t] + j * (run - s)];
  }
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    const int px = tid + t * kOvThreads;
    const int ar = px / tw, X = s * J0 + (px - ar * tw);
    if (nj[t] > 0) hr[(int64_t)(s * I + ar) * W + X] = acc[t] / (float)(ni * nj[t]);
  }
}

// The same average in two passes, for callers with nq * PH^2 floats of
// scratch.  Pass 1 blends the patches of 32 consecutive queries of one patch
// row: the neighbours' residual rows are read whole, in order and 16 bytes
// per load, each thread blending 4 adjacent patch pixels (the one-pass form
// reads each 4-byte value from the pixels it covers, scattered over the
// row), and the blended values leave through shared memory,
// transposed to the layout [patch row i][patch pixel p][patch column j].
// Pass 2 averages them per HR pixel: for one covering patch the lanes of a
// warp then read s runs of consecutive j.  Each blended value is computed
// with the same operations in the same order as in the one-pass form, and
// pass 2 sums them in its order, so both forms give the same bits.
constexpr int kBlendQ = 32;       // queries of one patch row per block
constexpr int kBlendPC = 128;     // patch pixels per shared-memory round
constexpr int kBlendMaxK = 64;

__global__ void __launch_bounds__(256) k_blend_rows(const int32_t* __restrict__ nbr,
                                                    const float* __restrict__ wgt,
                                                    const float* __restrict__ mu,
                                                    const float* __restrict__ hr_res, int ph2pad, int K,
                                                    int nw, int ph2, float* __restrict__ out) {
  __shared__ int32_t s_nbr[kBlendQ * kBlendMaxK];
  __shared__ float s_w[kBlendQ * kBlendMaxK];
  __shared__ float s_mu[kBlendQ];
  __shared__ float s_t[kBlendPC * (kBlendQ + 1)];
  const int i = blockIdx.y;
  const int j0 = blockIdx.x * kBlendQ;
  const int nqc = min(kBlendQ, nw - j0);
  const int64_t n0 = (int64_t)i * nw + j0;
  for (int e = threadIdx.x; e < nqc * K; e += blockDim.x) {
    s_nbr[e] = nbr[n0 * K + e];
    s_w[e] = wgt[n0 * K + e];
  }
  if ((int)threadIdx.x < nqc) s_mu[threadIdx.x] = mu[n0 + threadIdx.x];
  __syncthreads();
  for (int p0 = 0; p0 < ph2; p0 += kBlendPC) {
    const int pc = min(kBlendPC, ph2 - p0);
    const int pq = (pc + 3) / 4;   // 4-pixel groups; the last may reach into the row's padding
    for (int e = threadIdx.x; e < nqc * pq; e += blockDim.x) {
      const int q = e / pq, pl = 4 * (e - q * pq);
      const int32_t* nb = s_nbr + q * K;
      const float* wq = s_w + q * K;
      const float* col = hr_res + p0 + pl;
      float4 v = make_float4(s_mu[q], s_mu[q], s_mu[q], s_mu[q]);
      for (int m0 = 0; m0 < K; m0 += 8) {
        float4 r[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          r[u] = m0 + u < K ? __ldg(reinterpret_cast<const float4*>(col + (int64_t)nb[m0 + u] * ph2pad))
                            : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (m0 + u < K) {
            const float wm = wq[m0 + u];
            v.x = fmaf(wm, r[u].x, v.x);
            v.y = fmaf(wm, r[u].y, v.y);
            v.z = fmaf(wm, r[u].z, v.z);
            v.w = fmaf(wm, r[u].w, v.w);
          }
      }
      float* t = s_t + pl * (kBlendQ + 1) + q;
      t[0] = v.x;
      if (pl + 1 < pc) t[kBlendQ + 1] = v.y;
      if (pl + 2 < pc) t[2 * (kBlendQ + 1)] = v.z;
      if (pl + 3 < pc) t[3 * (kBlendQ + 1)] = v.w;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < pc * kBlendQ; e += blockDim.x) {
      const int pl = e / kBlendQ, q = e % kBlendQ;
      if (q < nqc) out[((int64_t)i * ph2 + p0 + pl) * nw + j0 + q] = s_t[pl * (kBlendQ + 1) + q];
    }
    __syncthreads();
  }
}

__global__ void k_overlap_average(const float* __restrict__ pb, int h, int w, int s, int P,
                                  float* __restrict__ hr) {
  const int W = s * w, H = s * h;
  const int X = blockIdx.x * blockDim.x + threadIdx.x;
  const int Y = blockIdx.y * blockDim.y + threadIdx.y;
  if (X >= W || Y >= H) return;
  const int PH = s * P, nh = h - P + 1, nw = w - P + 1, ph2 = PH * PH;
  const int i_hi = min(Y / s, nh - 1), j_hi = min(X / s, nw - 1);
  const int i_lo = Y >= PH ? (Y - PH) / s + 1 : 0;
  const int j_lo = X >= PH ? (X - PH) / s + 1 : 0;
  float acc = 0.f;
  int cnt = 0;
  for (int i = i_lo; i <= i_hi; ++i) {
    const float* row = pb + ((int64_t)i * ph2 + (Y - s * i) * PH) * nw;
    for (int j = j_lo; j <= j_hi; ++j) {
      acc += __ldg(row + (int64_t)(X - s * j) * nw + j);
      ++cnt;
    }
  }
  hr[(int64_t)Y * W + X] = acc / (float)cnt;
}

// e = D(B x) - y on the LR grid (FP32).  The blur and the box mean combine
// into separable 1-D weights over the (s+2)-wide window.
struct Wts1D {
  int n;
  float w[8];
};

// An NR x NC window of x at (r0, c0) into shared memory, borders clamped: all of
// a thread's loads are issued before the first is stored.
template <int NR, int NC, int STRIDE>
__device__ __forceinline__ void load_window(const float* __restrict__ x, int H, int W, int r0, int c0, int tid,
                                            float (*dst)[STRIDE]) {
  constexpr int N = NR * NC, IT = (N + 255) / 256;
  float v[IT];
#pragma unroll
  for (int k = 0; k < IT; ++k) {
    const int i = min(tid + k * 256, N - 1);
    const int r = i / NC, c = i - r * NC;
    v[k] = __ldg(x + (int64_t)zoom_clampi(r0 + r, 0, H - 1) * W + zoom_clampi(c0 + c, 0, W - 1));
  }
#pragma unroll
  for (int k = 0; k < IT; ++k) {
    const int i = tid + k * 256;
    if (i < N) dst[i / NC][i % NC] = v[k];
  }
}

// A block takes 32 x 8 LR pixels: their HR rows and columns in shared memory
// (clamped), the weighted row sums of every HR row, then the column sums; the
// same products and sums in the same order for every pixel as one thread's
// double loop.  Bound by issue (77 % of the slots; reading the image once is 36 %
// of the DRAM's rate); with each thread reading its
// (s + 2)^2 values from memory 1920 x 1080 at 3x took 61 us, and as much
// with one load of the window in flight a thread; 32 us so.
constexpr int kErrW = 32, kErrH = 8;

template <int S>
__global__ void __launch_bounds__(256) k_bp_error(const float* __restrict__ x, int H, int W,
                                                  const float* __restrict__ y, int h, int w, Wts1D wt,
                                                  float* __restrict__ e) {
  constexpr int NR = S * kErrH + 2, NC = S * kErrW + 2;
  __shared__ float xs[NR][NC];
  __shared__ float rows[NR][kErrW];
  const int j0 = blockIdx.x * kErrW, i0 = blockIdx.y * kErrH;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  load_window<NR, NC, NC>(x, H, W, S * i0 - 1, S * j0 - 1, tid, xs);
  __syncthreads();
  for (int r = warp; r < NR; r += kErrH) {
    float row = 0.f;
#pragma unroll
    for (int b = 0; b < S + 2; ++b) row = fmaf(wt.w[b], xs[r][S * lane + b], row);
    rows[r][lane] = row;
  }
  __syncthreads();
  const int i = i0 + warp, j = j0 + lane;
  if (i >= h || j >= w) return;
  float acc = 0.f;
#pragma unroll
  for (int a = 0; a < S + 2; ++a) acc = fmaf(wt.w[a], rows[S * warp + a][lane], acc);
  e[(int64_t)i * w + j] = acc - y[(int64_t)i * w + j];
}

// x' = x - r * G, G = normalised spatial Gaussian over the replicated LR
// error, r = exp(-(x - mean_Gamma x)^2 / (2 sigma_r^2)); clamped borders.
struct Gauss1D {
  int R;
  float c[16];
};

// One block computes a 64-row x 32-column tile of x' from shared memory: the
// tile of x with its R-pixel halo (clamped), then the separable sums -- each
// row's box sum over the 2R+1 columns, and for each LR error row the
// Gaussian-weighted sum over the 2R+1 replicated columns -- and per pixel the
// column sums over 2R+1 rows.  The summation order is that of the direct
// double loop (columns t within a row, then rows u), so the result is the
// same bit for bit; x is read from memory once (with the halo) instead of
// (2R+1)^2 times, and the LR row and column of every clamped tile row and
// column are computed once per block.  Was bound by shared-memory reads: a thread
// sums eight neighbouring columns of a row, then eight neighbouring rows of a
// column, from registers, and a thread's loads are issued together (5760 x
// 3240, R = 3: 125 us with 2R + 1 reads a sum and one load in flight, 93 us so).
// Bound by issue now: 82 % of the slots, shared memory 45 %, DRAM 16 %.
constexpr int kBpTileW = 32, kBpTileH = 64;
template <int R>
__global__ void __launch_bounds__(256) k_bp_update(const float* __restrict__ x, float* __restrict__ xo, int H,
                                                   int W, const float* __restrict__ e, int w, int s, Gauss1D g,
                                                   float inv_two_sr2) {
  constexpr int T = 2 * R + 1;
  constexpr int NW = kBpTileW + 2 * R, NH = kBpTileH + 2 * R;   // the tile with its halo
  constexpr int kRun = 8;               // columns, then rows, a thread sums side by side
  constexpr int XP = (NW | 1);          // odd strides: lanes on neighbouring rows hit different banks
  __shared__ float xs[NH][XP];          // x, clamped
  __shared__ float hs[NH][kBpTileW + 1];   // row box sums
  __shared__ float hg[NH][kBpTileW];    // per LR row: Gaussian row sums of the replicated error
  __shared__ int lrow[NH], lcol[NW];    // LR row (relative to lr0) / column of each clamped tile row / column
  const int X0 = blockIdx.x * kBpTileW, Y0 = blockIdx.y * kBpTileH;
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  const int lr0 = zoom_clampi(Y0 - R, 0, H - 1) / s;
  const int nlr = zoom_clampi(Y0 + kBpTileH - 1 + R, 0, H - 1) / s - lr0 + 1;
  for (int i = tid; i < NH; i += 256) lrow[i] = zoom_clampi(Y0 - R + i, 0, H - 1) / s - lr0;
  for (int i = tid; i < NW; i += 256) lcol[i] = zoom_clampi(X0 - R + i, 0, W - 1) / s;
  load_window<NH, NW, XP>(x, H, W, Y0 - R, X0 - R, tid, xs);
  __syncthreads();
  for (int i = tid; i < nlr * kBpTileW; i += 256) {
    const int r = i / kBpTileW, c = i % kBpTileW;
    const float* er = e + (int64_t)(lr0 + r) * w;
    float grow = 0.f;
#pragma unroll
    for (int t = 0; t < T; ++t) grow = fmaf(g.c[t], er[lcol[c + t]], grow);
    hg[r][c] = grow;
  }
  for (int i = tid; i < NH * (kBpTileW / kRun); i += 256) {
    const int r = i % NH, c = i / NH * kRun;
    float v[kRun + 2 * R];
#pragma unroll
    for (int t = 0; t < kRun + 2 * R; ++t) v[t] = xs[r][c + t];
#pragma unroll
    for (int k = 0; k < kRun; ++k) {
      float brow = 0.f;
#pragma unroll
      for (int t = 0; t < T; ++t) brow += v[k + t];
      hs[r][c + k] = brow;
    }
  }
  __syncthreads();
  static_assert(kBpTileH == kRun * 8 && kBpTileW == 32, "one run of rows a thread");
  const int c = threadIdx.x, y0 = threadIdx.y * kRun;
  const int X = X0 + c;
  if (X >= W) return;
  float b[kRun + 2 * R], q[kRun + 2 * R];
#pragma unroll
  for (int t = 0; t < kRun + 2 * R; ++t) {
    b[t] = hs[y0 + t][c];
    q[t] = hg[lrow[y0 + t]][c];
  }
#pragma unroll
  for (int k = 0; k < kRun; ++k) {
    const int Y = Y0 + y0 + k;
    if (Y >= H) break;
    float gs = 0.f, box = 0.f;
#pragma unroll
    for (int u = 0; u < T; ++u) {
      gs = fmaf(g.c[u], q[k + u], gs);
      box += b[k + u];
    }
    const float m = box / (float)(T * T);
    const float xv = xs[y0 + k + R][c + R];
    const float dv = xv - m;
    const float r = expf(-dv * dv * inv_two_sr2);
    xo[(int64_t)Y * W + X] = xv - r * gs;
  }
}

}  // namespace

cudaError_t launch_overlap_add(const int32_t* nbr, const float* wgt, const float* mu,
                               const float* hr_res, int ph2pad, int K, int h, int w, int s, int P,
                               float* hr, cudaStream_t st) {
  // at most two pixels a thread (s <= 4); 128 KB of shared memory at K = 64, P = 5, s = 4
  const size_t smem = (size_t)(kOvTile + P - 1) * (2 * s * s * P + 2 * P * K) * 4;
  if (s * s * kOvTile > 2 * kOvThreads) return cudaErrorInvalidValue;
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(k_overlap_add, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  // an LR row per block row: at most 65,535 in a grid's second dimension
  for (int i0 = 0; i0 < h; i0 += 65535)
    k_overlap_add<<<dim3((w + kOvTile - 1) / kOvTile, std::min(h - i0, 65535)), kOvThreads, smem, st>>>(
        nbr, wgt, mu, hr_res, ph2pad, K, h, w, s, P, i0, hr);
  return cudaGetLastError();
}

cudaError_t launch_overlap_add_staged(const int32_t* nbr, const float* wgt, const float* mu,
                                      const float* hr_res, int ph2pad, int K, int h, int w, int s, int P,
                                      float* patches, float* hr, cudaStream_t st) {
  const int nh = h - P + 1, nw = w - P + 1, PH = s * P;
  // 16-byte loads of the residual rows: 16-byte aligned rows, padded to 4
  if (K > kBlendMaxK || nh > 65535 || !patches || ph2pad % 4 != 0 || ph2pad < PH * PH ||
      reinterpret_cast<uintptr_t>(hr_res) % 16 != 0)
    return launch_overlap_add(nbr, wgt, mu, hr_res, ph2pad, K, h, w, s, P, hr, st);
  dim3 g1((nw + kBlendQ - 1) / kBlendQ, nh);
  k_blend_rows<<<g1, 256, 0, st>>>(nbr, wgt, mu, hr_res, ph2pad, K, nw, PH * PH, patches);
  dim3 blk(32, 8), g2((s * w + 31) / 32, (s * h + 7) / 8);
  k_overlap_average<<<g2, blk, 0, st>>>(patches, h, w, s, P, hr);
  return cudaGetLastError();
}

cudaError_t launch_bp_iteration(const float* x, float* x_out, const float* lr, float* err, int h,
                                int w, int s, double blur_sigma, float sigma_sp, float sigma_r,
                                int radius, cudaStream_t st) {
  const int H = s * h, W = s * w;
  Wts1D wt;
  {
    double e = exp(-1.0 / (2.0 * blur_sigma * blur_sigma));
    double t[3] = {e / (1.0 + 2.0 * e), 1.0 / (1.0 + 2.0 * e), e / (1.0 + 2.0 * e)};
    double acc[8] = {0};
    for (int b = 0; b < s; ++b)
      for (int u = 0; u < 3; ++u) acc[b + u] += t[u] / s;
    wt.n = s + 2;
    for (int a = 0; a < 8; ++a) wt.w[a] = (float)acc[a];
  }
  Gauss1D g;
  {
    g.R = radius;
    double c[16], tot = 0.0;
    for (int d = -radius; d <= radius; ++d) {
      c[d + radius] = exp(-(double)(d * d) / (2.0 * (double)sigma_sp * (double)sigma_sp));
      tot += c[d + radius];
    }
    for (int d = 0; d < 16; ++d) g.c[d] = d < 2 * radius + 1 ? (float)(c[d] / tot) : 0.f;
  }
  dim3 blk(32, 8);
  dim3 g1((w + kErrW - 1) / kErrW, (h + kErrH - 1) / kErrH);
  switch (s) {
    case 1: k_bp_error<1><<<g1, 256, 0, st>>>(x, H, W, lr, h, w, wt, err); break;
    case 2: k_bp_error<2><<<g1, 256, 0, st>>>(x, H, W, lr, h, w, wt, err); break;
    case 3: k_bp_error<3><<<g1, 256, 0, st>>>(x, H, W, lr, h, w, wt, err); break;
    case 4: k_bp_error<4><<<g1, 256, 0, st>>>(x, H, W, lr, h, w, wt, err); break;
    default: return cudaErrorInvalidValue;
  }
  dim3 g2((W + kBpTileW - 1) / kBpTileW, (H + kBpTileH - 1) / kBpTileH);
  const float inv = (float)(1.0 / (2.0 * (double)sigma_r * (double)sigma_r));
  switch (radius) {
#define ZOOM_BPU(RR) \
  case RR: k_bp_update<RR><<<g2, blk, 0, st>>>(x, x_out, H, W, err, w, s, g, inv); break;
    ZOOM_BPU(1) ZOOM_BPU(2) ZOOM_BPU(3) ZOOM_BPU(4) ZOOM_BPU(5) ZOOM_BPU(6) ZOOM_BPU(7)
#undef ZOOM_BPU
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}
