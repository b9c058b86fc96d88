// Dictionary and LSH index construction (Sec. 2.1, Sec. 3.2, Sec. 4.1).
#include <math.h>

#include <algorithm>
#include <vector>

#include "device_common.cuh"
#include "zoom_internal.h"

namespace {

constexpr int kMaxScale = 4;

// Combined blur+box weights of one output pixel, W_a * W_b over the
// (s+2) x (s+2) window, as unevaluated float pairs hi + lo.
struct PairWeights {
  int n;  // s + 2
  float hi[(kMaxScale + 2) * (kMaxScale + 2)];
  float lo[(kMaxScale + 2) * (kMaxScale + 2)];
};

// 1-D weights of "3-tap Gaussian then s-box mean": output i reads input
// s*i + a - 1, a in [0, s+2), with weight (1/s) * sum_{b + u = a} taps[u].
void degrade_weights_1d(int s, double sigma, double* wts) {
  double e = exp(-1.0 / (2.0 * sigma * sigma));
  double t[3] = {e / (1.0 + 2.0 * e), 1.0 / (1.0 + 2.0 * e), e / (1.0 + 2.0 * e)};
  for (int a = 0; a < s + 2; ++a) wts[a] = 0.0;
  for (int b = 0; b < s; ++b)
    for (int u = 0; u < 3; ++u) wts[b + u] += t[u] / s;
}

// LR[i][j] = sum_{a,b} W_a W_b HR[clamp(s i + a - 1)][clamp(s j + b - 1)],
// accumulated as a float pair (two-sum / fma two-product) so that the final
// float is the correctly rounded value of the exact sum in all but
// vanishingly rare cases.  The dictionary stores this rounded LR image.
__global__ void k_degrade_exact(const float* __restrict__ hr, int H, int W, int s, PairWeights pw,
                                float* __restrict__ lr, int h, int w) {
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  int i = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= h || j >= w) return;
  float shi = 0.f, slo = 0.f;
  for (int a = 0; a < pw.n; ++a) {
    int r = zoom_clampi(s * i + a - 1, 0, H - 1);
    for (int b = 0; b < pw.n; ++b) {
      int c = zoom_clampi(s * j + b - 1, 0, W - 1);
      float x = hr[(size_t)r * W + c];
      float whi = pw.hi[a * pw.n + b], wlo = pw.lo[a * pw.n + b];
      float p = x * whi;
      float pe = fmaf(x, whi, -p);
      pe = fmaf(x, wlo, pe);
      float t = shi + p;
      float bp = t - shi;
      float err = (shi - (t - bp)) + (p - bp);
      shi = t;
      slo += err + pe;
    }
  }
  lr[(size_t)i * w + j] = shi + slo;
}

// Patch pairs of the dictionary: one thread computes an entry's LR patch and
// feature, the block then writes its 128 entries' rows through shared memory
// and copies their HR patches, neighbouring lanes on neighbouring values.
// Bound by the rows written (620 bytes an entry at P = 5, s = 2).  With each
// thread writing its own rows every store instruction touched 32 lines: 1M
// entries 935 us, 225 us so.
constexpr int kGatherRows = 128;

template <int P, int F>
__global__ void __launch_bounds__(kGatherRows) k_dict_gather(
    const float* const* __restrict__ lr_images, const int32_t* __restrict__ lr_h,
    const int32_t* __restrict__ lr_w, const float* const* __restrict__ hr_images,
    const int32_t* __restrict__ hr_w, const int32_t* __restrict__ pos, int64_t n, int s, int ph2pad,
    float* __restrict__ lr_pix, float* __restrict__ feat, float* __restrict__ mu,
    float* __restrict__ norm2, float* __restrict__ hr_res) {
  constexpr int P2 = P * P;
  constexpr int D = zoom_feature_dim(P, F);
  constexpr int DP = (D + 3) / 4 * 4;
  __shared__ float s_pix[kGatherRows * P2];
  __shared__ float s_feat[F == 0 ? 1 : kGatherRows * (D | 1)];   // odd stride: no bank conflicts
  __shared__ const float* s_hr[kGatherRows];   // the entry's HR patch
  __shared__ int s_hw[kGatherRows];
  __shared__ float s_mean[kGatherRows];
  const int r = threadIdx.x;
  const int64_t e0 = (int64_t)blockIdx.x * kGatherRows, e = e0 + r;
  const int rows = (int)(n - e0 < kGatherRows ? n - e0 : kGatherRows);
  if (r < rows) {
    const int m = pos[e * 3 + 0], i = pos[e * 3 + 1], j = pos[e * 3 + 2];
    const float* lr = lr_images[m];
    const int lw = lr_w[m];
    float px[P2], v[P2], mean, n2;
#pragma unroll
    for (int a = 0; a < P; ++a)
#pragma unroll
      for (int b = 0; b < P; ++b) px[a * P + b] = lr[(size_t)(i + a) * lw + j + b];
    zoom_patch_feature<P2>(px, v, mean, n2);
#pragma unroll
    for (int q = 0; q < P2; ++q) s_pix[r * P2 + q] = px[q];
    if constexpr (F != 0) {
      float g[D];
      zoom_gradient_feature<P, F>(lr, lr_h[m], lw, (size_t)lw, i, j, g, n2);
#pragma unroll
      for (int q = 0; q < D; ++q) s_feat[r * (D | 1) + q] = g[q];
    }
    mu[e] = mean;
    norm2[e] = n2;
    const int hw = hr_w[m];
    s_hr[r] = hr_images[m] + (size_t)(s * i) * hw + s * j;
    s_hw[r] = hw;
    s_mean[r] = mean;
  }
  __syncthreads();
  for (int t = r; t < rows * P2; t += kGatherRows) lr_pix[e0 * P2 + t] = s_pix[t];
  for (int t = r; t < rows * DP; t += kGatherRows) {
    const int x = t / DP, q = t % DP;
    float f = 0.f;
    // a mean-free patch is the pixels less their mean (zoom_patch_feature)
    if (q < D) f = F == 0 ? s_pix[x * P2 + q] - s_mean[x] : s_feat[x * (D | 1) + q];
    feat[e0 * DP + t] = f;
  }
  // a warp per HR patch, four entries at a time in flight
  const int PH = s * P, ph2 = PH * PH;
  const float inv = 1.f / (float)PH;   // (q + 0.5) / PH is far enough from whole numbers
  const int lane = r & 31;
  for (int q = lane; q < ph2pad; q += 32) {
    const int a = (int)(((float)q + 0.5f) * inv), b = q - a * PH;
#pragma unroll 4
    for (int x = r >> 5; x < rows; x += kGatherRows / 32) {
      float o = 0.f;
      if (q < ph2) o = s_hr[x][(size_t)a * s_hw[x] + b] - s_mean[x];
      hr_res[(e0 + x) * ph2pad + q] = o;
    }
  }
}

// Eq. 10 for every projection and the key fold of every table; a thread takes
// R feature rows and the block's tables (blockIdx.y: a share of the L), whose
// alpha / beta are staged in shared memory.  Bound by the multiply-adds (L k D
// a row) and the operations beside them:
// - two rows a thread share each 16-byte read of the projections, where the rows
//   are many and long enough (launch_hash);
// - floor(t / w) comes from a multiplication with 1 / w unless the product
//   lies within its error of a whole number (or is not finite, or so small
//   that it could have been rounded to 0), which takes the division (one short
//   row a thread divides: its multiply-adds leave no room for the tests);
// - a pair of keys leaves in one 16-byte store.
// 1M rows, D = 25, L = k = 16: 755 us with one row a thread and a division a
// projection, 631 us so.  Few rows split the tables over blocks instead.
template <int D, int R>
__global__ void __launch_bounds__(128) k_hash(const float* __restrict__ feat, int dpad, int64_t n,
                                              const float* __restrict__ alpha, const float* __restrict__ beta,
                                              int L, int per, int k, float w, uint64_t* __restrict__ keys) {
  // projections staged with rows padded to DP floats (16-byte loads; the
  // multiply-adds keep the order of the feature's values)
  constexpr int DP = (D + 3) / 4 * 4;
  extern __shared__ float4 s_ab4[];
  float* s_ab = reinterpret_cast<float*>(s_ab4);
  const int l0 = blockIdx.y * per, l1 = min(L, l0 + per);
  const int nproj = (l1 - l0) * k, p0 = l0 * k;
  for (int t = threadIdx.x; t < nproj * DP; t += blockDim.x) {
    const int pj = t / DP, q = t % DP;
    s_ab[t] = q < D ? alpha[(p0 + pj) * D + q] : 0.f;
  }
  for (int t = threadIdx.x; t < nproj; t += blockDim.x) s_ab[nproj * DP + t] = beta[p0 + t];
  __syncthreads();
  const int64_t r0 = (int64_t)blockIdx.x * (128 * R) + threadIdx.x;
  if (r0 >= n) return;
  float v[R][DP];
#pragma unroll
  for (int y = 0; y < R; ++y) {
    const int64_t r = r0 + y * 128 < n ? r0 + y * 128 : r0;   // past the end: the first row again, not stored
    const float4* f4 = reinterpret_cast<const float4*>(feat + r * dpad);
#pragma unroll
    for (int q4 = 0; q4 < DP / 4; ++q4) {
      const float4 x = f4[q4];
      v[y][4 * q4] = x.x;
      v[y][4 * q4 + 1] = x.y;
      v[y][4 * q4 + 2] = x.z;
      v[y][4 * q4 + 3] = x.w;
    }
  }
  const float* s_beta = s_ab + nproj * DP;
  const float rw = w < 1e37f ? __frcp_rn(w) : NAN;   // a reciprocal too small for 24 bits: always divide
  // rows of keys start on 16 bytes (l0 is even; a caller's buffer may not)
  const bool pairs = (L & 1) == 0 && ((uintptr_t)keys & 15) == 0;
  uint64_t held[R];
  for (int l = l0; l < l1; ++l) {
    uint64_t x[R];
#pragma unroll
    for (int y = 0; y < R; ++y) x[y] = (uint64_t)l;
    for (int j = 0; j < k; ++j) {
      const int pj = (l - l0) * k + j;
      const float4* a4 = s_ab4 + pj * (DP / 4);
      float acc[R];
#pragma unroll
      for (int y = 0; y < R; ++y) acc[y] = 0.f;
#pragma unroll
      for (int q4 = 0; q4 < DP / 4; ++q4) {
        const float4 av = a4[q4];
#pragma unroll
        for (int y = 0; y < R; ++y) {
          acc[y] = fmaf(av.x, v[y][4 * q4], acc[y]);
          if (4 * q4 + 1 < D) acc[y] = fmaf(av.y, v[y][4 * q4 + 1], acc[y]);
          if (4 * q4 + 2 < D) acc[y] = fmaf(av.z, v[y][4 * q4 + 2], acc[y]);
          if (4 * q4 + 3 < D) acc[y] = fmaf(av.w, v[y][4 * q4 + 3], acc[y]);
        }
      }
      const float be = s_beta[pj];
#pragma unroll
      for (int y = 0; y < R; ++y) {
        const float t = acc[y] + be;
        // t * rw is within 2^-23 |t / w| of t / w, the quotient within 2^-24
        float fl;
        bool divide = true;
        if constexpr (R > 1 || D >= 25) {
          const float u = t * rw;
          fl = floorf(u);
          const float off = fabsf(u - rintf(u));
          divide = !(off > 4e-7f * fabsf(u) && off > 1e-30f && fabsf(u) < 1e9f);
        }
        if (divide) fl = floorf(__fdiv_rn(t, w));
        x[y] = zoom_fold_step(x[y], (int)fl, j);
      }
    }
#pragma unroll
    for (int y = 0; y < R; ++y) {
      const int64_t r = r0 + y * 128;
      if (r >= n) continue;
      if (!pairs) keys[r * L + l] = x[y];
      else if (l & 1) *reinterpret_cast<ulonglong2*>(keys + r * L + l - 1) = make_ulonglong2(held[y], x[y]);
      held[y] = x[y];
    }
  }
  // Launched beside the kernel before it (launch_hash): that one has to be
  // complete before this one is, for what follows both on the stream.
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ---------------------------------------------------------------------------
// LSD radix sort of (uint64 key, int32 id) pairs, 8 bits per pass, stable.
// ---------------------------------------------------------------------------

constexpr int RS_THREADS = 256;
constexpr int RS_TILE = 4096;
constexpr int SCAN_SEG = 4096;

__global__ void k_extract_column(const uint64_t* __restrict__ src, int L, int l, int64_t n,
                                 uint64_t* __restrict__ keys, int32_t* __restrict__ ids) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  keys[i] = src[i * L + l];
  ids[i] = (int32_t)i;
}

__global__ void k_radix_hist(const uint64_t* __restrict__ keys, int64_t n, int shift,
                             int32_t* __restrict__ hist, int ntiles) {
  __shared__ int h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  int64_t base = (int64_t)blockIdx.x * RS_TILE;
  // lanes of equal digit add their count once (digits of compacted ranks
  // take few values, which would pile the atomics onto a few counters)
  const unsigned lt = (1u << (threadIdx.x & 31)) - 1u;
  for (int t = threadIdx.x; t < RS_TILE; t += RS_THREADS) {
    int64_t g = base + t;
    const int digit = g < n ? (int)((keys[g] >> shift) & 255) : 256;
    const unsigned peers = __match_any_sync(0xffffffffu, digit);
    if (digit < 256 && (peers & lt) == 0) atomicAdd(&h[digit], __popc(peers));
  }
  __syncthreads();
  hist[(int64_t)threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}

// Stable scatter: items of a tile are ranked in index order.  The tile is
// processed in chunks of 256 (one item per thread); within a chunk,
// __match_any_sync groups lanes of equal digit, and per-digit prefix counts
// over the warps give each item its place after all earlier items.
__global__ void k_radix_scatter(const uint64_t* __restrict__ kin, const int32_t* __restrict__ vin,
                                uint64_t* __restrict__ kout, int32_t* __restrict__ vout, int64_t n,
                                int shift, const int32_t* __restrict__ offs, int ntiles) {
  __shared__ int run[256];
  __shared__ int wh[RS_THREADS / 32][256];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  run[tid] = offs[(int64_t)tid * ntiles + blockIdx.x];
  const unsigned lt = (1u << lane) - 1u;
  for (int c = 0; c < RS_TILE / RS_THREADS; ++c) {
    int64_t g = (int64_t)blockIdx.x * RS_TILE + c * RS_THREADS + tid;
    bool valid = g < n;
    uint64_t key = valid ? kin[g] : 0ull;
    int32_t val = valid ? vin[g] : 0;
    int digit = valid ? (int)((key >> shift) & 255) : 256;
    for (int q = tid; q < (RS_THREADS / 32) * 256; q += RS_THREADS) (&wh[0][0])[q] = 0;
    __syncthreads();
    unsigned peers = __match_any_sync(0xffffffffu, digit);
    int rank = __popc(peers & lt);
    if (valid && rank == 0) wh[warp][digit] = __popc(peers);
    __syncthreads();
    {
      int s = run[tid];
#pragma unroll
      for (int q = 0; q < RS_THREADS / 32; ++q) {
        int t = wh[q][tid];
        wh[q][tid] = s;
        s += t;
      }
      run[tid] = s;
    }
    __syncthreads();
    if (valid) {
      int p = wh[warp][digit] + rank;
      kout[p] = key;
      vout[p] = val;
    }
    __syncthreads();
  }
}

// Exclusive scan of int32 in three phases: per-segment sums, a one-block
// scan of the sums, per-segment scans with the segment offset.
__device__ __forceinline__ int block_exclusive_scan(int v, int* s_warp, int& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int w = lane < nw ? s_warp[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    s_warp[lane] = w;
  }
  __syncthreads();
  int excl = x - v + (warp > 0 ? s_warp[warp - 1] : 0);
  total = s_warp[nw - 1];
  __syncthreads();
  return excl;
}

__global__ void k_scan_reduce(const int32_t* __restrict__ in, int64_t n, int32_t* __restrict__ part) {
  __shared__ int s_warp[32];
  int64_t base = (int64_t)blockIdx.x * SCAN_SEG;
  int acc = 0;
  for (int t = threadIdx.x; t < SCAN_SEG; t += blockDim.x) {
    int64_t g = base + t;
    if (g < n) acc += in[g];
  }
  int total;
  block_exclusive_scan(acc, s_warp, total);
  if (threadIdx.x == 0) part[blockIdx.x] = total;
}

__global__ void k_scan_partials(int32_t* __restrict__ part, int np) {
  __shared__ int s_warp[32];
  // each thread scans a contiguous run of parts sequentially
  const int per = (np + blockDim.x - 1) / blockDim.x;
  int b0 = threadIdx.x * per;
  int acc = 0;
  for (int q = 0; q < per; ++q)
    if (b0 + q < np) acc += part[b0 + q];
  int total;
  int ex = block_exclusive_scan(acc, s_warp, total);
  for (int q = 0; q < per; ++q)
    if (b0 + q < np) {
      int t = part[b0 + q];
      part[b0 + q] = ex;
      ex += t;
    }
}

__global__ void k_scan_apply(const int32_t* __restrict__ in, int64_t n, const int32_t* __restrict__ part,
                             int32_t* __restrict__ out) {
  __shared__ int s_warp[32];
  constexpr int PER = SCAN_SEG / 256;  // launched with 256 threads
  int64_t base = (int64_t)blockIdx.x * SCAN_SEG + threadIdx.x * PER;
  int v[PER];
  int acc = 0;
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    int64_t g = base + q;
    v[q] = g < n ? in[g] : 0;
    acc += v[q];
  }
  int total;
  int ex = block_exclusive_scan(acc, s_warp, total) + part[blockIdx.x];
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    int64_t g = base + q;
    if (g < n) out[g] = ex;
    ex += v[q];
  }
}

cudaError_t exclusive_scan(const int32_t* in, int32_t* out, int64_t n, int32_t* part, cudaStream_t st) {
  int nseg = (int)((n + SCAN_SEG - 1) / SCAN_SEG);
  k_scan_reduce<<<nseg, 256, 0, st>>>(in, n, part);
  k_scan_partials<<<1, 1024, 0, st>>>(part, nseg);
  k_scan_apply<<<nseg, 256, 0, st>>>(in, n, part, out);
  return cudaGetLastError();
}

__global__ void k_csr_heads(const uint64_t* __restrict__ keys, int64_t n, int32_t* __restrict__ head) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  head[i] = (i == 0 || keys[i] != keys[i - 1]) ? 1 : 0;
}

__global__ void k_csr_write(const uint64_t* __restrict__ keys, const int32_t* __restrict__ head,
                            const int32_t* __restrict__ pos, int64_t n, uint64_t* __restrict__ ukeys,
                            int32_t* __restrict__ offs, int32_t* __restrict__ nuniq) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  if (head[i]) {
    ukeys[pos[i]] = keys[i];
    offs[pos[i]] = (int32_t)i;
  }
  if (i == n - 1) {
    int32_t u = pos[i] + head[i];
    offs[u] = (int32_t)n;
    *nuniq = u;
  }
}

// ---------------------------------------------------------------------------
// Key compaction for the bins (a3): a table of N entries holds few distinct
// keys (68 to 661 per table with 1M pairs), so the 64-bit keys are replaced by
// their rank among the table's distinct keys, and the stable sort by key
// becomes a stable sort by a 12-bit rank: 2 radix passes of 8 bits instead
// of 8.  Distinct keys go into a small open-addressing set per table (linear
// probing, a slot claimed by a 64-bit compare-and-swap; the one key equal to
// the empty marker is recorded by a flag); one block per table sorts them in
// shared memory and gives every slot its rank.  A table with more distinct
// keys than kKeySetCap keeps the 64-bit radix sort.
// ---------------------------------------------------------------------------
constexpr int kKeySetCap = 4096;            // distinct keys per table for the compacted sort
constexpr int kKeySetSlots = 2 * kKeySetCap;
constexpr uint64_t kEmptyKey = ~0ull;

__device__ __forceinline__ uint32_t keyset_hash(uint64_t k) {
  k ^= k >> 31;
  k *= 0x7FB5D329728EA185ull;
  return (uint32_t)(k >> 51) & (kKeySetSlots - 1);
}

// One thread per entry: its L keys (one 128-byte row) into the L sets.
__global__ void k_keyset_insert(const uint64_t* __restrict__ dkeys, int64_t n, int L, uint64_t* slots,
                                uint32_t* __restrict__ count, uint32_t* __restrict__ eflag,
                                uint32_t* __restrict__ full) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  for (int l = 0; l < L; ++l) {
    const uint64_t key = dkeys[i * L + l];
    if (key == kEmptyKey) {
      if (atomicOr(eflag + l, 1u) == 0u) atomicAdd(count + l, 1u);
      continue;
    }
    uint64_t* set = slots + (int64_t)l * kKeySetSlots;
    uint32_t h = keyset_hash(key);
    int p = 0;
    for (; p < kKeySetSlots; ++p, h = (h + 1) & (kKeySetSlots - 1)) {
      const uint64_t cur = *(volatile uint64_t*)(set + h);
      if (cur == key) break;
      if (cur == kEmptyKey) {
        const unsigned long long old = atomicCAS((unsigned long long*)(set + h), (unsigned long long)kEmptyKey,
                                                 (unsigned long long)key);
        if (old == kEmptyKey) {
          atomicAdd(count + l, 1u);
          break;
        }
        if (old == key) break;
      }
    }
    if (p == kKeySetSlots) atomicOr(full + l, 1u);   // no free slot left: the table keeps the 64-bit sort
  }
}

// One block (1024 threads) per table with at most kKeySetCap distinct keys:
// the set's keys sorted ascending (bitonic, in shared memory) into ukeys,
// and the rank of each slot's key (and of the empty-marker key) recorded.
__global__ void __launch_bounds__(1024) k_keyset_rank(const uint64_t* __restrict__ slots,
                                                      const uint32_t* __restrict__ eflag,
                                                      const uint32_t* __restrict__ compact, int64_t n,
                                                      uint64_t* __restrict__ ukeys, int32_t* __restrict__ nuniq,
                                                      uint16_t* __restrict__ slot_rank,
                                                      uint16_t* __restrict__ erank) {
  __shared__ uint64_t sk[kKeySetCap];
  __shared__ uint16_t ss[kKeySetCap];   // slot of each key (kKeySetSlots: the empty-marker key)
  __shared__ int m;
  const int l = blockIdx.x;
  if (!compact[l]) return;   // block-uniform
  if (threadIdx.x == 0) m = 0;
  __syncthreads();
  const uint64_t* set = slots + (int64_t)l * kKeySetSlots;
  for (int h = threadIdx.x; h < kKeySetSlots; h += blockDim.x) {
    const uint64_t k = set[h];
    if (k != kEmptyKey) {
      const int j = atomicAdd(&m, 1);
      sk[j] = k;
      ss[j] = h;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && eflag[l]) {   // the empty-marker key is the largest of all
    sk[m] = kEmptyKey;
    ss[m] = kKeySetSlots;
    ++m;
  }
  __syncthreads();
  const int u = m;
  int pw = 1;
  while (pw < u) pw <<= 1;
  for (int j = u + threadIdx.x; j < pw; j += blockDim.x) {   // padding sorts after every real key
    sk[j] = kEmptyKey;
    ss[j] = 0xFFFF;
  }
  __syncthreads();
  for (int k = 2; k <= pw; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < pw; i += blockDim.x) {
        const int o = i ^ j;
        if (o > i) {
          const bool up = (i & k) == 0;
          const bool gt = sk[i] > sk[o] || (sk[i] == sk[o] && ss[i] > ss[o]);
          if (gt == up) {
            const uint64_t tk = sk[i];
            sk[i] = sk[o];
            sk[o] = tk;
            const uint16_t ts = ss[i];
            ss[i] = ss[o];
            ss[o] = ts;
          }
        }
      }
      __syncthreads();
    }
  }
  for (int r = threadIdx.x; r < u; r += blockDim.x) {
    ukeys[(int64_t)l * n + r] = sk[r];
    if (ss[r] < kKeySetSlots) slot_rank[(int64_t)l * kKeySetSlots + ss[r]] = (uint16_t)r;
    else erank[l] = (uint16_t)r;
  }
  if (threadIdx.x == 0) nuniq[l] = u;
}

// One thread per entry: the rank of each of its keys in its table's set
// (compacted tables only).
__global__ void k_keyset_lookup(const uint64_t* __restrict__ dkeys, int64_t n, int L,
                                const uint64_t* __restrict__ slots, const uint16_t* __restrict__ slot_rank,
                                const uint16_t* __restrict__ erank, const uint32_t* __restrict__ compact,
                                uint16_t* __restrict__ rank) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  for (int l = 0; l < L; ++l) {
    if (!compact[l]) continue;
    const uint64_t key = dkeys[i * L + l];
    uint16_t r = 0;
    if (key == kEmptyKey) {
      r = erank[l];
    } else {
      const uint64_t* set = slots + (int64_t)l * kKeySetSlots;
      uint32_t h = keyset_hash(key);
      for (int p = 0; p < kKeySetSlots; ++p, h = (h + 1) & (kKeySetSlots - 1)) {
        if (set[h] == key) {
          r = slot_rank[(int64_t)l * kKeySetSlots + h];
          break;
        }
      }
    }
    rank[(int64_t)l * n + i] = r;
  }
}

__global__ void k_rank_pairs(const uint16_t* __restrict__ rank, int64_t n, uint64_t* __restrict__ keys,
                             int32_t* __restrict__ ids) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  keys[i] = rank[i];
  ids[i] = (int32_t)i;
}

// The same stable radix sort by rank for every table at once (blockIdx.y:
// the table).  The histogram is laid out [table][digit][tile], so one
// exclusive scan over all of it gives each item its position in the
// concatenated [table][n] output: a table's items land after every earlier
// table's n items.  ids_in == nullptr: the items' ids are their indices.
__global__ void k_rank_hist_b(const uint16_t* __restrict__ r, int64_t n, int shift, int32_t* __restrict__ hist,
                              int ntiles) {
  __shared__ int h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  const uint16_t* rt = r + (int64_t)blockIdx.y * n;
  const int64_t base = (int64_t)blockIdx.x * RS_TILE;
  const unsigned lt = (1u << (threadIdx.x & 31)) - 1u;
  for (int t = threadIdx.x; t < RS_TILE; t += RS_THREADS) {
    const int64_t g = base + t;
    const int digit = g < n ? (int)((rt[g] >> shift) & 255) : 256;
    const unsigned peers = __match_any_sync(0xffffffffu, digit);
    if (digit < 256 && (peers & lt) == 0) atomicAdd(&h[digit], __popc(peers));
  }
  __syncthreads();
  hist[((int64_t)blockIdx.y * 256 + threadIdx.x) * ntiles + blockIdx.x] = h[threadIdx.x];
}

__global__ void k_rank_scatter_b(const uint16_t* __restrict__ rin, const int32_t* __restrict__ ids_in,
                                 uint16_t* __restrict__ rout, int32_t* __restrict__ ids_out, int64_t n, int shift,
                                 const int32_t* __restrict__ offs, int ntiles) {
  __shared__ int run[256];
  __shared__ int wh[RS_THREADS / 32][256];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t tb = (int64_t)blockIdx.y * n;   // this table's slice of the inputs
  run[tid] = offs[((int64_t)blockIdx.y * 256 + tid) * ntiles + blockIdx.x];
  const unsigned lt = (1u << lane) - 1u;
  for (int c = 0; c < RS_TILE / RS_THREADS; ++c) {
    const int64_t g = (int64_t)blockIdx.x * RS_TILE + c * RS_THREADS + tid;
    const bool valid = g < n;
    const uint16_t key = valid ? rin[tb + g] : 0;
    const int32_t val = valid ? (ids_in ? ids_in[tb + g] : (int32_t)g) : 0;
    const int digit = valid ? (int)((key >> shift) & 255) : 256;
    for (int q = tid; q < (RS_THREADS / 32) * 256; q += RS_THREADS) (&wh[0][0])[q] = 0;
    __syncthreads();
    const unsigned peers = __match_any_sync(0xffffffffu, digit);
    const int rank = __popc(peers & lt);
    if (valid && rank == 0) wh[warp][digit] = __popc(peers);
    __syncthreads();
    {
      int sacc = run[tid];
#pragma unroll
      for (int q = 0; q < RS_THREADS / 32; ++q) {
        const int t = wh[q][tid];
        wh[q][tid] = sacc;
        sacc += t;
      }
      run[tid] = sacc;
    }
    __syncthreads();
    if (valid) {
      const int64_t pos = (int64_t)wh[warp][digit] + rank;
      rout[pos] = key;
      ids_out[pos] = val;
    }
    __syncthreads();
  }
}

// Bin offsets of every table from its rank-sorted ranks (blockIdx.y: table).
__global__ void k_csr_rank_offsets_b(const uint16_t* __restrict__ r, int64_t n, int32_t* __restrict__ offs) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint16_t* rt = r + (int64_t)blockIdx.y * n;
  int32_t* ot = offs + (int64_t)blockIdx.y * (n + 1);
  if (i == 0 || rt[i] != rt[i - 1]) ot[rt[i]] = (int32_t)i;
  if (i == n - 1) ot[rt[i] + 1] = (int32_t)n;
}

// Offsets of the runs of a rank-sorted table (its keys already written by
// k_keyset_rank): a run starts where the rank changes, and the rank is the
// run's index.
__global__ void k_csr_rank_offsets(const uint64_t* __restrict__ r, int64_t n, int32_t* __restrict__ offs) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  if (i == 0 || r[i] != r[i - 1]) offs[r[i]] = (int32_t)i;
  if (i == n - 1) offs[r[i] + 1] = (int32_t)n;
}

}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------

cudaError_t launch_degrade_exact(const float* hr, int H, int W, int s, double sigma, float* lr,
                                 cudaStream_t st) {
  double w1[kMaxScale + 2];
  degrade_weights_1d(s, sigma, w1);
  PairWeights pw;
  pw.n = s + 2;
  for (int a = 0; a < s + 2; ++a)
    for (int b = 0; b < s + 2; ++b) {
      double p = w1[a] * w1[b];
      float hi = (float)p;
      pw.hi[a * pw.n + b] = hi;
      pw.lo[a * pw.n + b] = (float)(p - (double)hi);
    }
  int h = H / s, w = W / s;
  dim3 blk(32, 8), grd((w + 31) / 32, (h + 7) / 8);
  k_degrade_exact<<<grd, blk, 0, st>>>(hr, H, W, s, pw, lr, h, w);
  return cudaGetLastError();
}

cudaError_t launch_dict_gather(const float* const* d_lr_images, const int32_t* d_lr_h,
                               const int32_t* d_lr_w, const float* const* d_hr_images,
                               const int32_t* d_hr_w, const int32_t* d_pos, int64_t n, int P, int s,
                               zoom_dict d, cudaStream_t st) {
  int blocks = (int)((n + kGatherRows - 1) / kGatherRows);
#define ZOOM_GATHER(PP, FF)                                                                     \
  k_dict_gather<PP, FF><<<blocks, kGatherRows, 0, st>>>(d_lr_images, d_lr_h, d_lr_w, d_hr_images, \
                                                        d_hr_w, d_pos, n, s, d->ph2pad, d->lr_pix, \
                                                        d->feat, d->mu, d->norm2, d->hr_res)
  if (P == 3 && d->feature == 0) ZOOM_GATHER(3, 0);
  else if (P == 5 && d->feature == 0) ZOOM_GATHER(5, 0);
  else if (P == 3 && d->feature == 1) ZOOM_GATHER(3, 1);
  else if (P == 5 && d->feature == 1) ZOOM_GATHER(5, 1);
  else if (P == 3 && d->feature == 2) ZOOM_GATHER(3, 2);
  else if (P == 5 && d->feature == 2) ZOOM_GATHER(5, 2);
  else return cudaErrorInvalidValue;
#undef ZOOM_GATHER
  return cudaGetLastError();
}

cudaError_t launch_hash(const float* feat, int dpad, int d, int64_t n, const float* alpha,
                        const float* beta, int L, int k, float w, uint64_t* keys, cudaStream_t st,
                        bool beside) {
  if (n == 0) return cudaSuccess;
  // Two rows a thread where that was faster (L = k = 16, one / two rows, us):
  // D = 9 never (258,064 rows 136 / 144, 1M 450 / 452), D = 18 from 800,000 rows
  // (515,524: 307 / 311, 1M: 564 / 546), D = 25 from 100,000 (81,796: 101 / 108,
  // 112,896: 112 / 102, 1M: 706 / 641), D = 50 from two blocks of 128 for each
  // of about 150 SMs (81,796: 194 / 157).  With one row the tables (in twos: see
  // the stores) go over blocks until there are as many (the 2x zoom of 64x64
  // with 3,844 queries: 189.6 us on 31 blocks, 182.9 us so).
  const bool two = n >= (d == 50 ? 2 * 128 * 304 : d == 25 ? 100000 : d == 18 ? 800000 : INT64_MAX);
  const int64_t rows = two ? 256 : 128, blocks = (n + rows - 1) / rows;
  int per = (L + 1) / 2 * 2;
  while (per > 2 && blocks * ((L + per - 1) / per) < 304) per = (per / 2 + 1) / 2 * 2;
  const size_t smem = (size_t)(per < L ? per : L) * k * ((d + 3) / 4 * 4 + 1) * sizeof(float);
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks, (unsigned)((L + per - 1) / per));
  cfg.blockDim = dim3(128);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = beside ? 1 : 0;
  cudaError_t e = cudaSuccess;
#define ZOOM_HASH1(DD, RR)                                                                                  \
  do {                                                                                                      \
    if (smem > 48 * 1024) {                                                                                 \
      e = cudaFuncSetAttribute(k_hash<DD, RR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);     \
      if (e != cudaSuccess) return e;                                                                       \
    }                                                                                                       \
    e = cudaLaunchKernelEx(&cfg, k_hash<DD, RR>, feat, dpad, n, alpha, beta, L, per, k, w, keys);           \
  } while (0)
#define ZOOM_HASH(DD)            \
  do {                           \
    if (two) ZOOM_HASH1(DD, 2);  \
    else ZOOM_HASH1(DD, 1);      \
  } while (0)
  switch (d) {
    case 9: ZOOM_HASH(9); break;
    case 25: ZOOM_HASH(25); break;
    case 18: ZOOM_HASH(18); break;
    case 50: ZOOM_HASH(50); break;
    default: return cudaErrorInvalidValue;
  }
#undef ZOOM_HASH1
#undef ZOOM_HASH
  return e != cudaSuccess ? e : cudaGetLastError();
}

namespace {
__global__ void k_make_pairs(const int32_t* __restrict__ keys32, int64_t n, uint64_t* __restrict__ keys,
                             int32_t* __restrict__ vals) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  keys[i] = (uint64_t)(uint32_t)keys32[i];
  vals[i] = (int32_t)i;
}
}  // namespace

// Stable sort of the positions 0..n-1 by a non-negative int32 key, then the
// CSR of equal-key runs: sorted_pos[n] (positions grouped by key, ascending
// within a run), ukeys[u] (run keys, ascending), offs[u+1], *nuniq = u.
cudaError_t sort_keys_csr(const int32_t* keys32, int64_t n, int32_t* sorted_pos, uint64_t* ukeys,
                          int32_t* offs, int32_t* nuniq, void* scratch, size_t scratch_bytes,
                          cudaStream_t st) {
  if (scratch_bytes < csr_scratch_bytes(n)) return cudaErrorInvalidValue;
  const int ntiles = (int)((n + RS_TILE - 1) / RS_TILE);
  char* p = (char*)scratch;
  uint64_t* ka = (uint64_t*)p; p += n * 8;
  uint64_t* kb = (uint64_t*)p; p += n * 8;
  int32_t* va = (int32_t*)p; p += n * 4;
  int32_t* vb = (int32_t*)p; p += n * 4;
  int32_t* hist = (int32_t*)p; p += (int64_t)256 * ntiles * 4;
  int32_t* head = (int32_t*)p; p += n * 4;
  int32_t* pos = (int32_t*)p; p += n * 4;
  int32_t* part = (int32_t*)p;
  const int eb = (int)((n + 255) / 256);
  k_make_pairs<<<eb, 256, 0, st>>>(keys32, n, ka, va);
  uint64_t* kin = ka; uint64_t* kout = kb;
  int32_t* vin = va; int32_t* vout = vb;
  for (int shift = 0; shift < 32; shift += 8) {   // keys fit in 32 bits
    k_radix_hist<<<ntiles, RS_THREADS, 0, st>>>(kin, n, shift, hist, ntiles);
    cudaError_t e = exclusive_scan(hist, hist, (int64_t)256 * ntiles, part, st);
    if (e != cudaSuccess) return e;
    k_radix_scatter<<<ntiles, RS_THREADS, 0, st>>>(kin, vin, kout, vout, n, shift, hist, ntiles);
    std::swap(kin, kout);
    std::swap(vin, vout);
  }
  k_csr_heads<<<eb, 256, 0, st>>>(kin, n, head);
  cudaError_t e = exclusive_scan(head, pos, n, part, st);
  if (e != cudaSuccess) return e;
  k_csr_write<<<eb, 256, 0, st>>>(kin, head, pos, n, ukeys, offs, nuniq);
  cudaMemcpyAsync(sorted_pos, vin, n * 4, cudaMemcpyDeviceToDevice, st);
  return cudaGetLastError();
}

size_t csr_scratch_bytes(int64_t n) {
  int64_t ntiles = (n + RS_TILE - 1) / RS_TILE;
  int64_t hist = 256 * ntiles;
  int64_t nseg = (std::max<int64_t>(hist, n) + SCAN_SEG - 1) / SCAN_SEG;
  // keys x2, ids x2, hist, head, pos, parts
  return (size_t)(2 * n * 8 + 2 * n * 4 + hist * 4 + 2 * n * 4 + nseg * 4 + 1024);
}

size_t csr_build_scratch_bytes(int64_t n, int L) {
  // the radix sort's buffers, then the key sets, the slot ranks, the per-table
  // flags, the 16-bit ranks of every entry in every table (twice) and their
  // ids, and the all-table histogram with its scan partials
  const int64_t ntiles = (n + RS_TILE - 1) / RS_TILE;
  const int64_t hist = (int64_t)L * 256 * ntiles;
  return csr_scratch_bytes(n) + 256 + (size_t)L * kKeySetSlots * 8 + (size_t)L * kKeySetSlots * 2 +
         (size_t)5 * L * 4 + 256 + (size_t)L * n * 2 + 256 + (size_t)L * n * 2 + 256 + (size_t)L * n * 4 + 256 +
         (size_t)hist * 4 + 256 + (size_t)((hist + SCAN_SEG - 1) / SCAN_SEG) * 4 + 1024;
}

cudaError_t build_csr_tables(zoom_index ix, void* scratch, size_t scratch_bytes, cudaStream_t st) {
  const int64_t n = ix->dict->n;
  const int L = ix->L;
  if (scratch_bytes < csr_build_scratch_bytes(n, L)) return cudaErrorInvalidValue;
  const int ntiles = (int)((n + RS_TILE - 1) / RS_TILE);
  char* p = (char*)scratch;
  uint64_t* ka = (uint64_t*)p; p += n * 8;
  uint64_t* kb = (uint64_t*)p; p += n * 8;
  int32_t* va = (int32_t*)p; p += n * 4;
  int32_t* vb = (int32_t*)p; p += n * 4;
  int32_t* hist = (int32_t*)p; p += (int64_t)256 * ntiles * 4;
  int32_t* head = (int32_t*)p; p += n * 4;
  int32_t* pos = (int32_t*)p; p += n * 4;
  int32_t* part = (int32_t*)p;
  // compaction arrays after the radix sort's (csr_scratch_bytes(n) of them)
  char* q = (char*)scratch + ((csr_scratch_bytes(n) + 255) & ~(size_t)255);
  uint64_t* slots = (uint64_t*)q; q += (size_t)L * kKeySetSlots * 8;
  uint16_t* slot_rank = (uint16_t*)q; q += (size_t)L * kKeySetSlots * 2;
  uint32_t* flags = (uint32_t*)q; q += (size_t)5 * L * 4;   // count, eflag, full, compact, erank (16-bit)
  uint32_t* count = flags;
  uint32_t* eflag = flags + L;
  uint32_t* full = flags + 2 * L;
  uint32_t* compact = flags + 3 * L;
  uint16_t* erank = (uint16_t*)(flags + 4 * L);
  q = (char*)(((uintptr_t)q + 255) & ~(uintptr_t)255);
  uint16_t* rank = (uint16_t*)q; q += (size_t)L * n * 2;
  q = (char*)(((uintptr_t)q + 255) & ~(uintptr_t)255);
  uint16_t* rank_b = (uint16_t*)q; q += (size_t)L * n * 2;
  q = (char*)(((uintptr_t)q + 255) & ~(uintptr_t)255);
  int32_t* ids_b = (int32_t*)q; q += (size_t)L * n * 4;
  q = (char*)(((uintptr_t)q + 255) & ~(uintptr_t)255);
  int32_t* hist_b = (int32_t*)q; q += (size_t)L * 256 * ntiles * 4;
  q = (char*)(((uintptr_t)q + 255) & ~(uintptr_t)255);
  int32_t* part_b = (int32_t*)q;
  const int eb = (int)((n + 255) / 256);

  // distinct keys per table; the host reads the counts (the build ends with
  // a stream synchronisation anyway)
  cudaError_t e = cudaMemsetAsync(slots, 0xFF, (size_t)L * kKeySetSlots * 8, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(flags, 0, (size_t)5 * L * 4, st);
  if (e != cudaSuccess) return e;
  k_keyset_insert<<<eb, 256, 0, st>>>(ix->dkeys, n, L, slots, count, eflag, full);
  std::vector<uint32_t> h_flags((size_t)3 * L);
  e = cudaMemcpyAsync(h_flags.data(), flags, (size_t)3 * L * 4, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return e;
  std::vector<uint32_t> h_compact(L);
  bool any = false;
  for (int l = 0; l < L; ++l) {
    h_compact[l] = h_flags[2 * L + l] == 0 && h_flags[l] <= (uint32_t)kKeySetCap ? 1u : 0u;
    any = any || h_compact[l];
  }
  if (any) {
    e = cudaMemcpyAsync(compact, h_compact.data(), (size_t)L * 4, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return e;
    k_keyset_rank<<<L, 1024, 0, st>>>(slots, eflag, compact, n, ix->ukeys, ix->nuniq, slot_rank, erank);
    k_keyset_lookup<<<eb, 256, 0, st>>>(ix->dkeys, n, L, slots, slot_rank, erank, compact, rank);
    // the copy of h_compact must finish before the vector goes
    e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
  }
  bool all = true;
  uint32_t umax = 0;
  for (int l = 0; l < L; ++l) {
    all = all && h_compact[l];
    umax = std::max(umax, h_flags[l]);
  }
  if (all && (int64_t)L * n < (int64_t{1} << 31)) {   // positions in 32-bit scans
    // every table at once: 1 pass of 8 bits when no table has more than 256
    // distinct keys, else 2; the last pass writes the ids into the index
    const int passes = umax <= 256u ? 1 : 2;
    const dim3 grid(ntiles, L);
    const uint16_t* rin = rank;
    uint16_t* rout = rank_b;
    const int32_t* iin = nullptr;
    for (int ps = 0; ps < passes; ++ps) {
      int32_t* iout = ps == passes - 1 ? ix->ids : ids_b;
      k_rank_hist_b<<<grid, RS_THREADS, 0, st>>>(rin, n, 8 * ps, hist_b, ntiles);
      e = exclusive_scan(hist_b, hist_b, (int64_t)L * 256 * ntiles, part_b, st);
      if (e != cudaSuccess) return e;
      k_rank_scatter_b<<<grid, RS_THREADS, 0, st>>>(rin, iin, rout, iout, n, 8 * ps, hist_b, ntiles);
      iin = iout;
      rin = rout;
      rout = rout == rank_b ? rank : rank_b;
    }
    k_csr_rank_offsets_b<<<dim3(eb, L), 256, 0, st>>>(rin, n, ix->offs);
    return cudaGetLastError();
  }
  for (int l = 0; l < L; ++l) {
    uint64_t* kin = ka; uint64_t* kout = kb;
    int32_t* vin = va; int32_t* vout = vb;
    if (h_compact[l]) {
      // stable sort of the entries by their rank (below 4096): 2 passes of
      // 8 bits, 1 when the table has at most 256 distinct keys
      k_rank_pairs<<<eb, 256, 0, st>>>(rank + (int64_t)l * n, n, ka, va);
      const int bits = h_flags[l] <= 256u ? 8 : 16;
      for (int shift = 0; shift < bits; shift += 8) {
        k_radix_hist<<<ntiles, RS_THREADS, 0, st>>>(kin, n, shift, hist, ntiles);
        e = exclusive_scan(hist, hist, (int64_t)256 * ntiles, part, st);
        if (e != cudaSuccess) return e;
        k_radix_scatter<<<ntiles, RS_THREADS, 0, st>>>(kin, vin, kout, vout, n, shift, hist, ntiles);
        std::swap(kin, kout);
        std::swap(vin, vout);
      }
      k_csr_rank_offsets<<<eb, 256, 0, st>>>(kin, n, ix->offs + (int64_t)l * (n + 1));
    } else {
      k_extract_column<<<eb, 256, 0, st>>>(ix->dkeys, L, l, n, ka, va);
      for (int shift = 0; shift < 64; shift += 8) {
        k_radix_hist<<<ntiles, RS_THREADS, 0, st>>>(kin, n, shift, hist, ntiles);
        e = exclusive_scan(hist, hist, (int64_t)256 * ntiles, part, st);
        if (e != cudaSuccess) return e;
        k_radix_scatter<<<ntiles, RS_THREADS, 0, st>>>(kin, vin, kout, vout, n, shift, hist, ntiles);
        std::swap(kin, kout);
        std::swap(vin, vout);
      }
      k_csr_heads<<<eb, 256, 0, st>>>(kin, n, head);
      e = exclusive_scan(head, pos, n, part, st);
      if (e != cudaSuccess) return e;
      k_csr_write<<<eb, 256, 0, st>>>(kin, head, pos, n, ix->ukeys + (int64_t)l * n,
                                      ix->offs + (int64_t)l * (n + 1), ix->nuniq + l);
    }
    e = cudaMemcpyAsync(ix->ids + (int64_t)l * n, vin, n * 4, cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

