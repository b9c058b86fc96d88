// Search order of the dictionary (index build): the entries sorted along a
// splitting tree, so that 256 consecutive entries (a tile of the tensor-core
// filter) lie close together and have a small bounding box.  A query then
// needs only the tiles whose box comes within its K-th distance
// (kernels_prune.cu).
//
// The tree splits each node at its sample median in the bound coordinate of
// largest variance.  Two levels of sampling keep it to a few launches: one
// block builds the first d1 levels from up to 2048 entries in shared memory; up
// to 1536 further samples per leaf are routed there, and one block per leaf
// builds d2 more levels.  Every entry is then routed (a lookup per level) and
// numbered by arrival at its leaf; the leaves' counts summed give its place
// (two 8-bit radix passes instead took ten launches, 90 us with 65,536 entries,
// 15 us so).
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <float.h>
#include <math.h>

#include <algorithm>

#include "device_common.cuh"
#include "search_tree.cuh"
#include "zoom_internal.h"

namespace {

constexpr int kTreeThreads = 1024;
// The first level's sample counts lie in cache lines of their own: 98,304
// samples that all counted in two lines took 35 us, 15 us so.
constexpr int kCountStride = 32;

// Order-preserving 32-bit key of an FP32 value.
__device__ __forceinline__ uint32_t order_key(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

struct TreeSmem {
  float z[PZ][PT_TOP];
  uint32_t key[PT_TOP];
  uint16_t perm[PT_TOP];
  float var[128 * PZ];
  int dim[128];
};

// Splits n (a power of two, at most PT_TOP) samples depth (at most 7) times;
// block of kTreeThreads.  A node of fewer than two samples sends everything
// left.
__device__ void kd_build(TreeSmem& s, int n, int depth, TreeNode* __restrict__ out) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int t = tid; t < n; t += kTreeThreads) s.perm[t] = (uint16_t)t;
  __syncthreads();
  for (int l = 0; l < depth; ++l) {
    const int nn = 1 << l, m = n >> l;
    if (m < 2) {
      for (int q = tid; q < nn; q += kTreeThreads) out[nn + q] = TreeNode{FLT_MAX, 0};
      continue;
    }
    for (int pr = warp; pr < nn * PZ; pr += kTreeThreads / 32) {
      const int node = pr / PZ, c = pr % PZ;
      float a = 0.f, b = 0.f;
      for (int j = lane; j < m; j += 32) {
        const float v = s.z[c][s.perm[node * m + j]];
        a += v;
        b = fmaf(v, v, b);
      }
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
      }
      if (lane == 0) s.var[pr] = b - a * a / (float)m;
    }
    __syncthreads();
    for (int q = tid; q < nn; q += kTreeThreads) {
      int best = 0;
      for (int c = 1; c < PZ; ++c)
        if (s.var[q * PZ + c] > s.var[q * PZ + best]) best = c;
      s.dim[q] = best;
    }
    __syncthreads();
    for (int t = tid; t < n; t += kTreeThreads) {
      const uint16_t p = s.perm[t];
      // (the value's upper 21 bits: what they round only moves a split a little)
      s.key[t] = (order_key(s.z[s.dim[t / m]][p]) & ~(uint32_t)(PT_TOP - 1)) | p;
    }
    __syncthreads();
    // bitonic sort of every node's m keys, all nodes ascending; a thread has
    // one pair a stage, so that a warp's pairs at distances up to 32 lie in 64
    // keys of its own and only the longer distances need the block's barrier
    static_assert(PT_TOP <= 2 * kTreeThreads && (PT_TOP & (PT_TOP - 1)) == 0, "one pair a thread");
    for (int k = 2; k <= m; k <<= 1) {
      if (k > 64) __syncthreads();
      for (int j = k >> 1; j > 0; j >>= 1) {
        const int a = ((tid & ~(j - 1)) << 1) | (tid & (j - 1)), b = a | j;
        if (tid < n / 2) {
          const bool up = k == m || (a & k) == 0;
          const uint32_t x = s.key[a], y = s.key[b];
          if ((x > y) == up) {
            s.key[a] = y;
            s.key[b] = x;
          }
        }
        if (j > 32) __syncthreads();
        else __syncwarp();
      }
    }
    __syncthreads();
    for (int t = tid; t < n; t += kTreeThreads) s.perm[t] = (uint16_t)(s.key[t] & (PT_TOP - 1));
    __syncthreads();
    for (int q = tid; q < nn; q += kTreeThreads)
      out[nn + q] = TreeNode{s.z[s.dim[q]][s.perm[q * m + m / 2 - 1]], s.dim[q]};
    __syncthreads();
  }
}

struct DctBasis {
  float b[25 * 25];   // [pixel][coefficient] of a P x P block
};

// One block: the variances of all D coefficients over ns (a power of two, at
// most PT_TOP) entries spread over the dictionary, the PZ largest as the basis,
// and the first d1 levels.  Bound by the barriers and shared memory of its one
// SM (73 us with 512 entries, 108 with 2048), so the next kernel is let in at
// once: with the hash beside it the build of 200,000 pairs takes 675 us instead
// of 780.
template <int D>
__global__ void __launch_bounds__(kTreeThreads) k_tree_top(const float* __restrict__ feat, int dpad, int64_t n,
                                                           DctBasis dct, int P2, int ns, int d1,
                                                           float* __restrict__ basis,
                                                           TreeNode* __restrict__ node1) {
  extern __shared__ __align__(16) unsigned char raw[];
  TreeSmem& s = *reinterpret_cast<TreeSmem*>(raw);
  __shared__ float s_dct[25 * 25];
  __shared__ float s_part[D][2][kTreeThreads / 32];
  __shared__ float s_v[D];
  __shared__ int s_pick[PZ];
  __shared__ __align__(16) float s_b[D * PZ];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  for (int t = tid; t < P2 * P2; t += kTreeThreads) s_dct[t] = dct.b[t];
  float f[2][D];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
#pragma unroll
    for (int i = 0; i < D; ++i) f[h][i] = 0.f;
    const int j = tid + h * kTreeThreads;
    if (j < ns) load_feature<D>(feat + (int64_t)j * n / ns * dpad, f[h]);
  }
  __syncthreads();
  constexpr int kBlocks = D == 18 ? 2 : 1;   // [g_x | g_y]
  constexpr int kP2 = D / kBlocks;
#pragma unroll
  for (int blk = 0; blk < kBlocks; ++blk) {
    for (int c = 0; c < kP2; ++c) {
      float v0 = 0.f, v1 = 0.f;
#pragma unroll
      for (int i = 0; i < kP2; ++i) {
        v0 = fmaf(f[0][blk * kP2 + i], s_dct[i * kP2 + c], v0);
        v1 = fmaf(f[1][blk * kP2 + i], s_dct[i * kP2 + c], v1);
      }
      float a = v0 + v1, b = fmaf(v0, v0, v1 * v1);
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
      }
      if (lane == 0) {
        s_part[blk * kP2 + c][0][warp] = a;
        s_part[blk * kP2 + c][1][warp] = b;
      }
    }
  }
  __syncthreads();
  if (tid < D) {
    float a = 0.f, b = 0.f;
    for (int w = 0; w < kTreeThreads / 32; ++w) {
      a += s_part[tid][0][w];
      b += s_part[tid][1][w];
    }
    s_v[tid] = b - a * a / (float)ns;
  }
  __syncthreads();
  if (warp == 0) {
    // the PZ largest, one after the other (equal ones: the lower number); NaN
    // is none
    static_assert(D <= 32, "a coefficient a lane");
    uint64_t key =
        lane < D && s_v[lane] > -FLT_MAX ? ((uint64_t)order_key(s_v[lane]) << 32) | (uint32_t)(64 - lane) : 0ull;
    for (int c = 0; c < PZ; ++c) {
      uint64_t g = key;
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        const uint64_t x = __shfl_xor_sync(0xffffffffu, g, o);
        g = g > x ? g : x;
      }
      const int best = g ? 64 - (int)(uint32_t)g : -1;
      if (lane == 0) s_pick[c] = best;   // -1: fewer coefficients than PZ (the column is zero)
      if (best == lane) key = 0;
    }
  }
  __syncthreads();
  for (int t = tid; t < D * PZ; t += kTreeThreads) {
    const int i = t / PZ, p = s_pick[t % PZ];
    const float b = p >= 0 && i / kP2 == p / kP2 ? s_dct[(i % kP2) * kP2 + p % kP2] : 0.f;
    s_b[t] = b;
    basis[t] = b;
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float z[PZ];
    bound_coords<D>(f[h], reinterpret_cast<const float4*>(s_b), z);
#pragma unroll
    for (int c = 0; c < PZ; ++c) s.z[c][tid + h * kTreeThreads] = z[c];
  }
  __syncthreads();
  kd_build(s, ns, d1, node1);
}

// m samples spread over the dictionary, routed through the first d1 levels
// into their leaf's list (at most PT_TOP each).
template <int D>
__global__ void __launch_bounds__(128) k_tree_sample(const float* __restrict__ feat, int dpad, int64_t n, int64_t m,
                                                     const float* __restrict__ basis,
                                                     const TreeNode* __restrict__ node1, int d1,
                                                     uint32_t* __restrict__ cnt, float* __restrict__ zl) {
  __shared__ __align__(16) float s_b[D * PZ];
  __shared__ float s_z[PZ][128];
  for (int t = threadIdx.x; t < D * PZ; t += 128) s_b[t] = basis[t];
  __syncthreads();
  const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x;
  if (i >= m) return;
  float f[D], z[PZ];
  load_feature<D>(feat + (i * n / m) * dpad, f);
  bound_coords<D>(f, reinterpret_cast<const float4*>(s_b), z);
#pragma unroll
  for (int c = 0; c < PZ; ++c) s_z[c][threadIdx.x] = z[c];
  const int leaf = tree_descend(node1, d1, [&](int c) { return s_z[c][threadIdx.x]; });
  const uint32_t slot = atomicAdd(cnt + leaf * kCountStride, 1u);
  if (slot < PT_TOP) {
    float4* o = reinterpret_cast<float4*>(zl + ((size_t)leaf * PT_TOP + slot) * PZ);
#pragma unroll
    for (int c4 = 0; c4 < PZ / 4; ++c4) o[c4] = make_float4(z[4 * c4], z[4 * c4 + 1], z[4 * c4 + 2], z[4 * c4 + 3]);
  }
}

// One block per first-level leaf: d2 more levels from its samples.
__global__ void __launch_bounds__(kTreeThreads) k_tree_sub(const uint32_t* __restrict__ cnt,
                                                           const float* __restrict__ zl, int d2,
                                                           TreeNode* __restrict__ node2) {
  extern __shared__ __align__(16) unsigned char raw[];
  TreeSmem& s = *reinterpret_cast<TreeSmem*>(raw);
  const int have = (int)min(cnt[blockIdx.x * kCountStride], (uint32_t)PT_TOP);
  int n = 1;
  while (2 * n <= have) n *= 2;
  if (have == 0) n = 0;
  const float* z = zl + (size_t)blockIdx.x * PT_TOP * PZ;
  for (int t = threadIdx.x; t < n * PZ; t += kTreeThreads) s.z[t % PZ][t / PZ] = z[t];
  __syncthreads();
  kd_build(s, n, d2, node2 + ((size_t)blockIdx.x << d2));
}

// Leaf of every entry, and its arrival number there (counts: hist).
template <int D>
__global__ void __launch_bounds__(128) k_tree_route(const float* __restrict__ feat, int dpad, int64_t n,
                                                    const float* __restrict__ basis,
                                                    const TreeNode* __restrict__ node1,
                                                    const TreeNode* __restrict__ node2, int d1, int d2,
                                                    uint16_t* __restrict__ leaf, uint32_t* __restrict__ rank,
                                                    uint32_t* __restrict__ hist) {
  __shared__ __align__(16) float s_b[D * PZ];
  __shared__ float s_z[PZ][128];
  for (int t = threadIdx.x; t < D * PZ; t += 128) s_b[t] = basis[t];
  __syncthreads();
  const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x;
  const unsigned active = __ballot_sync(0xffffffffu, i < n);
  if (i >= n) return;
  float f[D], z[PZ];
  load_feature<D>(feat + i * dpad, f);
  bound_coords<D>(f, reinterpret_cast<const float4*>(s_b), z);
#pragma unroll
  for (int c = 0; c < PZ; ++c) s_z[c][threadIdx.x] = z[c];
  const int lf = tree_leaf(node1, node2, d1, d2, [&](int c) { return s_z[c][threadIdx.x]; });
  leaf[i] = (uint16_t)lf;
  rank[i] = leaf_arrival(hist, lf, active);
}

__global__ void __launch_bounds__(256) k_tree_place(const uint16_t* __restrict__ leaf, const uint32_t* __restrict__ rank,
                                                    const uint32_t* __restrict__ offs, int64_t n,
                                                    int32_t* __restrict__ order) {
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i < n) order[(int64_t)offs[leaf[i]] + rank[i]] = (int32_t)i;
}

// Scaled FP16 box of [lo, hi] with the coordinates' rounding allowed for:
// centre and query are rounded to 11 bits (2^-11 of their magnitude each,
// |query| <= |centre| + half width + gap), |q - c| - h adds 2^-11 of
// itself, and the FP32 coordinates are within about 8e-6 of the largest
// feature norm R.  A box outside FP16's range excludes nothing.
__device__ __forceinline__ void write_box(float lo, float hi, float R, __half* c_out, __half* h_out) {
  const float c = 0.5f * (lo + hi) * PT_SCALE;
  const float h = 0.5f * (hi - lo) * PT_SCALE;
  const float w = h + (h + fabsf(c)) * 1.1e-3f + 8e-6f * PT_SCALE * R + 1e-6f;
  const bool fits = fabsf(c) + w < 30000.f;   // false for NaN too
  *c_out = __float2half_rn(fits ? c : 0.f);
  *h_out = fits ? __float2half_ru(w) : __ushort_as_half((unsigned short)0x7C00u);
}

// One block per tile: the single-term FP16 and BF16 operand rows of its 256
// entries in search order (the layout of the wide-step filter, with three
// ones after the norm's terms), its box and its mean.  stat [tiles][3 PZ + 1]: lo, hi, sum of the coordinates, largest
// ||f||^2.
template <int D, int KC>
__global__ void __launch_bounds__(PT_ROWS) k_tile_operands(
    const float* __restrict__ feat, int dpad, int64_t n, const int32_t* __restrict__ order,
    const float* __restrict__ basis, uint16_t* __restrict__ op_f1, uint16_t* __restrict__ op_bf,
    uint4* __restrict__ box, float* __restrict__ mid, float* __restrict__ stat) {
  static_assert(D + 6 <= KC * 8, "operand layout");
  __shared__ __align__(16) float s_b[D * PZ];
  __shared__ float s_z[PZ + 1][PT_ROWS + 1];
  __shared__ __align__(16) __half s_box[2 * PZ];
  const int r = threadIdx.x;
  const int64_t tile = blockIdx.x, pos = tile * PT_ROWS + r;
  for (int t = r; t < D * PZ; t += PT_ROWS) s_b[t] = basis[t];
  __syncthreads();
  const bool real = pos < n;
  const int id = real ? order[pos] : -1;
  float f[D];
#pragma unroll
  for (int i = 0; i < D; ++i) f[i] = 0.f;
  float n2 = 0.f;
  uint16_t h[KC * 8], b[KC * 8];
#pragma unroll
  for (int k = 0; k < KC * 8; ++k) h[k] = b[k] = 0;
  if (real) {
    load_feature<D>(feat + (int64_t)id * dpad, f);
#pragma unroll
    for (int i = 0; i < D; ++i) {
      n2 = fmaf(f[i], f[i], n2);
      h[i] = __half_as_ushort(__float2half_rn(-2.f * f[i]));
      b[i] = __bfloat16_as_ushort(__float2bfloat16_rn(-2.f * f[i]));
    }
    const __half n1 = __float2half_rn(n2);
    const float r1 = n2 - __half2float(n1);
    const __half nb = __float2half_rn(r1);
    h[D] = __half_as_ushort(n1);
    h[D + 1] = __half_as_ushort(nb);
    h[D + 2] = __half_as_ushort(__float2half_rn(r1 - __half2float(nb)));
    const __nv_bfloat16 m1 = __float2bfloat16_rn(n2);
    const float s1 = n2 - __bfloat162float(m1);
    const __nv_bfloat16 mb = __float2bfloat16_rn(s1);
    b[D] = __bfloat16_as_ushort(m1);
    b[D + 1] = __bfloat16_as_ushort(mb);
    b[D + 2] = __bfloat16_as_ushort(__float2bfloat16_rn(s1 - __bfloat162float(mb)));
#pragma unroll
    for (int t = 0; t < 3; ++t) {   // ones against the queries' thresholds
      h[D + 3 + t] = 0x3C00u;
      b[D + 3 + t] = 0x3F80u;
    }
  } else {
    h[D] = __half_as_ushort(__float2half_rn(60000.f));   // padding never ranks
    b[D] = __bfloat16_as_ushort(__float2bfloat16_rn(60000.f));
  }
#pragma unroll
  for (int kc = 0; kc < KC; ++kc) {
    const size_t o = ((size_t)tile * KC + kc) * (PT_ROWS * 8) + (size_t)r * 8;
    uint4 a, c;
    uint32_t* pa = &a.x;
    uint32_t* pc = &c.x;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      pa[t] = (uint32_t)h[kc * 8 + 2 * t] | ((uint32_t)h[kc * 8 + 2 * t + 1] << 16);
      pc[t] = (uint32_t)b[kc * 8 + 2 * t] | ((uint32_t)b[kc * 8 + 2 * t + 1] << 16);
    }
    *reinterpret_cast<uint4*>(op_f1 + o) = a;
    *reinterpret_cast<uint4*>(op_bf + o) = c;
  }
  float z[PZ];
  bound_coords<D>(f, reinterpret_cast<const float4*>(s_b), z);
#pragma unroll
  for (int c = 0; c < PZ; ++c) s_z[c][r] = z[c];
  s_z[PZ][r] = n2;
  __syncthreads();
  const int rows = (int)min((int64_t)PT_ROWS, n - tile * PT_ROWS);
  const int lane = r & 31, warp = r >> 5;
  float R2 = 0.f;   // every warp needs the largest norm
  for (int j = lane; j < rows; j += 32) R2 = fmaxf(R2, s_z[PZ][j]);
#pragma unroll
  for (int o = 16; o; o >>= 1) R2 = fmaxf(R2, __shfl_xor_sync(0xffffffffu, R2, o));
  for (int c = warp; c < PZ; c += PT_ROWS / 32) {
    float lo = FLT_MAX, hi = -FLT_MAX, sum = 0.f;
    for (int j = lane; j < rows; j += 32) {
      const float v = s_z[c][j];
      lo = fminf(lo, v);
      hi = fmaxf(hi, v);
      sum += v;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
      sum += __shfl_xor_sync(0xffffffffu, sum, o);
    }
    if (lane == 0) {
      write_box(lo, hi, sqrtf(R2), s_box + c, s_box + PZ + c);
      mid[tile * PZ + c] = sum / (float)rows;
      float* st = stat + tile * (3 * PZ + 1);
      st[c] = lo;
      st[PZ + c] = hi;
      st[2 * PZ + c] = sum;
      if (c == 0) st[3 * PZ] = R2;
    }
  }
  __syncthreads();
  if (r < 4) box[tile * 4 + r] = reinterpret_cast<const uint4*>(s_box)[r];
}

// Boxes and means of the super tiles: one warp each, lane c < PZ a coordinate.
__global__ void k_super_boxes(const float* __restrict__ stat, int64_t n, int nt, int ns, uint4* __restrict__ sbox,
                              float* __restrict__ smid) {
  __shared__ __align__(16) __half s_box[4][2 * PZ];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int s = blockIdx.x * 4 + w;
  if (s < ns && lane < PZ) {
    float lo = FLT_MAX, hi = -FLT_MAX, sum = 0.f, R2 = 0.f;
    const int t1 = min(nt, (s + 1) * PT_SUPER);
    for (int t = s * PT_SUPER; t < t1; ++t) {
      const float* st = stat + (size_t)t * (3 * PZ + 1);
      lo = fminf(lo, st[lane]);
      hi = fmaxf(hi, st[PZ + lane]);
      sum += st[2 * PZ + lane];
      R2 = fmaxf(R2, st[3 * PZ]);
    }
    const int64_t rows = min(n, (int64_t)t1 * PT_ROWS) - (int64_t)s * PT_SUPER * PT_ROWS;
    write_box(lo, hi, sqrtf(R2), &s_box[w][lane], &s_box[w][PZ + lane]);
    smid[s * PZ + lane] = sum / (float)rows;
  }
  __syncwarp();
  if (s < ns && lane < 4) sbox[s * 4 + lane] = reinterpret_cast<const uint4*>(s_box[w])[lane];
}

DctBasis dct_basis(int P) {
  DctBasis d;
  for (int i = 0; i < P * P; ++i)
    for (int c = 0; c < P * P; ++c) {
      auto one = [&](int x, int k) {
        return (k == 0 ? sqrt(1.0 / P) : sqrt(2.0 / P)) * cos(M_PI * (2 * x + 1) * k / (2.0 * P));
      };
      d.b[i * P * P + c] = (float)(one(i / P, c / P) * one(i % P, c % P));
    }
  return d;
}

}  // namespace

// Depths of the two tree levels for n entries: leaves of about 192 entries,
// at most 2^14 of them (leaf numbers are radix-sorted as 16-bit ranks).
void tree_depths(int64_t n, int* d1, int* d2) {
  int d = 2;
  while (d < 14 && ((int64_t)192 << d) < n) ++d;
  *d1 = (d + 1) / 2;
  *d2 = d / 2;
}

size_t tree_scratch_bytes(int64_t n) {
  int d1, d2;
  tree_depths(n, &d1, &d2);
  const int64_t nt = (n + PT_ROWS - 1) / PT_ROWS;
  return ((size_t)1 << d1) * (kCountStride * 4 + (size_t)PT_TOP * PZ * 4) + 256 + (size_t)n * (2 + 4) + 512 +
         (size_t)nt * (3 * PZ + 1) * 4 + 256 + ((size_t)4 << (d1 + d2)) + 256;
}

cudaError_t launch_tree_top(zoom_index ix, cudaStream_t st) {
  zoom_dict d = ix->dict;
  const int top = std::min(PT_TOP, 32 << ix->tree_d1);   // samples: 32 or so for every leaf
  const DctBasis dct = dct_basis(d->P);
  const int smem = (int)sizeof(TreeSmem);
  cudaError_t e;
#define ZOOM_TREE_TOP(DD)                                                                                        \
  do {                                                                                                           \
    e = cudaFuncSetAttribute(k_tree_top<DD>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);                  \
    if (e != cudaSuccess) return e;                                                                              \
    k_tree_top<DD><<<1, kTreeThreads, smem, st>>>(d->feat, d->dpad, d->n, dct, d->P * d->P, top, ix->tree_d1,      \
                                                  ix->tree_basis, (TreeNode*)ix->tree_node1);                    \
  } while (0)
  switch (d->d) {
    case 9: ZOOM_TREE_TOP(9); break;
    case 25: ZOOM_TREE_TOP(25); break;
    case 18: ZOOM_TREE_TOP(18); break;
    default: return cudaErrorInvalidValue;
  }
#undef ZOOM_TREE_TOP
  return cudaGetLastError();
}

// Builds the index's search order below the first levels: tree, order,
// operands, boxes.
cudaError_t build_search_tree(zoom_index ix, void* scratch, size_t scratch_bytes, cudaStream_t st) {
  zoom_dict d = ix->dict;
  const int64_t n = d->n;
  if (scratch_bytes < tree_scratch_bytes(n)) return cudaErrorInvalidValue;
  const int d1 = ix->tree_d1, d2 = ix->tree_d2;
  const int nt = (int)ix->tree_tiles, ns = (nt + PT_SUPER - 1) / PT_SUPER;
  char* p = (char*)scratch;
  auto take = [&](size_t bytes) {
    char* r = p;
    p += (bytes + 255) & ~(size_t)255;
    return r;
  };
  float* zl = (float*)take(((size_t)1 << d1) * PT_TOP * PZ * 4);
  uint32_t* cnt = (uint32_t*)take(((size_t)1 << d1) * kCountStride * 4);
  uint16_t* leaf = (uint16_t*)take((size_t)n * 2);
  float* stat = (float*)take((size_t)nt * (3 * PZ + 1) * 4);
  uint32_t* rank = (uint32_t*)take((size_t)n * 4);
  uint32_t* hist = (uint32_t*)take((size_t)4 << (d1 + d2));
  const int leaves = 1 << (d1 + d2);
  // samples: 48 or so for every leaf
  const int64_t m = std::min<int64_t>(n, (int64_t)std::min(1536, 48 << d2) << d1);
  cudaError_t e = cudaMemsetAsync(cnt, 0, ((size_t)1 << d1) * kCountStride * 4, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(hist, 0, (size_t)leaves * 4, st);
  if (e != cudaSuccess) return e;
  const int smem = (int)sizeof(TreeSmem);
  TreeNode* node1 = (TreeNode*)ix->tree_node1;
  TreeNode* node2 = (TreeNode*)ix->tree_node2;
#define ZOOM_TREE_A(DD)                                                                                       \
  k_tree_sample<DD><<<(unsigned)((m + 127) / 128), 128, 0, st>>>(d->feat, d->dpad, n, m, ix->tree_basis, node1, \
                                                                 d1, cnt, zl)
#define ZOOM_TREE_B(DD)                                                                                      \
  k_tree_route<DD><<<(unsigned)((n + 127) / 128), 128, 0, st>>>(d->feat, d->dpad, n, ix->tree_basis, node1, node2, \
                                                                d1, d2, leaf, rank, hist)
#define ZOOM_TREE_C(DD)                                                                                       \
  k_tile_operands<DD, 4><<<nt, PT_ROWS, 0, st>>>(d->feat, d->dpad, n, ix->tree_order,        \
                                                                      ix->tree_basis, ix->tree_f1, ix->tree_bf, \
                                                                      (uint4*)ix->tree_box, ix->tree_mid, stat)
#define ZOOM_TREE(X)                   \
  switch (d->d) {                      \
    case 9: X(9); break;               \
    case 25: X(25); break;             \
    case 18: X(18); break;             \
    default: return cudaErrorInvalidValue; \
  }
  ZOOM_TREE(ZOOM_TREE_A)
  e = cudaFuncSetAttribute(k_tree_sub, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  k_tree_sub<<<1 << d1, kTreeThreads, smem, st>>>(cnt, zl, d2, node2);
  ZOOM_TREE(ZOOM_TREE_B)
  k_leaf_scan<<<1, 1024, 0, st>>>(hist, leaves);
  k_tree_place<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(leaf, rank, hist, n, ix->tree_order);
  ZOOM_TREE(ZOOM_TREE_C)
  k_super_boxes<<<(ns + 3) / 4, 128, 0, st>>>(stat, n, nt, ns, (uint4*)ix->tree_sbox, ix->tree_smid);
  return cudaGetLastError();
#undef ZOOM_TREE
#undef ZOOM_TREE_A
#undef ZOOM_TREE_B
#undef ZOOM_TREE_C
}
