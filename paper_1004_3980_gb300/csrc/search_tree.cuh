// Shared by the index side (kernels_tree.cu) and the query side
// (kernels_prune.cu) of the search order: the bound coordinates, the
// splitting tree's routing and the tiles' boxes.
//
// Bound coordinates: the PZ coefficients of largest variance of the
// feature's orthonormal two-dimensional DCT (per P x P block).  The squared
// distance of two features over any subset of orthonormal coordinates is a
// lower bound of their squared distance, and the DCT concentrates the
// variance of image patches nearly as well as their principal components
// (1M pairs of 5 x 5 patches: the fraction of 256-entry tiles whose box lies
// within a query's 8th-nearest distance is 3.8 % with 16 DCT coefficients,
// 3.9 % with all 25 principal components), without an eigenproblem per
// dictionary.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

constexpr int PZ = 16;             // bound coordinates
constexpr int PT_ROWS = 256;       // entries per tile (the filter's step)
constexpr int PT_SUPER = 16;       // tiles per super tile
constexpr int PT_TOP = 2048;       // samples a (sub)tree is built from
constexpr float PT_SCALE = 4.f;    // bound coordinates are kept as 4 z in FP16

struct TreeNode {   // right iff z[dim] > thr
  float thr;
  int dim;
};

namespace {

// z = B^T f with B [D][PZ] in shared memory (16-byte rows).
template <int D>
__device__ __forceinline__ void bound_coords(const float (&f)[D], const float4* s_b, float (&z)[PZ]) {
#pragma unroll
  for (int c = 0; c < PZ; ++c) z[c] = 0.f;
#pragma unroll
  for (int i = 0; i < D; ++i) {
#pragma unroll
    for (int c4 = 0; c4 < PZ / 4; ++c4) {
      const float4 b = s_b[i * (PZ / 4) + c4];
      z[4 * c4 + 0] = fmaf(f[i], b.x, z[4 * c4 + 0]);
      z[4 * c4 + 1] = fmaf(f[i], b.y, z[4 * c4 + 1]);
      z[4 * c4 + 2] = fmaf(f[i], b.z, z[4 * c4 + 2]);
      z[4 * c4 + 3] = fmaf(f[i], b.w, z[4 * c4 + 3]);
    }
  }
}

// A feature row (dpad floats, 16-byte aligned) in registers.
template <int D>
__device__ __forceinline__ void load_feature(const float* __restrict__ row, float (&f)[D]) {
  const float4* r4 = reinterpret_cast<const float4*>(row);
#pragma unroll
  for (int i4 = 0; i4 < (D + 3) / 4; ++i4) {
    const float4 v = __ldg(r4 + i4);
    const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int t = 0; t < 4; ++t)
      if (4 * i4 + t < D) f[4 * i4 + t] = x[t];
  }
}

// Leaf of the first `depth` levels of the tree `nodes` (heap order, root 1);
// zc(c) gives coordinate c.
template <typename Z>
__device__ __forceinline__ int tree_descend(const TreeNode* __restrict__ nodes, int depth, Z zc) {
  int n = 1;
  for (int l = 0; l < depth; ++l) {
    const TreeNode nd = nodes[n];
    n = 2 * n + (zc(nd.dim) > nd.thr ? 1 : 0);
  }
  return n - (1 << depth);
}

// Leaf number of a point in the two-level tree: node1 [1 << d1], node2
// [1 << d1][1 << d2].
template <typename Z>
__device__ __forceinline__ int tree_leaf(const TreeNode* __restrict__ node1, const TreeNode* __restrict__ node2,
                                         int d1, int d2, Z zc) {
  const int a = tree_descend(node1, d1, zc);
  return (a << d2) | tree_descend(node2 + ((size_t)a << d2), d2, zc);
}

// This lane's arrival number at leaf lf, counted in hist; one atomic per leaf
// and warp (flat images send thousands of rows to one leaf).  active: the lanes
// here.
__device__ __forceinline__ uint32_t leaf_arrival(uint32_t* __restrict__ hist, int lf, unsigned active) {
  const int lane = threadIdx.x & 31;
  const unsigned same = __match_any_sync(active, lf);
  const int lead = __ffs(same) - 1;
  uint32_t base = 0;
  if (lane == lead) base = atomicAdd(hist + lf, (uint32_t)__popc(same));
  base = __shfl_sync(active, base, lead);
  return base + (uint32_t)__popc(same & ((1u << lane) - 1u));
}

// One block: hist[n] -> exclusive prefix sums in place.
__global__ void __launch_bounds__(1024) k_leaf_scan(uint32_t* __restrict__ hist, int n) {
  __shared__ uint32_t s_w[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = (n + 1023) / 1024, b0 = threadIdx.x * per;
  uint32_t acc = 0;
  for (int i = 0; i < per; ++i)
    if (b0 + i < n) acc += hist[b0 + i];
  uint32_t x = acc;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_w[warp] = x;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = s_w[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    s_w[lane] = w;
  }
  __syncthreads();
  uint32_t ex = x - acc + (warp ? s_w[warp - 1] : 0u);
  for (int i = 0; i < per; ++i)
    if (b0 + i < n) {
      const uint32_t t = hist[b0 + i];
      hist[b0 + i] = ex;
      ex += t;
    }
}

// A box in the scaled FP16 bound coordinates: 16 centres, 16 half widths
// (64 bytes).
struct alignas(16) BoxH {
  __half2 c[PZ / 2], h[PZ / 2];
};
__device__ __forceinline__ BoxH load_box(const uint4* __restrict__ b) {
  BoxH x;
  uint4* u = reinterpret_cast<uint4*>(&x);
#pragma unroll
  for (int i = 0; i < 4; ++i) u[i] = __ldg(b + i);
  return x;
}

// sum over the coordinates of max(|z - c| - h, 0)^2.  FP16 throughout: the
// result exceeds the exact value by less than 1 % (2^-11 per operation, at
// most 8 additions a lane), which the caller's threshold allows for; the
// operands' own rounding is in the half widths.  NaN compares as "not
// above", so a coordinate outside FP16's range never excludes anything.
__device__ __forceinline__ float box_bound(const __half2 (&z)[PZ / 2], const BoxH& b) {
  const __half2 one = __float2half2_rn(1.f);
  __half2 a0 = __float2half2_rn(0.f), a1 = a0;
#pragma unroll
  for (int i = 0; i < PZ / 2; i += 2) {
    const __half2 g0 = __hfma2_relu(__habs2(__hsub2(z[i], b.c[i])), one, __hneg2(b.h[i]));
    const __half2 g1 = __hfma2_relu(__habs2(__hsub2(z[i + 1], b.c[i + 1])), one, __hneg2(b.h[i + 1]));
    a0 = __hfma2(g0, g0, a0);
    a1 = __hfma2(g1, g1, a1);
  }
  const float2 s0 = __half22float2(a0), s1 = __half22float2(a1);
  return (s0.x + s0.y) + (s1.x + s1.y);
}

}  // namespace
