// Exact neighbour search over the dictionary's search order (kernels_tree.cu):
// every query is compared only with the tiles (256 entries) whose bounding
// box comes within its search radius.
//
// Steps, for queries sorted along the same tree (neighbouring queries need
// nearly the same tiles):
//  1. seeds: 256 queries at a time against 64 tiles near them (k_seed_tiles;
//     the dense wide-step filter over a tile list); the r-th smallest chunk
//     minimum, r a little above K, is the query's radius T;
//  2. visits: every (query, tile) pair whose box bound does not exceed T,
//     appended to the tile's query list (k_visit);
//  3. the filter over the lists (k_knn_tg): 128 listed queries x 256 entries
//     per tensor-core step; entries with d~ <= T + delta (delta bounds
//     |d~ - d|) are appended to their query's candidates;
//  4. the candidates' exact FP32 distances, membership and selection
//     (k_rerank_list).
// Every entry within distance T of the query is then among its candidates:
// its tile's box bound is at most T, and its d~ at most T + delta.  So if the
// K-th member found lies within T, the K nearest members are proven; every
// other query (too few members within T, or more candidates than the list
// holds) goes to the dense filters and the scan.
//
// Where the boxes exclude little (features that do not cluster: noise, a
// dictionary unlike the image) a round of queries is given up once its lists
// are longer than the list filter is worth, and its queries go to the dense
// filters too (PrunePlan::give_up).
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <float.h>
#include <limits.h>

#include "device_common.cuh"
#include "search_tree.cuh"
#include "tc_ptx.cuh"
#include "warp_select.cuh"
#include "zoom_internal.h"

namespace {

constexpr int PQ_ROWS = 128;        // queries per filter step (M)
constexpr int PQ_SEEDS = kPruneSeeds;

__device__ __forceinline__ unsigned lanes_below(int lane) { return (1u << lane) - 1u; }

// ---------------------------------------------------------------------------
// queries sorted along the tree
// ---------------------------------------------------------------------------

// Leaf of every query, and its arrival number there (counts: hist).  Bound by
// the tree walk's dependent lookups, up to 14 a query (2.06M queries: 138 us).
template <int D>
__global__ void __launch_bounds__(128) k_query_route(const float* __restrict__ feat, int dpad, int64_t nq,
                                                     const float* __restrict__ basis,
                                                     const TreeNode* __restrict__ node1,
                                                     const TreeNode* __restrict__ node2, int d1, int d2,
                                                     uint16_t* __restrict__ leaf, uint32_t* __restrict__ rank,
                                                     uint32_t* __restrict__ hist) {
  __shared__ __align__(16) float s_b[D * PZ];
  __shared__ float s_z[PZ][128];
  for (int t = threadIdx.x; t < D * PZ; t += 128) s_b[t] = basis[t];
  __syncthreads();
  const int64_t q = (int64_t)blockIdx.x * 128 + threadIdx.x;
  const unsigned active = __ballot_sync(kFull, q < nq);
  if (q >= nq) return;
  float f[D], z[PZ];
  load_feature<D>(feat + q * dpad, f);
  bound_coords<D>(f, reinterpret_cast<const float4*>(s_b), z);
#pragma unroll
  for (int c = 0; c < PZ; ++c) s_z[c][threadIdx.x] = z[c];
  const int lf = tree_leaf(node1, node2, d1, d2, [&](int c) { return s_z[c][threadIdx.x]; });
  leaf[q] = (uint16_t)lf;
  rank[q] = leaf_arrival(hist, lf, active);
}

// Writes every query's operand row (row-major, and in the tile layout of the
// seed filter), ||q||^2, scaled FP16 bound coordinates and number to its
// sorted place.  Bound by the scattered rows written, 150 bytes or so a query
// (2.06M queries: 255 us).  FORM 1: BF16, 2: single-term FP16 ([q | 1 1 1]).
template <int D, int KC, int FORM>
__global__ void __launch_bounds__(128) k_query_sorted(const float* __restrict__ feat, int dpad, int64_t nq,
                                                      const float* __restrict__ basis,
                                                      const uint16_t* __restrict__ leaf,
                                                      const uint32_t* __restrict__ rank,
                                                      const uint32_t* __restrict__ offs, uint16_t* __restrict__ qrow,
                                                      uint16_t* __restrict__ qop, float* __restrict__ qn,
                                                      uint4* __restrict__ qz, int32_t* __restrict__ perm) {
  __shared__ __align__(16) float s_b[D * PZ];
  for (int t = threadIdx.x; t < D * PZ; t += 128) s_b[t] = basis[t];
  __syncthreads();
  const int64_t q = (int64_t)blockIdx.x * 128 + threadIdx.x;
  if (q >= nq) return;
  float f[D], z[PZ];
  load_feature<D>(feat + q * dpad, f);
  const int64_t pos = (int64_t)offs[leaf[q]] + rank[q];
  uint16_t h[KC * 8];
#pragma unroll
  for (int k = 0; k < KC * 8; ++k) h[k] = 0;
  float n2 = 0.f;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    n2 = fmaf(f[i], f[i], n2);
    h[i] = FORM == 1 ? __bfloat16_as_ushort(__float2bfloat16_rn(f[i])) : __half_as_ushort(__float2half_rn(f[i]));
  }
  h[D] = h[D + 1] = h[D + 2] = FORM == 1 ? (uint16_t)0x3F80u : (uint16_t)0x3C00u;   // 1.0
#pragma unroll
  for (int kc = 0; kc < KC; ++kc) {
    uint4 a;
    uint32_t* pa = &a.x;
#pragma unroll
    for (int t = 0; t < 4; ++t) pa[t] = (uint32_t)h[kc * 8 + 2 * t] | ((uint32_t)h[kc * 8 + 2 * t + 1] << 16);
    *reinterpret_cast<uint4*>(qrow + pos * (KC * 8) + kc * 8) = a;
    *reinterpret_cast<uint4*>(qop + (pos / PQ_ROWS) * (KC * PQ_ROWS * 8) + kc * (PQ_ROWS * 8) +
                              (pos % PQ_ROWS) * 8) = a;
  }
  bound_coords<D>(f, reinterpret_cast<const float4*>(s_b), z);
  uint4 u[2];
  __half2* hz = reinterpret_cast<__half2*>(u);
#pragma unroll
  for (int c = 0; c < PZ / 2; ++c) hz[c] = __floats2half2_rn(z[2 * c] * PT_SCALE, z[2 * c + 1] * PT_SCALE);
  qz[pos * 2] = u[0];
  qz[pos * 2 + 1] = u[1];
  qn[pos] = n2;
  perm[pos] = (int32_t)q;
}

// ---------------------------------------------------------------------------
// seeds of 256 sorted queries: every warp lists the 32 tiles nearest the mean
// of its 32 queries (among the tiles of the kSeedSupers nearest super tiles),
// and the block takes PQ_SEEDS distinct tiles from the eight lists in turn.
// One mean of all 256 queries served those that straddle distant leaves of
// the tree badly: 1 to 3 % of the queries then had radii with up to 200,000
// entries inside (4M pairs).  Bound by the selection among a block's
// candidates (2.06M queries on 4M entries: 716 us, 258,064 on 1M: 64 us).
// ---------------------------------------------------------------------------
constexpr int kSeedSupers = 16;
constexpr int kMaxTiles = (int)(kPruneMaxEntries / PT_ROWS);
static_assert(kMaxTiles / PT_SUPER <= 2048 && PQ_SEEDS <= 128, "key layout of the seeds");

__global__ void __launch_bounds__(256) k_seed_tiles(const uint4* __restrict__ qz, int64_t nq,
                                                    const float4* __restrict__ smid, int ns,
                                                    const float4* __restrict__ mid, int nt,
                                                    int32_t* __restrict__ seeds) {
  extern __shared__ uint32_t s_key[];          // [8][ns] keys of the super tiles
  __shared__ int s_list[8][32];                // the warps' lists (-1: none)
  __shared__ uint32_t s_taken[kMaxTiles / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < (nt + 31) / 32; i += 256) s_taken[i] = 0;
  const int64_t pos = (int64_t)blockIdx.x * 256 + tid;
  float m[PZ];
#pragma unroll
  for (int c = 0; c < PZ; ++c) m[c] = 0.f;
  const bool valid = pos < nq;
  if (valid) {
    const uint4 u[2] = {qz[pos * 2], qz[pos * 2 + 1]};
    const __half2* hz = reinterpret_cast<const __half2*>(u);
#pragma unroll
    for (int c = 0; c < PZ / 2; ++c) {
      const float2 v = __half22float2(hz[c]);
      m[2 * c] = v.x;
      m[2 * c + 1] = v.y;
    }
  }
  const int rows = __popc(__ballot_sync(kFull, valid));
  s_list[warp][lane] = -1;
  if (rows > 0) {   // warp-uniform
#pragma unroll
    for (int c = 0; c < PZ; ++c) {
#pragma unroll
      for (int o = 16; o; o >>= 1) m[c] += __shfl_xor_sync(kFull, m[c], o);
      m[c] /= PT_SCALE * (float)rows;
    }
    auto dist = [&](const float4* __restrict__ c) {
      float d = 0.f;
#pragma unroll
      for (int i = 0; i < PZ / 4; ++i) {
        const float4 x = __ldg(c + i);
        const float a = x.x - m[4 * i], b = x.y - m[4 * i + 1], e = x.z - m[4 * i + 2], f = x.w - m[4 * i + 3];
        d = fmaf(a, a, fmaf(b, b, fmaf(e, e, fmaf(f, f, d))));
      }
      return d;
    };
    // the nearest super tiles: each lane keeps the keys of every 32nd one in
    // shared memory and their minimum in a register (a distance's low bits
    // hold the number: the order is a heuristic)
    uint32_t* key = s_key + warp * ns;
    uint32_t mn = 0xFFFFFFFFu;
    for (int s = lane; s < ns; s += 32) {
      const uint32_t k = (__float_as_uint(dist(smid + s * (PZ / 4))) & 0x7FFFF800u) | (uint32_t)s;
      key[s] = k;
      mn = min(mn, k);
    }
    int sup = -1;   // lane j: the j-th nearest super tile
    for (int j = 0; j < kSeedSupers; ++j) {
      const uint32_t g = __reduce_min_sync(kFull, mn);
      if (g == 0xFFFFFFFFu) break;
      const int s = (int)(g & 2047u);
      if (lane == j) sup = s;
      if (lane == (s & 31)) {
        key[s] = 0xFFFFFFFFu;
        mn = 0xFFFFFFFFu;
        for (int t = lane; t < ns; t += 32) mn = min(mn, key[t]);
      }
      __syncwarp();
    }
    // the nearest of their tiles
    constexpr int kPer = kSeedSupers * PT_SUPER / 32;
    uint32_t k2[kPer];
#pragma unroll
    for (int h = 0; h < kPer; ++h) {
      const int i = lane + 32 * h;   // tile i % 16 of super tile number i / 16
      const int s = __shfl_sync(kFull, sup, i / PT_SUPER);
      const int t = s * PT_SUPER + i % PT_SUPER;
      k2[h] = s >= 0 && t < nt ? (__float_as_uint(dist(mid + (size_t)t * (PZ / 4))) & 0x7FFFFF00u) | (uint32_t)i
                               : 0xFFFFFFFFu;
    }
    for (int j = 0; j < 32; ++j) {
      uint32_t l = k2[0];
#pragma unroll
      for (int h = 1; h < kPer; ++h) l = min(l, k2[h]);
      const uint32_t g = __reduce_min_sync(kFull, l);
      if (g == 0xFFFFFFFFu) break;
#pragma unroll
      for (int h = 0; h < kPer; ++h)
        if (k2[h] == g) k2[h] = 0xFFFFFFFFu;
      const int i = (int)(g & 255u);
      const int s = __shfl_sync(kFull, sup, i / PT_SUPER);
      if (lane == 0) s_list[warp][j] = s * PT_SUPER + i % PT_SUPER;
    }
  }
  __syncthreads();
  if (warp != 0) return;
  int32_t* out = seeds + (int64_t)blockIdx.x * PQ_SEEDS;
  int n = 0;
  // rank j of every list in turn, then (never in practice) the first tiles
  for (int j = 0; n < PQ_SEEDS; ++j) {
    int t = -1;
    if (j < 32) t = lane < 8 ? s_list[lane][j] : -1;
    else if ((j - 32) * 32 + lane < nt) t = (j - 32) * 32 + lane;
    else if ((j - 32) * 32 >= nt) break;
    bool mine = false;
    if (t >= 0 && t < nt) mine = (atomicOr(&s_taken[t >> 5], 1u << (t & 31)) >> (t & 31) & 1u) == 0;
    const unsigned who = __ballot_sync(kFull, mine);
    const int at = n + __popc(who & lanes_below(lane));
    if (mine && at < PQ_SEEDS) out[at] = t;
    n += __popc(who);
  }
}

// ---------------------------------------------------------------------------
// search radius of every query
// ---------------------------------------------------------------------------

// delta(T): bound on |d~ - d| for an entry within distance T (see launch_rerank)
__device__ __forceinline__ float filter_error(float T, float qn, const FilterError& fe) {
  const float nrm = sqrtf(qn);
  const float rc = nrm + sqrtf(T) * 1.001f + 1e-6f;
  return fe.c_qr * nrm * rc + fe.c_sq * (rc * rc + qn) + fe.c_rel * T + fe.c_abs * (nrm + rc) + 1e-12f;
}

// T: the r-th smallest seed chunk minimum (at least its own error bound, so
// that near duplicates do not shrink it to nothing).  rad: T, or -1 where
// the query is left to the dense search (nothing finite, or values whose
// products leave FP16); vis: the bound's threshold in scaled coordinates,
// with 1 % for its FP16 arithmetic.  The query's operand row gets minus the
// largest accumulator value that can belong to an entry within T, T + delta -
// ||q||^2, as three terms (the dictionary's rows have ones there), rounded up
// by the terms' own error and the accumulation's.  pad: the row that no entry
// passes.
template <int FORM>
__global__ void k_radius(const float* __restrict__ ld, int MC, int r, const float* __restrict__ qn, int64_t nq,
                         FilterError fe, float trunc, int D, int row_len, float* __restrict__ rad, float* __restrict__ vis,
                         uint16_t* __restrict__ qrow, uint16_t* __restrict__ pad) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  auto bits = [](float x, float& back) -> uint16_t {
    if (FORM == 1) {
      const __nv_bfloat16 h = __float2bfloat16_rn(x);
      back = __bfloat162float(h);
      return __bfloat16_as_ushort(h);
    }
    const __half h = __float2half_rn(x);
    back = __half2float(h);
    return __half_as_ushort(h);
  };
  float back;
  if (q < row_len) {
    const float x = q >= D && q < D + 3 ? 1.f : (q == D + 3 ? 60000.f : 0.f);
    pad[q] = bits(x, back);
  }
  if (q >= nq) return;
  const float n = qn[q];
  const float v = ld[q * MC + r - 1];
  const bool ok = n < 1000.f && v < 1000.f && v > -1000.f;   // false for NaN
  float T = -1.f, vs = -1.f;   // nothing is visited, nothing proven
  if (ok) {
    T = fmaxf(v, 0.f);
    if (FORM == 1) T *= 1.f + trunc;
    T = fmaxf(T, filter_error(T, n, fe));
    const float dl = filter_error(T, n, fe);
    vs = T;
    if (FORM == 1) {
      // every entry with d~ <= T is a candidate: those of the tiles left out
      // have d > vs, hence d~ > vs - (error at vs) >= T
      vs = T + filter_error(T + 2.f * dl, n, fe);
      if (vs > T + 2.f * dl) {   // (the error grows slower than that)
        rad[q] = vis[q] = -1.f;
        return;
      }
    }
    vs = vs * (PT_SCALE * PT_SCALE) * 1.01f + 1e-5f;
    float x = n - (T + dl + (T + dl + n) * 1e-6f + 2e-7f);   // - thr
    uint16_t* o = qrow + q * row_len + D + 3;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      o[i] = bits(x, back);
      x -= back;
    }
  }
  rad[q] = T;
  vis[q] = vs;
}

// ---------------------------------------------------------------------------
// visits: a warp takes 32 sorted queries and the super tiles part, part +
// parts, ... (32 at a time, one per lane): box of the queries against the
// super tiles' boxes, then against their tiles' boxes; the tiles that are
// left queue up, and 32 of them at a time are tested against every query, one
// tile per lane with its box in registers and the queries' coordinates
// broadcast from shared memory.  Bound by that test, half by its issue and half by
// its latency (24 paired FP16 operations of about 32 instructions a pair; 280 x
// 280 queries on 300,000 entries: 53 % of the issue slots, 17 % of the warps
// that fit, no memory above 36 %); with a query per lane and the boxes
// broadcast it took 45 and waited for every box.  A lane ends up
// with the mask of the queries that need its tile: one round of atomics gives
// the 32 masks their places in the tiles' lists.  The pairs of the round are
// counted, too: past `give_up` the warps stop.  2.06M queries on 4M entries:
// 20.4 ms in 32 rounds; 258,064 on 1M: 1.19 ms.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_visit(const uint4* __restrict__ qz, const float* __restrict__ vis,
                                               int nslab, const uint4* __restrict__ box, int nt,
                                               const uint4* __restrict__ sbox, int ns, int parts,
                                               uint16_t* __restrict__ list, uint32_t stride,
                                               uint32_t* __restrict__ tcnt, unsigned long long give_up,
                                               unsigned long long* __restrict__ pairs) {
  __shared__ uint4 s_z[8][32][2];
  __shared__ float s_T[8][32];
  __shared__ int s_queue[8][64];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int gw = blockIdx.x * 8 + wib;
  const int group = gw / parts, part = gw % parts;
  const int q = group * 32 + lane;   // query of the slab
  if (group * 32 >= nslab) return;   // warp-uniform
  const float T = q < nslab ? vis[q] : -1.f;
  const bool active = T >= 0.f;
  const unsigned act = __ballot_sync(kFull, active);
  if (!act) return;
  __half2 z[PZ / 2];
  {
    uint4 u[2] = {make_uint4(0, 0, 0, 0), make_uint4(0, 0, 0, 0)};
    if (active) {
      u[0] = qz[q * 2];
      u[1] = qz[q * 2 + 1];
    }
    const __half2* hz = reinterpret_cast<const __half2*>(u);
#pragma unroll
    for (int i = 0; i < PZ / 2; ++i) z[i] = hz[i];
    s_z[wib][lane][0] = u[0];
    s_z[wib][lane][1] = u[1];
    s_T[wib][lane] = active ? T : -1.f;
  }
  __syncwarp();
  // the box of the warp's queries: centre g, half width e with the FP16
  // rounding of the box-to-box test (2^-11 of each operand and of the sum of
  // the half widths) allowed for
  __half2 g[PZ / 2], e[PZ / 2];
#pragma unroll
  for (int i = 0; i < PZ / 2; ++i) {
    __half2 lo = active ? z[i] : __float2half2_rn(65504.f);
    __half2 hi = active ? z[i] : __float2half2_rn(-65504.f);
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      lo = __hmin2(lo, __shfl_xor_sync(kFull, lo, o));
      hi = __hmax2(hi, __shfl_xor_sync(kFull, hi, o));
    }
    const float2 l = __half22float2(lo), h = __half22float2(hi);
    g[i] = __floats2half2_rn(0.5f * (l.x + h.x), 0.5f * (l.y + h.y));
    const float2 c = __half22float2(g[i]);
    const float wx = fmaxf(h.x - c.x, c.x - l.x), wy = fmaxf(h.y - c.y, c.y - l.y);
    e[i] = __halves2half2(__float2half_ru(wx * 1.004f + fabsf(c.x) * 2e-3f + 1e-6f),
                          __float2half_ru(wy * 1.004f + fabsf(c.y) * 2e-3f + 1e-6f));
  }
  float Tg = active ? T : -1.f;
#pragma unroll
  for (int o = 16; o; o >>= 1) Tg = fmaxf(Tg, __shfl_xor_sync(kFull, Tg, o));
  Tg *= 1.01f;
  // box-to-box bound: the query box's half width joins the tile's, enlarged
  // by 2^-9 of itself for the rounding of the sum
  auto group_bound = [&](const uint4* __restrict__ b) {
    BoxH x = load_box(b);
    const __half2 grow = __float2half2_rn(1.002f);
#pragma unroll
    for (int i = 0; i < PZ / 2; ++i) x.h[i] = __hfma2(x.h[i], grow, e[i]);
    return box_bound(g, x);
  };
  int* queue = s_queue[wib];
  int qd = 0;   // tiles queued
  // Pairs not yet in the round's count: a warp adds them an eighth of its
  // (query, tile) pairs at a time, so that few do where the boxes exclude much
  // (an atomic on one address per 32 tiles made 258,064 queries on 1M entries
  // 5.34 -> 5.47 ms).  k_step_scan sees what stays uncounted in the lists.
  const uint32_t hold = (uint32_t)(4 * nt / parts + 1);
  uint32_t held = 0;
  bool stop = false;
  auto test = [&](int m) {   // the first m (at most 32) queued tiles
    const int t = lane < m ? queue[lane] : -1;
    unsigned mk = 0;
    {
      const BoxH x = load_box(box + (size_t)(t < 0 ? 0 : t) * 4);
#pragma unroll 4
      for (int j = 0; j < 32; ++j) {
        const uint4 u[2] = {s_z[wib][j][0], s_z[wib][j][1]};
        const __half2* hz = reinterpret_cast<const __half2*>(u);
        __half2 zj[PZ / 2];
#pragma unroll
        for (int i = 0; i < PZ / 2; ++i) zj[i] = hz[i];
        mk |= (box_bound(zj, x) > s_T[wib][j] ? 0u : 1u) << j;   // NaN: not excluded
      }
    }
    mk = t < 0 ? 0u : mk & act;
    held += __reduce_add_sync(kFull, (uint32_t)__popc(mk));
    const uint32_t p = mk ? atomicAdd(tcnt + t, (uint32_t)__popc(mk)) : 0u;
    if (held >= hold) {
      const unsigned long long before = lane == 0 ? atomicAdd(pairs, (unsigned long long)held) : 0ull;
      stop = __any_sync(kFull, before > give_up);
      held = 0;
    }
    for (unsigned any = __ballot_sync(kFull, mk != 0); any; any &= any - 1) {
      const int j = __ffs(any) - 1;
      const int tj = __shfl_sync(kFull, t, j);
      const unsigned mj = __shfl_sync(kFull, mk, j);
      const uint32_t at = __shfl_sync(kFull, p, j);
      if ((mj >> lane) & 1u) list[(size_t)tj * stride + at + __popc(mj & lanes_below(lane))] = (uint16_t)q;
    }
    const int rest = qd - m, v = lane < rest ? queue[m + lane] : 0;
    __syncwarp();
    if (lane < rest) queue[lane] = v;
    __syncwarp();
    qd = rest;
  };
  for (int s0 = part * 32; s0 < ns && !stop; s0 += parts * 32) {
    const int s = s0 + lane;
    bool keep = false;
    if (s < ns) keep = !(group_bound(sbox + (size_t)s * 4) > Tg);
    unsigned ms = __ballot_sync(kFull, keep);
    while (ms && !stop) {
      // the tiles of two super tiles at a time, one per lane
      const int b0 = __ffs(ms) - 1;
      ms &= ms - 1;
      const int b1 = ms ? __ffs(ms) - 1 : -1;
      if (ms) ms &= ms - 1;
      const int sup = lane < PT_SUPER ? b0 : b1;
      const int tile = (s0 + sup) * PT_SUPER + (lane & (PT_SUPER - 1));
      bool k2 = false;
      if (sup >= 0 && tile < nt) k2 = !(group_bound(box + (size_t)tile * 4) > Tg);
      const unsigned mt = __ballot_sync(kFull, k2);
      if (k2) queue[qd + __popc(mt & lanes_below(lane))] = tile;   // at most 31 + 32
      qd += __popc(mt);
      __syncwarp();
      if (qd >= 32) test(32);
    }
  }
  if (qd > 0 && !stop) test(qd);
}

// ---------------------------------------------------------------------------
// filter steps: the lists cut into steps of 128 queries
// ---------------------------------------------------------------------------

// One block: per tile the number of steps before it (off) and of non-empty
// tiles before it (ord); off[nt] is the total, or 0 where the round is given
// up, and off[nt + 1] says so.
__global__ void __launch_bounds__(1024) k_step_scan(const uint32_t* __restrict__ tcnt, int nt,
                                                    uint32_t* __restrict__ off, uint32_t* __restrict__ ord,
                                                    unsigned long long give_up,
                                                    const unsigned long long* __restrict__ pairs) {
  __shared__ unsigned long long s_w[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = (nt + 1023) / 1024, b0 = threadIdx.x * per;
  unsigned long long acc = 0;   // steps in the low half, non-empty tiles above
  for (int i = 0; i < per; ++i)
    if (b0 + i < nt) {
      const uint32_t c = tcnt[b0 + i];
      acc += (unsigned long long)((c + PQ_ROWS - 1) / PQ_ROWS) | ((unsigned long long)(c ? 1u : 0u) << 32);
    }
  unsigned long long x = acc;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_w[warp] = x;
  __syncthreads();
  if (warp == 0) {
    unsigned long long w = s_w[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(kFull, w, o);
      if (lane >= o) w += y;
    }
    s_w[lane] = w;
  }
  __syncthreads();
  unsigned long long ex = x - acc + (warp ? s_w[warp - 1] : 0ull);
  for (int i = 0; i < per; ++i)
    if (b0 + i < nt) {
      const uint32_t c = tcnt[b0 + i];
      off[b0 + i] = (uint32_t)ex;
      ord[b0 + i] = (uint32_t)(ex >> 32);
      ex += (unsigned long long)((c + PQ_ROWS - 1) / PQ_ROWS) | ((unsigned long long)(c ? 1u : 0u) << 32);
    }
  if (threadIdx.x == 1023) {
    const uint32_t steps = (uint32_t)s_w[31];
    const bool up = *pairs > give_up || (unsigned long long)steps * PQ_ROWS > give_up + (unsigned long long)nt * PQ_ROWS;
    off[nt] = up ? 0u : steps;
    off[nt + 1] = up ? 1u : 0u;
  }
}

// A step: x the tile, y its first list entry, z the number of queries, w the
// tile's number among the non-empty ones.
__global__ void k_steps(const uint32_t* __restrict__ tcnt, int nt, const uint32_t* __restrict__ off,
                        const uint32_t* __restrict__ ord, int4* __restrict__ steps, int32_t* __restrict__ tile_of) {
  const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 3;   // 8 lanes per tile
  if (t >= nt) return;
  const int c = (int)tcnt[t];
  const uint32_t o = off[t];
  const int od = (int)ord[t];
  if ((threadIdx.x & 7) == 0 && c > 0) tile_of[od] = t;
  for (int j = threadIdx.x & 7; j * PQ_ROWS < c; j += 8)
    steps[o + j] = make_int4(t, j * PQ_ROWS, min(PQ_ROWS, c - j * PQ_ROWS), od);
}

// ---------------------------------------------------------------------------
// the filter over query lists: one CTA per SM, each pieces of consecutive
// steps, so that a tile's operand (one bulk copy) serves its steps in a row.
// The operand rows of the queries carry -thr (three terms against ones of the
// dictionary's rows), so an accumulator is negative exactly where the entry
// may lie within the query's radius.
//   warps 18..23  gather the queries' operand rows (64 bytes each)
//                 through registers into a ring of stages, a step each in turn
//   warps 0, 1    issue the MMAs of the even / odd steps, M = 128 queries x
//                 N = 256 entries, into an accumulator each (the two fill the
//                 TMEM); warp 0 also copies the tiles
//   warps 2..17   epilogue: per parity two warps for each TMEM lane
//                 quadrant, one for the first 128 columns and one for the
//                 others, 32 columns at a time (twenty-four warps leave 80
//                 registers a thread)
// A chunk of 32 columns with a negative minimum in some lane (one warp vote)
// becomes a record (first position, 32 sign bits) in a shared-memory column of
// that lane; one atomic per lane and step gives the records their places in
// the query's candidate list, and they are written at the next step, when the
// atomic has long returned.  (Extracting the positions one by one in the
// epilogue cost about 350 cycles each.)  Bound by the hand-offs between the
// roles: with two 128-column accumulators a parity, one read while the other
// is computed, a step took 1250 cycles against 1080 here -- each hand-off costs
// the slowest of eight warps some 400 cycles whatever it covers; the counters have
// nothing near its limit (280 x 280 queries on 300,000 entries: tensor pipe 22 %
// of the cycles, issue slots 55 %, L1 and shared memory 49 %, L2 and DRAM below
// 10 %).  2.06M queries
// on 4M entries (BF16): 34.1 ms where the dense filter took 394 ms; 258,064 on
// 1M (FP16): 2.11 ms and 13.1 ms.
// ---------------------------------------------------------------------------
constexpr int kHits = PT_ROWS / 64;   // records per lane and step, at most: 128 columns
constexpr int kEpi = 16;              // epilogue warps
constexpr int kGather = 6;   // gathering warps
// polls of an accumulator's barrier before the suspending wait (1 to 32 the
// same; 256 made a step 5 % longer: the polling warps slow the others)
constexpr int kAccPolls = 8;
constexpr int kStagesTg = 6;   // a multiple of kGather / 2
// at least 3: a tile's slot is free once both parities are past it, and the
// parity that waits for a tile may be two tiles ahead of the other
constexpr int kSlotsTg = 4;
constexpr int kTgThreads = (2 + kEpi + kGather) * 32;
constexpr int kTgBar = 512;
__host__ __device__ constexpr int tg_smem(int KC) {
  return 1024 + 2 * kStagesTg * KC * PQ_ROWS * 16 + kSlotsTg * KC * PT_ROWS * 16 + kTgBar +
         2 * kStagesTg * PQ_ROWS * 2 + 2 * kHits * kEpi * 32 * 8;
}
static_assert(tg_smem(4) <= 232448, "shared memory of the list filter");
static_assert(kSlotsTg >= 3, "tile slots");
static_assert(kStagesTg % (kGather / 2) == 0, "a stage belongs to one gathering warp");

// The steps of one CTA, numbered 0 .. count - 1: pieces of `len` consecutive
// steps dealt out to the CTAs in turn, so that tiles many entries of which
// pass (a step then takes several times as long) spread over the CTAs.
// tile(k): the number of step k's tile among this CTA's tiles in order (a
// piece's first tile counts as a new one).
constexpr uint32_t kPieces = 8;   // pieces per CTA, at least (their length is a power of two, 32 or more)
struct StepIter {
  const int4* steps;
  uint32_t len, shift, count;
  uint32_t piece = 0, base = 0;   // current piece, tiles of the pieces before it
  int w0 = 0;                     // number of the current piece's first tile
  __device__ StepIter(const int4* s, uint32_t n) : steps(s), shift(5) {
    while ((gridDim.x * kPieces) << (shift + 1) <= n) ++shift;
    len = 1u << shift;
    const uint32_t round = len * gridDim.x, full = n / round, rest = n - full * round;
    const uint32_t mine = blockIdx.x * len;
    count = full * len + (rest > mine ? min(len, rest - mine) : 0u);
    if (count > 0) w0 = steps[start(0)].w;
  }
  __device__ uint32_t start(uint32_t p) const { return (p * gridDim.x + blockIdx.x) * len; }
  __device__ uint32_t global(uint32_t k) const { return start(k >> shift) + (k & (len - 1u)); }
  __device__ int4 step(uint32_t k) const { return steps[global(k)]; }
  // tile number of step k, whose entry is s (k non-decreasing over the calls)
  __device__ uint32_t tile(uint32_t k, const int4& s) {
    while (piece < k >> shift) {   // len >= 32 steps: at most one piece on
      base += (uint32_t)(steps[start(piece) + len - 1].w - w0) + 1u;
      ++piece;
      w0 = steps[start(piece)].w;
    }
    return base + (uint32_t)(s.w - w0);
  }
};

struct TgArgs {
  const uint16_t* qrow;     // operand rows of the slab's queries [m][KC * 8]
  const uint16_t* pad;      // a row that no entry passes
  int m;                    // queries of the slab
  const uint16_t* list;     // [nt][stride]
  uint32_t stride;
  int nt;
  const int4* steps;
  const uint32_t* n_steps;  // on the device
  const int32_t* tile_of;   // tile of each non-empty tile number
  const uint16_t* dop;      // [nt][KC][256][8]
  uint32_t* qcnt;           // [m] records found
  uint2* cand;              // [m][cap] records: first position in the search order, bit 31 - k for position + k
  uint32_t cap;
  unsigned int* status;
  uint64_t wait_ns;
  int inject;               // testing aid: withhold the accumulators from a CTA's third step on
};

// kind::f16, D fp32, A and B of one type, K-major, M = 128, N = 256
__host__ __device__ constexpr uint32_t tg_idesc(uint32_t ab_type) {
  return (1u << 4) | (ab_type << 7) | (ab_type << 10) | ((uint32_t)(PT_ROWS >> 3) << 17) |
         ((uint32_t)(PQ_ROWS >> 4) << 24);
}

template <int KC, uint32_t AB_TYPE>
__global__ void __maxnreg__(80) k_knn_tg(TgArgs a) {
  constexpr uint32_t kATile = KC * PQ_ROWS * 16;
  constexpr uint32_t kBTile = KC * PT_ROWS * 16;
  constexpr uint32_t kA = kStagesTg, kSlots = kSlotsTg;
  constexpr uint32_t kIdesc = tg_idesc(AB_TYPE);
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  unsigned char* sA = smem;                               // [2][kA] query stages
  unsigned char* sB = sA + 2 * kA * kATile;               // [kSlots] tiles
  uint64_t* bars = (uint64_t*)(sB + kSlots * kBTile);
  uint64_t* a_full = bars;                                // [2][kA]
  uint64_t* a_empty = a_full + 2 * kA;                    // [2][kA]
  uint64_t* b_full = a_empty + 2 * kA;                    // [kSlots]
  uint64_t* b_empty = b_full + kSlots;                    // [kSlots]
  uint64_t* acc_full = b_empty + kSlots;                  // [2] per parity
  uint64_t* acc_empty = acc_full + 2;                     // [2]
  uint64_t* drain = acc_empty + 2;                        // [2]
  uint64_t* tmem_done = drain + 2;                        // nobody uses the TMEM any more
  uint32_t* tmem_slot = (uint32_t*)(tmem_done + 1);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  static_assert((4 * kA + 2 * kSlots + 7) * 8 + 8 <= kTgBar, "barrier area");
  uint16_t* s_idx = (uint16_t*)((unsigned char*)bars + kTgBar);   // [2][kA][128] query of a row (0xFFFF: none)
  uint2* s_hit = (uint2*)(s_idx + 2 * kA * PQ_ROWS);   // [2][kHits][kEpi * 32], a column per epilogue lane

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (uint32_t i = 0; i < 2 * kA; ++i) {
      mbar_init(a_full + i, 1);
      mbar_init(a_empty + i, 8);      // the step's eight epilogue warps
    }
    for (uint32_t i = 0; i < kSlots; ++i) {
      mbar_init(b_full + i, 1);
      mbar_init(b_empty + i, 2);      // even and odd steps are past the tile
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(acc_full + i, 1);
      mbar_init(acc_empty + i, 8);
      mbar_init(drain + i, 1);
    }
    mbar_init(tmem_done, kEpi + 2);   // the epilogue warps and the issuing threads
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncwarp();   // the allocation is warp-collective: lane 0 comes from the initialisation
  if (warp == 0) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // Steps with k even have parity 0, the others parity 1.
  StepIter it(a.steps, *a.n_steps);
  const uint32_t count = it.count;

  if (warp >= 2 + kEpi) {
    // ---------------- query rows: steps g, g + kGather, ... ----------------
    const int g = warp - 2 - kEpi;
    const int p = g & 1;
    // A load takes four 16-byte pieces of eight rows, eight lanes a piece:
    // their stores then fill the banks (a row's pieces are 2 KB apart; with a
    // row's pieces in neighbouring lanes the stores took four times as long).
    constexpr int kQuads = KC / 4;                // loads per eight rows
    auto row_of = [&](int j) { return (j / kQuads) * 8 + (lane & 7); };
    auto piece_of = [&](int j) { return (j % kQuads) * 4 + (lane >> 3); };
    // The steps are read three steps of this warp ahead, the lists two, the
    // candidate counts one: a query whose candidate list has overflowed is
    // unproven whatever follows, so it is dropped.
    int idx[4], idx1[4], idx2[4];
    uint32_t qc[4];
    const int4 none = make_int4(0, 0, 0, 0);
    auto load_idx = [&](const int4& s, int (&x)[4]) {
      const uint16_t* l = a.list + (size_t)min((uint32_t)s.x, (uint32_t)a.nt - 1u) * a.stride;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t e = (uint32_t)(s.y + lane + 32 * j);
        x[j] = lane + 32 * j < s.z && e < a.stride ? min((int)l[e], a.m - 1) : -1;
      }
    };
    auto step_at = [&](uint32_t i) { return i < count ? it.step(i) : none; };
    load_idx(step_at(g), idx);
    load_idx(step_at(g + kGather), idx1);
    int4 s2 = step_at(g + 2 * kGather);
    uint32_t n = (uint32_t)(g >> 1);   // the step's number among its parity's
    for (uint32_t i = g; i < count; i += kGather, n += kGather / 2) {
      const uint32_t st = n % kA;
      load_idx(s2, idx2);
      s2 = step_at(i + 3 * kGather);
#pragma unroll
      for (int j = 0; j < 4; ++j) qc[j] = idx1[j] >= 0 ? __ldcg(a.qcnt + idx1[j]) : 0u;
      bool w = true;
      unsigned char* dst = sA + (p * kA + st) * kATile;
#pragma unroll
      for (int h = 0; h < KC / 2; ++h) {   // eight loads in flight
        uint4 v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int jj = h * 8 + j;
          const int q = __shfl_sync(kFull, idx[jj / kQuads / 4], row_of(jj) & 31);
          const uint4* src = reinterpret_cast<const uint4*>(q < 0 ? a.pad : a.qrow + (size_t)q * (KC * 8));
          v[j] = __ldg(src + piece_of(jj));
        }
        if (h == 0)
          w = __all_sync(kFull, mbar_wait_fast(a_empty + p * kA + st, ((n / kA) & 1u) ^ 1u, abort_flag, a.status,
                                               a.wait_ns));
        if (!w) break;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          *reinterpret_cast<uint4*>(dst + piece_of(h * 8 + j) * (PQ_ROWS * 16) + row_of(h * 8 + j) * 16) = v[j];
      }
      if (!w) break;
      uint16_t* si = s_idx + (p * kA + st) * PQ_ROWS;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        si[lane + 32 * j] = (uint16_t)idx[j];
        idx[j] = qc[j] <= a.cap ? idx1[j] : -1;
        idx1[j] = idx2[j];
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // this lane's rows, for the MMA's reads
      __syncwarp();
      if (lane == 0) mbar_arrive(a_full + p * kA + st);
    }
  } else if (warp <= 1) {
    // ---------------- MMA issue (and, warp 0, the tiles) ----------------
    if (lane == 0) {
      const int p = warp;
      const uint64_t ad0 = smem_desc(smem_u32(sA + p * kA * kATile), PQ_ROWS * 16, 128);
      const uint64_t bd0 = smem_desc(smem_u32(sB), PT_ROWS * 16, 128);
      constexpr uint64_t kAStep = (2 * PQ_ROWS * 16) >> 4, kBStep = (2 * PT_ROWS * 16) >> 4;
      // Warp 0 copies the tiles in order, up to kSlots - 1 ahead of the MMAs:
      // cw .. cl are the numbers of the current piece's tiles left to copy.
      uint32_t copied = 0, cp = 0;
      int cw = 0, cl = -1;
      auto enter = [&]() {   // the tiles of piece cp (none past the last)
        cl = -1;
        cw = 0;
        if (cp * it.len < count) {
          cw = it.steps[it.start(cp)].w;
          cl = it.steps[it.start(cp) + min(it.len, count - cp * it.len) - 1].w;
        }
      };
      if (p == 0) enter();
      // copies the tiles up to number `want` (block: waits for their slots;
      // else stops at the first that is still in use)
      auto copy_tiles = [&](uint32_t want, bool block) -> bool {
        for (; copied <= want && cw <= cl; ++copied) {
          const uint32_t slot = copied % kSlots, par = ((copied / kSlots) & 1u) ^ 1u;
          if (!mbar_test_wait(b_empty + slot, par)) {
            if (!block) return true;
            if (!mbar_wait_fast(b_empty + slot, par, abort_flag, a.status, a.wait_ns)) return false;
          }
          const uint32_t t = min((uint32_t)a.tile_of[cw], (uint32_t)a.nt - 1u);
          mbar_arrive_expect_tx(b_full + slot, kBTile);
          bulk_g2s(sB + slot * kBTile, (const unsigned char*)a.dop + (size_t)t * kBTile, kBTile, b_full + slot);
          if (cw++ == cl) {
            ++cp;
            enter();
          }
        }
        return true;
      };
      uint32_t n = 0;
      uint32_t o = (uint32_t)p < count ? it.tile(p, it.step(p)) : 0u;
      uint32_t at = 0xFFFFFFFFu;   // tile of this parity's step before
      bool ok = true;
      for (uint32_t i = p; i < count; i += 2, ++n) {
        const uint32_t st = n % kA, slot = o % kSlots;
        if (o != at) {
          ok = (p == 1 || copy_tiles(o, true)) &&
               mbar_wait_fast(b_full + slot, (o / kSlots) & 1u, abort_flag, a.status, a.wait_ns);
          at = o;
        }
        ok = ok && mbar_wait_fast(a_full + p * kA + st, (n / kA) & 1u, abort_flag, a.status, a.wait_ns);
        if (!ok) break;
        const uint64_t ad = ad0 + (uint64_t)st * (kATile >> 4), bd = bd0 + (uint64_t)slot * (kBTile >> 4);
        int4 s2;
        if (i + 2 < count) s2 = it.step(i + 2);
        ok = mbar_wait_fast(acc_empty + p, (n & 1u) ^ 1u, abort_flag, a.status, a.wait_ns);
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int ks = 0; ks < KC / 2; ++ks)
          mma_f16(tmem + (uint32_t)(p * PT_ROWS), ad + ks * kAStep, bd + ks * kBStep, kIdesc, ks > 0 ? 1u : 0u);
        mma_commit(acc_full + p);
        if (i + 2 < count) o = it.tile(i + 2, s2);
        // the next tiles, while their slots are free (tried at two steps of a
        // tile in 16: the poll costs an issuing thread about 100 cycles)
        if (p == 0 && (n & 7u) == 0u) copy_tiles(o + kSlots - 2, false);
      }
      if (p == 0 && ok) copy_tiles(0xFFFFFFFEu, true);   // what only the odd steps still need
      mma_commit(drain + p);
      mbar_drain(drain + p, 0u, a.status);
      // no copy may still be writing into shared memory at exit
      if (p == 0)
        for (uint32_t t = copied > kSlots ? copied - kSlots : 0; t < copied; ++t)
          mbar_drain(b_full + t % kSlots, (t / kSlots) & 1u, a.status);
      mbar_arrive(tmem_done);
    }
  } else {
    // ---------------- epilogue ----------------
    const int ew = warp - 2;
    const int p = (ew >> 2) & 1, sub = ew >> 3, quad = warp & 3;
    const int row = quad * 32 + lane;
    uint2* hit = s_hit + ew * 32 + lane;   // slot j of set t at [(t * kHits + j) * kEpi * 32]
    int set = 0, cnt = 0;
    // the records of the step before: cnt0 of them, for query q0 at place at0
    int q0 = 0, cnt0 = 0;
    uint32_t at0 = 0;
    auto put = [&]() {
      for (int j = 0; j < cnt0; ++j)
        if (at0 + j < a.cap) a.cand[(size_t)q0 * a.cap + at0 + j] = hit[((set ^ 1) * kHits + j) * (kEpi * 32)];
    };
    // the columns of a chunk whose values are negative (the entry may lie
    // within the radius of this lane's query): sign bits, four independent chains
    auto take = [&](const float (&v)[32], float m, uint32_t pos) {
      if (!__any_sync(kFull, m < 0.f)) return;
      uint32_t g[4] = {0, 0, 0, 0};
#pragma unroll
      for (int k = 0; k < 8; ++k)
#pragma unroll
        for (int b = 0; b < 4; ++b) g[b] = __funnelshift_l(__float_as_uint(v[8 * b + k]), g[b], 1);
      const uint32_t mine = (g[0] << 24) | (g[1] << 16) | (g[2] << 8) | g[3];
      if (mine) hit[(set * kHits + cnt) * (kEpi * 32)] = make_uint2(pos, mine);
      cnt += mine ? 1 : 0;
    };
    uint32_t n = 0;
    uint32_t passed = 0;   // tiles this parity is past (one lane releases them)
    const bool releaser = sub == 0 && quad == 0 && lane == 0;
    int4 s = (uint32_t)p < count ? it.step(p) : make_int4(0, 0, 0, 0);
    const uint32_t tb0 = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(p * PT_ROWS + sub * 128);
    bool ok = true;
    for (uint32_t i = p; ok && i < count; i += 2, ++n) {
      const uint32_t st = n % kA;
      const uint32_t pos0 = (uint32_t)s.x * PT_ROWS;
      const uint32_t ord = releaser ? it.tile(i, s) : 0u;
      if (i + 2 < count) s = it.step(i + 2);
      // (the stage's barrier has completed by then; waiting on it too orders
      // the read of the queries' numbers after their writes)
      ok = __all_sync(kFull, mbar_wait_fast<kAccPolls>(acc_full + p, n & 1u, abort_flag, a.status, a.wait_ns) &&
                                 mbar_wait_fast(a_full + p * kA + st, (n / kA) & 1u, abort_flag, a.status, a.wait_ns));
      if (!ok) break;
      tc_fence_after();
      // the MMAs of this parity's earlier steps have read their tiles
      if (releaser)
        for (; passed < ord; ++passed) mbar_arrive(b_empty + passed % kSlots);
      const int q = s_idx[(p * kA + st) * PQ_ROWS + row];
#pragma unroll 1
      for (int c = 0; c < 128; c += 32) {
        float v[32], m;
        __syncwarp();   // the TMEM loads are warp-collective: converge after the branches before
        tmem_ld32_min_issue(tb0 + (uint32_t)c, v, m);
        tmem_ld_wait(v, m);
        if (c == 96) {   // every read of the accumulator is done (and the MMAs have read the stage)
          tc_fence_before();
          __syncwarp();
          if (lane == 0) {
            if (a.inject != 1 || n < 1) mbar_arrive(acc_empty + p);
            mbar_arrive(a_empty + p * kA + st);
          }
        }
        take(v, m, pos0 + (uint32_t)(sub * 128 + c));
      }
      put();   // the step before's records
      cnt0 = (uint32_t)q < (uint32_t)a.m ? cnt : 0;
      q0 = q;
      // (in place: a copy of the result would wait for it here)
      asm volatile(
          "{\n\t.reg .pred p;\n\t"
          "setp.ne.s32 p, %2, 0;\n\t"
          "@p atom.global.add.u32 %0, [%1], %2;\n\t}\n"
          : "+r"(at0)
          : "l"(a.qcnt + (cnt0 > 0 ? q : 0)), "r"(cnt0)
          : "memory");
      cnt = 0;
      set ^= 1;
    }
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(tmem_done);
    put();
  }
  // The TMEM is freed once every epilogue warp is past its last read and every
  // MMA has completed.  The roles end at very different times, so this hangs
  // on a barrier of its own and not on the block's.
  __syncwarp();
  if (warp == 0) {
    const uint64_t t0 = globaltimer();
    while (!mbar_try_wait_sleep(tmem_done, 0u, 100000u))
      if (globaltimer() - t0 > a.wait_ns + kWaitNs) break;
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// ---------------------------------------------------------------------------
// exact selection among a query's candidates: one warp per query, one
// candidate per lane and round, the records expanded in shared memory (FP32
// difference form in the order of the other searches, so the distances are
// the same bits).  Queries whose K-th member is not within the radius are
// listed in fb.  Bound by the hits' rows, gathered from L2, and the sort of 32
// a round (258,064 queries on 1M entries: 401 us; the chunk rerank of the
// dense search 1.60 ms; the BF16 form with 2.06M on 4M: 6.2 ms, 15.7 ms).
//
// FORM 1, the precision form: its result is the K best members among the
// entries of the `chunks` dictionary chunks (32 consecutive entries) with the
// smallest BF16 distance d~.  That is the exact result here wherever the K
// members' chunks are all listed, and they are if no more than `chunks`
// chunks have an entry with d~ <= M, the largest d~ of the K members.  The
// candidates hold every entry with d~ <= T (k_radius), so it is enough to
// compute d~ of the candidates (BF16 operands, FP32 sums; mg bounds what the
// sums' order and the norm's three terms can change, and `trunc` the rounding
// of packed list keys) and count the chunks up to M + mg.  A query that
// fails this is searched by the dense filter like any query before:
// those past tail_q0, whose lists that filter cuts into parts, are listed
// apart.
// ---------------------------------------------------------------------------
constexpr int kDtRoom = 128;   // d~ kept per query: chunks past it fail the count anyway

template <int D>
__device__ __forceinline__ float bf16_distance(const float4* __restrict__ r4, const float4* q4, float qn) {
  // ||q||^2 + ||c||^2 - 2 q~ . c~
  float n2 = 0.f, dot = 0.f;
#pragma unroll
  for (int k = 0; k < (D + 3) / 4; ++k) {
    const float4 v4 = __ldg(r4 + k);
    const float x4[4] = {v4.x, v4.y, v4.z, v4.w};
    const float4 b4 = q4[k];
    const float b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      if (4 * k + t < D) {
        n2 = fmaf(x4[t], x4[t], n2);
        dot = fmaf(b[t], __bfloat162float(__float2bfloat16_rn(x4[t])), dot);
      }
    }
  }
  return qn + (n2 - 2.f * dot);
}

template <int D, int FORM>
__global__ void __launch_bounds__(128) k_rerank_list(
    const int32_t* __restrict__ perm, const float* __restrict__ rad, int nslab, const uint32_t* __restrict__ qcnt,
    const uint2* __restrict__ cand, uint32_t cap, const int32_t* __restrict__ order, int64_t nd,
    const float* __restrict__ qfeat, int dpad, const uint64_t* __restrict__ qkeys, const float* __restrict__ dfeat,
    const uint64_t* __restrict__ dkeys, int L, int tmin, int K, FilterError fe, int chunks, float trunc,
    int64_t tail_q0, const uint32_t* __restrict__ given_up, int32_t* __restrict__ nbr, float* __restrict__ dist, int32_t* __restrict__ fb_list,
    unsigned long long* __restrict__ fb_count, int32_t* __restrict__ tail_list,
    unsigned long long* __restrict__ tail_count) {
  constexpr int kRow4 = (D + 3) / 4;
  __shared__ float4 s_qb[FORM == 1 ? 4 : 1][kRow4];            // the query in BF16
  __shared__ float s_dt[FORM == 1 ? 4 : 1][kDtRoom];           // d~ <= T of the candidates
  __shared__ int s_ch[FORM == 1 ? 4 : 1][kDtRoom];             // and their chunks
  uint32_t kept = 0;
  float qn = 0.f, mg = 0.f;
  __shared__ uint64_t s_qk[4][32];
  __shared__ float4 s_q4[4][kRow4];
  __shared__ float2 s_m[4][32];
  __shared__ uint32_t s_pos[4][32 * 32];   // positions of 32 records
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int64_t q = (int64_t)blockIdx.x * 4 + wib;
  if (q >= nslab) return;   // warp-uniform
  const int64_t oq = perm[q];
  const float T = rad[q];
  const uint32_t n = qcnt[q];
  bool flagged = !(T >= 0.f) || n > cap || *given_up != 0;
  if (!flagged) {
    if (lane < L) s_qk[wib][lane] = qkeys[oq * L + lane];
    if (lane < kRow4) s_q4[wib][lane] = reinterpret_cast<const float4*>(qfeat + oq * dpad)[lane];
    __syncwarp();
    if constexpr (FORM == 1) {
      const float4* q4 = s_q4[wib];
#pragma unroll
      for (int k = 0; k < kRow4; ++k) {
        const float4 v = q4[k];
        if (4 * k < D) qn = fmaf(v.x, v.x, qn);
        if (4 * k + 1 < D) qn = fmaf(v.y, v.y, qn);
        if (4 * k + 2 < D) qn = fmaf(v.z, v.z, qn);
        if (4 * k + 3 < D) qn = fmaf(v.w, v.w, qn);
      }
      if (lane < kRow4) {
        float4 v = q4[lane];
        v.x = __bfloat162float(__float2bfloat16_rn(v.x));
        v.y = __bfloat162float(__float2bfloat16_rn(v.y));
        v.z = __bfloat162float(__float2bfloat16_rn(v.z));
        v.w = __bfloat162float(__float2bfloat16_rn(v.w));
        s_qb[wib][lane] = v;
      }
      const float rc = sqrtf(qn) + sqrtf(T) * 1.1f;
      // twice the sums' bound for the member that sets M and for the other entry
      mg = 4.f * (fe.c_sq * (rc * rc + qn) + fe.c_abs * (sqrtf(qn) + rc)) + 1e-12f;
      __syncwarp();
    }
    float bd = FLT_MAX, dK = FLT_MAX;
    int bi = INT_MAX, iK = INT_MAX, members = 0;
    // the records' positions, 32 records at a time, then 32 entries at a time
    uint32_t rec = 0, have = 0, b = 0;
    while (true) {
      if (b >= have) {
        if (rec >= n) break;
        const uint2 rc = rec + lane < n ? cand[q * cap + rec + lane] : make_uint2(0u, 0u);
        const uint32_t c = (uint32_t)__popc(rc.y);
        uint32_t x = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(kFull, x, o);
          if (lane >= o) x += y;
        }
        have = __shfl_sync(kFull, x, 31);
        __syncwarp();   // every lane is past its reads of the positions before
        uint32_t at = x - c;
        for (uint32_t m = rc.y; m; m &= m - 1) s_pos[wib][at++] = rc.x + (uint32_t)(32 - __ffs(m));
        __syncwarp();
        rec += 32;
        b = 0;
        continue;
      }
      float dd = FLT_MAX;
      int eid = INT_MAX;
      if (b + lane < have) {
        const int64_t pos = s_pos[wib][b + lane];
        if (pos < nd) eid = order[pos];   // not a padding row
      }
      b += 32;
      if (eid != INT_MAX) {
        const float4* r4 = reinterpret_cast<const float4*>(dfeat + (int64_t)eid * dpad);
        dd = 0.f;
#pragma unroll
        for (int k = 0; k < kRow4; ++k) {
          const float4 v4 = __ldg(r4 + k);
          const float x4[4] = {v4.x, v4.y, v4.z, v4.w};
          const float4 q4 = s_q4[wib][k];
          const float qx4[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            if (4 * k + t < D) {
              const float df = qx4[t] - x4[t];
              dd = fmaf(df, df, dd);
            }
          }
        }
      }
      if constexpr (FORM == 1) {
        bool keep = false;
        float dt = 0.f;
        if (eid != INT_MAX) {
          dt = bf16_distance<D>(reinterpret_cast<const float4*>(dfeat + (int64_t)eid * dpad), s_qb[wib], qn);
          keep = dt <= T;
        }
        const unsigned km = __ballot_sync(kFull, keep);
        const uint32_t at = kept + (uint32_t)__popc(km & lanes_below(lane));
        if (keep && at < (uint32_t)kDtRoom) {
          s_dt[wib][at] = dt;
          s_ch[wib][at] = eid >> 5;
        }
        kept += (uint32_t)__popc(km);
      }
      // ascending (distance, ID); membership is tested in that order until K
      // members of this round are known (no later one can enter) or the
      // entries lie past the K best of the rounds before
      warp_sort32(dd, eid, lane);
      bool mem = false;
      int found = 0;
      for (int j0 = 0; j0 < 32 && found < K;) {
        const int j1 = min(32, j0 + K - found + 2);
        const bool in = lane >= j0 && lane < j1 && eid != INT_MAX && lex_less(dd, eid, dK, iK);
        if (!__any_sync(kFull, in)) break;
        if (in) mem = lsh_member(dkeys + (int64_t)eid * L, s_qk[wib], L, tmin);
        found = __popc(__ballot_sync(kFull, mem));
        j0 = j1;
      }
      members += found;
      if (found > 0) {
        // close the gaps the non-members left (the members are in order)
        const unsigned mm = __ballot_sync(kFull, mem);
        if (mem) s_m[wib][__popc(mm & lanes_below(lane))] = make_float2(dd, __int_as_float(eid));
        __syncwarp();
        const float2 c = s_m[wib][lane];
        __syncwarp();
        const float v = lane < found ? c.x : FLT_MAX;
        const int id = lane < found ? __float_as_int(c.y) : INT_MAX;
        if (members == found) {   // the first members
          bd = v;
          bi = id;
        } else {
          warp_merge_best(bd, bi, v, id, K, lane);
        }
      }
      if (members >= K) {
        dK = __shfl_sync(kFull, bd, K - 1);
        iK = __shfl_sync(kFull, bi, K - 1);
      }
    }
    flagged = members < K || !(dK <= T);
    if constexpr (FORM == 1) {
      if (!flagged) {   // warp-uniform
        float M = -FLT_MAX;
        if (lane < K)
          M = bf16_distance<D>(reinterpret_cast<const float4*>(dfeat + (int64_t)bi * dpad), s_qb[wib], qn);
#pragma unroll
        for (int o = 16; o; o >>= 1) M = fmaxf(M, __shfl_xor_sync(kFull, M, o));
        M += fabsf(M) * trunc + mg;
        flagged = !(M <= T) || kept > (uint32_t)kDtRoom;
        if (!flagged) {
          __syncwarp();
          // distinct chunks with d~ <= M: an entry counts if no earlier one
          // of its chunk does
          uint32_t c = 0;
          for (uint32_t i = lane; i < kept; i += 32)
            c += s_dt[wib][i] <= M ? 1u : 0u;
          c = __reduce_add_sync(kFull, c);
          if (c > (uint32_t)chunks) {
            c = 0;
            for (uint32_t i = lane; i < kept; i += 32) {
              bool first = s_dt[wib][i] <= M;
              for (uint32_t j = 0; first && j < i; ++j) first = !(s_dt[wib][j] <= M && s_ch[wib][j] == s_ch[wib][i]);
              c += first ? 1u : 0u;
            }
            c = __reduce_add_sync(kFull, c);
          }
          flagged = c > (uint32_t)chunks;
        }
      }
    }
    if (!flagged && lane < K) {
      nbr[oq * K + lane] = bi;
      dist[oq * K + lane] = bd;
    }
  }
  if (flagged && lane == 0) {
    if (FORM == 1 && oq >= tail_q0) tail_list[atomicAdd(tail_count, 1ull)] = (int32_t)oq;
    else fb_list[atomicAdd(fb_count, 1ull)] = (int32_t)oq;
  }
}

template <int KC, uint32_t T>
cudaError_t run_tg(const TgArgs& a, int grid, cudaStream_t st) {
  auto kern = k_knn_tg<KC, T>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, tg_smem(KC));
  if (e != cudaSuccess) return e;
  cudaFuncAttributes fa;
  e = cudaFuncGetAttributes(&fa, kern);
  if (e != cudaSuccess) return e;
  if (fa.maxThreadsPerBlock < kTgThreads) return cudaErrorLaunchOutOfResources;
  kern<<<grid, kTgThreads, tg_smem(KC), st>>>(a);
  return cudaGetLastError();
}

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

// Where the search order is the faster search (zoom_internal.h has both sides).
static bool takes_search_order(int64_t n, int form, int K, int chunks, int64_t nq) {
  const bool bf16 = form == 1, few = bf16 && chunks < 2 * K;
  if (few && K > 12) return false;
  if (nq >= kPruneMinQueries) return !(bf16 && K < 6 && n < 131072 && nq < 4 * kPruneMinQueries);
  return nq * n >= kPruneMinPairs[bf16] && nq >= kPruneFewQueries[few ? 2 : bf16];
}

bool prune_plan(zoom_index ix, int form, int K, int chunks, int64_t nq, PrunePlan* p) {
  if (ix->tree_tiles == 0 || K > 16 || !takes_search_order(ix->dict->n, form, K, chunks, nq)) return false;
  p->form = form;
  p->kc = tc_kc(ix->dict->d, form);
  // the seeds' list must hold the r-th chunk minimum: two more than K, so
  // that K of the entries below it are members of the candidate set
  p->mc = K + 2 <= 16 ? 16 : 32;
  p->r = K + 2;
  p->cap = 128;
  const int64_t nt = ix->tree_tiles;
  // the tiles' query lists: one 16-bit number per query of the slab, at most 2 GB
  int64_t slab = (int64_t{1} << 31) / (2 * nt) / 256 * 256;
  slab = slab < 65280 ? slab : 65280;   // 0xFFFF marks no query
  const int64_t all = (nq + 255) / 256 * 256;
  p->slab = slab < all ? slab : all;
  return p->slab >= 256;
}

namespace {

struct Ws {
  char* base;
  size_t off = 0;
  template <typename T>
  T* take(size_t n) {
    off = (off + 255) & ~(size_t)255;
    T* r = (T*)(base ? base + off : nullptr);
    off += n * sizeof(T);
    return r;
  }
};

struct PruneBufs {
  uint32_t* hist;
  uint16_t *leaf, *qrow, *qop, *list;
  uint32_t *rank, *tcnt, *qcnt, *off, *ord;
  unsigned long long* pairs;
  uint2* cand;
  float *qn, *ld, *rad, *vis;
  uint4* qz;
  int32_t *perm, *seeds, *li, *tile_of;
  int4* steps;
};

size_t carve(zoom_index ix, const PrunePlan& p, int64_t nq, void* ws, PruneBufs* b) {
  Ws w{(char*)ws};
  const int64_t nqp = (nq + 255) / 256 * 256, nt = ix->tree_tiles;
  b->hist = w.take<uint32_t>((size_t)1 << (ix->tree_d1 + ix->tree_d2));
  b->leaf = w.take<uint16_t>(nq);
  b->rank = w.take<uint32_t>(nq);
  b->perm = w.take<int32_t>(nq);
  b->qrow = w.take<uint16_t>((size_t)(nqp + 1) * p.kc * 8);   // and the padding row
  b->qop = w.take<uint16_t>((size_t)nqp * p.kc * 8);
  b->qn = w.take<float>(nqp);
  b->qz = w.take<uint4>(2 * nqp);
  b->seeds = w.take<int32_t>(nqp / 256 * PQ_SEEDS);
  b->ld = w.take<float>((size_t)nq * p.mc);
  b->li = w.take<int32_t>((size_t)nq * p.mc);
  b->rad = w.take<float>(nq);
  b->vis = w.take<float>(nq);
  b->tcnt = w.take<uint32_t>(2 + nt + p.slab);   // pairs (64 bits), tile counts, candidate counts: one memset
  b->pairs = (unsigned long long*)b->tcnt;
  b->tcnt = b->tcnt ? b->tcnt + 2 : nullptr;
  b->qcnt = b->tcnt ? b->tcnt + nt : nullptr;
  b->off = w.take<uint32_t>(nt + 2);
  b->ord = w.take<uint32_t>(nt);
  b->tile_of = w.take<int32_t>(nt);
  b->steps = w.take<int4>((size_t)nt + (size_t)nt * p.slab / PQ_ROWS);
  b->cand = w.take<uint2>((size_t)p.slab * p.cap);
  b->list = w.take<uint16_t>((size_t)nt * p.slab);
  return w.off;
}

}  // namespace

size_t prune_ws_bytes(zoom_index ix, const PrunePlan& p, int64_t nq) {
  PruneBufs b;
  return carve(ix, p, nq, nullptr, &b) + 256;
}

cudaError_t run_pruned(zoom_index ix, const PrunePlan& p, const float* qfeat, const uint64_t* qkeys, int64_t nq,
                       int K, int32_t* nbr, float* dist, void* ws, int32_t* fb, unsigned long long* fb_count,
                       int32_t* fb_tail, unsigned long long* tail_count, cudaStream_t st) {
  zoom_dict d = ix->dict;
  zoom_ctx ctx = d->ctx;
  PruneBufs b;
  carve(ix, p, nq, ws, &b);
  const int d1 = ix->tree_d1, d2 = ix->tree_d2, nt = (int)ix->tree_tiles, ns = (nt + PT_SUPER - 1) / PT_SUPER;
  const int leaves = 1 << (d1 + d2);
  const TreeNode* n1 = (const TreeNode*)ix->tree_node1;
  const TreeNode* n2 = (const TreeNode*)ix->tree_node2;
  const uint4* box = (const uint4*)ix->tree_box;
  const uint4* sbox = (const uint4*)ix->tree_sbox;
  const FilterError fe = tc_filter_error(d->d, p.form);
  const uint16_t* dop = p.form == 1 ? ix->tree_bf : ix->tree_f1;
  const unsigned qb = (unsigned)((nq + 127) / 128);
  cudaError_t e = cudaMemsetAsync(b.hist, 0, (size_t)leaves * 4, st);
  if (e != cudaSuccess) return e;
#define ZOOM_PR_SORT(DD)                                                                                          \
  do {                                                                                                            \
    constexpr int kKc = 4;                                                                                        \
    k_query_route<DD><<<qb, 128, 0, st>>>(qfeat, d->dpad, nq, ix->tree_basis, n1, n2, d1, d2, b.leaf, b.rank, b.hist); \
    k_leaf_scan<<<1, 1024, 0, st>>>(b.hist, leaves);                                                              \
    if (p.form == 1)                                                                                              \
      k_query_sorted<DD, kKc, 1><<<qb, 128, 0, st>>>(qfeat, d->dpad, nq, ix->tree_basis, b.leaf, b.rank, b.hist,    \
                                                     b.qrow, b.qop, b.qn, b.qz, b.perm);                          \
    else                                                                                                          \
      k_query_sorted<DD, kKc, 2><<<qb, 128, 0, st>>>(qfeat, d->dpad, nq, ix->tree_basis, b.leaf, b.rank, b.hist,    \
                                                     b.qrow, b.qop, b.qn, b.qz, b.perm);                          \
  } while (0)
  switch (d->d) {
    case 9: ZOOM_PR_SORT(9); break;
    case 25: ZOOM_PR_SORT(25); break;
    case 18: ZOOM_PR_SORT(18); break;
    default: return cudaErrorInvalidValue;
  }
#undef ZOOM_PR_SORT
  const int seed_smem = 8 * ns * 4;   // at most 64 KB
  e = cudaFuncSetAttribute(k_seed_tiles, cudaFuncAttributeMaxDynamicSharedMemorySize, 8 * 2048 * 4);
  if (e != cudaSuccess) return e;
  k_seed_tiles<<<(unsigned)((nq + 255) / 256), 256, seed_smem, st>>>(
      b.qz, nq, (const float4*)ix->tree_smid, ns, (const float4*)ix->tree_mid, nt, b.seeds);
  e = cudaGetLastError();
  zoom_stage_mark(ctx, 8, st);   // start of the tensor-core filter kernels
  if (e == cudaSuccess)
    e = launch_knn_seeds(b.qop, b.qn, nq, dop, d->n, p.form, p.kc, p.mc, b.seeds, ctx->n_sm, b.ld, b.li,
                         ctx->d_status, st, ctx->wait_ns, ctx->inject);
  if (e != cudaSuccess) return e;
  uint16_t* pad = b.qrow + (size_t)((nq + 255) / 256 * 256) * p.kc * 8;
  {
    const unsigned blocks = (unsigned)((nq + 255) / 256);
    if (p.form == 1)
      k_radius<1><<<blocks, 256, 0, st>>>(b.ld, p.mc, p.r, b.qn, nq, fe, p.trunc, d->d, p.kc * 8, b.rad, b.vis, b.qrow, pad);
    else
      k_radius<2><<<blocks, 256, 0, st>>>(b.ld, p.mc, p.r, b.qn, nq, fe, p.trunc, d->d, p.kc * 8, b.rad, b.vis, b.qrow, pad);
  }
  // enough warps to fill the SMs: a warp takes 32 queries and every parts-th
  // group of 32 super tiles
  int parts = 1;
  while (parts < 16 && parts * 32 < ns && (p.slab / 32) * parts < (int64_t)ctx->n_sm * 48) parts *= 2;
  const int tmin = ix->t;
  for (int64_t q0 = 0; q0 < nq; q0 += p.slab) {
    const int m = (int)(nq - q0 < p.slab ? nq - q0 : p.slab);
    e = cudaMemsetAsync(b.pairs, 0, (size_t)(2 + nt + p.slab) * 4, st);
    if (e != cudaSuccess) return e;
    const int warps = (m + 31) / 32 * parts;
    const unsigned long long give_up = (unsigned long long)m * nt / p.give_up;
    k_visit<<<(warps + 7) / 8, 256, 0, st>>>(b.qz + 2 * q0, b.vis + q0, m, box, nt, sbox, ns, parts, b.list,
                                             (uint32_t)p.slab, b.tcnt, give_up, b.pairs);
    k_step_scan<<<1, 1024, 0, st>>>(b.tcnt, nt, b.off, b.ord, give_up, b.pairs);
    k_steps<<<(nt * 8 + 255) / 256, 256, 0, st>>>(b.tcnt, nt, b.off, b.ord, b.steps, b.tile_of);
    TgArgs a;
    a.qrow = b.qrow + (size_t)q0 * p.kc * 8;
    a.pad = pad;
    a.m = m;
    a.nt = nt;
    a.list = b.list;
    a.stride = (uint32_t)p.slab;
    a.steps = b.steps;
    a.n_steps = b.off + nt;
    a.tile_of = b.tile_of;
    a.dop = dop;
    a.qcnt = b.qcnt;
    a.cand = b.cand;
    a.cap = p.cap;
    a.status = ctx->d_status;
    a.wait_ns = ctx->wait_ns > 0 ? ctx->wait_ns : kWaitNs;
    a.inject = ctx->inject;
    e = p.form == 1 ? run_tg<4, 1>(a, ctx->n_sm, st) : run_tg<4, 0>(a, ctx->n_sm, st);
    if (e != cudaSuccess) return e;
#define ZOOM_PR_LIST(DD, FF)                                                                                      \
  k_rerank_list<DD, FF><<<(m + 3) / 4, 128, 0, st>>>(                                                           \
      b.perm + q0, b.rad + q0, m, b.qcnt, b.cand, p.cap, ix->tree_order, d->n, qfeat, d->dpad, qkeys, d->feat,  \
      ix->dkeys, ix->L, tmin, K, fe, p.chunks, p.trunc, p.tail_q0, b.off + nt + 1, nbr, dist, fb, fb_count, fb_tail, tail_count)
    switch (d->d + (p.form == 1 ? 100 : 0)) {
      case 9: ZOOM_PR_LIST(9, 2); break;
      case 25: ZOOM_PR_LIST(25, 2); break;
      case 18: ZOOM_PR_LIST(18, 2); break;
      case 109: ZOOM_PR_LIST(9, 1); break;
      case 125: ZOOM_PR_LIST(25, 1); break;
      default: ZOOM_PR_LIST(18, 1); break;
    }
#undef ZOOM_PR_LIST
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  zoom_stage_mark(ctx, 9, st);   // end of the filter kernels (their reranks included)
  return cudaGetLastError();
}
