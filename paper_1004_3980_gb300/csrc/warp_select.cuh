// Warp-wide selection helpers of the reranks: (distance, ID) order, a bitonic
// sort of one pair per lane, the merge with the K best, and the t-of-L
// membership test.
#pragma once
#include <cuda_runtime.h>
#include <float.h>
#include <limits.h>
#include <stdint.h>

namespace {

__device__ __forceinline__ bool lex_less(float a, int ai, float b, int bi) {
  return a < b || (a == b && ai < bi);
}

// Bitonic sort of one (value, ID) pair per lane, ascending across the lanes.
__device__ __forceinline__ void warp_sort32(float& v, int& id, int lane) {
#pragma unroll
  for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, v, j);
      const int oi = __shfl_xor_sync(0xffffffffu, id, j);
      const bool keep_small = ((lane & j) == 0) == ((lane & k) == 0);
      if (keep_small == lex_less(ov, oi, v, id)) {
        v = ov;
        id = oi;
      }
    }
  }
}

// Merges 32 ascending candidates (one per lane) into the ascending K best
// held by lanes 0..K-1: min(A[j], B[31 - j]) is a bitonic sequence holding
// the 32 smallest of both, which a bitonic merge sorts.
__device__ __forceinline__ void warp_merge_best(float& bd, int& bi, float v, int id, int K, int lane) {
  float a = lane < K ? bd : FLT_MAX;
  int ai = lane < K ? bi : INT_MAX;
  const float rb = __shfl_sync(0xffffffffu, v, 31 - lane);
  const int rbi = __shfl_sync(0xffffffffu, id, 31 - lane);
  if (lex_less(rb, rbi, a, ai)) {
    a = rb;
    ai = rbi;
  }
#pragma unroll
  for (int j = 16; j > 0; j >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, a, j);
    const int oi = __shfl_xor_sync(0xffffffffu, ai, j);
    if (((lane & j) == 0) == lex_less(ov, oi, a, ai)) {
      a = ov;
      ai = oi;
    }
  }
  bd = a;
  bi = ai;
}

// t-of-L membership: at least tmin of the entry's L bucket keys equal the
// query's.  Eight tables at a time (loads issued together); stops at tmin
// hits.
__device__ __forceinline__ bool lsh_member(const uint64_t* __restrict__ dk, const uint64_t* qk, int L,
                                           int tmin) {
  int hits = 0;
  for (int l0 = 0; l0 < L && hits < tmin; l0 += 8) {
    uint64_t kk[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) kk[j] = l0 + j < L ? __ldg(dk + l0 + j) : 0ull;
#pragma unroll
    for (int j = 0; j < 8; ++j) hits += (l0 + j < L && kk[j] == qk[l0 + j]) ? 1 : 0;
  }
  return hits >= tmin;
}

}  // namespace
