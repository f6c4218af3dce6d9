// Merge of a row's split-vocab partials, shared by the row kernels.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "molt_internal.cuh"
#include "ptx.cuh"

namespace molt {

// A block of kTileM * kMergeGroups threads merges kTileM rows: thread (r, g) =
// (tid % kTileM, tid / kTileM) reads every kMergeGroups-th partial of row r, so
// that neighbouring threads read neighbouring rows and a row's partials, up to
// two per 256 vocab columns when the call has few rows, are read eight at a time
// instead of one after another (T = 1031, V = 151936: 89 us with one thread per
// row).
constexpr int kMergeGroups = 8;
constexpr int kMergeThreads = kTileM * kMergeGroups;

struct RowStats {
  float M, S, Q;   // max z, sum e^(z - M), sum e^(z - M)(z - M)
};

// The statistics of packed row k (any value where !act), valid in the threads
// of group 0; every thread of the block calls it.
__device__ __forceinline__ RowStats merge_row_parts(const float4* __restrict__ part, int64_t stride, int n_parts,
                                                    int k, bool act) {
  __shared__ float sh_m[kMergeGroups][kTileM];
  __shared__ float2 sh_sq[kMergeGroups][kTileM];
  constexpr float kLog2e = 1.4426950408889634f;
  const int r = threadIdx.x % kTileM, g = threadIdx.x / kTileM;
  const float4* p0 = part + k;
  float M = -INFINITY;
  if (act) {
#pragma unroll 4
    for (int s = g; s < n_parts; s += kMergeGroups) M = fmaxf(M, p0[s * stride].x);
  }
  sh_m[g][r] = M;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kMergeGroups; ++i) M = fmaxf(M, sh_m[i][r]);
  float S = 0.f, Q = 0.f;
  if (act) {
#pragma unroll 4
    for (int s = g; s < n_parts; s += kMergeGroups) {
      const float4 p = p0[s * stride];
      if (p.y > 0.f) {
        const float d = p.x - M;
        const float f = ex2_approx(d * kLog2e);
        S += f * p.y;
        Q += f * (p.z + d * p.y);
      }
    }
  }
  sh_sq[g][r] = make_float2(S, Q);
  __syncthreads();
  S = Q = 0.f;
#pragma unroll
  for (int i = 0; i < kMergeGroups; ++i) {
    S += sh_sq[i][r].x;
    Q += sh_sq[i][r].y;
  }
  return {M, S, Q};
}

}  // namespace molt
