// Merge of a row's split-vocab partials, shared by the row kernels.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "molt_internal.cuh"
#include "ptx.cuh"

namespace molt {

// A block of kRedRows * kGroups threads merges kRedRows rows: thread (r, g) = (lane,
// warp) reads every kGroups-th partial of row r, so that a warp reads whole lines
// and a row's partials, one per vocab split and as many as 594 when the call has
// few rows, are read kGroups at a time.  Few rows are spread over more blocks than
// tiles of 128 would give (T = 100, V = 151936: 51 us with 128 rows and eight
// groups to a block).
constexpr int kMergeGroupsMany = 32, kMergeGroupsFew = 8;
inline int merge_groups(int n_parts) { return n_parts > 32 ? kMergeGroupsMany : kMergeGroupsFew; }

struct RowStats {
  float M, S, Q;   // max z, sum e^(z - M), sum e^(z - M)(z - M)
};

// The statistics of packed row k (any value where !act), valid in warp 0; every
// thread of the block calls it.
template <int kGroups>
__device__ __forceinline__ RowStats merge_row_parts(const float4* __restrict__ part, int64_t stride, int n_parts,
                                                    int k, bool act) {
  __shared__ float sh_m[kGroups][kRedRows];
  __shared__ float2 sh_sq[kGroups][kRedRows];
  constexpr float kLog2e = 1.4426950408889634f;
  const int r = threadIdx.x % kRedRows, g = threadIdx.x / kRedRows;
  const float4* p0 = part + k;
  float M = -INFINITY;
  if (act) {
#pragma unroll 4
    for (int s = g; s < n_parts; s += kGroups) M = fmaxf(M, p0[s * stride].x);
  }
  sh_m[g][r] = M;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kGroups; ++i) M = fmaxf(M, sh_m[i][r]);
  float S = 0.f, Q = 0.f;
  if (act) {
#pragma unroll 4
    for (int s = g; s < n_parts; s += kGroups) {
      const float4 p = p0[s * stride];
      if (p.y != 0.f) {   // 0: no columns.  A NaN passes
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
  if (g == 0) {
#pragma unroll
    for (int i = 0; i < kGroups; ++i) {
      S += sh_sq[i][r].x;
      Q += sh_sq[i][r].y;
    }
  }
  return {M, S, Q};
}

}  // namespace molt
