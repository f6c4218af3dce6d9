// Row-level kernels of the policy-update path: GRPO advantages, advantage
// broadcast, mask count, the packing of the active rows and of the rows with a
// gradient, the split-vocab merge with the clipped surrogate, the fixed-order loss
// reduction and the dhidden cast.  None of these is a contraction; they are launch- or HBM-bound.
#include <cstdint>
#include <cuda_runtime.h>

#include "merge.cuh"
#include "molt_internal.cuh"
#include "ptx.cuh"

namespace molt {
namespace {

constexpr float kLog2e = 1.4426950408889634f;

// ---------------------------------------------------------------------------
// Advantage estimators (Sec. 4.5: GRPO, a group-mean baseline, Dr. GRPO, RLOO,
// REINFORCE++; Sec. 4.2: one reward per rollout).  One warp per response index;
// the warp whose index starts a run of equal ids processes that group (for
// REINFORCE++, gid == nullptr and warp 0 normalises the whole batch).  Lanes
// load the rewards coalesced, 32 at a time, and fold them with shuffles in
// index order, so the fp64 sums run in the same order as a sequential loop.
// Explicit _rn intrinsics keep the compiler from contracting a multiply and an
// add into an FMA.
// ---------------------------------------------------------------------------
__global__ void group_adv_kernel(const float* __restrict__ r, const int32_t* __restrict__ gid, int n, double eps,
                                 int est, float* __restrict__ out, unsigned* err) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (warp >= n) return;
  int start = warp, end = n;
  if (gid == nullptr) {
    if (warp != 0) return;
  } else {
    const int g = gid[start];
    if (start > 0) {
      const int gp = gid[start - 1];
      if (gp == g) return;
      if (gp > g && lane == 0) atomicOr(err, kDevErrUnsortedGroups);
    }
    // end of the run
    for (int base = start;; base += 32) {
      const int j = base + lane;
      const bool same = (j < n) && (gid[j] == g);
      const unsigned m = __ballot_sync(0xffffffffu, same);
      if (m == 0xffffffffu) {
        end = base + 32;
        continue;
      }
      end = base + __ffs(~m) - 1;
      break;
    }
  }
  const int cnt = end - start;
  if (cnt == 1) {
    if (lane == 0) out[start] = 0.0f;
    return;
  }
  double s = 0.0;
  for (int base = start; base < end; base += 32) {
    const int j = base + lane;
    const double v = (j < end) ? static_cast<double>(r[j]) : 0.0;
    const int k = min(32, end - base);
    for (int i = 0; i < k; ++i) {
      const double vi = __shfl_sync(0xffffffffu, v, i);
      s = __dadd_rn(s, vi);
    }
  }
  s = __shfl_sync(0xffffffffu, s, 0);
  if (est == kAdvRloo) {
    // leave-one-out baseline (sum - r_j) / (n - 1)
    for (int base = start; base < end; base += 32) {
      const int j = base + lane;
      if (j < end) {
        const double rj = static_cast<double>(r[j]);
        const double b = __ddiv_rn(__dsub_rn(s, rj), static_cast<double>(cnt - 1));
        out[j] = __double2float_rn(__dsub_rn(rj, b));
      }
    }
    return;
  }
  const double mean = __ddiv_rn(s, static_cast<double>(cnt));
  if (est == kAdvGroupMean || est == kAdvDrGrpo) {
    for (int base = start; base < end; base += 32) {
      const int j = base + lane;
      if (j < end) out[j] = __double2float_rn(__dsub_rn(static_cast<double>(r[j]), mean));
    }
    return;
  }
  double ss = 0.0;
  for (int base = start; base < end; base += 32) {
    const int j = base + lane;
    const double d = (j < end) ? __dsub_rn(static_cast<double>(r[j]), mean) : 0.0;
    const double d2 = __dmul_rn(d, d);
    const int k = min(32, end - base);
    for (int i = 0; i < k; ++i) ss = __dadd_rn(ss, __shfl_sync(0xffffffffu, d2, i));
  }
  ss = __shfl_sync(0xffffffffu, ss, 0);
  const double sd = __dsqrt_rn(__ddiv_rn(ss, static_cast<double>(cnt - 1)));
  const double den = __dadd_rn(sd, eps);
  for (int base = start; base < end; base += 32) {
    const int j = base + lane;
    if (j < end) {
      const double d = __dsub_rn(static_cast<double>(r[j]), mean);
      out[j] = __double2float_rn(__ddiv_rn(d, den));
    }
  }
}

__global__ void broadcast_kernel(const float* __restrict__ adv, const int32_t* __restrict__ rot, int n_resp, int T,
                                 float* __restrict__ out) {
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < T; t += gridDim.x * blockDim.x) {
    const int k = rot[t];
    out[t] = (k >= 0 && k < n_resp) ? adv[k] : 0.0f;
  }
}

// sum of a uint8 mask: 16 bytes per load, per-block total, one atomic per block
__global__ void mask_count_kernel(const uint8_t* __restrict__ mask, int64_t T,
                                  unsigned long long* __restrict__ out) {
  unsigned long long c = 0;
  const int64_t nvec = T / 16;
  const uint4* m4 = reinterpret_cast<const uint4*>(mask);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nvec; i += (int64_t)gridDim.x * blockDim.x) {
    const uint4 v = m4[i];
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) c += (w[q] & 0xFFu ? 1 : 0) + (w[q] & 0xFF00u ? 1 : 0) +
                                     (w[q] & 0xFF0000u ? 1 : 0) + (w[q] & 0xFF000000u ? 1 : 0);
  }
  for (int64_t i = nvec * 16 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < T;
       i += (int64_t)gridDim.x * blockDim.x)
    c += mask[i] ? 1 : 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  __shared__ unsigned long long sh[32];
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long tot = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += sh[w];
    if (tot) atomicAdd(out, tot);
  }
}

// ---------------------------------------------------------------------------
// Order-preserving packing.  A grid of kPackThreads-thread blocks splits the rows
// evenly; each block counts the live rows before its own (a vectorised scan of the
// flags up to there, a few us at most: they sit in L2), so the count, the maps and
// the copies are one launch.  Before, one block compacted and a second kernel
// copied: 4 us more on the smallest call, 13 of 46 at T = 32768.
// ---------------------------------------------------------------------------
constexpr int kPackThreads = 256;

__device__ __forceinline__ int block_sum(int v) {
  __shared__ int ws[kPackThreads / 32];
  v = __reduce_add_sync(0xffffffffu, v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
  __syncthreads();
  int t = 0;
#pragma unroll
  for (int i = 0; i < kPackThreads / 32; ++i) t += ws[i];
  return t;
}

// nonzero bytes of m[0, n), by the whole block
__device__ __forceinline__ int count_bytes(const uint8_t* __restrict__ m, int n) {
  const int head = min(n, static_cast<int>((16 - (reinterpret_cast<uintptr_t>(m) & 15)) & 15));
  const int nvec = (n - head) / 16;
  const uint4* v = reinterpret_cast<const uint4*>(m + head);
  auto word = [](uint32_t w) { return __popc((((w & 0x7f7f7f7fu) + 0x7f7f7f7fu) | w) & 0x80808080u); };
  int c = 0;
  for (int i = threadIdx.x; i < head; i += kPackThreads) c += m[i] ? 1 : 0;
#pragma unroll 4
  for (int i = threadIdx.x; i < nvec; i += kPackThreads) {
    const uint4 x = v[i];
    c += word(x.x) + word(x.y) + word(x.z) + word(x.w);
  }
  for (int i = head + 16 * nvec + threadIdx.x; i < n; i += kPackThreads) c += m[i] ? 1 : 0;
  return block_sum(c);
}

// The block's share of rows [0, n), 256 at a time: row(k, live, j) for every row k
// (j its index among the live ones, `before` of which precede the share), then the
// live rows' hidden rows copied from src row k to dst row j (src nullptr: none).
// Returns the number of live rows up to the end of the share.
template <class Live, class Row>
__device__ __forceinline__ int pack_rows(int k0, int k1, int before, int H, const uint16_t* __restrict__ src,
                                         uint16_t* __restrict__ dst, Live live_of_row, Row row) {
  __shared__ int wsum[kPackThreads / 32];
  __shared__ int list[kPackThreads];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int vpr = H / 8;   // 16-byte vectors per row
  for (int base = k0; base < k1; base += kPackThreads) {
    const int k = base + threadIdx.x;
    const bool live = k < k1 && live_of_row(k);
    const unsigned m = __ballot_sync(0xffffffffu, live);
    __syncthreads();
    if (lane == 0) wsum[w] = __popc(m);
    __syncthreads();
    int pre = 0, cnt = 0;
#pragma unroll
    for (int i = 0; i < kPackThreads / 32; ++i) {
      pre += i < w ? wsum[i] : 0;
      cnt += wsum[i];
    }
    const int j = pre + __popc(m & ((1u << lane) - 1u));
    if (live) list[j] = k;
    if (k < k1) row(k, live, before + j);
    __syncthreads();
    if (src != nullptr) {
#pragma unroll 4
      for (int i = threadIdx.x; i < cnt * vpr; i += kPackThreads) {
        const int q = i / vpr, v = i - q * vpr;
        reinterpret_cast<uint4*>(dst + static_cast<int64_t>(before + q) * H)[v] =
            reinterpret_cast<const uint4*>(src + static_cast<int64_t>(list[q]) * H)[v];
      }
    }
    before += cnt;
  }
  return before;
}

// The active rows (mask != 0) packed: maps, and with `hidden` their hidden rows,
// tokens, behaviour log-probs and advantages.  (Rows past the last one stay as they
// are: the forward's products are independent by row.)  Also the call's zeroing:
// the outputs of masked rows and the backward's counters, which separate memsets
// cost a launch each.
__global__ void __launch_bounds__(kPackThreads) pack_kernel(
    const uint8_t* __restrict__ mask, int T, int H, const uint16_t* __restrict__ hidden,
    const int32_t* __restrict__ tokens, const float* __restrict__ b, const float* __restrict__ adv, int tok_shift,
    int32_t* __restrict__ row_map, int32_t* __restrict__ pos, int32_t* __restrict__ counts,
    uint16_t* __restrict__ h_p, int32_t* __restrict__ tok_p, float* __restrict__ b_p, float* __restrict__ adv_p,
    ZeroRows z, uint32_t* __restrict__ ctl, int ctl_words) {
  for (int i = blockIdx.x * kPackThreads + threadIdx.x; i < ctl_words; i += gridDim.x * kPackThreads) ctl[i] = 0u;
  const int share = (T + gridDim.x - 1) / gridDim.x;
  const int64_t first = static_cast<int64_t>(blockIdx.x) * share;
  if (first >= T) return;
  const int t0 = static_cast<int>(first), t1 = min(T, t0 + share);
  const int before = mask == nullptr ? t0 : count_bytes(mask, t0);
  const int total = pack_rows(
      t0, t1, before, H, hidden, h_p, [&](int t) { return mask == nullptr || mask[t] != 0; },
      [&](int t, bool live, int k) {
        pos[t] = live ? k : -1;
        if (live) {
          row_map[k] = t;
          if (tokens) tok_p[k] = tokens[t] - tok_shift;
          if (b) b_p[k] = b[t];
          if (adv) adv_p[k] = adv[t];
        } else {
#pragma unroll
          for (int i = 0; i < ZeroRows::kMax; ++i)
            if (z.out[i]) z.out[i][t] = 0.f;
        }
      });
  if (t1 == T && threadIdx.x == 0) {
    counts[0] = total;
    counts[1] = 0;
    counts[2] = 0;
    counts[4] = 0;
  }
}

// sums over a warp in a fixed tree
template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Eq. 2 terms of one active row (Sec. 4.5: ratio against the behaviour
// log-prob, PPO clipped surrogate with asymmetric bounds, m c / D).
struct RowLoss {
  float tl, coef, ratio;
  int clip_lo_hit, clip_hi_hit;
  double alr;
};
__device__ __forceinline__ RowLoss surrogate_row(float logp, float b, float A, float clip_lo, float clip_hi,
                                                 double D) {
  RowLoss r;
  r.ratio = expf(logp - b);
  const float lo = 1.0f - clip_lo, hi = 1.0f + clip_hi;
  const bool clipped = (A > 0.f && r.ratio > hi) || (A < 0.f && r.ratio < lo);
  const float rc = fminf(fmaxf(r.ratio, lo), hi);
  r.tl = clipped ? -(rc * A) : -(r.ratio * A);
  const float c = clipped ? 0.f : r.ratio * A;
  r.coef = (D > 0.0) ? static_cast<float>(static_cast<double>(c) / D) : 0.f;
  r.clip_lo_hit = (clipped && A < 0.f) ? 1 : 0;
  r.clip_hi_hit = (clipped && A > 0.f) ? 1 : 0;
  r.alr = fabs(static_cast<double>(logp) - static_cast<double>(b));
  return r;
}

// partial sums of a warp's 32 packed rows (loss, ratio, entropy, max |log ratio|,
// clip counts, KL, rejections): red[8 * row tile ..]
__device__ void warp_partials(bool act, const RowLoss& rl, float ent, float kl, int rejected,
                              double* __restrict__ r) {
  const double s_loss = warp_sum<double>(act ? (double)rl.tl : 0.0);
  const double s_ratio = warp_sum<double>(act ? (double)rl.ratio : 0.0);
  const double s_ent = warp_sum<double>(act ? (double)ent : 0.0);
  const double m_alr = warp_max(act ? rl.alr : 0.0);
  const int c_lo = __reduce_add_sync(0xffffffffu, act ? rl.clip_lo_hit : 0);
  const int c_hi = __reduce_add_sync(0xffffffffu, act ? rl.clip_hi_hit : 0);
  const double s_kl = warp_sum<double>(act ? (double)kl : 0.0);
  const int c_rej = __reduce_add_sync(0xffffffffu, rejected);
  if ((threadIdx.x & 31) == 0) {
    r[0] = s_loss;
    r[1] = s_ratio;
    r[2] = s_ent;
    r[3] = m_alr;
    r[4] = static_cast<double>(c_lo);
    r[5] = static_cast<double>(c_hi);
    r[6] = s_kl;
    r[7] = static_cast<double>(c_rej);
  }
}

// One block per kRedRows packed rows (merge_row_parts' threads): merge the per-split
// online softmax partials of each row into lse, logp and entropy; in loss mode also
// the ratio, the clipped surrogate (Sec. 4.5, PPO form), the Eq. 2 coefficient
// m c / D and the rows' partial sums.
template <int kGroups>
__global__ void __launch_bounds__(kRedRows * kGroups) merge_kernel(
    int loss_mode, int Tcap, int V, int n_parts, double denom, float clip_lo, float clip_hi,
    const int32_t* __restrict__ counts, const int32_t* __restrict__ row_map, const int32_t* __restrict__ tok_p,
    const float* __restrict__ b_p, const float* __restrict__ adv_p, const float4* __restrict__ part,
    const float* __restrict__ zx, float* __restrict__ lse_o, float* __restrict__ coef_o,
    double* __restrict__ red, float* __restrict__ logp_out, float* __restrict__ ent_out,
    float* __restrict__ tokloss_out, float* __restrict__ lp_p,
    float* __restrict__ ent_p, unsigned* err) {
  const int n = counts[0];
  if ((int)blockIdx.x * kRedRows >= n) return;
  const int k = blockIdx.x * kRedRows + threadIdx.x % kRedRows;
  const bool act = k < n;
  const RowStats st = merge_row_parts<kGroups>(part, Tcap, n_parts, k, act);
  if (threadIdx.x >= kRedRows) return;
  const double D = denom > 0.0 ? denom : static_cast<double>(n);
  float logp = 0.f, ent = 0.f;
  RowLoss rl{0.f, 0.f, 0.f, 0, 0, 0.0};
  if (act) {
    const float logS = logf(st.S);
    const float lse = st.M + logS;
    const int x = tok_p[k];
    if (x < 0 || x >= V) atomicOr(err, kDevErrTokenRange);
    logp = zx[k] - lse;
    ent = logS - st.Q / st.S;
    lse_o[k] = lse;
    if (loss_mode) rl = surrogate_row(logp, b_p[k], adv_p[k], clip_lo, clip_hi, D);
    const int t = row_map[k];
    if (logp_out) logp_out[t] = logp;
    if (ent_out) ent_out[t] = ent;
    if (tokloss_out) tokloss_out[t] = rl.tl;
    if (lp_p) lp_p[k] = logp;
    if (ent_p) ent_p[k] = ent;
  }
  if (!loss_mode) return;
  if (act) coef_o[k] = rl.coef;
  warp_partials(act, rl, ent, 0.f, 0, red + (int64_t)blockIdx.x * kRedSlots);
}

// ---------------------------------------------------------------------------
// Vocabulary-parallel pieces: the LM head split into vocabulary shards (one per
// tensor-parallel rank).  Each shard reduces its own columns to per-row
// statistics; the statistics of all shards, exchanged by the caller, merge into
// the row's lse, logp and entropy exactly as the forward's own vocab splits do.
// ---------------------------------------------------------------------------

// Statistics of one shard per original row: the forward's split partials
// combined in split order into (M, S, Q, z_x): M the shard's max logit, S =
// sum exp(z - M), Q = sum exp(z - M) (z - M), z_x the target logit if the
// target lies in the shard (tok_p holds the shard-local token) and -inf
// otherwise.  Masked rows get the empty statistics (-inf, 0, 0, -inf).
template <int kGroups>
__global__ void __launch_bounds__(kRedRows * kGroups) vp_local_kernel(
    int T, int Tcap, int V_s, int n_parts, const int32_t* __restrict__ pos, const int32_t* __restrict__ tok_p,
    const float4* __restrict__ part, const float* __restrict__ zx, float4* __restrict__ out) {
  const int t = blockIdx.x * kRedRows + threadIdx.x % kRedRows;
  const int k = t < T ? pos[t] : -1;
  const RowStats st = merge_row_parts<kGroups>(part, Tcap, n_parts, k, k >= 0);
  if (threadIdx.x >= kRedRows || t >= T) return;
  if (k < 0) {
    out[t] = make_float4(-INFINITY, 0.f, 0.f, -INFINITY);
    return;
  }
  const int xl = tok_p[k];
  out[t] = make_float4(st.M, st.S, st.Q, (xl >= 0 && xl < V_s) ? zx[k] : -INFINITY);
}

// One block of 128 threads per packed tile of active rows: merge the shards'
// statistics of each row (parts [n_shards, T], shard order fixed) into lse,
// logp and entropy, then the Eq. 2 terms as merge_kernel does.  A row whose
// target lies in no shard raises the token-range flag.  Per-row outputs go to
// the original row order (lse and m c / D for the shards' backward).
__global__ void __launch_bounds__(128) vp_merge_kernel(
    int T, int n_shards, double denom, float clip_lo, float clip_hi, const int32_t* __restrict__ counts,
    const int32_t* __restrict__ row_map, const float4* __restrict__ parts, const float* __restrict__ b,
    const float* __restrict__ adv, float* __restrict__ coef_p, double* __restrict__ red, float* __restrict__ lse_out, float* __restrict__ coef_out,
    float* __restrict__ logp_out, float* __restrict__ ent_out, float* __restrict__ tokloss_out, unsigned* err) {
  const int n = counts[0];
  const int n_tiles = (n + kTileM - 1) / kTileM;
  if ((int)blockIdx.x >= n_tiles) return;
  const int k = blockIdx.x * kTileM + threadIdx.x;
  const bool act = k < n;
  const double D = denom > 0.0 ? denom : static_cast<double>(n);
  float ent = 0.f;
  RowLoss rl{0.f, 0.f, 0.f, 0, 0, 0.0};
  if (act) {
    const int t = row_map[k];
    float M = -INFINITY, zxv = -INFINITY;
    for (int s = 0; s < n_shards; ++s) {
      const float4 p = parts[(int64_t)s * T + t];
      M = fmaxf(M, p.x);
      zxv = fmaxf(zxv, p.w);
    }
    float S = 0.f, Q = 0.f;
    for (int s = 0; s < n_shards; ++s) {
      const float4 p = parts[(int64_t)s * T + t];
      if (p.y != 0.f) {   // 0: no columns.  A NaN passes
        const float d = p.x - M;
        const float f = ex2_approx(d * kLog2e);
        S += f * p.y;
        Q += f * (p.z + d * p.y);
      }
    }
    if (zxv == -INFINITY) atomicOr(err, kDevErrTokenRange);
    const float logS = logf(S);
    const float lse = M + logS;
    const float logp = zxv == -INFINITY ? 0.f : zxv - lse;
    ent = logS - Q / S;
    rl = surrogate_row(logp, b[t], adv[t], clip_lo, clip_hi, D);
    lse_out[t] = lse;
    coef_out[t] = rl.coef;
    if (logp_out) logp_out[t] = logp;
    if (ent_out) ent_out[t] = ent;
    if (tokloss_out) tokloss_out[t] = rl.tl;
  }
  if (act) coef_p[k] = rl.coef;
  if (k / kRedRows * kRedRows < n) warp_partials(act, rl, ent, 0.f, 0, red + (int64_t)(k / kRedRows) * kRedSlots);
}

// one shard's dhidden contribution in the original row order, fp32: the
// accumulator row of t's backward row, 0 for rows without a gradient
__global__ void vp_dh_out_kernel(const float* __restrict__ dh32, const int32_t* __restrict__ live_of, int T, int H,
                                 float* __restrict__ out) {
  const int vpr = H / 4;
  const int64_t total = (int64_t)T * vpr;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int t = (int)(i / vpr), v = (int)(i - (int64_t)t * vpr);
    const int j = live_of[t];
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
    if (j >= 0) o = reinterpret_cast<const float4*>(dh32 + (int64_t)j * H)[v];
    reinterpret_cast<float4*>(out + (int64_t)t * H)[v] = o;
  }
}

// ---------------------------------------------------------------------------
// Extended objective (Sec. 4.5: KL control, rejection rules).
// ---------------------------------------------------------------------------

// Sequence gate.  Thread i checks that the ids do not decrease at token i; warp
// w owns packed rows [32 w, 32 w + 32) and handles every sequence that starts
// there: it walks the sequence 32 packed rows at a time (packing keeps the
// original order, so a sequence is a run of packed rows), sums logp - b in
// fp64 with a fixed shuffle tree, and writes the gate weight of every row.
// Reject when exp(mean) lies outside [lo, hi].
__global__ void __launch_bounds__(256) seq_gate_kernel(int T, const int32_t* __restrict__ seq,
                                                       const int32_t* __restrict__ counts,
                                                       const int32_t* __restrict__ row_map,
                                                       const float* __restrict__ lp_p, const float* __restrict__ b_p,
                                                       double lo, double hi, uint8_t* __restrict__ gate_p,
                                                       int32_t* __restrict__ n_rej, unsigned* err) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  if (i < T && i > 0 && seq[i] < seq[i - 1]) atomicOr(err, kDevErrUnsortedGroups);
  const int n = counts[0];
  const int base = i - lane;
  if (base >= n) return;   // whole warp leaves together
  const int k = base + lane;
  const int sid = (k < n) ? seq[row_map[k]] : 0;
  const bool start = (k < n) && (k == 0 || seq[row_map[k - 1]] != sid);
  unsigned starts = __ballot_sync(0xffffffffu, start);
  while (starts) {
    const int s0 = base + __ffs(starts) - 1;
    starts &= starts - 1;
    const int sid0 = __shfl_sync(0xffffffffu, sid, s0 - base);
    double acc = 0.0;
    int len = 0;
    for (int w0 = s0;; w0 += 32) {
      const int kk = w0 + lane;
      const bool in = kk < n && seq[row_map[kk]] == sid0;
      const unsigned m = __ballot_sync(0xffffffffu, in);
      const int run = (m == 0xffffffffu) ? 32 : __ffs(~m) - 1;   // leading rows of this sequence
      double v = (lane < run) ? static_cast<double>(lp_p[kk]) - static_cast<double>(b_p[kk]) : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      acc += v;
      len += run;
      if (run < 32) break;
    }
    const double g = exp(acc / static_cast<double>(len));
    const uint8_t keep = (g < lo || g > hi) ? 0 : 1;
    for (int j = s0 + lane; j < s0 + len; j += 32) gate_p[j] = keep;
    if (lane == 0 && !keep) atomicAdd(n_rej, 1);
  }
}

// One block of 128 threads per packed tile: the per-token loss of the extended
// objective and the two backward coefficients
//   coef  = m w (c + kl_coef (e^r - 1)) / D      on (p - onehot)
//   ecoef = m w entropy_coef / D                 on p (z - mu),  mu = lse - H
__global__ void __launch_bounds__(128) loss_rows_ex_kernel(
    int Tcap, double denom, float clip_lo, float clip_hi, LossEx ex, const int32_t* __restrict__ counts,
    const int32_t* __restrict__ row_map, const float* __restrict__ b_p, const float* __restrict__ adv_p,
    const float* __restrict__ lp_p, const float* __restrict__ ent_p, const float* __restrict__ lse,
    const uint8_t* __restrict__ gate_p, float* __restrict__ coef_o, float* __restrict__ ecoef_o,
    float* __restrict__ mu_o, double* __restrict__ red, float* __restrict__ tokloss_out) {
  const int n = counts[0];
  const int n_tiles = (n + kTileM - 1) / kTileM;
  if ((int)blockIdx.x >= n_tiles) return;
  const int k = blockIdx.x * kTileM + threadIdx.x;
  const bool act = k < n;
  const double D = denom > 0.0 ? denom : static_cast<double>(n);
  float ecoef = 0.f, mu = 0.f, ent = 0.f, kl = 0.f;
  int rejected = 0;
  RowLoss rl{0.f, 0.f, 0.f, 0, 0, 0.0};
  if (act) {
    const float logp = lp_p[k], b = b_p[k], A = adv_p[k];
    ent = ent_p[k];
    const float ratio = expf(logp - b);
    rl.ratio = ratio;
    const float lo = 1.0f - clip_lo, hi = 1.0f + clip_hi;
    const bool clipped = (A > 0.f && ratio > hi) || (A < 0.f && ratio < lo);
    const float rc = fminf(fmaxf(ratio, lo), hi);
    const float l_pg = clipped ? -(rc * A) : -(ratio * A);
    const float c = clipped ? 0.f : ratio * A;
    float c_kl = 0.f;
    if (ex.kl_coef != 0.f) {
      const float r = ex.ref_logp[row_map[k]] - logp;
      const float em1 = expm1f(r);
      kl = em1 - r;             // e^r - r - 1 without cancellation near r = 0
      c_kl = ex.kl_coef * em1;
    }
    const bool keep = gate_p == nullptr || gate_p[k] != 0;
    if (keep) {
      rl.tl = l_pg + ex.kl_coef * kl - ex.entropy_coef * ent;
      rl.coef = (D > 0.0) ? static_cast<float>(static_cast<double>(c + c_kl) / D) : 0.f;
      ecoef = (D > 0.0) ? static_cast<float>(static_cast<double>(ex.entropy_coef) / D) : 0.f;
      rl.clip_lo_hit = (clipped && A < 0.f) ? 1 : 0;
      rl.clip_hi_hit = (clipped && A > 0.f) ? 1 : 0;
    } else {
      kl = 0.f;
      rejected = 1;
    }
    mu = lse[k] - ent;
    rl.alr = fabs(static_cast<double>(logp) - static_cast<double>(b));
    if (tokloss_out) tokloss_out[row_map[k]] = rl.tl;
  }
  if (k < Tcap) {
    coef_o[k] = rl.coef;
    ecoef_o[k] = ecoef;
    mu_o[k] = mu;
  }
  if (k / kRedRows * kRedRows < n) warp_partials(act, rl, ent, kl, rejected, red + (int64_t)(k / kRedRows) * kRedSlots);
}

struct StatsDev {
  double denom, loss, sum_ratio, sum_entropy, max_abs_log_ratio;
  long long n_active, n_clip_low, n_clip_high, n_grad_rows;
};
struct StatsExDev {
  StatsDev base;
  double sum_kl;
  long long n_tokens_rejected, n_seq_rejected;
};
constexpr int kFinSlots = 8;

// fixed-order reduction of the rows' partial sums, the loss scalar and the stats;
// by one block of kPackThreads threads, a warp to each slot
__device__ __forceinline__ void reduce_loss(int n, double denom, const int32_t* __restrict__ counts,
                                            const double* __restrict__ red, float* __restrict__ loss_out,
                                            StatsDev* __restrict__ stats, StatsExDev* __restrict__ stats_ex,
                                            unsigned* err) {
  static_assert(kFinSlots == kPackThreads / 32, "a warp to each slot");
  __shared__ double tot[kFinSlots];
  const int n_rt = (n + kRedRows - 1) / kRedRows, n_tiles = (n_rt + 3) / 4;
  const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
  // In the order in which these sums have always been taken, so that the loss and
  // the stats stay the same bits: four sets of rows to a tile of 128, tile i to
  // column i % 1024, the columns 32 at a time by a shuffle tree (here 32 kBatch at
  // a time), and those 32 totals by another.
  auto join = [&](double x, double y) { return q == 3 ? fmax(x, y) : x + y; };
  auto part = [&](int r) { return r < n_rt ? red[(int64_t)r * kRedSlots + q] : 0.0; };
  constexpr int kBatch = 4;
  double a = 0.0;
  for (int w = 0; w < 32 && 32 * w < n_tiles; w += kBatch) {
    double x[kBatch] = {};
    for (int base = 32 * w + lane; base < n_tiles; base += 1024) {
#pragma unroll
      for (int i = 0; i < kBatch; ++i) {
        const int r = 4 * (base + 32 * i);
        x[i] = join(x[i], join(join(part(r), part(r + 1)), join(part(r + 2), part(r + 3))));
      }
    }
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
      const double total = q == 3 ? warp_max(x[i]) : warp_sum(x[i]);
      if (lane == w + i) a = total;
    }
  }
  a = (q == 3) ? warp_max(a) : warp_sum(a);
  if (lane == 0) tot[q] = a;
  __syncthreads();
  if (threadIdx.x != 0) return;
  const double D = denom > 0.0 ? denom : static_cast<double>(n);
  if (!(D > 0.0)) atomicOr(err, kDevErrZeroDenom);
  const double loss = D > 0.0 ? tot[0] / D : 0.0;
  if (loss_out) *loss_out = static_cast<float>(loss);
  StatsDev* st[2] = {stats, stats_ex ? &stats_ex->base : nullptr};
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    if (!st[i]) continue;
    st[i]->denom = D;
    st[i]->loss = loss;
    st[i]->sum_ratio = tot[1];
    st[i]->sum_entropy = tot[2];
    st[i]->max_abs_log_ratio = tot[3];
    st[i]->n_active = n;
    st[i]->n_clip_low = static_cast<long long>(tot[4]);
    st[i]->n_clip_high = static_cast<long long>(tot[5]);
  }
  if (stats_ex) {
    stats_ex->sum_kl = tot[6];
    stats_ex->n_tokens_rejected = static_cast<long long>(tot[7]);
    stats_ex->n_seq_rejected = counts[2];
  }
}

// Packs the rows whose gradient coefficient is nonzero (coef, or ecoef with an
// entropy bonus), the rows the backward processes, into whole tiles of 128: with
// `src` their hidden rows, tokens, lse, m c / D and, with an entropy bonus, its
// coefficient and mu; rows in [n_live, round_up(n_live, pad)) are zeroed, which the
// backward's products read with them (64 over chunks, 128 else; the last block does
// it alone: 127 rows of H = 5120 took 10 us).  n_rows < 0: rows are the packed
// active ones and the first block also reduces the loss.  Writes counts[1] (tiles)
// and counts[3] (rows), and for a shard's backward zeroes the chunk counters.
__global__ void __launch_bounds__(kPackThreads) finish_kernel(
    int n_rows, int pad, double denom, int32_t* __restrict__ counts, int32_t* __restrict__ tile_list,
    const double* __restrict__ red, float* __restrict__ loss_out, StatsDev* __restrict__ stats,
    StatsExDev* __restrict__ stats_ex, int H, int tok_shift, const uint16_t* __restrict__ src,
    const int32_t* __restrict__ tok, const float* __restrict__ lse, const float* __restrict__ coef,
    const float* __restrict__ ecoef, const float* __restrict__ mu, int32_t* __restrict__ live_of,
    uint16_t* __restrict__ h_l, int32_t* __restrict__ tok_l, float* __restrict__ lse_l, float* __restrict__ coef_l,
    float* __restrict__ ecoef_l, float* __restrict__ mu_l, uint32_t* __restrict__ ctl, int ctl_words, unsigned* err) {
  for (int i = blockIdx.x * kPackThreads + threadIdx.x; i < ctl_words; i += gridDim.x * kPackThreads) ctl[i] = 0u;
  const int n = n_rows < 0 ? counts[0] : n_rows;
  if (n_rows < 0 && blockIdx.x == 0) reduce_loss(n, denom, counts, red, loss_out, stats, stats_ex, err);
  const int share = (n + gridDim.x - 1) / gridDim.x;
  const int64_t first = static_cast<int64_t>(blockIdx.x) * share;
  if (first >= n && !(n == 0 && blockIdx.x == 0)) return;
  const int k0 = static_cast<int>(first), k1 = min(n, k0 + share);
  auto live = [&](int k) { return coef[k] != 0.f || (ecoef != nullptr && ecoef[k] != 0.f); };
  int c = 0;
#pragma unroll 8
  for (int k = threadIdx.x; k < k0; k += kPackThreads) c += live(k) ? 1 : 0;
  const int total = pack_rows(k0, k1, block_sum(c), H, src, h_l, live, [&](int k, bool is_live, int j) {
    live_of[k] = is_live ? j : -1;
    if (is_live && src != nullptr) {
      tok_l[j] = tok[k] - tok_shift;
      lse_l[j] = lse[k];
      coef_l[j] = coef[k];
      if (ecoef) {
        ecoef_l[j] = ecoef[k];
        mu_l[j] = mu[k];
      }
    }
  });
  if (k1 != n) return;
  const int n_lt = (total + kTileM - 1) / kTileM;
  for (int b = threadIdx.x; b < n_lt; b += kPackThreads) tile_list[b] = b;
  if (threadIdx.x == 0) {
    counts[1] = n_lt;
    counts[3] = total;
    if (stats) stats->n_grad_rows = total;
    if (stats_ex) stats_ex->base.n_grad_rows = total;
  }
  if (src == nullptr) return;
  const int n_pad = (total + pad - 1) / pad * pad;
  for (int j = total + threadIdx.x; j < n_pad; j += kPackThreads) {
    tok_l[j] = 0;
    lse_l[j] = 0.f;
    coef_l[j] = 0.f;
    if (ecoef) {
      ecoef_l[j] = 0.f;
      mu_l[j] = 0.f;
    }
  }
  const int64_t v0 = static_cast<int64_t>(total) * (H / 8), v1 = static_cast<int64_t>(n_pad) * (H / 8);
#pragma unroll 4
  for (int64_t v = v0 + threadIdx.x; v < v1; v += kPackThreads) reinterpret_cast<uint4*>(h_l)[v] = make_uint4(0, 0, 0, 0);
}

// dhidden_out[t] = bf16(dh32[live_of[pos[t]]]) for rows with a gradient, 0 for
// masked rows and rows whose gradient coefficient is 0
__global__ void cast_dh_kernel(const float* __restrict__ dh32, const int32_t* __restrict__ pos,
                               const int32_t* __restrict__ live_of, int T, int H, uint16_t* __restrict__ out) {
  const int vpr = H / 8;
  const int64_t total = (int64_t)T * vpr;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int t = (int)(i / vpr), v = (int)(i - (int64_t)t * vpr);
    const int kp = pos[t];
    const int k = kp >= 0 ? live_of[kp] : -1;
    uint4 o = make_uint4(0, 0, 0, 0);
    if (k >= 0) {
      const float4* src = reinterpret_cast<const float4*>(dh32 + (int64_t)k * H) + 2 * v;
      const float4 a = src[0], c = src[1];
      o.x = pack_bf16x2(a.x, a.y);
      o.y = pack_bf16x2(a.z, a.w);
      o.z = pack_bf16x2(c.x, c.y);
      o.w = pack_bf16x2(c.z, c.w);
    }
    reinterpret_cast<uint4*>(out + (int64_t)t * H)[v] = o;
  }
}

}  // namespace

// words[0]: the call's abort word, words[1]: a counter nothing raises,
// words[2]: 1 if the wait returned true, 2 if it gave up
__global__ void wait_selftest_kernel(uint32_t* words, unsigned* err) {
  __shared__ int abort_sh;
  if (threadIdx.x == 0) {
    abort_sh = 0;
    volatile int* abort_flag = &abort_sh;
    words[2] = turn_wait(words + 1, 1u, abort_flag, words, err) ? 1u : 2u;
  }
}

cudaError_t launch_wait_selftest(uint32_t* words, unsigned* err, cudaStream_t s) {
  wait_selftest_kernel<<<1, 32, 0, s>>>(words, err);
  return cudaGetLastError();
}

cudaError_t launch_group_advantages(const float* rewards, const int32_t* gids, int n, double eps, float* out,
                                    unsigned* err, cudaStream_t s) {
  return launch_advantages(rewards, gids, n, kAdvGrpo, eps, out, err, s);
}

cudaError_t launch_advantages(const float* rewards, const int32_t* gids, int n, int estimator, double eps,
                              float* out, unsigned* err, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (estimator == kAdvReinforcePP) {
    // one warp over the whole batch; zero everything first so a batch of one gives 0
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(float) * n, s);
    if (e != cudaSuccess) return e;
    group_adv_kernel<<<1, 32, 0, s>>>(rewards, nullptr, n, eps, estimator, out, err);
    return cudaGetLastError();
  }
  const int threads = 256;
  const int blocks = (int)(((int64_t)n * 32 + threads - 1) / threads);
  group_adv_kernel<<<blocks, threads, 0, s>>>(rewards, gids, n, eps, estimator, out, err);
  return cudaGetLastError();
}

cudaError_t launch_broadcast(const float* adv, const int32_t* rot, int n_resp, int T, float* out, cudaStream_t s) {
  if (T <= 0) return cudaSuccess;
  const int blocks = min((T + 255) / 256, 4096);
  broadcast_kernel<<<blocks, 256, 0, s>>>(adv, rot, n_resp, T, out);
  return cudaGetLastError();
}

cudaError_t launch_mask_count(const uint8_t* mask, int64_t T, int64_t* out, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(int64_t), s);
  if (e != cudaSuccess || T <= 0) return e;
  const int64_t nb = (T / 16 + 255) / 256 + 1;
  const int blocks = (int)(nb < 1024 ? nb : 1024);
  mask_count_kernel<<<blocks, 256, 0, s>>>(mask, T, reinterpret_cast<unsigned long long*>(out));
  return cudaGetLastError();
}

cudaError_t launch_pack(const uint8_t* mask, int T, int H, const uint16_t* hidden, const int32_t* tokens, const float* b,
                        const float* adv, int tok_shift, const Workspace& ws, const ZeroRows& z, int64_t ctl_words,
                        int n_sm, cudaStream_t s) {
  pack_kernel<<<n_sm * 8, kPackThreads, 0, s>>>(mask, T, H, hidden, tokens, b, adv, tok_shift, ws.row_map, ws.pos_of_row,
                                                ws.counts, ws.h_p, ws.tok_p, ws.b_p, ws.adv_p, z, ws.ctl,
                                                static_cast<int>(ctl_words));
  return cudaGetLastError();
}

cudaError_t launch_merge(bool loss_mode, bool ordered, int Tcap, int V, int n_parts, double denom, float clip_lo, float clip_hi,
                         const Workspace& ws, float* logp_out, float* ent_out, float* tokloss_out, float* lp_p,
                         float* ent_p, unsigned* err, cudaStream_t s) {
  const int blocks = Tcap / kRedRows;
  if (blocks == 0) return cudaSuccess;
  const int groups = ordered ? 1 : merge_groups(n_parts);
  auto* k = groups == 1                  ? &merge_kernel<1>
            : groups == kMergeGroupsMany ? &merge_kernel<kMergeGroupsMany>
                                         : &merge_kernel<kMergeGroupsFew>;
  k<<<blocks, kRedRows * groups, 0, s>>>(loss_mode ? 1 : 0, Tcap, V, n_parts, denom, clip_lo, clip_hi, ws.counts,
                                         ws.row_map, ws.tok_p, ws.b_p, ws.adv_p, ws.part, ws.zx, ws.lse, ws.coef,
                                         ws.red, logp_out, ent_out, tokloss_out, lp_p, ent_p, err);
  return cudaGetLastError();
}

cudaError_t launch_seq_gate(int T, int Tcap, const LossEx& ex, const Workspace& ws, unsigned* err, cudaStream_t s) {
  const int blocks = (Tcap + 255) / 256;
  if (blocks == 0 || ex.seq == nullptr) return cudaSuccess;
  seq_gate_kernel<<<blocks, 256, 0, s>>>(T, ex.seq, ws.counts, ws.row_map, ws.lp_p, ws.b_p, ex.gate_lo, ex.gate_hi,
                                         ws.gate_p, ws.counts + 2, err);
  return cudaGetLastError();
}

cudaError_t launch_loss_rows_ex(int Tcap, double denom, float clip_lo, float clip_hi, const LossEx& ex,
                                const Workspace& ws, float* tokloss_out, cudaStream_t s) {
  const int blocks = Tcap / kTileM;
  if (blocks == 0) return cudaSuccess;
  loss_rows_ex_kernel<<<blocks, kTileM, 0, s>>>(Tcap, denom, clip_lo, clip_hi, ex, ws.counts, ws.row_map, ws.b_p,
                                                 ws.adv_p, ws.lp_p, ws.ent_p, ws.lse,
                                                 ex.seq ? ws.gate_p : nullptr, ws.coef, ws.ecoef, ws.mu,
                                                 ws.red, tokloss_out);
  return cudaGetLastError();
}

cudaError_t launch_finish(int H, int pad, bool with_ecoef, double denom, const Workspace& ws, float* loss_out,
                          void* stats_out, void* stats_ex_out, unsigned* err, int n_sm, cudaStream_t s) {
  finish_kernel<<<n_sm * 8, kPackThreads, 0, s>>>(
      -1, pad, denom, ws.counts, ws.tile_list, ws.red, loss_out, reinterpret_cast<StatsDev*>(stats_out),
      reinterpret_cast<StatsExDev*>(stats_ex_out), H, 0, pad > 0 ? ws.h_p : nullptr, ws.tok_p, ws.lse, ws.coef,
      with_ecoef ? ws.ecoef : nullptr, ws.mu, ws.live_of, ws.h_l, ws.tok_l, ws.lse_l, ws.coef_l, ws.ecoef_l, ws.mu_l,
      nullptr, 0, err);
  return cudaGetLastError();
}

cudaError_t launch_vp_pack(int T, int H, int pad, const uint16_t* hidden, const int32_t* tokens, const float* lse,
                           const float* coef, int tok_shift, const Workspace& ws, int64_t ctl_words, int n_sm,
                           cudaStream_t s) {
  finish_kernel<<<n_sm * 8, kPackThreads, 0, s>>>(T, pad, 0.0, ws.counts, ws.tile_list, nullptr, nullptr, nullptr, nullptr, H,
                                                  tok_shift, hidden, tokens, lse, coef, nullptr, nullptr, ws.live_of,
                                                  ws.h_l, ws.tok_l, ws.lse_l, ws.coef_l, ws.ecoef_l, ws.mu_l, ws.ctl,
                                                  static_cast<int>(ctl_words), nullptr);
  return cudaGetLastError();
}

cudaError_t launch_vp_local(int T, int Tcap, int V_s, int n_parts, const Workspace& ws, float4* out,
                            cudaStream_t s) {
  if (T <= 0) return cudaSuccess;
  const int groups = merge_groups(n_parts);
  auto* k = groups == kMergeGroupsMany ? &vp_local_kernel<kMergeGroupsMany> : &vp_local_kernel<kMergeGroupsFew>;
  k<<<(T + kRedRows - 1) / kRedRows, kRedRows * groups, 0, s>>>(T, Tcap, V_s, n_parts, ws.pos_of_row, ws.tok_p, ws.part,
                                                                ws.zx, out);
  return cudaGetLastError();
}

cudaError_t launch_vp_merge(int T, int Tcap, int n_shards, double denom, float clip_lo, float clip_hi,
                            const float4* parts, const float* b, const float* adv, const Workspace& ws,
                            float* lse_out, float* coef_out, float* logp_out, float* ent_out, float* tokloss_out,
                            unsigned* err, cudaStream_t s) {
  const int blocks = Tcap / kTileM;
  if (blocks == 0) return cudaSuccess;
  vp_merge_kernel<<<blocks, kTileM, 0, s>>>(T, n_shards, denom, clip_lo, clip_hi, ws.counts, ws.row_map, parts, b,
                                            adv, ws.coef, ws.red, lse_out, coef_out, logp_out,
                                            ent_out, tokloss_out, err);
  return cudaGetLastError();
}

cudaError_t launch_vp_dh_out(const Workspace& ws, int T, int H, float* out, int n_sm, cudaStream_t s) {
  if (T <= 0) return cudaSuccess;
  vp_dh_out_kernel<<<n_sm * 8, 256, 0, s>>>(ws.dh32, ws.live_of, T, H, out);
  return cudaGetLastError();
}

cudaError_t launch_cast_dh(const Workspace& ws, int T, int H, uint16_t* dh_out, int n_sm, cudaStream_t s) {
  if (T <= 0) return cudaSuccess;
  cast_dh_kernel<<<n_sm * 8, 256, 0, s>>>(ws.dh32, ws.pos_of_row, ws.live_of, T, H, dh_out);
  return cudaGetLastError();
}

}  // namespace molt
