// Forward pass of the LM head with a fused online log-softmax (Sec. 4.5: the
// actor's recomputed log-probabilities of the generated tokens, plus entropy).
//
// z = h W^T is never written to global memory.  Each work unit is one tile of
// 256 packed token rows times one contiguous split of the vocabulary.  For
// every 256-column vocab tile of the split, the tensor cores of a CTA pair
// accumulate the 256 x 256 fp32 logit tile in TMEM (128 rows in each CTA; K = H
// in 64-element steps fed by TMA), and the epilogue warps fold it into per-row
// running statistics:
//   m = running max, s = sum exp(z - m), q = sum exp(z - m) (z - m)
// and pick the target logit z[x].  The split's (m, s, q) go to a small workspace;
// a row-level merge kernel combines the splits into
//   lse = m + log s,  logp = z[x] - lse,  entropy = log s - q / s.
//
// What bounds it: the tensor cores under the board's power cap, so the bytes
// moved per product count as much as the time they take.  A pair loads 64 bytes
// of operands per clock and SM at full rate where a single CTA's 128 x 256 tile
// loads 96.  Units are taken 16 token tiles at a time, all of them on one vocab
// split before the next, so that W comes from HBM once per 4096 rows and the
// pairs in flight read the same W tiles.  Measured in a loop at the power cap
// (T = 32768, H = 4096, V = 151936): 22.98 ms, 1.78 PFLOP/s, against 25.44 ms for
// 128 x 256 tiles on single CTAs; with groups of 8, 32 and 76 token tiles 23.20,
// 24.73 and 27.04 ms.  T = 1031: 0.90 against 1.72 ms (W came from HBM once per
// 128 rows); T = 5003, H = 320, V = 50257: 0.162 against 0.174 ms.
//
// Roles per CTA (384 threads; clusters of two CTAs, persistent, units claimed
// from a counter):
//   warps 0, 11  TMA producers: h tile [128 x 64] and W tile [128 x 64] of this
//                CTA per stage, 128-byte swizzle, 7-stage ring
//   warp 1       MMA issuer (even CTA): tcgen05.mma cta_group::2 kind::f16, M=256
//                N=256 K=16, double-buffered accumulators (2 x 256 TMEM columns)
//   warps 2-9    epilogue, two per TMEM lane quarter: each thread owns one TMEM
//                lane = one token row, and 128 of the 256 columns
//   warp 10      even CTA: claims units and hands them to every role of both CTAs
#include <atomic>
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

#include "molt_internal.cuh"
#include "ptx.cuh"

namespace molt {
namespace {

constexpr int kStages = 7;
constexpr int kHalf = 128 * kBK * 2;             // one operand's half of a stage, 16 KB
constexpr int kStageBytes = 2 * kHalf;           // 32 KB per CTA
constexpr int kEpiWarps = 8;
constexpr int kThreads = 128 + 32 * kEpiWarps;
constexpr int kSmemBytes = kStages * kStageBytes + 1024;
constexpr int kSlots = 2;                        // units handed from the claiming warp to the other roles
constexpr int kGroup = 16;                       // token tiles that share a pass over the vocabulary
constexpr uint32_t kIdesc = idesc_bf16_f32(256, 256, false, false);
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

template <bool kOrdered>
__device__ __forceinline__ void split_range(int s, int S, int n_vt, int& vt0, int& vt1) {
  if constexpr (kOrdered) {
    vt0 = static_cast<int>(static_cast<int64_t>(s) * n_vt / S);
    vt1 = static_cast<int>(static_cast<int64_t>(s + 1) * n_vt / S);
  } else {
    const int per = n_vt / S, more = n_vt - per * S;   // the first `more` splits take one tile more
    vt0 = s * per + min(s, more);
    vt1 = vt0 + per + (s < more ? 1 : 0);
  }
}

// Running statistics of one row.  q2 is in log2 units: q2 = sum e (z - m) log2(e).
// s is summed with its rounding carried along in c (Kahan), so that log s hardly
// depends on how the columns are split; in the ordered sums it is not (c stays 0).
struct Stats {
  float m = -INFINITY, s = 0.f, c = 0.f, q2 = 0.f;
  __device__ __forceinline__ void raise(float cmax) {
    if (cmax > m) {
      if (m != -INFINITY) {
        const float d2 = (m - cmax) * kLog2e;
        const float sc = ex2_approx(d2);
        q2 = sc * fmaf(d2, s, q2);
        s *= sc;
        c *= sc;
      }
      m = cmax;
    }
  }
  template <bool kOrdered>
  __device__ __forceinline__ void add(float ds, float dq) {
    if constexpr (kOrdered) {
      s += ds;
    } else {
      const float y = ds - c, t = s + y;
      c = (t - s) - y;
      s = t;
    }
    q2 += dq;
  }
};

// fold 32 logits (all columns valid) into the row's statistics
template <bool kOrdered>
__device__ __forceinline__ void fold_full(const float (&v)[32], Stats& r) {
  float cm[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
  for (int j = 4; j < 32; ++j) cm[j & 3] = fmaxf(cm[j & 3], v[j]);
  r.raise(fmaxf(fmaxf(cm[0], cm[1]), fmaxf(cm[2], cm[3])));
  const float mL = r.m * kLog2e;
  constexpr int kSums = kOrdered ? 2 : 4;
  float s[4] = {0.f, 0.f, 0.f, 0.f}, q[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const float y = fmaf(v[j], kLog2e, -mL);
    const float e = ex2_approx(y);
    s[j % kSums] += e;
    q[j % kSums] = fmaf(e, y, q[j % kSums]);
  }
  if constexpr (kOrdered)
    r.add<true>(s[0] + s[1], q[0] + q[1]);
  else
    r.add<false>((s[0] + s[1]) + (s[2] + s[3]), (q[0] + q[1]) + (q[2] + q[3]));
}

// same for a chunk where only the first `nv` (1..31) columns are valid
template <bool kOrdered>
__device__ __forceinline__ void fold_partial(const float (&v)[32], int nv, Stats& r) {
  float cmax = v[0];
#pragma unroll
  for (int j = 1; j < 32; ++j)
    if (j < nv) cmax = fmaxf(cmax, v[j]);
  r.raise(cmax);
  const float mL = r.m * kLog2e;
  float s = kOrdered ? r.s : 0.f, q = kOrdered ? r.q2 : 0.f;
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    if (j < nv) {
      const float y = fmaf(v[j], kLog2e, -mL);
      const float e = ex2_approx(y);
      s += e;
      q = fmaf(e, y, q);
    }
  }
  if constexpr (kOrdered) {
    r.s = s;
    r.q2 = q;
  } else {
    r.add<false>(s, q);
  }
}

// unit u of the list: 256-row token tile and vocab split
__device__ __forceinline__ void unit_of(int u, int n_mt, int S, int& mt, int& s) {
  const int g = u / (kGroup * S);
  const int r = u - g * kGroup * S;
  const int g_mt = min(kGroup, n_mt - g * kGroup);
  s = r / g_mt;
  mt = g * kGroup + (r - s * g_mt);
}

// kOrdered: the sums of the reproducible loss call.  Its results stay the same bits
// from one version of the library to the next, so a row's columns are summed one
// after the other by one thread (the four warps of the lower column half take all
// 256 columns, the others none), uncompensated, in the splits of ordered_splits
// (api.cu) and merged in their order.  T = 16384, V = 65536: 0.49 against
// 0.38 ms at H = 256, 0.73 and 0.62 at H = 512, 1.33 and 1.21 at H = 1024; at H = 4096
// the products hide it (4.94 and 4.93).
template <bool kOrdered>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    lmhead_fwd_kernel(const __grid_constant__ CUtensorMap tm_h, const __grid_constant__ CUtensorMap tm_w,
                      const FwdArgs a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kStages];    // even CTA: both CTAs' bytes land here
  __shared__ __align__(8) uint64_t empty_bar[kStages];   // both CTAs
  __shared__ __align__(8) uint64_t accf_bar[2];          // both CTAs: accumulator full
  __shared__ __align__(8) uint64_t acce_bar[2];          // even CTA: one arrival per reading warp of the pair
  __shared__ __align__(8) uint64_t ufull_bar[kSlots];    // both CTAs: unit index written
  __shared__ __align__(8) uint64_t uempty_bar[kSlots];   // even CTA: every reader of both CTAs has it
  __shared__ __align__(8) uint64_t hfull_bar[4], hempty_bar[4];   // the upper column half's (m, s, q) written / read
  __shared__ float half_sh[4][3][32];
  __shared__ __align__(8) uint64_t done_bar;
  __shared__ int unit_sh[kSlots];
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_sh;

  const uint32_t smem0 = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  volatile int* abort_flag = &abort_sh;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&accf_bar[b]), 1);
      mbar_init(smem_u32(&acce_bar[b]), kOrdered ? kEpiWarps : 2 * kEpiWarps);
    }
    for (int s = 0; s < kSlots; ++s) {
      mbar_init(smem_u32(&ufull_bar[s]), 1);
      // readers: the MMA issuer, four producer warps, every epilogue warp
      mbar_init(smem_u32(&uempty_bar[s]), 5 + 2 * kEpiWarps);
    }
    for (int i = 0; i < 4; ++i) {
      mbar_init(smem_u32(&hfull_bar[i]), 1);
      mbar_init(smem_u32(&hempty_bar[i]), 1);
    }
    mbar_init(smem_u32(&done_bar), 1);
    abort_sh = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(&tmem_base_sh), 512);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();   // both CTAs' barriers exist before any remote arrival
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_sh;

  const int n_rows = a.counts[0];
  const int n_mt = (n_rows + 255) / 256;
  const int S = a.n_split;
  const int n_units = n_mt * S;
  const int kblocks = a.H / kBK;

  // the next unit for a reader of the slot ring (called by one lane); -1 ends
  // the walk, also after a wait that ran out
  const uint32_t uempty_lead0 = mapa_shared(smem_u32(&uempty_bar[0]), 0);
  auto next_unit = [&](uint32_t i) -> int {
    const uint32_t s = i % kSlots;
    if (!mbar_wait_cluster(smem_u32(&ufull_bar[s]), (i / kSlots) & 1u, abort_flag, a.err)) return -1;
    const int u = *reinterpret_cast<volatile int*>(&unit_sh[s]);
    if (u >= -1) mbar_arrive_cluster_relaxed(uempty_lead0 + s * 8);   // always; orders the arrival after the read
    return u;
  };

  if (warp == 0 || warp == 3 + kEpiWarps) {
    if (lane == 0) {
      const bool is_a = warp == 0;
      const CUtensorMap* map = is_a ? &tm_h : &tm_w;
      prefetch_tmap(map);
      const uint32_t full_lead0 = mapa_shared(smem_u32(&full_bar[0]), 0);
      const uint32_t dst0 = smem0 + (is_a ? 0 : kHalf);
      uint32_t st = 0, ph = 0, n_it = 0;
      bool ok = true;
      int u = next_unit(0);
      for (uint32_t ui = 0; u >= 0 && ok; ++ui) {
        int mt, s, vt0, vt1;
        unit_of(u, n_mt, S, mt, s);
        split_range<kOrdered>(s, S, a.n_vtiles, vt0, vt1);
        for (int vt = vt0; vt < vt1 && ok; ++vt) {
          const int y = (is_a ? mt : vt) * 256 + static_cast<int>(rank) * 128;
          for (int kb = 0; kb < kblocks; ++kb) {
            if (!(ok = mbar_wait(smem_u32(&empty_bar[st]), ph ^ 1u, abort_flag, a.err))) break;
            if (is_a && leader) mbar_arrive_expect_tx(smem_u32(&full_bar[st]), 2 * kStageBytes);
            tma_load_2d_pair(dst0 + st * kStageBytes, map, full_lead0 + st * 8, kb * kBK, y);
            ++n_it;
            if (++st == kStages) {
              st = 0;
              ph ^= 1u;
            }
          }
        }
        if (ok) u = next_unit(ui + 1);
      }
      if (leader && is_a) {
        // every copy into both CTAs completes on these barriers: wait for the
        // last issued stages before the pair may exit
        const uint32_t first = n_it > (uint32_t)kStages ? n_it - kStages : 0u;
        for (uint32_t j = first; j < n_it; ++j)
          mbar_wait_drain(smem_u32(&full_bar[j % kStages]), (j / kStages) & 1u, a.err);
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && leader) {
      uint32_t st = 0, ph = 0, acc_it = 0;
      bool ok = true;
      const uint64_t ad0 = sdesc_sw128(smem0, 16, 1024), bd0 = sdesc_sw128(smem0 + kHalf, 16, 1024);
      int u = next_unit(0);
      for (uint32_t ui = 0; u >= 0 && ok; ++ui) {
        int mt, s, vt0, vt1;
        unit_of(u, n_mt, S, mt, s);
        split_range<kOrdered>(s, S, a.n_vtiles, vt0, vt1);
        for (int vt = vt0; vt < vt1 && ok; ++vt) {
          const uint32_t buf = acc_it & 1u;
          if (!(ok = mbar_wait(smem_u32(&acce_bar[buf]), ((acc_it >> 1) & 1u) ^ 1u, abort_flag, a.err))) break;
          tc_fence_after();
          const uint32_t d = tmem_base + buf * 256;
          auto issue = [&](uint32_t stage, uint32_t accumulate) {
            umma4_bf16_pair(d, ad0 + stage * (kStageBytes >> 4), bd0 + stage * (kStageBytes >> 4), 2u, 2u, kIdesc,
                            accumulate);
            umma_commit_pair_mc(smem_u32(&empty_bar[stage]), 3);
          };
          // two stages per turn: one wait of the issuing thread for eight products
          for (int kb = 0; kb < kblocks; kb += 2) {
            const bool two = kb + 1 < kblocks;
            const uint32_t st0 = st;
            if (!(ok = mbar_wait(smem_u32(&full_bar[st]), ph, abort_flag, a.err))) break;
            if (++st == kStages) {
              st = 0;
              ph ^= 1u;
            }
            if (two && !(ok = mbar_wait(smem_u32(&full_bar[st]), ph, abort_flag, a.err))) break;
            tc_fence_after();
            issue(st0, kb != 0 ? 1u : 0u);
            if (two) {
              issue(st, 1u);
              if (++st == kStages) {
                st = 0;
                ph ^= 1u;
              }
            }
          }
          if (!ok) break;
          umma_commit_pair_mc(smem_u32(&accf_bar[buf]), 3);
          ++acc_it;
        }
        if (ok) u = next_unit(ui + 1);
      }
      umma_commit_pair_mc(smem_u32(&done_bar), 1);
      mbar_wait_drain(smem_u32(&done_bar), 0, a.err);
    }
  } else if (warp == 2 + kEpiWarps) {
    if (lane == 0 && leader) {
      const uint32_t unit_peer0 = mapa_shared(smem_u32(&unit_sh[0]), 1);
      const uint32_t ufull_peer0 = mapa_shared(smem_u32(&ufull_bar[0]), 1);
      for (uint32_t i = 0;; ++i) {
        // claimed ahead of the slot: the counter's round trip is over when it frees
        int u = atomicAdd(a.next_unit, 1);
        if (u >= n_units) u = -1;
        const uint32_t s = i % kSlots;
        if (!mbar_wait_cluster(smem_u32(&uempty_bar[s]), ((i / kSlots) & 1u) ^ 1u, abort_flag, a.err)) break;
        *reinterpret_cast<volatile int*>(&unit_sh[s]) = u;
        mbar_arrive(smem_u32(&ufull_bar[s]));
        st_shared_cluster_u32(unit_peer0 + s * 4, static_cast<uint32_t>(u));
        mbar_arrive_cluster(ufull_peer0 + s * 8);
        if (u < 0) break;
      }
    }
  } else {
    // epilogue: warp w may read TMEM lanes [32 (w % 4), 32 (w % 4) + 32)
    const int q = warp & 3;
    const int hf = (warp - 2) >> 2;
    constexpr int kCols = kOrdered ? 256 : 128;   // columns of a tile that one warp reads
    const int r_in_tile = static_cast<int>(rank) * 128 + q * 32 + lane;
    const uint32_t acce_lead0 = mapa_shared(smem_u32(&acce_bar[0]), 0);
    uint32_t acc_it = 0;
    bool ok = true;
    for (uint32_t ui = 0; ok; ++ui) {
      int u = -1;
      if (lane == 0) u = next_unit(ui);
      u = __shfl_sync(0xffffffffu, u, 0);
      if (u < 0) break;
      if (kOrdered && hf == 1) continue;
      int mt, s, vt0, vt1;
      unit_of(u, n_mt, S, mt, s);
      split_range<kOrdered>(s, S, a.n_vtiles, vt0, vt1);
      const int row = mt * 256 + r_in_tile;
      const bool valid = row < n_rows;
      const int x = valid ? a.tok_p[row] : -1;
      Stats st;
      float zxv = 0.f;
      bool found = false;
      for (int vt = vt0; vt < vt1; ++vt) {
        const uint32_t buf = acc_it & 1u;
        if (!(ok = mbar_wait(smem_u32(&accf_bar[buf]), (acc_it >> 1) & 1u, abort_flag, a.err))) break;
        tc_fence_after();
        const int col0 = vt * 256 + hf * 128;
        const int ncols = min(kCols, a.V - col0);   // may be <= 0 in the last tile
        const int lx = x - col0;
        const uint32_t taddr = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + buf * 256 + hf * 128;
#pragma unroll 1
        for (int c0 = 0; c0 < kCols; c0 += 32) {
          if (c0 >= ncols) break;
          float v[32];
          tmem_ld32(taddr + c0, v);
          const int lxc = lx - c0;
          if (static_cast<unsigned>(lxc) < 32u) {
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if (j == lxc) zxv = v[j];
            found = true;
          }
          if (c0 + 32 <= ncols)
            fold_full<kOrdered>(v, st);
          else
            fold_partial<kOrdered>(v, ncols - c0, st);
        }
        // every lane's TMEM reads are complete: one arrival per warp hands it back
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster_relaxed(acce_lead0 + buf * 8);
        ++acc_it;
      }
      if (!ok) break;
      if (valid && found) a.zx[row] = zxv;
      if constexpr (kOrdered) {
        if (valid) a.part[static_cast<int64_t>(s) * a.rows_cap + row] = make_float4(st.m, st.s, st.q2 * kLn2, 0.f);
        continue;
      }
      // the two warps of a lane quarter put their column halves together
      if (hf == 1) {
        if (!(ok = mbar_wait(smem_u32(&hempty_bar[q]), (ui & 1u) ^ 1u, abort_flag, a.err))) break;
        half_sh[q][0][lane] = st.m;
        half_sh[q][1][lane] = st.s;
        half_sh[q][2][lane] = st.q2;
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&hfull_bar[q]));
      } else {
        if (!(ok = mbar_wait(smem_u32(&hfull_bar[q]), ui & 1u, abort_flag, a.err))) break;
        const float mo = half_sh[q][0][lane], so = half_sh[q][1][lane], qo = half_sh[q][2][lane];
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&hempty_bar[q]));
        const float M = fmaxf(st.m, mo);
        float S2 = 0.f, Q2 = 0.f;
        auto add = [&](float mi, float si, float qi) {
          if (si != 0.f) {   // 0: no columns.  A NaN passes, so that the row shows it
            const float d = (mi - M) * kLog2e;
            const float f = ex2_approx(d);
            S2 = fmaf(f, si, S2);
            Q2 = fmaf(f, fmaf(d, si, qi), Q2);
          }
        };
        add(st.m, st.s, st.q2);
        add(mo, so, qo);
        if (valid) a.part[static_cast<int64_t>(s) * a.rows_cap + row] = make_float4(M, S2, Q2 * kLn2, 0.f);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  cluster_sync_all();   // no CTA leaves while the other may still touch its memory
  tc_fence_after();
  if (warp == 1) {
    __syncwarp();
    tmem_dealloc_pair(tmem_base, 512);
  }
}

}  // namespace

cudaError_t launch_lmhead_fwd(const CUtensorMap& tm_h, const CUtensorMap& tm_w, const FwdArgs& a, int grid,
                              cudaStream_t s) {
  // the shared-memory attribute is per device: set it on each device once
  static std::atomic<unsigned long long> attr_set[2] = {};
  auto* const k = a.ordered ? &lmhead_fwd_kernel<true> : &lmhead_fwd_kernel<false>;
  auto& set = attr_set[a.ordered ? 1 : 0];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if ((set.load(std::memory_order_acquire) & bit) == 0) {
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e != cudaSuccess) return e;
    set.fetch_or(bit, std::memory_order_release);
  }
  k<<<grid / 2 * 2, kThreads, kSmemBytes, s>>>(tm_h, tm_w, a);
  return cudaGetLastError();
}

}  // namespace molt
