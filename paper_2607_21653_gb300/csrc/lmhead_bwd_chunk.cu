// Backward pass of the fused LM-head + policy loss over chunks of the
// tokens x vocabulary plane.
//
//   g_tv = coef_t (softmax(z_t)_v - [v == x_t]),  coef_t = m_t c_t / D   (Eq. 2)
//          (+ ecoef_t softmax(z_t)_v (z_tv - mu_t) with an entropy bonus)
//   dH_t = sum_v g_tv W_v          dW_v = sum_t g_tv h_t
//
// A chunk is up to 4096 tokens x 4096 vocab columns.  Its g (bf16, at most
// 32 MB) passes from the products that form it to the products that read it
// through a ring of a few chunk buffers, 64 MB together, that the 129 MB L2 holds
// while they are used (as any store it is also written back: 3.5 of the 52.9 GB of
// DRAM traffic at T = 11626 rows, H = 4096, V = 151936); neither the logits nor g of
// the whole plane exist anywhere.  All three products are then plain 256 x 256
// tiles on CTA pairs (tcgen05 cta_group::2):
//   Z    z = h W^T, M = 256 tokens, N = 256 vocab, K = H; the epilogue turns z
//        into g and stores it to the chunk buffer
//   dH   M = 256 tokens, N = 256 of H, K = the chunk's vocab; stored to the fp32
//        dhidden accumulator by the first vocab chunk, reduce-added by the others
//   dW   M = 256 vocab, N = 256 of H, K = the chunk's tokens; stored to dW by the
//        first token chunk (unless the call adds to it), reduce-added by the others
//
// Why chunks.  Every unit that holds g in one cluster's memory (512 x 512 at
// most) drains 4 H (Tu + Vu) bytes of fp32 partial sums for 6 Tu Vu H flops
// through its SMs' path to L2, and those drains held the operand loads back.
// A chunk is eight times wider in both directions, so the drains fall to an
// eighth, and no tile waits for a chain Z -> g -> dH -> dW inside one cluster.
// (Reproducible sums keep the drains: see kDetK.)
//
// One persistent launch walks all tiles of all chunks.  The tiles form one list,
//   step s:  dH tiles of chunk s - L, Z tiles of chunk s, dW tiles of chunk s - L
// (L < buffers, see chunk_plan in api.cu), and CTA pairs claim them in list order from
// a counter.  A dH or dW tile waits until every Z tile of its chunk is stored (zdone), a
// Z tile's epilogue until every tile that read the buffer's previous chunk is through
// (cdone).  Both are earlier in the list, so they were claimed earlier by pairs
// that are running: the waits end whatever share of the grid is resident.  L steps
// lie between a chunk's Z tiles and what reads them, buffers - L between those and the
// buffer's next Z tiles: each has to cover the tiles in flight.
//
// Roles per CTA (384 threads): warps 0 and 11 TMA producers of the A and the B
// operand (each CTA loads its half of both), warp 1 MMA issuer (even CTA) and
// TMEM owner, warps 2-9 epilogue, two per TMEM lane quarter (128 columns each),
// warp 10 (even CTA) claims tiles and hands them to the other roles of both CTAs
// through a ring of two slots.  TMEM holds two 256-column accumulators, so a
// tile's epilogue runs under the next tile's products.
//
// What bounds it, measured on T = 16384, H = 4096, V = 151936 (61.2 TFLOP in
// three products): 36.8 ms, 1.66 PFLOP/s, at the board's power cap (1.49 GHz of
// 2.07, 1375 W), where a cuBLAS 8192^3 product reaches 1.72 at the same clock; the
// cluster kernel takes 54.4-57.3 ms.  A tile of 64 K blocks takes 35.2K clocks of
// 32.8K ideal.  Issue decides what is left of the clock: one thread that waits for
// one stage at a time, with address arithmetic between the products, kept the
// tensor pipe at 67 % even with all loads left out, two stages per turn with the
// four products of each in one statement at 96 %; one producer thread with four
// 8 KB boxes per stage needed 830 clocks per K block of 512; and tiles decoded by
// the claiming warp, instead of by every role from their index, took 1 to 2K
// clocks off each.  A tile of few K blocks (short H) is bound by its epilogue,
// which converts without the target's and the edge's selects wherever the warp has
// neither and signals a Z tile's stores one tile later (T = 4000, H = 320, V =
// 50257: 0.51 ms, before these three 0.57; T = 3000, H = 1024, V = 32000: 0.355,
// before 0.399), and by the waits between the tiles of a chunk (see
// chunk_plan in api.cu).  Counters on T = 8192, H = 4096,
// V = 32768: tensor pipe active 93 % of the cycles, DRAM 28 %, L2 61 %.
#include <atomic>
#include <climits>
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

#include "molt_internal.cuh"
#include "ptx.cuh"

namespace molt {
namespace {

constexpr int kStages = 6;
constexpr int kHalf = 128 * kBK * 2;              // one operand's half of a stage, 16 KB
constexpr int kStageBytes = 2 * kHalf;            // 32 KB per CTA
constexpr int kOffBox = kStages * kStageBytes;    // 192 KB
constexpr int kBoxBytes = 4096;                   // 32 rows x 128 bytes
constexpr int kEpiWarps = 8;
constexpr int kThreads = 128 + 32 * kEpiWarps;
constexpr int kSmemBytes = 1024 + kOffBox + kEpiWarps * kBoxBytes;
constexpr int kSlots = 2;                         // tiles handed from the claiming warp to the other roles
// Tokens (columns) per term of a reproducible sum.  The mode's results stay the same
// bits from one version of the library to the next, so a term is what the cluster
// kernel adds at a time, and the two kernels give the same bits.  A whole chunk to a
// term, an eighth of the additions into global memory, takes 14.8 ms for the call at
// T = 16384, H = 4096, V = 65536 (30 % masked), terms of 512 18.2, the cluster kernel 23.1.
constexpr int kDetK = 512;
constexpr float kLog2e = 1.4426950408889634f;

enum TileKind : int { kTileZ = 0, kTileDH = 1, kTileDW = 2 };

// What one claimed tile is, as the claiming warp hands it to the other roles.
// t, v, h, t0 and v0 count 256-row / 256-column tiles.
struct __align__(16) Tile {
  int kind;      // TileKind, or -1 at the end of the walk
  int chunk;     // in list order
  int buf;       // chunk buffer
  int nk;        // K blocks
  int t, v, h;   // global tile indices (those the kind uses)
  int order;     // dH: the vocab chunk, dW: the token chunk
  int t0, v0;    // the chunk's first token and vocab tile
  int need;      // dH, dW: warps that store the chunk's g; Z: tiles that read the
                 // buffer's previous chunk (0: none)
  int first;     // dH, dW: warps that store the first contribution to this sum, which
                 // the tile's own is added to (0: it is the first, or dW is added to
                 // what the caller has there)
};

// The tile list, walked forwards by the claiming thread: claimed indices only grow.
// kAlign: chunks begin at a multiple of so many tiles.
template <int kAlign>
struct TileList {
  int n_rows, V, H;
  bool add_dw;
  int n_t, n_v, n_h, n_tc, n_vc, n_chunks, nb, lag;
  int total;                             // tiles in the list
  int step, base;                        // list step and its first index
  int n_dh, n_z, n_dw;                   // tiles of the step
  int c_t0, c_ct, c_v0, c_cv;            // chunk step - L
  int z_t0, z_ct, z_v0, z_cv;            // chunk step
  __device__ __forceinline__ void init(const ChunkArgs& a, int rows) {
    n_rows = rows;
    V = a.V;
    H = a.H;
    n_t = (n_rows + 255) / 256;
    n_v = (a.V + 255) / 256;
    n_h = (a.H + 255) / 256;
    n_tc = (n_t + a.chunk_t - 1) / a.chunk_t;
    // no rows: unless dW is added to, one chunk of no tokens whose dW tiles store zeros
    add_dw = a.add_dw != 0;
    if (n_t == 0 && !add_dw) n_tc = 1;
    n_vc = (n_v + a.chunk_v - 1) / a.chunk_v;
    n_chunks = n_tc * n_vc;
    total = n_t * n_v + (n_t * n_vc + n_v * n_tc) * n_h;   // Z + dH + dW tiles of all chunks
    nb = a.n_buf;
    lag = a.lag;
    step = 0;
    base = 0;
    fill();
  }
  __device__ __forceinline__ void span(int c, int& t0, int& ct, int& v0, int& cv) const {
    const int tc = c / n_vc, vc = c - tc * n_vc;
    t0 = begin(tc, n_tc, n_t);
    ct = begin(tc + 1, n_tc, n_t) - t0;
    v0 = begin(vc, n_vc, n_v);
    cv = begin(vc + 1, n_vc, n_v) - v0;
  }
  // first of n tiles, cut evenly into `parts`, that part i holds
  __device__ __forceinline__ int begin(int i, int parts, int n) const {
    const int64_t blocks = (n + kAlign - 1) / kAlign;
    return min(n, static_cast<int>(i * blocks / parts) * kAlign);
  }
  __device__ __forceinline__ void fill() {
    n_dh = n_z = n_dw = 0;
    const int c = step - lag;
    if (c >= 0 && c < n_chunks) {
      span(c, c_t0, c_ct, c_v0, c_cv);
      n_dh = c_ct * n_h;
      n_dw = c_cv * n_h;
    }
    if (step < n_chunks) {
      span(step, z_t0, z_ct, z_v0, z_cv);
      n_z = z_ct * z_cv;
    }
  }
  // the tile at index j (< total)
  __device__ __forceinline__ void seek(int j, Tile& x) {
    while (j >= base + n_dh + n_z + n_dw) {
      base += n_dh + n_z + n_dw;
      ++step;
      fill();
    }
    int i = j - base;
    const bool z = i >= n_dh && i < n_dh + n_z;
    x.chunk = z ? step : step - lag;
    const int tc = x.chunk / n_vc, vc = x.chunk - tc * n_vc;
    x.buf = x.chunk % nb;
    x.t0 = z ? z_t0 : c_t0;
    x.v0 = z ? z_v0 : c_v0;
    x.t = x.t0;
    x.v = x.v0;
    x.h = 0;
    x.order = 0;
    x.first = 0;
    uint32_t nz, nr;
    if (z) {
      i -= n_dh;
      x.kind = kTileZ;
      x.nk = H / kBK;
      x.v += i / z_ct;
      x.t += i % z_ct;
      nr = 0;
      if (x.chunk >= nb) chunk_counts(x.chunk - nb, nz, nr);
      x.need = static_cast<int>(nr);
      return;
    }
    chunk_counts(x.chunk, nz, nr);
    x.need = static_cast<int>(nz) * (2 * kEpiWarps);
    if (i < n_dh) {
      x.kind = kTileDH;
      x.order = vc;
      x.nk = (min(V, (c_v0 + c_cv) * 256) - c_v0 * 256 + kBK - 1) / kBK;
      x.h = i / c_ct;
      x.t += i % c_ct;
      if (vc > 0) x.first = c_ct * n_h * (2 * kEpiWarps);
    } else {
      i -= n_dh + n_z;
      x.kind = kTileDW;
      x.order = tc;
      x.nk = (min(n_rows, (c_t0 + c_ct) * 256) - c_t0 * 256 + kBK - 1) / kBK;   // 0 without rows
      x.h = i / c_cv;
      x.v += i % c_cv;
      if (tc > 0 && !add_dw) x.first = c_cv * n_h * (2 * kEpiWarps);
    }
  }
  // tiles of chunk c that write (z) or read its buffer
  __device__ __forceinline__ void chunk_counts(int c, uint32_t& z, uint32_t& rd) const {
    int t0, ct, v0, cv;
    span(c, t0, ct, v0, cv);
    z = static_cast<uint32_t>(ct * cv);
    rd = static_cast<uint32_t>((ct + cv) * n_h);
  }
};

__device__ __forceinline__ void write_box32(uint32_t box, int lane, const float (&v)[32]) {
  const uint32_t rowp = box + lane * 128;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t pos = static_cast<uint32_t>(i ^ (lane & 7));
    st_shared_v4(rowp + pos * 16, __float_as_uint(v[4 * i]), __float_as_uint(v[4 * i + 1]),
                 __float_as_uint(v[4 * i + 2]), __float_as_uint(v[4 * i + 3]));
  }
}

// kEnt: with an entropy bonus; kDet: reproducible sums
template <bool kEnt, bool kDet>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    lmhead_bwd_chunk_kernel(const __grid_constant__ ChunkMaps m, const ChunkArgs a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kStages];    // even CTA: both CTAs' bytes land here
  __shared__ __align__(8) uint64_t empty_bar[kStages];   // both CTAs
  __shared__ __align__(8) uint64_t accf_bar[2];          // both CTAs: accumulator full
  __shared__ __align__(8) uint64_t acce_bar[2];          // even CTA: one arrival per epilogue warp of the pair
  __shared__ __align__(8) uint64_t jfull_bar[kSlots];    // both CTAs: tile written
  __shared__ __align__(8) uint64_t jempty_bar[kSlots];   // even CTA: every reader of both CTAs has it
  __shared__ __align__(8) uint64_t done_bar;
  __shared__ Tile tile_sh[kSlots];
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_sh;

  const uint32_t smem0 = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t box_base = smem0 + kOffBox;
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
      mbar_init(smem_u32(&acce_bar[b]), 2 * kEpiWarps);
    }
    for (int s = 0; s < kSlots; ++s) {
      mbar_init(smem_u32(&jfull_bar[s]), 1);
      // readers: the MMA issuer, four producer warps, every epilogue warp
      mbar_init(smem_u32(&jempty_bar[s]), 5 + 2 * kEpiWarps);
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
  cluster_sync_all();   // every CTA's barriers exist before any remote arrival
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_sh;

  const int n_rows = a.counts[3];
  const int H = a.H, V = a.V;
  // columns of H that tile h covers: 256, less in the last one
  auto tile_w = [&](int h) -> int { return min(256, H - h * 256); };
  // N of its products: each CTA brings one or two whole 64-column boxes, zero past H
  auto mma_n = [&](int h) -> int { return H - h * 256 > 128 ? 256 : 128; };
  uint32_t* zdone = a.ctl + kChunkCtlHead;
  uint32_t* cdone = zdone + a.max_chunks;
  // per token chunk (vocab chunk), at its first chunk: warps that have stored the
  // first contributions to its dhidden (dW) rows
  uint32_t* dh_first = cdone + a.max_chunks;
  uint32_t* dw_first = dh_first + a.max_chunks;
  const int n_vc = ((V + 255) / 256 + a.chunk_v - 1) / a.chunk_v;

  // the i-th tile for a reader of the slot ring; false at the end of the walk, also
  // after a wait that ran out.  Single threads give the slot back here, a warp's
  // lane 0 for all of them (the condition always holds: it puts the arrival after
  // the reads).
  const uint32_t jempty_lead0 = mapa_shared(smem_u32(&jempty_bar[0]), 0);
  auto next_tile = [&](uint32_t i, Tile& x, bool whole_warp = false) -> bool {
    const uint32_t s = i % kSlots;
    // CTA scope in both CTAs: the odd one's copy arrives as bytes of the barrier (a
    // cluster-scope acquire here cost about 1000 clocks between two tiles)
    if (!mbar_wait(smem_u32(&jfull_bar[s]), (i / kSlots) & 1u, abort_flag, a.err)) return false;
    const uint32_t src = smem_u32(&tile_sh[s]);
    int4 q[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) q[k] = ld_shared_v4(src + 16 * k);
    if (whole_warp) __syncwarp();
    if ((!whole_warp || lane == 0) && (q[0].x & q[1].x & q[2].x) != INT_MIN)
      mbar_arrive_cluster_relaxed(jempty_lead0 + s * 8);
    x.kind = q[0].x;
    x.chunk = q[0].y;
    x.buf = q[0].z;
    x.nk = q[0].w;
    x.t = q[1].x;
    x.v = q[1].y;
    x.h = q[1].z;
    x.order = q[1].w;
    x.t0 = q[2].x;
    x.v0 = q[2].y;
    x.need = q[2].z;
    x.first = q[2].w;
    return x.kind >= 0;
  };

  // K blocks that one accumulator sums: all of a tile's, or in a reproducible sum one
  // term's, which a chunk's begin is a multiple of
  auto term_k = [&](const Tile& x) -> int { return kDet && x.kind != kTileZ ? kDetK / kBK : INT_MAX / 2; };

  if (warp == 0) {
    // A: 128 rows of h (Z) or g (dH), or 64 token rows of two panels of g (dW)
    if (lane == 0) {
      prefetch_tmap(&m.h128);
      prefetch_tmap(&m.g128);
      prefetch_tmap(&m.g64x2);
      const uint32_t full_lead0 = mapa_shared(smem_u32(&full_bar[0]), 0);
      uint32_t st = 0, ph = 0, n_it = 0;
      int ready = -1;   // last chunk seen whole: both kinds of tiles that read it come in runs
      bool ok = true;
      Tile x;
      for (uint32_t ji = 0; ok && next_tile(ji, x); ++ji) {
        const int nk = x.nk;
        if (x.kind != kTileZ && x.chunk != ready) {
          if (!turn_wait(zdone + x.chunk, static_cast<uint32_t>(x.need), abort_flag, a.ctl + 1, a.err)) break;
          fence_proxy_async_global();
          ready = x.chunk;
        }
        const int trow = x.t * 256 + static_cast<int>(rank) * 128;
        const int gpanel = x.buf * a.buf_panels + (x.v - x.v0) * 4 + static_cast<int>(rank) * 2;   // dW
        const int grow = x.buf * a.buf_panels * a.panel_rows + trow - x.t0 * 256;                  // dH
        for (int kb = 0; kb < nk; ++kb) {
          if (!(ok = mbar_wait(smem_u32(&empty_bar[st]), ph ^ 1u, abort_flag, a.err))) break;
          const uint32_t sa = smem0 + st * kStageBytes, fb = full_lead0 + st * 8;
          if (leader) mbar_arrive_expect_tx(smem_u32(&full_bar[st]), 2 * kStageBytes);
          ++n_it;
          if (x.kind == kTileZ)
            tma_load_2d_pair(sa, &m.h128, fb, kb * kBK, trow);
          else if (x.kind == kTileDH)
            tma_load_2d_pair(sa, &m.g128, fb, 0, grow + kb * a.panel_rows);
          else
            tma_load_3d_pair(sa, &m.g64x2, fb, 0, kb * kBK, gpanel);
          if (++st == kStages) {
            st = 0;
            ph ^= 1u;
          }
        }
      }
      if (leader) {
        // every copy into both CTAs completes on these barriers: wait for the
        // last issued stages before the pair may exit
        const uint32_t first = n_it > (uint32_t)kStages ? n_it - kStages : 0u;
        for (uint32_t j = first; j < n_it; ++j)
          mbar_wait_drain(smem_u32(&full_bar[j % kStages]), (j / kStages) & 1u, a.err);
      }
    }
  } else if (warp == 3 + kEpiWarps) {
    // B: 128 W rows (Z), or 64 rows of W (dH) or h (dW) by 128 columns
    if (lane == 0) {
      prefetch_tmap(&m.w128);
      prefetch_tmap(&m.w64x2);
      prefetch_tmap(&m.h64x2);
      const uint32_t full_lead0 = mapa_shared(smem_u32(&full_bar[0]), 0);
      uint32_t st = 0, ph = 0;
      bool ok = true;
      Tile x;
      for (uint32_t ji = 0; ok && next_tile(ji, x); ++ji) {
        const int nk = x.nk;
        const bool z = x.kind == kTileZ;
        const CUtensorMap* map = x.kind == kTileDH ? &m.w64x2 : &m.h64x2;
        const int vrow = x.v * 256 + static_cast<int>(rank) * 128;
        const int hc = x.h * 4 + static_cast<int>(rank) * (mma_n(x.h) / 128);   // in 64-column boxes
        const int row0 = (x.kind == kTileDH ? x.v0 : x.t0) * 256;
        for (int kb = 0; kb < nk; ++kb) {
          if (!(ok = mbar_wait(smem_u32(&empty_bar[st]), ph ^ 1u, abort_flag, a.err))) break;
          const uint32_t sb = smem0 + st * kStageBytes + kHalf, fb = full_lead0 + st * 8;
          if (z)
            tma_load_2d_pair(sb, &m.w128, fb, kb * kBK, vrow);
          else
            tma_load_3d_pair(sb, map, fb, 0, row0 + kb * kBK, hc);
          if (++st == kStages) {
            st = 0;
            ph ^= 1u;
          }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && leader) {
      uint32_t st = 0, ph = 0, ai = 0;
      bool ok = true;
      Tile x;
      for (uint32_t ji = 0; ok && next_tile(ji, x); ++ji) {
        const int nk = x.nk;
        // K-major operands advance 32 bytes per K = 16, MN-major ones 16 rows of 128
        const bool a_mn = x.kind == kTileDW, b_mn = x.kind != kTileZ;
        const uint32_t idesc = idesc_bf16_f32(256, b_mn ? mma_n(x.h) : 256, a_mn, b_mn);
        const uint32_t a_step = a_mn ? 128u : 2u, b_step = b_mn ? 128u : 2u;
        const uint64_t ad0 = sdesc_sw128(smem0, a_mn ? 8192u : 16u, 1024);
        const uint64_t bd0 = sdesc_sw128(smem0 + kHalf, b_mn ? 8192u : 16u, 1024);
        uint32_t d = 0;
        auto issue = [&](uint32_t stage, uint32_t accumulate) {
          umma4_bf16_pair(d, ad0 + stage * (kStageBytes >> 4), bd0 + stage * (kStageBytes >> 4), a_step, b_step,
                          idesc, accumulate);
          umma_commit_pair_mc(smem_u32(&empty_bar[stage]), 3);
        };
        // one accumulator after the other: one to a tile, or to a term
        int kb = 0;
        do {
          const uint32_t buf = ai & 1u;
          if (!(ok = mbar_wait(smem_u32(&acce_bar[buf]), ((ai >> 1) & 1u) ^ 1u, abort_flag, a.err))) break;
          tc_fence_after();
          d = tmem_base + buf * 256;
          // two stages per turn: one wait of the issuing thread for eight products.
          // The copies' complete_tx makes both CTAs' bytes visible to the MMAs
          // issued after the phase flips; a CTA-scope wait is enough.
          const int k0 = kb, k1 = kDet ? min(nk, kb + term_k(x)) : nk;
          for (; kb < k1; kb += 2) {
            const bool two = kb + 1 < k1;
            const uint32_t st0 = st;
            if (!(ok = mbar_wait(smem_u32(&full_bar[st]), ph, abort_flag, a.err))) break;
            if (++st == kStages) {
              st = 0;
              ph ^= 1u;
            }
            if (two && !(ok = mbar_wait(smem_u32(&full_bar[st]), ph, abort_flag, a.err))) break;
            tc_fence_after();
            issue(st0, kb != k0 ? 1u : 0u);
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
          ++ai;
        } while (kDet && kb < nk);
      }
      umma_commit_pair_mc(smem_u32(&done_bar), 1);
      mbar_wait_drain(smem_u32(&done_bar), 0, a.err);
    }
  } else if (warp == 2 + kEpiWarps) {
    if (lane == 0 && leader) {
      const uint32_t tile_peer0 = mapa_shared(smem_u32(&tile_sh[0]), 1);
      const uint32_t jfull_peer0 = mapa_shared(smem_u32(&jfull_bar[0]), 1);
      TileList<kDet ? kDetK / 256 : 1> list;
      list.init(a, n_rows);
      Tile x{};
      for (uint32_t i = 0; x.kind >= 0; ++i) {
        const uint32_t s = i % kSlots;
        // claimed when the slot frees and no earlier, so that pairs run at most
        // kSlots tiles ahead of one another's claims
        if (!mbar_wait_cluster(smem_u32(&jempty_bar[s]), ((i / kSlots) & 1u) ^ 1u, abort_flag, a.err)) break;
        const int j = static_cast<int>(atomicAdd(a.ctl, 1u));
        if (j < list.total)
          list.seek(j, x);
        else
          x.kind = -1;
        const int4 q[3] = {make_int4(x.kind, x.chunk, x.buf, x.nk), make_int4(x.t, x.v, x.h, x.order),
                           make_int4(x.t0, x.v0, x.need, x.first)};
        const uint32_t own = smem_u32(&tile_sh[s]), peer = tile_peer0 + s * static_cast<uint32_t>(sizeof(Tile));
        const uint32_t peer_bar = jfull_peer0 + s * 8;
        mbar_arrive_expect_tx_cluster(peer_bar, sizeof(Tile));
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          st_shared_v4(own + 16 * k, q[k].x, q[k].y, q[k].z, q[k].w);
          st_async_v4(peer + 16 * k, peer_bar, q[k]);
        }
        mbar_arrive(smem_u32(&jfull_bar[s]));
      }
    }
  } else {
    const int q = warp & 3;
    const int hf = (warp - 2) >> 2;
    const uint32_t lane_off = static_cast<uint32_t>(q * 32) << 16;
    const uint32_t box = box_base + (warp - 2) * kBoxBytes;
    const uint32_t acce_lead0 = mapa_shared(smem_u32(&acce_bar[0]), 0);
    const int slab = static_cast<int>(rank) * kEpiWarps + (warp - 2);
    bool ok = true;
    // waits until this warp's box has been read out
    auto box_free = [&]() {
      if (lane == 0) bulk_wait_group_read<0>();
      __syncwarp();
    };
    // counter that this warp still has to raise for its last tile's stores, or
    // nullptr: they are awaited when the warp would wait anyway, and at the latest
    // in the next tile, so nothing that waits for them is held up
    uint32_t* pending = nullptr;
    auto raise = [&]() {
      if (pending == nullptr) return;
      if (lane == 0) {
        bulk_wait_group<0>();
        fence_proxy_async_global();
        red_add_release_gpu(pending, 1u);
      }
      __syncwarp();
      pending = nullptr;
    };
    // waits (bounded) until a counter that earlier tiles raise reaches `count`
    auto wait_count = [&](const uint32_t* counter, int count) -> bool {
      raise();
      int good = 1;
      if (lane == 0) {
        good = turn_wait(counter, static_cast<uint32_t>(count), abort_flag, a.ctl + 1, a.err) ? 1 : 0;
        fence_proxy_async_global();
      }
      return __shfl_sync(0xffffffffu, good, 0) != 0;
    };
    int seen_dh = -1, seen_dw = -1;   // last first chunks seen stored
    uint32_t ai = 0;   // accumulators read
    // the next accumulator's products
    auto acc_full = [&]() -> bool {
      const uint32_t bar = smem_u32(&accf_bar[ai & 1u]), ph = (ai >> 1) & 1u;
      if (pending != nullptr && !__all_sync(0xffffffffu, mbar_test_wait(bar, ph))) raise();
      const bool full = mbar_wait(bar, ph, abort_flag, a.err);
      tc_fence_after();
      return full;
    };
    Tile x;
    for (uint32_t ji = 0; ok && next_tile(ji, x, true); ++ji) {
      const int r0 = static_cast<int>(rank) * 128 + q * 32;   // this warp's first row of the tile
      auto taddr = [&]() -> uint32_t { return tmem_base + lane_off + (ai & 1u) * 256 + hf * 128; };
      // accumulator read out: one arrival per warp hands it back
      auto release_acc = [&]() {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster_relaxed(acce_lead0 + (ai & 1u) * 8);
        ++ai;
      };
      if (x.kind == kTileZ) {
        const int row = x.t * 256 + r0 + lane;
        const bool in = row < n_rows;
        const float coef = in ? a.coef[row] : 0.f;
        float ecoef = 0.f, mu = 0.f;
        if constexpr (kEnt) {
          if (in) {
            ecoef = a.ecoef[row];
            mu = a.mu[row];
          }
        }
        const float lseL = in ? a.lse[row] * kLog2e : 0.f;
        const int vbase = x.v * 256 + hf * 128;
        const int lx = in ? a.tok_p[row] - vbase : -1;
        const int nvalid = in ? V - vbase : 0;
        // the buffer's previous chunk must have been read
        if (x.need > 0 && !(ok = wait_count(cdone + x.chunk - a.n_buf, x.need))) break;
        if (!(ok = acc_full())) break;
        const int p0 = (x.v - x.v0) * 4 + hf * 2;
        const int gy = (x.buf * a.buf_panels + p0) * a.panel_rows + (x.t - x.t0) * 256 + r0;
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
          uint32_t w[32];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            float v[32];
            tmem_ld32(taddr() + c * 64 + u * 32, v);
            const int lxc = lx - c * 64 - u * 32;
            const int nv = nvalid - c * 64 - u * 32;
            auto p_of = [&](int j) -> float {   // g without the target's term
              const float e = ex2_approx(fmaf(v[j], kLog2e, -lseL));
              if constexpr (kEnt) return fmaf(ecoef, v[j] - mu, coef) * e;
              return coef * e;
            };
            // a target or an invalid column among the warp's 32 x 32 values is rare
            if (__any_sync(0xffffffffu, static_cast<unsigned>(lxc) < 32u || nv < 32)) {
#pragma unroll
              for (int j = 0; j < 32; j += 2) {
                float g0 = p_of(j), g1 = p_of(j + 1);
                if (j == lxc) g0 -= coef;
                if (j + 1 == lxc) g1 -= coef;
                if (j >= nv) g0 = 0.f;
                if (j + 1 >= nv) g1 = 0.f;
                w[u * 16 + j / 2] = pack_bf16x2(g0, g1);
              }
            } else {
#pragma unroll
              for (int j = 0; j < 32; j += 2) w[u * 16 + j / 2] = pack_bf16x2(p_of(j), p_of(j + 1));
            }
          }
          if (c == 1) release_acc();
          if (c == 0) raise();   // of the tile before, long stored
          box_free();
          const uint32_t rowp = box + lane * 128;
#pragma unroll
          for (int i = 0; i < 8; ++i)
            st_shared_v4(rowp + static_cast<uint32_t>(i ^ (lane & 7)) * 16, w[4 * i], w[4 * i + 1], w[4 * i + 2],
                         w[4 * i + 3]);
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            tma_store_2d(&m.g32, box, 0, gy + c * a.panel_rows);
            bulk_commit_group();
          }
        }
        pending = zdone + x.chunk;
        continue;
      }
      const bool dh = x.kind == kTileDH;
      const bool empty = !dh && n_rows == 0;   // dW of no rows: zeros, no products
      const int w = tile_w(x.h);
      const int y = (dh ? x.t : x.v) * 256 + r0;
      const bool rows_in = y < (dh ? n_rows : V);
      const CUtensorMap* map = dh ? &m.dh : &m.dw;
      // the first contribution to a sum is stored, so nothing has to be zeroed
      // before; the others are added once it is there: it was a tile of an earlier
      // step, so the wait is a formality
      const bool first = x.order == 0 && (dh || !a.add_dw);
      uint32_t* turn = nullptr;
      const int n_term = kDet ? max(1, (x.nk + kDetK / kBK - 1) / (kDetK / kBK)) : 1;
      for (int term = 0; ok && term < n_term; ++term) {
        if (!(ok = acc_full())) break;
        // the products have read the chunk buffer
        if (term == n_term - 1 && leader && warp == 2 && lane == 0) red_add_release_gpu(cdone + x.chunk, 1u);
        if (term == 0) {
          if constexpr (kDet) {
            // reproducible sums: the contributions to a slab take turns in chunk order
            const int n_h = (H + 255) / 256;
            const int64_t tile = static_cast<int64_t>(dh ? x.t : a.max_t + x.v) * n_h + x.h;
            turn = a.det_turns + tile * (2 * kEpiWarps) + slab;
            if (!(ok = wait_count(turn, x.order))) break;
          } else if (x.first > 0) {
            const int c0 = dh ? x.chunk - x.order : x.chunk - x.order * n_vc;
            int& seen = dh ? seen_dh : seen_dw;
            if (seen != c0) {
              if (!(ok = wait_count((dh ? dh_first : dw_first) + c0, x.first))) break;
              seen = c0;
            }
          }
        }
        const bool store = first && term == 0;
#pragma unroll 1
        for (int s = 0; s < 4; ++s) {
          const int col = hf * 128 + s * 32;
          if (col >= w) break;
          float v[32];
          tmem_ld32(taddr() + s * 32, v);
          if (empty) {
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = 0.f;
          }
          if (kDet && store) {
            // what adding to +0 would leave: no negative zeros
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = __fadd_rn(v[j], 0.f);
          }
          if (s == 3 || col + 32 >= w) release_acc();
          if (s == 0) raise();
          box_free();
          write_box32(box, lane, v);
          fence_proxy_async_smem();
          if (term > 0 && lane == 0) {
            // this warp's box of the term before is in the sum
            if (w - hf * 128 >= 128)
              bulk_wait_group<3>();
            else
              bulk_wait_group<0>();
            fence_proxy_async_global();
          }
          __syncwarp();
          if (lane == 0 && rows_in) {
            if (store)
              tma_store_2d(map, box, x.h * 256 + col, y);
            else
              tma_reduce_add_2d(map, box, x.h * 256 + col, y);
          }
          if (lane == 0) bulk_commit_group();
        }
        if (hf * 128 >= w) release_acc();   // no columns for this warp
      }
      if (!ok) break;
      raise();
      if (!kDet && first) pending = dh ? dh_first + x.chunk : dw_first + x.chunk;
      if constexpr (kDet) {
        if (lane == 0) {
          bulk_wait_group<0>();
          fence_proxy_async_global();
          st_release_gpu(turn, static_cast<uint32_t>(x.order) + 1u);
        }
        __syncwarp();
      }
    }
    raise();
    if (lane == 0) bulk_wait_group<0>();
    __syncwarp();
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

cudaError_t launch_lmhead_bwd_chunk(const ChunkMaps& m, const ChunkArgs& a, int n_ctas, cudaStream_t s) {
  const bool ent = a.ecoef != nullptr;
  auto* k = a.det_turns != nullptr ? (ent ? &lmhead_bwd_chunk_kernel<true, true> : &lmhead_bwd_chunk_kernel<false, true>)
                                   : (ent ? &lmhead_bwd_chunk_kernel<true, false> : &lmhead_bwd_chunk_kernel<false, false>);
  const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
  if (e != cudaSuccess) return e;
  k<<<n_ctas / 2 * 2, kThreads, kSmemBytes, s>>>(m, a);
  return cudaGetLastError();
}

}  // namespace molt
