// Decode attention for wide multi-query groups (33..128 query heads per KV head, head_dim 64,
// bf16) on the 5th-generation tensor cores.  With g = 71 (Falcon-shaped MQA) the step needs
// g flop per byte of K/V -- hundreds of TFLOP/s at HBM speed -- so both contractions run as
// tcgen05.mma with accumulators in tensor memory:
//   S[head rows x 128 tokens] = Q K_tile^T      (Q, K tile in shared memory, K-major)
//   O[head rows x 64]        += P V_tile         (P bf16 in TENSOR memory, V tile MN-major)
// One CTA per (layer, unit, split), two CTAs per SM; per 128-token tile the roles are
//   warp 0      TMA: K and V tiles into a ring of stages (128-byte swizzle, every CTA its own tiles)
//   warp 1      MMA issue (one thread)
//   warps 2..5  p = exp2(s*scale - m_ref) from S to P, packed to bf16 and kept in tensor memory as the A
//               operand of the second MMA, four threads to a head row and the heads spread over the
//               four quarters of tensor memory (sq_tc_rows.cuh)
// Measured on B200: one M=128, K=16 MMA costs 45-48 cycles for N <= 64 and 64 cycles for N = 128,
// and operands read from shared memory compete with the TMA writes for its 128 B/clk; keeping P
// in tensor memory (64 columns) removes 56 KB of shared-memory traffic per tile.  Inside the
// kernel, two CTAs sharing the pipe, an MMA holds the issuing thread for about 80 cycles and a
// tcgen05.commit for about 180.
// A row's reference m_ref is its maximum over the first tile; later tiles reuse it and only
// when a weight would exceed 2^16 is the reference moved (O and the sums rescaled through
// tcgen05.ld/st, the tile redone): every weight stays finite and the result is that of the
// exact softmax.  Every barrier wait is bounded.
// What bounds the kernel (measured on B200 with per-tile clock stamps and with copies that leave
// work out, when a thread had a whole row; now the rows are spread evenly over the four schedulers,
// which took 3855 to 3663 us per token of 224 sequences of 8192 tokens): a softmax warp needed 1250 cycles per tile alone on its scheduler and 2150-2250 when
// it shared it with the other CTA's (the special-function unit: 128 exp2 per row and tile at one
// warp instruction per 8 cycles), against 2780 cycles of HBM time per pair of tiles at 1.9 GHz;
// a polynomial exp2 on the FMA pipe for a part of the weights was slower at every share tried.
// Cluster form (up to 96 heads, launches whose units leave room for at least two CTAs each, all at a time): the
// pieces of a unit are the CTAs of one cluster.  They read one another's row sums and un-normalised outputs over
// distributed shared memory and each stores its share of the output, where split-K sends them through memory to the
// last piece to arrive, which took 12 us to merge a unit of 71 heads in 8 pieces while the launch waited.  With H2O each
// piece then knows the log-sum-exps and runs the score pass (k_decode_gain.cu has it as a launch of its own) over its
// tokens: S^T = K_tile Q^T again, K from L2, a thread owns a token, and the first piece picks the next victim.  33
// sequences of 8191 tokens, 50 %, H2O, one launch (before: two) per layer: 1228 to 833 us per token.  Bound now by the chain
// of a launch: with caches of 10 tiles, 5 pieces, of 13.5 us 4 for a piece's two tiles, 1.3 its epilogue, 2 the cluster barrier
// (pieces of unlike speed), 2.3 the row sums and the output, 2.3 the scores, 1.2 the victim.
// Streaming K and V alone (no products, no softmax) reaches 7.3 TB/s and draws 970 W of the
// board's 1000 W; with the products 6.4 TB/s, with the softmax as well 4.6-4.7 TB/s, both at the
// power limit with the SM clock near 1.5-1.6 GHz: run for longer than a few milliseconds the
// kernel is bound by power, and what helps is fewer instructions per weight.
#include <algorithm>
#include <numeric>
#include <type_traits>

#include "sq_decode_common.cuh"
#include "sq_device.cuh"
#include "sq_internal.h"
#include "sq_scores.cuh"
#include "sq_select.cuh"
#include "sq_tc.cuh"
#include "sq_tc_rows.cuh"

namespace sq {

using namespace tc;

namespace {
constexpr int kD = 64;
constexpr int kTileBytes = kTM * kD * 2;  // 16 KB: one K or V tile
constexpr int kColS = 0, kColP = 128, kColO = 192, kTmemCols = 256;
__host__ __device__ constexpr uint32_t idesc(int n, bool b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (b_mn_major ? (1u << 16) : 0u) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(128 >> 4) << 24);
}

// Cluster form: what the pieces read of one another, and scratch, in the V stages once the last tile is done.
constexpr int kMaxPieces = 14;  // CTAs of a cluster (a B200 has room for no more than 14 clusters of 13 to 16 such CTAs)
constexpr int kClusterHeads = 96;
constexpr int kORow = kD + 4;  // floats from one head's partial output to the next (no bank conflicts)
struct ClusterShared {
  float o[kClusterHeads * kORow];          // un-normalised output
  float stat[kClusterHeads * kStatStride]; // maximum, sum, sum of the rounded weights
  float factor[kMaxPieces][kClusterHeads]; // a piece's weight in the merged row
  float nlse[kTM];                         // minus the row log-sum-exps, by row of the Q tile
  ScoreCandidate offer[kMaxPieces];        // one per piece (the first CTA's is read)
  ScoreCandidate warp_best[4];
};

// (bar.sync is an .aligned form as well)
__device__ __forceinline__ void softmax_sync() {
  __syncwarp();
  asm volatile("bar.sync 1, 128;" ::: "memory");
}

// Cluster form, the four softmax warps after the last tile: the piece's partial result to shared memory, then (behind
// the cluster's barrier) the unit's row sums from all pieces, this CTA's share of the output, and with H2O the
// score pass over its own tokens and its candidate for the next victim.  The warps reach both cluster barriers
// whether or not something gave up before.
template <bool H2O, class Args, class Rows>
__device__ __forceinline__ void finish_cluster(const Args& a, const LayerDesc* ldp, int unit, int n_tiles, int t0, int t1, int len,
                                               size_t out_at, Rows& rows, const WideLayout& layout, bool ok, ClusterShared& sh,
                                               uint32_t bar_odone, uint32_t bar_gfull, uint32_t bar_gfree, uint32_t tmem_base,
                                               volatile int* abort_flag) {
  const int tid = (int)threadIdx.x - 64, lane = tid & 31, warp = tid >> 5, quarter = (warp + 2) & 3;
  const int G = a.group, n = cluster_size(), me = cluster_rank();
  if (ok) ok = __all_sync(0xffffffffu, mbar_wait(bar_odone, (n_tiles - 1) & 1, abort_flag));
  if (ok) {
    tc_fence_after();
    float m_ref, l, l_w;
    rows.finish(&m_ref, &l, &l_w);
    const int row = layout.head_of_lane(quarter, lane);
    const bool live = row < G;
#pragma unroll 1
    for (int c = 0; c < 2; ++c) {
      float o[32];
      tmem_ld32(rows.o_addr + c * 32, o);
      if (live) {
#pragma unroll
        for (int q4 = 0; q4 < 8; ++q4)
          *reinterpret_cast<float4*>(sh.o + row * kORow + c * 32 + q4 * 4) =
              make_float4(o[q4 * 4], o[q4 * 4 + 1], o[q4 * 4 + 2], o[q4 * 4 + 3]);
      }
      __syncwarp();  // the loads of tensor memory are warp-wide
    }
    if (live) *reinterpret_cast<float4*>(sh.stat + row * kStatStride) = make_float4(m_ref, H2O ? l : l_w, l_w, 0.f);
    if (H2O) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(bar_gfree);
        mbar_arrive(bar_gfree + 8);
      }
    }
  }
  cluster_arrive();
  // the first tile's scores and positions are on their way meanwhile
  const int b = ldp->b, cap = ldp->cap;
  const bool full = (len == b);
  const int* pos = reinterpret_cast<const int*>(a.pool + ldp->pos_off) + (size_t)unit * cap;
  float* acc = reinterpret_cast<float*>(a.pool + ldp->acc_off) + (size_t)unit * cap;
  const int row = quarter * 32 + lane;
  float old[2];
  int p[2];
  auto fetch = [&](int i, int u) {
    const int slot = t0 + i * kTM + row;
    old[u] = 0.f;
    p[u] = 0x7fffffff;
    if (slot < t1) {
      old[u] = acc[slot];
      if (full) p[u] = pos[slot];
    }
  };
  if (H2O) {
    fetch(0, 0);
    fetch(1, 1);
  }
  cluster_wait();
  // Every read crosses the cluster: several at a time, this thread's part of the output (four consecutive values of a
  // head from every piece) on its way while the row sums are worked out.
  const int n4 = G * kD / 4;
  auto fetch_o = [&](int i4, int r0, float4 (&v)[8]) {
    const float* src = sh.o + (i4 * 4 / kD) * kORow + (i4 * 4) % kD;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (i4 < n4 && r0 + u < n) v[u] = ld_cluster4(map_rank(src, r0 + u));
    }
  };
  float4 v[8];
  int i4 = (n - 1 - me) * 128 + tid;
  fetch_o(i4, 0, v);
  if (tid < G) {
    float M = -INFINITY, L = 0.f, Lw = 0.f;
    for (int r0 = 0; r0 < n; r0 += 8) {
      float4 st[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        st[u] = make_float4(-INFINITY, 0.f, 0.f, 0.f);
        if (r0 + u < n) st[u] = ld_cluster4(map_rank(sh.stat + tid * kStatStride, r0 + u));
      }
      float m2 = M;
#pragma unroll
      for (int u = 0; u < 8; ++u) m2 = fmaxf(m2, st[u].x);
      const float f0 = M > -INFINITY ? exp2f(M - m2) : 0.f;
      L *= f0;
      Lw *= f0;
      M = m2;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (r0 + u >= n) continue;
        const float f = exp2f(st[u].x - M);
        L += st[u].y * f;
        Lw += st[u].z * f;
        sh.factor[r0 + u][tid] = st[u].x;
      }
    }
    const float inv = 1.f / Lw;
    for (int r = 0; r < n; ++r) sh.factor[r][tid] = exp2f(sh.factor[r][tid] - M) * inv;
    if (H2O) sh.nlse[layout.row_of_group(tid >> 3) + (tid & 7)] = -(M + log2f(L));
  }
  // columns past the group: a query of zeros (tm_q), so their weight is exp2(0 - inf) = 0
  if (H2O && tid >= G && tid < (G + 7) / 8 * 8) sh.nlse[layout.row_of_group(tid >> 3) + (tid & 7)] = -INFINITY;
  softmax_sync();
  for (; i4 < n4; i4 += n * 128) {
    const int h = i4 * 4 / kD;
    float4 O = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int r0 = 0; r0 < n; r0 += 8) {
      if (r0 > 0) fetch_o(i4, r0, v);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float f = r0 + u < n ? sh.factor[r0 + u][h] : 0.f;
        O.x += v[u].x * f;
        O.y += v[u].y * f;
        O.z += v[u].z * f;
        O.w += v[u].w * f;
      }
    }
    *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(a.out) + out_at + i4 * 4) =
        make_uint2(pack_bf16x2(O.x, O.y), pack_bf16x2(O.z, O.w));
    if (i4 + n * 128 < n4) fetch_o(i4 + n * 128, 0, v);
  }
  if constexpr (H2O) {
    // ---------------- scores: thread = one token ----------------
    const int thr = a.n_tok + 1 - ldp->b_recent;  // next step: positions <= thr are outside the recent window
    const uint32_t lane_sel = (uint32_t)(quarter * 32) << 16;
    const float c = a.scale_log2;
    unsigned long long best = ~0ull;
    int best_slot = -1;
    // (a tile's scores and positions are fetched two tiles ahead: one tile takes about as long as a trip to memory)
    auto one = [&](int i, int u) {
      const int slot = t0 + i * kTM + row;
      ok = __all_sync(0xffffffffu, mbar_wait(bar_gfull + 8 * u, (i >> 1) & 1, abort_flag));
      if (!ok) return;
      tc_fence_after();
      const uint32_t s_addr = tmem_base + lane_sel + u * kTM;
      float g0 = 0.f, g1 = 0.f;
      uint32_t r[2][32];
      tmem_ld32_nowait(s_addr, r[0]);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        tmem_wait_ld(r[q & 1]);
        if (q < 3) tmem_ld32_nowait(s_addr + (q + 1) * 32, r[(q + 1) & 1]);
        const int live = layout.groups(q, G);
#pragma unroll
        for (int s = 0; s < kClusterHeads / 32; ++s) {
          if (s >= live) continue;
          const float4* nl = reinterpret_cast<const float4*>(sh.nlse + q * 32 + s * 8);
#pragma unroll
          for (int q4 = 0; q4 < 2; ++q4) {
            const float4 l4 = nl[q4];
            const uint32_t* x = r[q & 1] + s * 8 + q4 * 4;
            g0 += ex2(fmaf(__uint_as_float(x[0]), c, l4.x));
            g1 += ex2(fmaf(__uint_as_float(x[1]), c, l4.y));
            g0 += ex2(fmaf(__uint_as_float(x[2]), c, l4.z));
            g1 += ex2(fmaf(__uint_as_float(x[3]), c, l4.w));
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_gfree + 8 * u);
      if (slot < t1) {
        const float v = old[u] + (g0 + g1);
        acc[slot] = v;
        if (full && p[u] <= thr) {
          const unsigned long long rank = victim_rank(v, p[u]);
          if (rank < best) {
            best = rank;
            best_slot = slot;
          }
        }
      }
      if (i + 2 < n_tiles) fetch(i + 2, u);
    };
    for (int i = 0; ok && i < n_tiles; i += 2) {
      one(i, 0);
      if (ok && i + 1 < n_tiles) one(i + 1, 1);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long r2 = __shfl_xor_sync(0xffffffffu, best, o);
      const int s2 = __shfl_xor_sync(0xffffffffu, best_slot, o);
      if (r2 < best) {
        best = r2;
        best_slot = s2;
      }
    }
    if (lane == 0) {
      sh.warp_best[warp].rank = best;
      sh.warp_best[warp].slot = best_slot;
    }
    softmax_sync();
    if (tid == 0) {
      for (int w = 1; w < 4; ++w)
        if (sh.warp_best[w].rank < best) {
          best = sh.warp_best[w].rank;
          best_slot = sh.warp_best[w].slot;
        }
      st_cluster_candidate(map_rank(&sh.offer[me], 0), best, best_slot);
    }
  }
  cluster_arrive();
}
}  // namespace

// ROWS: rows of the Q tile held in shared memory (120 for up to 96 heads, else 128; see sq_tc_rows.cuh).
// FORM: split-K, or the pieces of a unit as the CTAs of a cluster (Args: DecodeArgsBase), see the head of the file; kClusterMax: with a
// row's maximum so far as its reference throughout.
enum WideForm { kSplitK, kCluster, kClusterMax };
template <int STAGES, int ROWS, bool H2O, WideForm FORM, class Args>
__global__ void __launch_bounds__(192, 2)
    decode_attn_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                          const __grid_constant__ CUtensorMap tm_v, Args a) {
  constexpr bool CLUSTER = FORM != kSplitK;
  constexpr int kQBytes = ROWS * 128;
  constexpr int kSlots = ROWS == 120 ? 3 : 4;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  // The first MMA addresses 128 rows of Q, of which groups of eight hold heads; the others hold anything
  // and with ROWS = 120 the last eight alias the K stage that follows (rows are independent, those
  // accumulator rows are never read).
  unsigned char* q_s = smem;
  unsigned char* k_s = q_s + kQBytes;              // STAGES tiles
  unsigned char* v_s = k_s + STAGES * kTileBytes;  // STAGES tiles
  unsigned long long* bars = reinterpret_cast<unsigned long long*>(v_s + STAGES * kTileBytes);
  static_assert(10 + 2 * STAGES <= 16 || !CLUSTER, "barrier block");
  static_assert(6 + 2 * STAGES <= 16, "barrier block");
  static_assert(!CLUSTER || sizeof(ClusterShared) <= STAGES * kTileBytes, "scratch of the cluster form");
  const uint32_t bar_q = s_u32(bars + 0), bar_odone = s_u32(bars + 1), bar_sfull = s_u32(bars + 2),
                 bar_sfree = s_u32(bars + 3), bar_pready = s_u32(bars + 4), bar_pfree = s_u32(bars + 5);
  auto bar_full = [&](int s) { return s_u32(bars + 6 + s); };
  auto bar_empty = [&](int s) { return s_u32(bars + 6 + STAGES + s); };
  // cluster form with scores: the score pass's two accumulator buffers
  auto bar_gfull = [&](int j) { return s_u32(bars + 6 + 2 * STAGES + j); };
  auto bar_gfree = [&](int j) { return s_u32(bars + 8 + 2 * STAGES + j); };
  constexpr bool SCORES = H2O && CLUSTER;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 16);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  ItemLoc it;
  if constexpr (CLUSTER) {
    it.n_split = cluster_size();
    const int k = (int)blockIdx.x / (a.n_unit * it.n_split);
    it.layer = a.order[k];
    it.base = k * a.n_unit * it.n_split;
    it.local = (int)blockIdx.x - it.base;
  } else {
    if (!locate(a, blockIdx.x, it)) return;
  }
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const LayerDesc* ldp = a.layers + it.layer;
  const int b = ldp->b, cap = ldp->cap, G = a.group;
  const int unit = it.local / it.n_split, split = it.local - unit * it.n_split;
  const int len = min(a.n_tok + 1, b);
  if (!a.early) grid_wait();
  int w;
  if (H2O) {
    w = (a.n_tok < b) ? a.n_tok : __ldcg(reinterpret_cast<const int*>(a.pool + ldp->victim_off) + unit);
    if (w < 0 || w >= b) {
      if (tid == 0) atomicOr(a.status, 2);
      w = 0;
    }
  } else {
    w = ring_slot(a.n_tok, b, ldp->ring_base, ldp->ring_origin);
  }
  int t0, t1;
  if constexpr (CLUSTER) {  // the unit's tiles, dealt out evenly (the launcher sees to it that no piece is empty)
    const int n = (len + kTM - 1) / kTM;
    t0 = split * n / it.n_split * kTM;
    t1 = min(len, (split + 1) * n / it.n_split * kTM);
  } else {
    t0 = split * a.split_tokens;
    t1 = min(len, t0 + a.split_tokens);
  }
  const int n_tiles = (t1 - t0 + kTM - 1) / kTM;
  const int seq = unit / a.n_kv_head, kvh = unit - seq * a.n_kv_head;
  const size_t tok = (size_t)(it.layer - a.layer_begin) * a.batch + seq;
  using bf16 = __nv_bfloat16;
  // (pointers are formed where they are used: the softmax loop needs the registers)

  if (tid == 0) {
    mbar_init(bar_q, 1);
    mbar_init(bar_odone, 1);
    mbar_init(bar_sfull, 1);
    mbar_init(bar_sfree, 4);   // one arrival per softmax warp
    mbar_init(bar_pready, 4);
    mbar_init(bar_pfree, 1);
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(bar_full(s), 1);
      mbar_init(bar_empty(s), 1);
    }
    if (SCORES) {
      for (int j = 0; j < 2; ++j) {
        mbar_init(bar_gfull(j), 1);
        mbar_init(bar_gfree(j), 4);
      }
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_u32(tmem_slot)), "n"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const WideLayout layout(CLUSTER ? split & 3 : WideLayout::wave());

  // fetch of K and V tile i (its stage is free); rows of this unit in the [rows][64] view of the pool
  auto load_tile = [&](int i) {
    const int st = i % STAGES;
    const long long k_row0 = ldp->k_off / (kD * 2) + (long long)unit * cap;
    const long long v_row0 = ldp->v_off / (kD * 2) + (long long)unit * cap;
    mbar_expect_tx(bar_full(st), 2 * kTileBytes);
    tma_load_2d(s_u32(k_s + st * kTileBytes), &tm_k, 0, (int)(k_row0 + t0 + i * kTM), bar_full(st));
    tma_load_2d(s_u32(v_s + st * kTileBytes), &tm_v, 0, (int)(v_row0 + t0 + i * kTM), bar_full(st));
  };
  // The first tiles are under way before the launch ahead is done, up to the one that holds slot w
  int issued = 0;
  if (a.early) {
    if (tid == 0) {
      const int n_pre = min(min(STAGES, n_tiles), (w >= t0 && w < t1) ? (w - t0) / kTM : STAGES);
      for (; issued < n_pre; ++issued) load_tile(issued);
    }
    grid_wait();
  }
  if (warp == 0) {  // Q, eight heads per copy
    const int n_group = (G + 7) / 8;
    if (lane == 0) mbar_expect_tx(bar_q, n_group * 1024);
    __syncwarp();
    if (lane < n_group)
      tma_load_3d(s_u32(q_s + layout.row_of_group(lane) * 128), &tm_q, 0, 8 * lane, (int)(tok * a.n_kv_head) + kvh, bar_q);
  }
  // the CTA whose range holds slot w stores the new token (generic proxy), then lets the TMA reads
  // (async proxy) see it
  if (w >= t0 && w < t1) {
    if (tid < 16) {
      bf16* Kb = reinterpret_cast<bf16*>(a.pool + ldp->k_off) + (size_t)unit * cap * kD;
      bf16* Vb = reinterpret_cast<bf16*>(a.pool + ldp->v_off) + (size_t)unit * cap * kD;
      const bf16* kn = reinterpret_cast<const bf16*>(a.k_new) + (tok * a.n_kv_head + kvh) * kD;
      const bf16* vn = reinterpret_cast<const bf16*>(a.v_new) + (tok * a.n_kv_head + kvh) * kD;
      const bool is_v = tid >= 8;
      const int c = tid & 7;
      const uint4 val = *reinterpret_cast<const uint4*>((is_v ? vn : kn) + c * 8);
      *reinterpret_cast<uint4*>((is_v ? Vb : Kb) + (size_t)w * kD + c * 8) = val;
    }
    if (tid == 16) {
      reinterpret_cast<int*>(a.pool + ldp->pos_off)[(size_t)unit * cap + w] = a.n_tok;
      if (H2O) reinterpret_cast<float*>(a.pool + ldp->acc_off)[(size_t)unit * cap + w] = 0.f;
    }
    __threadfence();
    fence_proxy_async();
  }
  __syncthreads();

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      for (; issued < n_tiles; ++issued) {
        const int i = issued;
        if (i >= STAGES && !mbar_wait(bar_empty(i % STAGES), ((i / STAGES) - 1) & 1, abort_flag)) break;
        load_tile(i);
      }
    }
    if constexpr (SCORES) {
      // the score pass reads the K tiles again (from L2), through the same ring of stages
      cluster_arrive();
      if (lane == 0 && !*abort_flag) {
        for (; issued < 2 * n_tiles; ++issued) {
          const int st = issued % STAGES;
          if (issued >= STAGES && !mbar_wait(bar_empty(st), ((issued / STAGES) - 1) & 1, abort_flag)) break;
          mbar_expect_tx(bar_full(st), kTileBytes);
          tma_load_2d(s_u32(k_s + st * kTileBytes), &tm_k, 0,
                      (int)(ldp->k_off / (kD * 2) + (long long)unit * cap + t0 + (issued - n_tiles) * kTM), bar_full(st));
        }
      }
      __syncwarp();
    }
    if (lane == 0) {
      if (*abort_flag) {
        mbar_wait(bar_q, 0, abort_flag);
        for (int i = max(0, issued - STAGES); i < issued; ++i)
          for (int k = 0; k < kSpinLimit && !mbar_try_wait(bar_full(i % STAGES), (i / STAGES) & 1); ++k) {
          }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: one thread ----------------
    if (lane == 0) {
      const uint32_t q_addr = s_u32(q_s);
      auto issue_s = [&](int i) -> bool {
        const int st = i % STAGES;
        if (!mbar_wait(bar_full(st), (i / STAGES) & 1, abort_flag)) return false;
        if (i >= 1 && !mbar_wait(bar_sfree, (i - 1) & 1, abort_flag)) return false;
        tc_fence_after();
        const uint32_t k_addr = s_u32(k_s + st * kTileBytes);
#pragma unroll
        for (int k = 0; k < kD / 16; ++k)
          umma_bf16(tmem_base + kColS, umma_desc(q_addr + k * 32), umma_desc(k_addr + k * 32), idesc(128, false),
                    k > 0 ? 1u : 0u);
        umma_commit(bar_sfull);
        return true;
      };
      bool ok = mbar_wait(bar_q, 0, abort_flag);
      if (ok) ok = issue_s(0);
      for (int i = 0; ok && i < n_tiles; ++i) {
        if (i + 1 < n_tiles) ok = issue_s(i + 1);
        if (!ok) break;
        const int st = i % STAGES;
        ok = mbar_wait(bar_pready, i & 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint32_t v_addr = s_u32(v_s + st * kTileBytes);
#pragma unroll
        for (int k = 0; k < kTM / 16; ++k)
          // A = P in tensor memory: 16 tokens = 8 columns per step; B = V, MN-major: 2 KB per step
          umma_bf16_ta(tmem_base + kColO, tmem_base + kColP + k * 8, umma_desc(v_addr + k * 2048), idesc(kD, true),
                       (i > 0 || k > 0) ? 1u : 0u);
        umma_commit(bar_empty(st));
        umma_commit(bar_pfree);
        umma_commit(bar_odone);
      }
    }
    __syncwarp();
    if constexpr (SCORES) {
      // S^T = K_tile Q^T: tokens on the lanes, rows of the Q tile (dead ones too) on the columns
      cluster_arrive();
      if (lane == 0 && !*abort_flag) {
        const uint32_t q_addr = s_u32(q_s);
        for (int i = 0; i < n_tiles; ++i) {
          const int j = n_tiles + i, st = j % STAGES;
          if (!mbar_wait(bar_full(st), (j / STAGES) & 1, abort_flag)) break;
          if (!mbar_wait(bar_gfree(i & 1), (i >> 1) & 1, abort_flag)) break;
          tc_fence_after();
          const uint32_t k_addr = s_u32(k_s + st * kTileBytes);
#pragma unroll
          for (int k = 0; k < kD / 16; ++k)
            umma_bf16(tmem_base + (i & 1) * kTM, umma_desc(k_addr + k * 32), umma_desc(q_addr + k * 32), idesc(128, false),
                      k > 0 ? 1u : 0u);
          umma_commit(bar_empty(st));
          umma_commit(bar_gfull(i & 1));
        }
      }
      __syncwarp();
    }
  } else {
    // ---------------- softmax: four threads = one head row (sq_tc_rows.cuh) ----------------
    const int quarter = warp & 3;
    const uint32_t lane_sel = (uint32_t)(quarter * 32) << 16;
    WideRows<H2O, kSlots> rows;
    rows.s_addr = tmem_base + lane_sel + kColS;
    rows.p_addr = tmem_base + lane_sel + kColP;
    rows.o_addr = tmem_base + lane_sel + kColO;
    rows.scale_log2 = a.scale_log2;
    rows.lane = lane;
    rows.n_slot = layout.groups(quarter, G);
    rows.begin();
    bool ok = true;

    for (int i = 0; ok && i < n_tiles; ++i) {
      const int st = i % STAGES;
      const int n_valid = min(kTM, t1 - (t0 + i * kTM));
      ok = mbar_wait(bar_sfull, i & 1, abort_flag);
      if (ok && n_valid < kTM) {
        // rows of the V tile past the unit's last token may hold anything: zero them
        ok = mbar_wait(bar_full(st), (i / STAGES) & 1, abort_flag);
        const int row = quarter * 32 + lane;
        if (ok && row >= n_valid) {
          uint4* vrow = reinterpret_cast<uint4*>(v_s + st * kTileBytes + row * 128);
#pragma unroll
          for (int c = 0; c < 8; ++c) vrow[c] = make_uint4(0, 0, 0, 0);
        }
        fence_proxy_async();  // the zeroed rows must be visible to the tensor core
      }
      ok = __all_sync(0xffffffffu, ok);  // tcgen05.ld / st are warp-wide
      if (!ok) break;
      tc_fence_after();
      float f_o = 1.f;
      const bool moved = FORM == kClusterMax && i > 0 && rows.follow(n_valid, &f_o);
      bool s_released = rows.template tile<FORM == kClusterMax>(n_valid, i == 0, bar_sfree, [&]() {
        if (i >= 1) ok = __all_sync(0xffffffffu, mbar_wait(bar_pfree, (i - 1) & 1, abort_flag));
        if (FORM == kClusterMax && ok && moved) {  // (P is free once the product that O is waiting for is complete)
          tc_fence_after();
          rows.scale_o(f_o);
        }
      });
      if (!ok) break;
      if (FORM != kClusterMax && rows.too_large()) {
        ok = __all_sync(0xffffffffu, mbar_wait(bar_odone, (i - 1) & 1, abort_flag));
        if (!ok) break;
        tc_fence_after();
        rows.redo(n_valid);
        s_released = rows.tile(n_valid, false, bar_sfree, []() {});
      }
      rows.add_tile();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(bar_pready);
        if (!s_released) mbar_arrive(bar_sfree);
      }
    }
    if constexpr (CLUSTER) {
      finish_cluster<H2O>(a, ldp, unit, n_tiles, t0, t1, len, (tok * a.n_q_head + (size_t)kvh * G) * kD, rows, layout, ok,
                          *reinterpret_cast<ClusterShared*>(v_s), bar_odone, bar_gfull(0), bar_gfree(0), tmem_base, abort_flag);
    } else {
      // ---------------- epilogue: O / l -> out (or the split-K partial) ----------------
      if (ok) ok = __all_sync(0xffffffffu, mbar_wait(bar_odone, (n_tiles - 1) & 1, abort_flag));
      if (ok) {
        tc_fence_after();
        bf16* ob = reinterpret_cast<bf16*>(a.out) + (tok * a.n_q_head + (size_t)kvh * G) * kD;
        float* stat = a.part_stat + (size_t)blockIdx.x * G * kStatStride;
        float* po = a.part_o + (size_t)blockIdx.x * G * kD;
        float m_ref, l, l_w;
        rows.finish(&m_ref, &l, &l_w);
        const int row = layout.head_of_lane(quarter, lane);
        const bool live = row < G;  // this lane's row is a real head
        const float inv = 1.f / l_w;
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
          float o[32];
          tmem_ld32(rows.o_addr + c * 32, o);
          if (live && it.n_split == 1) {
#pragma unroll
            for (int q4 = 0; q4 < 4; ++q4)
              *reinterpret_cast<uint4*>(ob + (size_t)row * kD + c * 32 + q4 * 8) =
                  make_uint4(pack_bf16x2(o[q4 * 8] * inv, o[q4 * 8 + 1] * inv), pack_bf16x2(o[q4 * 8 + 2] * inv, o[q4 * 8 + 3] * inv),
                             pack_bf16x2(o[q4 * 8 + 4] * inv, o[q4 * 8 + 5] * inv), pack_bf16x2(o[q4 * 8 + 6] * inv, o[q4 * 8 + 7] * inv));
          } else if (live) {
#pragma unroll
            for (int q4 = 0; q4 < 8; ++q4)
              *reinterpret_cast<float4*>(po + (size_t)row * kD + c * 32 + q4 * 4) =
                  make_float4(o[q4 * 4], o[q4 * 4 + 1], o[q4 * 4 + 2], o[q4 * 4 + 3]);
          }
          __syncwarp();  // the loads of tensor memory are warp-wide
        }
        if (live) {
          stat[row * kStatStride] = m_ref;
          stat[row * kStatStride + 1] = H2O ? l : l_w;
          stat[row * kStatStride + 2] = l_w;
          // H2O: the unit's row log-sum-exps (log2 domain), read by the score-update pass that follows
          if (H2O && it.n_split == 1) (a.logits + ldp->lse_off + (size_t)unit * G)[row] = m_ref + log2f(l);
        }
      }
    }
  }
  if constexpr (CLUSTER) {
    // every offer is in; nothing of another CTA's shared memory is touched after this
    if (warp < 2) {
      if (!SCORES) cluster_arrive();
      cluster_wait();
      cluster_arrive();
    }
    cluster_wait();
    if (H2O && split == 0 && tid == 64 && len == b && !*abort_flag) {
      const ClusterShared& sh = *reinterpret_cast<const ClusterShared*>(v_s);
      ScoreCandidate best = sh.offer[0];
      for (int r = 1; r < it.n_split; ++r)
        if (sh.offer[r].rank < best.rank) best = sh.offer[r];
      reinterpret_cast<int*>(a.pool + ldp->victim_off)[unit] = best.slot;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "n"(kTmemCols) : "memory");
  }
  if (tid == 0 && *abort_flag) atomicOr(a.status, kStatusTimeout);
  if constexpr (!CLUSTER)
    if (it.n_split > 1) merge_if_last<bf16>(a, it, unit, reinterpret_cast<float*>(q_s), H2O ? a.logits + ldp->lse_off + (size_t)unit * G : nullptr);
}

// The occupancy calculator takes the attention kernel's registers to leave room for one CTA per SM; two run (seen
// by their clocks: 264 CTAs at a time).  It is asked for a kernel that has the same threads and shared memory.
__global__ void __launch_bounds__(192) cluster_room_kernel() {}

// Pieces per unit: as many as all units' clusters find room for at the same time, then as few as give the longest
// piece as many tiles.  Measured, us per launch with 4, 5, 6, 7, 8 pieces: 33 units of 58 tiles 47, 44, 38, 36, 34; of
// 10 tiles 17, 15, 14, 14, 15.5.
// *follow: bf16 holds the weight of a piece's reference exactly, so that the more pieces a unit has, the closer its outputs are
// to fp64.  Where split-K would cut shorter pieces than these, the references follow the rows' maxima instead (kClusterMax).  Error
// against fp64 of 8 sequences of 8191 tokens, logits of standard deviation 1, 2, 3, split-K / a fixed reference / this: 2.25e-3 /
// 2.32e-3 / 2.21e-3, 2.01e-3 / 2.17e-3 / 1.79e-3, 1.89e-3 / 2.00e-3 / 1.70e-3; us per launch 49.8 / 17.5 / 20.1.
// 0 where not even two fit, or where units of unlike length leave the longest piece too far above an even share of the
// launch's tiles (a cluster cuts every unit into the same number of pieces; split-K cuts the long ones into more).  Time of
// split-K, two launches with H2O, over this form, 32 layers in one launch, by the excess in tiles: without scores 4: 1.85, 7:
// 1.16, 10: 1.05 and 1.07, 15: 0.98, 40: 0.63; H2O 4: 1.63, 5: 1.10, 7: 1.17 (8 pieces), 1.06 and 0.92 (2 pieces: the less
// to merge, the less this form saves), 10: 0.95 and 0.96, 15: 0.85.  With references that follow the line falls with the pieces, by
// pieces and excess: without scores 2 pieces 4: 1.10, 5: 0.99, 6: 0.93; 3: 4: 1.01, 7: 0.93; 4: 5: 1.07, 6: 0.99, 8: 0.92; 5: 7: 1.18, 9:
// 1.05 and 0.97; 6: 6: 1.10, 8: 0.99; 8: 8: 1.30; H2O 2: 3: 1.06, 5: 0.97; 3: 4: 0.87; 4: 4: 1.09, 5: 0.95; 5: 5: 1.14, 7: 0.95; 6: 3: 1.12, 6: 0.98; 8:
// 4: 1.18 and 1.40, 8: 1.07.
// Launches of one layer, split-K / this form, us: 1 sequence of 4096 tokens 28.0 / 12.9, 16384: 84 / 25.5, 16 of 8191 35.6 / 22.6, 20 of 4000
// 29.5 / 16.4, 33 of 8191 32.3 / 24.3; H2O 1 of 16384 96 / 37.6, 8 of 8191 61 / 28.6, 33 of 8191 49.6 / 38.4, of 2457 34.4 / 20.0.
template <class Room>
static int cluster_pieces(const DecodeArgs& a, const int* desc_tiles, Room room, bool* follow) {
  const long long units = (long long)a.n_layer_total * a.n_unit;
  const auto [lo, hi] = std::minmax_element(desc_tiles, desc_tiles + a.n_layer_total);
  const int min_tiles = *lo, max_tiles = *hi;
  int n = most_ctas(std::min(kMaxPieces, min_tiles), units, room);
  if (n == 0) return 0;
  const int longest = (max_tiles + n - 1) / n;
  const long long total = std::accumulate(desc_tiles, desc_tiles + a.n_layer_total, 0LL) * a.n_unit;
  const long long even = std::max(total / (2LL * sm_count()), (long long)max_tiles / kMaxPieces);
  const bool h2o = a.policy == SQ_POLICY_H2O;
  *follow = longest * kTM > a.split_tokens;
  const int excess = *follow ? (h2o ? n : n + 2) : !h2o ? 12 : n == 2 ? 6 : 8;
  if (min_tiles < max_tiles && longest > even + excess) return 0;
  while (n > 2 && (max_tiles + n - 2) / (n - 1) == longest && units <= room(n - 1)) --n;
  return n;
}

template <bool H2O>
static cudaError_t launch_tc_cluster(const DecodeArgs& a, const int* desc_tiles, const CUtensorMap& tq, const CUtensorMap& tk,
                                     const CUtensorMap& tv, cudaStream_t s) {
  constexpr int STAGES = 3, ROWS = 120;
  constexpr size_t smem = 1024 + (size_t)ROWS * 128 + (size_t)2 * STAGES * kTileBytes + 8 * 16 + 16;
  auto kern = decode_attn_tc_kernel<STAGES, ROWS, H2O, kCluster, DecodeArgsBase>;
  auto kern_max = decode_attn_tc_kernel<STAGES, ROWS, H2O, kClusterMax, DecodeArgsBase>;
  const void* const all[3] = {reinterpret_cast<const void*>(cluster_room_kernel), reinterpret_cast<const void*>(kern),
                              reinterpret_cast<const void*>(kern_max)};
  static PerDevice set_up;
  const cudaError_t e = set_up.once([&] {
    cudaError_t r = cudaSuccess;
    for (const void* k : all) {
      if (r == cudaSuccess) r = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (r == cudaSuccess) r = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    }
    return r;
  });
  if (e != cudaSuccess) return e;
  static ClusterCount count[3];
  auto room = [&](int ctas) {  // (none of a size that the device does not hold for one of the kernels at all)
    int n = count[0].active(all[0], ctas, 192, smem);
    for (int k = 1; k < 3; ++k)
      if (count[k].active(all[k], ctas, 192, smem) == 0) n = 0;
    return n;
  };
  bool follow = false;
  const int n = cluster_pieces(a, desc_tiles, room, &follow);
  if (n == 0) return cudaErrorNotSupported;
  return launch_chained_cluster(follow ? kern_max : kern, n, a.n_layer_total * a.n_unit * n, 192, smem, s, tq, tk, tv,
                                static_cast<const DecodeArgsBase&>(a));
}

template <int STAGES, int ROWS, bool H2O>
static cudaError_t launch_tc_cfg(const DecodeArgs& a, int n_items, const CUtensorMap& tq, const CUtensorMap& tk,
                                 const CUtensorMap& tv, cudaStream_t s) {
  constexpr size_t smem = 1024 + (size_t)ROWS * 128 + (size_t)2 * STAGES * kTileBytes + 8 * 16 + 16;
  static_assert(2 * (smem + 1024 + 64) <= 228 * 1024, "two CTAs per SM");
  auto kern = decode_attn_tc_kernel<STAGES, ROWS, H2O, kSplitK, DecodeArgs>;
  static PerDevice set_up;
  const cudaError_t e = allow_smem(set_up, smem, kern);
  if (e != cudaSuccess) return e;
  return launch_chained(kern, n_items, 192, smem, s, tq, tk, tv, a);
}

static bool make_maps(const DecodeArgs& a, size_t pool_bytes, size_t q_rows, CUtensorMap* tm_q, CUtensorMap* tm_k, CUtensorMap* tm_v) {
  if (a.head_dim != kD || a.group <= 32 || a.group > 128) return false;
  const long long pool_rows = (long long)(pool_bytes / (kD * 2));
  if (pool_rows + kTM > 0x7fffffffLL || (long long)q_rows + kTM > 0x7fffffffLL) return false;
  return make_block_tile_map(tm_q, a.q, (long long)q_rows / a.group, a.group, kD, 8) && make_tile_map(tm_k, a.pool, pool_rows, kD, kTM) &&
         make_tile_map(tm_v, a.pool, pool_rows, kD, kTM);
}

// The cluster form.  desc_tiles: as for the even-deal form.  Returns cudaErrorNotSupported where it is not taken.
cudaError_t launch_decode_attn_tc_cluster(const DecodeArgs& a, const int* desc_tiles, size_t pool_bytes, size_t q_rows, cudaStream_t s) {
  if (a.group > kClusterHeads) return cudaErrorNotSupported;
  CUtensorMap tm_q, tm_k, tm_v;
  if (!make_maps(a, pool_bytes, q_rows, &tm_q, &tm_k, &tm_v)) return cudaErrorNotSupported;
  return a.policy == SQ_POLICY_H2O ? launch_tc_cluster<true>(a, desc_tiles, tm_q, tm_k, tm_v, s)
                                   : launch_tc_cluster<false>(a, desc_tiles, tm_q, tm_k, tm_v, s);
}

// Returns cudaErrorNotSupported when the shape is outside this kernel's range.
cudaError_t launch_decode_attn_tc(const DecodeArgs& a, int n_items, size_t pool_bytes, size_t q_rows, cudaStream_t s) {
  CUtensorMap tm_q, tm_k, tm_v;
  if (!make_maps(a, pool_bytes, q_rows, &tm_q, &tm_k, &tm_v)) return cudaErrorNotSupported;
  const bool h2o = a.policy == SQ_POLICY_H2O;
  if (a.group <= 96)
    return h2o ? launch_tc_cfg<3, 120, true>(a, n_items, tm_q, tm_k, tm_v, s)
               : launch_tc_cfg<3, 120, false>(a, n_items, tm_q, tm_k, tm_v, s);
  return h2o ? launch_tc_cfg<2, 128, true>(a, n_items, tm_q, tm_k, tm_v, s)
             : launch_tc_cfg<2, 128, false>(a, n_items, tm_q, tm_k, tm_v, s);
}

}  // namespace sq
