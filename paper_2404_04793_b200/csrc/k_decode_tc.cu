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
// Streaming K and V alone (no products, no softmax) reaches 7.3 TB/s and draws 970 W of the
// board's 1000 W; with the products 6.4 TB/s, with the softmax as well 4.6-4.7 TB/s, both at the
// power limit with the SM clock near 1.5-1.6 GHz: run for longer than a few milliseconds the
// kernel is bound by power, and what helps is fewer instructions per weight.
#include <type_traits>

#include "sq_decode_common.cuh"
#include "sq_device.cuh"
#include "sq_internal.h"
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
}  // namespace

// ROWS: rows of the Q tile held in shared memory (120 for up to 96 heads, else 128; see sq_tc_rows.cuh).
template <int STAGES, int ROWS, bool H2O>
__global__ void __launch_bounds__(192, 2)
    decode_attn_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                          const __grid_constant__ CUtensorMap tm_v, DecodeArgs a) {
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
  static_assert(6 + 2 * STAGES <= 16, "barrier block");
  const uint32_t bar_q = s_u32(bars + 0), bar_odone = s_u32(bars + 1), bar_sfull = s_u32(bars + 2),
                 bar_sfree = s_u32(bars + 3), bar_pready = s_u32(bars + 4), bar_pfree = s_u32(bars + 5);
  auto bar_full = [&](int s) { return s_u32(bars + 6 + s); };
  auto bar_empty = [&](int s) { return s_u32(bars + 6 + STAGES + s); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 16);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  ItemLoc it;
  if (!locate(a, blockIdx.x, it)) return;
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
  const int t0 = split * a.split_tokens, t1 = min(len, t0 + a.split_tokens);
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
  const WideLayout layout;

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
      tma_load_2d(s_u32(q_s + layout.row_of_group(lane) * 128), &tm_q, 0, (int)(tok * a.n_q_head + (size_t)kvh * G) + 8 * lane, bar_q);
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
      bool s_released = rows.tile(n_valid, i == 0, bar_sfree, [&]() {
        if (i >= 1) ok = __all_sync(0xffffffffu, mbar_wait(bar_pfree, (i - 1) & 1, abort_flag));
      });
      if (!ok) break;
      if (rows.too_large()) {
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
        if (!live) continue;
        if (it.n_split == 1) {
#pragma unroll
          for (int q4 = 0; q4 < 4; ++q4)
            *reinterpret_cast<uint4*>(ob + (size_t)row * kD + c * 32 + q4 * 8) =
                make_uint4(pack_bf16x2(o[q4 * 8] * inv, o[q4 * 8 + 1] * inv), pack_bf16x2(o[q4 * 8 + 2] * inv, o[q4 * 8 + 3] * inv),
                           pack_bf16x2(o[q4 * 8 + 4] * inv, o[q4 * 8 + 5] * inv), pack_bf16x2(o[q4 * 8 + 6] * inv, o[q4 * 8 + 7] * inv));
        } else {
#pragma unroll
          for (int q4 = 0; q4 < 8; ++q4)
            *reinterpret_cast<float4*>(po + (size_t)row * kD + c * 32 + q4 * 4) =
                make_float4(o[q4 * 4], o[q4 * 4 + 1], o[q4 * 4 + 2], o[q4 * 4 + 3]);
        }
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
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "n"(kTmemCols) : "memory");
  }
  if (tid == 0 && *abort_flag) atomicOr(a.status, kStatusTimeout);
  if (it.n_split > 1) merge_if_last<bf16>(a, it, unit, reinterpret_cast<float*>(q_s), H2O ? a.logits + ldp->lse_off + (size_t)unit * G : nullptr);
}

template <int STAGES, int ROWS, bool H2O>
static cudaError_t launch_tc_cfg(const DecodeArgs& a, int n_items, const CUtensorMap& tq, const CUtensorMap& tk,
                                 const CUtensorMap& tv, cudaStream_t s) {
  constexpr size_t smem = 1024 + (size_t)ROWS * 128 + (size_t)2 * STAGES * kTileBytes + 8 * 16 + 16;
  static_assert(2 * (smem + 1024 + 64) <= 228 * 1024, "two CTAs per SM");
  auto kern = decode_attn_tc_kernel<STAGES, ROWS, H2O>;
  static PerDevice set_up;
  const cudaError_t e = allow_smem(set_up, smem, kern);
  if (e != cudaSuccess) return e;
  return launch_chained(kern, n_items, 192, smem, s, tq, tk, tv, a);
}

// Returns cudaErrorNotSupported when the shape is outside this kernel's range.
cudaError_t launch_decode_attn_tc(const DecodeArgs& a, int n_items, size_t pool_bytes, size_t q_rows, cudaStream_t s) {
  if (a.head_dim != kD || a.group <= 32 || a.group > 128) return cudaErrorNotSupported;
  const long long pool_rows = (long long)(pool_bytes / (kD * 2));
  if (pool_rows + kTM > 0x7fffffffLL || (long long)q_rows + kTM > 0x7fffffffLL) return cudaErrorNotSupported;
  CUtensorMap tm_q, tm_k, tm_v;
  if (!make_tile_map(&tm_q, a.q, (long long)q_rows, kD, 8) || !make_tile_map(&tm_k, a.pool, pool_rows, kD, kTM) ||
      !make_tile_map(&tm_v, a.pool, pool_rows, kD, kTM))
    return cudaErrorNotSupported;
  const bool h2o = a.policy == SQ_POLICY_H2O;
  if (a.group <= 96)
    return h2o ? launch_tc_cfg<3, 120, true>(a, n_items, tm_q, tm_k, tm_v, s)
               : launch_tc_cfg<3, 120, false>(a, n_items, tm_q, tm_k, tm_v, s);
  return h2o ? launch_tc_cfg<2, 128, true>(a, n_items, tm_q, tm_k, tm_v, s)
             : launch_tc_cfg<2, 128, false>(a, n_items, tm_q, tm_k, tm_v, s);
}

}  // namespace sq
