// Tensor-core decode attention for grouped / multi-query heads (bf16; groups of 9 and more, smaller ones in
// k_decode_mma_low.cu): with g query heads
// sharing a KV head the step is a dense [g x d] . [d x tokens] contraction (g flop per byte of
// K/V), too much for the fp32 pipes at HBM speed once g >= 4.  The g heads of a unit are
// padded to 16-row tiles and run through mma.sync m16n8k16 (bf16 in, fp32 accumulate):
//   S = Q K^T   (K tile in shared memory, B operand through ldmatrix)
//   O += P V    (P = exp2(S*scale - max) re-used from the S accumulators as the A operand,
//                V tile through ldmatrix.trans)
// K/V tiles of 64 tokens stream through a multi-stage cp.async pipeline (16-byte copies,
// XOR-swizzled rows so ldmatrix is bank-conflict free).  Warps split the tile's tokens (WN)
// and, for very wide groups, the head tiles (WM); partial results merge through shared memory.
#include <algorithm>

#include "sq_decode_common.cuh"
#include "sq_device.cuh"
#include "sq_internal.h"
#include "sq_mma.cuh"
#include "sq_scores.cuh"

namespace sq {

// SCORES: H2O with the score update in the same launch (sq_scores.cuh): the pieces of a unit are the
// CTAs of a cluster, piece_tiles(len) tiles each, and the logits stay in shared memory.
template <int D, int MT, int WM, int WN, int STAGES, bool SCORES, class Args>
__global__ void __launch_bounds__(32 * WM * WN) decode_attn_mma_kernel(Args a) {
  constexpr int NT = 32 * WM * WN;
  constexpr int CH = D / 8;            // 16-byte chunks per row
  constexpr int KS = D / 16;           // k-steps of Q K^T / pairs of output n-blocks
  constexpr int NB = D / 8;            // output n-blocks of 8 columns
  constexpr int QROWS = WM * MT * 16;  // padded head rows
  constexpr int TILE_BYTES = kTile * D * 2;
  static_assert(kTile / WN == 16, "each warp owns 16 tokens of a tile");
  using bf16 = __nv_bfloat16;
  extern __shared__ __align__(128) unsigned char smem[];
  // Q is read into registers before the last stage is filled for the first time: with SCORES, which
  // needs the room, it starts out there
  static_assert(!SCORES || QROWS * D * 2 <= TILE_BYTES, "Q in a stage");
  unsigned char* k_s = smem + (SCORES ? 0 : QROWS * D * 2);
  unsigned char* v_s = k_s + STAGES * TILE_BYTES;
  unsigned char* q_s = SCORES ? k_s + (STAGES - 1) * TILE_BYTES : smem;

  ItemLoc it;
  int split;
  if constexpr (SCORES) {
    const int c = cluster_size(), item = blockIdx.x / c;
    const int k = item / a.n_unit;
    it.layer = a.order[k];
    it.n_split = 1;
    it.base = 0;
    it.local = item - k * a.n_unit;
    split = cluster_rank();
  } else {
    if (!locate(a, blockIdx.x, it)) return;
  }
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = warp / WN, wn = warp % WN;
  const int gq = lane >> 2, tq = lane & 3;
  const LayerDesc* ldp = a.layers + it.layer;
  const int b = ldp->b, cap = ldp->cap, G = a.group;
  const int unit = it.local / it.n_split;
  const int len = min(a.n_tok + 1, b);
  const bool h2o = SCORES || (a.policy == SQ_POLICY_H2O);
  int piece_tokens;
  if constexpr (SCORES) {
    piece_tokens = piece_tiles(len, cluster_size()) * kTile;
  } else {
    split = it.local - unit * it.n_split;
    piece_tokens = a.split_tokens;
  }
  if (!a.early) grid_wait();
  int w;
  if (h2o) {
    w = (a.n_tok < b) ? a.n_tok : __ldcg(reinterpret_cast<const int*>(a.pool + ldp->victim_off) + unit);
    if (w < 0 || w >= b) {
      if (tid == 0) atomicOr(a.status, 2);
      w = 0;
    }
  } else {
    w = ring_slot(a.n_tok, b, ldp->ring_base, ldp->ring_origin);
  }
  const int t0 = split * piece_tokens, t1 = min(len, t0 + piece_tokens);  // (a piece may be empty under SCORES)
  const int seq = unit / a.n_kv_head, kvh = unit - seq * a.n_kv_head;
  const size_t tok = (size_t)(it.layer - a.layer_begin) * a.batch + seq;
  bf16* Kb = reinterpret_cast<bf16*>(a.pool + ldp->k_off) + (size_t)unit * cap * D;
  bf16* Vb = reinterpret_cast<bf16*>(a.pool + ldp->v_off) + (size_t)unit * cap * D;
  const bf16* qb = reinterpret_cast<const bf16*>(a.q) + (tok * a.n_q_head + (size_t)kvh * G) * D;
  const bf16* kn = reinterpret_cast<const bf16*>(a.k_new) + (tok * a.n_kv_head + kvh) * D;
  const bf16* vn = reinterpret_cast<const bf16*>(a.v_new) + (tok * a.n_kv_head + kvh) * D;
  bf16* ob = reinterpret_cast<bf16*>(a.out) + (tok * a.n_q_head + (size_t)kvh * G) * D;
  float* logit;  // [token][G]
  if constexpr (SCORES) logit = reinterpret_cast<float*>(smem + 2 * STAGES * TILE_BYTES) - (size_t)t0 * G;
  else logit = a.logits + ldp->logit_off + (size_t)unit * cap * G;
  float* stat = a.part_stat + (size_t)blockIdx.x * G * kStatStride;  // (unused under SCORES)
  float* po = a.part_o + (size_t)blockIdx.x * G * D;

  const int n_tiles = (t1 - t0 + kTile - 1) / kTile;
  // `skip`: a row that is left out (the new token's, in the tiles fetched before it is in the cache)
  auto load_tile = [&](int tile, int skip) {
    if (tile < n_tiles) {
      const int stage = tile % STAGES;
      const int row0 = t0 + tile * kTile;
      const uint32_t kdst = smem_u32(k_s + stage * TILE_BYTES), vdst = smem_u32(v_s + stage * TILE_BYTES);
      for (int i = tid; i < kTile * CH; i += NT) {
        const int r = i / CH, c = i - r * CH;
        if (row0 + r == skip) continue;
        const bool ok = row0 + r < t1;
        const size_t src = (size_t)(ok ? row0 + r : t0) * D + c * 8;
        const uint32_t off = swz<D>(r, c);
        cp_async16(kdst + off, Kb + src, ok);
        cp_async16(vdst + off, Vb + src, ok);
      }
    }
    cp_async_commit();
  };
  // The first tiles of the cache, but for the new token's row, are under way before the launch ahead
  // is done (a.early) and before q is read.
#pragma unroll
  for (int s = 0; s < STAGES - 1; ++s) load_tile(s, w);
  if (a.early) grid_wait();

  // the CTA whose range holds slot w stores the new token: in the cache, where later tiles read it
  // like any other row, and in the tile already fetched around it
  if (w >= t0 && w < t1) {
    if (tid < 2 * CH) {
      const bool is_v = tid >= CH;
      const int c = is_v ? tid - CH : tid;
      const uint4 val = *reinterpret_cast<const uint4*>((is_v ? vn : kn) + c * 8);
      *reinterpret_cast<uint4*>((is_v ? Vb : Kb) + (size_t)w * D + c * 8) = val;
      const int tile = (w - t0) / kTile;
      if (tile < STAGES - 1)
        *reinterpret_cast<uint4*>((is_v ? v_s : k_s) + tile * TILE_BYTES + swz<D>((w - t0) % kTile, c)) = val;
    }
    if (tid == 2 * CH) {
      reinterpret_cast<int*>(a.pool + ldp->pos_off)[(size_t)unit * cap + w] = a.n_tok;
      if (h2o) reinterpret_cast<float*>(a.pool + ldp->acc_off)[(size_t)unit * cap + w] = 0.f;
    }
    __threadfence_block();
  }
  // query rows (zero beyond the group) into shared memory
  for (int i = tid; i < QROWS * CH; i += NT) {
    const int row = i / CH, c = i - row * CH;
    uint4 val = make_uint4(0, 0, 0, 0);
    if (row < G) val = *reinterpret_cast<const uint4*>(qb + (size_t)row * D + c * 8);
    *reinterpret_cast<uint4*>(q_s + swz<D>(row, c)) = val;
  }
  __syncthreads();

  // A fragments of Q, kept for the whole item
  uint32_t qa[MT][KS][4];
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) {
    const int mi = lane >> 3, r = lane & 7;
    const int row = (wm * MT + mt) * 16 + (mi & 1) * 8 + r;
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
      ldmatrix_x4(smem_u32(q_s + swz<D>(row, 2 * ks + (mi >> 1))), qa[mt][ks][0], qa[mt][ks][1], qa[mt][ks][2],
                  qa[mt][ks][3]);
  }
  float o[MT][NB][4];
  float m_run[MT][2], l_true[MT][2], l_w[MT][2];
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) {
#pragma unroll
    for (int nb = 0; nb < NB; ++nb)
#pragma unroll
      for (int j = 0; j < 4; ++j) o[mt][nb][j] = 0.f;
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      m_run[mt][hf] = -INFINITY;
      l_true[mt][hf] = 0.f;
      l_w[mt][hf] = 0.f;
    }
  }

  for (int tile = 0; tile < n_tiles; ++tile) {
    cp_async_wait<STAGES - 2>();
    __syncthreads();
    load_tile(tile + STAGES - 1, -1);
    const int stage = tile % STAGES;
    const uint32_t kst = smem_u32(k_s + stage * TILE_BYTES), vst = smem_u32(v_s + stage * TILE_BYTES);
    const int tok0 = t0 + tile * kTile + wn * 16;  // first token of this warp's 16
    if (tok0 >= t1) continue;                      // warp-uniform: nothing of this tile is ours

    // ---- S = Q K^T over the warp's 16 tokens (two 8-token blocks) ----
    float s[MT][2][4];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
      for (int nb = 0; nb < 2; ++nb)
#pragma unroll
        for (int j = 0; j < 4; ++j) s[mt][nb][j] = 0.f;
    {
      const int mi = lane >> 3, r = lane & 7;
      const int trow = wn * 16 + (mi >> 1) * 8 + r;
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        uint32_t b0, b1, b2, b3;
        ldmatrix_x4(kst + swz<D>(trow, 2 * ks + (mi & 1)), b0, b1, b2, b3);
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
          if ((wm * MT + mt) * 16 < G) {
            mma_bf16(s[mt][0], qa[mt][ks], b0, b1);
            mma_bf16(s[mt][1], qa[mt][ks], b2, b3);
          }
        }
      }
    }
    // ---- online softmax in the log2 domain; P packed to bf16 as the next A operand ----
    uint32_t pa[MT][4];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        float v[4];
#pragma unroll
        for (int nb = 0; nb < 2; ++nb)
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const int t = tok0 + nb * 8 + 2 * tq + j;
            v[nb * 2 + j] = (t < t1) ? s[mt][nb][hf * 2 + j] * a.scale_log2 : -INFINITY;
          }
        if (h2o) {
          const int h = (wm * MT + mt) * 16 + hf * 8 + gq;
          if (h < G) {
#pragma unroll
            for (int nb = 0; nb < 2; ++nb)
#pragma unroll
              for (int j = 0; j < 2; ++j) {
                const int t = tok0 + nb * 8 + 2 * tq + j;
                if (t < t1) logit[(size_t)t * G + h] = v[nb * 2 + j];
              }
          }
        }
        float mx = fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3]));
        mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, 2));
        const float m_new = fmaxf(m_run[mt][hf], mx);  // finite: token tok0 is valid
        const float corr = exp2f(m_run[mt][hf] - m_new);
        m_run[mt][hf] = m_new;
        float p[4], pr[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) p[j] = exp2f(v[j] - m_new);
        pa[mt][hf] = pack_bf16(p[0], p[1], pr[0], pr[1]);      // tokens 0-7 of the 16
        pa[mt][hf + 2] = pack_bf16(p[2], p[3], pr[2], pr[3]);  // tokens 8-15
        l_true[mt][hf] = l_true[mt][hf] * corr + ((p[0] + p[1]) + (p[2] + p[3]));
        l_w[mt][hf] = l_w[mt][hf] * corr + ((pr[0] + pr[1]) + (pr[2] + pr[3]));
#pragma unroll
        for (int nb = 0; nb < NB; ++nb) {
          o[mt][nb][hf * 2] *= corr;
          o[mt][nb][hf * 2 + 1] *= corr;
        }
      }
    }
    // ---- O += P V ----
    {
      const int mi = lane >> 3, r = lane & 7;
      const int trow = wn * 16 + (mi & 1) * 8 + r;
#pragma unroll
      for (int nb2 = 0; nb2 < KS; ++nb2) {
        uint32_t b0, b1, b2, b3;
        ldmatrix_x4_trans(vst + swz<D>(trow, 2 * nb2 + (mi >> 1)), b0, b1, b2, b3);
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
          if ((wm * MT + mt) * 16 < G) {
            mma_bf16(o[mt][2 * nb2], pa[mt], b0, b1);
            mma_bf16(o[mt][2 * nb2 + 1], pa[mt], b2, b3);
          }
        }
      }
    }
  }
  cp_async_wait<0>();
  // sums over the four lanes that share a row
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      l_true[mt][hf] += __shfl_xor_sync(kFull, l_true[mt][hf], 1);
      l_true[mt][hf] += __shfl_xor_sync(kFull, l_true[mt][hf], 2);
      l_w[mt][hf] += __shfl_xor_sync(kFull, l_w[mt][hf], 1);
      l_w[mt][hf] += __shfl_xor_sync(kFull, l_w[mt][hf], 2);
    }
  ScoreAhead ahead;
  if constexpr (SCORES)
    fetch_scores<NT>(ahead, reinterpret_cast<const float*>(a.pool + ldp->acc_off) + (size_t)unit * cap,
                     reinterpret_cast<const int*>(a.pool + ldp->pos_off) + (size_t)unit * cap, t0 + tid, t1, len == b);
  __syncthreads();  // the pipeline buffers are free: reuse them for the merge

  // ---- merge the WN token groups (tree over shared memory) ----
  constexpr int SLOT_FLOATS = MT * 16 * (D + 4);
  float* mg = reinterpret_cast<float*>(k_s);
#pragma unroll
  for (int stride = WN / 2; stride >= 1; stride >>= 1) {
    float* slot = mg + (size_t)(wm * (WN / 2) + (wn % stride)) * SLOT_FLOATS;
    if (wn >= stride && wn < 2 * stride) {
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          float* row = slot + (size_t)(mt * 16 + hf * 8 + gq) * (D + 4);
#pragma unroll
          for (int nb = 0; nb < NB; ++nb)
            *reinterpret_cast<float2*>(row + nb * 8 + 2 * tq) = make_float2(o[mt][nb][hf * 2], o[mt][nb][hf * 2 + 1]);
          if (tq == 0) {
            row[D] = m_run[mt][hf];
            row[D + 1] = l_true[mt][hf];
            row[D + 2] = l_w[mt][hf];
          }
        }
    }
    __syncthreads();
    if (wn < stride) {
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          const float* row = slot + (size_t)(mt * 16 + hf * 8 + gq) * (D + 4);
          const float m2 = row[D], m1 = m_run[mt][hf];
          const float mx = fmaxf(m1, m2);
          const float f1 = (m1 > -INFINITY) ? exp2f(m1 - mx) : 0.f;
          const float f2 = (m2 > -INFINITY) ? exp2f(m2 - mx) : 0.f;
          m_run[mt][hf] = mx;
          l_true[mt][hf] = l_true[mt][hf] * f1 + row[D + 1] * f2;
          l_w[mt][hf] = l_w[mt][hf] * f1 + row[D + 2] * f2;
#pragma unroll
          for (int nb = 0; nb < NB; ++nb) {
            const float2 o2 = *reinterpret_cast<const float2*>(row + nb * 8 + 2 * tq);
            o[mt][nb][hf * 2] = o[mt][nb][hf * 2] * f1 + o2.x * f2;
            o[mt][nb][hf * 2 + 1] = o[mt][nb][hf * 2 + 1] * f1 + o2.y * f2;
          }
        }
    }
    __syncthreads();
  }
  if constexpr (SCORES) {
    // the piece's partial and the scratch of the update in shared memory, past the merge area
    static_assert(WM == 1, "one row of warps");
    float* part_o = reinterpret_cast<float*>(v_s);
    float* part_stat = part_o + MT * 16 * D;
    ScoreShared<kMaxPieces>& sh = *reinterpret_cast<ScoreShared<kMaxPieces>*>(part_stat + MT * 16 * 4);
    static_assert(MT * 16 * (D + 4) * 4 + sizeof(sh) <= STAGES * TILE_BYTES, "partial area");
    if (wn == 0) {
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          const int h = mt * 16 + hf * 8 + gq;
          if (h >= G) continue;
#pragma unroll
          for (int nb = 0; nb < NB; ++nb)
            *reinterpret_cast<float2*>(part_o + h * D + nb * 8 + 2 * tq) = make_float2(o[mt][nb][hf * 2], o[mt][nb][hf * 2 + 1]);
          if (tq == 0) *reinterpret_cast<float4*>(part_stat + h * 4) = make_float4(m_run[mt][hf], l_true[mt][hf], l_w[mt][hf], 0.f);
        }
    }
    finish_scores<bf16, D, NT, kMaxPieces>(a, ldp, unit, t0, t1, len, ob, logit + (size_t)t0 * G, part_o, part_stat, sh, &ahead, w);
    return;
  }
  if (wn == 0) {
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      const int h = (wm * MT + mt) * 16 + hf * 8 + gq;
      if (h >= G) continue;
      if (it.n_split == 1) {
        const float inv = 1.f / l_w[mt][hf];
#pragma unroll
        for (int nb = 0; nb < NB; ++nb)
          *reinterpret_cast<__nv_bfloat162*>(ob + (size_t)h * D + nb * 8 + 2 * tq) =
              __floats2bfloat162_rn(o[mt][nb][hf * 2] * inv, o[mt][nb][hf * 2 + 1] * inv);
      } else {
#pragma unroll
        for (int nb = 0; nb < NB; ++nb)
          *reinterpret_cast<float2*>(po + (size_t)h * D + nb * 8 + 2 * tq) =
              make_float2(o[mt][nb][hf * 2], o[mt][nb][hf * 2 + 1]);
      }
      if (tq == 0) {
        stat[h * kStatStride] = m_run[mt][hf];
        stat[h * kStatStride + 1] = l_true[mt][hf];
        stat[h * kStatStride + 2] = l_w[mt][hf];
      }
    }
  }
  if (!h2o && it.n_split > 1) merge_if_last<bf16>(a, it, unit, reinterpret_cast<float*>(k_s));
}

template <int D, int MT, int WM, int WN, int STAGES>
static cudaError_t launch_cfg(const DecodeArgs& a, int n_items, cudaStream_t s) {
  constexpr int QROWS = WM * MT * 16;
  constexpr size_t pipe = (size_t)2 * STAGES * kTile * D * 2;
  constexpr size_t merge = (size_t)WM * (WN / 2) * MT * 16 * (D + 4) * 4;
  static_assert(merge <= pipe, "the merge area reuses the pipeline stages");
  constexpr size_t smem = (size_t)QROWS * D * 2 + pipe;
  auto kern = decode_attn_mma_kernel<D, MT, WM, WN, STAGES, false, DecodeArgs>;
  static PerDevice set_up;
  const cudaError_t e = allow_smem(set_up, smem, kern);
  if (e != cudaSuccess) return e;
  return launch_chained(kern, n_items, 32 * WM * WN, smem, s, a);
}

template <int D, int MT, int STAGES>
static cudaError_t launch_scores_cfg(const DecodeArgs& a, int pieces, size_t logit_bytes, cudaStream_t s) {
  const size_t smem = (size_t)2 * STAGES * kTile * D * 2 + logit_bytes;
  auto kern = decode_attn_mma_kernel<D, MT, 1, 4, STAGES, true, DecodeArgsBase>;
  static PerDevice set_up;
  const cudaError_t e = set_up.once([&] {
    const cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kScoresSmem);
    return r == cudaSuccess ? cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) : r;
  });
  if (e != cudaSuccess) return e;
  static ClusterFit wide;
  if (pieces > 8 && !wide.fits(reinterpret_cast<const void*>(kern), kMaxPieces, 128, kScoresSmem)) return cudaErrorNotSupported;
  return launch_chained_cluster(kern, pieces, a.n_layer_total * a.n_unit * pieces, 128, smem, s, static_cast<const DecodeArgsBase&>(a));
}

// H2O with the score update in the launch.  max_len: slots of the longest unit.  Returns
// cudaErrorNotSupported where the second launch (decode_combine_kernel, h2o_update_warp_kernel) is the
// better form or the logits of a piece do not fit.  The better form it is for launches of more CTAs than are resident at
// once, unless the pieces are equal (one layer, or few units) or the group is small and its pieces are short (one per
// unit) or long: all units are cut into the same number of pieces, which for short layers beside long ones, and
// where the logits ask for more pieces than the launch does, are too small.  us per token, second launch / this form, 8
// layers: one launch, 64 sequences of 1500 tokens, 32 / 1 heads of 64 99 / 163, 16 / 1 56 / 85; 8 of 1500, 64 / 8 heads of 128 76 /
// 97; 16 of 100, 32 / 1 of 128 19 / 24; 8 of 1500, 32 / 1 of 64 45 / 24; one launch per layer, 64 of 1500, 20 / 1 244 / 127, 64 / 8 514
// / 637.
// Pieces: as many as leave all CTAs resident at once (two per SM), a tile or more each; up to 16 where few
// clusters of that size are enough (more of them do not all fit at once beside smaller ones).  Measured, us
// per token of 32 layers of 32 / 8 heads of 128, one launch per layer, second launch / this form: 1 sequence
// 385 / 266 (at most eight pieces of two tiles or more: 281), its 16384-token caches 1309 / 560 (their
// logits do not fit eight pieces: 1138), 4: 451 / 358, 16: 660 / 534 (four pieces per unit, more than fit at
// once: 629), 64: 1060 / 983; 20 / 1 heads of 64, 64 sequences: 435 / 237; 80 layers of 64 / 8 heads, 4 sequences:
// 1372 / 859.  All 32 layers in one launch, 4096 units: 322 / 446.  (With the kernel for up to 8 heads
// k_decode_mma_low.cu gives 1 sequence 231, 4: 309, 16: 480, 64: 877.)
cudaError_t launch_decode_mma_scores(const DecodeArgs& a, int max_len, cudaStream_t s) {
  const int G = a.group;
  if (G > 32 || (a.head_dim != 64 && a.head_dim != 128)) return cudaErrorNotSupported;
  const int n_sm = sm_count();
  const long long units = (long long)a.n_layer_total * a.n_unit;
  if (units >= 6 * n_sm) return cudaErrorNotSupported;
  const int tiles = (max_len + kTile - 1) / kTile;
  const int stages = a.head_dim == 128 ? 3 : 4;
  const size_t fixed = (size_t)2 * stages * kTile * a.head_dim * 2;
  auto logit_bytes = [&](int p) { return (size_t)piece_tiles(max_len, p) * kTile * G * 4; };
  auto launch = [&](int limit) {
    const int wanted = (int)std::min<long long>({limit, std::max<long long>(1, 2 * n_sm / units), tiles});
    int pieces = wanted;
    while (pieces < 8 && fixed + logit_bytes(pieces) > kScoresSmem) ++pieces;
    const size_t lb = logit_bytes(pieces);
    if (fixed + lb > kScoresSmem) return cudaErrorNotSupported;
    const long long ctas = units * pieces;
    // (one head of 64: the fp32-pipe kernel and a second launch, see one_head_on_pipe())
    if (G == 1 && a.head_dim == 64 && a.n_layer_total > 1 && units > n_sm && max_len > 2048) return cudaErrorNotSupported;
    if (ctas > 2 * n_sm) {  // more than one wave
      if (pieces > wanted && piece_tiles(max_len, pieces) == 1) return cudaErrorNotSupported;
      const int len = max_len / pieces;
      const bool even = units <= n_sm || a.n_layer_total == 1;
      const bool low = G <= 4 && ((pieces == 1 && len <= 2432 && ctas <= 4 * n_sm) || (len >= 2560 && len <= 5120 && ctas <= 12 * n_sm));
      if (!(even && ctas <= 7 * n_sm) && !low) return cudaErrorNotSupported;
    }
    if (G <= 8) return launch_decode_mma_low(a, 0, pieces, lb, s);
    if (a.head_dim == 128) return G <= 16 ? launch_scores_cfg<128, 1, 3>(a, pieces, lb, s) : launch_scores_cfg<128, 2, 3>(a, pieces, lb, s);
    return G <= 16 ? launch_scores_cfg<64, 1, 4>(a, pieces, lb, s) : launch_scores_cfg<64, 2, 4>(a, pieces, lb, s);
  };
  return with_portable_clusters(units <= 16 ? kMaxPieces : 8, launch);
}

// Returns cudaErrorNotSupported when no tensor-core configuration covers the shape.
cudaError_t launch_decode_attn_mma(const DecodeArgs& a, int n_items, cudaStream_t s) {
  const int G = a.group;
  if (G <= 8 && (a.head_dim == 64 || a.head_dim == 128)) return launch_decode_mma_low(a, n_items, 0, 0, s);
  if (a.head_dim == 128) {
    // Two stages of 32 KB let three CTAs share an SM, which wins once the launch has CTAs to
    // spare (measured: Mistral- and Llama-2-70B-shaped fused steps 5-9 % faster); a launch of
    // about one wave (one layer at a time) is better off with the deeper ring per CTA.
    const bool many = n_items >= 6 * sm_count();
    if (G <= 16) return many ? launch_cfg<128, 1, 1, 4, 2>(a, n_items, s) : launch_cfg<128, 1, 1, 4, 3>(a, n_items, s);
    if (G <= 32) return many ? launch_cfg<128, 2, 1, 4, 2>(a, n_items, s) : launch_cfg<128, 2, 1, 4, 3>(a, n_items, s);
  } else if (a.head_dim == 64) {
    if (G <= 16) return launch_cfg<64, 1, 1, 4, 4>(a, n_items, s);
    if (G <= 32) return launch_cfg<64, 2, 1, 4, 4>(a, n_items, s);
    if (G <= 96) return launch_cfg<64, 3, 2, 4, 4>(a, n_items, s);
  }
  return cudaErrorNotSupported;
}

}  // namespace sq
