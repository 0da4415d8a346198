// Tensor-core decode attention for 1..8 bf16 query heads per KV head (mma.sync m16n8k16).  The heads are the
// N side of both products, so no row of a tile is padding (k_decode_mma.cu has them on the M side, 16 rows at
// a time):
//   S^T[16 tokens x 8 heads] = K Q^T      (K rows as the A operand, Q as B, kept in registers)
//   O^T[D x 8 heads]        += V^T P^T    (V through ldmatrix.trans as A; P^T is S^T turned by movmatrix)
// A warp owns 16 of a tile's 64 tokens.  What bounds a CTA is the chain per tile (wait, products, softmax,
// products; two or three CTAs per SM hide it), so the chain is kept short: a head's reference is the maximum of the
// warp's first tile and moves only when a weight would pass 2^16 (no reduction or rescaling per tile), and a
// full tile is fetched with constant strides.
// Measured, us per token, heads on the M side / this: 80 layers of 64 / 8 heads of 128, one launch per layer, 32
// sequences 2371 / 2109, 4: 933 / 784; 32 layers of 32 / 8 heads, 16 sequences 489 / 407, H2O 535 / 480, 1 sequence
// 264 / 212, H2O 265 / 231; all layers in one launch, 37 sequences with their own budgets 272 / 226.
#include <algorithm>

#include "sq_decode_common.cuh"
#include "sq_device.cuh"
#include "sq_internal.h"
#include "sq_mma.cuh"
#include "sq_scores.cuh"

namespace sq {

// SCORES: H2O with the score update in the same launch (sq_scores.cuh): the pieces of a unit are the CTAs of
// a cluster and the logits stay in shared memory.
// A reference that stays leaves the largest weight anywhere up to 2^16, where a running maximum makes it 1, exact in
// bf16.  So a weight enters the second product as a sum of bf16 numbers, and the normaliser is the sum of the
// fp32 weights.  HEADS: 1: three parts (fp32 precision), in the columns 0, 1, 2 of P^T; 4: up to four heads, two parts, head h in
// the columns h and h + 4; 8: two parts, the second by a product of its own.  Error of the outputs against fp64 (2-norm; bf16 rounding
// of the outputs alone gives 1.66e-3), 32 / 8 heads of 128, caches of 5000: one part under a running maximum 1.73e-3, one
// under a fixed reference 2.20e-3, two 1.67e-3 (80 layers of 64 / 8 heads, 32 sequences: 2142 us per token with one, 2164 with two).
template <int D, int STAGES, bool SCORES, int HEADS, class Args>
__global__ void __launch_bounds__(128) decode_attn_mma_low_kernel(Args a) {
  constexpr int NT = 128, WN = 4, NH = 8;
  constexpr int CH = D / 8;              // 16-byte chunks per row
  constexpr int KS = D / 16;             // k-steps of K Q^T = 16-row blocks of O^T
  constexpr int RPP = NT / CH;           // rows of a tile that the CTA fetches at a time
  constexpr int TILE_BYTES = kTile * D * 2;
  constexpr int SLOT = NH * (D + 4);     // a warp's result: [head][D], its maximum and sums
  static_assert(kTile / WN == 16 && RPP % 8 == 0, "tile split");
  using bf16 = __nv_bfloat16;
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char* k_s = smem;
  unsigned char* v_s = k_s + STAGES * TILE_BYTES;
  // Q is read into registers before the last stage is filled for the first time: it starts out there
  unsigned char* q_s = k_s + (STAGES - 1) * TILE_BYTES;

  ItemLoc it;
  int split, n_split;
  if constexpr (SCORES) {
    n_split = cluster_size();
    const int item = blockIdx.x / n_split, k = item / a.n_unit;
    it.layer = a.order[k];
    it.n_split = 1;
    it.base = 0;
    it.local = item - k * a.n_unit;
    split = cluster_rank();
  } else {
    if (!locate(a, blockIdx.x, it)) return;
    n_split = it.n_split;
  }
  const int tid = threadIdx.x, lane = tid & 31, wn = tid >> 5;
  const int gq = lane >> 2, tq = lane & 3, mi = lane >> 3, r8 = lane & 7;
  const LayerDesc* ldp = a.layers + it.layer;
  const int b = ldp->b, cap = ldp->cap, G = a.group;
  const int unit = it.local / it.n_split;
  const int len = min(a.n_tok + 1, b);
  const bool h2o = SCORES || (a.policy == SQ_POLICY_H2O);
  int piece_tokens;
  if constexpr (SCORES) {
    piece_tokens = piece_tiles(len, n_split) * kTile;
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
  const int n_tiles = (t1 - t0 + kTile - 1) / kTile;
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

  // this thread's chunk of row tid / CH of a tile, then of every RPP-th row after it
  const int my_row = tid / CH, my_c = tid - my_row * CH;
  const uint32_t my_off = swz<D>(my_row, my_c);
  const size_t my_src = (size_t)(t0 + my_row) * D + my_c * 8;
  // `skip`: a row that is left out (the new token's, in the tiles fetched before it is in the cache)
  auto load_tile = [&](int tile, int skip) {
    if (tile < n_tiles) {
      const int stage = tile % STAGES, row0 = t0 + tile * kTile;
      const uint32_t kdst = smem_u32(k_s) + stage * TILE_BYTES + my_off, vdst = smem_u32(v_s) + stage * TILE_BYTES + my_off;
      const bf16 *ks = Kb + my_src + (size_t)tile * kTile * D, *vs = Vb + my_src + (size_t)tile * kTile * D;
      if (row0 + kTile <= t1 && (skip < row0 || skip >= row0 + kTile)) {
#pragma unroll
        for (int p = 0; p < kTile / RPP; ++p) {  // (a step of RPP rows leaves the swizzle as it is)
          cp_async16(kdst + p * RPP * D * 2, ks + p * RPP * D, true);
          cp_async16(vdst + p * RPP * D * 2, vs + p * RPP * D, true);
        }
      } else {
#pragma unroll
        for (int p = 0; p < kTile / RPP; ++p) {
          const int row = row0 + my_row + p * RPP;
          if (row == skip) continue;
          const bool ok = row < t1;
          const size_t src = ok ? (size_t)row * D + my_c * 8 : (size_t)t0 * D;
          cp_async16(kdst + p * RPP * D * 2, Kb + src, ok);
          cp_async16(vdst + p * RPP * D * 2, Vb + src, ok);
        }
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
  for (int i = tid; i < NH * CH; i += NT) {  // query rows, zero beyond the group
    const int row = i / CH, c = i - row * CH;
    uint4 val = make_uint4(0, 0, 0, 0);
    // (a head stands once more in the row of its other parts, so that the threads of that column have its weights as well)
    const int h = HEADS == 1 ? (row == 2 ? 0 : row) : HEADS == 4 ? row & 3 : row;
    if (h < G) val = *reinterpret_cast<const uint4*>(qb + (size_t)h * D + c * 8);
    *reinterpret_cast<uint4*>(q_s + swz<D>(row, c)) = val;
  }
  __syncthreads();
  uint32_t qf[KS][2];  // B fragments of Q^T
#pragma unroll
  for (int ks = 0; ks < KS; ks += 2)
    ldmatrix_x4(smem_u32(q_s + swz<D>(r8, 2 * ks + mi)), qf[ks][0], qf[ks][1], qf[ks + 1][0], qf[ks + 1][1]);

  // this thread's heads are 2 tq and 2 tq + 1; of O^T it holds the rows gq and gq + 8 of each block
  float o[KS][4], m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
#pragma unroll
  for (int d = 0; d < KS; ++d)
#pragma unroll
    for (int j = 0; j < 4; ++j) o[d][j] = 0.f;
  bool first = true;
  // maximum of the warp's tokens, per head
  auto head_max = [&](const float (&v)[4], float (&mx)[2]) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      mx[j] = fmaxf(v[j], v[2 + j]);
#pragma unroll
      for (int off = 4; off < 32; off <<= 1) mx[j] = fmaxf(mx[j], __shfl_xor_sync(kFull, mx[j], off));
    }
  };

  for (int tile = 0; tile < n_tiles; ++tile) {
    cp_async_wait<STAGES - 2>();
    __syncthreads();
    load_tile(tile + STAGES - 1, -1);
    const int tok0 = t0 + tile * kTile + wn * 16;  // first token of this warp's 16
    if (tok0 >= t1) continue;                      // warp-uniform: nothing of this tile is ours
    const uint32_t kst = smem_u32(k_s) + (tile % STAGES) * TILE_BYTES, vst = smem_u32(v_s) + (tile % STAGES) * TILE_BYTES;
    // ---- S^T = K Q^T: token gq (v[0], v[1]) and gq + 8 (v[2], v[3]), heads 2 tq, 2 tq + 1; two chains ----
    float s0[4] = {0.f, 0.f, 0.f, 0.f}, s1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
      uint32_t kf[4];
      ldmatrix_x4(kst + swz<D>(wn * 16 + (mi & 1) * 8 + r8, 2 * ks + (mi >> 1)), kf[0], kf[1], kf[2], kf[3]);
      mma_bf16(ks & 1 ? s1 : s0, kf, qf[ks][0], qf[ks][1]);
    }
    float v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = (s0[j] + s1[j]) * a.scale_log2;
    if (tok0 + 16 > t1) {
      if (tok0 + gq >= t1) v[0] = v[1] = -INFINITY;
      if (tok0 + gq + 8 >= t1) v[2] = v[3] = -INFINITY;
    }
    if (h2o) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int t = tok0 + gq + (j >> 1) * 8, h = 2 * tq + (j & 1);
        if (t < t1 && h < G) logit[(size_t)t * G + h] = v[j];
      }
    }
    if (first) {
      head_max(v, m);  // finite: token tok0 is valid
      first = false;
    }
    float p[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) p[j] = exp2f(v[j] - m[j & 1]);
    if (__any_sync(kFull, fmaxf(fmaxf(p[0], p[1]), fmaxf(p[2], p[3])) > 65536.f)) {
      // rare: move the references; what is there so far shrinks with them
      float mx[2], f[2];
      head_max(v, mx);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float m_new = fmaxf(m[j], mx[j]);
        f[j] = exp2f(m[j] - m_new);
        m[j] = m_new;
        l[j] *= f[j];
      }
      if constexpr (HEADS == 1) f[1] = f[0];  // column 1 is the head of column 0
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int d = 0; d < KS; ++d) {
          o[d][j] *= f[j];
          o[d][2 + j] *= f[j];
        }
#pragma unroll
      for (int j = 0; j < 4; ++j) p[j] = exp2f(v[j] - m[j & 1]);
    }
    uint32_t pa[2], pb[2];  // tokens gq and gq + 8: the weights' parts, and with HEADS == 8 their second parts
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float x = p[2 * j], y = p[2 * j + 1];
      float xr, yr, d0, d1;
      if constexpr (HEADS == 1) {
        const float x1 = __bfloat162float(__float2bfloat16_rn(x)), r1 = x - x1;
        const float x2 = __bfloat162float(__float2bfloat16_rn(r1)), x3 = r1 - x2;
        pa[j] = pack_bf16(tq == 0 ? x1 : tq == 1 ? x3 : 0.f, tq == 0 ? x2 : 0.f, d0, d1);
      } else {
        pa[j] = pack_bf16(x, y, xr, yr);
        const uint32_t rest = pack_bf16(x - xr, y - yr, d0, d1);
        if constexpr (HEADS == 4) pa[j] = tq < 2 ? pa[j] : rest;
        else pb[j] = rest;
      }
      l[j] += p[j] + p[2 + j];
    }
    const uint32_t a0 = movmatrix_trans(pa[0]), a1 = movmatrix_trans(pa[1]);
    uint32_t b0 = 0, b1 = 0;
    if constexpr (HEADS == 8) {
      b0 = movmatrix_trans(pb[0]);
      b1 = movmatrix_trans(pb[1]);
    }
    // ---- O^T += V^T P^T ----
#pragma unroll
    for (int d = 0; d < KS; ++d) {
      uint32_t vf[4];
      ldmatrix_x4_trans(vst + swz<D>(wn * 16 + (mi >> 1) * 8 + r8, 2 * d + (mi & 1)), vf[0], vf[1], vf[2], vf[3]);
      mma_bf16(o[d], vf, a0, a1);
      if constexpr (HEADS == 8) mma_bf16(o[d], vf, b0, b1);
    }
  }
  cp_async_wait<0>();
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int off = 4; off < 32; off <<= 1) l[j] += __shfl_xor_sync(kFull, l[j], off);
  ScoreAhead ahead;
  if constexpr (SCORES)
    fetch_scores<NT>(ahead, reinterpret_cast<const float*>(a.pool + ldp->acc_off) + (size_t)unit * cap,
                     reinterpret_cast<const int*>(a.pool + ldp->pos_off) + (size_t)unit * cap, t0 + tid, t1, len == b);
  __syncthreads();  // the pipeline buffers are free: the four warps' results meet there
  float* mg = reinterpret_cast<float*>(k_s);
  static_assert(WN * SLOT * 4 <= STAGES * TILE_BYTES, "merge area");
  {
    float* slot = mg + wn * SLOT;
#pragma unroll
    for (int d = 0; d < KS; ++d)
#pragma unroll
      for (int j = 0; j < 4; ++j) slot[(2 * tq + (j & 1)) * (D + 4) + d * 16 + gq + (j >> 1) * 8] = o[d][j];
    if (gq == 0)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        float* row = slot + (2 * tq + j) * (D + 4) + D;
        row[0] = m[j];
        row[1] = l[j];
      }
  }
  __syncthreads();
  // four consecutive elements of a head per step
  float* part_o = reinterpret_cast<float*>(v_s);  // SCORES: [G][D], then the statistics [G][4]
  float* part_stat = part_o + NH * D;
  for (int i4 = tid; i4 < G * D / 4; i4 += NT) {
    const int h = i4 * 4 / D, e = i4 * 4 - h * D;
    float M = -INFINITY, f[WN];
#pragma unroll
    for (int x = 0; x < WN; ++x) {
      f[x] = mg[x * SLOT + h * (D + 4) + D];
      M = fmaxf(M, f[x]);
    }
    float L = 0.f;
    float4 O = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int x = 0; x < WN; ++x) {
      const float* row = mg + x * SLOT + h * (D + 4);
      f[x] = (f[x] > -INFINITY) ? exp2f(f[x] - M) : 0.f;
      L += row[D + 1] * f[x];
      float4 v = *reinterpret_cast<const float4*>(row + e);
      [[maybe_unused]] auto add = [&](int other) {  // the result of another part of the weights
        const float4 u = *reinterpret_cast<const float4*>(row + other * (D + 4) + e);
        v.x += u.x;
        v.y += u.y;
        v.z += u.z;
        v.w += u.w;
      };
      if constexpr (HEADS == 1) {
        add(1);
        add(2);
      }
      if constexpr (HEADS == 4) add(4);
      O.x += v.x * f[x];
      O.y += v.y * f[x];
      O.z += v.z * f[x];
      O.w += v.w * f[x];
    }
    if constexpr (SCORES) {
      *reinterpret_cast<float4*>(part_o + h * D + e) = O;
      if (e == 0) *reinterpret_cast<float4*>(part_stat + h * 4) = make_float4(M, L, L, 0.f);
    } else {
      if (n_split == 1) {
        const float inv = 1.f / L;
        const __nv_bfloat162 lo = __floats2bfloat162_rn(O.x * inv, O.y * inv), hi = __floats2bfloat162_rn(O.z * inv, O.w * inv);
        uint2 pk;
        pk.x = *reinterpret_cast<const unsigned*>(&lo);
        pk.y = *reinterpret_cast<const unsigned*>(&hi);
        *reinterpret_cast<uint2*>(ob + (size_t)h * D + e) = pk;
      } else {
        *reinterpret_cast<float4*>(a.part_o + (size_t)blockIdx.x * G * D + h * D + e) = O;
      }
      if (e == 0)
        *reinterpret_cast<float4*>(a.part_stat + ((size_t)blockIdx.x * G + h) * kStatStride) = make_float4(M, L, L, 0.f);
    }
  }
  if constexpr (SCORES) {
    ScoreShared<kMaxPieces>& sh = *reinterpret_cast<ScoreShared<kMaxPieces>*>(part_stat + NH * 4);
    static_assert(NH * (D + 4) * 4 + sizeof(sh) <= STAGES * TILE_BYTES, "partial area");
    finish_scores<bf16, D, NT, kMaxPieces>(a, ldp, unit, t0, t1, len, ob, logit + (size_t)t0 * G, part_o, part_stat, sh, &ahead, w);
  } else {
    if (!h2o && n_split > 1) merge_if_last<bf16>(a, it, unit, part_o);
  }
}

template <int D, int STAGES, int HEADS>
static cudaError_t launch_low_cfg(const DecodeArgs& a, int n_items, int pieces, size_t logit_bytes, cudaStream_t s) {
  constexpr size_t pipe = (size_t)2 * STAGES * kTile * D * 2;
  auto plain = decode_attn_mma_low_kernel<D, STAGES, false, HEADS, DecodeArgs>;
  auto scores = decode_attn_mma_low_kernel<D, STAGES, true, HEADS, DecodeArgsBase>;
  static PerDevice set_up;
  const cudaError_t e = set_up.once([&] {
    cudaError_t r = cudaFuncSetAttribute(plain, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pipe);
    if (r == cudaSuccess) r = cudaFuncSetAttribute(scores, cudaFuncAttributeMaxDynamicSharedMemorySize, kScoresSmem);
    return r == cudaSuccess ? cudaFuncSetAttribute(scores, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) : r;
  });
  if (e != cudaSuccess) return e;
  static ClusterFit wide;
  if (pieces > 8 && !wide.fits(reinterpret_cast<const void*>(scores), kMaxPieces, 128, kScoresSmem)) return cudaErrorNotSupported;
  if (pieces > 0)
    return launch_chained_cluster(scores, pieces, a.n_layer_total * a.n_unit * pieces, 128, pipe + logit_bytes, s,
                                  static_cast<const DecodeArgsBase&>(a));
  return launch_chained(plain, n_items, 128, pipe, s, a);
}

template <int HEADS>
static cudaError_t launch_low(const DecodeArgs& a, int n_items, int pieces, size_t logit_bytes, cudaStream_t s) {
  if (a.head_dim == 64) return launch_low_cfg<64, 4, HEADS>(a, n_items, pieces, logit_bytes, s);
  // Two stages of 32 KB let three CTAs share an SM, which wins once the launch has CTAs to spare; a launch of
  // about one wave (one layer at a time) is better off with the deeper ring per CTA.  us per token, three /
  // two stages: 800 units per layer 305 / 277, 512: 694 / 797, 256: 2109 / 2372.
  if (pieces == 0 && n_items >= 5 * sm_count()) return launch_low_cfg<128, 2, HEADS>(a, n_items, 0, 0, s);
  return launch_low_cfg<128, 3, HEADS>(a, n_items, pieces, logit_bytes, s);
}

cudaError_t launch_decode_mma_low(const DecodeArgs& a, int n_items, int pieces, size_t logit_bytes, cudaStream_t s) {
  if (a.group == 1) return launch_low<1>(a, n_items, pieces, logit_bytes, s);
  return a.group <= 4 ? launch_low<4>(a, n_items, pieces, logit_bytes, s) : launch_low<8>(a, n_items, pieces, logit_bytes, s);
}

}  // namespace sq
