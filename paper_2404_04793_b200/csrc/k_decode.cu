// Decode step of Algorithm 1 (steps 15-22) for a range of layers in one launch: append the new
// token into the slot C_seq frees, attend over the kept slots (split-K flash-decode, all query
// heads of a KV head share one pass over K/V), and for H2O add the received probabilities to
// the per-token scores and choose the slot the next append will reuse.  This file: the dispatch, and
// the kernel on the fp32 pipes (fp32 inputs, and bf16 groups that no tensor-core kernel takes).
#include <algorithm>
#include <cstdlib>
#include <cstring>

#include "sq_device.cuh"
#include "sq_internal.h"
#include "sq_select.cuh"
#include "sq_decode_common.cuh"
#include "sq_scores.cuh"

namespace sq {

constexpr int kMaxPieces = 8;  // CTAs of a cluster (the portable limit)

template <bool FIRST, class A>
__device__ __forceinline__ A& either(A& x, A& y) {
  if constexpr (FIRST) return x;
  else return y;
}

// One CTA (NW warps) per (layer, unit, split).  A K or V row is D*sizeof(T) bytes = LPR lanes
// x 16 bytes, so a warp reads 32/LPR consecutive rows per load instruction, fully coalesced.
// Each lane keeps its 16-byte slice of up to GT query heads (pre-scaled by log2(e)/sqrt(d))
// and of their output accumulators in fp32; logits are reduced over the LPR lanes by
// shuffles, and the softmax runs online in the log2 domain over batches of U rows.
// UNIFORM: the launch has no split-K (see locate()).
// NW = 4 everywhere but in the build for launches of few, unsplit units (one layer of a small
// batch): those leave most warp slots of the GPU empty with 4 warps per unit, and each warp then
// walks its rows in a chain of dependent round trips to memory; 16 warps per unit make the chain
// a quarter as long.
// SCORES: H2O with the score update in the same launch (sq_scores.cuh): the pieces of a unit are the
// CTAs of a cluster and the logits stay in shared memory.
// AHEAD: rows are fetched ahead of grid_wait() where a.early.
template <typename T, int D, int GT, int UNIFORM, class Args, int NW = 4, bool SCORES = false, bool AHEAD = false>
__global__ void __launch_bounds__(NW * 32, NW == 4 ? (GT == 1 ? (UNIFORM == 1 ? 8 : 6) : 1) : 2) decode_attn_kernel(Args a) {
  constexpr int EPV = Elem<T>::kPerVec;
  constexpr int LPR = D / EPV;   // lanes per row
  constexpr int RPW = 32 / LPR;  // rows per warp per load
  constexpr int U = 4;           // rows in flight per lane
  __shared__ float sm_o[NW][GT][D];
  __shared__ float sm_m[NW][GT], sm_l[NW][GT];

  extern __shared__ __align__(16) float dyn[];  // SCORES: logits [token of the piece][group], partial O [group][D], its sums [group][4]
  ItemLoc it;
  int item = blockIdx.x;
  if constexpr (SCORES) item /= cluster_size();
  if (!locate<UNIFORM, Args>(a, item, it)) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int sub = lane % LPR, rg = lane / LPR;
  const LayerDesc* ldp = a.layers + it.layer;
  const int b = ldp->b, cap = ldp->cap;
  const int unit = it.local / it.n_split;
  const int len = min(a.n_tok + 1, b);
  const bool h2o = SCORES || (a.policy == SQ_POLICY_H2O);
  if (!AHEAD || !a.early) grid_wait();
  int w;  // slot that receives the new token
  if (h2o) {
    w = (a.n_tok < b) ? a.n_tok : __ldcg(reinterpret_cast<const int*>(a.pool + ldp->victim_off) + unit);
    if (w < 0 || w >= b) {
      if (tid == 0) atomicOr(a.status, 2);
      w = 0;
    }
  } else {
    w = ring_slot(a.n_tok, b, ldp->ring_base, ldp->ring_origin);
  }
  int t0, piece;
  if constexpr (SCORES) {
    piece = piece_slots(len, cluster_size());
    t0 = cluster_rank() * piece;
  } else {
    piece = a.split_tokens;
    t0 = (it.local - unit * it.n_split) * piece;
  }
  const int t1 = min(len, t0 + piece);  // (a piece may be empty under SCORES)
  const int seq = unit / a.n_kv_head, kvh = unit - seq * a.n_kv_head;
  const size_t tok = (size_t)(it.layer - a.layer_begin) * a.batch + seq;
  const T* Kb = reinterpret_cast<const T*>(a.pool + ldp->k_off) + (size_t)unit * cap * D;
  const T* Vb = reinterpret_cast<const T*>(a.pool + ldp->v_off) + (size_t)unit * cap * D;
  const T* qb = reinterpret_cast<const T*>(a.q) + (tok * a.n_q_head + (size_t)kvh * a.group) * D;
  const T* kn = reinterpret_cast<const T*>(a.k_new) + (tok * a.n_kv_head + kvh) * D;
  const T* vn = reinterpret_cast<const T*>(a.v_new) + (tok * a.n_kv_head + kvh) * D;
  T* ob = reinterpret_cast<T*>(a.out) + (tok * a.n_q_head + (size_t)kvh * a.group) * D;
  float* logit;  // [slot][group]
  if constexpr (SCORES) logit = dyn - (size_t)t0 * a.group;
  else logit = a.logits + ldp->logit_off + (size_t)unit * cap * a.group;
  float* part_o = dyn + ((size_t)piece * a.group + 3) / 4 * 4;  // SCORES
  float* part_stat = part_o + (size_t)a.group * D;
  float* stat = a.part_stat + (size_t)blockIdx.x * a.group * kStatStride;
  float* po = a.part_o + (size_t)blockIdx.x * a.group * D;

  // The first batch of this lane's rows, ahead of grid_wait(): the new token's slot still holds the row that it
  // replaces, which is put right afterwards.
  uint4 k_ahead[U], v_ahead[U];
  bool ok_ahead[U];
  if (AHEAD && a.early) {
    const int r0 = t0 + warp * (U * RPW);
    if (t0 < t1) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int row = r0 + u * RPW + rg;
        ok_ahead[u] = row < t1;
        const int rr = ok_ahead[u] ? row : t0;
        k_ahead[u] = ld_stream(Kb + (size_t)rr * D + sub * EPV);
        v_ahead[u] = ld_stream(Vb + (size_t)rr * D + sub * EPV);
      }
    }
    grid_wait();
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int row = r0 + u * RPW + rg, rr = ok_ahead[u] ? row : t0;
      if (t0 < t1 && rr == w) {
        k_ahead[u] = ld_stream(kn + sub * EPV);
        v_ahead[u] = ld_stream(vn + sub * EPV);
      }
    }
  }

  for (int hb = 0; hb < a.group; hb += GT) {
    float qr[GT][EPV], o[GT][EPV], m[GT], l[GT];
#pragma unroll
    for (int g = 0; g < GT; ++g) {
      m[g] = -INFINITY;
      l[g] = 0.f;
      if (hb + g < a.group) {
        widen<T>(ld_stream(qb + (size_t)(hb + g) * D + sub * EPV), qr[g]);
      } else {
#pragma unroll
        for (int e = 0; e < EPV; ++e) qr[g][e] = 0.f;
      }
#pragma unroll
      for (int e = 0; e < EPV; ++e) {
        qr[g][e] *= a.scale_log2;
        o[g][e] = 0.f;
      }
    }
    for (int r0 = t0 + warp * (U * RPW); r0 < t1; r0 += NW * U * RPW) {
      // (arrays of the loop's own where nothing is fetched ahead, and no function for the loads: either costs the
      // register-capped builds up to 18 spilled registers)
      uint4 k_here[U], v_here[U];
      bool ok_here[U];
      auto& kq = either<AHEAD>(k_ahead, k_here);
      auto& vq = either<AHEAD>(v_ahead, v_here);
      auto& ok = either<AHEAD>(ok_ahead, ok_here);
      if (!(AHEAD && a.early && hb == 0 && r0 == t0 + warp * (U * RPW))) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int row = r0 + u * RPW + rg;
          ok[u] = row < t1;
          const int rr = ok[u] ? row : t0;
          const T* kp = (rr == w) ? kn : Kb + (size_t)rr * D;
          const T* vp = (rr == w) ? vn : Vb + (size_t)rr * D;
          kq[u] = ld_stream(kp + sub * EPV);
          vq[u] = ld_stream(vp + sub * EPV);
        }
      }
      float s[U][GT];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        float kf[EPV];
        widen<T>(kq[u], kf);
#pragma unroll
        for (int g = 0; g < GT; ++g) {
          float d = 0.f;
#pragma unroll
          for (int e = 0; e < EPV; ++e) d = fmaf(qr[g][e], kf[e], d);
#pragma unroll
          for (int off = LPR / 2; off > 0; off >>= 1) d += __shfl_xor_sync(kFull, d, off);
          s[u][g] = ok[u] ? d : -INFINITY;
        }
      }
      if (h2o) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (!ok[u]) continue;
          const int row = r0 + u * RPW + rg;
#pragma unroll
          for (int g = 0; g < GT; ++g)
            if (sub == g && hb + g < a.group) logit[(size_t)row * a.group + hb + g] = s[u][g];
        }
      }
      float mn[GT];
#pragma unroll
      for (int g = 0; g < GT; ++g) {
        float mx = s[0][g];
#pragma unroll
        for (int u = 1; u < U; ++u) mx = fmaxf(mx, s[u][g]);
        mn[g] = fmaxf(m[g], mx);
        if (mn[g] > -INFINITY) {
          const float corr = exp2f(m[g] - mn[g]);
          l[g] *= corr;
#pragma unroll
          for (int e = 0; e < EPV; ++e) o[g][e] *= corr;
          m[g] = mn[g];
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        float vf[EPV];
        widen<T>(vq[u], vf);
#pragma unroll
        for (int g = 0; g < GT; ++g) {
          const float p = (s[u][g] > -INFINITY) ? exp2f(s[u][g] - mn[g]) : 0.f;
          l[g] += p;
#pragma unroll
          for (int e = 0; e < EPV; ++e) o[g][e] = fmaf(p, vf[e], o[g][e]);
        }
      }
    }
    // merge the row groups of the warp
#pragma unroll
    for (int off = LPR; off < 32; off <<= 1) {
#pragma unroll
      for (int g = 0; g < GT; ++g) {
        const float m2 = __shfl_xor_sync(kFull, m[g], off);
        const float l2 = __shfl_xor_sync(kFull, l[g], off);
        const float mx = fmaxf(m[g], m2);
        const float f1 = (m[g] > -INFINITY) ? exp2f(m[g] - mx) : 0.f;
        const float f2 = (m2 > -INFINITY) ? exp2f(m2 - mx) : 0.f;
        l[g] = l[g] * f1 + l2 * f2;
#pragma unroll
        for (int e = 0; e < EPV; ++e) {
          const float o2 = __shfl_xor_sync(kFull, o[g][e], off);
          o[g][e] = o[g][e] * f1 + o2 * f2;
        }
        m[g] = mx;
      }
    }
    if (rg == 0) {
#pragma unroll
      for (int g = 0; g < GT; ++g) {
        if (sub == 0) {
          sm_m[warp][g] = m[g];
          sm_l[warp][g] = l[g];
        }
#pragma unroll
        for (int e = 0; e < EPV; ++e) sm_o[warp][g][sub * EPV + e] = o[g][e];
      }
    }
    __syncthreads();
    for (int idx = tid; idx < GT * D; idx += NW * 32) {
      const int g = idx / D, e = idx - g * D, h = hb + g;
      if (h >= a.group) continue;
      float M = -INFINITY;
#pragma unroll
      for (int ww = 0; ww < NW; ++ww) M = fmaxf(M, sm_m[ww][g]);
      float L = 0.f, O = 0.f;
#pragma unroll
      for (int ww = 0; ww < NW; ++ww) {
        const float mw = sm_m[ww][g];
        const float f = (mw > -INFINITY) ? exp2f(mw - M) : 0.f;
        L += sm_l[ww][g] * f;
        O += sm_o[ww][g][e] * f;
      }
      if constexpr (SCORES) {
        part_o[h * D + e] = O;
        if (e == 0) *reinterpret_cast<float4*>(part_stat + h * 4) = make_float4(M, L, L, 0.f);
        continue;
      }
      if (it.n_split == 1)
        ob[(size_t)h * D + e] = narrow<T>(O / L);
      else
        po[(size_t)h * D + e] = O;
      if (e == 0) {
        stat[h * kStatStride] = M;
        stat[h * kStatStride + 1] = L;
        stat[h * kStatStride + 2] = L;
      }
    }
    __syncthreads();
  }

  // the CTA whose range holds slot w stores the new token (nobody reads that slot this step)
  if (w >= t0 && w < t1) {
    if (tid < 2 * LPR) {
      const bool is_v = tid >= LPR;
      const int v = is_v ? tid - LPR : tid;
      const T* src = (is_v ? vn : kn) + v * EPV;
      T* dst = const_cast<T*>(is_v ? Vb : Kb) + (size_t)w * D + v * EPV;
      *reinterpret_cast<uint4*>(dst) = ld_stream(src);
    }
    if (tid == 64) {
      reinterpret_cast<int*>(a.pool + ldp->pos_off)[(size_t)unit * cap + w] = a.n_tok;
      if (h2o) reinterpret_cast<float*>(a.pool + ldp->acc_off)[(size_t)unit * cap + w] = 0.f;
    }
  }
  if constexpr (SCORES) {
    __shared__ ScoreShared<kMaxPieces> sh;
    finish_scores<T, D, NW * 32, kMaxPieces>(a, ldp, unit, t0, t1, len, ob, logit + (size_t)t0 * a.group, part_o, part_stat, sh, nullptr, w);
  } else {
    if (!h2o && it.n_split > 1) merge_if_last<T, 1>(a, it, unit, &sm_o[0][0][0]);
  }
}

// One CTA per (layer, unit): merges the split-K partials into the output and, for H2O, adds
// each kept token's probabilities (summed over the group's heads in head order) to its score
// and picks the slot the next append replaces.
template <typename T>
__global__ void __launch_bounds__(kSelThreads, 5) decode_combine_kernel(DecodeArgs a) {
  __shared__ SelScratch sc;
  __shared__ __align__(16) float s_M[kMaxGroup], s_invL[kMaxGroup], s_invLw[kMaxGroup];
  // one CTA per (descriptor of the launch, unit)
  const int unit = blockIdx.x % a.n_unit;
  ItemLoc it;
  if (!locate_desc(a, blockIdx.x / a.n_unit, it)) return;
  const int layer = it.layer;
  const int tid = threadIdx.x, D = a.head_dim, G = a.group, ns = it.n_split;
  grid_wait();
  const LayerDesc* ldp = a.layers + layer;
  const int b = ldp->b, cap = ldp->cap;
  const size_t item0 = (size_t)it.base + (size_t)unit * ns;
  const float* stat = a.part_stat + item0 * G * kStatStride;
  for (int h = tid; h < G; h += kSelThreads) {
    float M = -INFINITY;
    for (int s = 0; s < ns; ++s) M = fmaxf(M, stat[((size_t)s * G + h) * kStatStride]);
    float L = 0.f, Lw = 0.f;
    for (int s = 0; s < ns; ++s) {
      const float* st = stat + ((size_t)s * G + h) * kStatStride;
      const float f = (st[0] > -INFINITY) ? exp2f(st[0] - M) : 0.f;
      L += st[1] * f;
      Lw += st[2] * f;
    }
    s_M[h] = M;
    s_invL[h] = 1.f / L;     // normaliser of the probabilities (H2O scores)
    s_invLw[h] = 1.f / Lw;   // normaliser matching the weights the output was accumulated with
  }
  __syncthreads();
  if (ns > 1) {
    const int seq = unit / a.n_kv_head, kvh = unit - seq * a.n_kv_head;
    const size_t tok = (size_t)(layer - a.layer_begin) * a.batch + seq;
    T* ob = reinterpret_cast<T*>(a.out) + (tok * a.n_q_head + (size_t)kvh * G) * D;
    const float* po = a.part_o + item0 * G * D;
    for (int idx = tid; idx < G * D; idx += kSelThreads) {
      const int h = idx / D;
      float O = 0.f;
      for (int s = 0; s < ns; ++s) {
        const float ms = stat[((size_t)s * G + h) * kStatStride];
        O += po[(size_t)s * G * D + idx] * ((ms > -INFINITY) ? exp2f(ms - s_M[h]) : 0.f);
      }
      ob[idx] = narrow<T>(O * s_invLw[h]);
    }
  }
  if (a.policy != SQ_POLICY_H2O) return;
  const int len = min(a.n_tok + 1, b);
  const bool full = (len == b);
  const int thr = a.n_tok + 1 - ldp->b_recent;  // next step: positions <= thr are outside the recent window
  const int* pos = reinterpret_cast<const int*>(a.pool + ldp->pos_off) + (size_t)unit * cap;
  float* acc = reinterpret_cast<float*>(a.pool + ldp->acc_off) + (size_t)unit * cap;
  const float* logit = a.logits + ldp->logit_off + (size_t)unit * cap * G;
  unsigned long long best = ~0ull;
  int best_slot = -1;
  // four slots per thread in flight: their logits, score and position loads are independent
  constexpr int kIl = 4;
  for (int s0 = tid; s0 < len; s0 += kIl * kSelThreads) {
    float gain[kIl], old[kIl];
    int p[kIl];
#pragma unroll
    for (int u = 0; u < kIl; ++u) {
      const int slot = s0 + u * kSelThreads;
      gain[u] = 0.f;
      old[u] = 0.f;
      p[u] = 0x7fffffff;
      if (slot < len) {
        old[u] = acc[slot];
        if (full) p[u] = pos[slot];
      }
    }
    if ((G & 3) == 0) {
      for (int h = 0; h < G; h += 4) {
        const float4 m4 = *reinterpret_cast<const float4*>(s_M + h), i4 = *reinterpret_cast<const float4*>(s_invL + h);
#pragma unroll
        for (int u = 0; u < kIl; ++u) {
          const int slot = s0 + u * kSelThreads;
          if (slot < len) {
            const float4 l4 = *reinterpret_cast<const float4*>(logit + (size_t)slot * G + h);
            gain[u] += exp2f(l4.x - m4.x) * i4.x;
            gain[u] += exp2f(l4.y - m4.y) * i4.y;
            gain[u] += exp2f(l4.z - m4.z) * i4.z;
            gain[u] += exp2f(l4.w - m4.w) * i4.w;
          }
        }
      }
    } else {
      // odd group sizes: one slot at a time, so a slot's G consecutive logits stay in L1
#pragma unroll 1
      for (int u = 0; u < kIl; ++u) {
        const int slot = s0 + u * kSelThreads;
        if (slot >= len) continue;
        float g1 = 0.f;
        for (int h = 0; h < G; ++h) g1 += exp2f(logit[(size_t)slot * G + h] - s_M[h]) * s_invL[h];
        gain[u] = g1;
      }
    }
#pragma unroll
    for (int u = 0; u < kIl; ++u) {
      const int slot = s0 + u * kSelThreads;
      if (slot >= len) continue;
      const float v = old[u] + gain[u];
      acc[slot] = v;
      if (full && p[u] <= thr) {
        const unsigned long long r = victim_rank(v, p[u]);
        if (r < best) {
          best = r;
          best_slot = slot;
        }
      }
    }
  }
  if (full) {
    best_slot = block_argmin(sc, best, best_slot);
    if (tid == 0) reinterpret_cast<int*>(a.pool + ldp->victim_off)[unit] = best_slot;
  }
}

// H2O bookkeeping for launches without split-K and groups of at most 32 heads: one WARP per
// (descriptor, unit) instead of one CTA.  A unit holds a few hundred to a few thousand slots,
// too little to occupy 256 threads for longer than the block's set-up and reductions take; as
// warps, every unit of a step is resident at once and nothing synchronises beyond a warp.
// The arithmetic per slot (head order of the sum, the reciprocal of the row sum) is that of
// decode_combine_kernel, so both give the same bits.
constexpr int kWarpUpdWarps = 8;
__global__ void __launch_bounds__(32 * kWarpUpdWarps, 3) h2o_update_warp_kernel(DecodeArgsBase a) {
  __shared__ __align__(16) float s_M[kWarpUpdWarps][32], s_invL[kWarpUpdWarps][32];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int idx = blockIdx.x * kWarpUpdWarps + wib;
  if (idx >= a.n_layer_total * a.n_unit) return;
  const int k = idx / a.n_unit, unit = idx - k * a.n_unit;
  const int layer = a.order[k], G = a.group;
  const LayerDesc* ldp = a.layers + layer;
  const int b = ldp->b, cap = ldp->cap;
  const float* stat = a.part_stat + ((size_t)k * a.n_unit + unit) * G * kStatStride;
  grid_wait();
  if (lane < G) {
    const float2 ml = *reinterpret_cast<const float2*>(stat + lane * kStatStride);
    s_M[wib][lane] = ml.x;
    s_invL[wib][lane] = 1.f / ml.y;
  }
  __syncwarp();
  const float* wM = s_M[wib];
  const float* wI = s_invL[wib];
  const int len = min(a.n_tok + 1, b);
  const bool full = (len == b);
  const int thr = a.n_tok + 1 - ldp->b_recent;  // next step: positions <= thr are outside the recent window
  const int* pos = reinterpret_cast<const int*>(a.pool + ldp->pos_off) + (size_t)unit * cap;
  float* acc = reinterpret_cast<float*>(a.pool + ldp->acc_off) + (size_t)unit * cap;
  const float* logit = a.logits + ldp->logit_off + (size_t)unit * cap * G;
  unsigned long long best = ~0ull;
  int best_slot = -1;
  constexpr int kIl = 8;  // slots per lane in flight: their logits, score and position loads are independent
  for (int s0 = lane; s0 < len; s0 += kIl * 32) {
    float gain[kIl], old[kIl];
    int p[kIl];
#pragma unroll
    for (int u = 0; u < kIl; ++u) {
      const int slot = s0 + u * 32;
      gain[u] = 0.f;
      old[u] = 0.f;
      p[u] = 0x7fffffff;
      if (slot < len) {
        old[u] = acc[slot];
        if (full) p[u] = pos[slot];
      }
    }
    if ((G & 3) == 0) {
      for (int h = 0; h < G; h += 4) {
        const float4 m4 = *reinterpret_cast<const float4*>(wM + h), i4 = *reinterpret_cast<const float4*>(wI + h);
        float4 l4[kIl];
#pragma unroll
        for (int u = 0; u < kIl; ++u) {
          const int slot = s0 + u * 32;
          l4[u] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (slot < len) l4[u] = *reinterpret_cast<const float4*>(logit + (size_t)slot * G + h);
        }
#pragma unroll
        for (int u = 0; u < kIl; ++u) {
          gain[u] += exp2f(l4[u].x - m4.x) * i4.x;
          gain[u] += exp2f(l4[u].y - m4.y) * i4.y;
          gain[u] += exp2f(l4[u].z - m4.z) * i4.z;
          gain[u] += exp2f(l4[u].w - m4.w) * i4.w;
        }
      }
    } else {
#pragma unroll 1
      for (int u = 0; u < kIl; ++u) {
        const int slot = s0 + u * 32;
        if (slot >= len) continue;
        float g1 = 0.f;
        for (int h = 0; h < G; ++h) g1 += exp2f(logit[(size_t)slot * G + h] - wM[h]) * wI[h];
        gain[u] = g1;
      }
    }
#pragma unroll
    for (int u = 0; u < kIl; ++u) {
      const int slot = s0 + u * 32;
      if (slot >= len) continue;
      const float v = old[u] + gain[u];
      acc[slot] = v;
      if (full && p[u] <= thr) {
        const unsigned long long r = victim_rank(v, p[u]);
        if (r < best) {
          best = r;
          best_slot = slot;
        }
      }
    }
  }
  if (full) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long c2 = __shfl_xor_sync(kFull, best, o);
      const int s2 = __shfl_xor_sync(kFull, best_slot, o);
      if (c2 < best) {
        best = c2;
        best_slot = s2;
      }
    }
    if (lane == 0) reinterpret_cast<int*>(a.pool + ldp->victim_off)[unit] = best_slot;
  }
}

// CTAs that start while the launch ahead runs out go where its short units have ended and crowd those SMs.  With long
// pieces, or a wave or more of CTAs of unequal layers, that costs more than a launch's start.  us per token, chained /
// not, fp32, 8 layers, 32 / 8 heads of 128: one launch, 1 sequence of 6000 tokens 141 / 132, 2 of 1500 74.6 / 70.2; one
// per layer, 8 of 6000 1055 / 987.  Short pieces, one launch per layer, against the un-chained build: 1 of 600 180 / 160.
template <typename K, typename A>
static cudaError_t launch_pipe(K kern, const A& args, size_t elem, int n_items, int threads, cudaStream_t s) {
  const size_t piece_bytes = 2 * elem * args.split_tokens * args.head_dim;
  if ((args.early || n_items <= 2 * sm_count()) && piece_bytes <= 512 * 1024) return launch_chained(kern, n_items, threads, 0, s, args);
  kern<<<n_items, threads, 0, s>>>(args);
  return cudaGetLastError();
}

// One head: register-capped, so each form has its own build: with rows ahead of the wait or without (they
// spill 8 to 60 bytes, which is worth it only where they hide a launch's start), with split-K (which takes the
// table) or without, and for few unsplit units (at most two 16-warp CTAs per SM, all resident at once) 16 warps per unit.
// More heads: no rows ahead.  With four heads they take 162 registers to 184, three CTAs per SM to two (12 layers
// of 16 / 4 heads, 40 sequences, one launch: 446 us with rows ahead and a wider merge, 311 without).
template <typename T, int D, bool AHEAD>
static cudaError_t launch_attn_one(const DecodeArgs& a, int n_items, cudaStream_t s) {
  const DecodeArgsBase& base = a;
  if (a.uniform && n_items <= 2 * sm_count())
    return launch_pipe(decode_attn_kernel<T, D, 1, 1, DecodeArgsBase, 16, false, AHEAD>, base, sizeof(T), n_items, 512, s);
  if (a.uniform) return launch_pipe(decode_attn_kernel<T, D, 1, 1, DecodeArgsBase, 4, false, AHEAD>, base, sizeof(T), n_items, 128, s);
  return launch_pipe(decode_attn_kernel<T, D, 1, 0, DecodeArgs, 4, false, AHEAD>, a, sizeof(T), n_items, 128, s);
}
template <typename T, int D>
static cudaError_t launch_attn_g(const DecodeArgs& a, int n_items, cudaStream_t s) {
  if (a.group == 1) return a.early ? launch_attn_one<T, D, true>(a, n_items, s) : launch_attn_one<T, D, false>(a, n_items, s);
  if constexpr (sizeof(T) == 4)  // (bf16 comes here with one head or more than 32)
    if (a.group <= 4) return launch_pipe(decode_attn_kernel<T, D, 4, -1, DecodeArgs>, a, sizeof(T), n_items, 128, s);
  return launch_pipe(decode_attn_kernel<T, D, 8, -1, DecodeArgs>, a, sizeof(T), n_items, 128, s);
}

constexpr int kScoresLimit = 96 * 1024;  // dynamic shared memory of a CTA with the score update
template <auto KERN>
static cudaError_t launch_scores_kernel(const DecodeArgs& a, int pieces, int n_cta, int threads, size_t smem, cudaStream_t s) {
  static PerDevice set_up;
  const cudaError_t e = allow_smem(set_up, kScoresLimit, KERN);
  if (e != cudaSuccess) return e;
  return launch_chained_cluster(KERN, pieces, n_cta, threads, smem, s, static_cast<const DecodeArgsBase&>(a));
}

// H2O with the score update in the launch.  Returns cudaErrorNotSupported where the second launch
// (decode_combine_kernel, h2o_update_warp_kernel) is needed, because a piece's logits do not fit, or the better form: a
// unit has at most eight pieces here, so that long caches of few units leave the GPU idle, and the logits of long pieces
// leave room for fewer CTAs on an SM.  us per token, second launch / this form, fp32: 12 layers of 16 / 4 heads of 128, 8
// sequences 331 / 271; 8 layers of 32 / 8 heads of 128: one launch per layer, 1 sequence of 1500 tokens 264 / 193, 4000: 320 /
// 379, 12000: 539 / 1018; one launch, 1 of 1500 60 / 76, 8 of 4000 491 / 916; 16 / 2 heads of 64, 64 of 1500, one launch per
// layer 501 / 444; 4 / 4 heads of 64, one launch, 4 of 400 14.3 / 10.6, 16 of 4000 142 / 159; 32 / 32 of 128, one launch, 1
// of 1500 75 / 83, 4000: 182 / 206, 12000: 543 / 635.
template <typename T, int D>
static cudaError_t launch_attn_scores(const DecodeArgs& a, int max_len, cudaStream_t s) {
  const int G = a.group;
  if (G > 32) return cudaErrorNotSupported;
  const long long units = (long long)a.n_layer_total * a.n_unit;
  // few units: 16 warps each (two such CTAs per SM); else 4 warps, eight CTAs per SM
  const int n_sm = sm_count();
  const bool wide = G == 1 && units <= 2 * n_sm;
  const long long slots = G == 1 && !wide ? 8LL * n_sm : 2LL * n_sm;
  int pieces = (int)std::min<long long>(kMaxPieces, std::max<long long>(1, slots / units));
  pieces = std::min(pieces, std::max(1, max_len / (wide ? 256 : 128)));
  const size_t limit = (wide || G > 1) ? kScoresLimit : 24 * 1024;
  auto bytes = [&](int p) { return (((size_t)piece_slots(max_len, p) * G + 3) / 4 * 4 + (size_t)G * (D + 4)) * 4; };
  while (pieces < kMaxPieces && bytes(pieces) > limit) ++pieces;
  const size_t smem = bytes(pieces);
  if (smem > limit) return cudaErrorNotSupported;
  const long long ctas = units * pieces;
  const int len = (max_len + pieces - 1) / pieces;
  const bool one_layer = a.n_layer_total == 1;
  if (G == 1) {
    if (ctas > (one_layer ? 8 : 4) * n_sm || (!one_layer && units > n_sm && len > 1200)) return cudaErrorNotSupported;
  } else {
    const bool filled = G > 4 && one_layer && 5 * ctas >= 8 * n_sm;  // equal pieces on nearly every slot
    if (ctas > 4 * n_sm || (len > (one_layer ? 600 : 320) && !filled)) return cudaErrorNotSupported;
  }
  const int n_cta = (int)ctas;
  // (rows ahead of the wait, us per token, one launch per layer: four heads, 12 layers, 8 sequences 329 with, 340
  // without; 80 layers of 64 / 8 heads, 2 sequences 2352 with, 2315 without)
  if (wide) return launch_scores_kernel<decode_attn_kernel<T, D, 1, 1, DecodeArgsBase, 16, true, true>>(a, pieces, n_cta, 512, smem, s);
  if (G == 1) return launch_scores_kernel<decode_attn_kernel<T, D, 1, 1, DecodeArgsBase, 4, true, true>>(a, pieces, n_cta, 128, smem, s);
  if (G <= 4) return launch_scores_kernel<decode_attn_kernel<T, D, 4, 1, DecodeArgsBase, 4, true, true>>(a, pieces, n_cta, 128, smem, s);
  return launch_scores_kernel<decode_attn_kernel<T, D, 8, 1, DecodeArgsBase, 4, true>>(a, pieces, n_cta, 128, smem, s);
}

// The second launch of H2O (scores and next victim, and for split units the merge), by a warp or a CTA per unit.
// It walks a slot's logits four at a time and leaves the rest of their lines to L1.  A launch that starts while the
// attention kernel runs out shares the SMs with that kernel's shared memory, which beside the bf16 kernels' tiles
// leaves a fraction of the L1: it saves a launch's start (about 2 us) and pays by the logit.  So launches of more than
// three quarters of a million logits start after that kernel.  us per token, chained / after, 8 layers: one launch
// for all, 16 sequences, 32 / 1 heads of 64, 12000 tokens 689 / 244, 4000: 235 / 93, 100: 15.7 / 19.0; one launch per
// layer, 64 sequences, 32 / 1 heads of 128, 4000 tokens 887 / 687; 16 sequences, 16 / 1 heads of 64, 400 tokens 83 / 102;
// geometric means over groups of 9 to 32: a quarter of a million logits 0.92 to 0.97, half 0.95 to 1.2, two 1.05 to 1.12.
// fp32 (no tiles in shared memory) and up to four heads (one read per logit line): chained at most 6 % slower.
static cudaError_t launch_second(const DecodeArgs& a, int dtype, const int* desc_tiles, cudaStream_t s) {
  const int n_cta = a.n_layer_total * a.n_unit;
  // More units than the CTA-per-unit kernel holds in one wave (5 CTAs per SM), and nothing to
  // merge: only the scores and the next victim remain, one warp per unit.  Smaller launches
  // (one layer of a small batch) finish sooner with a CTA per unit.
  const bool by_warp = a.policy == SQ_POLICY_H2O && a.uniform && a.group <= 32 && n_cta > 5 * sm_count();
  long long logits = 0;
  for (int k = 0; k < a.n_layer_total; ++k) logits += 128LL * desc_tiles[k];
  logits *= (long long)a.n_unit * a.group;
  const bool chained = dtype == SQ_F32 || a.group <= 4 || logits <= 3 << 18;
  auto go = [&](auto kern, int grid, int block, const auto& args) {
    if (chained) return launch_chained(kern, grid, block, 0, s, args);
    kern<<<grid, block, 0, s>>>(args);
    return cudaGetLastError();
  };
  if (by_warp)
    return go(h2o_update_warp_kernel, (n_cta + kWarpUpdWarps - 1) / kWarpUpdWarps, 32 * kWarpUpdWarps, static_cast<const DecodeArgsBase&>(a));
  if (dtype == SQ_F32) return go(decode_combine_kernel<float>, n_cta, kSelThreads, a);
  return go(decode_combine_kernel<__nv_bfloat16>, n_cta, kSelThreads, a);
}

// One bf16 head per KV head: the mma.sync kernel, but for short caches, where a unit is over before its pipeline of
// tiles pays, and for launches of very many units, where the fp32-pipe kernel's eight CTAs per SM keep as much in flight.
// Between one and two units per SM the mma.sync kernel wins at any length.  Time of the fp32-pipe kernel over the other's,
// 32 / 32 heads of 128 in launches of one layer: caches of 60 tokens 0.62 to 0.95, 200 0.83 to 1.08, 300 1.44 and more up to
// 512 units, 0.98 for 2048; of 8 layers: 60 0.61 to 0.93, 200 0.77 to 0.94, 300 1.09 and more up to 1024 units, 0.93 for 4096, 700
// 0.97 for 4096; heads of 64 cross over at twice the length.  One launch per layer, 32 layers, caches of 409 on average, us per
// token, fp32 pipe / mma.sync: 2 sequences 305 / 198, 8: 417 / 342, 40: 1835 / 1417.
// Under H2O the logits go to memory, where the scores are not updated in the launch: with layers of unequal length the
// fp32-pipe kernel is then the faster one up to eight units per SM (8 layers of 8 / 8 heads of 64 in one launch, 16
// sequences of 1500 tokens 80 / 123, 4000: 184 / 300; 32 / 32 of 128, 4 of 1500 146 / 177).
static bool one_head_on_pipe(int n_desc, int n_unit, int head_dim, int max_len, bool h2o) {
  const long long units = (long long)n_desc * n_unit, n_sm = sm_count(), row_elems = (long long)max_len * head_dim;
  if (units <= n_sm) return max_len <= 320;
  const bool uneven = h2o && n_desc > 1;
  if (units <= 2 * n_sm) return uneven && head_dim == 64 && max_len > 2048;
  if (units < 8 * n_sm) return uneven || max_len <= 200;
  return row_elems <= 64 * 1024 || (units >= 24 * n_sm && n_desc > 1 && row_elems <= 160 * 1024);
}

DecodeKernel decode_kernel_for(int dtype, int head_dim, int group, int n_desc, int n_unit, int max_len, bool h2o) {
  if (dtype != SQ_BF16) return DecodeKernel::kPipe;
  if (group > 32) return head_dim == 64 ? DecodeKernel::kTcgen05 : DecodeKernel::kPipe;
  if (group == 1 && one_head_on_pipe(n_desc, n_unit, head_dim, max_len, h2o)) return DecodeKernel::kPipe;
  return DecodeKernel::kMma;
}

// decode_kernel_for() names the attention kernel; where the tcgen05 kernels refuse a launch (a pool or a batch
// beyond 32-bit tile coordinates), the mma.sync kernel takes up to 96 heads of it and the fp32-pipe kernel the rest.
cudaError_t launch_decode(const DecodeArgs& a, int dtype, int n_items, bool need_combine, size_t pool_bytes,
                          size_t q_rows, const int* desc_tiles, int max_len, cudaStream_t s) {
  if (n_items <= 0) return cudaSuccess;
  bool done = false;
  if (dtype == SQ_BF16 && a.group > 32) {
    // long units that do not fill the CTA slots: the even deal; else one CTA per unit and piece
    cudaError_t e = launch_decode_attn_tc_stream(a, desc_tiles, pool_bytes, q_rows, s);
    if (e == cudaErrorNotSupported) {
      // few units: the pieces of a unit as a cluster, under H2O with the scores and the next victim
      e = launch_decode_attn_tc_cluster(a, desc_tiles, pool_bytes, q_rows, s);
      if (e != cudaErrorNotSupported) return e;
    }
    if (e == cudaErrorNotSupported) e = launch_decode_attn_tc(a, n_items, pool_bytes, q_rows, s);
    if (e == cudaSuccess) {
      // H2O: the attention kernel left the row log-sum-exps; the scores and the next victim come
      // from a second pass over K instead of logits carried through memory
      if (a.policy == SQ_POLICY_H2O) return launch_h2o_gain_tc(a, n_items, pool_bytes, q_rows, s);
      done = true;
    } else if (e != cudaErrorNotSupported) {
      return e;
    }
  }
  // every other kernel needs the per-slot logits for H2O: a context sized for the tcgen05 pair
  // does not hold them, and nothing may fall back silently
  if (!done && a.policy == SQ_POLICY_H2O && !a.has_logits) return cudaErrorNotSupported;
  if (!done && a.policy == SQ_POLICY_H2O) {
    cudaError_t e;
    if (dtype == SQ_BF16) e = launch_decode_mma_scores(a, max_len, s);
    else e = a.head_dim == 64 ? launch_attn_scores<float, 64>(a, max_len, s) : launch_attn_scores<float, 128>(a, max_len, s);
    if (e != cudaErrorNotSupported) return e;
  }
  if (!done && decode_kernel_for(dtype, a.head_dim, a.group, a.n_layer_total, a.n_unit, max_len, a.policy == SQ_POLICY_H2O) != DecodeKernel::kPipe) {
    cudaError_t e = launch_decode_attn_mma(a, n_items, s);
    if (e == cudaSuccess) done = true;
    else if (e != cudaErrorNotSupported) return e;
  }
  if (!done) {
    cudaError_t e;
    if (dtype == SQ_F32) e = a.head_dim == 64 ? launch_attn_g<float, 64>(a, n_items, s) : launch_attn_g<float, 128>(a, n_items, s);
    else e = a.head_dim == 64 ? launch_attn_g<__nv_bfloat16, 64>(a, n_items, s) : launch_attn_g<__nv_bfloat16, 128>(a, n_items, s);
    if (e != cudaSuccess) return e;
  }
  if (!need_combine) return cudaSuccess;
  return launch_second(a, dtype, desc_tiles, s);
}

}  // namespace sq
