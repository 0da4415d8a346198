// End of a decode step under H2O inside the attention kernel, for groups of at most 32 query heads.
// The pieces of a unit (a range of its slots each) are the CTAs of one thread-block cluster: once
// every piece has its partial result in shared memory they read one another's over the cluster
// (distributed shared memory), so each knows the unit's row maxima and sums, and
//   * merges and stores its share of the output,
//   * adds each of its tokens' probabilities, from the logits it kept in shared memory, to the
//     token's score, and
//   * offers its candidate for the slot that the next append replaces; the first CTA picks.
// Against a second launch that reads the logits back from memory this saves that launch, g fp32
// logits per token written and read, and the partials' trip through L2.
#pragma once
#include "sq_decode_common.cuh"
#include "sq_device.cuh"
#include "sq_select.cuh"

namespace sq {

constexpr int kMaxPieces = 8;  // CTAs of a cluster (the portable limit)

__device__ __forceinline__ int cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return (int)r;
}
__device__ __forceinline__ int cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return (int)r;
}
// Barrier over the cluster's threads; shared memory written before it is visible to the others after it.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Address, in the cluster's shared window, of this CTA's shared-memory location p in CTA `rank`.
__device__ __forceinline__ uint32_t map_rank(const void* p, int rank) {
  uint32_t d;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return d;
}
__device__ __forceinline__ float4 ld_cluster4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void st_cluster_candidate(uint32_t addr, unsigned long long rank, int slot) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(rank) : "memory");
  asm volatile("st.shared::cluster.u32 [%0+8], %1;" ::"r"(addr), "r"(slot) : "memory");
}

// slots of a piece when a unit of `len` slots is cut into `pieces` (whole groups of 32)
__host__ __device__ inline int piece_slots(int len, int pieces) { return ((len + pieces - 1) / pieces + 31) / 32 * 32; }

struct ScoreCandidate {
  unsigned long long rank;
  int slot, pad;
};
// Small shared scratch of finish_scores.
struct ScoreShared {
  float m[32], inv_l[32], inv_w[32];
  float scale[kMaxPieces][32];        // weight of a piece's partial in the merged row
  ScoreCandidate offer[kMaxPieces];   // one per piece (the first CTA's is read)
  ScoreCandidate warp_best[16];
};

// part_o [G][D] (un-normalised) and part_stat [G][4] (maximum, sum, sum of the weights O was made with):
// this piece's partial in shared memory, where every thread of the CTA has written it; logit [token of
// the piece][G], log2 domain, complete too.  t0, t1: the piece's slots; len: the unit's.  NT threads.
template <typename T, int D, int NT>
__device__ __forceinline__ void finish_scores(const DecodeArgsBase& a, const LayerDesc* ldp, int unit, int t0, int t1, int len, T* ob,
                                              const float* logit, const float* part_o, const float* part_stat, ScoreShared& sh) {
  const int tid = threadIdx.x, lane = tid & 31, G = a.group;
  const int n = cluster_size(), me = cluster_rank();
  const int b = ldp->b, cap = ldp->cap;
  const bool full = (len == b);
  if (n > 1) cluster_sync();
  else __syncthreads();
  if (tid < G) {
    float M = -INFINITY;
    float4 st[kMaxPieces];
#pragma unroll
    for (int r = 0; r < kMaxPieces; ++r) {
      st[r] = make_float4(-INFINITY, 0.f, 0.f, 0.f);
      if (r < n) st[r] = n > 1 ? ld_cluster4(map_rank(part_stat + tid * 4, r)) : *reinterpret_cast<const float4*>(part_stat + tid * 4);
      M = fmaxf(M, st[r].x);
    }
    float L = 0.f, Lw = 0.f;
#pragma unroll
    for (int r = 0; r < kMaxPieces; ++r) {
      if (r >= n) continue;
      const float f = (st[r].x > -INFINITY) ? exp2f(st[r].x - M) : 0.f;
      L += st[r].y * f;
      Lw += st[r].z * f;
      sh.scale[r][tid] = f;
    }
    sh.m[tid] = M;
    sh.inv_l[tid] = 1.f / L;
    sh.inv_w[tid] = 1.f / Lw;
  }
  __syncthreads();
  // this CTA's share of the output, four values at a time
  const int n4 = G * D / 4;
  for (int i4 = me * NT + tid; i4 < n4; i4 += n * NT) {
    const int h = i4 * 4 / D;
    float4 O = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int r = 0; r < kMaxPieces; ++r) {
      if (r >= n) break;
      const float4 v = n > 1 ? ld_cluster4(map_rank(part_o + i4 * 4, r)) : *reinterpret_cast<const float4*>(part_o + i4 * 4);
      const float f = sh.scale[r][h];
      O.x += v.x * f;
      O.y += v.y * f;
      O.z += v.z * f;
      O.w += v.w * f;
    }
    const float inv = sh.inv_w[h];
    if (sizeof(T) == 2) {
      __nv_bfloat162 lo = __floats2bfloat162_rn(O.x * inv, O.y * inv), hi = __floats2bfloat162_rn(O.z * inv, O.w * inv);
      uint2 pk;
      pk.x = *reinterpret_cast<unsigned*>(&lo);
      pk.y = *reinterpret_cast<unsigned*>(&hi);
      reinterpret_cast<uint2*>(ob)[i4] = pk;
    } else {
      reinterpret_cast<float4*>(ob)[i4] = make_float4(O.x * inv, O.y * inv, O.z * inv, O.w * inv);
    }
  }
  // scores of this piece's tokens
  const int thr = a.n_tok + 1 - ldp->b_recent;  // next step: positions <= thr are outside the recent window
  const int* pos = reinterpret_cast<const int*>(a.pool + ldp->pos_off) + (size_t)unit * cap;
  float* acc = reinterpret_cast<float*>(a.pool + ldp->acc_off) + (size_t)unit * cap;
  unsigned long long best = ~0ull;
  int best_slot = -1;
  constexpr int kIl = 4;  // slots per thread in flight
  for (int s0 = t0 + tid; s0 < t1; s0 += kIl * NT) {
    float old[kIl];
    int p[kIl];
#pragma unroll
    for (int u = 0; u < kIl; ++u) {
      const int slot = s0 + u * NT;
      old[u] = 0.f;
      p[u] = 0x7fffffff;
      if (slot < t1) {
        old[u] = acc[slot];
        if (full) p[u] = pos[slot];
      }
    }
#pragma unroll
    for (int u = 0; u < kIl; ++u) {
      const int slot = s0 + u * NT;
      if (slot >= t1) continue;
      const float* lg = logit + (size_t)(slot - t0) * G;
      float gain = 0.f;  // in head order
      if ((G & 3) == 0) {
        for (int h = 0; h < G; h += 4) {
          const float4 l4 = *reinterpret_cast<const float4*>(lg + h);
          gain += exp2f(l4.x - sh.m[h]) * sh.inv_l[h];
          gain += exp2f(l4.y - sh.m[h + 1]) * sh.inv_l[h + 1];
          gain += exp2f(l4.z - sh.m[h + 2]) * sh.inv_l[h + 2];
          gain += exp2f(l4.w - sh.m[h + 3]) * sh.inv_l[h + 3];
        }
      } else {
        for (int h = 0; h < G; ++h) gain += exp2f(lg[h] - sh.m[h]) * sh.inv_l[h];
      }
      const float v = old[u] + gain;
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
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long r2 = __shfl_xor_sync(kFull, best, o);
    const int s2 = __shfl_xor_sync(kFull, best_slot, o);
    if (r2 < best) {
      best = r2;
      best_slot = s2;
    }
  }
  if (lane == 0) {
    sh.warp_best[tid >> 5].rank = best;
    sh.warp_best[tid >> 5].slot = best_slot;
  }
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < NT / 32; ++w)
      if (sh.warp_best[w].rank < best) {
        best = sh.warp_best[w].rank;
        best_slot = sh.warp_best[w].slot;
      }
    if (n > 1) st_cluster_candidate(map_rank(&sh.offer[me], 0), best, best_slot);
  }
  if (n > 1) {
    cluster_sync();  // every offer is in; nothing of another CTA's shared memory is touched after this
    if (tid == 0 && me == 0)
      for (int r = 1; r < n; ++r)
        if (sh.offer[r].rank < best) {
          best = sh.offer[r].rank;
          best_slot = sh.offer[r].slot;
        }
  }
  if (full && me == 0 && tid == 0) reinterpret_cast<int*>(a.pool + ldp->victim_off)[unit] = best_slot;
}

}  // namespace sq
