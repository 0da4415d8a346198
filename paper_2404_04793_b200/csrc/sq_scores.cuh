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
// Barrier over the cluster's threads, in two parts; shared memory written before it is visible to the others after it.  The
// .aligned forms want a warp's threads together, so the warp meets first: loops and branches ahead may end in its lanes at
// different times.
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_sync() {
  cluster_arrive();
  cluster_wait();
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
// Shared scratch of finish_scores for up to PIECES CTAs per cluster.
template <int PIECES>
struct ScoreShared {
  float4 stat[PIECES][32];        // the pieces' partial statistics; .w: a piece's weight in the merged row
  float m[32], inv_l[32], inv_w[32];
  ScoreCandidate offer[PIECES];   // one per piece (the first CTA's is read)
  ScoreCandidate warp_best[16];
};
constexpr int kScoreIl = 4;  // slots per thread in flight in the score update
// A thread's first slots' scores and positions, which a kernel with registers to spare fetches ahead of
// its merge so that the trip to memory runs under it (no value is looked at before the update).
struct ScoreAhead {
  float old[kScoreIl];
  int p[kScoreIl];
};
template <int NT>
__device__ __forceinline__ void fetch_scores(ScoreAhead& ah, const float* acc, const int* pos, int s0, int t1, bool full) {
#pragma unroll
  for (int u = 0; u < kScoreIl; ++u) {
    const int slot = s0 + u * NT;
    ah.old[u] = 0.f;
    ah.p[u] = 0x7fffffff;
    if (slot < t1) {
      ah.old[u] = acc[slot];
      if (full) ah.p[u] = pos[slot];
    }
  }
}

// part_o [G][D] (un-normalised) and part_stat [G][4] (maximum, sum, sum of the weights O was made with):
// this piece's partial in shared memory, where every thread of the CTA has written it; logit [token of
// the piece][G], log2 domain, complete too.  t0, t1: the piece's slots; len: the unit's; w: the new
// token's slot.  fetched: scores of the thread's first slots, or null.  NT threads.
template <typename T, int D, int NT, int PIECES>
__device__ __forceinline__ void finish_scores(const DecodeArgsBase& a, const LayerDesc* ldp, int unit, int t0, int t1, int len, T* ob,
                                              const float* logit, const float* part_o, const float* part_stat,
                                              ScoreShared<PIECES>& sh, const ScoreAhead* fetched, int w) {
  const int tid = threadIdx.x, lane = tid & 31, G = a.group;
  const int n = cluster_size(), me = cluster_rank();
  const int b = ldp->b, cap = ldp->cap;
  const bool full = (len == b);
  const int* pos = reinterpret_cast<const int*>(a.pool + ldp->pos_off) + (size_t)unit * cap;
  float* acc = reinterpret_cast<float*>(a.pool + ldp->acc_off) + (size_t)unit * cap;
  if (n > 1) {
    cluster_sync();
    for (int i = tid; i < n * 32; i += NT) {  // one read over the cluster per (piece, head)
      const int r = i >> 5, h = i & 31;
      if (h < G) sh.stat[r][h] = ld_cluster4(map_rank(part_stat + h * 4, r));
    }
  } else {
    __syncthreads();
    if (tid < G) sh.stat[0][tid] = *reinterpret_cast<const float4*>(part_stat + tid * 4);
  }
  __syncthreads();
  if (tid < G) {
    float M = -INFINITY;
    for (int r = 0; r < n; ++r) M = fmaxf(M, sh.stat[r][tid].x);
    float L = 0.f, Lw = 0.f;
    for (int r = 0; r < n; ++r) {
      const float4 st = sh.stat[r][tid];
      const float f = (st.x > -INFINITY) ? exp2f(st.x - M) : 0.f;
      L += st.y * f;
      Lw += st.z * f;
      sh.stat[r][tid].w = f;
    }
    sh.m[tid] = M;
    sh.inv_l[tid] = 1.f / L;
    sh.inv_w[tid] = 1.f / Lw;
  }
  __syncthreads();
  // this CTA's share of the output, four values at a time; the last CTA, whose piece is the shortest, first
  const int n4 = G * D / 4;
  for (int i4 = (n - 1 - me) * NT + tid; i4 < n4; i4 += n * NT) {
    const int h = i4 * 4 / D;
    float4 O = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int r0 = 0; r0 < n; r0 += 4) {
      float4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r0 + u < n)
          v[u] = n > 1 ? ld_cluster4(map_rank(part_o + i4 * 4, r0 + u)) : *reinterpret_cast<const float4*>(part_o + i4 * 4);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float f = (r0 + u < n) ? sh.stat[r0 + u][h].w : 0.f;
        O.x += v[u].x * f;
        O.y += v[u].y * f;
        O.z += v[u].z * f;
        O.w += v[u].w * f;
      }
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
  unsigned long long best = ~0ull;
  int best_slot = -1;
  for (int s0 = t0 + tid; s0 < t1; s0 += kScoreIl * NT) {
    ScoreAhead ahead;
    if (fetched && s0 < t0 + kScoreIl * NT) ahead = *fetched;
    else fetch_scores<NT>(ahead, acc, pos, s0, t1, full);
#pragma unroll
    for (int u = 0; u < kScoreIl; ++u) {
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
      // the new token's entries may have been fetched before they were stored
      const float v = (slot == w ? 0.f : ahead.old[u]) + gain;
      const int p = slot == w ? a.n_tok : ahead.p[u];
      acc[slot] = v;
      if (full && p <= thr) {
        const unsigned long long r = victim_rank(v, p);
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
