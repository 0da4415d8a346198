// Layer importance (Section 3 cosine-similarity equation; Algorithm 1, steps 1-4) and the
// layer-wise budget allocator (Algorithm 1, steps 5-12; Appendix A.2).
#include <algorithm>

#include "sq_device.cuh"
#include "sq_internal.h"

namespace sq {

// One warp per token: streams the token's two hidden-state rows once, keeps the three sums
// (A.B, A.A, B.B) in fp32 registers, and adds the token's cosine to the warp's running sum (fp64: with few
// warps a sum runs over many tokens; in fp32 the mean of 3 million was off by 3.7e-8).
// CTA sums go to cta_partial; the CTA that finishes last adds them up in index order,
// so the result does not depend on scheduling.
// FUSED: the rows are the residual stream (a) and the attention block's output (b); the kernel
// writes their sum, rounded to T, to sum_out and takes the cosine between a and that sum, i.e.
// between the hidden state before and after self-attention, in the pass that produces the latter.
// Bound by HBM: what counts is bytes in flight.  Few warps with long batches of loads (kU 16-byte pieces
// of each row per lane) keep more in flight per SM than many warps with short ones, and leave the
// partial sums of fewer CTAs to add up at the end.  Measured, us per layer (TB/s) of 16384 tokens of 4096
// bf16 elements (10006 of 4544), kU x CTAs per SM: two rows read: 4 x 8 (before) 48.4 (42.2), 4 x 6 46.1 (34.3),
// 8 x 4 43.8 (33.5), 16 x 2 41.2 (36.2), 8 x 3 42.0 = 6.4 TB/s (31.1); fused (two read, one written): 4 x 8
// started, 5 resident (before) 83.2 (58.5), 4 x 4 72.3 (53.3), 4 x 3 70.4 (49.7), 8 x 2 67.3 = 6.0 TB/s (52.2).
template <bool FUSED>
struct ImportanceCfg {
  static constexpr int kU = 8;
  static constexpr int kCtas = FUSED ? 2 : 3;  // per SM
};
// SHORT: rows of at most 32 pieces (512 bytes) would leave kU - 1 of a lane's loads empty, so a warp takes kU
// rows at a time instead.  us per layer of 61039 tokens of 128 bf16 elements, two rows read (fused): 4 batches,
// 8 CTAs per SM, a row at a time (before) 26.6 (34.9); a batch of kU rows 15.4 (20.5).
template <typename T, bool FUSED, bool SHORT>
__global__ void __launch_bounds__(256, ImportanceCfg<FUSED>::kCtas) cos_sim_reduce_kernel(ImportanceArgs a) {
  constexpr int EPV = Elem<T>::kPerVec;
  const int nvec = a.hidden / EPV;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long n_warp = (long long)gridDim.x * 8;
  double wsum = 0.0;
  grid_wait();
  // one 16-byte piece of each row: its part of the three sums; FUSED: the sum's piece to *out
  auto piece = [&](const uint4& va, const uint4& vb, uint4* out, float& dot, float& na, float& nb) {
    float fa[EPV], fb[EPV];
    widen<T>(va, fa);
    widen<T>(vb, fb);
    if (FUSED) {
      // the sum as it is stored: one fp32 addition, rounded to T
      T r[EPV];
#pragma unroll
      for (int e = 0; e < EPV; ++e) {
        r[e] = narrow<T>(fa[e] + fb[e]);
        fb[e] = to_float<T>(r[e]);
      }
      if (out) *out = *reinterpret_cast<const uint4*>(r);
    }
#pragma unroll
    for (int e = 0; e < EPV; ++e) {
      dot = fmaf(fa[e], fb[e], dot);
      na = fmaf(fa[e], fa[e], na);
      nb = fmaf(fb[e], fb[e], nb);
    }
  };
  auto cosine = [&](float dot, float na, float nb) {
    dot = warp_sum(dot);
    na = warp_sum(na);
    nb = warp_sum(nb);
    const float den = sqrtf(na) * sqrtf(nb);
    return (den > 0.f) ? dot / den : 0.f;
  };
  constexpr int U = ImportanceCfg<FUSED>::kU;
  const uint4* rows_a = reinterpret_cast<const uint4*>(a.a);
  const uint4* rows_b = reinterpret_cast<const uint4*>(a.b);
  uint4* rows_o = FUSED ? reinterpret_cast<uint4*>(a.sum_out) : nullptr;
  if constexpr (SHORT) {
    for (long long row0 = ((long long)blockIdx.x * 8 + warp) * U; row0 < a.n_tok; row0 += n_warp * U) {
      uint4 va[U], vb[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        va[u] = vb[u] = make_uint4(0, 0, 0, 0);
        if (lane < nvec && row0 + u < a.n_tok) {
          va[u] = ld_stream(rows_a + (row0 + u) * nvec + lane);
          vb[u] = ld_stream(rows_b + (row0 + u) * nvec + lane);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        float dot = 0.f, na = 0.f, nb = 0.f;
        piece(va[u], vb[u], FUSED && lane < nvec && row0 + u < a.n_tok ? rows_o + (row0 + u) * nvec + lane : nullptr, dot, na, nb);
        wsum += cosine(dot, na, nb);  // (0 for a row past the end)
      }
    }
  } else {
    for (long long row = (long long)blockIdx.x * 8 + warp; row < a.n_tok; row += n_warp) {
      float dot = 0.f, na = 0.f, nb = 0.f;
      for (int v0 = lane; v0 < nvec; v0 += 32 * U) {
        uint4 va[U], vb[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int v = v0 + 32 * u;
          va[u] = vb[u] = make_uint4(0, 0, 0, 0);
          if (v < nvec) {
            va[u] = ld_stream(rows_a + row * nvec + v);
            vb[u] = ld_stream(rows_b + row * nvec + v);
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
          piece(va[u], vb[u], FUSED && v0 + 32 * u < nvec ? rows_o + row * nvec + v0 + 32 * u : nullptr, dot, na, nb);
      }
      wsum += cosine(dot, na, nb);
    }
  }
  __shared__ double s_w[8];
  __shared__ bool s_last;
  if (lane == 0) s_w[warp] = wsum;
  __syncthreads();
  if (threadIdx.x == 0) {
    double c = 0.0;
    for (int i = 0; i < 8; ++i) c += s_w[i];
    a.cta_partial[blockIdx.x] = c;
    __threadfence();
    unsigned int t = atomicAdd(a.ticket, 1u);
    s_last = (t == gridDim.x - 1);
  }
  __syncthreads();
  if (s_last) {
    __threadfence();
    __shared__ double s_acc[8];
    double acc = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += 256) acc += __ldcg(a.cta_partial + i);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) s_acc[warp] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int i = 1; i < 8; ++i) acc += s_acc[i];
      *a.cos_sum += acc;
      *a.ticket = 0u;
    }
  }
}

cudaError_t launch_importance(const ImportanceArgs& a, int dtype, int n_sm, cudaStream_t s) {
  // all CTAs resident at once; at most kMaxImportanceCtas partial sums
  const long long slots = std::min<long long>(kMaxImportanceCtas, (long long)n_sm * (a.sum_out ? ImportanceCfg<true>::kCtas : ImportanceCfg<false>::kCtas));
  const bool is_short = a.hidden / (dtype == SQ_F32 ? 4 : 8) <= 32;
  const int per_cta = 8 * (is_short ? ImportanceCfg<false>::kU : 1);  // rows in flight
  const int n_cta = (int)std::min<long long>((a.n_tok + per_cta - 1) / per_cta, slots);
  auto go = [&](auto kern) { return launch_chained(kern, n_cta, 256, 0, s, a); };
  if (a.sum_out) {
    if (dtype == SQ_F32) return is_short ? go(cos_sim_reduce_kernel<float, true, true>) : go(cos_sim_reduce_kernel<float, true, false>);
    return is_short ? go(cos_sim_reduce_kernel<__nv_bfloat16, true, true>) : go(cos_sim_reduce_kernel<__nv_bfloat16, true, false>);
  }
  if (dtype == SQ_F32) return is_short ? go(cos_sim_reduce_kernel<float, false, true>) : go(cos_sim_reduce_kernel<float, false, false>);
  return is_short ? go(cos_sim_reduce_kernel<__nv_bfloat16, false, true>) : go(cos_sim_reduce_kernel<__nv_bfloat16, false, false>);
}

// ---------------------------------------------------------------------------------------
// Budget allocator: one CTA.  The clustering is the exact optimum of one-dimensional k-means
// (optimal clusters of scalars are runs of the sorted values): every cut of the sorted list
// into k runs is costed in fp64 and the cheapest wins, the first in lexicographic order on
// equal cost.  A run's cost is evaluated in index order -- mean = (x0 + x1 + ...)/n, then
// (x0-mean)^2 + (x1-mean)^2 + ... -- with individually rounded operations, so the decision
// is reproducible on any IEEE machine.
// ---------------------------------------------------------------------------------------
__device__ double run_cost(const double* x, int lo, int hi) {
  double s = 0.0;
  for (int i = lo; i < hi; ++i) s = __dadd_rn(s, x[i]);
  double mean = __ddiv_rn(s, (double)(hi - lo));
  double c = 0.0;
  for (int i = lo; i < hi; ++i) {
    double d = __dsub_rn(x[i], mean);
    c = __dadd_rn(c, __dmul_rn(d, d));
  }
  return c;
}

constexpr int kAllocThreads = 1024;

// Smallest (cost, id) over the block, id < 0 meaning none; the result is valid in thread 0.
__device__ __forceinline__ int block_best(double cost, int id, double* s_cost, int* s_id) {
  auto better = [](double c1, int i1, double c2, int i2) { return i1 >= 0 && (i2 < 0 || c1 < c2 || (c1 == c2 && i1 < i2)); };
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double c2 = __shfl_xor_sync(0xffffffffu, cost, o);
    const int i2 = __shfl_xor_sync(0xffffffffu, id, o);
    if (better(c2, i2, cost, id)) {
      cost = c2;
      id = i2;
    }
  }
  if ((threadIdx.x & 31) == 0) {
    s_cost[threadIdx.x >> 5] = cost;
    s_id[threadIdx.x >> 5] = id;
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < kAllocThreads / 32; ++w)
      if (better(s_cost[w], s_id[w], cost, id)) {
        cost = s_cost[w];
        id = s_id[w];
      }
  return id;
}

// Bound by latency (one chain of dependent fp64 additions per run of layers): one thread per cut, nothing
// done by a single thread that the block can share.  32 layers: 22 us with 256 threads and serial ends.
__global__ void __launch_bounds__(kAllocThreads) allocate_budgets_kernel(AllocateArgs a) {
  __shared__ double s_x[kMaxLayers];         // sorted values
  __shared__ int s_rank[kMaxLayers];         // rank of each layer's value
  __shared__ double s_head[kMaxLayers + 1];  // cost of run [0, i)
  __shared__ double s_tail[kMaxLayers + 1];  // cost of run [i, n)
  __shared__ double s_best_cost[kAllocThreads / 32];
  __shared__ int s_best_id[kAllocThreads / 32];
  __shared__ int s_cut;
  __shared__ unsigned s_rest[kMaxLayers / 32];  // per 32 layers: those outside G3
  const int n = a.n_layer, tid = threadIdx.x;
  const int st = a.stride, off = blockIdx.x;  // this CTA's budget vector: entries i * st + off
  const long long cnt = tid < n ? a.tok_count[tid] : 0;
  grid_wait();

  // layer averages, rounded to fp32 (the value reported to the caller), ranked by (value, layer)
  if (tid < n) {
    const float c = cnt > 0 ? (float)(a.cos_sum[tid * st + off] / (double)cnt) : 0.f;
    a.cos_sim[tid * st + off] = c;
    s_head[tid] = (double)c;  // scratch: unsorted values
  }
  __syncthreads();
  if (tid < n) {
    const double v = s_head[tid];
    int r = 0;
    for (int j = 0; j < n; ++j) {
      const double w = s_head[j];
      r += (w < v) || (w == v && j < tid);
    }
    s_x[r] = v;
    s_rank[tid] = r;
  }
  __syncthreads();
  const int distinct = 1 + __syncthreads_count(tid >= 1 && tid < n && s_x[tid] != s_x[tid - 1]);
  const int k = min(a.n_cluster, distinct);
  // heads and tails on different warps: their chains run side by side
  if (tid <= n) s_head[tid] = (tid > 0) ? run_cost(s_x, 0, tid) : 0.0;
  else if (tid >= 512 && tid - 512 <= n) s_tail[tid - 512] = (tid - 512 < n) ? run_cost(s_x, tid - 512, n) : 0.0;
  __syncthreads();
  double best = 0.0;
  int best_id = -1;
  if (k == 2) {
    for (int i = 1 + tid; i < n; i += kAllocThreads) {
      const double c = __dadd_rn(s_head[i], s_tail[i]);
      if (best_id < 0 || c < best) {
        best = c;
        best_id = i;
      }
    }
  } else if (k == 3) {
    // candidate id = i * n + j, visited in increasing id per thread
    for (int id = tid; id < n * n; id += kAllocThreads) {
      const int i = id / n, j = id - i * n;
      if (i < 1 || i > n - 2 || j <= i || j > n - 1) continue;
      const double c = __dadd_rn(__dadd_rn(s_head[i], run_cost(s_x, i, j)), s_tail[j]);
      if (best_id < 0 || c < best) {
        best = c;
        best_id = id;
      }
    }
  }
  const int bi = block_best(best, best_id, s_best_cost, s_best_id);
  if (tid == 0) s_cut = bi < 0 ? n : (k == 2 ? bi : bi % n);  // G3 = sorted ranks [cut, n)
  __syncthreads();
  // budgets (Algorithm 1, steps 6-12): G3 gets floor(b_init*p), the rest share what is left
  const int n3 = n - s_cut;
  const bool split = n3 > 0 && n3 < n;
  const bool g3 = split && tid < n && s_rank[tid] >= s_cut;
  const unsigned rest_here = __ballot_sync(0xffffffffu, tid < n && !g3);
  if (tid < kMaxLayers && (tid & 31) == 0) s_rest[tid >> 5] = rest_here;
  __syncthreads();
  if (tid >= n) return;
  long long b = a.b_init;
  if (split) {
    long long b_low = (long long)floor(__dmul_rn((double)a.b_init, a.p));
    if (b_low < 1) b_low = 1;
    if (g3) {
      b = b_low;
    } else {
      const long long rest = (long long)n * a.b_init - (long long)n3 * b_low;
      const long long m = n - n3, base = rest / m, extra = rest % m;
      long long seen = __popc(rest_here & ((1u << (tid & 31)) - 1u));  // layers outside G3 before this one
      for (int w = 0; w < (tid >> 5); ++w) seen += __popc(s_rest[w]);
      b = base + (seen < extra ? 1 : 0);
    }
  }
  a.is_g3[tid * st + off] = g3 ? 1 : 0;
  a.budget[tid * st + off] = (int)b;
}

cudaError_t launch_allocate(const AllocateArgs& a, cudaStream_t s) {
  return launch_chained(allocate_budgets_kernel, a.stride, kAllocThreads, 0, s, a);
}

}  // namespace sq
