// Prefill side of Algorithm 1 (step 13 with the first compression of steps 16-18 applied at
// once): H2O prompt scores, C_seq selection over the prompt, and the gather of the kept K/V
// rows into the layer's cache region.
#include <algorithm>
#include <cstdlib>
#include <cstring>

#include "sq_device.cuh"
#include "sq_internal.h"
#include "sq_select.cuh"

namespace sq {

// ---------------------------------------------------------------------------------------
// H2O prompt scores on the fp32 pipes.  acc[t] = sum over the query heads sharing the KV head and over
// query rows r >= t of softmax_row_r(Q K^T / sqrt(d))[t] (causal).  Two sweeps over TQ x 64 score tiles
// (rows: queries, columns: keys): row log-sum-exp, then column sums of exp(s - lse).
// Thread (tx, ty) of the 16 x TQ/4 block owns rows 4 ty .. +3 and columns 4 tx .. +3 of a tile.  Both
// operands lie transposed in shared memory, so one 16-byte read of each feeds sixteen FMAs; the next
// streamed tile is on its way to registers while this one is worked on.  Bound by the FMA pipe for large
// prompts and by the chain of tiles of a CTA for small ones: there TQ is 32, and the second sweep's
// stream is cut into pieces whose column sums the last to finish adds up in order (deterministic).
// Measured, us per layer of scores, selection and gather, fp32, 64 x 64 tiles with scalar reads and one CTA per
// key tile / this: 2 sequences of 777 tokens, 16 / 4 heads of 128: 798 / 286; 20 of 500, 20 / 1 heads of 64: 1627 / 585; 1 of
// 2048, 32 / 32 heads of 128: 2143 / 1395.  (Short prompts: prefill_rows_kernel.)
// ---------------------------------------------------------------------------------------
constexpr int TK = 64;

// four consecutive elements of a row, widened
template <typename T>
__device__ __forceinline__ float4 load4(const T* p);
template <>
__device__ __forceinline__ float4 load4<float>(const float* p) {
  return *reinterpret_cast<const float4*>(p);
}
template <>
__device__ __forceinline__ float4 load4<__nv_bfloat16>(const __nv_bfloat16* p) {
  const uint2 v = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                     __uint_as_float(v.y & 0xffff0000u));
}

// A tile of ROWS rows of D elements on its way from global memory to shared memory, where it lies
// transposed: element (row, e) at [e * (ROWS + 4) + row].  Rows at or past `limit` read as 0.
template <typename T, int D, int ROWS, int NT>
struct TileLoad {
  static constexpr int N = ROWS * D / 4 / NT;
  float4 v[N];
  __device__ __forceinline__ void fetch(const T* base, int row0, int limit) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int idx = threadIdx.x + i * NT, row = idx % ROWS, e = idx / ROWS * 4;
      v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (row0 + row < limit) v[i] = load4<T>(base + (size_t)(row0 + row) * D + e);
    }
  }
  __device__ __forceinline__ void store(float* s) const {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int idx = threadIdx.x + i * NT, row = idx % ROWS, e = idx / ROWS * 4;
      s[(e + 0) * (ROWS + 4) + row] = v[i].x;
      s[(e + 1) * (ROWS + 4) + row] = v[i].y;
      s[(e + 2) * (ROWS + 4) + row] = v[i].z;
      s[(e + 3) * (ROWS + 4) + row] = v[i].w;
    }
  }
};

template <int D, int TQ>
__device__ __forceinline__ void score_tile(const float* qs, const float* ks, float (&s)[4][4]) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) s[r][c] = 0.f;
#pragma unroll 8
  for (int e = 0; e < D; ++e) {
    const float4 q = *reinterpret_cast<const float4*>(qs + e * (TQ + 4) + 4 * ty);
    const float4 k = *reinterpret_cast<const float4*>(ks + e * (TK + 4) + 4 * tx);
    const float qv[4] = {q.x, q.y, q.z, q.w}, kv[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) s[r][c] = fmaf(qv[r], kv[c], s[r][c]);
  }
}

template <int D, int TQ>
constexpr size_t score_smem() {
  return (size_t)D * (TQ + 4 + TK + 4) * 4;
}

template <typename T, int D, int TQ>
__global__ void __launch_bounds__(4 * TQ) prefill_row_lse_kernel(ScoreArgs a, float scale_log2) {
  constexpr int NT = 4 * TQ;
  extern __shared__ __align__(16) float sm[];
  float* qs = sm;
  float* ks = sm + D * (TQ + 4);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int P = a.prompt, n_qt = (P + TQ - 1) / TQ;
  const int qt = n_qt - 1 - blockIdx.x, hq = blockIdx.y, bi = blockIdx.z;  // longest rows first
  const int g = a.n_q_head / a.n_kv_head;
  const T* qbase = reinterpret_cast<const T*>(a.q) + ((size_t)bi * a.n_q_head + hq) * P * D;
  const T* kbase = reinterpret_cast<const T*>(a.k) + ((size_t)bi * a.n_kv_head + hq / g) * P * D;
  const int q0 = qt * TQ, n_kt = (min(q0 + TQ, P) + TK - 1) / TK;
  grid_wait();
  {
    TileLoad<T, D, TQ, NT> ql;
    ql.fetch(qbase, q0, P);
    ql.store(qs);
  }
  TileLoad<T, D, TK, NT> kl;
  kl.fetch(kbase, 0, P);
  float m[4], l[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    m[r] = -INFINITY;
    l[r] = 0.f;
  }
  for (int kt = 0; kt < n_kt; ++kt) {
    const int k0 = kt * TK;
    __syncthreads();
    kl.store(ks);
    __syncthreads();
    if (kt + 1 < n_kt) kl.fetch(kbase, k0 + TK, P);
    float s[4][4];
    score_tile<D, TQ>(qs, ks, s);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int qr = q0 + 4 * ty + r;
      float tmax = -INFINITY;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int kr = k0 + 4 * tx + c;
        s[r][c] = (kr <= qr && qr < P) ? s[r][c] * scale_log2 : -INFINITY;
        tmax = fmaxf(tmax, s[r][c]);
      }
      // every thread keeps the maximum and sum of its own columns; the row's are formed at the end
      const float m_new = fmaxf(m[r], tmax);
      if (m_new > -INFINITY) {
        float sum = 0.f;
#pragma unroll
        for (int c = 0; c < 4; ++c) sum += exp2f(s[r][c] - m_new);
        l[r] = l[r] * exp2f(m[r] - m_new) + sum;
        m[r] = m_new;
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    float mm = m[r];
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) mm = fmaxf(mm, __shfl_xor_sync(0xffffffffu, mm, o));
    float ll = (m[r] > -INFINITY) ? l[r] * exp2f(m[r] - mm) : 0.f;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) ll += __shfl_xor_sync(0xffffffffu, ll, o);
    const int qr = q0 + 4 * ty + r;
    if (tx == 0 && qr < P) a.lse2[((size_t)bi * a.n_q_head + hq) * P + qr] = mm + log2f(ll);
  }
}

// Grid: (key tile, KV head, sequence * n_piece).  The (head, query tile) pairs that a key tile sees,
// heads outermost, go to its pieces `chunk` at a time.
template <typename T, int D, int TQ>
__global__ void __launch_bounds__(4 * TQ) prefill_col_sum_kernel(ScoreArgs a, float scale_log2, int n_piece, int chunk) {
  constexpr int NT = 4 * TQ;
  extern __shared__ __align__(16) float sm[];
  __shared__ float red[TQ / 4][TK];
  __shared__ int s_last;
  float* qs = sm;
  float* ks = sm + D * (TQ + 4);
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int kt = blockIdx.x, hk = blockIdx.y, bi = blockIdx.z / n_piece, piece = blockIdx.z - bi * n_piece;
  const int g = a.n_q_head / a.n_kv_head, P = a.prompt;
  const int n_qt = (P + TQ - 1) / TQ, k0 = kt * TK, qt0 = k0 / TQ, per = n_qt - qt0;
  const int n_stream = g * per, i0 = piece * chunk, i1 = min(n_stream, i0 + chunk);
  const int pieces_here = (n_stream + chunk - 1) / chunk;
  if (i0 >= n_stream) return;
  const T* kbase = reinterpret_cast<const T*>(a.k) + ((size_t)bi * a.n_kv_head + hk) * P * D;
  const T* qhead0 = reinterpret_cast<const T*>(a.q) + ((size_t)bi * a.n_q_head + hk * g) * P * D;
  const float* lse0 = a.lse2 + ((size_t)bi * a.n_q_head + hk * g) * P;
  int h = i0 / per, qt = qt0 + (i0 - h * per);
  {
    TileLoad<T, D, TK, NT> kl;
    kl.fetch(kbase, k0, P);
    kl.store(ks);
  }
  TileLoad<T, D, TQ, NT> ql;
  ql.fetch(qhead0 + (size_t)h * P * D, qt * TQ, P);
  grid_wait();  // the inputs are older than the launch ahead, the row sums are its result
  float col[4] = {0.f, 0.f, 0.f, 0.f};
  for (int i = i0; i < i1; ++i) {
    const int q0 = qt * TQ;
    float lse[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int qr = q0 + 4 * ty + r;
      lse[r] = qr < P ? lse0[(size_t)h * P + qr] : INFINITY;  // a query past the end attends to nothing
    }
    __syncthreads();
    ql.store(qs);
    __syncthreads();
    if (++qt == n_qt) {
      qt = qt0;
      ++h;
    }
    if (i + 1 < i1) ql.fetch(qhead0 + (size_t)h * P * D, qt * TQ, P);
    float s[4][4];
    score_tile<D, TQ>(qs, ks, s);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int qr = q0 + 4 * ty + r;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float p = exp2f(s[r][c] * scale_log2 - lse[r]);
        if (k0 + 4 * tx + c <= qr) col[c] += p;
      }
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) red[ty][4 * tx + c] = col[c];
  __syncthreads();
  const size_t unit = (size_t)bi * a.n_kv_head + hk, stride = (size_t)a.batch * a.n_kv_head * P;
  const int kr = k0 + tid;
  if (tid < TK && kr < P) {
    float sum = 0.f;
    for (int y = 0; y < TQ / 4; ++y) sum += red[y][tid];
    (pieces_here == 1 ? a.acc_prompt : a.partial + piece * stride)[unit * P + kr] = sum;
  }
  if (pieces_here == 1) return;
  // the key tile's last piece to finish adds all pieces up, in order (no piece waits)
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    int* ticket = a.tickets + unit * gridDim.x + kt;
    s_last = atomicAdd(ticket, 1) == pieces_here - 1;
    if (s_last) *ticket = 0;
  }
  __syncthreads();
  if (s_last && tid < TK && kr < P) {
    __threadfence();
    float sum = 0.f;
#pragma unroll 8
    for (int p = 0; p < pieces_here; ++p) sum += __ldcg(a.partial + p * stride + unit * P + kr);
    a.acc_prompt[unit * P + kr] = sum;
  }
}

// Short prompts in one launch: a CTA has a query tile of one head and keeps its logits of all keys in shared memory, so
// that once the row sums are known it adds up its rows' weights per key.  The sums of a KV head's (head, query tile)
// pairs go to scratch, pair by pair; a key tile's last pair to finish adds them in order (no pair waits).  Against the
// two sweeps that is one launch and one product less.  us per layer of scores, selection and copies, fp32, two sweeps / this:
// 2 / 2 heads of 64: 1 sequence of 128 tokens 17.2 / 13.3, 256: 23.4 / 19.7, 30 of 256: 59.4 / 36.9; 32 / 32 of 128, 1 of 256: 70.1 /
// 43.8, 500: 165 / 133; 16 / 4 of 128, 6 of 150: 69.6 / 54.2; 8 / 8 of 128, 2 of 600: 144 / 113.
// The chain of a CTA (all keys of its rows) and of the last pair grow with the prompt: of more than 20 pairs per KV head
// launches of few CTAs are no faster (1 sequence of 700, 2 / 2 heads of 64, 45.8 / 46.5).
constexpr int kRowsPairs = 20;
template <int D>
constexpr size_t rows_smem(int n_kt) {
  return score_smem<D, 32>() + (size_t)32 * (n_kt * TK + 4) * 4;
}

template <typename T, int D>
__global__ void __launch_bounds__(128) prefill_rows_kernel(ScoreArgs a, float scale_log2) {
  constexpr int TQ = 32, NT = 4 * TQ;
  extern __shared__ __align__(16) float sm[];
  __shared__ float s_lse[TQ];
  __shared__ int s_last[NT];
  float* qs = sm;
  float* ks = qs + D * (TQ + 4);
  float* logit = ks + D * (TK + 4);  // [TQ][row_len]
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int P = a.prompt, n_qt = (P + TQ - 1) / TQ, n_kt_all = (P + TK - 1) / TK, row_len = n_kt_all * TK + 4;
  const int qt = n_qt - 1 - blockIdx.x, hq = blockIdx.y, bi = blockIdx.z;  // longest rows first
  const int g = a.n_q_head / a.n_kv_head, hk = hq / g;
  const T* qbase = reinterpret_cast<const T*>(a.q) + ((size_t)bi * a.n_q_head + hq) * P * D;
  const T* kbase = reinterpret_cast<const T*>(a.k) + ((size_t)bi * a.n_kv_head + hk) * P * D;
  const int q0 = qt * TQ, n_kt = (min(q0 + TQ, P) + TK - 1) / TK;
  grid_wait();
  {
    TileLoad<T, D, TQ, NT> ql;
    ql.fetch(qbase, q0, P);
    ql.store(qs);
  }
  TileLoad<T, D, TK, NT> kl;
  kl.fetch(kbase, 0, P);
  float m[4], l[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    m[r] = -INFINITY;
    l[r] = 0.f;
  }
  for (int kt = 0; kt < n_kt; ++kt) {
    const int k0 = kt * TK;
    __syncthreads();
    kl.store(ks);
    __syncthreads();
    if (kt + 1 < n_kt) kl.fetch(kbase, k0 + TK, P);
    float s[4][4];
    score_tile<D, TQ>(qs, ks, s);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int qr = q0 + 4 * ty + r;
      float tmax = -INFINITY;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int kr = k0 + 4 * tx + c;
        if (kr > qr || qr >= P) s[r][c] = -INFINITY;
      }
      // (unscaled: the scaling is rounded once, with the subtraction of the log-sum-exp)
      *reinterpret_cast<float4*>(logit + (4 * ty + r) * row_len + k0 + 4 * tx) = make_float4(s[r][0], s[r][1], s[r][2], s[r][3]);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        s[r][c] *= scale_log2;
        tmax = fmaxf(tmax, s[r][c]);
      }
      const float m_new = fmaxf(m[r], tmax);
      if (m_new > -INFINITY) {
        float sum = 0.f;
#pragma unroll
        for (int c = 0; c < 4; ++c) sum += exp2f(s[r][c] - m_new);
        l[r] = l[r] * exp2f(m[r] - m_new) + sum;
        m[r] = m_new;
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    float mm = m[r];
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) mm = fmaxf(mm, __shfl_xor_sync(0xffffffffu, mm, o));
    float ll = (m[r] > -INFINITY) ? l[r] * exp2f(m[r] - mm) : 0.f;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) ll += __shfl_xor_sync(0xffffffffu, ll, o);
    if (tx == 0) s_lse[4 * ty + r] = q0 + 4 * ty + r < P ? mm + log2f(ll) : INFINITY;  // a query past the end attends to nothing
  }
  __syncthreads();
  const size_t unit = (size_t)bi * a.n_kv_head + hk, stride = (size_t)a.batch * a.n_kv_head * P;
  const int pair = (hq - hk * g) * n_qt + qt;
  float* mine = a.partial + pair * stride + unit * P;
  const int n_key = min(n_kt * TK, P);
  for (int key = tid; key < n_key; key += NT) {
    float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
    for (int r = 0; r < TQ; r += 4)
#pragma unroll
      for (int u = 0; u < 4; ++u) sum[u] += exp2f(fmaf(logit[(r + u) * row_len + key], scale_log2, -s_lse[r + u]));  // (-inf before the key: 0)
    mine[key] = (sum[0] + sum[1]) + (sum[2] + sum[3]);
  }
  // the pair's key tiles: a ticket each, query tiles from kt * TK / TQ on see tile kt
  __threadfence();
  __syncthreads();
  if (tid < n_kt) {
    int* ticket = a.tickets + unit * n_kt_all + tid;
    s_last[tid] = atomicAdd(ticket, 1) == g * (n_qt - tid * TK / TQ) - 1;
    if (s_last[tid]) *ticket = 0;
  }
  __syncthreads();
  for (int key = tid; key < n_key; key += NT) {
    if (!s_last[key / TK]) continue;
    __threadfence();
    float sum = 0.f;
    for (int h = 0; h < g; ++h) {
      float part = 0.f;  // of the head
#pragma unroll 8
      for (int t = key / TK * TK / TQ; t < n_qt; ++t) part += __ldcg(a.partial + (size_t)(h * n_qt + t) * stride + unit * P + key);
      sum += part;
    }
    a.acc_prompt[unit * P + key] = sum;
  }
}

template <typename T, int D>
static cudaError_t launch_scores_rows(const ScoreArgs& a, cudaStream_t s) {
  const int n_qt = (a.prompt + 31) / 32, n_kt = (a.prompt + TK - 1) / TK, g = a.n_q_head / a.n_kv_head;
  const long long pairs = (long long)g * n_qt;
  if (pairs > kRowsPairs) return cudaErrorNotSupported;
  constexpr size_t kMost = rows_smem<D>((kRowsPairs * 32 + TK - 1) / TK);  // of one head per KV head
  static_assert(kMost <= 227 * 1024, "shared memory of a CTA");
  if (pairs * a.batch * a.n_kv_head * a.prompt > (long long)a.partial_floats) return cudaErrorNotSupported;
  auto kern = prefill_rows_kernel<T, D>;
  static PerDevice set_up;
  const cudaError_t e = allow_smem(set_up, kMost, kern);
  if (e != cudaSuccess) return e;
  return launch_chained(kern, dim3(n_qt, a.n_q_head, a.batch), 128, rows_smem<D>(n_kt), s, a, 1.4426950408889634f / sqrtf((float)D));
}

template <typename T, int D, int TQ>
static cudaError_t launch_scores_tq(const ScoreArgs& a, cudaStream_t s) {
  auto k1 = prefill_row_lse_kernel<T, D, TQ>;
  auto k2 = prefill_col_sum_kernel<T, D, TQ>;
  constexpr size_t smem = score_smem<D, TQ>();
  static PerDevice set_up;
  cudaError_t e = allow_smem(set_up, smem, k1, k2);
  if (e != cudaSuccess) return e;
  const float scale_log2 = 1.4426950408889634f / sqrtf((float)D);
  const int n_qt = (a.prompt + TQ - 1) / TQ, n_kt = (a.prompt + TK - 1) / TK, g = a.n_q_head / a.n_kv_head;
  const long long units = (long long)a.batch * a.n_kv_head;
  // pieces of about an eighth of an SM's share, as far as the scratch and the grid go
  const long long longest = (long long)g * n_qt, tiles = units * longest * (n_kt + 1) / 2;
  long long chunk = std::max(1LL, std::min(longest, tiles / (8LL * sm_count())));
  auto pieces = [&](long long c) { return (longest + c - 1) / c; };
  while (chunk < longest && (pieces(chunk) * units * a.prompt > (long long)a.partial_floats || pieces(chunk) * a.batch > 65535))
    chunk = std::min(longest, chunk * 2);
  e = launch_chained(k1, dim3(n_qt, a.n_q_head, a.batch), 4 * TQ, smem, s, a, scale_log2);
  if (e != cudaSuccess) return e;
  return launch_chained(k2, dim3(n_kt, a.n_kv_head, a.batch * (unsigned)pieces(chunk)), 4 * TQ, smem, s, a, scale_log2,
                        (int)pieces(chunk), (int)chunk);
}

template <typename T, int D>
static cudaError_t launch_scores_t(const ScoreArgs& a, cudaStream_t s) {
  const cudaError_t e = launch_scores_rows<T, D>(a, s);
  if (e != cudaErrorNotSupported) return e;
  // small problems: more and shorter CTAs
  const long long ctas = (long long)((a.prompt + 63) / 64) * a.n_q_head * a.batch;
  return ctas < 2LL * sm_count() ? launch_scores_tq<T, D, 32>(a, s) : launch_scores_tq<T, D, 64>(a, s);
}

// fp32-pipe kernels (any dtype)
cudaError_t launch_prefill_scores_alu(const ScoreArgs& a, int dtype, cudaStream_t s) {
  if (dtype == SQ_F32) {
    return a.head_dim == 64 ? launch_scores_t<float, 64>(a, s) : launch_scores_t<float, 128>(a, s);
  }
  return a.head_dim == 64 ? launch_scores_t<__nv_bfloat16, 64>(a, s) : launch_scores_t<__nv_bfloat16, 128>(a, s);
}

// bf16 prompts go to the tcgen05 kernels; fp32 (and anything those cannot serve) stays on the
// fp32 pipes.
cudaError_t launch_prefill_scores(const ScoreArgs& a, int dtype, int* status, cudaStream_t s) {
  if (dtype == SQ_BF16) {
    cudaError_t e = launch_prefill_scores_tc(a, status, s);
    if (e != cudaErrorNotSupported) return e;
  }
  return launch_prefill_scores_alu(a, dtype, s);
}

// ---------------------------------------------------------------------------------------
// Copies of kept prompt rows of K and V into the unit's slots (16-byte vectors).
// Bound by HBM (a kept row is read and written once).  Each thread moves 16-byte pieces of K and V of
// several slots, all loads before the first store.  Measured, 256 units of 409 rows of 256 bytes on average
// per layer (107 MB read + written): 20.1 us with one piece of K and V per thread, 18 with this.
// ---------------------------------------------------------------------------------------
__host__ __device__ constexpr int copy_slots(int nt) { return nt / 4; }  // slots per CTA of nt threads

// The slots s0 .. s0 + copy_slots(NT) - 1 of a unit; pos_of(j): the prompt position of slot s0 + j, -1 past the last.
// ug: unit of the batch (sequence, KV head), unit: its index within the descriptor.
template <int ROW_BYTES, int NT, class Pos>
__device__ __forceinline__ void copy_rows(const GatherArgs& a, const LayerDesc& ld, int ug, int unit, int s0, Pos pos_of) {
  constexpr int VPR = ROW_BYTES / 16;            // 16-byte pieces per row
  constexpr int N = copy_slots(NT) * VPR / NT;   // pieces of K (and of V) per thread
  constexpr int B = N < 4 ? N : 4;               // of them in flight
  const uint4* ksrc = reinterpret_cast<const uint4*>(a.k_prompt) + (size_t)ug * a.prompt * VPR;
  const uint4* vsrc = reinterpret_cast<const uint4*>(a.v_prompt) + (size_t)ug * a.prompt * VPR;
  uint4* kdst = reinterpret_cast<uint4*>(a.pool + ld.k_off) + ((size_t)unit * ld.cap + s0) * VPR;
  uint4* vdst = reinterpret_cast<uint4*>(a.pool + ld.v_off) + ((size_t)unit * ld.cap + s0) * VPR;
#pragma unroll
  for (int n0 = 0; n0 < N; n0 += B) {
    uint4 kv[B], vv[B];
    int p[B];
#pragma unroll
    for (int n = 0; n < B; ++n) {
      const int idx = threadIdx.x + (n0 + n) * NT;
      p[n] = pos_of(idx / VPR);
      if (p[n] >= 0) {
        kv[n] = ld_stream(ksrc + (size_t)p[n] * VPR + idx % VPR);
        vv[n] = ld_stream(vsrc + (size_t)p[n] * VPR + idx % VPR);
      }
    }
#pragma unroll
    for (int n = 0; n < B; ++n) {
      const int idx = threadIdx.x + (n0 + n) * NT;
      if (p[n] >= 0) {
        kdst[idx] = kv[n];
        vdst[idx] = vv[n];
      }
    }
  }
}

// Where a unit's heavy rows are few, the CTA that selects them copies them too: up to 100 KB of K and V, in less time than a launch
// takes to start, and no launch follows.  us per layer, copied by a launch / here: fp32, 1 sequence of 256, two heads, 102 kept
// 11.4 / 7.1; 8 KV heads of 128, 16 sequences, 286 kept 20.0 / 17.2, 180: 18.0 / 14.7, 4 sequences, 140: 12.2 / 10.4; 32 KV heads, 8
// sequences, 240 kept 21.7 / 17.3; one head of 64, 33 sequences, 400 kept 12.7 / 11.5.
constexpr int kOwnSlots = 256;
constexpr int kOwnBytes = 100 * 1024;

// The slots of an H2O cache whose position needs no selection: the recent window behind the heavy slots, or the whole prompt
// where the budget holds it.  Slot s of them has position s + prompt - min(prompt, b).
struct FixedSlots {
  int begin, end;
};
__host__ __device__ inline FixedSlots fixed_slots(int prompt, int b, int b_heavy) {
  return prompt > b ? FixedSlots{b_heavy, b} : FixedSlots{0, prompt};
}

// ---------------------------------------------------------------------------------------
// C_seq over the prompt for H2O (one block per unit): keeps the b_recent highest positions
// and, of the others, the b_heavy with the largest score (equal scores: lower position).
// Writes the kept positions, ascending, and their scores to the layer's tables.
// ---------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kSelThreads) select_prompt_kernel(const float* __restrict__ acc_prompt, int P,
                                                                    const LayerDesc* __restrict__ descs,
                                                                    int units_per_desc, char* pool) {
  __shared__ SelScratch sc;
  const int tid = threadIdx.x;
  const LayerDesc ld = descs[blockIdx.x / units_per_desc];  // the descriptor this unit belongs to
  const int unit = blockIdx.x % units_per_desc;             // its index within the descriptor
  const float* acc = acc_prompt + (size_t)blockIdx.x * P;
  int* pos_out = reinterpret_cast<int*>(pool + ld.pos_off) + (size_t)unit * ld.cap;
  float* acc_out = reinterpret_cast<float*>(pool + ld.acc_off) + (size_t)unit * ld.cap;
  if (P <= ld.b) {
    for (int i = tid; i < P; i += kSelThreads) {
      pos_out[i] = i;
      acc_out[i] = acc[i];
    }
    return;
  }
  const int n_cand = P - ld.b_recent;  // positions [0, n_cand) compete for the heavy slots
  uint32_t thr = 0u;
  unsigned int n_at = 0u, ties = 0u;
  int pos_thr = -1;  // among entries with key == thr keep positions <= pos_thr
  if (ld.b_heavy > 0) {
    auto key = [&](int i) { return score_key(acc[i]); };
    auto all = [&](int) { return true; };
    thr = block_radix_select(sc, n_cand, (unsigned)ld.b_heavy, key, all, &n_at, &ties);
    if (ties == n_at) {
      pos_thr = P;
    } else {
      // the n_at lowest positions among the tied: select on the key (2^31-1 - position)
      auto pkey = [&](int i) { return 0x7fffffffu - (uint32_t)i; };
      auto tied = [&](int i) { return score_key(acc[i]) == thr; };
      unsigned int d0, d1;
      uint32_t pt = block_radix_select(sc, n_cand, n_at, pkey, tied, &d0, &d1);
      pos_thr = (int)(0x7fffffffu - pt);
    }
  }
  int written = 0;
  for (int i0 = 0; i0 < P; i0 += kSelThreads) {
    const int i = i0 + tid;
    bool keep = false;
    if (i < P) {
      if (i >= n_cand) {
        keep = true;
      } else if (ld.b_heavy > 0) {
        uint32_t kk = score_key(acc[i]);
        keep = (kk > thr) || (kk == thr && i <= pos_thr);
      }
    }
    int tot;
    int off = block_excl_count(sc, keep, &tot);
    if (keep && written + off < ld.b) {
      pos_out[written + off] = i;
      acc_out[written + off] = acc[i];
    }
    written += tot;
  }
}

// The same for prompts of at most NT * KPT tokens: a token's key stays in a register (token j * NT + tid
// in key j), so the scores are read once; the threshold is found two bits per step by counting keys
// (no histogram: prompt scores share their leading bits, which serialises its atomics) and the search
// ends as soon as a threshold keeps exactly the right number; the kept tokens' scores and the
// cache's first victim come out of the same registers.
// Measured, us per layer of 128 units, 4096 tokens (16 sequences, 8 KV heads): 17.8 with the histogram
// form and its victim launch, about 5 with this one (one sq_evict pass over 32 layers: 2275 -> 1930).
// The CTAs behind one per unit copy the rows of the slots that need no selection (with the default split of a budget half
// of them) meanwhile: the selection is a chain of block-wide steps on one CTA per unit, 12 us in which HBM idled.
// Measured, us per layer, selection and copy one after the other / this, 16 sequences of 4096, 8 KV heads of 128: 1423 rows kept
// 45 / 36, 286 rows 21 / 20; 33 of 8191, one head of 64, 7000 rows 43 / 35.
template <int NT, int KPT, int ROW_BYTES>
__global__ void __launch_bounds__(NT) select_prompt_regs_kernel(const GatherArgs a) {
  constexpr int NW = NT / 32;
  const LayerDesc* descs = a.descs;
  const int P = a.prompt, units_per_desc = a.units_per_desc;
  char* pool = a.pool;
  __shared__ unsigned s_cnt[2][NW];
  __shared__ int s_off[KPT * NW];
  __shared__ unsigned long long s_best[NW];
  __shared__ int s_slot[NW];
  __shared__ int s_heavy[kOwnSlots];  // own_copy: the heavy slots' positions
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  grid_wait();
  const int ug = blockIdx.x % a.n_unit;
  const LayerDesc ld = descs[ug / units_per_desc];
  const int unit = ug % units_per_desc;
  if (blockIdx.x >= a.n_unit) {
    const FixedSlots f = fixed_slots(P, ld.b, ld.b_heavy);
    const int s0 = f.begin + ((int)blockIdx.x / a.n_unit - 1) * copy_slots(NT), shift = P - min(P, ld.b);
    if (s0 < f.end) copy_rows<ROW_BYTES, NT>(a, ld, ug, unit, s0, [&](int j) { return s0 + j < f.end ? s0 + j + shift : -1; });
    return;
  }
  const float* acc = a.scores + (size_t)ug * P;
  int* pos_out = reinterpret_cast<int*>(pool + ld.pos_off) + (size_t)unit * ld.cap;
  float* acc_out = reinterpret_cast<float*>(pool + ld.acc_off) + (size_t)unit * ld.cap;
  const bool drop = P > ld.b;
  const int n_cand = drop ? P - ld.b_recent : 0;  // positions [0, n_cand) compete for the heavy slots
  float val[KPT];
  // of the competing tokens; 0 for the others.  (A score with every bit set, a NaN, has key 0 as well: it takes the lowest other, since
  // there have to be as many competing tokens as the heavy slots were reckoned to get.)
  uint32_t key[KPT];
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    const int i = j * NT + tid;
    val[j] = (i < P) ? acc[i] : 0.f;
  }
#pragma unroll
  for (int j = 0; j < KPT; ++j) key[j] = (j * NT + tid < n_cand) ? max(score_key(val[j]), 1u) : 0u;

  // Competing tokens with key >= lo stay: the largest lo that leaves at least b_heavy of them.  With
  // ties at lo (need_ties < all of them) the lowest positions among those stay.
  uint32_t lo = 0xffffffffu;
  int n_tied_kept = 0x7fffffff;
  if (drop && ld.b_heavy > 0) {
    const unsigned want = (unsigned)ld.b_heavy;
    lo = 0u;
    unsigned n_lo = (unsigned)n_cand;  // competing tokens with key >= lo
    int turn = 0;
    for (int shift = 30; shift >= 0 && n_lo != want; shift -= 2, turn ^= 1) {
      const uint32_t c1 = lo | (1u << shift), c2 = lo | (2u << shift), c3 = lo | (3u << shift);
      unsigned cnt = 0u;  // three counts of at most KPT * 32 <= 512 per warp, ten bits each
#pragma unroll
      for (int j = 0; j < KPT; ++j)
        cnt += (key[j] >= c1 ? 1u : 0u) + (key[j] >= c2 ? 1u << 10 : 0u) + (key[j] >= c3 ? 1u << 20 : 0u);
      cnt = __reduce_add_sync(0xffffffffu, cnt);
      if (lane == 0) s_cnt[turn][warp] = cnt;
      __syncthreads();  // (the other buffer is written next: one barrier per step is enough)
      const unsigned w = lane < NW ? s_cnt[turn][lane] : 0u;
      const unsigned n1 = __reduce_add_sync(0xffffffffu, w & 1023u), n2 = __reduce_add_sync(0xffffffffu, (w >> 10) & 1023u),
                     n3 = __reduce_add_sync(0xffffffffu, w >> 20);
      if (n3 >= want) {
        lo = c3;
        n_lo = n3;
      } else if (n2 >= want) {
        lo = c2;
        n_lo = n2;
      } else if (n1 >= want) {
        lo = c1;
        n_lo = n1;
      }
    }
    if (n_lo != want) {  // all bits decided: n_lo - want of the tokens whose key is lo go
      unsigned c = 0u;
#pragma unroll
      for (int j = 0; j < KPT; ++j) c += key[j] == lo ? 1u : 0u;
      c = __reduce_add_sync(0xffffffffu, c);
      __syncthreads();
      if (lane == 0) s_cnt[0][warp] = c;
      __syncthreads();
      const unsigned ties = __reduce_add_sync(0xffffffffu, lane < NW ? s_cnt[0][lane] : 0u);
      n_tied_kept = (int)(ties - (n_lo - want));
    }
  }
  // Numbers of the flagged tokens before each of this thread's, in token order; every thread calls.
  auto ranks = [&](const bool (&flag)[KPT], int (&rank)[KPT]) {
    __syncthreads();
    unsigned bal[KPT];
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
      bal[j] = __ballot_sync(0xffffffffu, flag[j]);
      if (lane == 0) s_off[j * NW + warp] = __popc(bal[j]);
    }
    __syncthreads();
    if (warp == 0) {  // exclusive scan of the KPT * NW counts
      int running = 0;
#pragma unroll 1
      for (int b0 = 0; b0 < KPT * NW; b0 += 32) {
        const int i = b0 + lane;
        const int c = i < KPT * NW ? s_off[i] : 0;
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += t;
        }
        if (i < KPT * NW) s_off[i] = running + incl - c;
        running += __shfl_sync(0xffffffffu, incl, 31);
      }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < KPT; ++j) rank[j] = s_off[j * NW + warp] + __popc(bal[j] & ((1u << lane) - 1u));
  };
  bool keep[KPT];
  int rank[KPT];
  if (n_tied_kept != 0x7fffffff) {
#pragma unroll
    for (int j = 0; j < KPT; ++j) keep[j] = key[j] == lo && j * NT + tid < n_cand;
    ranks(keep, rank);
#pragma unroll
    for (int j = 0; j < KPT; ++j)
      if (keep[j] && rank[j] >= n_tied_kept) key[j] = 0u;  // a tie that goes
  }
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    const int i = j * NT + tid;
    keep[j] = i < P && (i >= n_cand || (ld.b_heavy > 0 && key[j] >= lo && key[j] != 0u));
  }
  ranks(keep, rank);
  const bool full = P >= ld.b;
  const int last_old = P - ld.b_recent;  // positions up to it are outside the next step's recent window
  unsigned long long best = ~0ull;
  int best_slot = -1;
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    const int i = j * NT + tid;
    if (keep[j] && rank[j] < ld.b) {
      pos_out[rank[j]] = i;
      acc_out[rank[j]] = val[j];
      if (a.own_copy && rank[j] < kOwnSlots) s_heavy[rank[j]] = i;
      if (i <= last_old) {
        const unsigned long long r = victim_rank(val[j], i);
        if (r < best) {
          best = r;
          best_slot = rank[j];
        }
      }
    }
  }
  if (!full) return;  // the cache still grows: the next token takes a fresh slot (and nothing was selected)
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
    s_best[warp] = best;
    s_slot[warp] = best_slot;
  }
  __syncthreads();
  if (a.own_copy) {
    const int n = drop ? ld.b_heavy : 0;
    for (int s0 = 0; s0 < n; s0 += copy_slots(NT))
      copy_rows<ROW_BYTES, NT>(a, ld, ug, unit, s0, [&](int j) { return s0 + j < n ? s_heavy[s0 + j] : -1; });
  }
  if (tid == 0) {
    for (int w = 1; w < NW; ++w)
      if (s_best[w] < best) {
        best = s_best[w];
        best_slot = s_slot[w];
      }
    reinterpret_cast<int*>(pool + ld.victim_off)[unit] = best_slot;
  }
}

// First victim of a full H2O cache (the token the next append will replace).
__global__ void __launch_bounds__(kSelThreads) pick_victim_kernel(char* pool, const LayerDesc* __restrict__ descs,
                                                                  int units_per_desc, int prompt, int next_pos) {
  __shared__ SelScratch sc;
  const LayerDesc ld = descs[blockIdx.x / units_per_desc];
  const int unit = blockIdx.x % units_per_desc;
  const int len = min(prompt, ld.b);
  if (len < ld.b) return;  // the cache still grows: the next token takes a fresh slot
  const int* pos = reinterpret_cast<const int*>(pool + ld.pos_off) + (size_t)unit * ld.cap;
  const float* acc = reinterpret_cast<const float*>(pool + ld.acc_off) + (size_t)unit * ld.cap;
  const int thr = next_pos - ld.b_recent;
  unsigned long long best = ~0ull;
  int slot = -1;
  for (int i = threadIdx.x; i < len; i += kSelThreads) {
    int p = pos[i];
    if (p <= thr) {
      unsigned long long r = victim_rank(acc[i], p);
      if (r < best) {
        best = r;
        slot = i;
      }
    }
  }
  slot = block_argmin(sc, best, slot);
  if (threadIdx.x == 0) reinterpret_cast<int*>(pool + ld.victim_off)[unit] = slot;
}

// The rows of the slots [0, n) of a unit.  Sliding Window / StreamingLLM: all, the kept position of a slot in closed form, which
// also goes to the position table; H2O: those whose position the selection wrote there, with `heavy` only the heavy ones.
template <int ROW_BYTES>
__global__ void __launch_bounds__(256) gather_kernel(const GatherArgs a, bool heavy) {
  __shared__ int s_pos[copy_slots(256)];
  const int ug = blockIdx.x, s0 = blockIdx.y * copy_slots(256);
  grid_wait();
  const LayerDesc ld = a.descs[ug / a.units_per_desc];
  const int unit = ug % a.units_per_desc;
  const int n = heavy ? fixed_slots(a.prompt, ld.b, ld.b_heavy).begin : min(a.prompt, ld.b);
  if (s0 >= n) return;                                   // the grid covers the longest descriptor
  int* pos_tab = reinterpret_cast<int*>(a.pool + ld.pos_off) + (size_t)unit * ld.cap;
  if (threadIdx.x < copy_slots(256)) {
    const int slot = s0 + threadIdx.x;
    int p = -1;
    if (slot < n) {
      if (a.policy == SQ_POLICY_H2O) {
        p = pos_tab[slot];
      } else {
        p = (slot < ld.ring_base) ? slot : ld.ring_origin + (slot - ld.ring_base);
        pos_tab[slot] = p;
      }
    }
    s_pos[threadIdx.x] = p;
  }
  __syncthreads();
  copy_rows<ROW_BYTES, 256>(a, ld, ug, unit, s0, [&](int j) { return s_pos[j]; });
}

template <int ROW_BYTES>
static cudaError_t launch_gather(const GatherArgs& a, int max_slots, bool heavy, cudaStream_t s) {
  if (max_slots <= 0) return cudaSuccess;
  return launch_chained(gather_kernel<ROW_BYTES>, dim3(a.n_unit, (max_slots + copy_slots(256) - 1) / copy_slots(256)), 256, 0, s, a, heavy);
}

template <int NT, int KPT, int ROW_BYTES>
static cudaError_t launch_select(const GatherArgs& a, cudaStream_t s) {
  const long long chunks = (a.max_fixed + copy_slots(NT) - 1) / copy_slots(NT);
  return launch_chained(select_prompt_regs_kernel<NT, KPT, ROW_BYTES>, (unsigned)(a.n_unit * (1 + chunks)), NT, 0, s, a);
}

// H2O: selection over the prompt and the first victim of the caches it fills.  The register form covers
// prompts of up to 16384 tokens; its block is sized by the prompt, so that short prompts of many units
// do not start warps that hold nothing.
template <int ROW_BYTES>
static cudaError_t launch_fill(const GatherArgs& a, bool any_full, cudaStream_t s) {
  if (a.policy != SQ_POLICY_H2O) return launch_gather<ROW_BYTES>(a, a.max_keep, false, s);
  if (a.prompt > 16384) {
    select_prompt_kernel<<<a.n_unit, kSelThreads, 0, s>>>(a.scores, a.prompt, a.descs, a.units_per_desc, a.pool);
    if (any_full) pick_victim_kernel<<<a.n_unit, kSelThreads, 0, s>>>(a.pool, a.descs, a.units_per_desc, a.prompt, a.prompt);
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e : launch_gather<ROW_BYTES>(a, a.max_keep, false, s);
  }
  GatherArgs b = a;
  b.own_copy = a.max_heavy <= kOwnSlots && a.max_heavy * 2 * ROW_BYTES <= kOwnBytes;
  const cudaError_t e = b.prompt <= 1024   ? launch_select<256, 4, ROW_BYTES>(b, s)
                        : b.prompt <= 4096 ? launch_select<512, 8, ROW_BYTES>(b, s)
                                           : launch_select<1024, 16, ROW_BYTES>(b, s);
  return e != cudaSuccess || b.own_copy ? e : launch_gather<ROW_BYTES>(b, b.max_heavy, true, s);
}

cudaError_t launch_fill_cache(const GatherArgs& a, int dtype, bool any_full, cudaStream_t s) {
  const int row_bytes = a.head_dim * (dtype == SQ_F32 ? 4 : 2);
  if (row_bytes == 128) return launch_fill<128>(a, any_full, s);
  if (row_bytes == 256) return launch_fill<256>(a, any_full, s);
  if (row_bytes == 512) return launch_fill<512>(a, any_full, s);
  return cudaErrorInvalidValue;
}

}  // namespace sq
