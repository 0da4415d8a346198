// H2O prompt scores on the 5th-generation tensor cores (bf16).
//
// acc[t] = sum over the query heads sharing a KV head and over query rows r >= t of
//          softmax_row_r(Q K^T / sqrt(d))[t]                       (causal)
// is two sweeps over tiles of 128 rows by TN columns of the score matrix, each tile one tcgen05.mma chain
// (M = 128, N = TN, K = head_dim, bf16 in, fp32 accumulators in tensor memory):
//   sweep 1, CTA = (sequence, query head, 128 query rows): S = Q_tile K_tile^T for the key tiles
//     up to the diagonal; a drain thread owns one TMEM lane = one query row and
//     keeps its running maximum / sum -> row log-sum-exp.
//   sweep 2, CTA = (sequence, KV head, 128 keys, some heads of the group): the operands swap,
//     S^T = K_tile Q_tile^T for all query tiles from the diagonal down and the CTA's heads; thread t
//     owns one key and adds exp2(s*scale - lse[row]) over the tile's columns -> the key's column sum,
//     with no cross-thread reduction and no atomics; a key tile cut into several CTAs by heads is
//     added up, in head order, by the one that finishes last (deterministic).
// Roles per CTA: warp 0 issues TMA tile loads (128-byte swizzle, every CTA its own tiles)
// into a ring of shared-memory stages; warp 1 allocates tensor memory, issues the MMAs, signalling
// completion through tcgen05.commit -> mbarrier, and stages the row log-sum-exps of sweep 2; the others
// drain the accumulators with tcgen05.ld.  Two accumulator buffers let the next tile's MMA run under
// this tile's exponentials.
// What bounds it: the drain's exponentials and what they share a scheduler with.  Per element and warp a sweep takes 9
// cycles, the exponential arithmetic alone 7 (special-function unit 6), the rest is waits for accumulators and
// their loads; without the exponentials a sweep still takes 60 % of its time, without loads or products 98 %; at head_dim 128 the
// board's power limit comes first (1.7 GHz).  us per layer of sweeps 1 / 2: 4 sequences of 4096, 32 / 8 heads of 128: 314 / 367
// with two loads in flight and tiles of 128 columns only, now 305 / 363; 2 of 5003, 71 / 1 heads of 64: 499 / 507, now 482 / 483.
// Built and taken back: in sweep 1 a row's maximum over its first tile as its reference throughout (298 and 457 us).  Rows that
// rise above it then have their exponents formed at the size of the rise, 31 for a key of 2^1 after keys of 2^-30: such
// a key's score was off by up to 1.3e-6, where under a running maximum roundings come to 3.8e-7 at most.
// Built to parity and measured slower (sweeps 1 / 2, against 313 / 366 and 499 / 508): queries on the lanes in both sweeps, with
// one register per key in sweep 2 (315 / 416 as one persistent CTA per SM with 128x256 tiles, 334 / 511 as two CTAs of nine
// warps) or four queries and 16 keys per thread (356 and 515); no issuing warps, the last warp to empty a buffer issues
// its MMAs (413 / 481: an MMA holds the thread that issues it for about 80 cycles); 16 drain warps per CTA of 32 columns
// (310 / 409 and 496 / 556).
// Every mbarrier wait is bounded: on expiry the CTA raises a status bit and winds down.
#include <algorithm>
#include <type_traits>

#include "sq_device.cuh"
#include "sq_internal.h"
#include "sq_tc.cuh"

namespace sq {

using namespace tc;

// TN: columns of a tile (streamed rows), 64 or 128.  A CTA has a TMA warp, an MMA warp and TN / 16 drain warps: a warp
// reaches only the 32 tensor-memory lanes of its quarter (warp index mod 4) and takes 64 of a tile's columns.  An SM's 16
// drain warps are four CTAs of 64 columns, whose waits for an accumulator fall at different times, where shared memory
// holds four (head_dim 64, 2 sequences of 5003, 71 / 1 heads: 992 us a layer against 998 with two of 128; 1136 CTAs 73 against 80), else
// two of 128.
constexpr int prefill_threads(int tn) { return 64 + 2 * tn; }

// exp2 of a pair on the FMA pipe: x = n + f with n the nearest integer (the usual 1.5 * 2^23
// addition), 2^f for |f| <= 1/2 from a degree-5 polynomial (fitted here by a Remez exchange on the
// relative error; in fp32 within 2.1e-7 of the exact value, ex2.approx's own bound is 1.7e-7), the
// exponent added to the bits.  Arguments below -126 give 2^-126 (times at most sqrt 2) instead of a
// smaller number or 0.
__device__ __forceinline__ unsigned long long ex2_pair_fma(unsigned long long x2) {
  constexpr float kMagic = 12582912.f;
  float x0, x1;
  f32x2_split(x2, x0, x1);
  x2 = f32x2(fmaxf(x0, -126.f), fmaxf(x1, -126.f));
  const unsigned long long t2 = add_f32x2(x2, f32x2(kMagic, kMagic));
  const unsigned long long n2 = add_f32x2(t2, f32x2(-kMagic, -kMagic));
  const unsigned long long f2 = fma_f32x2(n2, f32x2(-1.f, -1.f), x2);
  unsigned long long p2 = f32x2(1.3276472454890609e-3f, 1.3276472454890609e-3f);
  p2 = fma_f32x2(p2, f2, f32x2(9.675540961325169e-3f, 9.675540961325169e-3f));
  p2 = fma_f32x2(p2, f2, f32x2(5.550713092088699e-2f, 5.550713092088699e-2f));
  p2 = fma_f32x2(p2, f2, f32x2(2.4022120237350464e-1f, 2.4022120237350464e-1f));
  p2 = fma_f32x2(p2, f2, f32x2(6.931469440460205e-1f, 6.931469440460205e-1f));
  p2 = fma_f32x2(p2, f2, f32x2(1.f, 1.f));
  float t0, t1, p0, p1;
  f32x2_split(t2, t0, t1);
  f32x2_split(p2, p0, p1);
  return f32x2(__uint_as_float(__float_as_uint(p0) + (__float_as_uint(t0) << 23)),
               __uint_as_float(__float_as_uint(p1) + (__float_as_uint(t1) << 23)));
}
__device__ __forceinline__ unsigned long long ex2_pair_sfu(unsigned long long x2) {
  float x0, x1;
  f32x2_split(x2, x0, x1);
  return f32x2(ex2(x0), ex2(x1));
}
// Of every eight pairs of score elements two take the FMA-pipe form, spread evenly, in sweep 1 at head_dim 128 one.  With none the
// special-function unit bounds the drain (16 exponentials per cycle and SM: 1024 cycles per 128 x 128 elements); an FMA-pipe
// pair costs 25 cycles of a scheduler where the unit's takes 16.  Measured on B200, us per layer with 1, 2, 3 of eight: head_dim 128 (4
// sequences of 4096, 32 / 8 heads), sweep 1 305, 320, 321, sweep 2 364, 360, 374; head_dim 64 (2 sequences of 5003, 71 / 1 heads)
// 485, 482, 504 and 501, 485, 505.
template <int D, int SWEEP>
__device__ __forceinline__ constexpr bool on_fma(int pair) {  // `pair` is a constant after unrolling
  return SWEEP == 1 && D == 128 ? (pair & 7) == 7 : (pair & 3) == 3;
}

// SWEEP 1: rows = queries, streamed tiles = keys; SWEEP 2: rows = keys, streamed tiles = queries.
template <int D, int TN, int STAGES, int SWEEP>
__global__ void __launch_bounds__(prefill_threads(TN), TN == 64 ? 4 : 2)
    prefill_scores_tc_kernel(const __grid_constant__ CUtensorMap tm_rows, const __grid_constant__ CUtensorMap tm_stream,
                             ScoreArgs a, ScorePieces pc, float scale_log2, int* status) {
  constexpr int SUB = D / 64;               // 64-column sub-tiles per operand tile
  constexpr int STREAM_SUB = TN * 128;      // one [TN rows x 64 bf16] swizzled sub-tile
  constexpr int ROWS_BYTES = SUB * kSubBytes, TILE_BYTES = SUB * STREAM_SUB;  // the fixed tile, a streamed tile
  constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TN >> 3) << 17) | ((uint32_t)(kTM >> 4) << 24);
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* a_s = smem;
  unsigned char* b_s = smem + ROWS_BYTES;
  unsigned long long* bars = reinterpret_cast<unsigned long long*>(b_s + STAGES * TILE_BYTES);
  // barriers (at most 15 of the 16 slots), then the TMEM base, the abort flag and the lse staging
  static_assert(7 + 2 * STAGES <= 16, "barrier block");
  const uint32_t bar_a = s_u32(bars + 0);
  auto bar_full = [&](int s) { return s_u32(bars + 1 + s); };
  auto bar_empty = [&](int s) { return s_u32(bars + 1 + STAGES + s); };
  auto bar_sfull = [&](int b) { return s_u32(bars + 1 + 2 * STAGES + b); };
  auto bar_sfree = [&](int b) { return s_u32(bars + 3 + 2 * STAGES + b); };
  auto bar_lse = [&](int b) { return s_u32(bars + 5 + 2 * STAGES + b); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 16);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* lse_s = reinterpret_cast<float*>(tmem_slot + 4);  // [2][128]: sweep 2, minus the row log-sum-exps

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int P = a.prompt, g = a.n_q_head / a.n_kv_head;
  const int n_tile = (P + kTM - 1) / kTM, n_col_tile = (P + TN - 1) / TN;
  // grid = (head, sequence, tile): the tile index varies slowest, so the CTAs with the most streamed
  // tiles of every head and sequence start first and the short ones fill the tail of the launch
  const int bi = blockIdx.y;
  int row_tile, n_stream, piece = 0, head0 = 0;
  int rows_head, stream_head;  // (sequence, head) of the fixed tile in the rows tensor, of the first streamed one in the other
  int hq = 0, hk = 0;
  if (SWEEP == 1) {
    hq = blockIdx.x;
    hk = hq / g;
    row_tile = n_tile - 1 - blockIdx.z;  // longest rows first
    n_stream = min(kTM / TN * (row_tile + 1), n_col_tile);
    rows_head = bi * a.n_q_head + hq;
    stream_head = bi * a.n_kv_head + hk;
  } else {
    hk = blockIdx.x;
    row_tile = blockIdx.z / pc.n_piece;  // key tile 0 sees every query tile: longest first
    piece = blockIdx.z - row_tile * pc.n_piece;
    head0 = piece * pc.heads;            // this piece's heads of the group
    n_stream = min(pc.heads, g - head0) * (n_col_tile - kTM / TN * row_tile);
    rows_head = bi * a.n_kv_head + hk;
    stream_head = bi * a.n_q_head + hk * g;
  }
  // Walks the streamed tiles in order: (sweep 1) key tiles 0..row_tile, (sweep 2) per head of the
  // piece the query tiles from the diagonal down.
  struct Walk {
    int h, qt;
  };
  auto walk_begin = [&]() {
    Walk w;
    w.h = head0;
    w.qt = SWEEP == 1 ? 0 : kTM / TN * row_tile;
    return w;
  };
  auto walk_next = [&](Walk& w) {
    ++w.qt;
    if (SWEEP == 2 && w.qt == n_col_tile) {
      w.qt = kTM / TN * row_tile;
      ++w.h;
    }
  };

  if (tid == 0) {
    mbar_init(bar_a, 1);
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(bar_full(s), 1);
      mbar_init(bar_empty(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar_sfull(b), 1);
      mbar_init(bar_sfree(b), TN / 16);  // one arrival per drain warp
      mbar_init(bar_lse(b), 1);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_u32(tmem_slot)), "n"(2 * TN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = *tmem_slot;
  grid_wait();

  // drain threads: sweep 1: running maximum of the row and the sum of its weights; sweep 2: the key's sum (even and odd columns)
  // (a tile's 64 weights are added up by themselves, so that a sum over thousands of tiles is no less precise than they are)
  float m = -INFINITY, sum = 0.f;
  bool ok = true;
  if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      mbar_expect_tx(bar_a, ROWS_BYTES);
#pragma unroll
      for (int sb = 0; sb < SUB; ++sb) tma_load_3d(s_u32(a_s + sb * kSubBytes), &tm_rows, sb * 64, row_tile * kTM, rows_head, bar_a);
      int issued = 0;
      Walk w = walk_begin();
      for (int i = 0; i < n_stream; ++i) {
        const int st = i % STAGES;
        if (i >= STAGES && !mbar_wait(bar_empty(st), ((i / STAGES) - 1) & 1, abort_flag)) break;
        mbar_expect_tx(bar_full(st), TILE_BYTES);
#pragma unroll
        for (int sb = 0; sb < SUB; ++sb)
          tma_load_3d(s_u32(b_s + st * TILE_BYTES + sb * STREAM_SUB), &tm_stream, sb * 64, w.qt * TN, stream_head + w.h, bar_full(st));
        issued = i + 1;
        walk_next(w);
      }
      if (*abort_flag) {
        // winding down early: let the copies already in flight land before the CTA exits
        mbar_wait(bar_a, 0, abort_flag);
        for (int i = max(0, issued - STAGES); i < issued; ++i) {
          for (int k = 0; k < kSpinLimit && !mbar_try_wait(bar_full(i % STAGES), (i / STAGES) & 1); ++k) {
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer; sweep 2: also stages the tile's row log-sum-exps ----------------
    // (fetched one tile ahead, so that the trip to memory runs under the tile before)
    constexpr int kLse = TN / 32;  // per lane
    struct alignas(4 * kLse) Lse {
      float x[kLse];
    };
    auto fetch_lse = [&](const Walk& w) {
      const float* src = a.lse2 + ((size_t)bi * a.n_q_head + hk * g + w.h) * P;
      const int q = w.qt * TN + lane * kLse;
      Lse v;
#pragma unroll
      for (int e = 0; e < kLse; ++e) v.x[e] = (q + e < P) ? -src[q + e] : -INFINITY;  // a query past the end attends to nothing
      return v;
    };
    Walk w = walk_begin();
    Lse lse_next = {};
    if (SWEEP == 2) lse_next = fetch_lse(w);
    ok = mbar_wait(bar_a, 0, abort_flag);
    for (int i = 0; ok && i < n_stream; ++i) {
      const int st = i % STAGES, buf = i & 1;
      ok = mbar_wait(bar_full(st), (i / STAGES) & 1, abort_flag);
      if (ok && i >= 2) ok = mbar_wait(bar_sfree(buf), ((i >> 1) - 1) & 1, abort_flag);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (lane == 0) {
        const uint32_t d_tmem = tmem_base + buf * TN;
#pragma unroll
        for (int k = 0; k < D / 16; ++k) {
          const uint32_t a_addr = s_u32(a_s + (k / 4) * kSubBytes) + (k % 4) * 32;
          const uint32_t b_addr = s_u32(b_s + st * TILE_BYTES + (k / 4) * STREAM_SUB) + (k % 4) * 32;
          umma_bf16(d_tmem, umma_desc(a_addr), umma_desc(b_addr), kIdesc, k > 0 ? 1u : 0u);
        }
        umma_commit(bar_empty(st));  // the stage may be refilled once these MMAs have read it
        umma_commit(bar_sfull(buf)); // the accumulator buffer is complete
      }
      __syncwarp();
      if (SWEEP == 2) {
        // (behind the products, which do not wait for them)
        *reinterpret_cast<Lse*>(lse_s + buf * TN + lane * kLse) = lse_next;
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_lse(buf));
        if (i + 1 < n_stream) {
          walk_next(w);
          lse_next = fetch_lse(w);
        }
      }
    }
  } else {
    // ---------------- accumulator drain: thread = one row of the fixed tile, 64 columns ----------------
    const int quarter = warp & 3;
    const int col0 = TN == 64 ? 0 : ((warp - 2) >> 2) * 64;  // of the 64 columns of every tile that this warp drains
    const int row = quarter * 32 + lane;
    const uint32_t s_addr = tmem_base + ((uint32_t)(quarter * 32) << 16) + col0;
    const unsigned long long scale2 = f32x2(scale_log2, scale_log2);
    unsigned long long acc_a, acc_b;  // of the tile, even and odd columns
    Walk w = walk_begin();
    // The tiles on the diagonal mask a part of their elements, the others none: they are separate
    // instantiations of the drain, so that tiles off the diagonal carry no compare / select per element.
    struct Tile {
      int buf, off;  // off: of the tile's first column from the fixed tile's first row
    };
    auto chunk = [&](auto diag_c, const Tile& t, uint32_t (&r)[32], int c0) {  // columns c0 .. c0+31 of the tile
      constexpr bool DIAG = decltype(diag_c)::value;
      if (SWEEP == 1) {
        if (DIAG) {
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (t.off + c0 + j > row) r[j] = 0xff800000u;  // key after the query: -inf
        }
        float mx = __uint_as_float(r[0]);
#pragma unroll
        for (int j = 1; j + 1 < 32; j += 2) mx = max3(mx, __uint_as_float(r[j]), __uint_as_float(r[j + 1]));
        const float m_new = fmaxf(m, fmaxf(mx, __uint_as_float(r[31])) * scale_log2);
        if (DIAG && m_new == -INFINITY) return;  // nothing of the row so far (second half of the first rows)
        if (m_new > m) {
          const float f = ex2(m - m_new);
          const unsigned long long f2 = f32x2(f, f), zero = f32x2(0.f, 0.f);
          acc_a = fma_f32x2(acc_a, f2, zero);
          acc_b = fma_f32x2(acc_b, f2, zero);
          sum *= f;
          m = m_new;
        }
        const unsigned long long neg_m2 = f32x2(-m, -m);
#pragma unroll
        for (int jp = 0; jp < 16; ++jp) {
          const unsigned long long x2 =
              fma_f32x2(f32x2(__uint_as_float(r[2 * jp]), __uint_as_float(r[2 * jp + 1])), scale2, neg_m2);
          // (a masked tile keeps to the form that gives an exact 0)
          const unsigned long long e2 = !DIAG && on_fma<D, SWEEP>(jp) ? ex2_pair_fma(x2) : ex2_pair_sfu(x2);
          if (jp & 1) acc_b = add_f32x2(acc_b, e2);
          else acc_a = add_f32x2(acc_a, e2);
        }
      } else {
        const ulonglong2* ls = reinterpret_cast<const ulonglong2*>(lse_s + t.buf * TN + c0);
#pragma unroll
        for (int j4 = 0; j4 < 8; ++j4) {
          const ulonglong2 lv = ls[j4];
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int jp = 2 * j4 + q;
            const unsigned long long x2 = fma_f32x2(f32x2(__uint_as_float(r[2 * jp]), __uint_as_float(r[2 * jp + 1])),
                                                    scale2, q ? lv.y : lv.x);
            unsigned long long e2 = on_fma<D, SWEEP>(jp) ? ex2_pair_fma(x2) : ex2_pair_sfu(x2);
            if (DIAG) {  // query before the key: no attention
              float e0, e1;
              f32x2_split(e2, e0, e1);
              e2 = f32x2(t.off + c0 + 2 * jp >= row ? e0 : 0.f, t.off + c0 + 2 * jp + 1 >= row ? e1 : 0.f);
            }
            if (q) acc_b = add_f32x2(acc_b, e2);
            else acc_a = add_f32x2(acc_a, e2);
          }
        }
      }
    };
    auto drain_tile = [&](auto diag_c, const Tile& t) {
      auto hand_back = [&]() {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_sfree(t.buf));
      };
      // (32 columns at a time: with the second half's load in flight under the first's exponentials the registers
      // held the FMA-pipe form back, 497 against 482 us a sweep at head_dim 64)
      acc_a = acc_b = f32x2(0.f, 0.f);
      uint32_t r[32];
      tmem_ld32_nowait(s_addr + t.buf * TN, r);
      tmem_wait_ld(r);
      chunk(diag_c, t, r, col0);
      __syncwarp();
      tmem_ld32_nowait(s_addr + t.buf * TN + 32, r);
      tmem_wait_ld(r);
      if (SWEEP == 1) hand_back();  // the tile is in registers: the tensor core may have the buffer back
      chunk(diag_c, t, r, col0 + 32);
      if (SWEEP == 2) hand_back();  // the buffer's lse staging is in use until here
      float a0, a1;
      f32x2_split(add_f32x2(acc_a, acc_b), a0, a1);
      sum += a0 + a1;
    };
    for (int i = 0; ok && i < n_stream; ++i) {
      const Tile t{i & 1, (w.qt - kTM / TN * row_tile) * TN};
      const bool diag = (unsigned)t.off < (unsigned)kTM;
      walk_next(w);
      if (SWEEP == 2) ok = mbar_wait(bar_lse(t.buf), (i >> 1) & 1, abort_flag);
      if (ok) ok = mbar_wait(bar_sfull(t.buf), (i >> 1) & 1, abort_flag);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (diag) drain_tile(std::true_type{}, t);
      else drain_tile(std::false_type{}, t);
    }
  }
  if (warp >= 2) {
    const int row = (warp & 3) * 32 + lane, row_idx = row_tile * kTM + row;  // query (sweep 1) / key (sweep 2)
    const bool second_half = warp >= 6;
    float l = sum;
    if constexpr (TN == 128) {
      // the two halves of a row meet in shared memory (the staging area is free once every drain
      // thread is past its last tile); every drain thread reaches both barriers, aborted or not
      __syncwarp();
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (second_half) {
        lse_s[2 * row] = m;
        lse_s[2 * row + 1] = l;
      }
      __syncwarp();
      asm volatile("bar.sync 1, 256;" ::: "memory");
      const float o0 = lse_s[2 * row], o1 = lse_s[2 * row + 1];
      if (SWEEP == 1) {
        // this half holds column 0 of every tile, so m is finite; the other half may be empty
        const float mm = fmaxf(m, o0);
        l = l * ex2(m - mm) + o1 * ex2(o0 - mm);
        m = mm;
      } else {
        l += o1;
      }
    }
    if (!second_half && ok && !*abort_flag && row_idx < P) {
      if (SWEEP == 1) {
        a.lse2[((size_t)bi * a.n_q_head + hq) * P + row_idx] = m + log2f(l);
      } else {
        float* dst = pc.n_piece == 1 ? a.acc_prompt : pc.partial + (size_t)piece * a.batch * a.n_kv_head * P;
        dst[((size_t)bi * a.n_kv_head + hk) * P + row_idx] = l;
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "n"(2 * TN) : "memory");
  }
  if (tid == 0 && *abort_flag) atomicOr(status, kStatusTimeout);
  if (SWEEP == 2 && pc.n_piece > 1) {
    // the key tile's last piece to finish adds all pieces up, in head order (no piece waits)
    __shared__ int s_last;
    if (tid == 0) {
      int* ticket = pc.tickets + ((size_t)bi * a.n_kv_head + hk) * n_tile + row_tile;
      __threadfence();
      s_last = atomicAdd(ticket, 1) == pc.n_piece - 1;
      if (s_last) *ticket = 0;
    }
    __syncthreads();
    const int key = row_tile * kTM + tid;
    if (s_last && tid < kTM && key < P) {
      __threadfence();
      const size_t at = ((size_t)bi * a.n_kv_head + hk) * P + key, stride = (size_t)a.batch * a.n_kv_head * P;
      float sum = 0.f;
#pragma unroll 8
      for (int p = 0; p < pc.n_piece; ++p) sum += __ldcg(pc.partial + at + p * stride);
      a.acc_prompt[at] = sum;
    }
  }
}

// ---------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

namespace tc {
bool make_tile_map(CUtensorMap* tm, const void* base, long long rows, int d, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)d, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)d * 2};
  cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
bool make_block_tile_map(CUtensorMap* tm, const void* base, long long blocks, int rows, int d, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)rows, (cuuint64_t)blocks};
  cuuint64_t strides[2] = {(cuuint64_t)d * 2, (cuuint64_t)rows * d * 2};
  cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
}  // namespace tc

template <int D, int TN, int STAGES>
static cudaError_t launch_tc_t(const ScoreArgs& a, int* status, cudaStream_t s) {
  // Blocks of the maps: a head's prompt.  (A query past the end of one has weight exp2(x - inf), which is 0 for a row of zeros; the
  // next head's query, if it is NaN or inf, would make it NaN.)
  CUtensorMap tm_q, tm_k;
  const long long q_heads = (long long)a.batch * a.n_q_head, k_heads = (long long)a.batch * a.n_kv_head;
  if (q_heads * a.prompt + kTM > 0x7fffffffLL) return cudaErrorNotSupported;
  CUtensorMap ts_q, ts_k;  // streamed
  auto map = [&](CUtensorMap* tm, const void* base, long long heads, int rows) {
    return tc::make_block_tile_map(tm, base, heads, a.prompt, D, rows);
  };
  if (!map(&tm_q, a.q, q_heads, kTM) || !map(&tm_k, a.k, k_heads, kTM)) return cudaErrorNotSupported;
  if (!map(&ts_q, a.q, q_heads, TN) || !map(&ts_k, a.k, k_heads, TN)) return cudaErrorNotSupported;
  constexpr size_t smem = 1024 + (size_t)(D / 64) * (kSubBytes + STAGES * TN * 128) + 8 * 16 + 16 + 2 * TN * 4;
  const float scale_log2 = 1.4426950408889634f / sqrtf((float)D);
  const int n_tile = (a.prompt + kTM - 1) / kTM;
  auto k1 = prefill_scores_tc_kernel<D, TN, STAGES, 1>;
  auto k2 = prefill_scores_tc_kernel<D, TN, STAGES, 2>;
  static PerDevice set_up;
  cudaError_t e = allow_smem(set_up, smem, k1, k2);
  if (e != cudaSuccess) return e;
  // Sweep 2 walks the heads of a group one after the other.  A launch of few key tiles and many heads
  // (71 heads on one KV head) would be over when its longest CTA is: it is cut into pieces of `heads`
  // heads so that the longest CTA has at most about a quarter of a CTA slot's share of the work.
  // Measured, us per layer, one CTA per key tile / cut: 2 sequences of 5003 tokens, 71 heads on one KV
  // head (80 key tiles): 3283 / 559; 1 sequence of 777, 32 on 8: 37 / 15; 4 of 4096, 32 on 8: 410 / 395.
  ScorePieces pc;
  const int g = a.n_q_head / a.n_kv_head;
  const long long units = (long long)a.batch * a.n_kv_head;
  const long long slots = 2LL * sm_count();  // (of 128 columns; finer pieces for the CTAs of 64 were slower, 497 against 488 us)
  long long heads = std::max(1LL, std::min((long long)g, units * g * (n_tile + 1) / (8 * slots)));
  auto pieces = [&](long long h) { return (g + h - 1) / h; };
  while (heads < g && (pieces(heads) * units * a.prompt > (long long)a.partial_floats || pieces(heads) * n_tile > 65535)) ++heads;
  pc.heads = (int)heads;
  pc.n_piece = (int)pieces(heads);
  pc.partial = a.partial;
  pc.tickets = a.tickets;
  // Short launches start while the one ahead runs out; where CTAs are longer than a few tiles those that start early crowd the
  // SMs that are done first.  us per layer, after / chained: 71 / 1 heads of 64, 1 sequence of 128 tokens 22.7 / 17.4, 512: 31.1 /
  // 27.3, 700: 38.0 / 36.8, 1000: 49.4 / 52.7; 2 heads, 4 of 4000 72 / 82.
  const bool chained = n_tile <= 6;
  auto go = [&](auto kern, dim3 grid, const CUtensorMap& rows, const CUtensorMap& stream) {
    if (chained) return launch_chained(kern, grid, prefill_threads(TN), smem, s, rows, stream, a, pc, scale_log2, status);
    kern<<<grid, prefill_threads(TN), smem, s>>>(rows, stream, a, pc, scale_log2, status);
    return cudaGetLastError();
  };
  e = go(k1, dim3(a.n_q_head, a.batch, n_tile), tm_q, ts_k);
  return e != cudaSuccess ? e : go(k2, dim3(a.n_kv_head, a.batch, n_tile * pc.n_piece), tm_k, ts_q);
}

// Returns cudaErrorNotSupported when the shape or the driver cannot serve the tensor-core path.
cudaError_t launch_prefill_scores_tc(const ScoreArgs& a, int* status, cudaStream_t s) {
  if (a.n_q_head > 65535 || a.batch > 65535 || (a.prompt + kTM - 1) / kTM > 65535) return cudaErrorNotSupported;
  if ((reinterpret_cast<uintptr_t>(a.q) | reinterpret_cast<uintptr_t>(a.k)) & 15u) return cudaErrorNotSupported;
  // Tiles of 64 columns put four CTAs with four drain warps each on an SM; a launch that fills no more than two of them is over
  // sooner with eight warps per CTA.  us per layer, 64 / 128 columns, by CTAs of sweep 1: 32 (1 sequence of 4096, one head) 95 / 66, 256
  // (4 of 4000, two) 101 / 79, 284 28.1 / 26.6, 296 40 / 34, 300 27.9 / 28.1, 568 48.0 / 49.4, 1136 73 / 80.
  const long long ctas = (long long)a.n_q_head * a.batch * ((a.prompt + kTM - 1) / kTM);
  if (a.head_dim == 64) return ctas > 2LL * sm_count() ? launch_tc_t<64, 64, 3>(a, status, s) : launch_tc_t<64, 128, 4>(a, status, s);
  if (a.head_dim == 128) return launch_tc_t<128, 128, 2>(a, status, s);
  return cudaErrorNotSupported;
}

}  // namespace sq
