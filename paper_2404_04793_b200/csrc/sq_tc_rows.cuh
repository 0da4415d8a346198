// Softmax role of the wide-group decode kernels: p = exp2(s * scale - m_ref) for one 128-token tile, from the
// accumulators S in tensor memory to bf16 weights P in tensor memory, by four warps.
//
// A warp reaches only the 32 tensor-memory lanes of its quarter and runs on the scheduler of the same
// number, so the heads are laid out to give the four schedulers the same work: groups of eight heads
// go to the quarters in turn (group j: quarter j % 4, lanes 8 * (j / 4) ...).  The 16-lane shapes of
// tcgen05.ld / st give thread t the columns 8k + 2(t%4), +1 of the rows t/4 and t/4 + 8: four threads
// share a row, and every lane of a warp has a head's weight to work on.  With 71 heads the special-function
// unit of a scheduler is busy for 512 cycles per tile (768 in the quarter with the ninth group); with a
// thread per row and the heads on lanes 0..70 two schedulers took 1024 and one idled.
// Measured, us per token, 32 layers, one launch per layer, thread per row / this: 224 sequences of 16384, 50 %
// 3855 / 3663 (at the board's power limit); 33 sequences of 8191, 50 %, H2O 1328 / 1278.
#pragma once
#include "sq_tc.cuh"

namespace sq {
namespace tc {

constexpr float kMaxWeight = 65536.f;  // 2^16

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// The layout turns by one quarter with the CTA's wave number: where one quarter has a group more than
// the others, the two CTAs of an SM have it on different schedulers (with a B200's 148 SMs; any other turn gives the same
// results).
struct WideLayout {
  int rot;
  __device__ __forceinline__ explicit WideLayout(int turn) : rot(turn & 3) {}
  static __device__ __forceinline__ int wave() { return blockIdx.x / 148; }
  // head of tensor-memory lane `lane` of a quarter
  __device__ __forceinline__ int head_of_lane(int quarter, int lane) const {
    return 8 * (4 * (lane >> 3) + ((quarter - rot) & 3)) + (lane & 7);
  }
  // row of the Q tile in which group j of eight heads starts
  __device__ __forceinline__ int row_of_group(int j) const { return 32 * ((j + rot) & 3) + 8 * (j >> 2); }
  // groups of eight heads in a quarter
  __device__ __forceinline__ int groups(int quarter, int n_head) const { return ((n_head + 7) / 8 - ((quarter - rot) & 3) + 3) / 4; }
};

// State of one softmax warp.  SLOTS: most groups of eight heads in a quarter (3: up to 96 heads, 4: 128).
template <bool H2O, int SLOTS>
struct WideRows {
  uint32_t s_addr, p_addr, o_addr;  // S, P, O of the quarter's first lane
  float scale_log2;
  int lane, n_slot;
  // by slot, of the row lane / 4 of the slot's eight: the reference (equal in the row's four threads) and
  // this thread's part of the sums of the weights, exact (H2O) and as rounded to bf16; t_*: of the tile
  float m[SLOTS], l[SLOTS], l_w[SLOTS], t_l[SLOTS], t_w[SLOTS];

  __device__ __forceinline__ void begin() {
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      m[s] = -INFINITY;
      l[s] = l_w[s] = t_l[s] = t_w[s] = 0.f;
    }
  }
  // columns at or past n_valid count for nothing
  __device__ __forceinline__ void mask(uint32_t (&r)[32], int c, int n_valid) const {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int col = c * 64 + 8 * k + 2 * (lane & 3);
      if (col >= n_valid) r[4 * k] = r[4 * k + 2] = 0xff800000u;
      if (col + 1 >= n_valid) r[4 * k + 1] = r[4 * k + 3] = 0xff800000u;
    }
  }
  static __device__ __forceinline__ float row_max(const uint32_t (&r)[32], int b, float mx) {
#pragma unroll
    for (int k = 0; k < 8; ++k) mx = max3(mx, __uint_as_float(r[4 * k + b]), __uint_as_float(r[4 * k + b + 1]));
    return mx;
  }
  // maximum over the four threads of a row
  static __device__ __forceinline__ float quad_max(float x) {
    x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 1));
    return fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 2));
  }
  // the rows' maxima over the tile's valid tokens, log2 domain
  __device__ __forceinline__ void tile_max(int n_valid, float (&mx)[SLOTS]) {
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) mx[s] = -INFINITY;
#pragma unroll
    for (int hf = 0; hf < (SLOTS + 1) / 2; ++hf) {
      if (2 * hf >= n_slot) continue;
#pragma unroll 1
      for (int c = 0; c < 2; ++c) {
        uint32_t r[32];
        tmem_ld16x256_x8_nowait(s_addr + ((uint32_t)(16 * hf) << 16) + c * 64, r);
        tmem_wait_ld(r);
        if (n_valid < kTM) mask(r, c, n_valid);
        mx[2 * hf] = row_max(r, 0, mx[2 * hf]);
        if (2 * hf + 1 < SLOTS) mx[(2 * hf + 1) % SLOTS] = row_max(r, 2, mx[(2 * hf + 1) % SLOTS]);
      }
    }
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) mx[s] = quad_max(mx[s]) * scale_log2;
  }
  // 64 columns (tokens) of the rows of slot A and, with TWO, of slot B, which are eight lanes apart
  template <bool TWO>
  __device__ __forceinline__ void chunk(const uint32_t (&r)[32], uint32_t (&pk)[16], float m_a, float m_b, unsigned long long& l_a,
                                        unsigned long long& l_b, float (&w)[4]) {
    const unsigned long long scale2 = f32x2(scale_log2, scale_log2), na2 = f32x2(-m_a, -m_a), nb2 = f32x2(-m_b, -m_b);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        if (b == 1 && !TWO) {
          pk[2 * k + 1] = 0u;
          continue;
        }
        float p0, p1;
        f32x2_split(fma_f32x2(f32x2(__uint_as_float(r[4 * k + 2 * b]), __uint_as_float(r[4 * k + 2 * b + 1])), scale2, b ? nb2 : na2),
                    p0, p1);
        p0 = ex2(p0);
        p1 = ex2(p1);
        if (H2O) {
          if (b) l_b = add_f32x2(l_b, f32x2(p0, p1));
          else l_a = add_f32x2(l_a, f32x2(p0, p1));
        }
        const uint32_t u = pack_bf16x2(p0, p1);
        w[2 * b] = add_bf16_lo(w[2 * b], u);
        w[2 * b + 1] = add_bf16_hi(w[2 * b + 1], u);
        pk[2 * k + b] = u;
      }
    }
  }

  // The tile's weights of the slots 2 * HF (and 2 * HF + 1).  LAST: nothing of S is read after this, so it is
  // handed back before its last 64 columns are worked out, unless the tile may have to be redone;
  // returns whether it was.
  // p_free() waits for the product that still reads the tile before's P: before the first store only, so
  // that the first 64 columns are worked out meanwhile.
  // SCALES: p_free() may also have O to scale, for which the load in flight has to be complete.
  template <int HF, bool TWO, bool LAST, bool SCALES, class PFree>
  __device__ __forceinline__ bool half(int n_valid, bool first, uint32_t bar_sfree, bool wait_p, PFree p_free) {
    constexpr int A = 2 * HF, B = TWO ? 2 * HF + 1 : 2 * HF;
    const uint32_t s = s_addr + ((uint32_t)(16 * HF) << 16), p = p_addr + ((uint32_t)(16 * HF) << 16);
    unsigned long long la = f32x2(0.f, 0.f), lb = la;
    float w[4] = {0.f, 0.f, 0.f, 0.f};
    uint32_t ra[32], rb[32];
    tmem_ld16x256_x8_nowait(s, ra);
    tmem_wait_ld(ra);
    tmem_ld16x256_x8_nowait(s + 64, rb);
    if (n_valid < kTM) mask(ra, 0, n_valid);
    if (first) {
      // The reference: the maximum of the tile, so that a unit of one tile has its largest weight at 1, which bf16
      // holds exactly (the maximum of 64 columns put the outputs 2 to 7 % further from fp64).
      tmem_wait_ld(rb);
      if (n_valid < kTM) mask(rb, 1, n_valid);
      m[A] = quad_max(row_max(rb, 0, row_max(ra, 0, -INFINITY))) * scale_log2;
      if (TWO) m[B] = quad_max(row_max(rb, 2, row_max(ra, 2, -INFINITY))) * scale_log2;
    }
    uint32_t pk[16];
    chunk<TWO>(ra, pk, m[A], m[B], la, lb, w);
    if (SCALES && wait_p) tmem_wait_ld(rb);
    if (wait_p) p_free();
    tmem_st16x128_x8_u32(p, pk);
    tmem_wait_ld(rb);
    if (n_valid < kTM) mask(rb, 1, n_valid);
    bool released = false;
    if (LAST) {
      // 16 weights of at most 2^10 and 2^15 before them stay below kMaxWeight
      bool safe = w[0] + w[1] <= 32768.f && fmaf(row_max(rb, 0, -INFINITY), scale_log2, -m[A]) <= 10.f;
      if (TWO) safe = safe && w[2] + w[3] <= 32768.f && fmaf(row_max(rb, 2, -INFINITY), scale_log2, -m[B]) <= 10.f;
#pragma unroll
      for (int q = 2; q < SLOTS; ++q)
        if (HF == 0) safe = safe && t_w[q] <= kMaxWeight;
      released = __all_sync(0xffffffffu, safe);
      if (released) {
        tc_fence_before();
        if (lane == 0) mbar_arrive(bar_sfree);
      }
    }
    chunk<TWO>(rb, pk, m[A], m[B], la, lb, w);
    tmem_st16x128_x8_u32(p + 32, pk);
    float s0, s1;
    f32x2_split(la, s0, s1);
    t_l[A] = s0 + s1;
    t_w[A] = w[0] + w[1];
    if (TWO) {
      f32x2_split(lb, s0, s1);
      t_l[B] = s0 + s1;
      t_w[B] = w[2] + w[3];
    }
    return released;
  }
  // A whole tile; returns whether S was handed back.  A row's weights are too large when one of its
  // threads' sums is: redo() follows.
  template <bool SCALES = false, class PFree>
  __device__ __forceinline__ bool tile(int n_valid, bool first, uint32_t bar_sfree, PFree p_free) {
    const bool upper = n_slot >= 3;
    if (SLOTS == 4 && n_slot == 4) half<1, SLOTS == 4, false, SCALES>(n_valid, first, bar_sfree, true, p_free);
    else if (upper) half<1, false, false, SCALES>(n_valid, first, bar_sfree, true, p_free);
    const bool released = n_slot >= 2 ? half<0, true, true, SCALES>(n_valid, first, bar_sfree, !upper, p_free)
                                      : half<0, false, true, SCALES>(n_valid, first, bar_sfree, !upper, p_free);
    tmem_wait_st();
    return released;
  }
  __device__ __forceinline__ bool too_large() const {
    float w = 0.f;
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) w = fmaxf(w, t_w[s]);
    return __any_sync(0xffffffffu, w > kMaxWeight);
  }
  __device__ __forceinline__ void add_tile() {
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      l[s] += t_l[s];
      l_w[s] += t_w[s];
    }
  }
  // the value that the threads of this lane's row hold
  __device__ __forceinline__ float of_lane(const float (&v)[SLOTS]) const {
    float x = 0.f;
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      const float y = __shfl_sync(0xffffffffu, v[s], (lane & 7) * 4);
      if ((lane >> 3) == s) x = y;
    }
    return x;
  }
  // Rare: moves the reference of the rows that need it; O and the sums (complete up to the tile before, and
  // no product running) shrink with it.  The tile is then done again.
  __device__ __forceinline__ void redo(int n_valid) {
    float mx[SLOTS], f[SLOTS];
    tile_max(n_valid, mx);
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      const bool need = __any_sync(0xfu << (lane & 28), t_w[s] > kMaxWeight);
      f[s] = need ? ex2(m[s] - mx[s]) : 1.f;
      l[s] *= f[s];
      l_w[s] *= f[s];
      if (need) m[s] = mx[s];
    }
    float f_o = of_lane(f);
    if ((lane >> 3) >= n_slot) f_o = 1.f;
    scale_o(f_o);
  }
  // Ahead of a tile: the references of the rows that have their largest logit so far in it move there, and the sums shrink with
  // them.  Returns whether any did; O is to be multiplied by f_o once the tile before's product is complete.
  __device__ __forceinline__ bool follow(int n_valid, float* f_o) {
    float mx[SLOTS], f[SLOTS];
    bool up = false;
    tile_max(n_valid, mx);
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      const bool rise = s < n_slot && mx[s] > m[s];
      f[s] = rise ? ex2(m[s] - mx[s]) : 1.f;
      l[s] *= f[s];
      l_w[s] *= f[s];
      if (rise) m[s] = mx[s];
      up = up || rise;
    }
    *f_o = of_lane(f);
    return __any_sync(0xffffffffu, up);
  }
  // O times this lane's factor
  __device__ __forceinline__ void scale_o(float f_o) {
#pragma unroll 1
    for (int c = 0; c < 2; ++c) {
      float o[32];
      tmem_ld32(o_addr + c * 32, o);
#pragma unroll
      for (int j = 0; j < 32; ++j) o[j] *= f_o;
      tmem_st32(o_addr + c * 32, o);
    }
  }
  // Sums over the rows' four threads, brought with the references to the lanes that hold the rows.
  __device__ __forceinline__ void finish(float* ref, float* sum, float* sum_w) {
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      l[s] += __shfl_xor_sync(0xffffffffu, l[s], 1);
      l[s] += __shfl_xor_sync(0xffffffffu, l[s], 2);
      l_w[s] += __shfl_xor_sync(0xffffffffu, l_w[s], 1);
      l_w[s] += __shfl_xor_sync(0xffffffffu, l_w[s], 2);
    }
    *ref = of_lane(m);
    *sum = of_lane(l);
    *sum_w = of_lane(l_w);
  }
};

}  // namespace tc
}  // namespace sq
