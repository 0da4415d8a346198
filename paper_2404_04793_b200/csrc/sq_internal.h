// Internal declarations shared by the libsq translation units (host context + kernel launchers).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "sq.h"
#include "sq_device_state.h"

namespace sq {

constexpr int kMaxLayers = 256;
constexpr int kMaxImportanceCtas = 4096;  // partial sums of one importance launch
constexpr int kMaxGroup = 128;          // query heads per KV head
constexpr int kTargetItems = 148 * 16;  // room for split-K pieces beyond one per (layer, unit)

// Per-layer cache geometry, resident in device memory once the budgets are known.
// k/v/pos/acc/victim offsets are BYTES from the pool base; logit_off and lse_off count floats from the
// start of the logits area of the workspace.
struct LayerDesc {
  long long k_off, v_off, pos_off, acc_off, victim_off, logit_off;
  long long lse_off;      // H2O: [unit][group] row log-sum-exps for the score pass of wide groups
  int b;                  // budget: tokens kept per unit
  int cap;                // slots per unit (b rounded up to page_tokens)
  int b_heavy, b_recent;  // H2O split of b
  int ring_base;          // Sliding Window 0, StreamingLLM n_sink: slots below it never rotate
  int ring_origin;        // the position that maps to slot ring_base
};

// Slot of position x in a ring-managed (Sliding Window / StreamingLLM) cache.
__host__ __device__ inline int ring_slot(int x, int b, int base, int origin) {
  if (x < base) return x;
  return base + (x - origin) % (b - base);
}

struct ImportanceArgs {
  const void* a;
  const void* b;
  void* sum_out;         // fused form: receives a + b (rounded to the dtype), which then plays the part of b; else null
  long long n_tok;
  int hidden;
  double* cta_partial;   // [n_cta]
  unsigned int* ticket;  // zero on entry, zero again on exit
  double* cos_sum;       // += sum over tokens of the cosine
};

struct AllocateArgs {  // entry of layer i: [i * stride + blockIdx.x] (one CTA per budget vector); budget, is_g3: page-locked host memory
  const double* cos_sum;
  long long tok_count[kMaxLayers];  // by layer
  int n_layer, n_cluster, stride;
  long long b_init;
  double p;
  float* cos_sim;
  int* budget;
  unsigned char* is_g3;
};

struct GatherArgs {  // prompt rows -> cache slots of one layer (all its descriptors in one launch)
  const void* k_prompt;
  const void* v_prompt;
  char* pool;
  const LayerDesc* descs;   // the layer's descriptors (device); unit u belongs to descs[u / units_per_desc]
  int units_per_desc;
  int n_unit, prompt, max_keep, policy, head_dim;
  const float* scores;      // H2O: [n_unit][prompt]
  int max_fixed, max_heavy; // H2O: most slots of a descriptor that need no selection, and that do
  bool own_copy;            // H2O: the selecting CTA copies the heavy rows of its unit
};

struct ScoreArgs {  // H2O prompt scores of one layer
  const void* q;
  const void* k;
  float* lse2;        // [B, Hq, P]  log2-domain row log-sum-exp
  float* acc_prompt;  // [B, Hkv, P]
  int batch, n_q_head, n_kv_head, prompt, head_dim;
  float* partial;       // scratch for the column sums of a key tile's pieces, partial_floats of it (0: no pieces)
  size_t partial_floats;
  int* tickets;         // [B * Hkv][key tiles of 64 or 128] arrival counters, zero between launches
};
// How sweep 2 of the prompt scores is cut: pieces of `heads` query heads of a group; with more than
// one piece, piece p's column sums go to partial + p * B * Hkv * P and the last to finish adds them.
struct ScorePieces {
  int heads, n_piece;
  float* partial;
  int* tickets;
};

// "Layer" below means one cache descriptor: a layer of the whole batch, or, with per-sequence
// budgets, a (layer, sequence) pair holding that sequence's n_kv_head units (batch = 1 then).
struct DecodeArgsBase {
  const LayerDesc* layers;
  const int* order;  // the launch's descriptors, n_layer_total of them, in launch order (largest budget first)
  char* pool;
  float* logits;
  float* part_stat;  // [item][group][4]   (max, sum, sum of rounded weights, pad) in the log2 domain
  float* part_o;     // [item][group][head_dim]
  const void* q;
  const void* k_new;
  const void* v_new;
  void* out;
  int* status;
  int* tickets;  // [n_layer_total][n_unit] arrival counters of the split-K pieces, zero between launches
  int n_layer_total, layer_begin, layer_end;
  int n_tok;  // tokens seen before this step == position of the new token
  int batch, n_q_head, n_kv_head, head_dim, group;
  int n_unit;  // batch * n_kv_head
  int split_tokens, policy;
  int uniform;  // every descriptor of the launch has n_unit items (no split-K): items are found in O(1)
  int has_logits;  // H2O: the workspace holds the per-slot logits the kernels other than the tcgen05 pair need
  float scale_log2;  // log2(e) / sqrt(head_dim)
  int early;  // the launch before this one touched none of these layers: their cache may be read ahead of grid_wait()
};
// With split-K: items before the k-th descriptor of the launch (k <= n_layer_total <= kMaxLayers).
// Rides in the kernel parameters, so a lookup is a binary search in constant memory; the kernel
// build for launches without split-K takes the base only (1 KB less to pass per launch).
struct DecodeArgs : DecodeArgsBase {
  int cum[kMaxLayers + 1];
};

struct EvictLayer {  // one layer of an explicit eviction
  LayerDesc ld_old, ld_new;
  int len, n_tok;
};

struct EvictArgs {
  char* pool;
  const EvictLayer* tab;  // [n_layers] in device memory
  int n_layers, max_cap;
  int n_unit, policy, n_sink, row_bytes;
  int* status;
};

// Launch of a kernel that starts while the one before it in the stream is still running out
// (programmatic dependent launch): it may start once every CTA of that kernel has passed its own
// grid_wait(), and what it does ahead of its own grid_wait() (setting up, reading what older launches
// wrote) overlaps that kernel's tail.
// Measured per generated token, one launch (H2O: two) per layer, without / with it: 32 layers, 32 / 8 heads of
// 128, H2O: 1 sequence 580 / 388 us, 16 sequences 825 / 661 us; 32 / 32 heads, 8 sequences 552 / 474 us; 80 layers,
// 64 / 8 heads, 32 sequences 2651 / 2397 us; 71 / 1 heads of 64, 33 sequences, H2O 1507 / 1331 us.
template <typename... P, typename... A>
inline cudaError_t launch_chained_cluster(void (*kern)(P...), int cluster, dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                          A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}
template <typename... P, typename... A>
inline cudaError_t launch_chained(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
  return launch_chained_cluster(kern, 1, grid, block, smem, s, std::forward<A>(args)...);
}

// Launchers: each returns the cudaError_t of its launches.
cudaError_t launch_importance(const ImportanceArgs& a, int dtype, int n_sm, cudaStream_t s);
cudaError_t launch_allocate(const AllocateArgs& a, cudaStream_t s);
cudaError_t launch_fill_cache(const GatherArgs& a, int dtype, bool any_full, cudaStream_t s);
cudaError_t launch_prefill_scores(const ScoreArgs& a, int dtype, int* status, cudaStream_t s);
cudaError_t launch_prefill_scores_alu(const ScoreArgs& a, int dtype, cudaStream_t s);
cudaError_t launch_prefill_scores_tc(const ScoreArgs& a, int* status, cudaStream_t s);
// Attention kernel of a launch over n_desc descriptors of n_unit units, the longest of max_len slots.
enum class DecodeKernel { kTcgen05, kMma, kPipe };  // wide groups; mma.sync; fp32 pipes
DecodeKernel decode_kernel_for(int dtype, int head_dim, int group, int n_desc, int n_unit, int max_len, bool h2o);
// desc_tiles: per descriptor of the launch (launch order) the 128-token tiles of one unit; max_len: slots of the longest unit
cudaError_t launch_decode(const DecodeArgs& a, int dtype, int n_items, bool need_combine, size_t pool_bytes,
                          size_t q_rows, const int* desc_tiles, int max_len, cudaStream_t s);
cudaError_t launch_decode_attn_tc(const DecodeArgs& a, int n_items, size_t pool_bytes, size_t q_rows, cudaStream_t s);
cudaError_t launch_decode_attn_tc_cluster(const DecodeArgs& a, const int* desc_tiles, size_t pool_bytes, size_t q_rows,
                                          cudaStream_t s);
cudaError_t launch_decode_attn_tc_stream(const DecodeArgs& a, const int* desc_tiles, size_t pool_bytes, size_t q_rows,
                                         cudaStream_t s);
cudaError_t launch_h2o_gain_tc(const DecodeArgs& a, int n_items, size_t pool_bytes, size_t q_rows, cudaStream_t s);
cudaError_t launch_decode_attn_mma(const DecodeArgs& a, int n_items, cudaStream_t s);
// groups of at most 8 heads; pieces > 0: H2O with the score update, that many CTAs per unit
cudaError_t launch_decode_mma_low(const DecodeArgs& a, int n_items, int pieces, size_t logit_bytes, cudaStream_t s);
cudaError_t launch_decode_mma_scores(const DecodeArgs& a, int max_len, cudaStream_t s);
cudaError_t launch_evict(const EvictArgs& a, cudaStream_t s);

}  // namespace sq
