// Launch parameters shared by the host side of the library and its kernels.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cstdint>

#include "ebd.h"
#include "lm_params.h"

namespace ebd {

// Checked builds (compiled with -DEBD_CHECKS): a global access whose index
// comes from device data (row offsets, positions, counts) is preceded by a
// check of the index against the buffer's extent; a failed check records
// EBD_ERR_BOUNDS in the status word and the access is skipped (nothing traps
// or waits).  In other builds the check compiles away.
__device__ __forceinline__ bool in_bounds(long long i, long long n, int* status) {
#ifdef EBD_CHECKS
  if (i >= 0 && i < n) return true;
  if (status != nullptr) atomicCAS(status, 0, EBD_ERR_BOUNDS);
  return false;
#else
  (void)i;
  (void)n;
  (void)status;
  return true;
#endif
}

constexpr int kMaxWindow = 64;        // window rows per sequence in the block-window setting
constexpr int kMaxSeqRows = 512;      // in the full-sequence setting
constexpr int kUnit = 64;             // vocabulary rows per work unit of the LM head
constexpr int kLmThreads = 320;  // TMA warp, MMA warp, two epilogue warpgroups of 4 warps
constexpr int kMaxGroupRows = 512;    // rows per LM-head launch (TMEM: 512 columns)
constexpr int kRowsThreads = 256;
constexpr int kAttnThreads = 128;
constexpr int kAttnChunk = 64;        // keys per K/V tile
constexpr int kAttnStages = 3;        // at most
constexpr int kMaxAttnSplits = 8;
constexpr int kAttnParts = 4;         // split tiles per SM that the attention's partials hold, at most
constexpr int kAttnTcThreads = 352;   // tcgen05 attention: K and V load warps, MMA warp, 8 softmax warps
constexpr int kAttnTcRows = 64;       // query rows per tile of the tcgen05 attention

// ------------------------------------------------------------------ attention
struct AttnParams {
  int B, Hq, Hkv, D, group;
  int R;                    // rows of the step (extent of q and out)
  int max_prefix;
  int max_qtiles, splits;   // key splits of a tile with at least
  int split_from;           // split_from chunks of keys; the others have one
  int stages;               // ring of the mma.sync kernel: kAttnStages, or 2 for three CTAs per SM
  int two;                  // at most two of its CTAs per SM, whatever they take
  int tc;                   // 1: the tcgen05 kernel, 0: the mma.sync kernel (64-row tiles)
  const int* cu_rows;
  const int* prefix_len;
  const int* suffix;        // [B][2] {s0, S} cached keys after the window, or null
  const __nv_bfloat16* q;   // [R][Hq][D]
  float* out;               // [R][Hq][D]
  float* part;              // [B*Hkv*max_qtiles*splits][tile rows][D] unnormalised O
  float* part_ml;           // [B*Hkv*max_qtiles*splits][tile rows][2] (max, sum) in log2 units
  int* tickets;             // [B*Hkv*max_qtiles]
  int* status;
  uint64_t limit_ns;
  int wait_prior;           // every CTA waits for the grid it depends on before exiting
  const unsigned* ready;     // non-null: q and the window K/V are being copied in by
  unsigned ready_ticket;    // another stream, which then writes ready_ticket to *ready
};

// ------------------------------------------------------------------ decision
// Rows of the decision's scratch.  A sequence of n rows takes ceil(n / 8) whole
// groups of 8 from scratch_row on: of the b sequences before it at most
// min(b, r0) hold a row, and each of those ends in at most one part of a group.
// A launch within max_rows and max_batch thus stays below scratch_rows, which
// counts no more sequences than rows (65535 sequences of 4096 rows: 36864).
__host__ __device__ inline int scratch_row(int r0, int b) { return 8 * (r0 / 8 + (b < r0 ? b : r0)); }
inline int scratch_rows(int max_rows, int max_batch) {
  return 8 * (max_rows / 8 + (max_batch < max_rows ? max_batch : max_rows));
}

struct RowsParams {
  int B, R, V, grid_lm;     // grid_lm: LM-head partials per row
  int features_in;          // 1: s_conf/s_ent/s_gap/s_arg are inputs
  int cap;                  // rows per sequence the launch has to hold: 32, 64 or kMaxSeqRows
  int strict;               // cu_rows[B] has to be R
  int warm;                 // launched behind the LM head: first passes on stand-in rows
  int spare_row;            // a row of s_* that no window row uses
  int mode, top_m, gen_len, g_max, l_min, l_b, eos_id, lps_enabled;
  float tau, tau_psi, inv_log_v;
  const int* cu_rows;
  const int* row_pos;
  const float4* part_f;
  const int* part_i;
  const int* tokens;        // decode state in: read before the LM head's grid completes
  const uint8_t* mask;
  const uint8_t* in_block;
  const int* blk_meta;
  int* tokens_out;          // decode state out: the same buffers as the state in,
  uint8_t* mask_out;        // unless the state in is a staged copy of the caller's
  uint8_t* in_block_out;
  int* blk_meta_out;
  float *conf, *entropy, *ent_norm, *gap, *lbs_logit, *lps_prob;  // outputs, may be null
  int* argmax;
  uint8_t* accepted;
  float *s_conf, *s_ent, *s_gap;  // statistics of every row [R]: scratch, or inputs
  int* s_arg;
  const uint4* mat;         // router image (rows_image.h)
  const float* vec;
  const float* tok_table;   // [V][64]
  int cap_rows;             // rows of the scratch below (scratch_rows)
  __nv_bfloat16* kv;        // LBS keys and values [2 layers][2][planes][cap_rows][128]
  __nv_bfloat16* kvp;       // windows of more than 64 rows: LPS keys and values [2 blocks][2][planes][cap_rows][32]
  float* z;                 // and, between launches, LBS activations [cap_rows][128]
  __nv_bfloat16* q;         // and queries [planes][cap_rows][128]
  float *O, *P;             // [cap_rows] LBS logits by rank in M, p_psi by rank in B n M
  int* status;
};

// host launchers (defined next to their kernels)
cudaError_t launch_lm_stats(const CUtensorMap& tmap_w, const CUtensorMap& tmap_h,
                            const LmParams& p, cudaStream_t st);
int lm_grid(int num_sms, int n_units);       // CTAs of the unpaired LM head
int lm_pair_grid(int num_sms, int n_units);  // CTAs of the paired (cta_group::2) LM head
// rows of an LM-head launch from which CTA pairs run it (and up to kMaxGroupRows)
constexpr int kLmPairMinRows = 65;
void lm_plan(LmParams& p, int rows, int V, int d, int num_sms, bool pair = false);
// pdl: launched as a programmatic dependent of the kernel before it on
// `st` (that kernel's CTAs release it early; the attention reads nothing the
// earlier kernel writes)
cudaError_t launch_attention(const CUtensorMap& kc, const CUtensorMap& vc, const CUtensorMap& kw,
                             const CUtensorMap& vw, const AttnParams& p, cudaStream_t st,
                             bool pdl = false);
// the decision, the rows of a sequence split over a cluster of CTAs
// (k_decide.cu)
struct DecideSlots {        // clusters that fit the GPU at once
  int c8, c4;               // windows of up to 64 rows: of 8 and of 4 CTAs
  int wide16, wide8, wide4; // of more: of 16, 8 and 4
};
cudaError_t decide_rows_configure(DecideSlots& n);
cudaError_t launch_decide_rows(const RowsParams& p, const DecideSlots& n, cudaStream_t st, bool pdl);
// vocabulary-parallel LM head: one state per row from a launch's partials,
// and the statistics from the states of several shards (k_stats.cu)
cudaError_t launch_shard_state(const float4* part_f, const int* part_i, int rows, int grid,
                               float* state, cudaStream_t st);
cudaError_t launch_merge_shards(const float* states, int shards, int rows, int V, float inv_log_v,
                                float* conf, float* entropy, float* ent_norm, float* gap,
                                int* argmax, int* status, cudaStream_t st);
// prefix-cache append on commit: window row r of sequence b with mask[r] == 0
// is copied (K and V, Hkv * D bf16 each) to cache position row_pos[r] < Pmax
cudaError_t launch_kv_append(uint16_t* k_cache, uint16_t* v_cache, const uint16_t* k_win,
                             const uint16_t* v_win, const int* cu_rows, const int* row_pos,
                             const uint8_t* mask, int B, int rows, int Pmax, int hkvd,
                             cudaStream_t st, bool pdl);
cudaError_t launch_pack_lm(const __nv_bfloat16* w, __nv_bfloat16* out, int V, int d,
                           cudaStream_t st);
cudaError_t launch_fold_tok(const __nv_bfloat16* w_tok, const __nv_bfloat16* w_emb, float* table,
                            int V, int d_base, cudaStream_t st);

}  // namespace ebd
