// Internal interface between the surrogate / compaction code and the fused
// LM-head entry point.
#pragma once

#include "pace_internal.cuh"

namespace pace {

struct SurrogateWs {
  double* seq_sum;    // SEQ_MEAN: per sequence, the part in the tile it begins in
  double* seq_cnt;
  double* head_sum;   // SEQ_MEAN: per tile, the part of a sequence that began earlier
  double* head_cnt;
  double* block_sum;  // TOKEN_MEAN: per block
  double* block_cnt;
  float* adv;
  unsigned* counter;  // finished blocks
};

struct RowCounts {
  long long* block;  // rows in the loss per block of the row walk,
  int* warp;         // and per warp
};

struct CompactWs {
  RowCounts counts;
  long long* total;     // M, the number of rows in the loss
  int32_t* rowidx;      // [n_rows]: compact row -> original row
};

// The group advantages of a call, computed by some blocks of a launch (adv_blocks).
struct AdvJob {
  const float* reward;
  const uint8_t* accepted;
  int64_t n_groups;  // 0: none
  int G;
  int L;             // lanes per group, or 0: a thread per group
  double eps;
  int unbiased;
  float* adv;
};

// Workspace of the log-prob pipeline (compaction, gathered rows, split partials).
struct LmWs {
  CompactWs cw;
  SurrogateWs sw;
  void* hidden_c;  // dense copy of the rows in the loss [max(n_rows, 128)][H] (backward
                   // only; null for the forward, whose LM head reads rows by index)
  float* part_m;
  float* part_s;
  float* tgt;
  unsigned* round_ctr;  // the LM head's pacing counter (items whose loads were issued)
};

void carve_surrogate_ws(Carver& cv, int64_t n_rows, int64_t n_seq, SurrogateWs* w);
AdvJob adv_job(const float* reward, const uint8_t* accepted, int64_t n_seq, int G, float eps,
               int unbiased, float* adv);
pace_status launch_group_adv(const AdvJob& j, const PaceBatch* b, unsigned* counter,
                             int32_t* status, cudaStream_t st);
void carve_lm_ws(Carver& cv, int64_t n_rows, int64_t n_seq, int H, bool dense_rows,
                 LmWs* w);
bool lm_needs_compaction(const PaceBatch* b);
pace_status check_lm_args(const PaceBatch* batch, const void* hidden, const void* w_vocab,
                          const int32_t* targets, int H, int V, float temperature,
                          const float* logprob);
pace_status run_logprob(const PaceBatch* batch, const void* hidden, const void* w_vocab,
                        const int32_t* targets, int H, int V, float temperature, float* logprob,
                        float* lse, const LmWs& ws, const AdvJob& adv, unsigned* counter,
                        int32_t* status_dev, cudaStream_t st);
void carve_compact_ws(Carver& cv, int64_t n_rows, CompactWs* w);
pace_status check_batch(const PaceBatch* b);
pace_status check_loss_args(const PaceBatch* b, const PaceLossArgs* l);
pace_status run_surrogate(const PaceBatch* b, const float* logprob, const PaceLossArgs* l,
                          const SurrogateWs& ws, bool adv_done, int32_t* status, cudaStream_t st);
// Counts the rows in the loss and lists them; clears counter0 and counter1 and lp /
// lse of the rows outside the loss (any may be null), and computes the advantages.
pace_status run_compaction(const PaceBatch* b, const CompactWs& ws, const AdvJob& adv,
                           unsigned* counter0, unsigned* counter1, float* lp, float* lse,
                           int32_t* status, cudaStream_t st);
RowCounts carve_row_counts(Carver& cv, int64_t n_rows);
pace_status launch_count_rows(const PaceBatch* b, RowCounts counts, unsigned long long* seq_in,
                              int* n_used, const AdvJob& adv, unsigned* counter0,
                              unsigned* counter1, int32_t* status, cudaStream_t st);
pace_status run_gather(const void* hidden, int H, int64_t n_rows, const CompactWs& ws,
                       void* out, cudaStream_t st);

}  // namespace pace
