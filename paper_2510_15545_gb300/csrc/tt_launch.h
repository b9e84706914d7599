// tt_launch.h -- kernel argument blocks and launchers (internal to libtt).
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "tt.h"

namespace tt {

struct Partial;

constexpr int kAlignWarpsMax = 8;             // warps (pairs at a time) per align CTA
constexpr int kAlignWarpsStep = 4;            // the same inside tt_step, beside the row pass
constexpr int kAlignSmemMax = 200 * 1024;     // dynamic shared memory cap of one align CTA
constexpr int kMaxChunksPerRow = 1024;        // rows up to 1024 * 2048 = 2,097,152 columns

struct AlignArgs {
  int B, n_draft, n_target, max_k, max_m, window;
  const int32_t* draft_off;
  const int32_t* draft_ids;
  const int32_t* target_off;
  const int32_t* target_ids;
  tt_vocab vd, vt;
  int32_t* path;
  int32_t* path_len;
  int32_t* cost;
  int32_t* map;
  int32_t* status;
  uint8_t* need;               // needed draft rows (may be NULL)
  unsigned long long* work;    // row-pass work counters to zero (may be NULL)
  const int32_t* target_cols;  // scored column of each target position
  int32_t* excl;               // [n_target + B] written: scored column of each target row
                               // (-1 for the bonus row), may be NULL
  int after_grid;      // 1: launched while the grid before it (the penalty's sets) may run;
                       // the row pass, which reads those, starts after both
  int tile_blocks;     // 16-byte blocks of a pair's cost tile
  size_t smem_per_pair;
  int pairs_per_block; // (set by launch_align)
};

constexpr int kNucNarrowRows = 1;  // RowSet::nucleus
constexpr int kNucWideRows = 2;
// How a nucleus family's rows of V columns (unit_cols to an 8 KB unit) are
// settled: rows of more than kNucRowUnits units, and at most kNucWideMax
// columns, by the nucleus row kernel. It hands each unit to another of its
// warps, so in rows of few units most warps and most of its room for candidates
// stay unused. Against the row pass and the kernels after it, on Zipf logits
// (both families of one width):
//                        64 requests, top-p 0.95   512 requests, top-p 0.9
//   bf16 10,000 (2.4 units)     94 us to 79             411 us to 392
//   bf16 16,323 (4.0)           88 us to 87             394 us to 459
//   bf16 20,419 (5.0)           84 us to 94             387 us to 509
//   fp32  9,155 (4.5)           80 us to 87             371 us to 456
//   fp32 16,323 (8.0)           80 us to 98             367 us to 527
constexpr int kNucRowUnits = 4;
constexpr int kNucWideMax = 480 * 2048;
inline int nucleus_rows(bool nucleus, int V, int unit_cols) {
  if (!nucleus) return 0;
  return V > kNucRowUnits * unit_cols && V <= kNucWideMax ? kNucWideRows : kNucNarrowRows;
}

// One family of logits rows seen by the row pass.
struct RowSet {
  const char* data;
  int64_t stride_bytes;
  int V;
  int nch;
  float scale;  // log2(e) / T
  int64_t n_rows;
  Partial* part;
  const uint8_t* need;  // rows to visit (NULL = all)
  int top_k;            // > 0: filtered rows, the row pass writes top-k lists to cand
  Cand* cand;           // [n_rows * nlist * cand_stride(top_k)]: one list per row unit
  int nlist;            // units (8 KB stages: 2048 fp32 or 4096 bf16 columns) per row
  int nucleus;          // top-p without top-k (top_k = 0). kNucNarrowRows: the row pass
                        // writes the compensated partials of all its columns and the
                        // nucleus kernels find each row's kept set; kNucWideRows: the
                        // nucleus row kernel streams the rows and finds it at once
  // Repetition penalty (top-k families only; pen = NULL: none): the row pass
  // gives each request's penalized columns the row's own (penalized or raw)
  // value in fp32 units; bf16 units leave them out of their lists and the
  // kept-set kernel adds them back.
  const PenEntry* pen;    // penalized columns of request b at pbase[b] (pcnt[b]), by unit
  const int32_t* pbase;
  const int32_t* pcnt;
  const int32_t* pstart;  // [B * (nch + 1)]: first entry of each row unit, then pcnt
  float penalty;          // theta
  int unit_cols;          // columns per row unit (2048 fp32, 4096 bf16)
};

struct RowPassArgs {
  RowSet d, t;
  int64_t rows_d, rows_t;    // rows of each family to stream (0 = family absent)
  int B, n_target, n_draft;
  const int32_t* target_off;
  const int32_t* target_cols;
  const int32_t* draft_off;  // to find a penalized draft row's request
  int32_t* err;              // err[0] = epoch of a failed call, err[1] = its TT_REQ_* bits
  int32_t epoch;             // identifies this call
  const int32_t* excl_late;  // [target rows] column left out of the sum, written by the grid
                             // this one depends on: read only after the grid-dependency
                             // wait, before it (and when NULL) found from target_off /
                             // target_cols
  // Work counter for the items past each CTA's fixed share, zeroed by the grid
  // this one depends on and read only after the grid-dependency wait; NULL:
  // every item belongs to a fixed share.
  unsigned long long* work;
  int32_t keep;              // 1: the decision reads whole rows again, so the streamed ones
                             // are not marked to leave L2 first
  int32_t pre_eighths;       // with work: eighths of the target items streamed in fixed
                             // blocks before the grid-dependency wait (1..7)
  int32_t stall_stage;       // test hook (-1 = off): in CTA 0 the stage consumed at
                             // consumer step stall_stage is never freed, so the
                             // bounded waits run out
  uint64_t wait_ns;          // limit of every pipeline wait (set by launch_rowpass: 2 s)
};

// The row pass over several column shards of the target rows at once.
struct ShardRows {
  const char* data;
  int64_t stride_bytes, n_rows;
  Partial* part;
  const int32_t* excl;  // [target rows] the shard's own scored column or -1: read only
                        // after the grid-dependency wait
  int64_t end;          // row units of the shards up to this one
  int V, col0, nch;
};
struct ShardPassArgs : RowPassArgs {  // (t: V of the whole row, scale; rows_t)
  int S;
  ShardRows sh[TT_MAX_SHARDS];
};

struct DecideArgs {
  int B, n_draft, n_target, max_k, max_m, full_q, mode_transfer_only;
  const int32_t* draft_off;
  const int32_t* draft_cols;
  const int32_t* target_off;
  const int32_t* target_cols;
  const int32_t* map;
  const float* q_hat_in;     // given q_hat (verify) or NULL (computed here)
  const float* draft_probs;  // given draft probabilities or NULL
  RowSet d, t;
  int dt_d, dt_t;
  const int32_t* status_in;  // status of an earlier stage (align) or NULL
  int32_t* err;              // row-pass error words (NULL when no row pass ran)
  int32_t epoch;
  uint64_t seed, request_base;
  int32_t* accepted;
  int32_t* next_token;
  int32_t* status;
  float* q_hat_out;
  float* p_hat;
  float* lse;
  int warm_ctas;  // CTAs b < warm_ctas run a warming pass before the wait (see decide.cu)
  int sm_count;   // SMs of the device (sizes the decision kernel's CTAs)
  float top_p_d, top_p_t;    // top-p of filtered families (d.top_k / t.top_k > 0)
  const int32_t* status_q;   // status of the kernel that produced q_hat_in, or NULL
  const Cand* kept_d;        // kept sets of filtered families (written by the kept kernel)
  const Cand* kept_t;
  const KeptHead* head_d;
  const KeptHead* head_t;
  const float* um_d;         // per-chunk kept masses of nucleus families
  const float* um_t;
  const int32_t* status_p;   // problems of the repetition-penalty histories, or NULL
};

// The kept-set stage of filtered families: one warp per row merges the row's
// unit lists into its top-k and applies temperature and top-p.
struct KeptArgs {
  RowSet d, t;             // families with top_k > 0 (kept_kernel) or nucleus (nucleus_kernel)
                           // are done, the others skipped
  int64_t rows_d, rows_t;  // rows of each family (draft rows with d.need[row] == 0 skipped)
  float top_p_d, top_p_t;
  Cand* kept_d;
  Cand* kept_t;
  KeptHead* head_d;
  KeptHead* head_t;
  float* um_d;             // nucleus families: kept probability mass per chunk
  float* um_t;
  int dt_d, dt_t;          // logits types (nucleus rows are read again)
  int B, n_target;         // the batch, to find a nucleus target row's scored column
  const int32_t* target_off;
  const int32_t* target_cols;
  const int32_t* draft_off;  // and a penalized draft row's request
  int n_draft;
};

// The nucleus row kernel (nucrow.cu): the rows of families with nucleus =
// kNucWideRows, each streamed once and its kept set found.
struct NucRowArgs {
  RowSet d, t;
  int64_t rows_d, rows_t;  // rows of each such family (0: none)
  float top_p_d, top_p_t;
  KeptHead* head_d;
  KeptHead* head_t;
  float* um_d;
  float* um_t;
  int32_t* err;
  int32_t epoch;
  unsigned long long* work;  // row counter, zeroed by a grid this one depends on, or NULL:
                             // every row belongs to a fixed share
  int32_t stall_stage;       // as in RowPassArgs
  uint64_t wait_ns;
};

// The repetition penalty's per-request sets (pen.cu): for each penalized
// family, every request's history and sequence columns, one entry each (with
// its first sequence position), by row unit, and the start of each unit.
struct PenArgs {
  int B;
  int on_d, on_t;
  int V_d, V_t, nch_d, nch_t, unit_d, unit_t, nlist_d, nlist_t;
  int n_draft, n_target, n_hist_d, n_hist_t;
  const int32_t* hist_off_d;
  const int32_t* hist_cols_d;
  const int32_t* hist_off_t;
  const int32_t* hist_cols_t;
  const int32_t* draft_off;
  const int32_t* draft_cols;
  const int32_t* target_off;
  const int32_t* target_cols;
  PenEntry* pen_d;
  int32_t* pbase_d;
  int32_t* pcnt_d;
  int32_t* pstart_d;
  PenEntry* pen_t;
  int32_t* pbase_t;
  int32_t* pcnt_t;
  int32_t* pstart_t;
  int32_t* pstatus;
  int32_t* fell;  // two words of scratch: whether a family's offsets fall anywhere
};

struct PrepArgs {
  int B, n_draft, n_target;
  const int32_t* draft_off;
  const int32_t* target_off;
  const int32_t* map;
  uint8_t* need;   // needed-draft-row flags, written from map
  unsigned long long* work;  // row-pass work counter to zero (may be NULL)
};

size_t align_smem_per_pair(int max_k, int max_m, int tile_blocks);
int align_window(int window);
int align_tile_blocks(int max_k, int max_m, int window);
cudaError_t launch_align(const AlignArgs& args, cudaStream_t stream);
// All shards of one type in one grid; `end` is filled in here.
cudaError_t launch_shard_rowpass(const ShardPassArgs& args, int dt, cudaStream_t stream,
                                 int sm_count, bool pdl);
cudaError_t launch_rowpass(const RowPassArgs& args, int dt_d, int dt_t, cudaStream_t stream,
                           int sm_count, bool pdl);
cudaError_t launch_decide(const DecideArgs& args, cudaStream_t stream, bool pdl);
cudaError_t launch_prep(const PrepArgs& args, cudaStream_t stream);

// Filtered families (filter.cu): the kept sets of the filtered rows from their
// top-k lists, then q_hat of every target position from the kept sets of the
// mapped draft rows, and the decision over filtered target rows
// (args.t.top_k > 0) with q_hat_in given.
cudaError_t launch_kept(const KeptArgs& args, cudaStream_t stream, int sm_count, bool pdl);
// Nucleus families (top-p without top-k, App. F): the exact kept set of every
// nucleus row from its logits and the row pass's partials, and the decision
// over nucleus target rows.
cudaError_t launch_nucleus(const KeptArgs& args, cudaStream_t stream, int sm_count, bool pdl);
cudaError_t launch_nucleus_rows(const NucRowArgs& args, int dt_d, int dt_t, cudaStream_t stream,
                                int sm_count, bool pdl);
cudaError_t launch_decide_nucleus(const DecideArgs& args, cudaStream_t stream, bool pdl);
cudaError_t launch_pen_prep(const PenArgs& args, cudaStream_t stream);
cudaError_t launch_filter_q(const DecideArgs& args, cudaStream_t stream, bool pdl);
cudaError_t launch_decide_filtered(const DecideArgs& args, cudaStream_t stream, bool pdl);

// Loads every kernel of the library on the current device and sets its launch
// attributes, so that no module is loaded lazily inside a dependent-launch chain.
cudaError_t preload_align();
cudaError_t preload_rowpass();
cudaError_t preload_decide();
cudaError_t preload_filter();
cudaError_t preload_nucleus();
cudaError_t preload_nucleus_rows();

// Test hook of the bounded waits (rowpass.cu): the stage to hold and the wait
// limit of the next streaming launch; false (and the defaults) when off.
bool next_launch_stall(int32_t* stall_stage, uint64_t* wait_ns);
cudaError_t preload_pen();

// Records a failed CUDA call for tt_last_cuda_error() and returns TT_ERR_CUDA.
tt_status record_cuda_error(cudaError_t e);

// Every argument check of tt_step, on the host only (nothing is queued on a
// stream): TT_OK and the workspace bytes the step needs (0 for an empty batch),
// or the status tt_step would return for these arguments.
tt_status step_check(const tt_batch* batch, const tt_vocab* vd, const tt_vocab* vt,
                     const tt_logits* draft, const float* draft_probs, const tt_logits* target,
                     const tt_params* prm, const tt_step_out* out, size_t* need);

}  // namespace tt
