// Host-visible declarations shared by the translation units of the library.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include "ps.h"
#include "ps_device.cuh"

// ---- the opaque handles of ps.h
#include <mutex>
#include <utility>
#include <vector>
struct HostWords {
  volatile u32 status[8];      // one word per ST_* bit, set by the kernel that meets the problem (report)
  ps_front_entry entry;        // ps_check_composition's answer,
  volatile u32 answered;       // and the number of the call that it answers
};
struct ps_ctx {
  int device;
  cudaStream_t stream;
  void* scratch;
  size_t scratch_bytes;
  u32* d_lengths;     // the compaction's counters (EvalArgs: n_nonempty, n_listed, blocks_done)
  HostWords* h;       // pinned host memory that kernels write to (nothing has to be copied back)
  std::mutex* check;  // one ps_check_composition at a time uses h->entry
  u32 checks;
  int sm_count;
};

struct ps_space {
  ps_ctx* ctx;
  ps_space_desc desc;             // pointers inside are not kept
  std::vector<u32> n_values;
  std::vector<Fact> facts;        // all N concatenated
  std::vector<u32> fact_begin;    // per N, offset into facts (n_n + 1 entries)
  std::vector<u32> modes;         // allowed modes ascending
  ps_model_shape* d_shapes;
  ModelRec* d_recs;
  Fact* d_facts;
  u32* d_order;                   // see SpaceDev::order
  std::vector<u32> order;
  std::vector<std::pair<u32, std::vector<std::pair<u32, u32>>>> degrees;   // see sweep_order
  SpaceDev dev;
};

// ---- sweep
#define SWEEP_MAX_WARPS 16        /* warps of a block at most */
#define PS_MAX_CAPS 8

struct SweepArgs {
  u64 caps[PS_MAX_CAPS];
  u64 cap_max;          // the largest of them
  u64 host_cap;
  u32 require_flags;    // without PS_F_FEASIBLE
  u32 comm_kind;
  u32 n_caps;
  u32 max_entries;      // entries of an output row; top-k: entries kept
  u32 skip_rejected;    // do not evaluate factorisations whose composition bits miss a required flag
  ps_front_entry* out;
  u32* counts;
  volatile u32* status;
};

cudaError_t launch_sweep(int kind, const SpaceDev& sp, const SweepArgs& a, int sm_count, cudaStream_t stream);

// ---- batch evaluation
/* Block shape of the window kernels: blocks of four warps, four of them resident (128 registers a
   thread; the write pass five, see EVAL_MIN_BLOCKS_WRITE).  Against two
   blocks of eight warps: materialise -5 % (625 codes a group) to -13 % (256 codes); short blocks
   spread the warps' set-up and store phases better. */
#ifndef EVAL_THREADS
#define EVAL_THREADS 128
#endif
#ifndef EVAL_MIN_BLOCKS
#define EVAL_MIN_BLOCKS 4
#endif
#define EVAL_RUN_UNITS 32

struct EvalArgs {
  u64 first, count;         // the window
  u64 first_group;          // global group index of the tile 0's first group
  u32 n_tiles;
  // filter (compaction modes)
  u64 cap_bytes, host_cap;
  u32 require_flags;        // without PS_F_FEASIBLE
  ps_out_soa out;
  u64* idx_out;
  u64* n_out;
  // compaction scratch.  The window's factorisations ("units", counted through all models)
  // are taken in runs of EVAL_RUN_UNITS, a block of the count pass each.
  u64 first_unit;
  u32 n_units, n_runs;
  u32* group_offset;        // [n_tiles] survivors of the earlier groups of the group's run
  u32* nonempty;            // [n_units] the units that have survivors, counted from first_unit, in any order
  // Counters of the count pass: places given out in the list and blocks that have finished.  Both
  // are zero between calls: the last block leaves the list's length in n_listed and clears them.  So
  // no call needs a memset of its own, and a captured call can be replayed.
  u32* n_nonempty;
  u32* blocks_done;
  u32* n_listed;
  u64* run_offset;          // [n_runs] survivors of each run, then of all runs before it
};

void eval_plan_runs(const SpaceDev& sp, EvalArgs& a);   // fills first_unit, n_units, n_runs
cudaError_t launch_eval_materialise(const SpaceDev& sp, const EvalArgs& a, cudaStream_t stream);
cudaError_t launch_eval_count(const SpaceDev& sp, const EvalArgs& a, cudaStream_t stream);
cudaError_t launch_eval_write(const SpaceDev& sp, const EvalArgs& a, cudaStream_t stream);

// ---- small kernels
cudaError_t launch_model_derive(const ps_model_shape* d_shapes, ModelRec* d_recs, u32 n,
                                volatile u32* status, cudaStream_t stream);
cudaError_t launch_check_point(const ps_model_shape& shape, Fact f, u32 v, u32 tau, u32 code_dp,
                               u32 tp_max_valid, u32 tp_coll, u32 axis_form, u32 comm_kind,
                               u64 cap_bytes, HostWords* h, u32 call, cudaStream_t stream);
cudaError_t launch_select(const ps_select_query* d_q, u64 n, u32 head_num, u32 head_den, u32 layer_num,
                          u32 layer_den, u32 tp_degree, ps_select_result* d_out, cudaStream_t stream);
cudaError_t launch_int_peak(u32 blocks, u32 iters, u32* d_sink, cudaStream_t stream);

// ---- brute-force verifier
cudaError_t launch_verify(const ps_verify_shape& s, const ps_verify_case* d_cases, u64 n, const double* d_data,
                          u64 data_len, double* d_theta_out, ps_verify_result* d_out, volatile u32* status,
                          cudaStream_t stream);

cudaError_t launch_select_compare(const SpaceDev& sp, u32 unit_begin, u32 unit_end, u32 N, u64 device_bytes, u32 fast,
                                  u32 head_num, u32 head_den, u32 layer_num, u32 layer_den, u32 tp_degree,
                                  u64 host_cap, u32 require_flags, u32 comm_kind, const ps_front_entry* d_frontier,
                                  const u32* d_counts, u32 n_caps, u32 cap_index, u32 max_entries,
                                  ps_select_compare_result* d_out, cudaStream_t stream);
