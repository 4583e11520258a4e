// stride_internal.h -- launch interfaces between the C-ABI layer and the
// kernels.  Not installed; callers use include/stride.h.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "stride.h"

namespace stride {

// One published scan element of a lookback (32 bytes): running-sum terms, and
// the open turn's sums of log pi_T, d and logp_S * d.  (The running sum before
// the open turn is published in the flag's line: row_scan.cuh.)
struct alignas(32) ScanSlot {
  double c, st, sd, sl;
};

// The scan flag of row r (one CTA per row) or of 32-row tile r (persistent
// kernel) is flags[r * kFlagStride]: one flag per 128-byte line.  Each polls
// and reads its predecessors' flags; packed 32 to a line, a few lines took all
// of that traffic, and GB300 windows of 512-1,024 rows scored 3-12 % faster,
// with a flag per row, with the flags spread out.
constexpr int kFlagStride = 32;

constexpr uint64_t kWaitTimeoutNs = 2000000000ull;  // bound on any single device-side wait

struct BatchParams {
  const void* S;
  const void* T;
  const void* const* T_rows;  // per-window-row teacher row pointers (multi-teacher), or NULL
  int64_t ld;
  int32_t V;
  int32_t mode;
  const int32_t* tokens;
  const int64_t* traj_row_off;
  const int64_t* turn_row_off;
  const int32_t* traj_turn_off;
  int32_t n_traj;
  int32_t n_turns;
  int64_t row_begin;
  int64_t row_end;
  int64_t n_rows;
  const float* lambda;
  float lambda_all;
  stride_scan_state* state;
  stride_row_outputs out;
  stride_turn_stats* turn_stats;
  double* profile;  // [STRIDE_PROFILE_BINS * 3] or NULL, added to
  int32_t* dev_status;
  // workspace views
  uint32_t* ticket;
  uint32_t* flags;
  ScanSlot* agg;
  ScanSlot* incl;
  float* ws_logp_s;  // per window row, for the scan on log-probs and the persistent kernel's tiles
  float* ws_logp_t;
  uint64_t timeout_ns;
  uint32_t first_wave;  // CTAs of the split kernel that are resident from the start
  int32_t scan_inside;  // the persistent kernel completes its window's scan
  // A shard pass through the persistent kernel: per row (m, s) of S and T and
  // the token's logits, its column counted from col0; nothing else is written.
  float* partials;
  int64_t col0;
};

struct StepParams {
  const void* S;
  const void* T;
  int64_t ld;
  int32_t V;
  int32_t mode;
  const int32_t* tokens;
  const uint8_t* turn_end;
  const int32_t* rollout_idx;  // compacted rows: row b is rollout rollout_idx[b]; NULL = row b is rollout b
  int32_t B;                   // rows of this step
  int32_t n_state;             // rollouts in state / lambda (compacted form: bound of rollout_idx)
  const float* lambda;
  float lambda_all;
  stride_scan_state* state;
  stride_row_outputs out;
  uint8_t* stopped_now;
  stride_turn_stats* turn_out;
  int32_t* dev_status;
};

struct SelectParams {
  const float* turn_mean;
  const int32_t* n_turns;
  const uint8_t* correct;
  float alpha;
  int32_t N;
  int32_t T_max;
  int32_t* k_star;
  int32_t* k_max;
};

// Workspace layout of stride_score_batch (all offsets 256-byte aligned).
struct BatchWorkspaceLayout {
  size_t ticket_off, flags_off, agg_off, incl_off, logp_s_off, logp_t_off, clear_bytes, total;
};
BatchWorkspaceLayout batch_workspace_layout(int64_t n_rows);

// Teacher row address of window row `tile`: the aligned T buffer, or the
// multi-teacher row table.
template <typename LT>
__device__ __forceinline__ const LT* teacher_row(const BatchParams& p, int64_t tile) {
  return p.T_rows ? reinterpret_cast<const LT*>(p.T_rows[tile])
                  : reinterpret_cast<const LT*>(p.T) + tile * p.ld;
}

constexpr int kMaxTeacherDomains = 8;
struct TeacherTable {
  const void* base[kMaxTeacherDomains];
  int64_t rows[kMaxTeacherDomains];
  int32_t n_domains;
  int64_t ld_bytes;
};
cudaError_t launch_teacher_rows(const BatchParams& p, const TeacherTable& tt, const uint8_t* traj_domain,
                                const int64_t* traj_T_row0, const void** rows_out, cudaStream_t stream);

// Multiprocessor count of the current device, looked up once per device
// (thread-safe); 0 with the CUDA error in *err if it cannot be queried.
int current_device_sms(int* dev_out, cudaError_t* err);

// Launches kern as a programmatic dependent of the previous kernel on the
// stream: its CTAs may be scheduled before that kernel has ended, so kern
// waits (griddepcontrol.wait) before it touches what that kernel writes.  Every
// kernel of the library waits, in every thread, so a completed one's
// predecessors are complete too.  Ahead of its wait a kernel may give L2 hints,
// and, where its predecessor is known to release it only past its own wait,
// read what was there before that one (the scans after a scoring kernel: layout,
// carried state, lambda; the second pass: the log-probs too) and write what
// that one does not use (the first pass's workspace).
template <typename... K, typename... A>
cudaError_t launch_dependent(void (*kern)(K...), unsigned grid, unsigned block, cudaStream_t stream, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, static_cast<K>(args)...);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// Launchers return a cudaError_t from the launch.
// Clears what the chosen kernel needs at zero in the workspace (at most
// clear_bytes from its start) and launches the batch scoring kernels.
cudaError_t launch_score_batch(const BatchParams& p, int dtype, bool vec, size_t clear_bytes, cudaStream_t stream);
cudaError_t launch_score_batch_stream(const BatchParams& p, int dtype, bool aligned, cudaStream_t stream);
// Whether that kernel scans its window itself, and what it needs at zero from
// the workspace's start: the header (ticket), and one flag line per tile.
bool stream_scan_inside(int V);
size_t stream_clear_bytes(int64_t n_rows, int V);
// Zeroes `bytes` (a multiple of 16) at ws as a programmatic dependent of the
// previous kernel on the stream (it waits for that kernel first).
cudaError_t launch_clear_workspace(void* ws, size_t bytes, int sms, cudaStream_t stream);
cudaError_t launch_score_step(const StepParams& p, int dtype, bool vec, cudaStream_t stream);
// Diagnostic overrides of the automatic kernel choices (process-wide; 0 on
// success, -1 for a value out of range).
int set_step_shape_override(int threads, int C);  // 0 = automatic; 128 or 512 threads, 1..16 CTAs per row
int set_batch_kernel_override(const char* name);  // NULL / "" / "auto" = automatic
cudaError_t launch_select_restart(const SelectParams& p, cudaStream_t stream);
cudaError_t launch_state_init(stride_scan_state* state, int32_t n, cudaStream_t stream);
cudaError_t launch_partial_lse(const void* S, const void* T, int dtype, bool vec, int64_t ld,
                               int32_t V_shard, int64_t col0, const int32_t* tokens, int64_t rows,
                               float* partials, int32_t* dev_status, cudaStream_t stream);
cudaError_t launch_combine_partials(const float* parts, int32_t n_shards, int64_t rows, float* logp_s,
                                    float* logp_t, float* lse_s, float* lse_t, int32_t* dev_status,
                                    cudaStream_t stream);
// What the scan on log-probs follows: a scoring kernel of this library, which
// lets its dependents in only after its own wait; one that has checked the
// layout; one wave of the split kernel (whose window may run as one cluster).
struct ScanAfter {
  bool scoring, checked, small;
};
cudaError_t launch_scan_logprobs(const BatchParams& p, const float* logp_s, const float* logp_t,
                                 cudaStream_t stream, const ScanAfter& after);
cudaError_t launch_buffer_record(float* buf_mean, int32_t* buf_n_turns, int32_t n_tasks, int32_t T_max,
                                 const int32_t* task, const int32_t* k0, const stride_turn_stats* ts,
                                 const int32_t* traj_turn_off, int32_t n_traj, int32_t* dev_status,
                                 cudaStream_t stream);

}  // namespace stride
