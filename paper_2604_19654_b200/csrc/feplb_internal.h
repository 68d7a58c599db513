// Internal declarations shared by the translation units of libfeplb (not part of the ABI).
#ifndef FEPLB_INTERNAL_H_
#define FEPLB_INTERNAL_H_

#include <cstddef>
#include <cstdint>

#include "feplb.h"

#define FEPLB_MAX_EXPERTS 1024
#define FEPLB_MAX_GROUPS 1024
#define FEPLB_SLOTS_PER_BLOCK 1024   // slots ranked by one CTA of the permutation kernels
#define FEPLB_FRONT_SMALL_SLOTS 8192 // most slots of a batch whose routing and gather run as one launch
#define FEPLB_MAX_RANGES 4           // token ranges a host-buffer forward is cut into at most
#define FEPLB_TILE_M 128             // rows of one GEMM tile
#ifndef FEPLB_NOALLOC_MAX_HIST_INTS
#error "feplb.h must define FEPLB_NOALLOC_MAX_HIST_INTS"
#endif

// bits of the device status word
#define FEPLB_ST_RANGE 1u      // expert id outside [0, E)
#define FEPLB_ST_COUNTS 2u     // counts passed to dispatch disagree with the ids
#define FEPLB_ST_WAIT 4u       // a bounded mbarrier wait gave up inside the GEMM
#define FEPLB_ST_GROUP 8u      // a group entry was malformed (expert or rows out of range)
#define FEPLB_ST_PLAN 16u      // the GEMM's bounded wait for the planner's dynamic group table gave up
#define FEPLB_MERGED_MAX_ROWS_PER_EXPERT 768   // static and dynamic groups share launches below this many rows per expert ...
#define FEPLB_MERGED_ANY_ROWS_WEIGHT (6 << 20)  // ... and at any number where a weight matrix has fewer elements than this
#define FEPLB_WM_MAX_ROWS_PER_EXPERT 1280       // the weights-on-M form ends here in launches over static and dynamic groups together
#define FEPLB_SHORT_TILE_WEIGHT (1 << 19)       // below this many elements tiles are short, single-CTA tiles better ...
#define FEPLB_SHORT_TILE_MIN_ROWS 288           // ... from this many rows per expert
#define FEPLB_PAIR_DEEP_WEIGHT (2 << 20)        // two-CTA tiles with deep stages: matrices of at least so many elements,
#define FEPLB_PAIR_DEEP_EXPERTS 25              // or so many experts, or two waves of tiles
#define FEPLB_PAIR_MIN_ROWS_PER_EXPERT 256     // launches over static and dynamic groups, or all: two-CTA tiles from here
#define FEPLB_FEW_LARGE_WEIGHT (1 << 20)       // weight matrices of at least so many elements: the form for few rows per expert up to WM_MIN_ROWS
#define FEPLB_FEW_GUARD_WEIGHT (3 << 17)        // its guard against a nearly empty wave of long units, from so many elements
#define FEPLB_WM_MIN_ROWS_PER_EXPERT 64        // the weights-on-M form from here to WM_MAX_ROWS (in launches of one table to MERGED_MAX_ROWS)
#define FEPLB_WM_MIN_WEIGHT (1 << 19)          // ... for weight matrices of at least so many elements and with enough units;
#define FEPLB_WM_ANY_UNITS_WEIGHT (3 << 20)     // ... from this many elements whatever their number
// No launch of a forward waits for the plan below this many rows per expert, or where the expert FFN takes less than this long
#define FEPLB_DIRECT_ROWS_PER_EXPERT 128
#define FEPLB_DIRECT_SMALL_FRONT_ROWS 192      // ... or, in the merged order behind the one-launch front, from this many
#define FEPLB_DIRECT_FFN_US 150
#define FEPLB_WM_MAX_ENTRIES 1024    // group entries (static + dynamic table) one weights-on-M launch can hold

int feplb_validate_config(const feplb_config* c);

#ifdef __CUDACC__
#include <cuda_runtime.h>

// Kernel launchers (each enqueues on `st` and returns the cudaError_t of the launch).
// n_launch is incremented by the number of kernels enqueued.
// totals: E + 1 ints of scratch, zero between calls.
cudaError_t feplb_launch_route_hist(const int32_t* ids, int64_t S, int E, int R, int32_t* totals, int32_t* counts,
                                    int32_t* rank_load, uint32_t* status, cudaStream_t st, int64_t* n_launch);
cudaError_t feplb_launch_permute(const int32_t* ids, int64_t S, int K, int E, int A, const int32_t* counts,
                                 int32_t* block_hist, int32_t* pad_off, int32_t* slot_to_row,
                                 int32_t* row_to_token, int64_t s_cap, uint32_t* status,
                                 cudaStream_t st, int64_t* n_launch);
// A launch per pass walks a.groups (filtered by a.which) and then, if dyn.seq != 0, the planner's dynamic
// table, which it picks up on the device once the host-side ready word carries (seq << 32) | number of
// groups; the CTA that wins `claim` copies it to table_dev (feplb_dyn.cuh).
struct feplb_wm_dyn {
  // the table travels as 32-byte entries {expert, row_start, rows, exec_rank, is_dynamic, seq, 0, 0}
  void* table_dev = nullptr;                         // device copy of the table, written by the claiming CTA
  const void* table_host = nullptr;                  // device address of the planner's table in mapped host memory
  unsigned long long* ready_dev = nullptr;           // set by the claiming CTA after table_dev
  const unsigned long long* ready_host = nullptr;    // device address of the word the planner thread sets after table_host
  uint32_t* claim = nullptr;                         // device word the CTAs race for
  unsigned long long* early = nullptr;               // device word: seq of the forward whose table the gather brought over
  uint32_t* gather_done = nullptr;                   // device word: seq of the forward whose gather has a CTA without work left
  uint32_t seq = 0;                                  // 0: no dynamic table
  int max_groups = 0;                                // capacity of the tables
  unsigned long long* stamps = nullptr;              // optional: globaltimer marks, [0..7] of the two launches, [9] early delivery
  unsigned long long wait_limit_ns = 0;              // bound of the wait for the table (0: the library's default)
};
// Must follow feplb_launch_permute or feplb_launch_route_fused on the same stream: turns the ranks those
// left in slot_to_row into rows (block_base = the scanned per-CTA histograms), fills row_to_token and
// copies the rows of x.
cudaError_t feplb_launch_gather(const void* x, const int32_t* ids, const int32_t* block_base, int32_t* slot_to_row,
                                const int32_t* counts, const int32_t* pad_off, void* x_perm, int T, int K, int E, int d,
                                int A, int64_t s_cap, int num_sms, cudaStream_t st, int64_t* n_launch,
                                int32_t* row_to_token, bool programmatic, int t0 = 0,          // tokens [t0, t0 + T)
                                const feplb_wm_dyn* dyn = nullptr, uint32_t* status = nullptr);   // pick the planner's table up along the way
// Whole-layer path: histogram (+ ranks inside each CTA's slots) + one scan kernel that emits counts, rank
// loads, offsets, the home group table and the -1 tail of row_to_token.
cudaError_t feplb_launch_route_fused(const int32_t* ids, int64_t S, int E, int R, int A, int dyn,
                                     const uint8_t* mask_in, int32_t* block_hist, int32_t* counts,
                                     int32_t* rank_load, int32_t* pad_off, feplb_group* groups, uint8_t* mask_out,
                                     int32_t* slot_to_row, int32_t* row_to_token, int64_t s_cap, uint32_t* status,
                                     unsigned long long* counts_host_tagged, int32_t seq, unsigned long long* t_counts,
                                     cudaStream_t st, int64_t* n_launch);
// A batch processed in n_ranges token ranges (first_token[r] * K a multiple of FEPLB_SLOTS_PER_BLOCK): the group table of
// range r goes to out + r * E.  block_base and home as feplb_launch_route_fused leaves them.
cudaError_t feplb_launch_range_groups(const int32_t* block_base, int64_t S, int K, int E, const feplb_group* home,
                                      const int* first_token, int n_ranges, feplb_group* out, cudaStream_t st, int64_t* n_launch);
// Small batches: feplb_launch_route_fused and feplb_launch_gather in one launch; with groups == nullptr (and no mask,
// counts, rank_load, pad_off) feplb_launch_permute and feplb_launch_gather, counts_in being the caller's counts.
bool feplb_front_is_small(int64_t S, int E);
cudaError_t feplb_launch_front_small(const void* x, const int32_t* ids, int T, int K, int E, int R, int d, int A, int dyn,
                                     const uint8_t* mask_in, const int32_t* counts_in, int32_t* counts, int32_t* rank_load,
                                     int32_t* pad_off, feplb_group* groups, int32_t* slot_to_row, int32_t* row_to_token, void* x_perm,
                                     int64_t s_cap, uint32_t* status, unsigned long long* counts_host_tagged, int32_t seq,
                                     unsigned long long* t_counts, int num_sms, cudaStream_t st, int64_t* n_launch);
cudaError_t feplb_launch_upload_groups(const feplb_group* src_host_mapped, feplb_group* dst, int n, cudaStream_t st);
cudaError_t feplb_launch_home_groups(const int32_t* counts, const uint8_t* mask_in, int E, int R, int A, int dyn,
                                     feplb_group* groups, uint8_t* mask_out, cudaStream_t st, int64_t* n_launch);
cudaError_t feplb_launch_combine(const void* y_perm, const int32_t* slot_to_row, const float* gates, void* out,
                                 int T, int K, int d, int num_sms, cudaStream_t st, int64_t* n_launch);

cudaError_t feplb_launch_route_topk(const float* logits, int T, int E, int K, int32_t* ids, float* gates,
                                    int num_sms, cudaStream_t st, int64_t* n_launch);

struct feplb_gemm_args {
  const void* x_perm; const void* w1; const void* w3; const void* w2;
  void* h; void* y;
  const feplb_group* groups; int n_groups; int which;
  int E, d, f; int64_t s_cap;
  uint32_t* status;
  int num_sms;
  int deep;   // pair: stages of 128 elements of K, 128-row last tiles
  int pair;   // 1: clusters of two CTAs on 256-row tiles (cta_group::2); 0: one CTA per 128-row tile
  // receive buffer of migrated experts' weights ([n_recv_slots, f, d] x2 and [n_recv_slots, d, f]); may be null
  const void* recv_w1; const void* recv_w3; const void* recv_w2; int n_recv_slots;
  const void* recv_x = nullptr;   // optional [s_cap, d]: rows of pieces that run from a receive slot are read here (pass 1)
  void* ab_out;   // optional [s_cap, 2f]: pass 1 also saves the pre-activations a | b (for the backward pass)
};
// Returns FEPLB_OK or a feplb_status; text of a failure goes to err (size errn).
// One thread waits (bounded by limit_ns) on an mbarrier nobody completes; *gave_up = 1 and FEPLB_ST_WAIT expected.
cudaError_t feplb_launch_wait_selftest(uint32_t* status, unsigned long long limit_ns, int* gave_up, cudaStream_t st);
// Tokens-on-M forms (feplb_gemm.cu): single CTA per 128-row tile or, with a.pair, clusters of two on 256-row tiles.
int feplb_launch_expert_ffn(const feplb_gemm_args& a, cudaStream_t st, int64_t* n_launch, char* err, size_t errn,
                            const feplb_wm_dyn* dyn = nullptr);
// Weights-on-M form (feplb_gemm_wm.cu).  FEPLB_E_STATE, with nothing launched, where no tensor map covers W1 and W3 together.
bool feplb_wm_supported(int E, int n_entries_max);
int feplb_launch_expert_ffn_wm(const feplb_gemm_args& a, const feplb_wm_dyn& dyn, cudaStream_t st, int64_t* n_launch,
                               char* err, size_t errn);
// The same for few rows per expert (feplb_gemm_few.cu): one table, no receive slots.  stamps: as feplb_wm_dyn::stamps.
// nmax: most token rows per unit, 32, 64 or 128.  FEPLB_E_STATE, with nothing launched, where no tensor map covers W1 and W3 together.
int feplb_launch_expert_ffn_few(const feplb_gemm_args& a, cudaStream_t st, int64_t* n_launch, char* err, size_t errn,
                                int nmax, unsigned long long* stamps);
// ---- backward pass ---------------------------------------------------------------------------
struct feplb_bwd_args {
  const void* x_perm; const void* ab_saved; void* h; void* d_y_perm;   // padding rows of h, d_y_perm, d_ab get zeros
  const void* w1t; const void* w3t; const void* w2t;        // [E,d,f], [E,d,f], [E,f,d]
  const feplb_group* groups; int n_groups; int which;
  const feplb_group* expert_table;                          // E entries {e, first row, rows}: the K ranges of the weight gradients
  void* d_ab; void* d_x_perm;                               // [s_cap, 2f], [s_cap, d]
  float* dw1; float* dw3; float* dw2; int accumulate;       // fp32 [E,f,d], [E,f,d], [E,d,f]; dw1 == nullptr: skip
  int E, d, f; int64_t s_cap;
  uint32_t* status; int num_sms;
  bool pads_zeroed = false;                                 // the padding rows hold zeros already
  int pair_dgrad, pair_wgrad;                               // 1: cta_group::2 form (256 x 256 tiles per cluster of two CTAs)
};
cudaError_t feplb_launch_transpose_weights(const void* w1, const void* w3, const void* w2, void* w1t, void* w3t, void* w2t,
                                           int E, int d, int f, cudaStream_t st, int64_t* n_launch);
// The padding rows of h, d_y_perm and d_ab that the combine's backward kernel zeroes along the way.
struct feplb_bwd_pads { const feplb_group* table; int E, f; void* h; void* d_ab; };
cudaError_t feplb_launch_combine_bwd(const void* d_out, const void* y_perm, const int32_t* slot_to_row, const float* gates,
                                     void* d_y_perm, float* d_gates, int T, int K, int d, cudaStream_t st, int64_t* n_launch,
                                     const feplb_bwd_pads* pads = nullptr);
int feplb_launch_expert_ffn_bwd(const feplb_bwd_args& a, cudaStream_t st, int64_t* n_launch, char* err, size_t errn);
#endif

#endif  // FEPLB_INTERNAL_H_
