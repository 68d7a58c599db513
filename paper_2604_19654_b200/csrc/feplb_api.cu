// C ABI of libfeplb: context, argument checks, the planner thread (paper Section 2.3: the CPU
// load balancer runs on a dedicated thread, triggered by router completion, while the GPU
// computes the static experts) and the per-micro-batch orchestration.
#include <cuda_runtime.h>

#include <atomic>
#include <algorithm>
#include <chrono>
#include <climits>
#include <cmath>
#include <condition_variable>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <numeric>
#include <thread>
#include <vector>

#include "feplb.h"
#include "feplb_internal.h"

namespace {
using clk = std::chrono::steady_clock;
inline double us_since(clk::time_point t0) {
  return std::chrono::duration<double, std::micro>(clk::now() - t0).count();
}
enum JobState { JOB_IDLE = 0, JOB_PENDING = 1, JOB_RUNNING = 2, JOB_DONE = 3 };
enum { EV_T0 = 0, EV_HIST, EV_DISPATCH, EV_STATIC0, EV_STATIC1, EV_DYN0, EV_DYN1, EV_COMBINE, EV_COUNTS, EV_COPIES, EV_STAMPS, EV_N };
constexpr int kEvRing = 16;   // forwards whose stage events may be outstanding
constexpr int kStampWords = 16;   // [0..3] pass 1, [4..7] pass 2 (see WmParams::stamps), [8] counts left the device, [9] table
                                  // brought over by the gather
}  // namespace

struct feplb_ctx {
  feplb_config cfg;
  int device = 0, num_sms = 0;
  size_t s_cap = 0;
  int nb = 0;   // CTAs of the permutation kernels
  char err[512] = {0};
  int64_t launches = 0;
  int32_t path = 0;            // FEPLB_PATH_* of the last forward
  int32_t detail = 0;          // FEPLB_DETAIL_* of the last forward
  int gemm_pair_default = 0;   // GEMM form for launches whose group sizes the host does not know
  int gemm_pair_forced = -1;   // feplb_set_gemm_form: 0/1 forces one form everywhere, -1 = chosen per table
  int bwd_pair = 0;            // backward GEMMs in the pair form: bit 0 activation gradients, bit 1 weight gradients
  int gemm_pair_auto = 0, bwd_pair_auto = 0;   // the choices feplb_create derived from the geometry
  bool wm_ok = false;          // the weights-on-M form may be asked for: widths of whole units
  int few = 0, few_auto = 0;   // > 0: single group tables go through the form for few rows per expert, in units of that many
  bool wm = false;             // ... and is the form in use (feplb_create's choice or feplb_set_gemm_form)
  bool wm_auto = false;
  bool wm_merged = false, wm_merged_auto = false;   // the same for launches over static and dynamic groups together
  bool wm_static = false, wm_static_auto = false;   // the static launches of the four-launch order use it
  bool pair_deep = false;      // the two-CTA form runs with stages of 128 elements and 128-row last tiles
  bool merged_ok = false;      // both group tables of a forward fit one launch (static, then dynamic groups)
  bool merged = false;         // ... and feplb_moe_forward runs that way: two GEMM launches instead of four
  bool merged_auto = false;
  bool direct = false;         // no launch of a forward depends on the plan: both passes walk the home table (small batches)
  bool direct_auto = false;
  bool merged_pair = false;    // form of the merged launches when none is forced
  int32_t planner_delay_us = 0;        // test aid: the planner sleeps before it publishes its table
  int32_t device_wait_limit_us = 0;    // bound of the GEMM's wait for the table (0: default)
  // weights-on-M form: the words through which a running GEMM launch learns that the dynamic table exists
  int32_t* h_dyn_tab32 = nullptr;                    // pinned + mapped: the dynamic table as 32-byte entries tagged with the sequence number
  int32_t* h_dyn_tab32_dev = nullptr;                // its device address
  int32_t* d_dyn_tab32 = nullptr;                    // device copy, made by the GEMM's claiming CTA
  unsigned long long* d_dyn_ready = nullptr;         // device words: [0] ready, [1] claim, [2] early, [3] gather done
  unsigned long long* h_dyn_ready = nullptr;         // pinned + mapped word, set by the planner thread
  unsigned long long* h_dyn_ready_dev = nullptr;     // its device address
  unsigned long long* d_stamps = nullptr;            // [kEvRing][kStampWords] globaltimer marks of the kernels
  unsigned long long* h_stamps = nullptr;            // pinned copy, filled at the end of a timed forward
  bool job_wm = false;

  // device scratch
  int32_t* d_block_hist = nullptr;
  int32_t* d_pad_off = nullptr;
  int32_t* d_totals = nullptr;       // [E + 1] accumulators and ticket of feplb_route_hist, zero between calls
  uint32_t* d_status = nullptr;
  feplb_group* d_home_groups = nullptr;
  feplb_group* d_dyn_groups = nullptr;
  feplb_group* d_range_groups = nullptr;        // [FEPLB_MAX_RANGES, E] (host-buffer forward)
  uint8_t* d_mask = nullptr;
  // Phase-2 receive buffer: R*max_num_dyn slots of one expert's weights each (phase2_copy)
  void* d_recv_w1 = nullptr;
  void* d_recv_w3 = nullptr;
  void* d_recv_w2 = nullptr;
  int n_recv_slots = 0;
  void* d_recv_x = nullptr;    // Phase-2 receive region of the migrated pieces' rows: [s_cap, d], same row numbers as x_perm
  cudaEvent_t ev_gather = nullptr;          // the permuted rows of the current forward are written
  std::atomic<int32_t> gather_seq{0};       // ... recorded for the forward with this sequence number
  const void* job_x_perm = nullptr;
  void* d_preact = nullptr;   // caller-owned [s_cap, 2f]: pass 1 saves a | b there when set (training)
  // pinned staging
  int32_t* h_counts = nullptr;
  feplb_group* h_dyn_groups = nullptr;          // pinned and mapped: the upload kernel reads it through h_dyn_groups_dev
  feplb_group* h_dyn_groups_dev = nullptr;
  uint32_t* h_status = nullptr;
  uint8_t* h_mask = nullptr;
  unsigned long long* h_counts_tagged = nullptr;   // pinned, written by the scan kernel: (sequence number << 32) | count
  int32_t flag_seq = 0;
  int32_t job_flag_seq = 0;          // 0: the job waits on ev_counts instead
  int32_t planner_timeout_ms = 2000; // bound of the planner's wait for the counts

  cudaStream_t copy_stream = nullptr;
  // pipelined host-buffer path: input and output copy streams and per-slot events
  cudaStream_t in_stream = nullptr, out_stream = nullptr;
  cudaEvent_t ev_in[FEPLB_HOST_SLOTS] = {}, ev_done[FEPLB_HOST_SLOTS] = {}, ev_out[FEPLB_HOST_SLOTS] = {};
  bool slot_used[FEPLB_HOST_SLOTS] = {};
  bool slot_staged[FEPLB_HOST_SLOTS] = {};     // inputs already on their way (feplb_host_stage_inputs)
  cudaEvent_t ev_range_in[FEPLB_MAX_RANGES] = {}, ev_range_out[FEPLB_MAX_RANGES] = {};   // host-buffer forward in token ranges
  cudaEvent_t ev_range_ids = nullptr;
  bool order_forced = false;       // feplb_set_launch_merging chose the launch order
  cudaEvent_t ev_counts = nullptr, ev_plan = nullptr;
  cudaEvent_t evr[kEvRing][EV_N] = {{nullptr}};
  cudaEvent_t* ev = evr[0];        // event set of the current forward
  bool ev_used[kEvRing] = {false};
  feplb_timeline ev_host[kEvRing]; // host fields of the forward that used the set
  int ev_slot = 0;
  bool timeline_on = false, timeline_valid = false;
  feplb_timeline tl;               // host fields of the current forward
  feplb_timeline tl_sum;           // totals over harvested forwards
  feplb_timeline tl_last;          // last harvested forward
  int64_t tl_n = 0;
  clk::time_point t0;

  // planner thread
  std::thread th;
  std::mutex mu;
  std::condition_variable cv;
  bool quit = false;
  int job = JOB_IDLE;
  std::atomic<bool> job_abort{false};   // the counts of the pending job will not come: its launches failed
  const uint8_t* job_mask = nullptr;
  const void* job_w1 = nullptr;   // weights of the current forward (sources of the Phase-2 copies)
  const void* job_w3 = nullptr;
  const void* job_w2 = nullptr;
  double copy_bytes = 0;
  int job_rc = FEPLB_OK;
  int n_dyn_groups = 0;
  int dyn_pair = 0;   // GEMM form chosen by the planner for the dynamic groups (it knows their sizes)
  // plan storage owned by the context
  std::vector<feplb_move> moves;
  std::vector<feplb_group> groups;
  std::vector<int64_t> load_before, load_after;
  std::vector<uint8_t> mask;
  std::vector<int64_t> score;
  feplb_plan_out plan;
};

namespace {

int fail(feplb_ctx* c, int code, const char* fmt, ...) {
  if (c) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(c->err, sizeof(c->err), fmt, ap);
    va_end(ap);
  }
  return code;
}
#define CUDA_TRY(ctx, call)                                                                      \
  do {                                                                                           \
    cudaError_t e_ = (call);                                                                     \
    if (e_ != cudaSuccess) return fail(ctx, FEPLB_E_CUDA, "%s: %s", #call, cudaGetErrorString(e_)); \
  } while (0)

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Bounded wait for the counts of job `seq`: either the front of the layer pass writes them straight into pinned
// host memory, each tagged with the forward's sequence number (whole-layer path), or (seq = 0) a copy was
// enqueued and its event is polled (stand-alone feplb_plan_async); no blocking driver call either way.
int await_counts(feplb_ctx* c, int32_t seq) {
  int rc = FEPLB_OK;
  const auto w0 = clk::now();
  for (uint32_t spin = 0;; ++spin) {
    if (seq) {
      int e = 0;
      for (; e < c->cfg.E; ++e) {
        const unsigned long long v = *(volatile unsigned long long*)(c->h_counts_tagged + e);
        if ((int32_t)(v >> 32) != seq) break;
        c->h_counts[e] = (int32_t)(uint32_t)v;
      }
      if (e == c->cfg.E) break;
      if (c->job_abort.load(std::memory_order_relaxed)) { rc = FEPLB_E_CUDA; break; }
    } else {
      cudaError_t q = cudaEventQuery(c->ev_counts);
      if (q == cudaSuccess) break;
      if (q != cudaErrorNotReady) { rc = FEPLB_E_CUDA; break; }
    }
    if ((spin & 1023u) == 1023u && std::chrono::duration<double>(clk::now() - w0).count() > 1e-3 * c->planner_timeout_ms) { rc = FEPLB_E_TIMEOUT; break; }
#if defined(__x86_64__) || defined(__i386__)
    __builtin_ia32_pause();     // a polite spin: the sibling hyper-thread (another rank's host thread) keeps its issue slots
#endif
  }
  std::atomic_thread_fence(std::memory_order_acquire);
  c->tl.host_counts_ready_us = us_since(c->t0);
  return rc;
}

// Mask (given, or derived from the counts) and plan of the counts in h_counts.
int make_plan(feplb_ctx* c, const uint8_t* mask) {
  const feplb_config& cfg = c->cfg;
  if (!mask) {
    for (int e = 0; e < cfg.E; ++e) c->score[e] = c->h_counts[e];
    feplb_select_dynamic(c->score.data(), cfg.E, cfg.R, cfg.dyn, c->mask.data());
  } else {
    memcpy(c->mask.data(), mask, cfg.E);
  }
  const auto p0 = clk::now();
  const int rc = feplb_plan(&cfg, c->h_counts, c->mask.data(), &c->plan);
  c->tl.plan_us = us_since(p0);
  c->tl.host_plan_done_us = us_since(c->t0);
  return rc;
}

// The planner thread: waits for the counts, derives mask and plan, uploads the dynamic groups.
void planner_main(feplb_ctx* c) {
  cudaSetDevice(c->device);
  for (;;) {
    {
      std::unique_lock<std::mutex> lk(c->mu);
      c->cv.wait(lk, [&] { return c->quit || c->job == JOB_PENDING; });
      if (c->quit) return;
      c->job = JOB_RUNNING;
    }
    int rc = await_counts(c, c->job_flag_seq);
    if (rc == FEPLB_OK) {
      const feplb_config& cfg = c->cfg;
      rc = make_plan(c, c->job_mask);
      if (rc == FEPLB_OK) {
        int n = 0;
        for (int i = 0; i < c->plan.n_groups; ++i)
          if (c->plan.groups[i].is_dynamic) c->h_dyn_groups[n++] = c->plan.groups[i];
        c->n_dyn_groups = n;
        cudaError_t ce = cudaSuccess;
        c->copy_bytes = 0;
        if (cfg.phase2_copy && c->job_w1) {
          // Phase 2 (Section 2.2): the weights of every migrated expert travel to the receiving
          // rank's buffer on the copy engines while the SMs compute the static experts.  Move i
          // takes the next free slot of its destination rank; the piece's group then reads slot s.
          const int L = cfg.E / cfg.R;
          const size_t per = (size_t)cfg.d * cfg.f * 2;
          std::vector<int> next_slot(cfg.R, 0), move_slot(c->plan.n_moves, 0);
          for (int i = 0; i < c->plan.n_moves && ce == cudaSuccess; ++i) {
            const feplb_move& m = c->plan.moves[i];
            const int s = m.dst * cfg.max_num_dyn + next_slot[m.dst]++;
            move_slot[i] = s;
            const char* src[3] = {(const char*)c->job_w1, (const char*)c->job_w3, (const char*)c->job_w2};
            char* dst[3] = {(char*)c->d_recv_w1, (char*)c->d_recv_w3, (char*)c->d_recv_w2};
            for (int k = 0; k < 3 && ce == cudaSuccess; ++k)
              ce = cudaMemcpyAsync(dst[k] + per * s, src[k] + per * m.expert, per, cudaMemcpyDeviceToDevice, c->copy_stream);
            c->copy_bytes += 3.0 * per;
          }
          std::vector<int> next_move(cfg.E, 0);   // per expert: moves consumed so far, in move order
          for (int g = 0; g < n; ++g) {
            feplb_group& gr = c->h_dyn_groups[g];
            if (gr.exec_rank == gr.expert / L) continue;      // home remainder: home weights
            int i = next_move[gr.expert];
            while (i < c->plan.n_moves && c->plan.moves[i].expert != gr.expert) ++i;
            next_move[gr.expert] = i + 1;
            if (i < c->plan.n_moves) gr.is_dynamic = 2 + move_slot[i];
          }
          // ... and so do the rows of the moved pieces (Section 2.2: Phase 2 redistributes tokens and
          // weights): each piece's rows go to the same row numbers of the receive region, once the
          // gather kernel of this forward has written them (the event is recorded by the calling thread,
          // which then publishes the forward's sequence number)
          if (ce == cudaSuccess && c->plan.n_moves > 0 && c->job_x_perm) {
            const auto g0 = clk::now();
            while (c->gather_seq.load(std::memory_order_acquire) != c->job_flag_seq &&
                   std::chrono::duration<double>(clk::now() - g0).count() < 1e-3 * c->planner_timeout_ms) {
#if defined(__x86_64__) || defined(__i386__)
              __builtin_ia32_pause();
#endif
            }
            if (c->gather_seq.load(std::memory_order_acquire) != c->job_flag_seq) ce = cudaErrorNotReady;
            if (ce == cudaSuccess) ce = cudaStreamWaitEvent(c->copy_stream, c->ev_gather, 0);
            const size_t row_bytes = (size_t)cfg.d * 2;
            for (int g = 0; g < n && ce == cudaSuccess; ++g) {
              const feplb_group& gr = c->h_dyn_groups[g];
              if (gr.is_dynamic < 2 || gr.rows <= 0) continue;
              ce = cudaMemcpyAsync((char*)c->d_recv_x + row_bytes * gr.row_start, (const char*)c->job_x_perm + row_bytes * gr.row_start,
                                   row_bytes * gr.rows, cudaMemcpyDeviceToDevice, c->copy_stream);
              c->copy_bytes += (double)row_bytes * gr.rows;
            }
          }
          if (ce == cudaSuccess && c->copy_bytes > 0) ce = cudaEventRecord(c->ev[EV_COPIES], c->copy_stream);
          if (ce != cudaSuccess) c->copy_bytes = 0;
          c->tl.phase2_copy_bytes = c->copy_bytes;
        }
        if (ce != cudaSuccess) rc = FEPLB_E_CUDA;
        int64_t dyn_rows = 0;
        for (int i = 0; i < n; ++i) dyn_rows += c->h_dyn_groups[i].rows;
        c->dyn_pair = c->gemm_pair_forced >= 0 ? c->gemm_pair_forced == FEPLB_FORM_PAIR : (n > 0 && dyn_rows >= (int64_t)512 * n);
        cudaError_t e = cudaSuccess;
        if (c->job_wm) {
          // A GEMM launch may already be running and waiting for this table (the merged launches
          // are never combined with Phase-2 copies): publish it from here, with a plain store into
          // mapped host memory, so that the waiting kernel depends on this thread alone.  The first
          // CTA that sees the word brings the table into device memory for the others; there is no
          // upload kernel on this path (it could not be relied on to run beside a kernel that holds
          // every SM, and a late one would overwrite the next forward's table).
          if (c->planner_delay_us > 0) std::this_thread::sleep_for(std::chrono::microseconds(c->planner_delay_us));
          const unsigned long long word = ((unsigned long long)(uint32_t)c->job_flag_seq << 32) | (uint32_t)n;
          for (int i = 0; i < n; ++i) {
            const feplb_group& gr = c->h_dyn_groups[i];
            volatile int32_t* t = c->h_dyn_tab32 + 8 * i;
            t[0] = gr.expert; t[1] = gr.row_start; t[2] = gr.rows; t[3] = gr.exec_rank;
            t[4] = gr.is_dynamic; t[5] = c->job_flag_seq; t[6] = 0; t[7] = 0;
          }
          std::atomic_thread_fence(std::memory_order_release);
          *(volatile unsigned long long*)c->h_dyn_ready = word;
          c->tl.host_upload_enqueued_us = us_since(c->t0);
        } else {
          if (n) e = feplb_launch_upload_groups(c->h_dyn_groups_dev, c->d_dyn_groups, n, c->copy_stream);
          if (e == cudaSuccess) e = cudaEventRecord(c->ev_plan, c->copy_stream);
          c->tl.host_upload_enqueued_us = us_since(c->t0);
        }
        if (e != cudaSuccess) rc = FEPLB_E_CUDA;
      }
    }
    if (rc != FEPLB_OK && c->job_wm && c->job_flag_seq) {
      // the launches of this forward must not wait for a table that will not come: an empty one
      std::atomic_thread_fence(std::memory_order_release);
      *(volatile unsigned long long*)c->h_dyn_ready = (unsigned long long)(uint32_t)c->job_flag_seq << 32;
    }
    {
      std::lock_guard<std::mutex> lk(c->mu);
      c->job_rc = rc;
      c->job = JOB_DONE;
    }
    c->cv.notify_all();
  }
}

int check_dev_ptrs(feplb_ctx* c, std::initializer_list<const void*> ptrs) {
  for (const void* p : ptrs)
    if (!p || !aligned16(p)) return fail(c, FEPLB_E_INVALID, "null or unaligned device pointer");
  return FEPLB_OK;
}

}  // namespace

// Most token rows per unit of the form for few rows per expert (feplb_gemm_few.cu), or 0 where the others are better.
// us per layer, single-CTA 128-row tiles -> units of 32 / 64 / 128 rows:
//   one wave of units: 8 experts, d = 128, f = 64: T = 256 18.7 -> 15.6 / 16.8 / 18.5, T = 1000 18.6 -> 16.6 / 17.6 / 20.0;
//     16 experts, d = 512, f = 256, 125 rows per expert 23.9 -> 24.5 / 23.0 / 21.4: the smallest units that fit
//   T <= 64 (an expert has two units of 32 at most): 64 experts, d = 2048, f = 768, top-6, T = 64 82.5 -> 77.0 / 81.0 / 82.7;
//     T = 96 83.5 -> 78.0 / 78.4 / 82.6; 64 experts, d = 4096, T = 90 134.7 -> 134.9 / 122.5 / 126.8
//   128 experts, d = 6144, f = 2048: 8 rows per expert 925 -> 855 / 815 / 822, 16 1052 -> 1140 / 984 / 961, 32 1225 -> 1641 /
//     1293 / 1144, 64 1402 -> 2427 / 1719 / 1386 (weights-on-M form 1334): small units leave room for more weights in flight,
//     but a busy expert's weights are read again for each
//   128 experts, d = 2560: f = 128 8 rows 55.1 -> 57.5 (64), 22 rows 65.1 -> 68.3; f = 192 8 rows 75.4 -> 66.1; f = 256 38
//     rows 106 -> 105 (128); f = 320 130 -> 123: units of a short second pass have mostly fixed costs
static int few_rows(const feplb_config& g, int num_sms) {
  const int64_t S = (int64_t)g.T * g.K, E = g.E, touched = S < E ? S : E, weight = (int64_t)g.d * g.f;
  const int64_t blocks = g.f / 64 > g.d / 128 ? g.f / 64 : g.d / 128;        // weight blocks of the wider pass
  for (int n = 32; n <= 128 && S < FEPLB_PAIR_MIN_ROWS_PER_EXPERT * E; n *= 2)
    if ((touched + S / n) * blocks <= num_sms) return n;
  int n = 0;
  if (S < 7 * E) n = g.T <= 64 ? 32 : 64;
  else if (g.f <= 128) n = 0;
  else if (weight < FEPLB_FEW_LARGE_WEIGHT) n = S < 24 * E ? 64 : 0;
  else n = S < 14 * E ? 64 : S < FEPLB_WM_MIN_ROWS_PER_EXPERT * E ? 128 : 0;
  if (!n) return 0;
  // A second wave of units that is mostly empty costs a whole one where units are long (their weights' 64 rows of f; the single
  // form's tiles are twice as wide).  How many experts a batch touches is known on the device alone: from 2048 columns on the guard
  // takes what an even routing would touch and stays clear of 1.125 to 2.25 waves of that, which are 1.0 to 1.4 waves of a skewed
  // one; a single token's experts are certain, and a wave is the line.  us per layer, waves of pass 1: 24 experts, d = 6144, f =
  // 1216, T = 1 (1.03) 83.4 -> 90.9; 60, d = 4608, f = 960, T = 21 (1.01) 69.4 -> 74.1; 128, d = 4992, f = 320, T = 10 (1.28) 80.8
  // -> 87.6; 64, d = 3840, f = 384, T = 9 (1.22) 65.0 -> 69.4; 64, d = 3584, f = 640, T = 5 (1.08) 60.6 -> 63.9; 128, d = 2048, f =
  // 192, T = 30 (1.38) 47.3 -> 51.2; 96, d = 2176, f = 192, T = 50 (1.07) 45.0 -> 48.2; below one wave and above 1.5 it gains 5 to
  // 24 % (32, d = 4224, f = 320, T = 34, 0.54 waves, 1.04 if even, 53.7 -> 42.2; 96, d = 4864, f = 1920, T = 2, 1.62 waves 6 %).
  // Shorter units lose less: 16, d = 1408, f = 576, T = 174 (1.3 waves if every expert is touched) 30.1 -> 31.7.  Units of 128 rows
  // need more waves: 4.4 waves 64, d = 2944, f = 576, T = 178 104 -> 112, 4.7 waves 128, d = 4992, f = 256, T = 745 224 -> 238, 5.0
  // waves 128, d = 5888, f = 320, T = 330 1.03 times faster.
  if (n < 128 && g.d >= 2048) {
    const double even = E * (1.0 - pow(1.0 - (double)g.K / E, g.T));
    const double units = g.f / 64 * (even > (double)S / n ? even : (double)S / n);
    if (weight >= FEPLB_FEW_GUARD_WEIGHT && units > (g.T == 1 ? 1.0 : 1.125) * num_sms && units < 2.25 * num_sms) return 0;
  } else if (weight >= FEPLB_WM_MIN_WEIGHT) {
    const int64_t units = g.f / 64 * (touched + S / n);
    if (5 * units > 6 * num_sms && units < (n == 128 ? 5 : 2) * num_sms) return 0;
  }
  // Narrow layers: a unit of pass 1 is its fixed costs, and busy experts have many: 128 experts, d = 128, f = 1152, T = 1679, top-1
  // 35.3 -> 39.4; 96, d = 256, f = 384, T = 344, top-5 29.2 -> 30.8; 128, d = 128, f = 768, 10.5 rows per expert 35.7 -> 36.7; but 64, d =
  // 128, f = 768, 9.98 rows 27.0 -> 25.4.
  if (g.d <= 256 && S >= 10 * E && g.f / 64 * touched >= 3 * num_sms) return 0;
  return n;
}

extern "C" int feplb_version(void) { return 100; }

extern "C" const char* feplb_strerror(int s) {
  switch (s) {
    case FEPLB_OK: return "ok";
    case FEPLB_E_INVALID: return "invalid argument";
    case FEPLB_E_RANGE: return "expert id out of range";
    case FEPLB_E_CUDA: return "CUDA error";
    case FEPLB_E_NOMEM: return "out of memory or capacity too small";
    case FEPLB_E_TIMEOUT: return "timed out";
    case FEPLB_E_STATE: return "invalid call order";
    case FEPLB_E_DEVICE: return "device-side check failed";
    default: return "unknown status";
  }
}

extern "C" int feplb_create(const feplb_config* cfg, feplb_ctx** out) {
  if (!out) return FEPLB_E_INVALID;
  *out = nullptr;
  int rc = feplb_validate_config(cfg);
  if (rc != FEPLB_OK) return rc;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return FEPLB_E_CUDA;
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, dev) != cudaSuccess) return FEPLB_E_CUDA;
  if (prop.major != 10) return FEPLB_E_CUDA;   // sm_100a code only
  feplb_ctx* c = new (std::nothrow) feplb_ctx();
  if (!c) return FEPLB_E_NOMEM;
  c->cfg = *cfg;
  c->device = dev;
  c->num_sms = prop.multiProcessorCount;
  c->s_cap = feplb_s_pad(cfg);
  // 256-row pair tiles pay off when an expert's segment is several tiles long on average
  c->gemm_pair_auto = c->gemm_pair_default = (int64_t)cfg->T * cfg->K >= (int64_t)2048 * cfg->E;
  // a launch over static and dynamic groups runs them in one form: the two-CTA form from 256 rows per expert, but small
  // weights, where a tile is short, from 288 rows in single-CTA tiles (us per layer: 16 experts, d = 512, f = 256, T = 30000,
  // top-2 107.9 -> 99.4; 48, d = 128, f = 64, 293 rows 33.6 -> 26.9; 24, d = 640, f = 256, 300 rows 40.2 -> 36.0; 128, d = 1792,
  // f = 128, 330 rows 187 -> 173; 8, d = 6144, f = 64, 1761 rows 260 -> 245; 128, d = 1792, f = 256, 604 rows 396 -> 386; d = 2688,
  // f = 192, 2262 rows 379 -> 361; d = 1152, f = 384, 1903 rows 92.6 -> 91.9; but d = 1536, f = 576, 6713 rows 302 -> 359,
  // and d = 512, f = 832, 6118 rows 150 -> 160: from 256 Ki elements on only where f is short).  From 256 rows to that line
  // small weights would gain as well (258 rows, two-CTA -> single: 8, d = 128, f = 64 21.2 -> 18.2; 24, d = 640, f = 256 40.2 -> 34.8; 64,
  // d = 1792, f = 128 95.9 -> 87.7; 32, d = 1152, f = 384 64.9 -> 57.5; 48, d = 256, f = 512 47.6 -> 40.2).
  const int64_t weight = (int64_t)cfg->d * cfg->f;
  const bool short_tiles = (weight < FEPLB_SHORT_TILE_WEIGHT / 2 || (weight < FEPLB_SHORT_TILE_WEIGHT && cfg->f <= 384)) && (int64_t)cfg->T * cfg->K >= (int64_t)FEPLB_SHORT_TILE_MIN_ROWS * cfg->E;
  c->merged_pair = (int64_t)cfg->T * cfg->K >= (int64_t)FEPLB_PAIR_MIN_ROWS_PER_EXPERT * cfg->E && !short_tiles;
  // Deep stages of that form (128 elements of K, and tiles of 128 rows): the epilogue that serves both tile heights costs
  // every tile a little, a stage of 128 elements is half empty where the width is an odd number of 64, and a ring of three is
  // less in flight while weights stream.  us per layer at the power cap, 64-element stages / deep ones:
  //   large: 128 experts, d = 6144, f = 2048, 1024 rows per expert 9855 / 9547, 4096 rows 37217 / 36420; 32, d = 4096, f = 1024,
  //     4096 rows 3091 / 3035; 16, d = 6144, f = 768, 3000 rows 1404 / 1375; d = 1536, f = 1408, 300 rows 107.8 / 103.3
  //   many groups, i.e. many last tiles: 128, d = 2560, f = 320, 264 rows 406 / 389; 96, d = 384, f = 1024, 313 rows 158 / 151
  //   short second pass: 48, d = 3584, f = 192, 8300 rows 3187 / 3435; 24, d = 3072, f = 192, 15000 rows 2502 / 2676; 16, d = 2560,
  //     f = 256, 1294 rows 199.5 / 205.0; 16, d = 4736, f = 256, 269 rows 85.5 / 87.9; short first pass: 96, d = 128, f = 512, 286
  //     rows 58.3 / 61.7
  //   ... and few groups: 8, d = 512, f = 832, 6118 rows 169.5 / 173.6; 16, d = 512, f = 1024, 1754 rows 122.5 / 124.6; 8, d = 512, f =
  //     704, 2088 rows 63.5 / 64.9; d = 640 level
  //   less than two waves of tiles: 16, d = 1536, f = 640, 290 rows 55.2 / 57.9; 16, d = 3328, f = 320, 306 rows 89.4 / 90.5; 16, d =
  //     512, f = 640, 441 rows 41.9 / 42.9; 16, d = 1664, f = 448, 304 rows 59.2 / 61.5
  {
    const int64_t m_tiles = (int64_t)cfg->T * cfg->K / 256 + cfg->E / 2, clusters = c->num_sms / 2;
    const int64_t blocks = std::min((cfg->f + 127) / 128, (cfg->d + 255) / 256);     // N tiles of the narrower pass
    c->pair_deep = cfg->f > 256 && cfg->d >= 256 &&
                   (weight >= FEPLB_PAIR_DEEP_WEIGHT || cfg->E >= FEPLB_PAIR_DEEP_EXPERTS || (cfg->d >= 768 && m_tiles * blocks >= 2 * clusters));
  }
  // backward GEMMs: the pair form pays once an expert's segment spans several 256-row tiles
  // (measured: -7.5 % backward time at 1024 rows per expert, slower at 384)
  c->bwd_pair_auto = c->bwd_pair = (int64_t)cfg->T * cfg->K >= (int64_t)512 * cfg->E ? 3 : 0;
  const int64_t S = (int64_t)cfg->T * cfg->K;
  c->nb = (int)((S + FEPLB_SLOTS_PER_BLOCK - 1) / FEPLB_SLOTS_PER_BLOCK);
  const int cap_moves = cfg->R * cfg->max_num_dyn;
  const int cap_groups = cfg->E + cap_moves;
  // Weights-on-M form: no padding rows to speak of, and an expert's weights cross the L2 ports once per 256 rows.
  // us per layer, single-CTA 128-row tiles / two-CTA 256-row tiles / weights on M:
  //   128 experts, d = 6144, f = 2048: 64 rows per expert 1498 / 1485 / 1363, 128 2212 / 2160 / 1940, 512 5645 / 5383 / 5163,
  //     1024 10110 / 9500 / 9622;  32 experts, d = 4096, f = 1024: 88 194 / 193 / 178, 512 525 / 494 / 478
  //   64 experts, d = 2048, f = 768: 66 136.6 / 142.0 / 132.9, 131 188.7 / 184.2 / 173.5, 384 342 / 330 / 322, 768 607 / 577 / 572,
  //     2812 1917 / 1815 / 1832
  //   half-empty last weight blocks (60 experts, d = 1920, f = 704): 102 145.8 / 152.4 / 140.0, 400 312 / 304 / 298
  //   32 experts, d = 1024, f = 512: 112 44.8 / 44.6 / 43.2, 250 63.2 / 61.4 / 59.6;  16, d = 512, f = 256: 375 28.4 / 30.9 / 31.3
  // Below 3 Mi elements the launch must have six waves of units and at most an eighth of them empty: 24 experts, d = 2304, f =
  // 320, 113 rows, 1.4 waves 48 -> 59; 16, d = 2944, f = 448, 132 rows, 1.3 waves 55 -> 65; 48, d = 2688, f = 384, 169 rows, 3.2
  // waves 112 -> 123; 64, d = 2816, f = 512, 135 rows, 5.3 waves 163 -> 172; 128, d = 2560, f = 320 (a sixth empty), 264 rows,
  // 10.5 waves 355 -> 365; but 60, d = 1920, f = 704, 6.8 waves 146 -> 141, 32, d = 1920, f = 448, 9 waves 1.08 times faster.
  const int64_t f_blocks = (cfg->f + 127) / 128;
  const bool wm_units = f_blocks * (cfg->E + S / 256) >= 6 * (c->num_sms / 2) && f_blocks * 128 * 7 <= (int64_t)cfg->f * 8;
  const bool wm_can = feplb_wm_supported(cfg->E, cfg->E + cap_groups);
  c->few_auto = c->few = few_rows(*cfg, c->num_sms);
  c->wm_ok = wm_can && cfg->f % 128 == 0 && cfg->d % 256 == 0;
  const bool large = weight >= FEPLB_MERGED_ANY_ROWS_WEIGHT;
  c->wm_merged_auto = c->wm_merged = wm_can && S >= (int64_t)FEPLB_WM_MIN_ROWS_PER_EXPERT * cfg->E &&
                                     S < (int64_t)FEPLB_WM_MAX_ROWS_PER_EXPERT * cfg->E &&
                                     (weight >= FEPLB_WM_ANY_UNITS_WEIGHT || (weight >= FEPLB_WM_MIN_WEIGHT && wm_units));
  c->wm_auto = c->wm = c->wm_merged && S < (int64_t)FEPLB_MERGED_MAX_ROWS_PER_EXPERT * cfg->E;
  // In the four-launch order the static experts are the less busy ones and stay in the range above for longer: d = 6144,
  // f = 2048, 128 experts, 1024 rows per expert on average 9911 -> 9750 us per layer, 1500 rows 13828 -> 13785.
  c->wm_static_auto = c->wm_static = wm_can && S < (int64_t)2048 * cfg->E && weight >= FEPLB_WM_ANY_UNITS_WEIGHT;
  // One launch per pass over the static and then the dynamic groups (the table of the latter is
  // picked up on the device): saves two launch ramps and two partly filled last waves per forward,
  // which matters while a forward's GEMMs take up to a few milliseconds.  Launches of their own -> one, us per layer
  // (weights on M / two-CTA tiles): 64 experts, d = 2048, f = 768, 768 rows per expert 549 -> 533 / 535, 1536 994 ->
  // 979 / 978, 2812 1735 -> 1717 / 1687, 6144 3654 -> 3656 / 3611; 32, d = 4096, f = 1024, 1024 rows 866 -> 834 / 841, 2048
  // 1555 -> 1562 / 1543; 64, d = 3072, f = 1536, 1250 2087 -> 2065 / 2103.  At large weights (d = 6144, f = 2048) the two
  // are within 1 %, and static and dynamic groups keep a form each from 768 rows per expert.
  c->merged_ok = cfg->E + cap_groups <= FEPLB_MAX_GROUPS;
  c->merged_auto = c->merged = c->merged_ok && (!large || S < (int64_t)FEPLB_MERGED_MAX_ROWS_PER_EXPERT * cfg->E);
  // Small batches: a migration only relabels the rank that executes rows whose weights are the same everywhere, so
  // the launches need not wait for the plan at all.  They do where the static groups keep the GPU busy for longer
  // than the planner takes (its table is then there in time); below that the wait and the table's way to the
  // device cost up to 10 us per forward, and the plan (returned as ever) is made by the calling thread
  // instead.  Whole layer, table order -> this: 27.9 -> 19.6 us (T = 256, top-2, d = 128, 8 experts), 30.8 ->
  // 20.3 (the same at T = 1200), 97.9 -> 88.7 (T = 64, top-6, d = 2048, 64 experts), 156.7 -> 148.9 (102 rows
  // per expert, d = 1920), 181 -> 170 (128 of d = 2048).  Above the line, where the table comes with the gather, the two
  // are level: 173.6 and 172.0 at 131 rows per expert of d = 2048, 211 and 211 at 188, 286 and 284 at 281, 2001 and 1989
  // at 128 of d = 6144; at 1024 of d = 6144 the order that gives the static groups launches of their own is 4 % ahead.
  // Up to 8192 slots no CTA of the front picks the table up, the launches always take the late way, and the line lies
  // elsewhere: 192 rows per expert.  Table order -> this: 32 experts of d = 6144, f = 2048, 256 rows each 789 -> 764 us, 32 of
  // d = f = 2048, 256 rows 285 -> 266, 24 of d = 3072, f = 1536, 333 rows 321 -> 296, 16 of d = 6144, f = 2048, 512 rows
  // 707 -> 678; at 171 rows (48 experts, d = 6144) 952 -> 932, within the runs of one side.  From 768 rows per expert of large weights static and dynamic groups keep the launches of
  // their own that feplb_forward_path reports there.
  // The time is an estimate: all weights streamed at 6.5 TB/s plus the products at 1 PFLOP/s.
  const double ffn_us = 6.0 * cfg->d * cfg->f * ((double)cfg->E / 6.5e6 + (double)S / 1e9);
  c->direct_auto = c->direct = S < (int64_t)FEPLB_DIRECT_ROWS_PER_EXPERT * cfg->E || ffn_us < FEPLB_DIRECT_FFN_US ||
                                (c->merged && feplb_front_is_small(S, cfg->E) && S >= (int64_t)FEPLB_DIRECT_SMALL_FRONT_ROWS * cfg->E);
  bool ok = true;
  ok = ok && cudaMalloc(&c->d_dyn_ready, 4 * sizeof(unsigned long long)) == cudaSuccess &&
       cudaMemset(c->d_dyn_ready, 0, 4 * sizeof(unsigned long long)) == cudaSuccess;
  ok = ok && cudaHostAlloc(&c->h_dyn_ready, sizeof(unsigned long long), cudaHostAllocMapped) == cudaSuccess &&
       cudaHostGetDevicePointer(&c->h_dyn_ready_dev, c->h_dyn_ready, 0) == cudaSuccess;
  if (ok) *c->h_dyn_ready = 0;
  ok = ok && cudaHostAlloc(&c->h_dyn_tab32, 32 * (size_t)(cap_groups > 0 ? cap_groups : 1), cudaHostAllocMapped) == cudaSuccess &&
       cudaHostGetDevicePointer(&c->h_dyn_tab32_dev, c->h_dyn_tab32, 0) == cudaSuccess;
  if (ok) memset(c->h_dyn_tab32, 0, 32 * (size_t)(cap_groups > 0 ? cap_groups : 1));
  ok = ok && cudaMalloc(&c->d_dyn_tab32, 32 * (size_t)(cap_groups > 0 ? cap_groups : 1)) == cudaSuccess &&
       cudaMemset(c->d_dyn_tab32, 0, 32 * (size_t)(cap_groups > 0 ? cap_groups : 1)) == cudaSuccess;
  ok = ok && cudaMalloc(&c->d_stamps, sizeof(unsigned long long) * kEvRing * kStampWords) == cudaSuccess;
  ok = ok && cudaMallocHost(&c->h_stamps, sizeof(unsigned long long) * kEvRing * kStampWords) == cudaSuccess;
  ok = ok && cudaMalloc(&c->d_block_hist, sizeof(int32_t) * (size_t)(c->nb > 0 ? c->nb : 1) * cfg->E) == cudaSuccess;
  ok = ok && cudaMalloc(&c->d_pad_off, sizeof(int32_t) * (cfg->E + 1)) == cudaSuccess;
  ok = ok && cudaMalloc(&c->d_totals, sizeof(int32_t) * (cfg->E + 1)) == cudaSuccess &&
       cudaMemset(c->d_totals, 0, sizeof(int32_t) * (cfg->E + 1)) == cudaSuccess;
  ok = ok && cudaMalloc(&c->d_status, sizeof(uint32_t)) == cudaSuccess;
  ok = ok && cudaMalloc(&c->d_home_groups, sizeof(feplb_group) * cfg->E) == cudaSuccess;
  ok = ok && cudaMalloc(&c->d_dyn_groups, (sizeof(feplb_group) * cap_groups + 15) / 16 * 16) == cudaSuccess;
  ok = ok && cudaMalloc(&c->d_range_groups, sizeof(feplb_group) * cfg->E * FEPLB_MAX_RANGES) == cudaSuccess;
  ok = ok && cudaMalloc(&c->d_mask, cfg->E) == cudaSuccess;
  if (cfg->phase2_copy && (int64_t)cfg->R * cfg->max_num_dyn > 30000) ok = false;   // slot ids travel in 15 bits
  if (ok && cfg->phase2_copy) {
    c->n_recv_slots = cfg->R * cfg->max_num_dyn;
    const size_t per = (size_t)cfg->d * cfg->f * 2, n = (size_t)(c->n_recv_slots > 0 ? c->n_recv_slots : 1);
    ok = ok && cudaMalloc(&c->d_recv_w1, per * n) == cudaSuccess;
    ok = ok && cudaMalloc(&c->d_recv_w3, per * n) == cudaSuccess;
    ok = ok && cudaMalloc(&c->d_recv_w2, per * n) == cudaSuccess;
    ok = ok && cudaMalloc(&c->d_recv_x, (size_t)(c->s_cap > 0 ? c->s_cap : 1) * cfg->d * 2) == cudaSuccess;
    ok = ok && cudaEventCreateWithFlags(&c->ev_gather, cudaEventDisableTiming) == cudaSuccess;
  }
  ok = ok && cudaMallocHost(&c->h_counts, sizeof(int32_t) * cfg->E) == cudaSuccess;
  ok = ok && cudaHostAlloc(&c->h_dyn_groups, (sizeof(feplb_group) * cap_groups + 15) / 16 * 16, cudaHostAllocMapped) == cudaSuccess &&
       cudaHostGetDevicePointer(&c->h_dyn_groups_dev, c->h_dyn_groups, 0) == cudaSuccess;
  ok = ok && cudaMallocHost(&c->h_status, sizeof(uint32_t)) == cudaSuccess;
  ok = ok && cudaMallocHost(&c->h_mask, cfg->E) == cudaSuccess;
  ok = ok && cudaMallocHost(&c->h_counts_tagged, sizeof(unsigned long long) * (cfg->E > 0 ? cfg->E : 1)) == cudaSuccess;
  if (ok) memset(c->h_counts_tagged, 0, sizeof(unsigned long long) * cfg->E);
  ok = ok && cudaMemset(c->d_status, 0, sizeof(uint32_t)) == cudaSuccess;
  ok = ok && cudaStreamCreateWithFlags(&c->copy_stream, cudaStreamNonBlocking) == cudaSuccess;
  ok = ok && cudaStreamCreateWithFlags(&c->in_stream, cudaStreamNonBlocking) == cudaSuccess;
  ok = ok && cudaStreamCreateWithFlags(&c->out_stream, cudaStreamNonBlocking) == cudaSuccess;
  for (int i = 0; ok && i < FEPLB_HOST_SLOTS; ++i)
    ok = cudaEventCreateWithFlags(&c->ev_in[i], cudaEventDisableTiming) == cudaSuccess &&
         cudaEventCreateWithFlags(&c->ev_done[i], cudaEventDisableTiming) == cudaSuccess &&
         cudaEventCreateWithFlags(&c->ev_out[i], cudaEventDisableTiming) == cudaSuccess;
  for (int i = 0; ok && i < FEPLB_MAX_RANGES; ++i)
    ok = cudaEventCreateWithFlags(&c->ev_range_in[i], cudaEventDisableTiming) == cudaSuccess &&
         cudaEventCreateWithFlags(&c->ev_range_out[i], cudaEventDisableTiming) == cudaSuccess;
  ok = ok && cudaEventCreateWithFlags(&c->ev_range_ids, cudaEventDisableTiming) == cudaSuccess;
  ok = ok && cudaEventCreate(&c->ev_counts) == cudaSuccess;
  ok = ok && cudaEventCreateWithFlags(&c->ev_plan, cudaEventDisableTiming) == cudaSuccess;
  for (int r = 0; ok && r < kEvRing; ++r)
    for (int i = 0; ok && i < EV_N; ++i) ok = cudaEventCreate(&c->evr[r][i]) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    feplb_destroy(c);
    return FEPLB_E_NOMEM;
  }
  c->moves.resize(cap_moves > 0 ? cap_moves : 1);
  c->groups.resize(cap_groups);
  c->load_before.resize(cfg->R);
  c->load_after.resize(cfg->R);
  c->mask.resize(cfg->E);
  c->score.resize(cfg->E);
  c->plan = feplb_plan_out{0, 0, cap_moves, cap_groups, c->moves.data(), c->groups.data(),
                           c->load_before.data(), c->load_after.data()};
  memset(&c->tl, 0, sizeof(c->tl));
  memset(&c->tl_sum, 0, sizeof(c->tl_sum));
  memset(&c->tl_last, 0, sizeof(c->tl_last));
  c->th = std::thread(planner_main, c);
  *out = c;
  return FEPLB_OK;
}

extern "C" int feplb_destroy(feplb_ctx* c) {
  if (!c) return FEPLB_OK;
  if (c->th.joinable()) {
    {
      std::lock_guard<std::mutex> lk(c->mu);
      c->quit = true;
    }
    c->cv.notify_all();
    c->th.join();
  }
  cudaSetDevice(c->device);
  cudaDeviceSynchronize();
  cudaFree(c->d_block_hist);
  cudaFree(c->d_pad_off);
  cudaFree(c->d_totals);
  cudaFree(c->d_status);
  cudaFree(c->d_home_groups);
  cudaFree(c->d_dyn_groups);
  cudaFree(c->d_range_groups);
  cudaFree(c->d_mask);
  cudaFree(c->d_recv_w1);
  cudaFree(c->d_recv_w3);
  cudaFree(c->d_recv_w2);
  cudaFree(c->d_recv_x);
  if (c->ev_gather) cudaEventDestroy(c->ev_gather);
  cudaFree(c->d_dyn_ready);
  cudaFree(c->d_dyn_tab32);
  cudaFreeHost(c->h_dyn_tab32);
  cudaFree(c->d_stamps);
  cudaFreeHost(c->h_dyn_ready);
  cudaFreeHost(c->h_stamps);
  cudaFreeHost(c->h_counts);
  cudaFreeHost(c->h_dyn_groups);
  cudaFreeHost(c->h_status);
  cudaFreeHost(c->h_mask);
  cudaFreeHost(c->h_counts_tagged);
  if (c->copy_stream) cudaStreamDestroy(c->copy_stream);
  if (c->in_stream) cudaStreamDestroy(c->in_stream);
  if (c->out_stream) cudaStreamDestroy(c->out_stream);
  for (int i = 0; i < FEPLB_HOST_SLOTS; ++i) {
    if (c->ev_in[i]) cudaEventDestroy(c->ev_in[i]);
    if (c->ev_done[i]) cudaEventDestroy(c->ev_done[i]);
    if (c->ev_out[i]) cudaEventDestroy(c->ev_out[i]);
  }
  for (int i = 0; i < FEPLB_MAX_RANGES; ++i) {
    if (c->ev_range_in[i]) cudaEventDestroy(c->ev_range_in[i]);
    if (c->ev_range_out[i]) cudaEventDestroy(c->ev_range_out[i]);
  }
  if (c->ev_range_ids) cudaEventDestroy(c->ev_range_ids);
  if (c->ev_counts) cudaEventDestroy(c->ev_counts);
  if (c->ev_plan) cudaEventDestroy(c->ev_plan);
  for (int r = 0; r < kEvRing; ++r)
    for (int i = 0; i < EV_N; ++i)
      if (c->evr[r][i]) cudaEventDestroy(c->evr[r][i]);
  cudaGetLastError();
  delete c;
  return FEPLB_OK;
}

extern "C" const char* feplb_last_error(const feplb_ctx* c) { return c ? c->err : ""; }

extern "C" int32_t feplb_forward_path(const feplb_ctx* c) { return c ? c->path : 0; }

extern "C" int32_t feplb_forward_detail(const feplb_ctx* c) { return c ? c->detail : 0; }

extern "C" int64_t feplb_launch_count(const feplb_ctx* c) { return c ? c->launches : 0; }

extern "C" int feplb_check_status(feplb_ctx* c, void* stream) {
  if (!c) return FEPLB_E_INVALID;
  cudaStream_t st = (cudaStream_t)stream;
  CUDA_TRY(c, cudaMemcpyAsync(c->h_status, c->d_status, sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
  CUDA_TRY(c, cudaMemsetAsync(c->d_status, 0, sizeof(uint32_t), st));
  CUDA_TRY(c, cudaStreamSynchronize(st));
  const uint32_t s = *c->h_status;
  if (s & FEPLB_ST_WAIT) return fail(c, FEPLB_E_DEVICE, "a bounded device-side wait gave up (status 0x%x)", s);
  if (s & FEPLB_ST_PLAN)
    return fail(c, FEPLB_E_TIMEOUT, "the expert GEMM gave up waiting for the planner's dynamic group table (status 0x%x)", s);
  if (s & FEPLB_ST_GROUP) return fail(c, FEPLB_E_DEVICE, "malformed group entry (status 0x%x)", s);
  if (s & FEPLB_ST_COUNTS) return fail(c, FEPLB_E_DEVICE, "counts disagree with topk_ids (status 0x%x)", s);
  if (s & FEPLB_ST_RANGE) return fail(c, FEPLB_E_RANGE, "expert id outside [0, E) (status 0x%x)", s);
  return FEPLB_OK;
}

extern "C" int feplb_route_hist(feplb_ctx* c, const int32_t* topk_ids, int32_t* counts, int32_t* rank_load, void* stream) {
  if (!c) return FEPLB_E_INVALID;
  if (!counts || !rank_load || (!topk_ids && c->cfg.T > 0)) return fail(c, FEPLB_E_INVALID, "route_hist: null pointer");
  const int64_t S = (int64_t)c->cfg.T * c->cfg.K;
  CUDA_TRY(c, feplb_launch_route_hist(topk_ids, S, c->cfg.E, c->cfg.R, c->d_totals, counts, rank_load, c->d_status,
                                      (cudaStream_t)stream, &c->launches));
  return FEPLB_OK;
}

static int dispatch_impl(feplb_ctx* c, const void* x, const int32_t* topk_ids, const int32_t* counts, void* x_perm,
                         int32_t* slot_to_row, int32_t* row_to_token, cudaStream_t st) {
  const feplb_config& g = c->cfg;
  const int64_t S = (int64_t)g.T * g.K;
  if (!counts || !row_to_token) return fail(c, FEPLB_E_INVALID, "dispatch: null pointer");
  if (g.T > 0) {
    int rc = check_dev_ptrs(c, {x, x_perm});
    if (rc != FEPLB_OK) return rc;
    if (!topk_ids || !slot_to_row) return fail(c, FEPLB_E_INVALID, "dispatch: null pointer");
  }
  if (feplb_front_is_small(S, g.E)) {
    CUDA_TRY(c, feplb_launch_front_small(x, topk_ids, g.T, g.K, g.E, g.R, g.d, g.row_align, 0, nullptr, counts, nullptr, nullptr,
                                         nullptr, nullptr, slot_to_row, row_to_token, x_perm, (int64_t)c->s_cap, c->d_status,
                                         nullptr, 0, nullptr, c->num_sms, st, &c->launches));
    return FEPLB_OK;
  }
  CUDA_TRY(c, feplb_launch_permute(topk_ids, S, g.K, g.E, g.row_align, counts, c->d_block_hist, c->d_pad_off,
                                   slot_to_row, row_to_token, (int64_t)c->s_cap, c->d_status, st, &c->launches));
  CUDA_TRY(c, feplb_launch_gather(x, topk_ids, c->d_block_hist, slot_to_row, counts, c->d_pad_off, x_perm, g.T, g.K, g.E,
                                  g.d, g.row_align, (int64_t)c->s_cap, c->num_sms, st, &c->launches, row_to_token, true));
  return FEPLB_OK;
}

extern "C" int feplb_dispatch(feplb_ctx* c, const void* x, const int32_t* topk_ids, const int32_t* counts,
                              void* x_perm, int32_t* slot_to_row, int32_t* row_to_token, void* stream) {
  if (!c) return FEPLB_E_INVALID;
  return dispatch_impl(c, x, topk_ids, counts, x_perm, slot_to_row, row_to_token, (cudaStream_t)stream);
}

extern "C" int feplb_home_groups(feplb_ctx* c, const int32_t* counts, const uint8_t* dyn_mask,
                                 feplb_group* groups_out, uint8_t* dyn_mask_out, void* stream) {
  if (!c) return FEPLB_E_INVALID;
  if (!counts || !groups_out) return fail(c, FEPLB_E_INVALID, "home_groups: null pointer");
  if (!dyn_mask && c->cfg.mask_policy != FEPLB_MASK_REACTIVE)
    return fail(c, FEPLB_E_INVALID, "home_groups: dyn_mask is required unless mask_policy is REACTIVE");
  CUDA_TRY(c, feplb_launch_home_groups(counts, dyn_mask, c->cfg.E, c->cfg.R, c->cfg.row_align, c->cfg.dyn,
                                       groups_out, dyn_mask_out, (cudaStream_t)stream, &c->launches));
  return FEPLB_OK;
}

// `dyn` != nullptr: weights-on-M launches that go on to the planner's dynamic table after `groups`.
static int ffn_impl(feplb_ctx* c, const void* x_perm, const void* w1, const void* w3, const void* w2,
                    const feplb_group* groups, int32_t n_groups, int32_t which, void* h, void* y, cudaStream_t st,
                    int pair = -1, const feplb_wm_dyn* dyn = nullptr, bool weights_on_m = false) {
  if (pair < 0) pair = c->gemm_pair_default;
  if (n_groups < 0 || n_groups > FEPLB_MAX_GROUPS) return fail(c, FEPLB_E_INVALID, "expert_ffn: n_groups out of range");
  if (which != FEPLB_FFN_ALL && which != FEPLB_FFN_STATIC && which != FEPLB_FFN_DYNAMIC)
    return fail(c, FEPLB_E_INVALID, "expert_ffn: bad selector");
  if ((n_groups == 0 && !dyn) || c->s_cap == 0) return FEPLB_OK;
  int rc = check_dev_ptrs(c, {x_perm, w1, w3, w2, h, y});
  if (rc != FEPLB_OK) return rc;
  if (!groups) return fail(c, FEPLB_E_INVALID, "expert_ffn: null group table");
  feplb_gemm_args a;
  a.x_perm = x_perm; a.w1 = w1; a.w3 = w3; a.w2 = w2; a.h = h; a.y = y;
  a.groups = groups; a.n_groups = n_groups; a.which = which;
  a.E = c->cfg.E; a.d = c->cfg.d; a.f = c->cfg.f; a.s_cap = (int64_t)c->s_cap;
  a.status = c->d_status; a.num_sms = c->num_sms; a.pair = pair; a.deep = c->pair_deep;
  a.ab_out = c->d_preact;
  a.recv_w1 = c->d_recv_w1; a.recv_w3 = c->d_recv_w3; a.recv_w2 = c->d_recv_w2; a.n_recv_slots = c->n_recv_slots;
  a.recv_x = c->d_recv_x;
  // k_ffn_few reads home weights only and one table: not with receive slots, not where a launch picks the planner's table up
  if (c->few && !weights_on_m && !a.n_recv_slots && !(dyn && dyn->seq)) {
    rc = feplb_launch_expert_ffn_few(a, st, &c->launches, c->err, sizeof(c->err), c->few, dyn ? dyn->stamps : nullptr);
    if (rc != FEPLB_E_STATE) {
      c->path |= FEPLB_PATH_SINGLE;
      c->detail |= c->few;             // FEPLB_DETAIL_UNITS_*
      return rc;
    }
  }
  if ((weights_on_m || (dyn ? c->wm_merged : c->wm)) && n_groups + (dyn ? dyn->max_groups : 0) <= FEPLB_WM_MAX_ENTRIES) {
    const feplb_wm_dyn none;
    rc = feplb_launch_expert_ffn_wm(a, dyn ? *dyn : none, st, &c->launches, c->err, sizeof(c->err));
    if (rc != FEPLB_E_STATE) {
      c->path |= FEPLB_PATH_WEIGHT_M;
      return rc;
    }
  }
  c->path |= pair ? FEPLB_PATH_PAIR : FEPLB_PATH_SINGLE;
  if (pair && a.deep) c->detail |= FEPLB_DETAIL_DEEP_STAGES;
  return feplb_launch_expert_ffn(a, st, &c->launches, c->err, sizeof(c->err), dyn);
}

extern "C" int feplb_expert_ffn(feplb_ctx* c, const void* x_perm, const void* w1, const void* w3, const void* w2,
                                const feplb_group* groups, int32_t n_groups, int32_t which,
                                void* h_scratch, void* y_perm, void* stream) {
  if (!c) return FEPLB_E_INVALID;
  const int32_t path = c->path, detail = c->detail;         // of the last forward, which this call is not
  const int rc = ffn_impl(c, x_perm, w1, w3, w2, groups, n_groups, which, h_scratch, y_perm, (cudaStream_t)stream);
  c->path = path;
  c->detail = detail;
  return rc;
}

extern "C" int feplb_combine(feplb_ctx* c, const void* y_perm, const int32_t* slot_to_row, const float* gates,
                             void* out, void* stream) {
  if (!c) return FEPLB_E_INVALID;
  if (c->cfg.T == 0) return FEPLB_OK;
  int rc = check_dev_ptrs(c, {y_perm, out});
  if (rc != FEPLB_OK) return rc;
  if (!slot_to_row || !gates) return fail(c, FEPLB_E_INVALID, "combine: null pointer");
  CUDA_TRY(c, feplb_launch_combine(y_perm, slot_to_row, gates, out, c->cfg.T, c->cfg.K, c->cfg.d, c->num_sms,
                                   (cudaStream_t)stream, &c->launches));
  return FEPLB_OK;
}

extern "C" int feplb_plan_async(feplb_ctx* c, const int32_t* counts, const uint8_t* dyn_mask_host, void* stream) {
  if (!c) return FEPLB_E_INVALID;
  if (!counts) return fail(c, FEPLB_E_INVALID, "plan_async: null counts");
  if (!dyn_mask_host && c->cfg.mask_policy != FEPLB_MASK_REACTIVE)
    return fail(c, FEPLB_E_INVALID, "plan_async: dyn_mask_host is required unless mask_policy is REACTIVE");
  {
    std::lock_guard<std::mutex> lk(c->mu);
    if (c->job != JOB_IDLE) return fail(c, FEPLB_E_STATE, "plan_async: a plan is already pending");
  }
  cudaStream_t st = (cudaStream_t)stream;
  if (!c->timeline_valid) c->t0 = clk::now();
  CUDA_TRY(c, cudaMemcpyAsync(c->h_counts, counts, sizeof(int32_t) * c->cfg.E, cudaMemcpyDeviceToHost, st));
  CUDA_TRY(c, cudaEventRecord(c->ev_counts, st));
  {
    std::lock_guard<std::mutex> lk(c->mu);
    c->job_mask = dyn_mask_host;
    c->job_flag_seq = 0;
    c->job_wm = false;
    c->job = JOB_PENDING;
  }
  c->cv.notify_all();
  return FEPLB_OK;
}

// Whole-layer path: the counts of this forward arrive in h_counts with sequence number `seq`.
static int plan_kick_flag(feplb_ctx* c, const uint8_t* dyn_mask_host, int32_t seq, bool wm) {
  {
    std::lock_guard<std::mutex> lk(c->mu);
    if (c->job != JOB_IDLE) return fail(c, FEPLB_E_STATE, "moe_forward: a plan is already pending");
    c->job_mask = dyn_mask_host;
    c->job_wm = wm;
    c->job_flag_seq = seq;
    c->job_abort.store(false, std::memory_order_relaxed);
    c->job = JOB_PENDING;
  }
  c->cv.notify_all();
  return FEPLB_OK;
}

// The context's plan -> the caller's arrays (NULL: not wanted).
static int copy_plan(feplb_ctx* c, feplb_plan_out* plan_copy) {
  if (!plan_copy) return FEPLB_OK;
  if (plan_copy->cap_moves < c->plan.n_moves || plan_copy->cap_groups < c->plan.n_groups ||
      !plan_copy->load_before || !plan_copy->load_after)
    return fail(c, FEPLB_E_NOMEM, "plan_wait: plan_copy too small");
  plan_copy->n_moves = c->plan.n_moves;
  plan_copy->n_groups = c->plan.n_groups;
  if (c->plan.n_moves) memcpy(plan_copy->moves, c->plan.moves, sizeof(feplb_move) * c->plan.n_moves);
  if (c->plan.n_groups) memcpy(plan_copy->groups, c->plan.groups, sizeof(feplb_group) * c->plan.n_groups);
  memcpy(plan_copy->load_before, c->plan.load_before, sizeof(int64_t) * c->cfg.R);
  memcpy(plan_copy->load_after, c->plan.load_after, sizeof(int64_t) * c->cfg.R);
  return FEPLB_OK;
}

// Waits for the planner's job and returns the context to idle; copies the plan out.
static int join_planner(feplb_ctx* c, int32_t timeout_ms, feplb_plan_out* plan_copy) {
  int rc;
  {
    std::unique_lock<std::mutex> lk(c->mu);
    if (c->job == JOB_IDLE) return fail(c, FEPLB_E_STATE, "plan_wait: no plan was requested");
    if (!c->cv.wait_for(lk, std::chrono::milliseconds(timeout_ms < 0 ? 0 : timeout_ms), [&] { return c->job == JOB_DONE; }))
      return fail(c, FEPLB_E_TIMEOUT, "plan_wait: planner did not finish within %d ms", timeout_ms);
    rc = c->job_rc;
    c->job = JOB_IDLE;
  }
  if (rc != FEPLB_OK) return fail(c, rc, "planner failed: %s", feplb_strerror(rc));
  if ((rc = copy_plan(c, plan_copy)) != FEPLB_OK) return rc;
  if (c->n_dyn_groups > 0 && !c->job_wm) ++c->launches;     // the planner thread's table upload kernel
  return FEPLB_OK;
}

extern "C" int feplb_plan_wait(feplb_ctx* c, int32_t timeout_ms, feplb_plan_out* plan_copy,
                               const feplb_group** dyn_groups_dev, int32_t* n_dyn_groups, void* stream) {
  if (!c) return FEPLB_E_INVALID;
  int rc = join_planner(c, timeout_ms, plan_copy);
  if (rc != FEPLB_OK) return rc;
  if (dyn_groups_dev) *dyn_groups_dev = c->d_dyn_groups;
  if (n_dyn_groups) *n_dyn_groups = c->n_dyn_groups;
  CUDA_TRY(c, cudaStreamWaitEvent((cudaStream_t)stream, c->ev_plan, 0));
  return FEPLB_OK;
}

// Reads the stage events of ring slot r (waiting for them if needed) and adds them to the totals.
static int harvest_slot(feplb_ctx* c, int r) {
  if (!c->ev_used[r]) return FEPLB_OK;
  cudaEvent_t* ev = c->evr[r];
  CUDA_TRY(c, cudaEventSynchronize(ev[EV_COMBINE]));
  if (c->ev_host[r].ffn_launches == 2) CUDA_TRY(c, cudaEventSynchronize(ev[EV_STAMPS]));
  float ms = 0;
  auto el = [&](cudaEvent_t a, cudaEvent_t b) { return cudaEventElapsedTime(&ms, a, b) == cudaSuccess ? ms * 1e3 : 0.0; };
  feplb_timeline t = c->ev_host[r];
  t.dev_hist_us = el(ev[EV_T0], ev[EV_HIST]);
  t.dev_dispatch_us = el(ev[EV_HIST], ev[EV_DISPATCH]);
  const bool merged = t.ffn_launches == 2;
  t.dev_static_ffn_us = el(ev[EV_STATIC0], ev[EV_STATIC1]);
  t.dev_dynamic_ffn_us = merged ? 0.0 : el(ev[EV_DYN0], ev[EV_DYN1]);
  t.dev_combine_us = el(ev[merged ? EV_STATIC1 : EV_DYN1], ev[EV_COMBINE]);
  t.dev_counts_to_static_start_us = el(ev[EV_COUNTS], ev[EV_STATIC0]);
  t.dev_counts_to_static_end_us = el(ev[EV_COUNTS], ev[EV_STATIC1]);
  t.dev_total_us = el(ev[EV_T0], ev[EV_COMBINE]);
  t.dev_counts_to_copies_done_us = t.phase2_copy_bytes > 0 ? el(ev[EV_COUNTS], ev[EV_COPIES]) : 0.0;
  if (t.ffn_launches == 2) {
    // weights-on-M form: marks taken inside the kernels (all ones = never written)
    const unsigned long long* sp = c->h_stamps + (size_t)r * kStampWords;
    const unsigned long long none = ~0ull;
    auto span = [&](unsigned long long a, unsigned long long b) { return a != none && b != none && b >= a ? (b - a) * 1e-3 : 0.0; };
    const unsigned long long t_counts = sp[8], p1_start = sp[0], p1_first_dyn = sp[1], p1_end = sp[2] == none ? none : ~sp[2];
    const unsigned long long p2_start = sp[4], p2_end = sp[6] == none ? none : ~sp[6];
    t.dev_ffn_pass1_us = span(p1_start, p1_end);
    t.dev_ffn_pass2_us = span(p2_start, p2_end);
    t.dev_counts_to_static_start_us = span(t_counts, p1_start);
    // table there before the launch: static and dynamic groups side by side, no static part of its own;
    // no CTA ran out of static work otherwise: every group counts as static (the order that does not need the plan)
    t.dev_counts_to_static_end_us = span(t_counts, sp[9] != none ? p1_start : p1_first_dyn != none ? p1_first_dyn : p1_end);
    const unsigned long long w1 = sp[3] == none ? 0 : ~sp[3], w2 = sp[7] == none ? 0 : ~sp[7];
    t.dev_plan_wait_us = (w1 > w2 ? w1 : w2) * 1e-3;
  }
  cudaGetLastError();
  const double* src = reinterpret_cast<const double*>(&t);
  double* dst = reinterpret_cast<double*>(&c->tl_sum);
  for (size_t i = 0; i < sizeof(feplb_timeline) / sizeof(double); ++i) dst[i] += src[i];
  c->tl_last = t;
  c->tl_n += 1;
  c->ev_used[r] = false;
  return FEPLB_OK;
}

extern "C" int feplb_set_timeline(feplb_ctx* c, int32_t enable) {
  if (!c) return FEPLB_E_INVALID;
  c->timeline_on = enable != 0;
  return FEPLB_OK;
}

#define TL_EVENT(i)                                                  \
  do {                                                               \
    if (c->timeline_on) CUDA_TRY(c, cudaEventRecord(c->ev[i], st));  \
  } while (0)

extern "C" int feplb_moe_forward(feplb_ctx* c, const void* x, const int32_t* topk_ids, const float* gates,
                                 const void* w1, const void* w3, const void* w2, const uint8_t* dyn_mask_host,
                                 int32_t* counts, int32_t* rank_load, void* x_perm, void* h_scratch, void* y_perm,
                                 int32_t* slot_to_row, int32_t* row_to_token, void* out,
                                 feplb_plan_out* plan_copy, void* stream) {
  if (!c) return FEPLB_E_INVALID;
  cudaStream_t st = (cudaStream_t)stream;
  const feplb_config& g = c->cfg;
  if (!dyn_mask_host && g.mask_policy != FEPLB_MASK_REACTIVE)
    return fail(c, FEPLB_E_INVALID, "moe_forward: dyn_mask_host is required unless mask_policy is REACTIVE");
  int rc;
  if (c->timeline_on) {
    c->ev_slot = (c->ev_slot + 1) % kEvRing;
    if ((rc = harvest_slot(c, c->ev_slot)) != FEPLB_OK) return rc;   // long finished unless the ring wrapped quickly
    c->ev = c->evr[c->ev_slot];
  }
  c->t0 = clk::now();
  c->timeline_valid = true;
  c->tl.phase2_copy_bytes = 0;
  c->tl.dev_counts_to_copies_done_us = 0;
  // Weights-on-M form: one launch per pass runs the static groups and then the dynamic ones, whose
  // table it picks up on the device, so everything is enqueued before the planner is joined.
  // Not with Phase-2 weight copies: the dynamic groups would then wait, inside a kernel that holds
  // every SM, for device-to-device copies that the driver may carry out with kernels of its own;
  // that case keeps the four-launch order (the dynamic launches follow the copies in stream order).
  // (the test aids of feplb_set_planner_timing are about the table a launch waits for: they keep that order)
  const bool direct = c->direct && !g.phase2_copy && !c->planner_delay_us && !c->device_wait_limit_us;
  const bool wm = direct || (c->merged && !g.phase2_copy);
  c->tl.ffn_launches = wm ? 2 : 4;
  c->tl.dev_ffn_pass1_us = c->tl.dev_ffn_pass2_us = c->tl.dev_plan_wait_us = 0;
  unsigned long long* stamps = nullptr;
  if (wm && c->timeline_on) {
    stamps = c->d_stamps + (size_t)c->ev_slot * kStampWords;
    CUDA_TRY(c, cudaMemsetAsync(stamps, 0xFF, sizeof(unsigned long long) * kStampWords, st));
  }
  TL_EVENT(EV_T0);
  // step 1: counts, rank loads, segment offsets and the home group table in two launches; the
  // planner thread starts as soon as the counts reach the host
  if (!counts || !rank_load || !row_to_token) return fail(c, FEPLB_E_INVALID, "moe_forward: null pointer");
  if (g.T > 0) {
    if ((rc = check_dev_ptrs(c, {x, x_perm})) != FEPLB_OK) return rc;
    if (!topk_ids || !slot_to_row) return fail(c, FEPLB_E_INVALID, "moe_forward: null pointer");
  }
  const int64_t S = (int64_t)g.T * g.K;
  const uint8_t* mask_dev = nullptr;
  if (dyn_mask_host) {
    memcpy(c->h_mask, dyn_mask_host, g.E);
    CUDA_TRY(c, cudaMemcpyAsync(c->d_mask, c->h_mask, g.E, cudaMemcpyHostToDevice, st));
    mask_dev = c->d_mask;
  }
  if (direct) {
    std::lock_guard<std::mutex> lk(c->mu);
    if (c->job != JOB_IDLE) return fail(c, FEPLB_E_STATE, "moe_forward: a plan is already pending");
  }
  c->flag_seq = c->flag_seq == INT32_MAX ? 1 : c->flag_seq + 1;
  const int32_t seq = c->flag_seq;
  const bool small_front = feplb_front_is_small(S, g.E);
  c->path = (small_front ? FEPLB_PATH_SMALL_FRONT : 0) | (direct ? FEPLB_PATH_HOME_TABLE : wm ? FEPLB_PATH_MERGED : 0);
  c->detail = 0;
  c->job_w1 = w1; c->job_w3 = w3; c->job_w2 = w2;   // read by the planner thread after it is woken
  c->job_x_perm = x_perm;
  // Where the gather looks for the planner's table the thread is woken before the launches whose counts it waits for: a
  // forward on an idle GPU has its counts about 10 us after them, as long as a sleeping thread takes to wake.  Elsewhere
  // the launches go first.
  const bool kick_first = wm && !direct && !small_front;
  if (kick_first && (rc = plan_kick_flag(c, dyn_mask_host, seq, wm)) != FEPLB_OK) return rc;
  const cudaError_t front =
      small_front ? feplb_launch_front_small(x, topk_ids, g.T, g.K, g.E, g.R, g.d, g.row_align, g.dyn, mask_dev, nullptr, counts,
                                             rank_load, c->d_pad_off, c->d_home_groups, slot_to_row, row_to_token, x_perm,
                                             (int64_t)c->s_cap, c->d_status, c->h_counts_tagged, seq, stamps ? stamps + 8 : nullptr,
                                             c->num_sms, st, &c->launches)
                  : feplb_launch_route_fused(topk_ids, S, g.E, g.R, g.row_align, g.dyn, mask_dev, c->d_block_hist, counts,
                                             rank_load, c->d_pad_off, c->d_home_groups, nullptr, slot_to_row, row_to_token,
                                             (int64_t)c->s_cap, c->d_status, c->h_counts_tagged, seq,
                                             stamps ? stamps + 8 : nullptr, st, &c->launches);
  if (front != cudaSuccess) {
    if (kick_first) {
      c->job_abort.store(true, std::memory_order_relaxed);
      join_planner(c, c->planner_timeout_ms + 500, nullptr);
      c->job_abort.store(false, std::memory_order_relaxed);      // the next forward may wait for its counts by itself
    }
    return fail(c, FEPLB_E_CUDA, "routing launch: %s", cudaGetErrorString(front));
  }
  if (!direct && !kick_first && (rc = plan_kick_flag(c, dyn_mask_host, seq, wm)) != FEPLB_OK) return rc;
  TL_EVENT(EV_COUNTS);
  TL_EVENT(EV_HIST);
  // how the merged launches, and the gather in front of them, get the planner's table
  feplb_wm_dyn dyn;
  dyn.table_dev = c->d_dyn_tab32; dyn.table_host = c->h_dyn_tab32_dev;
  dyn.ready_dev = c->d_dyn_ready; dyn.ready_host = c->h_dyn_ready_dev;
  dyn.claim = reinterpret_cast<uint32_t*>(c->d_dyn_ready + 1); dyn.early = c->d_dyn_ready + 2;
  dyn.gather_done = reinterpret_cast<uint32_t*>(c->d_dyn_ready + 3);
  dyn.seq = direct || !wm ? 0u : (uint32_t)seq; dyn.max_groups = direct ? 0 : c->plan.cap_groups; dyn.stamps = stamps;
  dyn.wait_limit_ns = 1000ull * (unsigned long long)c->device_wait_limit_us;
  // step 3: permutation (does not depend on the plan: a migration relabels rows, it does not move
  // them here).  From here on a failure must still join the planner, so errors are carried in rc.
  {
    cudaError_t e = cudaSuccess;
    if (!small_front)
      e = feplb_launch_gather(x, topk_ids, c->d_block_hist, slot_to_row, counts, c->d_pad_off, x_perm, g.T, g.K, g.E, g.d,
                              g.row_align, (int64_t)c->s_cap, c->num_sms, st, &c->launches, row_to_token, true, 0, &dyn, c->d_status);
    if (e == cudaSuccess && g.phase2_copy) {
      // the planner's row copies of Phase 2 wait for the permuted rows
      e = cudaEventRecord(c->ev_gather, st);
      c->gather_seq.store(seq, std::memory_order_release);
    }
    if (e != cudaSuccess) rc = fail(c, FEPLB_E_CUDA, "dispatch launch: %s", cudaGetErrorString(e));
  }
  TL_EVENT(EV_DISPATCH);
  TL_EVENT(EV_STATIC0);
  if (wm) {
    // steps 4 + 5 in two launches: static groups from the table built on the device, then the dynamic
    // groups as soon as the planner has published them (bounded wait inside the kernel)
    if (rc == FEPLB_OK)
      rc = ffn_impl(c, x_perm, w1, w3, w2, c->d_home_groups, g.E, direct ? FEPLB_FFN_ALL : FEPLB_FFN_STATIC, h_scratch, y_perm, st,
                    c->gemm_pair_forced >= 0 ? c->gemm_pair_forced : (int)c->merged_pair, &dyn);
    TL_EVENT(EV_STATIC1);          // both launches lie between EV_STATIC0 and here; no events of their own for the dynamic part
    c->tl.host_enqueue_static_done_us = us_since(c->t0);
    int rc_comb = rc == FEPLB_OK ? feplb_combine(c, y_perm, slot_to_row, gates, out, stream) : FEPLB_OK;
    if (c->timeline_on && rc == FEPLB_OK && rc_comb == FEPLB_OK) {
      cudaError_t e = cudaEventRecord(c->ev[EV_COMBINE], st);
      if (e == cudaSuccess && stamps)      // the kernels' own marks follow the last stage event to the host
        e = cudaMemcpyAsync(c->h_stamps + (size_t)c->ev_slot * kStampWords, stamps, sizeof(unsigned long long) * kStampWords,
                            cudaMemcpyDeviceToHost, st);
      if (e == cudaSuccess) e = cudaEventRecord(c->ev[EV_STAMPS], st);
      if (e != cudaSuccess) rc_comb = fail(c, FEPLB_E_CUDA, "timeline records: %s", cudaGetErrorString(e));
    }
    // Everything is enqueued.  Join the planner (always, so that the context returns to idle); where no launch needs
    // the plan it is made right here, which spares waking the planner thread and being woken by it.
    int rc_join;
    if (direct) {
      rc_join = await_counts(c, seq);
      if (rc_join == FEPLB_OK) rc_join = make_plan(c, dyn_mask_host);
      if (rc_join != FEPLB_OK) rc_join = fail(c, rc_join, "planner failed: %s", feplb_strerror(rc_join));
      else rc_join = copy_plan(c, plan_copy);
      c->tl.host_upload_enqueued_us = us_since(c->t0);
    } else {
      rc_join = join_planner(c, c->planner_timeout_ms + 500, plan_copy);
    }
    c->tl.host_join_us = us_since(c->t0);
    if (rc != FEPLB_OK) return rc;
    if (rc_comb != FEPLB_OK) return rc_comb;
    if (rc_join != FEPLB_OK) return rc_join;
  } else {
    // step 4: static experts on their home ranks, from the group table built on the device
    if (rc == FEPLB_OK)
      rc = ffn_impl(c, x_perm, w1, w3, w2, c->d_home_groups, g.E, FEPLB_FFN_STATIC, h_scratch, y_perm, st, -1, nullptr, c->wm_static);
    TL_EVENT(EV_STATIC1);
    c->tl.host_enqueue_static_done_us = us_since(c->t0);
    // join the planner (always, so that the context returns to idle), then step 5
    const feplb_group* dyn_groups = nullptr;
    int32_t n_dyn = 0;
    int rc_join = feplb_plan_wait(c, c->planner_timeout_ms + 500, plan_copy, &dyn_groups, &n_dyn, stream);
    c->tl.host_join_us = us_since(c->t0);
    if (rc != FEPLB_OK) return rc;
    if (rc_join != FEPLB_OK) return rc_join;
    TL_EVENT(EV_DYN0);
    if ((rc = ffn_impl(c, x_perm, w1, w3, w2, dyn_groups, n_dyn, FEPLB_FFN_ALL, h_scratch, y_perm, st, c->dyn_pair)) != FEPLB_OK) return rc;
    TL_EVENT(EV_DYN1);
    // step 6
    if ((rc = feplb_combine(c, y_perm, slot_to_row, gates, out, stream)) != FEPLB_OK) return rc;
    TL_EVENT(EV_COMBINE);
  }
  c->tl.host_return_us = us_since(c->t0);
  if (c->timeline_on) {
    c->ev_host[c->ev_slot] = c->tl;
    c->ev_used[c->ev_slot] = true;
  }
  return FEPLB_OK;
}

// Token ranges of a host-buffer forward.  Copying a batch in, computing and copying the result out one after the other
// leaves each of the three idle two thirds of the time.  In ranges they overlap, but every range streams the experts'
// weights again: with per-direction copy time c, weight time w and the rest of the compute time v, n equal
// ranges take about c/n + (w + v/n) + c/n + (n - 1) * (longest of the three).  n is the smallest that is within 2 % of
// the best and gains at least 5 %.  Rates: 55 GB/s per direction of PCIe, 6.5 TB/s of HBM, 1.1 PFLOP/s, all measured
// on this layer; 30 us of launches and ramps per range.  Measured, whole batch -> ranges (64 experts, d = 2048, f = 768,
// top-6): T = 4096 937 -> 704 us (two), T = 8192 1748 -> 1139, T = 2048 544 -> 462; below that one range.
static int host_ranges(const feplb_ctx* c, int* first_token) {
  const feplb_config& g = c->cfg;
  const double S = (double)g.T * g.K, df = (double)g.d * g.f;
  const double copy = 2.0 * g.T * g.d / 55e3, weights = 30.0 + 6.0 * df * g.E / 6.5e6, rest = 6.0 * S * df / 1.1e9 + 8.0 * S * g.d / 6.5e6;
  const int step = FEPLB_SLOTS_PER_BLOCK / std::gcd(FEPLB_SLOTS_PER_BLOCK, (int)g.K);   // tokens whose slots are whole CTAs of 1024
  double cost[FEPLB_MAX_RANGES + 1], best = 1e30;
  for (int n = 1; n <= FEPLB_MAX_RANGES; ++n) {
    const double a = copy / n, b = weights + rest / n;
    cost[n] = n > 1 && g.T / n < step ? 1e30 : 2 * a + b + (n - 1) * (a > b ? a : b);
    if (cost[n] < best) best = cost[n];
  }
  int n = 1;
  if (best < 0.95 * cost[1])
    while (cost[n] > 1.02 * best) ++n;
  // to the nearest boundary: a range that is a step longer than the others holds them all up (T = 6000, top-3, three ranges at
  // 1024 and 3072 972 us, at 2048 and 4096 806)
  for (int i = 0; i <= n; ++i) first_token[i] = i == n ? g.T : (int)(((int64_t)g.T * i + (int64_t)n * step / 2) / ((int64_t)n * step) * step);
  return n;
}

// One range after the other on `st`, input copies on the context's input stream, result copies on its output stream.
// All launches are enqueued before the plan is made (by the calling thread, as for small batches): they walk the
// home groups of their range.  Rows, indices and sums are those of the whole-batch path.
static int host_forward_ranges(feplb_ctx* c, int n, const int* first, const void* x_host, const int32_t* topk_ids_host,
                               const float* gates_host, void* x_dev, int32_t* ids_dev, float* gates_dev, const void* w1,
                               const void* w3, const void* w2, const uint8_t* dyn_mask_host, int32_t* counts, int32_t* rank_load,
                               void* x_perm, void* h_scratch, void* y_perm, int32_t* slot_to_row, int32_t* row_to_token,
                               void* out_dev, void* out_host, feplb_plan_out* plan_copy, cudaStream_t st) {
  const feplb_config& g = c->cfg;
  const int64_t S = (int64_t)g.T * g.K;
  const size_t row = (size_t)g.d * 2, nk = (size_t)S * 4;
  int rc = check_dev_ptrs(c, {x_dev, x_perm, w1, w3, w2, h_scratch, y_perm, out_dev});
  if (rc != FEPLB_OK) return rc;
  if (!counts || !rank_load || !row_to_token || !slot_to_row) return fail(c, FEPLB_E_INVALID, "moe_forward_host: null pointer");
  {
    std::lock_guard<std::mutex> lk(c->mu);
    if (c->job != JOB_IDLE) return fail(c, FEPLB_E_STATE, "moe_forward: a plan is already pending");
  }
  c->t0 = clk::now();
  c->timeline_valid = true;
  memset(&c->tl, 0, sizeof(c->tl));
  c->tl.ffn_launches = 2 * n;
  c->path = FEPLB_PATH_RANGES;
  c->detail = 0;
  // inputs: after whatever `st` still does with the staging buffers
  CUDA_TRY(c, cudaEventRecord(c->ev_range_ids, st));
  CUDA_TRY(c, cudaStreamWaitEvent(c->in_stream, c->ev_range_ids, 0));
  CUDA_TRY(c, cudaMemcpyAsync(ids_dev, topk_ids_host, nk, cudaMemcpyHostToDevice, c->in_stream));
  CUDA_TRY(c, cudaEventRecord(c->ev_range_ids, c->in_stream));
  CUDA_TRY(c, cudaStreamWaitEvent(st, c->ev_range_ids, 0));
  for (int i = 0; i < n; ++i) {
    const size_t o = row * first[i];
    CUDA_TRY(c, cudaMemcpyAsync((char*)x_dev + o, (const char*)x_host + o, row * (first[i + 1] - first[i]), cudaMemcpyHostToDevice, c->in_stream));
    CUDA_TRY(c, cudaEventRecord(c->ev_range_in[i], c->in_stream));
    if (i > 0) continue;
    // not needed before the first combine
    CUDA_TRY(c, cudaMemcpyAsync(gates_dev, gates_host, nk, cudaMemcpyHostToDevice, c->in_stream));
    CUDA_TRY(c, cudaEventRecord(c->ev_range_ids, c->in_stream));
  }
  // routing of the whole batch
  const uint8_t* mask_dev = nullptr;
  if (dyn_mask_host) {
    memcpy(c->h_mask, dyn_mask_host, g.E);
    CUDA_TRY(c, cudaMemcpyAsync(c->d_mask, c->h_mask, g.E, cudaMemcpyHostToDevice, st));
    mask_dev = c->d_mask;
  }
  c->flag_seq = c->flag_seq == INT32_MAX ? 1 : c->flag_seq + 1;
  CUDA_TRY(c, feplb_launch_route_fused(ids_dev, S, g.E, g.R, g.row_align, g.dyn, mask_dev, c->d_block_hist,
                                       counts, rank_load, c->d_pad_off, c->d_home_groups, nullptr, slot_to_row, row_to_token,
                                       (int64_t)c->s_cap, c->d_status, c->h_counts_tagged, c->flag_seq, nullptr, st, &c->launches));
  CUDA_TRY(c, feplb_launch_range_groups(c->d_block_hist, S, g.K, g.E, c->d_home_groups, first, n, c->d_range_groups, st, &c->launches));
  for (int i = 0; i < n; ++i) {
    const int t0 = first[i], T = first[i + 1] - first[i];
    CUDA_TRY(c, cudaStreamWaitEvent(st, c->ev_range_in[i], 0));
    CUDA_TRY(c, feplb_launch_gather(x_dev, ids_dev, c->d_block_hist, slot_to_row, counts, c->d_pad_off, x_perm, T, g.K, g.E, g.d,
                                    i == 0 ? g.row_align : 1, (int64_t)c->s_cap, c->num_sms, st, &c->launches, row_to_token, true, t0));
    const int pair = c->gemm_pair_forced >= 0 ? c->gemm_pair_forced : (int64_t)T * g.K >= (int64_t)256 * g.E;
    if ((rc = ffn_impl(c, x_perm, w1, w3, w2, c->d_range_groups + (size_t)i * g.E, g.E, FEPLB_FFN_ALL, h_scratch, y_perm, st, pair)) != FEPLB_OK)
      return rc;
    if (i == 0) CUDA_TRY(c, cudaStreamWaitEvent(st, c->ev_range_ids, 0));
    CUDA_TRY(c, feplb_launch_combine(y_perm, slot_to_row + (size_t)t0 * g.K, gates_dev + (size_t)t0 * g.K, (char*)out_dev + row * t0, T,
                                     g.K, g.d, c->num_sms, st, &c->launches));
    CUDA_TRY(c, cudaEventRecord(c->ev_range_out[i], st));
  }
  c->tl.host_enqueue_static_done_us = us_since(c->t0);
  for (int i = 0; i < n; ++i) {
    const size_t o = row * first[i];
    CUDA_TRY(c, cudaStreamWaitEvent(c->out_stream, c->ev_range_out[i], 0));
    CUDA_TRY(c, cudaMemcpyAsync((char*)out_host + o, (const char*)out_dev + o, row * (first[i + 1] - first[i]), cudaMemcpyDeviceToHost, c->out_stream));
  }
  rc = await_counts(c, c->flag_seq);
  if (rc == FEPLB_OK) rc = make_plan(c, dyn_mask_host);
  if (rc != FEPLB_OK) return fail(c, rc, "planner failed: %s", feplb_strerror(rc));
  rc = copy_plan(c, plan_copy);
  c->tl.host_upload_enqueued_us = c->tl.host_join_us = c->tl.host_return_us = us_since(c->t0);
  return rc;
}

extern "C" int feplb_moe_forward_host(feplb_ctx* c, const void* x_host, const int32_t* topk_ids_host,
                                      const float* gates_host, void* x_dev, int32_t* ids_dev, float* gates_dev,
                                      const void* w1, const void* w3, const void* w2, const uint8_t* dyn_mask_host,
                                      int32_t* counts, int32_t* rank_load, void* x_perm, void* h_scratch, void* y_perm,
                                      int32_t* slot_to_row, int32_t* row_to_token, void* out_dev, void* out_host,
                                      feplb_plan_out* plan_copy, void* stream) {
  if (!c) return FEPLB_E_INVALID;
  cudaStream_t st = (cudaStream_t)stream;
  const feplb_config& g = c->cfg;
  const size_t nx = (size_t)g.T * g.d * 2, nk = (size_t)g.T * g.K * 4;
  if (g.T > 0) {
    if (!x_host || !topk_ids_host || !gates_host || !out_host || !x_dev || !ids_dev || !gates_dev || !out_dev)
      return fail(c, FEPLB_E_INVALID, "moe_forward_host: null pointer");
    int first[FEPLB_MAX_RANGES + 1];
    const int n = host_ranges(c, first);
    const bool whole = g.phase2_copy || c->timeline_on || c->order_forced || c->planner_delay_us || c->device_wait_limit_us ||
                       (!dyn_mask_host && g.mask_policy != FEPLB_MASK_REACTIVE);
    if (n > 1 && !whole) {
      const int rc = host_forward_ranges(c, n, first, x_host, topk_ids_host, gates_host, x_dev, ids_dev, gates_dev, w1, w3, w2,
                                         dyn_mask_host, counts, rank_load, x_perm, h_scratch, y_perm, slot_to_row, row_to_token,
                                         out_dev, out_host, plan_copy, st);
      // everything drains before the call returns, also after a failure
      const cudaError_t e[3] = {cudaStreamSynchronize(c->in_stream), cudaStreamSynchronize(st), cudaStreamSynchronize(c->out_stream)};
      if (rc != FEPLB_OK) return rc;
      for (cudaError_t x : e) CUDA_TRY(c, x);
      return FEPLB_OK;
    }
    CUDA_TRY(c, cudaMemcpyAsync(ids_dev, topk_ids_host, nk, cudaMemcpyHostToDevice, st));
    CUDA_TRY(c, cudaMemcpyAsync(gates_dev, gates_host, nk, cudaMemcpyHostToDevice, st));
    CUDA_TRY(c, cudaMemcpyAsync(x_dev, x_host, nx, cudaMemcpyHostToDevice, st));
  }
  int rc = feplb_moe_forward(c, x_dev, ids_dev, gates_dev, w1, w3, w2, dyn_mask_host, counts, rank_load, x_perm,
                             h_scratch, y_perm, slot_to_row, row_to_token, out_dev, plan_copy, stream);
  if (rc != FEPLB_OK) return rc;
  if (g.T > 0) CUDA_TRY(c, cudaMemcpyAsync(out_host, out_dev, nx, cudaMemcpyDeviceToHost, st));
  CUDA_TRY(c, cudaStreamSynchronize(st));
  return FEPLB_OK;
}

extern "C" int feplb_host_stage_inputs(feplb_ctx* c, int32_t slot, const void* x_host, const int32_t* topk_ids_host,
                                       const float* gates_host, void* x_dev, int32_t* ids_dev, float* gates_dev) {
  if (!c) return FEPLB_E_INVALID;
  if (slot < 0 || slot >= FEPLB_HOST_SLOTS) return fail(c, FEPLB_E_INVALID, "host_stage_inputs: slot out of range");
  if (c->slot_staged[slot]) return fail(c, FEPLB_E_STATE, "host_stage_inputs: slot %d already holds staged inputs", slot);
  const feplb_config& g = c->cfg;
  const size_t nx = (size_t)g.T * g.d * 2, nk = (size_t)g.T * g.K * 4;
  if (g.T > 0 && (!x_host || !topk_ids_host || !gates_host || !x_dev || !ids_dev || !gates_dev))
    return fail(c, FEPLB_E_INVALID, "host_stage_inputs: null pointer");
  // the slot's device staging was last read by the forward that used this slot before
  if (c->slot_used[slot]) CUDA_TRY(c, cudaStreamWaitEvent(c->in_stream, c->ev_done[slot], 0));
  if (g.T > 0) {
    CUDA_TRY(c, cudaMemcpyAsync(ids_dev, topk_ids_host, nk, cudaMemcpyHostToDevice, c->in_stream));
    CUDA_TRY(c, cudaMemcpyAsync(gates_dev, gates_host, nk, cudaMemcpyHostToDevice, c->in_stream));
    CUDA_TRY(c, cudaMemcpyAsync(x_dev, x_host, nx, cudaMemcpyHostToDevice, c->in_stream));
  }
  CUDA_TRY(c, cudaEventRecord(c->ev_in[slot], c->in_stream));
  c->slot_staged[slot] = true;
  return FEPLB_OK;
}

extern "C" int feplb_moe_forward_host_async(feplb_ctx* c, int32_t slot, const void* x_host, const int32_t* topk_ids_host,
                                            const float* gates_host, void* x_dev, int32_t* ids_dev, float* gates_dev,
                                            const void* w1, const void* w3, const void* w2, const uint8_t* dyn_mask_host,
                                            int32_t* counts, int32_t* rank_load, void* x_perm, void* h_scratch,
                                            void* y_perm, int32_t* slot_to_row, int32_t* row_to_token, void* out_dev,
                                            void* out_host, feplb_plan_out* plan_copy, void* stream) {
  if (!c) return FEPLB_E_INVALID;
  if (slot < 0 || slot >= FEPLB_HOST_SLOTS) return fail(c, FEPLB_E_INVALID, "moe_forward_host_async: slot out of range");
  cudaStream_t st = (cudaStream_t)stream;
  const feplb_config& g = c->cfg;
  const size_t nx = (size_t)g.T * g.d * 2;
  if (g.T > 0 && (!out_host || !x_dev || !ids_dev || !gates_dev || !out_dev))
    return fail(c, FEPLB_E_INVALID, "moe_forward_host_async: null pointer");
  if (c->slot_staged[slot]) {
    c->slot_staged[slot] = false;        // inputs were started by feplb_host_stage_inputs; ev_in[slot] marks their end
  } else {
    int rc = feplb_host_stage_inputs(c, slot, x_host, topk_ids_host, gates_host, x_dev, ids_dev, gates_dev);
    if (rc != FEPLB_OK) return rc;
    c->slot_staged[slot] = false;
  }
  // compute: after its inputs have arrived and the slot's previous result has left out_dev
  CUDA_TRY(c, cudaStreamWaitEvent(st, c->ev_in[slot], 0));
  if (c->slot_used[slot]) CUDA_TRY(c, cudaStreamWaitEvent(st, c->ev_out[slot], 0));
  int rc = feplb_moe_forward(c, x_dev, ids_dev, gates_dev, w1, w3, w2, dyn_mask_host, counts, rank_load, x_perm,
                             h_scratch, y_perm, slot_to_row, row_to_token, out_dev, plan_copy, stream);
  if (rc != FEPLB_OK) return rc;
  CUDA_TRY(c, cudaEventRecord(c->ev_done[slot], st));
  // output
  CUDA_TRY(c, cudaStreamWaitEvent(c->out_stream, c->ev_done[slot], 0));
  if (g.T > 0) CUDA_TRY(c, cudaMemcpyAsync(out_host, out_dev, nx, cudaMemcpyDeviceToHost, c->out_stream));
  CUDA_TRY(c, cudaEventRecord(c->ev_out[slot], c->out_stream));
  c->slot_used[slot] = true;
  return FEPLB_OK;
}

extern "C" int feplb_host_wait(feplb_ctx* c, int32_t slot) {
  if (!c) return FEPLB_E_INVALID;
  if (slot < 0 || slot >= FEPLB_HOST_SLOTS) return fail(c, FEPLB_E_INVALID, "host_wait: slot out of range");
  if (c->slot_used[slot]) CUDA_TRY(c, cudaEventSynchronize(c->ev_out[slot]));
  return FEPLB_OK;
}

extern "C" int feplb_get_timeline(feplb_ctx* c, feplb_timeline* out) {
  if (!c || !out) return FEPLB_E_INVALID;
  if (!c->timeline_valid) return fail(c, FEPLB_E_STATE, "get_timeline: no forward pass yet");
  if (c->timeline_on || c->tl_n) {
    for (int i = 1; i <= kEvRing; ++i) {   // oldest first, so that tl_last is the newest forward
      int rc = harvest_slot(c, (c->ev_slot + i) % kEvRing);
      if (rc != FEPLB_OK) return rc;
    }
    *out = c->tl_last;
  } else {
    *out = c->tl;   // host fields only
  }
  return FEPLB_OK;
}

extern "C" int feplb_timeline_totals(feplb_ctx* c, feplb_timeline* sum, int64_t* n_forwards, int32_t reset) {
  if (!c || !sum || !n_forwards) return FEPLB_E_INVALID;
  for (int i = 1; i <= kEvRing; ++i) {
    int rc = harvest_slot(c, (c->ev_slot + i) % kEvRing);
    if (rc != FEPLB_OK) return rc;
  }
  *sum = c->tl_sum;
  *n_forwards = c->tl_n;
  if (reset) {
    memset(&c->tl_sum, 0, sizeof(c->tl_sum));
    c->tl_n = 0;
  }
  return FEPLB_OK;
}

extern "C" int feplb_set_planner_timeout(feplb_ctx* c, int32_t timeout_ms) {
  if (!c || timeout_ms < 1) return FEPLB_E_INVALID;
  std::lock_guard<std::mutex> lk(c->mu);
  if (c->job != JOB_IDLE) return fail(c, FEPLB_E_STATE, "set_planner_timeout: a plan is pending");
  c->planner_timeout_ms = timeout_ms;
  return FEPLB_OK;
}

extern "C" int feplb_set_gemm_form(feplb_ctx* c, int32_t forward_form, int32_t backward_pair) {
  if (!c) return FEPLB_E_INVALID;
  if (forward_form < FEPLB_FORM_AUTO || forward_form > FEPLB_FORM_WEIGHT_M)
    return fail(c, FEPLB_E_INVALID, "set_gemm_form: forward_form must be FEPLB_FORM_AUTO, _SINGLE, _PAIR or _WEIGHT_M");
  if (forward_form == FEPLB_FORM_WEIGHT_M && !c->wm_ok)
    return fail(c, FEPLB_E_INVALID, "set_gemm_form: the weights-on-M form needs f %% 128 == 0, d %% 256 == 0 and "
                                    "2*E + R*max_num_dyn <= %d", FEPLB_WM_MAX_ENTRIES);
  if (backward_pair < -1 || backward_pair > 3)
    return fail(c, FEPLB_E_INVALID, "set_gemm_form: backward_pair must be -1 (auto) or a 2-bit mask");
  std::lock_guard<std::mutex> lk(c->mu);
  if (c->job != JOB_IDLE) return fail(c, FEPLB_E_STATE, "set_gemm_form: a plan is pending");
  c->wm_static = forward_form == FEPLB_FORM_AUTO && c->wm_static_auto;
  c->few = forward_form == FEPLB_FORM_AUTO ? c->few_auto : 0;
  c->wm = forward_form == FEPLB_FORM_AUTO ? c->wm_auto : forward_form == FEPLB_FORM_WEIGHT_M;
  c->wm_merged = forward_form == FEPLB_FORM_AUTO ? c->wm_merged_auto : c->wm;
  c->gemm_pair_forced = forward_form == FEPLB_FORM_SINGLE || forward_form == FEPLB_FORM_PAIR ? forward_form : -1;
  c->gemm_pair_default = c->gemm_pair_forced < 0 ? c->gemm_pair_auto : forward_form;
  c->bwd_pair = backward_pair < 0 ? c->bwd_pair_auto : backward_pair;
  return FEPLB_OK;
}

extern "C" int feplb_set_launch_merging(feplb_ctx* c, int32_t merged) {
  if (!c || merged < -1 || merged > 1) return FEPLB_E_INVALID;
  if (merged == 1 && !c->merged_ok)
    return fail(c, FEPLB_E_INVALID, "set_launch_merging: needs 2*E + R*max_num_dyn <= %d", FEPLB_MAX_GROUPS);
  std::lock_guard<std::mutex> lk(c->mu);
  if (c->job != JOB_IDLE) return fail(c, FEPLB_E_STATE, "set_launch_merging: a plan is pending");
  c->merged = merged < 0 ? c->merged_auto : merged != 0;
  c->direct = merged < 0 && c->direct_auto;
  c->order_forced = merged >= 0;
  return FEPLB_OK;
}

extern "C" int feplb_set_planner_timing(feplb_ctx* c, int32_t planner_delay_us, int32_t device_wait_limit_us) {
  if (!c || planner_delay_us < 0 || planner_delay_us > 1000000 || device_wait_limit_us < 0) return FEPLB_E_INVALID;
  std::lock_guard<std::mutex> lk(c->mu);
  if (c->job != JOB_IDLE) return fail(c, FEPLB_E_STATE, "set_planner_timing: a plan is pending");
  c->planner_delay_us = planner_delay_us;
  c->device_wait_limit_us = device_wait_limit_us;
  return FEPLB_OK;
}

extern "C" int feplb_pack_weights(feplb_ctx* c, const void* w1_in, const void* w3_in, const void* w2_in, void* w1, void* w3,
                                  void* w2, void* stream) {
  if (!c) return FEPLB_E_INVALID;
  int rc = check_dev_ptrs(c, {w1_in, w3_in, w2_in, w1, w3, w2});
  if (rc != FEPLB_OK) return rc;
  // [E,d,f] -> [E,f,d] and [E,f,d] -> [E,d,f]: the transposition of feplb_transpose_weights with d and f exchanged
  CUDA_TRY(c, feplb_launch_transpose_weights(w1_in, w3_in, w2_in, w1, w3, w2, c->cfg.E, c->cfg.f, c->cfg.d,
                                             (cudaStream_t)stream, &c->launches));
  return FEPLB_OK;
}

extern "C" int feplb_selftest_bounded_wait(feplb_ctx* c, int32_t limit_us, void* stream) {
  if (!c || limit_us < 1 || limit_us > 1000000) return FEPLB_E_INVALID;
  cudaStream_t st = (cudaStream_t)stream;
  int rc = feplb_check_status(c, stream);          // start from a clean status word
  if (rc != FEPLB_OK) return rc;
  int* d_flag = reinterpret_cast<int*>(c->d_pad_off);   // scratch word, rewritten by the next dispatch
  CUDA_TRY(c, cudaMemsetAsync(d_flag, 0xFF, sizeof(int), st));
  CUDA_TRY(c, feplb_launch_wait_selftest(c->d_status, 1000ull * limit_us, d_flag, st));
  ++c->launches;
  int gave_up = -1;
  CUDA_TRY(c, cudaMemcpyAsync(&gave_up, d_flag, sizeof(int), cudaMemcpyDeviceToHost, st));
  rc = feplb_check_status(c, stream);              // synchronises; expected: FEPLB_E_DEVICE from the wait
  if (rc == FEPLB_E_DEVICE && gave_up == 1) return FEPLB_OK;
  return fail(c, FEPLB_E_STATE, "bounded-wait self-test: status %d, gave_up %d", rc, gave_up);
}

extern "C" int feplb_route_topk(feplb_ctx* c, const float* logits, int32_t* topk_ids, float* gates, void* stream) {
  if (!c) return FEPLB_E_INVALID;
  if (c->cfg.K > c->cfg.E) return fail(c, FEPLB_E_INVALID, "route_topk: K > E");
  if (c->cfg.T > 0 && (!logits || !topk_ids || !gates)) return fail(c, FEPLB_E_INVALID, "route_topk: null pointer");
  CUDA_TRY(c, feplb_launch_route_topk(logits, c->cfg.T, c->cfg.E, c->cfg.K, topk_ids, gates, c->num_sms,
                                      (cudaStream_t)stream, &c->launches));
  return FEPLB_OK;
}

// ---- backward pass ---------------------------------------------------------------------------

extern "C" int feplb_set_preact_buffer(feplb_ctx* c, void* ab) {
  if (!c) return FEPLB_E_INVALID;
  if (ab && !aligned16(ab)) return fail(c, FEPLB_E_INVALID, "set_preact_buffer: unaligned pointer");
  c->d_preact = ab;
  return FEPLB_OK;
}

extern "C" int feplb_transpose_weights(feplb_ctx* c, const void* w1, const void* w3, const void* w2, void* w1t, void* w3t,
                                       void* w2t, void* stream) {
  if (!c) return FEPLB_E_INVALID;
  int rc = check_dev_ptrs(c, {w1, w3, w2, w1t, w3t, w2t});
  if (rc != FEPLB_OK) return rc;
  CUDA_TRY(c, feplb_launch_transpose_weights(w1, w3, w2, w1t, w3t, w2t, c->cfg.E, c->cfg.d, c->cfg.f, (cudaStream_t)stream,
                                             &c->launches));
  return FEPLB_OK;
}

static int combine_bwd_impl(feplb_ctx* c, const void* d_out, const void* y_perm, const int32_t* slot_to_row,
                            const float* gates, void* d_y_perm, float* d_gates, const feplb_bwd_pads* pads, void* stream) {
  if (!c) return FEPLB_E_INVALID;
  if (c->cfg.T == 0) return FEPLB_OK;
  int rc = check_dev_ptrs(c, {d_out, y_perm, d_y_perm});
  if (rc != FEPLB_OK) return rc;
  if (!slot_to_row || !gates || !d_gates) return fail(c, FEPLB_E_INVALID, "combine_bwd: null pointer");
  CUDA_TRY(c, feplb_launch_combine_bwd(d_out, y_perm, slot_to_row, gates, d_y_perm, d_gates, c->cfg.T, c->cfg.K, c->cfg.d,
                                       (cudaStream_t)stream, &c->launches, pads));
  return FEPLB_OK;
}

extern "C" int feplb_combine_bwd(feplb_ctx* c, const void* d_out, const void* y_perm, const int32_t* slot_to_row,
                                 const float* gates, void* d_y_perm, float* d_gates, void* stream) {
  return combine_bwd_impl(c, d_out, y_perm, slot_to_row, gates, d_y_perm, d_gates, nullptr, stream);
}

extern "C" int feplb_dispatch_bwd(feplb_ctx* c, const void* d_x_perm, const int32_t* slot_to_row, void* d_x, void* stream) {
  if (!c) return FEPLB_E_INVALID;
  if (c->cfg.T == 0) return FEPLB_OK;
  int rc = check_dev_ptrs(c, {d_x_perm, d_x});
  if (rc != FEPLB_OK) return rc;
  if (!slot_to_row) return fail(c, FEPLB_E_INVALID, "dispatch_bwd: null pointer");
  CUDA_TRY(c, feplb_launch_combine(d_x_perm, slot_to_row, nullptr, d_x, c->cfg.T, c->cfg.K, c->cfg.d, c->num_sms,
                                   (cudaStream_t)stream, &c->launches));
  return FEPLB_OK;
}

static int expert_ffn_bwd_impl(feplb_ctx* c, const void* x_perm, const void* ab_saved, void* h,
                               void* d_y_perm, const void* w1t, const void* w3t, const void* w2t,
                               const feplb_group* groups, int32_t n_groups, int32_t which,
                               const feplb_group* expert_table, void* d_ab,
                               void* d_x_perm, float* dw1, float* dw3, float* dw2, int32_t accumulate,
                               bool pads_zeroed, void* stream) {
  if (!c) return FEPLB_E_INVALID;
  if (n_groups < 0 || n_groups > FEPLB_MAX_GROUPS) return fail(c, FEPLB_E_INVALID, "expert_ffn_bwd: n_groups out of range");
  if (n_groups == 0 || c->s_cap == 0) return FEPLB_OK;
  int rc = check_dev_ptrs(c, {x_perm, ab_saved, h, d_y_perm, w1t, w3t, w2t, d_ab, d_x_perm});
  if (rc != FEPLB_OK) return rc;
  if (!groups) return fail(c, FEPLB_E_INVALID, "expert_ffn_bwd: null group table");
  const bool want_w = dw1 || dw3 || dw2;
  if (want_w) {
    if (!dw1 || !dw3 || !dw2 || !expert_table)
      return fail(c, FEPLB_E_INVALID, "expert_ffn_bwd: weight gradients need dw1, dw3, dw2 and expert_table");
    if (c->cfg.row_align != 128)
      return fail(c, FEPLB_E_INVALID, "expert_ffn_bwd: weight gradients need row_align = 128 (an expert's rows are the K range)");
  }
  feplb_bwd_args a;
  a.x_perm = x_perm; a.ab_saved = ab_saved; a.h = h; a.d_y_perm = d_y_perm;
  a.w1t = w1t; a.w3t = w3t; a.w2t = w2t;
  a.groups = groups; a.n_groups = n_groups; a.which = which;
  a.expert_table = expert_table;
  a.d_ab = d_ab; a.d_x_perm = d_x_perm;
  a.dw1 = want_w ? dw1 : nullptr; a.dw3 = dw3; a.dw2 = dw2; a.accumulate = accumulate != 0;
  a.E = c->cfg.E; a.d = c->cfg.d; a.f = c->cfg.f; a.s_cap = (int64_t)c->s_cap;
  a.status = c->d_status; a.num_sms = c->num_sms;
  a.pads_zeroed = pads_zeroed;
  a.pair_dgrad = c->bwd_pair & 1; a.pair_wgrad = (c->bwd_pair >> 1) & 1;
  return feplb_launch_expert_ffn_bwd(a, (cudaStream_t)stream, &c->launches, c->err, sizeof(c->err));
}

extern "C" int feplb_expert_ffn_bwd(feplb_ctx* c, const void* x_perm, const void* ab_saved, void* h,
                                    void* d_y_perm, const void* w1t, const void* w3t, const void* w2t,
                                    const feplb_group* groups, int32_t n_groups, int32_t which,
                                    const feplb_group* expert_table, void* d_ab,
                                    void* d_x_perm, float* dw1, float* dw3, float* dw2, int32_t accumulate,
                                    void* stream) {
  return expert_ffn_bwd_impl(c, x_perm, ab_saved, h, d_y_perm, w1t, w3t, w2t, groups, n_groups, which, expert_table, d_ab,
                             d_x_perm, dw1, dw3, dw2, accumulate, false, stream);
}

extern "C" int feplb_moe_backward(feplb_ctx* c, const void* d_out, const float* gates, const void* w1t, const void* w3t,
                                  const void* w2t, const void* x_perm, const void* ab_saved, void* h,
                                  const void* y_perm, const int32_t* slot_to_row,
                                  void* d_y_perm, void* d_ab, void* d_x_perm, void* d_x, float* d_gates,
                                  float* dw1, float* dw3, float* dw2, int32_t accumulate, void* stream) {
  if (!c) return FEPLB_E_INVALID;
  // weight gradients: the padding rows are zeroed by the first kernel; what is wrong with the arguments has to be
  // found before it writes to them
  const bool zero_pads = (dw1 || dw3 || dw2) && c->cfg.row_align == 128 && c->cfg.T > 0;
  int rc = FEPLB_OK;
  if (zero_pads && (rc = check_dev_ptrs(c, {h, d_ab})) != FEPLB_OK) return rc;
  const feplb_bwd_pads pads = {c->d_home_groups, c->cfg.E, c->cfg.f, h, d_ab};
  rc = combine_bwd_impl(c, d_out, y_perm, slot_to_row, gates, d_y_perm, d_gates, zero_pads ? &pads : nullptr, stream);
  if (rc != FEPLB_OK) return rc;
  // every expert's rows in one table: the home table of the forward pass that ran last on this context
  rc = expert_ffn_bwd_impl(c, x_perm, ab_saved, h, d_y_perm, w1t, w3t, w2t, c->d_home_groups, c->cfg.E, FEPLB_FFN_ALL,
                           c->d_home_groups, d_ab, d_x_perm, dw1, dw3, dw2, accumulate, zero_pads, stream);
  if (rc != FEPLB_OK) return rc;
  return feplb_dispatch_bwd(c, d_x_perm, slot_to_row, d_x, stream);
}
