// Integer side of the FEPLB hot path on sm_100a: routing histogram (paper Section 2.2: per-expert
// token counts known after Phase 1), the stable counting-sort permutation of (token, k) slots
// into expert-contiguous rows (Section 2.2, Phase 1: expert order for the grouped GEMM), the row
// gather, and the home (pre-plan) group table the static-expert GEMM runs on (Section 2.3).
//
// Ranks inside an expert's segment must not depend on the order in which atomics land, so
// ranking is done in three deterministic levels: a warp ranks its 32 slots with match_any and
// a lane mask, warps of a CTA are chained through per-warp histograms in shared memory, CTAs
// are chained through an exclusive scan of per-CTA histograms.  Atomics are used only for the
// per-expert totals (integer adds commute).  The first two levels run in the histogram kernel,
// which already holds the ids and match masks and leaves each slot's rank inside its CTA's 1024
// slots behind; the gather kernel adds the segment offset and the CTA's base from the scan, so no
// ranking kernel of its own sits between the counts and the row copies.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "feplb_dyn.cuh"
#include "feplb_internal.h"

namespace {

struct RangeBlocks { int first[FEPLB_MAX_RANGES + 1]; };   // first CTA-of-1024-slots of every token range, and the end

// Programmatic dependent launch: a kernel launched with the attribute below may be scheduled
// while the kernel before it in the stream drains; pdl_sync() holds it until that kernel's
// results are complete (a no-op for ordinary launches) and lets its own successor do the same.
__device__ __forceinline__ void pdl_sync() {
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename... KArgs, typename... Args>
cudaError_t launch(void (*kernel)(KArgs...), int grid, int block, size_t smem, cudaStream_t st, bool programmatic,
                   Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = programmatic ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kChunks = FEPLB_SLOTS_PER_BLOCK / kThreads;   // 32-slot chunks per warp (4)
static_assert(FEPLB_SLOTS_PER_BLOCK == kWarps * kChunks * 32, "slot tiling");

// Warp w of CTA b owns slots [b*1024 + w*128, +128) as kChunks chunks of 32 consecutive slots.
// Fills the per-warp histograms wh[kWarps][E] and returns each lane's ids and match masks.
__device__ __forceinline__ bool warp_histograms(const int32_t* __restrict__ ids, int64_t S, int E, int* wh,
                                                int (&id)[kChunks], unsigned (&mk)[kChunks]) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < kWarps * E; i += kThreads) wh[i] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * FEPLB_SLOTS_PER_BLOCK + w * (kChunks * 32);
  bool bad = false;
#pragma unroll
  for (int c = 0; c < kChunks; ++c) {
    const int64_t s = base + c * 32 + lane;
    int v = -1;
    if (s < S) {
      v = ids[s];
      if ((unsigned)v >= (unsigned)E) { bad = true; v = -1; }
    }
    id[c] = v;
    mk[c] = __match_any_sync(0xffffffffu, v);
    if (v >= 0 && lane == __ffs(mk[c]) - 1) wh[w * E + v] += __popc(mk[c]);
    __syncwarp();
  }
  return bad;
}

// A slot's rank among the slots of its expert inside its CTA's 1024 slots, as k_block_hist leaves it in
// slot_to_row for the gather kernel: -2 - rank (final rows are >= 0, -1 marks an id outside [0, E)).
__device__ __forceinline__ int encode_local_rank(int r) { return -2 - r; }

// Step 1: per-CTA histograms; with totals != nullptr (E accumulators and a ticket, all zero between calls) also counts
// and rank_load, by one atomic per CTA and expert and a last CTA, so that no memset has to precede the kernel;
// with local_rank != nullptr also every slot's encoded rank inside this CTA's slots.
__global__ void __launch_bounds__(kThreads)
k_block_hist(const int32_t* __restrict__ ids, int64_t S, int E, int L, int32_t* __restrict__ block_hist,
             int32_t* __restrict__ counts, int32_t* __restrict__ rank_load, int32_t* totals, uint32_t* status,
             int32_t* __restrict__ local_rank) {
  extern __shared__ int wh[];
  int id[kChunks];
  unsigned mk[kChunks];
  pdl_sync();
  if (warp_histograms(ids, S, E, wh, id, mk)) atomicOr(status, FEPLB_ST_RANGE);
  __syncthreads();
  // chain the warps: wh[w][e] becomes the rank of warp w's first slot of expert e; the sum is the CTA's count
  for (int e = threadIdx.x; e < E; e += kThreads) {
    int sum = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const int t = wh[w * E + e];
      wh[w * E + e] = sum;
      sum += t;
    }
    if (block_hist) block_hist[(int64_t)blockIdx.x * E + e] = sum;
    if (totals && sum) atomicAdd(&totals[e], sum);
  }
  if (totals) {
    // The CTA that arrives last writes the result and leaves the accumulators zero for the next call; the ticket
    // wraps to zero by itself.
    __shared__ int last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicInc(reinterpret_cast<unsigned*>(totals + E), gridDim.x - 1) == gridDim.x - 1;
    __syncthreads();
    if (last) {
      __threadfence();
      for (int e = threadIdx.x; e < E; e += kThreads) {
        const int n = __ldcg(totals + e);
        wh[e] = n;
        counts[e] = n;
        totals[e] = 0;
      }
      __syncthreads();
      for (int r = threadIdx.x; r < E / L; r += kThreads) {
        int n = 0;
        for (int e = r * L; e < (r + 1) * L; ++e) n += wh[e];
        rank_load[r] = n;
      }
    }
  }
  if (!local_rank) return;
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int64_t base = (int64_t)blockIdx.x * FEPLB_SLOTS_PER_BLOCK + w * (kChunks * 32);
#pragma unroll
  for (int c = 0; c < kChunks; ++c) {
    const int64_t s = base + c * 32 + lane;
    const int v = id[c];
    int r = 0;
    if (v >= 0) r = wh[w * E + v] + __popc(mk[c] & lt);
    __syncwarp();
    if (v >= 0 && lane == __ffs(mk[c]) - 1) wh[w * E + v] += __popc(mk[c]);
    __syncwarp();
    if (s < S) local_rank[s] = v >= 0 ? encode_local_rank(r) : -1;
  }
}

// Block-wide exclusive scan of v over the 1024 threads of the block; tmp holds 64 values.
template <typename V = int>
__device__ __forceinline__ V block_exclusive_scan(V v, V* tmp, V* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  V x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    V y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) tmp[w] = x;
  __syncthreads();
  if (w == 0) {
    V s = tmp[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      V y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    tmp[32 + lane] = s;   // inclusive scan of the warp sums
  }
  __syncthreads();
  const V warp_off = w ? tmp[32 + w - 1] : 0;
  if (total) *total = tmp[32 + 31];
  return warp_off + x - v;
}

// Exclusive scan over CTAs of the per-CTA histograms by one block of 1024 threads, in three steps: who takes which part
// of which expert's column (before the histograms are there), the sums, the prefixes in place.  Several threads
// share an expert, each taking at least four CTAs, so that the loads of a column are a few round trips.
// From the end of the histogram to the end of the scan, 64 CTAs, 128 experts: 9.9 us with one thread per expert, 5.6
// this way.  More parts cost more in the sums over the parts than they save (118 CTAs, 8 experts, route + gather +
// combine: up to 128 parts 65.9 us, up to 16 57.3).
struct ScanRows { int p, parts, e, r0, r1, base; int v[8]; };
__device__ __forceinline__ ScanRows scan_rows(int nb, int E) {
  ScanRows q;
  q.parts = max(1, min(min(1024 / E, 16), (nb + 3) / 4));
  q.p = threadIdx.x / E;
  q.e = threadIdx.x - q.p * E;
  const int per = (nb + q.parts - 1) / q.parts;
  q.r0 = q.p < q.parts ? min(nb, per * q.p) : 0;
  q.r1 = q.p < q.parts ? min(nb, q.r0 + per) : 0;
  return q;
}
// Returns the expert's total (threads < E).  part: 1024 ints of shared memory.
__device__ __forceinline__ int sum_rows(const int32_t* __restrict__ block_hist, int E, int* part, ScanRows& q) {
  int sum = 0;
  for (int b0 = q.r0; b0 < q.r1; b0 += 8) {          // eight independent loads in flight per round
#pragma unroll
    for (int j = 0; j < 8; ++j) q.v[j] = b0 + j < q.r1 ? block_hist[(int64_t)(b0 + j) * E + q.e] : 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) sum += q.v[j];
  }
  part[threadIdx.x] = sum;
  __syncthreads();
  q.base = 0;
  int total = 0;
  if (q.p < q.parts)
    for (int o = 0; o < q.parts; ++o) {
      const int t = part[o * E + q.e];
      if (o < q.p) q.base += t;
      total += t;
    }
  return total;
}
__device__ __forceinline__ void store_scan(int32_t* __restrict__ block_hist, int E, ScanRows& q) {
  int run = q.base;
  const bool kept = q.r1 - q.r0 <= 8;
  for (int b0 = q.r0; b0 < q.r1; b0 += 8) {
    if (!kept) {
#pragma unroll
      for (int j = 0; j < 8; ++j) q.v[j] = b0 + j < q.r1 ? block_hist[(int64_t)(b0 + j) * E + q.e] : 0;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (b0 + j < q.r1) block_hist[(int64_t)(b0 + j) * E + q.e] = run;
      run += q.v[j];
    }
  }
}

// Exclusive scan of the per-CTA histograms over CTAs (in place), check against counts, and
// pad_off[e] = sum_{e'<e} round_up(counts[e'], A); pad_off[E] = padded total.
// The counts are the caller's: when they disagree with the ids (FEPLB_ST_COUNTS) the result is
// wrong but every later access stays inside the caller's buffers -- a negative count is taken as
// zero, offsets are summed in 64 bits and clamped to s_cap, a padded total beyond s_cap is reported;
// the gather kernel then drops the rows that do not fit.
__global__ void __launch_bounds__(1024)
k_scan(int32_t* __restrict__ block_hist, int nb, int E, int A, const int32_t* __restrict__ counts,
       int32_t* __restrict__ pad_off, int64_t s_cap, uint32_t* status, int32_t* __restrict__ row_to_token) {
  __shared__ long long tmp[64];
  __shared__ int part[1024];
  const int e = threadIdx.x;
  int c = 0;
  ScanRows q = scan_rows(nb, E);
  pdl_sync();
  const int run = sum_rows(block_hist, E, part, q);
  store_scan(block_hist, E, q);
  if (e < E) {
    c = counts[e];
    if (run != c) atomicOr(status, FEPLB_ST_COUNTS);
    if (c < 0) c = 0;
  }
  long long total;
  const long long off = block_exclusive_scan<long long>(((long long)c + A - 1) / A * A, tmp, &total);
  if (e < E) pad_off[e] = (int32_t)(off < s_cap ? off : s_cap);
  if (e == 0) {
    pad_off[E] = (int32_t)(total < s_cap ? total : s_cap);
    if (total > s_cap) atomicOr(status, FEPLB_ST_COUNTS);
  }
  // rows behind the last segment hold no token (the padding rows inside segments and the
  // live rows are marked by k_gather: with counts that agree with the ids that covers every row)
  for (int64_t i = total + threadIdx.x; i < s_cap; i += blockDim.x) row_to_token[i] = -1;
}

// Whole-layer variant of k_scan: from the per-CTA histograms alone it produces everything the
// rest of the pass needs -- counts, per-rank loads, segment offsets, the home group table (with
// the dynamic-expert mask, given or derived from the counts) and the -1 tail of row_to_token --
// so that no memset, atomic or extra launch sits between the histogram and the plan.
__global__ void __launch_bounds__(1024)
k_scan_fused(int32_t* __restrict__ block_hist, int nb, int E, int L, int A, int dyn,
             const uint8_t* __restrict__ mask_in, int32_t* __restrict__ counts_out,
             int32_t* __restrict__ rank_load_out, int32_t* __restrict__ pad_off,
             feplb_group* __restrict__ groups, uint8_t* __restrict__ mask_out,
             int32_t* __restrict__ row_to_token, int64_t s_cap,
             unsigned long long* __restrict__ counts_host_tagged, int32_t seq, unsigned long long* t_counts) {
  __shared__ int tmp[64];
  __shared__ int part[1024];
  __shared__ int sc[FEPLB_MAX_EXPERTS];
  const int e = threadIdx.x;
  int c = 0;
  ScanRows q = scan_rows(nb, E);
  pdl_sync();
  const int run = sum_rows(block_hist, E, part, q);
  if (e < E) {
    c = run;
    counts_out[e] = c;
    sc[e] = c;
    // Straight into pinned host memory for the planner thread, each count in one 8-byte word that
    // carries this forward's sequence number: the reader polls until every word shows the
    // number, so no system-scope fence and no separate flag hold this kernel up (under bulk
    // host<->device copies such a fence was measured to cost tens of microseconds).
    if (counts_host_tagged)
      *reinterpret_cast<volatile unsigned long long*>(counts_host_tagged + e) =
          ((unsigned long long)(uint32_t)seq << 32) | (uint32_t)c;
  }
  store_scan(block_hist, E, q);
  if (t_counts && e == 0) {            // timeline: when the counts left for the host (globaltimer, ns)
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    *t_counts = t;
  }
  int total;
  const int off = block_exclusive_scan((c + A - 1) / A * A, tmp, &total);   // also orders sc[] for all threads
  if (e < E) {
    pad_off[e] = off;
    int is_dyn;
    if (mask_in) {
      is_dyn = mask_in[e] != 0;
    } else {
      const int b0 = e / L * L;
      int better = 0;
      for (int o = b0; o < b0 + L; ++o) better += (sc[o] > c) || (sc[o] == c && o < e);
      is_dyn = better < dyn;
    }
    groups[e] = feplb_group{e, off, c, e / L, is_dyn};
    if (mask_out) mask_out[e] = (uint8_t)is_dyn;
  }
  if (e == 0) pad_off[E] = total;
  if (e < E / L) {
    int sum = 0;
    for (int o = e * L; o < (e + 1) * L; ++o) sum += sc[o];
    rank_load_out[e] = sum;
  }
  for (int64_t i = (int64_t)total + threadIdx.x; i < s_cap; i += blockDim.x) row_to_token[i] = -1;
}

__device__ __forceinline__ uint4 ld_nc_v4(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// Row gather, token-major: one warp reads a token's row once (16-byte vectors, coalesced) and
// writes it to the K rows of its slots.  A slot's row = segment offset of its expert + first row of
// its CTA-of-1024-slots within the segment (both from the scan) + its rank inside that CTA (left in
// slot_to_row by k_block_hist); the warp that copies the first slice of a token writes the final
// slot_to_row and row_to_token entries (tokens [t0, t0 + T) of the batch).  Another warp working on a later slice of the same token may
// read either form of the entry, and gets the same row from both.
constexpr int kGatherUnroll = 4;
// How long the gather's first CTA looks for the planner's table even if the rows are copied in less: a planner whose
// thread is awake publishes it 2-3 us after the scan, one that has to be woken (a forward on an idle GPU) some 5 us later.
// One such forward and the wait for it, T = 2000 / 4096: 208 / 298 us with a fixed wait of 15 us, 216 / 299 with 4 us at
// least, 205 / 296 with 8 and the thread woken before the routing launches.  When the planner is late (held back 60 us), 64 experts,
// d = 2048, us per layer without an early table -> a fixed wait of 15 us -> this: T = 1400 190 -> 194 -> 188, T = 2000
// 227 -> 231 -> 227, T = 4096 343 -> 343 -> 341; when it is not: 191 -> 185 -> 181, 228 -> 220 -> 216, 343 -> 334 -> 333.
constexpr unsigned long long kEarlyTableNs = 8000;
// Work unit = (token, slice of 4 x 32 chunks = 2 KiB of its row).  Unit u goes to warp u mod #warps of a grid
// sized to the machine: all warps work on neighbouring tokens at any time, and the rows of an expert, which
// follow the token order, are written in one moving window per expert, so that DRAM pages are written while
// they are open.  With a contiguous range of units per warp (every warp in a place of its own) the gather and
// the combine together, T = 8192, top-8, d = 6144, ran at 5.5 TB/s; this way at 6.0 (route + gather +
// combine 353 -> 330 us).  Slices of 1 KiB: 347 us, of 4 KiB: the same.
__global__ void __launch_bounds__(kThreads, 6)     // 40 registers; with 48 (five CTAs per SM) route + gather + combine 310 -> 315 us
k_gather(const uint4* __restrict__ x, const int32_t* __restrict__ ids, const int32_t* __restrict__ pad_off,
         const int32_t* __restrict__ block_base, int32_t* slot_to_row, int32_t* __restrict__ row_to_token,
         uint4* __restrict__ x_perm, int t0, int T, int K, int E, int chunks, int64_t s_cap, const int32_t* __restrict__ counts,
         int A, const DynTable dyn, uint32_t* status) {
  pdl_sync();
  const int lane = threadIdx.x & 31;
  const int first = dyn.seq != 0;        // the first CTA picks the planner's table up
  if (first && blockIdx.x == 0) {
    if (threadIdx.x < 32) dyn_deliver_early(dyn, lane, status, kEarlyTableNs);
    return;
  }
  const int64_t warp = ((int64_t)(blockIdx.x - first) * kThreads + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)(gridDim.x - first) * kThreads) >> 5;
  const int slices = (chunks + 32 * kGatherUnroll - 1) / (32 * kGatherUnroll);
  const int64_t units = (int64_t)T * slices;
  for (int64_t u = warp; u < units; u += nwarps) {
    const int tu = (int)(u / slices), t = t0 + tu;
    const int c0 = (int)(u - (int64_t)tu * slices) * 32 * kGatherUnroll;
    const uint4* src = x + (int64_t)t * chunks;
    uint4 v[kGatherUnroll];
#pragma unroll
    for (int i = 0; i < kGatherUnroll; ++i) {
      const int c = c0 + i * 32 + lane;
      if (c < chunks) v[i] = ld_nc_v4(src + c);
    }
    int myrow = -1;
    if (lane < K) {
      const int64_t s = (int64_t)t * K + lane;
      const int r = __ldcg(slot_to_row + s);
      const int e = ids[s];      // in flight together with r; its offsets follow in one more round trip
      if (r >= 0) {
        myrow = r;               // already final
      } else if (r <= -2) {      // implies 0 <= e < E (checked by k_block_hist)
        const int64_t row = (int64_t)pad_off[e] + block_base[s / FEPLB_SLOTS_PER_BLOCK * E + e] + (-2 - r);
        // rows beyond the buffer: only with counts that disagree with the ids (reported by the scan)
        myrow = row < s_cap ? (int)row : -1;
      }
      if (c0 == 0) {             // the token's first slice: this warp publishes the rows
        slot_to_row[s] = myrow;
        if (myrow >= 0) row_to_token[myrow] = t;
      }
    }
    for (int k = 0; k < K; ++k) {
      const int row = __shfl_sync(0xffffffffu, myrow, k);
      if (row < 0) continue;
      uint4* dst = x_perm + (int64_t)row * chunks;
#pragma unroll
      for (int i = 0; i < kGatherUnroll; ++i) {
        const int c = c0 + i * 32 + lane;
        if (c < chunks) dst[c] = v[i];
      }
    }
  }
  if (first && threadIdx.x == 0) *reinterpret_cast<volatile uint32_t*>(dyn.gather_done) = dyn.seq;
  if (A > 1) {                   // zeros for the padding rows at the end of every expert's segment, one row per warp at a time
    for (int64_t q = warp; q < (int64_t)E * A; q += nwarps) {
      const int e = (int)(q / A), c = counts[e] > 0 ? counts[e] : 0;
      // clamped to the buffer: counts that disagree with the ids must not turn into wild writes
      const int64_t row = (int64_t)pad_off[e] + c + (q - (int64_t)e * A);
      if (row >= pad_off[e + 1] || row >= s_cap || row < 0) continue;
      for (int i = lane; i < chunks; i += 32) x_perm[row * chunks + i] = make_uint4(0, 0, 0, 0);
      if (lane == 0) row_to_token[row] = -1;
    }
  }
}

// The whole front of a layer pass for small batches -- histogram, ranks, scan, home group table and row gather --
// as ONE launch.  Chained, the three kernels it replaces take 11 us of launch and memory latency whatever the
// size; here every CTA computes the complete routing of the batch for itself (at most kSmallMaxSlots ids, read
// from L2; the ranks end up in shared memory), so that no CTA needs another one's result, and then copies
// its share of the rows.  CTA 0 alone publishes the tables (groups != nullptr) or compares the counts with the
// caller's (counts_in, stand-alone dispatch: the segments have the caller's sizes, clamped to the buffer, as in
// k_scan and k_gather).  The redundant part grows with the number of slots and ends the range: see
// feplb_front_is_small.
// Whole layer, chained front -> this: 32.3 -> 27.9 us at T = 256, top-2, d = 128, 8 experts; 102.0 -> 97.9 us at
// T = 64, top-6, d = 2048, 64 experts.
constexpr int kSmallThreads = 1024;
constexpr int kSmallWarps = kSmallThreads / 32;
constexpr int kSmallSlice = 64;              // 16-byte chunks of a row per work unit (2 per lane)

template <int CH>                            // chunks of 32 slots per warp
__global__ void __launch_bounds__(kSmallThreads, 1)
k_route_small(const uint4* __restrict__ x, const int32_t* __restrict__ ids, int T, int K, int E, int L, int A, int dyn,
              const uint8_t* __restrict__ mask_in, const int32_t* __restrict__ counts_in, int32_t* __restrict__ counts_out,
              int32_t* __restrict__ rank_load_out, int32_t* __restrict__ pad_off_out, feplb_group* __restrict__ groups, int32_t* __restrict__ slot_to_row,
              int32_t* __restrict__ row_to_token, uint4* __restrict__ x_perm, int chunks, int64_t s_cap, uint32_t* status,
              unsigned long long* __restrict__ counts_host_tagged, int32_t seq, unsigned long long* t_counts) {
  extern __shared__ int sm[];
  __shared__ int tmp[64];
  int* wh = sm;                              // [kSmallWarps][E] histograms per warp, then ranks of a warp's first slots
  int* sc = wh + kSmallWarps * E;            // [E] rows of the segment: the counts, or the caller's
  int* pad = sc + E;                         // [E] first row of the segment
  int* rows = pad + E;                       // [32 * 32 * CH] row of every slot, -1 for an id outside [0, E)
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int S = T * K;
  for (int i = threadIdx.x; i < kSmallWarps * E; i += kSmallThreads) wh[i] = 0;
  __syncthreads();
  pdl_sync();
  // the first work unit's row piece and this warp's ids, all in flight together
  const int slices = (chunks + kSmallSlice - 1) / kSmallSlice;
  const int units = T * slices;
  int u = blockIdx.x + gridDim.x * w;
  uint4 v[2];
  auto load_unit = [&](int unit) {
    const int t = unit / slices, c0 = (unit - t * slices) * kSmallSlice;
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (c0 + i * 32 + lane < chunks) v[i] = ld_nc_v4(x + (int64_t)t * chunks + c0 + i * 32 + lane);
  };
  int id[CH];
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    const int s = (w * CH + c) * 32 + lane;
    id[c] = s < S ? ids[s] : -1;
  }
  const int given = counts_in && (int)threadIdx.x < E ? counts_in[threadIdx.x] : 0;
  if (u < units) load_unit(u);
  unsigned mk[CH];
  bool bad = false;
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    if ((unsigned)id[c] >= (unsigned)E) {
      bad |= (w * CH + c) * 32 + lane < S;
      id[c] = -1;
    }
    mk[c] = __match_any_sync(0xffffffffu, id[c]);
    if (id[c] >= 0 && lane == __ffs(mk[c]) - 1) wh[w * E + id[c]] += __popc(mk[c]);
    __syncwarp();
  }
  if (bad && blockIdx.x == 0) atomicOr(status, FEPLB_ST_RANGE);
  __syncthreads();
  const int e = threadIdx.x;
  int cnt = 0;
  if (e < E) {
#pragma unroll
    for (int i = 0; i < kSmallWarps; ++i) {
      const int n = wh[i * E + e];
      wh[i * E + e] = cnt;
      cnt += n;
    }
    if (blockIdx.x == 0) {
      if (counts_in && given != cnt) atomicOr(status, FEPLB_ST_COUNTS);
      if (counts_out) counts_out[e] = cnt;
      if (counts_host_tagged)                // see k_scan_fused
        *reinterpret_cast<volatile unsigned long long*>(counts_host_tagged + e) =
            ((unsigned long long)(uint32_t)seq << 32) | (uint32_t)cnt;
    }
    // a segment larger than the buffer pushes the ones behind it out of it whatever its size: no sum overflows
    if (counts_in) cnt = min(max(given, 0), (int)s_cap);
    sc[e] = cnt;
  }
  if (blockIdx.x == 0 && e == 0 && t_counts) {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    *t_counts = t;
  }
  int total;
  const int off = block_exclusive_scan((cnt + A - 1) / A * A, tmp, &total);      // also orders sc[] and wh[] for all threads
  if (e < E) pad[e] = off;
  __syncthreads();
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    int r = -1;
    if (id[c] >= 0) r = pad[id[c]] + wh[w * E + id[c]] + __popc(mk[c] & lt);
    if (r >= s_cap) r = -1;                  // only with counts that disagree with the ids
    __syncwarp();
    if (id[c] >= 0 && lane == __ffs(mk[c]) - 1) wh[w * E + id[c]] += __popc(mk[c]);
    __syncwarp();
    rows[(w * CH + c) * 32 + lane] = r;
  }
  __syncthreads();
  for (; u < units; u += gridDim.x * kSmallWarps) {
    const int t = u / slices, c0 = (u - t * slices) * kSmallSlice;
    if (c0 == 0 && lane < K) {
      const int row = rows[t * K + lane];
      slot_to_row[t * K + lane] = row;
      if (row >= 0) row_to_token[row] = t;
    }
    for (int k = 0; k < K; ++k) {
      const int row = rows[t * K + k];
      if (row < 0) continue;
      uint4* dst = x_perm + (int64_t)row * chunks + c0 + lane;
      if (c0 + lane < chunks) dst[0] = v[0];
      if (c0 + 32 + lane < chunks) dst[32] = v[1];
    }
    if (u + gridDim.x * kSmallWarps < units) load_unit(u + gridDim.x * kSmallWarps);
  }
  if (groups && blockIdx.x == 0) {       // whole-layer path
    if (e < E) {
      pad_off_out[e] = off;
      int is_dyn;
      if (mask_in) {
        is_dyn = mask_in[e] != 0;
      } else {
        const int b0 = e / L * L;
        int better = 0;
        for (int o = b0; o < b0 + L; ++o) better += (sc[o] > cnt) || (sc[o] == cnt && o < e);
        is_dyn = better < dyn;
      }
      groups[e] = feplb_group{e, off, cnt, e / L, is_dyn};
    }
    if (e == 0) pad_off_out[E] = total;
    if (e < E / L) {
      int sum = 0;
      for (int o = e * L; o < (e + 1) * L; ++o) sum += sc[o];
      rank_load_out[e] = sum;
    }
  }
  for (int64_t i = (int64_t)total + (int64_t)blockIdx.x * kSmallThreads + threadIdx.x; i < s_cap;
       i += (int64_t)gridDim.x * kSmallThreads)
    row_to_token[i] = -1;
  if (A > 1) {                               // padding rows at the end of the segments
    for (int g = blockIdx.x; g < E; g += gridDim.x) {
      const int r0 = pad[g] + sc[g], r1 = (int)min((int64_t)pad[g] + (sc[g] + A - 1) / A * A, s_cap);
      for (int r = r0 + (int)threadIdx.x; r < r1; r += kSmallThreads) row_to_token[r] = -1;
      uint4* p = x_perm + (int64_t)r0 * chunks;
      const int64_t n = (int64_t)(r1 - r0) * chunks;
      for (int64_t i = threadIdx.x; i < n; i += kSmallThreads) p[i] = make_uint4(0, 0, 0, 0);
    }
  }
}

// Home group table {e, pad_off[e], counts[e], home(e), dynamic?} for all E experts.
__global__ void __launch_bounds__(1024)
k_home_groups(const int32_t* __restrict__ counts, const uint8_t* __restrict__ mask_in, int E, int L, int A, int dyn,
              feplb_group* __restrict__ groups, uint8_t* __restrict__ mask_out) {
  __shared__ int tmp[64];
  __shared__ int sc[FEPLB_MAX_EXPERTS];
  const int e = threadIdx.x;
  const int c = e < E ? counts[e] : 0;
  if (e < E) sc[e] = c;
  const int off = block_exclusive_scan<int>((c + A - 1) / A * A, tmp, nullptr);
  if (e >= E) return;
  int is_dyn;
  if (mask_in) {
    is_dyn = mask_in[e] != 0;
  } else {
    // dynamic iff fewer than `dyn` experts of the block are busier (ties: lower id is busier)
    const int b0 = e / L * L;
    int better = 0;
    for (int o = b0; o < b0 + L; ++o) better += (sc[o] > c) || (sc[o] == c && o < e);
    is_dyn = better < dyn;
  }
  groups[e] = feplb_group{e, off, c, e / L, is_dyn};
  if (mask_out) mask_out[e] = (uint8_t)is_dyn;
}

// Group tables of a batch processed in token ranges whose first slots are multiples of 1024: range r (one CTA) holds, per
// expert, the rows of its slots, which lie side by side in the expert's segment because rows follow the slots.
__global__ void __launch_bounds__(1024)
k_range_groups(const int32_t* __restrict__ block_base, int nb, int E, const feplb_group* __restrict__ home, RangeBlocks rb,
               feplb_group* __restrict__ out) {
  pdl_sync();
  const int e = threadIdx.x, b0 = rb.first[blockIdx.x], b1 = rb.first[blockIdx.x + 1];
  if (e >= E) return;
  feplb_group g = home[e];
  const int lo = b0 < nb ? block_base[(int64_t)b0 * E + e] : g.rows, hi = b1 < nb ? block_base[(int64_t)b1 * E + e] : g.rows;
  g.row_start += lo;
  g.rows = hi - lo;
  out[(int64_t)blockIdx.x * E + e] = g;
}

// Order-preserving map of finite floats to unsigned integers > 0; -0 and +0 map to the same value.
__device__ __forceinline__ unsigned sortable(float f) {
  const unsigned u = __float_as_uint(f + 0.f);
  return u & 0x80000000u ? ~u : u | 0x80000000u;
}
__device__ __forceinline__ float unsortable(unsigned u) { return __uint_as_float(u & 0x80000000u ? u & 0x7fffffffu : ~u); }

// Router top-k gating (paper Sections 2.3 and 3.1: top-k routing, no auxiliary loss): one warp per
// token.  Lane l holds logits l, l+32, ... as sortable integers (0 = none or taken); each of the K rounds finds the
// largest by one warp reduction and the lowest expert id that has it by a second one; gates = softmax over the K
// selected logits.  Bound by the instructions of the rounds, not by memory: with five shuffles of value and id
// per round in place of the two reductions 13.1 us
// at T = 8192, E = 128, top-8, this way 6.9.
template <int NPER>
__global__ void __launch_bounds__(kThreads)
k_route_topk(const float* __restrict__ logits, int T, int E, int K, int32_t* __restrict__ ids,
             float* __restrict__ gates) {
  pdl_sync();
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * kThreads + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * kThreads) >> 5;
  for (int t = warp; t < T; t += nwarps) {
    unsigned v[NPER];
#pragma unroll
    for (int i = 0; i < NPER; ++i) {
      const int e = i * 32 + lane;
      v[i] = e < E ? sortable(logits[(int64_t)t * E + e]) : 0u;
    }
    float sel_val = 0.f;
    int sel_idx = 0;
    for (int k = 0; k < K; ++k) {
      unsigned best = 0;
#pragma unroll
      for (int i = 0; i < NPER; ++i) best = max(best, v[i]);
      best = __reduce_max_sync(0xffffffffu, best);
      unsigned idx = 0xffffffffu;
#pragma unroll
      for (int i = NPER - 1; i >= 0; --i)
        if (v[i] == best) idx = i * 32 + lane;
      idx = __reduce_min_sync(0xffffffffu, idx);
#pragma unroll
      for (int i = 0; i < NPER; ++i)
        if (i * 32 + lane == idx) v[i] = 0u;
      if (lane == k) { sel_val = unsortable(best); sel_idx = (int)idx; }
    }
    const float m = __shfl_sync(0xffffffffu, sel_val, 0);       // the first pick is the maximum
    float ex = lane < K ? expf(sel_val - m) : 0.f;
    float sum = ex;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane < K) {
      ids[(int64_t)t * K + lane] = sel_idx;
      gates[(int64_t)t * K + lane] = ex / sum;
    }
  }
}

}  // namespace

cudaError_t feplb_launch_route_hist(const int32_t* ids, int64_t S, int E, int R, int32_t* totals, int32_t* counts,
                                    int32_t* rank_load, uint32_t* status, cudaStream_t st, int64_t* n_launch) {
  cudaError_t err;
  const int nb = (int)((S + FEPLB_SLOTS_PER_BLOCK - 1) / FEPLB_SLOTS_PER_BLOCK);
  if (nb == 0) {
    if ((err = cudaMemsetAsync(counts, 0, sizeof(int32_t) * E, st)) != cudaSuccess) return err;
    return cudaMemsetAsync(rank_load, 0, sizeof(int32_t) * R, st);
  }
  ++*n_launch;
  return launch(k_block_hist, nb, kThreads, sizeof(int) * kWarps * E, st, true, ids, S, E, E / R, (int32_t*)nullptr, counts,
                rank_load, totals, status, (int32_t*)nullptr);
}

cudaError_t feplb_launch_permute(const int32_t* ids, int64_t S, int K, int E, int A, const int32_t* counts,
                                 int32_t* block_hist, int32_t* pad_off, int32_t* slot_to_row,
                                 int32_t* row_to_token, int64_t s_cap, uint32_t* status,
                                 cudaStream_t st, int64_t* n_launch) {
  // two kernels chained by a programmatic launch (the second one's launch latency hides under the first);
  // feplb_launch_gather, which must follow, turns the ranks they leave in slot_to_row into rows
  (void)K;
  cudaError_t err;
  const int nb = (int)((S + FEPLB_SLOTS_PER_BLOCK - 1) / FEPLB_SLOTS_PER_BLOCK);
  if (nb) {
    err = launch(k_block_hist, nb, kThreads, sizeof(int) * kWarps * E, st, true, ids, S, E, E, block_hist,
                 (int32_t*)nullptr, (int32_t*)nullptr, (int32_t*)nullptr, status, slot_to_row);
    ++*n_launch;
    if (err != cudaSuccess) return err;
  }
  err = launch(k_scan, 1, 1024, 0, st, nb > 0, block_hist, nb, E, A, counts, pad_off, s_cap, status, row_to_token);
  ++*n_launch;
  return err;
}

cudaError_t feplb_launch_gather(const void* x, const int32_t* ids, const int32_t* block_base, int32_t* slot_to_row,
                                const int32_t* counts, const int32_t* pad_off, void* x_perm, int T, int K, int E, int d,
                                int A, int64_t s_cap, int num_sms, cudaStream_t st, int64_t* n_launch,
                                int32_t* row_to_token, bool programmatic, int t0, const feplb_wm_dyn* dyn, uint32_t* status) {
  const int chunks = d / 8;
  if (T == 0 && A == 1) return cudaSuccess;
  const int64_t units = (int64_t)T * ((chunks + 32 * kGatherUnroll - 1) / (32 * kGatherUnroll));
  int blocks = num_sms * 8;   // 8 CTAs of 256 threads per SM are resident
  const int64_t need = ((A > 1 && units < (int64_t)E * A ? (int64_t)E * A : units) + kWarps - 1) / kWarps;
  if (need < blocks) blocks = (int)need;
  const feplb_wm_dyn none;
  if (dyn && dyn->seq && blocks < num_sms * 8) ++blocks;
  ++*n_launch;
  return launch(k_gather, blocks, kThreads, 0, st, programmatic, (const uint4*)x, ids, pad_off, block_base, slot_to_row,
                row_to_token, (uint4*)x_perm, t0, T, K, E, chunks, s_cap, counts, A,
                feplb_dyn_table(dyn ? *dyn : none), status);
}

// Copies the planner's table of dynamic groups from mapped pinned host memory to the device.  A
// kernel rather than a host-to-device memcpy: a memcpy would queue on the copy engine behind
// whatever bulk input transfer is in flight, and the dynamic GEMM waits for this table.
__global__ void __launch_bounds__(256) k_upload_groups(const int4* __restrict__ src_host, int4* __restrict__ dst, int n16) {
  for (int i = threadIdx.x; i < n16; i += 256) dst[i] = src_host[i];
}

cudaError_t feplb_launch_upload_groups(const feplb_group* src_host_mapped, feplb_group* dst, int n, cudaStream_t st) {
  const int n16 = (int)(((size_t)n * sizeof(feplb_group) + 15) / 16);      // both tables are allocated in 16-byte multiples
  if (n16 == 0) return cudaSuccess;
  k_upload_groups<<<1, 256, 0, st>>>(reinterpret_cast<const int4*>(src_host_mapped), reinterpret_cast<int4*>(dst), n16);
  return cudaGetLastError();
}

cudaError_t feplb_launch_home_groups(const int32_t* counts, const uint8_t* mask_in, int E, int R, int A, int dyn,
                                     feplb_group* groups, uint8_t* mask_out, cudaStream_t st, int64_t* n_launch) {
  k_home_groups<<<1, 1024, 0, st>>>(counts, mask_in, E, E / R, A, dyn, groups, mask_out);
  ++*n_launch;
  return cudaGetLastError();
}

cudaError_t feplb_launch_route_fused(const int32_t* ids, int64_t S, int E, int R, int A, int dyn,
                                     const uint8_t* mask_in, int32_t* block_hist, int32_t* counts,
                                     int32_t* rank_load, int32_t* pad_off, feplb_group* groups, uint8_t* mask_out,
                                     int32_t* slot_to_row, int32_t* row_to_token, int64_t s_cap, uint32_t* status,
                                     unsigned long long* counts_host_tagged, int32_t seq, unsigned long long* t_counts,
                                     cudaStream_t st, int64_t* n_launch) {
  cudaError_t err;
  const int nb = (int)((S + FEPLB_SLOTS_PER_BLOCK - 1) / FEPLB_SLOTS_PER_BLOCK);
  if (nb) {
    err = launch(k_block_hist, nb, kThreads, sizeof(int) * kWarps * E, st, true, ids, S, E, E, block_hist,
                 (int32_t*)nullptr, (int32_t*)nullptr, (int32_t*)nullptr, status, slot_to_row);
    ++*n_launch;
    if (err != cudaSuccess) return err;
  }
  ++*n_launch;
  return launch(k_scan_fused, 1, 1024, 0, st, true, block_hist, nb, E, E / R, A, dyn, mask_in, counts, rank_load, pad_off,
                groups, mask_out, row_to_token, s_cap, counts_host_tagged, seq, t_counts);
}

cudaError_t feplb_launch_range_groups(const int32_t* block_base, int64_t S, int K, int E, const feplb_group* home,
                                      const int* first_token, int n_ranges, feplb_group* out, cudaStream_t st, int64_t* n_launch) {
  RangeBlocks rb = {};
  const int nb = (int)((S + FEPLB_SLOTS_PER_BLOCK - 1) / FEPLB_SLOTS_PER_BLOCK);
  for (int i = 0; i <= n_ranges; ++i)
    rb.first[i] = i == n_ranges ? nb : (int)((int64_t)first_token[i] * K / FEPLB_SLOTS_PER_BLOCK);
  ++*n_launch;
  return launch(k_range_groups, n_ranges, 1024, 0, st, true, block_base, nb, E, home, rb, out);
}

// The one-launch front pays while the routing that every CTA repeats is short: its eight match rounds at 8192
// slots take as long as the two launches it saves (T = 1537, top-4, d = 1920: 155.9 us per layer either way).
constexpr int kSmallMaxSlots = FEPLB_FRONT_SMALL_SLOTS, kSmallMaxExperts = 256;
bool feplb_front_is_small(int64_t S, int E) { return S > 0 && S <= kSmallMaxSlots && E <= kSmallMaxExperts; }

template <int CH>
static cudaError_t launch_small(const void* x, const int32_t* ids, int T, int K, int E, int R, int d, int A, int dyn,
                                const uint8_t* mask_in, const int32_t* counts_in, int32_t* counts, int32_t* rank_load, int32_t* pad_off,
                                feplb_group* groups, int32_t* slot_to_row, int32_t* row_to_token, void* x_perm, int64_t s_cap, uint32_t* status,
                                unsigned long long* counts_host_tagged, int32_t seq, unsigned long long* t_counts, int num_sms,
                                cudaStream_t st) {
  static bool ready[64] = {};                // per instantiation and device: the shared-memory attribute
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!ready[dev]) {
    const int most = (int)sizeof(int) * ((kSmallWarps + 2) * kSmallMaxExperts + kSmallThreads * CH);
    cudaError_t e = cudaFuncSetAttribute(k_route_small<CH>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e != cudaSuccess) return e;
    ready[dev] = true;
  }
  const int chunks = d / 8;
  const int64_t units = (int64_t)T * ((chunks + kSmallSlice - 1) / kSmallSlice);
  const int64_t want = A > 1 && units < E ? E : units;       // padding rows are zeroed one expert per CTA
  const int grid = (int)(want < num_sms ? want : num_sms);
  const size_t smem = sizeof(int) * ((size_t)(kSmallWarps + 2) * E + (size_t)kSmallThreads * CH);
  return launch(k_route_small<CH>, grid, kSmallThreads, smem, st, true, (const uint4*)x, ids, T, K, E, E / R, A, dyn, mask_in,
                counts_in, counts, rank_load, pad_off, groups, slot_to_row, row_to_token, (uint4*)x_perm, chunks, s_cap, status,
                counts_host_tagged, seq, t_counts);
}

cudaError_t feplb_launch_front_small(const void* x, const int32_t* ids, int T, int K, int E, int R, int d, int A, int dyn,
                                     const uint8_t* mask_in, const int32_t* counts_in, int32_t* counts, int32_t* rank_load,
                                     int32_t* pad_off, feplb_group* groups, int32_t* slot_to_row, int32_t* row_to_token, void* x_perm,
                                     int64_t s_cap, uint32_t* status, unsigned long long* counts_host_tagged, int32_t seq,
                                     unsigned long long* t_counts, int num_sms, cudaStream_t st, int64_t* n_launch) {
  const int S = T * K;
  auto go = [&](auto fn) {
    return fn(x, ids, T, K, E, R, d, A, dyn, mask_in, counts_in, counts, rank_load, pad_off, groups, slot_to_row, row_to_token, x_perm,
              s_cap, status, counts_host_tagged, seq, t_counts, num_sms, st);
  };
  ++*n_launch;
  if (S <= kSmallThreads) return go(launch_small<1>);
  if (S <= kSmallThreads * 2) return go(launch_small<2>);
  if (S <= kSmallThreads * 4) return go(launch_small<4>);
  static_assert(kSmallMaxSlots == kSmallThreads * 8, "slots of the largest instantiation");
  return go(launch_small<8>);
}

cudaError_t feplb_launch_route_topk(const float* logits, int T, int E, int K, int32_t* ids, float* gates,
                                    int num_sms, cudaStream_t st, int64_t* n_launch) {
  if (T == 0) return cudaSuccess;
  int blocks = (T + kWarps - 1) / kWarps;
  if (blocks > num_sms * 8) blocks = num_sms * 8;
  const int nper = (E + 31) / 32;
  auto kernel = nper <= 1 ? k_route_topk<1> : nper <= 2 ? k_route_topk<2> : nper <= 4 ? k_route_topk<4>
                : nper <= 8 ? k_route_topk<8> : nper <= 16 ? k_route_topk<16> : k_route_topk<32>;
  ++*n_launch;
  return launch(kernel, blocks, kThreads, 0, st, true, logits, T, E, K, ids, gates);
}
