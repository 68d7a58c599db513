// Grouped SwiGLU expert FFN of the FEPLB hot path on sm_100a (paper Section 2.3: static-expert,
// then dynamic-expert Grouped GEMM; Section 3.1: grouped GEMM over per-expert row segments).
//
// Two launches of one persistent, warp-specialised kernel:
//   pass 1 (SwiGLU): H[rows, n0:n0+bn] = silu(X W1[e]) * (X W3[e])   -- one MMA of N = 2*bn whose
//                    B tile is the W1 tile followed by the W3 tile; the epilogue multiplies
//                    the two halves of the accumulator and rounds to bf16
//   pass 2 (plain):  Y[rows, n0:n0+2bn] = H W2[e]
// Per CTA: warp 0 = TMA producer (one lane), warp 1 = tcgen05.mma issuer (one lane) and TMEM
// owner, the other warps = epilogue (tcgen05.ld -> registers -> global).  A and B tiles are
// staged by TMA (128-byte swizzle, K-major) through a shared-memory ring; the fp32 accumulators
// live in TMEM.  A tile covers rows of ONE group (row segment of one expert); the last tile of
// a group is ragged and its surplus rows are computed but never stored.
//
// Every mbarrier wait is bounded: when it gives up the CTA raises FEPLB_ST_WAIT in the status
// word, all roles leave their loops, TMEM is released and the kernel returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdio>

#include "feplb_internal.h"
#include "feplb_tc.cuh"
#include "feplb_dyn.cuh"

namespace {

constexpr int BM = FEPLB_TILE_M;       // rows per MMA (UMMA M) = rows of one sub-tile
constexpr int kChunk = 64;             // K elements of a 128-byte swizzle row
constexpr int UMMA_K = 16;             // K per tcgen05.mma for 16-bit inputs
constexpr int kAccCols = 256;          // TMEM columns of one accumulator
constexpr int kTmemCols = 512;         // all of TMEM: one CTA per SM
// A single-form tile with at most kFewRows valid rows loads a box of only so many: while weights stream from HBM the
// padding rows of full boxes would be a third of the bytes through an SM's L2 port.  Whole layer at T = 128, top-8,
// d = 6144, 128 experts: 966 -> 947 us; T = 300, top-6, d = 2048, 64 experts: 110.3 -> 108.6.
constexpr int kFewRows = 32;
constexpr int kABytes = BM * kChunk * 2;           // 16 KiB per sub-tile and chunk
constexpr int kBBytesMax = 256 * kChunk * 2;       // 32 KiB

// Two forms of one kernel.
//   single (PAIR = false): one CTA computes a 128 x 256 tile (UMMA M x N, cta_group::1); K step 64;
//     4 stages of 48 KiB (A 16 KiB + B 32 KiB).  The mainloop needs 96 bytes per MMA cycle from L2.
//   pair (PAIR = true): a cluster of two CTAs computes a 256 x 256 tile with cta_group::2 MMAs
//     issued by the even CTA: each CTA stages its own 128 rows of A and HALF of the B tile (the
//     W1 tile in the even CTA and the W3 tile in the odd one in pass 1), so a CTA needs only
//     64 bytes per MMA cycle from L2.  No load is shared between the CTAs: each brings its own halves.  Used for
//     launches whose groups are large.  K step 64, 6 stages of 32 KiB, or with deep stages (DEEP) K step 128, two 64-element
//     chunks in one TMA instruction per operand (3-d maps), 3 stages of 64 KiB: a stage costs the producer and the
//     issuer a fixed few hundred cycles, whatever it holds.  The last tile of a group then shrinks to 128 rows, 64 per
//     CTA, where no more are valid.  Which of the two: pair_deep in feplb_create.
// Both keep two accumulators in TMEM so that the epilogue of tile i overlaps the MMAs of tile i+1.
template <bool PAIR, bool DEEP> struct Ring {
  static constexpr int kChunks = DEEP ? 2 : 1;
  static constexpr int BK = kChunks * kChunk;                                          // K elements per stage
  static constexpr int kStages = DEEP ? 3 : PAIR ? 6 : 4;
  static constexpr int kStageBytes = kChunks * (kABytes + (PAIR ? kBBytesMax / 2 : kBBytesMax));   // multiple of 1024
  static constexpr int kTileRows = PAIR ? 2 * BM : BM;
};
constexpr int kMaxStages = 6;
constexpr int kAccStages = 2;
constexpr int kRingBytes = 4 * (kABytes + kBBytesMax);   // 192 KiB in both forms
static_assert(Ring<false, false>::kStages * Ring<false, false>::kStageBytes == kRingBytes &&
              Ring<true, false>::kStages * Ring<true, false>::kStageBytes == kRingBytes &&
              Ring<true, true>::kStages * Ring<true, true>::kStageBytes == kRingBytes, "ring size");
constexpr int kEpiWarps = 4;
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr int kEpiStageBytes = 32 * 128;            // per epilogue warp: 32 rows x 64 bf16

struct SmemTail {
  unsigned long long full[kMaxStages];
  unsigned long long empty[kMaxStages];
  unsigned long long tmem_full[kAccStages];
  unsigned long long tmem_empty[kAccStages];
  unsigned long long dyn_bar;         // completed by warp 0 once the dynamic entries are in place
  uint32_t idesc[kMaxStages];         // deep stages: instruction descriptor of the tile whose first K block is in the stage (leader)
  uint32_t tmem_base;
  int abort_flag;
  int n_entries;                      // entries in use (the table known at launch, then the planner's dynamic groups)
  int total_mtiles;                   // prefix[n_entries]
  int prefix[FEPLB_MAX_GROUPS + 1];   // prefix[g] = M tiles of groups before g
  int g_row_start[FEPLB_MAX_GROUPS];
  int g_rows[FEPLB_MAX_GROUPS];
  int g_expert[FEPLB_MAX_GROUPS];
};
constexpr size_t kSmemBytes = 1024 /* alignment slack */ + (size_t)kRingBytes +
                              (size_t)kEpiWarps * kEpiStageBytes + sizeof(SmemTail);
static_assert(kSmemBytes <= 232448, "shared memory budget");
static_assert(kSmemBytes > 116 * 1024, "two CTAs must never share an SM: each allocates all of TMEM");

struct GemmParams {
  const feplb_group* groups;
  int n_groups;
  int which;            // FEPLB_FFN_*
  int E;
  int64_t s_cap;        // rows of the A and output buffers
  int n_tiles_n;        // N tiles per M tile
  int half_width;       // rows of B over all half tiles of one M tile: f (pass 1), d / 2 (pass 2); a multiple of 64
  int b_box;            // rows of one box of the B tensor maps (64 or 128), which divides every half tile; with deep stages a
                        // box has bn rows, and a narrow last tile leaves some of them unused
  int early_weights;    // the group table was complete before this kernel's predecessor let it start: B loads of the
                        // first tile may be issued before griddepcontrol.wait
  int num_k_blocks;     // K / 64, with deep stages K / 128 rounded up (the chunk past the end reads as zeros and is not multiplied)
  int num_chunks;       // K / 64
  int halves;           // deep stages: tiles of at most 128 valid rows take the 128-row MMA (in pass 1 it needs w13 ...
  int b_first;          // ... which begins at W3 where that lies in front of W1)
  int b_rows_per_expert;  // rows of one expert in the B tensor maps
  int n_recv_slots;     // slots of the receive buffer of migrated experts' weights (0 = none)
  int bn;               // rows of one B half tile (64 or 128; the last N tile may be narrower); the MMA has N = 2 * rows
  __nv_bfloat16* out;
  int ld_out;           // elements between output rows
  uint32_t* status;
  __nv_bfloat16* ab_out;   // pass 1, optional: pre-activations a | b saved for the backward pass ([rows, 2f])
  DynTable dyn;            // the planner's table of dynamic groups, walked after `groups` (dyn.seq == 0: none in this launch)
  unsigned long long* stamps;   // optional, preset to all ones, globaltimer ns: [0] first CTA's start, [1] first time a CTA
                                // ran out of static tiles, [2] ~(last CTA's end), [3] ~(longest wait for the dynamic table)
};


// Tensor maps of one pass: rows (whole boxes, fewer rows, receive region), the two halves of B, the same of the receive
// buffer, the output in boxes of 32 rows x 64 columns.
template <bool DEEP> struct Maps { CUtensorMap a, as, ra, b0, b1, r0, r1, out; };
template <> struct Maps<true> : Maps<false> { CUtensorMap w13; };     // pass 1: W1 and W3 together, for tiles of 128 rows

struct TileCoord { int row0, rows_valid, expert, slot, n0, bn; };   // slot >= 0: weights in that receive slot;
                                                                   // n0 = first column of the half tile, bn its rows

// tile -> (group, M tile, N tile); N tiles of one M tile are consecutive so that CTAs running at
// the same time share the A rows and sweep one expert's weights together (both stay in L2).
template <int kRows, bool NARROW>
__device__ __forceinline__ TileCoord tile_coord(const SmemTail* t, int n_groups, const GemmParams& p, int tile) {
  const int mt = tile / p.n_tiles_n;
  int lo = 0, hi = n_groups;   // largest g with prefix[g] <= mt
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (t->prefix[mid] <= mt) lo = mid; else hi = mid;
  }
  const int local = mt - t->prefix[lo];
  TileCoord c;
  c.row0 = t->g_row_start[lo] + local * kRows;
  c.rows_valid = min(kRows, t->g_rows[lo] - local * kRows);
  c.expert = t->g_expert[lo] & 0xffff;
  c.slot = (t->g_expert[lo] >> 16) - 1;
  c.n0 = (tile - mt * p.n_tiles_n) * p.bn;
  c.bn = NARROW ? min(p.bn, p.half_width - c.n0) : p.bn;
  return c;
}

// Pair form, deep stages: a tile of at most 128 valid rows is a 128 x 256 MMA over the two CTAs, 64 rows of A each.  In pass 1 both
// halves of B then hold W1 and W3 rows of the same 64 hidden units (see the producer), which takes a full-width tile.
// Half the MMA time and half the A rows against a 256-row tile whose second half is empty: 64 experts, d = 2048, T =
// 4096 (a third of the tiles) 345.9 -> 340.2 us per layer, three hot experts 355.9 -> 345.0.
template <bool SWIGLU, bool DEEP>
__device__ __forceinline__ bool is_half(const TileCoord& c, const GemmParams& p) {
  return DEEP && c.rows_valid <= BM && c.slot < 0 && p.halves && (!SWIGLU || c.bn == 128);
}

// fp32 accumulator registers of 32 columns -> 16 packed bf16 pairs (SwiGLU: silu(a) * b first).
template <bool SWIGLU>
__device__ __forceinline__ void convert_slice(const uint32_t (&a)[32], const uint32_t (&b)[32], uint32_t* packed) {
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    float v0 = __uint_as_float(a[2 * i]), v1 = __uint_as_float(a[2 * i + 1]);
    if (SWIGLU) {
      v0 = silu_f(v0) * __uint_as_float(b[2 * i]);
      v1 = silu_f(v1) * __uint_as_float(b[2 * i + 1]);
    }
    packed[i] = pack_bf16x2(v0, v1);
  }
}

// 32 rows x 64 bf16 columns, one row per lane in packed[32]: through the warp's staging area (row
// `lane`, 16-byte chunk j at position j ^ (lane & 7)) and out again 4 rows per instruction, so
// that every global store covers whole 128-byte lines; rows >= rows_here are not written.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* m, uint32_t src, int c0, int c1) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
               ::"l"(reinterpret_cast<uint64_t>(m)), "r"(src), "r"(c0), "r"(c1) : "memory");
}
// The warp's staging area may still be read by the TMA store of its previous slice.
__device__ __forceinline__ void staging_ready(int lane) {
  if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
  __syncwarp();
}

// Full slices (all 32 rows valid) leave through one TMA store: the staging layout below IS the
// 128-byte-swizzled box layout, so lane 0 hands the 4 KiB to the copy unit and the warp moves on.
__device__ __forceinline__ void stage_and_tma_store(uint32_t stg, const uint32_t* packed, const CUtensorMap* m, int gcol,
                                                    int grow, int lane) {
  staging_ready(lane);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint32_t addr = stg + (uint32_t)(lane * 128 + ((j ^ (lane & 7)) << 4));
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(packed[4 * j]), "r"(packed[4 * j + 1]),
                 "r"(packed[4 * j + 2]), "r"(packed[4 * j + 3]) : "memory");
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
  if (lane == 0) {
    tma_store_2d(m, stg, gcol, grow);
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
  }
}

__device__ __forceinline__ void stage_and_store(uint32_t stg, const uint32_t* packed, __nv_bfloat16* obase, int ld,
                                                int col, int rows_here, int lane) {
  const int rd_row = lane >> 3, rd_chunk = lane & 7;
  staging_ready(lane);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint32_t addr = stg + (uint32_t)(lane * 128 + ((j ^ (lane & 7)) << 4));
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(packed[4 * j]), "r"(packed[4 * j + 1]),
                 "r"(packed[4 * j + 2]), "r"(packed[4 * j + 3]) : "memory");
  }
  __syncwarp();
#pragma unroll
  for (int it = 0; it < 8; ++it) {
    const int r = it * 4 + rd_row;
    const uint32_t addr = stg + (uint32_t)(r * 128 + ((rd_chunk ^ (r & 7)) << 4));
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    if (r < rows_here) *reinterpret_cast<uint4*>(obase + (int64_t)r * ld + col + rd_chunk * 8) = v;
  }
  __syncwarp();
}

// One entry of a group table -> shared-memory arrays; returns its number of M tiles (0 if not selected).
template <int kRows>
__device__ __forceinline__ int put_group(SmemTail* t, int idx, int expert, int row_start, int rows, int is_dynamic, bool selected,
                                         const GemmParams& p) {
  int tiles = 0;
  if (selected && rows > 0) {
    const bool ok = expert >= 0 && expert < p.E && row_start >= 0 && (int64_t)row_start + rows <= p.s_cap &&
                    is_dynamic - 2 < p.n_recv_slots;
    if (ok) tiles = (rows + kRows - 1) / kRows;
    else atomicOr(p.status, FEPLB_ST_GROUP);
  }
  t->g_row_start[idx] = row_start;
  t->g_rows[idx] = rows;
  // expert id in the low half; receive slot + 1 in the high half (0 = weights at home)
  t->g_expert[idx] = (expert & 0xffff) | ((is_dynamic >= 2 ? is_dynamic - 1 : 0) << 16);
  return tiles;
}

// NARROW: the last N tile of a row of tiles has fewer columns than the others.  An instantiation of its own, because a
// width that differs per tile costs the roles more than it saves where it does not: both passes of a large batch in the
// single form, 64 experts, d = 2048, f = 768, 1536 / 3750 rows per expert on average: 950 / 2187 us with one kernel
// for all widths, 920 / 2118 this way; the pair form 864 / 1967 and 851 / 1938.
template <bool SWIGLU, bool PAIR, bool NARROW, bool DEEP>
__global__ void __launch_bounds__(kThreads, 1)
k_grouped_gemm(const __grid_constant__ Maps<DEEP> tm, const GemmParams p) {
  static_assert(PAIR || !DEEP, "deep stages: pair form only");
  using F = Ring<PAIR, DEEP>;
  constexpr int kStages = F::kStages, kStageBytes = F::kStageBytes, kTileRows = F::kTileRows, kChunks = F::kChunks, BK = F::BK;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* epi_smem = smem + (size_t)kRingBytes;
  // pair form: rank of this CTA in its cluster of two (0 = leader, issues the MMAs), work is dealt
  // per cluster; single form: every CTA is its own leader
  const uint32_t cta_rank = PAIR ? cluster_ctarank() : 0u;
  const int worker = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
  const int n_workers = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
  SmemTail* tail = reinterpret_cast<SmemTail*>(epi_smem + (size_t)kEpiWarps * kEpiStageBytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort_flag = &tail->abort_flag;

  // ---- set-up: barriers, TMEM, group table ------------------------------------------------
  if (threadIdx.x == 0) {
    prefetch_tmap(&tm.a);
    prefetch_tmap(&tm.as);
    prefetch_tmap(&tm.ra);
    prefetch_tmap(&tm.b0);
    prefetch_tmap(&tm.b1);
    prefetch_tmap(&tm.r0);
    prefetch_tmap(&tm.r1);
    prefetch_tmap(&tm.out);
    if constexpr (DEEP) prefetch_tmap(&tm.w13);
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_u32(&tail->full[s]), 1);
      mbar_init(smem_u32(&tail->empty[s]), 1);
    }
    for (int a = 0; a < kAccStages; ++a) {
      mbar_init(smem_u32(&tail->tmem_full[a]), 1);
      // one arrival per epilogue warp (of both CTAs in the pair form: the leader's barrier collects them)
      mbar_init(smem_u32(&tail->tmem_empty[a]), PAIR ? 2 * kEpiWarps : kEpiWarps);
    }
    mbar_init(smem_u32(&tail->dyn_bar), 1);
    tail->abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 1) {
    __syncwarp();
    if (PAIR) {
      tmem_alloc_pair(smem_u32(&tail->tmem_base), kTmemCols);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(smem_u32(&tail->tmem_base), kTmemCols);
      tmem_relinquish();
    }
  }
  // Everything above touched only this CTA's resources; from here on the results of the kernels before
  // this one are read -- except, with early_weights, by the producer's first weight loads and the reads of
  // the group table: the kernel before this one had itself waited for the table's writer when it let this
  // one start.  For the same reason this kernel lets its successor start only after its own wait.
  if (!p.early_weights) asm volatile("griddepcontrol.wait;" ::: "memory");
  if (p.stamps && !p.early_weights && threadIdx.x == 0) atomicMin(&p.stamps[0], global_timer_ns());
  for (int g = threadIdx.x; g < p.n_groups; g += kThreads) {
    const feplb_group gr = p.groups[g];
    const bool selected = p.which == FEPLB_FFN_ALL || (p.which == FEPLB_FFN_STATIC) == (gr.is_dynamic == 0);
    tail->prefix[g + 1] = put_group<kTileRows>(tail, g, gr.expert, gr.row_start, gr.rows, gr.is_dynamic, selected, p);   // scanned below
  }
  if (threadIdx.x == 0) tail->prefix[0] = 0;
  const bool early = dyn_is_early(p.dyn);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    const int n = !early ? p.n_groups : dyn_merge_table(
        p.dyn, p.n_groups, FEPLB_MAX_GROUPS, p.status, lane,
        [&](int e, int rs) { return tail->g_row_start[e] == rs && tail->prefix[e + 1] == 0; },
        [&](int i, int e, int rs, int rw, int dy) { tail->prefix[i + 1] = put_group<kTileRows>(tail, i, e, rs, rw, dy, true, p); });
    warp_scan_prefix(tail->prefix, 0, n, lane);
    if (lane == 0) {
      tail->n_entries = n;
      tail->total_mtiles = tail->prefix[n];
    }
  }
  __syncthreads();
  if (PAIR) cluster_sync_all();   // the peer's barriers are initialised before anything signals them
  tc_fence_after();
  const uint32_t tmem_base = tail->tmem_base;
  const bool has_dyn = p.dyn.seq != 0 && !early;
  const int n_static_entries = early ? tail->n_entries : p.n_groups;
  const int n_static_tiles = tail->prefix[n_static_entries] * p.n_tiles_n;
  // (the producer waits on its own, after its first weight loads)
  if (p.early_weights && warp != 0) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (p.stamps && threadIdx.x == 32) atomicMin(&p.stamps[0], global_timer_ns());
  }
  if (warp != 0) asm volatile("griddepcontrol.launch_dependents;");

  if (warp == 0) {
    // ---- TMA producer (lane 0 issues; the whole warp fetches the dynamic table) ----------------
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true, dyn_known = !has_dyn;
    int n_entries = n_static_entries, total = n_static_tiles;
    // Reads the n_dyn groups of the dynamic table from its device copy, appends its entries and tells
    // the other roles; false if an entry does not carry this forward's sequence number yet.
    auto take_table = [&](int n_dyn) -> bool {
      if (n_dyn < 0 || n_static_entries + n_dyn > FEPLB_MAX_GROUPS) {
        if (lane == 0) atomicOr(p.status, FEPLB_ST_GROUP);
        n_dyn = 0;
      }
      bool good = true;
      for (int i = lane; i < n_dyn; i += 32) {
        int e, rs, rw, dy;
        if (!dyn_entry(p.dyn, i, e, rs, rw, dy)) { good = false; continue; }
        tail->prefix[n_static_entries + i + 1] = put_group<kTileRows>(tail, n_static_entries + i, e, rs, rw, dy, true, p);
      }
      if (!__all_sync(0xffffffffu, good)) return false;
      warp_scan_prefix(tail->prefix, n_static_entries, n_dyn, lane);
      n_entries = n_static_entries + n_dyn;
      total = tail->prefix[n_entries] * p.n_tiles_n;
      if (lane == 0) {
        tail->n_entries = n_entries;
        tail->total_mtiles = tail->prefix[n_entries];
        mbar_arrive(smem_u32(&tail->dyn_bar));      // release: the entries above are visible to the waiters
      }
      dyn_known = true;
      return true;
    };
    // What a tile's K blocks are loaded from, worked out once per tile and not in the K loop, which runs in one thread
    // beside the MMA issuer (d = 1920, f = 704, 60 experts, T = 1537: 148.7 -> 145.1 us per layer).
    // Pair form: both CTAs credit the LEADER's barrier; the leader announces the bytes of both.  For a tile whose
    // second 128 rows hold no valid row (a group of at most 128 rows, or a ragged tail) the peer's A box lies past
    // the end of the tensor and brings zeros (the counter of bytes from L2 to the SMs counts them like rows: 1.53 ->
    // 1.65 GB in pass 1).  Multiplying zeros takes less power than multiplying what a skipped load would leave in the
    // stage, which is clock at the power cap (64 experts, d = 2048, T = 4096: 343.2 -> 337.1 us per layer).  Zeros for the partly valid 128 rows as well, by boxes of 32 rows, cost
    // 4 % instead.
    struct Source { const CUtensorMap *a, *b0, *b1; int arow, brow0, brow1; uint32_t half, tx, idesc; bool two, split; };
    auto source = [&](const TileCoord& c) {
      Source q;
      const bool few = !PAIR && c.slot < 0 && c.rows_valid <= kFewRows;
      // weights of a migrated expert come from its slot of the receive buffer, and in pass 1 its rows from the
      // receive region (same row numbers as the permuted buffer)
      q.a = c.slot >= 0 ? &tm.ra : few ? &tm.as : &tm.a;
      q.b0 = c.slot >= 0 ? &tm.r0 : &tm.b0;
      q.b1 = c.slot >= 0 ? &tm.r1 : &tm.b1;
      q.arow = c.row0;
      q.brow0 = (c.slot >= 0 ? c.slot : c.expert) * p.b_rows_per_expert + (SWIGLU ? c.n0 : 2 * c.n0);
      q.brow1 = SWIGLU ? q.brow0 : q.brow0 + c.bn;
      q.half = (uint32_t)(DEEP ? p.bn : c.bn) * BK * 2;
      q.two = !DEEP && NARROW && c.bn > p.b_box;    // 128 rows in boxes of 64
      q.tx = (PAIR ? 2 * kChunks * kABytes : few ? kFewRows * kChunk * 2 : kABytes) + 2 * q.half;
      if (PAIR && cta_rank) {
        q.arow = c.rows_valid > BM ? c.row0 + BM : (int)p.s_cap;
        q.b0 = q.b1;
        q.brow0 = q.brow1;
      }
      q.idesc = make_idesc(kTileRows, 2 * c.bn);
      q.split = false;
      if (is_half<SWIGLU, DEEP>(c, p)) {
        // 64 rows of A per CTA (zeros where none of them is valid); pass 1: 64 rows of W1 and the same 64 of W3
        q.a = &tm.as;
        q.arow = !cta_rank ? c.row0 : c.rows_valid > BM / 2 ? c.row0 + BM / 2 : (int)p.s_cap;
        q.tx = kChunks * kABytes + 2 * q.half;
        q.idesc = make_idesc(BM, 2 * c.bn);
        q.split = SWIGLU;
        if (SWIGLU) q.brow0 = c.expert * p.b_rows_per_expert + c.n0 + (int)cta_rank * 64;
      }
      return q;
    };
    auto announce = [&](const Source& q, int st) {      // the bytes of a stage, and what the issuer does with them
      if (PAIR && cta_rank) return;
      if (DEEP) tail->idesc[st] = q.idesc;
      mbar_expect_tx(smem_u32(&tail->full[st]), q.tx);
    };
    auto load_b = [&](const Source& q, int kb, uint32_t full, uint32_t sb) {
      constexpr uint32_t kBox = 64 * BK * 2;
      if constexpr (DEEP) {
        const uint32_t full0 = map_to_cta(full, 0);
        if (SWIGLU && q.split)      // 64 rows of W1 and of W3, chunk after chunk
          asm volatile(
              "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %3, %5}], [%2];"
              ::"r"(sb), "l"(reinterpret_cast<uint64_t>(&tm.w13)), "r"(full0), "r"(0), "r"(q.brow0), "r"(kb * kChunks) : "memory");
        else
          tma_load_3d_pair(sb, q.b0, full0, 0, q.brow0, kb * kChunks);
      } else if (PAIR) {
        const uint32_t full0 = map_to_cta(full, 0);
        tma_load_2d_pair(sb, q.b0, full0, kb * BK, q.brow0);
        if (q.two) tma_load_2d_pair(sb + kBox, q.b0, full0, kb * BK, q.brow0 + 64);
      } else {
        tma_load_2d(sb, q.b0, full, kb * BK, q.brow0);
        tma_load_2d(sb + q.half, q.b1, full, kb * BK, q.brow1);
        if (q.two) {
          tma_load_2d(sb + kBox, q.b0, full, kb * BK, q.brow0 + 64);
          tma_load_2d(sb + q.half + kBox, q.b1, full, kb * BK, q.brow1 + 64);
        }
      }
    };
    auto load_a = [&](const Source& q, int kb, uint32_t full, uint32_t sa) {
      if (DEEP) tma_load_3d_pair(sa, q.a, map_to_cta(full, 0), 0, q.arow, kb * kChunks);
      else if (PAIR) tma_load_2d_pair(sa, q.a, map_to_cta(full, 0), kb * BK, q.arow);
      else tma_load_2d(sa, q.a, full, kb * BK, q.arow);
    };
    // Weights of the first tile, as far as the ring holds them, before the wait for the rows.
    int n_early = 0;
    if (p.early_weights) {
      if (worker < n_static_tiles) {
        n_early = min(kStages, p.num_k_blocks);
        if (lane == 0) {
          const Source q = source(tile_coord<kTileRows, NARROW>(tail, n_entries, p, worker));
          for (int kb = 0; kb < n_early; ++kb) {
            announce(q, kb);
            load_b(q, kb, smem_u32(&tail->full[kb]), smem_u32(smem + (size_t)kb * kStageBytes) + kChunks * kABytes);
          }
        }
        __syncwarp();
      }
      asm volatile("griddepcontrol.wait;" ::: "memory");
    }
    asm volatile("griddepcontrol.launch_dependents;");
    bool claimer = false, tried_claim = false;
    for (int tile = worker; ok; tile += n_workers) {
      if (!dyn_known && tile >= total) {
        // Out of static tiles: now the table is needed (bounded wait; see feplb_dyn.cuh).
        const unsigned long long t0 = global_timer_ns();
        if (p.stamps && lane == 0) atomicMin(&p.stamps[1], t0);
        while (!dyn_known) {
          const int n_dyn = dyn_wait_table(p.dyn, lane, abort_flag, p.status, t0, claimer, tried_claim);
          if (n_dyn == kDynAbort) { ok = false; break; }
          // no table within the limit: go on as if it were empty, so that the static tiles still in
          // flight in this CTA complete normally; the status word carries the reason
          if (!take_table(n_dyn == kDynGaveUp ? 0 : n_dyn) && global_timer_ns() - t0 > p.dyn.wait_limit_ns + kWaitLimitNs) {
            if (lane == 0) atomicOr(p.status, FEPLB_ST_PLAN);
            take_table(0);
          }
        }
        if (!ok) break;
        if (p.stamps && lane == 0) atomicMin(&p.stamps[3], ~(global_timer_ns() - t0));
      }
      if (tile >= total) break;
      const TileCoord c = tile_coord<kTileRows, NARROW>(tail, n_entries, p, tile);
      // While static tiles remain, peek at the device-side word once per tile: the load is in flight
      // during the K loop below and is looked at after it, so it costs the pipeline nothing.
      unsigned long long peek = 0;
      if (!dyn_known && lane == 0) peek = ld_relaxed_gpu_u64(p.dyn.ready_dev);
      if (lane == 0) {
        const Source q = source(c);
        int kb = 0;
        for (; kb < n_early; ++kb) {       // stages 0 .. n_early - 1, whose weights are on their way
          load_a(q, kb, smem_u32(&tail->full[stage]), smem_u32(smem + (size_t)stage * kStageBytes));
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
        for (; kb < p.num_k_blocks; ++kb) {
          if (!(ok = mbar_wait(smem_u32(&tail->empty[stage]), phase ^ 1u, abort_flag, p.status))) break;
          const uint32_t full = smem_u32(&tail->full[stage]);
          const uint32_t sa = smem_u32(smem + (size_t)stage * kStageBytes);
          announce(q, stage);
          load_a(q, kb, full, sa);
          load_b(q, kb, full, sa + kChunks * kABytes);
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
      }
      n_early = 0;
      ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
      if (ok && !dyn_known) {
        peek = __shfl_sync(0xffffffffu, peek, 0);
        if (dyn_peek_count(p.dyn, peek) >= 0) take_table(dyn_peek_count(p.dyn, peek));
      }
    }
    if (!ok && lane == 0) {
      // leave time for copies already issued to land before the CTA's shared memory goes away
      for (int i = 0; i < 2000; ++i) __nanosleep(100);
    }
  } else if (warp == 1) {
    // ---- MMA issuer -------------------------------------------------------------------------
    if (lane == 0 && cta_rank == 0) {
      uint32_t idesc = make_idesc(kTileRows, 2 * p.bn);
      // between the chunks of a stage's A (64 rows in a tile of 128) and B, >> 4
      uint32_t a_chunk = kABytes >> 4;
      const uint32_t b_chunk = (uint32_t)(p.bn * kChunk * 2) >> 4;
      int stage = 0, as = 0;
      uint32_t phase = 0, aphase = 0;
      bool ok = true, dyn_known = !has_dyn;
      int total = n_static_tiles;
      for (int tile = worker; ok; tile += n_workers) {
        if (tile >= total) {
          if (dyn_known) break;
          if (!(ok = mbar_wait(smem_u32(&tail->dyn_bar), 0, abort_flag, p.status, p.dyn.wait_limit_ns + 2 * kWaitLimitNs))) break;
          dyn_known = true;
          total = tail->total_mtiles * p.n_tiles_n;
          if (tile >= total) break;
        }
        if (!DEEP && NARROW) idesc = make_idesc(kTileRows, 2 * min(p.bn, p.half_width - tile % p.n_tiles_n * p.bn));
        if (!(ok = mbar_wait(smem_u32(&tail->tmem_empty[as]), aphase ^ 1u, abort_flag, p.status))) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(as * kAccCols);
        for (int kb = 0; kb < p.num_k_blocks; ++kb) {
          if (!(ok = mbar_wait(smem_u32(&tail->full[stage]), phase, abort_flag, p.status))) break;
          tc_fence_after();
          if (DEEP && kb == 0) {
            idesc = *reinterpret_cast<volatile uint32_t*>(&tail->idesc[stage]);
            a_chunk = idesc >> 24 == BM >> 4 ? kABytes / 2 >> 4 : kABytes >> 4;
          }
          const uint32_t sa = smem_u32(smem + (size_t)stage * kStageBytes);
          const uint64_t da = make_smem_desc(sa);
          const uint64_t db = make_smem_desc(sa + kChunks * kABytes);
#pragma unroll
          for (int k = 0; k < BK / UMMA_K; ++k) {
            // +32 bytes (>> 4 = 2) per K step inside the 128-byte swizzle row
            const int ch = k / (kChunk / UMMA_K), ks = 2 * (k % (kChunk / UMMA_K));
            if (ch > 0 && kb * kChunks + ch >= p.num_chunks) break;
            if (PAIR) umma_bf16_pair(d_tmem, da + (uint64_t)(ch * a_chunk + ks), db + (uint64_t)(ch * b_chunk + ks), idesc, (uint32_t)((kb | k) != 0));
            else umma_bf16(d_tmem, da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), idesc, (uint32_t)((kb | k) != 0));
          }
          // stage reusable (in both CTAs of a pair) once these MMAs have read it
          if (PAIR) umma_commit_pair(smem_u32(&tail->empty[stage]));
          else umma_commit(smem_u32(&tail->empty[stage]));
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        // accumulator complete (announced to the epilogue warps of both CTAs of a pair)
        if (PAIR) umma_commit_pair(smem_u32(&tail->tmem_full[as]));
        else umma_commit(smem_u32(&tail->tmem_full[as]));
        if (++as == kAccStages) { as = 0; aphase ^= 1u; }
      }
    }
  } else {
    // ---- epilogue: TMEM -> registers -> bf16 -> (warp-private smem transpose) -> global -------
    // A thread owns one accumulator row, so storing straight from registers would scatter 16-byte
    // pieces over 32 rows per instruction.  Instead each warp stages 32 rows x 64 columns (128 B
    // per row, 16-byte chunks XOR-swizzled by row) and writes them back out 4 rows per
    // instruction: every store covers whole 128-byte lines, masked per row for ragged tiles.
    const int q = warp & 3;                   // TMEM lane quarter this warp may read
    const uint32_t stg = smem_u32(epi_smem + (size_t)(warp - 2) * kEpiStageBytes);
    int as = 0;
    uint32_t aphase = 0;
    bool ok = true, dyn_known = !has_dyn;
    int n_entries = n_static_entries, total = n_static_tiles;
    for (int tile = worker; ok; tile += n_workers) {
      if (tile >= total) {
        if (dyn_known) break;
        ok = mbar_wait(smem_u32(&tail->dyn_bar), 0, abort_flag, p.status, p.dyn.wait_limit_ns + 2 * kWaitLimitNs);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        dyn_known = true;
        n_entries = tail->n_entries;
        total = tail->total_mtiles * p.n_tiles_n;
        if (tile >= total) break;
      }
      const TileCoord c = tile_coord<kTileRows, NARROW>(tail, n_entries, p, tile);
      // In a tile of 128 rows over two CTAs TMEM lanes 0-63 hold the CTA's 64 rows for the columns of the even CTA's half
      // of B, lanes 64-127 the same rows for those of the odd CTA's.
      const bool half = is_half<SWIGLU, DEEP>(c, p);
      // pass 1: TMEM columns of a and of b
      const uint32_t a_off = SWIGLU && half && p.b_first ? 64 : 0, b_off = half ? 64 - a_off : (uint32_t)c.bn;
      const int out_cols = half ? (SWIGLU ? 64 : c.bn) : SWIGLU ? c.bn : 2 * c.bn;
      const int col0 = (SWIGLU ? c.n0 : 2 * c.n0) + (half ? (q >> 1) * out_cols : 0);   // this warp's first output column
      ok = mbar_wait(smem_u32(&tail->tmem_full[as]), aphase, abort_flag, p.status);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(as * kAccCols);
      const int row_off = half ? (int)cta_rank * (BM / 2) + (q & 1) * 32 : (int)cta_rank * BM + q * 32;    // this warp's first row inside the tile
      const int rows_here = c.rows_valid - row_off;       // valid rows among this warp's 32
      __nv_bfloat16* obase = p.out + (int64_t)(c.row0 + row_off) * p.ld_out + col0;
      // Single form: a warp without valid rows only hands the accumulator back.  In the pair form, which has few of them,
      // this test costs more than it saves: d = 6144, T = 65536 35344 us per layer with it, 34903 without.
      if (PAIR || rows_here > 0) {
        uint32_t a0[32], a1[32], b0[32], b1[32], packed[32];
        tmem_ld32(taddr + a_off, a0);
        tmem_ld32(taddr + a_off + 32u, a1);
        if (SWIGLU) {
          tmem_ld32(taddr + b_off, b0);
          tmem_ld32(taddr + b_off + 32u, b1);
        }
        for (int col = 0; col < out_cols; col += 64) {
          tmem_ld_wait();
          if (SWIGLU && p.ab_out != nullptr) {
            // training: also keep the pre-activations a | b of these 64 hidden units (bf16) for the
            // backward pass, in [rows, 2f] with b at column offset f
            __nv_bfloat16* abase = p.ab_out + (int64_t)(c.row0 + row_off) * (2 * p.ld_out);
            const int hcol = col0 + col;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              packed[i] = pack_bf16x2(__uint_as_float(a0[2 * i]), __uint_as_float(a0[2 * i + 1]));
              packed[16 + i] = pack_bf16x2(__uint_as_float(a1[2 * i]), __uint_as_float(a1[2 * i + 1]));
            }
            stage_and_store(stg, packed, abase, 2 * p.ld_out, hcol, rows_here, lane);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              packed[i] = pack_bf16x2(__uint_as_float(b0[2 * i]), __uint_as_float(b0[2 * i + 1]));
              packed[16 + i] = pack_bf16x2(__uint_as_float(b1[2 * i]), __uint_as_float(b1[2 * i + 1]));
            }
            stage_and_store(stg, packed, abase, 2 * p.ld_out, p.ld_out + hcol, rows_here, lane);
          }
          convert_slice<SWIGLU>(a0, b0, packed);
          convert_slice<SWIGLU>(a1, b1, packed + 16);
          if (col + 64 < out_cols) {           // next slice's TMEM loads fly while this one is stored
            tmem_ld32(taddr + a_off + (uint32_t)(col + 64), a0);
            tmem_ld32(taddr + a_off + (uint32_t)(col + 96), a1);
            if (SWIGLU) {
              tmem_ld32(taddr + b_off + (uint32_t)(col + 64), b0);
              tmem_ld32(taddr + b_off + (uint32_t)(col + 96), b1);
            }
          }
          if (rows_here >= 32) stage_and_tma_store(stg, packed, &tm.out, col0 + col, c.row0 + row_off, lane);
          else stage_and_store(stg, packed, obase, p.ld_out, col, rows_here, lane);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (PAIR) mbar_arrive_cluster(map_to_cta(smem_u32(&tail->tmem_empty[as]), 0));
        else mbar_arrive(smem_u32(&tail->tmem_empty[as]));
      }
      if (++as == kAccStages) { as = 0; aphase ^= 1u; }
    }
    staging_ready(lane);      // the staging area must outlive the last TMA store that reads it
  }

  // ---- teardown ---------------------------------------------------------------------------------
  tc_fence_before();
  __syncthreads();
  if (p.stamps && threadIdx.x == 0) atomicMin(&p.stamps[2], ~global_timer_ns());
  if (PAIR) cluster_sync_all();   // the leader's MMAs read the peer's shared memory: leave together
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    if (PAIR) tmem_dealloc_pair(tmem_base, kTmemCols);
    else tmem_dealloc(tmem_base, kTmemCols);
  }
}

// Self-test of the bounded wait: one thread waits on an mbarrier that nothing will ever complete.
// The wait must give up after limit_ns, raise FEPLB_ST_WAIT and let the kernel return normally.
__global__ void k_wait_selftest(uint32_t* status, unsigned long long limit_ns, int* gave_up) {
  __shared__ unsigned long long bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    mbar_init(smem_u32(&bar), 1);
    fence_barrier_init();
    const bool ok = mbar_wait(smem_u32(&bar), 0, &abort_flag, status, limit_ns);
    *gave_up = ok ? 0 : 1;
  }
}

// ------------------------------------------------------------------------------------------ host

// Row-major bf16 matrix [rows, inner] -> tensor map with a [box_rows, 64] box, 128-byte swizzle.
bool make_tmap(CUtensorMap* m, const void* base, uint64_t rows, uint64_t inner, uint32_t box_rows) {
  const cuuint64_t dims[2] = {inner, rows}, strides[1] = {inner * 2};
  const cuuint32_t box[2] = {(cuuint32_t)kChunk, box_rows};
  return encode_tmap(m, 2, base, dims, strides, box);
}
// 64 rows of W1 and the same 64 of W3, two chunks: {64 columns, rows, W1 and W3, chunks}.
bool make_tmap_w13_tile(CUtensorMap* m, const void* w1, const void* w3, uint64_t rows, uint64_t inner) {
  const uint64_t apart = w13_apart(w1, w3);
  const cuuint64_t dims[4] = {(cuuint64_t)kChunk, rows, 2, inner / kChunk}, strides[3] = {inner * 2, apart, kChunk * 2};
  const cuuint32_t box[4] = {(cuuint32_t)kChunk, 64, 2, 2};
  return apart && encode_tmap(m, 4, w1 < w3 ? w1 : w3, dims, strides, box);
}

template <bool SWIGLU, bool PAIR, bool NARROW, bool DEEP>
cudaError_t launch_form(const Maps<DEEP>& m, const GemmParams& p, int num_sms, cudaStream_t st) {
  // per instantiation and device: the shared-memory attribute and the resident grid are set on first use
  static int grid_of[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  int& grid = grid_of[dev];
  const auto kernel = k_grouped_gemm<SWIGLU, PAIR, NARROW, DEEP>;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (PAIR) {
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = 2;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.numAttrs = 2;
  }
  if (!grid) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
    if (e != cudaSuccess) return e;
    int g = num_sms;
    if (PAIR) {
      // as many clusters of two as can be resident at once (one CTA per SM, both SMs in one GPC)
      int n_clusters = 0;
      cfg.gridDim = dim3(num_sms / 2 * 2);
      e = cudaOccupancyMaxActiveClusters(&n_clusters, kernel, &cfg);
      if (e != cudaSuccess) return e;
      if (n_clusters < 1) return cudaErrorLaunchOutOfResources;
      g = 2 * (n_clusters < num_sms / 2 ? n_clusters : num_sms / 2);
    }
    grid = g;
  }
  cfg.gridDim = dim3(grid);
  return cudaLaunchKernelEx(&cfg, kernel, m, p);
}

template <bool SWIGLU>
cudaError_t launch_one(const Maps<true>& m, const GemmParams& p, bool pair, bool deep, int num_sms, cudaStream_t st) {
  const bool narrow = p.half_width % p.bn != 0;
  if (!pair) return (narrow ? launch_form<SWIGLU, false, true, false> : launch_form<SWIGLU, false, false, false>)(m, p, num_sms, st);
  if (!deep) return (narrow ? launch_form<SWIGLU, true, true, false> : launch_form<SWIGLU, true, false, false>)(m, p, num_sms, st);
  return (narrow ? launch_form<SWIGLU, true, true, true> : launch_form<SWIGLU, true, false, true>)(m, p, num_sms, st);
}

}  // namespace

int feplb_launch_expert_ffn(const feplb_gemm_args& a, cudaStream_t st, int64_t* n_launch, char* err, size_t errn,
                            const feplb_wm_dyn* dyn) {
  if ((a.n_groups == 0 && !(dyn && dyn->seq)) || a.s_cap == 0) return FEPLB_OK;
  if (dyn && a.n_groups + dyn->max_groups > FEPLB_MAX_GROUPS) {
    snprintf(err, errn, "expert_ffn: the two group tables of a merged launch exceed %d entries", FEPLB_MAX_GROUPS);
    return FEPLB_E_INVALID;
  }
  // Half tiles of up to 128 rows of B (columns of H in pass 1, half the columns of Y in pass 2).  Where the
  // width is not a multiple of 128 the last N tile is narrower, and boxes of 64 rows serve both: a 128 x 256
  // tile moves 48 KiB per 512 MMA cycles into the SM, two 128 x 128 tiles (64-row half tiles throughout,
  // as narrow widths such as 64 still have) 64 KiB.  Whole layer at d = 1920, f = 704, E = 60, T = 1537,
  // top-4: 171.2 -> 150.9 us together with the early weight loads of pass 2.
  const int hw1 = a.f, hw2 = a.d / 2;
  const int bn1 = hw1 < 128 ? 64 : 128, bn2 = hw2 < 128 ? 64 : 128;
  const bool deep = a.pair && a.deep;
  const int bb1 = deep ? bn1 : hw1 % 128 ? 64 : 128, bb2 = deep ? bn2 : hw2 % 128 ? 64 : 128;
  const auto map = deep ? make_tmap_chunks : make_tmap;
  const int few = a.pair ? BM / 2 : kFewRows;            // rows of the smaller boxes of A
  const uint64_t rows = (uint64_t)a.s_cap, w1_rows = (uint64_t)a.E * a.f, w2_rows = (uint64_t)a.E * a.d, d = (uint64_t)a.d, f = (uint64_t)a.f;
  Maps<true> m1, m2;
  if (!map(&m1.a, a.x_perm, rows, d, BM) || !map(&m1.as, a.x_perm, rows, d, few) || !map(&m1.b0, a.w1, w1_rows, d, bb1) ||
      !map(&m1.b1, a.w3, w1_rows, d, bb1) || !map(&m2.a, a.h, rows, f, BM) || !map(&m2.as, a.h, rows, f, few) ||
      !map(&m2.b0, a.w2, w2_rows, f, bb2) || !make_tmap(&m1.out, a.h, rows, f, 32) || !make_tmap(&m2.out, a.y, rows, d, 32)) {
    snprintf(err, errn, "cuTensorMapEncodeTiled failed (driver entry point missing or bad pointer/shape)");
    return FEPLB_E_CUDA;
  }
  m2.b1 = m2.w13 = m2.b0;
  m1.w13 = m1.b0;
  const bool halves = deep && make_tmap_w13_tile(&m1.w13, a.w1, a.w3, w1_rows, d);
  // receive buffer of migrated experts' weights, addressed by slot like the home weights by expert, and the rows of
  // migrated pieces: pass 1 reads them from the receive region when there is one
  m1.r0 = m1.b0; m1.r1 = m1.b1; m2.r0 = m2.b0; m1.ra = m1.a; m2.ra = m2.a;
  const bool has_recv = a.recv_w1 && a.recv_w3 && a.recv_w2 && a.n_recv_slots > 0;
  const uint64_t slots = (uint64_t)a.n_recv_slots;
  if (has_recv && (!map(&m1.r0, a.recv_w1, slots * f, d, bb1) || !map(&m1.r1, a.recv_w3, slots * f, d, bb1) ||
                   !map(&m2.r0, a.recv_w2, slots * d, f, bb2) || (a.recv_x && !map(&m1.ra, a.recv_x, rows, d, BM)))) {
    snprintf(err, errn, "cuTensorMapEncodeTiled failed for the receive buffer");
    return FEPLB_E_CUDA;
  }
  m2.r1 = m2.r0;
  GemmParams p1;
  p1.n_recv_slots = has_recv ? a.n_recv_slots : 0;
  p1.groups = a.groups; p1.n_groups = a.n_groups; p1.which = a.which; p1.E = a.E; p1.s_cap = a.s_cap;
  p1.n_tiles_n = (hw1 + bn1 - 1) / bn1; p1.half_width = hw1; p1.b_box = bb1; p1.early_weights = 0;
  const int chunks = deep ? 2 : 1;
  p1.halves = halves; p1.b_first = a.w3 < a.w1;
  p1.num_k_blocks = (a.d / kChunk + chunks - 1) / chunks; p1.num_chunks = a.d / kChunk; p1.b_rows_per_expert = a.f; p1.bn = bn1;
  p1.out = (__nv_bfloat16*)a.h; p1.ld_out = a.f; p1.status = a.status; p1.ab_out = (__nv_bfloat16*)a.ab_out;
  const feplb_wm_dyn none;
  p1.dyn = feplb_dyn_table(dyn ? *dyn : none);
  p1.stamps = dyn ? dyn->stamps : nullptr;
  GemmParams p2 = p1;
  p2.n_tiles_n = (hw2 + bn2 - 1) / bn2; p2.half_width = hw2; p2.b_box = bb2; p2.early_weights = 1;
  p2.halves = 1;
  p2.num_k_blocks = (a.f / kChunk + chunks - 1) / chunks; p2.num_chunks = a.f / kChunk; p2.b_rows_per_expert = a.d; p2.bn = bn2;
  p2.out = (__nv_bfloat16*)a.y; p2.ld_out = a.d; p2.ab_out = nullptr;
  p2.stamps = p1.stamps ? p1.stamps + 4 : nullptr;

  cudaError_t e = launch_one<true>(m1, p1, a.pair, deep, a.num_sms, st);
  ++*n_launch;
  if (e == cudaSuccess) {
    e = launch_one<false>(m2, p2, a.pair, deep, a.num_sms, st);
    ++*n_launch;
  }
  if (e != cudaSuccess) {
    snprintf(err, errn, "k_grouped_gemm launch: %s", cudaGetErrorString(e));
    return FEPLB_E_CUDA;
  }
  return FEPLB_OK;
}

cudaError_t feplb_launch_wait_selftest(uint32_t* status, unsigned long long limit_ns, int* gave_up, cudaStream_t st) {
  k_wait_selftest<<<1, 32, 0, st>>>(status, limit_ns, gave_up);
  return cudaGetLastError();
}
