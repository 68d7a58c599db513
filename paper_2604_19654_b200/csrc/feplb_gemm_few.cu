// Grouped SwiGLU expert FFN for batches that bring an expert few rows each (decode), for sm_100a (paper Section 2.3:
// the expert Grouped GEMM; Section 3.1: its cost depends strongly on the per-expert batch size).
//
// Such a batch lives on how fast the weights of the touched experts stream in, and two things besides the loads
// themselves decide that: how many bytes are in flight, and the power that the tensor cores burn on padding (a memory-bound
// launch at the power cap runs its L2 and its SMs at a lower clock too).  So weight rows are on the M side of the
// MMA and the token rows, padded to 16, on the N side:
//
//   unit   = (row block of one group: n <= NMAX rows) x (128 weight rows of the group's expert), one CTA
//   pass 1 : 64 rows of W1[e] and the same 64 of W3[e], 16 of the one and 16 of the other in turn, so that each warp's
//            quarter of TMEM holds a = x W1 in its lower and b = x W3 of the same hidden units in its upper 16
//            lanes, and one thread reads both;  H = silu(a) * b
//   pass 2 : 128 rows of W2[e];  Y = H W2
//
// A stage holds 128 elements of K: 32 KiB of weights in one TMA instruction (pass 1 through a map whose third dimension
// leads from W1 to W3), the token rows in another.  NMAX decides between weights in flight and weights read again: units of
// at most 32, 64 or 128 token rows leave room for five, four or three stages, i.e. 160, 128 or 96 KiB of weights per
// SM (few_rows in feplb_api.cu has the measurements).  Pass 2 starts with
// the weights of its first unit before it waits for pass 1.  Per CTA: warp 0 = TMA producer, warp 1 = tcgen05.mma
// issuer and TMEM owner, warps 2..5 or 2..9 = epilogue.  Every wait is bounded and ends in a status bit, a clean TMEM
// release and a normal return.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdio>

#include "feplb_internal.h"
#include "feplb_tc.cuh"

namespace {

constexpr int UMMA_K = 16;
constexpr int kChunk = 64;                          // K elements of a 128-byte swizzle row
constexpr int BK = 2 * kChunk;                      // K elements per stage
constexpr int kWRows = 128;                         // weight rows per unit
constexpr int kWBytes = kWRows * BK * 2;            // 32 KiB
// NMAX: most token rows per unit (UMMA N); they come in boxes of NMAX, NMAX / 2, ... 16 rows
template <int NMAX> struct Form {
  static constexpr int kStages = NMAX == 32 ? 5 : NMAX == 64 ? 4 : 3;
  static constexpr int kStageBytes = kWBytes + NMAX * BK * 2;     // 40, 48, 64 KiB
  static constexpr int kBoxes = NMAX == 32 ? 2 : NMAX == 64 ? 3 : 4;
  static constexpr int kTmemCols = 2 * NMAX;                      // two accumulators
  static constexpr int kEpiWarps = NMAX == 128 ? 8 : 4;           // one warp, or two, per TMEM lane quarter
  static constexpr int kThreads = 64 + 32 * kEpiWarps;
};
constexpr int kMaxStages = 5;
constexpr int kMaxBoxes = 4;
constexpr int kEpiStageBytes = 32 * 64;             // per epilogue warp: 32 tokens x 32 columns of bf16

struct Tail {
  unsigned long long full[kMaxStages], empty[kMaxStages];
  unsigned long long tmem_full[2], tmem_empty[2];
  uint32_t tmem_base;
  int abort_flag;
  int prefix[FEPLB_MAX_GROUPS + 1];                 // prefix[g] = units of the entries before g
  int row_start[FEPLB_MAX_GROUPS];
  int rows[FEPLB_MAX_GROUPS];
  int expert[FEPLB_MAX_GROUPS];
};
template <int NMAX> constexpr size_t smem_bytes() {
  constexpr size_t n = 1024 + (size_t)Form<NMAX>::kStages * Form<NMAX>::kStageBytes + (size_t)Form<NMAX>::kEpiWarps * kEpiStageBytes + sizeof(Tail);
  static_assert(n <= 232448 && n > 116 * 1024, "one CTA per SM");
  return n;
}

struct FewParams {
  const feplb_group* groups;
  int n_groups;
  int which;                                        // FEPLB_FFN_* filter
  int E;
  int64_t s_cap;
  int n_wt;                                         // weight blocks per row block
  int num_k_blocks;                                 // K / 128, rounded up
  int num_chunks;                                   // K / 64; a chunk past the end reads as zeros and is not multiplied
  int w_rows_per_expert;
  int unit_cols;                                    // output columns of a unit: 64 (pass 1) or 128 (pass 2)
  int b_first;                                      // pass 1: the lower lanes hold b (W3 lies in front of W1 in memory)
  int early_weights;                                // the group table was complete before this kernel's predecessor let it start
  __nv_bfloat16* out;
  int ld_out;
  __nv_bfloat16* ab_out;                            // pass 1, optional: pre-activations a | b ([rows, 2f])
  uint32_t* status;
  unsigned long long* stamps;                       // optional, as in feplb_gemm.cu: [0] first CTA's start, [2] ~(last CTA's end)
};

struct RowMaps { CUtensorMap m[kMaxBoxes]; };

struct Unit { int row0, n_rows, n_pad, expert, wt; };

// unit -> (entry, row block, weight block); the weight blocks of one row block are consecutive.
template <int NMAX>
__device__ __forceinline__ Unit unit_coord(const Tail* t, const FewParams& p, int u) {
  int lo = 0, hi = p.n_groups;                      // largest g with prefix[g] <= u
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (t->prefix[mid] <= u) lo = mid; else hi = mid;
  }
  const int local = u - t->prefix[lo];
  const int blk = local / p.n_wt;
  const int rows = t->rows[lo];
  const int nb = (rows + NMAX - 1) / NMAX;
  const int bs = ((rows + nb - 1) / nb + 15) & ~15; // rows per block, a multiple of 16, <= NMAX
  Unit c;
  c.wt = local - blk * p.n_wt;
  c.row0 = t->row_start[lo] + blk * bs;
  c.n_rows = min(bs, rows - blk * bs);
  c.n_pad = (c.n_rows + 15) & ~15;
  c.expert = t->expert[lo];
  return c;
}

__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* m, uint32_t bar, int c0, int c1, int c2, int c3, int c4) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4) : "memory");
}

// 16 or 32 columns (HALVES fragments of 16) x 32 token rows -> rows of global memory: stmatrix transposes into token rows of
// 64 bytes whose 16-byte pieces are exchanged by bits 1 and 2 of the row number, and 16-byte pieces go out.
template <int HALVES>
__device__ __forceinline__ void store_transposed(uint32_t stg, const float* v, __nv_bfloat16* out, int64_t ld, int n_valid, int lane) {
  const uint32_t octet = lane >> 3, tok = lane & 7;
  __syncwarp();                                     // the staging area has been read
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    if (HALVES == 2) {
      const uint32_t addr = stg + (8 * g + tok) * 64 + ((octet ^ ((tok >> 1) & 3)) << 4);
      asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr),
                   "r"(pack_bf16x2(v[4 * g], v[4 * g + 1])), "r"(pack_bf16x2(v[4 * g + 2], v[4 * g + 3])),
                   "r"(pack_bf16x2(v[16 + 4 * g], v[16 + 4 * g + 1])), "r"(pack_bf16x2(v[16 + 4 * g + 2], v[16 + 4 * g + 3])) : "memory");
    } else {
      const uint32_t addr = stg + (8 * g + tok) * 64 + (((octet & 1) ^ ((tok >> 1) & 3)) << 4);
      asm volatile("stmatrix.sync.aligned.m8n8.x2.trans.shared.b16 [%0], {%1, %2};" ::"r"(addr),
                   "r"(pack_bf16x2(v[4 * g], v[4 * g + 1])), "r"(pack_bf16x2(v[4 * g + 2], v[4 * g + 3])) : "memory");
    }
  }
  __syncwarp();
  constexpr int kPieces = 2 * HALVES, kRows = 32 / kPieces;       // 16-byte pieces per token, tokens per instruction
  const int tj = lane / kPieces, piece = lane % kPieces;
#pragma unroll
  for (int it = 0; it < 32 / kRows; ++it) {
    const int j = it * kRows + tj;
    uint4 w;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w.x), "=r"(w.y), "=r"(w.z), "=r"(w.w)
                 : "r"(stg + (uint32_t)(j * 64 + ((piece ^ ((j >> 1) & 3)) << 4))));
    if (j < n_valid) *reinterpret_cast<uint4*>(out + (int64_t)j * ld + piece * 8) = w;
  }
}

template <bool SWIGLU, int NMAX>
__global__ void __launch_bounds__(Form<NMAX>::kThreads, 1)
k_ffn_few(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ RowMaps tm_x, const FewParams p) {
  using F = Form<NMAX>;
  constexpr int kStages = F::kStages, kStageBytes = F::kStageBytes, kEpiWarps = F::kEpiWarps, kThreads = F::kThreads;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* epi_smem = smem + (size_t)kStages * kStageBytes;
  Tail* tail = reinterpret_cast<Tail*>(epi_smem + (size_t)kEpiWarps * kEpiStageBytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int worker = (int)blockIdx.x, n_workers = (int)gridDim.x;
  volatile int* abort_flag = &tail->abort_flag;

  if (threadIdx.x == 0) {
    prefetch_tmap(&tm_w);
    for (int i = 0; i < F::kBoxes; ++i) prefetch_tmap(&tm_x.m[i]);
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_u32(&tail->full[s]), 1);
      mbar_init(smem_u32(&tail->empty[s]), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&tail->tmem_full[a]), 1);
      mbar_init(smem_u32(&tail->tmem_empty[a]), kEpiWarps);
    }
    tail->abort_flag = 0;
    tail->prefix[0] = 0;
    fence_barrier_init();
  }
  if (warp == 1) {
    __syncwarp();
    tmem_alloc(smem_u32(&tail->tmem_base), F::kTmemCols);
    tmem_relinquish();
  }
  // As in feplb_gemm.cu: with early_weights the group table and the first weights are read before the wait, and the
  // kernel behind may start only after this one's own wait.
  if (!p.early_weights) asm volatile("griddepcontrol.wait;" ::: "memory");
  if (p.stamps && !p.early_weights && threadIdx.x == 0) atomicMin(&p.stamps[0], global_timer_ns());
  for (int g = threadIdx.x; g < p.n_groups; g += kThreads) {
    const feplb_group gr = p.groups[g];
    const bool selected = p.which == FEPLB_FFN_ALL || (p.which == FEPLB_FFN_STATIC) == (gr.is_dynamic == 0);
    int units = 0;
    if (selected && gr.rows > 0) {
      if (gr.expert >= 0 && gr.expert < p.E && gr.row_start >= 0 && (int64_t)gr.row_start + gr.rows <= p.s_cap && gr.is_dynamic < 2)
        units = (gr.rows + NMAX - 1) / NMAX * p.n_wt;
      else atomicOr(p.status, FEPLB_ST_GROUP);
    }
    tail->prefix[g + 1] = units;
    tail->row_start[g] = gr.row_start;
    tail->rows[g] = gr.rows;
    tail->expert[g] = gr.expert;
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) warp_scan_prefix(tail->prefix, 0, p.n_groups, lane);
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tail->tmem_base;
  const int total = tail->prefix[p.n_groups];
  if (p.early_weights && warp != 0) {               // (the producer waits on its own, after its first weight loads)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (p.stamps && threadIdx.x == 32) atomicMin(&p.stamps[0], global_timer_ns());
  }
  if (warp != 0) asm volatile("griddepcontrol.launch_dependents;");

  if (warp == 0) {
    // ---- TMA producer -------------------------------------------------------------------------------
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      struct Source { const CUtensorMap* x; int wrow, xrow; uint32_t tx; };
      auto source = [&](const Unit& c) {
        Source q;
        q.wrow = c.expert * p.w_rows_per_expert + c.wt * p.unit_cols;
        q.xrow = c.row0;
        int bi = F::kBoxes - 1;                     // the smallest box that covers the rows
        while ((NMAX >> bi) < c.n_pad) --bi;
        q.x = &tm_x.m[bi];
        q.tx = (uint32_t)(kWBytes + (NMAX >> bi) * (BK * 2));
        return q;
      };
      auto load_weights = [&](const Source& q, int kb, int st) {
        const uint32_t full = smem_u32(&tail->full[st]), sa = smem_u32(smem + (size_t)st * kStageBytes);
        mbar_expect_tx(full, q.tx);
        if (SWIGLU) tma_load_5d(sa, &tm_w, full, 0, 0, 0, q.wrow / 16, kb * 2);       // 64 rows of W1 and of W3
        else tma_load_3d(sa, &tm_w, full, 0, q.wrow, kb * 2);                         // 128 rows of W2
      };
      auto load_rows = [&](const Source& q, int kb, int st) {
        tma_load_3d(smem_u32(smem + (size_t)st * kStageBytes) + kWBytes, q.x, smem_u32(&tail->full[st]), 0, q.xrow, kb * 2);
      };
      int n_early = 0;
      if (p.early_weights) {
        if (worker < total) {
          n_early = min(kStages, p.num_k_blocks);
          const Source q = source(unit_coord<NMAX>(tail, p, worker));
          for (int kb = 0; kb < n_early; ++kb) load_weights(q, kb, kb);
        }
        asm volatile("griddepcontrol.wait;" ::: "memory");
      }
      asm volatile("griddepcontrol.launch_dependents;");
      for (int u = worker; ok && u < total; u += n_workers) {
        const Source q = source(unit_coord<NMAX>(tail, p, u));
        int kb = 0;
        for (; kb < n_early; ++kb) {                // stages 0 .. n_early - 1, whose weights are on their way
          load_rows(q, kb, stage);
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
        n_early = 0;
        for (; kb < p.num_k_blocks; ++kb) {
          if (!(ok = mbar_wait(smem_u32(&tail->empty[stage]), phase ^ 1u, abort_flag, p.status))) break;
          load_weights(q, kb, stage);
          load_rows(q, kb, stage);
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
      }
      if (!ok)
        for (int i = 0; i < 2000; ++i) __nanosleep(100);   // copies already issued land before the CTA's shared memory goes away
    }
  } else if (warp == 1) {
    // ---- MMA issuer -----------------------------------------------------------------------------------
    if (lane == 0) {
      int stage = 0, as = 0;
      uint32_t phase = 0, aphase = 0;
      bool ok = true;
      for (int u = worker; ok && u < total; u += n_workers) {
        const Unit c = unit_coord<NMAX>(tail, p, u);
        const uint32_t idesc = make_idesc(kWRows, c.n_pad);
        int box = 16;
        while (box < c.n_pad) box *= 2;
        const uint32_t x_chunk = (uint32_t)(box * kChunk * 2) >> 4;       // between the two chunks of the rows
        if (!(ok = mbar_wait(smem_u32(&tail->tmem_empty[as]), aphase ^ 1u, abort_flag, p.status))) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(as * NMAX);
        for (int kb = 0; kb < p.num_k_blocks; ++kb) {
          if (!(ok = mbar_wait(smem_u32(&tail->full[stage]), phase, abort_flag, p.status))) break;
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + (size_t)stage * kStageBytes);
          const uint64_t da = make_smem_desc(sa), db = make_smem_desc(sa + kWBytes);
#pragma unroll
          for (int k = 0; k < BK / UMMA_K; ++k) {
            // +32 bytes (>> 4 = 2) per K step inside a chunk
            const int ch = k / (kChunk / UMMA_K), ks = 2 * (k % (kChunk / UMMA_K));
            if (ch > 0 && kb * 2 + ch >= p.num_chunks) break;
            umma_bf16(d_tmem, da + (uint64_t)(ch * (kWBytes / 2 >> 4) + ks), db + (uint64_t)(ch * x_chunk + ks), idesc,
                      (uint32_t)((kb | k) != 0));
          }
          umma_commit(smem_u32(&tail->empty[stage]));
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        umma_commit(smem_u32(&tail->tmem_full[as]));
        if (++as == 2) { as = 0; aphase ^= 1u; }
      }
    }
  } else {
    // ---- epilogue: TMEM -> registers -> (SwiGLU) -> bf16 -> transposed rows in global memory ------------
    const int q = warp & 3;                         // TMEM lane quarter this warp may read
    const uint32_t stg = smem_u32(epi_smem + (size_t)(warp - 2) * kEpiStageBytes);
    int as = 0;
    uint32_t aphase = 0;
    for (int u = worker; u < total; u += n_workers) {
      const Unit c = unit_coord<NMAX>(tail, p, u);
      bool ok = mbar_wait(smem_u32(&tail->tmem_full[as]), aphase, abort_flag, p.status);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(as * NMAX);
      const int col0 = c.wt * p.unit_cols + (SWIGLU ? q * 16 : q * 32);
      for (int j0 = 32 * ((warp - 2) >> 2); j0 < c.n_rows; j0 += 8 * kEpiWarps) {
        uint32_t r[32];
        tmem_ld_frag(taddr + (uint32_t)j0, r);
        tmem_ld_frag(taddr + (16u << 16) + (uint32_t)j0, r + 16);
        tmem_ld_wait();
        float v[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
        const int64_t row = c.row0 + j0;
        if (SWIGLU) {
          if (p.ab_out != nullptr) {
            __nv_bfloat16* lower = p.ab_out + row * (2 * p.ld_out) + col0;
            store_transposed<1>(stg, v, lower + (p.b_first ? p.ld_out : 0), 2 * p.ld_out, c.n_rows - j0, lane);
            store_transposed<1>(stg, v + 16, lower + (p.b_first ? 0 : p.ld_out), 2 * p.ld_out, c.n_rows - j0, lane);
          }
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = p.b_first ? silu_f(v[16 + i]) * v[i] : silu_f(v[i]) * v[16 + i];
        }
        store_transposed<SWIGLU ? 1 : 2>(stg, v, p.out + row * p.ld_out + col0, p.ld_out, c.n_rows - j0, lane);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&tail->tmem_empty[as]));
      if (++as == 2) { as = 0; aphase ^= 1u; }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (p.stamps && threadIdx.x == 0) atomicMin(&p.stamps[2], ~global_timer_ns());
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, F::kTmemCols);
  }
}

// ------------------------------------------------------------------------------------------ host

bool make_row_maps(RowMaps* x, const void* base, uint64_t rows, uint64_t inner, int nmax) {
  for (int i = 0; (nmax >> i) >= 16; ++i)
    if (!make_tmap_chunks(&x->m[i], base, rows, inner, (uint32_t)(nmax >> i))) return false;
  return true;
}

template <bool SWIGLU, int NMAX>
cudaError_t launch(const CUtensorMap& w, const RowMaps& x, const FewParams& p, int num_sms, cudaStream_t st) {
  // per instantiation and device: the shared-memory attribute is set on first use
  static bool ready[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!ready[dev]) {
    const cudaError_t e = cudaFuncSetAttribute(k_ffn_few<SWIGLU, NMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes<NMAX>());
    if (e != cudaSuccess) return e;
    ready[dev] = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(num_sms);
  cfg.blockDim = dim3(Form<NMAX>::kThreads);
  cfg.dynamicSmemBytes = smem_bytes<NMAX>();
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_ffn_few<SWIGLU, NMAX>, w, x, p);
}

// Both passes.
template <int NMAX>
cudaError_t launch_both(const CUtensorMap& w13, const CUtensorMap& w2, const RowMaps& x, const RowMaps& h, const FewParams& p1,
                        const FewParams& p2, int num_sms, cudaStream_t st, int64_t* n_launch) {
  ++*n_launch;
  const cudaError_t e = launch<true, NMAX>(w13, x, p1, num_sms, st);
  if (e != cudaSuccess) return e;
  ++*n_launch;
  return launch<false, NMAX>(w2, h, p2, num_sms, st);
}

}  // namespace

int feplb_launch_expert_ffn_few(const feplb_gemm_args& a, cudaStream_t st, int64_t* n_launch, char* err, size_t errn,
                                int nmax, unsigned long long* stamps) {
  if (a.n_groups == 0 || a.s_cap == 0) return FEPLB_OK;
  CUtensorMap w13, w2;
  RowMaps x, h;
  if (!make_tmap_w13(&w13, a.w1, a.w3, (uint64_t)a.E * a.f, (uint64_t)a.d)) return FEPLB_E_STATE;
  if (!make_tmap_chunks(&w2, a.w2, (uint64_t)a.E * a.d, (uint64_t)a.f, kWRows) ||
      !make_row_maps(&x, a.x_perm, (uint64_t)a.s_cap, (uint64_t)a.d, nmax) ||
      !make_row_maps(&h, a.h, (uint64_t)a.s_cap, (uint64_t)a.f, nmax)) {
    snprintf(err, errn, "cuTensorMapEncodeTiled failed (driver entry point missing or bad pointer/shape)");
    return FEPLB_E_CUDA;
  }
  FewParams p1;
  p1.groups = a.groups; p1.n_groups = a.n_groups; p1.which = a.which; p1.E = a.E; p1.s_cap = a.s_cap;
  p1.unit_cols = kWRows / 2; p1.n_wt = a.f / p1.unit_cols; p1.num_k_blocks = (a.d + BK - 1) / BK; p1.num_chunks = a.d / kChunk; p1.w_rows_per_expert = a.f;
  p1.early_weights = 0; p1.b_first = a.w3 < a.w1;
  p1.out = (__nv_bfloat16*)a.h; p1.ld_out = a.f; p1.ab_out = (__nv_bfloat16*)a.ab_out; p1.status = a.status; p1.stamps = stamps;
  FewParams p2 = p1;
  p2.unit_cols = kWRows; p2.n_wt = a.d / p2.unit_cols; p2.num_k_blocks = (a.f + BK - 1) / BK; p2.num_chunks = a.f / kChunk; p2.w_rows_per_expert = a.d;
  p2.early_weights = 1;
  p2.out = (__nv_bfloat16*)a.y; p2.ld_out = a.d; p2.ab_out = nullptr; p2.stamps = stamps ? stamps + 4 : nullptr;
  const auto both = nmax == 32 ? launch_both<32> : nmax == 64 ? launch_both<64> : launch_both<128>;
  const cudaError_t e = both(w13, w2, x, h, p1, p2, a.num_sms, st, n_launch);
  if (e != cudaSuccess) {
    snprintf(err, errn, "k_ffn_few launch: %s", cudaGetErrorString(e));
    return FEPLB_E_CUDA;
  }
  return FEPLB_OK;
}
