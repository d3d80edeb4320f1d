// The kernels of the serving loop, instantiated per (operand type, head_dim, query heads per
// kv head) so that each instance carries exactly one attention variant: the persistent
// cooperative loop and the one-phase kernel of stepped mode.
#pragma once
#include <cuda_runtime.h>

#include "../../include/blink.h"
#include "attention.cuh"
#include "control.cuh"
#include "dev_ctx.cuh"
#include "forward.cuh"
#include "gemm_dec.cuh"
#include "gemm_tc.cuh"
#include "kernel_set.h"

namespace blink {

// What the phases of a step depend on besides the layer: made once per step, kept in shared memory.
struct StepInfo {
  int T, R;      // rows of the step, rows that sample
  bool dec;      // decode-sized: the GEMMs of gemm_dec.cuh
  bool small;    // of at most 16 rows: norms, SwiGLU and final norm run inside those GEMMs
  bool fuse;     // RoPE and the K/V write run inside the attention
  bool fold;     // fp32: norms, RoPE and SwiGLU run inside the CUDA-core GEMMs
  bool fold_out; // and the final norm inside the LM head
  bool nuc;      // some row samples from the nucleus of its whole row
  bool att_cta;  // the attention phase leaves the first half of the weight ring alone
};
__shared__ StepInfo g_step;
// The phases of a layer and of the output part, in order, for the current step: phase | (expert or AttKind) << 8 | PLAN_BARRIER when a
// grid barrier closes it.
constexpr int PLAN_BARRIER = 1 << 16, PLAN_MAX = 2 * MAX_EXPERTS + 14;
__shared__ int g_plan[2][PLAN_MAX];   // each ends with -1
__shared__ int g_pos[FWD_THREADS];   // layer << 16 | place in the two lists: a copy per thread, so that none waits for another
static_assert(N_PHASE_TIMERS <= 32, "copied by one warp");
__shared__ unsigned long long g_phase_ns[N_PHASE_TIMERS];   // device time per phase kind of the open step (CTA 0)
__shared__ unsigned long long g_phase_t;                    // when the last phase ended
// Phases that a step does not have because others do their work.
__device__ __forceinline__ bool phase_absorbed(const DevCtx& c, const StepInfo& st, int ph) {
  if (c.fused) return ph == PH_ROPE || ph == PH_SILU;   // done by the epilogues of the QKV and gate/up GEMMs
  if (st.fold && ph != PH_FNORM) return ph == PH_NORM1 || ph == PH_ROPE || ph == PH_NORM2 || ph == PH_SILU;
  if (st.fold_out) return ph == PH_FNORM;
  if (ph == PH_ROPE) return st.fuse;
  if (!st.small) return false;
  return ph == PH_NORM1 || ph == PH_FNORM || (c.E == 0 && (ph == PH_NORM2 || ph == PH_SILU));
}
// (one thread)
__device__ __forceinline__ void make_plan(const DevCtx& c, const StepInfo& st) {
  int n = 0;
  for (int ph = PH_NORM1; ph <= PH_DOWN; ++ph) {
    if (phase_absorbed(c, st, ph)) continue;
    if (ph == PH_ATTN && c.dtype == 0) {   // (every step has rows: at least one of the three)
      const AttStep& a = g_att_step;
      if (a.npp > 0) g_plan[0][n++] = ph | ATT_PAIRS << 8;
      if (a.npf > 0) g_plan[0][n++] = ph | ATT_TILES << 8;
      if (a.n_dec > 0) g_plan[0][n++] = ph | (a.C == 0 ? ATT_DEC_STREAM : a.half ? ATT_DEC_HALF : ATT_DEC_CTA) << 8;
      g_plan[0][n - 1] |= PLAN_BARRIER;
    } else if (c.E > 0 && (ph == PH_GU || ph == PH_DOWN)) {
      if (ph == PH_GU) g_plan[0][n++] = PH_MOE_GROUP | PLAN_BARRIER;   // routing lists and gathered rows first
      // The experts' GEMMs are independent of one another (own weights, own gathered rows; the down projections add
      // into the residual rows with reductions): one grid barrier after the last expert, none in between, so every
      // CTA streams its share of all experts back to back.  (With fused epilogues the barriers stay: their tile
      // counters are per GEMM.)
      for (int e = 0; e < c.E; ++e) g_plan[0][n++] = ph | e << 8 | (c.fused || e + 1 == c.E ? PLAN_BARRIER : 0);
    } else {
      g_plan[0][n++] = ph | PLAN_BARRIER;
    }
  }
  g_plan[0][n] = -1;
  // the output part; long rows are prepared for sampling by all CTAs, rows that sample from a whole-row nucleus with one
  // more pass over the logits
  n = 0;
  for (int i = 0; i < 5; ++i) {
    const int ph = output_phase(i);
    if (phase_absorbed(c, st, ph) || ((ph == PH_SMAX || ph == PH_SNUC) && !sample_split_rows(c.V)) || (ph == PH_SNUC && !st.nuc)) continue;
    g_plan[1][n++] = ph | PLAN_BARRIER;
  }
  g_plan[1][n] = -1;
}
template <typename WT, bool PAIR>
static __device__ __noinline__ void step_begin(const DevCtx& c) {
  StepInfo s;
  const SchedState* ss = c.ss;
  s.T = __ldcg(&ss->cur_T);
  s.R = __ldcg(&ss->cur_rows);
  s.nuc = __ldcg(&ss->cur_nuc) != 0;
  const int C = __ldcg(&ss->cur_C), npf = __ldcg(&ss->cur_npf) + __ldcg(&ss->cur_npp), fuse = __ldcg(&ss->cur_fuse);
  if constexpr (sizeof(WT) == 2) {
    s.small = dec_small(c, s.T);
    s.dec = dec_step(c, s.T);
    s.fuse = fuse != 0;
    s.fold = s.fold_out = false;
    s.att_cta = C > 0 && npf == 0;
    if (s.dec) dec_geometry<PAIR>(c, s.T, s.R);
    att_lists(c);
    const int tiles = (c.qkv_dim + 127) / 128;
    if (c.gemm_tc && threadIdx.x == 0)
      g_qkv_passes = tc_passes(s.T, c.d >> 6, PAIR ? (tiles + 1) / 2 : tiles, PAIR ? (int)gridDim.x / 2 : (int)gridDim.x);
  } else {
    s.small = s.dec = s.fuse = s.att_cta = false;
    s.fold = fold_step(c, s.T);
    s.fold_out = s.fold && fold_lm_head(c, s.R);
  }
  if (threadIdx.x < N_PHASE_TIMERS) g_phase_ns[threadIdx.x] = 0ull;
  if (threadIdx.x == 0) {
    g_step = s;
    make_plan(c, s);
    g_phase_t = global_timer_ns();
  }
  __syncthreads();
}
// The GEMM whose weights the producer may fetch while the grid waits at the end of `phase` (-1: none), and how many stages
// of them: the attention between QKV and O leaves half of the ring alone at most.
__device__ __forceinline__ int dec_next_gemm(const DevCtx& c, const StepInfo& st, int phase, int layer, int& count) {
  count = DEC_STAGES;
  if (!st.dec) return -1;
  if (phase == PH_QKV) { count = ATT_CTA_OFF / DEC_STAGE_BYTES; return st.att_cta ? GEMM_O : -1; }
  if (c.E > 0) return -1;
  if (phase == PH_O) return GEMM_GU;
  if (phase == PH_GU) return GEMM_DOWN;
  if (phase == PH_DOWN) return layer + 1 < c.L ? GEMM_QKV : st.R > 0 ? GEMM_LMHEAD : -1;
  return -1;
}

// The GEMM phases of a decode-sized step; false when the phase is none of them.  `chain`: weights of the GEMM that
// follows may be fetched ahead (not when every phase is a launch of its own).
template <bool PAIR>
__device__ __forceinline__ bool run_phase_dec(const DevCtx& c, const StepInfo& st, int phase, int layer, float* smem, bool chain) {
  int which;
  switch (phase) {
    case PH_QKV: which = GEMM_QKV; break;
    case PH_O: which = GEMM_O; break;
    case PH_GU: if (c.E > 0) return false; which = GEMM_GU; break;
    case PH_DOWN: if (c.E > 0) return false; which = GEMM_DOWN; break;
    case PH_LMHEAD: which = GEMM_LMHEAD; break;
    default: return false;
  }
  int count;
  const int next = chain ? dec_next_gemm(c, st, phase, layer, count) : -1;
  phase_gemm_dec<PAIR>(c, which, layer, st.T, st.R, next, count, smem);
  return true;
}
// The grid barrier that closes a phase.  CTA 0 keeps a device time per phase kind (a phase's time includes this
// barrier), recorded when per-iteration statistics are kept.
__device__ __forceinline__ bool end_phase(const DevCtx& c, int ph) {
  const bool gemm = ph == PH_QKV || ph == PH_O || ph == PH_GU || ph == PH_DOWN;
  const bool ok = g_step.dec && gemm ? dec_barrier(c) : grid_barrier(c);
  if (c.stats_cap > 0 && blockIdx.x == 0 && threadIdx.x == 0) {
    const unsigned long long t = global_timer_ns();
    g_phase_ns[ph >= PH_SMAX ? (int)PH_SAMPLE : ph] += t - g_phase_t;   // the parts of sampling share a timer
    g_phase_t = t;
  }
  return ok;
}
// One GEMM phase.  (A function of its own, arguments and all: built in the dispatcher, the arguments went by way of its stack and
// it kept registers of its own there.)
template <typename WT, bool PAIR>
static __device__ __noinline__ void phase_gemm(const DevCtx& c, int phase, int layer, int sub, float* smem) {
  const size_t esz = sizeof(WT);
  const int T = g_step.T;
  GemmArgs a;
  int which;
  if (phase == PH_QKV) {
    which = GEMM_QKV;
    a = GemmArgs{c.xn, c.w_base + c.w_off[1] + (size_t)layer * c.qkv_dim * c.d * esz, c.qkv, T, c.qkv_dim, c.d, c.qkv_dim, 0};
    a.w_row0 = (long long)layer * c.qkv_dim;
    if (c.fused) a.fix = FIX_ROPE_KV;
  } else if (phase == PH_O) {
    which = GEMM_O;
    a = GemmArgs{c.attn, c.w_base + c.w_off[2] + (size_t)layer * c.d * c.q_dim * esz, c.h, T, c.d, c.q_dim, c.d, 1};
    a.w_row0 = (long long)layer * c.d;
    if (c.fused_norm) { a.fix = FIX_SUMSQ; a.fix_rowss = c.rowss_a; }
  } else if (phase == PH_LMHEAD) {
    which = GEMM_LMHEAD;
    a = GemmArgs{c.xs, c.w_base + c.w_off[9], c.logits, g_step.R, c.V, c.d, c.V, 0};
  } else {
    // the dense FFN, or expert `sub` on the rows routed to it (gathered, contiguous from moe_off[sub])
    const int off = c.E > 0 ? c.moe_off[sub] : 0, cnt = c.E > 0 ? c.moe_off[sub + 1] - off : T;
    const long long we = c.E > 0 ? (long long)layer * c.E + sub : layer;
    if (phase == PH_GU) {
      which = GEMM_GU;
      a = GemmArgs{reinterpret_cast<const char*>(c.E > 0 ? c.xg : c.xn) + (size_t)off * c.d * esz, c.w_base + c.w_off[3] + (size_t)we * 2 * c.F * c.d * esz,
                   c.gu + (size_t)off * 2 * c.F, cnt, 2 * c.F, c.d, 2 * c.F, 0};
      a.w_row0 = we * 2 * c.F;
      if (c.fused) { a.fix = FIX_SILU; a.fix_out = reinterpret_cast<char*>(c.act) + (size_t)off * c.F * esz; }
    } else {
      which = GEMM_DOWN;
      a = GemmArgs{reinterpret_cast<const char*>(c.act) + (size_t)off * c.F * esz, c.w_base + c.w_off[4] + (size_t)we * c.d * c.F * esz, c.h, cnt, c.d, c.F,
                   c.d, 1};
      a.w_row0 = we * c.d;
      if (c.E > 0) {   // result row i belongs to token moe_tok[off + i], weighted by its gate
        a.row_map = c.moe_tok + off;
        a.row_scale = c.moe_gate + off;
      } else if (c.fused_norm) {
        a.fix = FIX_SUMSQ;
        a.fix_rowss = c.rowss_b;
      }
    }
    a.x_row0 = off;
  }
  if constexpr (PAIR) {   // (on the tensor cores, and without fused epilogues)
    phase_gemm_tc<PAIR>(c, a, which, layer, smem);
  } else {
    if constexpr (sizeof(WT) == 2) {
      if (c.gemm_tc) {
        phase_gemm_tc<PAIR>(c, a, which, layer, smem);
        return;
      }
    }
    phase_gemm_simt<WT>(a);
  }
}
template <typename WT, int HD, int NREP, bool PAIR>
__device__ __forceinline__ void run_phase(const DevCtx& c, int phase, int layer, int sub, float* smem, bool chain) {
  const StepInfo& st = g_step;
  const int T = st.T;
  if constexpr (sizeof(WT) == 2) {
    if (st.dec && run_phase_dec<PAIR>(c, st, phase, layer, smem, chain)) return;
  }
  if constexpr (sizeof(WT) == 4) {
    if (st.fold) {
      if (phase == PH_QKV) { phase_gemm_fold<FOLD_ROPE>(c, layer); return; }
      if (phase == PH_GU) { phase_gemm_fold<FOLD_SILU>(c, layer); return; }
      if (phase == PH_LMHEAD && st.fold_out) { phase_gemm_fold<FOLD_NORM>(c, 0); return; }
    }
  }
  switch (phase) {
    case PH_NORM1:
      if constexpr (!PAIR)
        if (c.fused_norm && layer > 0) { phase_norm_apply<WT>(c, layer, 0, T); break; }
      phase_norm<WT>(c, layer, 0);
      break;
    case PH_ROPE: phase_rope_kv<WT>(c, layer); break;
    case PH_ATTN:
      if constexpr (sizeof(WT) == 2) phase_attention_bf16<HD, NREP, PAIR>(c, layer, sub, smem);
      else phase_attention<WT, HD, NREP>(c, layer, smem);
      break;
    case PH_NORM2:
      if constexpr (!PAIR)
        if (c.fused_norm) { phase_norm_apply<WT>(c, layer, 1, T); break; }
      phase_norm<WT>(c, layer, 1);
      break;
    case PH_SILU:
      phase_silu_mul<WT>(c, layer, smem);
      break;
    case PH_MOE_GROUP: phase_moe_group<WT>(c, smem); break;
    case PH_FNORM:
      phase_final_norm<WT>(c);
      break;
    case PH_QKV: case PH_O: case PH_GU: case PH_DOWN: case PH_LMHEAD: phase_gemm<WT, PAIR>(c, phase, layer, sub, smem); break;
    case PH_SMAX: phase_sample_max(c); break;
    case PH_SNUC: phase_sample_weights(c, smem); break;
    case PH_SAMPLE: phase_sample(c, smem); break;
    default: break;
  }
}

// ---- persistent loop -----------------------------------------------------------------
template <typename WT, int HD, int NREP, bool PAIR>
__global__ void __launch_bounds__(FWD_THREADS, 1) blink_loop_kernel(const __grid_constant__ DevCtx param) {
  extern __shared__ __align__(1024) float smem[];
  const DevCtx& c = ctx_to_shared(param);
  long long launch_iters = 0;
  tc_init<PAIR>(c);
  att_init(c);
  dec_init<PAIR>(c);
  if constexpr (PAIR) cluster_sync_all();   // the other CTA's barriers exist before they are signalled
  else __syncthreads();
  while (true) {
    if (blockIdx.x == 0) control_phase(c, launch_iters);
    if (!grid_barrier(c)) break;
    if (*(volatile int*)&c.ss->cmd != CMD_RUN) break;
    if (!c.control_only) {
      bool ok = true;
      step_begin<WT, PAIR>(c);
      // Everything that a phase needs is in shared memory, the place in the plan too: what the dispatcher keeps in registers
      // across a phase is saved and read back on the way from one phase to the next, and the phase functions save
      // registers of their own for it.  With layer and index in registers the dispatcher spilled 100 / 212 bytes and
      // steps were longer: one row of the 1B shape 774 -> 754 us, of 8 layers of the 8B shape 911 -> 887, 64 rows of 4 layers
      // 914 -> 896, the smallest shape's 8 rows 103.7 -> 101.4.
      // (Place and entry are two dependent reads; with list length and layer count read beside them the fp32 steps of the
      // small configuration, which have the most phases, were 2 % longer.)
      volatile int* pos = &g_pos[threadIdx.x];
      volatile int* plan = &g_plan[0][0];
      *pos = 0;
      while (true) {
        const int at = *pos, todo = plan[at & 0xffff];
        if (todo < 0) {   // end of the layer: the next one, or the output part, which follows the last
          const int layer = (at >> 16) + 1, L = g_ctx.L;
          if (layer > L) break;
          *pos = layer << 16 | (layer == L ? PLAN_MAX : 0);
          continue;
        }
        run_phase<WT, HD, NREP, PAIR>(g_ctx, todo & 255, at >> 16, (todo >> 8) & 255, smem, true);
        const int now = *pos, done = plan[now & 0xffff];
        *pos = now + 1;
        if ((done & PLAN_BARRIER) && !end_phase(g_ctx, done & 255)) { ok = false; break; }
      }
      if (!ok) break;
      if (c.stats_cap > 0 && blockIdx.x == 0 && threadIdx.x < 32) {
        __syncwarp();   // thread 0 has added the last phase after the barrier
        if (threadIdx.x < N_PHASE_TIMERS) c.ss->cur_phase_ns[threadIdx.x] = g_phase_ns[threadIdx.x];
      }
    } else if (!grid_barrier(c)) break;
  }
  dec_drain<PAIR>(c, PAIR ? cluster_ctarank() : 0u);
  tc_fini<PAIR>(c);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const int aborted = *(volatile int*)&c.ss->abort_flag;
    __threadfence_system();
    c.mbox->loop_state = aborted ? (uint32_t)BLINK_LOOP_EXIT_ERROR : (uint32_t)c.ss->exit_reason;
    __threadfence_system();
  }
}

template <typename WT, int HD, int NREP, bool PAIR>
__global__ void __launch_bounds__(FWD_THREADS, 1) blink_phase_kernel(const __grid_constant__ DevCtx param, int phase, int layer, int sub) {
  extern __shared__ __align__(1024) float smem[];
  const DevCtx& c = ctx_to_shared(param);
  if (c.ss->cmd != CMD_RUN) return;
  tc_init<PAIR>(c);
  att_init(c);
  dec_init<PAIR>(c);
  if constexpr (PAIR) cluster_sync_all();
  else __syncthreads();
  step_begin<WT, PAIR>(c);
  if (phase == PH_ATTN && sizeof(WT) == 2) {   // all of its pieces
    for (int i = 0; g_plan[0][i] >= 0; ++i)
      if ((g_plan[0][i] & 255) == PH_ATTN) run_phase<WT, HD, NREP, PAIR>(c, phase, layer, (g_plan[0][i] >> 8) & 255, smem, false);
  } else if (!phase_absorbed(c, g_step, phase)) {
    run_phase<WT, HD, NREP, PAIR>(c, phase, layer, sub, smem, false);
  }
  tc_fini<PAIR>(c);
}

// `pair`: the variant whose GEMMs run on CTA pairs (tcgen05 cta_group::2; launched with clusters of two).
// Built for 16-bit operands with four query heads per kv head, the shape of the large configurations.
template <typename WT, int HD>
inline KernelSet kernel_set_for(int n_rep, bool pair) {
  if (pair) {
    if constexpr (sizeof(WT) == 2) {
      if (n_rep == 4) return {(const void*)blink_loop_kernel<WT, HD, 4, true>, (const void*)blink_phase_kernel<WT, HD, 4, true>};
    }
    return {nullptr, nullptr};
  }
  switch (n_rep) {
    case 1: return {(const void*)blink_loop_kernel<WT, HD, 1, false>, (const void*)blink_phase_kernel<WT, HD, 1, false>};
    case 2: return {(const void*)blink_loop_kernel<WT, HD, 2, false>, (const void*)blink_phase_kernel<WT, HD, 2, false>};
    case 4: return {(const void*)blink_loop_kernel<WT, HD, 4, false>, (const void*)blink_phase_kernel<WT, HD, 4, false>};
    case 8: return {(const void*)blink_loop_kernel<WT, HD, 8, false>, (const void*)blink_phase_kernel<WT, HD, 8, false>};
    default: return {nullptr, nullptr};
  }
}

}  // namespace blink
