// Control plane of the serving loop, executed by CTA 0 (256 threads) once per
// iteration: retire the previous step (publish tokens, free blocks), move newly
// submitted requests into the HBM ring, scan + claim, FCFS admission, step
// composition, block allocation and metadata build.
//
// Paper: Section 4.2 "Persistent scheduler" (scan, claim, launch, poll, publish),
// "Parallel slot scanning" (256 threads over contiguous slot ranges, CAS claim),
// "Continuous batching with inline prefill" (FCFS), "Ring buffer" (state machine,
// fences order the externally visible updates).
#pragma once
#include "../../include/blink.h"
#include "dev_ctx.cuh"
#include "mailbox.h"
#include "att_plan.h"

namespace blink {

// The kernels work on a copy of their parameter block in shared memory.  The phase functions take the block by
// reference, and through a reference the parameter space is read like global memory: by way of L1, which every grid
// barrier's acquire empties, so that each phase began with round trips to L2 for its own sizes and pointers.
__shared__ DevCtx g_ctx;
__shared__ unsigned long long g_bar_target;   // arrivals the CTA expects at its next grid barrier, zero when the kernel starts
__device__ __forceinline__ const DevCtx& ctx_to_shared(const DevCtx& param) {
  static_assert(sizeof(DevCtx) % 4 == 0, "copied by words");
  const uint32_t* src = reinterpret_cast<const uint32_t*>(&param);
  uint32_t* dst = reinterpret_cast<uint32_t*>(&g_ctx);
  for (int i = threadIdx.x; i < (int)(sizeof(DevCtx) / 4); i += blockDim.x) dst[i] = src[i];
  if (threadIdx.x == 0) g_bar_target = 0ull;
  __syncthreads();
  return g_ctx;
}

// ---- memory-ordering helpers ------------------------------------------------------
__device__ __forceinline__ uint64_t ld_acquire_sys_u64(const volatile uint64_t* p) {
  uint64_t v;
  asm volatile("ld.acquire.sys.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t ld_relaxed_sys_u32(const volatile uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.sys.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t ld_acquire_sys_u32(const volatile uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.sys.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
struct MailboxWords {   // see read_mailbox
  const Mailbox* m;
  __device__ __forceinline__ uint32_t stop_relaxed() const { return ld_relaxed_sys_u32(&m->stop); }
  __device__ __forceinline__ uint32_t start_acquire() const { return ld_acquire_sys_u32(&m->start); }
  __device__ __forceinline__ uint64_t sub_tail_acquire() const { return ld_acquire_sys_u64(&m->sub_tail); }
};
__device__ __forceinline__ uint64_t global_timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void dev_fail(const DevCtx& c, int code) {
  if (atomicCAS((int*)&c.mbox->device_status, 0, code) == 0) __threadfence_system();
  atomicExch(&c.ss->abort_flag, 1);
}

__device__ __forceinline__ unsigned long long ld_acquire_gpu_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// Grid-wide barrier with a bounded wait: every CTA adds one to a monotone counter (reset by the
// host before each launch) and waits until it reaches the next multiple of the grid size.
// Returns false when the loop must unwind (time-out here or abort raised elsewhere).  g_bar_target
// is the CTA's running total.  Out of line: one copy of the code for all phases.
__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}

// Arrival and wait of the CTA, by one thread after a barrier of the threads whose stores it stands for.
__device__ __forceinline__ bool grid_arrive_and_wait(const DevCtx& c) {
  SchedState* ss = c.ss;
  const unsigned long long target = g_bar_target + gridDim.x;
  g_bar_target = target;
  // release at gpu scope is cumulative: the stores of the CTA's other threads, ordered before this
  // point by the barrier before, are covered without a separate fence
  asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(&ss->bar_ctr) : "memory");
  long long t0 = 0;
  unsigned int polls = 0;
  while (ld_acquire_gpu_u64(&ss->bar_ctr) < target) {
    if ((++polls & 63u) == 0) {
      if (*(volatile int*)&ss->abort_flag) return false;
      if (t0 == 0) t0 = clock64();
      if ((unsigned long long)(clock64() - t0) > c.barrier_timeout_cycles) {
        dev_fail(c, DEV_ERR_BARRIER_TIMEOUT);
        return false;
      }
      if (polls > 4096u) __nanosleep(200);
    }
  }
  return *(volatile int*)&ss->abort_flag == 0;
}
__shared__ int g_bar_ok;
static __device__ __noinline__ bool grid_barrier(const DevCtx& c) {
  // Buffers written with ordinary stores in one phase (normed rows, K/V rows, attention output, ...)
  // are read by TMA / bulk copies (the async proxy) in a later phase: every thread orders its
  // stores against that proxy before it arrives, and again before it issues copies afterwards.
  fence_proxy_async_global();
  __syncthreads();
  if (threadIdx.x == 0) g_bar_ok = grid_arrive_and_wait(c) ? 1 : 0;
  __syncthreads();
  fence_proxy_async_global();
  return g_bar_ok != 0;
}

// Exclusive prefix sums of N values over the 256 threads of the control CTA, all at once (two barriers; one scan after
// another took 0.4 us each, nine of them in a step); tot gets the sums, v the prefixes.
template <int N>
__device__ __forceinline__ void block_exscan(int (&v)[N], int (&tot)[N]) {
  constexpr int W = CTRL_THREADS / 32;
  __shared__ __align__(16) int s_scan[N][W];
  static_assert(W == 8, "a row of warp sums is two 16-byte vectors");
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int x[N];
#pragma unroll
  for (int n = 0; n < N; ++n) x[n] = v[n];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1)
#pragma unroll
    for (int n = 0; n < N; ++n) {
      const int y = __shfl_up_sync(0xffffffffu, x[n], o);
      if (lane >= o) x[n] += y;
    }
  __syncthreads();   // the previous call's sums have been read
  if (lane == 31)
#pragma unroll
    for (int n = 0; n < N; ++n) s_scan[n][w] = x[n];
  __syncthreads();
#pragma unroll
  for (int n = 0; n < N; ++n) {
    const int4 a = *reinterpret_cast<const int4*>(&s_scan[n][0]), b = *reinterpret_cast<const int4*>(&s_scan[n][4]);
    const int p[W] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    int before = 0, all = 0;
#pragma unroll
    for (int i = 0; i < W; ++i) {
      if (i < w) before += p[i];
      all += p[i];
    }
    v[n] = x[n] - v[n] + before;
    tot[n] = all;
  }
}

// Of the batch table while a step is composed; the attention's between the steps (attn_decode_cta).
struct CtlScratch {
  long long ticket[MAX_BATCH];
  int phase[MAX_BATCH], rem[MAX_BATCH];
};
__shared__ __align__(16) CtlScratch g_ctl;

__device__ __forceinline__ int32_t fake_token(unsigned long long ticket, int gen, int vocab) {
  // control-only stand-in sampler: a fixed hash of (ticket, index)
  uint32_t x = (uint32_t)(ticket * 2654435761ull + (unsigned long long)gen * 40503ull + 12345ull);
  return (int32_t)(x % (uint32_t)vocab);
}

__device__ __forceinline__ bool trace_on(const DevCtx& c) { return c.trace_cap > 0 && !c.ss->trace_off; }

// ---- step 5 of the iteration: publish, retire, free -------------------------------------
static __device__ void post_step(const DevCtx& c) {
  SchedState* ss = c.ss;
  const int tid = threadIdx.x;
  const int n_items = ss->cur_items;
  const int n_rows = ss->cur_rows;
  const bool tr = trace_on(c) && ss->cur_hdr >= 0;
  int32_t* rec_post = c.trace + ss->cur_post;
  __shared__ unsigned long long s_ptok;
  __shared__ int s_need_sum;
  // the host's cancel marks are a round trip to host memory away: asked for first, looked at after the rest
  int cslot = 0;
  uint32_t cmark = 0u;
  if (c.cancel != nullptr && tid < c.MB && c.b_phase[tid] != PHASE_FREE) {
    cslot = c.b_slot[tid];
    cmark = ld_relaxed_sys_u32(&c.cancel[cslot]);
  }
  if (tid == 0) { s_ptok = 0; s_need_sum = 0; }
  __syncthreads();

  int fin = 0, nfree = 0, b = -1, row = -1, out_slot = -1, out_gen = 0;
  long long ticket = 0;
  if (tid < n_items) {
    b = c.it_bslot[tid];
    const int n = c.it_ntok[tid];
    row = c.it_row[tid];
    const int slot = c.b_slot[b];
    ticket = c.b_ticket[b];
    int phase = c.b_phase[b];
    if (phase == PHASE_PREFILL) {
      c.b_prefilled[b] += n;
      atomicAdd(&s_ptok, (unsigned long long)n);
    }
    if (row >= 0) {
      const int gen = c.b_generated[b];
      const int32_t sampled = c.control_only ? fake_token((unsigned long long)ticket, gen, c.V) : c.row_sampled[row];
      const int32_t fed = (c.b_flags[b] & REQ_FLAG_FORCED) ? c.forced_arena[(size_t)slot * c.max_new + gen] : sampled;
      c.gen_arena[(size_t)slot * c.max_new + gen] = fed;
      c.b_last[b] = fed;
      c.b_generated[b] = gen + 1;
      fin = (gen + 1 == c.b_N[b]) || (c.b_eos[b] >= 0 && fed == c.b_eos[b]);
      // externally visible: token and timestamp first, then the generation count
      c.out_tokens[(size_t)slot * c.max_new + gen] = sampled;
      c.out_time[(size_t)slot * c.max_new + gen] = global_timer_ns();
      c.slot_hot[slot].generated = gen + 1;
      if (phase == PHASE_PREFILL) c.b_phase[b] = PHASE_DECODE;
      c.slot_hot[slot].state = fin ? SLOT_DECODE_COMPLETED : SLOT_DECODE_PROCESSING;
      out_slot = slot;
      out_gen = gen + 1;
      if (tr) { rec_post[2 * row] = b; rec_post[2 * row + 1] = sampled; }
      if (fin) {
        nfree = c.b_have[b];
        atomicAdd(&s_need_sum, c.b_need[b]);
      }
    }
  }
  const int top = ss->free_top;
  int sc[2] = {fin, nfree}, sc_tot[2];
  block_exscan(sc, sc_tot);
  const int fin_idx = sc[0], free_off = sc[1], tot_fin = sc_tot[0], tot_free = sc_tot[1];
  if (fin) {
    if (tr) rec_post[2 * n_rows + fin_idx] = (int32_t)ticket;
    for (int j = 0; j < nfree; ++j) {
      const int blk = c.block_table[(size_t)b * c.max_blocks_seq + j];
      c.free_stack[top + free_off + j] = blk;
      if (tr) rec_post[2 * n_rows + tot_fin + free_off + j] = blk;
    }
    c.b_have[b] = 0;
    c.b_phase[b] = PHASE_FREE;
  }
  if (out_slot >= 0) {   // (the writes above have had the time of the scans to reach the host)
    __threadfence_system();
    c.out_count[out_slot] = (uint32_t)out_gen | (fin ? 0x80000000u : 0u);
  }
  __syncthreads();
  // Cancellation (an early exit the host asks for): every request that is still live after the step's
  // own completions and whose slot carries the host's cancel mark is retired here, in ascending batch
  // slot, exactly as at a normal end: blocks pushed back in logical order, reservation released.
  int cfin = 0, cfree = 0;
  long long cticket = 0;
  if (cmark != 0u && c.b_phase[tid] != PHASE_FREE) {
    cfin = 1;
    cfree = c.b_have[tid];
    cticket = c.b_ticket[tid];
    atomicAdd(&s_need_sum, c.b_need[tid]);
  }
  int cfin_idx = 0, cfree_off = 0, tot_cfin = 0, tot_cfree = 0;
  if (__syncthreads_or(cfin)) {
    int cs[2] = {cfin, cfree}, cs_tot[2];
    block_exscan(cs, cs_tot);
    cfin_idx = cs[0]; cfree_off = cs[1]; tot_cfin = cs_tot[0]; tot_cfree = cs_tot[1];
  }
  if (cfin) {
    if (tr) rec_post[2 * n_rows + tot_fin + tot_free + cfin_idx] = (int32_t)cticket;
    for (int j = 0; j < cfree; ++j) {
      const int blk = c.block_table[(size_t)tid * c.max_blocks_seq + j];
      c.free_stack[top + tot_free + cfree_off + j] = blk;
      if (tr) rec_post[2 * n_rows + tot_fin + tot_free + tot_cfin + cfree_off + j] = blk;
    }
    c.b_have[tid] = 0;
    c.b_phase[tid] = PHASE_FREE;
    c.slot_hot[cslot].state = SLOT_DECODE_COMPLETED;
    __threadfence_system();
    c.out_count[cslot] = (uint32_t)c.b_generated[tid] | 0xC0000000u;   // finished + cancelled
  }
  __syncthreads();
  if (tid == 0) {
    ss->free_top = top + tot_free + tot_cfree;
    ss->reserved -= s_need_sum;
    ss->tokens_out += (unsigned long long)n_rows;
    ss->prompt_tokens += s_ptok;
    ss->sample_rows_total += (unsigned long long)n_rows;
    const uint64_t t_end = global_timer_ns();
    if (tr) {
      // The record lists finished tickets then freed blocks; with cancellations the order is: tickets
      // that ended by themselves, their blocks, cancelled tickets, their blocks -- rewritten below into
      // the record's two lists (tickets first, then blocks) when both kinds occur.
      int32_t* hdr = c.trace + ss->cur_hdr;
      if (tot_cfin > 0 && tot_free > 0) {
        // move the cancelled tickets in front of the first group's blocks (few words, one thread)
        int32_t* base = rec_post + 2 * n_rows + tot_fin;
        for (int k = 0; k < tot_cfin; ++k) {
          const int32_t tk = base[tot_free + k];
          for (int j = tot_free + k; j > k; --j) base[j] = base[j - 1];
          base[k] = tk;
        }
      }
      hdr[6] = n_rows;
      hdr[7] = tot_fin + tot_cfin;
      hdr[8] = tot_free + tot_cfree;
      hdr[9] = ss->free_top;
      hdr[10] = ss->reserved;
      const long long end = ss->cur_post + 2 * n_rows + tot_fin + tot_cfin + tot_free + tot_cfree;
      hdr[11] = (int32_t)(end - ss->cur_hdr);
      ss->trace_pos = end;
    }
    if (c.stats_cap > 0 && (long long)ss->iter < c.stats_cap) {
      IterStat& st = c.stats[ss->iter];
      st.t_begin_ns = ss->cur_t_begin;
      st.t_forward_ns = ss->cur_t_forward;
      st.t_end_ns = t_end;
      st.n_tokens = ss->cur_T;
      st.n_decode = ss->cur_decode;
      st.n_sample_rows = n_rows;
      st.n_items = n_items;
      st.ctx_tokens = ss->cur_ctx;
      st.kv_tokens = ss->cur_kv;
      for (int i = 0; i < N_PHASE_TIMERS; ++i) st.phase_ns[i] = ss->cur_phase_ns[i];
    }
    for (int i = 0; i < N_PHASE_TIMERS; ++i) ss->cur_phase_ns[i] = 0;
    ss->iter += 1;
    ss->cur_hdr = -1;
    ss->pending_post = 0;
    c.mbox->heartbeat = ss->iter;
  }
  __syncthreads();
}

// ---- stand-in for the frontend's RDMA write: pinned submit area -> HBM ring --------------
// (a warp per request: entry and prompt are reads from host memory, a microsecond or two each)
static __device__ void ingress(const DevCtx& c, unsigned long long tail) {
  SchedState* ss = c.ss;
  const int tid = threadIdx.x, lane = tid & 31;
  const unsigned long long seen = ss->seen;
  for (unsigned long long e = seen + (unsigned)(tid >> 5); e < tail; e += CTRL_THREADS / 32) {
    const SubEntry en = c.sub_q[e % (unsigned long long)c.n_slots];
    const uint32_t slot = en.slot, np = en.n_prompt;
    if (slot >= (uint32_t)c.n_slots || np > (uint32_t)c.max_prompt || en.max_new > (uint32_t)c.max_new || en.ticket != e) {
      if (lane == 0) dev_fail(c, DEV_ERR_BAD_INDEX);
      break;
    }
    auto copy = [&](int32_t* dst, const int32_t* src, uint32_t n) {
      for (uint32_t i0 = 0; i0 < n; i0 += 256) {   // eight words per lane on their way at a time
        int32_t v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = src[min(i0 + 32u * k + lane, n - 1u)];
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if (i0 + 32u * k + lane < n) dst[i0 + 32u * k + lane] = v[k];
      }
    };
    copy(c.in_arena + (size_t)slot * c.max_prompt, c.sub_tokens + (size_t)slot * c.max_prompt, np);
    if (en.flags & REQ_FLAG_FORCED)
      copy(c.forced_arena + (size_t)slot * c.max_new, c.sub_forced + (size_t)slot * c.max_new, en.max_new);
    if (lane == 0) {
      SlotCold& cold = c.slot_cold[slot];
      cold.ticket = en.ticket;
      cold.max_new = en.max_new;
      cold.top_k = en.top_k;
      cold.temperature = en.temperature;
      cold.eos_id = en.eos_id;
      cold.seed = en.seed;
      cold.user_tag = en.user_tag;
      cold.flags = en.flags;
      cold.top_p = en.top_p;
      SlotHot& hot = c.slot_hot[slot];
      hot.n_prompt = np;
      hot.generated = 0;
      hot.arena_off = slot;
    }
    __threadfence();   // payload before the state flip
    __syncwarp();
    if (lane == 0) c.slot_hot[slot].state = SLOT_PREFILL_PENDING;
  }
  __syncthreads();
  if (tid == 0) ss->seen = tail;
  __syncthreads();
}

// ---- parallel slot scan + CAS claim (Section 4.2 "Parallel slot scanning") ----------------
static __device__ void scan_and_claim(const DevCtx& c) {
  const int per = (c.n_slots + CTRL_THREADS - 1) / CTRL_THREADS;
  const int lo = threadIdx.x * per;
  const int hi = min(c.n_slots, lo + per);
  for (int s = lo; s < hi; ++s) {
    if (c.slot_hot[s].state == SLOT_PREFILL_PENDING) {
      if (atomicCAS(&c.slot_hot[s].state, (uint32_t)SLOT_PREFILL_PENDING, (uint32_t)SLOT_PREFILL_PROCESSING) ==
          SLOT_PREFILL_PENDING) {
        const unsigned long long t = c.slot_cold[s].ticket;
        c.ticket_to_slot[t % (unsigned long long)c.n_slots] = (uint32_t)s;
      }
    }
  }
  __syncthreads();
}

// ---- steps 1-3: admit, compose, allocate, build metadata ----------------------------------
// Returns the number of rows T of the composed step (0 = nothing to run).
static __device__ int schedule_step(const DevCtx& c, unsigned long long visible) {
  SchedState* ss = c.ss;
  const int tid = threadIdx.x;
  const int MB = c.MB;
  int(&s_phase)[MAX_BATCH] = g_ctl.phase;
  long long(&s_ticket)[MAX_BATCH] = g_ctl.ticket;
  int(&s_rem)[MAX_BATCH] = g_ctl.rem;
  __shared__ int s_qstart[MAX_BATCH + 1];
  __shared__ int s_item_b[MAX_BATCH];
  __shared__ int s_n_admit;
  __shared__ int s_trace_ok;
  __shared__ unsigned long long s_ctx, s_kv;
  __shared__ int s_ndec;
  __shared__ int s_nkb[MAX_BATCH];
  __shared__ int s_maxkb, s_C, s_Citems, s_nuc;

  const uint64_t t_begin = global_timer_ns();
  s_phase[tid] = tid < MB ? c.b_phase[tid] : -1;
  if (tid == 0) { s_n_admit = 0; s_ctx = 0; s_kv = 0; s_ndec = 0; s_maxkb = 0; s_C = 0; s_Citems = 0; s_nuc = 0; }
  __syncthreads();

  // open a trace record (header is completed later)
  long long hdr = -1;
  if (trace_on(c)) hdr = ss->trace_pos;
  int32_t* rec = c.trace + (hdr >= 0 ? hdr : 0);

  // 1. FCFS admission.  The decisions are serial (each depends on the one before), what they need is read and what they
  // cause is written by all threads.
  const unsigned long long na = ss->next_admit;
  const int n_cand = (int)min(visible - na, (unsigned long long)MB);
  if (n_cand > 0) {   // uniform over the CTA
    uint32_t slot = 0;
    int P = 0;
    SlotCold cold;
    if (tid < n_cand) {
      slot = c.ticket_to_slot[(na + tid) % (unsigned long long)c.n_slots];
      bool bad = slot >= (uint32_t)c.n_slots;
      if (!bad) {
        cold = c.slot_cold[slot];
        P = (int)c.slot_hot[slot].n_prompt;
        bad = cold.ticket != na + tid || c.slot_hot[slot].state != SLOT_PREFILL_PROCESSING;
      }
      s_qstart[tid] = bad ? -1 : (P + (int)cold.max_new - 1 + c.bs - 1) / c.bs;   // blocks needed
    }
    __syncthreads();
    if (tid == 0) {
      int n = 0, reserved = ss->reserved, cursor = 0;
      for (; n < n_cand; ++n) {
        const int need = s_qstart[n];
        if (need < 0) { dev_fail(c, DEV_ERR_TICKET_TABLE); break; }
        while (cursor < MB && s_phase[cursor] != PHASE_FREE) ++cursor;
        if (cursor >= MB || reserved + need > c.n_blocks) break;  // head of line blocks
        s_phase[cursor] = PHASE_PREFILL;
        s_item_b[n] = cursor;
        reserved += need;
      }
      ss->next_admit = na + n;
      ss->reserved = reserved;
      s_n_admit = n;
    }
    __syncthreads();
    if (tid < s_n_admit) {
      const int b = s_item_b[tid];
      c.b_phase[b] = PHASE_PREFILL;
      c.b_ticket[b] = (long long)(na + tid);
      c.b_slot[b] = (int)slot;
      c.b_P[b] = P;
      c.b_N[b] = (int)cold.max_new;
      c.b_prefilled[b] = 0;
      c.b_generated[b] = 0;
      c.b_have[b] = 0;
      c.b_need[b] = s_qstart[tid];
      c.b_last[b] = 0;
      c.b_eos[b] = cold.eos_id;
      c.b_topk[b] = (int)cold.top_k;
      c.b_temp[b] = cold.temperature;
      c.b_topp[b] = cold.top_p;
      c.b_seed[b] = cold.seed;
      c.b_flags[b] = (int)cold.flags;
      if (hdr >= 0 && hdr + TRACE_HDR_WORDS + 2 * (tid + 1) <= c.trace_cap) {
        rec[TRACE_HDR_WORDS + 2 * tid] = (int32_t)(na + tid);
        rec[TRACE_HDR_WORDS + 2 * tid + 1] = b;
      }
    }
    __threadfence();
    __syncthreads();
  }
  const int n_admit = s_n_admit;

  // 2. compose
  int phase = PHASE_FREE, P = 0, prefilled = 0, gen = 0, have = 0, slot = 0;
  long long ticket = 0;
  if (tid < MB) {
    phase = s_phase[tid];
    if (phase != PHASE_FREE) {
      P = c.b_P[tid];
      prefilled = c.b_prefilled[tid];
      gen = c.b_generated[tid];
      have = c.b_have[tid];
      slot = c.b_slot[tid];
      ticket = c.b_ticket[tid];
    }
  }
  s_ticket[tid] = ticket;
  s_rem[tid] = (phase == PHASE_PREFILL) ? (P - prefilled) : 0;
  __syncthreads();
  int take = 0, start = 0;
  // prompt tokens already promised to earlier tickets in this iteration
  long long before = 0;
  if (phase == PHASE_PREFILL)
    for (int j = 0; j < MB; ++j)
      if (s_rem[j] > 0 && s_ticket[j] < ticket) before += s_rem[j];
  bool prefill_turn = false;
  if (c.policy == BLINK_POLICY_PAUSE_RESUME) {
    // Section 4.2 "Continuous batching with inline prefill": a step is a decode step, or a prefill step
    // for the whole prompts of the newly admitted requests while decoding is paused for this one step
    const int has_pf = __syncthreads_or(phase == PHASE_PREFILL);
    const int has_dec = __syncthreads_or(phase == PHASE_DECODE);
    prefill_turn = has_pf && (!ss->last_was_prefill || !has_dec);
    if (prefill_turn) {
      if (phase == PHASE_PREFILL && before + P <= (long long)c.chunk) take = P;   // whole prompts, nobody overtakes
      if (phase == PHASE_DECODE) c.slot_hot[slot].state = SLOT_DECODE_PAUSED;
    } else if (phase == PHASE_DECODE) {
      take = 1;
      start = P + gen - 1;
      c.slot_hot[slot].state = SLOT_DECODE_PROCESSING;
    }
  } else if (phase == PHASE_DECODE) {
    take = 1;
    start = P + gen - 1;
  } else if (phase == PHASE_PREFILL) {
    const long long left = (long long)c.chunk - before;
    take = (int)max(0ll, min((long long)(P - prefilled), left));
    start = prefilled;
  }
  const int f = take > 0;
  const int new_len = start + take;
  const int want = f ? (new_len + c.bs - 1) / c.bs - have : 0;
  const int sample = f && (phase == PHASE_DECODE || new_len == P);
  // attention work lists: single-row requests stream their KV blocks, multi-row requests are
  // cut into blocks of 128 / n_rep query rows
  const int q_rows = 128 / c.n_rep;
  const int is_dec = f && take == 1;
  const int nkb_att = is_dec ? (new_len + c.bs - 1) / c.bs : 0;
  const int n_blk = f && take > 1 ? (take + q_rows - 1) / q_rows : 0;
  const bool pairs_ok = c.att_pair && take > 1 && att_on_pairs(new_len);
  // (entries 7 and 8: blocks that post_step may free at most, and tickets that may end, by completion or
  // cancellation, for the trace space check; 6, 9 and 10: blocks of query rows for single CTAs, for CTA pairs, the latter in blocks for
  // single CTAs; the upper half of 8: requests for the pairs that have a long context)
  const int is_long = pairs_ok && new_len > ATT_ONE_ROUND_KEYS;
  int sc[11] = {f, take, want, sample, is_dec, nkb_att, pairs_ok ? 0 : n_blk, phase != PHASE_FREE ? have + want : 0, (phase != PHASE_FREE ? 1 : 0) | is_long << 16,
                pairs_ok ? (take + ATT_PAIR_ROWS - 1) / ATT_PAIR_ROWS : 0, pairs_ok ? n_blk : 0};
  int sc_tot[11];
  block_exscan(sc, sc_tot);
  const int n_ctas = c.n_warps_grid / (CTRL_THREADS / 32);
  const bool no_pairs = att_one_round_on_ctas(sc_tot[9] * c.Hkv, (sc_tot[6] + sc_tot[10]) * c.Hkv, n_ctas, sc_tot[8] >> 16 ? ATT_ONE_ROUND_KEYS + 1 : 0);
  const bool on_pairs = pairs_ok && !no_pairs;
  const int n_qp = on_pairs ? (take + ATT_PAIR_ROWS - 1) / ATT_PAIR_ROWS : 0, n_qb = on_pairs ? 0 : n_blk;
  const int n_pp = no_pairs ? 0 : sc_tot[9], n_pf = sc_tot[6] + (no_pairs ? sc_tot[10] : 0);
  const int item = sc[0], qstart = sc[1], aoff = sc[2], row = sc[3], dec_idx = sc[4], kb_pre = sc[5],
            pf_off = on_pairs ? sc[9] : n_pp + sc[6] + (no_pairs ? sc[10] : 0);
  const int n_items = sc_tot[0], T = sc_tot[1], n_alloc = sc_tot[2], n_rows = sc_tot[3], n_dec_att = sc_tot[4], tot_kb = sc_tot[5],
            tot_may_free = sc_tot[7], n_live = sc_tot[8] & 0xffff;

  if (T == 0) return 0;  // uniform: every thread sees the same T

  if (tid == 0) {
    int ok = 1;
    if (hdr >= 0) {
      const long long worst = hdr + TRACE_HDR_WORDS + 2ll * n_admit + 5ll * n_items + 3ll * n_alloc + 2ll * n_rows +
                              n_live + tot_may_free;
      if (worst > c.trace_cap) {
        ok = 0;
        ss->trace_off = 1;
        atomicCAS((int*)&c.mbox->device_status, 0, DEV_ERR_TRACE_OVERFLOW);
      }
    }
    s_trace_ok = ok;
    if (ss->free_top < n_alloc) dev_fail(c, DEV_ERR_STACK_UNDERFLOW);
  }
  __syncthreads();
  if (ss->free_top < n_alloc) return 0;
  const bool tr = hdr >= 0 && s_trace_ok;
  int32_t* rec_sched = rec + TRACE_HDR_WORDS + 2 * n_admit;
  int32_t* rec_alloc = rec_sched + 5 * n_items;

  // 3. allocate: ascending batch slot, the stack pops from its top
  const int top = ss->free_top;
  if (f) {
    for (int j = 0; j < want; ++j) {
      const int blk = c.free_stack[top - 1 - (aoff + j)];
      c.block_table[(size_t)tid * c.max_blocks_seq + have + j] = blk;
      if (tr) {
        rec_alloc[3 * (aoff + j)] = tid;
        rec_alloc[3 * (aoff + j) + 1] = have + j;
        rec_alloc[3 * (aoff + j) + 2] = blk;
      }
    }
    c.b_have[tid] = have + want;
    c.it_bslot[item] = tid;
    c.it_start[item] = start;
    c.it_ntok[item] = take;
    c.it_qstart[item] = qstart;
    c.it_row[item] = sample ? row : -1;
    s_qstart[item] = qstart;
    s_item_b[item] = tid;
    if (sample) {
      c.row_tok[row] = qstart + take - 1;
      c.row_item[row] = item;
      const float tp = c.b_topp[tid];
      if (c.b_topk[tid] <= 0 && tp > 0.f && tp < 1.f) s_nuc = 1;
    }
    if (c.dec_row != nullptr) {
      if (is_dec) {
        c.dec_row[dec_idx] = qstart;
        c.dec_bslot[dec_idx] = tid;
        c.dec_nctx[dec_idx] = new_len;
        c.dec_kbpre[dec_idx] = kb_pre;
        s_nkb[dec_idx] = nkb_att;
        atomicMax(&s_maxkb, nkb_att);
      }
      for (int q = 0; q < n_qb + n_qp; ++q) {   // (one of the two is zero) heaviest (last) row block first
        c.pf_item[pf_off + q] = item;
        c.pf_qb[pf_off + q] = n_qb + n_qp - 1 - q;
        if (n_qp > 0) c.pf_unit[pf_off + q] = make_int4(start, take, qstart, tid);
      }
    }
    if (tr) {
      rec_sched[5 * item] = tid;
      rec_sched[5 * item + 1] = (int32_t)ticket;
      rec_sched[5 * item + 2] = phase;
      rec_sched[5 * item + 3] = start;
      rec_sched[5 * item + 4] = take;
    }
    unsigned long long ctx = (phase == PHASE_DECODE) ? (unsigned long long)(start + 1)
                                                     : (unsigned long long)take * start +
                                                           (unsigned long long)take * (take + 1) / 2;
    atomicAdd(&s_ctx, ctx);
    atomicAdd(&s_kv, (unsigned long long)new_len);
    if (phase == PHASE_DECODE) atomicAdd(&s_ndec, 1);
  }
  if (tid == 0) s_qstart[n_items] = T;
  __threadfence();
  __syncthreads();

  // CTA-wide decode attention for few units: the smallest part size (of 32 candidates from a fair share up, at
  // least 24 tiles: a cut unit costs a merge through memory, about the time of three tiles per warp) whose parts fit
  // the grid at once; when none does, units stay whole
  if (tid < 32 && c.dec_row != nullptr && n_dec_att > 0 && n_dec_att * c.Hkv <= 2 * n_ctas) {
    const int share = max(24, (tot_kb * c.Hkv + n_ctas - 1) / n_ctas);
    const int C = share + tid * ((share + 7) / 8);
    int parts = 0;
    for (int i = 0; i < n_dec_att; ++i) parts += (s_nkb[i] + C - 1) / C;
    const unsigned fit = __ballot_sync(0xffffffffu, parts * c.Hkv <= n_ctas);
    const int pick = fit ? __ffs(fit) - 1 : 31;
    if (tid == pick) {
      s_C = fit ? C : s_maxkb;
      s_Citems = fit ? parts * c.Hkv : n_dec_att * c.Hkv;
    }
  }

  // per-row metadata: token id, position, owning item, KV slot
  // every warp of the grid starts on the sub-range of its own index; the counter hands out the rest
  if (c.att_ctr != nullptr)
    for (int i = tid; i < c.L; i += CTRL_THREADS) c.att_ctr[i] = c.n_warps_grid;
  for (int r = tid; r < T; r += CTRL_THREADS) {
    int lo = 0, hi = n_items;  // last item with qstart <= r
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (s_qstart[mid] <= r) lo = mid; else hi = mid;
    }
    const int b = s_item_b[lo];
    const int st = c.it_start[lo];
    const int pos = st + (r - s_qstart[lo]);
    int32_t tok;
    if (c.b_phase[b] == PHASE_DECODE) tok = c.b_last[b];
    else tok = c.in_arena[(size_t)c.b_slot[b] * c.max_prompt + pos];
    c.tok_id[r] = tok;
    c.tok_pos[r] = pos;
    c.tok_item[r] = lo;
    c.tok_slotmap[r] = c.block_table[(size_t)b * c.max_blocks_seq + pos / c.bs] * c.bs + pos % c.bs;
  }
  __syncthreads();
  if (tid == 0) {
    ss->free_top = top - n_alloc;
    ss->cur_T = T;
    ss->cur_items = n_items;
    ss->cur_rows = n_rows;
    ss->cur_decode = s_ndec;
    ss->cur_nuc = s_nuc;
    ss->cur_ctx = (long long)s_ctx;
    ss->cur_kv = (long long)s_kv;
    ss->cur_t_begin = t_begin;
    ss->pending_post = 1;
    ss->last_was_prefill = prefill_turn ? 1 : 0;
    if (c.dec_row != nullptr) {
      const long long TT = (long long)tot_kb * c.Hkv;
      const AttDecodeWay way =
          att_decode_way({TT, n_dec_att * c.Hkv, s_maxkb, s_C, s_Citems, n_ctas, CTRL_THREADS / 32, n_pf + n_pp > 0, c.att_sub_max});
      // a decode step of few rows: the CTA-wide kernel also applies RoPE and writes the new keys and values
      const int fuse = c.dec_small && T <= DEC_SMALL_ROWS && n_pf + n_pp == 0 && s_C > 0;
      ss->cur_fuse = fuse;
      c.dec_kbpre[n_dec_att] = tot_kb;
      ss->cur_ndec = n_dec_att;
      ss->cur_TT = (int)TT;
      ss->cur_S = (int)way.S;
      ss->cur_C = fuse ? s_C : way.C;
      ss->cur_half = way.half;
      ss->cur_npf = n_pf;
      ss->cur_npp = n_pp;
    }
    if (tr) {
      rec[0] = TRACE_MAGIC;
      rec[1] = (int32_t)ss->iter;
      rec[2] = (int32_t)((long long)visible - 1);
      rec[3] = n_admit;
      rec[4] = n_items;
      rec[5] = n_alloc;
      ss->cur_hdr = hdr;
      ss->cur_post = hdr + TRACE_HDR_WORDS + 2ll * n_admit + 5ll * n_items + 3ll * n_alloc;
    } else {
      ss->cur_hdr = -1;
    }
    ss->cur_t_forward = global_timer_ns();
    __threadfence();
  }
  __syncthreads();
  return T;
}

// One pass of the control plane.  `launch_iters` counts the iterations this kernel
// launch has started.  Sets ss->cmd to CMD_RUN (a step was composed), CMD_EXIT
// (leave the GPU; reason in ss->exit_reason) or CMD_NONE (stepped mode, idle).
// (a function of its own: inlined, its code shares the register allocation of the dispatcher of the loop kernel,
// which then spills more on the path of every phase: 1-1.5 % of a decode step)
static __device__ __noinline__ void control_phase(const DevCtx& c, long long& launch_iters) {
  SchedState* ss = c.ss;
  const int tid = threadIdx.x;
  __shared__ int s_cmd;
  __shared__ int s_started;
  __shared__ int s_leave;
  __shared__ unsigned long long s_tail;
  if (ss->pending_post) post_step(c);
  const long long idle_t0 = clock64();   // (thread 0 compares)
  unsigned int spins = 0;
  while (true) {
    if (tid == 0) {
      int cmd = CMD_NONE;
      MailboxWords words{c.mbox};
      const MailboxView mail = read_mailbox(words, c.start_paused && launch_iters == 0);   // (a launch that has run a step has seen the start)
      if (mail.stop) { cmd = CMD_EXIT; ss->exit_reason = 2; }
      else if (*(volatile int*)&ss->abort_flag) { cmd = CMD_EXIT; ss->exit_reason = 5; }
      else if (c.iteration_budget > 0 && launch_iters >= c.iteration_budget) { cmd = CMD_EXIT; ss->exit_reason = 3; }
      s_cmd = cmd;
      s_tail = cmd == CMD_NONE && mail.started ? mail.tail : ss->seen;
      s_started = mail.started;
    }
    __syncthreads();
    if (s_cmd == CMD_EXIT) break;
    const unsigned long long tail = s_tail;
    const bool started = s_started != 0;
    int T = 0;
    if (started) {
      if (tail > ss->seen) {   // slots become pending here and nowhere else
        ingress(c, tail);
        scan_and_claim(c);
      }
      T = schedule_step(c, ss->seen);
    }
    __syncthreads();
    if (T > 0) {
      if (tid == 0) s_cmd = CMD_RUN;
      launch_iters += 1;
      __syncthreads();
      break;
    }
    // One thread reads the flag (another CTA may raise it at any time) and the clock, so that the whole CTA takes the
    // same branch: with a clock of its own every warp may pass the limit in another turn, the barriers of the CTA then
    // no longer match and the kernel does not end.  Idle: poll the submit mailbox, leave the GPU when nothing comes.
    if (tid == 0) {
      const int reason = *(volatile int*)&ss->abort_flag ? 5 : !c.stepped && (unsigned long long)(clock64() - idle_t0) > c.idle_exit_cycles ? 4 : 0;
      if (reason) { s_cmd = CMD_EXIT; ss->exit_reason = reason; }
      s_leave = reason != 0 || c.stepped;   // (stepped: CMD_NONE)
    }
    __syncthreads();
    if (s_leave) break;
    if (++spins > 16) __nanosleep(1000);
    __syncthreads();
  }
  if (tid == 0) {
    ss->cmd = s_cmd;
    __threadfence();
  }
  __syncthreads();
}

}  // namespace blink
