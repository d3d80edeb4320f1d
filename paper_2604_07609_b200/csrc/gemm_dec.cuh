// Dense contractions of decode-sized steps (up to 128 token rows): the weights are the work, so they keep coming.
//
// The GEMM phases of gemm_tc.cuh start with an empty pipeline: a phase of a one-row step spends about 4 us until its
// first MMA and 3 us from its last one to the next phase, and between two GEMMs lie element-wise phases of 3 to 6 us
// each, while HBM idles (8B shape, one row: 112 us per layer for 67 us of weight streaming).  Here
//   * weights have a shared-memory ring of their own (4 stages of 32 KiB), and the weight producer of a GEMM goes on
//     with the first stages of the NEXT GEMM as the last stages of its own are released, so that 19 MB of the next
//     weights arrive during the tail, the grid barrier and whatever lies between the two GEMMs (prefetching more of
//     them into L2 as well gained nothing at 4, 8 and 16 further stages);
//   * steps of up to 16 rows have no norm, SwiGLU and final-norm phases: every CTA makes the token operand it needs
//     itself (normed rows, or silu(gate) * up of its own K range) and keeps it in shared memory for the whole phase
//     (1 KiB per k-block and CTA of a pair).  The rows are a few KiB to read; a phase and its grid barrier cost more;
//   * steps of 17 to 128 rows bring their token tiles through a second ring by TMA, as gemm_tc.cuh does.
// Geometry (who computes what) is that of tc_geom, taken once per step for all five GEMMs.
// Loops of unknown length stay rolled (a quarter less code for the instruction cache of 32 KB; the times are the same).
#pragma once
#include "gemm_tc.cuh"

namespace blink {

constexpr int DEC_MID_ROWS = 128;
static_assert(DEC_SMALL_ROWS == 16, "made operands are two groups of eight rows");
constexpr int DEC_STAGES = 4, DEC_STAGE_BYTES = 2 * TC_A_BYTES;   // two k-blocks of a 128-row weight tile
constexpr int DEC_B_OFF = DEC_STAGES * DEC_STAGE_BYTES, DEC_B_BYTES = 65536;
constexpr int DEC_B_STAGES = 8;
static_assert(DEC_B_OFF + DEC_B_BYTES <= TC_TILE_BUDGET, "rings exceed the dynamic shared memory");

struct DecShared {
  TcGeom g[GEMM_KINDS];
  uint64_t a_full[DEC_STAGES], a_empty[DEC_STAGES];
  uint64_t b_full[DEC_B_STAGES], b_empty[DEC_B_STAGES];   // token ring (17 rows and more)
  uint64_t b_made;    // token operand made by the CTAs themselves: one arrival per CTA, counted in CTA 0 of a pair
  uint64_t b_loaded;  // token operand of the O projection brought whole by TMA
};
__shared__ __align__(8) DecShared g_dec;

// per-warp bookkeeping (parities), see TcState
struct DecState {
  uint32_t fill_a, use_a, fill_b, use_b, made, loaded;
  int pre;   // weight producer: stages of the coming GEMM that are already on their way
};

__shared__ DecState g_dec_state[FWD_THREADS / 32];

template <bool PAIR>
__device__ __forceinline__ void dec_init(const DevCtx& c) {
  if ((threadIdx.x & 31) == 0) g_dec_state[threadIdx.x >> 5] = DecState{0u, 0u, 0u, 0u, 0u, 0u, 0};
  if (!c.gemm_tc) return;
  if (threadIdx.x == 32) {
    for (int i = 0; i < DEC_STAGES; ++i) { mbar_init(&g_dec.a_full[i], 1); mbar_init(&g_dec.a_empty[i], 1); }
    for (int i = 0; i < DEC_B_STAGES; ++i) { mbar_init(&g_dec.b_full[i], 1); mbar_init(&g_dec.b_empty[i], 1); }
    mbar_init(&g_dec.b_made, PAIR ? 2 : 1);
    mbar_init(&g_dec.b_loaded, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
}
// The loop may be abandoned between two GEMMs: wait (bounded) for weights that are still on their way into this CTA's
// shared memory.  Run by warp 0 of every CTA, before the cluster's last barrier.
template <bool PAIR>
__device__ __forceinline__ void dec_drain(const DevCtx& c, uint32_t rank) {
  if (!c.gemm_tc || (threadIdx.x >> 5) != 0) return;
  const DecState s = g_dec_state[0];
  if (!PAIR || rank == 0) {   // all bytes of a pair are counted in CTA 0
    const long long t0 = clock64();
    for (int i = 0; i < s.pre; ++i)
      while (!mbar_try_wait(&g_dec.a_full[i], ((s.fill_a >> i) & 1u) ^ 1u) && clock64() - t0 < 200000000ll) {}
  }
}

__device__ __forceinline__ bool dec_small(const DevCtx& c, int T) { return c.dec_small && T <= DEC_SMALL_ROWS; }
__device__ __forceinline__ bool dec_step(const DevCtx& c, int T) { return dec_small(c, T) || (c.dec_mid && T <= DEC_MID_ROWS); }

__device__ __forceinline__ int dec_n(const DevCtx& c, int which) {
  return which == GEMM_QKV ? c.qkv_dim : which == GEMM_GU ? 2 * c.F : which == GEMM_LMHEAD ? c.V : c.d;
}
__device__ __forceinline__ int dec_k(const DevCtx& c, int which) {
  return which == GEMM_O ? c.q_dim : which == GEMM_DOWN ? c.F : c.d;
}
// Once per step, by five threads; the caller synchronises the CTA afterwards.
template <bool PAIR>
__device__ __forceinline__ void dec_geometry(const DevCtx& c, int T, int R) {
  const int which = threadIdx.x;
  if (which < GEMM_KINDS) {
    const int rows = which == GEMM_LMHEAD ? R : T, N = dec_n(c, which);
    const int tiles = (N + 127) / 128;
    g_dec.g[which] = tc_geom(c, max(rows, 1), N, dec_k(c, which), which == GEMM_LMHEAD && lm_head_whole_tiles(c),
                             PAIR ? (int)gridDim.x / 2 : (int)gridDim.x, PAIR ? (int)blockIdx.x / 2 : (int)blockIdx.x,
                             PAIR ? (tiles + 1) / 2 : tiles, PAIR, 1);
  }
}

// Weight producer (warp 0): stage-sized pieces [first, first + count) of this CTA's range of a GEMM; piece i goes to
// stage i % DEC_STAGES.  Returns the number of pieces issued, and in the low four bits the new parities.
template <bool PAIR>
static __device__ __noinline__ int dec_fill_weights(const DevCtx& c, const TcGeom& g, int which, int layer, char* tiles, uint32_t fill_a,
                                                    uint32_t rank, int first, int count) {
  const TcMaps* maps = reinterpret_cast<const TcMaps*>(c.tc_maps);
  const uint64_t policy = l2_evict_first();
  const int row0 = which == GEMM_LMHEAD ? 0 : layer * dec_n(c, which);
  int i = 0, issued = 0;
#pragma unroll 1
  for (TcSeg sg = tc_seg_first(g); sg.left > 0; tc_seg_next(g, sg)) {
    const int nt = tc_my_tile<PAIR>(sg.nt, rank);
    const int tile0 = ((row0 >> 7) + nt) * g.kblocks;
    const int pieces = (sg.kb1 - sg.kb0 + 1) >> 1;
    if (i + pieces <= first) { i += pieces; continue; }
    int kb = sg.kb0;
    if (first > i) { kb += 2 * (first - i); i = first; }
#pragma unroll 1
    for (; kb < sg.kb1; kb += 2, ++i) {
      if (i >= first + count) return (issued << 4) | (int)fill_a;
      const int nk = min(2, sg.kb1 - kb), stage = i % DEC_STAGES;
      if (!mbar_wait_warp(c, &g_dec.a_empty[stage], ((fill_a >> stage) & 1u) ^ 1u)) return (issued << 4) | (int)fill_a;
      fill_a ^= 1u << stage;
      char* sa = tiles + stage * DEC_STAGE_BYTES;
      if (elect_one()) {
        uint64_t* bar = &g_dec.a_full[stage];
        if constexpr (PAIR) {
          if (rank == 0) mbar_expect_tx(bar, 2u * (uint32_t)nk * TC_A_BYTES);
          if (c.w_streaming) {
            tma_pair_load_3d(sa, &maps->ws[which][nk - 1], 0, 0, tile0 + kb, bar, policy);
          } else {
            for (int j = 0; j < nk; ++j)
              tma_pair_load_2d(sa + j * TC_A_BYTES, &maps->w[which], (kb + j) * 64, row0 + nt * 128, bar, policy);
          }
        } else {
          mbar_expect_tx(bar, (uint32_t)nk * TC_A_BYTES);
          if (c.w_streaming) {
            tma_load_3d_hint(sa, &maps->ws[which][nk - 1], 0, 0, tile0 + kb, bar, policy);
          } else {
            for (int j = 0; j < nk; ++j)
              tma_load_2d_hint(sa + j * TC_A_BYTES, &maps->w[which], (kb + j) * 64, row0 + nt * 128, bar, policy);
          }
        }
      }
      ++issued;
    }
  }
  return (issued << 4) | (int)fill_a;
}

// ---- token operands made by the CTA --------------------------------------------------------------------------
// Slot i of the operand holds the k-block of the i-th unit of the CTA's range (a range longer than K wraps round), so
// a CTA makes only the k-blocks it will use.  Inside a slot: 8 rows of 128 bytes, 16-byte chunks swizzled by the row.
// Of a pair, CTA r makes the rows of tokens r, r + 2, r + 4, ..: column j of the accumulator then belongs to token
// dec_token(j), and a step of few rows is halved between the two.
struct DecSlots {
  int kb_first, kblocks, n, bytes;   // first k-block, k-blocks of K, slots, bytes of a slot
};
template <bool PAIR>
__device__ __forceinline__ int dec_token(int j) { return PAIR ? ((j & 7) << 1) | (j >> 3) : j; }
template <bool PAIR>
__device__ __forceinline__ int dec_rows_here(int rows, uint32_t rank) { return PAIR ? (rows - (int)rank + 1) >> 1 : rows; }
template <bool PAIR>
__device__ __forceinline__ DecSlots dec_slots(const TcGeom& g) {
  DecSlots d;
  d.kblocks = g.kblocks;
  d.kb_first = (int)((unsigned)g.u0 % (unsigned)g.kblocks);
  d.n = min(g.u1 - g.u0, g.kblocks);
  d.bytes = PAIR ? 1024 : 2048;
  return d;
}
__device__ __forceinline__ int dec_slot_of(const DecSlots& d, int kb) {   // may be >= n: not needed by this CTA
  const int s = kb - d.kb_first;
  return s < 0 ? s + d.kblocks : s;
}

// RMSNorm of the step's rows into the operand slots, 8 / NV rows at a time by the whole CTA (NV vectors of 4 per thread
// and row; the gains are loaded once).  The code of a phase comes from beyond the instruction cache every time, so
// short code beats unrolled code here: with 64 elements per thread and everything unrolled the stores alone took 3.4 us.
template <bool PAIR, int NV>
static __device__ __noinline__ void dec_make_normed(const DevCtx& c, int which, int layer, int rows, const DecSlots sl, char* bt,
                                                    uint32_t rank) {
  constexpr int WARPS = FWD_THREADS / 32, RP = 8 / NV;
  __shared__ float s_ss[2][WARPS][8];
  const int tid = threadIdx.x;
  const int d = c.d;
  const int n_here = dec_rows_here<PAIR>(rows, rank);
  const bool embed = which == GEMM_QKV && layer == 0;
  const bool live = tid * 4 < d;   // d = 256: the first two warps
  const float* g = which == GEMM_QKV ? wptr_f(c, 6) + (size_t)layer * d : which == GEMM_GU ? wptr_f(c, 7) + (size_t)layer * d
                                                                                          : wptr_f(c, 8);
  float4 gg[NV];
  if (live)
#pragma unroll
    for (int k = 0; k < NV; ++k) gg[k] = __ldg(reinterpret_cast<const float4*>(g + tid * 4 + k * 1024));
  const float inv_d = __fdividef(1.0f, (float)d);
  const int col = (tid & 15) * 4;
#pragma unroll 1
  for (int r0 = 0; r0 < n_here; r0 += RP) {   // uniform over the CTA
    float4 v[RP][NV];
    float ss[RP];
#pragma unroll
    for (int q = 0; q < RP; ++q) {
      const int r = min(r0 + q, n_here - 1), t = PAIR ? 2 * r + (int)rank : r;   // past the end: the last row again
      if (embed) {
        const __nv_bfloat16* e = wptr<__nv_bfloat16>(c, 0) + (size_t)c.tok_id[t] * d + tid * 4;
#pragma unroll
        for (int k = 0; k < NV; ++k) v[q][k] = live ? load4<__nv_bfloat16>(e + k * 1024) : make_float4(0.f, 0.f, 0.f, 0.f);
      } else {
        const float* h = c.h + (size_t)(which == GEMM_LMHEAD ? c.row_tok[t] : t) * d + tid * 4;
#pragma unroll
        for (int k = 0; k < NV; ++k)
          v[q][k] = live ? __ldcg(reinterpret_cast<const float4*>(h + k * 1024)) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
#pragma unroll
    for (int q = 0; q < RP; ++q) {
      ss[q] = 0.f;
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        ss[q] = fmaf(v[q][k].x, v[q][k].x, ss[q]); ss[q] = fmaf(v[q][k].y, v[q][k].y, ss[q]);
        ss[q] = fmaf(v[q][k].z, v[q][k].z, ss[q]); ss[q] = fmaf(v[q][k].w, v[q][k].w, ss[q]);
      }
    }
    float(*red)[8] = s_ss[(r0 / RP) & 1];   // two buffers: one barrier per round
    const float own = warp_sum_many<RP>(ss);
    if ((tid & (32 / RP - 1)) == 0) red[tid >> 5][(tid & 31) / (32 / RP)] = own;
    __syncthreads();
    if (live) {
#pragma unroll
      for (int q = 0; q < RP; ++q) {
        const int r = r0 + q;
        if (r < n_here) {
          float tot = 0.f;
#pragma unroll
          for (int i = 0; i < WARPS; ++i) tot += red[i][q];
          const float inv = rsqrtf(tot * inv_d + c.rms_eps);
          char* row = bt + (r >> 3) * 1024 + (r & 7) * 128 + (((col >> 3) ^ (r & 7)) << 4) + (col & 7) * 2;
          // the embedding row also goes into the residual stream, by one CTA
          const int t = PAIR ? 2 * r + (int)rank : r;
          const bool keep = embed && (int)blockIdx.x == t;
#pragma unroll
          for (int k = 0; k < NV; ++k) {
            const float4 x = v[q][k];
            if (keep) *reinterpret_cast<float4*>(c.h + (size_t)t * d + tid * 4 + k * 1024) = x;
            const int slot = dec_slot_of(sl, k * 16 + (tid >> 4));
            if (slot < sl.n)
              store4<__nv_bfloat16>(reinterpret_cast<__nv_bfloat16*>(row + slot * sl.bytes), x.x * inv * gg[k].x, x.y * inv * gg[k].y,
                                    x.z * inv * gg[k].z, x.w * inv * gg[k].w);
          }
        }
      }
    }
  }
}
// silu(gate) * up of the step's rows into the operand slots of the down projection
template <bool PAIR>
static __device__ __noinline__ void dec_make_silu(const DevCtx& c, int rows, const DecSlots sl, char* bt, uint32_t rank) {
  constexpr int U = 2;
  const int nr = dec_rows_here<PAIR>(rows, rank);
  const int per_row = sl.n * 8, total = nr * per_row;   // items of 8 features
  for (int base = FWD_THREADS - 1 - threadIdx.x; base < total; base += U * FWD_THREADS) {   // warp 0, busy with the weights, last
    float4 g[U][2], u[U][2];
    int dst[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int idx = min(base + k * FWD_THREADS, total - 1);   // clamped: the tail repeats the last item
      const int r = (int)((unsigned)idx / (unsigned)per_row), q = idx - r * per_row;
      const int slot = q >> 3, c8 = q & 7;
      int kb = sl.kb_first + slot;
      if (kb >= sl.kblocks) kb -= sl.kblocks;
      const float* src = c.gu + (size_t)(PAIR ? 2 * r + (int)rank : r) * 2 * c.F + kb * 64 + c8 * 8;
      dst[k] = slot * sl.bytes + (r >> 3) * 1024 + (r & 7) * 128 + ((c8 ^ (r & 7)) << 4);
      g[k][0] = __ldcg(reinterpret_cast<const float4*>(src));
      g[k][1] = __ldcg(reinterpret_cast<const float4*>(src) + 1);
      u[k][0] = __ldcg(reinterpret_cast<const float4*>(src + c.F));
      u[k][1] = __ldcg(reinterpret_cast<const float4*>(src + c.F) + 1);
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
      uint4 o;
      uint32_t* ow = reinterpret_cast<uint32_t*>(&o);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float4 a = g[k][e], b = u[k][e];
        const __nv_bfloat162 lo = __floats2bfloat162_rn(__fdividef(a.x, 1.0f + __expf(-a.x)) * b.x, __fdividef(a.y, 1.0f + __expf(-a.y)) * b.y);
        const __nv_bfloat162 hi = __floats2bfloat162_rn(__fdividef(a.z, 1.0f + __expf(-a.z)) * b.z, __fdividef(a.w, 1.0f + __expf(-a.w)) * b.w);
        ow[2 * e] = *reinterpret_cast<const uint32_t*>(&lo);
        ow[2 * e + 1] = *reinterpret_cast<const uint32_t*>(&hi);
      }
      *reinterpret_cast<uint4*>(bt + dst[k]) = o;
    }
  }
}

// What the roles of a phase share.
struct DecPhase {
  int which, layer, rows;
  bool made, loaded;   // token operand made by the CTAs / brought whole by TMA; neither: ring
};

// MMA issuer (warp 1 of CTA 0)
template <bool PAIR>
__device__ __forceinline__ void dec_issue_mmas(const DevCtx& c, const DecPhase& p, const TcGeom& g, char* tiles, TcState& tc,
                                               DecState& s) {
  const int n_mma = (p.rows + 15) & ~15;   // one token pass
  const uint32_t idesc = PAIR ? idesc_bf16_pair(n_mma) : idesc_bf16(n_mma);
  const uint64_t desc_a = smem_desc_sw128(smem_u32(tiles)), desc_b = smem_desc_sw128(smem_u32(tiles + DEC_B_OFF));
  const bool ring = !p.made && !p.loaded;
  const uint32_t slot_step = (PAIR ? 1024u : 2048u) >> 4, b_step = g.b_bytes >> 4;
  const int nb = min(DEC_B_STAGES, (int)((unsigned)DEC_B_BYTES / (2u * g.b_bytes)));
  const int slots = min(g.u1 - g.u0, g.kblocks);
  if (g.u0 < g.u1) {
    if (p.made) {
      if (!(PAIR ? mbar_wait_warp_acquire(c, &g_dec.b_made, s.made & 1u) : mbar_wait_warp(c, &g_dec.b_made, s.made & 1u))) return;
    } else if (p.loaded) {
      if (!mbar_wait_warp(c, &g_dec.b_loaded, s.loaded & 1u)) return;
    }
  }
  int piece = 0, bstage = 0, slot = 0, abuf = 0;
#pragma unroll 1
  for (TcSeg sg = tc_seg_first(g); sg.left > 0; tc_seg_next(g, sg)) {
    const uint32_t d_tmem = tc.tmem_base + (uint32_t)abuf * 256u;
    if (!mbar_wait_warp(c, &g_tc.acc_empty[abuf], ((tc.acc_mma >> abuf) & 1u) ^ 1u)) return;
    tc.acc_mma ^= 1u << abuf;
    tc_fence_after();
#pragma unroll 1
    for (int kb = sg.kb0; kb < sg.kb1; kb += 2, ++piece) {
      const int stage = piece % DEC_STAGES;
      const bool two = kb + 1 < sg.kb1;
      if (ring) {
        if (!mbar_wait_warp(c, &g_dec.b_full[bstage], (s.use_b >> bstage) & 1u)) return;
        s.use_b ^= 1u << bstage;
      }
      if (!mbar_wait_warp(c, &g_dec.a_full[stage], (s.use_a >> stage) & 1u)) return;
      s.use_a ^= 1u << stage;
      tc_fence_after();
      const uint64_t da = desc_a + (uint64_t)(uint32_t)(stage * (DEC_STAGE_BYTES >> 4));
      const int slot1 = slot + 1 == slots ? 0 : slot + 1;
      const uint64_t db = desc_b + (uint64_t)(ring ? (uint32_t)bstage * 2u * b_step : (uint32_t)slot * slot_step);
      const uint64_t db1 = desc_b + (uint64_t)(ring ? (uint32_t)bstage * 2u * b_step + b_step : (uint32_t)slot1 * slot_step);
      const uint32_t more = kb > sg.kb0 ? 1u : 0u;
      if (elect_one()) {
#pragma unroll
        for (int k16 = 0; k16 < 4; ++k16) {
          if constexpr (PAIR) umma_bf16_pair(d_tmem, da + (uint64_t)(2 * k16), db + (uint64_t)(2 * k16), idesc, k16 ? 1u : more);
          else umma_bf16(d_tmem, da + (uint64_t)(2 * k16), db + (uint64_t)(2 * k16), idesc, k16 ? 1u : more);
        }
        if (two) {
          const uint64_t da1 = da + (uint64_t)(TC_A_BYTES >> 4);
#pragma unroll
          for (int k16 = 0; k16 < 4; ++k16) {
            if constexpr (PAIR) umma_bf16_pair(d_tmem, da1 + (uint64_t)(2 * k16), db1 + (uint64_t)(2 * k16), idesc, 1u);
            else umma_bf16(d_tmem, da1 + (uint64_t)(2 * k16), db1 + (uint64_t)(2 * k16), idesc, 1u);
          }
        }
        if constexpr (PAIR) {
          umma_commit_pair(&g_dec.a_empty[stage]);
          if (ring) umma_commit_pair(&g_dec.b_empty[bstage]);
        } else {
          umma_commit(&g_dec.a_empty[stage]);
          if (ring) umma_commit(&g_dec.b_empty[bstage]);
        }
      }
      __syncwarp();
      if (++bstage == nb) bstage = 0;
      slot = two ? (slot1 + 1 == slots ? 0 : slot1 + 1) : slot1;
    }
    if (elect_one()) {
      if constexpr (PAIR) umma_commit_pair(&g_tc.acc_full[abuf]);
      else umma_commit(&g_tc.acc_full[abuf]);
    }
    __syncwarp();
    abuf ^= 1;
  }
}

// Token tiles by TMA (warp 2): through the ring, or (O projection of a small step) all of the range's k-blocks at once.
template <bool PAIR>
__device__ __forceinline__ void dec_load_tokens(const DevCtx& c, const DecPhase& p, const TcGeom& g, char* tiles, DecState& s,
                                                uint32_t rank) {
  const TcMaps* maps = reinterpret_cast<const TcMaps*>(c.tc_maps);
  const int act_id = p.which == GEMM_O ? ACT_ATTN : p.which == GEMM_DOWN ? ACT_ACT : p.which == GEMM_LMHEAD ? ACT_XS : ACT_XN;
  const uint64_t keep_policy = l2_evict_normal();
  const int n_mma = (p.rows + 15) & ~15;
  const int row0 = PAIR ? (int)rank * (n_mma / 2) : 0;
  char* bt = tiles + DEC_B_OFF;
  if (p.loaded) {
    const DecSlots sl = dec_slots<PAIR>(g);
    if (sl.n <= 0) return;
    const CUtensorMap* map = &maps->act[act_id][PAIR ? 0 : 1];   // 8 or 16 rows
    if (elect_one()) {
      if (!PAIR || rank == 0) mbar_expect_tx(&g_dec.b_loaded, (PAIR ? 2u : 1u) * (uint32_t)(sl.n * sl.bytes));
#pragma unroll 1
      for (int i = 0, kb = sl.kb_first; i < sl.n; ++i) {
        if constexpr (PAIR) tma_pair_load_2d(bt + i * sl.bytes, map, kb * 64, row0, &g_dec.b_loaded, keep_policy);
        else tma_load_2d(bt + i * sl.bytes, map, kb * 64, row0, &g_dec.b_loaded);
        if (++kb == sl.kblocks) kb = 0;
      }
    }
    return;
  }
  const CUtensorMap* map = &maps->act[act_id][g.load_box];
  const int nb = min(DEC_B_STAGES, (int)((unsigned)DEC_B_BYTES / (2u * g.b_bytes)));
  int bstage = 0;
#pragma unroll 1
  for (TcSeg sg = tc_seg_first(g); sg.left > 0; tc_seg_next(g, sg)) {
#pragma unroll 1
    for (int kb = sg.kb0; kb < sg.kb1; kb += 2) {
      const int nk = min(2, sg.kb1 - kb);
      if (!mbar_wait_warp(c, &g_dec.b_empty[bstage], ((s.fill_b >> bstage) & 1u) ^ 1u)) return;
      s.fill_b ^= 1u << bstage;
      char* sb = bt + (size_t)bstage * 2 * g.b_bytes;
      if (elect_one()) {
        if (!PAIR || rank == 0) mbar_expect_tx(&g_dec.b_full[bstage], (PAIR ? 2u : 1u) * (uint32_t)nk * g.b_bytes);
        for (int j = 0; j < nk; ++j) {
          if constexpr (PAIR) tma_pair_load_2d(sb + j * g.b_bytes, map, (kb + j) * 64, row0, &g_dec.b_full[bstage], keep_policy);
          else tma_load_2d(sb + j * g.b_bytes, map, (kb + j) * 64, row0, &g_dec.b_full[bstage]);
        }
      }
      if (++bstage == nb) bstage = 0;
    }
  }
}

// The 16 columns of an accumulator whose token operand was made by the CTAs -> out
template <bool PAIR>
__device__ __forceinline__ void dec_epi_made(const TcEpiOut& e, uint32_t taddr, int n, bool plain) {
  float v[16];
  tmem_ld16(taddr, v);
  if (n >= e.N) return;
  float* o = e.out + (e.ilv_F ? (n & 1) * e.ilv_F + (n >> 1) : n);
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int t = dec_token<PAIR>(j);
    if (t < e.T) {
      if (plain) o[(size_t)t * e.ldo] = v[j];
      else red_add_f32(o + (size_t)t * e.ldo, v[j]);
    }
  }
}

// The grid barrier after a GEMM of a decode-sized step.  Warp 0 may still be bringing weights of the next GEMM (it has
// nothing in memory that the grid waits for): the others arrive without it.
static __device__ __noinline__ bool dec_barrier(const DevCtx& c) {
  if (threadIdx.x >= 32) {
    fence_proxy_async_global();
    asm volatile("bar.sync 3, %0;" ::"n"(FWD_THREADS - 32) : "memory");
    if (threadIdx.x == 32) g_bar_ok = grid_arrive_and_wait(c) ? 1 : 0;
  }
  __syncthreads();
  fence_proxy_async_global();
  return g_bar_ok != 0;
}

// One GEMM of a decode-sized step.  `next_which` (or -1): the GEMM whose weights follow; `next_pre`: how many of its
// stages may be filled before it starts.
template <bool PAIR>
static __device__ __noinline__ void phase_gemm_dec(const DevCtx& c, int which, int layer, int T, int R, int next_which, int next_pre,
                                                   float* smem_f) {
  const TcGeom g = g_dec.g[which];
  const bool small = dec_small(c, T);
  DecPhase p;
  p.which = which;
  p.layer = layer;
  p.rows = which == GEMM_LMHEAD ? R : T;
  p.loaded = small && which == GEMM_O;
  p.made = small && which != GEMM_O && !(c.E > 0 && which != GEMM_QKV && which != GEMM_LMHEAD);
  const uint32_t rank = PAIR ? cluster_ctarank() : 0u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  char* tiles = tc_tiles(smem_f);
  TcState tc = g_tc_state[warp];
  DecState s = g_dec_state[warp];
  auto fill = [&](int w, int l, int from, int count) {   // (warp 0)
    const int r = dec_fill_weights<PAIR>(c, g_dec.g[w], w, l, tiles, s.fill_a, rank, from, count);
    s.fill_a = (uint32_t)r & 15u;
    return r >> 4;
  };
  // Small steps have no phases that clear what the split-K GEMMs add into: gate/up rows (read by the down projection of
  // the layer before) are cleared in the QKV and LM head phases, QKV rows (read by the attention) in the O phase, and in
  // the last of those the logits, where the LM head splits K.
  const bool clear_gu = small && c.E == 0 && ((which == GEMM_QKV && layer > 0) || which == GEMM_LMHEAD);
  if (p.rows <= 0) {   // uniform over the grid: no row samples (and nothing has been prefetched for it)
    if (clear_gu) zero_floats(c.gu, (long long)T * 2 * c.F);
    return;
  }

  int first = 0;
  if (warp == 0) {   // whatever the phase before could not bring yet
    first = s.pre;
    if (first < DEC_STAGES) first += fill(which, layer, first, DEC_STAGES - first);
    s.pre = 0;
  }
  if (p.made) {
    const DecSlots sl = dec_slots<PAIR>(g);
    char* bt = tiles + DEC_B_OFF;
    if (sl.n > 0 || (which == GEMM_QKV && layer == 0)) {   // (no share of the GEMM, but perhaps an embedding row to copy)
      if (which == GEMM_DOWN) dec_make_silu<PAIR>(c, p.rows, sl, bt, rank);
      else if (c.d == 4096) dec_make_normed<PAIR, 4>(c, which, layer, p.rows, sl, bt, rank);
      else if (c.d == 2048) dec_make_normed<PAIR, 2>(c, which, layer, p.rows, sl, bt, rank);
      else dec_make_normed<PAIR, 1>(c, which, layer, p.rows, sl, bt, rank);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // read by the MMAs next
    __syncthreads();
    if (threadIdx.x == 0 && g.u0 < g.u1) {
      if constexpr (PAIR) mbar_arrive_cta0_release(&g_dec.b_made);   // the MMAs that read this CTA's half are issued by CTA 0
      else mbar_arrive(&g_dec.b_made);
    }
  }

  if (warp == 0) {
    fill(which, layer, first, 0x4000000);
    if (next_which >= 0 && *(volatile int*)&g_tc.dead == 0)
      s.pre = fill(next_which, next_which == GEMM_QKV ? layer + 1 : layer, 0, next_pre);
  } else if (warp == 2) {
    if (!p.made) dec_load_tokens<PAIR>(c, p, g, tiles, s, rank);
  } else if (warp == 1) {
    if (rank == 0) dec_issue_mmas<PAIR>(c, p, g, tiles, tc, s);
  } else if (warp >= 4) {
    const int id = blockIdx.x * 128 + (threadIdx.x - 128), n = gridDim.x * 128;
    if (small && (which == GEMM_O || which == GEMM_DOWN)) {   // the gains of the coming norm into L2, one line per thread
      const float* gn = which == GEMM_O ? wptr_f(c, 7) + (size_t)layer * c.d
                        : layer + 1 < c.L ? wptr_f(c, 6) + (size_t)(layer + 1) * c.d : wptr_f(c, 8);
#pragma unroll 1
      for (int i = id * 32; i < c.d; i += n * 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(gn + i));
    }
    if (clear_gu) {
      float4* q = reinterpret_cast<float4*>(c.gu);
#pragma unroll 1
      for (int i = id; i < T * c.F / 2; i += n) q[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    } else if (which == GEMM_O && small) {
      if (c.ss->cur_fuse) {   // (else the RoPE phase has cleared them)
        float4* q = reinterpret_cast<float4*>(c.qkv);
#pragma unroll 1
        for (int i = id; i < T * c.qkv_dim / 4; i += n) q[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
      if (layer == c.L - 1 && !lm_head_whole_tiles(c)) {
        float4* q = reinterpret_cast<float4*>(c.logits);
#pragma unroll 1
        for (int i = id; i < R * (c.V / 4); i += n) q[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    const int q = warp & 3;
    const bool accumulate = which == GEMM_O || which == GEMM_DOWN;
    float* out = which == GEMM_QKV ? c.qkv : which == GEMM_GU ? c.gu : which == GEMM_LMHEAD ? c.logits : c.h;
    const int N = dec_n(c, which);
    const TcEpiOut eo{out, (size_t)N, nullptr, nullptr, p.rows, N, (which == GEMM_GU && c.w_streaming) ? c.F : 0, nullptr};
    const int n_mma = (p.rows + 15) & ~15;
    int abuf = 0;
#pragma unroll 1
    for (TcSeg sg = tc_seg_first(g); sg.left > 0; tc_seg_next(g, sg)) {
      const int nt = tc_my_tile<PAIR>(sg.nt, rank);
      const bool plain = sg.kb0 == 0 && sg.kb1 == g.kblocks && !accumulate;
      if (!mbar_wait_warp(c, &g_tc.acc_full[abuf], (tc.acc_epi >> abuf) & 1u)) break;
      tc.acc_epi ^= 1u << abuf;
      tc_fence_after();
      const uint32_t taddr = tc.tmem_base + (uint32_t)abuf * 256u + ((uint32_t)(q * 32) << 16);
      if (p.made) dec_epi_made<PAIR>(eo, taddr, nt * 128 + q * 32 + lane, plain);
      else tc_epi_columns(eo, taddr, nt * 128 + q * 32 + lane, 0, 0, n_mma, plain);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if constexpr (PAIR) mbar_arrive_cta0(&g_tc.acc_empty[abuf]);
        else mbar_arrive(&g_tc.acc_empty[abuf]);
      }
      abuf ^= 1;
    }
  }
  __syncwarp();
  if (g.u0 < g.u1) {
    if (p.made) s.made ^= 1u;
    if (p.loaded) s.loaded ^= 1u;
  }
  if (lane == 0) {
    g_tc_state[warp] = tc;
    g_dec_state[warp] = s;
  }
  __syncwarp();   // (the grid barrier that follows brings the warps together)
}

// ---- host side: which steps may take this path --------------------------------------------------------------
// Up to 16 rows: every CTA's token operand has to fit (in k-blocks of its range of each GEMM), and the norm is built for
// four widths.  17 to 128 rows: CTA pairs only (a single CTA's token tile is twice as large, its ring too short).
inline void dec_host_setup(DevCtx& c, bool pair, int grid) {
  c.dec_small = c.dec_mid = 0;
  if (!c.gemm_tc || c.fused || c.control_only) return;
  const int nb = pair ? grid / 2 : grid;
  const int N[GEMM_KINDS] = {c.qkv_dim, c.d, 2 * c.F, c.d, c.V}, K[GEMM_KINDS] = {c.d, c.q_dim, c.d, c.F, c.d};
  bool fits = c.d == 256 || c.d == 1024 || c.d == 2048 || c.d == 4096;
  for (int i = 0; i < GEMM_KINDS; ++i) {
    if (c.E > 0 && (i == GEMM_GU || i == GEMM_DOWN)) continue;
    const int kblocks = K[i] / 64, tiles128 = (N[i] + 127) / 128, tiles = pair ? (tiles128 + 1) / 2 : tiles128;
    long long slots = ((long long)tiles * kblocks + nb - 1) / nb + 1;       // even shares
    const int split = nb / tiles;
    if (split >= 2 && (kblocks + split - 1) / split > slots) slots = (kblocks + split - 1) / split;   // whole CTAs per tile
    if (slots > kblocks || i == GEMM_LMHEAD) slots = kblocks;
    fits = fits && slots * (pair ? 1024 : 2048) <= DEC_B_BYTES;
  }
  c.dec_small = fits;
  c.dec_mid = pair;
}

}  // namespace blink
