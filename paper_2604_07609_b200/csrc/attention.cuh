// Paged attention of the bf16 data path (Section 4.2 / 6.1 of the paper: the engine's paged
// KV cache with decode attention and context attention inside the step).
//
// Two kinds of work share the phase:
//   * decode rows (one query token per request): bandwidth-bound.  All (row, kv head, KV block)
//     tiles of the step form one flat sequence that is cut into sub-ranges; warps fetch
//     sub-ranges from a counter, stream the 16-key K and V tiles (contiguous in the pool) into
//     a private shared-memory ring with TMA tile copies (mbarrier completion), and keep an
//     online softmax per (row, kv head) unit.  The query heads of a GQA group share every K/V
//     load.  A unit cut by a sub-range boundary leaves partial (m, l, acc) records; whoever
//     finishes the last part merges them in a fixed order.
//   * prefill-chunk rows (several query tokens of one request): a dense contraction, so it
//     runs on tensor cores (mma.sync m16n8k16, flash-attention style tiling): one CTA per
//     (request, block of query rows, kv head), 64-key K/V tiles through a double-buffered
//     cp.async pipeline, scores and probabilities in registers.  Requests of more than a few hundred keys
//     go to CTA pairs instead where the shape allows (attn_pair.cuh).
#pragma once
#include "attn_pair.cuh"
#include "gemm_tc.cuh"

namespace blink {

constexpr int ATT_NS = 3;  // ring stages per warp (decode path)
constexpr int ATT_WARPS = FWD_THREADS / 32;

struct AttShared {
  uint64_t bar[ATT_WARPS][ATT_NS];
  int ids[ATT_WARPS][8];
  int dead;
};
__shared__ __align__(8) AttShared g_att;
__shared__ int g_att_pre[MAX_BATCH + 1];   // prefix of KV blocks over the decode rows of the step
__shared__ int g_att_bslot[MAX_BATCH];
__shared__ int g_att_nctx[MAX_BATCH];
__shared__ int g_att_row[MAX_BATCH];
// the step's scalars: like the arrays above they do not change between layers and are read from memory once per step
struct AttStep {
  int n_dec, TT, S, C, half, npf, npp, fuse;   // (half: the units of C are for half CTAs)
};
__shared__ AttStep g_att_step;

__shared__ uint32_t g_att_par[ATT_WARPS];   // mbarrier parities of the warps' rings
__shared__ int g_att_blk[FWD_THREADS];      // CTA-wide decode: the lane's block id of the CTA's first item (the same in all layers of a step)

__device__ __forceinline__ void att_init(const DevCtx& c) {
  g_att_blk[threadIdx.x] = 0;
  if ((threadIdx.x & 31) == 0) g_att_par[threadIdx.x >> 5] = 0u;
  if (c.dtype != 0 || c.control_only) return;
  if ((threadIdx.x & 31) == 0) {
    for (int i = 0; i < ATT_NS; ++i) mbar_init(&g_att.bar[threadIdx.x >> 5][i], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x == 0) {
    g_att.dead = 0;
    ap_init();
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
}

__device__ __forceinline__ uint32_t pack_bf2(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
// one TMA tile copy from a rank-5 tensor map
__device__ __forceinline__ void tma_load_5d(void* smem_dst, const CUtensorMap* map, int c0, int c1, int c2, int c3, int c4,
                                            uint64_t* bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4, "
      "%5, %6}], [%7], %8;" ::"r"(smem_u32(smem_dst)),
      "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}

// flat tile sequence of the decode rows: unit (d, g) owns tiles [Hkv*pre[d] + g*nkb, +nkb)
struct DecCursor {
  int f, f_end;      // next tile and end of the current sub-range
  int d, g, kb, nkb; // decoded position of f
};
__device__ __forceinline__ void dec_seek(DecCursor& cur, int f, int f_end, int n_dec, int Hkv) {
  cur.f = f;
  cur.f_end = f_end;
  int lo = 0, hi = n_dec;  // last d with Hkv * pre[d] <= f
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (Hkv * g_att_pre[mid] <= f) lo = mid; else hi = mid;
  }
  cur.d = lo;
  cur.nkb = g_att_pre[lo + 1] - g_att_pre[lo];
  const int rem = f - Hkv * g_att_pre[lo];
  cur.g = rem / cur.nkb;
  cur.kb = rem - cur.g * cur.nkb;
}
// tiles [b0, b1) of sub-range `id`: S tiles of the flat sequence, or (S == 0) one whole unit
__device__ __forceinline__ void dec_sub_range(int id, int S, int TT, int Hkv, int& b0, int& b1) {
  if (S > 0) {
    b0 = id * S;
    b1 = min(TT, b0 + S);
  } else {
    const int d = id / Hkv, g = id - d * Hkv;
    const int pre = g_att_pre[d], nkb = g_att_pre[d + 1] - pre;
    b0 = Hkv * pre + g * nkb;
    b1 = b0 + nkb;
  }
}
__device__ __forceinline__ void dec_advance(DecCursor& cur, int n_dec, int Hkv) {
  cur.f += 1;
  if (++cur.kb == cur.nkb) {
    cur.kb = 0;
    if (++cur.g == Hkv) {
      cur.g = 0;
      cur.d += 1;
      if (cur.d < n_dec) cur.nkb = g_att_pre[cur.d + 1] - g_att_pre[cur.d];
    }
  }
}

// ---- tensor-core and matrix-load wrappers ---------------------------------------------------------
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void mma_bf16_16816(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// One 16-key tile of a (row, kv head) unit by one warp: scores, online softmax, out += P V (see below).
template <int HD>
__device__ __forceinline__ void att_tile_math(uint32_t kt, uint32_t vt, int n_valid, float qscale, const uint32_t (&qf)[HD / 16][2],
                                              float (&o)[HD / 16][4], float (&m2)[2], float (&l2)[2]) {
  constexpr int KS = HD / 16, NBOX = HD / 64;
  const int lane = threadIdx.x & 31;
  const int gq = lane >> 2;
  // The matrix loads and MMAs below are issued in program order, so all loads of an operand are
  // issued before the MMAs that use them, and V is fetched before the softmax arithmetic.
  uint32_t kf[KS][4];    // A operand of the scores: K tile, keys x dims
#pragma unroll
  for (int ks = 0; ks < KS; ++ks) {
    const int key = (lane & 7) + ((lane >> 3) & 1) * 8;
    const int ck = ks * 2 + (lane >> 4);
    const int line = key * NBOX + (ck >> 3);   // 128-byte line of the tile; chunks are swizzled with the line index
    ldsm_x4(kt + line * 128 + (((ck & 7) ^ (line & 7)) << 4), kf[ks][0], kf[ks][1], kf[ks][2], kf[ks][3]);
  }
  uint32_t vf[HD / 16][4];   // A operand of the output: V tile transposed, dims x keys
#pragma unroll
  for (int i = 0; i < HD / 16; ++i) {
    const int key = (lane & 7) + ((lane >> 4) & 1) * 8;
    const int ck = i * 2 + ((lane >> 3) & 1);
    const int line = key * NBOX + (ck >> 3);
    ldsm_x4_t(vt + line * 128 + (((ck & 7) ^ (line & 7)) << 4), vf[i][0], vf[i][1], vf[i][2], vf[i][3]);
  }
  // scores^T [16 keys][8 heads]: four accumulators (k-step mod 4) keep the dependent chains short
  float sacc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) { sacc[i][0] = sacc[i][1] = sacc[i][2] = sacc[i][3] = 0.f; }
#pragma unroll
  for (int ks = 0; ks < KS; ++ks) mma_bf16_16816(sacc[ks & 3], kf[ks], qf[ks][0], qf[ks][1]);
  float sv[4];   // keys gq (0, 1) and gq + 8 (2, 3), heads 2 tq (0, 2) and 2 tq + 1 (1, 3)
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float v = (sacc[0][e] + sacc[1][e]) + (sacc[2][e] + sacc[3][e]);
    sv[e] = (gq + (e >> 1) * 8 < n_valid) ? v * qscale : -INFINITY;
  }
  // online softmax per head: maxima over the 16 keys live in the lanes with the same tq
  float mx0 = fmaxf(sv[0], sv[2]), mx1 = fmaxf(sv[1], sv[3]);
#pragma unroll
  for (int sh = 4; sh <= 16; sh <<= 1) {
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, sh));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, sh));
  }
  const float mn0 = fmaxf(m2[0], mx0), mn1 = fmaxf(m2[1], mx1);   // finite: key 0 of the tile is always valid
  if (__any_sync(0xffffffffu, mn0 > m2[0] || mn1 > m2[1])) {
    const float c0 = fast_ex2(m2[0] - mn0), c1 = fast_ex2(m2[1] - mn1);
    l2[0] *= c0; l2[1] *= c1;
#pragma unroll
    for (int i = 0; i < HD / 16; ++i) { o[i][0] *= c0; o[i][1] *= c1; o[i][2] *= c0; o[i][3] *= c1; }
  }
  m2[0] = mn0; m2[1] = mn1;
  const float p0 = fast_ex2(sv[0] - mn0), p1 = fast_ex2(sv[1] - mn1), p2 = fast_ex2(sv[2] - mn0), p3 = fast_ex2(sv[3] - mn1);
  l2[0] += p0 + p2;
  l2[1] += p1 + p3;
  // P^T as the B operand of the output: transpose the two 8 x 8 (key, head) blocks in registers
  uint32_t pb0, pb1;
  {
    const uint32_t plo = pack_bf2(p0, p1), phi = pack_bf2(p2, p3);
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(pb0) : "r"(plo));
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(pb1) : "r"(phi));
  }
  // out^T += V^T P^T: 16 dims per MMA, one k-step of 16 keys
#pragma unroll
  for (int i = 0; i < HD / 16; ++i) mma_bf16_16816(o[i], vf[i], pb0, pb1);
}

// ---- decode rows: warp-level streaming kernel -------------------------------------------------
// One warp owns a (row, kv head) unit at a time and walks its 16-key tiles.  A tile's K and V
// ([16 keys][head_dim] each, contiguous in the pool) arrive through one TMA tile copy with the
// 128-byte swizzle, so both can be read with ldmatrix (at most two-way bank conflicts).  The two small contractions
// of a tile (scores and out += P V for the query heads of the group) run as m16n8k16 MMAs with
// the 16 keys (or 16 output dims) as the rows and the group's heads as the columns: written with
// CUDA-core FMAs the same loop needs about 800 instructions per tile and the SM runs out of issue
// slots at about half the HBM bandwidth; this form needs about 110.  Softmax statistics stay in
// fp32 registers and are combined with shuffles.
template <int HD, int NREP>
static __device__ __noinline__ void attn_decode_stream(const DevCtx& c, int layer) {
  extern __shared__ __align__(1024) float smem[];
  char* ring = tc_tiles(smem) + (threadIdx.x >> 5) * (ATT_NS * 2 * 16 * HD * 2);
  constexpr int RB = HD * 2;         // bytes per key row
  constexpr int TILE = 16 * RB;      // bytes of one K (or V) tile of a (block, kv head)
  constexpr int STAGE = 2 * TILE;
  constexpr int KS = HD / 16;        // k-steps of Q K^T
  constexpr int REC = NREP * HD + ((2 * NREP + 3) & ~3);  // floats per partial record, 16-byte multiple
  constexpr unsigned FULL = 0xffffffffu;
  static_assert(NREP <= 8, "the group's heads must fit the first eight operand rows");
  const int n_dec = g_att_step.n_dec, TT = g_att_step.TT, S = g_att_step.S;   // S == 0: a sub-range is a unit
  if (TT <= 0) return;
  const int Hkv = c.Hkv;
  const int n_sub = S > 0 ? (TT + S - 1) / S : n_dec * Hkv;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int gq = lane >> 2, tq = lane & 3;   // operand row (= head of the group) and column pair
  const bool live = gq < NREP;   // this lane loads the q of head gq
  uint64_t* bars = g_att.bar[w];
  volatile int* dead = &g_att.dead;
  int* ctr = c.att_ctr + layer;
  const CUtensorMap* kv_map = reinterpret_cast<const CUtensorMap*>(c.kv_map);
  const __nv_bfloat16* qb = reinterpret_cast<const __nv_bfloat16*>(c.qb);
  __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(c.attn);
  const float qscale = c.attn_scale * 1.4426950408889634f;
  const uint32_t ring_s = smem_u32(ring);
  const uint64_t kv_policy = l2_evict_first();   // the cache is read once per step

  uint32_t par = g_att_par[w];
  int n_issued = 0, n_consumed = 0, p_k = 0, c_k = 0;
  bool p_done = false, first_fetch = true;
  DecCursor pc{0, 0, 0, 0, 0, 1}, cc{0, 0, 0, 0, 0, 1};
  int p_blk = 0, p_blk_d = -1, p_blk_base = -1;
  int sub_start = 0, sub_id = 0;
  bool in_unit = false;

  // Both contractions are written with the 16 keys (scores) or 16 dims (output) as the M rows of
  // the MMA and the group's heads as the 8 columns, so a tile costs 8 + 8 MMAs.  Column pair
  // (2 tq, 2 tq + 1) of every accumulator belongs to this lane: two heads, softmax state for each.
  uint32_t qf[KS][2];     // B operand of the scores: q of head gq, dims 16 ks + 2 tq .. and + 8
  float o[HD / 16][4];    // out^T: dims gq + 16 i (c0, c1) and gq + 8 + 16 i (c2, c3), heads 2 tq, 2 tq + 1
  float m2[2] = {-INFINITY, -INFINITY}, l2[2] = {0.f, 0.f};

  while (true) {
    // ---- producer: keep up to ATT_NS tiles in flight ----
    while (!p_done && n_issued - n_consumed < ATT_NS) {
      if (pc.f == pc.f_end) {
        // next non-empty sub-range: the warp's own index first, then whatever the counter hands out
        int id = 0, b0 = 0, b1 = 0;
        while (true) {
          if (first_fetch) {
            id = blockIdx.x * ATT_WARPS + w;
            first_fetch = false;
          } else {
            if (lane == 0) id = atomicAdd(ctr, 1);
            id = __shfl_sync(FULL, id, 0);
          }
          if (id >= n_sub) { p_done = true; break; }
          dec_sub_range(id, S, TT, Hkv, b0, b1);
          if (b0 < b1) break;
        }
        if (p_done) break;
        if (lane == 0) g_att.ids[w][p_k & 7] = id;
        __syncwarp();
        p_k += 1;
        dec_seek(pc, b0, b1, n_dec, Hkv);
      }
      if (pc.d != p_blk_d || (pc.kb & ~31) != p_blk_base) {
        p_blk_d = pc.d;
        p_blk_base = pc.kb & ~31;
        const int idx = p_blk_base + lane;
        p_blk = idx < pc.nkb ? c.block_table[(size_t)g_att_bslot[pc.d] * c.max_blocks_seq + idx] : 0;
      }
      const int blk = __shfl_sync(FULL, p_blk, pc.kb & 31);
      if (lane == 0) {
        const int s = n_issued % ATT_NS;
        // one copy brings the K tile and the V tile: box {64 dims, HD / 64 halves, 16 keys, K and V, this layer}
        mbar_expect_tx(&bars[s], STAGE);
        tma_load_5d(ring + s * STAGE, kv_map, 0, 0, (blk * Hkv + pc.g) * 16, 0, layer, &bars[s], kv_policy);
      }
      dec_advance(pc, n_dec, Hkv);
      n_issued += 1;
    }
    if (n_consumed == n_issued) break;

    // ---- consumer: one tile ----
    while (cc.f == cc.f_end) {   // next non-empty sub-range (the producer already issued a tile of it)
      sub_id = g_att.ids[w][c_k & 7];
      c_k += 1;
      int sub_end;
      dec_sub_range(sub_id, S, TT, Hkv, sub_start, sub_end);
      dec_seek(cc, sub_start, sub_end, n_dec, Hkv);
      in_unit = false;
    }
    const int t_row = g_att_row[cc.d];
    const int n_ctx = g_att_nctx[cc.d];
    if (!in_unit) {  // a unit (or this sub-range's part of it) starts here
      in_unit = true;
      m2[0] = m2[1] = -INFINITY;
      l2[0] = l2[1] = 0.f;
      const __nv_bfloat16* qrow = qb + (size_t)t_row * c.q_dim + (size_t)(cc.g * NREP + (live ? gq : 0)) * HD;
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        qf[ks][0] = live ? *reinterpret_cast<const uint32_t*>(qrow + ks * 16 + 2 * tq) : 0u;
        qf[ks][1] = live ? *reinterpret_cast<const uint32_t*>(qrow + ks * 16 + 8 + 2 * tq) : 0u;
      }
#pragma unroll
      for (int i = 0; i < HD / 16; ++i) { o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f; }
    }
    const int s = n_consumed % ATT_NS;
    if (!__all_sync(FULL, mbar_wait(c, &bars[s], (par >> s) & 1u, dead))) break;  // uniform exit
    par ^= 1u << s;
    const uint32_t kt = ring_s + s * STAGE, vt = kt + TILE;
    const int key0 = cc.kb * 16;
    const int n_valid = min(16, n_ctx - key0);   // >= 1
    if (n_valid < 16) {
      // the tail of the last block holds whatever the pool held: clear those V rows (0 x NaN)
      uint4* vg = reinterpret_cast<uint4*>(ring + s * STAGE + TILE + n_valid * RB);
      for (int i = lane; i < (16 - n_valid) * RB / 16; i += 32) vg[i] = make_uint4(0u, 0u, 0u, 0u);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // before TMA refills this stage
      __syncwarp();
    }
    att_tile_math<HD>(kt, vt, n_valid, qscale, qf, o, m2, l2);
    __syncwarp();  // all reads of this stage are done before it is refilled
    n_consumed += 1;

    const bool unit_ends = (cc.kb == cc.nkb - 1) || (cc.f + 1 == cc.f_end);
    if (unit_ends) {
      in_unit = false;
      float lt0 = l2[0], lt1 = l2[1];   // sums over the keys: lanes with the same tq
#pragma unroll
      for (int sh = 4; sh <= 16; sh <<= 1) {
        lt0 += __shfl_xor_sync(FULL, lt0, sh);
        lt1 += __shfl_xor_sync(FULL, lt1, sh);
      }
      const int us = Hkv * g_att_pre[cc.d] + cc.g * cc.nkb, ue = us + cc.nkb;
      const int j_first = S > 0 ? us / S : 0, j_last = S > 0 ? (ue - 1) / S : 0;
      const int h0 = 2 * tq;   // this lane's heads: h0, h0 + 1
      if (j_first == j_last) {   // the whole unit was handled here
        __nv_bfloat16* obase = out + (size_t)t_row * c.q_dim + (size_t)(cc.g * NREP) * HD;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          if (h0 + e < NREP) {
            const float inv = __fdividef(1.0f, e ? lt1 : lt0);
#pragma unroll
            for (int i = 0; i < HD / 16; ++i) {
              obase[(h0 + e) * HD + 16 * i + gq] = __float2bfloat16_rn(o[i][e] * inv);
              obase[(h0 + e) * HD + 16 * i + 8 + gq] = __float2bfloat16_rn(o[i][2 + e] * inv);
            }
          }
        }
      } else {
        // partial record: [NREP][HD] accumulators, then m[NREP], then l[NREP]
        const int unit = cc.d * Hkv + cc.g;
        float* rec = c.att_part + (size_t)(2 * sub_id + (us <= sub_start ? 0 : 1)) * REC;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          if (h0 + e < NREP) {
#pragma unroll
            for (int i = 0; i < HD / 16; ++i) {
              rec[(h0 + e) * HD + 16 * i + gq] = o[i][e];
              rec[(h0 + e) * HD + 16 * i + 8 + gq] = o[i][2 + e];
            }
            if (gq == 0) { rec[NREP * HD + h0 + e] = m2[e]; rec[NREP * HD + NREP + h0 + e] = e ? lt1 : lt0; }
          }
        }
        __threadfence();
        __syncwarp();
        int old = 0;
        if (lane == 0) old = atomicAdd(&c.att_cnt[unit], 1);
        old = __shfl_sync(FULL, old, 0);
        if (old == j_last - j_first) {  // this warp delivered the last part: merge in sub-range order
          __threadfence();
          // each lane merges four consecutive dims at a time; loads of the parts are independent
          for (int i4 = lane; i4 < NREP * HD / 4; i4 += 32) {
            const int h = (i4 * 4) / HD;
            float M = -INFINITY;
#pragma unroll 4
            for (int j = j_first; j <= j_last; ++j) {
              const float* r = c.att_part + (size_t)(2 * j + (us <= j * S ? 0 : 1)) * REC;
              M = fmaxf(M, __ldcg(r + NREP * HD + h));
            }
            float4 num = make_float4(0.f, 0.f, 0.f, 0.f);
            float den = 0.f;
#pragma unroll 4
            for (int j = j_first; j <= j_last; ++j) {
              const float* r = c.att_part + (size_t)(2 * j + (us <= j * S ? 0 : 1)) * REC;
              const float f = fast_ex2(__ldcg(r + NREP * HD + h) - M);
              const float4 a4 = __ldcg(reinterpret_cast<const float4*>(r) + i4);
              num.x += f * a4.x; num.y += f * a4.y; num.z += f * a4.z; num.w += f * a4.w;
              den += f * __ldcg(r + NREP * HD + NREP + h);
            }
            const float inv = __fdividef(1.0f, den);
            uint2 o2;
            o2.x = pack_bf2(num.x * inv, num.y * inv);
            o2.y = pack_bf2(num.z * inv, num.w * inv);
            *reinterpret_cast<uint2*>(out + (size_t)t_row * c.q_dim + (size_t)(cc.g * NREP) * HD + i4 * 4) = o2;
          }
          if (lane == 0) c.att_cnt[unit] = 0;
        }
      }
    }
    dec_advance(cc, n_dec, Hkv);
  }
  __syncwarp();
  if (lane == 0) g_att_par[w] = par;
}

// ---- decode rows: one CTA per part of a unit -----------------------------------------------------------
// Few (row, kv head) units, as a handful of requests make them: the streaming kernel above gives a unit to one
// warp, or cuts it and pays a record, a fence, a counter and a merge by one warp for every cut, so that one row of
// 300 keys took 22 us and one of 4000 keys 51 us per layer, nearly all of it latency.  Here the eight warps of a
// CTA share a part of a unit (C tiles, no part crosses units): their tiles are in flight at once, their sums are
// merged in shared memory, and only units of more than C tiles leave records, merged by the whole last CTA.  Where there
// are more units than CTAs, half CTAs take one each instead of CTAs two in turn: 8B shape, us a layer, 20 rows of 160 keys 15.5 ->
// 12.4, 24 of 300 19.7 -> 15.3, 37 of 100 20.1 -> 15.5, 37 of 300 24.3 -> 19.2.
// In steps of at most 16 rows without prompt rows this kernel also takes over RoPE and the K/V write (a phase and a grid
// barrier less): every CTA rotates the queries it needs, and the warp that meets a unit's last tile computes the new key
// and value row, writes it to the pool and into its copy of the tile.
constexpr int ATT_NSC = 2;   // ring stages per warp here
constexpr int ATT_CTA_OFF = 65536;   // the space before it may be receiving weights of the O projection already
struct AttCta {
  float m[ATT_WARPS][8], l[ATT_WARPS][8];   // maxima and sums of the warps
  int last;
};
__shared__ AttCta g_att_cta;
// GW: warps that share a unit, all of the CTA's or half of them (two groups, which go their own ways).
template <int HD, int NREP, int GW>
static __device__ __noinline__ void attn_decode_cta(const DevCtx& c, int layer) {
  extern __shared__ __align__(1024) float smem[];
  char* base = tc_tiles(smem) + ATT_CTA_OFF;
  constexpr int RB = HD * 2;
  constexpr int TILE = 16 * RB;
  constexpr int STAGE = 2 * TILE;
  constexpr int KS = HD / 16;
  constexpr int REC = NREP * HD + ((2 * NREP + 3) & ~3);
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int GT = GW * 32, NG = ATT_WARPS / GW;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int grp = NG == 1 ? 0 : w / GW, w0 = grp * GW, wg = w - w0, tg = (int)threadIdx.x - grp * GT;
  const int n_groups = NG * (int)gridDim.x;
  auto group_sync = [&]() {
    if constexpr (NG == 1) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(4 + grp), "n"(GT) : "memory");
  };
  float(*s_m)[8] = g_att_cta.m + w0;
  float(*s_l)[8] = g_att_cta.l + w0;
  // the unit's queries, in what the control plane uses between the steps
  static_assert(NG * NREP * HD * 2 <= (int)sizeof(g_ctl), "no room for the queries");
  __nv_bfloat16* s_q = reinterpret_cast<__nv_bfloat16*>(&g_ctl) + grp * NREP * HD;
  const int gq = lane >> 2, tq = lane & 3;
  const bool live = gq < NREP;
  const int n_dec = g_att_step.n_dec, C = g_att_step.C, Hkv = c.Hkv;
  char* ring = base + w * ATT_NSC * STAGE;
  float* s_o = reinterpret_cast<float*>(base + w0 * ATT_NSC * STAGE);   // a warp's sums [NREP][HD] go where its ring stages were
  constexpr int S_O = ATT_NSC * STAGE / 4;       // floats from one warp's sums to the next
  static_assert(NREP * HD * 4 <= ATT_NSC * STAGE, "a warp's sums exceed its stages");
  const bool fuse = g_att_step.fuse != 0;
  uint64_t* bars = g_att.bar[w];
  volatile int* dead = &g_att.dead;
  const CUtensorMap* kv_map = reinterpret_cast<const CUtensorMap*>(c.kv_map);
  const __nv_bfloat16* qb = reinterpret_cast<const __nv_bfloat16*>(c.qb);
  __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(c.attn);
  const float qscale = c.attn_scale * 1.4426950408889634f;
  const uint64_t kv_policy = l2_evict_first();
  uint32_t par = g_att_par[w];

  // items in unit order, from the last CTA: prompt rows of a step sit on the first ones (those that single CTAs take only while no
  // pair has any)
  for (int item = (int)gridDim.x - 1 - (int)blockIdx.x + grp * (int)gridDim.x; ; item += n_groups) {   // uniform over the group
    int d = 0, rest = item, nkb = 0, ns = 1;   // (the units of half CTAs are whole)
    for (; d < n_dec; ++d) {
      nkb = g_att_pre[d + 1] - g_att_pre[d];
      if constexpr (NG == 1) ns = (nkb + C - 1) / C;
      if (rest < Hkv * ns) break;
      rest -= Hkv * ns;
    }
    if (d >= n_dec) break;
    const int g = rest / ns, part = rest - g * ns;
    const int kb0 = part * C, kb1 = min(nkb, kb0 + C);
    const int n_tiles = kb0 + wg < kb1 ? (kb1 - kb0 - wg + GW - 1) / GW : 0;   // kb0 + wg, + GW, ...
    const int t_row = g_att_row[d], n_ctx = g_att_nctx[d];
    const int32_t* table = c.block_table + (size_t)g_att_bslot[d] * c.max_blocks_seq;
    // block ids of the warp's first 32 tiles, one per lane; the first item's are kept from layer to layer
    const bool first = item < n_groups;
    int blk = g_att_blk[threadIdx.x];
    if (!(first && layer > 0 && !c.stepped)) {
      blk = lane < n_tiles ? table[kb0 + wg + GW * lane] : 0;
      if (first) g_att_blk[threadIdx.x] = blk;
    }
    auto issue = [&](int i) {
      if (i >= 32 && (i & 31) == 0) blk = i + lane < n_tiles ? table[kb0 + wg + GW * (i + lane)] : 0;
      const int b = __shfl_sync(FULL, blk, i & 31);
      if (lane == 0) {
        const int s = i % ATT_NSC;
        mbar_expect_tx(&bars[s], STAGE);
        tma_load_5d(ring + s * STAGE, kv_map, 0, 0, (b * Hkv + g) * 16, 0, layer, &bars[s], kv_policy);
      }
    };
#pragma unroll
    for (int i = 0; i < ATT_NSC; ++i)
      if (i < n_tiles) issue(i);
    uint32_t qf[KS][2];
    float o[HD / 16][4];
    float m2[2] = {-INFINITY, -INFINITY}, l2[2] = {0.f, 0.f};
    // this warp meets the unit's last tile: the new key and value row is its business
    const bool newest = fuse && n_tiles > 0 && kb0 + wg + GW * (n_tiles - 1) == nkb - 1;
    uint2 new_k = make_uint2(0u, 0u), new_v = make_uint2(0u, 0u);
    // The queries by way of shared memory, a thread per rotation pair: with every warp rotating all of them for itself the
    // code of this was 64 loads long, and met beyond the instruction cache.
    if (fuse) {
      constexpr int H2 = HD / 2;
      const int pos = n_ctx - 1;
      const float* row = c.qkv + (size_t)t_row * c.qkv_dim;
      const float* cs = c.rope_cos + (size_t)pos * H2;
      const float* sn = c.rope_sin + (size_t)pos * H2;
      float4 kx = make_float4(0.f, 0.f, 0.f, 0.f), vx = kx, kc = kx, ks4 = kx;
      const int d0 = (lane * 4) & (HD - 1);   // four dims of the new row (HD 64: the upper lanes repeat the lower ones)
      if (newest) {
        kx = __ldcg(reinterpret_cast<const float4*>(row + c.q_dim + g * HD + d0));
        vx = __ldcg(reinterpret_cast<const float4*>(row + c.q_dim + c.kv_dim + g * HD + d0));
        kc = *reinterpret_cast<const float4*>(cs + (d0 & (H2 - 1)));
        ks4 = *reinterpret_cast<const float4*>(sn + (d0 & (H2 - 1)));
      }
#pragma unroll
      for (int k = tg; k < NREP * H2; k += GT) {
        const int i = k % H2, at = k / H2 * HD + i;
        const float x1 = __ldcg(row + g * NREP * HD + at), x2 = __ldcg(row + g * NREP * HD + at + H2), cc = cs[i], ss = sn[i];
        // the same fused forms as the RoPE phase
        s_q[at] = __float2bfloat16_rn(fmaf(x1, cc, -__fmul_rn(x2, ss)));
        s_q[at + H2] = __float2bfloat16_rn(fmaf(x2, cc, __fmul_rn(x1, ss)));
      }
      if (newest) {   // uniform over the warp
        float4 px;
        constexpr int PL = HD / 8;   // lanes between the two halves of a pair
        px.x = __shfl_xor_sync(FULL, kx.x, PL); px.y = __shfl_xor_sync(FULL, kx.y, PL);
        px.z = __shfl_xor_sync(FULL, kx.z, PL); px.w = __shfl_xor_sync(FULL, kx.w, PL);
        float4 y;
        if (d0 < H2) {
          y = make_float4(fmaf(kx.x, kc.x, -__fmul_rn(px.x, ks4.x)), fmaf(kx.y, kc.y, -__fmul_rn(px.y, ks4.y)),
                          fmaf(kx.z, kc.z, -__fmul_rn(px.z, ks4.z)), fmaf(kx.w, kc.w, -__fmul_rn(px.w, ks4.w)));
        } else {
          y = make_float4(fmaf(kx.x, kc.x, __fmul_rn(px.x, ks4.x)), fmaf(kx.y, kc.y, __fmul_rn(px.y, ks4.y)),
                          fmaf(kx.z, kc.z, __fmul_rn(px.z, ks4.z)), fmaf(kx.w, kc.w, __fmul_rn(px.w, ks4.w)));
        }
        new_k = make_uint2(pack_bf2(y.x, y.y), pack_bf2(y.z, y.w));
        new_v = make_uint2(pack_bf2(vx.x, vx.y), pack_bf2(vx.z, vx.w));
        const int b = table[nkb - 1];
        if (lane * 4 < HD) {
          *reinterpret_cast<uint2*>(kv_tile<__nv_bfloat16>(c, layer, 0, b, g) + (size_t)(pos & 15) * HD + d0) = new_k;
          *reinterpret_cast<uint2*>(kv_tile<__nv_bfloat16>(c, layer, 1, b, g) + (size_t)(pos & 15) * HD + d0) = new_v;
        }
      }
    } else if (tg < NREP * HD / 8) {
      reinterpret_cast<uint4*>(s_q)[tg] =
          __ldcg(reinterpret_cast<const uint4*>(qb + (size_t)t_row * c.q_dim + (size_t)g * NREP * HD) + tg);
    }
    group_sync();
    const uint32_t* qs = reinterpret_cast<const uint32_t*>(s_q + (live ? gq : 0) * HD + 2 * tq);
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
      qf[ks][0] = live ? qs[ks * 8] : 0u;
      qf[ks][1] = live ? qs[ks * 8 + 4] : 0u;
    }
#pragma unroll
    for (int i = 0; i < HD / 16; ++i) { o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f; }
    for (int i = 0; i < n_tiles; ++i) {
      const int s = i % ATT_NSC;
      if (!__all_sync(FULL, mbar_wait(c, &bars[s], (par >> s) & 1u, dead))) break;
      par ^= 1u << s;
      char* st = ring + s * STAGE;
      const int n_valid = min(16, n_ctx - (kb0 + wg + GW * i) * 16);   // >= 1
      if (n_valid < 16) {   // the tail of the last block holds whatever the pool held: clear those V rows (0 x NaN)
        uint4* vg = reinterpret_cast<uint4*>(st + TILE + n_valid * RB);
        for (int k = lane; k < (16 - n_valid) * RB / 16; k += 32) vg[k] = make_uint4(0u, 0u, 0u, 0u);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
      }
      if (newest && i == n_tiles - 1) {   // the copy holds what the pool held before the row was written
        if (lane * 4 < HD) {
          const int d0 = lane * 4, line = ((n_ctx - 1) & 15) * (HD / 64) + (d0 >> 6);
          char* dst = st + line * 128 + ((((d0 & 63) >> 3) ^ (line & 7)) << 4) + (d0 & 7) * 2;
          *reinterpret_cast<uint2*>(dst) = new_k;
          *reinterpret_cast<uint2*>(dst + TILE) = new_v;
        }
        __syncwarp();
      }
      att_tile_math<HD>(smem_u32(st), smem_u32(st) + TILE, n_valid, qscale, qf, o, m2, l2);
      __syncwarp();   // all reads of this stage are done before it is refilled
      if (i + ATT_NSC < n_tiles) issue(i + ATT_NSC);
    }
    // the warp's sums to shared memory
    float lt0 = l2[0], lt1 = l2[1];
#pragma unroll
    for (int sh = 4; sh <= 16; sh <<= 1) {
      lt0 += __shfl_xor_sync(FULL, lt0, sh);
      lt1 += __shfl_xor_sync(FULL, lt1, sh);
    }
    const int h0 = 2 * tq;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      if (h0 + e < NREP) {
        if (n_tiles > 0) {
          float* ow = s_o + wg * S_O + (h0 + e) * HD;
#pragma unroll
          for (int i = 0; i < HD / 16; ++i) {
            ow[16 * i + gq] = o[i][e];
            ow[16 * i + 8 + gq] = o[i][2 + e];
          }
        }
        if (gq == 0) { s_m[wg][h0 + e] = m2[e]; s_l[wg][h0 + e] = e ? lt1 : lt0; }
      }
    }
    group_sync();
    // merge the warps: a thread takes two consecutive dims of a head at a time
    const int n_warps = min(GW, kb1 - kb0);   // the first n_warps of the group had tiles
    float* rec = c.att_part + (size_t)item * REC;
    __nv_bfloat16* obase = out + (size_t)t_row * c.q_dim + (size_t)(g * NREP) * HD;
    for (int i2 = tg; i2 < NREP * HD / 2; i2 += GT) {
      const int h = i2 * 2 / HD;
      float M = -INFINITY;
      for (int k = 0; k < n_warps; ++k) M = fmaxf(M, s_m[k][h]);
      float2 num = make_float2(0.f, 0.f);
      float den = 0.f;
      for (int k = 0; k < n_warps; ++k) {
        const float f = fast_ex2(s_m[k][h] - M);
        const float2 a = *reinterpret_cast<const float2*>(s_o + k * S_O + i2 * 2);
        num.x = fmaf(f, a.x, num.x);
        num.y = fmaf(f, a.y, num.y);
        den = fmaf(f, s_l[k][h], den);
      }
      if (NG > 1 || ns == 1) {
        const float inv = __fdividef(1.0f, den);
        *reinterpret_cast<uint32_t*>(obase + i2 * 2) = pack_bf2(num.x * inv, num.y * inv);
      } else {
        *reinterpret_cast<float2*>(rec + i2 * 2) = num;
        if ((i2 * 2) % HD == 0) { rec[NREP * HD + h] = M; rec[NREP * HD + NREP + h] = den; }
      }
    }
    if (NG == 1 && ns > 1) {
      const int unit = d * Hkv + g;
      __threadfence();
      group_sync();
      if (tg == 0) g_att_cta.last = atomicAdd(&c.att_cnt[unit], 1) == ns - 1;
      group_sync();
      if (g_att_cta.last) {   // this CTA delivered the last part: merge in part order (records of a unit are consecutive)
        __threadfence();
        const float* r0 = c.att_part + (size_t)(item - part) * REC;
        for (int i2 = tg; i2 < NREP * HD / 2; i2 += GT) {
          const int h = i2 * 2 / HD;
          float M = -INFINITY;
#pragma unroll 8
          for (int k = 0; k < ns; ++k) M = fmaxf(M, __ldcg(r0 + (size_t)k * REC + NREP * HD + h));
          float2 num = make_float2(0.f, 0.f);
          float den = 0.f;
#pragma unroll 8
          for (int k = 0; k < ns; ++k) {
            const float f = fast_ex2(__ldcg(r0 + (size_t)k * REC + NREP * HD + h) - M);
            const float2 a = __ldcg(reinterpret_cast<const float2*>(r0 + (size_t)k * REC) + i2);
            num.x = fmaf(f, a.x, num.x);
            num.y = fmaf(f, a.y, num.y);
            den = fmaf(f, __ldcg(r0 + (size_t)k * REC + NREP * HD + NREP + h), den);
          }
          const float inv = __fdividef(1.0f, den);
          *reinterpret_cast<uint32_t*>(obase + i2 * 2) = pack_bf2(num.x * inv, num.y * inv);
        }
        if (tg == 0) c.att_cnt[unit] = 0;
      }
    }
    // the sums are free for the next item, and before copies land there again
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    group_sync();
  }
  if (lane == 0) g_att_par[w] = par;
}

// ---- prefill-chunk rows: tensor-core tile kernel ---------------------------------------------------
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}

// One CTA: query rows [qblk*QROWS, +QROWS) of one request's chunk, one kv head; the NREP query
// heads of the group are stacked along M (M row = head * QROWS + row), 16 M rows per warp.
// Shared memory: Q [128][HD] then two stages of K [64][HD], V [64][HD]; 16-byte chunks of a row
// are XOR-swizzled with the row index so that ldmatrix reads are conflict-free.
template <int HD, int NREP>
static __device__ __noinline__ void attn_prefill_tile(const DevCtx& c, int layer, int item, int qblk, int g, char* smem) {
  constexpr int QROWS = 128 / NREP;
  constexpr int RB = HD * 2;          // bytes per row
  constexpr int CPR = RB / 16;        // 16-byte chunks per row
  constexpr int KT = 64;              // keys per tile
  constexpr int QBYTES = 128 * RB, KVBYTES = KT * RB;
  constexpr int TILE = 16 * HD * 2;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int bslot = c.it_bslot[item], start = c.it_start[item], ntok = c.it_ntok[item], qstart = c.it_qstart[item];
  const int r_base = qblk * QROWS;
  const int n_keys = start + min(ntok, r_base + QROWS);
  const int nkt = (n_keys + KT - 1) / KT;
  const int32_t* table = c.block_table + (size_t)bslot * c.max_blocks_seq;
  const __nv_bfloat16* qb = reinterpret_cast<const __nv_bfloat16*>(c.qb);
  __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(c.attn);
  const char* kv_base = reinterpret_cast<const char*>(c.kv_base);
  const size_t kv_stride = (size_t)c.n_blocks * c.Hkv * TILE;
  const char* k_plane = kv_base + (size_t)layer * 2 * kv_stride;
  const uint32_t s_q = smem_u32(smem), s_kv = s_q + QBYTES;
  const float qscale = c.attn_scale * 1.4426950408889634f;

  __syncthreads();  // the previous user of this shared memory is done
  // Q tile
  for (int id = tid; id < 128 * CPR; id += FWD_THREADS) {
    const int mrow = id / CPR, ck = id % CPR;
    const int h = mrow / QROWS, r = r_base + mrow % QROWS;
    const bool ok = r < ntok;
    const __nv_bfloat16* src = qb + (size_t)(qstart + (ok ? r : 0)) * c.q_dim + (size_t)(g * NREP + h) * HD + ck * 8;
    cp_async16(s_q + mrow * RB + ((ck ^ (mrow & 7)) << 4), src, ok ? 16u : 0u);
  }
  auto load_kv = [&](int kt, int stage) {
    const uint32_t dk = s_kv + stage * 2 * KVBYTES, dv = dk + KVBYTES;
    for (int id = tid; id < KT * CPR; id += FWD_THREADS) {
      const int key = id / CPR, ck = id % CPR;
      const int kpos = kt * KT + key;
      const bool ok = kpos < n_keys;
      const int blk = table[ok ? (kpos >> 4) : 0];
      const char* src = k_plane + ((size_t)blk * c.Hkv + g) * TILE + (size_t)(kpos & 15) * RB + ck * 16;
      const uint32_t off = key * RB + ((ck ^ (key & 7)) << 4);
      cp_async16(dk + off, src, ok ? 16u : 0u);
      cp_async16(dv + off, src + kv_stride, ok ? 16u : 0u);
    }
  };
  load_kv(0, 0);
  asm volatile("cp.async.commit_group;" ::: "memory");

  const int mrow0 = w * 16;
  const int gq = lane >> 2, tq = lane & 3;
  // positions of the two rows this lane holds in the accumulator layout
  const int pos_lo = start + r_base + (mrow0 + gq) % QROWS;
  const int pos_hi = start + r_base + (mrow0 + gq + 8) % QROWS;
  uint32_t qf[HD / 16][4];
  float o[HD / 8][4];
#pragma unroll
  for (int i = 0; i < HD / 8; ++i) { o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f; }
  float m_lo = -INFINITY, m_hi = -INFINITY, l_lo = 0.f, l_hi = 0.f;

  for (int kt = 0; kt < nkt; ++kt) {
    const int stage = kt & 1;
    if (kt + 1 < nkt) load_kv(kt + 1, stage ^ 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    if (kt == 0) {
#pragma unroll
      for (int ks = 0; ks < HD / 16; ++ks) {
        const int row = mrow0 + (lane & 7) + ((lane >> 3) & 1) * 8;
        const int ck = ks * 2 + (lane >> 4);
        ldsm_x4(s_q + row * RB + ((ck ^ (row & 7)) << 4), qf[ks][0], qf[ks][1], qf[ks][2], qf[ks][3]);
      }
    }
    const uint32_t sk = s_kv + stage * 2 * KVBYTES, sv = sk + KVBYTES;
    // S = Q K^T for 64 keys: 8 n-tiles of 8 keys
    float sacc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i) { sacc[i][0] = sacc[i][1] = sacc[i][2] = sacc[i][3] = 0.f; }
#pragma unroll
    for (int ks = 0; ks < HD / 16; ++ks) {
      uint32_t bf[4][4];   // all loads of the k-step first, then its MMAs (both are issued in program order)
#pragma unroll
      for (int np = 0; np < 4; ++np) {
        const int key = np * 16 + (lane & 7) + (lane >> 4) * 8;
        const int ck = ks * 2 + ((lane >> 3) & 1);
        ldsm_x4(sk + key * RB + ((ck ^ (key & 7)) << 4), bf[np][0], bf[np][1], bf[np][2], bf[np][3]);
      }
#pragma unroll
      for (int np = 0; np < 4; ++np) {
        mma_bf16_16816(sacc[2 * np], qf[ks], bf[np][0], bf[np][1]);
        mma_bf16_16816(sacc[2 * np + 1], qf[ks], bf[np][2], bf[np][3]);
      }
    }
    // scale, causal mask, online softmax (rows gq and gq + 8 of the warp's 16)
    float mx_lo = -INFINITY, mx_hi = -INFINITY;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      const int k0 = kt * KT + nt * 8 + 2 * tq;
      sacc[nt][0] = (k0 <= pos_lo) ? sacc[nt][0] * qscale : -INFINITY;
      sacc[nt][1] = (k0 + 1 <= pos_lo) ? sacc[nt][1] * qscale : -INFINITY;
      sacc[nt][2] = (k0 <= pos_hi) ? sacc[nt][2] * qscale : -INFINITY;
      sacc[nt][3] = (k0 + 1 <= pos_hi) ? sacc[nt][3] * qscale : -INFINITY;
      mx_lo = fmaxf(mx_lo, fmaxf(sacc[nt][0], sacc[nt][1]));
      mx_hi = fmaxf(mx_hi, fmaxf(sacc[nt][2], sacc[nt][3]));
    }
    mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 1));
    mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 2));
    mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 1));
    mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 2));
    // key 0 is visible to every row, so after the first tile the maxima are finite
    const float mn_lo = fmaxf(m_lo, mx_lo), mn_hi = fmaxf(m_hi, mx_hi);
    const float c_lo = fast_ex2(m_lo - mn_lo), c_hi = fast_ex2(m_hi - mn_hi);
    m_lo = mn_lo; m_hi = mn_hi;
    l_lo *= c_lo; l_hi *= c_hi;
#pragma unroll
    for (int i = 0; i < HD / 8; ++i) { o[i][0] *= c_lo; o[i][1] *= c_lo; o[i][2] *= c_hi; o[i][3] *= c_hi; }
    uint32_t pf[4][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      const float p0 = fast_ex2(sacc[nt][0] - mn_lo), p1 = fast_ex2(sacc[nt][1] - mn_lo);
      const float p2 = fast_ex2(sacc[nt][2] - mn_hi), p3 = fast_ex2(sacc[nt][3] - mn_hi);
      l_lo += p0 + p1;
      l_hi += p2 + p3;
      pf[nt >> 1][(nt & 1) * 2] = pack_bf2(p0, p1);
      pf[nt >> 1][(nt & 1) * 2 + 1] = pack_bf2(p2, p3);
    }
    // O += P V
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
#pragma unroll
      for (int d4 = 0; d4 < HD / 16; d4 += 4) {
        uint32_t bf[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int key = kk * 16 + (lane & 7) + ((lane >> 3) & 1) * 8;
          const int ck = (d4 + j) * 2 + (lane >> 4);
          ldsm_x4_t(sv + key * RB + ((ck ^ (key & 7)) << 4), bf[j][0], bf[j][1], bf[j][2], bf[j][3]);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          mma_bf16_16816(o[2 * (d4 + j)], pf[kk], bf[j][0], bf[j][1]);
          mma_bf16_16816(o[2 * (d4 + j) + 1], pf[kk], bf[j][2], bf[j][3]);
        }
      }
    }
    __syncthreads();  // everyone is done with this stage before it is refilled
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 1);
  l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 2);
  l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 1);
  l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 2);
  const int h = mrow0 / QROWS;   // 16 | QROWS, so a warp's rows belong to one head
  const int r_lo = r_base + (mrow0 + gq) % QROWS, r_hi = r_base + (mrow0 + gq + 8) % QROWS;
  const float i_lo = __fdividef(1.0f, l_lo), i_hi = __fdividef(1.0f, l_hi);
#pragma unroll
  for (int nt = 0; nt < HD / 8; ++nt) {
    const size_t col = (size_t)(g * NREP + h) * HD + nt * 8 + 2 * tq;
    if (r_lo < ntok)
      *reinterpret_cast<uint32_t*>(out + (size_t)(qstart + r_lo) * c.q_dim + col) = pack_bf2(o[nt][0] * i_lo, o[nt][1] * i_lo);
    if (r_hi < ntok)
      *reinterpret_cast<uint32_t*>(out + (size_t)(qstart + r_hi) * c.q_dim + col) = pack_bf2(o[nt][2] * i_hi, o[nt][3] * i_hi);
  }
}

// ---- the phase ---------------------------------------------------------------------------------------
template <int HD>
constexpr int att_smem_bytes() {
  constexpr int ring = ATT_WARPS * ATT_NS * 2 * 16 * HD * 2 + 1024;   // + alignment slack
  constexpr int cta = ATT_CTA_OFF + ATT_WARPS * ATT_NSC * 2 * 16 * HD * 2 + 1024;
  constexpr int tile = 128 * HD * 2 + 2 * 2 * 64 * HD * 2;
  return ring > cta ? (ring > tile ? ring : tile) : (cta > tile ? cta : tile);
}

// The attention of a step is up to three pieces of work, each an entry of the step's plan of its own: called from a phase
// function in between, the decode attention is one call deeper and saves 112 registers on its way in instead of 28, 17.8 us
// a layer instead of 13.8 for 64 rows of 50 keys; with that function inlined into the dispatcher every phase is a little longer
// (one-row step of the 8B shape 1.2 %).
enum AttKind : int { ATT_PAIRS = 0, ATT_TILES, ATT_DEC_CTA, ATT_DEC_HALF, ATT_DEC_STREAM };

// The step's work lists: once per step.
__device__ __forceinline__ void att_lists(const DevCtx& c) {
  const SchedState* ss = c.ss;
  const int n = ss->cur_ndec;
  if (threadIdx.x == 0) g_att_step = AttStep{n, ss->cur_TT, ss->cur_S, ss->cur_C, ss->cur_half, ss->cur_npf, ss->cur_npp, ss->cur_fuse};
  for (int i = threadIdx.x; i <= n; i += FWD_THREADS) {
    g_att_pre[i] = c.dec_kbpre[i];
    if (i < n) { g_att_bslot[i] = c.dec_bslot[i]; g_att_nctx[i] = c.dec_nctx[i]; g_att_row[i] = c.dec_row[i]; }
  }
}
// The prompt rows that single CTAs take.  (The pairs' units start from the first CTA, these then from the last.)
template <int HD, int NREP>
static __device__ __noinline__ void att_tiles(const DevCtx& c, int layer, float* smem_f) {
  const int n_pp = g_att_step.npp, n_pf = g_att_step.npf * c.Hkv;
  for (int u = n_pp > 0 ? (int)gridDim.x - 1 - (int)blockIdx.x : (int)blockIdx.x; u < n_pf; u += gridDim.x) {
    const int e = u / c.Hkv, g = u % c.Hkv;
    attn_prefill_tile<HD, NREP>(c, layer, c.pf_item[n_pp + e], c.pf_qb[n_pp + e], g, reinterpret_cast<char*>(smem_f));
  }
  __syncthreads();   // the tiles' shared memory is free
}
template <int HD, int NREP, bool PAIR>
__device__ __forceinline__ void phase_attention_bf16(const DevCtx& c, int layer, int kind, float* smem_f) {
  char* tiles = tc_tiles(smem_f);   // 1024-byte aligned: the tiles are swizzled
  if (kind == ATT_DEC_STREAM) attn_decode_stream<HD, NREP>(c, layer);
  else if (kind == ATT_DEC_CTA) attn_decode_cta<HD, NREP, ATT_WARPS>(c, layer);
  else if (kind == ATT_DEC_HALF) attn_decode_cta<HD, NREP, ATT_WARPS / 2>(c, layer);
  else if (kind == ATT_TILES) att_tiles<HD, NREP>(c, layer, smem_f);
  if constexpr (PAIR && HD == 128 && NREP == 4)
    if (kind == ATT_PAIRS) attn_prefill_pair(c, layer, tiles, g_att_step.npp);
}

}  // namespace blink
