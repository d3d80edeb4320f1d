// Prompt attention of the CTA pairs on tcgen05 (head_dim 128, four query heads per kv head).
//
// A unit is 64 query rows of one request and one kv head: M = 256 rows of (head, query row), 128 in each CTA of the pair
// (CTA r: query rows 32 r .. 32 r + 31, four heads).  Keys come in tiles of 128: for the scores each CTA holds 64 keys of
// the tile (both halves of the dims), for the output 64 dims of all 128 keys, so that a pair reads every key and value
// once for 256 rows.  Even and odd tiles are two independent streams with maxima, sums and accumulators of their own,
// one per half of the warps; while one stream is in its softmax the tensor core works for the other.  They are merged at the
// end of the unit, where the two threads that own a row of TMEM read both accumulators.
//
//   stream s of a unit, tile j (every warp of it in both CTAs unless said otherwise):
//     scores complete -> the warps ask for the stream's next keys
//     outputs of the stream's tile before complete
//       -> probabilities to shared memory; the accumulator is rescaled only when a row's maximum has grown by more than 2^8
//          (a smaller growth leaves probabilities above one, and their sum takes it up: nothing is lost)
//     -> arrival in CTA 0, where a warp of the stream issues the next tile's scores and another the output MMAs
//
// What bounds it: the softmax (128 exponentials a thread are 1024 cycles of a unit that both streams share; two warps per scheduler
// leave its latencies open); loads, hand-overs and the scores' MMAs are the rest.  512 rows of 512 keys: 27.4 us a layer with
// attn_prefill_tile, 14.4 here; behind 3500 keys 177 and 61.
#pragma once
#include "gemm_tc.cuh"

namespace blink {

constexpr int AP_ROWS = ATT_PAIR_ROWS;   // query rows of a unit
constexpr int AP_KT = 128;               // keys of a tile
constexpr int AP_Q = 0, AP_P = 32768, AP_K = AP_P + 2 * 32768, AP_V = AP_K + 2 * 16384, AP_END = AP_V + 4 * 16384;
static_assert(AP_END <= TC_TILE_BUDGET, "operands exceed the dynamic shared memory");

struct AttPairShared {
  // counted in CTA 0: queries (an arrival per CTA), keys (bytes of both CTAs), probabilities (an arrival per warp of the
  // stream in both CTAs).  In each CTA: its own values, and the completions of scores and outputs.
  uint64_t q_full, k_full[2], p_full[2], v_full[2][2], s_full[2], o_part[2], o_full[2];   // (o_part: every tile, o_full: the last)
  uint32_t units, tiles[2], outs[2];   // so far: units, tiles and finished accumulators per stream (the barriers' parities)
  struct {
    int4 req;       // start, rows, first row and batch slot of the unit's request
    int r0;         // first of the unit's query rows in it
    int ids[32];    // block ids of its first four tiles
  } unit[2];        // the first unit, which is the same in all layers of a step, and any other
};
__shared__ __align__(16) AttPairShared g_ap;

__device__ __forceinline__ void ap_init() {   // one thread; the caller makes the barriers visible to the cluster
  mbar_init(&g_ap.q_full, 2);
  for (int s = 0; s < 2; ++s) {
    mbar_init(&g_ap.k_full[s], 1);
    mbar_init(&g_ap.p_full[s], 8);
    mbar_init(&g_ap.v_full[s][0], 1);
    mbar_init(&g_ap.v_full[s][1], 1);
    mbar_init(&g_ap.s_full[s], 1);
    mbar_init(&g_ap.o_part[s], 1);
    mbar_init(&g_ap.o_full[s], 1);
    g_ap.tiles[s] = g_ap.outs[s] = 0u;
  }
  g_ap.units = 0u;
}

// A value that all lanes of the (converged) warp have in common, in a uniform register.
__device__ __forceinline__ uint32_t warp_uniform(uint32_t v) { return __reduce_max_sync(0xffffffffu, v); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {   // two at once
  float2 d;
  asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmov.b64 z, {%6, %7};\n\tfma.rn.f32x2 x, x, y, z;\n\t"
      "mov.b64 {%0, %1}, x;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tadd.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float fast_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// 32 lanes x 32 consecutive 32-bit columns, without the wait: the registers hold nothing before tmem_wait_ld() has named them, and
// even a copy of one may not stand in between, so load and wait lie in one block of straight code.
__device__ __forceinline__ void tmem_ld32_async(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, "
      "%18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
        "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
#define BLINK_RW8(r, i) "+r"(r[i]), "+r"(r[i + 1]), "+r"(r[i + 2]), "+r"(r[i + 3]), "+r"(r[i + 4]), "+r"(r[i + 5]), "+r"(r[i + 6]), "+r"(r[i + 7])
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&a)[32], uint32_t (&b)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : BLINK_RW8(a, 0), BLINK_RW8(a, 8), BLINK_RW8(a, 16), BLINK_RW8(a, 24), BLINK_RW8(b, 0), BLINK_RW8(b, 8), BLINK_RW8(b, 16),
                 BLINK_RW8(b, 24)
               :
               : "memory");
}
#undef BLINK_RW8
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float* v) {
  const uint32_t* r = reinterpret_cast<const uint32_t*>(v);
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
      "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// 16 keys x 64 dims of the pool, counted on CTA 0's barrier whichever CTA asks
__device__ __forceinline__ void tma_kv_pair(void* smem_dst, const CUtensorMap* map, int half, int row, uint32_t bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3}], "
      "[%4], %5;" ::"r"(smem_u32(smem_dst)),
      "l"(map), "r"(half * 64), "r"(row), "r"(bar & PAIR_CTA0_MASK), "l"(policy)
      : "memory");
}
// MN-major operand of 64 columns (128-byte rows of 64 bf16 along N, swizzled, eight k-rows every 1024 bytes).  One such
// block along N, so the offset between blocks is never used.
__device__ __forceinline__ uint64_t smem_desc_sw128_mn(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(1024 >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// One row of a score tile -> probabilities (bf16, swizzled rows of 64 keys, two slabs), their sum, and the largest score.
// One pass and no branch inside: with a pass for the maximum first and the accumulator's rescaling unrolled too, the body of a
// tile was beyond the 32 KB instruction cache (more than twice the time), and a conditional mask copies every value once more.
template <bool MASKED>
__device__ __forceinline__ void ap_probs(uint32_t t_s, uint32_t p_row, int swz, float qscale, float neg, int seen, float& mx, float2& sum) {
  const float2 scale2 = make_float2(qscale, qscale), neg2 = make_float2(neg, neg);
  float mx0 = -INFINITY, mx1 = -INFINITY;
  float2 s0 = make_float2(0.f, 0.f), s1 = s0;
  auto quarter = [&](const uint32_t(&r)[32], int k) {
    float v[32];
#pragma unroll
    for (int x = 0; x < 32; ++x) v[x] = __uint_as_float(r[x]);
    if constexpr (MASKED) {
#pragma unroll
      for (int x = 0; x < 32; ++x) v[x] = 32 * k + x <= seen ? v[x] : -INFINITY;
    }
#pragma unroll
    for (int x = 0; x < 32; x += 4) {
      mx0 = fmaxf(fmaxf(mx0, v[x]), v[x + 1]);
      mx1 = fmaxf(fmaxf(mx1, v[x + 2]), v[x + 3]);
    }
#pragma unroll
    for (int x = 0; x < 32; x += 8) {
      uint32_t o[4];
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        float2 e = fma2(make_float2(v[x + 2 * y], v[x + 2 * y + 1]), scale2, neg2);
        e.x = fast_ex2(e.x);
        e.y = fast_ex2(e.y);
        if (y & 1) s1 = add2(s1, e); else s0 = add2(s0, e);
        const __nv_bfloat162 b2 = __floats2bfloat162_rn(e.x, e.y);
        o[y] = *reinterpret_cast<const uint32_t*>(&b2);
      }
      const uint32_t dst = p_row + (uint32_t)((k >> 1) * 16384) + ((uint32_t)((((k & 1) * 4) + (x >> 3)) ^ swz) << 4);
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(o[0]), "r"(o[1]), "r"(o[2]), "r"(o[3]) : "memory");
    }
  };
  // (a wait for TMEM loads takes some 400 cycles: the second half is on its way while the first is worked on)
  uint32_t va[32], vb[32], vc[32], vd[32];
  tmem_ld32_async(t_s, va);
  tmem_ld32_async(t_s + 32u, vb);
  tmem_wait_ld(va, vb);
  tmem_ld32_async(t_s + 64u, vc);
  tmem_ld32_async(t_s + 96u, vd);
  quarter(va, 0);
  quarter(vb, 1);
  tmem_wait_ld(vc, vd);
  quarter(vc, 2);
  quarter(vd, 3);
  mx = fmaxf(mx0, mx1);
  sum = add2(s0, s1);
}

// The (entry, kv head) units of the first n_entries entries of the step's list, dealt to the pairs in turn.
static __device__ __noinline__ void attn_prefill_pair(const DevCtx& c, int layer, char* base, int n_entries) {
  constexpr int HD = 128, NREP = 4;
  // (warp-uniform values in uniform registers: from vector registers every operand of an MMA is moved first, 100 cycles each)
  const uint32_t rank = warp_uniform(cluster_ctarank());
  const int w = (int)warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int s = w >> 2, q = w & 3;   // stream, and the quarter of the TMEM lanes this warp reads (= its head)
  const int n_units = n_entries * c.Hkv;
  const CUtensorMap* map = reinterpret_cast<const CUtensorMap*>(c.kv_map) + 1;
  const uint32_t tmem = warp_uniform(g_tc_state[0].tmem_base);
  const uint32_t t_s = tmem + (uint32_t)s * 128u + ((uint32_t)(q * 32) << 16);
  const uint32_t t_o = tmem + 256u + ((uint32_t)(q * 32) << 16);
  const uint32_t b_s = smem_u32(base);
  const uint32_t idesc_s = idesc_bf16_pair(AP_KT), idesc_o = idesc_bf16_pair(HD) | (1u << 16);   // (bit 16: B is MN-major)
  const uint64_t d_q = smem_desc_sw128(b_s + AP_Q), d_k = smem_desc_sw128(b_s + AP_K + s * 16384),
                 d_p = smem_desc_sw128(b_s + AP_P + s * 32768), d_v = smem_desc_sw128_mn(b_s + AP_V + s * 32768);
  const uint64_t policy = l2_evict_normal();
  const float qscale = c.attn_scale * 1.4426950408889634f;
  uint32_t units = warp_uniform(g_ap.units), nt0 = warp_uniform(g_ap.tiles[0]), nt1 = warp_uniform(g_ap.tiles[1]),
           no0 = warp_uniform(g_ap.outs[0]), no1 = warp_uniform(g_ap.outs[1]);
  bool ok = true;   // false once a wait has run out: the rest is skipped, the barriers of the CTA are kept

  if (threadIdx.x == 32) asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  for (int u = (int)blockIdx.x >> 1; u < n_units; u += (int)gridDim.x >> 1) {
    const int e = u / c.Hkv, g = u - e * c.Hkv;
    const int which = u < (int)gridDim.x >> 1 ? 0 : 1;
    auto& rec = g_ap.unit[which];
    if (which || layer == 0 || c.stepped) {
      __syncthreads();   // (the unit before is done with its record)
      if (threadIdx.x < 32) {
        const int4 r = c.pf_unit[e];
        const int qb = c.pf_qb[e];
        if (lane == 0) {
          rec.req = r;
          rec.r0 = qb * AP_ROWS;
        }
        const int last = (r.x + min(r.y, qb * AP_ROWS + AP_ROWS) + 15) / 16 - 1;
        rec.ids[lane] = c.block_table[(size_t)r.w * c.max_blocks_seq + min(lane, last)];
      }
      __syncthreads();
    }
    const int start = (int)warp_uniform((uint32_t)rec.req.x), ntok = (int)warp_uniform((uint32_t)rec.req.y), qstart = rec.req.z,
              r0 = (int)warp_uniform((uint32_t)rec.r0);
    const int32_t* table = c.block_table + (size_t)rec.req.w * c.max_blocks_seq;
    const int n_keys = start + min(ntok, r0 + AP_ROWS), nkb = (n_keys + 15) >> 4;
    const int tiles = (n_keys + AP_KT - 1) / AP_KT;
    const int my_tiles = (tiles + 1 - s) >> 1;
    const uint32_t done = s ? nt1 : nt0;   // the stream's tiles before this unit
    const int r_base = r0 + (int)rank * 32;
    const int blk_rows = c.Hkv * 16;
    const int row_k = (layer * 2 * c.n_blocks * c.Hkv + g) * 16, row_v = row_k + c.n_blocks * c.Hkv * 16;   // pool rows of block 0

    // Keys and values: a quarter of the stream's copies by each of its warps (a copy takes its thread 100 cycles or so, and the
    // slowest warp sets the pace).  Blocks past the end repeat the last one (masked scores, left out of the output MMAs).
    int ids = 0;
    auto block_ids = [&](int i) { return lane < 8 ? table[min(8 * (s + 2 * i) + lane, nkb - 1)] : 0; };
    auto load_k = [&](int id) {
      const int blk = (int)warp_uniform((uint32_t)__shfl_sync(0xffffffffu, id, 4 * (int)rank + q));
      if (elect_one()) {
        if (rank == 0 && q == 0) mbar_expect_tx(&g_ap.k_full[s], 32768u);
        char* dst = base + AP_K + s * 16384 + q * 2048;
        const int row = row_k + blk * blk_rows;
        tma_kv_pair(dst, map, 0, row, smem_u32(&g_ap.k_full[s]), policy);
        tma_kv_pair(dst + 8192, map, 1, row, smem_u32(&g_ap.k_full[s]), policy);
      }
      __syncwarp();
    };
    auto load_v = [&](int id, uint32_t n) {   // n: the stream's tile, counted over the units
      const int b0 = (int)warp_uniform((uint32_t)__shfl_sync(0xffffffffu, id, 2 * q)),
                b1 = (int)warp_uniform((uint32_t)__shfl_sync(0xffffffffu, id, 2 * q + 1));
      if (elect_one()) {
        uint64_t* bar = &g_ap.v_full[s][n & 1u];
        char* dst = base + AP_V + (s * 2 + (int)(n & 1u)) * 16384 + q * 4096;
        if (q == 0) mbar_expect_tx(bar, 16384u);
        tma_load_2d_hint(dst, map, (int)rank * 64, row_v + b0 * blk_rows, bar, policy);
        tma_load_2d_hint(dst + 2048, map, (int)rank * 64, row_v + b1 * blk_rows, bar, policy);
      }
      __syncwarp();
    };
    // queries: row = head * 32 + query row, two slabs of 64 dims
#pragma unroll 2
    for (int k = 0; k < 8; ++k) {
      const int row = k * 16 + (int)(threadIdx.x >> 4), ck = threadIdx.x & 15;
      const int r = r_base + (row & 31);
      const bool live = r < ntok;
      const char* src = reinterpret_cast<const char*>(c.qb) + ((size_t)(qstart + (live ? r : 0)) * c.q_dim + (g * NREP + (row >> 5)) * HD) * 2 + ck * 16;
      const uint32_t dst = b_s + AP_Q + (ck >> 3) * 16384 + row * 128 + (((ck & 7) ^ (row & 7)) << 4);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(live ? 16u : 0u) : "memory");
    }
    if (my_tiles > 0 && ok) {
      const int id0 = rec.ids[8 * s + (lane & 7)];
      load_k(id0);
      load_v(id0, done);
      if (my_tiles > 1) {
        ids = rec.ids[16 + 8 * s + (lane & 7)];
        load_v(ids, done + 1u);
      }
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0) mbar_arrive_cta0_release(&g_ap.q_full);

    auto issue_scores = [&](uint32_t n) {   // (first warp of the stream in CTA 0)
      ok = ok && mbar_wait_warp(c, &g_ap.k_full[s], n & 1u);
      if (!ok) return;
      tc_fence_after();
      if (elect_one()) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          umma_bf16_pair(tmem + (uint32_t)s * 128u, d_q + (uint64_t)((i >> 2) * 1024 + (i & 3) * 2), d_k + (uint64_t)((i >> 2) * 512 + (i & 3) * 2),
                         idesc_s, i ? 1u : 0u);
        umma_commit_pair(&g_ap.s_full[s]);
      }
      __syncwarp();
    };
    if (rank == 0 && q == 0 && my_tiles > 0) {
      ok = ok && mbar_wait_warp_acquire(c, &g_ap.q_full, units & 1u);
      issue_scores(done);
    }

    float m = -INFINITY, l = 0.f;   // maximum in use (scaled, log2 domain) and sum of this row
    const int pos = start + r_base + lane;
    for (int i = 0; i < my_tiles; ++i) {
      const int j = s + 2 * i;
      const uint32_t n = done + (uint32_t)i;
      ok = ok && mbar_wait_warp(c, &g_ap.s_full[s], n & 1u);
      tc_fence_after();
      if (i + 1 < my_tiles && ok) load_k(ids);
      if (i > 0) {   // the output MMAs of the tile before are done with the probabilities, the accumulator and their values
        ok = ok && mbar_wait_warp(c, &g_ap.o_part[s], (n - 1u) & 1u);
        tc_fence_after();
      }
      // Probabilities against the maximum in use.  The largest score is followed on the way; when it turns out to have grown by
      // more than 2^8 (always so for the first tile, otherwise rare) the accumulator and the sum are rescaled and the pass is run again.
      const uint32_t p_row = b_s + AP_P + (uint32_t)(s * 32768 + (q * 32 + lane) * 128);
      const int seen = pos - j * AP_KT;   // keys of the tile up to this one are visible to the row
      const bool masked = AP_KT - 1 > start + r_base - j * AP_KT;   // some row of the warp does not see all keys
      float2 sum;
#pragma unroll 1
      while (true) {
        float mx;
        if (masked) ap_probs<true>(t_s, p_row, lane & 7, qscale, m == -INFINITY ? 0.f : -m, seen, mx, sum);
        else ap_probs<false>(t_s, p_row, lane & 7, qscale, m == -INFINITY ? 0.f : -m, seen, mx, sum);
        mx *= qscale;
        if (!__any_sync(0xffffffffu, mx > m + 8.f)) break;
        const float mn = fmaxf(m, mx);
        const float f = mn == -INFINITY ? 1.f : fast_ex2(m - mn);
        m = mn;
        l *= f;
        if (i > 0 && ok) {
          const uint32_t t = t_o + (uint32_t)s * 128u;
#pragma unroll 1
          for (int k = 0; k < 128; k += 16) {
            float o[16];
            tmem_ld16(t + (uint32_t)k, o);
#pragma unroll
            for (int x = 0; x < 16; ++x) o[x] *= f;
            tmem_st16(t + (uint32_t)k, o);
          }
          tmem_wait_st();
        }
      }
      l += sum.x + sum.y;
      if (q == 1) {   // this warp stands for the values of its CTA
        ok = ok && mbar_wait_warp(c, &g_ap.v_full[s][n & 1u], (n >> 1) & 1u);
        if (j == tiles - 1 && (n_keys & 15) != 0) {   // the tail of the last block holds whatever the pool held: 0 x NaN
          char* vt = base + AP_V + (s * 2 + (int)(n & 1u)) * 16384 + ((n_keys - j * AP_KT) >> 4) * 2048;
          for (int k = (n_keys & 15) * 8 + lane; k < 128; k += 32) *reinterpret_cast<uint4*>(vt + k * 16) = make_uint4(0u, 0u, 0u, 0u);
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cta0_release(&g_ap.p_full[s]);
      // The next scores before the outputs of this tile (by another warp, so that neither waits for the other's issue): the
      // softmax can go on while the tensor core works on the outputs.
      if (rank == 0 && q == 0 && i + 1 < my_tiles) {
        ok = ok && mbar_wait_warp_acquire(c, &g_ap.p_full[s], n & 1u);
        issue_scores(n + 1u);
      } else if (rank == 0 && q == 2) {
        ok = ok && mbar_wait_warp_acquire(c, &g_ap.p_full[s], n & 1u);
        if (ok) {
          tc_fence_after();
          const int nk = min(8, nkb - 8 * j);
          const uint64_t dv = d_v + (uint64_t)((n & 1u) * 1024u);
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < 8; ++k)
              if (k < nk) umma_bf16_pair(tmem + 256u + (uint32_t)s * 128u, d_p + (uint64_t)((k >> 2) * 1024 + (k & 3) * 2), dv + (uint64_t)(k * 128), idesc_o,
                             (i | k) ? 1u : 0u);
            umma_commit_pair(&g_ap.o_part[s]);
            if (i + 1 == my_tiles) umma_commit_pair(&g_ap.o_full[s]);
          }
          __syncwarp();
        }
      }
      if (i + 1 < my_tiles && ok) {
        if (i > 0) load_v(ids, n + 1u);
        if (i + 2 < my_tiles) ids = block_ids(i + 2);
      }
    }
    // merge the streams: each of the two threads of a row takes half of the dims
    // (maximum and sum of every row go where the stream's keys were: its scores are complete)
    float2* ml = reinterpret_cast<float2*>(base + AP_K) + q * 32 + lane;
    ml[s * 2048] = make_float2(m, l);
    const bool two = tiles > 1;
    ok = ok && mbar_wait_warp(c, &g_ap.o_full[0], no0 & 1u);
    if (two) ok = ok && mbar_wait_warp(c, &g_ap.o_full[1], no1 & 1u);
    tc_fence_after();
    __syncthreads();
    const float2 a = ml[0], b = ml[2048];
    const float M = two ? fmaxf(a.x, b.x) : a.x;
    float f0 = fast_ex2(a.x - M), f1 = two ? fast_ex2(b.x - M) : 0.f;   // (stream 0 has key 0, which every row sees: M is finite)
    const float inv = __fdividef(1.0f, two ? fmaf(f1, b.y, f0 * a.y) : a.y);
    f0 *= inv;
    f1 *= inv;
    // through shared memory (where the probabilities were), so that rows leave whole
    const uint32_t o_row = b_s + AP_P + (uint32_t)((q * 32 + lane) * 256);
    uint32_t a0[32], a1[32], b0[32], b1[32];   // (one stream: what the other's accumulator holds counts for nothing)
    tmem_ld32_async(t_o + (uint32_t)(s * 64), a0);
    tmem_ld32_async(t_o + (uint32_t)(s * 64 + 32), a1);
    tmem_ld32_async(t_o + 128u + (uint32_t)(s * 64), b0);
    tmem_ld32_async(t_o + 128u + (uint32_t)(s * 64 + 32), b1);
    tmem_wait_ld(a0, a1);
    tmem_wait_ld(b0, b1);
    auto half_row = [&](const uint32_t(&r0)[32], const uint32_t(&r1)[32], int h) {
      auto dim = [&](int x) { return fmaf(two ? __uint_as_float(r1[x]) : 0.f, f1, __uint_as_float(r0[x]) * f0); };
#pragma unroll
      for (int k = 0; k < 32; k += 8) {
        uint32_t o[4];
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          const __nv_bfloat162 b2 = __floats2bfloat162_rn(dim(k + 2 * y), dim(k + 2 * y + 1));
          o[y] = *reinterpret_cast<const uint32_t*>(&b2);
        }
        const uint32_t dst = o_row + (((s * 8 + h * 4 + (k >> 3)) ^ (lane & 7)) << 4);   // 16-byte pieces, swizzled by the row
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(o[0]), "r"(o[1]), "r"(o[2]), "r"(o[3]) : "memory");
      }
    };
    half_row(a0, b0, 0);
    half_row(a1, b1, 1);
    tc_fence_before();
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // copies land there again for the next unit
    __syncthreads();
#pragma unroll 2
    for (int k = 0; k < 8; ++k) {
      const int row = k * 16 + (int)(threadIdx.x >> 4), ck = threadIdx.x & 15, r = r_base + (row & 31);
      if (r < ntok && ok)
        *reinterpret_cast<uint4*>(reinterpret_cast<char*>(c.attn) + ((size_t)(qstart + r) * c.q_dim + (g * NREP + (row >> 5)) * HD) * 2 + ck * 16) =
            *reinterpret_cast<const uint4*>(base + AP_P + row * 256 + ((ck ^ (row & 7)) << 4));
    }
    units += 1u;
    nt0 += (uint32_t)((tiles + 1) >> 1);
    nt1 += (uint32_t)(tiles >> 1);
    no0 += 1u;
    no1 += two ? 1u : 0u;
  }
  if (!ok) {   // copies of this CTA may be on their way: let them land before the shared memory is given up
    const long long t0 = clock64();
    while (clock64() - t0 < 200000ll) {}
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0) {
    g_ap.units = units;
    g_ap.tiles[0] = nt0;
    g_ap.tiles[1] = nt1;
    g_ap.outs[0] = no0;
    g_ap.outs[1] = no1;
  }
}

}  // namespace blink
