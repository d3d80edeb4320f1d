// Sampling of the step's rows: greedy, top-k with temperature, nucleus (Section 4.2 of the paper: "Top-P with
// temperature", sampling captured inside the step).
//
// A row of 128 256 logits is half a megabyte.  One CTA reading it twice took 60 us for top-k (a single SM, and a
// single thread for the k exponentials) and 590 us for the nucleus, so the work is split in two:
//   * all CTAs together: the maximum of every chunk of the row (at most 1024 chunks), and, for nucleus rows, the
//     weights of the row per bucket of z (phase_sample_max, phase_sample_weights);
//   * one CTA per row (sample_row): the k-th largest of 256 maxima over chunks bounds the candidates from below, so
//     only the few dozen chunks whose maximum reaches the bound are read again; k weights by k threads.
// Measured on the 8B shape: top-k 60 -> 30 us for one row, 60 -> 40 for 58; nucleus 590 -> 72 for 20 (grid barriers
// included).
#pragma once
#include "control.cuh"
#include "dev_ctx.cuh"
#include "forward.cuh"

namespace blink {

// Philox4x32-10 (Salmon et al., SC'11): counter-based, so the draw for (ticket, index)
// does not depend on batch composition.
__device__ __forceinline__ uint32_t philox4x32_10_word0(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                                        uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
    const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
    k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
  }
  return c0;
}

// order-preserving map float -> uint32 (larger float => larger key)
__device__ __forceinline__ uint32_t float_key(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// ---- top-p (nucleus) arithmetic: Section 4.2 names "Top-P with temperature" as the in-step sampler ----
// Weights are integers, q = floor(exp(z - z0) * 2^40) with z0 the largest z of the row, so that every
// sum is exact and no result depends on the order in which a parallel machine adds: the nucleus is
// the smallest prefix of the order (z desc, index asc) with cum * 2^24 >= P24 * Q (Q = total weight,
// P24 = round(top_p * 2^24) in [1, 2^24]); the draw is renormalised to its weight M: with the 24-bit
// uniform x24, the token is the first of the order with cum > (x24 * M) >> 24.
__device__ __forceinline__ unsigned long long nucleus_weight(float z, float z0) {
  return __double2ull_rd(exp((double)z - (double)z0) * 1099511627776.0);
}
__device__ __forceinline__ unsigned long long nucleus_p24(float top_p) {
  long long p = (long long)rint((double)top_p * 16777216.0);
  return (unsigned long long)(p < 1 ? 1 : (p > 16777216 ? 16777216 : p));
}
// ceil(p24 * Q / 2^24): the weight the nucleus has to reach (Q < 2^58, p24 <= 2^24)
__device__ __forceinline__ unsigned long long nucleus_need(unsigned long long p24, unsigned long long Q) {
  unsigned long long lo = p24 * Q, hi = __umul64hi(p24, Q);
  const unsigned long long lo2 = lo + 16777215ull;
  if (lo2 < lo) hi += 1;
  return (hi << 40) | (lo2 >> 24);
}
// (x24 * M) >> 24
__device__ __forceinline__ unsigned long long nucleus_target(unsigned long long x24, unsigned long long M) {
  return (__umul64hi(x24, M) << 40) | ((x24 * M) >> 24);
}

// ---- chunks of a row ------------------------------------------------------------------------------------
// A chunk is a power of two of elements, at least 4, so that a row has at most SAMPLE_CHUNKS of them.
constexpr int SAMPLE_CHUNKS = 1024;
__device__ __forceinline__ int sample_chunk_len(int V) {
  int cl = 4;
  while ((long long)cl * SAMPLE_CHUNKS < V) cl <<= 1;
  return cl;
}
__device__ __forceinline__ bool sample_row_vec(const float* lg, int V) { return (V & 3) == 0 && ((size_t)lg & 15) == 0; }
// Four elements from i (a multiple of 4) on, -infinity past the row.  The two forms are chosen outside the loops: a
// branch around every load would make each wait for the one before.
template <bool VEC>
__device__ __forceinline__ float4 sample_load4(const float* lg, int V, int i) {
  if constexpr (VEC) {
    const float4 v = __ldcg(reinterpret_cast<const float4*>(lg + min(i, V - 4)));   // clamped: always a valid address
    return i < V ? v : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
  } else {
    float4 v;
    v.x = i < V ? lg[i] : -INFINITY;
    v.y = i + 1 < V ? lg[i + 1] : -INFINITY;
    v.z = i + 2 < V ? lg[i + 2] : -INFINITY;
    v.w = i + 3 < V ? lg[i + 3] : -INFINITY;
    return v;
  }
}
__device__ __forceinline__ float max4(const float4& v) { return fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)); }
// One warp: maxima of the chunks in elements [i0, i0 + SAMPLE_WARP_SPAN) of the row (eight loads in flight per lane).
constexpr int SAMPLE_WARP_SPAN = 1024;
__device__ __forceinline__ void sample_chunk_maxima(const float* lg, int V, int cl, int i0, float* cmax) {
  const int lane = threadIdx.x & 31;
  float m[8];
  if (sample_row_vec(lg, V)) {
    float4 v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = sample_load4<true>(lg, V, i0 + k * 128 + lane * 4);
#pragma unroll
    for (int k = 0; k < 8; ++k) m[k] = max4(v[k]);
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) m[k] = max4(sample_load4<false>(lg, V, i0 + k * 128 + lane * 4));
  }
  const int shift = 31 - __clz(cl);
  if (cl <= 128) {
    const int lanes = cl >> 2;   // lanes of one chunk
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      for (int o = lanes >> 1; o > 0; o >>= 1) m[k] = fmaxf(m[k], __shfl_xor_sync(0xffffffffu, m[k], o));
      const int i = i0 + k * 128 + lane * 4;
      if ((lane & (lanes - 1)) == 0 && i < V) cmax[i >> shift] = m[k];
    }
  } else {   // cl <= SAMPLE_WARP_SPAN: several 128-element blocks of one chunk
    float run = -INFINITY;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      run = fmaxf(run, m[k]);
      if ((((k + 1) * 128) & (cl - 1)) == 0) {
        const float t = warp_max(run);
        const int i = i0 + (k + 1) * 128 - cl;
        if (lane == 0 && i < V) cmax[i >> shift] = t;
        run = -INFINITY;
      }
    }
  }
}
// Rows whose maxima and weights are taken by all CTAs together: those of more than 24576 entries.  Sampling in the loop by
// the row's own CTA | with the extra phase, us, for greedy and the nucleus at 1, 20 and 100 rows:
//   16384 entries:  8.8 |  9.1, 8.4 | 8.9, 8.1 | 10.2     62 | 52,  72 | 66,  74 | 82
//   24576          10.9 |  9.8, 10.5 | 9.3, 10.5 | 12.5  103 | 83, 133 | 118, 137 | 144
//   28672          12.8 |  9.6, 12.5 | 9.5, 12.5 | 12.7  119 | 97, 155 | 133, 161 | 166
//   32000          12.9 |  9.6, 12.6 | 9.5, 12.6 | 12.8  134 | 104, 174 | 152, 178 | 187
// (top-k as greedy, 11 us more.)  Beyond 2^20 a chunk is longer than a warp's span.
__host__ __device__ __forceinline__ bool sample_split_rows(int V) { return V > 24576 && V <= SAMPLE_WARP_SPAN * SAMPLE_CHUNKS; }

// The lowest index whose value under `z` (monotone) is `top`, the largest of the row; the whole CTA, all threads get the
// answer.  NaN is never the largest, so a row of NaN alone has none: token 0.
template <typename F>
__device__ __forceinline__ int sample_first_max(const float* lg, int V, int cl, const float* s_cmax, float top, F z) {
  constexpr int NONE = 0x7fffffff;
  __shared__ int s_chunk, s_pick;
  __syncthreads();
  if (threadIdx.x == 0) { s_chunk = NONE; s_pick = NONE; }
  __syncthreads();
  int i0 = 0, i1 = V;
  if (top > -INFINITY) {   // (else the maximum of a chunk of NaN looks like a member)
    for (int i = threadIdx.x; i < (V + cl - 1) / cl; i += FWD_THREADS)
      if (z(s_cmax[i]) == top) { atomicMin(&s_chunk, i); break; }
    __syncthreads();
    if (s_chunk != NONE) { i0 = s_chunk * cl; i1 = min(V, i0 + cl); }
  }
  for (int i = i0 + threadIdx.x; i < i1; i += FWD_THREADS)
    if (z(lg[i]) == top) { atomicMin(&s_pick, i); break; }
  __syncthreads();
  return s_pick == NONE ? 0 : s_pick;
}

// all CTAs: chunk maxima of every sampled row; nucleus weights start at zero
static __device__ __noinline__ void phase_sample_max(const DevCtx& c) {
  const int R = c.ss->cur_rows, V = c.V;
  if (!sample_split_rows(V)) return;
  if (c.ss->cur_nuc)
    for (int i = blockIdx.x * FWD_THREADS + threadIdx.x; i < R * 256; i += gridDim.x * FWD_THREADS) {
      c.nuc_m[i] = 0ull;
      c.nuc_c[i] = 0u;
    }
  const int cl = sample_chunk_len(V);
  const int spans = (V + SAMPLE_WARP_SPAN - 1) / SAMPLE_WARP_SPAN;
  const int nw = gridDim.x * (FWD_THREADS / 32);
  for (int u = blockIdx.x * (FWD_THREADS / 32) + (threadIdx.x >> 5); u < R * spans; u += nw) {
    const int r = u / spans, sp = u - r * spans;
    sample_chunk_maxima(c.logits + (size_t)r * V, V, cl, sp * SAMPLE_WARP_SPAN, c.cmax + (size_t)r * SAMPLE_CHUNKS);
  }
}

// ---- weights of a row per bucket of z -------------------------------------------------------------------
// An entry more than 28 below the largest z has the weight floor(exp(-28) * 2^40) = 0 and is never the answer: bucket 0.
// Buckets 255 .. 1 divide the distances from 0 to the smaller of 28 and the spread of the row, which is taken from its
// first entries: what lies further down still has bucket 1.  Over a fixed 28 a row of small or nearly equal logits falls
// into a few buckets, whose sums every thread then adds to (100 such rows of 32000 entries in a step: 513 us, by their
// spread 187; of 128256 entries, shared by all CTAs, 1030 and 800).
constexpr float NUC_SPAN = 28.0f;
__device__ __forceinline__ int nuc_bucket(float z, float z0, float scale) {
  const float d = z0 - z;
  return d <= NUC_SPAN ? 255 - min((int)(d * scale), 254) : 0;
}
__device__ __forceinline__ bool nucleus_row(int top_k, float top_p) { return top_k <= 0 && top_p > 0.f && top_p < 1.f; }

// Weights and counts of elements [i0, i1) into shared memory.  A weight of up to 41 bits is added as three limbs of
// 14 bits: 32-bit adds into shared memory are native, the 64-bit one is a compare-and-swap loop.  Eight exponentials per
// thread are worked on before the first add: with a branch after each they wait for one another (20 rows of 32000 normal
// logits by a CTA each: 420 us, together 150).
constexpr int NUC_LIMB_BITS = 14;
constexpr int NUC_LIMB_ENTRIES = 1 << (32 - NUC_LIMB_BITS);   // so many entries of one bucket fit a 32-bit sum
struct NucLimbs {
  unsigned int w[3][256];
  unsigned int n[256];
};
__device__ __forceinline__ void nuc_add_range(NucLimbs& L, const float* lg, int V, int i0, int i1, float temp, float z0, float scale) {
  constexpr int U = 2;   // vectors per thread whose exponentials are worked on together
  const bool vec = sample_row_vec(lg, V);
  for (int base = i0 + threadIdx.x * 4; base < i1; base += U * FWD_THREADS * 4) {
    float e[4 * U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = base + u * FWD_THREADS * 4;
      const float4 v = vec ? sample_load4<true>(lg, V, i) : sample_load4<false>(lg, V, i);
      e[4 * u] = v.x; e[4 * u + 1] = v.y; e[4 * u + 2] = v.z; e[4 * u + 3] = v.w;
    }
    int b[4 * U];
    unsigned long long q[4 * U];
#pragma unroll
    for (int k = 0; k < 4 * U; ++k) {
      const float z = __fdiv_rn(e[k], temp);
      b[k] = base + (k >> 2) * FWD_THREADS * 4 + (k & 3) < i1 ? nuc_bucket(z, z0, scale) : 0;
      q[k] = nucleus_weight(z, z0);
    }
#pragma unroll
    for (int k = 0; k < 4 * U; ++k) {
      if (b[k]) {
        atomicAdd(&L.w[0][b[k]], (unsigned int)q[k] & 16383u);
        atomicAdd(&L.w[1][b[k]], (unsigned int)(q[k] >> NUC_LIMB_BITS) & 16383u);
        atomicAdd(&L.w[2][b[k]], (unsigned int)(q[k] >> (2 * NUC_LIMB_BITS)));
        atomicAdd(&L.n[b[k]], 1u);
      }
    }
  }
}
// The whole CTA: weight m and number n of the entries of bucket threadIdx.x among elements [i0, i1).
__device__ __forceinline__ void nuc_bucket_sums(NucLimbs& L, const float* lg, int V, int i0, int i1, float temp, float z0, float scale,
                                                unsigned long long& m, unsigned int& n) {
  const int b = threadIdx.x;
  m = 0ull;
  n = 0u;
  for (; i0 < i1; i0 += NUC_LIMB_ENTRIES) {   // (a thread clears and reads its own bucket)
    L.w[0][b] = L.w[1][b] = L.w[2][b] = L.n[b] = 0u;
    __syncthreads();
    nuc_add_range(L, lg, V, i0, min(i1 - i0, NUC_LIMB_ENTRIES) + i0, temp, z0, scale);
    __syncthreads();
    m += (unsigned long long)L.w[0][b] + ((unsigned long long)L.w[1][b] << NUC_LIMB_BITS) +
         ((unsigned long long)L.w[2][b] << (2 * NUC_LIMB_BITS));
    n += L.n[b];
  }
}
__device__ __forceinline__ float block_max(float v, float* s_red /*[8]*/) {
  v = warp_max(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
  __syncthreads();
  float t = -INFINITY;
#pragma unroll
  for (int i = 0; i < FWD_THREADS / 32; ++i) t = fmaxf(t, s_red[i]);
  return t;
}
// Buckets per unit of z, the same in every CTA that works on the row.
__device__ __forceinline__ float nuc_scale(const float* lg, int V, float temp, float z0, float* s_red) {
  float low = INFINITY;
  for (int i = threadIdx.x * 4; i < min(V, FWD_THREADS * 4); i += FWD_THREADS * 4)
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i + k < V) low = fminf(low, lg[i + k]);
  low = -block_max(-low, s_red);
  const float spread = fminf(NUC_SPAN, z0 - __fdiv_rn(low, temp));
  return spread > 0.f ? 254.0f / spread : 0.f;
}
__device__ __forceinline__ float sample_row_max(const float* cmax, int n, float* s_red) {
  float m = -INFINITY;
  for (int i = threadIdx.x; i < n; i += FWD_THREADS) m = fmaxf(m, cmax[i]);
  return block_max(m, s_red);
}

// all CTAs, after the maxima: the bucket weights of the nucleus rows, every row by as many CTAs as there are to share
static __device__ __noinline__ void phase_sample_weights(const DevCtx& c, float* smem) {
  if (!c.ss->cur_nuc || !sample_split_rows(c.V)) return;
  __shared__ float s_red[FWD_THREADS / 32];
  NucLimbs& L = *reinterpret_cast<NucLimbs*>(smem);
  const int R = c.ss->cur_rows, V = c.V;
  const int cl = sample_chunk_len(V), nch = (V + cl - 1) / cl;
  const int parts = max(1, (int)gridDim.x / R);
  const int len = ((V + parts - 1) / parts + SAMPLE_WARP_SPAN - 1) & ~(SAMPLE_WARP_SPAN - 1);
  for (int u = blockIdx.x; u < R * parts; u += gridDim.x) {
    const int r = u / parts, part = u - r * parts;
    const int b = c.it_bslot[c.row_item[r]];
    if (!nucleus_row(c.b_topk[b], c.b_topp[b]) || part * len >= V) continue;   // uniform over the CTA
    const float temp = c.b_temp[b];
    const float* lg = c.logits + (size_t)r * V;
    const float z0 = __fdiv_rn(sample_row_max(c.cmax + (size_t)r * SAMPLE_CHUNKS, nch, s_red), temp);
    const float scale = nuc_scale(lg, V, temp, z0, s_red);
    unsigned long long m;
    unsigned int n;
    nuc_bucket_sums(L, lg, V, part * len, min(V, (part + 1) * len), temp, z0, scale, m, n);
    if (n) {
      if (m) atomicAdd(&c.nuc_m[(size_t)r * 256 + threadIdx.x], m);
      atomicAdd(&c.nuc_c[(size_t)r * 256 + threadIdx.x], n);
    }
  }
}

// ---- whole-row nucleus search (one CTA per row) -----------------------------------------------------------
constexpr int NUC_CAND = 1024;
struct NucShared {
  unsigned long long m0[256];   // level 0: weight per bucket of z
  unsigned int c0[256];         //          and number of entries
  unsigned long long m[256];    // deeper levels: buckets linear in the float key inside [klo, khi]
  unsigned int cn[256];
  unsigned long long acc;       // weight of everything ahead of the current member set in the order
  unsigned long long res_cum;   // result: cumulative weight up to and including the entry found
  unsigned int klo, khi, cnt;
  int b0, first, done, res_idx, n, n_list;
  unsigned int chunk_cnt[FWD_THREADS];
};
// From bucket 255 down: the first bucket b >= 1 whose weight carries the running sum past t, or 0; acc gets the sum of
// the buckets above it.  One warp, eight buckets per lane.
__device__ __forceinline__ int nuc_pick_bucket(const unsigned long long* m, unsigned long long acc0, unsigned long long t,
                                               unsigned long long& acc) {
  const int lane = threadIdx.x & 31;
  unsigned long long own = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) own += (255 - 8 * lane - k) > 0 ? m[255 - 8 * lane - k] : 0ull;
  unsigned long long incl = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  const unsigned hit = __ballot_sync(0xffffffffu, acc0 + incl > t);
  int b = 0;
  unsigned long long a = acc0 + __shfl_sync(0xffffffffu, incl, 31);
  if (hit) {
    const int src = __ffs(hit) - 1;
    a = acc0 + incl - own;
    b = 255 - 8 * lane;
    for (int k = 0; k < 8 && a + m[b] <= t; ++k) a += m[b--];
    b = __shfl_sync(0xffffffffu, b, src);
    a = __shfl_sync(0xffffffffu, a, src);
  }
  acc = a;
  return b;
}
// Chunks of the row for which `wanted(chunk maximum)` holds, as a list (in no particular order).
template <typename F>
__device__ __forceinline__ int sample_list_chunks(const float* s_cmax, int nch, int* s_list, int* s_n, F wanted) {
  if (threadIdx.x == 0) *s_n = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < nch; i += FWD_THREADS)
    if (wanted(s_cmax[i])) s_list[atomicAdd(s_n, 1)] = i;
  __syncthreads();
  return *s_n;
}
// f(value, index) for every element of the listed chunks, four vectors in flight per thread
template <bool VEC, typename F>
__device__ __forceinline__ void sample_for_listed_as(const float* lg, int V, int cl, const int* s_list, int n_list, F f) {
  const int sh = 31 - __clz(cl) - 2;   // log2 of the chunk's vectors
  const int total = n_list << sh;
  for (int base = threadIdx.x; base < total; base += 4 * FWD_THREADS) {
    float4 v[4];
    int idx[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int q = base + k * FWD_THREADS;
      idx[k] = q < total ? s_list[q >> sh] * cl + ((q & ((1 << sh) - 1)) << 2) : V;
      v[k] = sample_load4<VEC>(lg, V, idx[k]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (idx[k] < V) f(v[k].x, idx[k]);
      if (idx[k] + 1 < V) f(v[k].y, idx[k] + 1);
      if (idx[k] + 2 < V) f(v[k].z, idx[k] + 2);
      if (idx[k] + 3 < V) f(v[k].w, idx[k] + 3);
    }
  }
}
template <typename F>
__device__ __forceinline__ void sample_for_listed(const float* lg, int V, int cl, const int* s_list, int n_list, F f) {
  if (sample_row_vec(lg, V)) sample_for_listed_as<true>(lg, V, cl, s_list, n_list, f);
  else sample_for_listed_as<false>(lg, V, cl, s_list, n_list, f);
}

// First entry of the order (z desc, index asc) whose cumulative weight exceeds t (t < total weight).
// The member set starts as one level-0 bucket and is narrowed 256-fold per pass over the chunks that can hold members
// (buckets over the float-key interval of the set) until it fits the candidate buffer, which is then ranked
// exactly.  A set that cannot be narrowed (more than NUC_CAND equal values) is resolved by index.
static __device__ __noinline__ void nucleus_locate(NucShared& st, const float* lg, int V, int cl, const float* s_cmax, float temp,
                                                   float z0, float scale, unsigned long long t, float* s_cz, int* s_ci, float* s_sz, int* s_si) {
  const int tid = threadIdx.x;
  const int nch = (V + cl - 1) / cl;
  if (tid < 32) {
    unsigned long long acc;
    const int b = nuc_pick_bucket(st.m0, 0ull, t, acc);
    if (tid == 0) {
      st.b0 = b; st.acc = acc; st.cnt = st.c0[b]; st.klo = 0u; st.khi = 0xffffffffu; st.first = 1; st.done = 0;
    }
  }
  __syncthreads();
  const int b0 = st.b0;
  int* s_list = reinterpret_cast<int*>(s_sz);   // free until the candidates are ranked
  for (int level = 0; level < 8; ++level) {   // a level divides the key interval by 256: four suffice
    const unsigned int klo = st.klo, khi = st.khi;
    const int n_list = sample_list_chunks(s_cmax, nch, s_list, &st.n_list,
                                          [&](float m) { return nuc_bucket(__fdiv_rn(m, temp), z0, scale) >= b0; });
    if (st.cnt <= (unsigned)NUC_CAND) {
      // ---- gather the members, rank them exactly, walk the cumulative weights ----
      if (tid == 0) st.n = 0;
      __syncthreads();
      sample_for_listed(lg, V, cl, s_list, n_list, [&](float v, int i) {
        const float z = __fdiv_rn(v, temp);
        const unsigned int key = float_key(z);
        if (nuc_bucket(z, z0, scale) == b0 && key >= klo && key <= khi) {
          const int p = atomicAdd(&st.n, 1);
          if (p < NUC_CAND) { s_cz[p] = z; s_ci[p] = i; }
        }
      });
      __syncthreads();
      const int nc = min(st.n, NUC_CAND);
      for (int a = tid; a < nc; a += FWD_THREADS) {
        const float za = s_cz[a];
        const int ia = s_ci[a];
        int rank = 0;
        for (int j = 0; j < nc; ++j) {
          const float zj = s_cz[j];
          rank += (zj > za) || (zj == za && s_ci[j] < ia);
        }
        s_sz[rank] = za; s_si[rank] = ia;
      }
      __syncthreads();
      if (tid < 32) {   // 32 weights at a time, their running sum by shuffles
        unsigned long long cum = st.acc;
        int pick = nc > 0 ? s_si[nc - 1] : 0;
        for (int j0 = 0; j0 < nc; j0 += 32) {
          const int j = j0 + tid;
          unsigned long long incl = j < nc ? nucleus_weight(s_sz[j], z0) : 0ull;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
            if (tid >= o) incl += y;
          }
          const unsigned hit = __ballot_sync(0xffffffffu, j < nc && cum + incl > t);
          if (hit) {
            const int src = __ffs(hit) - 1;
            pick = s_si[j0 + src];
            cum += __shfl_sync(0xffffffffu, incl, src);
            break;
          }
          cum += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (tid == 0) { st.res_idx = pick; st.res_cum = cum; st.done = 1; }
      }
      __syncthreads();
      return;
    }
    if (st.first) {   // key interval of the level-0 bucket's members
      __syncthreads();
      if (tid == 0) { st.klo = 0xffffffffu; st.khi = 0u; }
      __syncthreads();
      unsigned int lo = 0xffffffffu, hi = 0u;
      sample_for_listed(lg, V, cl, s_list, n_list, [&](float v, int) {
        const float z = __fdiv_rn(v, temp);
        if (nuc_bucket(z, z0, scale) == b0) {
          const unsigned int key = float_key(z);
          lo = min(lo, key);
          hi = max(hi, key);
        }
      });
      if (lo <= hi) { atomicMin(&st.klo, lo); atomicMax(&st.khi, hi); }
      __syncthreads();
      if (tid == 0) st.first = 0;
      __syncthreads();
      continue;   // same member set, now with its key interval
    }
    if (klo == khi) {
      // ---- more than NUC_CAND entries with one and the same z: equal weights, ordered by index ----
      const float z = __uint_as_float((klo & 0x80000000u) ? (klo & 0x7fffffffu) : ~klo);
      const unsigned long long q0 = nucleus_weight(z, z0);            // > 0: the set's weight exceeds t - acc
      const unsigned long long jl = q0 > 0 ? (t - st.acc) / q0 : 0;   // entries of the set ahead of the one sought
      const int ch = (V + FWD_THREADS - 1) / FWD_THREADS;
      const int i0 = tid * ch, i1 = min(V, i0 + ch);
      unsigned int mine = 0;
      for (int i = i0; i < i1; ++i) {
        const float zi = __fdiv_rn(lg[i], temp);
        mine += (nuc_bucket(zi, z0, scale) == b0 && float_key(zi) == klo) ? 1u : 0u;
      }
      st.chunk_cnt[tid] = mine;
      __syncthreads();
      unsigned long long before = 0;
      for (int k = 0; k < tid; ++k) before += st.chunk_cnt[k];
      if (jl >= before && jl < before + mine) {
        unsigned long long seen = before;
        for (int i = i0; i < i1; ++i) {
          const float zi = __fdiv_rn(lg[i], temp);
          if (nuc_bucket(zi, z0, scale) == b0 && float_key(zi) == klo) {
            if (seen == jl) { st.res_idx = i; st.res_cum = st.acc + (jl + 1) * q0; st.done = 1; break; }
            ++seen;
          }
        }
      }
      __syncthreads();
      if (tid == 0 && !st.done) { st.res_idx = 0; st.res_cum = st.acc; st.done = 1; }   // cannot happen for t < total
      __syncthreads();
      return;
    }
    // ---- one more level: 256 buckets over the key interval [klo, khi] ----
    st.m[tid] = 0ull;
    st.cn[tid] = 0u;
    __syncthreads();
    const unsigned long long W = (unsigned long long)khi - klo + 1ull;
    sample_for_listed(lg, V, cl, s_list, n_list, [&](float v, int) {
      const float z = __fdiv_rn(v, temp);
      const unsigned int key = float_key(z);
      if (nuc_bucket(z, z0, scale) == b0 && key >= klo && key <= khi) {
        const int b = (int)((((unsigned long long)(key - klo)) << 8) / W);
        atomicAdd(&st.m[b], nucleus_weight(z, z0));
        atomicAdd(&st.cn[b], 1u);
      }
    });
    __syncthreads();
    if (tid < 32) {
      unsigned long long acc;
      const int b = nuc_pick_bucket(st.m, st.acc, t, acc);
      if (tid == 0) {
        st.acc = acc;
        st.cnt = st.cn[b];
        // keys of bucket b: (key - klo) * 256 / W == b
        st.klo = klo + (unsigned int)(((unsigned long long)b * W + 255ull) >> 8);
        st.khi = klo + (unsigned int)((((unsigned long long)(b + 1) * W + 255ull) >> 8) - 1ull);
      }
    }
    __syncthreads();
  }
  if (tid == 0 && !st.done) { st.res_idx = 0; st.res_cum = st.acc; st.done = 1; }
  __syncthreads();
}

// Shared-memory layout of sample_row (floats).
constexpr int SAMPLE_CAND = 1024;
constexpr int SAMPLE_SMEM_FLOATS = 256 + 4 * SAMPLE_CAND + SAMPLE_CHUNKS;
static_assert(sizeof(NucLimbs) <= 4 * SAMPLE_CAND * sizeof(float), "the weight limbs use the candidates' place");

// Top-p over the whole row (no top-k cut): z = logit / T, weights and order as described above.  `nm`, `nc`: the row's
// bucket weights and counts, or null (then this CTA adds them up).  The result is returned by thread 0 (others: -1).
static __device__ __noinline__ int sample_row_nucleus(const float* lg, int V, int cl, const float* s_cmax, float lmax, float temp,
                                                      float top_p, unsigned long long ticket, int gen_index,
                                                      unsigned long long seed, float* smem, const unsigned long long* nm,
                                                      const unsigned int* nc) {
  __shared__ NucShared st;
  __shared__ unsigned long long s_t;
  __shared__ bool s_none;
  const int tid = threadIdx.x;
  float* s_cz = smem + 256;
  int* s_ci = reinterpret_cast<int*>(smem + 256 + SAMPLE_CAND);
  float* s_sz = smem + 256 + 2 * SAMPLE_CAND;
  int* s_si = reinterpret_cast<int*>(smem + 256 + 3 * SAMPLE_CAND);
  __shared__ float s_red[FWD_THREADS / 32];
  const float z0 = __fdiv_rn(lmax, temp);
  const float scale = nuc_scale(lg, V, temp, z0, s_red);
  __syncthreads();
  if (nm != nullptr) {
    st.m0[tid] = __ldcg(nm + tid);
    st.c0[tid] = __ldcg(nc + tid);
  } else {
    unsigned long long m;
    unsigned int n;
    nuc_bucket_sums(*reinterpret_cast<NucLimbs*>(s_cz), lg, V, 0, V, temp, z0, scale, m, n);
    st.m0[tid] = m;
    st.c0[tid] = n;
  }
  __syncthreads();
  if (tid < 32) {
    unsigned long long Q = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) Q += st.m0[tid * 8 + k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) Q += __shfl_xor_sync(0xffffffffu, Q, o);
    if (tid == 0) {
      s_none = Q == 0ull;
      s_t = nucleus_need(nucleus_p24(top_p), Q) - 1ull;   // first entry with cum >= need  <=>  cum > need - 1
    }
  }
  __syncthreads();
  if (s_none) {   // the largest z is infinite or there is no number in the row: no distance to it has a weight
    const int pick = sample_first_max(lg, V, cl, s_cmax, z0, [&](float v) { return __fdiv_rn(v, temp); });
    return tid == 0 ? pick : -1;
  }
  nucleus_locate(st, lg, V, cl, s_cmax, temp, z0, scale, s_t, s_cz, s_ci, s_sz, s_si);   // end of the nucleus: its weight is res_cum
  if (tid == 0) {
    const uint32_t x = philox4x32_10_word0((uint32_t)ticket, (uint32_t)(ticket >> 32), (uint32_t)gen_index, 0u,
                                           (uint32_t)seed, (uint32_t)(seed >> 32));
    s_t = nucleus_target((unsigned long long)(x >> 8), st.res_cum);
  }
  __syncthreads();
  nucleus_locate(st, lg, V, cl, s_cmax, temp, z0, scale, s_t, s_cz, s_ci, s_sz, s_si);
  const int result = tid == 0 ? st.res_idx : -1;
  __syncthreads();
  return result;
}

// One CTA per sampled row.  Greedy: lowest index among the maxima.  Top-k: z = logit / T
// (IEEE fp32 divide); the k largest by (z desc, index asc); weights exp(z - z0) and the inverse-CDF walk run in fp64.
// `cmax`: the row's chunk maxima in memory, or null (then this CTA takes them); `nm`, `nc` as above.
// The result is returned by thread 0 (other threads return -1).
static __device__ int sample_row(const float* lg, int V, int top_k, float temp, float top_p, unsigned long long ticket,
                                 int gen_index, unsigned long long seed, float* smem, const float* cmax,
                                 const unsigned long long* nm, const unsigned int* nc_) {
  constexpr int CAND_MAX = SAMPLE_CAND;
  const int tid = threadIdx.x;
  uint32_t* s_hist = reinterpret_cast<uint32_t*>(smem);             // [256]
  float* s_cz = smem + 256;                                          // [CAND_MAX]
  int* s_ci = reinterpret_cast<int*>(smem + 256 + CAND_MAX);         // [CAND_MAX]
  float* s_cmax = smem + 256 + 4 * CAND_MAX;                         // [SAMPLE_CHUNKS]
  __shared__ float s_red[FWD_THREADS / 32];
  __shared__ unsigned long long s_prefix, s_mask;
  __shared__ int s_remaining, s_ncand, s_nlist;
  __shared__ float s_tz[MAX_TOPK];
  __shared__ int s_ti[MAX_TOPK];
  __shared__ double s_tw[MAX_TOPK];
  int result = -1;
  const bool nucleus = top_p > 0.f && top_p < 1.f;   // outside (0, 1): no nucleus cut
  const int cl = sample_chunk_len(V), nch = (V + cl - 1) / cl;
  __syncthreads();
  if (cmax != nullptr) {
    for (int i = tid; i < nch; i += FWD_THREADS) s_cmax[i] = __ldcg(cmax + i);
  } else if (cl <= SAMPLE_WARP_SPAN) {
    for (int i0 = (tid >> 5) * SAMPLE_WARP_SPAN; i0 < V; i0 += (FWD_THREADS / 32) * SAMPLE_WARP_SPAN)
      sample_chunk_maxima(lg, V, cl, i0, s_cmax);
  } else {
    for (int ch = tid >> 5; ch < nch; ch += FWD_THREADS / 32) {
      float m = -INFINITY;
      for (int i = ch * cl + (tid & 31); i < min(V, (ch + 1) * cl); i += 32) m = fmaxf(m, lg[i]);
      m = warp_max(m);
      if ((tid & 31) == 0) s_cmax[ch] = m;
    }
  }
  if (tid == 0) s_ncand = 0;
  __syncthreads();
  // maximum over the chunks of this thread (tid, tid + 256, ...)
  float lmax = -INFINITY;
  for (int i = tid; i < nch; i += FWD_THREADS) lmax = fmaxf(lmax, s_cmax[i]);
  if (top_k <= 0) {
    const float gmax = block_max(lmax, s_red);
    if (nucleus) return sample_row_nucleus(lg, V, cl, s_cmax, gmax, temp, top_p, ticket, gen_index, seed, smem, nm, nc_);
    const int pick = sample_first_max(lg, V, cl, s_cmax, gmax, [](float v) { return v; });
    return tid == 0 ? pick : -1;
  }
  const int k = min(top_k, V);
  // Fast path.  The k-th largest of the 256 per-thread maxima, tau, is a lower bound of the k-th largest z of the row
  // (k threads hold an element >= tau each), so {z >= tau} contains the top k and is usually a few dozen elements.
  // z = logit / T is monotone in the logit, so the maxima can be taken on logits and divided once.
  {
    float* s_tm = smem;   // [FWD_THREADS] thread maxima of z (aliases the histogram, not live yet)
    const float zmax = __fdiv_rn(lmax, temp);
    s_tm[tid] = zmax;
    __syncthreads();
    int rank = 0;
#pragma unroll 8
    for (int j4 = 0; j4 < FWD_THREADS / 4; ++j4) {
      const float4 z4 = *reinterpret_cast<const float4*>(s_tm + 4 * j4);
      rank += (z4.x > zmax) || (z4.x == zmax && 4 * j4 < tid);
      rank += (z4.y > zmax) || (z4.y == zmax && 4 * j4 + 1 < tid);
      rank += (z4.z > zmax) || (z4.z == zmax && 4 * j4 + 2 < tid);
      rank += (z4.w > zmax) || (z4.w == zmax && 4 * j4 + 3 < tid);
    }
    if (rank == k - 1) s_red[0] = zmax;
    __syncthreads();
    const float tau = s_red[0];
    if (tau > -INFINITY) {
      // cheap conservative test on the logit first, the exact one on z for the survivors
      const float x = tau * temp;
      const float thr_l = x - fabsf(x) * 9.5367431640625e-7f - 1e-30f;
      int* s_list = reinterpret_cast<int*>(smem + 256 + 2 * CAND_MAX);
      const int n_list = sample_list_chunks(s_cmax, nch, s_list, &s_nlist, [&](float m) { return m >= thr_l; });
      sample_for_listed(lg, V, cl, s_list, n_list, [&](float v, int i) {
        if (v >= thr_l) {
          const float z = __fdiv_rn(v, temp);
          if (z >= tau) {
            const int p = atomicAdd(&s_ncand, 1);
            if (p < CAND_MAX) { s_cz[p] = z; s_ci[p] = i; }
          }
        }
      });
    }
    __syncthreads();
  }
  const bool fast_ok = s_ncand >= k && s_ncand <= CAND_MAX;
  __syncthreads();
  if (!fast_ok) {
  // Fallback (huge plateaus of equal values, or fewer than k finite thread maxima):
  // radix select over the composite key (z key, ~index): unique keys, so ties in z
  // break towards the lower index and the k-th key is exact.  Refine 8 bits at a time
  // until the set {key >= prefix} (>= k elements by construction) fits the sort buffer.
  if (tid == 0) { s_prefix = 0; s_mask = 0; s_remaining = k; }
  __syncthreads();
  for (int shift = 56; shift >= 0; shift -= 8) {
    s_hist[tid] = 0;   // FWD_THREADS == 256 bins
    __syncthreads();
    const unsigned long long prefix = s_prefix, mask = s_mask;
    for (int i = tid; i < V; i += FWD_THREADS) {
      const unsigned long long key =
          ((unsigned long long)float_key(__fdiv_rn(lg[i], temp)) << 32) | (uint32_t)(~(uint32_t)i);
      if ((key & mask) == prefix) atomicAdd(&s_hist[(unsigned)(key >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (tid == 0) {
      const int need = s_remaining;   // how many are still needed from inside the current prefix
      int bin = 255;
      uint32_t above = 0;
      for (; bin > 0; --bin) {
        if (above + s_hist[bin] >= (uint32_t)need) break;
        above += s_hist[bin];
      }
      s_remaining = need - (int)above;
      s_prefix = prefix | ((unsigned long long)bin << shift);
      s_mask = mask | (255ull << shift);
      // keys >= new prefix: those in strictly higher bins at every level so far, plus this bin
      s_ncand = (k - s_remaining) + (int)s_hist[bin];
    }
    __syncthreads();
    if (s_ncand <= CAND_MAX) break;
  }
  const unsigned long long thr = s_prefix;
  __syncthreads();
  if (tid == 0) s_ncand = 0;
  __syncthreads();
  for (int i = tid; i < V; i += FWD_THREADS) {
    const float z = __fdiv_rn(lg[i], temp);
    const unsigned long long key = ((unsigned long long)float_key(z) << 32) | (uint32_t)(~(uint32_t)i);
    if (key >= thr) {
      const int p = atomicAdd(&s_ncand, 1);
      if (p < CAND_MAX) { s_cz[p] = z; s_ci[p] = i; }
    }
  }
  __syncthreads();
  }  // fallback
  const int nc = min(s_ncand, CAND_MAX);
  // rank every candidate by (z desc, index asc); the k best land at their rank
  for (int a = tid; a < nc; a += FWD_THREADS) {
    const float za = s_cz[a];
    const int ia = s_ci[a];
    const uint32_t ka = float_key(za + 0.f);   // keys, so that NaN has a place too: every rank below nc is taken once
    int rank = 0;
    for (int j = 0; j < nc; ++j) {
      const uint32_t kj = float_key(s_cz[j] + 0.f);   // (-0 counts as 0)
      rank += (kj > ka) || (kj == ka && s_ci[j] < ia);
    }
    if (rank < k) { s_tz[rank] = za; s_ti[rank] = ia; }
  }
  __syncthreads();
  // the k weights by k threads, then one thread adds them in order
  unsigned long long* s_tq = reinterpret_cast<unsigned long long*>(s_tw);
  if (tid < min(k, nc)) {
    if (nucleus) s_tq[tid] = nucleus_weight(s_tz[tid], s_tz[0]);
    else s_tw[tid] = exp((double)s_tz[tid] - (double)s_tz[0]);
  }
  __syncthreads();
  if (tid == 0) {
    const uint32_t x = philox4x32_10_word0((uint32_t)ticket, (uint32_t)(ticket >> 32), (uint32_t)gen_index, 0u,
                                           (uint32_t)seed, (uint32_t)(seed >> 32));
    const int kk = min(k, nc);
    if (nucleus) {
      // nucleus inside the k candidates (already in the order), integer weights
      unsigned long long Q = 0;
      for (int j = 0; j < kk; ++j) Q += s_tq[j];
      const unsigned long long need = nucleus_need(nucleus_p24(top_p), Q);
      unsigned long long M = 0;
      int m = 0;
      for (; m < kk; ++m) {
        M += s_tq[m];
        if (M >= need) { ++m; break; }
      }
      const unsigned long long target = nucleus_target((unsigned long long)(x >> 8), M);
      unsigned long long cum = 0;
      int pick = s_ti[m - 1];
      for (int j = 0; j < m; ++j) {
        cum += s_tq[j];
        if (cum > target) { pick = s_ti[j]; break; }
      }
      result = pick;
    } else {
      const double u = (double)(x >> 8) * (1.0 / 16777216.0);
      double total = 0.0;
      for (int j = 0; j < kk; ++j) total += s_tw[j];
      const double target = u * total;
      double accum = 0.0;
      int pick = s_ti[kk - 1];
      for (int j = 0; j < kk; ++j) {
        accum += s_tw[j];
        if (accum > target) { pick = s_ti[j]; break; }
      }
      result = pick;
    }
  }
  __syncthreads();
  return result;
}

static __device__ __noinline__ void phase_sample(const DevCtx& c, float* smem) {
  const int R = c.ss->cur_rows;
  const int V = c.V;
  const int tid = threadIdx.x;
  const bool split = sample_split_rows(V);
  const unsigned long long rows_before = c.ss->sample_rows_total;
  for (int r = blockIdx.x; r < R; r += gridDim.x) {
    const float* lg = c.logits + (size_t)r * V;
    const int item = c.row_item[r];
    const int b = c.it_bslot[item];
    if (c.logits_capture != nullptr && (long long)(rows_before + r) < c.capture_rows) {
      float* dst = c.logits_capture + (size_t)(rows_before + r) * V;
      for (int i = tid; i < V; i += FWD_THREADS) dst[i] = lg[i];
    }
    const int tok = sample_row(lg, V, min(c.b_topk[b], MAX_TOPK), c.b_temp[b], c.b_topp[b], (unsigned long long)c.b_ticket[b],
                               c.b_generated[b], c.b_seed[b], smem, split ? c.cmax + (size_t)r * SAMPLE_CHUNKS : nullptr,
                               split ? c.nuc_m + (size_t)r * 256 : nullptr, split ? c.nuc_c + (size_t)r * 256 : nullptr);
    if (tid == 0) c.row_sampled[r] = tok;
  }
}

}  // namespace blink
