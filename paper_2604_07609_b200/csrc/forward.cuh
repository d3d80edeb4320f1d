// Data-parallel phases of one serving step (every CTA of the grid takes part):
// embedding + RMSNorm, CUDA-core reference GEMM, RoPE + paged-KV write, paged
// attention, SwiGLU gate, final norm, sampling.  Each phase is a __device__
// function that distributes its work over blockIdx.x / gridDim.x, so the same
// code runs inside the persistent loop (phases separated by grid barriers) and
// as host-launched kernels (stepped mode).
//
// Paper: the model step is the "inference engine" of Section 4.2 (paged KV cache,
// context attention, fused MLP, sampling captured inside the step); Section 6.1
// lists the engine features.  The math is the standard pre-norm decoder.
#pragma once
#include "control.cuh"
#include "dev_ctx.cuh"

namespace blink {

constexpr int FWD_THREADS = 256;

template <typename T> struct OpType;
template <> struct OpType<float> {
  static __device__ __forceinline__ float to_f(float v) { return v; }
  static __device__ __forceinline__ float from_f(float v) { return v; }
};
template <> struct OpType<__nv_bfloat16> {
  static __device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }
  static __device__ __forceinline__ __nv_bfloat16 from_f(float v) { return __float2bfloat16_rn(v); }
};

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
// Sums of NV values over the 32 lanes by halving exchange: lane l ends with the sum of value (l * NV) / 32.
template <int NV>
__device__ __forceinline__ float warp_sum_many(float (&v)[NV]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int n = NV, o = 16; o > 0; o >>= 1) {
    if (n > 1) {
      n >>= 1;
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int i = 0; i < NV / 2; ++i) {
        if (i < n) {
          const float send = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
          v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      }
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    }
  }
  return v[0];
}
__device__ __forceinline__ float block_sum(float v, float* s_red /*[8]*/) {
  v = warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
  __syncthreads();
  float t = 0.f;
#pragma unroll
  for (int i = 0; i < FWD_THREADS / 32; ++i) t += s_red[i];
  return t;
}

template <typename WT>
__device__ __forceinline__ const WT* wptr(const DevCtx& c, int id) {
  return reinterpret_cast<const WT*>(c.w_base + c.w_off[id]);
}
__device__ __forceinline__ const float* wptr_f(const DevCtx& c, int id) {
  return reinterpret_cast<const float*>(c.w_base + c.w_off[id]);
}

// zero n_floats (a multiple of 4) floats starting at p, grid-strided
__device__ __forceinline__ void zero_floats(float* p, long long n_floats) {
  float4* q = reinterpret_cast<float4*>(p);
  const long long n4 = n_floats >> 2;
  for (long long i = (long long)blockIdx.x * FWD_THREADS + threadIdx.x; i < n4; i += (long long)gridDim.x * FWD_THREADS)
    q[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// store four consecutive values in the operand type
template <typename WT>
__device__ __forceinline__ void store4(WT* p, float a, float b, float c, float d);
template <>
__device__ __forceinline__ void store4<float>(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
template <>
__device__ __forceinline__ void store4<__nv_bfloat16>(__nv_bfloat16* p, float a, float b, float c, float d) {
  const __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
  uint2 v;
  v.x = *reinterpret_cast<const uint32_t*>(&lo);
  v.y = *reinterpret_cast<const uint32_t*>(&hi);
  *reinterpret_cast<uint2*>(p) = v;
}
template <typename WT>
__device__ __forceinline__ float4 load4(const WT* p);
template <>
__device__ __forceinline__ float4 load4<float>(const float* p) { return *reinterpret_cast<const float4*>(p); }
template <>
__device__ __forceinline__ float4 load4<__nv_bfloat16>(const __nv_bfloat16* p) {
  const uint2 v = *reinterpret_cast<const uint2*>(p);
  const __nv_bfloat162 lo = *reinterpret_cast<const __nv_bfloat162*>(&v.x), hi = *reinterpret_cast<const __nv_bfloat162*>(&v.y);
  const float2 a = __bfloat1622float2(lo), b = __bfloat1622float2(hi);
  return make_float4(a.x, a.y, b.x, b.y);
}

// One CTA normalises one row: n = x / sqrt(mean(x^2) + eps) * g.  Every thread keeps its part of
// the row (16-byte vectors, up to NORM_MAXV of them: d <= 8192) in registers between the sum and
// the scaling, so the row is read once.  `src_embed` non-null: the row is first gathered from
// the embedding table into the residual stream.
constexpr int NORM_MAXV = 8;
template <typename WT>
__device__ __forceinline__ void norm_row_cta(const DevCtx& c, float* hrow, const WT* src_embed, const float* g, WT* orow,
                                             float* s_red, const float* wr = nullptr, int row_index = 0) {
  const int d = c.d;
  float4 v[NORM_MAXV];
  float ss = 0.f;
#pragma unroll
  for (int k = 0; k < NORM_MAXV; ++k) {
    const int i = (k * FWD_THREADS + threadIdx.x) * 4;
    if (i < d) {
      if (src_embed != nullptr) {
        v[k] = load4<WT>(src_embed + i);
        *reinterpret_cast<float4*>(hrow + i) = v[k];
      } else {
        v[k] = *reinterpret_cast<const float4*>(hrow + i);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < NORM_MAXV; ++k) {
    const int i = (k * FWD_THREADS + threadIdx.x) * 4;
    if (i < d) {  // fixed order
      ss = fmaf(v[k].x, v[k].x, ss); ss = fmaf(v[k].y, v[k].y, ss); ss = fmaf(v[k].z, v[k].z, ss); ss = fmaf(v[k].w, v[k].w, ss);
    }
  }
  ss = block_sum(ss, s_red);
  const float inv = rsqrtf(__fdividef(ss, (float)d) + c.rms_eps);
#pragma unroll
  for (int k = 0; k < NORM_MAXV; ++k) {
    const int i = (k * FWD_THREADS + threadIdx.x) * 4;
    if (i < d) {
      const float4 gg = *reinterpret_cast<const float4*>(g + i);
      v[k] = make_float4(v[k].x * inv * gg.x, v[k].y * inv * gg.y, v[k].z * inv * gg.z, v[k].w * inv * gg.w);
      store4<WT>(orow + i, v[k].x, v[k].y, v[k].z, v[k].w);
    }
  }
  if (wr != nullptr) {
    // Router of the routed-expert FFN on the normed row in fp32 (not its 16-bit copy): logits over
    // the E experts, top-k by (logit desc, expert id asc), weights = softmax restricted to the chosen.
    // Eight experts at a time, their weights for a vector of the row on the way together (expert by expert, each with a
    // reduction of its own, a row took 10 us).
    __shared__ float s_rl[FWD_THREADS / 32][MAX_EXPERTS];
    const int E = c.E;
    for (int e0 = 0; e0 < E; e0 += 8) {
      float p[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) p[j] = 0.f;
#pragma unroll
      for (int k = 0; k < NORM_MAXV; ++k) {
        const int i = (k * FWD_THREADS + threadIdx.x) * 4;
        if (i < d) {
          float4 w4[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) w4[j] = *reinterpret_cast<const float4*>(wr + (size_t)min(e0 + j, E - 1) * d + i);   // past the end: the last again
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            p[j] = fmaf(v[k].x, w4[j].x, p[j]); p[j] = fmaf(v[k].y, w4[j].y, p[j]); p[j] = fmaf(v[k].z, w4[j].z, p[j]); p[j] = fmaf(v[k].w, w4[j].w, p[j]);
          }
        }
      }
      const float t = warp_sum_many<8>(p);   // lanes 4 j .. 4 j + 3 hold expert e0 + j
      const int e = e0 + ((threadIdx.x & 31) >> 2);
      if ((threadIdx.x & 3) == 0 && e < E) s_rl[threadIdx.x >> 5][e] = t;
    }
    __syncthreads();
    if (threadIdx.x < 32) {   // a lane per expert
      const int lane = threadIdx.x;
      float lg = 0.f;
      if (lane < E)
        for (int w = 0; w < FWD_THREADS / 32; ++w) lg += s_rl[w][lane];
      bool open = lane < E;   // not chosen yet
      float den = 0.f, top = 0.f, mine = 0.f;
      int place = -1;
      for (int j = 0; j < c.topE; ++j) {
        // The first open expert, or one with a larger logit.  NaN is larger than nothing and nothing is larger than NaN: it
        // stays out of the exchange, where it would keep lanes from hearing of one another, unless it is the first.
        const int first = __ffs(__ballot_sync(0xffffffffu, open)) - 1;
        const float lg_first = __shfl_sync(0xffffffffu, lg, first);
        float bv = open && lg == lg ? lg : -INFINITY;
        int bi = open && lg == lg ? lane : 32;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
          const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
          if (oi < 32 && (bi == 32 || ov > bv || (ov == bv && oi < bi))) { bv = ov; bi = oi; }   // ties keep the lower id
        }
        if (lg_first != lg_first) { bv = lg_first; bi = first; }
        if (j == 0) top = bv;
        const float ex = expf(bv - top);
        den += ex;
        if (lane == bi) { open = false; place = j; mine = ex; }
      }
      if (place >= 0) {
        c.moe_sel[(size_t)row_index * c.topE + place] = lane;
        c.moe_wt[(size_t)row_index * c.topE + place] = mine / den;
      }
    }
    __syncthreads();
  }
}

// Two rows of a CTA at a time, one by each half of its threads (NV = d / 512 16-byte vectors per thread, all of a row's
// loads in flight at once, the gains held in registers).  With one row per CTA in turn a 500-row step had four rounds
// of load latency and reduction (9 us at d = 4096 although the next row was prefetched); this form has two.
template <typename WT, int NV>
static __device__ __noinline__ void norm_rows_halves(const float* __restrict__ h, const float* __restrict__ g, WT* __restrict__ out, int T,
                                                     float eps) {
  constexpr int d = NV * 512;
  __shared__ float s_half[2][2][4];
  const int half = threadIdx.x >> 7, tid = threadIdx.x & 127;
  // rows are dealt to the first halves of all CTAs, then to the second halves
  int t = half * gridDim.x + blockIdx.x;
  if (t >= T) return;
  float4 gg[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) gg[k] = __ldg(reinterpret_cast<const float4*>(g + (k * 128 + tid) * 4));
  int buf = 0;
#pragma unroll 1
  for (; t < T; t += 2 * gridDim.x) {
    const float* src = h + (size_t)t * d + tid * 4;
    float4 v[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = __ldcg(reinterpret_cast<const float4*>(src + k * 512));
    float ss = 0.f;
#pragma unroll
    for (int k = 0; k < NV; ++k) {   // fixed order
      ss = fmaf(v[k].x, v[k].x, ss); ss = fmaf(v[k].y, v[k].y, ss); ss = fmaf(v[k].z, v[k].z, ss); ss = fmaf(v[k].w, v[k].w, ss);
    }
    ss = warp_sum(ss);
    if ((tid & 31) == 0) s_half[half][buf][tid >> 5] = ss;
    asm volatile("bar.sync %0, 128;" ::"r"(half + 1) : "memory");   // two buffers: one barrier per row
    ss = (s_half[half][buf][0] + s_half[half][buf][1]) + (s_half[half][buf][2] + s_half[half][buf][3]);
    buf ^= 1;
    const float inv = rsqrtf(ss * (1.0f / (float)d) + eps);
    WT* orow = out + (size_t)t * d + tid * 4;
#pragma unroll
    for (int k = 0; k < NV; ++k)
      store4<WT>(orow + k * 512, v[k].x * inv * gg[k].x, v[k].y * inv * gg[k].y, v[k].z * inv * gg[k].z, v[k].w * inv * gg[k].w);
  }
}

// ---- RMSNorm of the residual rows into the operand buffer; layer 0 gathers the
// embedding first.
template <typename WT>
static __device__ __noinline__ void phase_norm(const DevCtx& c, int layer, int which /*0: norm1, 1: norm2*/) {
  __shared__ float s_red[FWD_THREADS / 32];
  const int T = c.ss->cur_T;
  const float* g = wptr_f(c, which == 0 ? 6 : 7) + (size_t)layer * c.d;
  WT* out = reinterpret_cast<WT*>(c.xn);
  // fused path: both sum-of-squares buffers start a step at zero (the last layer's leftovers)
  if (c.fused_norm && which == 0 && layer == 0)
    for (int i = blockIdx.x * FWD_THREADS + threadIdx.x; i < c.Tmax; i += gridDim.x * FWD_THREADS) {
      c.rowss_a[i] = 0.f;
      c.rowss_b[i] = 0.f;
    }
  const float* wr = (which == 1 && c.E > 0) ? wptr_f(c, 5) + (size_t)layer * c.E * c.d : nullptr;
  if (wr == nullptr && !(which == 0 && layer == 0) && (c.d == 4096 || c.d == 2048)) {
    if (c.d == 4096) norm_rows_halves<WT, 8>(c.h, g, out, T, c.rms_eps);
    else norm_rows_halves<WT, 4>(c.h, g, out, T, c.rms_eps);
    return;
  }
  for (int t = blockIdx.x; t < T; t += gridDim.x) {
    const WT* e = (which == 0 && layer == 0) ? wptr<WT>(c, 0) + (size_t)c.tok_id[t] * c.d : nullptr;
    norm_row_cta<WT>(c, c.h + (size_t)t * c.d, e, g, out + (size_t)t * c.d, s_red, wr, t);
  }
}

// The LM head gives every CTA whole weight tiles when there are at least as many tiles as CTAs: no
// partial sums, so the logits need no clearing.
__device__ __forceinline__ bool lm_head_whole_tiles(const DevCtx& c) { return (c.V + 127) / 128 >= (int)gridDim.x; }

// Fused path: the sum of squares of every residual row is already known (added up by the epilogue of
// the GEMM that completed the row), so the norm is element-wise: n = x * rsqrt(ss / d + eps) * g.
// `rows` null: rows 0 .. R-1 of h go to rows 0 .. R-1 of out; else row r of out comes from row rows[r].
template <typename WT>
__device__ __noinline__ void norm_apply_rows(const float* __restrict__ h, const float* __restrict__ rowss,
                                             const float* __restrict__ g, WT* __restrict__ out, const int32_t* rows, int R,
                                             int d, float eps) {
  constexpr int U = 4;   // items whose loads are in flight before the first store (one CTA per SM: latency-bound otherwise)
  const int d4 = d >> 2;
  const int total = R * d4;   // < 2^31
  const float inv_d = __fdividef(1.0f, (float)d);
  const int stride = gridDim.x * FWD_THREADS;
  for (int base = blockIdx.x * FWD_THREADS + threadIdx.x; base < total; base += U * stride) {
    float4 v[U], gg[U];
    float ss[U];
    int r[U], j[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int idx = min(base + k * stride, total - 1);   // clamped: the tail loads a valid item twice
      r[k] = idx / d4;
      j[k] = (idx - r[k] * d4) * 4;
      const int t = rows != nullptr ? rows[r[k]] : r[k];
      v[k] = __ldcg(reinterpret_cast<const float4*>(h + (size_t)t * d + j[k]));
      ss[k] = __ldcg(rowss + t);
      gg[k] = *reinterpret_cast<const float4*>(g + j[k]);
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
      if (base + k * stride < total) {
        const float inv = rsqrtf(ss[k] * inv_d + eps);
        store4<WT>(out + (size_t)r[k] * d + j[k], v[k].x * inv * gg[k].x, v[k].y * inv * gg[k].y, v[k].z * inv * gg[k].z,
                   v[k].w * inv * gg[k].w);
      }
    }
  }
}

// Norm phases of the fused path for layers whose input rows are complete with their sums of squares:
// which 0 = first norm of layer > 0 (reads rowss_b, clears rowss_a), 1 = second norm (reads rowss_a,
// clears rowss_b).  The cleared buffer is the one the next GEMM epilogue adds into.
template <typename WT>
static __device__ __noinline__ void phase_norm_apply(const DevCtx& c, int layer, int which, int T) {
  const float* g = wptr_f(c, which == 0 ? 6 : 7) + (size_t)layer * c.d;
  float* clear = which == 0 ? c.rowss_a : c.rowss_b;
  for (int i = blockIdx.x * FWD_THREADS + threadIdx.x; i < T; i += gridDim.x * FWD_THREADS) clear[i] = 0.f;
  norm_apply_rows<WT>(c.h, which == 0 ? c.rowss_b : c.rowss_a, g, reinterpret_cast<WT*>(c.xn), nullptr, T, c.d, c.rms_eps);
}

// Final norm of the sampled rows only (the LM head runs on those rows).
template <typename WT>
static __device__ __noinline__ void phase_final_norm(const DevCtx& c) {
  __shared__ float s_red[FWD_THREADS / 32];
  const int R = c.ss->cur_rows;
  const float* g = wptr_f(c, 8);
  WT* out = reinterpret_cast<WT*>(c.xs);
  if (c.gemm_tc && !lm_head_whole_tiles(c)) zero_floats(c.logits, (long long)R * c.V);
  if (c.fused_norm) {
    norm_apply_rows<WT>(c.h, c.rowss_b, g, out, c.row_tok, R, c.d, c.rms_eps);
    return;
  }
  for (int r = blockIdx.x; r < R; r += gridDim.x)
    norm_row_cta<WT>(c, c.h + (size_t)c.row_tok[r] * c.d, nullptr, g, out + (size_t)r * c.d, s_red);
}

// ---- dense contractions ------------------------------------------------------------------
enum GemmFix : int {
  FIX_NONE = 0,
  FIX_ROPE_KV,  // QKV: RoPE on q and k, q -> 16-bit attention operand, k and v -> paged pool; the tile is cleared
  FIX_SILU,     // gate/up: act = silu(gate) * up in the operand type; both tiles are cleared
  FIX_SUMSQ,    // O and down: add the tile's share of sum(x^2) of every residual row
};
struct GemmArgs {
  const void* x;   // [M][K] operand type
  const void* w;   // [N][K] operand type
  float* out;      // [M][ldo]
  int M, N, K, ldo;
  int accumulate;  // 1: out += result (residual), 0: out = result
  // routed experts: x rows start at row x_row0 of the activation buffer, the weights at row w_row0 of
  // the stacked weight tensor; with row_map the result row t goes to out row row_map[t], scaled by
  // row_scale[t], always added (several experts contribute to one token)
  int x_row0 = 0;
  long long w_row0 = 0;
  const int32_t* row_map = nullptr;
  const float* row_scale = nullptr;
  // tensor-core path: element-wise work that consumes the finished output tiles of this GEMM (run by
  // the CTA that delivers a tile's last partial sum, see tc_finish_tiles)
  int fix = 0;               // FIX_*
  void* fix_out = nullptr;   // FIX_SILU: the activation rows (operand type) matching `out`
  float* fix_rowss = nullptr;// FIX_SUMSQ: per-row sums of squares to add to
};

// One warp: GR token rows x NC output features, the 32 lanes side by side along K (four elements each), so that all
// loads of 256 elements of K are in flight at once.  The reference shapes are small (a few dozen rows, K of 256 to
// 1024): with 64 x 64 tiles and 16 elements of K per step only 4 to 64 CTAs had work and every step waited for
// its own loads (27 us for K = 256, 98 us for K = 1024 at 8 rows; now 3 and 5).
constexpr int SIMT_GR = 8;
template <typename WT, int NC>
__device__ __forceinline__ void gemm_simt_tasks(const GemmArgs& a) {
  const WT* X = reinterpret_cast<const WT*>(a.x);
  const WT* W = reinterpret_cast<const WT*>(a.w);
  const int lane = threadIdx.x & 31;
  const int groups_n = (a.N + NC - 1) / NC, groups_m = (a.M + SIMT_GR - 1) / SIMT_GR;
  const int nw = gridDim.x * (FWD_THREADS / 32);
  for (int task = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; task < groups_m * groups_n; task += nw) {
    const int gm = task / groups_n, gn = task - gm * groups_n;
    const int m0 = gm * SIMT_GR, n0 = gn * NC;
    float acc[SIMT_GR * NC];
#pragma unroll
    for (int i = 0; i < SIMT_GR * NC; ++i) acc[i] = 0.f;
#pragma unroll 2
    for (int k = lane * 4; k < a.K; k += 128) {
      float4 w[NC], x[SIMT_GR];
#pragma unroll
      for (int j = 0; j < NC; ++j) w[j] = load4<WT>(W + (size_t)min(n0 + j, a.N - 1) * a.K + k);   // clamped: rows past the end repeat
#pragma unroll
      for (int i = 0; i < SIMT_GR; ++i) x[i] = load4<WT>(X + (size_t)min(m0 + i, a.M - 1) * a.K + k);
#pragma unroll
      for (int i = 0; i < SIMT_GR; ++i)
#pragma unroll
        for (int j = 0; j < NC; ++j) {
          float& s = acc[i * NC + j];
          s = fmaf(x[i].x, w[j].x, s); s = fmaf(x[i].y, w[j].y, s); s = fmaf(x[i].z, w[j].z, s); s = fmaf(x[i].w, w[j].w, s);
        }
    }
    const float v = warp_sum_many<SIMT_GR * NC>(acc);
    constexpr int LPV = 32 / (SIMT_GR * NC);   // lanes that hold the same sum
    const int idx = lane / LPV, m = m0 + idx / NC, n = n0 + idx % NC;
    if (lane % LPV == 0 && m < a.M && n < a.N) {
      if (a.row_map != nullptr) {
        atomicAdd(a.out + (size_t)a.row_map[m] * a.ldo + n, a.row_scale[m] * v);
      } else {
        float* o = a.out + (size_t)m * a.ldo + n;
        *o = a.accumulate ? (*o + v) : v;
      }
    }
  }
}
// CUDA-core GEMM: out[t][n] (+)= sum_k x[t][k] * w[n][k], fp32 accumulate, deterministic (no split over CTAs).  Four
// features per warp load 12 vectors for 128 multiplications; fewer when the tasks would not fill the warps of the grid.
template <typename WT>
static __device__ __noinline__ void phase_gemm_simt(const GemmArgs& a) {
  const long long rows = (a.M + SIMT_GR - 1) / SIMT_GR, warps = (long long)gridDim.x * (FWD_THREADS / 32);
  if (rows * a.N >= 4 * warps) gemm_simt_tasks<WT, 4>(a);
  else if (rows * a.N >= 2 * warps) gemm_simt_tasks<WT, 2>(a);
  else gemm_simt_tasks<WT, 1>(a);
}

// ---- RoPE (rotate-half pairing) on q and k, then K/V into the paged pool --------------
// KV pool layout [L][2][n_blocks][Hkv][bs][hd]: one (block, kv head) tile is contiguous.
template <typename WT>
__device__ __forceinline__ WT* kv_tile(const DevCtx& c, int layer, int kv, int block, int head) {
  const size_t tile = (size_t)c.bs * c.hd;
  return reinterpret_cast<WT*>(c.kv_base) +
         ((((size_t)layer * 2 + kv) * c.n_blocks + block) * c.Hkv + head) * tile;
}

// One warp: four rounds of heads of one row (a lane owns four consecutive rotation pairs i .. i+3, i+half .. i+half+3 of
// a head; 32 lanes cover 2 heads of 128 or 4 of 64).  Position and table entries are read once per task and all loads
// are in flight before the first use; a thread per (row, head, quad) with its own index arithmetic, position and table
// loads took 16 us for 500 rows of the 8B shape (31 MB through L2).
template <typename WT>
static __device__ __noinline__ void phase_rope_kv(const DevCtx& c, int layer) {
  constexpr int U = 4;
  const int T = c.ss->cur_T;
  const int hd = c.hd, half = hd >> 1;
  const int lanes = half >> 2, per_round = 32 / lanes;   // lanes per head, heads per round
  const int heads = c.Hq + 2 * c.Hkv, rot_heads = c.Hq + c.Hkv;
  const int per_task = per_round * U, tasks_row = (heads + per_task - 1) / per_task;
  const int lane = threadIdx.x & 31;
  const int sub = lane / lanes, i = (lane - sub * lanes) * 4;
  const int total = T * tasks_row, step = gridDim.x * (FWD_THREADS / 32);
#pragma unroll 1
  for (int task = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; task < total; task += step) {
    const int t = (int)((unsigned)task / (unsigned)tasks_row), h0 = (task - t * tasks_row) * per_task + sub;
    float* row = c.qkv + (size_t)t * c.qkv_dim + i;
    float4 x1[U], x2[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int hh = min(h0 + u * per_round, heads - 1);   // past the end: the last head again (not stored)
      x1[u] = __ldcg(reinterpret_cast<const float4*>(row + hh * hd));
      x2[u] = __ldcg(reinterpret_cast<const float4*>(row + hh * hd + half));
    }
    const int pos = c.tok_pos[t], sm = c.tok_slotmap[t];
    const float4 cs = *reinterpret_cast<const float4*>(c.rope_cos + (size_t)pos * half + i);
    const float4 sn = *reinterpret_cast<const float4*>(c.rope_sin + (size_t)pos * half + i);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int hh = h0 + u * per_round;
      if (hh >= heads) break;
      float4 y1 = x1[u], y2 = x2[u];
      if (hh < rot_heads) {   // explicit fused forms: every instance of this code rounds the same way
#define BLINK_ROT1(a, b, cc, ss_) fmaf((a), (cc), -__fmul_rn((b), (ss_)))
#define BLINK_ROT2(a, b, cc, ss_) fmaf((b), (cc), __fmul_rn((a), (ss_)))
        y1 = make_float4(BLINK_ROT1(x1[u].x, x2[u].x, cs.x, sn.x), BLINK_ROT1(x1[u].y, x2[u].y, cs.y, sn.y),
                         BLINK_ROT1(x1[u].z, x2[u].z, cs.z, sn.z), BLINK_ROT1(x1[u].w, x2[u].w, cs.w, sn.w));
        y2 = make_float4(BLINK_ROT2(x1[u].x, x2[u].x, cs.x, sn.x), BLINK_ROT2(x1[u].y, x2[u].y, cs.y, sn.y),
                         BLINK_ROT2(x1[u].z, x2[u].z, cs.z, sn.z), BLINK_ROT2(x1[u].w, x2[u].w, cs.w, sn.w));
#undef BLINK_ROT1
#undef BLINK_ROT2
      }
      float* src = row + hh * hd;
      if (sizeof(WT) != 2 && hh < c.Hq) {   // fp32 mode: the attention reads q from this buffer
        *reinterpret_cast<float4*>(src) = y1;
        *reinterpret_cast<float4*>(src + half) = y2;
        continue;
      }
      WT* dst;
      if (hh < c.Hq) dst = reinterpret_cast<WT*>(c.qb) + (size_t)t * c.q_dim + hh * hd + i;   // operand of the attention contraction
      else dst = kv_tile<WT>(c, layer, hh < rot_heads ? 0 : 1, sm / c.bs, hh - (hh < rot_heads ? c.Hq : rot_heads)) +
                 (size_t)(sm % c.bs) * hd + i;
      store4<WT>(dst, y1.x, y1.y, y1.z, y1.w);
      store4<WT>(dst + half, y2.x, y2.y, y2.z, y2.w);
      if (c.gemm_tc) {   // the split-K GEMM of the next layer adds partial sums into this buffer: leave it cleared
        *reinterpret_cast<float4*>(src) = make_float4(0.f, 0.f, 0.f, 0.f);
        *reinterpret_cast<float4*>(src + half) = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
  }
}

// ---- fp32 steps of little work: the element-wise phases inside the GEMMs ------------------------------------
// A phase of the small configuration is 3 us, nearly all of it the grid barrier and the first round trip to L2, and a layer had
// nine.  Here the norm's sum of squares is added up beside the products, by every warp for its own rows (x is read anyway;
// the gains multiply the weights, the row's factor the result), and a warp owns pairs of features, so that it can rotate q and k
// and write K and V (QKV), or form silu(gate) * up (gate/up), from its own sums: five phases a layer, and no final norm.
// Steps of the small configuration: 8 rows 97 -> 72 us, 64 to 68 rows 142 -> 120.
enum FoldMode : int { FOLD_NORM = 0, FOLD_ROPE, FOLD_SILU };
// A sum of squares more per row and warp is up to half of the multiplications again: worth it while the largest GEMM of the layer
// has 10^8 of them.  One prompt of T rows, us a step without | with: 8 94 | 68, 64 142 | 125, 128 163 | 143, 190 199 | 183 (2 layers, d 256, F 1024).
__device__ __forceinline__ bool fold_step(const DevCtx& c, int T) {
  return c.dtype != 0 && c.E == 0 && (long long)T * c.d * 2 * c.F <= 100000000ll;
}
// The final norm is one phase (3.2 to 5 us), an LM head that does its work 5 % longer: 16 rows of 32000 entries 21.4 -> 23.4 us, 32 rows
// 38.2 -> 42.5, 128 rows of 128000 entries 725 -> 760 (d 256).
__device__ __forceinline__ bool fold_lm_head(const DevCtx& c, int R) { return (long long)R * c.d * c.V <= 200000000ll; }
template <int NC, int MODE>
__device__ __forceinline__ void gemm_fold_tasks(const DevCtx& c, const float* X, const int32_t* x_rows, const float* __restrict__ W,
                                                const float* __restrict__ gain, int M, int N, int layer) {
  constexpr int PAIRS = MODE == FOLD_NORM ? NC : NC / 2;   // results of a task and row
  constexpr int LPV = 32 / (SIMT_GR * NC);                 // lanes that hold the same sum
  const int K = c.d, lane = threadIdx.x & 31, half = c.hd >> 1;
  const int P = MODE == FOLD_NORM ? N : N / 2;
  const int groups_n = (P + PAIRS - 1) / PAIRS, groups_m = (M + SIMT_GR - 1) / SIMT_GR;
  const int nw = gridDim.x * (FWD_THREADS / 32);
  for (int task = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; task < groups_m * groups_n; task += nw) {
    const int gm = task / groups_n, gn = task - gm * groups_n;
    const int m0 = gm * SIMT_GR, p0 = gn * PAIRS;
    const float *w[NC], *x[SIMT_GR];
#pragma unroll
    for (int j = 0; j < NC; ++j) {   // clamped: rows past the end repeat
      const int q = min(p0 + (MODE == FOLD_NORM ? j : j % PAIRS), P - 1);
      const int n = MODE == FOLD_NORM ? q : MODE == FOLD_SILU ? q + (j < PAIRS ? 0 : P) : q / half * c.hd + q % half + (j < PAIRS ? 0 : half);
      w[j] = W + (size_t)n * K;
    }
#pragma unroll
    for (int i = 0; i < SIMT_GR; ++i) {
      const int m = min(m0 + i, M - 1);
      x[i] = X + (size_t)(x_rows != nullptr ? x_rows[m] : m) * K;
    }
    // what this lane's result needs besides, on its way with the first products
    const int idx = lane / LPV, r = idx / NC, j = idx % NC, m = m0 + r, q = p0 + j;
    const bool mine = lane % LPV == 0 && m < M && q < P && j < PAIRS;
    int sm = 0, hh = 0, d0 = 0;
    float cs = 1.f, sn = 0.f;
    if (MODE == FOLD_ROPE && mine) {
      hh = q / half;
      d0 = q - hh * half;
      sm = c.tok_slotmap[m];
      if (hh < c.Hq + c.Hkv) {
        const size_t at = (size_t)c.tok_pos[m] * half + d0;
        cs = c.rope_cos[at];
        sn = c.rope_sin[at];
      }
    }
    float acc[SIMT_GR * NC], ss[SIMT_GR];
#pragma unroll
    for (int i = 0; i < SIMT_GR * NC; ++i) acc[i] = 0.f;
#pragma unroll
    for (int i = 0; i < SIMT_GR; ++i) ss[i] = 0.f;
#pragma unroll 2
    for (int k = lane * 4; k < K; k += 128) {
      const float4 g = *reinterpret_cast<const float4*>(gain + k);
      float4 wv[NC], xv[SIMT_GR];
#pragma unroll
      for (int t = 0; t < NC; ++t) wv[t] = *reinterpret_cast<const float4*>(w[t] + k);
#pragma unroll
      for (int i = 0; i < SIMT_GR; ++i) xv[i] = *reinterpret_cast<const float4*>(x[i] + k);
#pragma unroll
      for (int t = 0; t < NC; ++t) wv[t] = make_float4(wv[t].x * g.x, wv[t].y * g.y, wv[t].z * g.z, wv[t].w * g.w);
#pragma unroll
      for (int i = 0; i < SIMT_GR; ++i) {
        ss[i] = fmaf(xv[i].x, xv[i].x, ss[i]); ss[i] = fmaf(xv[i].y, xv[i].y, ss[i]); ss[i] = fmaf(xv[i].z, xv[i].z, ss[i]); ss[i] = fmaf(xv[i].w, xv[i].w, ss[i]);
#pragma unroll
        for (int t = 0; t < NC; ++t) {
          float& s = acc[i * NC + t];
          s = fmaf(xv[i].x, wv[t].x, s); s = fmaf(xv[i].y, wv[t].y, s); s = fmaf(xv[i].z, wv[t].z, s); s = fmaf(xv[i].w, wv[t].w, s);
        }
      }
    }
    const float sq = __shfl_sync(0xffffffffu, warp_sum_many<SIMT_GR>(ss), r * (32 / SIMT_GR));
    const float v = warp_sum_many<SIMT_GR * NC>(acc) * rsqrtf(__fdividef(sq, (float)K) + c.rms_eps);
    if constexpr (MODE == FOLD_NORM) {
      if (mine) c.logits[(size_t)m * N + q] = v;
    } else {
      const float v2 = __shfl_down_sync(0xffffffffu, v, LPV * PAIRS);   // the second feature of the pair
      if (!mine) continue;
      if constexpr (MODE == FOLD_SILU) {
        reinterpret_cast<float*>(c.act)[(size_t)m * P + q] = __fdividef(v, 1.0f + __expf(-v)) * v2;
      } else {
        float y1 = v, y2 = v2;
        if (hh < c.Hq + c.Hkv) {   // the fused forms of the RoPE phase
          y1 = fmaf(v, cs, -__fmul_rn(v2, sn));
          y2 = fmaf(v2, cs, __fmul_rn(v, sn));
        }
        float* dst = hh < c.Hq ? c.qkv + (size_t)m * c.qkv_dim + hh * c.hd + d0
                               : kv_tile<float>(c, layer, hh < c.Hq + c.Hkv ? 0 : 1, sm / c.bs, (hh - c.Hq) % c.Hkv) + (size_t)(sm % c.bs) * c.hd + d0;
        dst[0] = y1;
        dst[half] = y2;
      }
    }
  }
}
template <int MODE>
static __device__ __noinline__ void phase_gemm_fold(const DevCtx& c, int layer) {
  const int M = MODE == FOLD_NORM ? c.ss->cur_rows : c.ss->cur_T;
  const int N = MODE == FOLD_NORM ? c.V : MODE == FOLD_ROPE ? c.qkv_dim : 2 * c.F;
  const float* W = MODE == FOLD_NORM ? wptr<float>(c, 9) : wptr<float>(c, MODE == FOLD_ROPE ? 1 : 3) + (size_t)layer * N * c.d;
  const float* gain = MODE == FOLD_NORM ? wptr_f(c, 8) : wptr_f(c, MODE == FOLD_ROPE ? 6 : 7) + (size_t)layer * c.d;
  const float* X = c.h;
  const int32_t* rows = MODE == FOLD_NORM ? c.row_tok : nullptr;
  if (MODE == FOLD_ROPE && layer == 0) {   // the embedding rows, which also start the residual stream
    X = wptr<float>(c, 0);
    rows = c.tok_id;
    for (int t = blockIdx.x; t < M; t += gridDim.x)
      for (int i = threadIdx.x * 4; i < c.d; i += FWD_THREADS * 4)
        *reinterpret_cast<float4*>(c.h + (size_t)t * c.d + i) = *reinterpret_cast<const float4*>(X + (size_t)rows[t] * c.d + i);
  }
  const long long groups = (M + SIMT_GR - 1) / SIMT_GR, warps = (long long)gridDim.x * (FWD_THREADS / 32);
  if (groups * N >= 4 * warps) gemm_fold_tasks<4, MODE>(c, X, rows, W, gain, M, N, layer);
  else gemm_fold_tasks<2, MODE>(c, X, rows, W, gain, M, N, layer);
}

// ---- element-wise consumers of finished GEMM output tiles (fused path) ----------------------------
// A tile is 128 consecutive output features of rows [t0, t1); the eight warps take rows in turn and a
// lane owns four consecutive features, so every access is one 512-byte line per row.  The fp32 sums
// were produced by reductions at L2 by several CTAs: they are read with .cg loads.

// QKV tile nt: RoPE on the q and k heads it covers (the rotation partner i + hd/2 of a feature lies in
// the same tile, hd/8 lanes away), q into the 16-bit attention operand, k and v into the paged pool;
// then the tile is cleared for the next GEMM that adds partial sums into this buffer.
constexpr int FIX_U = 8;   // rows per warp whose loads are issued before the first dependent use
constexpr int FIX_WARPS = FWD_THREADS / 32;

template <typename WT>
__device__ __noinline__ void fixup_rope_kv(const DevCtx& c, int layer, int nt, int t0, int t1) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int hd = c.hd, half = hd >> 1;
  const int f = nt * 128 + lane * 4;          // feature of this lane
  const int hh = f / hd, i0 = f - hh * hd;    // head and offset inside it
  const bool low = i0 < half;
  const int i = low ? i0 : i0 - half;         // rotation pair index
  const int partner = half >> 2;              // lanes between the two halves of a pair
  if (f >= c.qkv_dim) return;                 // whole warp: tiles are not ragged on this path
  const bool rot = hh < c.Hq + c.Hkv;
  const bool is_q = hh < c.Hq;
  const int kv = hh < c.Hq + c.Hkv ? 0 : 1;
  const int kvh = hh - c.Hq - kv * c.Hkv;
  for (int tb = t0 + w; tb < t1; tb += FIX_WARPS * FIX_U) {
    float4 x[FIX_U];
    int pos[FIX_U], sm[FIX_U];
#pragma unroll
    for (int u = 0; u < FIX_U; ++u) {
      const int t = min(tb + u * FIX_WARPS, t1 - 1);   // clamped: rows past the end repeat the last one (not stored)
      x[u] = __ldcg(reinterpret_cast<const float4*>(c.qkv + (size_t)t * c.qkv_dim + f));
      pos[u] = rot ? c.tok_pos[t] : 0;
      sm[u] = is_q ? 0 : c.tok_slotmap[t];
    }
#pragma unroll
    for (int u = 0; u < FIX_U; ++u) {
      const int t = tb + u * FIX_WARPS;
      float4 o;
      o.x = __shfl_xor_sync(0xffffffffu, x[u].x, partner);
      o.y = __shfl_xor_sync(0xffffffffu, x[u].y, partner);
      o.z = __shfl_xor_sync(0xffffffffu, x[u].z, partner);
      o.w = __shfl_xor_sync(0xffffffffu, x[u].w, partner);
      if (t >= t1) continue;   // uniform over the warp
      float4 y = x[u];
      float4 cs[FIX_U], sn[FIX_U];
      if (rot) {
        cs[u] = *reinterpret_cast<const float4*>(c.rope_cos + (size_t)pos[u] * half + i);
        sn[u] = *reinterpret_cast<const float4*>(c.rope_sin + (size_t)pos[u] * half + i);
        // the same explicit fused forms as the stand-alone RoPE phase: x1 = low half, x2 = high half
        if (low) {
          y = make_float4(fmaf(x[u].x, cs[u].x, -__fmul_rn(o.x, sn[u].x)), fmaf(x[u].y, cs[u].y, -__fmul_rn(o.y, sn[u].y)),
                          fmaf(x[u].z, cs[u].z, -__fmul_rn(o.z, sn[u].z)), fmaf(x[u].w, cs[u].w, -__fmul_rn(o.w, sn[u].w)));
        } else {
          y = make_float4(fmaf(x[u].x, cs[u].x, __fmul_rn(o.x, sn[u].x)), fmaf(x[u].y, cs[u].y, __fmul_rn(o.y, sn[u].y)),
                          fmaf(x[u].z, cs[u].z, __fmul_rn(o.z, sn[u].z)), fmaf(x[u].w, cs[u].w, __fmul_rn(o.w, sn[u].w)));
        }
      }
      WT* dst;
      if (is_q) dst = reinterpret_cast<WT*>(c.qb) + (size_t)t * c.q_dim + (size_t)hh * hd + i0;
      else dst = kv_tile<WT>(c, layer, kv, sm[u] / c.bs, kvh) + (size_t)(sm[u] % c.bs) * hd + i0;
      store4<WT>(dst, y.x, y.y, y.z, y.w);
      __stcg(reinterpret_cast<float4*>(c.qkv + (size_t)t * c.qkv_dim + f), make_float4(0.f, 0.f, 0.f, 0.f));
    }
  }
}

// gate tile j and up tile j of rows [t0, t1) of `gu` (row pitch 2F): act = silu(gate) * up; both cleared.
template <typename WT>
__device__ __noinline__ void fixup_silu(float* gu, WT* act, int F, int f0, int width, int t0, int t1) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int f = f0 + lane * 4;
  if (lane * 4 >= width || f >= F) return;
  for (int tb = t0 + w; tb < t1; tb += FIX_WARPS * FIX_U) {
    float4 g[FIX_U], u4[FIX_U];
#pragma unroll
    for (int u = 0; u < FIX_U; ++u) {
      const int t = min(tb + u * FIX_WARPS, t1 - 1);
      g[u] = __ldcg(reinterpret_cast<const float4*>(gu + (size_t)t * 2 * F + f));
      u4[u] = __ldcg(reinterpret_cast<const float4*>(gu + (size_t)t * 2 * F + F + f));
    }
#pragma unroll
    for (int u = 0; u < FIX_U; ++u) {
      const int t = tb + u * FIX_WARPS;
      if (t >= t1) continue;
      store4<WT>(act + (size_t)t * F + f, __fdividef(g[u].x, 1.0f + __expf(-g[u].x)) * u4[u].x, __fdividef(g[u].y, 1.0f + __expf(-g[u].y)) * u4[u].y,
                 __fdividef(g[u].z, 1.0f + __expf(-g[u].z)) * u4[u].z, __fdividef(g[u].w, 1.0f + __expf(-g[u].w)) * u4[u].w);
      __stcg(reinterpret_cast<float4*>(gu + (size_t)t * 2 * F + f), make_float4(0.f, 0.f, 0.f, 0.f));
      __stcg(reinterpret_cast<float4*>(gu + (size_t)t * 2 * F + F + f), make_float4(0.f, 0.f, 0.f, 0.f));
    }
  }
}

// residual tile nt of rows [t0, t1): its share of sum(x^2) per row
static __device__ __noinline__ void fixup_sumsq(const float* h, int ld, int N, float* rowss, int nt, int t0, int t1) {
  constexpr int U = 8;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int f = nt * 128 + lane * 4;
  for (int tb = t0 + w; tb < t1; tb += FIX_WARPS * U) {
    float4 x[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int t = min(tb + u * FIX_WARPS, t1 - 1);
      x[u] = f < N ? __ldcg(reinterpret_cast<const float4*>(h + (size_t)t * ld + f)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int t = tb + u * FIX_WARPS;
      float s = fmaf(x[u].x, x[u].x, fmaf(x[u].y, x[u].y, fmaf(x[u].z, x[u].z, x[u].w * x[u].w)));
      s = warp_sum(s);
      if (lane == 0 && t < t1) atomicAdd(rowss + t, s);
    }
  }
}

// ---- paged attention ---------------------------------------------------------------------
// Unit of work: (row t, kv head g): the n_rep query heads of the group share every K/V
// load.  The 8 warps of the CTA take KV blocks round-robin; within a warp a 16-byte
// vector load per lane covers whole (block, head) tiles with coalesced 512-byte rows.
// Online softmax per warp, merged across warps in shared memory at the end.
template <typename WT, int HD, int NREP>
static __device__ __noinline__ void phase_attention(const DevCtx& c, int layer, float* smem) {
  constexpr int CE = 16 / (int)sizeof(WT);  // elements per 16-byte chunk
  constexpr int LPK = HD / CE;              // lanes per key
  constexpr int KPP = 32 / LPK;             // keys per pass
  constexpr int MAXR = NREP;                // query heads per kv head
  constexpr int NW = FWD_THREADS / 32;
  static_assert(LPK <= 32 && KPP >= 1, "head_dim too large for this mapping");
  const int T = c.ss->cur_T;
  constexpr int n_rep = NREP;
  const int bs = c.bs;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int sub = lane / LPK;   // which key of the pass
  const int ch = lane % LPK;    // which 16-byte chunk of the head vector
  // shared: q [NREP][HD], per-warp m,l [NW][NREP], acc [NW][NREP][HD]
  float* s_q = smem;
  float* s_m = s_q + MAXR * HD;
  float* s_l = s_m + NW * MAXR;
  float* s_acc = s_l + NW * MAXR;
  WT* out = reinterpret_cast<WT*>(c.attn);

  const int units = T * c.Hkv;
  for (int u = blockIdx.x; u < units; u += gridDim.x) {
    const int t = u / c.Hkv, g = u % c.Hkv;
    const int item = c.tok_item[t];
    const int b = c.it_bslot[item];
    const int n_ctx = c.tok_pos[t] + 1;
    const int32_t* table = c.block_table + (size_t)b * c.max_blocks_seq;
    __syncthreads();
    for (int i = threadIdx.x; i < n_rep * HD; i += FWD_THREADS)
      s_q[i] = c.qkv[(size_t)t * c.qkv_dim + (size_t)g * n_rep * HD + i] * c.attn_scale;
    __syncthreads();
    float q[MAXR][CE];
    float acc[MAXR][CE];
    float m[MAXR], l[MAXR];
#pragma unroll
    for (int r = 0; r < MAXR; ++r) {
      m[r] = -INFINITY;
      l[r] = 0.f;
#pragma unroll
      for (int e = 0; e < CE; ++e) {
        acc[r][e] = 0.f;
        q[r][e] = (r < n_rep) ? s_q[r * HD + ch * CE + e] : 0.f;
      }
    }
    const int n_kb = (n_ctx + bs - 1) / bs;
    for (int kb = w; kb < n_kb; kb += NW) {
      const int blk = table[kb];
      const WT* kt = kv_tile<WT>(c, layer, 0, blk, g);
      const WT* vt = kv_tile<WT>(c, layer, 1, blk, g);
      for (int k0 = 0; k0 < bs; k0 += KPP) {
        const int key = k0 + sub;
        const int kpos = kb * bs + key;
        const bool valid = key < bs && kpos < n_ctx;
        float kf[CE], vf[CE];
        if (valid) {
          const uint4 kr = *reinterpret_cast<const uint4*>(kt + (size_t)key * HD + ch * CE);
          const uint4 vr = *reinterpret_cast<const uint4*>(vt + (size_t)key * HD + ch * CE);
          const WT* kp = reinterpret_cast<const WT*>(&kr);
          const WT* vp = reinterpret_cast<const WT*>(&vr);
#pragma unroll
          for (int e = 0; e < CE; ++e) { kf[e] = OpType<WT>::to_f(kp[e]); vf[e] = OpType<WT>::to_f(vp[e]); }
        } else {
#pragma unroll
          for (int e = 0; e < CE; ++e) { kf[e] = 0.f; vf[e] = 0.f; }
        }
#pragma unroll
        for (int r = 0; r < MAXR; ++r) {
          if (r >= n_rep) break;
          float s = 0.f;
#pragma unroll
          for (int e = 0; e < CE; ++e) s = fmaf(q[r][e], kf[e], s);
#pragma unroll
          for (int o = LPK / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
          if (!valid) s = -INFINITY;
          // max over the keys of this pass (lanes with different `sub`)
          float mx = s;
#pragma unroll
          for (int o = LPK; o < 32; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
          const float m_new = fmaxf(m[r], mx);
          if (m_new == -INFINITY) continue;   // nothing valid yet (uniform across the warp)
          const float corr = __expf(m[r] - m_new);
          const float p = valid ? __expf(s - m_new) : 0.f;
          // l and acc are per-lane partials over this lane's keys; lanes of other `sub`
          // hold the other keys and are merged at the end
          l[r] = l[r] * corr + p;
#pragma unroll
          for (int e = 0; e < CE; ++e) acc[r][e] = fmaf(p, vf[e], acc[r][e] * corr);
          m[r] = m_new;
        }
      }
    }
    // merge lanes that handled different keys (same chunk): sum over `sub`
#pragma unroll
    for (int r = 0; r < MAXR; ++r) {
      if (r >= n_rep) break;
#pragma unroll
      for (int o = LPK; o < 32; o <<= 1) {
        l[r] += __shfl_xor_sync(0xffffffffu, l[r], o);
#pragma unroll
        for (int e = 0; e < CE; ++e) acc[r][e] += __shfl_xor_sync(0xffffffffu, acc[r][e], o);
      }
      // every lane with the same `ch` now holds the warp's full partial
      if (sub == 0) {
#pragma unroll
        for (int e = 0; e < CE; ++e) s_acc[((size_t)w * MAXR + r) * HD + ch * CE + e] = acc[r][e];
        if (ch == 0) { s_m[w * MAXR + r] = m[r]; s_l[w * MAXR + r] = l[r]; }
      }
    }
    __syncthreads();
    // merge the warps: out = sum_w e^(m_w - M) acc_w / sum_w e^(m_w - M) l_w
    for (int i = threadIdx.x; i < n_rep * HD; i += FWD_THREADS) {
      const int r = i / HD, dim = i % HD;
      float M = -INFINITY;
#pragma unroll
      for (int ww = 0; ww < NW; ++ww) M = fmaxf(M, s_m[ww * MAXR + r]);
      float num = 0.f, den = 0.f;
#pragma unroll
      for (int ww = 0; ww < NW; ++ww) {
        const float mw = s_m[ww * MAXR + r];
        if (mw == -INFINITY) continue;
        const float f = __expf(mw - M);
        num += f * s_acc[((size_t)ww * MAXR + r) * HD + dim];
        den += f * s_l[ww * MAXR + r];
      }
      out[(size_t)t * c.q_dim + (size_t)(g * n_rep + r) * HD + dim] = OpType<WT>::from_f(num / den);
    }
  }
}
constexpr int ATTN_SMEM_FLOATS(int HD, int NREP) { return NREP * HD + 2 * 8 * NREP + 8 * NREP * HD; }

// ---- SwiGLU gate: act = silu(gate) * up ------------------------------------------------
// The gate/up buffer comes from HBM (the weight stream of the GEMM before has pushed it out of L2)
// and one CTA per SM leaves eight warps to cover that latency, so every thread has the loads of
// SILU_U items in flight before it stores.  A function of its own: inlined into the loop kernel
// the buffers of loaded values end up in local memory.
// silu(g) * u with the approximate division (2 ulp, then rounded to the operand type): the exact fp32 division
// took a quarter of the SwiGLU phase
template <typename WT>
__device__ __forceinline__ void silu_store(float* gu, WT* out, int t, int j, int F, const float4& g, const float4& u, bool clear) {
  store4<WT>(out + (size_t)t * F + j, __fdividef(g.x, 1.0f + __expf(-g.x)) * u.x, __fdividef(g.y, 1.0f + __expf(-g.y)) * u.y,
             __fdividef(g.z, 1.0f + __expf(-g.z)) * u.z, __fdividef(g.w, 1.0f + __expf(-g.w)) * u.w);
  if (clear) {   // consumed: the next split-K gate/up GEMM adds partial sums into a cleared buffer
    __stcg(reinterpret_cast<float4*>(gu + (size_t)t * 2 * F + j), make_float4(0.f, 0.f, 0.f, 0.f));
    __stcg(reinterpret_cast<float4*>(gu + (size_t)t * 2 * F + F + j), make_float4(0.f, 0.f, 0.f, 0.f));
  }
}
template <typename WT>
__device__ __noinline__ void silu_mul_rows(float* __restrict__ gu, WT* __restrict__ out, int T, int F, bool clear) {
  constexpr int SILU_U = 4;
  const int F4 = F / 4;
  const int total = T * F4;   // < 2^31: at most a few thousand rows
  const int stride = gridDim.x * FWD_THREADS;
  for (int base = blockIdx.x * FWD_THREADS + threadIdx.x; base < total; base += SILU_U * stride) {
    float4 g[SILU_U], u[SILU_U];
#pragma unroll
    for (int k = 0; k < SILU_U; ++k) {
      const int idx = min(base + k * stride, total - 1);   // clamped: the tail loads a valid item twice
      const int t = idx / F4, j = (idx - t * F4) * 4;
      g[k] = __ldcg(reinterpret_cast<const float4*>(gu + (size_t)t * 2 * F + j));
      u[k] = __ldcg(reinterpret_cast<const float4*>(gu + (size_t)t * 2 * F + F + j));
    }
#pragma unroll
    for (int k = 0; k < SILU_U; ++k) {
      const int idx = base + k * stride;
      if (idx < total) {
        const int t = idx / F4;
        silu_store<WT>(gu, out, t, (idx - t * F4) * 4, F, g[k], u[k], clear);
      }
    }
  }
}
// The same over the (token pass, gate/up weight tile) units that the GEMM has not already written as
// activations (a unit is up to 256 rows x 64 features; the GEMM stamps the units it wrote).  Every CTA
// compacts the pending units into shared memory once, then all threads of the grid share their items evenly.
static __device__ __noinline__ int silu_pending_units(const unsigned long long* done, unsigned long long stamp, int n_units, int* list) {
  __shared__ int s_warp[FWD_THREADS / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int count = 0;   // uniform over the CTA
  for (int b0 = 0; b0 < n_units; b0 += FWD_THREADS) {
    const int unit = b0 + threadIdx.x;
    const bool pend = unit < n_units && __ldcg(done + unit) != stamp;   // written by other SMs: not through L1
    const unsigned m = __ballot_sync(0xffffffffu, pend);
    if (lane == 0) s_warp[w] = __popc(m);
    __syncthreads();
    int off = count, tot = 0;
#pragma unroll
    for (int i = 0; i < FWD_THREADS / 32; ++i) {
      if (i < w) off += s_warp[i];
      tot += s_warp[i];
    }
    if (pend) list[off + __popc(m & ((1u << lane) - 1u))] = unit;
    count += tot;
    __syncthreads();
  }
  return count;
}
// A CTA takes up to a quarter of a pending unit at a time: 64 rows x 64 features, four items per thread.  The
// loads are asynchronous copies into a staging area in shared memory (each thread reads back only what it
// copied itself), so four items are in flight per thread without holding registers for them: a body that
// needs many registers here changes the register allocation of the other phase functions of the loop
// kernel, to their cost.
// Token rows per pass of a tensor-core GEMM over T rows in `passes` passes of at most 256: a multiple of 16, the passes
// as even as they go.
__device__ __forceinline__ int tc_pass_rows(int T, int passes) { return (int)((((unsigned)T + (unsigned)passes - 1u) / (unsigned)passes + 15u) & ~15u); }
__device__ __forceinline__ int tc_pass_rows(int T) { return tc_pass_rows(T, (int)((unsigned)(T + 255) >> 8)); }
constexpr int SILU_STAGE_OFF = 32768 * 4;   // bytes: the staging area follows the list of pending units
template <typename WT>
__device__ __noinline__ void silu_mul_pending(float* __restrict__ gu, WT* __restrict__ out, int T, int F, const int* list, int count) {
  const int tiles = F >> 6, pass_rows = tc_pass_rows(T);
  const int r_in = threadIdx.x >> 4, col = (threadIdx.x & 15) << 2;
  const char* stage = reinterpret_cast<const char*>(list) + SILU_STAGE_OFF + threadIdx.x * 16;   // [2][8][FWD_THREADS] x 16 bytes
  const uint32_t stage_s = (uint32_t)__cvta_generic_to_shared(stage);
  constexpr int BUF = 8 * FWD_THREADS * 16;
  auto where = [&](int q, int& row0, int& j, int& t_end) {
    const int unit = list[q >> 2];
    const int pass = unit / tiles, tile = unit - pass * tiles;
    row0 = pass * pass_rows + ((q & 3) << 6) + r_in;
    j = (tile << 6) + col;
    t_end = min(T, (pass + 1) * pass_rows);
  };
  auto fetch = [&](int q, int buf) {
    int row0, j, t_end;
    where(q, row0, j, t_end);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int t = row0 + 16 * k;
      if (t < t_end) {
        const float* src = gu + (size_t)t * 2 * F + j;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(stage_s + buf * BUF + (2 * k) * FWD_THREADS * 16), "l"(src) : "memory");
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(stage_s + buf * BUF + (2 * k + 1) * FWD_THREADS * 16), "l"(src + F) : "memory");
      }
    }
  };
  // the next piece is on its way while the current one is worked on (every thread reads back what it copied itself)
  int q = blockIdx.x, buf = 0;
  if (q < count * 4) fetch(q, 0);
  asm volatile("cp.async.commit_group;" ::: "memory");
#pragma unroll 1
  for (; q < count * 4; q += gridDim.x, buf ^= 1) {
    if (q + (int)gridDim.x < count * 4) fetch(q + gridDim.x, buf ^ 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    int row0, j, t_end;
    where(q, row0, j, t_end);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int t = row0 + 16 * k;
      if (t < t_end) {
        const float4 g = *reinterpret_cast<const float4*>(stage + buf * BUF + (2 * k) * FWD_THREADS * 16);
        const float4 u = *reinterpret_cast<const float4*>(stage + buf * BUF + (2 * k + 1) * FWD_THREADS * 16);
        silu_store<WT>(gu, out, t, j, F, g, u, true);
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}
// The GEMM writes activations itself only in steps of more than one token pass: there its epilogue hides
// behind the tensor-core work of the next tile, while at decode sizes the GEMM is bound by the weight
// stream and the longer epilogue would show.
__device__ __forceinline__ bool gu_direct_step(const DevCtx& c, int T) { return c.gu_direct && T > 256; }
template <typename WT>
static __device__ __noinline__ void phase_silu_mul(const DevCtx& c, int layer, float* smem) {
  const int T = c.E > 0 ? c.ss->cur_T * c.topE : c.ss->cur_T;   // rows of the gate/up buffer
  if (T <= 0) return;
  if (gu_direct_step(c, T)) {
    int* list = reinterpret_cast<int*>(smem);
    const int count = silu_pending_units(c.gu_done, c.ss->iter * (unsigned long long)c.L + (unsigned long long)layer + 1ull, ((T + 255) >> 8) * (c.F >> 6), list);
    silu_mul_pending<WT>(c.gu, reinterpret_cast<WT*>(c.act), T, c.F, list, count);
  } else
    silu_mul_rows<WT>(c.gu, reinterpret_cast<WT*>(c.act), T, c.F, c.gemm_tc != 0);
}

// ---- routed experts: group the (token, expert) pairs by expert and gather their rows ---------
// Every CTA builds the same lists in shared memory (stable: ascending token inside an expert, so
// the order does not depend on timing), CTA 0 publishes them, and all CTAs copy the normed rows
// of the tokens into expert-contiguous order for the per-expert GEMMs.
template <typename WT>
static __device__ __noinline__ void phase_moe_group(const DevCtx& c, float* smem) {
  const int T = c.ss->cur_T, K = c.topE, E = c.E;
  const int A = T * K;   // assignments
  __shared__ int s_off[MAX_EXPERTS + 1];
  int* s_tok = reinterpret_cast<int*>(smem);          // [A] token of each gathered row
  // the choices as bytes behind it, where they fit: every warp walks all of them for each of its experts, and a walk
  // over memory waits for every 32 (25 us for 960 choices)
  unsigned char* s_sel = reinterpret_cast<unsigned char*>(s_tok + A);
  const bool staged = c.gemm_tc && A <= 32768;        // (the GEMM rings are larger than 5 x 32768 bytes)
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  // counts, then offsets
  if (threadIdx.x <= E) s_off[threadIdx.x] = 0;
  __syncthreads();
  for (int a = threadIdx.x; a < A; a += FWD_THREADS) {
    const int e = c.moe_sel[a];
    if (staged) s_sel[a] = (unsigned char)e;
    atomicAdd(&s_off[e + 1], 1);
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int e = 0; e < E; ++e) s_off[e + 1] += s_off[e];
  __syncthreads();
  // stable placement: a warp walks all assignments in order for each of its experts
  for (int e = w; e < E; e += FWD_THREADS / 32) {
    int base = s_off[e];
    for (int a0 = 0; a0 < A; a0 += 32) {
      const int a = a0 + lane;
      const bool mine = a < A && (staged ? (int)s_sel[a] : c.moe_sel[a]) == e;
      const unsigned m = __ballot_sync(0xffffffffu, mine);
      if (mine) {
        const int pos = base + __popc(m & ((1u << lane) - 1u));
        s_tok[pos] = a / K;
        if (blockIdx.x == 0) { c.moe_tok[pos] = a / K; c.moe_gate[pos] = c.moe_wt[a]; }
      }
      base += __popc(m);
    }
  }
  if (blockIdx.x == 0 && threadIdx.x <= E) c.moe_off[threadIdx.x] = s_off[threadIdx.x];
  __syncthreads();
  // gather: one warp per row, 16-byte vectors
  const WT* xn = reinterpret_cast<const WT*>(c.xn);
  WT* xg = reinterpret_cast<WT*>(c.xg);
  const int vec_per_row = c.d * (int)sizeof(WT) / 16;
  for (int r = blockIdx.x * (FWD_THREADS / 32) + w; r < A; r += gridDim.x * (FWD_THREADS / 32)) {
    const uint4* src = reinterpret_cast<const uint4*>(xn + (size_t)s_tok[r] * c.d);
    uint4* dst = reinterpret_cast<uint4*>(xg + (size_t)r * c.d);
    for (int i0 = 0; i0 < vec_per_row; i0 += 256) {   // eight vectors per lane on their way at a time
      uint4 v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = src[min(i0 + 32 * k + lane, vec_per_row - 1)];
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (i0 + 32 * k + lane < vec_per_row) dst[i0 + 32 * k + lane] = v[k];
    }
  }
}

}  // namespace blink

#include "sampler.cuh"
