// Which way the attention of a step goes: rules on its sizes alone.  Plain C++, so that a test can ask them on the CPU.
#pragma once

#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace blink {

// ---- requests of several rows ----------------------------------------------------------------------------------
// Query rows that a CTA pair takes at a time, and the requests that may go to the pairs: a unit of a pair starts and ends in 11 us
// (with the phase) where one of a single CTA takes 6, but goes through 128 keys of 64 rows in 1.0 to 1.7 us where that takes 5.5
// for 32.  8B shape, us a layer, single CTAs | pairs, for prompts x rows: 1 x 128 10.9 | 13.1, 1 x 256 16.7 | 15.4, 1 x 257 17.9 | 13.2,
// 1 x 400 24.2 | 14.7, 1 x 512 27.4 | 15.7, 512 rows behind 3500 keys 177 | 63, 3 x 170 15.4 | 17.5, 8 x 64 12.1 | 18.2, 24 x 20 17.0 | 34.2,
// 3 x 257 35.7 | 25.2, 4 x 300 44.5 | 34.9, 6 x 300 59 | 45, 10 x 300 82 | 67, 14 x 270 103 | 83, 4 x 430 62 | 50, 10 x 430 142 | 100, 10 x 350 92 | 91,
// 4 x 512 90 | 53, 2 x 2000 355 | 144.
constexpr int ATT_PAIR_ROWS = 64;
__host__ __device__ __forceinline__ bool att_on_pairs(int keys) { return keys > 256; }
// All the same to single CTAs: the pairs would need a second round where the single CTAs have all the step's units in one, and the
// contexts are short.  2 x 257 19.0 | 21.0, 2 x 270 19.9 | 21.2, but 2 x 290 (two rounds both) 26.3 | 22.8; the lines cross at some 350 keys.
constexpr int ATT_ONE_ROUND_KEYS = 320;
__host__ __device__ __forceinline__ bool att_one_round_on_ctas(int pair_units, int cta_units, int n_ctas, int longest) {
  return pair_units > n_ctas / 2 && cta_units <= n_ctas && longest <= ATT_ONE_ROUND_KEYS;
}

// ---- single rows ---------------------------------------------------------------------------------------------------
struct AttDecodeWay {
  long long S;   // streaming: tiles per sub-range of the flat tile sequence, 0 = a sub-range is a (row, kv head) unit
  int C;         // > 0: units are shared by the warps of a CTA, C tiles per part
  int half;      // such units (whole ones) are shared by half of the warps of a CTA
};
struct AttDecodeStep {
  long long TT;        // (row, kv head, block) tiles, and the (row, kv head) units that hold them
  int units, maxkb;    // most tiles of a unit
  int cta_C, cta_items;   // parts that fit the CTAs at once (or whole units), 0 = too many units
  int n_ctas, warps;   // CTAs of the grid, warps of a CTA
  bool prompt_rows;    // beside rows of prompts
  long long sub_max;   // records that the streaming kernel has room for
};
__host__ __device__ __forceinline__ AttDecodeWay att_decode_way(const AttDecodeStep& a) {
  AttDecodeWay way{0, 0, 0};
  // Sub-ranges: k per warp of the grid.  Every cut of a unit costs a partial record and a merge,
  // so a pure decode step takes one sub-range per warp up to 96 tiles; with prefill tiles in the
  // step the CTAs reach their decode share at different times and smaller sub-ranges (up to 48
  // tiles, the later ones handed out by the counter) even that out.
  const long long NW = (long long)a.n_ctas * a.warps, TT = a.TT, U = a.units, maxkb = a.maxkb;
  const long long cap = a.prompt_rows ? 48 : 96;
  const long long k = (TT + cap * NW - 1) / (cap * NW) > 1 ? (TT + cap * NW - 1) / (cap * NW) : 1;
  long long S = (TT + k * NW - 1) / (k * NW);
  // at least 8 tiles per sub-range: a cut costs a partial record, a fence and a counter update (about the time of
  // two tiles), and a unit cut into n parts is merged by one warp in n steps; with few long rows one tile per
  // sub-range made a single 2048-token row take 120 us per layer, most of it the merge
  if (S < 8) S = 8;
  while ((TT + S - 1) / S > a.sub_max) S *= 2;   // cannot happen with the sizes set at create
  // Estimates in units of 0.2 us, fitted to the measurements below: the streaming
  // kernel cuts the flat sequence evenly, 8 a tile with all warps at work, 52 for the ends of cut units; whole units
  // per warp need no cuts, a tile 5 with few warps at work and 8 with all; a CTA per part shares a unit between its
  // eight warps, 6 a tile and 17 a round (start, merge in shared memory, two barriers).
  // 8B shape, us a layer, streaming | whole units | CTA, for rows x keys:
  //   17 x 40  17.9 | 11.9 | 10.2    17 x 300  26 | 30 | 12.7    17 x 1500  40 | 106 | 24    17 x 4000  70 | 280 | 50
  //   24 x 40  18.0 | 11.7    24 x 300  26 | 29    24 x 1500  48 | 110    24 x 4000  87 | 285
  //   37 x 40  18.1 | 12.0    37 x 300  27 | 30    37 x 1500  58 | 126    48 x 40  18.2 | 12.2
  //   48 x 300  28 | 30    100 x 40  20 | 15.5    100 x 300  41 | 36    100 x 900  88 | 91    200 x 40  26.5 | 24.5
  //   200 x 300  69 | 68    200 x 700  125 | 146    200 of 20 to 1500 keys  88 | 144
  const long long t_stream = 8 * S * ((((TT + S - 1) / S) + NW - 1) / NW) + 52;
  const long long t_unit = maxkb * ((U + NW - 1) / NW) * (5 * NW + 3 * (U < NW ? U : NW)) / NW + 14;
  // More units than CTAs: half CTAs, one round, 6 a tile of their warps and 24 for a CTA's worth of units.  Below what memory allows
  // where all units are long, but so is what the streaming kernel is charged; the better of the two others | half CTAs, measured together
  // (right after the prompts' steps, whose clocks make both longer):
  //   8B shape  19 x 40  9.8 | 9.7    19 x 300  25 | 13.4    19 x 1500  43 | 40    19 x 4000  83 | 91    24 x 40  10.0 | 10.9    24 x 300  25 | 14.8
  //             24 x 1500  55 | 43    24 x 4000  98 | 90    30 x 300  26 | 16.7    30 x 1500  59 | 47    30 x 4000  116 | 92
  //             37 x 40  10.0 | 14.1    37 x 100  14.7 | 15.0    37 x 300  26 | 18.6    37 x 1500  68 | 51    37 x 4000  129 | 104
  //             24 of 20 to 1500 keys  37 | 28.5    37 of 20 to 1500  46 | 41    24 of 100 to 4000  70 | 81
  //   1B shape  19 x 100  10.2 | 9.3    24 x 300  16.8 | 12.3    24 x 1500  25.4 | 23.6    24 x 4000  44 | 48    30 x 4000  52 | 50    37 x 4000  60 | 57
  //             24 of 100 to 4000 keys  31 | 44
  // The choice is the faster side or within 4 % of it for units of one length, except 24 x 4000 keys of the 8B shape (streaming,
  // 98); lengths from 20 to 1500 stream although half CTAs would be faster.
  way.half = a.cta_C > 0 && a.cta_items > a.n_ctas;
  if (a.cta_C > 0) {
    const long long part = a.cta_C < maxkb ? a.cta_C : maxkb;
    const long long t_cta = way.half ? 6 * ((maxkb + 3) / 4) + 24ll * a.cta_items / a.n_ctas + 1
                                     : 6 * ((part + 7) / 8) + 17 + (a.cta_C < maxkb ? 14 : 0);
    if (t_cta <= t_stream && t_cta <= t_unit) way.C = a.cta_C;
  }
  way.S = way.C == 0 && t_unit < t_stream ? 0 : S;
  return way;
}

}  // namespace blink
