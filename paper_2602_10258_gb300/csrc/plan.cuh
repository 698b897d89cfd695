// Per-query preparation shared by the batched search and the serve loop:
// filter validation, the boolean filter-distance table and the routing
// decision (graph search or exact scan).
#pragma once

#include "jag_internal.cuh"

namespace jag {

// Positions [*b, *e) of the values in [lo, hi] of a sorted column, by the
// calling warp: the lower bound by lanes 0..15, the upper by lanes 16..31, each
// cutting its range into 16 parts a round.  Five dependent reads for a million
// values where one lane's two binary searches made forty (preparation of 16
// label queries on 200K points: 15 us, now 7).
template <class V>
__device__ __forceinline__ void warp_bounds(const V *v, int64_t n, V lo, V hi, int64_t *b, int64_t *e) {
  const int lane = threadIdx.x & 31, half = lane >> 4, j = lane & 15;
  int64_t x = 0, y = n;   // the bound lies in [x, y]
  while (__any_sync(kFull, x < y)) {
    const int64_t s = (y - x + 15) >> 4;
    const int64_t p = x + (j + 1) * s - 1;   // the last value of part j
    bool below = false;
    if (s > 0 && p < y) {
      const V a = v[p];
      below = half ? a <= hi : a < lo;
    }
    const uint32_t m = __ballot_sync(kFull, below);
    x += __popc(half ? m >> 16 : m & 0xFFFFu) * s;
    if (s > 0) y = min64(y, x + s - 1);
  }
  *b = __shfl_sync(kFull, x, 0);
  *e = __shfl_sync(kFull, x, 16);
}

// Boolean distance table of one filter (Sec. 3.1, boolean example):
// lut[s] = least Hamming distance from assignment s of the m involved bits to
// an assignment where the truth table is 1 (255 if there is none).  Computed
// one dimension at a time: the Hamming metric is a sum over bits, so relaxing
// each pair (s, s ^ 2^j) once per bit j gives the exact distances.
__device__ inline void build_bool_lut(const uint8_t *tt, int m, uint8_t *lut) {
  const int lane = threadIdx.x & 31;
  const uint32_t S = 1u << m;
  for (uint32_t s = lane; s < S; s += 32) lut[s] = ((tt[s >> 3] >> (s & 7)) & 1) ? 0 : 255;
  __syncwarp();
  for (int j = 0; j < m; ++j) {
    const uint32_t low = (1u << j) - 1;
    for (uint32_t i = lane; i < (S >> 1); i += 32) {
      const uint32_t s = ((i & ~low) << 1) | (i & low);
      const uint32_t t = s | (1u << j);
      const int a = lut[s], b = lut[t];
      lut[s] = (uint8_t)min(a, b + 1);
      lut[t] = (uint8_t)min(b, a + 1);
    }
    __syncwarp();
  }
}

// Plan of one query by the calling warp (every lane returns the same):
// validate the filter (false: bad filter, route kRouteSkip); build the
// boolean table at lut_base + 8 * aux_off; label/range filters count their
// passing set exactly (binary search in the sorted column), subset/boolean
// filters estimate it on the fixed sample of S = min(4096, n) points with
// ids floor(j n / S).  With s0 > 0 a query whose count (estimate) is below s0
// goes to the exact scan (a slice of a sorted column, or, for subset/boolean
// filters, a list gathered by a pass over the mask column).  need_est: fill
// pl.est even when s0 = 0 (the learned policy's feature).
__device__ inline bool plan_query(const DevIndex &ix, const jag_filter &f, const uint8_t *aux, int64_t aux_bytes,
                                  int64_t s0, int64_t cap, int scan_all, int need_est, uint8_t *lut_base,
                                  QueryPlan &pl) {
  const int lane = threadIdx.x & 31;
  pl.route = kRouteGraph; pl.lut_off = -1; pl.begin = 0; pl.end = 0; pl.count = 0; pl.est = 0;
  bool ok;
  int m = 0;
  switch (f.kind) {
    case JAG_F_NONE: ok = true; break;
    case JAG_F_LABEL: case JAG_F_RANGE_I32: ok = ix.a_i32 != nullptr; break;
    case JAG_F_RANGE_F32: ok = ix.a_f32 != nullptr; break;
    case JAG_F_SUBSET: ok = ix.a_mask != nullptr; break;
    case JAG_F_BOOL: {
      m = __popcll(f.payload);
      ok = ix.a_mask != nullptr && aux != nullptr && m <= 16 && f.aux_off >= 0;
      if (ok) {
        const int64_t tbytes = ((int64_t)1 << m) / 8 > 0 ? ((int64_t)1 << m) / 8 : 1;
        ok = (int64_t)f.aux_off + tbytes <= aux_bytes;
      }
      break;
    }
    default: ok = false;
  }
  if (!ok) {
    pl.route = kRouteSkip;
    return false;
  }
  const uint8_t *tt = nullptr;
  if (f.kind == JAG_F_BOOL) {
    tt = aux + f.aux_off;
    pl.lut_off = f.aux_off * 8;
    build_bool_lut(tt, m, lut_base + pl.lut_off);
  }
  if (scan_all) {
    pl.route = kRouteBrute;
  } else if (s0 > 0 || need_est) {
    if (f.kind == JAG_F_LABEL || f.kind == JAG_F_RANGE_I32 || f.kind == JAG_F_RANGE_F32) {
      int64_t b = 0, e = 0;
      if (f.kind == JAG_F_RANGE_F32) {
        const float lo = u2f((uint32_t)lo32(f.payload)), hi = u2f((uint32_t)hi32(f.payload));
        if (lo <= hi) warp_bounds(ix.sf32_val, ix.n, lo, hi, &b, &e);
      } else {
        const int32_t lo = lo32(f.payload), hi = f.kind == JAG_F_LABEL ? lo : hi32(f.payload);
        if (lo <= hi) warp_bounds(ix.si32_val, ix.n, lo, hi, &b, &e);
      }
      pl.begin = b; pl.end = e;
      pl.est = (int32_t)min64(e - b, 0x7FFFFFFF);
      if (s0 > 0 && e - b < s0 && e - b <= cap) pl.route = kRouteSlice;
    } else if (f.kind == JAG_F_SUBSET || f.kind == JAG_F_BOOL) {
      const int64_t S = ix.n < 4096 ? ix.n : 4096;
      // the sample's masks are kept together (32 KB, read through L1): gathered
      // from the column, each was a sector of its own behind a 64-bit division
      // (the preparation kernel: 96 us for 5,000 subset filters, 18 us so; 110 us
      // for 777 boolean and range filters, 62 us so)
      int hits = 0;
      if (f.kind == JAG_F_SUBSET) {
#pragma unroll 8
        for (int j = lane; j < (int)S; j += 32) hits += (f.payload & __ldg(ix.mask_sample + j)) == f.payload ? 1 : 0;
      } else if (m <= 5) {   // the truth table in a register
        uint32_t word = tt[0];
        for (int b = 1; b < (1 << m) / 8; ++b) word |= (uint32_t)tt[b] << (8 * b);
#pragma unroll 8
        for (int j = lane; j < (int)S; j += 32)
          hits += (word >> compress_bits(__ldg(ix.mask_sample + j), f.payload)) & 1u;
      } else {
        for (int j = lane; j < (int)S; j += 32) {
          const uint32_t s = compress_bits(__ldg(ix.mask_sample + j), f.payload);
          hits += (tt[s >> 3] >> (s & 7)) & 1;
        }
      }
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) hits += __shfl_xor_sync(kFull, hits, o);
      pl.est = hits;
      if (s0 > 0 && (int64_t)hits * ix.n < s0 * S) pl.route = kRouteList;
    }
  }
  return true;
}

}  // namespace jag
