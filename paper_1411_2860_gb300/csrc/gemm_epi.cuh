// Epilogue helpers shared by the reduced-GEMM kernels (gemm_tc.cu, gemm_cg2.cu):
// the expansion of a gradient product's components back to samples, written
// straight from the registers that tcgen05.ld filled (ExpandArgs, common.hpp).
#pragma once

#include <cuda_bf16.h>

#include <type_traits>

#include "common.hpp"
#include "tc.cuh"

namespace pj {
namespace {

// Where entry e of the expansion's coefficient table (Cs: t (l+1) + p for mode 1, Ds:
// p 8 + t for mode 2) sits in a Coef8.
__device__ __forceinline__ int expand_c8_index(const ExpandArgs& ex, int e) {
  return ex.mode == 1 ? (e % ex.lp1) * 8 + e / ex.lp1 : e;
}

// Element stores of a chunk: NR accumulator values of output column j (one per row from
// i0 on), for outputs whose rows TMA cannot address.  A chunk whose rows all exist is
// walked by pointer; tested and addressed one by one, the stores took the epilogue
// warps (one per scheduler) three times the instructions.  add: atomic additions.
template <int NR, typename Op>
__device__ __forceinline__ void walk_rows(const uint32_t (&r)[NR], int64_t ldy, int i0, int M, Op op) {
  if (i0 + NR <= M) {
    int64_t off = 0;
#pragma unroll
    for (int u = 0; u < NR; ++u, off += ldy) op(off, __uint_as_float(r[u]));
  } else {
#pragma unroll
    for (int u = 0; u < NR; ++u)
      if (i0 + u < M) op(u * ldy, __uint_as_float(r[u]));
  }
}
template <int NR>
__device__ __forceinline__ void store_rows(const uint32_t (&r)[NR], void* Yv, int64_t ldy, bool out_bf16, bool add, int i0,
                                           int M, int j) {
  if (out_bf16) {
    __nv_bfloat16* Y = static_cast<__nv_bfloat16*>(Yv) + i0 * ldy + j;
    walk_rows(r, ldy, i0, M, [&](int64_t off, float v) { Y[off] = __float2bfloat16_rn(v); });
  } else if (add) {
    float* Y = static_cast<float*>(Yv) + i0 * ldy + j;
    walk_rows(r, ldy, i0, M, [&](int64_t off, float v) { atomicAdd(Y + off, v); });
  } else {
    float* Y = static_cast<float*>(Yv) + i0 * ldy + j;
    walk_rows(r, ldy, i0, M, [&](int64_t off, float v) { __stcs(Y + off, v); });
  }
}

// The same for a lowered correlation: element (i, j) is output sample i * 128 + j of a
// phase, `stride` floats apart, below `limit`.
template <int NR>
__device__ __forceinline__ void store_samples(const uint32_t (&r)[NR], float* Y, int64_t stride, int64_t limit,
                                              int i0, int j, bool jok) {
#pragma unroll
  for (int u = 0; u < NR; ++u) {
    const int64_t flat = static_cast<int64_t>(i0 + u) * 128 + j;
    if (jok && flat < limit) __stcs(Y + flat * stride, __uint_as_float(r[u]));
  }
}

template <bool kBF16>
__device__ __forceinline__ void store_run(void* out, int64_t off, const float (&y)[8], int n, int per) {
  if (kBF16) {
    __nv_bfloat16* o = static_cast<__nv_bfloat16*>(out) + off;
    if (n == per && per >= 2) {
      uint32_t w[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        w[k] = uint32_t(__bfloat16_as_ushort(__float2bfloat16_rn(y[2 * k]))) |
               (uint32_t(__bfloat16_as_ushort(__float2bfloat16_rn(y[2 * k + 1]))) << 16);
      if (per == 8) *reinterpret_cast<uint4*>(o) = make_uint4(w[0], w[1], w[2], w[3]);
      else if (per == 4) *reinterpret_cast<uint2*>(o) = make_uint2(w[0], w[1]);
      else *reinterpret_cast<uint32_t*>(o) = w[0];
    } else {
#pragma unroll
      for (int t = 0; t < 8; ++t)
        if (t < n) o[t] = __float2bfloat16_rn(y[t]);
    }
  } else {
    float* o = static_cast<float*>(out) + off;
    if (n == per && per >= 4) {
      reinterpret_cast<float4*>(o)[0] = make_float4(y[0], y[1], y[2], y[3]);
      if (per == 8) reinterpret_cast<float4*>(o)[1] = make_float4(y[4], y[5], y[6], y[7]);
    } else if (n == per && per == 2) {
      *reinterpret_cast<float2*>(o) = make_float2(y[0], y[1]);
    } else {
#pragma unroll
      for (int t = 0; t < 8; ++t)
        if (t < n) o[t] = y[t];
    }
  }
}

// The expansion runs over 8 TMEM columns at a time in a loop that is not
// unrolled: a fully unrolled 32-column step is several KB of straight-line
// code per (mode, l+1, dtype), and with one epilogue warp per scheduler the
// instruction fetch, not the stores, then bounds the epilogue.

// Mode 1 (components on the TMEM lanes): lane `lane` holds component p = kk % LP1
// of group g = kk / LP1 for 8 output rows i0 .. i0 + 7; the LP1 lanes of a group
// exchange their values and each writes 8 / LP1 of the group's 8 samples per row.
template <int LP1, bool kBF16>
__device__ __forceinline__ void expand_rows_x8(const uint32_t (&r)[8], int lane, int kk, int Kp, int i0, int M,
                                               const ExpandArgs& ex, const float* sc) {
  constexpr int per = 8 / LP1;
  const int g = kk / LP1, pc = kk - g * LP1, t0 = pc * per;
  const int lbase = lane & ~(LP1 - 1);
  const int64_t col0 = static_cast<int64_t>(g) * 8 + t0;
  void* const out = ex.out;
  const int64_t ld = ex.ld;
  int n = static_cast<int>(ex.K - col0);
  n = kk < Kp ? (n < 0 ? 0 : (n > per ? per : n)) : 0;
  float cf[per][LP1];
#pragma unroll
  for (int t = 0; t < per; ++t)
#pragma unroll
    for (int pp = 0; pp < LP1; ++pp) cf[t][pp] = sc[(t0 + t) * LP1 + pp];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    float v[LP1];
#pragma unroll
    for (int pp = 0; pp < LP1; ++pp) v[pp] = __shfl_sync(0xffffffffu, __uint_as_float(r[u]), lbase + pp);
    if (n > 0 && i0 + u < M) {
      float y[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        float acc = 0.0f;
        if (t < per) {
#pragma unroll
          for (int pp = 0; pp < LP1; ++pp) acc = fmaf(v[pp], cf[t < per ? t : 0][pp], acc);
        }
        y[t] = acc;
      }
      store_run<kBF16>(out, static_cast<int64_t>(i0 + u) * ld + col0, y, n, per);
    }
  }
}

// Mode 2 (components on the TMEM columns): this thread holds components
// k0 .. k0 + 7 of output column j; each group of LP1 gives 8 sample rows.
// The 8 x LP1 coefficients sit in registers for LP1 <= 4 (read from shared
// memory per use for LP1 = 8, where they would take 64 registers).
template <int LP1, bool kBF16>
__device__ __forceinline__ void expand_cols_x8(const uint32_t (&r)[8], int k0, int Kp, int j,
                                               const ExpandArgs& ex, const float* sd) {
  constexpr bool kRegs = LP1 <= 4;
  float cr[kRegs ? LP1 * 8 : 1];
  if (kRegs) {
#pragma unroll
    for (int e = 0; e < (kRegs ? LP1 * 8 : 1); ++e) cr[e] = sd[e];
  }
  const int64_t ld = ex.ld, K = ex.K;
  auto* out = static_cast<typename std::conditional<kBF16, __nv_bfloat16, float>::type*>(ex.out);
#pragma unroll
  for (int a = 0; a < 8 / LP1; ++a) {
    const int kk = k0 + a * LP1;
    if (kk >= Kp) break;
    const int64_t row0 = static_cast<int64_t>(kk / LP1) * 8;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      if (row0 + t >= K) break;
      float acc = 0.0f;
#pragma unroll
      for (int pp = 0; pp < LP1; ++pp)
        acc = fmaf(kRegs ? cr[kRegs ? pp * 8 + t : 0] : sd[pp * 8 + t], __uint_as_float(r[a * LP1 + pp]), acc);
      const int64_t off = (row0 + t) * ld + j;
      if (kBF16)
        out[off] = __float2bfloat16_rn(acc);
      else
        out[off] = acc;
    }
  }
}

// Mode 1 on a chunk of 8 rows and a warp of groups that all exist, walked by pointer with
// the coefficients held by the caller's loop.  With an address, two bounds and the
// coefficients' shared loads per row, the instructions of the eight epilogue warps bound
// the expansion: the backward of an 8192 x 4096 x 4096 BF16 layer (l+1 = 2) takes 147 us
// so, 152 before, and a 2048 x 2048 x 4096 FP32 one (l+1 = 8) 105 us, 113 before.  Not for
// l+1 = 1, whose rows exchange nothing (190 against 184 us), not for BF16 at l+1 = 8, whose
// lanes store two bytes each (526 against 520 us), nor for mode 2, whose stores in bursts
// slowed the products they overlap (l+1 = 4: 282 against 278 us).
template <int LP1, bool kBF16>
__device__ __forceinline__ void expand_rows_full(const uint32_t (&r)[8], int lbase, const float (&cf)[8 / LP1][LP1],
                                                 void* out, int64_t off, int64_t ld) {
  constexpr int per = 8 / LP1;
#pragma unroll
  for (int u = 0; u < 8; ++u, off += ld) {
    float v[LP1], y[8];
#pragma unroll
    for (int pp = 0; pp < LP1; ++pp) v[pp] = __shfl_sync(0xffffffffu, __uint_as_float(r[u]), lbase + pp);
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      y[t] = 0.0f;
      if (t < per) {
#pragma unroll
        for (int pp = 0; pp < LP1; ++pp) y[t] = fmaf(v[pp], cf[t < per ? t : 0][pp], y[t]);
      }
    }
    store_run<kBF16>(out, off, y, per, per);
  }
}

template <int LP1, bool kBF16>
__device__ __noinline__ void expand_tile_cols(uint32_t taddr, int ncols, const ExpandArgs ex, const float* sc,
                                              int lane, int kk_lane, int Kp, int i0, int M, int j, bool jok) {
  uint32_t r[8];
  constexpr bool kWhole = LP1 > 1 && !(LP1 == 8 && kBF16);
  if constexpr (kWhole) {
    if (ex.mode == 1) {
      constexpr int per = 8 / LP1;
      const int g = kk_lane / LP1, t0 = (kk_lane - g * LP1) * per;
      const int64_t col0 = static_cast<int64_t>(g) * 8 + t0;
      const bool whole = __all_sync(0xffffffffu, kk_lane < Kp && col0 + per <= ex.K);
      float cf[per][LP1];
#pragma unroll
      for (int t = 0; t < per; ++t)
#pragma unroll
        for (int pp = 0; pp < LP1; ++pp) cf[t][pp] = sc[(t0 + t) * LP1 + pp];
#pragma unroll 1
      for (int c = 0; c < ncols && i0 + c < M; c += 8) {
        tmem_ld_x8(taddr + c, r);
        tmem_wait_ld();
        if (whole && i0 + c + 8 <= M)
          expand_rows_full<LP1, kBF16>(r, lane & ~(LP1 - 1), cf, ex.out, (i0 + c) * ex.ld + col0, ex.ld);
        else
          expand_rows_x8<LP1, kBF16>(r, lane, kk_lane, Kp, i0 + c, M, ex, sc);
      }
      return;
    }
  }
#pragma unroll 1
  for (int c = 0; c < ncols; c += 8) {
    tmem_ld_x8(taddr + c, r);
    tmem_wait_ld();
    if (!kWhole && ex.mode == 1) {
      if (i0 + c < M) expand_rows_x8<LP1, kBF16>(r, lane, kk_lane, Kp, i0 + c, M, ex, sc);
    } else if (jok && i0 + c < Kp) {
      expand_cols_x8<LP1, kBF16>(r, i0 + c, Kp, j, ex, sc);
    }
  }
}

// Expands `ncols` (a multiple of 8) TMEM columns starting at taddr (this warp's
// lane quadrant), whose first column is output row i0 (mode 1: the lanes hold
// components kk_lane of Kp) or component i0 of Kp (mode 2: the lanes hold output
// column j).
__device__ __forceinline__ void expand_tile(uint32_t taddr, int ncols, const ExpandArgs& ex, const float* s_coef,
                                            int lane, int kk_lane, int Kp, int i0, int M, int j, bool jok) {
  if (ex.out_bf16) {
    switch (ex.lp1) {
      case 1: expand_tile_cols<1, true>(taddr, ncols, ex, s_coef, lane, kk_lane, Kp, i0, M, j, jok); break;
      case 2: expand_tile_cols<2, true>(taddr, ncols, ex, s_coef, lane, kk_lane, Kp, i0, M, j, jok); break;
      case 4: expand_tile_cols<4, true>(taddr, ncols, ex, s_coef, lane, kk_lane, Kp, i0, M, j, jok); break;
      default: expand_tile_cols<8, true>(taddr, ncols, ex, s_coef, lane, kk_lane, Kp, i0, M, j, jok); break;
    }
  } else {
    switch (ex.lp1) {
      case 1: expand_tile_cols<1, false>(taddr, ncols, ex, s_coef, lane, kk_lane, Kp, i0, M, j, jok); break;
      case 2: expand_tile_cols<2, false>(taddr, ncols, ex, s_coef, lane, kk_lane, Kp, i0, M, j, jok); break;
      case 4: expand_tile_cols<4, false>(taddr, ncols, ex, s_coef, lane, kk_lane, Kp, i0, M, j, jok); break;
      default: expand_tile_cols<8, false>(taddr, ncols, ex, s_coef, lane, kk_lane, Kp, i0, M, j, jok); break;
    }
  }
}

}  // namespace
}  // namespace pj
