// Projection kernels (Sec. III-B): every group of L consecutive inner-dimension
// values of a row of A is multiplied by the kept columns of C, every group of
// a column of B by the kept rows of D (Fig. 5 and its description), and the
// CONV signal / templates are projected per group (Fig. 6, Eq. 11-12).
// These kernels stream HBM; the arithmetic is FP32 (FP64 for the double path).
#include <cuda_bf16.h>

#include <atomic>
#include <type_traits>

#include "common.hpp"
#include "pdl.cuh"

namespace pj {
namespace {

__device__ __forceinline__ float load_as_float(const float* p) { return __ldg(p); }
__device__ __forceinline__ float load_as_float(const __nv_bfloat16* p) { return __bfloat162float(*p); }

__device__ __forceinline__ uint16_t bf16_bits(float x) {
  return __bfloat16_as_ushort(__float2bfloat16_rn(x));
}
__device__ __forceinline__ float bf16_value(uint16_t b) {
  return __bfloat162float(__ushort_as_bfloat16(b));
}

// Component order.  Every group of L consecutive inner-dimension values is
// projected on its own (the block-diagonal C_N, D_N of Eq. 15; the top-level
// block is a multiple of L, so no group straddles two blocks), and component
// p of global group gg sits at column gg * (l+1) + p of the reduced inner
// dimension.  A short last group (K not a multiple of L) is zero-extended.

// Widest aligned stores for a run of n BF16 values starting at dst, where dst
// is aligned to 2 * n bytes for n a power of two (n <= 16).
__device__ __forceinline__ void store_run(uint16_t* dst, const uint16_t* v, int n) {
  if (n == 8) {
    uint4 q;
    q.x = v[0] | (uint32_t(v[1]) << 16);
    q.y = v[2] | (uint32_t(v[3]) << 16);
    q.z = v[4] | (uint32_t(v[5]) << 16);
    q.w = v[6] | (uint32_t(v[7]) << 16);
    *reinterpret_cast<uint4*>(dst) = q;
  } else if (n == 4) {
    uint2 q;
    q.x = v[0] | (uint32_t(v[1]) << 16);
    q.y = v[2] | (uint32_t(v[3]) << 16);
    *reinterpret_cast<uint2*>(dst) = q;
  } else if (n == 2) {
    *reinterpret_cast<uint32_t*>(dst) = v[0] | (uint32_t(v[1]) << 16);
  } else {
    for (int i = 0; i < n; ++i) dst[i] = v[i];
  }
}

// The first n (<= 8) of v at dst: one vector store when n is 1, 2, 4 or 8 (dst
// aligned to 2 n bytes), else element stores with compile-time indices (v
// stays in registers).
__device__ __forceinline__ void store_upto8(uint16_t* dst, const uint16_t (&v)[8], int n) {
  if (n == 8 || n == 4 || n == 2) {
    store_run(dst, v, n);
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (i < n) dst[i] = v[i];
  }
}

// Zeroes elements [c0, c1) of a BF16 row whose start is 16-byte aligned; c1 is
// a multiple of 8 (the padded reduced dimension is a multiple of 64).
__device__ __forceinline__ void zero_run(uint16_t* row, int64_t c0, int64_t c1) {
  int64_t c = c0;
  for (; c < c1 && (c & 7) != 0; ++c) row[c] = 0;
  for (; c < c1; c += 8) *reinterpret_cast<uint4*>(row + c) = make_uint4(0u, 0u, 0u, 0u);
}

// ---- split parts (see gemm_tiered) ----------------------------------------
struct StoreUpto8 {
  __device__ __forceinline__ void operator()(uint16_t* dst, const uint16_t (&v)[8], int n) const {
    store_upto8(dst, v, n);
  }
};

// Component p of group gg, one value at a time (general L).
__device__ __forceinline__ void split_part_one(uint16_t* row, int64_t gg, int p, uint16_t h, uint16_t l, int lp1,
                                               int tl, int64_t Kp_pad, int64_t Kt_pad) {
  if (tl >= lp1) {
    row[Kp_pad + gg * lp1 + p] = l;
  } else if (p < tl) {
    row[Kp_pad + gg * tl + p] = h;
    row[Kp_pad + Kt_pad + gg * tl + p] = l;
  }
}

// Zero padding of every segment of one output row.
// from: the first component no other thread writes (at least NG (l+1); plain split only).
__device__ __forceinline__ void zero_split_rows(uint16_t* row, int64_t NG, int lp1, int nsplit, int tl,
                                                int64_t Kp_pad, int64_t Kt_pad, int64_t from = 0) {
  if (nsplit > 1 && tl < lp1) {
    zero_run(row, NG * lp1, Kp_pad);
    zero_run(row + Kp_pad, NG * tl, Kt_pad);
    zero_run(row + Kp_pad + Kt_pad, NG * tl, Kt_pad);
  } else {
    const int64_t c0 = from > NG * lp1 ? from : NG * lp1;
    for (int sg = 0; sg < nsplit; ++sg) zero_run(row + sg * Kp_pad, c0, Kp_pad);
  }
}

// 4-byte asynchronous copy global -> shared (bytes = 4, or 0 to write zeros).
__device__ __forceinline__ void cp_async4(float* dst, const void* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                   static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// Waits until at most N of this thread's groups are pending.
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ---- L = 8: components in pairs ------------------------------------------
// The l+1 components of one group of eight inputs: acc[k] holds components 2k
// and 2k+1, each one FMA chain over the inputs in order (paired FMAs), with the
// kept basis values at c[t * 8 + q] (element t, component q; zero past l+1;
// 16-byte aligned shared memory, read as 16-byte broadcasts).
template <int LP1>
__device__ __forceinline__ void group8_pairs(const float (&x)[8], const float* c, float2 (&acc)[(LP1 + 1) / 2]) {
  constexpr int NP = (LP1 + 1) / 2;
#pragma unroll
  for (int k = 0; k < NP; ++k) acc[k] = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    const float2 xx = make_float2(x[t], x[t]);
    const float4 c0 = *reinterpret_cast<const float4*>(c + t * 8);
    acc[0] = __ffma2_rn(xx, make_float2(c0.x, c0.y), acc[0]);
    if constexpr (NP > 1) acc[NP > 1 ? 1 : 0] = __ffma2_rn(xx, make_float2(c0.z, c0.w), acc[NP > 1 ? 1 : 0]);
    if constexpr (NP > 2) {
      const float4 c1 = *reinterpret_cast<const float4*>(c + t * 8 + 4);
      acc[NP > 2 ? 2 : 0] = __ffma2_rn(xx, make_float2(c1.x, c1.y), acc[NP > 2 ? 2 : 0]);
      if constexpr (NP > 3) acc[NP > 3 ? 3 : 0] = __ffma2_rn(xx, make_float2(c1.z, c1.w), acc[NP > 3 ? 3 : 0]);
    }
  }
}

// The same for two groups (the same chains, so the same bits): each read of the basis
// values feeds both.
template <int LP1>
__device__ __forceinline__ void group8_pairs2(const float (&x)[8], const float (&y)[8], const float* c,
                                              float2 (&ax)[(LP1 + 1) / 2], float2 (&ay)[(LP1 + 1) / 2]) {
  constexpr int NP = (LP1 + 1) / 2;
#pragma unroll
  for (int k = 0; k < NP; ++k) ax[k] = ay[k] = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    const float2 xx = make_float2(x[t], x[t]), yy = make_float2(y[t], y[t]);
#pragma unroll
    for (int h = 0; h < (NP + 1) / 2; ++h) {
      const float4 v = *reinterpret_cast<const float4*>(c + t * 8 + 4 * h);
      ax[2 * h] = __ffma2_rn(xx, make_float2(v.x, v.y), ax[2 * h]);
      ay[2 * h] = __ffma2_rn(yy, make_float2(v.x, v.y), ay[2 * h]);
      if (2 * h + 1 < NP) {
        ax[(2 * h + 1) % NP] = __ffma2_rn(xx, make_float2(v.z, v.w), ax[(2 * h + 1) % NP]);
        ay[(2 * h + 1) % NP] = __ffma2_rn(yy, make_float2(v.z, v.w), ay[(2 * h + 1) % NP]);
      }
    }
  }
}

// hi = bf16(component) and lo = bf16(component - hi), two components per conversion.
template <int LP1>
__device__ __forceinline__ void split_bf16(const float2 (&acc)[(LP1 + 1) / 2], uint16_t (&hi)[8], uint16_t (&lo)[8]) {
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    hi[q] = 0;
    lo[q] = 0;
  }
#pragma unroll
  for (int k = 0; k < (LP1 + 1) / 2; ++k) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(acc[k].x, acc[k].y);
    const float2 hf = __bfloat1622float2(h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(acc[k].x - hf.x, acc[k].y - hf.y);
    hi[2 * k] = __bfloat16_as_ushort(h.x);
    lo[2 * k] = __bfloat16_as_ushort(l.x);
    if (2 * k + 1 < LP1) {
      hi[2 * k + 1] = __bfloat16_as_ushort(h.y);
      lo[2 * k + 1] = __bfloat16_as_ushort(l.y);
    }
  }
}

// Stages the kept basis values of an L = 8 job as c[t * 8 + q] (zero past l+1)
// from the layout `at(t, q)` gives; every thread of the block calls it.
template <typename At>
__device__ __forceinline__ void stage_coef8(float* c, int lp1, At at) {
  for (int k = threadIdx.x; k < 64; k += blockDim.x) {
    const int t = k >> 3, q = k & 7;
    c[k] = q < lp1 ? at(t, q) : 0.0f;
  }
}

// ---- rows of A -> A_c (BF16, hi [+ lo]) -----------------------------------
// L = 8: one warp per two (row, run of 32 groups) units, both runs loaded before
// any arithmetic.  For each run the warp reads its 256
// inputs with lane-strided loads (each instruction reads 128 or 64 contiguous
// bytes, whatever the row's alignment), transposes them through a padded
// per-warp shared buffer (element e at e + e / 32: conflict-free both ways), and
// lane g projects group g of the run, writing its l+1 contiguous components.
// Other L (<= 64): one thread per (row, group), inputs staged in local memory.
// The thread of group 0 of a row also zeroes the row's padding columns.
// Every thread of the block reaches the one __syncthreads.
constexpr int kRowRun = 32;                         // groups per run (L = 8)
constexpr int kRowUnits = 2;                        // runs per warp, loaded together (2 consecutive: <= 2 rows)
constexpr int kRowBuf = 8 * kRowRun + 8;            // padded floats per run

template <int LP1>
__device__ __forceinline__ void rows_group8(const RowsJob& J, uint16_t* row, int64_t gg, const float (&x)[8],
                                            const float* sC) {
  float2 acc[(LP1 + 1) / 2];
  group8_pairs<LP1>(x, sC, acc);
  uint16_t hi[8], lo[8];
  split_bf16<LP1>(acc, hi, lo);
  store_upto8(row + gg * LP1, hi, LP1);
  if (J.nsplit > 1) store_split_part(row, gg, hi, lo, LP1, J.tl, J.Kp_pad, J.Kt_pad, StoreUpto8{});
}

// l+1 in {3, 5, 6, 7} without a tiered split: a run's 32 groups of components are one
// span of the row (64 (l+1) bytes from a 16-byte boundary), staged in the run's
// buffer (which the warp has read) and stored in 16-byte chunks clipped to the
// segment; lanes past the last group carry zeros.  Every lane of the warp takes part.
template <int LP1>
__device__ __forceinline__ void rows_span_odd(const RowsJob& J, const float (&x)[8], const float* sC, uint16_t* st,
                                              uint16_t* o0, int64_t room, int lane) {
  float2 acc[(LP1 + 1) / 2];
  group8_pairs<LP1>(x, sC, acc);
  uint16_t hi[8], lo[8];
  split_bf16<LP1>(acc, hi, lo);
  const int nch = static_cast<int>((room < 64 * LP1 ? room : 64 * LP1) / 16);
#pragma unroll 1
  for (int part = 0; part < (J.nsplit > 1 ? 2 : 1); ++part) {
    __syncwarp();   // the run's inputs (or the previous part) are read
#pragma unroll
    for (int p = 0; p < LP1; ++p) st[lane * LP1 + p] = part ? lo[p] : hi[p];
    __syncwarp();
    for (int k = lane; k < nch; k += 32)
      reinterpret_cast<uint4*>(o0 + part * J.Kp_pad)[k] = reinterpret_cast<const uint4*>(st)[k];
  }
}

// One group's components at the row's group gg, plain or with every lo term.
template <int LP1>
__device__ __forceinline__ void rows_store(uint16_t* row, int64_t gg, const float2 (&acc)[(LP1 + 1) / 2], bool two,
                                           int64_t Kp_pad) {
  uint16_t hi[8], lo[8];
  split_bf16<LP1>(acc, hi, lo);
  store_upto8(row + gg * LP1, hi, LP1);
  if (two) store_upto8(row + Kp_pad + gg * LP1, lo, LP1);
}

// Group gx of row rx and group gy of row ry (NULL: not stored), l+1 in {1, 2, 4, 8}.
template <int LP1>
__device__ __forceinline__ void rows_two(uint16_t* rx, int64_t gx, const float (&x)[8], uint16_t* ry, int64_t gy,
                                         const float (&y)[8], const float* sC, bool two, int64_t Kp_pad) {
  float2 ax[(LP1 + 1) / 2], ay[(LP1 + 1) / 2];
  group8_pairs2<LP1>(x, y, sC, ax, ay);
  if (rx) rows_store<LP1>(rx, gx, ax, two, Kp_pad);
  if (ry) rows_store<LP1>(ry, gy, ay, two, Kp_pad);
}

// Projects and stores run `run` of row i from buffer `buf` and, when live1, run `run1` of
// row i1 from buf1 (which may be overwritten).  Every lane of the warp takes part.
template <int LP1>
__device__ __forceinline__ void rows_two_runs(const RowsJob& J, int64_t i, int64_t run, float* buf, bool live1,
                                              int64_t i1, int64_t run1, float* buf1, const float* sC) {
  const int lane = threadIdx.x & 31;
  const int64_t g0 = run * kRowRun + lane, g1 = run1 * kRowRun + lane;
  uint16_t* const row0 = J.Ac + i * J.pitch;
  uint16_t* const row1 = J.Ac + i1 * J.pitch;
  const bool tiered = J.nsplit > 1 && J.tl < LP1;
  constexpr bool kOdd = LP1 == 3 || LP1 == 5 || LP1 == 6 || LP1 == 7;
  float x[8], y[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    x[t] = buf[8 * lane + t + (lane >> 2)];
    y[t] = buf1[8 * lane + t + (lane >> 2)];
  }
  if (tiered) {
    if (g0 < J.NG) rows_group8<LP1>(J, row0, g0, x, sC);
    if (live1 && g1 < J.NG) rows_group8<LP1>(J, row1, g1, y, sC);
  } else if constexpr (kOdd) {
    rows_span_odd<LP1>(J, x, sC, reinterpret_cast<uint16_t*>(buf), row0 + run * (kRowRun * LP1),
                       2 * (J.Kp_pad - run * (kRowRun * LP1)), lane);
    if (live1)   // the same for the whole warp
      rows_span_odd<LP1>(J, y, sC, reinterpret_cast<uint16_t*>(buf1), row1 + run1 * (kRowRun * LP1),
                         2 * (J.Kp_pad - run1 * (kRowRun * LP1)), lane);
  } else {
    rows_two<LP1>(g0 < J.NG ? row0 : nullptr, g0, x, live1 && g1 < J.NG ? row1 : nullptr, g1, y, sC, J.nsplit > 1,
                  J.Kp_pad);
  }
  if (g0 == 0) zero_split_rows(row0, J.NG, LP1, J.nsplit, J.tl, J.Kp_pad, J.Kt_pad);
  if (live1 && g1 == 0) zero_split_rows(row1, J.NG, LP1, J.nsplit, J.tl, J.Kp_pad, J.Kt_pad);
}

// The runs of one warp, w0 .. w0 + n - 1 (consecutive runs of a row, then of the next),
// two at a time.  FP32: a ring of kRowRing pairs filled by 4-byte asynchronous copies
// (rows start anywhere, and the copies need no registers), so a warp keeps two pairs in
// flight while it projects a third.  With one pair per warp, loaded, projected and
// stored before the block left, the kernel moved 0.56 of the copy rate however few
// instructions it took.  BF16 (rows may start at odd 2-byte offsets): plain loads, one
// pair at a time.
constexpr int kRowRing = 3;
constexpr int kRowsSmem = 8 * kRowRing * kRowUnits * kRowBuf * 4;   // bytes a block of either kind reserves (L = 8)

template <typename InT, int LP1, bool kArg>
__device__ __forceinline__ void rows_body8(const RowsJob& J, int64_t w0, float* sC, float* sX) {
  static_assert(kRowUnits == 2, "runs go in pairs");
  constexpr bool kAsync = sizeof(InT) == 4;
  const int lane = threadIdx.x & 31;
  const int64_t nrun = (J.NG + kRowRun - 1) / kRowRun;
  const int64_t units = J.M * nrun;
  const int n = static_cast<int>(units - w0 < J.upw ? (units > w0 ? units - w0 : 0) : J.upw);
  // (one 32-bit division per warp: 64-bit ones per run were more instructions than the
  // projection itself)
  int64_t li = units < (int64_t(1) << 32) ? static_cast<uint32_t>(w0) / static_cast<uint32_t>(nrun) : w0 / nrun;
  int64_t lr = w0 - li * nrun;      // the next run to load ...
  int64_t pi = li, pr = lr;         // ... and to project
  float* const bufs = sX + (threadIdx.x >> 5) * (kRowRing * kRowUnits * kRowBuf);
  auto load_run = [&](float* buf, bool live) {
    const InT* a = static_cast<const InT*>(J.A) + (live ? li * J.lda + lr * (8 * kRowRun) : 0);
    const int64_t left = live ? J.K - lr * (8 * kRowRun) : 0;
    const int nk = static_cast<int>(left < 8 * kRowRun ? left : 8 * kRowRun);
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const bool in = s * 32 + lane < nk;
      if constexpr (kAsync)
        cp_async4(buf + s * 33 + lane, in ? a + s * 32 + lane : a, in ? 4 : 0);
      else
        buf[s * 33 + lane] = in ? load_as_float(a + s * 32 + lane) : 0.0f;
    }
    if (++lr == nrun) {
      lr = 0;
      ++li;
    }
  };
  auto load_pair = [&](int k) {   // runs 2k and 2k + 1 into ring slot k % kRowRing
    if (2 * k < n) {
      float* b = bufs + (k % kRowRing) * (kRowUnits * kRowBuf);
      load_run(b, true);
      load_run(b + kRowBuf, 2 * k + 1 < n);
    }
    if constexpr (kAsync) cp_async_commit();
  };
  if constexpr (kAsync)
    for (int k = 0; k < kRowRing - 1; ++k) load_pair(k);
  if (!kArg) stage_coef8(sC, LP1, [&](int t, int q) { return J.Cs[t * LP1 + q]; });
  __syncthreads();
#pragma unroll 1
  for (int k = 0; 2 * k < n; ++k) {
    if constexpr (kAsync) {
      load_pair(k + kRowRing - 1);   // into the slot projected last
      cp_async_wait<kRowRing - 1>();
    } else {
      load_pair(k);
    }
    __syncwarp();
    const int64_t i0 = pi, r0 = pr;
    if (++pr == nrun) {
      pr = 0;
      ++pi;
    }
    float* b = bufs + (k % kRowRing) * (kRowUnits * kRowBuf);
    rows_two_runs<LP1>(J, i0, r0, b, 2 * k + 1 < n, pi, pr, b + kRowBuf, sC);
    if (++pr == nrun) {
      pr = 0;
      ++pi;
    }
    __syncwarp();   // the pair's buffers are read
  }
}

template <typename InT>
__device__ __forceinline__ void rows_body_any(const RowsJob& J, int64_t e, float* sC) {
  const bool live = e < J.M * J.NG;
  const int64_t i = live ? e / J.NG : 0, gg = live ? e - i * J.NG : 0;
  const int L = J.L, lp1 = J.lp1;
  const InT* A = static_cast<const InT*>(J.A);
  const int n = static_cast<int>(J.K - gg * L < L ? J.K - gg * L : L);
  for (int k = threadIdx.x; k < L * lp1; k += blockDim.x) sC[k] = J.Cs[k];
  __syncthreads();
  if (!live) return;
  uint16_t* out = J.Ac + i * J.pitch + gg * lp1;
  const InT* a = A + i * J.lda + gg * L;
  uint16_t* row = J.Ac + i * J.pitch;
  float xs[64];
  for (int t = 0; t < L; ++t) xs[t] = t < n ? load_as_float(a + t) : 0.0f;
  for (int p = 0; p < lp1; ++p) {
    float acc = 0.0f;
    for (int t = 0; t < L; ++t) acc = fmaf(xs[t], sC[t * lp1 + p], acc);
    const uint16_t h = bf16_bits(acc);
    out[p] = h;
    if (J.nsplit > 1) split_part_one(row, gg, p, h, bf16_bits(acc - bf16_value(h)), lp1, J.tl, J.Kp_pad, J.Kt_pad);
  }
  if (gg == 0) zero_split_rows(row, J.NG, lp1, J.nsplit, J.tl, J.Kp_pad, J.Kt_pad);
}

// LP = 0: any group size, thread t of block b handles unit b * 256 + t; LP > 0: groups
// of 8 with l+1 = LP, warp units (b * 8 + t / 32) * upw onwards.  One
// instantiation per l+1: with a switch over all of them in one kernel the column paths
// shared one register allocation and spilled.
template <typename InT, int LP, bool kArg>
__device__ __forceinline__ void rows_body(const RowsJob& J, int64_t b, float* sC, float* sX) {
  if constexpr (LP > 0)
    rows_body8<InT, LP, kArg>(J, (b * 8 + (threadIdx.x >> 5)) * J.upw, sC, sX);
  else
    rows_body_any<InT>(J, b * blockDim.x + threadIdx.x, sC);
}

// Arguments of a single operand's launch: the kept vectors (kArg; else they are in the
// job's table) and the call's error word when this is the call's first kernel.
struct SideArgs {
  Coef8 c8;
  int* clear;
};

template <bool kArg>
__device__ __forceinline__ void side_begin(const SideArgs& a, float* sC) {
  if (kArg && threadIdx.x < 64) sC[threadIdx.x] = a.c8.c[(threadIdx.x & 7) * 8 + (threadIdx.x >> 3)];   // [t * 8 + q]
  pdl_begin();
  if (a.clear && blockIdx.x == 0 && threadIdx.x == 0) *a.clear = 0;
}

template <typename InT, int LP, bool kArg>
__global__ void __launch_bounds__(256, LP ? 4 : 1) project_rows_kernel(const __grid_constant__ RowsJob J,
                                                           const __grid_constant__ SideArgs a) {
  __shared__ __align__(16) float sC[LP ? 64 : 64 * 64];
  extern __shared__ __align__(16) float sX[];   // kRowsSmem bytes for groups of 8
  side_begin<kArg>(a, sC);
  rows_body<InT, LP, kArg>(J, blockIdx.x, sC, sX);
}

template <typename InT, int LP>
__global__ void __launch_bounds__(256, LP ? 4 : 1) project_rows_jobs_kernel(const RowsJob* __restrict__ jobs,
                                                                const int* __restrict__ job_of) {
  __shared__ __align__(16) float sC[LP ? 64 : 64 * 64];
  extern __shared__ __align__(16) float sX[];   // kRowsSmem bytes for groups of 8
  pdl_begin();
  const RowsJob J = jobs[job_of[blockIdx.x]];   // a copy: read once, not again after every store
  rows_body<InT, LP, false>(J, static_cast<int64_t>(blockIdx.x) - J.block0, sC, sX);
}

// ---- columns of B -> B_d stored transposed (N x pitch, K-major) -----------
// One thread per (column, 4 consecutive groups): the reads of one row of B are
// coalesced across the block's columns; each thread writes 4 (l+1) contiguous
// components of its column with 16-byte stores.  The threads of the first
// group quad also zero their column's padding.
constexpr int kColGroups = 4;

// The components the quads of a column write: whole quads when they fit the row.
template <int LP1>
__device__ __forceinline__ int64_t staged_end(const ColsJob& J) {
  const int64_t end = (J.NG + kColGroups - 1) / kColGroups * kColGroups * LP1;
  return end <= J.Kp_pad ? end : J.NG * LP1;
}

// L = 8, l+1 = 4 or 8, four whole groups: the warp's 32 columns stage their
// runs in `stage` (4 KB per warp) and write them row by row (run_put_group /
// runs_write).  Every lane of the warp takes part; columns past N are not
// written back.
template <int LP1>
__device__ __forceinline__ void cols_staged(const ColsJob& J, int64_t j, int64_t g0, const float (&xa)[32],
                                            const float* sD, uint8_t* stage) {
  const int lane = threadIdx.x & 31;
  const bool live = j < J.N;
  const bool tiered = J.nsplit > 1 && J.tl < LP1, two = J.nsplit > 1 && !tiered;
  uint16_t* row = J.Bd + (live ? j : 0) * J.pitch;
  uint8_t* base = stage + (threadIdx.x >> 5) * 4096;
#pragma unroll
  for (int q = 0; q < kColGroups; q += 2) {   // two groups per read of the basis values
    float x8[8], y8[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      x8[t] = xa[q * 8 + t];
      y8[t] = xa[q * 8 + 8 + t];
    }
    float2 ax[(LP1 + 1) / 2], ay[(LP1 + 1) / 2];
    group8_pairs2<LP1>(x8, y8, sD, ax, ay);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint16_t hi[8], lo[8];
      split_bf16<LP1>(h ? ay : ax, hi, lo);
      run_put_group<LP1>(base, 128, 0, lane, q + h, hi);
      if (two) run_put_group<LP1>(base, 128, 1, lane, q + h, lo);
      if (tiered && live) store_split_part(row, g0 + q + h, hi, lo, LP1, J.tl, J.Kp_pad, J.Kt_pad, StoreUpto8{});
    }
  }
  __syncwarp();
  const int64_t jw = j - lane;
  const int ncols = J.N - jw < 32 ? static_cast<int>(J.N - jw) : 32;
  uint16_t* o0 = J.Bd + jw * J.pitch + g0 * LP1;
  runs_write<LP1>(base, 128, 0, lane, o0, J.pitch, ncols);
  if (two) runs_write<LP1>(base, 128, 1, lane, o0 + J.Kp_pad, J.pitch, ncols);
  if (g0 == 0 && live)
    zero_split_rows(row, J.NG, LP1, J.nsplit, J.tl, J.Kp_pad, J.Kt_pad, tiered ? 0 : staged_end<LP1>(J));
}

// L = 8, l+1 in {3, 5, 6, 7}, four whole groups, no tiered split: a column's run of
// 4 (l+1) components (8 (l+1) bytes of its row) packed into words, staged in the warp's
// area (2 KB per part; runs an odd number of 8 bytes apart, so the lanes' words fall in
// different banks but for pairs) and written by the warp run after run, in 8-byte
// chunks.  Stored by the lanes themselves, every chunk went to 32 rows at once and the
// words of all four groups were held in registers and spilled.  Every lane of the warp
// takes part; columns past N are not written back.
template <int LP1>
__device__ __forceinline__ void cols_quad_odd(const ColsJob& J, int64_t j, int64_t g0,
                                              const float (&xa)[kColGroups * 8], const float* sD, uint8_t* stage) {
  constexpr int kPitch = 8 * (LP1 | 1);
  static_assert(32 * kPitch <= 2048, "the runs of a warp fit their area");
  const int lane = threadIdx.x & 31;
  const bool two = J.nsplit > 1;
  uint8_t* base = stage + (threadIdx.x >> 5) * 4096;
#pragma unroll
  for (int q = 0; q < kColGroups; q += 2) {
    float x8[8], y8[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      x8[t] = xa[q * 8 + t];
      y8[t] = xa[q * 8 + 8 + t];
    }
    float2 ax[(LP1 + 1) / 2], ay[(LP1 + 1) / 2];
    group8_pairs2<LP1>(x8, y8, sD, ax, ay);
    uint16_t hx[8], lx[8], hy[8], ly[8];
    split_bf16<LP1>(ax, hx, lx);
    split_bf16<LP1>(ay, hy, ly);
    uint32_t* wh = reinterpret_cast<uint32_t*>(base + lane * kPitch + q * 2 * LP1);
    uint32_t* wl = wh + 2048 / 4;
#pragma unroll
    for (int k = 0; k < LP1; ++k) {   // word k: components 2k and 2k + 1 of the two groups' 2 (l+1)
      const int a = 2 * k, b = 2 * k + 1;
      wh[k] = (a < LP1 ? hx[a % 8] : hy[(a + 8 - LP1) % 8]) | (uint32_t(b < LP1 ? hx[b % 8] : hy[(b + 8 - LP1) % 8]) << 16);
      if (two)
        wl[k] = (a < LP1 ? lx[a % 8] : ly[(a + 8 - LP1) % 8]) |
                (uint32_t(b < LP1 ? lx[b % 8] : ly[(b + 8 - LP1) % 8]) << 16);
    }
  }
  __syncwarp();
  const int64_t jw = j - lane;
  const int ncols = J.N - jw < 32 ? static_cast<int>(J.N - jw) : 32;
  uint16_t* o0 = J.Bd + jw * J.pitch + g0 * LP1;
  for (int part = 0; part < (two ? 2 : 1); ++part)
#pragma unroll
    for (int s = 0; s < LP1; ++s) {
      const int gi = s * 32 + lane, c = gi / LP1, k = gi - c * LP1;
      if (c < ncols)
        *reinterpret_cast<uint2*>(o0 + part * J.Kp_pad + c * J.pitch + k * 4) =
            *reinterpret_cast<const uint2*>(base + part * 2048 + c * kPitch + k * 8);
    }
  if (g0 == 0 && j < J.N)
    zero_split_rows(J.Bd + j * J.pitch, J.NG, LP1, J.nsplit, J.tl, J.Kp_pad, J.Kt_pad, staged_end<LP1>(J));
}

// L = 8, unstaged: group gg of one column, l+1 components.
template <int LP1>
__device__ __forceinline__ void col_group8(const ColsJob& J, uint16_t* row, int64_t gg, const float (&x8)[8],
                                           const float* sD) {
  float2 acc[(LP1 + 1) / 2];
  group8_pairs<LP1>(x8, sD, acc);
  uint16_t hi[8], lo[8];
  split_bf16<LP1>(acc, hi, lo);
  store_upto8(row + gg * LP1, hi, LP1);
  if (J.nsplit > 1) store_split_part(row, gg, hi, lo, LP1, J.tl, J.Kp_pad, J.Kt_pad, StoreUpto8{});
}

template <typename InT, int LP, bool kArg>
__device__ __forceinline__ void cols_body(const ColsJob& J, int64_t j, int64_t qd, float* sD, uint8_t* stage) {
  constexpr int LMAX = LP ? 8 : 64;
  const int L = LP ? 8 : J.L;
  const int lp1 = LP ? LP : J.lp1;
  const bool live = j < J.N;
  const InT* B = static_cast<const InT*>(J.B);
  const int64_t g0 = qd * kColGroups;
  const int ng = static_cast<int>(J.NG - g0 < kColGroups ? J.NG - g0 : kColGroups);
  // L = 8: all kColGroups * 8 inputs are loaded before the staging barrier.
  float xa[LP ? kColGroups * 8 : 1];
  if (LP && (g0 + kColGroups) * 8 <= J.K) {
    // whole groups: no test per load (a column past N reads the last one, and is not written)
    const InT* __restrict__ b = B + g0 * 8 * J.ldb + (live ? j : J.N - 1);
    const int64_t ldb = J.ldb;
#pragma unroll
    for (int e = 0; e < (LP ? kColGroups * 8 : 1); ++e, b += ldb) xa[e] = load_as_float(b);
  } else if (LP) {
#pragma unroll
    for (int q = 0; q < kColGroups; ++q) {
      const int64_t k0 = (g0 + q) * 8;
      const int n = live && q < ng ? static_cast<int>(J.K - k0 < 8 ? J.K - k0 : 8) : 0;
#pragma unroll
      for (int t = 0; t < 8; ++t) xa[q * 8 + t] = t < n ? load_as_float(B + (k0 + t) * J.ldb + j) : 0.0f;
    }
  }
  if (kArg) {
  } else if (LP)
    stage_coef8(sD, lp1, [&](int t, int q) { return J.Ds[q * 8 + t]; });
  else
    for (int k = threadIdx.x; k < L * lp1; k += blockDim.x) sD[k] = J.Ds[k];
  __syncthreads();
  // Four whole groups, or fewer whose missing components (zeros) still lie in the row's
  // padding (as in project_tma.cu); the same for the whole block.
  const bool tiered = J.nsplit > 1 && J.tl < lp1;
  if constexpr (LP == 4 || LP == 8) {
    if (ng == kColGroups || (!tiered && (g0 + kColGroups) * LP <= J.Kp_pad)) {
      cols_staged<LP>(J, j, g0, xa, sD, stage);
      return;
    }
  }
  if constexpr (LP == 3 || LP == 5 || LP == 6 || LP == 7) {
    if (!tiered && (g0 + kColGroups) * LP <= J.Kp_pad) {
      cols_quad_odd<LP>(J, j, g0, xa, sD, stage);
      return;
    }
  }
  if (!live) return;
  uint16_t* row = J.Bd + j * J.pitch;
  if constexpr (LP > 0) {
#pragma unroll
    for (int q = 0; q < kColGroups; ++q) {
      if (q >= ng) break;
      float x8[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) x8[t] = xa[(q * 8 + t) % (LP ? kColGroups * 8 : 1)];
      col_group8<LP>(J, row, g0 + q, x8, sD);
    }
  } else {
    for (int q = 0; q < ng; ++q) {
      const int64_t k0 = (g0 + q) * L;
      const int n = static_cast<int>(J.K - k0 < L ? J.K - k0 : L);
      float x[LMAX];
#pragma unroll
      for (int t = 0; t < LMAX; ++t)
        if (t < L) x[t] = t < n ? load_as_float(B + (k0 + t) * J.ldb + j) : 0.0f;
      for (int p = 0; p < lp1; ++p) {
        float acc = 0.0f;
#pragma unroll
        for (int t = 0; t < LMAX; ++t)
          if (t < L) acc = fmaf(sD[p * L + t], x[t], acc);
        const uint16_t h = bf16_bits(acc);
        row[(g0 + q) * lp1 + p] = h;
        if (J.nsplit > 1)
          split_part_one(row, g0 + q, p, h, bf16_bits(acc - bf16_value(h)), lp1, J.tl, J.Kp_pad, J.Kt_pad);
      }
    }
  }
  if (qd == 0) zero_split_rows(row, J.NG, lp1, J.nsplit, J.tl, J.Kp_pad, J.Kt_pad);
}

template <typename InT, int LP, bool kArg>
__global__ void __launch_bounds__(256, LP == 7 ? 2 : LP ? 3 : 2) project_cols_kernel(const __grid_constant__ ColsJob J,
                                                                            const __grid_constant__ SideArgs a) {
  __shared__ __align__(16) float sD[LP ? 64 : 64 * 64];
  __shared__ __align__(16) uint8_t sStage[LP ? 8 * 4096 : 16];
  side_begin<kArg>(a, sD);
  const uint32_t b = blockIdx.x, nbx = static_cast<uint32_t>(J.nbx);
  cols_body<InT, LP, kArg>(J, static_cast<int64_t>(b % nbx) * blockDim.x + threadIdx.x, b / nbx, sD, sStage);
}

template <typename InT, int LP>
__global__ void __launch_bounds__(256, LP == 7 ? 2 : LP ? 3 : 2) project_cols_jobs_kernel(const ColsJob* __restrict__ jobs,
                                                                const int* __restrict__ job_of) {
  __shared__ __align__(16) float sD[LP ? 64 : 64 * 64];
  __shared__ __align__(16) uint8_t sStage[LP ? 8 * 4096 : 16];
  pdl_begin();
  const ColsJob J = jobs[job_of[blockIdx.x]];   // (as for rows)
  const uint32_t b = blockIdx.x - static_cast<uint32_t>(J.block0), nbx = static_cast<uint32_t>(J.nbx);
  cols_body<InT, LP, false>(J, static_cast<int64_t>(b % nbx) * blockDim.x + threadIdx.x, b / nbx, sD, sStage);
}

// ---- FP64 path ------------------------------------------------------------
// Blocks [0, row_blocks): one thread per (row, group) of A; the rest: one thread per
// (column, group) of B.
struct PairF64 {
  const double* A;
  const double* B;
  double* Ac;
  double* Bd;
  const double* Cs;
  const double* Ds;
  int64_t lda, ldb, M, N, K, NG, Kp, row_blocks;
  int L, lp1;
  int* clear;   // the call's error word (NULL: not cleared here)
  Coef8d c8;    // the kept vectors (kArg: groups of 8)
};

template <bool kArg>
__global__ void __launch_bounds__(128) project_pair_f64_kernel(const __grid_constant__ PairF64 p) {
  pdl_begin();
  if (p.clear && blockIdx.x == 0 && threadIdx.x == 0) *p.clear = 0;
  const int L = kArg ? 8 : p.L, lp1 = p.lp1;
  const bool rows = static_cast<int64_t>(blockIdx.x) < p.row_blocks;
  const int64_t e = (static_cast<int64_t>(blockIdx.x) - (rows ? 0 : p.row_blocks)) * blockDim.x + threadIdx.x;
  if (e >= (rows ? p.M : p.N) * p.NG) return;
  const int64_t i = rows ? e / p.NG : 0, j = rows ? 0 : e % p.N;
  const int64_t gg = rows ? e - i * p.NG : e / p.N;
  const double* x = rows ? p.A + i * p.lda + gg * L : p.B + gg * L * p.ldb + j;
  const int64_t xs = rows ? 1 : p.ldb;
  double* o = rows ? p.Ac + i * p.Kp + gg * lp1 : p.Bd + gg * lp1 * p.N + j;
  const int64_t os = rows ? 1 : p.N;
  const int n = static_cast<int>(p.K - gg * L < L ? p.K - gg * L : L);
  if constexpr (kArg) {
    double v[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) v[t] = t < n ? x[t * xs] : 0.0;
    for (int q = 0; q < lp1; ++q) {
      double acc = 0.0;
#pragma unroll
      for (int t = 0; t < 8; ++t) acc = fma(v[t], p.c8.c[q * 8 + t], acc);
      o[q * os] = acc;
    }
  } else {
    for (int q = 0; q < lp1; ++q) {
      double acc = 0.0;
      for (int t = 0; t < n; ++t) acc = fma(x[t * xs], rows ? p.Cs[t * lp1 + q] : p.Ds[q * L + t], acc);
      o[q * os] = acc;
    }
  }
}

// ---- CONV: signal and templates -------------------------------------------
// Box-basis form of the Haar projection with l+1 a power of two: the kept
// span is the functions constant on aligned runs of Lb = T / R samples, with
// orthonormal basis 1/sqrt(Lb) on each run.  The projected signal at
// position x is b[x] = sum_{u < Lb} s[x + u] / sqrt(Lb).  It is stored phase-
// split, with eight element shifts so every row view starts 16-byte aligned:
//   G[(sigma * Lb + phi) * P + y] = b[phi + Lb * (y + sigma)]  (0 where b is undefined).
// The templates are stored as lag-paired chunks of 64 projected components:
//   TP[c][e * 64 + t][i] = kb_t[(c - e) * 64 + i] for 0 <= c - e < R / 64, else 0,
// with kb_t[g] = sum_{u < Lb} k_t[g * Lb + u] / sqrt(Lb).
//
// One launch does both.  Signal blocks come first: block j owns the output
// columns y in [Y0, Y0 + YB) of every (sigma, phi) row, Y0 = j * YB, with
// YB = 2048 / Lb (one instantiation per Lb).  It loads s over [Lb Y0, Lb (Y0 + YB + 8)), forms the box
// sums by log2(Lb) pairwise doubling passes in shared memory (sums of 2, 4,
// ... Lb samples), and each thread writes 8 consecutive y of one (sigma, phi)
// row with one 16-byte store.  Template blocks follow (conv_template_part).
// Block 0 also clears the
// call's error word (no kernel of the call has run before it).
constexpr int kConvXB = 2048;            // box-sum positions per signal block (YB = kConvXB / Lb)
constexpr int kConvSpanMax = 64 * 40;    // samples a signal block loads: Lb (YB + 8), largest at Lb = 64
// Shared-memory index of box-sum position u: Lb floats of padding after every
// 8 Lb positions, so the reads of the output phase (lanes over phi and over
// octets 8 Lb positions apart) fall in distinct banks for every Lb.
template <int LB>
__device__ __forceinline__ int conv_pad(int u) { return u + (u / (8 * LB)) * LB; }
constexpr int kConvBuf = kConvSpanMax + kConvSpanMax / 8 + 64;  // + the over-read of the last vector

struct ConvProjParams {
  const float* s;
  int64_t S, P;
  int Lb;
  float scale;
  uint16_t* G;
  int64_t sig_blocks;
  const float* k;     // NULL: no templates in this launch
  int64_t T, nt, R;
  int Kc;
  uint16_t* TP;
  int* err;
};

template <int LB>
__device__ __forceinline__ void conv_signal_block(const ConvProjParams& p, int64_t blk, float (*buf)[kConvBuf]) {
  constexpr int YB = kConvXB / LB;
  constexpr int span = LB * (YB + 8);  // a multiple of 8; x0 too, so the span is read with 16-byte loads
  const int64_t Y0 = blk * YB;
  const int64_t x0 = Y0 * LB;
  for (int u4 = threadIdx.x; u4 < span / 4; u4 += blockDim.x) {
    const int64_t x = x0 + 4 * u4;
    float4 v;
    if (x + 4 <= p.S) {
      v = __ldg(reinterpret_cast<const float4*>(p.s + x));
    } else {
      v.x = x < p.S ? __ldg(p.s + x) : 0.0f;
      v.y = x + 1 < p.S ? __ldg(p.s + x + 1) : 0.0f;
      v.z = x + 2 < p.S ? __ldg(p.s + x + 2) : 0.0f;
      v.w = x + 3 < p.S ? __ldg(p.s + x + 3) : 0.0f;
    }
    const int u = 4 * u4;   // the four stay inside one padded run of 8 LB
    float* d = buf[0] + conv_pad<LB>(u);
    if (LB % 4 == 0) {      // the padding keeps 16-byte alignment
      *reinterpret_cast<float4*>(d) = v;
    } else {
      d[0] = v.x;
      d[1] = v.y;
      d[2] = v.z;
      d[3] = v.w;
    }
  }
  __syncthreads();
  int cur = 0;
#pragma unroll
  for (int w = 1; w < LB; w *= 2) {
    const int n = span - 2 * w + 1;  // valid sums of 2w after this pass
    if (LB >= 4) {
      // Four consecutive positions per thread (the padding keeps every
      // 4-aligned run of four contiguous and 16-byte aligned).  The last
      // vector may form up to three sums past n; they are never read.
      for (int u = 4 * threadIdx.x; u < n; u += 4 * blockDim.x) {
        const float4 a = *reinterpret_cast<const float4*>(&buf[cur][conv_pad<LB>(u)]);
        float4 r;
        if (w >= 4) {
          const float4 b = *reinterpret_cast<const float4*>(&buf[cur][conv_pad<LB>(u + w)]);
          r = make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
        } else {
          const float4 b = *reinterpret_cast<const float4*>(&buf[cur][conv_pad<LB>(u + 4)]);
          const float e[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
          r = make_float4(e[0] + e[w], e[1] + e[1 + w], e[2] + e[2 + w], e[3] + e[3 + w]);
        }
        *reinterpret_cast<float4*>(&buf[cur ^ 1][conv_pad<LB>(u)]) = r;
      }
    } else {
      for (int u = threadIdx.x; u < n; u += blockDim.x)
        buf[cur ^ 1][conv_pad<LB>(u)] = buf[cur][conv_pad<LB>(u)] + buf[cur][conv_pad<LB>(u + w)];
    }
    __syncthreads();
    cur ^= 1;
  }
  // BF16 once per box sum, staged transposed as bt[phi][Y - Y0] (row length
  // RL = YB + 8: 16-byte aligned rows whose stride in 16-byte units is odd).
  constexpr int RL = YB + 8;
  uint16_t* bt = reinterpret_cast<uint16_t*>(buf[cur ^ 1]);
  for (int u = threadIdx.x; u < LB * RL; u += blockDim.x) {
    const int phi = u % LB, yr = u / LB;
    const bool ok = yr < YB + 7 && x0 + u + LB <= p.S;
    bt[phi * RL + yr] = ok ? bf16_bits(buf[cur][conv_pad<LB>(u)] * p.scale) : 0;
  }
  __syncthreads();
  // Thread (octet j8, phi) holds bt[phi][8 j8 .. 8 j8 + 16) and writes the
  // eight shifted copies: copy sigma is the 8 values starting at sigma.
  static_assert(8 * LB * (YB / 8) == 8 * 256, "one (octet, phi) per thread");
  const int phi = threadIdx.x % LB, j8 = threadIdx.x / LB;
  const int64_t y0 = Y0 + 8 * j8;
  if (y0 >= p.P) return;
  const uint4* row = reinterpret_cast<const uint4*>(bt + phi * RL + 8 * j8);
  const uint4 lo4 = row[0], hi4 = row[1];
  const uint32_t w[8] = {lo4.x, lo4.y, lo4.z, lo4.w, hi4.x, hi4.y, hi4.z, hi4.w};
  uint16_t* g = p.G + static_cast<int64_t>(phi) * p.P + y0;
  const int64_t copy_stride = static_cast<int64_t>(LB) * p.P;
#pragma unroll
  for (int sigma = 0; sigma < 8; ++sigma) {
    uint4 o;
    if (sigma % 2 == 0) {
      o = make_uint4(w[sigma / 2], w[sigma / 2 + 1], w[sigma / 2 + 2], w[sigma / 2 + 3]);
    } else {
      const int q = sigma / 2;
      o = make_uint4(__funnelshift_r(w[q], w[q + 1], 16), __funnelshift_r(w[q + 1], w[q + 2], 16),
                     __funnelshift_r(w[q + 2], w[q + 3], 16), __funnelshift_r(w[q + 3], w[q + 4], 16));
    }
    *reinterpret_cast<uint4*>(g + sigma * copy_stride) = o;
  }
}

// Template pairs.  Lb < 8: four consecutive entries of one row per thread,
// their 4 Lb samples read with Lb 16-byte loads.  Lb >= 8: one entry per
// thread, its Lb samples read with Lb / 4 independent 16-byte loads (all in
// flight at once).  The samples of a group are contiguous and 16-byte aligned.
template <int LB>
constexpr int conv_tpl_per_thread() { return LB < 8 ? 4 : 1; }

template <int LB>
__device__ __forceinline__ void conv_template_part(const ConvProjParams& p, int64_t e) {
  constexpr int EPT = conv_tpl_per_thread<LB>();
  const int64_t total = static_cast<int64_t>(p.Kc + 1) * 128 * (64 / EPT);
  if (e >= total) return;
  const int i0 = static_cast<int>(e % (64 / EPT)) * EPT;
  const int row = static_cast<int>((e / (64 / EPT)) % 128);
  const int c = static_cast<int>(e / ((64 / EPT) * 128));
  const int ee = row / 64, t = row % 64;
  const int cc = c - ee;
  float acc[EPT];
#pragma unroll
  for (int j = 0; j < EPT; ++j) acc[j] = 0.0f;
  // (components at or past R pad the last chunk with zeros; R is a multiple of EPT)
  if (t < p.nt && cc >= 0 && cc < p.Kc && cc * 64 + i0 < p.R) {
    const float4* kt = reinterpret_cast<const float4*>(p.k + t * p.T + (static_cast<int64_t>(cc) * 64 + i0) * LB);
    if (LB == 1) {
      const float4 v = __ldg(kt);
      acc[0] = v.x; acc[EPT > 1 ? 1 : 0] = v.y; acc[EPT > 2 ? 2 : 0] = v.z; acc[EPT > 3 ? 3 : 0] = v.w;
    } else if (LB == 2) {
      const float4 a = __ldg(kt), b = __ldg(kt + 1);
      acc[0] = a.x + a.y; acc[EPT > 1 ? 1 : 0] = a.z + a.w;
      acc[EPT > 2 ? 2 : 0] = b.x + b.y; acc[EPT > 3 ? 3 : 0] = b.z + b.w;
    } else {
      constexpr int Q = LB >= 4 ? LB / 4 : 1;  // 16-byte loads per entry
      float4 v[EPT * Q];
#pragma unroll
      for (int q = 0; q < EPT * Q; ++q) v[q] = __ldg(kt + q);
#pragma unroll
      for (int j = 0; j < EPT; ++j)
#pragma unroll
        for (int q = 0; q < Q; ++q) {
          acc[j] += v[j * Q + q].x;
          acc[j] += v[j * Q + q].y;
          acc[j] += v[j * Q + q].z;
          acc[j] += v[j * Q + q].w;
        }
    }
  }
  uint16_t* dst = p.TP + e * EPT;
  if (EPT == 4) {
    uint16_t h[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) h[j] = bf16_bits(acc[j < EPT ? j : 0] * p.scale);
    store_run(dst, h, 4);
  } else {
    *dst = bf16_bits(acc[0] * p.scale);
  }
}

template <int LB>
__global__ void __launch_bounds__(256) conv_project_kernel(const __grid_constant__ ConvProjParams p) {
  __shared__ __align__(16) float buf[2][kConvBuf];
  pdl_begin();
  if (blockIdx.x == 0 && threadIdx.x == 0) *p.err = 0;
  if (blockIdx.x < p.sig_blocks)
    conv_signal_block<LB>(p, blockIdx.x, buf);
  else
    conv_template_part<LB>(p, (static_cast<int64_t>(blockIdx.x) - p.sig_blocks) * blockDim.x + threadIdx.x);
}

// ---- CONV projection for any basis (the general path) ----------------------
// Signal: G[(sigma PH + phi) P + y lp1 + p] = bf16( sum_{i<L} s[x + i] c[i, p] ) with
// x = phi + L (y + sigma): for every phase phi < L of the lags, the projections of
// the groups starting at phi + L y, all lp1 of them side by side, in copies shifted
// by sigma positions (zero extension past the signal).  Templates: the template-pair
// chunks of the box path with kd_t[g lp1 + p] = sum_{i<L} d[p, i] k_t[g L + i].
struct ConvGenParams {
  const float* s;
  int64_t S, P;
  int L, PH;
  uint16_t* G;
  int64_t sig_threads;
  const float* k;     // NULL: no templates in this launch
  int64_t T, nt, R;
  int Kc;
  uint16_t* TP;
  const float* Cs;    // L x lp1, Cs[i * lp1 + p] = c[i, p]
  const float* Ds;    // lp1 x L, Ds[p * L + i] = d[p, i]
  int inl;            // the kept vectors are in c8 (L = 8), and block 0 clears *err
  Coef8 c8;
  int* err;
};

template <int LP1>
__global__ void __launch_bounds__(256) conv_project_general_kernel(const __grid_constant__ ConvGenParams p) {
  __shared__ float sC[kMaxL * LP1];
  __shared__ float sD[LP1 * kMaxL];
  pdl_begin();
  if (p.inl) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *p.err = 0;
    for (int e = threadIdx.x; e < 8 * LP1; e += blockDim.x) {
      sC[e] = p.c8.c[(e % LP1) * 8 + e / LP1 & 63];
      sD[e] = p.c8.c[e & 63];
    }
  } else {
    for (int e = threadIdx.x; e < p.L * LP1; e += blockDim.x) {
      sC[e] = p.Cs[e];
      sD[e] = p.Ds[e];
    }
  }
  __syncthreads();
  const int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (e < p.sig_threads) {
    const int64_t npos = p.P / LP1;
    const int64_t y = e % npos, rest = e / npos;
    const int phi = static_cast<int>(rest % p.PH), sigma = static_cast<int>(rest / p.PH);
    const int64_t x = phi + static_cast<int64_t>(p.L) * (y + sigma);
    float acc[LP1];
#pragma unroll
    for (int q = 0; q < LP1; ++q) acc[q] = 0.0f;
    for (int i = 0; i < p.L; ++i) {
      const float v = x + i < p.S ? __ldg(p.s + x + i) : 0.0f;
#pragma unroll
      for (int q = 0; q < LP1; ++q) acc[q] = fmaf(v, sC[i * LP1 + q], acc[q]);
    }
    uint16_t* o = p.G + (static_cast<int64_t>(sigma) * p.PH + phi) * p.P + y * LP1;
    if (LP1 >= 8) {
#pragma unroll
      for (int q = 0; q < LP1; q += 8) {
        uint16_t v8[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v8[u] = bf16_bits(acc[q + u]);
        *reinterpret_cast<uint4*>(o + q) = make_uint4(v8[0] | (uint32_t(v8[1]) << 16), v8[2] | (uint32_t(v8[3]) << 16),
                                                      v8[4] | (uint32_t(v8[5]) << 16), v8[6] | (uint32_t(v8[7]) << 16));
      }
    } else {
#pragma unroll
      for (int q = 0; q < LP1; ++q) o[q] = bf16_bits(acc[q]);
    }
    return;
  }
  if (!p.k) return;
  const int64_t te = e - p.sig_threads;
  if (te >= static_cast<int64_t>(p.Kc + 1) * 128 * 64) return;
  const int i = static_cast<int>(te % 64);
  const int row = static_cast<int>((te / 64) % 128);
  const int c = static_cast<int>(te / (64 * 128));
  const int ee = row / 64, t = row % 64, cc = c - ee;
  const int64_t kk = static_cast<int64_t>(cc) * 64 + i;   // reduced component (g, q): kk = g lp1 + q
  float acc = 0.0f;
  if (t < p.nt && cc >= 0 && kk < p.R) {
    const int64_t g = kk / LP1;
    const int q = static_cast<int>(kk - g * LP1);
    const float* kt = p.k + t * p.T + g * p.L;
    for (int u = 0; u < p.L; ++u) acc = fmaf(sD[q * p.L + u], __ldg(kt + u), acc);
  }
  p.TP[te] = bf16_bits(acc);
}

}  // namespace

static cudaError_t launch_conv_project_general(const float* s, const float* k, const ConvGeom& g, uint16_t* G,
                                               uint16_t* TP, const float* Cs, const float* Ds, const Coef8* c8,
                                               int* err, cudaStream_t st) {
  ConvGenParams p{};
  p.s = s;
  p.S = g.S;
  p.P = g.P;
  p.L = g.L;
  p.PH = g.PH;
  p.G = G;
  p.sig_threads = static_cast<int64_t>(g.ncopy) * g.PH * (g.P / g.lp1);
  p.k = k;
  p.T = g.T;
  p.nt = g.nt;
  p.R = g.R;
  p.Kc = g.Kc;
  p.TP = TP;
  p.Cs = Cs;
  p.Ds = Ds;
  if (c8) {
    p.inl = 1;
    p.c8 = *c8;
  }
  p.err = err;
  const int64_t threads = p.sig_threads + (k ? static_cast<int64_t>(g.Kc + 1) * 128 * 64 : 0);
  const unsigned blocks = static_cast<unsigned>(ceil_div(threads, 256));
  switch (g.lp1) {   // a power of two in [1, 64]
    case 1: return launch_plain(conv_project_general_kernel<1>, dim3(blocks), 256, 0, st, p);
    case 2: return launch_plain(conv_project_general_kernel<2>, dim3(blocks), 256, 0, st, p);
    case 4: return launch_plain(conv_project_general_kernel<4>, dim3(blocks), 256, 0, st, p);
    case 8: return launch_plain(conv_project_general_kernel<8>, dim3(blocks), 256, 0, st, p);
    case 16: return launch_plain(conv_project_general_kernel<16>, dim3(blocks), 256, 0, st, p);
    case 32: return launch_plain(conv_project_general_kernel<32>, dim3(blocks), 256, 0, st, p);
    case 64: return launch_plain(conv_project_general_kernel<64>, dim3(blocks), 256, 0, st, p);
    default: return cudaErrorInvalidValue;
  }
}

RowsJob make_rows_job(const void* A, int64_t lda, int in_dtype, const GemmGeom& g, const float* Cs, uint16_t* Ac) {
  RowsJob J{};
  J.A = A;
  J.Ac = Ac;
  J.Cs = Cs;
  J.lda = lda;
  J.M = g.M;
  J.K = g.K;
  J.NG = ceil_div(g.K, g.L);
  J.pitch = gemm_pitch(g);
  J.Kp_pad = g.Kp_pad;
  J.Kt_pad = g.Kt_pad;
  J.tl = g.tl;
  J.L = g.L;
  J.lp1 = g.lp1;
  J.nsplit = g.nsplit;
  J.in_bf16 = in_dtype == PJ_BF16;
  // Runs per warp: eight where that leaves the chip full (4 blocks of 8 warps an SM),
  // fewer for small operands; BF16 input loads one pair at a time, so its warps take one.
  int sms = 0;
  if (device_sms(&sms) != PJ_OK) sms = 152;
  const int64_t units = J.M * ceil_div(J.NG, kRowRun), warps = static_cast<int64_t>(sms) * 32;
  J.upw = J.in_bf16 || units <= 2 * warps ? 2 : (units >= 8 * warps ? 8 : static_cast<int>(units / warps / 2 * 2));
  return J;
}

ColsJob make_cols_job(const void* B, int64_t ldb, int in_dtype, const GemmGeom& g, const float* Ds, uint16_t* Bd) {
  ColsJob J{};
  J.B = B;
  J.Bd = Bd;
  J.Ds = Ds;
  J.ldb = ldb;
  J.N = g.N;
  J.K = g.K;
  J.NG = ceil_div(g.K, g.L);
  J.pitch = gemm_pitch(g);
  J.Kp_pad = g.Kp_pad;
  J.Kt_pad = g.Kt_pad;
  J.tl = g.tl;
  J.nbx = ceil_div(g.N, 256);
  J.L = g.L;
  J.lp1 = g.lp1;
  J.nsplit = g.nsplit;
  J.in_bf16 = in_dtype == PJ_BF16;
  return J;
}

int64_t rows_job_blocks(const RowsJob& J) {
  return J.L == 8 ? ceil_div(J.M * ceil_div(J.NG, kRowRun), 8 * J.upw) : ceil_div(J.M * J.NG, 256);
}
int64_t cols_job_blocks(const ColsJob& J) { return J.nbx * ceil_div(J.NG, kColGroups); }

int projection_class(int in_bf16, int L, int lp1) { return (in_bf16 ? 9 : 0) + (L == 8 ? lp1 : 0); }

// f(InT value, std::integral_constant<int, LP>) for the kernels of one class.
template <typename InT, typename F>
static cudaError_t with_lp(int lp, F f) {
  switch (lp) {
    case 0: return f(InT(), std::integral_constant<int, 0>());
    case 1: return f(InT(), std::integral_constant<int, 1>());
    case 2: return f(InT(), std::integral_constant<int, 2>());
    case 3: return f(InT(), std::integral_constant<int, 3>());
    case 4: return f(InT(), std::integral_constant<int, 4>());
    case 5: return f(InT(), std::integral_constant<int, 5>());
    case 6: return f(InT(), std::integral_constant<int, 6>());
    case 7: return f(InT(), std::integral_constant<int, 7>());
    default: return f(InT(), std::integral_constant<int, 8>());
  }
}
// The shared-memory opt-in of a row kernel (a block's static share is added to the ring:
// above 48 KB), recorded per kernel and device; a racing repeat is harmless.
template <typename K>
static cudaError_t rows_smem(K* kern, int smem) {
  static std::atomic<const void*> done[64][80] = {};
  if (smem == 0) return cudaSuccess;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const void* key = reinterpret_cast<const void*>(kern);
  if (dev >= 0 && dev < 64)
    for (auto& d : done[dev]) {
      const void* k = d.load(std::memory_order_acquire);
      if (k == key) return cudaSuccess;
      if (!k) break;
    }
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess && dev >= 0 && dev < 64)
    for (auto& d : done[dev]) {
      const void* none = nullptr;
      if (d.compare_exchange_strong(none, key) || none == key) break;
    }
  return e;
}
template <typename F>
static cudaError_t with_class(int cls, F f) {
  return cls >= 9 ? with_lp<__nv_bfloat16>(cls - 9, f) : with_lp<float>(cls, f);
}

cudaError_t launch_project_pair_simt(const void* A, int64_t lda, const void* B, int64_t ldb, int in_dtype,
                                     const GemmGeom& g, const float* Cs, const float* Ds, const Coef8* c8,
                                     uint16_t* Ac, uint16_t* Bd, int* clear_err, cudaStream_t st) {
  if (g.K == 0) return cudaSuccess;
  const bool rows = A && g.M > 0, cols = B && g.N > 0;
  if (!rows && !cols) return cudaSuccess;
  SideArgs a{};
  if (c8) a.c8 = *c8;
  a.clear = clear_err;
  if (rows) {
    const RowsJob J = make_rows_job(A, lda, in_dtype, g, Cs, Ac);
    const dim3 grid(static_cast<unsigned>(rows_job_blocks(J)));
    const cudaError_t e = with_class(projection_class(J.in_bf16, J.L, J.lp1), [&](auto in, auto lp) {
      using InT = decltype(in);
      constexpr int LP = decltype(lp)::value;
      auto kern = c8 ? project_rows_kernel<InT, LP, (LP > 0)> : project_rows_kernel<InT, LP, false>;
      const int smem = LP ? kRowsSmem : 0;
      const cudaError_t e = rows_smem(kern, smem);
      return e != cudaSuccess ? e : launch_plain(kern, grid, 256, smem, st, J, a);
    });
    if (e != cudaSuccess) return e;
    a.clear = nullptr;
  }
  if (!cols) return cudaSuccess;
  const ColsJob J = make_cols_job(B, ldb, in_dtype, g, Ds, Bd);
  const dim3 grid(static_cast<unsigned>(cols_job_blocks(J)));
  return with_class(projection_class(J.in_bf16, J.L, J.lp1), [&](auto in, auto lp) {
    using InT = decltype(in);
    constexpr int LP = decltype(lp)::value;
    return launch_plain(c8 ? project_cols_kernel<InT, LP, (LP > 0)> : project_cols_kernel<InT, LP, false>, grid, 256, 0,
                        st, J, a);
  });
}

cudaError_t launch_project_rows_jobs(int cls, const RowsJob* jobs, const int* job_of, int64_t blocks, cudaStream_t st) {
  if (blocks == 0) return cudaSuccess;
  const unsigned nb = static_cast<unsigned>(blocks);
  return with_class(cls, [&](auto in, auto lp) {
    auto kern = project_rows_jobs_kernel<decltype(in), decltype(lp)::value>;
    const int smem = decltype(lp)::value ? kRowsSmem : 0;
    const cudaError_t e = rows_smem(kern, smem);
    return e != cudaSuccess ? e : launch_plain(kern, dim3(nb), 256, smem, st, jobs, job_of);
  });
}

cudaError_t launch_project_cols_jobs(int cls, const ColsJob* jobs, const int* job_of, int64_t blocks, cudaStream_t st) {
  if (blocks == 0) return cudaSuccess;
  const unsigned nb = static_cast<unsigned>(blocks);
  return with_class(cls, [&](auto in, auto lp) {
    return launch_plain(project_cols_jobs_kernel<decltype(in), decltype(lp)::value>, dim3(nb), 256, 0, st, jobs, job_of);
  });
}


cudaError_t launch_project_pair_f64(const double* A, int64_t lda, const double* B, int64_t ldb, const GemmGeom& g,
                                    const double* Cs, const double* Ds, const Coef8d* c8, double* Ac, double* Bd,
                                    int* clear_err, cudaStream_t st) {
  const int64_t NG = ceil_div(g.K, g.L);
  const int64_t rb = A ? ceil_div(g.M * NG, 128) : 0, cb = B ? ceil_div(g.N * NG, 128) : 0;
  if (rb + cb == 0) return cudaSuccess;
  PairF64 p{A, B, Ac, Bd, Cs, Ds, lda, ldb, g.M, g.N, g.K, NG, g.Kp, rb, g.L, g.lp1, clear_err, {}};
  if (c8) p.c8 = *c8;
  return launch_plain(c8 ? project_pair_f64_kernel<true> : project_pair_f64_kernel<false>,
                      dim3(static_cast<unsigned>(rb + cb)), 128, 0, st, p);
}

cudaError_t launch_conv_project(const float* s, const float* k, const ConvGeom& g, uint16_t* G, uint16_t* TP,
                                int* err, cudaStream_t st, const float* Cs, const float* Ds, const Coef8* c8) {
  if (!g.box) return launch_conv_project_general(s, k, g, G, TP, Cs, Ds, c8, err, st);
  ConvProjParams p{};
  p.s = s;
  p.S = g.S;
  p.P = g.P;
  p.Lb = g.Lb;
  p.scale = 1.0f / sqrtf(static_cast<float>(g.Lb));
  p.G = G;
  p.sig_blocks = ceil_div(g.P, kConvXB / g.Lb);
  p.k = k;
  p.T = g.T;
  p.nt = g.nt;
  p.R = g.R;
  p.Kc = g.Kc;
  p.TP = TP;
  p.err = err;
  const int64_t tpl_threads = static_cast<int64_t>(g.Kc + 1) * 128 * (g.Lb < 8 ? 16 : 64);
  const int64_t tpl_blocks = k ? ceil_div(tpl_threads, 256) : 0;
  const unsigned blocks = static_cast<unsigned>(p.sig_blocks + tpl_blocks);
  switch (g.Lb) {  // Lb = T / R is a power of two in [1, 64]
    case 1: return launch_plain(conv_project_kernel<1>, dim3(blocks), 256, 0, st, p);
    case 2: return launch_plain(conv_project_kernel<2>, dim3(blocks), 256, 0, st, p);
    case 4: return launch_plain(conv_project_kernel<4>, dim3(blocks), 256, 0, st, p);
    case 8: return launch_plain(conv_project_kernel<8>, dim3(blocks), 256, 0, st, p);
    case 16: return launch_plain(conv_project_kernel<16>, dim3(blocks), 256, 0, st, p);
    case 32: return launch_plain(conv_project_kernel<32>, dim3(blocks), 256, 0, st, p);
    case 64: return launch_plain(conv_project_kernel<64>, dim3(blocks), 256, 0, st, p);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace pj
