// Reduced GEMM on tcgen05 tensor cores (the (l+1) smaller products of
// Sec. III-B, Fig. 5, accumulated over blocks as in Eq. 2 and Eq. 8).
//
// Y[i][j] = sum_k A_c[i][k] B_d[j][k] over the reduced inner dimension k
// (all blocks and kept projections; with split components, three passes
// hi*hi + hi*lo + lo*hi).  The per-block partial products are summed in the
// FP32 TMEM accumulator as part of the MMA K loop.
//
// Tile: 128 output columns (rows of B_d, the MMA M side) x up to 256 output
// rows (rows of A_c, the MMA N side; a grouped launch picks the height per
// instance, a multiple of 32), K step 64 (one 128-byte swizzle row).
// Persistent CTAs, one per SM; warp 0 issues TMA loads, warp 1 issues UMMA,
// warps 2-5 drain the two TMEM accumulators (2 x 256 columns) so the epilogue
// of one tile overlaps the main loop of the next.  TMEM lane = output column,
// so each warp's stores of one output row are 128 contiguous bytes.
//
// A tile moves (128 + rows) x 128 bytes from L2 per K stage; at the tensor
// rate that is more than the SMs can draw from L2, so products whose tile columns
// pair up, and batches, run on 2-SM MMAs instead (gemm_cg2.cu); this kernel serves
// the odd ones, stream-K and solo CTAs.
// With the hi/lo split, the hi and lo tiles of a K chunk take two ring slots and
// serve all three products (hi*hi, lo*hi, hi*lo) from there: four tile loads per
// chunk instead of six, and the same shared memory covers 1.5x the MMA time.
//
// A grouped launch walks a per-CTA tile list planned on the host; a tile may
// cover only a range of the K stages of its instance (a split reduced
// dimension), in which case its partial product is added to the output by a
// TMA reduction (or FP32 atomics) instead of stored.
#include <cuda_bf16.h>
#include <string.h>

#include "common.hpp"
#include "gemm_epi.cuh"
#include "pdl.cuh"
#include "tc.cuh"
#include "tmap.hpp"
#if PJ_CTA_PAIRS
#include "tc_pair.cuh"   // (nothing here uses it: the build's multicast forms are looked for in this file)
#endif

namespace pj {
namespace {

constexpr int BM = 128;  // output columns per tile (MMA M)
constexpr int BN = 256;  // output rows per tile (MMA N)
constexpr int BK = 64;
// The ring holds as many slots of (128 + tile height) operand rows as its memory takes:
// four at 256 rows, eight at 64.  (With four slots at every height, the 64-row tiles of a
// 1000 x 777 product over 2256 split components waited on their loads: 28.6 us.)
constexpr int kMaxStages = 8;
constexpr int kThreads = 192;
constexpr uint32_t kStageP = BM * BK * 2;
constexpr uint32_t kStageOut = 32 * BM * 4;          // output staging: 32 rows x 128 columns (FP32 max)
constexpr uint32_t kCtl = 256;                       // barriers, TMEM slot and votes
constexpr size_t kSmemBytes = 232448 - 512;          // a block's shared memory less the static coefficients
constexpr uint32_t kRing = 232448 - 512 - 1024 - kStageOut - kCtl;
static_assert((2 * kMaxStages + 5) * 8 + 16 + 8 * 4 <= kCtl, "control area");

// Ring slots at a tile height of bn rows (a multiple of 32).
__host__ __device__ constexpr int ring_slots(int bn) {
  const int n = static_cast<int>(kRing / (kStageP + static_cast<uint32_t>(bn) * BK * 2));
  return n < kMaxStages ? n : kMaxStages;
}
static_assert(ring_slots(BN) >= 4, "at least two K chunks of a split product");

struct GemmParams {
  GemmInst single;           // the instance when `tiles` is null
  const GemmInst* insts;     // grouped launch: instance table in global memory
  const GemmTile* tiles;     // grouped launch: tiles ordered CTA by CTA (null for a single instance)
  const int* cta_off;        // grouped launch: tiles of CTA c are [cta_off[c], cta_off[c+1])
  int num_tiles;             // single instance: tiles, walked with a grid stride
  int streamk;               // single instance: CTAs share the K stages of all tiles evenly
  int slot_rows;             // tile height the ring slots are sized for (the instance's, or 256 when grouped)
  int stall;                 // failure-detection self-test: the producer stops after this many stages (-1: never)
  int* err;
  ExpandArgs ex;             // single instance: expansion to samples in the epilogue (mode 0: none)
  Coef8 ex_c8;               // its vectors when ex.coef is null
};

// The n-th tile of this CTA: instance, coordinates and K-stage range; false past the last.
__device__ __forceinline__ const GemmInst* tile_of(const GemmParams& p, int n, GemmTile& t) {
  if (p.tiles) {
    const int k = p.cta_off[blockIdx.x] + n;
    if (k >= p.cta_off[blockIdx.x + 1]) return nullptr;
    t = p.tiles[k];
    return p.insts + t.inst;
  }
  const int unit = p.single.share ? 3 : 1;   // a shared-tile chunk is three stages, never cut
  const int S = p.single.kc / unit;
  if (p.streamk) {
    // Stream-K: CTA b owns the K chunks [U b / G, U (b+1) / G) of the U = tiles * S
    // chunks of the whole product, tile by tile; a tile cut between CTAs adds its
    // partial products into the (zeroed) output.
    const int64_t U = static_cast<int64_t>(p.num_tiles) * S;
    const int64_t u0 = U * blockIdx.x / gridDim.x, u1 = U * (blockIdx.x + 1) / gridDim.x;
    const int64_t start = n == 0 ? u0 : (u0 / S + n) * S;
    if (start >= u1) return nullptr;
    const int tile = static_cast<int>(start / S);
    const int64_t end = u1 < static_cast<int64_t>(tile + 1) * S ? u1 : static_cast<int64_t>(tile + 1) * S;
    t.tj = tile % p.single.tiles_n;
    t.ti = tile / p.single.tiles_n;
    t.k0 = unit * static_cast<int>(start - static_cast<int64_t>(tile) * S);
    t.k1 = unit * static_cast<int>(end - static_cast<int64_t>(tile) * S);
    t.red = (t.k0 != 0 || t.k1 != p.single.kc) ? 1 : 0;
    return &p.single;
  }
  const int tile = blockIdx.x + n * gridDim.x;
  if (tile >= p.num_tiles) return nullptr;
  t.tj = tile % p.single.tiles_n;
  t.ti = tile / p.single.tiles_n;
  t.k0 = 0;
  t.k1 = p.single.kc;
  t.red = 0;
  return &p.single;
}

// kMN: the launch may hold MN-major operands (the K-major instantiation carries none of
// their branches).
template <bool kMN>
__global__ void __launch_bounds__(kThreads, 1) gemm_tc_kernel(const __grid_constant__ GemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* sm = smem_raw + (((raw + 1023u) & ~1023u) - raw);
  const int nst = ring_slots(p.slot_rows);
  const uint32_t slot_bytes = kStageP + static_cast<uint32_t>(p.slot_rows) * BK * 2;   // P rows, then Q rows
  uint8_t* stage = sm + kRing;                         // output staging
  uint64_t* bars = reinterpret_cast<uint64_t*>(stage + kStageOut);
  uint64_t* full = bars;
  uint64_t* empty = bars + kMaxStages;
  uint64_t* acc_full = bars + 2 * kMaxStages;
  uint64_t* acc_empty = acc_full + 2;
  uint64_t* drain = acc_empty + 2;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(drain + 1);
  int* vote = reinterpret_cast<int*>(tslot + 4);       // [2][4] epilogue warps' wait outcomes

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (threadIdx.x == 0) {
    for (int s = 0; s < nst; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&acc_full[a], 1);
      mbar_init(&acc_empty[a], 4);
    }
    mbar_init(drain, 1);
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tslot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  pdl_begin();

  if (warp == 0) {
    {
      // ---------------- TMA producer (the whole warp; one lane issues)
      int stage = 0;
      uint32_t phase = 0;
      uint32_t used = 0, last_phase = 0;   // bit s: slot s was filled; the phase of its last fill
      bool ok = true;
      int issued = 0;
      GemmTile T{};
      for (int n = 0; ok; ++n) {
        const GemmInst* I = tile_of(p, n, T);
        if (!I) break;
        // Everything the loop needs, read once: the copies are asm volatile with a memory
        // clobber, so a value read through I would be read again for every one of them,
        // and this thread's chain of loads would set the pace of the whole CTA.
        const CUtensorMap* const mapP = &I->mapP;
        const CUtensorMap* const mapQ = &I->mapQ;
        if (lane == 0) {
          tma_prefetch(mapP);
          tma_prefetch(mapQ);
        }
        __syncwarp();
        const int tj = T.tj, bn = I->bn;
        const int y0 = T.ti * bn;
        const bool conv = I->conv_mode != 0;
        const bool mnP = kMN && I->mnP != 0, mnQ = kMN && I->mnQ != 0;
        const uint32_t stage_bytes = kStageP + static_cast<uint32_t>(bn) * BK * 2;
        const int qchunks = bn / 64;
        // Shared tiles: K chunk c is ring slots 2c (hi P, hi Q) and 2c + 1 (lo P, lo Q).
        const bool share = I->share != 0;
        const int f0 = share ? 2 * share_chunk(T.k0) : T.k0, f1 = share ? 2 * share_chunk(T.k1) : T.k1;
        const int sP0 = I->segP[0], sP1 = I->segP[1], sP2 = I->segP[2];
        const int sQ0 = I->segQ[0], sQ1 = I->segQ[1], sQ2 = I->segQ[2];
        const int e0 = I->nseg > 1 ? I->segKc[0] : 0x7fffffff, e1 = I->nseg > 2 ? e0 + I->segKc[1] : 0x7fffffff;
        for (int kk = f0; kk < f1; ++kk, ++issued) {
          if (issued == p.stall) {  // self-test only: the consumers' bounded waits must run out
            ok = false;
            break;
          }
          if (!mbar_wait_warp(&empty[stage], phase ^ 1u, p.err, DEV_TIMEOUT_EMPTY)) {
            ok = false;
            break;
          }
          int kin, oP, oQ;   // chunk, and the segments' offsets in P and Q
          if (share) {
            kin = kk >> 1;
            oP = (kk & 1) ? sP1 : sP0;
            oQ = (kk & 1) ? sQ2 : sQ0;
          } else {
            kin = kk < e0 ? kk : (kk < e1 ? kk - e0 : kk - e1);
            oP = kk < e0 ? sP0 : (kk < e1 ? sP1 : sP2);
            oQ = kk < e0 ? sQ0 : (kk < e1 ? sQ1 : sQ2);
          }
          const int px = oP + kin * BK;
          // Row-split mode: Q row r, K chunk k lives at row r + k / 2, half k mod 2 of a
          // 128-wide view (the signal segments of a lowered correlation); there a segment's
          // Q offset counts rows (the split residual rows follow the hi rows).
          const int qx = conv ? (kin & 1) * BK : oQ + kin * BK;
          const int qy = conv ? y0 + (kin >> 1) + oQ : y0;
          uint64_t* const bar = &full[stage];
          uint8_t* const dP = sm + stage * slot_bytes;
          uint8_t* const dQ = dP + kStageP;
          if (elect_one()) {
            mbar_arrive_expect_tx(bar, stage_bytes);
            if (mnP) {  // 64-wide MN chunks of 64 K rows (8 KB each)
              tma_load_2d(dP, mapP, bar, tj * BM, px);
              tma_load_2d(dP + 8192, mapP, bar, tj * BM + 64, px);
            } else {
              tma_load_2d(dP, mapP, bar, px, tj * BM);
            }
            if (mnQ) {
              for (int c = 0; c < qchunks; ++c) tma_load_2d(dQ + c * 8192, mapQ, bar, y0 + 64 * c, qx);
            } else {
              tma_load_2d(dQ, mapQ, bar, qx, qy);
            }
          }
          __syncwarp();
          used |= 1u << stage;
          last_phase = (last_phase & ~(1u << stage)) | (phase << stage);
          if (++stage == nst) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      // Every issued copy must land before the CTA may exit.
      for (int s = 0; s < nst; ++s)
        if (lane == 0 && (used >> s & 1u) && !mbar_wait_drain(&full[s], last_phase >> s & 1u))
          atomicCAS(p.err, 0, DEV_TIMEOUT_DRAIN);
    }
  } else if (warp == 1) {
    {
      // ---------------- UMMA issuer (the whole warp; one lane issues)
      const uint32_t slot_units = slot_bytes / 16;
      int stage = 0;
      uint32_t phase = 0;
      int it = 0;
      bool ok = true;
      bool issued_any = false;
      GemmTile T{};
      for (int n = 0; ok; ++n, ++it) {
        const GemmInst* I = tile_of(p, n, T);
        if (!I) break;
        const bool mnP = kMN && I->mnP != 0, mnQ = kMN && I->mnQ != 0;
        const uint32_t idesc = idesc_bf16_f32(BM, I->bn) | (static_cast<uint32_t>(mnP) << 15) |
                               (static_cast<uint32_t>(mnQ) << 16);
        const int acc = it & 1;
        const uint32_t acc_phase = (it >> 1) & 1;
        if (!mbar_wait_warp(&acc_empty[acc], acc_phase ^ 1u, p.err, DEV_TIMEOUT_ACC_FREE)) break;
        tc_fence_after();
        const uint32_t d = tmem + acc * BN;
        // One 64-component product of the P tile in slot sp and the Q tile in slot sq.
        // (A K step of 16 moves a K-major start by 32 bytes, an MN-major one by 2048.)
        const uint32_t a0 = smem_u32(sm);
        const uint64_t bP = mnP ? sdesc_sw128_mn(a0, 8192) : sdesc_sw128(a0, 0);
        const uint64_t bQ = mnQ ? sdesc_sw128_mn(a0 + kStageP, 8192) : sdesc_sw128(a0 + kStageP, 0);
        const uint32_t kP = mnP ? 128 : 2, kQ = mnQ ? 128 : 2;
        auto products = [&](int sp, int sq, bool first) {
          const uint64_t dp = sdesc_advance(bP, sp * slot_units), dq = sdesc_advance(bQ, sq * slot_units);
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)
            umma_f16(d, sdesc_advance(dp, k * kP), sdesc_advance(dq, k * kQ), idesc, !first || (k != 0));
        };
        auto release = [&](int sl) { umma_commit(&empty[sl]); };
        const bool share = I->share != 0;
        const int c0 = share ? share_chunk(T.k0) : T.k0, c1 = share ? share_chunk(T.k1) : T.k1;
        for (int kk = c0; kk < c1; ++kk) {
          if (!mbar_wait_warp(&full[stage], phase, p.err, DEV_TIMEOUT_FULL)) {
            ok = false;
            break;
          }
          tc_fence_after();
          if (elect_one()) {
            products(stage, stage, kk == c0);
            if (!share) release(stage);
          }
          __syncwarp();
          issued_any = true;
          if (share) {  // hi*hi issued; then lo(P)*hi(Q) and hi(P)*lo(Q) from the same four tiles
            const int hi = stage;
            if (++stage == nst) {
              stage = 0;
              phase ^= 1u;
            }
            if (!mbar_wait_warp(&full[stage], phase, p.err, DEV_TIMEOUT_FULL)) {
              ok = false;
              break;
            }
            tc_fence_after();
            if (elect_one()) {
              products(stage, hi, false);
              products(hi, stage, false);
              release(hi);
              release(stage);
            }
            __syncwarp();
          }
          if (++stage == nst) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (ok && elect_one()) umma_commit(&acc_full[acc]);
        __syncwarp();
      }
      // Commit only behind issued MMAs: a commit with nothing to track is never issued.
      if (issued_any) {
        if (elect_one()) umma_commit(drain);
        __syncwarp();
        if (lane == 0 && !mbar_wait_drain(drain, 0)) atomicCAS(p.err, 0, DEV_TIMEOUT_DRAIN);
      }
    }
  } else {
    // ---------------- epilogue: TMEM -> registers -> shared staging -> TMA store
    // (direct stores when Y's pitch does not allow TMA; or the expansion to
    // samples of a gradient product, written straight from registers)
    const int q = warp & 3;  // TMEM lane quadrant this warp may access
    const bool leader = warp == 2 && lane == 0;
    bool pending = false;
    __shared__ float s_coef[64];
    // read once: the stores go through generic pointers, after which values read
    // through a pointer to the parameters would be read again
    const ExpandArgs ex = p.ex;
    if (ex.mode) {
      const int ncoef = 8 * ex.lp1;
      for (int e = threadIdx.x - 64; e < ncoef; e += 128)
        s_coef[e] = ex.coef ? ex.coef[e] : p.ex_c8.c[expand_c8_index(ex, e)];
      named_barrier(1, 128);
    }
    int it = 0;
    GemmTile T{};
    for (int n = 0;; ++n, ++it) {
      const GemmInst* I = tile_of(p, n, T);
      if (!I) break;
      const int ti = T.ti, tj = T.tj;
      const bool red = T.red != 0;
      const int acc = it & 1;
      const uint32_t acc_phase = (it >> 1) & 1;
      const bool okw = __all_sync(0xffffffffu, mbar_wait(&acc_full[acc], acc_phase, p.err, DEV_TIMEOUT_ACC));
      // The four epilogue warps take the same decision, so none is left alone at a barrier.
      if (lane == 0) vote[(it & 1) * 4 + q] = okw ? 1 : 0;
      named_barrier(1, 128);
      const int* v = vote + (it & 1) * 4;
      if (!(v[0] && v[1] && v[2] && v[3])) break;
      tc_fence_after();
      // read once: the stores go through generic pointers, after which a field read
      // through I would be read again
      const int M = I->M, N = I->N, bn = I->bn;
      const bool out_bf16 = I->out_bf16 != 0;
      const int64_t ldy = I->ldy;
      void* const Yout = I->Y;
      const int tma_rows = I->tma_out && (tj + 1) * BM <= I->tma_cols ? I->tma_rows : 0;
      const int jl = q * 32 + lane;
      const int j = tj * BM + jl;
      const bool jok = j < N;
      if (ex.mode) {
        // Y[i][j] (i: row of Q, j: row of P) expanded to samples: mode 1 has the
        // components on j (N = their count), mode 2 on i (M = their count).
        const int ncomp = ex.mode == 1 ? N : M;
        expand_tile(tmem + acc * BN + (static_cast<uint32_t>(q * 32) << 16), I->bn, ex, s_coef, lane, j, ncomp,
                    ti * I->bn, M, j, jok);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[acc]);
        continue;
      }
      for (int c0 = 0; c0 < bn; c0 += 32) {
        uint32_t r[32];
        tmem_ld_x32(tmem + acc * BN + c0 + (static_cast<uint32_t>(q * 32) << 16), r);
        tmem_wait_ld();
        const int i0 = ti * bn + c0;
        if (i0 >= M) continue;  // uniform: no rows of this chunk exist
        if (i0 + 32 <= tma_rows) {
          if (leader && pending) bulk_wait_read_all();
          named_barrier(1, 128);  // staging free
          if (out_bf16) {
            __nv_bfloat16* st = reinterpret_cast<__nv_bfloat16*>(stage);
#pragma unroll
            for (int u = 0; u < 32; ++u) st[u * BM + jl] = __float2bfloat16_rn(__uint_as_float(r[u]));
          } else {
            float* st = reinterpret_cast<float*>(stage);
#pragma unroll
            for (int u = 0; u < 32; ++u) st[u * BM + jl] = __uint_as_float(r[u]);
          }
          fence_proxy_async_smem();
          named_barrier(1, 128);  // staging written
          if (leader) {
            if (red)
              tma_reduce_add_2d(&I->mapY, stage, tj * BM, i0);
            else
              tma_store_2d(&I->mapY, stage, tj * BM, i0);
            bulk_commit_group();
            pending = true;
          }
        } else if (I->conv_mode) {
          // lowered correlation: element (i, j) is output sample i * 128 + j of this phase
          store_samples<32>(r, static_cast<float*>(Yout), I->conv_stride, I->conv_limit, i0, j, jok);
        } else if (jok) {
          store_rows<32>(r, Yout, ldy, out_bf16, red, i0, M, j);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[acc]);
    }
    if (leader && pending) bulk_wait_all();
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

}  // namespace

bool build_gemm_inst(const GemmTcArgs& a, GemmInst* I) {
  memset(I, 0, sizeof(GemmInst));
  if ((a.mnQ && (a.bn % 64 || a.conv_mode)) || (a.mnP && a.conv_mode)) return false;
  if (a.mnP) {  // stored as xdim K rows of rowsP values: boxes of 64 values x 64 K rows
    const uint64_t dims[2] = {static_cast<uint64_t>(a.rowsP), static_cast<uint64_t>(a.xdim)};
    const uint64_t strides[1] = {static_cast<uint64_t>(a.ldp) * 2};
    const uint32_t box[2] = {64, BK};
    if (!make_tmap_bf16(&I->mapP, a.P, 2, dims, strides, box)) return false;
  } else {
    const uint64_t dims[2] = {static_cast<uint64_t>(a.xdim), static_cast<uint64_t>(a.rowsP)};
    const uint64_t strides[1] = {static_cast<uint64_t>(a.ldp) * 2};
    const uint32_t box[2] = {BK, BM};
    if (!make_tmap_bf16(&I->mapP, a.P, 2, dims, strides, box)) return false;
  }
  if (a.mnQ) {
    const uint64_t dims[2] = {static_cast<uint64_t>(a.rowsQ), static_cast<uint64_t>(a.xdim)};
    const uint64_t strides[1] = {static_cast<uint64_t>(a.ldq) * 2};
    const uint32_t box[2] = {64, BK};
    if (!make_tmap_bf16(&I->mapQ, a.Q, 2, dims, strides, box)) return false;
  } else {
    const uint64_t dims[2] = {static_cast<uint64_t>(a.conv_mode ? BM : a.xdim),
                              static_cast<uint64_t>(a.conv_mode ? a.q_rows_alloc : a.rowsQ)};
    const uint64_t strides[1] = {static_cast<uint64_t>(a.ldq) * 2};
    const uint32_t box[2] = {BK, static_cast<uint32_t>(a.pair ? a.bn / 2 : a.bn)};
    if (!make_tmap_bf16(&I->mapQ, a.Q, 2, dims, strides, box)) return false;
  }
  I->bn = a.bn;
  I->mnQ = a.mnQ;
  I->mnP = a.mnP;
  I->Y = a.Y;
  I->ldy = a.ldy;
  I->out_bf16 = a.out_dtype == PJ_BF16;
  I->M = static_cast<int>(a.rowsQ);
  I->N = static_cast<int>(a.rowsP);
  I->nseg = a.nseg;
  I->kc = 0;
  for (int s = 0; s < 3; ++s) {
    I->segP[s] = static_cast<int>(a.segP[s]);
    I->segQ[s] = static_cast<int>(a.segQ[s]);
    I->segKc[s] = s < a.nseg ? static_cast<int>(ceil_div(a.segK[s] ? a.segK[s] : a.kdim, BK)) : 0;
    I->kc += I->segKc[s];
  }
  // The plain split's three segments (hi*hi, lo(P)*hi(Q), hi(P)*lo(Q)) share their
  // tiles: four loads per K chunk instead of six (see GemmInst::share).
  I->share = a.nseg == 3 && I->segKc[0] == I->segKc[1] && I->segKc[1] == I->segKc[2] && I->segP[0] == I->segP[2] &&
             I->segQ[0] == I->segQ[1];
  I->tiles_n = static_cast<int>(ceil_div(a.rowsP, BM));
  I->conv_mode = a.conv_mode;
  I->conv_stride = a.conv_stride;
  I->conv_limit = a.conv_limit;
  I->tma_out = 0;
  I->tma_rows = static_cast<int>(a.rowsQ);
  I->tma_cols = 1 << 30;
  const size_t es = I->out_bf16 ? 2 : 4;
  if (a.conv_mode) {
    // contiguous output rows of 128 samples only when samples are adjacent in memory
    const int64_t full_rows = a.conv_limit / BM;
    if (a.conv_stride == 1 && !I->out_bf16 && full_rows > 0 && reinterpret_cast<uintptr_t>(a.Y) % 16 == 0) {
      const uint64_t dims[2] = {static_cast<uint64_t>(BM), static_cast<uint64_t>(full_rows)};
      const uint64_t strides[1] = {static_cast<uint64_t>(BM) * 4};
      const uint32_t box[2] = {BM, 32};
      I->tma_out = make_tmap_f32(&I->mapY, a.Y, 2, dims, strides, box) ? 1 : 0;
      I->tma_rows = static_cast<int>(full_rows);
    }
  } else if ((a.ldy * es) % 16 == 0 && reinterpret_cast<uintptr_t>(a.Y) % 16 == 0) {
    const uint64_t dims[2] = {static_cast<uint64_t>(a.rowsP), static_cast<uint64_t>(a.rowsQ)};
    const uint64_t strides[1] = {static_cast<uint64_t>(a.ldy) * es};
    const uint32_t box[2] = {BM, 32};
    I->tma_out = (I->out_bf16 ? make_tmap_bf16_plain(&I->mapY, a.Y, 2, dims, strides, box)
                              : make_tmap_f32(&I->mapY, a.Y, 2, dims, strides, box)) ? 1 : 0;
    I->tma_rows = 1 << 30;   // TMA clips ragged rows itself
    if ((a.rowsP * static_cast<int64_t>(es)) % 16) I->tma_cols = static_cast<int>(a.rowsP);
  }
  return true;
}

// K stages of all segments of a product.
static int args_stages(const GemmTcArgs& a) {
  int n = 0;
  for (int s = 0; s < a.nseg && s < 3; ++s) n += static_cast<int>(ceil_div(a.segK[s] ? a.segK[s] : a.kdim, BK));
  return n;
}

int gemm_tiles_of(const GemmInst& I) { return I.tiles_n * static_cast<int>(ceil_div(I.M, I.bn)); }

static cudaError_t set_smem_attr() {
  static bool done[64] = {false};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
  const int bytes = static_cast<int>(kSmemBytes);
  e = cudaFuncSetAttribute(gemm_tc_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gemm_tc_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = true;
  return e;
}

cudaError_t launch_gemm_tc_generic(const GemmTcArgs& a_in, int* err, int num_sms, cudaStream_t st) {
  GemmParams p;
  if (a_in.rowsQ == 0 || a_in.rowsP == 0) return cudaSuccess;
  GemmTcArgs a = a_in;
  if (!a.conv_mode)
    a.bn = single_launch_bn(a.rowsQ, ceil_div(a.rowsP, BM), args_stages(a), num_sms, a.mnQ ? 64 : 32, BN);
  const int64_t tiles_n = ceil_div(a.rowsP, BM);
  const int64_t tiles = tiles_n * ceil_div(a.rowsQ, a.bn);
  // (the expansion writes samples, which partial products could not be added into)
  const bool streamk = !a.conv_mode && !a.ex.mode && a.out_dtype != PJ_BF16 &&
                       use_stream_k(tiles, args_stages(a), num_sms, a.nseg > 1);
  // 256-row tiles on 2-SM MMAs wherever the tile columns pair up (gemm_cg2.cu).
  if (!streamk && gemm_cg2_eligible(a, num_sms)) return launch_gemm_cg2(a, err, num_sms, st);
  if (!build_gemm_inst(a, &p.single)) return cudaErrorInvalidValue;
  p.insts = nullptr;
  p.tiles = nullptr;
  p.cta_off = nullptr;
  p.num_tiles = gemm_tiles_of(p.single);
  p.slot_rows = a.bn;
  p.err = err;
  p.stall = a.stall_stage;
  p.ex = a.ex;
  p.ex_c8 = a.ex_c8 ? *a.ex_c8 : Coef8{};
  cudaError_t e = set_smem_attr();
  if (e != cudaSuccess) return e;
  int grid = p.num_tiles < num_sms ? p.num_tiles : num_sms;
  p.streamk = 0;
  if (streamk) {
    e = cudaMemset2DAsync(a.Y, a.ldy * 4, 0, a.rowsP * 4, a.rowsQ, st);
    if (e != cudaSuccess) return e;
    p.streamk = 1;
    grid = num_sms;
  }
  return launch_pdl(a.mnP || a.mnQ ? gemm_tc_kernel<true> : gemm_tc_kernel<false>,
                    dim3(static_cast<unsigned>(grid)), kThreads, kSmemBytes, st, 1, p);
}

cudaError_t launch_gemm_tc_grouped(const GemmInst* insts, const GemmTile* tiles, const int* cta_off, int ctas,
                                   int* err, cudaStream_t st) {
  if (ctas == 0) return cudaSuccess;
  GemmParams p;
  memset(&p.single, 0, sizeof(GemmInst));
  p.insts = insts;
  p.tiles = tiles;
  p.cta_off = cta_off;
  p.num_tiles = 0;
  p.streamk = 0;
  p.slot_rows = BN;   // instances of any height share the ring
  p.stall = -1;
  p.err = err;
  p.ex = ExpandArgs{};
  p.ex_c8 = Coef8{};
  cudaError_t e = set_smem_attr();
  if (e != cudaSuccess) return e;
  // grouped instances are K-major
  return launch_pdl(gemm_tc_kernel<false>, dim3(static_cast<unsigned>(ctas)), kThreads, kSmemBytes, st, 1, p);
}

cudaError_t launch_gemm_tc(const uint16_t* Ac, const uint16_t* Bd, void* Y, int64_t ldy, int out_dtype,
                           const GemmGeom& g, int* err, int num_sms, cudaStream_t st) {
  GemmTcArgs a;
  const int64_t pitch = gemm_pitch(g);
  a.Q = Ac;
  a.ldq = pitch;
  a.rowsQ = g.M;
  a.P = Bd;
  a.ldp = pitch;
  a.rowsP = g.N;
  a.xdim = pitch;      // components are zero-padded inside each segment
  a.kdim = g.Kp_pad;
  a.Y = Y;
  a.ldy = ldy;
  a.out_dtype = out_dtype;
  if (g.nsplit == 1) {
    a.nseg = 1;
    a.segP[0] = a.segQ[0] = 0;
  } else if (!gemm_tiered(g)) {  // hi*hi + hi(A)*lo(B) + lo(A)*hi(B)
    a.nseg = 3;
    a.segQ[0] = 0;        a.segP[0] = 0;
    a.segQ[1] = 0;        a.segP[1] = g.Kp_pad;
    a.segQ[2] = g.Kp_pad; a.segP[2] = 0;
  } else {  // hi*hi over every component, then hi*lo and lo*hi over the lead ones
    const int64_t hl = g.Kp_pad, ll = g.Kp_pad + g.Kt_pad;
    a.nseg = 3;
    a.segQ[0] = 0;  a.segP[0] = 0;  a.segK[0] = g.Kp_pad;
    a.segQ[1] = hl; a.segP[1] = ll; a.segK[1] = g.Kt_pad;
    a.segQ[2] = ll; a.segP[2] = hl; a.segK[2] = g.Kt_pad;
  }
  return launch_gemm_tc_generic(a, err, num_sms, st);
}

}  // namespace pj
