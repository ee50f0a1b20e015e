// Reduced GEMM of a single product on 2-SM MMAs (tcgen05.mma.cta_group::2):
// the same Y[i][j] = sum_k A_c[i][k] B_d[j][k] as gemm_tc.cu (the (l+1)
// smaller products of Sec. III-B, accumulated over blocks as in Eq. 2 and
// Eq. 8), with the two CTAs of a cluster acting as one 256-row MMA.
//
// Why: a CTA of gemm_tc.cu keeps its whole 128 x 256 operand pair in shared
// memory per K stage (48 KB), so four stages hold about 1 us of MMA work -- less
// than the time a TMA load from L2 takes under load on this GPU, and the tensor
// pipe waits.  In a 2-SM MMA the pair computes a 256 x N tile and each CTA holds
// only its 128 rows of P and N/2 rows of Q: 32 KB per stage, so six stages fit
// and the same shared memory covers 1.5x the MMA time.
//
// Tile: the pair takes P rows [256 c, 256 c + 256) (CTA r: its 128) and Q rows
// [bn t, bn t + bn) (CTA r loads bn/2 of them); each CTA's tensor memory holds
// the accumulator of its 128 P rows x bn Q rows, so the epilogue is the one of
// gemm_tc.cu, CTA by CTA.  The leader's (rank 0) thread issues every MMA; the
// TMA loads of both CTAs count on the leader's stage barriers, and each MMA
// commit frees the stage in both CTAs.  Both CTAs' epilogue warps arrive on the
// leader's accumulator barriers.
//
// The producer's and the issuer's instruction chains set the pace: with the instance's
// fields read in the loop (again after every copy) and descriptors built per MMA, a slot
// of the 4096 x 2048 product over 12,880 components took 0.34 us whatever was
// prefetched; with everything held in registers it takes 0.30 us (137 -> 122 us, 1.77
// PFLOP/s).
//
// A batch's products run here too (kGrouped): on CTAs of their own (gemm_tc.cu) they
// drew 96 KB of operands per 64-component chunk through SMs that take in about 70 bytes a
// clock each (tc.cuh), and the grouped launch of 40 products and 20 correlations took 818
// us; here it took 64 KB and 733 us at 98 % of the tensor pipe's cycles, under the power
// cap (1.74 GHz).  (The correlations have since moved to a launch of their own, batch.cu.)
#include <cuda_bf16.h>
#include <string.h>

#include "common.hpp"
#include "gemm_epi.cuh"
#include "pdl.cuh"
#include "tc.cuh"
#include "tmap.hpp"
#if PJ_CTA_PAIRS
#include "tc_pair.cuh"
#endif

namespace pj {

#if PJ_CTA_PAIRS
namespace {

constexpr int CM = 128;   // P rows per CTA (the pair's MMA M is 256)
constexpr int CN = 256;   // most Q rows per pair tile (MMA N); each CTA holds half
constexpr int CK = 64;
// The ring holds as many slots as its memory takes: six at 256 Q rows, eight at 128.
constexpr int kCMaxStages = 8;
// warp 0: TMA producer; warp 1: MMA issuer (leader CTA); warps 2-9: epilogue.
// Eight epilogue warps (two per TMEM lane quadrant) split an expansion tile's
// columns in halves; the plain epilogue runs on warps 2-5.
constexpr int kCThreads = 320;
constexpr uint32_t kCStageP = CM * CK * 2;
// Output staging of the TMA-store epilogue: 32 KB, four 32-column chunks of BF16
// or two of FP32 in flight, so a chunk is staged while earlier ones are stored.
constexpr uint32_t kCStageOut = 2 * 32 * CM * 4;
constexpr uint32_t kCCtl = 320;
constexpr uint32_t kCRing = 6 * (kCStageP + (CN / 2) * CK * 2);
constexpr size_t kCSmemBytes = 1024 + kCRing + kCStageOut + kCCtl;
static_assert(kCSmemBytes + 64 * sizeof(float) <= 232448, "shared memory per block (dynamic + static)");

__host__ __device__ constexpr int cg2_slots(int bn) {
  const int n = static_cast<int>(kCRing / (kCStageP + static_cast<uint32_t>(bn / 2) * CK * 2));
  return n < kCMaxStages ? n : kCMaxStages;
}

struct Cg2Params {
  GemmInst I;       // P map box {CK, CM} (MN-major: {64, CK}); Q map box {CK, bn/2} (MN-major: {64, CK})
  const GemmInst* insts;   // grouped launch: the instances, the tiles pair by pair (tj counts pair
  const GemmTile* tiles;   // columns), and where each pair's tiles start
  const int* pair_off;
  int slot_rows;    // tile height the ring slots are sized for (the instance's, or 256 when grouped)
  ExpandArgs ex;
  Coef8 ex_c8;      // the expansion's vectors when ex.coef is null
  int npp;          // pair columns: P tile columns of 256
  int num_pairs;    // npp x Q tile rows
  int stall;        // failure-detection self-test: the producers stop after this many stages (-1: never)
  int* err;
};

// The n-th tile of this pair: instance, pair column tj, tile row ti and K-stage range;
// null past the last.
template <bool kGrouped>
__device__ __forceinline__ const GemmInst* cg2_tile(const Cg2Params& p, int n, GemmTile& t) {
  if (kGrouped) {
    const int k = p.pair_off[blockIdx.x / 2] + n;
    if (k >= p.pair_off[blockIdx.x / 2 + 1]) return nullptr;
    t = p.tiles[k];
    return p.insts + t.inst;
  }
  const int pi = static_cast<int>(blockIdx.x / 2) + n * static_cast<int>(gridDim.x / 2);
  if (pi >= p.num_pairs) return nullptr;
  t.tj = pi % p.npp;
  t.ti = pi / p.npp;
  t.k0 = 0;
  t.k1 = p.I.kc;
  t.red = 0;
  return &p.I;
}

// kGrouped: the batch's launch, many instances (K-major, no expansion) over planned tile
// lists; see launch_gemm_cg2_grouped.
template <bool kMN, bool kGrouped>
__global__ void __launch_bounds__(kCThreads, 1) gemm_cg2_kernel(const __grid_constant__ Cg2Params p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* sm = smem_raw + (((raw + 1023u) & ~1023u) - raw);
  const int nst = cg2_slots(p.slot_rows);
  const uint32_t slot_bytes = kCStageP + static_cast<uint32_t>(p.slot_rows / 2) * CK * 2;   // P rows, then Q rows
  uint8_t* stage_out = sm + kCRing;
  uint64_t* bars = reinterpret_cast<uint64_t*>(stage_out + kCStageOut);
  uint64_t* full = bars;
  uint64_t* empty = bars + kCMaxStages;
  uint64_t* acc_full = bars + 2 * kCMaxStages;
  uint64_t* acc_empty = acc_full + 2;
  uint64_t* drain = acc_empty + 2;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(drain + 1);
  int* vote = reinterpret_cast<int*>(tslot + 4);   // 2 x 8 flags
  static_assert((2 * kCMaxStages + 5) * 8 + 16 + 16 * 4 <= kCCtl, "barriers, TMEM slot and votes");
  __shared__ float s_coef[64];

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < nst; ++s) {
      mbar_init(&full[s], 1);    // the leader's expect_tx; both CTAs' copies count their bytes on it
      mbar_init(&empty[s], 1);   // the leader's MMA commit, delivered to both CTAs
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&acc_full[a], 1);
      mbar_init(&acc_empty[a], 16);  // eight epilogue warps in each CTA (the leader's is used)
    }
    mbar_init(drain, 1);
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc_cg2(tslot, 512);
    tmem_relinquish_cg2();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // both CTAs' barriers exist before any copy, commit or remote arrive reaches them
  tc_fence_after();
  const uint32_t tmem = *tslot;
  const uint32_t full_leader = mapa_shared(smem_u32(full), 0);
  const uint32_t acc_empty_leader = mapa_shared(smem_u32(acc_empty), 0);
  pdl_begin();

  if (warp == 0) {
    {
      // ---------------- TMA producer (both CTAs; the whole warp, one lane issues): this
      // CTA's P rows and half of the Q rows
      int stage = 0;
      uint32_t phase = 0;
      uint32_t used = 0, last_phase = 0;   // bit s: slot s was filled; the phase of its last fill
      bool ok = true;
      int issued = 0;
      const int stall = p.stall;
      GemmTile T{};
      for (int n = 0; ok; ++n) {
        const GemmInst* I = cg2_tile<kGrouped>(p, n, T);
        if (!I) break;
        // read once (see gemm_tc.cu: a value read through I would be read again after every copy)
        const CUtensorMap* const mapP = &I->mapP;
        const CUtensorMap* const mapQ = &I->mapQ;
        if (lane == 0 && (kGrouped || n == 0)) {
          tma_prefetch(mapP);
          tma_prefetch(mapQ);
        }
        __syncwarp();
        const int bn = I->bn, half = bn / 2;
        const bool mnP = kMN && I->mnP != 0, mnQ = kMN && I->mnQ != 0;
        const bool share = I->share != 0;   // hi and lo tiles in alternate slots (GemmInst::share)
        const int f0 = share ? 2 * share_chunk(T.k0) : T.k0, f1 = share ? 2 * share_chunk(T.k1) : T.k1;
        const int sP0 = I->segP[0], sP1 = I->segP[1], sP2 = I->segP[2];
        const int sQ0 = I->segQ[0], sQ1 = I->segQ[1], sQ2 = I->segQ[2];
        const int e0 = I->nseg > 1 ? I->segKc[0] : 0x7fffffff, e1 = I->nseg > 2 ? e0 + I->segKc[1] : 0x7fffffff;
        const uint32_t pair_bytes = 2 * (kCStageP + static_cast<uint32_t>(half) * CK * 2);
        const int prow = T.tj * 2 * CM + static_cast<int>(rank) * CM;
        const int qrow = T.ti * bn + static_cast<int>(rank) * half;
        for (int kk = f0; kk < f1; ++kk, ++issued) {
          if (issued == stall) {
            ok = false;
            break;
          }
          if (!mbar_wait_warp(&empty[stage], phase ^ 1u, p.err, DEV_TIMEOUT_EMPTY)) {
            ok = false;
            break;
          }
          int kin, oP, oQ;
          if (share) {
            kin = kk >> 1;
            oP = (kk & 1) ? sP1 : sP0;
            oQ = (kk & 1) ? sQ2 : sQ0;
          } else {
            kin = kk < e0 ? kk : (kk < e1 ? kk - e0 : kk - e1);
            oP = kk < e0 ? sP0 : (kk < e1 ? sP1 : sP2);
            oQ = kk < e0 ? sQ0 : (kk < e1 ? sQ1 : sQ2);
          }
          const int px = oP + kin * CK;
          const int qx = oQ + kin * CK;
          const uint32_t bar = full_leader + stage * 8;
          uint8_t* const dP = sm + stage * slot_bytes;
          uint8_t* const dQ = dP + kCStageP;
          if (elect_one()) {
            if (leader) mbar_arrive_expect_tx(&full[stage], pair_bytes);
            if (mnP) {
              tma_load_2d_cg2(dP, mapP, bar, prow, px);
              tma_load_2d_cg2(dP + 8192, mapP, bar, prow + 64, px);
            } else {
              tma_load_2d_cg2(dP, mapP, bar, px, prow);
            }
            if (mnQ) {
              for (int c = 0; c < half / 64; ++c) tma_load_2d_cg2(dQ + c * 8192, mapQ, bar, qrow + 64 * c, qx);
            } else {
              tma_load_2d_cg2(dQ, mapQ, bar, qx, qrow);
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
      // The leader's barriers count both CTAs' copies: once the leader has seen every
      // issued phase complete, no copy of either CTA is still writing shared memory
      // (the peer leaves only after the cluster barrier below).
      if (leader && lane == 0)
        for (int s = 0; s < nst; ++s)
          if ((used >> s & 1u) && !mbar_wait_drain(&full[s], last_phase >> s & 1u))
            atomicCAS(p.err, 0, DEV_TIMEOUT_DRAIN);
    }
  } else if (warp == 1) {
    if (leader) {
      // ---------------- MMA issuer (the leader's whole warp; one lane issues)
      const uint32_t a0 = smem_u32(sm), slot_units = slot_bytes / 16;
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      bool issued_any = false;
      GemmTile T{};
      for (int n = 0, it = 0; ok; ++n, ++it) {
        const GemmInst* I = cg2_tile<kGrouped>(p, n, T);
        if (!I) break;
        const bool mnP = kMN && I->mnP != 0, mnQ = kMN && I->mnQ != 0;
        const uint32_t idesc = idesc_bf16_f32(2 * CM, I->bn) | (static_cast<uint32_t>(mnP) << 15) |
                               (static_cast<uint32_t>(mnQ) << 16);
        // (A K step of 16 moves a K-major start by 32 bytes, an MN-major one by 2048.)
        const uint64_t bP = mnP ? sdesc_sw128_mn(a0, 8192) : sdesc_sw128(a0, 0);
        const uint64_t bQ = mnQ ? sdesc_sw128_mn(a0 + kCStageP, 8192) : sdesc_sw128(a0 + kCStageP, 0);
        const uint32_t kP = mnP ? 128 : 2, kQ = mnQ ? 128 : 2;
        const bool share = I->share != 0;
        const int c0 = share ? share_chunk(T.k0) : T.k0, c1 = share ? share_chunk(T.k1) : T.k1;
        const int acc = it & 1;
        const uint32_t acc_phase = (it >> 1) & 1;
        if (!mbar_wait_warp(&acc_empty[acc], acc_phase ^ 1u, p.err, DEV_TIMEOUT_ACC_FREE)) break;
        tc_fence_after();
        const uint32_t d = tmem + acc * CN;
        // One 64-component product of the P tiles in slot sp and the Q tiles in slot sq.
        auto products = [&](int sp, int sq, bool first) {
          const uint64_t dp = sdesc_advance(bP, sp * slot_units), dq = sdesc_advance(bQ, sq * slot_units);
#pragma unroll
          for (int k = 0; k < CK / 16; ++k)
            umma_f16_cg2(d, sdesc_advance(dp, k * kP), sdesc_advance(dq, k * kQ), idesc, !first || (k != 0));
        };
        for (int kk = c0; kk < c1; ++kk) {
          if (!mbar_wait_warp(&full[stage], phase, p.err, DEV_TIMEOUT_FULL)) {
            ok = false;
            break;
          }
          tc_fence_after();
          if (elect_one()) {
            products(stage, stage, kk == c0);
            if (!share) umma_commit_cg2_mc(&empty[stage], 0x3);
          }
          __syncwarp();
          issued_any = true;
          if (share) {
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
              umma_commit_cg2_mc(&empty[hi], 0x3);
              umma_commit_cg2_mc(&empty[stage], 0x3);
            }
            __syncwarp();
          }
          if (++stage == nst) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (ok && elect_one()) umma_commit_cg2_mc(&acc_full[acc], 0x3);
        __syncwarp();
      }
      if (issued_any) {
        if (elect_one()) umma_commit_cg2_mc(drain, 0x1);
        __syncwarp();
        if (lane == 0 && !mbar_wait_drain(drain, 0)) atomicCAS(p.err, 0, DEV_TIMEOUT_DRAIN);
      }
    }
  } else {
    // ---------------- epilogue (both CTAs): this CTA's 128 P rows of the accumulator
    const int ew = warp - 2;   // epilogue warp 0..7
    const int q = warp & 3;    // the TMEM lane quadrant this warp may read
    const int h = ew >> 2;     // the half of an expansion tile's columns it expands
    const bool store_leader = warp == 2 && lane == 0;
    bool pending = false;
    // Everything the stores need, read from the parameters once: the stores go
    // through generic pointers, so values read through a pointer to the
    // parameters would be read again after every store.
    const ExpandArgs ex = kGrouped ? ExpandArgs{} : p.ex;
    int sbuf = 0, last_nbuf = 0;
    bool relaid = false;
    if (ex.mode)
      for (int e = threadIdx.x - 64; e < 8 * ex.lp1; e += 256)
        s_coef[e] = ex.coef ? ex.coef[e] : p.ex_c8.c[expand_c8_index(ex, e)];
    named_barrier(1, 256);
    GemmTile T{};
    for (int n = 0, it = 0;; ++n, ++it) {
      const GemmInst* I = cg2_tile<kGrouped>(p, n, T);
      if (!I) break;
      const int ti = T.ti, tj = T.tj * 2 + static_cast<int>(rank);
      const bool red = T.red != 0;
      const int M = I->M, N = I->N, bn = I->bn;
      const bool out_bf16 = I->out_bf16 != 0;
      const int tma_rows = I->tma_out && (tj + 1) * CM <= I->tma_cols ? I->tma_rows : 0;
      const int64_t ldy = I->ldy;
      void* const Yout = I->Y;
      const uint32_t chunk_bytes = 32u * CM * (out_bf16 ? 2u : 4u);
      const int nbuf = static_cast<int>(kCStageOut / chunk_bytes);
      // another element size lays the staging out anew: the next store waits for all under way
      if (kGrouped && last_nbuf != 0 && nbuf != last_nbuf) {
        relaid = true;
        sbuf = 0;
      }
      last_nbuf = nbuf;
      const int acc = it & 1;
      const uint32_t acc_phase = (it >> 1) & 1;
      const bool okw = __all_sync(0xffffffffu, mbar_wait(&acc_full[acc], acc_phase, p.err, DEV_TIMEOUT_ACC));
      if (lane == 0) vote[(it & 1) * 8 + ew] = okw ? 1 : 0;
      named_barrier(1, 256);
      const int* v = vote + (it & 1) * 8;
      bool all_ok = true;
#pragma unroll
      for (int w = 0; w < 8; ++w) all_ok = all_ok && v[w] != 0;
      if (!all_ok) break;
      tc_fence_after();
      const int jl = q * 32 + lane;
      const int j = tj * CM + jl;
      const bool jok = j < N;
      if (ex.mode) {
        const int ncomp = ex.mode == 1 ? N : M;
        const int hb = bn / 2;   // a multiple of 16
        expand_tile(tmem + acc * CN + h * hb + (static_cast<uint32_t>(q * 32) << 16), hb, ex, s_coef, lane,
                    j, ncomp, ti * bn + h * hb, M, j, jok);
      }
      // (a pair's second column past an odd number of columns writes nothing)
      for (int c0 = 0; c0 < (ex.mode || h || tj * CM >= N ? 0 : bn); c0 += 32) {
        uint32_t r[32];
        tmem_ld_x32(tmem + acc * CN + c0 + (static_cast<uint32_t>(q * 32) << 16), r);
        tmem_wait_ld();
        const int i0 = ti * bn + c0;
        if (i0 >= M) continue;  // uniform: no rows of this chunk exist
        if (i0 + 32 <= tma_rows) {
          // buffer sbuf was last read by the store nbuf chunks ago
          if (store_leader && pending) {
            if (relaid) bulk_wait_read_all();
            else if (nbuf == 4) bulk_wait_read_3();
            else bulk_wait_read_1();
          }
          relaid = false;
          named_barrier(2, 128);  // staging buffer free
          uint8_t* buf = stage_out + sbuf * chunk_bytes;
          if (out_bf16) {
            __nv_bfloat16* st = reinterpret_cast<__nv_bfloat16*>(buf);
#pragma unroll
            for (int u = 0; u < 32; ++u) st[u * CM + jl] = __float2bfloat16_rn(__uint_as_float(r[u]));
          } else {
            float* st = reinterpret_cast<float*>(buf);
#pragma unroll
            for (int u = 0; u < 32; ++u) st[u * CM + jl] = __uint_as_float(r[u]);
          }
          fence_proxy_async_smem();
          named_barrier(2, 128);  // staging written
          if (store_leader) {
            if (kGrouped && red)
              tma_reduce_add_2d(&I->mapY, buf, tj * CM, i0);
            else
              tma_store_2d(&I->mapY, buf, tj * CM, i0);
            bulk_commit_group();
            pending = true;
          }
          if (++sbuf == nbuf) sbuf = 0;
        } else if (jok) {
          store_rows<32>(r, Yout, ldy, out_bf16, kGrouped && red, i0, M, j);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(acc_empty_leader + acc * 8);
    }
    if (store_leader && pending) bulk_wait_all();
  }

  tc_fence_before();
  __syncthreads();
  // Neither CTA leaves while the leader's MMAs or the other CTA's copies may still
  // reach its shared or tensor memory.
  cluster_sync_all();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc_cg2(tmem, 512);
  }
}

cudaError_t set_cg2_smem_attr() {
  static bool done[64] = {false};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
  const int bytes = static_cast<int>(kCSmemBytes);
  e = cudaFuncSetAttribute(gemm_cg2_kernel<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gemm_cg2_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gemm_cg2_kernel<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = true;
  return e;
}

}  // namespace

// Rows of Q per pair tile: the height whose whole waves of pair tiles over the SM
// pairs finish first (each pair tile counted as its K stages scaled by its height
// plus a fixed cost of 4 stages); a multiple of 32 (of 128 for an MN-major Q, whose
// halves are whole 64-row chunks).
static int cg2_bn(int64_t rowsQ, int64_t pair_cols, int64_t stages, int sms, bool mnQ) {
  const int gran = mnQ ? 128 : 32;
  int best = CN;
  double best_t = 0;
  for (int bn = CN; bn >= (mnQ ? 128 : 64); bn -= gran) {
    const int64_t tiles = (rowsQ + bn - 1) / bn * pair_cols;
    const int64_t waves = (tiles + sms / 2 - 1) / (sms / 2);
    const double t = static_cast<double>(waves) * (static_cast<double>(stages) * bn / 256.0 + 4.0);
    if (bn == CN || t < best_t * 0.99) {
      best = bn;
      best_t = t;
    }
  }
  return best;
}

bool gemm_cg2_eligible(const GemmTcArgs& a, int num_sms) {
  return !a.conv_mode && num_sms >= 2 && a.rowsP > 0 && ceil_div(a.rowsP, CM) % 2 == 0;
}

static int cg2_stages(const GemmTcArgs& a) {
  int stages = 0;
  for (int s = 0; s < a.nseg && s < 3; ++s) stages += static_cast<int>(ceil_div(a.segK[s] ? a.segK[s] : a.kdim, CK));
  return stages;
}

static cudaError_t launch_cg2(Cg2Params& p, bool mn, int num_sms, cudaStream_t st) {
  cudaError_t e = set_cg2_smem_attr();
  if (e != cudaSuccess) return e;
  const int slots = num_sms / 2;
  return launch_pdl(mn ? gemm_cg2_kernel<true, false> : gemm_cg2_kernel<false, false>,
                    dim3(static_cast<unsigned>(2 * (p.num_pairs < slots ? p.num_pairs : slots))), kCThreads, kCSmemBytes,
                    st, 2, p);
}

cudaError_t launch_gemm_cg2(const GemmTcArgs& a_in, int* err, int num_sms, cudaStream_t st) {
  GemmTcArgs a = a_in;
  const int64_t pair_cols = ceil_div(a.rowsP, CM) / 2;
  a.bn = cg2_bn(a.rowsQ, pair_cols, cg2_stages(a), num_sms, a.mnQ != 0);
  a.pair = 1;   // Q boxes of bn/2 rows (K-major), one CTA's half of the tile
  Cg2Params p{};
  if (!build_gemm_inst(a, &p.I)) return cudaErrorInvalidValue;
  p.npp = static_cast<int>(pair_cols);
  p.num_pairs = static_cast<int>(pair_cols * ceil_div(a.rowsQ, a.bn));
  p.slot_rows = a.bn;
  p.stall = a.stall_stage;
  p.err = err;
  p.ex = a.ex;
  if (a.ex_c8) p.ex_c8 = *a.ex_c8;
  return launch_cg2(p, a.mnP || a.mnQ, num_sms, st);
}

cudaError_t launch_gemm_cg2_grouped(const GemmInst* insts, const GemmTile* tiles, const int* pair_off, int pairs,
                                    int* err, cudaStream_t st) {
  if (pairs == 0) return cudaSuccess;
  cudaError_t e = set_cg2_smem_attr();
  if (e != cudaSuccess) return e;
  Cg2Params p{};
  p.insts = insts;
  p.tiles = tiles;
  p.pair_off = pair_off;
  p.slot_rows = CN;   // instances of any height share the ring
  p.stall = -1;
  p.err = err;
  return launch_pdl(gemm_cg2_kernel<false, true>, dim3(static_cast<unsigned>(2 * pairs)), kCThreads, kCSmemBytes, st, 2, p);
}

#else   // the solo build has no CTA pairs

cudaError_t launch_gemm_cg2_grouped(const GemmInst*, const GemmTile*, const int*, int, int*, cudaStream_t) {
  return cudaErrorNotSupported;   // a build without CTA pairs plans none
}

bool gemm_cg2_eligible(const GemmTcArgs&, int) { return false; }
cudaError_t launch_gemm_cg2(const GemmTcArgs&, int*, int, cudaStream_t) { return cudaErrorNotSupported; }

#endif

}  // namespace pj
