// Reduced product in double precision on CUDA cores (the FP64 correctness
// path): Y = A_c B_d with A_c M x Kp and B_d Kp x N, both row-major.
#include "common.hpp"
#include "pdl.cuh"

namespace pj {
namespace {

// The tile of block b, counted along the rows of tiles: its first output row and column.
// One grid dimension holds them all: 65,535 rows of tiles, all that gridDim.y takes, are
// 524,280 rows of outputs at 8 x 8.
template <int TILE>
__device__ __forceinline__ void f64_tile_origin(int64_t N, int64_t& i0, int64_t& j0) {
  const uint32_t tn = static_cast<uint32_t>((N + TILE - 1) / TILE);
  const uint32_t ti = blockIdx.x / tn;
  i0 = static_cast<int64_t>(ti) * TILE;
  j0 = static_cast<int64_t>(blockIdx.x - ti * tn) * TILE;
}

// A block of 256 threads computes a TILE x TILE block of Y, K' in chunks of TILE
// staged in shared memory; each thread owns TILE * TILE / 256 outputs.
template <int TILE>
__global__ void __launch_bounds__(256) gemm_f64_kernel(const double* __restrict__ A, const double* __restrict__ B,
                                                       double* __restrict__ Y, int64_t ldy, int64_t M, int64_t N,
                                                       int64_t K) {
  constexpr int ROWS = 256 / TILE;      // thread rows
  constexpr int PER = TILE / ROWS;      // outputs per thread
  __shared__ double sA[TILE][TILE + 1];
  __shared__ double sB[TILE][TILE + 1];
  const int tx = threadIdx.x % TILE, ty = threadIdx.x / TILE;
  int64_t i0, j0;
  f64_tile_origin<TILE>(N, i0, j0);
  pdl_begin();
  double acc[PER];
#pragma unroll
  for (int r = 0; r < PER; ++r) acc[r] = 0.0;
  for (int64_t k0 = 0; k0 < K; k0 += TILE) {
#pragma unroll
    for (int r = 0; r < PER; ++r) {
      const int row = ty + ROWS * r;
      sA[row][tx] = (i0 + row < M && k0 + tx < K) ? A[(i0 + row) * K + k0 + tx] : 0.0;
      sB[row][tx] = (k0 + row < K && j0 + tx < N) ? B[(k0 + row) * N + j0 + tx] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < TILE; ++kk) {
      const double b = sB[kk][tx];
#pragma unroll
      for (int r = 0; r < PER; ++r) acc[r] = fma(sA[ty + ROWS * r][kk], b, acc[r]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int r = 0; r < PER; ++r) {
    const int64_t i = i0 + ty + ROWS * r, j = j0 + tx;
    if (i < M && j < N) Y[i * ldy + j] = acc[r];
  }
}

// An 8 x 8 block of Y per 256 threads: thread t sums the quarter t / 64 of every chunk of
// 64 reduced components for output t % 64, and the quarters are added at the end.
// Why: the SM's FP64 units (two FMAs a clock) bound these products, so what counts is
// that the SMs get equal shares.  The 256 x 256 output of 512 components is 256 tiles of
// 16, two on 104 SMs and one on 48 (78 us); as 1024 tiles of 8 every SM gets six or
// seven.  The quarters give a small output four times the warps.
constexpr int kF8 = 8, kF8Chunk = 64, kF8Parts = 4;

__global__ void __launch_bounds__(256) gemm_f64_tile8_kernel(const double* __restrict__ A,
                                                             const double* __restrict__ B, double* __restrict__ Y,
                                                             int64_t ldy, int64_t M, int64_t N, int64_t K) {
  __shared__ double sA[kF8][kF8Chunk + 1];
  __shared__ double sB[kF8Chunk][kF8 + 1];
  __shared__ double sR[kF8Parts][kF8 * kF8];
  const int t = threadIdx.x, o = t & 63, part = t >> 6, oy = o >> 3, ox = o & 7;
  int64_t i0, j0;
  f64_tile_origin<kF8>(N, i0, j0);
  // what this thread stages of a chunk: two values of A (rows ar, ar + 4) and of B (rows bk, bk + 32)
  const int ar = t >> 6, ak = t & 63, bk = t >> 3, bj = t & 7;
  pdl_begin();
  auto load_a = [&](int64_t k0, int r) {
    return i0 + r < M && k0 + ak < K ? A[(i0 + r) * K + k0 + ak] : 0.0;
  };
  auto load_b = [&](int64_t k0, int k) {
    return k0 + k < K && j0 + bj < N ? B[(k0 + k) * N + j0 + bj] : 0.0;
  };
  double a0 = load_a(0, ar), a1 = load_a(0, ar + 4), b0 = load_b(0, bk), b1 = load_b(0, bk + 32);
  double acc = 0.0;
  for (int64_t k0 = 0; k0 < K; k0 += kF8Chunk) {
    sA[ar][ak] = a0;
    sA[ar + 4][ak] = a1;
    sB[bk][bj] = b0;
    sB[bk + 32][bj] = b1;
    __syncthreads();
    const int64_t kn = k0 + kF8Chunk;   // the next chunk, in flight during the sums
    if (kn < K) {
      a0 = load_a(kn, ar);
      a1 = load_a(kn, ar + 4);
      b0 = load_b(kn, bk);
      b1 = load_b(kn, bk + 32);
    }
#pragma unroll
    for (int kk = 0; kk < kF8Chunk / kF8Parts; ++kk) {
      const int k = part * (kF8Chunk / kF8Parts) + kk;
      acc = fma(sA[oy][k], sB[k][ox], acc);
    }
    __syncthreads();
  }
  sR[part][o] = acc;
  __syncthreads();
  if (part == 0 && i0 + oy < M && j0 + ox < N)
    Y[(i0 + oy) * ldy + j0 + ox] = ((sR[0][o] + sR[1][o]) + (sR[2][o] + sR[3][o]));
}

}  // namespace

// Tiles of 8, 16 or 32: the size whose fullest SM computes the fewest outputs (the FP64
// units run at one rate for all of them); a larger tile unless a smaller saves 5 %.
// Calls with 32, or 16 below 304 tiles of 32, at every size, and with this rule:
// 256 x 256 x 512 107 us and 73; 4096 x 40 x 512 268 and 183; 100,000 x 40 x 64 811 and
// 552; 1000 x 1000 x 300 598 and 545; 2048 x 2056 x 512 3632 and 3616.
static int f64_tile(int64_t M, int64_t N, int sms) {
  int best = 32;
  int64_t best_w = 0;
  for (int tile = 32; tile >= 8; tile /= 2) {
    const int64_t tiles = ceil_div(M, tile) * ceil_div(N, tile);
    const int64_t w = ceil_div(tiles, sms) * tile * tile;
    if (tile == 32 || w * 20 < best_w * 19) {
      best = tile;
      best_w = w;
    }
  }
  return best;
}

cudaError_t launch_gemm_f64(const double* Ac, const double* Bd, double* Y, int64_t ldy, int64_t M, int64_t N,
                            int64_t Kp, cudaStream_t st) {
  if (M == 0 || N == 0) return cudaSuccess;
  int sms = 0;
  if (device_sms(&sms) != PJ_OK) sms = 152;
  const int tile = f64_tile(M, N, sms);
  const int64_t tiles = ceil_div(N, tile) * ceil_div(M, tile);
  if (tiles > INT32_MAX) return cudaErrorInvalidConfiguration;
  const dim3 grid(static_cast<unsigned>(tiles));
  if (tile == 8) return launch_plain(gemm_f64_tile8_kernel, grid, 256, 0, st, Ac, Bd, Y, ldy, M, N, Kp);
  if (tile == 16) return launch_plain(gemm_f64_kernel<16>, grid, 256, 0, st, Ac, Bd, Y, ldy, M, N, Kp);
  return launch_plain(gemm_f64_kernel<32>, grid, 256, 0, st, Ac, Bd, Y, ldy, M, N, Kp);
}

}  // namespace pj
