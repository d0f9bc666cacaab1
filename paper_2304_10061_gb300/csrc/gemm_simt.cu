// Float32 GEMM on the CUDA cores (the all-float32 path of the MLPs):
//   C[M x N] = A[M x K] B^T,  A row-major [M][lda], B row-major [N][ldb]
// (B is a weight matrix W [out x in] for the forward, W^T for input gradients),
// with the epilogues of epilogue.cuh.
//
// Register-blocked SGEMM: BM x 64 block tiles, k-slices of SB_K, an 8 x 8
// outer-product block per thread (rows {4 ty ..} and {BM / 2 + 4 ty ..}, columns
// {4 tx ..} and {32 + 4 tx ..}), column pairs accumulated in packed fp32 (two IEEE
// multiply-adds per instruction, the results of the scalar ones).  Operands are
// read from global memory as float4 rows (when the row starts and strides allow
// it), stored k-major into a double-buffered shared-memory tile, and the next
// k-slice is loaded into registers while the current one is multiplied (one
// barrier per slice).  The column tiles of one row block are neighbouring blocks
// of the grid, so the A rows are read from HBM once and the other column tiles
// hit L2.
// Bound: the fp32 pipe, 65 TFLOP/s with operands in registers on this part, and
// beside it the shared-memory reads (a 16-byte read costs a warp four wavefronts
// however many lanes share an address).  128 x 64 tiles of 128 threads with
// slices of 16, three to a SM: 52-55 TFLOP/s at 590,000 rows, 42-46 at 25,000
// (N = 192..384, K = 192..384); scalar multiply-adds in 128 x 128 tiles of 256
// threads: 44-50 and 23-35 (a block per SM left over in the last wave costs most
// at the small size); also tried: 8 x 16 blocks per thread 49-53 and 31-40, 64 x
// 64 tiles 47-50 and 36-43, 128 x 128 tiles packed 38-43 and 33-37.
#include <cuda_runtime.h>

#include "epilogue.cuh"
#include "internal.h"
#include "launch.cuh"

namespace alg {

constexpr int SB_PAD = 4;

// One 4-wide k group of row r (global row index), zero beyond M and K.
__device__ __forceinline__ float4 ld_k4(const float* __restrict__ P, int ld, int rows, int r, int K, int k,
                                        bool vec) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (r >= rows) return v;
  const float* p = P + (size_t)r * ld + k;
  if (vec && k + 3 < K) return __ldg(reinterpret_cast<const float4*>(p));
  if (k < K) v.x = __ldg(p);
  if (k + 1 < K) v.y = __ldg(p + 1);
  if (k + 2 < K) v.z = __ldg(p + 2);
  if (k + 3 < K) v.w = __ldg(p + 3);
  return v;
}

// Four consecutive columns [n, n+4) of row m (n + 3 < N, 16-byte aligned rows).
__device__ __forceinline__ void epi_apply4_f32(const EpiParams& ep, int m, int n, float4 a) {
  float v[4] = {a.x, a.y, a.z, a.w};
  if (ep.epi == EPI_FWD_SILU) {
    if (ep.pre) *reinterpret_cast<float4*>(reinterpret_cast<float*>(ep.pre) + (size_t)m * ep.ldp + n) = a;
    const float rs = ep.rowscale ? ep.rowscale[m] : 1.0f;
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = v[j] * epi_sigmoid(v[j]) * rs;
  } else if (ep.epi == EPI_F32) {
    if (ep.add) {
      const float4 x = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(ep.add) +
                                                        (size_t)m * ep.ld_add + n);
      v[0] += x.x; v[1] += x.y; v[2] += x.z; v[3] += x.w;
    }
  } else if (ep.epi == EPI_BWD_SILU) {
    const float4 z4 = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(ep.pre) + (size_t)m * ep.ldp + n);
    const float z[4] = {z4.x, z4.y, z4.z, z4.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float s = epi_sigmoid(z[j]);
      v[j] = v[j] * s * (1.0f + z[j] * (1.0f - s));
    }
  }
  *reinterpret_cast<float4*>(reinterpret_cast<float*>(ep.out) + (size_t)m * ep.ldo + n) =
      make_float4(v[0], v[1], v[2], v[3]);
}

template <int BM, int SB_K>
__global__ void __launch_bounds__(BM) gemm_simt_kernel(
    const float* __restrict__ A, int lda, const float* __restrict__ B, int ldb, int M, int N, int K, EpiParams ep,
    int vecA, int vecB) {
  pdl_wait();
  constexpr int BN = 64, TM = 8, TN = 8, kThreads = BM;   // BM BN / (TM TN)
  constexpr int kRows = kThreads / (SB_K / 4);    // rows of a slice loaded per pass (four k per thread)
  constexpr int ALOADS = BM / kRows, BLOADS = BN / kRows;
  static_assert(BM % kRows == 0 && BN % kRows == 0, "whole passes");
  constexpr int GM = TM / 4, GN = TN / 4;         // groups of four rows / columns of a thread
  constexpr int kTx = BN / TN;                    // threads across the columns
  __shared__ __align__(16) float As[2][SB_K][BM + SB_PAD];
  __shared__ __align__(16) float Bs[2][SB_K][BN + SB_PAD];
  const int tid = threadIdx.x;
  const int tx = tid % kTx, ty = tid / kTx;
  // linear block index: the column tiles of a row block are consecutive
  const int ntn = (N + BN - 1) / BN;
  const int n0 = (int)(blockIdx.x % ntn) * BN, m0 = (int)(blockIdx.x / ntn) * BM;
  // load mapping: row tid / (SB_K / 4) (+ kRows h), k group of four
  const int lr = tid / (SB_K / 4), lk = tid % (SB_K / 4) * 4;
  float4 ra[ALOADS], rb[BLOADS];
  auto gload = [&](int k0) {
#pragma unroll
    for (int h = 0; h < ALOADS; ++h) ra[h] = ld_k4(A, lda, M, m0 + lr + kRows * h, K, k0 + lk, vecA != 0);
#pragma unroll
    for (int h = 0; h < BLOADS; ++h) rb[h] = ld_k4(B, ldb, N, n0 + lr + kRows * h, K, k0 + lk, vecB != 0);
  };
  auto sstore = [&](int buf) {
#pragma unroll
    for (int h = 0; h < ALOADS; ++h) {
      As[buf][lk + 0][lr + kRows * h] = ra[h].x;
      As[buf][lk + 1][lr + kRows * h] = ra[h].y;
      As[buf][lk + 2][lr + kRows * h] = ra[h].z;
      As[buf][lk + 3][lr + kRows * h] = ra[h].w;
    }
#pragma unroll
    for (int h = 0; h < BLOADS; ++h) {
      Bs[buf][lk + 0][lr + kRows * h] = rb[h].x;
      Bs[buf][lk + 1][lr + kRows * h] = rb[h].y;
      Bs[buf][lk + 2][lr + kRows * h] = rb[h].z;
      Bs[buf][lk + 3][lr + kRows * h] = rb[h].w;
    }
  };
  float2 acc[TM][TN / 2];   // row i x column pair
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) acc[i][j] = make_float2(0.0f, 0.0f);

  const int nk = (K + SB_K - 1) / SB_K;
  gload(0);
  sstore(0);
  __syncthreads();
  for (int kt = 0; kt < nk; ++kt) {
    const int buf = kt & 1;
    if (kt + 1 < nk) gload((kt + 1) * SB_K);
#pragma unroll
    for (int k = 0; k < SB_K; ++k) {
      float4 a4[GM];
      float2 b[TN / 2];
#pragma unroll
      for (int g = 0; g < GM; ++g) a4[g] = *reinterpret_cast<const float4*>(&As[buf][k][g * (BM / GM) + 4 * ty]);
#pragma unroll
      for (int g = 0; g < GN; ++g) {
        const float4 v = *reinterpret_cast<const float4*>(&Bs[buf][k][g * (BN / GN) + 4 * tx]);
        b[2 * g] = make_float2(v.x, v.y);
        b[2 * g + 1] = make_float2(v.z, v.w);
      }
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const float4 v = a4[i / 4];
        const float x = (i & 3) == 0 ? v.x : ((i & 3) == 1 ? v.y : ((i & 3) == 2 ? v.z : v.w));
        const float2 aa = make_float2(x, x);
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = __ffma2_rn(aa, b[j], acc[i][j]);
      }
    }
    if (kt + 1 < nk) sstore(buf ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = m0 + (i / 4) * (BM / GM) + 4 * ty + (i & 3);
    if (m >= M) continue;
#pragma unroll
    for (int g = 0; g < GN; ++g) {
      const int n = n0 + g * (BN / GN) + 4 * tx;
      const float2 lo = acc[i][2 * g], hi = acc[i][2 * g + 1];
      if (ep.vec && n + 3 < N) {
        epi_apply4_f32(ep, m, n, make_float4(lo.x, lo.y, hi.x, hi.y));
      } else {
        const float v[4] = {lo.x, lo.y, hi.x, hi.y};
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (n + j < N) epi_apply<float>(ep, m, n + j, v[j]);
      }
    }
  }
}

template <int BM, int SB_K>
static void launch_simt(const GemmArgs& g, const float* A, const float* B, int ldb, const EpiParams& ep, int vecA,
                        int vecB, cudaStream_t st) {
  const unsigned tiles = (unsigned)((g.M + BM - 1) / BM) * (unsigned)((g.N + 63) / 64);
  launch(gemm_simt_kernel<BM, SB_K>, tiles, BM, 0, st, A, g.lda, B, ldb, g.M, g.N, g.K, ep, vecA, vecB);
}

void gemm_simt_f32(const GemmArgs& g, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0) return;
  const float* A = reinterpret_cast<const float*>(g.A);
  const float* B = g.trans ? g.W->f32T : g.W->f32;
  const int ldb = g.trans ? g.W->ldT : g.W->ld;
  auto al16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  const int vecA = al16(A) && g.lda % 4 == 0;
  const int vecB = al16(B) && ldb % 4 == 0;
  const EpiParams ep = make_epi(g);
  // 64-row tiles when 128-row ones would leave SMs without a tile, and slices of 8 for short sums
  // (every output's sum runs over k in the same order in each)
  if ((int64_t)((g.M + 127) / 128) * ((g.N + 63) / 64) < 152) launch_simt<64, 8>(g, A, B, ldb, ep, vecA, vecB, st);
  else if (g.K <= 64) launch_simt<128, 8>(g, A, B, ldb, ep, vecA, vecB, st);
  else launch_simt<128, 16>(g, A, B, ldb, ep, vecA, vecB, st);
}

}  // namespace alg
