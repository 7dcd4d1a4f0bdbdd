// qgemm_f64.cu -- FP64 quaternion GEMM on the CUDA cores.
//
// C = A B with the Hamilton product per scalar (Sec. 2):
//   (a0 + a1 i + a2 j + a3 k)(b0 + b1 i + b2 j + b3 k) =
//     (a0b0 - a1b1 - a2b2 - a3b3) + (a0b1 + a1b0 + a2b3 - a3b2) i
//   + (a0b2 - a1b3 + a2b0 + a3b1) j + (a0b3 + a1b2 - a2b1 + a3b0) k.
// GB300 has a small FP64 pipe (two FMAs per clock and SM), so this kernel is
// bound by FP64 issue at any tiling, and what a tiling can lose is padding and
// the last wave: 8 x 8 quaternion tiles, one output per thread of a 64-thread
// block, up to 32 blocks per SM.  With 32 x 32 tiles a 238^3 product ran on 64
// of the 152 SMs (1.1 ms, 0.36 at the pipe's rate) and a 1000-row one padded
// 2.4 % per side.  The tiles' operand traffic (512 bytes per k) stays far below
// what L2 delivers in the 2048 cycles their FMAs take.
#include <algorithm>

#include "common.cuh"

namespace qp {
namespace {

constexpr int BM = 8, BN = 8, BK = 16;

__global__ void __launch_bounds__(BM * BN) k_qgemm_f64(int M, int K, int N, Planes<const double> A,
                                                       Planes<const double> B, Planes<double> C) {
  __shared__ double sa[4][BK][BM + 1];  // sa[c][k][i]
  __shared__ double sb[4][BK][BN + 1];  // sb[c][k][j]
  const int tx = threadIdx.x % BN, ty = threadIdx.x / BN;
  const int i0 = blockIdx.y * BM, j0 = blockIdx.x * BN;
  double o[4] = {0.0, 0.0, 0.0, 0.0};

  for (int k0 = 0; k0 < K; k0 += BK) {
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const int t = threadIdx.x + h * BM * BN;
      const int ia = t / BK, ka = t % BK, kb = t / BN, jb = t % BN;
      const bool oka = i0 + ia < M && k0 + ka < K, okb = k0 + kb < K && j0 + jb < N;
#pragma unroll
      for (int c = 0; c < 4; c++) {
        sa[c][ka][ia] = oka ? A.p[c * A.ps + (long)(i0 + ia) * A.ld + k0 + ka] : 0.0;
        sb[c][kb][jb] = okb ? B.p[c * B.ps + (long)(k0 + kb) * B.ld + j0 + jb] : 0.0;
      }
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < BK; kk++) {
      double p[4], q[4];
#pragma unroll
      for (int c = 0; c < 4; c++) {
        p[c] = sa[c][kk][ty];
        q[c] = sb[c][kk][tx];
      }
      o[0] = fma(p[0], q[0], fma(-p[1], q[1], fma(-p[2], q[2], fma(-p[3], q[3], o[0]))));
      o[1] = fma(p[0], q[1], fma(p[1], q[0], fma(p[2], q[3], fma(-p[3], q[2], o[1]))));
      o[2] = fma(p[0], q[2], fma(-p[1], q[3], fma(p[2], q[0], fma(p[3], q[1], o[2]))));
      o[3] = fma(p[0], q[3], fma(p[1], q[2], fma(-p[2], q[1], fma(p[3], q[0], o[3]))));
    }
    __syncthreads();
  }
  const int gi = i0 + ty, gj = j0 + tx;
  if (gi < M && gj < N)
#pragma unroll
    for (int c = 0; c < 4; c++) C.p[c * C.ps + (long)gi * C.ld + gj] = o[c];
}

}  // namespace

cudaError_t launch_qgemm_f64(int M, int K, int N, const Planes<const double>& A, const Planes<const double>& B,
                             const Planes<double>& C, cudaStream_t st) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  // rows in slabs: the grid's y extent is limited to 65535 blocks (64-bit row
  // counter: the last slab may end at the largest int)
  const dim3 grid((unsigned)(((long)N + BN - 1) / BN), (unsigned)(((long)M + BM - 1) / BM));
  if (grid.y > 65535) {
    constexpr long slab = 65535L * BM;
    for (long i = 0; i < M; i += slab) {
      Planes<const double> a = A;
      Planes<double> c = C;
      a.p += i * A.ld;
      c.p += i * C.ld;
      const cudaError_t e = launch_qgemm_f64((int)std::min(M - i, slab), K, N, a, B, c, st);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
  k_qgemm_f64<<<grid, BM * BN, 0, st>>>(M, K, N, A, B, C);
  ++g_kernel_launches;
  return cudaGetLastError();
}

}  // namespace qp
