// krylov.cu -- vector kernels of the global quaternion Krylov solvers
// (Gl-QGMRES / Gl-QFOM, Sec. 3.5).  A block is an n x m quaternion matrix
// stored as L = 4 n m contiguous doubles (four planes); the global inner
// product <V, W> = Re tr(V^H W) is the plain dot product of those arrays.
// The basis V_0, V_1, ... is one array of blocks with stride L.  Reductions
// are deterministic (fixed block shapes, tree sums in shared memory).
#include "common.cuh"

namespace qp {
namespace {

constexpr int KT = 256;

__device__ double block_reduce(double v, double* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 32) {
    t = threadIdx.x < (int)(blockDim.x >> 5) ? sh[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  }
  return t;  // valid in thread 0
}

// h[i] = <V_i, W>, i < c: block i reduces over the L elements.
__global__ void __launch_bounds__(KT) k_block_dot(const double* __restrict__ V, int c, const double* __restrict__ W,
                                                   long L, double* __restrict__ h) {
  __shared__ double sh[KT / 32];
  const double* v = V + (long)blockIdx.x * L;
  double s = 0.0;
  for (long e = threadIdx.x; e < L; e += KT) s += v[e] * W[e];
  s = block_reduce(s, sh);
  if (threadIdx.x == 0) h[blockIdx.x] = s;
}

// W += sign * sum_{i<c} h[i] V_i.  A block takes 32 consecutive elements
// (one per lane, coalesced across the basis), its warps split the basis
// index i, and the warps' partial sums are added in a fixed order.  Block 0
// also adds h into the Hessenberg column when hcol is given.
constexpr int kCombWarps = 16;
__global__ void __launch_bounds__(32 * kCombWarps) k_block_combine(double* __restrict__ W, const double* __restrict__ V,
                                                                   const double* __restrict__ h, int c, long L,
                                                                   double sign, double* __restrict__ hcol) {
  __shared__ double part[kCombWarps][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long e = (long)blockIdx.x * 32 + lane;
  double s = 0.0;
  if (e < L)
    for (int i = w; i < c; i += kCombWarps) s += h[i] * V[(long)i * L + e];
  part[w][lane] = s;
  __syncthreads();
  if (w == 0 && e < L) {
    double t = 0.0;
    for (int q = 0; q < kCombWarps; q++) t += part[q][lane];
    W[e] += sign * t;
  }
  if (blockIdx.x == 0 && hcol)
    for (int i = threadIdx.x; i < c; i += 32 * kCombWarps) hcol[i] += h[i];
}

// nrm = ||W||; out = W / nrm (out may alias W; left unscaled when nrm = 0).
// One block: the blocks of these solvers are small (L = 4 n m).
__global__ void __launch_bounds__(1024) k_norm_scale(const double* W, long L, double* __restrict__ nrm, double* out) {
  __shared__ double sh[32];
  __shared__ double tot;
  double s = 0.0;
  for (long e = threadIdx.x; e < L; e += blockDim.x) s += W[e] * W[e];
  s = block_reduce(s, sh);
  if (threadIdx.x == 0) {
    tot = sqrt(s);
    *nrm = tot;
  }
  __syncthreads();
  const double t = tot;
  if (out && t > 0.0)
    for (long e = threadIdx.x; e < L; e += blockDim.x) out[e] = W[e] / t;
}

// out = a - b
__global__ void k_sub(double* __restrict__ out, const double* __restrict__ a, const double* __restrict__ b, long L) {
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < L; e += (long)gridDim.x * blockDim.x)
    out[e] = a[e] - b[e];
}

// C = A B for a skinny right-hand side (m <= kSkinnyMax columns): block i
// computes row i of C; its threads stride over k, accumulate the Hamilton
// products for every column, and reduce across the block.  The general GEMM
// kernels tile 64 x 64 outputs and leave almost every SM idle at m <= 16.
constexpr int kSkinnyMax = 16;
__global__ void __launch_bounds__(128) k_qgemm_skinny(Planes<const double> A, Planes<const double> B, int K, int m,
                                                      Planes<double> C) {
  __shared__ double sh[4 * kSkinnyMax][4];
  const int i = blockIdx.x;
  double acc[4 * kSkinnyMax];
#pragma unroll
  for (int t = 0; t < 4 * kSkinnyMax; t++) acc[t] = 0.0;
  for (int k = threadIdx.x; k < K; k += blockDim.x) {
    const long ai = (long)i * A.ld + k;
    const double as = A.p[ai], ax = A.p[A.ps + ai], ay = A.p[2 * A.ps + ai], az = A.p[3 * A.ps + ai];
#pragma unroll
    for (int l = 0; l < kSkinnyMax; l++) {
      if (l < m) {
        const long bi = (long)k * B.ld + l;
        const double bs = B.p[bi], bx = B.p[B.ps + bi], by = B.p[2 * B.ps + bi], bz = B.p[3 * B.ps + bi];
        acc[4 * l + 0] += as * bs - ax * bx - ay * by - az * bz;
        acc[4 * l + 1] += as * bx + ax * bs + ay * bz - az * by;
        acc[4 * l + 2] += as * by - ax * bz + ay * bs + az * bx;
        acc[4 * l + 3] += as * bz + ax * by - ay * bx + az * bs;
      }
    }
  }
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int t = 0; t < 4 * kSkinnyMax; t++) {
    if (t < 4 * m) {
      double v = acc[t];
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) sh[t][w] = v;
    }
  }
  __syncthreads();
  if (threadIdx.x < 4 * m) {
    const int t = threadIdx.x, l = t >> 2, q = t & 3;
    C.p[q * C.ps + (long)i * C.ld + l] = sh[t][0] + sh[t][1] + sh[t][2] + sh[t][3];
  }
}

// Givens steps j0 .. j0 + nb - 1 (nb <= 32) of the GMRES / FOM least-squares
// update, on the device so that the host need not read every Hessenberg
// column.  Thread t owns column j0 + t: it applies the rotations of steps
// 0 .. j0 - 1 (in place; h_{j+1,j} = col[j+1] is kept) alongside the other
// columns' threads, then the batch's own rotations in order as they are formed:
// the serial chain is j0 + nb rotations per batch instead of one launch of up
// to j rotations per step (28 % of the solve's kernel time).  Rotation j forms
// c, s, updates g, and writes the residual estimate |g_{j+1}| (GMRES) or
// |g_{j+1}| / |c_j| (FOM).
__global__ void __launch_bounds__(32) k_givens(double* __restrict__ H, long hstride, double* __restrict__ cs,
                                               double* __restrict__ sn, double* __restrict__ g, int j0, int nb,
                                               int fom, double* __restrict__ res) {
  const int t = threadIdx.x, j = j0 + t;
  double* col = H + hstride * j;
  double a = 0.0;
  if (t < nb) {
    // the running entry stays in a register: every load is of an entry not yet
    // written, so the loads pipeline and only the rotation chain is serial
    a = col[0];
    for (int i = 0; i < j0; i++) {
      const double b = col[i + 1], c = cs[i], s = sn[i];
      col[i] = c * a + s * b;
      a = -s * a + c * b;
    }
  }
  double gp = g[j0];
  for (int q = 0; q < nb; q++) {
    double c = 0.0, s = 0.0;
    if (t == q) {
      const double b = col[j + 1];
      const double rho = hypot(a, b);
      c = rho > 0.0 ? a / rho : 1.0;
      s = rho > 0.0 ? b / rho : 0.0;
      cs[j] = c;
      sn[j] = s;
      col[j] = rho;
    }
    c = __shfl_sync(0xffffffffu, c, q);
    s = __shfl_sync(0xffffffffu, s, q);
    if (t > q && t < nb) {
      const int i = j0 + q;
      const double b = col[i + 1];
      col[i] = c * a + s * b;
      a = -s * a + c * b;
    }
    const double gn = -s * gp;
    if (t == 0) {
      g[j0 + q] = c * gp;
      g[j0 + q + 1] = gn;
      res[j0 + q] = fom ? (c != 0.0 ? fabs(gn) / fabs(c) : INFINITY) : fabs(gn);
    }
    gp = gn;
  }
}

// nb Arnoldi steps (global Gram-Schmidt, applied twice) in one cooperative
// launch: W = A V_j, h = V^T W, W -= V h, h' = V^T W, W -= V h', hcol = h + h',
// V_{j+1} = W / ||W||, with a grid barrier between the phases.  Eight launches
// of 2-27 us per step left the GPU idle between them (0.24 ms a step; the FP64
// work of a 238 x 3 block at step 100 is 8 us).  Work is cut so that no phase
// needs atomics: rows of A over the grid's warps, basis vectors over blocks
// (dots), groups of 32 elements over blocks (updates).
constexpr int AT = 256, AW = AT / 32;

// Grid barrier: all blocks are resident (cooperative launch).  Bounded: false
// once a wait has run out (the flag then makes every later wait return).
__device__ bool grid_barrier(unsigned int* bar, unsigned int target, volatile int* err) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    int good = 1;
    __threadfence();
    atomicAdd(bar, 1u);
    unsigned long long t0 = 0;
    for (unsigned int it = 0; *reinterpret_cast<volatile unsigned int*>(bar) < target; it++) {
      if ((it & 1023u) == 1023u) {
        unsigned long long t;
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
        if (t0 == 0) t0 = t;
        if (*err != 0 || t - t0 > 2000000000ull) {
          *err = 51;
          good = 0;
          break;
        }
      }
    }
    __threadfence();
    ok = good;
  }
  __syncthreads();
  return ok != 0;
}

__device__ __forceinline__ double block_sum_at(double v, double* sh) {  // valid in thread 0
  __syncthreads();
  sh[threadIdx.x] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x < 32) {
    r = sh[threadIdx.x];
#pragma unroll
    for (int k = 1; k < AW; k++) r += sh[threadIdx.x + 32 * k];
    for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  }
  return r;
}

struct ArnoldiArgs {
  Planes<const double> A;
  int n, m;
  long L;
  double *V, *W, *h, *H;  // basis, work block, 2 x hlen dots, Hessenberg columns
  long hstride, hlen;
  double* part;           // one sum per element group
  int j0, nb;
  unsigned int* bar;      // 0 at launch
  int* err;
};

template <int MC>
__global__ void __launch_bounds__(AT, 1) k_arnoldi(ArnoldiArgs P) {
  __shared__ double sh[AT];
  __shared__ double nrm_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, G = gridDim.x;
  const long L = P.L, pl = (long)P.n * P.m;
  const int groups = (int)((L + 31) / 32);
  unsigned int target = 0;
  for (int b = 0; b < P.nb; b++) {
    const int j = P.j0 + b, c = j + 1;
    const double* Vj = P.V + (long)j * L;
    double* hcol = P.H + P.hstride * j;
    // ---- W = A V_j: a warp per row, lanes over k ----
    for (int i = warp * G + blockIdx.x; i < P.n; i += AW * G) {
      double acc[4 * MC];
#pragma unroll
      for (int t = 0; t < 4 * MC; t++) acc[t] = 0.0;
      for (int k = lane; k < P.n; k += 32) {
        const long ai = (long)i * P.A.ld + k;
        const double as = P.A.p[ai], ax = P.A.p[P.A.ps + ai], ay = P.A.p[2 * P.A.ps + ai],
                     az = P.A.p[3 * P.A.ps + ai];
#pragma unroll
        for (int l = 0; l < MC; l++) {
          if (l < P.m) {
            const long bi = (long)k * P.m + l;
            const double bs = __ldcg(Vj + bi), bx = __ldcg(Vj + pl + bi), by = __ldcg(Vj + 2 * pl + bi),
                         bz = __ldcg(Vj + 3 * pl + bi);
            acc[4 * l + 0] += as * bs - ax * bx - ay * by - az * bz;
            acc[4 * l + 1] += as * bx + ax * bs + ay * bz - az * by;
            acc[4 * l + 2] += as * by - ax * bz + ay * bs + az * bx;
            acc[4 * l + 3] += as * bz + ax * by - ay * bx + az * bs;
          }
        }
      }
#pragma unroll
      for (int t = 0; t < 4 * MC; t++) {
        if (t < 4 * P.m) {
          double v = acc[t];
          for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          if (lane == 0) P.W[(t & 3) * pl + (long)i * P.m + (t >> 2)] = v;
        }
      }
    }
    if (!grid_barrier(P.bar, target += G, P.err)) return;
    for (int pass = 0; pass < 2; pass++) {
      double* h = P.h + pass * P.hlen;
      // ---- h = V^T W: a block per basis vector ----
      for (int i = blockIdx.x; i < c; i += G) {
        const double* v = P.V + (long)i * L;
        double s = 0.0;
        for (long e = threadIdx.x; e < L; e += AT) s += __ldcg(v + e) * __ldcg(P.W + e);
        s = block_sum_at(s, sh);
        if (threadIdx.x == 0) h[i] = s;
      }
      if (!grid_barrier(P.bar, target += G, P.err)) return;
      // ---- W -= V h: a block per 32 elements, warps over the basis ----
      for (int q = blockIdx.x; q < groups; q += G) {
        const long e = (long)q * 32 + lane;
        double s = 0.0;
        if (e < L)
#pragma unroll 4
          for (int i = warp; i < c; i += AW) s += __ldcg(h + i) * __ldcg(P.V + (long)i * L + e);
        __syncthreads();
        sh[threadIdx.x] = s;
        __syncthreads();
        if (warp == 0) {
          double x = 0.0;
          if (e < L) {
            double t = 0.0;
#pragma unroll
            for (int k = 0; k < AW; k++) t += sh[lane + 32 * k];
            x = __ldcg(P.W + e) - t;
            P.W[e] = x;
          }
          if (pass == 1) {
            x *= x;
            for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            if (lane == 0) P.part[q] = x;
          }
        }
      }
      if (pass == 1 && blockIdx.x == G - 1)
        for (int i = threadIdx.x; i < c; i += AT) hcol[i] = __ldcg(P.h + i) + __ldcg(h + i);
      if (!grid_barrier(P.bar, target += G, P.err)) return;
    }
    // ---- ||W|| (every block adds the group sums in the same order), V_{j+1} ----
    double s = 0.0;
    for (int q = threadIdx.x; q < groups; q += AT) s += __ldcg(P.part + q);
    s = block_sum_at(s, sh);
    if (threadIdx.x == 0) {
      nrm_s = sqrt(s);
      if (blockIdx.x == 0) hcol[j + 1] = nrm_s;
    }
    __syncthreads();
    const double nrm = nrm_s;
    if (nrm > 0.0)
      for (long e = (long)blockIdx.x * AT + threadIdx.x; e < L; e += (long)G * AT)
        P.V[(long)(j + 1) * L + e] = __ldcg(P.W + e) / nrm;
    if (!grid_barrier(P.bar, target += G, P.err)) return;
  }
}

int grid_of(long L) {
  long b = (L + KT - 1) / KT;
  return (int)(b < 1 ? 1 : b > 4096 ? 4096 : b);
}

}  // namespace

bool skinny_ok(int m) { return m >= 1 && m <= kSkinnyMax; }

cudaError_t launch_qgemm_skinny(int M, int K, int m, const Planes<const double>& A, const Planes<const double>& B,
                                const Planes<double>& C, cudaStream_t st) {
  k_qgemm_skinny<<<M, 128, 0, st>>>(A, B, K, m, C);
  ++g_kernel_launches;
  return cudaGetLastError();
}

cudaError_t launch_givens(double* H, long hstride, double* cs, double* sn, double* g, int j0, int nb, int fom,
                          double* res, cudaStream_t st) {
  if (nb < 1 || nb > 32) return cudaErrorInvalidValue;
  k_givens<<<1, 32, 0, st>>>(H, hstride, cs, sn, g, j0, nb, fom, res);
  ++g_kernel_launches;
  return cudaGetLastError();
}

// Blocks of up to 64 KB in the cooperative kernel, larger ones a launch per phase.
// Measured on both sides (times of whole unrestarted solves, launch per phase
// divided by cooperative): 1.08 to 1.45 for 1 to 4 columns at 8192 numbers (2048 x
// 1 to 512 x 4), 1.02 to 1.2 for 5 to 8 columns; even at 8192 numbers of 8 columns
// and 8568 of 9; 0.95 at 238 x 12 (11424 numbers).  The line is a compromise: 12 to
// 16 columns of 80 to 150 rows, where one block of 128 threads per row holds the
// product in one wave, lose in the cooperative kernel (0.85 to 0.93), and 1 to 4
// columns gain beyond the line too (1024 x 4 1.36, 2048 x 2 1.11).
bool arnoldi_ok(long L, int m) { return skinny_ok(m) && L <= 8192; }

cudaError_t launch_arnoldi(const Planes<const double>& A, int n, int m, double* V, double* W, double* h, long hlen,
                           double* H, long hstride, double* part, int j0, int nb, unsigned int* bar, int* err,
                           cudaStream_t st) {
  int dev = 0, nsm = 0, coop = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (e != cudaSuccess) return e;
  if (!coop) return cudaErrorNotSupported;
  ArnoldiArgs P{A, n, m, 4L * n * m, V, W, h, H, hstride, hlen, part, j0, nb, bar, err};
  if ((e = cudaMemsetAsync(bar, 0, sizeof(unsigned int), st)) != cudaSuccess) return e;
  void* args[] = {&P};
  const void* k = m <= 4 ? (const void*)k_arnoldi<4> : (const void*)k_arnoldi<kSkinnyMax>;
  e = cudaLaunchCooperativeKernel(k, dim3(nsm), dim3(AT), args, 0, st);
  ++g_kernel_launches;
  return e;
}

cudaError_t launch_block_dot(const double* V, int c, const double* W, long L, double* h, cudaStream_t st) {
  k_block_dot<<<c, KT, 0, st>>>(V, c, W, L, h);
  ++g_kernel_launches;
  return cudaGetLastError();
}

cudaError_t launch_block_sub(double* W, const double* V, const double* h, int c, long L, double* hcol,
                             cudaStream_t st) {
  k_block_combine<<<(int)((L + 31) / 32), 32 * kCombWarps, 0, st>>>(W, V, h, c, L, -1.0, hcol);
  ++g_kernel_launches;
  return cudaGetLastError();
}

cudaError_t launch_norm_scale(const double* W, long L, double* nrm, double* out, cudaStream_t st) {
  k_norm_scale<<<1, 1024, 0, st>>>(W, L, nrm, out);
  ++g_kernel_launches;
  return cudaGetLastError();
}

cudaError_t launch_basis_add(double* X, const double* V, const double* y, int k, long L, cudaStream_t st) {
  k_block_combine<<<(int)((L + 31) / 32), 32 * kCombWarps, 0, st>>>(X, V, y, k, L, 1.0, nullptr);
  ++g_kernel_launches;
  return cudaGetLastError();
}

cudaError_t launch_sub(double* out, const double* a, const double* b, long L, cudaStream_t st) {
  k_sub<<<grid_of(L), KT, 0, st>>>(out, a, b, L);
  ++g_kernel_launches;
  return cudaGetLastError();
}

}  // namespace qp
