// common.cuh -- internal types shared by the CUDA sources of libqpinv.
//
// A quaternion matrix lives in HBM as four real planes (s, x, y, z), the
// layout of the C ABI.  Besides the FP64 "master" planes, a matrix that
// feeds the tensor cores also carries BF16 split copies:
//   A-form: row-major rows x cols (K-major when the matrix is the left
//           operand, K = cols);
//   B-form: the plane-wise transpose, cols x rows (K-major when the matrix
//           is the right operand, K = rows).
// Split level L stores L BF16 terms v = t0 + t1 + ... (each the BF16
// rounding of the remainder), level-major then component-major.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

namespace qp {

// kernels launched by this thread through the launch_* functions below
extern thread_local long long g_kernel_launches;

typedef __nv_bfloat16 bf16;

// Row-major plane set: element (c, i, j) at p[c * ps + i * ld + j].
template <typename T>
struct Planes {
  T* p = nullptr;
  long ld = 0;  // elements between rows
  long ps = 0;  // elements between component planes
};

// BF16 split forms of one matrix (either pointer may be null).
struct Split16 {
  bf16* a = nullptr;  // A-form [level][comp][rows][lda]
  long lda = 0, psa = 0;
  bf16* b = nullptr;  // B-form [level][comp][cols][ldb]
  long ldb = 0, psb = 0;
  int levels = 0;
};

// Programmatic dependent launch: a kernel launched this way may start while
// its predecessor in the stream still runs.  It does its own setup, then
// pdl_wait() before its first access to global memory (the predecessor has
// then completed, and transitively everything before it); pdl_trigger() lets
// its successor start the same way.  Every kernel launched through launch_pdl
// calls both.  Small solves are strings of 5-15 us kernels, of which launch
// and setup (barriers, TMEM, descriptors) were 2-3 us each (64 x 48 solve 1.15
// -> 1.00 ms, image completion 34.9 -> 31.9).  Grids of more than two blocks
// per SM do not trigger: their successor's waiting blocks gain nothing and
// held slots of the last wave (exact 2048^3 product 1.5 % slower).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() {
  if (gridDim.x * gridDim.y <= 2 * 152) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// launch_pdl inside a function that returns cudaError_t
#define QP_LAUNCH(...)                                                   \
  do {                                                                   \
    if (cudaError_t qp_le = qp::launch_pdl(__VA_ARGS__)) return qp_le;   \
  } while (0)

// A coefficient as the kernels read it: GB300's FP64 pipe does two operations
// per clock and SM, so even a comparison of a double with 0 or 1 costs as much
// as the arithmetic it saves; the host decides the kind once per launch.
enum { CK_ZERO = 0, CK_ONE = 1, CK_MINUS = 2, CK_GENERAL = 3 };
struct Coef {
  double d = 0.0;
  float f = 0.f;
  int kind = CK_ZERO;
  void set(double x) {
    d = x;
    f = (float)x;
    kind = x == 0.0 ? CK_ZERO : x == 1.0 ? CK_ONE : x == -1.0 ? CK_MINUS : CK_GENERAL;
  }
};
template <typename T>
__device__ __forceinline__ T coef(const Coef& c);
template <>
__device__ __forceinline__ float coef<float>(const Coef& c) { return c.f; }
template <>
__device__ __forceinline__ double coef<double>(const Coef& c) { return c.d; }

// FP32 <-> FP64 conversions from the bits, on the integer pipe (64 operations
// per clock and SM) instead of the FP64 pipe's.  Zeros, subnormals, infinities
// and NaN take the instruction.
__device__ __forceinline__ double widen(float x) {
  const uint32_t b = __float_as_uint(x);
  if (((b >> 23) & 0xFFu) - 1u >= 254u) return (double)x;
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + 0x38000000u)), (int)(b << 29));
}
__device__ __forceinline__ float narrow(double x) {  // round to nearest even, as the cast
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t ex = (hi >> 20) & 0x7FFu;
  if (ex - 897u >= 253u) return (float)x;  // below the FP32 normal range, or near overflow
  const uint32_t m = ((ex - 896u) << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29);
  const uint32_t rem = lo & 0x1FFFFFFFu;
  const uint32_t up = (rem > 0x10000000u || (rem == 0x10000000u && (m & 1u))) ? 1u : 0u;
  return __uint_as_float((hi & 0x80000000u) | (m + up));
}
// The same for N values with one branch for all: round a single value's
// instruction the compiler predicates instead of branching, and the FP64 pipe
// then takes its 16 cycles for it all the same (8.6 % of a 4096^3 product's time,
// in an epilogue that no MMA overlaps: 1.23 -> 1.20 ms; 2048^3 200 -> 188 us).
template <int N>
__device__ __forceinline__ void to_master_all(const float* x, double* y) {
  bool special = false;  // an exponent of 0 or 255
#pragma unroll
  for (int t = 0; t < N; t++) special |= ((__float_as_uint(x[t]) + 0x00800000u) & 0x7F000000u) == 0u;
  if (special) {
#pragma unroll
    for (int t = 0; t < N; t++) y[t] = (double)x[t];
  } else {
#pragma unroll
    for (int t = 0; t < N; t++) {
      const uint32_t b = __float_as_uint(x[t]);
      y[t] = __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + 0x38000000u)), (int)(b << 29));
    }
  }
}
template <int N>
__device__ __forceinline__ void to_master_all(const float* x, float* y) {
#pragma unroll
  for (int t = 0; t < N; t++) y[t] = x[t];
}
__device__ __forceinline__ float flip_sign(float x) { return -x; }
__device__ __forceinline__ double flip_sign(double x) {
  return __hiloint2double((int)((uint32_t)__double2hiint(x) ^ 0x80000000u), __double2loint(x));
}
template <typename T>
__device__ __forceinline__ T to_master(float x);
template <>
__device__ __forceinline__ float to_master<float>(float x) { return x; }
template <>
__device__ __forceinline__ double to_master<double>(float x) { return widen(x); }
__device__ __forceinline__ float to_float(float x) { return x; }
__device__ __forceinline__ float to_float(double x) { return narrow(x); }

// Block partial sums finished in the kernel that wrote them: the last block
// to arrive (counted in *count, which it resets) adds the blocks' partials in
// a fixed order (strided threads, shuffle, warp order), so the result does not
// depend on the blocks' timing.  A pass with a stop test or a norm is then one
// launch instead of two (a separate one-block reduction: 4-10 us each, 23 of
// the 142 launches of a 64 x 48 solve).
struct Reduce {
  double* partials = nullptr;  // [block][nvals]
  double* out = nullptr;       // nvals sums
  unsigned int* count = nullptr;  // 0 between launches
};
// Every thread of the block calls this after its block's partials are
// written (by any of its threads); sh: 32 doubles of shared memory.
template <int NVALS>
__device__ __forceinline__ void reduce_last_block(const Reduce& r, long nblocks, double* sh) {
  __shared__ int last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned int total = gridDim.x * gridDim.y;
    last = atomicAdd(r.count, 1u) == total - 1 ? 1 : 0;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  // the warps share the values: warp w adds value w % NVALS over every
  // (warps / NVALS)-th group of 32 blocks (one value after another with the
  // whole block took 12-15 k cycles, mostly barriers and FP64 shuffles)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, per = (int)(blockDim.x >> 5) / NVALS;
  const int v = warp % NVALS, w = warp / NVALS;
  double s = 0.0;
  if (w < per) {
#pragma unroll 4
    for (long b = 32L * w + lane; b < nblocks; b += 32L * per) s += __ldcg(r.partials + b * NVALS + v);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) sh[warp] = s;
  }
  __syncthreads();
  if (threadIdx.x < NVALS) {
    double t = 0.0;
    for (int k = 0; k < per; k++) t += sh[k * NVALS + threadIdx.x];
    r.out[threadIdx.x] = t;
  }
  if (threadIdx.x == 0) *r.count = 0;
}

// Output specification of the fused combine kernel:
//   out = cacc * acc + sum_t caux[t] * aux_t + diag * I   (diag on plane s)
// The master output (and every aux input) has the master type of the pass:
// float (tensor-core phase) or double (FP64 phase).  BF16 outputs are
// round-to-nearest splits of the FP32 value (t0 = bf16(v), t1 = bf16(v - t0),
// ...).
struct OutSpec {
  void* mp = nullptr;  // master output planes (type of the pass), may be null
  long mld = 0, mps = 0;
  Split16 s16;         // BF16 outputs (a and/or b may be null)
  double cacc = 0.0;
  double caux[4] = {0, 0, 0, 0};
  double diag = 0.0;
  Coef kacc, kaux[4], kdiag;  // set by the launch function
  void set_coefs() {
    kacc.set(cacc);
    for (int t = 0; t < 4; t++) kaux[t].set(caux[t]);
    kdiag.set(diag);
  }
};

enum { ACC_F32 = 0, ACC_F64 = 1, ACC_Q8 = 2 };

constexpr int kMaxOut = 3;

struct CombineArgs {
  int rows = 0, cols = 0;
  int f64 = 0;                // master type of aux inputs and outputs: 0 float, 1 double
  const void* acc = nullptr;  // accumulator planes, may be null
  // ACC_Q8: the eight real products of the exact-slice GEMM (qgemm_emu.cu),
  // int64 planes [set][8], the sets summed; twice a component is an integer
  // combination q of them, its value q * 2^(erow[i] + ecol[j] - shift)
  int acc_kind = ACC_F32;
  int acc_sets = 1;
  long ld_acc = 0, ps_acc = 0;
  const int* acc_erow = nullptr;
  const int* acc_ecol = nullptr;
  int acc_shift = 0;
  const void* aux[4] = {nullptr, nullptr, nullptr, nullptr};
  long ld_aux[4] = {0, 0, 0, 0}, ps_aux[4] = {0, 0, 0, 0};
  OutSpec out[kMaxOut];
  int nout = 0;
  Reduce red;  // red.partials: sums of ||out0 - aux0||^2, ||out0||^2 and the non-finite count into red.out
};

}  // namespace qp

// Host-side launch helpers implemented in elementwise.cu / qgemm_*.cu.
namespace qp {

// blocks (and partials) launch_combine will use for these arguments
int combine_blocks(const CombineArgs& a);
cudaError_t launch_combine(const CombineArgs& a, cudaStream_t st);
// ||A||_F^2, the non-finite count, the largest row and column modulus sums into
// out[0..3]; scratch: norms_scratch(m, n) doubles
long norms_scratch(int m, int n);
cudaError_t launch_matrix_norms(const Planes<const double>& A, int m, int n, double* scratch, double* out,
                                unsigned int* count, cudaStream_t st);
// scratch entries of a column reduction over `cols` columns
inline long COL_SCRATCH(long cols) { return 64 * cols; }
// ||A - B||_F^2 (B optional) and the non-finite count of A into r.out[0..1];
// partials for kFroBlocks blocks.
constexpr int kFroBlocks = 1024;
cudaError_t launch_fro2(const Planes<const double>& A, const Planes<const double>* B, int m, int n, const Reduce& r,
                        cudaStream_t st);
// The norms of a residual plane set R (n x n, FP64) that the Penrose pass
// needs, in one read, into r.out[0..3] (partials of penrose_norm_blocks(n)
// blocks): ||R||_F^2 without its diagonal's s plane, the sum of R_s(i, i)^2,
// the sum of (sr R_s(i, i) + 1)^2 (sr = +-1), and ||R^H - R||_F^2.
int penrose_norm_blocks(int n);
cudaError_t launch_penrose_norms(const Planes<const double>& R, int n, double sr, const Reduce& r, cudaStream_t st);
cudaError_t launch_init_x0(const Planes<const double>& A, int m, int n, double alpha, const Planes<double>& X,
                           cudaStream_t st);
cudaError_t launch_init_x0(const Planes<const double>& A, int m, int n, double alpha, const Planes<float>& X,
                           cudaStream_t st);
// D = S (FP64 planes, any strides)
cudaError_t launch_copy_planes(const Planes<const double>& S, int rows, int cols, const Planes<double>& D,
                               cudaStream_t st);
cudaError_t launch_f64_to_f32(const Planes<const double>& src, int rows, int cols, const Planes<float>& dst,
                              cudaStream_t st);
cudaError_t launch_f32_to_f64(const Planes<const float>& src, int rows, int cols,
                              const Planes<double>& dst, cudaStream_t st);

// Exact slices of a product's operands for the eight-product exact-slice GEMM
// (qgemm_emu.cu): S balanced 7-bit digits of v * 2^-e per component (slice s
// an integer in [-64, 63], [-128, 128] for s = 0, of weight 2^-7(s+1)), stored
// as the BF16 digit sums of products p0 .. p0 + np - 1.  P (M x K): A-form with
// the left combinations, za [S][np][M][lda], row exponents eP; Q (K x N): the
// transposed B-form with the right combinations, zb [S][np][N][ldb], column
// exponents eQ.  A null za or zb leaves that operand out.  Padding up to the
// next multiple of 8 along the slice rows is written as 0.
struct SliceArgs {
  int M = 0, N = 0, K = 0, S = 0, p0 = 0, np = 8;
  int *eP = nullptr, *eQ = nullptr;
  int* scratch = nullptr;  // COL_SCRATCH(N) ints, kept between the groups of one product
  bf16* za = nullptr;
  long lda = 0, psa = 0;
  bf16* zb = nullptr;
  long ldb = 0, psb = 0;
};
cudaError_t launch_slices(const SliceArgs& a, const Planes<const double>& P, const Planes<const double>& Q,
                          cudaStream_t st);
cudaError_t launch_slices(const SliceArgs& a, const Planes<const float>& P, const Planes<const float>& Q,
                          cudaStream_t st);

cudaError_t launch_qgemm_f64(int M, int K, int N, const Planes<const double>& A,
                             const Planes<const double>& B, const Planes<double>& C,
                             cudaStream_t st);

// Combine pass fused into the epilogue of the tensor-core GEMM: the product
// never goes to HBM; each output o is
//   out_o = cacc * (A B) + sum_t caux[t] * aux_t + diag * I   (diag on plane s)
// evaluated in the master type (FP32, or FP64 with f64 = 1) and written as a
// master and/or round-to-nearest BF16 splits of its FP32 rounding (A-form
// row-major, B-form transposed); in the FP32 case optionally with the
// stop-test sums of output 0 (||out0 - aux0||^2, ||out0||^2, non-finite count).
// Outputs must not alias the product's operand forms (other CTAs are still
// reading them); an output may alias an aux plane (same element, same thread).
struct EpiOut {
  void* mp = nullptr;  // master planes, float (double when EpiArgs::f64); may be null
  long mld = 0, mps = 0;
  bf16* a = nullptr;  // A-form splits [level][comp][rows][lda] (may be null)
  long lda = 0, psa = 0;
  bf16* b = nullptr;  // B-form splits [level][comp][cols][ldb] (may be null)
  long ldb = 0, psb = 0;
  int levels = 0;
  Coef cacc, caux[3], diag;
};
constexpr int kEpiAux = 3;
struct EpiArgs {
  int nout = 0;  // 0: plain FP32 store of the product into TcGemmArgs::C
  EpiOut out[kMaxOut];
  const void* aux[kEpiAux] = {nullptr, nullptr, nullptr};  // planes of the master type
  long ld_aux[kEpiAux] = {0, 0, 0}, ps_aux[kEpiAux] = {0, 0, 0};
  Reduce red;  // red.partials: 3 values per (CTA, epilogue warp), tc_partial_blocks() of them (f64 == 0 only)
  int f64 = 0;  // 1: aux inputs and output masters are double planes (FP64 arithmetic in the epilogue)
};

// Tensor-core quaternion GEMM on BF16 split operands.  acc (FP32) = sum over
// the listed (i, j) term pairs of A_i * B_j, restricted to k in [k0, k1).
struct TcGemmArgs {
  int M = 0, N = 0, K = 0;
  int k0 = 0, k1 = 0;
  const Split16* A = nullptr;  // uses the A-form
  const Split16* B = nullptr;  // uses the B-form
  int npairs = 0;
  int pair_i[16] = {0}, pair_j[16] = {0};
  Planes<float> C;  // FP32 output
  EpiArgs epi;      // epi.nout > 0: fused combine instead of the plain store (FP32 output only)
  int broad = -1;   // tile shapes: 1 128 columns, 0 64 columns, -1 chosen by size
  int* err = nullptr;  // device error word (bounded-wait expiry)
};
cudaError_t launch_qgemm_tc(const TcGemmArgs& a, cudaStream_t st);
int tc_partial_blocks(const TcGemmArgs& a);  // blocks of partials a fused launch of these arguments writes

// FP64-accurate product from S exact slices per operand in one launch
// (qgemm_emu.cu).  emu_plan chooses the tile width, the split of an item's
// levels and K range into parts, and the fixed point; the launch writes the
// int64 planes C64 [nparts][8][M][ld64] of products p0 .. p0 + np - 1 (units
// 2^-F; written, not added to).  ld64 and ps64 are multiples of 4.
struct EmuPlan {
  int bn = 128, ngroups = 1, nk = 1, nparts = 1;
  int F = 0;
};
EmuPlan emu_plan(int M, int N, int K, int S);
struct EmuGemmArgs {
  int M = 0, N = 0, K = 0;
  const Split16* A = nullptr;  // A-form slices of np combinations (levels >= S)
  const Split16* B = nullptr;  // B-form slices
  int S = 0, p0 = 0, np = 8;
  long long* C64 = nullptr;
  long ld64 = 0, ps64 = 0;
  int* err = nullptr;
};
cudaError_t launch_qgemm_emu(const EmuGemmArgs& a, const EmuPlan& plan, cudaStream_t st);
bool tc_supported();

// Batched solver (batched_impl.cuh: host side in batched.cu, kernels in batched_tile<t>.cu).
struct BatchResultHost {
  int status, iters, side, gemms;
  double alpha, delta, delta_rel;
  double E[4], E_rel[4];
};
}  // namespace qp
#include <vector>
namespace qp {
// CTA GEMM engines of the batched kernel: CUDA-core double-FP32 tiles
// (quaternion entries) 0: 16x16, 1: 32x32, 2: 64x32, 3: 32x64, 4: 64x64, and
// 5: the tensor-core exact-slice engine (batched_tc.cu).
constexpr int BATCH_TILES = 6;
constexpr int BATCH_TILE_TC = 5;
const char* batched_tile_name(int tile);
// Device and pinned host buffers of one batched call (owned by the context).
struct BatchRun {
  int tile = 1, slots = 0;
  void* ws = nullptr;  // slots * batched_slot_bytes()
  void* tc_ws = nullptr;    // tensor-core engine: slots * batched_tc_slot_bytes()
  void* tc_maps = nullptr;  // ... its TMA maps on the device (2 per slot)
  void* host_maps = nullptr;  // pinned staging of the maps
  int* err = nullptr;       // device error word
  void *dev_items = nullptr, *dev_order = nullptr, *dev_results = nullptr;
  int* dev_counter = nullptr;
  void *host_items = nullptr, *host_order = nullptr, *host_results = nullptr;  // pinned
};
// A captured CUDA graph of the call (upload, counter reset, the persistent
// kernel, result download), replayed while the launch shape is unchanged.
struct BatchGraph {
  cudaStream_t stream = nullptr;  // capture / replay stream (non-blocking)
  cudaGraphExec_t exec = nullptr;
  unsigned long long key = 0;
  int replays = 0;
};
cudaError_t run_batched(int batch, const int* m, const int* n, const double* const* A, const long* lda,
                        double* const* X, const long* ldx, int method, double tol, int max_iter, int mparam,
                        int stop_rule, int alpha_mode, double alpha_user, const double* hpi19_k, const BatchRun& r,
                        BatchGraph* graph, std::vector<BatchResultHost>& out, cudaStream_t st);
size_t batched_slot_bytes();
size_t batched_tc_slot_bytes();  // slice scratch of one tensor-core engine slot
// Learned alpha (alpha.cu).
int alpha_nweights();
int alpha_ntrain();
int alpha_feature_scratch_floats(int m, int n);
int power_radius_doubles(int s, int steps);  // dscratch entries of power_radius
cudaError_t power_radius(const Planes<const float>& M, int s, int steps, float* scratch, double* dscratch,
                         double* pin, cudaStream_t st, double* rho);
cudaError_t alpha_features(const Planes<const float>& A, int m, int n, double fro2, double norm1, double norminf,
                           float* scratch, double* dscratch, double* pin, cudaStream_t st, float* feat,
                           double* theta1_out);
void alpha_init_weights(float* W, unsigned long long seed);
size_t alpha_scratch_floats(int B);
cudaError_t alpha_forward(const float* dW, const float* dX, int B, float* scratch, float* dy_out, cudaStream_t st);
cudaError_t alpha_gradient(const float* dW, const float* dX, const float* dT, int B, float* scratch, float* dG,
                           double* dloss, cudaStream_t st);
cudaError_t alpha_adam(float* dW, const float* dG, float* dM1, float* dM2, int t, float lr, cudaStream_t st);
size_t batched_item_bytes();
size_t batched_result_bytes();
int batched_max_dim();
int batched_slots_per_sm(int tile);

// CUR image completion (cur.cu): the data-consistency fill, the gather of the
// CUR factors and the Gaussian filter, on contiguous planes (ps = m * n).
struct CurFill {
  const double* M[4] = {nullptr, nullptr, nullptr, nullptr};  // observed planes, row stride ldm
  long ldm = 0;
  const unsigned char* mask = nullptr;  // nonzero = observed, row stride ldk
  long ldk = 0;
  const double* X = nullptr;  // estimate for the unobserved pixels (null: 0); may alias C
  double* C = nullptr;
  int m = 0, n = 0;
};
constexpr int kMaxGaussRadius = 16;
struct GaussTaps {
  int radius = 0;
  double w[2 * kMaxGaussRadius + 1];
};
cudaError_t launch_cur_fill(const CurFill& f, cudaStream_t st);
cudaError_t launch_cur_gather(const double* C, int m, int n, int r, const int* I, const int* J, double* CJ,
                              double* RI, double* W, cudaStream_t st);
cudaError_t launch_cur_gauss(const double* in, double* out, int m, int n, const GaussTaps& g, cudaStream_t st);
// Signal filtering (toeplitz.cu): X(i, j) = x(t0 + i - j), (p+1) x (p+1),
// from planes of samples with plane stride xps; X contiguous.
cudaError_t launch_toeplitz(const double* x, long xps, int p, int t0, double* X, cudaStream_t st);
// Global Krylov solvers (krylov.cu): blocks of L doubles, basis stride L.
cudaError_t launch_block_dot(const double* V, int c, const double* W, long L, double* h, cudaStream_t st);
cudaError_t launch_block_sub(double* W, const double* V, const double* h, int c, long L, double* hcol,
                             cudaStream_t st);
cudaError_t launch_norm_scale(const double* W, long L, double* nrm, double* out, cudaStream_t st);
cudaError_t launch_basis_add(double* X, const double* V, const double* y, int k, long L, cudaStream_t st);
cudaError_t launch_sub(double* out, const double* a, const double* b, long L, cudaStream_t st);
// Givens rotations of Hessenberg columns j0 .. j0 + nb - 1 (columns hstride apart, nb <= 32).
cudaError_t launch_givens(double* H, long hstride, double* cs, double* sn, double* g, int j0, int nb, int fom,
                          double* res, cudaStream_t st);
// nb Arnoldi steps on blocks of L = 4 n m doubles in one cooperative launch
// (arnoldi_ok(L, m)): writes V_{j0+1} .. and Hessenberg columns j0 .. (unrotated);
// h: 2 hlen doubles, part: (L + 31) / 32 doubles of scratch, bar: a counter.
bool arnoldi_ok(long L, int m);
cudaError_t launch_arnoldi(const Planes<const double>& A, int n, int m, double* V, double* W, double* h, long hlen,
                           double* H, long hstride, double* part, int j0, int nb, unsigned int* bar, int* err,
                           cudaStream_t st);
// C = A B (FP64) for B with 1..16 columns: one block per row of C.
bool skinny_ok(int m);
cudaError_t launch_qgemm_skinny(int M, int K, int m, const Planes<const double>& A, const Planes<const double>& B,
                                const Planes<double>& C, cudaStream_t st);

}  // namespace qp
