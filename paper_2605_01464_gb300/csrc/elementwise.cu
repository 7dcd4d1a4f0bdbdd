// elementwise.cu -- HBM-bound kernels of the solve: the fused combine pass
// that follows every quaternion product (residual R = I - AX, polynomial
// blocks, X update with the stop-test norms), BF16 operand splitting and
// exact slicing with transposed copies, initialisation X_0 = alpha A^H, and
// the norm and Penrose-residual reductions.
//
// GB300's FP64 pipe is a small fraction of its FP32 rate, so the
// tensor-core phase runs these passes on FP32 masters; only the FP64 phase
// (polish, Penrose) uses double arithmetic, and exact slicing and exponent
// extraction use integer operations on the bit patterns.  Reductions are
// deterministic: each block writes partial sums and one block adds them in a
// fixed order.
#include <algorithm>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace qp {

thread_local long long g_kernel_launches = 0;

namespace {

constexpr int TILE = 32;
constexpr int TROWS = 8;  // block = 32 x 8 threads, each thread 4 rows of the tile

// Sum over a block of 256 threads, valid in thread 0; sh: 256 doubles.  The
// first warp adds eight entries per lane and then shuffles: 13 FP64
// instructions per block (a shuffle tree in every warp takes 48, and GB300's
// FP64 pipe needs 16 cycles for each).
__device__ __forceinline__ double block_sum(double v, double* sh) {
  __syncthreads();
  sh[threadIdx.x] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x < 32) {
    r = sh[threadIdx.x];
#pragma unroll
    for (int k = 1; k < 8; k++) r += sh[threadIdx.x + 32 * k];
    for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  }
  return r;
}
__device__ __forceinline__ double block_count(int v, double* sh) {  // the same for counts
  __syncthreads();
  const int w = __reduce_add_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) reinterpret_cast<int*>(sh)[threadIdx.x >> 5] = w;
  __syncthreads();
  int r = 0;
  if (threadIdx.x == 0)
    for (int k = 0; k < (int)(blockDim.x >> 5); k++) r += reinterpret_cast<int*>(sh)[k];
  return (double)r;
}

// Inf / NaN from the exponent bits (integer instructions: GB300's FP64 pipe
// is the scarce resource in these passes).
__device__ __forceinline__ int nonfinite_bits(double x) {
  return ((__double_as_longlong(x) >> 52) & 0x7FF) == 0x7FF ? 1 : 0;
}
__device__ __forceinline__ int nonfinite_bits(float x) { return ((__float_as_int(x) >> 23) & 0xFF) == 0xFF ? 1 : 0; }

// round(v * 2^sh) as an integer, from the bits of v (integer arithmetic only).
// Requires |v * 2^sh| < 2^62; subnormal inputs count as zero.
__device__ __forceinline__ long long to_fixed(double v, int sh) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int ex = (int)((b >> 52) & 0x7FF);
  if (ex == 0) return 0;
  const long long mant = (long long)((b & 0xFFFFFFFFFFFFFull) | (1ull << 52));
  const int k = ex - 1075 + sh;  // v * 2^sh = mant * 2^k
  long long F;
  if (k >= 0) F = mant << k;
  else if (k <= -55) F = 0;
  else F = (mant + (1ll << (-k - 1))) >> (-k);
  return (b >> 63) ? -F : F;
}
__device__ __forceinline__ long long to_fixed(float v, int sh) {
  const unsigned b = __float_as_uint(v);
  const int ex = (int)((b >> 23) & 0xFF);
  if (ex == 0) return 0;
  const long long mant = (long long)((b & 0x7FFFFFu) | (1u << 23));
  const int k = ex - 150 + sh;
  long long F;
  if (k >= 0) F = mant << k;
  else if (k <= -26) F = 0;
  else F = (mant + (1ll << (-k - 1))) >> (-k);
  return (b >> 31) ? -F : F;
}

// Magnitudes as integers, in the order of the values: a maximum is taken over
// these, and its exponent once at the end.
template <typename T>
struct Bits;
template <>
struct Bits<double> {
  using U = unsigned long long;
  static constexpr int MANT = 53, BIAS = 1022;
};
template <>
struct Bits<float> {
  using U = unsigned;
  static constexpr int MANT = 24, BIAS = 126;
};
__device__ __forceinline__ unsigned long long abs_bits(double v) {
  return (unsigned long long)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
}
__device__ __forceinline__ unsigned abs_bits(float v) { return __float_as_uint(v) & 0x7FFFFFFFu; }

// Binary exponent e of a slicing with S slices, from the largest magnitude:
// |v| < 2^e for every v and for every v rounded to 7S bits (-100000 when all are
// zero or subnormal).  Where 7S bits do not hold the mantissa, half of the last
// kept bit carries a maximum that rounds up to its power of two into the next
// exponent, so that no sliced entry reaches 1 in its row's or column's units: the
// exact-slice GEMM's fixed point has no room for a component of 4K (see emu_plan).
template <typename T>
__device__ __forceinline__ int exp_of(typename Bits<T>::U mx, int S) {
  using B = Bits<T>;
  const typename B::U half = 7 * S < B::MANT ? (typename B::U)1 << (B::MANT - 1 - 7 * S) : 0;
  const int ex = (int)((mx + half) >> (B::MANT - 1));
  return ex == 0 ? -100000 : ex - B::BIAS;
}

// q 2^e rounded to nearest (ties to even) as a double or float, from the
// integer bits: the same value as ldexp((T)q, e) without FP64 arithmetic or
// 64-bit conversion instructions.  Results outside the normal range take ldexp.
// The leading one is shifted to bit 63; the kept bits including it are added
// to the exponent field one too low, so that a rounding carry moves into it.
__device__ __noinline__ double i64_scaled_slow(long long q, int e) { return ldexp((double)q, e); }
__device__ __noinline__ float i64_scaledf_slow(long long q, int e) { return ldexpf((float)q, e); }
__device__ __forceinline__ unsigned long long i64_norm(long long q, uint32_t& sign, int& lz) {
  sign = (uint32_t)((unsigned long long)q >> 32) & 0x80000000u;
  const unsigned long long mag = q < 0 ? 0ull - (unsigned long long)q : (unsigned long long)q;
  lz = __clzll((long long)mag);
  return mag << (lz & 63);
}
__device__ __forceinline__ double i64_scaled(long long q, int e) {
  uint32_t sign;
  int lz;
  const unsigned long long mag = i64_norm(q, sign, lz);
  const int biased = 1023 + 63 - lz + e;
  if ((unsigned)(biased - 1) >= 2045u) return q == 0 ? 0.0 : i64_scaled_slow(q, e);
  const unsigned long long m = mag >> 11;
  const uint32_t up = (((uint32_t)mag & 0x7FFu) + 0x3FFu + ((uint32_t)m & 1u)) >> 11;
  const unsigned long long b = m + up + ((unsigned long long)(uint32_t)(biased - 1) << 52);
  return q == 0 ? 0.0 : __longlong_as_double((long long)(b | ((unsigned long long)sign << 32)));
}
__device__ __forceinline__ float i64_scaledf(long long q, int e) {
  uint32_t sign;
  int lz;
  const unsigned long long mag = i64_norm(q, sign, lz);
  const int biased = 127 + 63 - lz + e;
  if ((unsigned)(biased - 1) >= 253u) return q == 0 ? 0.f : i64_scaledf_slow(q, e);
  const uint32_t hi = (uint32_t)(mag >> 32), m = hi >> 8;
  // bits below the last kept one, the low word folded into a sticky bit
  const uint32_t rest = ((hi & 0xFFu) << 1) | ((uint32_t)mag != 0 ? 1u : 0u);
  const uint32_t up = (rest + 0xFFu + (m & 1u)) >> 9;
  const uint32_t b = m + up + ((uint32_t)(biased - 1) << 23);
  return q == 0 ? 0.f : __uint_as_float(b | sign);
}

// Twice the four components from the eight real products of the exact-slice
// GEMM (see qgemm_emu.cu).  Wrapping arithmetic: a doubled component is below
// 2^63 in modulus (emu_plan), the partial sums need not be.
__device__ __forceinline__ void quad_of(const unsigned long long* p, long long* q) {
  const unsigned long long a = p[4] + p[5], b = p[4] - p[5], c = p[6] + p[7], d = p[6] - p[7];
  q[0] = (long long)(2 * p[1] - a + c);
  q[1] = (long long)(2 * p[0] - a - c);
  q[2] = (long long)(2 * p[2] + b + d);
  q[3] = (long long)(2 * p[3] + b - d);
}
template <typename T>
__device__ __forceinline__ T q8_value(long long q, int e) {
  if (sizeof(T) == 4) return (T)i64_scaledf(q, e);
  return (T)i64_scaled(q, e);
}

// Two adjacent values (the second if `two`), one access where the address allows.
template <typename T2, typename T>
__device__ __forceinline__ void load_pair(const T* p, bool two, T& x, T& y) {
  if (two && (reinterpret_cast<uintptr_t>(p) & (sizeof(T2) - 1)) == 0) {
    const T2 t = *reinterpret_cast<const T2*>(p);
    x = t.x;
    y = t.y;
  } else {
    x = p[0];
    y = two ? p[1] : (T)0;
  }
}
__device__ __forceinline__ void ld2(const float* p, bool two, float& x, float& y) { load_pair<float2>(p, two, x, y); }
__device__ __forceinline__ void ld2(const double* p, bool two, double& x, double& y) {
  load_pair<double2>(p, two, x, y);
}
__device__ __forceinline__ void st2(float* p, bool two, float x, float y) {
  if (two && (reinterpret_cast<uintptr_t>(p) & 7) == 0) *reinterpret_cast<float2*>(p) = make_float2(x, y);
  else {
    p[0] = x;
    if (two) p[1] = y;
  }
}
__device__ __forceinline__ void st2(double* p, bool two, double x, double y) {
  if (two && (reinterpret_cast<uintptr_t>(p) & 15) == 0) *reinterpret_cast<double2*>(p) = make_double2(x, y);
  else {
    p[0] = x;
    if (two) p[1] = y;
  }
}

// cacc times the accumulator's four components at (i, j) and (i, j + 1);
// cacc = +-1 is a sign (for the fixed-point planes, of the integer).
template <typename T>
__device__ __forceinline__ void acc_pairs(const CombineArgs& a, const Coef& k, int i, int j, bool two, T (*v)[2]) {
  const long off = (long)i * a.ld_acc + j;
  if (a.acc_kind == ACC_Q8) {
    // the planes' rows are padded to a multiple of 4: the pair loads stay inside
    unsigned long long p0[8], p1[8];
    const unsigned long long* src = (const unsigned long long*)a.acc + off;
#pragma unroll
    for (int t = 0; t < 8; t++) {
      const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(src + t * a.ps_acc);
      p0[t] = u.x;
      p1[t] = u.y;
    }
    for (int s = 1; s < a.acc_sets; s++) {
      src += 8 * a.ps_acc;
#pragma unroll
      for (int t = 0; t < 8; t++) {
        const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(src + t * a.ps_acc);
        p0[t] += u.x;
        p1[t] += u.y;
      }
    }
    long long q0[4], q1[4];
    quad_of(p0, q0);
    quad_of(p1, q1);
    const int er = a.acc_erow[i] - a.acc_shift;
    const int e0 = er + a.acc_ecol[j], e1 = two ? er + a.acc_ecol[j + 1] : 0;
    const bool neg = k.kind == CK_MINUS;
#pragma unroll
    for (int c = 0; c < 4; c++) {
      v[c][0] = q8_value<T>(neg ? -q0[c] : q0[c], e0);
      v[c][1] = two ? q8_value<T>(neg ? -q1[c] : q1[c], e1) : (T)0;
    }
  } else {
#pragma unroll
    for (int c = 0; c < 4; c++) {
      if (a.acc_kind == ACC_F64) {
        double x, y;
        ld2((const double*)a.acc + c * a.ps_acc + off, two, x, y);
        v[c][0] = (T)x;
        v[c][1] = (T)y;
      } else {
        float x, y;
        ld2((const float*)a.acc + c * a.ps_acc + off, two, x, y);
        v[c][0] = to_master<T>(x);
        v[c][1] = to_master<T>(y);
      }
      if (k.kind == CK_MINUS) {
        v[c][0] = flip_sign(v[c][0]);
        v[c][1] = flip_sign(v[c][1]);
      }
    }
  }
  if (k.kind == CK_GENERAL) {
    const T x = coef<T>(k);
#pragma unroll
    for (int c = 0; c < 4; c++) {
      v[c][0] *= x;
      v[c][1] *= x;
    }
  }
}

// Round-to-nearest BF16 splits of two adjacent FP32 values.
__device__ __forceinline__ void split_store2(bf16* base, long idx, long lstride, int levels, float x, float y) {
  float rx = x, ry = y;
  for (int l = 0; l < levels; l++) {
    const __nv_bfloat162 t = __floats2bfloat162_rn(rx, ry);
    *reinterpret_cast<__nv_bfloat162*>(base + l * lstride + idx) = t;
    rx -= __low2float(t);
    ry -= __high2float(t);
  }
}

// Combine pass over column pairs: a block takes 8 `groups` rows x 64 columns,
// a thread two adjacent columns of one row per group (8- or 16-byte accesses,
// packed BF16 pairs).  Bound: HBM, once nothing but the pass's own additions
// runs on the FP64 pipe: coefficients carry a host-side kind (comparing a
// double with 0 or 1 is FP64 work; it was most of the former kernel's 6 FP64
// instructions per value), conversions and sign flips are integer operations.
template <typename T>
__global__ void __launch_bounds__(256) k_combine(const __grid_constant__ CombineArgs a, int groups) {
  pdl_wait();
  pdl_trigger();
  __shared__ float stage[4][2 * TILE][TILE + 1];  // [plane][column][row]
  __shared__ double red[256];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int rows_b = TROWS * groups, r0 = blockIdx.y * rows_b, c0 = blockIdx.x * 2 * TILE;
  const int j = c0 + 2 * tx;
  T s_dx = 0, s_x = 0;
  int s_bad = 0;

  for (int o = 0; o < a.nout; o++) {
    const OutSpec& O = a.out[o];
    for (int q = 0; q < groups; q++) {
      const int i = r0 + ty + q * TROWS;
      T v[4][2] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}};
      const bool in0 = i < a.rows && j < a.cols, two = in0 && j + 1 < a.cols;
      if (in0) {
        const bool acc_in = a.acc && O.kacc.kind != CK_ZERO;
        if (acc_in) acc_pairs<T>(a, O.kacc, i, j, two, v);
#pragma unroll
        for (int t = 0; t < 4; t++) {
          if (!a.aux[t] || O.kaux[t].kind == CK_ZERO) continue;
          const T* ap = (const T*)a.aux[t] + (long)i * a.ld_aux[t] + j;
          const T ct = coef<T>(O.kaux[t]);
          T u[4][2];
#pragma unroll
          for (int c = 0; c < 4; c++) ld2(ap + c * a.ps_aux[t], two, u[c][0], u[c][1]);
          if (t == 0 && !acc_in && O.kaux[0].kind == CK_ONE) {  // a plain copy takes no arithmetic
#pragma unroll
            for (int c = 0; c < 4; c++) {
              v[c][0] = u[c][0];
              v[c][1] = u[c][1];
            }
            continue;
          }
#pragma unroll
          for (int c = 0; c < 4; c++) {
            v[c][0] += ct * u[c][0];
            v[c][1] += ct * u[c][1];
          }
        }
        if (O.kdiag.kind != CK_ZERO) {
          if (i == j) v[0][0] += coef<T>(O.kdiag);
          if (two && i == j + 1) v[0][1] += coef<T>(O.kdiag);
        }
        if (o == 0 && a.red.partials) {
          const T* x0p = (const T*)a.aux[0];
#pragma unroll
          for (int c = 0; c < 4; c++) {
            T x0[2] = {0, 0};
            if (x0p) ld2(x0p + c * a.ps_aux[0] + (long)i * a.ld_aux[0] + j, two, x0[0], x0[1]);
#pragma unroll
            for (int h = 0; h < 2; h++) {
              if (h && !two) continue;
              s_x += v[c][h] * v[c][h];
              if (x0p) {
                const T dx = v[c][h] - x0[h];
                s_dx += dx * dx;
              }
              s_bad += nonfinite_bits(v[c][h]);
            }
          }
        }
        if (O.mp) {
          T* dst = (T*)O.mp + (long)i * O.mld + j;
#pragma unroll
          for (int c = 0; c < 4; c++) st2(dst + c * O.mps, two, v[c][0], v[c][1]);
        }
        if (O.s16.a) {
          // operand rows are padded to 64 entries: the pair's second half is
          // written beyond an odd width too (zero)
          const long idx = (long)i * O.s16.lda + j;
#pragma unroll
          for (int c = 0; c < 4; c++)
            split_store2(O.s16.a, c * O.s16.psa + idx, 4 * O.s16.psa, O.s16.levels, to_float(v[c][0]),
                         to_float(v[c][1]));
        }
      }
      if (O.s16.b) {
#pragma unroll
        for (int c = 0; c < 4; c++) {
          stage[c][2 * tx][ty + q * TROWS] = to_float(v[c][0]);
          stage[c][2 * tx + 1][ty + q * TROWS] = to_float(v[c][1]);
        }
      }
    }
    if (O.s16.b) {
      __syncthreads();
      // B-form row jj (an output column) holds the block's rows in pairs
      const int np = rows_b / 2;
      for (int t = threadIdx.x; t < 2 * TILE * np; t += 256) {
        const int jl = t / np, p = t % np, jj = c0 + jl, ii = r0 + 2 * p;
        if (jj < a.cols && ii < a.rows) {
          const long idx = (long)jj * O.s16.ldb + ii;
#pragma unroll
          for (int c = 0; c < 4; c++)
            split_store2(O.s16.b, c * O.s16.psb + idx, 4 * O.s16.psb, O.s16.levels, stage[c][jl][2 * p],
                         stage[c][jl][2 * p + 1]);
        }
      }
      __syncthreads();
    }
  }
  if (a.red.partials) {
    if (!a.aux[0]) s_dx = s_x;  // ||v - 0||^2
    const long b = (long)blockIdx.y * gridDim.x + blockIdx.x;
    const double t0 = block_sum((double)s_dx, red);
    const double t1 = block_sum((double)s_x, red);
    const double t2 = block_count(s_bad, red);
    if (threadIdx.x == 0) {
      a.red.partials[3 * b + 0] = t0;
      a.red.partials[3 * b + 1] = t1;
      a.red.partials[3 * b + 2] = t2;
    }
    reduce_last_block<3>(a.red, (long)gridDim.x * gridDim.y, red);
  }
}

// Row groups of 8 per block: four, or one while that leaves SMs without work.
static int combine_groups(const CombineArgs& a) {
  const long blocks = (long)((a.cols + 2 * TILE - 1) / (2 * TILE)) * ((a.rows + TILE - 1) / TILE);
  return blocks < 2 * 152 ? 1 : TILE / TROWS;
}

// ---------------------------------------------------------------- exact slicing
// The exact-slice GEMM computes a quaternion product as eight real products
// of digit sums (qgemm_emu.cu).  A thread takes 8 consecutive entries along
// the slice row: its four components become 64-bit integers F = round(v
// 2^(7S - e)), biased so that every balanced 7-bit digit is a plain bit field
// (F + 64 (1 + 2^7 + ... + 2^(7(S-2))): field - 64 in [-64, 63]; the top digit
// is what is left above them), and each slice writes one 16-byte store per
// product.  Digits become floats by inserting the field into the mantissa of
// 2^23, so the sums and the conversion are FP32 adds and packed BF16
// conversions (exact: the sums are integers of at most 8 bits).
// Bound: HBM writes, 16 S bytes per entry (double the four-plane form's; the
// product it feeds does half the tensor work).
//
// Up to four slices of FP32 values (28 bits and the bias) are 32-bit integers:
// half the integer instructions, which bound the FP32 phase's slicing.
__device__ __forceinline__ int to_fixed32(float v, int sh) {  // as to_fixed, |v 2^sh| <= 2^28
  const unsigned b = __float_as_uint(v);
  const int ex = (int)((b >> 23) & 0xFF);
  const int mant = (int)((b & 0x7FFFFFu) | (1u << 23));
  const int k = ex - 150 + sh;
  int F;
  if (k >= 0) F = mant << k;
  else if (k <= -26) F = 0;
  else F = (mant + (1 << (-k - 1))) >> (-k);
  if (ex == 0) F = 0;
  return (b >> 31) ? -F : F;
}
template <typename T>
__device__ __forceinline__ void slice_bias(const T* v, int S, int e, long long* G) {
  long long bias = 0;
  for (int q = 0; q < S - 1; q++) bias = (bias << 7) + 64;
#pragma unroll
  for (int t = 0; t < 8; t++) G[t] = to_fixed(v[t], 7 * S - e) + bias;
}
__device__ __forceinline__ void slice_bias(const float* v, int S, int e, int* G) {
  int bias = 0;
  for (int q = 0; q < S - 1; q++) bias = (bias << 7) + 64;
#pragma unroll
  for (int t = 0; t < 8; t++) G[t] = to_fixed32(v[t], 7 * S - e) + bias;
}
template <typename I>
__device__ __forceinline__ float digit_of(I G, int sh, bool top) {
  if (top) return (float)(int)(G >> sh);
  return __uint_as_float(0x4B000000u | ((unsigned)(G >> sh) & 127u)) - 8388672.0f;
}
// LEFT: w+x, z-y, w-x, y+z, x+z, x-z, w+y, w-y; right: w+x, y-z, y+z, w-x, x+y, x-y, w-z, w+z.
template <bool LEFT>
__device__ __forceinline__ void digit_sums(float w, float x, float y, float z, float* c) {
  if (LEFT) {
    c[0] = w + x; c[1] = z - y; c[2] = w - x; c[3] = y + z;
    c[4] = x + z; c[5] = x - z; c[6] = w + y; c[7] = w - y;
  } else {
    c[0] = w + x; c[1] = y - z; c[2] = y + z; c[3] = w - x;
    c[4] = x + y; c[5] = x - y; c[6] = w - z; c[7] = w + z;
  }
}
// dst: the entries' place in slice 0, product p0; planes ps apart, slices np ps apart.
template <bool LEFT, typename I>
__device__ __forceinline__ void slices_store(bf16* dst, long ps, int S, int p0, int np, const I (*G)[8]) {
  for (int l = 0; l < S; l++) {
    const int sh = 7 * (S - 1 - l);
    uint32_t pk[8][4];
#pragma unroll
    for (int t = 0; t < 8; t += 2) {
      float a[8], b[8];
      digit_sums<LEFT>(digit_of(G[0][t], sh, l == 0), digit_of(G[1][t], sh, l == 0), digit_of(G[2][t], sh, l == 0),
                       digit_of(G[3][t], sh, l == 0), a);
      digit_sums<LEFT>(digit_of(G[0][t + 1], sh, l == 0), digit_of(G[1][t + 1], sh, l == 0),
                       digit_of(G[2][t + 1], sh, l == 0), digit_of(G[3][t + 1], sh, l == 0), b);
#pragma unroll
      for (int p = 0; p < 8; p++) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(a[p], b[p]);
        pk[p][t >> 1] = *reinterpret_cast<const uint32_t*>(&h);
      }
    }
    bf16* dl = dst + (long)l * np * ps;
#pragma unroll
    for (int p = 0; p < 8; p++)
      if (p >= p0 && p < p0 + np)
        *reinterpret_cast<uint4*>(dl + (p - p0) * ps) = make_uint4(pk[p][0], pk[p][1], pk[p][2], pk[p][3]);
  }
}

// A-form: WPR warps per row find the row's exponent (one read of the row),
// then slice it (the second read hits L1 / L2: a row is at most a few
// hundred KB), so no separate exponent pass is needed.
//
// Blocks past the slicing (blockIdx.x >= cx.first) find the column exponents'
// partial maxima of the product's other operand: both are needed before the
// columns can be sliced, and neither depends on the other (one launch less).
template <typename T>
struct ColExp {
  Planes<const T> A;
  int rows = 0, cols = 0, chunk_rows = 0, colblocks = 0, first = 0x7fffffff;
  int S = 0;            // slices
  int* part = nullptr;  // [chunk][cols]
};
template <typename T>
__device__ __forceinline__ void col_maxexp_block(const ColExp<T>& cx, int blk, int (*sh)[32]) {
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int j = (blk % cx.colblocks) * 32 + tx, ch = blk / cx.colblocks;
  const int r0 = ch * cx.chunk_rows, r1 = min(cx.rows, r0 + cx.chunk_rows);
  typename Bits<T>::U top = 0;
  if (j < cx.cols)
#pragma unroll 2
    for (int i = r0 + ty; i < r1; i += 8)
#pragma unroll
      for (int c = 0; c < 4; c++) top = max(top, abs_bits(cx.A.p[c * cx.A.ps + (long)i * cx.A.ld + j]));
  int mx = exp_of<T>(top, cx.S);
  sh[ty][tx] = mx;
  __syncthreads();
  if (ty == 0 && j < cx.cols) {
#pragma unroll
    for (int t = 1; t < 8; t++) mx = max(mx, sh[t][tx]);
    cx.part[(long)ch * cx.cols + j] = mx;
  }
}
template <typename T, int WPR, typename I>
__global__ void __launch_bounds__(256, 2) k_slice_rows(Planes<const T> A, int rows, int cols, int* __restrict__ e_out,
                                                    int S, int p0, int np, bf16* dst, long ld, long ps, ColExp<T> cx) {
  pdl_wait();
  pdl_trigger();
  __shared__ int sh2[8][32];
  if ((int)blockIdx.x >= cx.first) {
    col_maxexp_block<T>(cx, blockIdx.x - cx.first, sh2);
    return;
  }
  int* sh = sh2[0];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * (8 / WPR) + warp / WPR, tr = (warp % WPR) * 32 + lane;
  const bool ok = i < rows;
  const T* row = A.p + (long)(ok ? i : 0) * A.ld;
  typename Bits<T>::U top = 0;
  if (ok) {
#pragma unroll 4
    for (int j = tr; j < cols; j += 32 * WPR)
#pragma unroll
      for (int c = 0; c < 4; c++) top = max(top, abs_bits(row[c * A.ps + j]));
  }
  int mx = exp_of<T>(top, S);
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (WPR > 1) {
    if (lane == 0) sh[warp] = mx;
    __syncthreads();
    const int w0 = warp / WPR * WPR;
#pragma unroll
    for (int q = 0; q < WPR; q++) mx = max(mx, sh[w0 + q]);
  }
  if (!ok) return;
  const int e = mx == -100000 ? 0 : mx;
  if (tr == 0) e_out[i] = e;
  const int g8 = (cols + 7) / 8;
  for (int g = tr; g < g8; g += 32 * WPR) {
    I G[4][8];
#pragma unroll
    for (int c = 0; c < 4; c++) {
      const T* src = row + c * A.ps + 8 * g;
      T v[8];
#pragma unroll
      for (int q = 0; q < 8; q++) v[q] = 8 * g + q < cols ? src[q] : (T)0;
      slice_bias(v, S, e, G[c]);
    }
    slices_store<true, I>(dst + (long)i * ld + 8 * g, ps, S, p0, np, G);
  }
}

// B-form (the plane-wise transpose): a block takes 64
// rows x 32 columns of the four planes through shared memory (and finishes its
// columns' exponents from the chunk maxima), then each thread slices 8 consecutive rows of one column (a warp's stores cover 128
// bytes of each of 4 slice rows).  Rows past `rows` up to the padded pitch are 0.
constexpr int SC_ROWS = 64, SC_COLS = 32;
template <typename T, typename I>
__global__ void __launch_bounds__(256, 2) k_slice_cols(Planes<const T> A, int rows, int cols, const int* __restrict__ part,
                                                       int chunks, int* __restrict__ e, int S, int p0, int np,
                                                       bf16* dst, long ld, long ps) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) unsigned char sc_smem[];
  __shared__ int ecol[SC_COLS];
  T(*tile)[SC_COLS][SC_ROWS + 1] = reinterpret_cast<T(*)[SC_COLS][SC_ROWS + 1]>(sc_smem);
  const int i0 = blockIdx.y * SC_ROWS, j0 = blockIdx.x * SC_COLS;
  {
    const int jl = threadIdx.x & 31;
#pragma unroll 2
    for (int il = threadIdx.x >> 5; il < SC_ROWS; il += 8) {
      const bool in = i0 + il < rows && j0 + jl < cols;
#pragma unroll
      for (int c = 0; c < 4; c++) tile[c][jl][il] = in ? A.p[c * A.ps + (long)(i0 + il) * A.ld + j0 + jl] : (T)0;
    }
  }
  if (threadIdx.x < SC_COLS) {  // the columns' exponents from their chunks' maxima
    const int j = j0 + threadIdx.x;
    int mx = -100000;
    if (j < cols)
      for (int ch = 0; ch < chunks; ch++) mx = max(mx, part[(long)ch * cols + j]);
    mx = mx == -100000 ? 0 : mx;
    ecol[threadIdx.x] = mx;
    if (blockIdx.y == 0 && j < cols) e[j] = mx;
  }
  __syncthreads();
  const int jl = threadIdx.x >> 3, ig = (threadIdx.x & 7) * 8;
  const int j = j0 + jl;
  if (j < cols && i0 + ig < ((rows + 7) / 8) * 8) {
    const int ej = ecol[jl];
    I G[4][8];
#pragma unroll
    for (int c = 0; c < 4; c++) {
      T v[8];
#pragma unroll
      for (int q = 0; q < 8; q++) v[q] = tile[c][jl][ig + q];
      slice_bias(v, S, ej, G[c]);
    }
    slices_store<false, I>(dst + (long)j * ld + i0 + ig, ps, S, p0, np, G);
  }
}

// ||A||_F^2, the non-finite count and the modulus sums of A's rows and columns
// in one read: a block takes 64 rows x 32 columns and writes one partial sum
// per row and per column of its tile (the moduli meet in shared memory).
// Bound: the FP64 pipe's square roots (about 15 instructions each), so they
// are taken once per entry: a pass each for the norm, the row sums and the
// column sums, and three more launches for their ends, took 340 us at 2048^2.
constexpr int MN_ROWS = 64, MN_COLS = 32;
__global__ void __launch_bounds__(256) k_matrix_norms(Planes<const double> A, int m, int n, double* rowpart,
                                                      double* colpart, Reduce r) {
  pdl_wait();
  pdl_trigger();
  __shared__ double mod[MN_ROWS][MN_COLS + 1];
  __shared__ double sh[256];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  // tiles in one dimension, the columns' first: a grid's y extent is limited to 65535
  const int cb = (n + MN_COLS - 1) / MN_COLS, bx = blockIdx.x % cb, by = blockIdx.x / cb;
  const int j = bx * MN_COLS + tx, r0 = by * MN_ROWS;
  double s = 0.0, col = 0.0;
  int bad = 0;
#pragma unroll 2
  for (int il = ty; il < MN_ROWS; il += 8) {
    const int i = r0 + il;
    double x[4] = {0.0, 0.0, 0.0, 0.0};
    if (i < m && j < n) {
#pragma unroll
      for (int c = 0; c < 4; c++) x[c] = A.p[c * A.ps + (long)i * A.ld + j];
    }
    const double q = fma(x[3], x[3], fma(x[2], x[2], fma(x[1], x[1], x[0] * x[0])));
#pragma unroll
    for (int c = 0; c < 4; c++) bad += nonfinite_bits(x[c]);
    const double d = sqrt(q);
    s += q;
    col += d;
    mod[il][tx] = d;
  }
  const double t0 = block_sum(s, sh);
  const double t1 = block_count(bad, sh);
  if (threadIdx.x == 0) {
    double* p = r.partials + 2 * (long)blockIdx.x;
    p[0] = t0;
    p[1] = t1;
  }
  __syncthreads();
  sh[threadIdx.x] = col;
  __syncthreads();
  if (ty == 0 && j < n) {
#pragma unroll
    for (int k = 1; k < 8; k++) col += sh[tx + 32 * k];
    colpart[(long)by * n + j] = col;
  }
  if (threadIdx.x >= 64 && threadIdx.x < 64 + MN_ROWS) {
    const int il = threadIdx.x - 64;
    double t = 0.0;
    for (int k = 0; k < MN_COLS; k++) t += mod[il][k];
    if (r0 + il < m) rowpart[(long)bx * m + r0 + il] = t;
  }
  reduce_last_block<2>(r, gridDim.x, sh);
}

// The largest row sum and column sum from the partials (summed in block
// order); the last block takes the maximum over the blocks.
__global__ void __launch_bounds__(256) k_norms_finish(const double* rowpart, int cb, int m, const double* colpart,
                                                      int rb, int n, int row_blocks, Reduce r) {
  pdl_wait();
  pdl_trigger();
  __shared__ double sh[256];
  __shared__ int last;
  const bool rows = (int)blockIdx.x < row_blocks;
  const int idx = (rows ? blockIdx.x : blockIdx.x - row_blocks) * 256 + threadIdx.x, len = rows ? m : n;
  const double* p = rows ? rowpart : colpart;
  const int parts = rows ? cb : rb;
  double s = 0.0;
  if (idx < len)
#pragma unroll 4
    for (int k = 0; k < parts; k++) s += p[(long)k * len + idx];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int k = 128; k > 0; k >>= 1) {
    if ((int)threadIdx.x < k) sh[threadIdx.x] = fmax(sh[threadIdx.x], sh[threadIdx.x + k]);
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    r.partials[blockIdx.x] = sh[0];
    __threadfence();
    last = atomicAdd(r.count, 1u) == gridDim.x - 1 ? 1 : 0;
  }
  __syncthreads();
  if (!last || threadIdx.x >= 2) return;
  __threadfence();
  double mx = 0.0;
  const int b0 = threadIdx.x == 0 ? 0 : row_blocks, b1 = threadIdx.x == 0 ? row_blocks : (int)gridDim.x;
  for (int b = b0; b < b1; b++) mx = fmax(mx, __ldcg(r.partials + b));
  r.out[2 + threadIdx.x] = mx;
  if (threadIdx.x == 0) *r.count = 0;
}

constexpr int CR_COLS = 32, CR_MAX_CHUNKS = 64;  // column blocks and row chunks of the column exponents

// ||A - B||_F^2 (B optional) and the non-finite count of A.  Work is split
// into tasks of one row and FRO_COLS consecutive columns; a block takes tasks
// blockIdx.x + k gridDim.x, FRO_U of them at a time with all their loads of A
// issued before the first use.  FP64 pipe: one FMA per value and nothing else
// (a run-time scale compared with 1.0 and a diagonal term compared with 0.0
// made it four: 136 us for a 2048^2 matrix, 20 at the copy bandwidth).
constexpr int FRO_COLS = 256, FRO_U = 2;
template <bool HASB>
__global__ void __launch_bounds__(FRO_COLS) k_fro2(Planes<const double> A, Planes<const double> B, int m, int n,
                                                   Reduce r) {
  pdl_wait();
  pdl_trigger();
  __shared__ double sh[256];
  const unsigned chunks = (n + FRO_COLS - 1) / FRO_COLS;
  const unsigned tasks = (unsigned)m * chunks;  // below 2^31 for any matrix that fits the device
  double s = 0.0;
  int bad = 0;
  for (unsigned t0 = blockIdx.x; t0 < tasks; t0 += FRO_U * gridDim.x) {
    double x[FRO_U][4];
    long off[FRO_U];
    int jj[FRO_U];
    bool ok[FRO_U];
#pragma unroll
    for (int u = 0; u < FRO_U; u++) {
      const unsigned t = t0 + u * gridDim.x, row = t / chunks;
      off[u] = row;
      jj[u] = (int)(t - row * chunks) * FRO_COLS + threadIdx.x;
      ok[u] = t < tasks && jj[u] < n;
#pragma unroll
      for (int c = 0; c < 4; c++) x[u][c] = ok[u] ? A.p[c * A.ps + off[u] * A.ld + jj[u]] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < FRO_U; u++) {
#pragma unroll
      for (int c = 0; c < 4; c++) {
        double v = x[u][c];
        bad += nonfinite_bits(v);
        if (HASB) v -= ok[u] ? B.p[c * B.ps + off[u] * B.ld + jj[u]] : 0.0;
        s = fma(v, v, s);
      }
    }
  }
  const double t0 = block_sum(s, sh);
  const double t1 = block_count(bad, sh);
  if (threadIdx.x == 0) {
    r.partials[2 * blockIdx.x] = t0;
    r.partials[2 * blockIdx.x + 1] = t1;
  }
  reduce_last_block<2>(r, gridDim.x, sh);
}

// The Penrose pass's sums over a residual plane set (see launch_penrose_norms)
// in one read: a block takes the tile pair (I, J), (J, I), I <= J, so that the
// anti-Hermitian part |conj(R_ji) - R_ij|^2 is formed once per pair and counted
// twice (diagonal tiles once).  Replaces three passes per residual (its norm,
// the norm of +-R + I, which differs on the diagonal's s plane only, and the
// anti-Hermitian part) at 2 FP64 operations per value instead of 7.
__global__ void __launch_bounds__(256) k_penrose_norms(Planes<const double> R, int n, int neg, Reduce r) {
  pdl_wait();
  pdl_trigger();
  __shared__ double t[4][TILE][TILE + 1];
  __shared__ double sh[256];
  // blockIdx.x = J (J + 1) / 2 + I
  int J = (int)((sqrtf(8.f * (float)blockIdx.x + 1.f) - 1.f) * 0.5f);
  while ((long)J * (J + 1) / 2 > blockIdx.x) J--;
  while ((long)(J + 1) * (J + 2) / 2 <= blockIdx.x) J++;
  const int I = (int)(blockIdx.x - (long)J * (J + 1) / 2);
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, r0 = I * TILE, c0 = J * TILE;
  double s = 0.0, sd = 0.0, s1 = 0.0, ah = 0.0;
  // the mirrored tile R[c0.., r0..], transposed into shared memory
  for (int q = 0; q < TILE / TROWS; q++) {
    const int i = c0 + ty + q * TROWS, j = r0 + tx;
#pragma unroll
    for (int c = 0; c < 4; c++) {
      const double v = (i < n && j < n) ? R.p[c * R.ps + (long)i * R.ld + j] : 0.0;
      t[c][tx][ty + q * TROWS] = v;
      if (I != J) s = fma(v, v, s);
    }
  }
  __syncthreads();
  for (int q = 0; q < TILE / TROWS; q++) {
    const int i = r0 + ty + q * TROWS, j = c0 + tx;
    if (i >= n || j >= n) continue;
#pragma unroll
    for (int c = 0; c < 4; c++) {
      const double v = R.p[c * R.ps + (long)i * R.ld + j], w = t[c][ty + q * TROWS][tx];  // R_ij, R_ji
      const double d = c == 0 ? w - v : w + v;
      ah = fma(d, d, ah);
      if (c == 0 && i == j) {
        sd = fma(v, v, sd);
        const double x = (neg ? flip_sign(v) : v) + 1.0;
        s1 = fma(x, x, s1);
      } else {
        s = fma(v, v, s);
      }
    }
  }
  const double b0 = block_sum(s, sh), b1 = block_sum(sd, sh), b2 = block_sum(s1, sh), b3 = block_sum(ah, sh);
  if (threadIdx.x == 0) {
    double* p = r.partials + 4 * (long)blockIdx.x;
    p[0] = b0;
    p[1] = b1;
    p[2] = b2;
    p[3] = I == J ? b3 : 2.0 * b3;
  }
  reduce_last_block<4>(r, gridDim.x, sh);
}

// X (n x m) = alpha * A^H, A m x n: X[j][i] = alpha * conj(A[i][j]).
template <typename T>
__global__ void __launch_bounds__(256) k_init_x0(Planes<const double> A, int m, int n, double al, Planes<T> X) {
  pdl_wait();
  pdl_trigger();
  __shared__ double t[4][TILE][TILE + 1];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int r0 = blockIdx.y * TILE, c0 = blockIdx.x * TILE;  // tile of A: rows r0.., cols c0..
  for (int q = 0; q < TILE / TROWS; q++) {
    const int i = r0 + ty + q * TROWS, j = c0 + tx;
    for (int c = 0; c < 4; c++)
      t[c][ty + q * TROWS][tx] = (i < m && j < n) ? A.p[c * A.ps + (long)i * A.ld + j] : 0.0;
  }
  __syncthreads();
  for (int q = 0; q < TILE / TROWS; q++) {
    const int j = c0 + ty + q * TROWS, i = r0 + tx;  // X element (j, i)
    if (i < m && j < n)
      for (int c = 0; c < 4; c++) {
        const double v = t[c][tx][ty + q * TROWS];
        const double x = al * (c == 0 ? v : flip_sign(v));
        X.p[c * X.ps + (long)j * X.ld + i] = sizeof(T) == 4 ? (T)narrow(x) : (T)x;
      }
  }
}

// Row chunks of a column reduction: about four blocks per SM of a 152-SM
// part in total, at least 64 rows per chunk.
static int col_chunks(int rows, int cols) {
  const int colblocks = (cols + CR_COLS - 1) / CR_COLS;
  int ch = (608 + colblocks - 1) / colblocks;
  ch = std::min(ch, (rows + 63) / 64);
  return std::max(1, std::min(ch, CR_MAX_CHUNKS));
}

__global__ void k_f32_to_f64(Planes<const float> S, int rows, int cols, Planes<double> D) {
  pdl_wait();
  pdl_trigger();
  const long total = (long)rows * cols;
  for (long t = (long)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
    const long i = t / cols, j = t % cols;
    for (int c = 0; c < 4; c++) D.p[c * D.ps + i * D.ld + j] = widen(S.p[c * S.ps + i * S.ld + j]);
  }
}

__global__ void k_f64_to_f32(Planes<const double> S, int rows, int cols, Planes<float> D) {
  pdl_wait();
  pdl_trigger();
  const long total = (long)rows * cols;
  for (long t = (long)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
    const long i = t / cols, j = t % cols;
    for (int c = 0; c < 4; c++) D.p[c * D.ps + i * D.ld + j] = narrow(S.p[c * S.ps + i * S.ld + j]);
  }
}

// D = S, four planes: a block takes 512 columns of a row (two per thread).
__global__ void __launch_bounds__(256) k_copy_planes(Planes<const double> S, int rows, int cols, Planes<double> D) {
  pdl_wait();
  pdl_trigger();
  const int j = (blockIdx.x * 256 + threadIdx.x) * 2;
  if (j >= cols) return;
  for (int i = blockIdx.y; i < rows; i += gridDim.y) {
    double u[4][2];
#pragma unroll
    for (int c = 0; c < 4; c++) ld2(S.p + c * S.ps + (long)i * S.ld + j, j + 1 < cols, u[c][0], u[c][1]);
#pragma unroll
    for (int c = 0; c < 4; c++) st2(D.p + c * D.ps + (long)i * D.ld + j, j + 1 < cols, u[c][0], u[c][1]);
  }
}

int grid_for(long total) {
  long blocks = (total + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  if (blocks < 1) blocks = 1;
  return (int)blocks;
}

}  // namespace

int combine_blocks(const CombineArgs& a) {
  const int rows = TROWS * combine_groups(a);
  return ((a.cols + 2 * TILE - 1) / (2 * TILE)) * ((a.rows + rows - 1) / rows);
}

cudaError_t launch_combine(const CombineArgs& args, cudaStream_t st) {
  CombineArgs a = args;
  for (int o = 0; o < a.nout; o++) a.out[o].set_coefs();
  if (a.rows <= 0 || a.cols <= 0) return cudaSuccess;
  const int groups = combine_groups(a), rows = TROWS * groups;
  dim3 grid((a.cols + 2 * TILE - 1) / (2 * TILE), (a.rows + rows - 1) / rows);
  if (a.f64)
    QP_LAUNCH(k_combine<double>, grid, dim3(256), 0, st, a, groups);
  else
    QP_LAUNCH(k_combine<float>, grid, dim3(256), 0, st, a, groups);
  ++g_kernel_launches;
  return cudaGetLastError();
}

long norms_scratch(int m, int n) {  // row and column partials, block partials of both launches
  const long cb = (n + MN_COLS - 1) / MN_COLS, rb = (m + MN_ROWS - 1) / MN_ROWS;
  return cb * m + rb * n + std::max(2 * cb * rb, (long)(m + 255) / 256 + (n + 255) / 256);
}
cudaError_t launch_matrix_norms(const Planes<const double>& A, int m, int n, double* scratch, double* out,
                                unsigned int* count, cudaStream_t st) {
  const int cb = (n + MN_COLS - 1) / MN_COLS, rb = (m + MN_ROWS - 1) / MN_ROWS;
  if ((long)cb * rb > 0x7fffffffL) return cudaErrorInvalidValue;  // 2^42 entries
  double *rowpart = scratch, *colpart = scratch + (long)cb * m;
  const Reduce r{colpart + (long)rb * n, out, count};
  QP_LAUNCH(k_matrix_norms, dim3(cb * rb), dim3(256), 0, st, A, m, n, rowpart, colpart, r);
  const int row_blocks = (m + 255) / 256;
  QP_LAUNCH(k_norms_finish, dim3(row_blocks + (n + 255) / 256), dim3(256), 0, st, rowpart, cb, m, colpart, rb, n,
            row_blocks, r);
  g_kernel_launches += 2;
  return cudaGetLastError();
}

cudaError_t launch_fro2(const Planes<const double>& A, const Planes<const double>* B, int m, int n, const Reduce& r,
                        cudaStream_t st) {
  const long tasks = (long)m * ((n + FRO_COLS - 1) / FRO_COLS);
  const int blocks = (int)std::max(1L, std::min<long>(tasks, kFroBlocks));
  if (B)
    QP_LAUNCH(k_fro2<true>, dim3(blocks), dim3(FRO_COLS), 0, st, A, *B, m, n, r);
  else
    QP_LAUNCH(k_fro2<false>, dim3(blocks), dim3(FRO_COLS), 0, st, A, A, m, n, r);
  ++g_kernel_launches;
  return cudaGetLastError();
}

int penrose_norm_blocks(int n) {
  const int t = (n + TILE - 1) / TILE;
  return t * (t + 1) / 2;
}
cudaError_t launch_penrose_norms(const Planes<const double>& R, int n, double sr, const Reduce& r, cudaStream_t st) {
  QP_LAUNCH(k_penrose_norms, dim3(penrose_norm_blocks(n)), dim3(TILE * TROWS), 0, st, R, n, sr < 0 ? 1 : 0, r);
  ++g_kernel_launches;
  return cudaGetLastError();
}

template <typename T>
static cudaError_t init_x0_t(const Planes<const double>& A, int m, int n, double alpha, const Planes<T>& X,
                             cudaStream_t st) {
  dim3 grid((n + TILE - 1) / TILE, (m + TILE - 1) / TILE);
  QP_LAUNCH(k_init_x0<T>, grid, dim3(TILE * TROWS), 0, st, A, m, n, alpha, X);
  ++g_kernel_launches;
  return cudaGetLastError();
}
cudaError_t launch_init_x0(const Planes<const double>& A, int m, int n, double alpha, const Planes<double>& X,
                           cudaStream_t st) {
  return init_x0_t<double>(A, m, n, alpha, X, st);
}
cudaError_t launch_init_x0(const Planes<const double>& A, int m, int n, double alpha, const Planes<float>& X,
                           cudaStream_t st) {
  return init_x0_t<float>(A, m, n, alpha, X, st);
}

cudaError_t launch_copy_planes(const Planes<const double>& S, int rows, int cols, const Planes<double>& D,
                               cudaStream_t st) {
  if (rows <= 0 || cols <= 0) return cudaSuccess;
  QP_LAUNCH(k_copy_planes, dim3((cols + 511) / 512, std::min(rows, 8192)), dim3(256), 0, st, S, rows, cols, D);
  ++g_kernel_launches;
  return cudaGetLastError();
}

cudaError_t launch_f32_to_f64(const Planes<const float>& src, int rows, int cols, const Planes<double>& dst,
                              cudaStream_t st) {
  QP_LAUNCH(k_f32_to_f64, dim3(grid_for((long)rows * cols)), dim3(256), 0, st, src, rows, cols, dst);
  ++g_kernel_launches;
  return cudaGetLastError();
}

cudaError_t launch_f64_to_f32(const Planes<const double>& src, int rows, int cols, const Planes<float>& dst,
                              cudaStream_t st) {
  QP_LAUNCH(k_f64_to_f32, dim3(grid_for((long)rows * cols)), dim3(256), 0, st, src, rows, cols, dst);
  ++g_kernel_launches;
  return cudaGetLastError();
}


// See common.cuh.  The row-slicing blocks of P and the exponent blocks of Q
// share a launch; either part may be absent.
template <typename T, typename I>
static cudaError_t slice_t(const SliceArgs& a, const Planes<const T>& P, const Planes<const T>& Q, cudaStream_t st) {
  auto bad = [](long ld, long ps, const bf16* dst, int k) {
    return (ld & 7) || (ps & 7) || (reinterpret_cast<uintptr_t>(dst) & 15) || ld < ((k + 7) / 8) * 8;
  };
  if (a.M <= 0 || a.N <= 0 || a.K <= 0) return cudaSuccess;
  if ((a.za && bad(a.lda, a.psa, a.za, a.K)) || (a.zb && bad(a.ldb, a.psb, a.zb, a.K))) return cudaErrorInvalidValue;
  // four warps per row once a row is more than two iterations of one warp
  const int wpr = a.K > 512 ? 4 : 1;
  const int row_blocks = a.za ? (wpr == 4 ? (a.M + 1) / 2 : (a.M + 7) / 8) : 0;
  const int chunks = col_chunks(a.K, a.N);
  ColExp<T> cx;
  int col_blocks = 0;
  if (a.zb && a.p0 == 0) {  // the exponents serve every group of products
    cx.A = Q;
    cx.S = a.S;
    cx.rows = a.K;
    cx.cols = a.N;
    cx.chunk_rows = (a.K + chunks - 1) / chunks;
    cx.colblocks = (a.N + 31) / 32;
    cx.first = row_blocks;
    cx.part = a.scratch;
    col_blocks = cx.colblocks * chunks;
  }
  if (row_blocks + col_blocks > 0) {
    if (wpr == 4)
      QP_LAUNCH(k_slice_rows<T, 4, I>, dim3(row_blocks + col_blocks), dim3(256), 0, st, P, a.M, a.K, a.eP, a.S, a.p0,
                a.np, a.za, a.lda, a.psa, cx);
    else
      QP_LAUNCH(k_slice_rows<T, 1, I>, dim3(row_blocks + col_blocks), dim3(256), 0, st, P, a.M, a.K, a.eP, a.S, a.p0,
                a.np, a.za, a.lda, a.psa, cx);
    ++g_kernel_launches;
    if (cudaError_t err = cudaGetLastError()) return err;
  }
  if (a.zb) {
    constexpr int smem = (int)sizeof(T) * 4 * SC_COLS * (SC_ROWS + 1);
    static std::atomic<unsigned long long> attr_done{0};
    if (cudaError_t err = ensure_smem_attr(k_slice_cols<T, I>, smem, attr_done)) return err;
    dim3 grid((a.N + SC_COLS - 1) / SC_COLS, (a.K + SC_ROWS - 1) / SC_ROWS);
    QP_LAUNCH(k_slice_cols<T, I>, grid, dim3(256), smem, st, Q, a.K, a.N, a.scratch, chunks, a.eQ, a.S, a.p0, a.np,
              a.zb, a.ldb, a.psb);
    ++g_kernel_launches;
  }
  return cudaGetLastError();
}
cudaError_t launch_slices(const SliceArgs& a, const Planes<const double>& P, const Planes<const double>& Q,
                          cudaStream_t st) {
  return slice_t<double, long long>(a, P, Q, st);
}
cudaError_t launch_slices(const SliceArgs& a, const Planes<const float>& P, const Planes<const float>& Q,
                          cudaStream_t st) {
  return a.S <= 4 ? slice_t<float, int>(a, P, Q, st) : slice_t<float, long long>(a, P, Q, st);
}

}  // namespace qp
