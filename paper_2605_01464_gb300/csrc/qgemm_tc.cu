// qgemm_tc.cu -- quaternion GEMM on the sm_103a tensor cores (tcgen05 + TMEM + TMA).
//
// The quaternion product C = A B (Hamilton product, Sec. 2) is one real
// contraction [C0 C1 C2 C3] = [A0 A1 A2 A3] M(B), where block (r, c) of the
// 4K x 4N matrix M(B) is +-B_{r xor c}:
//     c=0    c=1    c=2    c=3
//   r=0 +B0   +B1    +B2    +B3
//   r=1 -B1   +B0    -B3    +B2
//   r=2 -B2   +B3    +B0    -B1
//   r=3 -B3   -B2    +B1    +B0
// M(B) is never formed: per K step the kernel stages the four A planes and
// the four B planes of a tile in shared memory (TMA, 64-byte swizzle) and
// issues the (r, c) products as separate tcgen05.mma instructions, each
// reading plane r xor c of B and taking its sign from the instruction
// descriptor's negate-A bit.  Output components accumulate in FP32 in TMEM.
//
// Split operands: A and B are sums of BF16 terms (A = A_0 + A_1 + ...); the
// kernel accumulates A_i B_j over a list of (i, j) pairs, giving products
// accurate to about 2^-8 (1 term), 2^-16 (3 pairs) or 2^-24 (6 pairs).
//
// One persistent kernel, one CTA per SM, over work items (tile of 128 x BN
// entries, NC of the four output components); warp 0 issues TMA loads, warp 1
// owns TMEM and issues the MMAs (one elected lane), 16 warps drain finished
// items from TMEM, running the fused combine pass, while the MMA warp fills
// the next item's accumulators.  Four shapes (tc_shape): every output entry
// receives the same MMAs in the same order in all of them, so they give
// bit-identical products.
//
// Measured (GB300): single pass 4096^3 with FP64 output 1.17-1.21 ms = 1813-1875
// TFLOP/s (1.14 ms = 1930 with FP32 output; 1609 with one-lane issue loops, see
// elect_one); the fused products of a 60 x 512 solve 119 -> 18 us (all of a small
// product's epilogue ran on one SM's four warps), of a 500^2 one 93 -> 45 us.
// The 2048^2 solve's fused single-pass products take 216-263 us, their MMAs 157:
// the component pair's operand traffic (64 bytes per cycle and SM at full rate)
// and the last item's epilogue are what is left.
// Every wait is bounded (2 s of globaltimer); on expiry the kernel records
// an error code, stops at its next work item, drains what it started and frees TMEM.
#include <cuda.h>

#include <algorithm>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace qp {
namespace {

constexpr int BM = 128;      // output rows per tile = TMEM lanes
constexpr int BK = 32;       // K elements per stage: one 64-byte swizzle row
constexpr int GROUP_M = 16;  // rasterization: 16 row tiles per group share B tiles in L2
constexpr int A_PLANE = BM * BK * 2;
constexpr int EPI_WARPS = 16;
constexpr int THREADS = 32 * (2 + EPI_WARPS);
constexpr int TP = 48;       // row pitch (bytes) of the epilogue's 16 x 16 BF16 tiles: conflict-free stmatrix

template <int BN_, int NC_>
struct Cfg {
  static constexpr int BN = BN_, NC = NC_;
  static constexpr int B_PLANE = BN * BK * 2;
  static constexpr int STAGE = 4 * (A_PLANE + B_PLANE);
  static constexpr int STAGES = BN == 128 ? 3 : 4;
  static constexpr int STG_WARP = 2 * 16 * TP;  // A-form and B-form tile of an epilogue warp
  static constexpr int SMEM = STAGES * STAGE + EPI_WARPS * STG_WARP + 1024;
  static constexpr int ACC = NC * BN;                   // TMEM columns of one accumulator
  static constexpr int NBUF = 2 * ACC <= 512 ? 2 : 1;   // accumulators used in turn
  static constexpr int TMEM = NBUF * ACC;
  static constexpr int PIECES = ACC / 8;  // 16 x 16 epilogue pieces of a TMEM lane quarter
  // Instruction descriptor, kind::f16: D = F32, A = B = BF16, both K-major.
  static constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                                    ((uint32_t)(BM >> 4) << 24);
  static_assert(SMEM <= 227 * 1024, "shared memory per CTA");
  static_assert(PIECES % 4 == 0 && BN % 16 == 0, "four warps per lane quarter share its pieces");
  static_assert(TMEM >= 32 && (TMEM & (TMEM - 1)) == 0, "TMEM allocation");
};

struct KParams {
  int M, N;
  int Mt, Nt, items;
  int arows;     // rows of the A box: 128, or fewer when the whole matrix has fewer
  int kb0, kb1;  // K blocks [kb0, kb1) of BK elements
  int npairs;
  int pi[16], pj[16];
  Planes<float> C;
  EpiArgs E;     // E.nout > 0: fused combine epilogue
  int plain64;   // ... of one FP64 output that is the product itself
  int* err;
};

// Two adjacent entries (x, y) of a row; `two`: y is inside the matrix.
__device__ __forceinline__ void load2(const float* p, bool two, float* u) {
  if (two && (reinterpret_cast<uintptr_t>(p) & 7) == 0) {
    const float2 t = *reinterpret_cast<const float2*>(p);
    u[0] = t.x;
    u[1] = t.y;
  } else {
    u[0] = p[0];
    u[1] = two ? p[1] : 0.f;
  }
}
__device__ __forceinline__ void load2(const double* p, bool two, double* u) {
  if (two && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
    const double2 t = *reinterpret_cast<const double2*>(p);
    u[0] = t.x;
    u[1] = t.y;
  } else {
    u[0] = p[0];
    u[1] = two ? p[1] : 0.0;
  }
}
__device__ __forceinline__ void store2(float* p, bool two, float x, float y) {
  if (two && (reinterpret_cast<uintptr_t>(p) & 7) == 0) {
    *reinterpret_cast<float2*>(p) = make_float2(x, y);
  } else {
    p[0] = x;
    if (two) p[1] = y;
  }
}
__device__ __forceinline__ void store2(double* p, bool two, double x, double y) {
  if (two && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
    *reinterpret_cast<double2*>(p) = make_double2(x, y);
  } else {
    p[0] = x;
    if (two) p[1] = y;
  }
}

template <typename T>
__device__ __forceinline__ void store_piece(T* plane, long ld, int r0, int M, int j0, int N, const float* v) {
  const int lane = threadIdx.x & 31, i = r0 + (lane >> 2), j = j0 + 2 * (lane & 3);
  T* dst = plane + (long)i * ld + j;
  T w[8];
  to_master_all<8>(v, w);
#pragma unroll
  for (int t = 0; t < 8; t += 2) {
    const int k = (t >> 1) & 1, jj = j + 8 * (t >> 2);
    if (i + 8 * k < M && jj < N)
      store2(dst + 8 * k * ld + 8 * (t >> 2), jj + 1 < N, w[t], w[t + 1]);
  }
}

// An epilogue piece is 16 rows x 16 columns in the 16x256b fragment layout:
// value e of a lane is at row lane / 4 + 8 ((e >> 1) & 1), column 8 (e >> 2) +
// 2 (lane % 4) + (e & 1).  A warp access then covers 32-byte (FP32) or
// 64-byte (FP64) segments of 8 rows; with one row per lane every access
// touched 32 cache lines and the L1 tag stage was 61-68 % busy (single-pass
// fused products of the 2048^2 solve 229-354 us, their MMAs 157).
//
// Fused combine of one piece, plane c (see EpiArgs): v = the product's
// values.  The whole warp calls this: the BF16 forms go through `stg`, the
// warp's two 16 x 16 tiles of shared memory (stmatrix, transposed for the
// B-form), and leave as 16-byte pieces of 16 rows.  Columns up to the next
// multiple of 8 beyond N and rows beyond M are written as zeros (operand
// forms are padded; the GEMM's TMA maps end at K).
// The piece's auxiliary values towards L1 while its accumulator is not ready.
__device__ __forceinline__ void epi_prefetch(const EpiArgs& E, int c, int r0, int M, int j0, int N) {
  const int lane = threadIdx.x & 31, i0 = r0 + (lane >> 2), jc = j0 + 2 * (lane & 3);
  const int es = E.f64 ? 8 : 4;
#pragma unroll
  for (int a = 0; a < kEpiAux; a++) {
    if (!E.aux[a]) continue;
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int i = i0 + 8 * (q & 1), j = jc + 8 * (q >> 1);
      if (i < M && j < N)
        asm volatile("prefetch.global.L1 [%0];" ::"l"(reinterpret_cast<const char*>(E.aux[a]) +
                                                       (c * E.ps_aux[a] + (long)i * E.ld_aux[a] + j) * es));
    }
  }
}

template <typename T>
__device__ __forceinline__ void epi_piece(const EpiArgs& E, int c, int r0, int M, int j0, int N, const float* v,
                                          uint32_t stg, float& sdx, float& sx, int& bad) {
  const int lane = threadIdx.x & 31, i0 = r0 + (lane >> 2), jc = j0 + 2 * (lane & 3);
  // FP32: every auxiliary value of the piece is loaded before the first use
  constexpr bool PRE = sizeof(T) == 4;
  T u[PRE ? kEpiAux : 1][8];
  auto load_aux = [&](int a, T* x) {
    const T* ap = reinterpret_cast<const T*>(E.aux[a]) + c * E.ps_aux[a] + (long)i0 * E.ld_aux[a] + jc;
#pragma unroll
    for (int e = 0; e < 8; e += 2) {
      const int k = (e >> 1) & 1, j = jc + 8 * (e >> 2);
      x[e] = x[e + 1] = (T)0;
      if (i0 + 8 * k < M && j < N) load2(ap + 8 * k * E.ld_aux[a] + 8 * (e >> 2), j + 1 < N, x + e);
    }
  };
  if (PRE) {
#pragma unroll
    for (int a = 0; a < kEpiAux; a++)
      if (E.aux[a]) load_aux(a, u[PRE ? a : 0]);
  }
#pragma unroll 1
  for (int o = 0; o < E.nout; o++) {
    const EpiOut& O = E.out[o];
    T w[8];
    const int ck = O.cacc.kind;
#pragma unroll
    for (int t = 0; t < 8; t++)  // +-1 as a sign flip (the combine kernel's arithmetic)
      w[t] = ck == CK_ZERO ? (T)0 : to_master<T>(ck == CK_MINUS ? -v[t] : v[t]);
    if (ck == CK_GENERAL) {
#pragma unroll
      for (int t = 0; t < 8; t++) w[t] *= coef<T>(O.cacc);
    }
#pragma unroll
    for (int a = 0; a < kEpiAux; a++) {
      if (!E.aux[a] || O.caux[a].kind == CK_ZERO) continue;
      const T ca = coef<T>(O.caux[a]);
      if (!PRE) load_aux(a, u[0]);
#pragma unroll
      for (int t = 0; t < 8; t++) w[t] += ca * u[PRE ? a : 0][t];
    }
    if (c == 0 && O.diag.kind != CK_ZERO && r0 < j0 + 16 && j0 < r0 + 16) {
#pragma unroll
      for (int t = 0; t < 8; t++)
        if (i0 + 8 * ((t >> 1) & 1) == jc + 8 * (t >> 2) + (t & 1)) w[t] += coef<T>(O.diag);
    }
    if (PRE && o == 0 && E.red.partials) {
#pragma unroll
      for (int t = 0; t < 8; t++)
        if (i0 + 8 * ((t >> 1) & 1) < M && jc + 8 * (t >> 2) + (t & 1) < N) {
          const float x = (float)w[t], x0 = E.aux[0] ? (float)(w[t] - u[0][t]) : x;
          sdx += x0 * x0;
          sx += x * x;
          bad += isfinite(x) ? 0 : 1;
        }
    }
    if (O.mp) {
      T* mp = reinterpret_cast<T*>(O.mp) + c * O.mps + (long)i0 * O.mld + jc;
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        const int k = (e >> 1) & 1, j = jc + 8 * (e >> 2);
        if (i0 + 8 * k < M && j < N) store2(mp + 8 * k * O.mld + 8 * (e >> 2), j + 1 < N, w[e], w[e + 1]);
      }
    }
    if (O.a || O.b) {
      float r[8];
#pragma unroll
      for (int t = 0; t < 8; t++) r[t] = to_float(w[t]);
      // lane L stores row L % 8 of 8 x 8 matrix L / 8 = (row half, column half)
      const int mat = lane >> 3, rr = lane & 7, orow = lane >> 1, ochk = lane & 1;
      const uint32_t sa = stg + ((mat & 1) * 8 + rr) * TP + (mat >> 1) * 16;
      const uint32_t sb = stg + 16 * TP + ((mat >> 1) * 8 + rr) * TP + (mat & 1) * 16;
#pragma unroll 1
      for (int l = 0; l < O.levels; l++) {
        uint32_t h[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
          const __nv_bfloat162 b = __floats2bfloat162_rn(r[2 * q], r[2 * q + 1]);
          r[2 * q] -= __low2float(b);
          r[2 * q + 1] -= __high2float(b);
          h[q] = *reinterpret_cast<const uint32_t*>(&b);
        }
        __syncwarp();  // the previous level's tiles are read
        if (O.a) st_matrix(sa, h);
        if (O.b) st_matrix_trans(sb, h);
        __syncwarp();
        if (O.a && r0 + orow < M && j0 + 8 * ochk < N)
          *reinterpret_cast<uint4*>(O.a + (long)l * 4 * O.psa + c * O.psa + (long)(r0 + orow) * O.lda + j0 +
                                    8 * ochk) = ld_shared16(stg + orow * TP + ochk * 16);
        if (O.b && j0 + orow < N && r0 + 8 * ochk < M)
          *reinterpret_cast<uint4*>(O.b + (long)l * 4 * O.psb + c * O.psb + (long)(j0 + orow) * O.ldb + r0 +
                                    8 * ochk) = ld_shared16(stg + (16 + orow) * TP + ochk * 16);
      }
    }
  }
}

// The signed MMAs of one stage (BK / 16 steps of K = 16, r = 0..3 each) into
// components C0 .. C0 + NC - 1, accumulators BN columns apart.  Descriptors:
// the upper word is the same for all tiles, the lower one is an address / 16;
// ap = distance of the A planes / 16.  With fewer than 128 rows of A the MMAs
// read on into the next plane: those accumulator rows are not used.
template <class C, int C0>
__device__ __forceinline__ void stage_mmas(uint32_t d, uint32_t ad, uint32_t bd, uint32_t ap, uint32_t acc) {
  constexpr uint32_t NEG_A = 1u << 13;
  constexpr uint64_t hi = desc_hi(2 * BK);
#pragma unroll
  for (int kk = 0; kk < BK / 16; kk++)
#pragma unroll
    for (int r = 0; r < 4; r++)
#pragma unroll
      for (int q = 0; q < C::NC; q++) {
        const int c = C0 + q;
        mma_bf16(d + q * C::BN, hi | (ad + r * ap + kk * 2),
                 hi | (bd + (((r ^ c) * C::B_PLANE) >> 4) + kk * 2), qsign_neg(r, c) ? C::IDESC | NEG_A : C::IDESC,
                 (kk || r) ? 1u : acc);
      }
}

template <class C>
__global__ void __launch_bounds__(THREADS, 1)
    k_qgemm_tc(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ KParams P) {
  constexpr int STAGES = C::STAGES, BN = C::BN, NC = C::NC, NBUF = C::NBUF;
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t bar_full[STAGES], bar_empty[STAGES], bar_acc_full[NBUF], bar_acc_empty[NBUF], bar_drain;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  __shared__ double red_sh[32];

  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int units = (P.kb1 - P.kb0) * P.npairs;  // (K block, split pair) units per item

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < STAGES; s++) {
      mbar_init(smem_u32(&bar_full[s]), 1);
      mbar_init(smem_u32(&bar_empty[s]), 1);
    }
    for (int b = 0; b < NBUF; b++) {
      mbar_init(smem_u32(&bar_acc_full[b]), 1);
      mbar_init(smem_u32(&bar_acc_empty[b]), EPI_WARPS);  // one arrival per epilogue warp
    }
    mbar_init(smem_u32(&bar_drain), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(C::TMEM)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_slot;
  pdl_wait();  // the setup above touches no global memory
  pdl_trigger();
  int issued = 0;

  // grouped rasterization: consecutive items walk the component groups of a
  // tile, then GROUP_M row tiles, then the next column tile
  auto item_origin = [&](int item, int& m0, int& n0, int& c0) {
    const int t = item / (4 / NC);
    c0 = NC * (item % (4 / NC));
    const int per_group = GROUP_M * P.Nt, group = t / per_group, local = t % per_group;
    const int gm = min(GROUP_M, P.Mt - group * GROUP_M);
    m0 = (group * GROUP_M + local % gm) * BM;
    n0 = (local / gm) * BN;
  };

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
      int u = 0;
      bool ok = true;
      for (int item = blockIdx.x; item < P.items && ok; item += gridDim.x) {
        int m0, n0, c0;
        item_origin(item, m0, n0, c0);
        for (int x = 0; x < units; x++, u++) {
          const int s = u % STAGES;
          if (u >= STAGES && !mbar_wait(smem_u32(&bar_empty[s]), ((u / STAGES) - 1) & 1, &abort_flag, P.err, 41)) {
            ok = false;
            break;
          }
          const int kb = P.kb0 + x / P.npairs, pr = x % P.npairs;
          const uint32_t fb = smem_u32(&bar_full[s]);
          // one copy per operand: the box holds the four component planes (one
          // copy per plane: 0.064 against 0.055 ms for 500 x 1000 x 500, 2 terms,
          // and no difference for the 128-column shapes)
          mbar_expect_tx(fb, 4 * (P.arows * BK * 2 + C::B_PLANE));
          uint8_t* st = smem + (size_t)s * C::STAGE;
          tma_load_3d(smem_u32(st), &tmA, kb * BK, m0, P.pi[pr] * 4, fb);
          tma_load_3d(smem_u32(st + 4 * A_PLANE), &tmB, kb * BK, n0, P.pj[pr] * 4, fb);
          issued = u + 1;
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: warp-uniform loops, one elected lane ----------------
    const uint32_t a_lo = desc_lo(smem_u32(smem)), b_lo = desc_lo(smem_u32(smem + 4 * A_PLANE));
    const uint32_t ap = (uint32_t)(P.arows * BK * 2) >> 4;
    int s = 0, w = 0;
    uint32_t ph = 0;
    for (int item = blockIdx.x; item < P.items; item += gridDim.x, w++) {
      int m0, n0, c0;
      item_origin(item, m0, n0, c0);
      const int b = w % NBUF;
      if (w >= NBUF) {
        (void)mbar_wait(smem_u32(&bar_acc_empty[b]), ((w / NBUF) - 1) & 1, &abort_flag, P.err, 42);
        if (warp_aborted(&abort_flag)) break;
      }
      fence_after();
      const uint32_t dacc = tmem + b * C::ACC;
      for (int x = 0; x < units; x++) {
        (void)mbar_wait(smem_u32(&bar_full[s]), ph, &abort_flag, P.err, 43);
        fence_after();
        const uint32_t ad = a_lo + s * (C::STAGE >> 4), bd = b_lo + s * (C::STAGE >> 4), acc = x > 0 ? 1u : 0u;
        if (elect_one()) {
          if (NC == 4) stage_mmas<C, 0>(dacc, ad, bd, ap, acc);
          else if (NC == 2) {
            if (c0 == 0) stage_mmas<C, 0>(dacc, ad, bd, ap, acc);
            else stage_mmas<C, 2 & (4 - NC)>(dacc, ad, bd, ap, acc);
          } else {
            switch (c0) {
              case 0: stage_mmas<C, 0>(dacc, ad, bd, ap, acc); break;
              case 1: stage_mmas<C, 1 & (4 - NC)>(dacc, ad, bd, ap, acc); break;
              case 2: stage_mmas<C, 2 & (4 - NC)>(dacc, ad, bd, ap, acc); break;
              default: stage_mmas<C, 3 & (4 - NC)>(dacc, ad, bd, ap, acc); break;
            }
          }
          mma_commit(smem_u32(&bar_empty[s]));
        }
        __syncwarp();
        if (++s == STAGES) {
          s = 0;
          ph ^= 1;
        }
      }
      if (elect_one()) mma_commit(smem_u32(&bar_acc_full[b]));
      __syncwarp();
    }
  } else {
    // ---------------- epilogue: pieces of 16 rows x 16 columns ----------------
    // warp e = warp - 2: TMEM lane quarter warp % 4, every fourth piece of it
    // (16 columns and a half of the quarter's 32 rows each)
    const int quarter = warp & 3, e = warp - 2;
    const uint32_t tq = tmem + ((uint32_t)(quarter * 32) << 16);
    const uint32_t stg = smem_u32(smem + STAGES * C::STAGE + e * C::STG_WARP);
    // Touch every 64 bytes of the parameters while the first MMAs run: each
    // launch starts with them outside the constant cache, and the epilogue's
    // first use of each line otherwise waits for it in turn.
    {
      int warm = 0;
#pragma unroll
      for (int q = 0; q < (int)(sizeof(KParams) / 64); q++) warm ^= reinterpret_cast<const int*>(&P)[16 * q];
      asm volatile("" ::"r"(warm));
    }
    float sdx = 0.f, sx = 0.f;
    int bad = 0;
    int w = 0;
    for (int item = blockIdx.x; item < P.items; item += gridDim.x, w++) {
      int m0, n0, c0;
      item_origin(item, m0, n0, c0);
      const int b = w % NBUF;
      {  // while the item's MMAs run
        const int pc = e >> 2, col = (pc >> 1) * 16, j0 = n0 + col % BN, r0 = m0 + quarter * 32 + (pc & 1) * 16;
        if (P.E.nout > 0 && j0 < P.N && r0 < P.M) epi_prefetch(P.E, c0 + col / BN, r0, P.M, j0, P.N);
      }
      int have = 1;
      if (lane == 0) have = mbar_wait(smem_u32(&bar_acc_full[b]), (w / NBUF) & 1, &abort_flag, P.err, 44) ? 1 : 0;
      have = __shfl_sync(0xffffffffu, have, 0);
      fence_after();
      if (!have) break;
#pragma unroll 1
      for (int pc = e >> 2; pc < C::PIECES; pc += 4) {
        const int col = (pc >> 1) * 16, c = c0 + col / BN;
        const int j0 = n0 + col % BN, r0 = m0 + quarter * 32 + (pc & 1) * 16;
        if (pc + 4 < C::PIECES && P.E.nout > 0) {  // the next piece's auxiliary values
          const int col1 = ((pc + 4) >> 1) * 16, j1 = n0 + col1 % BN;
          if (j1 < P.N && r0 < P.M) epi_prefetch(P.E, c0 + col1 / BN, r0, P.M, j1, P.N);
        }
        if (j0 >= P.N || r0 >= P.M) continue;  // the same for the whole warp
        uint32_t raw[8];
        float v[8];
        if (units > 0) {
          tmem_ld_16x16(tq + b * C::ACC + col + ((uint32_t)((pc & 1) * 16) << 16), raw);
          tmem_wait_ld();
        }
#pragma unroll
        for (int t = 0; t < 8; t++) v[t] = units > 0 ? __uint_as_float(raw[t]) : 0.f;
        if (P.plain64) {  // the product itself as FP64 planes
          store_piece(reinterpret_cast<double*>(P.E.out[0].mp) + c * P.E.out[0].mps, P.E.out[0].mld, r0, P.M, j0, P.N,
                      v);
        } else if (P.E.nout == 0) {
          store_piece(P.C.p + c * P.C.ps, P.C.ld, r0, P.M, j0, P.N, v);
        } else if (P.E.f64) {
          epi_piece<double>(P.E, c, r0, P.M, j0, P.N, v, stg, sdx, sx, bad);
        } else {
          epi_piece<float>(P.E, c, r0, P.M, j0, P.N, v, stg, sdx, sx, bad);
        }
      }
      // the accumulator is read: release it to the MMA warp
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bar_acc_empty[b]));
    }
    if (P.E.red.partials) {
      double d0 = sdx, d1 = sx, d2 = bad;
      for (int o = 16; o > 0; o >>= 1) {
        d0 += __shfl_xor_sync(0xffffffffu, d0, o);
        d1 += __shfl_xor_sync(0xffffffffu, d1, o);
        d2 += __shfl_xor_sync(0xffffffffu, d2, o);
      }
      if (lane == 0) {
        double* pp = P.E.red.partials + 3 * ((long)blockIdx.x * EPI_WARPS + e);
        pp[0] = d0;
        pp[1] = d1;
        pp[2] = d2;
      }
    }
  }

  fence_before();
  __syncthreads();
  if (P.E.red.partials) reduce_last_block<3>(P.E.red, (long)gridDim.x * EPI_WARPS, red_sh);
  if (warp == 1 && abort_flag) drain_mmas(smem_u32(&bar_drain));
  if (warp == 0 && lane == 0 && abort_flag) {
    for (int u = (issued > STAGES ? issued - STAGES : 0); u < issued; u++)
      drain_wait(smem_u32(&bar_full[u % STAGES]), (u / STAGES) & 1);
  }
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TMEM) : "memory");
  }
}

int sm_count() {
  static int nsm[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (!nsm[dev] && cudaDeviceGetAttribute(&nsm[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  return nsm[dev];
}

enum TcShape { SHAPE_FULL, SHAPE_PAIR, SHAPE_64, SHAPE_32 };  // BN x NC: 128 x 4, 128 x 2, 64 x 1, 32 x 1
constexpr int SHAPE_BN[4] = {128, 128, 64, 32}, SHAPE_NC[4] = {4, 2, 1, 1};

long shape_items(int sh, int M, int N) {
  return (long)((M + BM - 1) / BM) * ((N + SHAPE_BN[sh] - 1) / SHAPE_BN[sh]) * (4 / SHAPE_NC[sh]);
}

// Shape of a product (qpinv_options.tc_broad: 1 the 128-column shapes, 0 the
// 64-column one, -1 by the time of the busiest SM): a stage costs its MMAs or
// its operand bytes, whichever is longer (cycles per stage below), an item
// its stages, and the last item of an SM its epilogue (every item of the
// four-component shape, which has one accumulator).  Storing the product itself
// (FP32, or FP64 for the caller) is a short epilogue: with the combine pass's
// cost there, one-term products took the pair shape and its twice the operand
// bytes (4096^3 1.37 against 1.20 ms, 2048^3 211 against 188 us).  Measured where
// the line lies: 500 x 1000 x 500, 2 terms, 0.053 ms with 64 columns against
// 0.082 with the component pair; 1000^3, 3 terms, 0.150 (component pair) against
// 0.252 (four components) and 0.36 (64 columns); 1100^3, 1 term, 63 us (four
// components) against 66; 2048^3, 1 term, 188 against 207 and 435; 2200 x 300 x
// 2200 72 (component pair) against 101.
TcShape tc_shape(int broad, bool fused, bool f64, bool plain64, int M, int N, int units) {
  if (broad == 0) return SHAPE_64;
  if (broad == 1) return fused ? SHAPE_PAIR : SHAPE_FULL;
  const double stage[4] = {1950, 1100, 600, 450};
  const double tail[4] = {!fused || plain64 ? 12000. : f64 ? 60000. : 45000., f64 ? 24000. : 12000., 5000, 4000};
  const int nsm = std::max(1, sm_count());
  int best = SHAPE_PAIR;
  double tb = 1e300;
  for (int sh = SHAPE_FULL; sh <= SHAPE_32; sh++) {
    const double waves = (double)((shape_items(sh, M, N) + nsm - 1) / nsm);
    const double t = waves * units * stage[sh] + tail[sh] * (sh == SHAPE_FULL ? waves : 1.0) +
                     (waves - 1) * 1000.0;
    if (t < tb) {
      tb = t;
      best = sh;
    }
  }
  return (TcShape)best;
}

template <class C>
cudaError_t launch_cfg(const TcGemmArgs& a, KParams& P, cudaStream_t st) {
  CUtensorMap mA, mB;
  P.arows = a.M >= BM ? BM : (a.M + 7) / 8 * 8;  // whole 8-row swizzle groups
  if (!make_map(&mA, a.A->a, a.K, a.M, 4 * a.A->levels, a.A->lda, a.A->psa, P.arows, BK, 4))
    return cudaErrorInvalidValue;
  if (!make_map(&mB, a.B->b, a.K, a.N, 4 * a.B->levels, a.B->ldb, a.B->psb, C::BN, BK, 4))
    return cudaErrorInvalidValue;
  static std::atomic<unsigned long long> attr_done{0};
  if (cudaError_t e = ensure_smem_attr(k_qgemm_tc<C>, C::SMEM, attr_done)) return e;
  P.Mt = (a.M + BM - 1) / BM;
  P.Nt = (a.N + C::BN - 1) / C::BN;
  const long items = (long)P.Mt * P.Nt * (4 / C::NC);
  const int nsm = sm_count();
  if (nsm < 1 || items > 0x7fffffffL) return cudaErrorInvalidValue;
  P.items = (int)items;
  ++g_kernel_launches;
  return launch_pdl(k_qgemm_tc<C>, dim3((unsigned)std::min<long>(items, nsm)), dim3(THREADS), C::SMEM, st, mA, mB, P);
}

int units_of(const TcGemmArgs& a) { return ((a.k1 + BK - 1) / BK - a.k0 / BK) * a.npairs; }

}  // namespace

int tc_partial_blocks(const TcGemmArgs& a) {
  const TcShape sh = tc_shape(a.broad, true, a.epi.f64 != 0, false, a.M, a.N, units_of(a));
  return (int)std::min<long>(shape_items(sh, a.M, a.N), std::max(1, sm_count())) * EPI_WARPS;
}

bool tc_supported() {  // sm_103; attributes only (cudaGetDeviceProperties takes tens of microseconds)
  int dev = 0, major = 0, minor = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev) != cudaSuccess)
    return false;
  return major == 10 && minor == 3 && get_encode() != nullptr;
}

cudaError_t launch_qgemm_tc(const TcGemmArgs& a, cudaStream_t st) {
  if (a.M <= 0 || a.N <= 0) return cudaSuccess;
  if (a.npairs < 1 || a.npairs > 16 || !a.A || !a.B || !a.A->a || !a.B->b) return cudaErrorInvalidValue;
  if ((a.A->lda % 8) || (a.A->psa % 8) || (a.B->ldb % 8) || (a.B->psb % 8)) return cudaErrorInvalidValue;
  if ((a.k0 % BK) != 0 || (a.k1 != a.K && (a.k1 % BK) != 0) || a.k0 < 0 || a.k1 > a.K || a.k0 > a.k1)
    return cudaErrorInvalidValue;
  for (int p = 0; p < a.npairs; p++)
    if (a.pair_i[p] < 0 || a.pair_i[p] >= a.A->levels || a.pair_j[p] < 0 || a.pair_j[p] >= a.B->levels)
      return cudaErrorInvalidValue;
  KParams P;
  P.M = a.M;
  P.N = a.N;
  P.kb0 = a.k0 / BK;
  P.kb1 = (a.k1 + BK - 1) / BK;
  P.npairs = a.npairs;
  for (int p = 0; p < 16; p++) {
    P.pi[p] = p < a.npairs ? a.pair_i[p] : 0;
    P.pj[p] = p < a.npairs ? a.pair_j[p] : 0;
  }
  P.C = a.C;
  P.E = a.epi;
  if (P.E.nout < 0 || P.E.nout > kMaxOut || (P.E.f64 && P.E.red.partials)) return cudaErrorInvalidValue;
  const EpiOut& O = P.E.out[0];
  P.plain64 = P.E.f64 && P.E.nout == 1 && O.mp && !O.a && !O.b && O.cacc.kind == CK_ONE && O.diag.kind == CK_ZERO;
  for (int t = 0; t < kEpiAux; t++)
    if (P.E.aux[t] && O.caux[t].kind != CK_ZERO) P.plain64 = 0;
  P.err = a.err;
  switch (tc_shape(a.broad, P.E.nout > 0, P.E.f64 != 0, P.plain64 != 0, a.M, a.N, units_of(a))) {
    case SHAPE_FULL: return launch_cfg<Cfg<128, 4>>(a, P, st);
    case SHAPE_PAIR: return launch_cfg<Cfg<128, 2>>(a, P, st);
    case SHAPE_64: return launch_cfg<Cfg<64, 1>>(a, P, st);
    default: return launch_cfg<Cfg<32, 1>>(a, P, st);
  }
}

}  // namespace qp
