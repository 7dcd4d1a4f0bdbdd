// qgemm_emu.cu -- FP64-accurate quaternion GEMM from exact BF16 slices in ONE
// tensor-core launch, with eight real products per quaternion product.
//
// Operands are cut into S exact slices per entry (row / column power-of-two
// scaling, balanced 7-bit digits), so A B = sum over slice pairs (s, t) of
// A_s B_t, and level d = s + t carries the weight 2^-7(d+2).  Levels 0..S-1
// are formed.
//
// Hamilton product with eight multiplications (the rank of the quaternion
// algebra over the reals is 8; Howell and Lafon, 1975): with a = (w, x, y, z),
//   P0 = (w+x)(w'+x')   P1 = (z-y)(y'-z')   P2 = (w-x)(y'+z')  P3 = (y+z)(w'-x')
//   P4 = (x+z)(x'+y')   P5 = (x-z)(x'-y')   P6 = (w+y)(w'-z')  P7 = (w-y)(w'+z')
//   2w" = 2 P1 - P4 - P5 + P6 + P7      2x" = 2 P0 - P4 - P5 - P6 - P7
//   2y" = 2 P2 + P4 - P5 + P6 - P7      2z" = 2 P3 + P4 - P5 - P6 + P7
// In floating point the sums would cost accuracy; here every quantity is an
// exact integer, so the regrouping changes nothing: the slicing kernels store
// the digit sums of the eight combinations (at most 128 in modulus, 256 for
// the first slice: exact in BF16), each product is a plain real contraction,
// and the combine pass adds the eight 64-bit accumulators.  Half the tensor
// work of the 16-product form: 8-slice 2048^3 issues 18 passes of 32 K^3
// flops instead of 36.
//
// Work item: (tile of 128 x BN entries, product p, part).  The tensor core
// has one FP32 accumulator per level, and levels are taken in pairs (h, h-1),
// h = S-1, S-3, ...: slice A_s meets B_{h-s} (level h) and B_{h-1-s} (level
// h-1), and B_t meets A_{h-t} and A_{h-1-t}, so one new A tile and one new B
// tile per step s feed both levels; a single-level loop would load twice the
// bytes per MMA (it has no reuse left once each real product has its own
// operand planes).  Stage u of the TMA pipeline holds (A_s, B_{h-s}); the B
// tiles lie in descending address order, so B_{h-1-s} (the next stage) sits
// right below B_{h-s} and one MMA of 2 BN columns computes A_s [B_{h-1-s} |
// B_{h-s}] into the adjacent accumulators [level h-1 | level h]; only at the
// ring's wrap it takes two MMAs of BN columns.  The wide MMA also reads A
// once for both levels: 96 bytes of shared memory per cycle instead of 128.
//
// K is taken in chunks short enough that every FP32 partial sum is an exact
// integer (the term bound is 2^16 for digit pair (0, 0), 2^15 for (0, t) and
// (s, 0), else 2^14: K chunk <= 2^10 / (h + 3), 256 for h = 0); the lowest
// pair, whose rounding lies below the result's, runs in chunks of 1024.  Two
// TMEM buffers (2 BN columns each) alternate, so the 16 epilogue warps drain
// one chunk into 64-bit integers in registers while the MMA warp fills the
// other.  The running sum moves from the lowest pair's unit 2^-7(h+2) up to
// the result's unit 2^-F with one rounded shift per pair, and each item
// writes its accumulator plane once: no clearing and no read-modify-write.
//
// Parts: a product with too few tiles for the chip splits an item's level
// pairs and K range over up to 16 parts, each with its own set of planes
// (combined with the eight products, exactly).
//
// Measured (GB300): the 8-slice 2048^3 product 2.89 ms against 5.31 ms of the
// 16-product kernel it replaced (1710 TFLOP/s issued of 1957 measured burst),
// 4096^3 23.9-24.3 against 44.9 ms, 60 x 512 x 60 14 against 155 us.  What is left
// at 2048: 2048 items on 152 SMs fill 13.5 of 14 waves, and the MMA warp's
// barrier waits between stages.
#include <cuda.h>

#include <algorithm>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace qp {
namespace {

constexpr int EBM = 128, EBK = 64;                  // BK = one 128-byte swizzle row
constexpr int EA_TILE = EBM * EBK * 2;              // 16 KB
constexpr int EEPI_WARPS = 16;                      // four per TMEM lane quarter
constexpr int EEPI0 = 2;                            // warp 0 TMA, warp 1 MMA
constexpr int ETHREADS = 32 * (EEPI0 + EEPI_WARPS);
constexpr int EGROUP_M = 16;

template <int BN_>
struct ECfg {
  static constexpr int BN = BN_;
  static constexpr int B_TILE = BN * EBK * 2;
  static constexpr int STAGES = BN == 128 ? 6 : 8;
  static constexpr int SMEM = STAGES * (EA_TILE + B_TILE) + 1024;  // + alignment slack
  static constexpr int BUF = 2 * BN;          // TMEM columns of a buffer: [level h-1 | level h]
  static constexpr int CW = BN / 4;           // columns per epilogue warp and level
  static constexpr uint32_t IDESC1 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                                     ((uint32_t)(EBM >> 4) << 24);
  static constexpr uint32_t IDESC2 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(2 * BN >> 3) << 17) |
                                     ((uint32_t)(EBM >> 4) << 24);
  static_assert(SMEM <= 227 * 1024, "shared memory per CTA");
  static_assert(2 * BUF <= 512, "TMEM columns");
};

struct EParams {
  int M, N, K;
  int Mt, Nt, tiles, items;
  int nk, kspan;             // K ranges per item and their length (multiple of EBK)
  int ngroups;               // level groups
  int np[4], h[4][4];        // level pairs of each group (upper level h), lowest weight first
  int kc[4][4];              // their K chunks (multiples of EBK)
  int F;                     // accumulator unit 2^-F
  int p0, nprod;             // products p0 .. p0 + nprod - 1 (operand planes [slice][nprod])
  long long* C64;            // [part][product][M][ld64]
  long ld64, ps64;
  int* err;
};

struct EItem {
  int m0, n0, p, part, g, k0, k1;
};
// Items run part-major, then product, then tile (16 row tiles per raster
// group), so that the CTAs at work at one time share one product's operands.
template <int BN>
__device__ __forceinline__ EItem item_of(const EParams& P, int item) {
  EItem it;
  const int t = item % P.tiles, q = item / P.tiles;
  it.p = q % P.nprod;
  it.part = q / P.nprod;
  it.g = it.part / P.nk;
  it.k0 = (it.part % P.nk) * P.kspan;
  it.k1 = min(P.K, it.k0 + P.kspan);
  const int per_group = EGROUP_M * P.Nt, group = t / per_group, local = t % per_group;
  const int gm = min(EGROUP_M, P.Mt - group * EGROUP_M);
  it.m0 = (group * EGROUP_M + local % gm) * EBM;
  it.n0 = (local / gm) * BN;
  return it;
}

// nkk MMAs of K = 16 along one stage (32 bytes of the swizzle row each); the
// first accumulates if acc, the others always.
template <uint32_t IDESC>
__device__ __forceinline__ void mma_steps(uint32_t d, uint32_t ad, uint32_t bd, int nkk, uint32_t acc) {
  constexpr uint64_t hi = desc_hi(2 * EBK);
  if (nkk == EBK / 16) {
#pragma unroll
    for (int kk = 0; kk < EBK / 16; kk++)
      mma_bf16(d, hi | (ad + kk * 2), hi | (bd + kk * 2), IDESC, kk ? 1u : acc);
  } else {
#pragma unroll 1
    for (int kk = 0; kk < nkk; kk++) mma_bf16(d, hi | (ad + kk * 2), hi | (bd + kk * 2), IDESC, kk ? 1u : acc);
  }
}

template <int BN>
__global__ void __launch_bounds__(ETHREADS, 1)
    k_qgemm_emu(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                const __grid_constant__ EParams P) {
  using C = ECfg<BN>;
  constexpr int STAGES = C::STAGES, CW = C::CW;
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t bar_full[STAGES], bar_empty[STAGES], bar_acc_full[2], bar_acc_empty[2], bar_drain;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;

  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* smemB = smem + STAGES * EA_TILE;  // stage st at (STAGES - 1 - st) * B_TILE
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < STAGES; s++) {
      mbar_init(smem_u32(&bar_full[s]), 1);
      mbar_init(smem_u32(&bar_empty[s]), 1);
    }
    for (int b = 0; b < 2; b++) {
      mbar_init(smem_u32(&bar_acc_full[b]), 1);
      mbar_init(smem_u32(&bar_acc_empty[b]), EEPI_WARPS);
    }
    mbar_init(smem_u32(&bar_drain), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(2 * C::BUF)
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

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
      int u = 0, st = 0;
      uint32_t ph = 1;  // parity of bar_empty's previous phase: the first pass over the ring does not wait
      bool ok = true;
      for (int item = blockIdx.x; item < P.items && ok; item += gridDim.x) {
        const EItem it = item_of<BN>(P, item);
        for (int li = 0; li < P.np[it.g] && ok; li++) {
          const int h = P.h[it.g][li];
          for (int k = it.k0; k < it.k1 && ok; k += EBK) {
            for (int s = 0; s <= h; s++, u++) {
              if (u >= STAGES && !mbar_wait(smem_u32(&bar_empty[st]), ph, &abort_flag, P.err, 11)) {
                ok = false;
                break;
              }
              const uint32_t fb = smem_u32(&bar_full[st]);
              mbar_expect_tx(fb, EA_TILE + C::B_TILE);
              tma_load_3d(smem_u32(smem + st * EA_TILE), &tmA, k, it.m0, s * P.nprod + it.p, fb);
              tma_load_3d(smem_u32(smemB + (STAGES - 1 - st) * C::B_TILE), &tmB, k, it.n0, (h - s) * P.nprod + it.p, fb);
              issued = u + 1;
              if (++st == STAGES) {
                st = 0;
                ph ^= 1;
              }
            }
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    // The whole warp walks the loops and one elected lane issues (elect_one).
    const uint32_t a_lo = desc_lo(smem_u32(smem)), b_lo = desc_lo(smem_u32(smemB));
    int w = 0, st = 0;
    uint32_t ph = 0;  // parity of stage st's current fill
    for (int item = blockIdx.x; item < P.items; item += gridDim.x) {
      const EItem it = item_of<BN>(P, item);
      for (int li = 0; li < P.np[it.g]; li++) {
        const int h = P.h[it.g][li], kc = P.kc[it.g][li];
        for (int c0 = it.k0; c0 < it.k1; c0 += kc, w++) {
          const int b = w & 1, c1 = min(it.k1, c0 + kc);
          if (w >= 2) (void)mbar_wait(smem_u32(&bar_acc_empty[b]), ((w >> 1) - 1) & 1, &abort_flag, P.err, 12);
          fence_after();
          const uint32_t dlo = tmem + b * C::BUF, dhi = dlo + BN;
          for (int k = c0; k < c1; k += EBK) {
            const int nkk = min(EBK / 16, (c1 - k + 15) / 16);
            (void)mbar_wait(smem_u32(&bar_full[st]), ph, &abort_flag, P.err, 13);
            for (int s = 0; s <= h; s++) {
              const int sn = st + 1 == STAGES ? 0 : st + 1;
              const uint32_t phn = st + 1 == STAGES ? ph ^ 1 : ph;
              const uint32_t ad = a_lo + st * (EA_TILE >> 4);
              const uint32_t bh = b_lo + (STAGES - 1 - st) * (C::B_TILE >> 4);
              const uint32_t bl = b_lo + (STAGES - 1 - sn) * (C::B_TILE >> 4);
              const uint32_t acc = (k > c0 || s > 0) ? 1u : 0u;
              if (s < h) (void)mbar_wait(smem_u32(&bar_full[sn]), phn, &abort_flag, P.err, 13);
              fence_after();
              if (elect_one()) {
                if (s < h && sn != 0) mma_steps<C::IDESC2>(dlo, ad, bl, nkk, acc);
                else {
                  if (s < h) mma_steps<C::IDESC1>(dlo, ad, bl, nkk, acc);
                  mma_steps<C::IDESC1>(dhi, ad, bh, nkk, acc);
                }
                mma_commit(smem_u32(&bar_empty[st]));
              }
              __syncwarp();
              st = sn;
              ph = phn;
            }
          }
          if (elect_one()) mma_commit(smem_u32(&bar_acc_full[b]));
          __syncwarp();
        }
      }
      // here: at every chunk 2048^3 takes 2.94 ms for 2.92, at the item's start 2.97
      if (warp_aborted(&abort_flag)) break;
    }
  } else {
    // ---------------- epilogue: exact FP32 chunk sums -> 64-bit integers in registers ----------------
    // Warp e reads TMEM lane quarter warp % 4 (its 32 rows) and CW columns of
    // both levels of the pair.
    const int e = warp - EEPI0, quarter = warp & 3, col0 = (e >> 2) * CW;
    const uint32_t tb0 = tmem + ((uint32_t)(quarter * 32) << 16) + col0;
    int w = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < P.items && ok; item += gridDim.x) {
      const EItem it = item_of<BN>(P, item);
      long long acc[CW];
#pragma unroll
      for (int t = 0; t < CW; t++) acc[t] = 0;
      int T = 1 << 20;  // unit 2^-T of acc (empty at first)
      for (int li = 0; li < P.np[it.g] && ok; li++) {
        const int h = P.h[it.g][li], kc = P.kc[it.g][li];
        const int unit = 7 * (h + 2), Tn = max(unit, P.F), sh = Tn - unit;
        if (li > 0 && T > Tn) {  // up to this pair's unit, rounded
          const int d = T - Tn;
#pragma unroll
          for (int t = 0; t < CW; t++) acc[t] = (acc[t] + (1LL << (d - 1))) >> d;
        }
        T = Tn;
        for (int c0 = it.k0; c0 < it.k1 && ok; c0 += kc, w++) {
          const int b = w & 1;
          int have = 1;
          if (lane == 0) have = mbar_wait(smem_u32(&bar_acc_full[b]), (w >> 1) & 1, &abort_flag, P.err, 14) ? 1 : 0;
          have = __shfl_sync(0xffffffffu, have, 0);
          if (!have) {
            ok = false;
            break;
          }
          fence_after();
          const uint32_t tb = tb0 + b * C::BUF;
#pragma unroll
          for (int q = 0; q < CW; q += 8) {
            uint32_t lo[8], hi[8];
            tmem_ld8u(tb + BN + q, hi);
            if (h > 0) tmem_ld8u(tb + q, lo);
            tmem_wait_ld();
#pragma unroll
            for (int t = 0; t < 8; t++) {
              long long v = (long long)__float2int_rn(__uint_as_float(hi[t]));
              if (h > 0) v += (long long)__float2int_rn(__uint_as_float(lo[t])) * 128;
              acc[q + t] += v << sh;
            }
          }
          fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&bar_acc_empty[b]));
        }
      }
      if (!ok) break;
      if (T > P.F) {
        const int d = T - P.F;
#pragma unroll
        for (int t = 0; t < CW; t++) acc[t] = (acc[t] + (1LL << (d - 1))) >> d;
      }
      const int row = it.m0 + quarter * 32 + lane;
      if (row < P.M) {
        const int j0 = it.n0 + col0;
        long long* dst = P.C64 + (long)(it.part * 8 + P.p0 + it.p) * P.ps64 + (long)row * P.ld64 + j0;
#pragma unroll
        for (int t = 0; t < CW; t += 4)  // ld64 is a multiple of 4: whole groups only
          if (j0 + t < P.N) {
            reinterpret_cast<longlong2*>(dst + t)[0] = make_longlong2(acc[t], acc[t + 1]);
            reinterpret_cast<longlong2*>(dst + t)[1] = make_longlong2(acc[t + 2], acc[t + 3]);
          }
      }
    }
  }

  fence_before();
  __syncthreads();
  if (warp == 1 && abort_flag) drain_mmas(smem_u32(&bar_drain));
  if (warp == 0 && lane == 0 && abort_flag) {
    for (int u = (issued > STAGES ? issued - STAGES : 0); u < issued; u++)
      drain_wait(smem_u32(&bar_full[u % STAGES]), (u / STAGES) & 1);
  }
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * C::BUF) : "memory");
  }
}

int emu_sm_count() {
  static int nsm[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (!nsm[dev] && cudaDeviceGetAttribute(&nsm[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  return nsm[dev];
}

template <int BN>
cudaError_t launch_bn(const EmuGemmArgs& a, EParams& P, int nsm, cudaStream_t st) {
  using C = ECfg<BN>;
  CUtensorMap mA, mB;
  if (!make_map(&mA, a.A->a, a.K, a.M, a.np * a.S, a.A->lda, a.A->psa, EBM, EBK)) return cudaErrorInvalidValue;
  if (!make_map(&mB, a.B->b, a.K, a.N, a.np * a.S, a.B->ldb, a.B->psb, BN, EBK)) return cudaErrorInvalidValue;
  static std::atomic<unsigned long long> attr_done{0};
  if (cudaError_t e = ensure_smem_attr(k_qgemm_emu<BN>, C::SMEM, attr_done)) return e;
  ++g_kernel_launches;
  return launch_pdl(k_qgemm_emu<BN>, dim3((unsigned)std::min(P.items, nsm)), dim3(ETHREADS), C::SMEM, st, mA, mB, P);
}

}  // namespace

EmuPlan emu_plan(int M, int N, int K, int S) {
  EmuPlan p;
  int lg = 0;
  while ((1L << lg) < 4L * K) lg++;
  // A product is at most 4K in normalised units: |acc| <= 2^62.  The combine pass
  // forms twice a component, which has to stay below 2^63, a component below 4K:
  // sliced entries are below 1 by at least 2^-7S (2^-53 where 8 slices hold an FP64
  // mantissa), so twice a component leaves 2^11 units or more for the roundings (a
  // few hundred) and for what the dropped levels would have subtracted.
  p.F = 62 - lg;
  const int npairs = (S + 1) / 2;
  const int nsm = std::max(1, emu_sm_count());
  // Tile width and parts by the time of the busiest SM, in units of one
  // 128 x 128 x 64 MMA step (256 cycles): an item costs its level pairs'
  // steps over its K range (a 64-column step about 0.55 of a 128-column one)
  // plus a fixed 12 for filling the pipeline, draining the last chunk and
  // storing; the accumulator planes of further parts are written and read
  // again by the combine pass.  With at least two waves of 128-column items
  // the plain form wins; below that the splits spread one product over the
  // chip (a 60 x 60 x 512 product is 8 items otherwise).
  double best = 1e300;
  for (int bn = 128; bn >= 64; bn -= 64) {
    const long tiles = (long)((M + EBM - 1) / EBM) * ((N + bn - 1) / bn);
    if (tiles > 0x7fffffffL / 128) continue;
    for (int ng = 1; ng <= npairs; ng <<= 1) {
      for (int nk = 1; nk <= 4; nk <<= 1) {
        if (nk > 1 && K < 128 * nk) break;
        const int kspan = (((K + nk - 1) / nk + EBK - 1) / EBK) * EBK;
        double cost[4] = {0, 0, 0, 0}, sum = 0, cmax = 0, cmin = 1e300;
        int load[4] = {0, 0, 0, 0};
        for (int q = 0, h = S - 1; h >= 0; h -= 2, q++) {
          int g = 0;
          for (int x = 1; x < ng; x++)
            if (load[x] < load[g]) g = x;
          load[g] += 2 * h + 1;
        }
        for (int g = 0; g < ng; g++) {
          cost[g] = load[g] * ((kspan + EBK - 1) / EBK) * (bn == 128 ? 1.0 : 0.55) + 12.0;
          sum += cost[g] * nk * 8.0 * tiles;
          cmax = std::max(cmax, cost[g]);
          cmin = std::min(cmin, cost[g]);
        }
        const double items = 8.0 * tiles * ng * nk;
        double t = ng == 1 ? std::ceil(items / nsm) * cmax : std::max(cmax, sum / nsm + 0.5 * cmin);
        // each further part: 64 bytes written and read per entry at about 5 TB/s,
        // and one more dependent load in the combine pass
        t += 3.0 * (ng * nk - 1);
        t += 128.0 * M * (double)N * ng * nk / 5e12 / (256 / 1.9e9);
        if (t < best * 0.97) {
          best = t;
          p.bn = bn;
          p.ngroups = ng;
          p.nk = nk;
        }
      }
    }
  }
  p.nparts = p.ngroups * p.nk;
  return p;
}

cudaError_t launch_qgemm_emu(const EmuGemmArgs& a, const EmuPlan& plan, cudaStream_t st) {
  if (a.M <= 0 || a.N <= 0 || a.K <= 0) return cudaSuccess;
  if (!a.A || !a.B || !a.A->a || !a.B->b || !a.C64 || a.S < 1 || a.S > 8) return cudaErrorInvalidValue;
  if (a.A->levels < a.S || a.B->levels < a.S) return cudaErrorInvalidValue;
  if ((a.A->lda % 8) || (a.A->psa % 8) || (a.B->ldb % 8) || (a.B->psb % 8) || (a.ld64 % 4) || (a.ps64 % 4) ||
      (reinterpret_cast<uintptr_t>(a.C64) & 15) || a.ld64 < a.N)
    return cudaErrorInvalidValue;
  if (a.p0 < 0 || a.np < 1 || a.p0 + a.np > 8) return cudaErrorInvalidValue;
  if ((plan.bn != 64 && plan.bn != 128) || plan.ngroups < 1 || plan.ngroups > 4 || plan.nk < 1)
    return cudaErrorInvalidValue;
  const int nsm = emu_sm_count();
  if (nsm < 1) return cudaErrorInvalidValue;
  EParams P;
  P.M = a.M;
  P.N = a.N;
  P.K = a.K;
  P.Mt = (a.M + EBM - 1) / EBM;
  P.Nt = (a.N + plan.bn - 1) / plan.bn;
  P.tiles = P.Mt * P.Nt;
  P.nk = plan.nk;
  P.kspan = (((a.K + plan.nk - 1) / plan.nk + EBK - 1) / EBK) * EBK;
  P.ngroups = plan.ngroups;
  int load[4] = {0, 0, 0, 0};
  for (int g = 0; g < 4; g++) P.np[g] = 0;
  for (int h = a.S - 1; h >= 0; h -= 2) {  // largest pair first, each to the lightest group
    int g = 0;
    for (int x = 1; x < plan.ngroups; x++)
      if (load[x] < load[g]) g = x;
    const int lim = h == a.S - 1 ? 1024 : h == 0 ? 256 : 1024 / (h + 3);
    P.h[g][P.np[g]] = h;
    P.kc[g][P.np[g]++] = std::max(EBK, lim / EBK * EBK);
    load[g] += 2 * h + 1;
  }
  P.F = plan.F;
  P.p0 = a.p0;
  P.nprod = a.np;
  P.items = P.tiles * a.np * plan.ngroups * plan.nk;
  P.C64 = a.C64;
  P.ld64 = a.ld64;
  P.ps64 = a.ps64;
  P.err = a.err;
  return plan.bn == 128 ? launch_bn<128>(a, P, nsm, st) : launch_bn<64>(a, P, nsm, st);
}

}  // namespace qp
