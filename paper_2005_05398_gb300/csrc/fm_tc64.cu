// Float64 mode products of the preconditioner on the tensor cores (Eq. prec-2, precision FM_PREC_FP64).
//
// The float64 z and x stages are batched GEMMs out = W^l . slab.  On GB300 the FP64 pipe gives 1.2 TFLOP/s, so
// the float64 CUDA-core kernels (k_zmix, k_mix) spend 0.70 + 2.4 ms on them per application at 3.7 M unknowns
// (He L=0, 96 x 96 x 24 intervals).  Here both operands are split into integer digits whose products the tensor
// cores add exactly (Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012; Mukunoki et al., ISC 2020):
//   * a row of W and a column of the slab are scaled by a power of two (its largest entry) to integers of 62 bits
//     (K <= 64) or 59 bits, seven balanced base-512 digits d_0 .. d_6 in [-256, 256], each exact in float16;
//   * the 34 products with i + j <= 7 run as tcgen05.mma kind::f16, those of one weight g = i + j into one
//     float32 accumulator D_g (8 accumulators in tensor memory).  A float32 sum of integers is exact up to 2^24:
//     |D_g| <= (g + 1) K 2^16 for K <= 64, so D_0 .. D_3 are; above, |d_0| <= 32 keeps D_0 and D_1 exact for any
//     input, and the split of W checks D_2 and D_3 from the digit sums of its rows (K > 192: each half of K has
//     accumulators of its own).  Beyond 2^24 a rounding of D_4 .. D_7 costs 2^-43 of the row's and column's maxima or
//     less; it takes slab digits that follow the signs of hundreds of digits of W (sums are about 2^19 otherwise);
//   * the epilogue adds sum_g 2^(9 (7 - g)) D_g as a fixed-point integer and rounds once to float64, in integer
//     arithmetic (the FP64 pipe is not touched).
// The columns of W_z are scaled to g_l^{M'}(1) and span up to 1e8 while the modes they meet are damped at high l: on
// the scale of the column's largest mode the products that matter would be cut off (base 256 without balance lost
// 1e-14 .. 6e-10 there).  The z inverse therefore takes column k of W_z by 2^-a_k and mode k of the slab by 2^a_k, a_k
// the exponent of that column's maximum: an integer add per value.
// Accuracy, against 64-bit-mantissa sums of the solver's own matrices, over both bases, J <= 10, n_z = 8 .. 130,
// n_x = 48 .. 256, with random and with smooth vectors taken through the chain (relative 2-norm per M' component):
// z stages 3e-17 .. 9e-17 where the float64 chain has 5e-17 .. 1.7e-15 (K > 64: up to 2e-15 against 8e-15), x
// stages 3e-17 .. 6e-16 against 1e-16 .. 1.6e-15.  The bound is normwise: an entry far below its column's largest
// product carries that product's last bits.  A column with an infinity, a NaN or a maximum outside 2^+-677 takes a
// float64 loop over the original values instead.
//
// One CTA per SM walks (slab, column tile) pairs: 16 worker warps load the tile's doubles (the next tile's are in
// flight during the MMAs), split them into K-major 128-byte-swizzled operands that stay for every row tile, and
// run the epilogue; one warp streams the digits of W by TMA, one issues the MMAs.  Two forms:
//   * K <= 64 (the z stages, small grids): A = 128 columns of the slab, B = the rows of W with all digits
//     resident, so that every tensor-memory lane holds a column and W is read once per mode.  (With W as the
//     128-row operand 50 of 128 rows were used and a z stage took 90 us instead of 32.)
//   * otherwise A = 128 rows of W streamed through a ring, B = NT columns of the slab: NT = 64 fills the tensor
//     memory (8 x 64 columns); K > 192 takes NT = 32 so that the digits fit in shared memory.
// Bound: the MMAs' shared-memory operands (6 KB per 128 x 64 x 16, 48 cycles to read for 32 of the tensor pipe, which
// ncu shows active for 26 % of the cycles at K = 192 and 15 % at K = 50) and the integer work of split and epilogue.
// Measured per stage, both components of He L = 0: K = 192, 100 slabs of 192 columns 104 us forward and 112 us inverse
// (k_mix 1.2 ms); K = 50, two of 36,864 columns 60 us (k_zmix 350 us).  Every wait is bounded; a wait
// that expires sets the context's wait flag and leaves NaN in what the CTA had to write.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "fm_internal.h"
#include "fm_tc.h"

namespace fmi {

namespace {

constexpr int kDig = 7;             // base-512 digits per value
constexpr int kAcc = 8;             // accumulators: weights g = i + j = 0 .. 7
constexpr int kWorkers = 512;       // load / split / epilogue threads
constexpr int kProducer = kWorkers / 32, kIssuer = kProducer + 1;  // warps
constexpr int kF64Threads = kWorkers + 64;
constexpr uint32_t kBlockA = 128 * 128;  // one A block: 128 rows x 64 float16

struct F64Comp {
  CUtensorMap tmA;         // digits of W: [nl * 7][rows][ld], box 64 x 128
  const double* W;         // [nl][M][M]
  const int* expA;         // [nl][M] biased exponent of the row maximum
  const int* bal;          // z inverse: [nl][M] exponents a_k the slab's values are raised by (<< 20), else null
  const double* in;
  double* out;
  int K, N;                // contraction length (= rows of W), columns
  int slabs, nz;           // slabs and z modes (l - M0 = slab / nz + slab % nz); nz = 0: l = slab
  int64_t in_slab, out_slab;
  int64_t sk, sn;          // element (k, n) of a slab at k sk + n sn (one of them 1)
  int64_t om, on;          // out element (m, n) at m om + n on (one of them 1)
  int ntile;               // column tiles
};

struct F64Args {
  F64Comp c[3];
  int ncomp, total;
  int kblocks;             // 64-element K blocks of the B region (largest component)
  int stages;
  int* err;
};

// four accumulator columns of this warp's 32 lanes (no wait)
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// named barrier whose threads all learn whether one of them came with 'v'
__device__ __forceinline__ bool named_sync_or(int id, int nthreads, bool v) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %3, 0;\n barrier.cta.red.or.pred q, %1, %2, p;\n selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"(id), "r"(nthreads), "r"((uint32_t)v)
      : "memory");
  return r != 0;
}

// bits of a value of 1 on the integers' scale: 62-bit integers for K <= 64, 59-bit ones (|d_0| <= 32) otherwise
constexpr int kBitsSmall = 61, kBitsLarge = 58;

// The integer of a double on the scale of a maximum with biased exponent 'emax' (2^(bits + 1023 - emax) times the
// value, rounded to nearest), plus 256 in every digit: bits 9 (6 - i) .. + 8 of the result (d_0: ten bits), less
// 256, are digit d_i.
__device__ __forceinline__ uint64_t digits_of(double v, int emax, int bits) {
  const uint64_t b = (uint64_t)__double_as_longlong(v);
  const int e = (int)((b >> 52) & 0x7FF);
  uint64_t m = (b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  const int sh = emax - (bits - 52) - e;
  if (e == 0 || sh > 54) m = 0;  // zero, denormal or below half a unit
  else if (sh <= 0) m <<= -sh;
  else m = (m + (1ull << (sh - 1))) >> sh;
  if ((int64_t)b < 0) m = 0ull - m;
  return m + 0x4020100804020100ull;
}

// The same for the slab's values (high and low word), truncated toward zero, in 32-bit words with few ALU
// instructions (that pipe bounds the splitting).  The error is below one unit, 2^-bits of the column's maximum.
// emax of an all-zero column must be large.
template <int BITS>
__device__ __forceinline__ void digits32(uint32_t bh, uint32_t bl, uint32_t emax, uint32_t& lo, uint32_t& hi) {
  const uint32_t mh = __funnelshift_l(bl, (bh & 0xFFFFFu) | 0x100000u, BITS - 52), ml = bl << (BITS - 52);
  const uint32_t sh = emax - ((bh >> 20) & 0x7FFu);  // >= 0; an exponent of 0 shifts everything out
  const uint32_t t = (uint32_t)max((int)sh - 32, 0);
  uint32_t l = __funnelshift_rc(ml, mh, sh), h;
  asm("shr.u32 %0, %1, %2;" : "=r"(l) : "r"(l), "r"(t));   // (PTX shifts clamp at 32)
  asm("shr.u32 %0, %1, %2;" : "=r"(h) : "r"(mh), "r"(sh));
  const uint32_t sg = (uint32_t)((int)bh >> 31);
  asm("add.cc.u32 %0, %2, %4;\n addc.u32 %1, %3, 0x40201008;\n"
      : "=r"(lo), "=r"(hi)
      : "r"(l ^ sg), "r"(h ^ sg), "r"(0x04020100u - sg));
}

// the high word of a slab value raised by 2^(sa >> 20) (sa >= 0); what leaves the range becomes an infinity, so that
// the column takes the float64 loop; zeros and denormals stay
__device__ __forceinline__ uint32_t raise(uint32_t bh, uint32_t sa) {
  const uint32_t h = bh & 0x7FFFFFFFu;
  const uint32_t t = h < 0x100000u ? h : min(h + sa, 0x7FF00000u);
  return t | (bh & 0x80000000u);
}

// The digit in bits S .. of the 16-bit half words PRM selects from the words of two consecutive k -> two float16
// digits: 1024 + field by bit pattern, less 1280.
template <uint32_t PRM, int S, uint32_t MASK = 0x01FF01FFu>
__device__ __forceinline__ uint32_t digit_pair(uint32_t a, uint32_t b) {
  uint32_t w = ((__byte_perm(a, b, PRM) >> S) & MASK) | 0x64006400u;
  asm("sub.f16x2 %0, %1, %2;" : "=r"(w) : "r"(w), "r"(0x65006500u));
  return w;
}
template <uint32_t PRM, int S, uint32_t MASK = 0x01FF01FFu>
__device__ __forceinline__ void store_digit(uint32_t addr, const uint32_t (&g)[8]) {
  st_shared_v4(addr, digit_pair<PRM, S, MASK>(g[0], g[1]), digit_pair<PRM, S, MASK>(g[2], g[3]),
               digit_pair<PRM, S, MASK>(g[4], g[5]), digit_pair<PRM, S, MASK>(g[6], g[7]));
}

// sum_g 2^(9 (12 - g)) D_g 2^(ea + ec - 2046 - 2 bits) rounded to a double, expo = (ea + ec - 879 - 2 bits) << 20: a
// 96-bit fixed-point sum (w2:w1:w0, in sixteenths of D_6) in integers, no FP64.  v: D_0 .. D_4, 16 (D_5 + ...)
__device__ __forceinline__ double combine(const int (&v)[6], int expo) {
  const int64_t mid = (int64_t)v[3] * (1ll << 31) + (int64_t)v[4] * (1 << 22) + (int64_t)v[5] * (1 << 9);
  const int64_t top = (int64_t)v[0] * (1 << 26) + (int64_t)v[1] * (1 << 17) + (int64_t)v[2] * 256 + (mid >> 32);
  uint32_t w0 = (uint32_t)mid, w1 = (uint32_t)top, w2 = (uint32_t)(top >> 32);
  const uint32_t s = (uint32_t)((int)w2 >> 31);
  asm("add.cc.u32 %0, %3, %6;\n addc.cc.u32 %1, %4, 0;\n addc.u32 %2, %5, 0;\n"
      : "=r"(w0), "=r"(w1), "=r"(w2)
      : "r"(w0 ^ s), "r"(w1 ^ s), "r"(w2 ^ s), "r"(s & 1u));
  if (w2 == 0) {  // the sum's leading words are zero
    w2 = w1;
    w1 = w0;
    w0 = 0;
    expo -= 32 << 20;
    if (w2 == 0) {
      w2 = w1;
      w1 = 0;
      expo -= 32 << 20;
      if (w2 == 0) return 0.0;
    }
  }
  const int lz = __clz((int)w2);
  const uint32_t nh = __funnelshift_l(w1, w2, lz), nl = __funnelshift_l(w0, w1, lz);
  uint32_t rl, rh;  // the top 53 bits, rounded (a carry raises the exponent)
  asm("add.cc.u32 %0, %2, %4;\n addc.u32 %1, %3, %5;\n"
      : "=r"(rl), "=r"(rh)
      : "r"(__funnelshift_r(nl, nh, 11)), "r"(nh >> 11), "r"((nl >> 10) & 1u), "r"((uint32_t)(expo - lz * (1 << 20))));
  return __hiloint2double((int)(rh | (s & 0x80000000u)), (int)rl);
}

// D_0 .. D_4 as integers, D_5 + D_6 / 512 + D_7 / 512^2 in sixteenths (float32: its rounding is 2^-57 of the row's and
// column's maxima; float to integer conversions run on the narrow XU pipe: six of them instead of eight)
__device__ __forceinline__ void sums_of(const uint32_t (&d)[kAcc][4], int e, int (&v)[6]) {
#pragma unroll
  for (int g = 0; g < 5; ++g) v[g] = __float2int_rn(__uint_as_float(d[g][e]));
  v[5] = __float2int_rn(fmaf(fmaf(__uint_as_float(d[7][e]), 0.001953125f, __uint_as_float(d[6][e])), 0.03125f,
                             __uint_as_float(d[5][e]) * 16.f));
}

// kind::f16 with float16 A and B, float32 accumulation, M = 128, N = n
__host__ __device__ constexpr uint32_t f16_idesc(int n) { return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24); }

// low word of sw128_desc (the high word is the same for every tile)
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr) { return ((addr & 0x3FFFFu) >> 4) | (1u << 16); }
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);

// one MMA from descriptor low words; acc = 0 overwrites the accumulator
__device__ __forceinline__ void mma_lo(uint32_t d, uint32_t alo, uint32_t blo, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 da, db;\n setp.ne.b32 p, %5, 0;\n"
      " mov.b64 da, {%1, %4};\n mov.b64 db, {%2, %4};\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n}\n" ::"r"(d),
      "r"(alo), "r"(blo), "r"(idesc), "r"(kDescHi), "r"(acc)
      : "memory");
}

// The MMAs of digit I of the one operand (descriptor 'flo') with the digits j <= 7 - I of the other ('rlo' for
// j = 0, 'step' apart) over the ks steps of one K block, for the elected lane; neighbours go to different
// accumulators.  FIXED_A: the fixed digit is operand A.  'first': the block starts the accumulators it is the
// first to touch.
template <int I, int N, bool FIXED_A>
__device__ __forceinline__ void issue_digit(uint32_t tmem, uint32_t flo, uint32_t rlo, uint32_t step, uint32_t id, int ks,
                                            bool first) {
  constexpr int NJ = kAcc - I < kDig ? kAcc - I : kDig;
  uint32_t acc = first ? 0u : 1u;
#pragma unroll 1
  for (int kk = 0; kk < ks; ++kk) {
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const uint32_t d = tmem + (uint32_t)((I + j) * N), r = rlo + (uint32_t)j * step;
      const uint32_t ac = (I == 0 || (I == 1 && j == kDig - 1)) ? acc : 1u;
      mma_lo(d, FIXED_A ? flo : r, FIXED_A ? r : flo, id, ac);
    }
    acc = 1u;
    flo += 2;
    rlo += 2;
  }
}
template <int N, bool FIXED_A>
__device__ __forceinline__ void issue_item(int i, uint32_t tmem, uint32_t flo, uint32_t rlo, uint32_t step, uint32_t id,
                                           int ks, bool first) {
  switch (i) {
    case 0: issue_digit<0, N, FIXED_A>(tmem, flo, rlo, step, id, ks, first); break;
    case 1: issue_digit<1, N, FIXED_A>(tmem, flo, rlo, step, id, ks, first); break;
    case 2: issue_digit<2, N, FIXED_A>(tmem, flo, rlo, step, id, ks, first); break;
    case 3: issue_digit<3, N, FIXED_A>(tmem, flo, rlo, step, id, ks, first); break;
    case 4: issue_digit<4, N, FIXED_A>(tmem, flo, rlo, step, id, ks, first); break;
    case 5: issue_digit<5, N, FIXED_A>(tmem, flo, rlo, step, id, ks, first); break;
    default: issue_digit<6, N, FIXED_A>(tmem, flo, rlo, step, id, ks, first); break;
  }
}

// SMALL (K <= 64): A = 128 columns of the slab (their digits in shared memory), B = the rows of W (all seven
// digits resident, reloaded when the mode l changes), D[column][row of W].
// Otherwise: A = 128 rows of W (streamed), B = NT columns of the slab, D[row of W][column].
template <int NT, bool SMALL>
__global__ void __launch_bounds__(kF64Threads, 1) k_tc_f64(const __grid_constant__ F64Args a) {
  constexpr int kRows = SMALL ? 128 : NT;          // slab columns of a tile
  constexpr int kN = SMALL ? 64 : NT;              // MMA N
  constexpr int kHalf = 2;                         // NT = 32: K blocks from here on use the second accumulators
  constexpr int kCols = kAcc * kN * (kN == 32 ? 2 : 1);  // tensor-memory columns: 512
  constexpr int kBits = SMALL ? kBitsSmall : kBitsLarge;
  constexpr int kOct = SMALL ? 2 : 3;              // octets of eight doubles a worker holds per tile
  constexpr uint32_t kWItem = SMALL ? 64 * 128 : kBlockA;  // bytes of one TMA item of W
  extern __shared__ unsigned char t64_smem[];
  const uint32_t raw = smem_u32(t64_smem);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* gbase = t64_smem + (base - raw);
  const uint32_t tileX = (uint32_t)kRows * 128u;                  // one digit of the slab, one K block
  const uint32_t digX = (uint32_t)a.kblocks * tileX;              // one digit
  const uint32_t sW = base + kDig * digX;
  const uint32_t sExp = sW + (uint32_t)a.stages * kWItem;  // largest |high word| [2][kRows]
  const uint32_t bars = sExp + 2u * kRows * 4u;
  const uint32_t full0 = bars, empty0 = bars + 64, bready = bars + 128, dfull = bars + 136, dfree = bars + 144,
                 mfin = bars + 152, slot = bars + 160;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(gbase + (bars - base) + 168);
  volatile int* n_items = reinterpret_cast<volatile int*>(gbase + (bars - base) + 172);
  int* s_max = reinterpret_cast<int*>(gbase + (sExp - base));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
  if (tid == 0) {
    for (int s = 0; s < a.stages; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(bready, kWorkers);
    mbar_init(dfull, 1);
    mbar_init(dfree, kWorkers);
    mbar_init(mfin, 1);
    *abort_flag = 0;
    *n_items = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kProducer) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(kCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid < 2 * kRows) s_max[tid] = 0;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(gbase + (slot - base));
  auto locate = [&](int q, int* ci, int* slab, int* n0) {
    int cq = 0;
    while (cq + 1 < a.ncomp && q >= a.c[cq].slabs * a.c[cq].ntile) {
      q -= a.c[cq].slabs * a.c[cq].ntile;
      ++cq;
    }
    *ci = cq;
    *slab = q / a.c[cq].ntile;
    *n0 = (q - *slab * a.c[cq].ntile) * kRows;
  };
  auto mode_of = [](const F64Comp& cp, int slab) { return cp.nz ? slab / cp.nz + slab % cp.nz : slab; };

  if (warp == kProducer) {
    if (lane == 0) {  // TMA producer: blocks of W in the order (row tile, K block, digit); SMALL: the digits, per mode
      int it = 0, cur = -1;
      for (int q = blockIdx.x; q < a.total && !*abort_flag; q += gridDim.x) {
        int ci, slab, n0;
        locate(q, &ci, &slab, &n0);
        const F64Comp& cp = a.c[ci];
        const int l = mode_of(cp, slab);
        if (SMALL && ci * 65536 + l == cur) continue;  // resident
        cur = ci * 65536 + l;
        const int mt = SMALL ? 1 : (cp.K + 127) / 128, kbs = SMALL ? 1 : (cp.K + 63) / 64;
        for (int m = 0; m < mt && !*abort_flag; ++m)
          for (int kb = 0; kb < kbs && !*abort_flag; ++kb)
            for (int i = 0; i < kDig; ++i, ++it) {
              const int s = it % a.stages;
              if (it >= a.stages && !mbar_wait(empty0 + 8 * s, ((uint32_t)(it / a.stages) & 1u) ^ 1u)) {
                *abort_flag = 1;
                break;
              }
              mbar_expect_tx(full0 + 8 * s, kWItem);
              tma_load_3d(sW + s * kWItem, &cp.tmA, kb * 64, m * 128, l * kDig + i, full0 + 8 * s);
              *n_items = it + 1;
            }
      }
    }
  } else if (warp == kIssuer) {
    // MMA issuer.  The elected lane issues each item's MMAs from straight code with constant offsets: 72 cycles
    // per 128 x 64 x 16 MMA (48 are the reads of its operands from shared memory); with a runtime loop over the
    // digits and 64-bit descriptor arithmetic the issue itself took 105.
    if (elect_one()) {
      int it = 0, si = 0, gc = 0, cur = -1, loads = 0;
      bool ok = true;
      const uint32_t id = f16_idesc(kN);
      for (int q = blockIdx.x; q < a.total && ok; q += gridDim.x, ++si) {
        int ci, slab, n0;
        locate(q, &ci, &slab, &n0);
        const F64Comp& cp = a.c[ci];
        const int K = cp.K;
        ok = mbar_wait(bready, (uint32_t)si & 1u);
        if (SMALL) {
          const int tag = ci * 65536 + mode_of(cp, slab);
          // the digits of this mode (seven items: item i of load n is number 7 n + i, stage i)
          const bool fresh = tag != cur;
          if (fresh) {
            cur = tag;
            ++loads;
          }
          if (ok && gc > 0) ok = mbar_wait(dfree, (uint32_t)(gc - 1) & 1u);
          if (*abort_flag) ok = false;
          if (!ok) break;
          tc_fence_after();
          const int ks = (K + 15) / 16;
          for (int j = 0; j < kDig && ok; ++j) {  // digit j of W against the digits of the slab it pairs with
            if (fresh) ok = mbar_wait(full0 + 8 * j, (uint32_t)(loads - 1) & 1u);
            if (!ok) break;
            tc_fence_after();
            const uint32_t blo = desc_lo(sW + j * kWItem);
            issue_item<kN, false>(j, tmem, blo, desc_lo(base), digX >> 4, id, ks, j < 2);
          }
          // the digits of W may be overwritten once these MMAs have completed, when the next tile needs others
          const int qn = q + (int)gridDim.x;
          bool next_fresh = false;
          if (qn < a.total) {
            int cn, sn, nn;
            locate(qn, &cn, &sn, &nn);
            next_fresh = cn * 65536 + mode_of(a.c[cn], sn) != cur;
          }
          if (ok && next_fresh)
            for (int j = 0; j < kDig; ++j) mma_commit(empty0 + 8 * j);
          if (ok) mma_commit(dfull);
          ++gc;
        } else {
          const int mt = (K + 127) / 128, kbs = (K + 63) / 64;
          for (int m = 0; m < mt && ok; ++m, ++gc) {
            if (gc > 0) ok = ok && mbar_wait(dfree, (uint32_t)(gc - 1) & 1u);
            if (*abort_flag) ok = false;
            if (!ok) break;
            tc_fence_after();
            for (int kb = 0; kb < kbs && ok; ++kb) {
              const int ks = min(4, (K - kb * 64 + 15) / 16);
              for (int i = 0; i < kDig; ++i, ++it) {
                const int s = it % a.stages;
                if (!mbar_wait(full0 + 8 * s, (uint32_t)(it / a.stages) & 1u)) {
                  ok = false;
                  break;
                }
                tc_fence_after();
                const uint32_t alo = desc_lo(sW + s * kWItem);
                const uint32_t blo = desc_lo(base) + (((uint32_t)kb * tileX) >> 4);
                const bool second = kN == 32 && kb >= kHalf;
                issue_item<kN, true>(i, tmem + (second ? kAcc * kN : 0), alo, blo, digX >> 4, id, ks,
                                     (kb == 0 || (kN == 32 && kb == kHalf)) && i < 2);
                mma_commit(empty0 + 8 * s);
              }
            }
            if (ok) mma_commit(dfull);
          }
        }
      }
      if (!ok) *abort_flag = 1;
      mma_commit(mfin);  // arrives once every MMA issued above has completed
    }
    __syncwarp();
  } else {  // workers
    double v[kOct][8];
    auto load_tile = [&](int q) {
      int ci, slab, n0;
      locate(q, &ci, &slab, &n0);
      const F64Comp& cp = a.c[ci];
      const double* src = cp.in + (int64_t)slab * cp.in_slab;
      const int octs = ((cp.K + 63) / 64) * 8 * kRows;
#pragma unroll
      for (int o = 0; o < kOct; ++o) {
        const int idx = o * kWorkers + tid;
        const int n = n0 + idx % kRows, k0 = (idx / kRows) * 8;
        const bool ok = idx < octs && n < cp.N;
        const double* p = src + (int64_t)n * cp.sn + (int64_t)k0 * cp.sk;
#pragma unroll
        for (int e = 0; e < 8; ++e) v[o][e] = (ok && k0 + e < cp.K) ? p[(int64_t)e * cp.sk] : 0.0;
      }
    };
    int si = 0, gc = 0;
    if ((int)blockIdx.x < a.total) load_tile(blockIdx.x);
    for (int q = blockIdx.x; q < a.total; q += gridDim.x, ++si) {
      int ci, slab, n0;
      locate(q, &ci, &slab, &n0);
      const F64Comp& cp = a.c[ci];
      const int octs = ((cp.K + 63) / 64) * 8 * kRows, l = mode_of(cp, slab);
      int* cmax = s_max + (si & 1) * kRows;  // high word of each column's largest magnitude (0: all zero)
      if (tid < kRows) s_max[((si + 1) & 1) * kRows + tid] = 0;  // the other buffer, for the next tile
#pragma unroll
      for (int o = 0; o < kOct; ++o) {
        const int idx = o * kWorkers + tid;
        if (idx >= octs) break;
        if (cp.bal) {  // balanced columns of W: the same exponents on the slab's modes
          const int k0 = (idx / kRows) * 8;
          const int* sa = cp.bal + (int64_t)l * cp.K;
#pragma unroll
          for (int e = 0; e < 8; ++e)
            v[o][e] = __hiloint2double((int)raise((uint32_t)__double2hiint(v[o][e]), (uint32_t)sa[min(k0 + e, cp.K - 1)]),
                                       __double2loint(v[o][e]));
        }
        uint32_t mx = 0, low = 0;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          mx = max(mx, (uint32_t)__double2hiint(v[o][e]) & 0x7FFFFFFFu);
          low |= (uint32_t)__double2loint(v[o][e]);
        }
        if (mx == 0 && low) mx = 1;
        atomicMax(&cmax[idx % kRows], (int)mx);
      }
      named_sync(1, kWorkers);
#pragma unroll
      for (int o = 0; o < kOct; ++o) {
        const int idx = o * kWorkers + tid;
        if (idx >= octs) break;
        const int n = idx % kRows, ko = idx / kRows;
        const uint32_t cm = (uint32_t)cmax[n], em = cm ? cm >> 20 : 4096u;
        uint32_t lo[8], hi[8];
#pragma unroll
        for (int e = 0; e < 8; ++e)
          digits32<kBits>((uint32_t)__double2hiint(v[o][e]), (uint32_t)__double2loint(v[o][e]), em, lo[e], hi[e]);
        const uint32_t at = base + (uint32_t)(ko >> 3) * tileX + sw128(n, (ko & 7) * 16);
        store_digit<0x7632, 6, 0x03FF03FFu>(at, hi);  // bits 54 .. 63
        store_digit<0x6521, 5>(at + digX, hi);        // 45 .. 53
        store_digit<0x5410, 4>(at + 2 * digX, hi);    // 36 .. 44
        store_digit<0x7632, 2>(at + 4 * digX, lo);    // 18 .. 26
        store_digit<0x6521, 1>(at + 5 * digX, lo);    // 9 .. 17
        store_digit<0x5410, 0>(at + 6 * digX, lo);    // 0 .. 8
#pragma unroll
        for (int e = 0; e < 8; ++e) lo[e] = __funnelshift_r(lo[e], hi[e], 24);
        store_digit<0x5410, 3>(at + 3 * digX, lo);    // 27 .. 35
      }
      fence_async_smem();
      mbar_arrive(bready);
      if (q + (int)gridDim.x < a.total) load_tile(q + gridDim.x);  // in flight during the MMAs
      const int mt = SMALL ? 1 : (cp.K + 127) / 128;
      // this warp's tensor-memory lanes and columns
      const int qd = warp & 3, part = kN / (kWorkers / 128), c_lo = (warp >> 2) * part;
      double* o = cp.out + (int64_t)slab * cp.out_slab;
      bool ok = true;
      for (int m = 0; m < mt; ++m, ++gc) {
        ok = ok && mbar_wait(dfull, (uint32_t)gc & 1u);
        tc_fence_after();
        if (!ok) *abort_flag = 1;
        // lane = row r of W and columns = slab columns (or the reverse when SMALL)
        const int lim_l = SMALL ? cp.N - n0 : cp.K, lim_c = SMALL ? cp.K : cp.N - n0;
        const int r0 = m * 128 + qd * 32, r = r0 + lane;
        if (__all_sync(0xffffffffu, ok) && r0 < lim_l) {
          int e_lane = 0, m_lane = 0;  // exponent of this lane's row (or column)
          if (r < lim_l) {
            m_lane = SMALL ? cmax[r] : 0;
            e_lane = SMALL ? m_lane >> 20 : cp.expA[(int64_t)l * cp.K + r];
          }
          for (int c0 = c_lo; c0 < c_lo + part && c0 < lim_c; c0 += 4) {
            uint32_t d[kAcc][4];
            int vs[4][6];
            const uint32_t at = tmem + ((uint32_t)(qd * 32) << 16) + (uint32_t)c0;
#pragma unroll
            for (int g = 0; g < kAcc; ++g) tmem_ld4(at + (uint32_t)(g * kN), d[g]);
            tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 4; ++e) sums_of(d, e, vs[e]);
            if (kN == 32 && cp.K > 64 * kHalf) {  // the second half of K
#pragma unroll
              for (int g = 0; g < kAcc; ++g) tmem_ld4(at + (uint32_t)((kAcc + g) * kN), d[g]);
              tmem_wait_ld();
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                int w2[6];
                sums_of(d, e, w2);
#pragma unroll
                for (int g = 0; g < 6; ++g) vs[e][g] += w2[g];
              }
            }
            double res[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int mc = SMALL ? m_lane : cmax[c0 + e];  // of the slab column
              const int ec = SMALL ? (c0 + e < cp.K ? cp.expA[(int64_t)l * cp.K + c0 + e] : 0) : mc >> 20;
              res[e] = combine(vs[e], (e_lane + ec - 879 - 2 * kBits) * (1 << 20));
              if ((mc >= 1701 << 20) || (mc < 346 << 20 && mc)) {  // (an all-zero column gave 0)
                const int n = n0 + (SMALL ? r : c0 + e), rw = min(SMALL ? c0 + e : r, cp.K - 1);
                const double* p = cp.in + (int64_t)slab * cp.in_slab + (int64_t)n * cp.sn;
                const double* w = cp.W + ((int64_t)l * cp.K + rw) * cp.K;
                double s = 0.0;
                if (n < cp.N)
                  for (int k = 0; k < cp.K; ++k) s = __fma_rn(w[k], p[(int64_t)k * cp.sk], s);
                res[e] = s;
              }
            }
            const int64_t ls = SMALL ? cp.on : cp.om, cs = SMALL ? cp.om : cp.on;  // out strides along lanes, columns
            double* ob = o + (int64_t)n0 * cp.on;
            if (ls == 1) {  // lanes hold consecutive elements
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (r < lim_l && c0 + e < lim_c) ob[(int64_t)(c0 + e) * cs + r] = res[e];
            } else {  // the thread's four elements are consecutive: one 32-byte sector
              double* ot = ob + (int64_t)r * ls + c0;
              if (r < lim_l && c0 + 3 < lim_c && (reinterpret_cast<uintptr_t>(ot) & 15u) == 0) {
                reinterpret_cast<double2*>(ot)[0] = make_double2(res[0], res[1]);
                reinterpret_cast<double2*>(ot)[1] = make_double2(res[2], res[3]);
              } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                  if (r < lim_l && c0 + e < lim_c) ot[e] = res[e];
              }
            }
          }
        }
        tc_fence_before();
        mbar_arrive(dfree);
      }
      // the exponents of this tile have been read by every warp; every worker takes the same way out
      if (named_sync_or(1, kWorkers, !ok || *abort_flag)) break;
    }
  }
  // tear-down: every issued MMA has completed (mfin) and every issued TMA load has landed
  __syncthreads();
  if (tid == 0) {
    if (!mbar_wait(mfin, 0)) *abort_flag = 1;
    if (*abort_flag) {
      const int n = *n_items;
      for (int it = (n > a.stages ? n - a.stages : 0); it < n; ++it)
        (void)mbar_wait(full0 + 8 * (it % a.stages), (uint32_t)(it / a.stages) & 1u);
    }
  }
  __syncthreads();
  if (warp == kProducer) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
  }
  if (*abort_flag) {  // a wait expired: no tile of this CTA may pass for a result
    if (tid == 0) atomicExch(a.err, 1);
    const double nan = __longlong_as_double(0x7FF8000000000000ll);
    for (int q = blockIdx.x; q < a.total; q += gridDim.x) {
      int ci, slab, n0;
      locate(q, &ci, &slab, &n0);
      const F64Comp& cp = a.c[ci];
      for (int e = tid; e < cp.K * kRows; e += kF64Threads) {
        const int m = e / kRows, n = n0 + e % kRows;
        if (n < cp.N) cp.out[(int64_t)slab * cp.out_slab + (int64_t)m * cp.om + (int64_t)n * cp.on] = nan;
      }
    }
  }
}

// a_k (<< 20) of the columns of each mode's W [M][M]: the exponent of the column's maximum above the smallest one.
// One block per mode, a thread per column.
__global__ void __launch_bounds__(256) k_col_exponents(const double* __restrict__ W, int M, int* __restrict__ bal) {
  __shared__ int low;
  const double* w = W + (int64_t)blockIdx.x * M * M;
  const int k = threadIdx.x;
  if (k == 0) low = 2047;
  __syncthreads();
  uint32_t mx = 0;
  if (k < M)
    for (int m = 0; m < M; ++m) mx = max(mx, (uint32_t)__double2hiint(w[(int64_t)m * M + k]) & 0x7FFFFFFFu);
  if (mx) atomicMin(&low, (int)(mx >> 20));
  __syncthreads();
  if (k < M) bal[(int64_t)blockIdx.x * M + k] = mx ? min((int)(mx >> 20) - low, 400) << 20 : 0;
}

// Digits of the rows of W [rows][K], its columns taken by 2^-a_k when 'bal' is given: D[((l 7 + i) M + m) ld + k] =
// digit i of W[l][m][k] (float16, zero for k >= K), expA[row] the biased exponent of the row's maximum.  One warp per
// row.  'bad' is set when a row is not finite or its maximum lies outside 2^+-200 (the split would not be exact), and
// for the 59-bit integers when its digits do not keep every D_3 (and so D_0 .. D_2) within 2^24: |d_0| <= 32 and
// |d_i| <= 256 on the slab's side, the first and second 128 of K > 192 apart.  (Digits of a matrix average half
// their range: 0.9 x 2^24 at K = 192.)  The components then keep the CUDA-core kernels.
__global__ void __launch_bounds__(256) k_split_rows(const double* __restrict__ W, int64_t rows, int M, int ld, int bits,
                                                    const int* __restrict__ bal, uint16_t* __restrict__ D,
                                                    int* __restrict__ expA, int* bad) {
  const int64_t row = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= rows) return;
  const int64_t l = row / M, m = row - l * M;
  const double* w = W + row * M;
  auto value = [&](int k) {
    return bal ? w[k] * __hiloint2double((1023 << 20) - bal[l * M + k], 0) : w[k];
  };
  uint32_t mx = 0;
  for (int k = lane; k < M; k += 32) mx = max(mx, (uint32_t)__double2hiint(value(k)) & 0x7FFFFFFFu);
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  const int em = (int)(mx >> 20);
  if (lane == 0) {
    expA[row] = em;
    if (em < 823 || em > 1223) *bad = 1;
  }
  int most[2] = {0, 0};  // this lane's part of the bound of D_3
  for (int k = lane; k < ld; k += 32) {
    const uint64_t g = digits_of(k < M ? value(k) : 0.0, em, bits);
    int b3 = 0;
#pragma unroll
    for (int i = 0; i < kDig; ++i) {
      const int dg = (int)((i == 0 ? g >> 54 : (g >> (9 * (6 - i))) & 0x1FFull)) - 256;
      D[((l * kDig + i) * M + m) * ld + k] = __half_as_ushort(__int2half_rn(k < M ? dg : 0));
      if (k < M && i < 4) b3 += abs(dg) * (i == 3 ? 32 : 256);
    }
    most[M > 192 && k >= 128] += b3;
  }
  for (int o = 16; o > 0; o >>= 1) {
    most[0] += __shfl_xor_sync(0xffffffffu, most[0], o);
    most[1] += __shfl_xor_sync(0xffffffffu, most[1], o);
  }
  if (lane == 0 && bits != kBitsSmall && max(most[0], most[1]) > 1 << 24) *bad = 1;
}

constexpr int kF64MaxK = 256;
size_t f64_smem(int nt, bool small, int kblocks, int stages) {
  const size_t rows = small ? 128 : nt;
  return 1024 + (size_t)kDig * kblocks * rows * 128 + (size_t)stages * (small ? 8192 : kBlockA) + 2 * rows * 4 + 192;
}
int pad8(int n) { return (n + 7) / 8 * 8; }

}  // namespace

int64_t f64_digit_bytes(int64_t nl, int n) { return nl * n * (int64_t)(pad8(n) * kDig * 2 + 4); }

// Splits W (nl matrices n x n) of a component into digits ('small': the form whose TMA box has 64 rows; 'balance': its
// columns taken by powers of two); *bad is set when a row cannot be split exactly, *mapped cleared when the digits have
// no tensor map.
static int split_matrix(fm_ctx* c, const double* W, int64_t nl, int n, bool small, bool balance, F64Mat* f, int* bad,
                        bool* mapped) {
  int rc;
  const int ld = pad8(n);
  void* D = nullptr;
  if ((rc = dev_alloc(c, &D, (size_t)nl * kDig * n * ld * 2))) return rc;
  if (!encode3t(&f->tm, D, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, ld, n, (int)(nl * kDig), 64, small ? 64 : 128)) {
    *mapped = false;
    return FM_OK;
  }
  if ((rc = dev_alloc(c, (void**)&f->exps, (size_t)nl * n * 4))) return rc;
  if (balance) {
    if ((rc = dev_alloc(c, (void**)&f->bal, (size_t)nl * n * 4))) return rc;
    k_col_exponents<<<(unsigned)nl, 256, 0, c->stream>>>(W, n, f->bal);
  }
  const int64_t rows = nl * n;
  k_split_rows<<<(unsigned)((rows + 7) / 8), 256, 0, c->stream>>>(W, rows, n, ld, small ? kBitsSmall : kBitsLarge, f->bal,
                                                                  (uint16_t*)D, f->exps, bad);
  FM_CUDA(cudaGetLastError());
  f->W = W;
  return FM_OK;
}

// longest contraction of a stage over the components (one launch serves them all)
static int stage_k(const fm_ctx* c, int stage) {
  int k = 1;
  for (auto& cp : c->comps) k = std::max(k, stage < 2 ? cp.nz : cp.nx);
  return k;
}

// FM_PREC_FP64: digits of the z and x matrices of every component they serve.  Without tensor maps for them (a driver
// without the encoder, an encoding refused) the CUDA-core kernels stay.
int f64_setup(fm_ctx* c) {
  if (c->opts.precision != FM_PREC_FP64 || c->opts.mma == FM_MMA_SIMT) return FM_OK;
  int rc;
  FM_CUDA(cudaFuncSetAttribute(k_tc_f64<64, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  FM_CUDA(cudaFuncSetAttribute(k_tc_f64<64, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  FM_CUDA(cudaFuncSetAttribute(k_tc_f64<32, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  int* bad = c->tc_err + 1;
  bool all = true;
  for (auto& cp : c->comps) all = all && cp.nx <= kF64MaxK && cp.nz <= kF64MaxK;
  if (!all) return FM_OK;
  const bool zs = stage_k(c, 0) <= 64, xs = stage_k(c, 2) <= 64;
  for (auto& cp : c->comps) {
    const double* W[4] = {cp.Wzb, cp.Wz, cp.Wxb, cp.Wx};
    for (int st = 0; st < 4; ++st) {
      bool mapped = true;
      if ((rc = split_matrix(c, W[st], st < 2 ? c->nM : cp.nl, st < 2 ? cp.nz : cp.nx, st < 2 ? zs : xs, st == 1,
                             &cp.f64[st], bad, &mapped)))
        return rc;
      if (!mapped) return FM_OK;
    }
  }
  int h = 0;
  FM_CUDA(cudaMemcpyAsync(&h, bad, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  FM_CUDA(cudaStreamSynchronize(c->stream));
  c->f64_tc = h == 0;
  return FM_OK;
}

// One stage of every component in one launch: 0 W-bar_z, 1 W_z, 2 W-bar_x, 3 W_x of the chain
//   z forward  in[M'][k][i][j] -> t[slab][i][j]      x forward  t[slab][i][j] -> u[slab][j][i]
//   x inverse  u[slab][j][i]   -> t[slab][i][j]      z inverse  t[slab][i][j] -> out[M'][k][i][j]
int f64_stage(fm_ctx* c, int stage, const double* in, double* out) {
  F64Args a;
  std::memset(&a, 0, sizeof(a));
  a.ncomp = (int)c->comps.size();
  const int kmax = stage_k(c, stage);
  const bool small = kmax <= 64;
  const int nt = kmax <= 192 ? 64 : 32, cols = small ? 128 : nt;
  double fl = 0.0, by = 0.0;
  for (int q = 0; q < a.ncomp; ++q) {
    const Comp& cp = c->comps[q];
    F64Comp& f = a.c[q];
    const F64Mat& m = cp.f64[stage];
    const int64_t nxy = (int64_t)cp.nx * cp.ny;
    f.tmA = m.tm;
    f.W = m.W;
    f.expA = m.exps;
    f.bal = m.bal;
    f.in = in + cp.off;
    f.out = out + cp.off;
    if (stage < 2) {
      f.K = cp.nz;
      f.N = (int)nxy;
      f.slabs = c->nM;
      f.in_slab = f.out_slab = cp.nz * nxy;
      f.sk = f.om = nxy;
      f.sn = f.on = 1;
    } else {
      f.K = cp.nx;
      f.N = cp.ny;
      f.slabs = c->nM * cp.nz;
      f.nz = cp.nz;
      f.in_slab = f.out_slab = nxy;
      f.sk = stage == 2 ? cp.ny : 1;
      f.sn = stage == 2 ? 1 : cp.nx;
      f.om = stage == 2 ? 1 : cp.ny;
      f.on = stage == 2 ? cp.nx : 1;
    }
    f.ntile = (f.N + cols - 1) / cols;
    a.total += f.slabs * f.ntile;
    const double nun = (double)nxy * cp.nz * c->nM;
    fl += 2.0 * f.K * nun;
    by += 16.0 * nun;
  }
  a.kblocks = (kmax + 63) / 64;
  a.stages = small ? kDig : 4;
  while (!small && a.stages > 2 && f64_smem(nt, small, a.kblocks, a.stages) > 227 * 1024) --a.stages;
  a.err = c->tc_err;
  const size_t smem = f64_smem(nt, small, a.kblocks, a.stages);
  const int grid = std::min(a.total, 152);
  const int tk_ = prof_begin(c, stage < 2 ? FM_KERNEL_ZMIX : FM_KERNEL_XMIX);
  if (small) k_tc_f64<64, true><<<grid, kF64Threads, smem, c->stream>>>(a);
  else if (nt == 64) k_tc_f64<64, false><<<grid, kF64Threads, smem, c->stream>>>(a);
  else k_tc_f64<32, false><<<grid, kF64Threads, smem, c->stream>>>(a);
  prof_end(c, tk_, fl, by);
  c->launches++;
  FM_CUDA(cudaGetLastError());
  return FM_OK;
}

}  // namespace fmi
