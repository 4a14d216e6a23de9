// Banded y solves of the preconditioner (Eq. prec-2, the y stage with the M' chain).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cstring>
#include <type_traits>
#include <vector>

#include "fm_apply.h"
#include "fm_internal.h"
#include "fm_tc.h"

namespace {

using fmi::mbar_arrive;
using fmi::mbar_expect_tx;
using fmi::mbar_init;
using fmi::mbar_wait;

// ---------------------------------------------------------------------------
// Banded y solves: one lane per (l, i_x) line of a component, 32 lines per CTA; the right-hand side of a line is the
// M' chain of y vectors u[iM][l - M'][j][i_x] interleaved as r = j n_c + c, solved in place by the banded LU factors
// (forward with row pivots, then backward by columns).  Bound by each line's chain of dependent rows, so a row is
// kept short:
//   * a producer warp feeds a ring in shared memory a few chunks of rows ahead.  The host lays the factors of a CTA's
//     lines out contiguously per row, so a chunk is one bulk copy; the line's own values ride along by cp.async.  The
//     solver warp only waits, multiplies and stores (it copied its own rows before: half of its instructions);
//   * both sweeps update a window of pending rows in registers (right-looking), whose shift is the destination of the
//     update: no moves, and one multiply-add between a row's value and the next;
//   * the pivots of a chain of n_c components only ever swap rows of the same component: with STEP = n_c two (cubic)
//     or four (quintic) candidates are compared instead of the whole window.  Chains whose factors pivot otherwise
//     take STEP = 1.
// Every wait is bounded; a wait that expires sets the context's wait flag and leaves NaN in the lines.
// ---------------------------------------------------------------------------
struct YArgs {
  int nx, ny, nz, M0, nl;
  int kq;                   // band half-width of the 1D y matrices (2 cubic, 4 quintic)
  int64_t comp_off;
  const int* chain_lo;   // [nl]
  const int* chain_n;    // [nl]
  const int* pstep;      // [nl] n_c when every pivot offset of the chain is a multiple of it, else 1
  const int64_t* band_off;  // [nl] offset into U: [block of 32 lines][n][2 kl + 1][lines of the block, padded to 4]
  const int64_t* lmul_off;  // [nl] offset into L: [block][n][kl + 1][lines]
};

// Row walker of a line: row r = j * n_c + c lives at P0 + c * DC + j * nx (DC the distance between the
// chain's neighbouring M' components), stepped without divisions.
template <typename T>
struct RowPtr {
  T* p;
  int c, nc;
  int64_t dc, nx;
  __device__ __forceinline__ void next() {
    p += dc;
    if (++c == nc) {
      c = 0;
      p += nx - (int64_t)nc * dc;
    }
  }
  __device__ __forceinline__ void prev() {
    p -= dc;
    if (--c < 0) {
      c = nc - 1;
      p -= nx - (int64_t)nc * dc;
    }
  }
};

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ int pivot_of(float v) { return __float_as_int(v); }   // an integer's bits, set by the host
__device__ __forceinline__ int pivot_of(double v) { return __double2loint(v); }

constexpr int kYStages = 3;

// The ring of one CTA: kYStages stages of 'rows' factor rows (slots x wd values each) and as many line values
template <typename T>
struct YRing {
  T* buf;
  uint32_t full, empty;  // barriers [kYStages]
  int rows, fstride;     // rows per stage; values of a stage's factor part
  __device__ __forceinline__ T* stage(int s) const { return buf + (size_t)s * (fstride + rows * 32); }
};

// The producer's sweep: chunk ch holds rows ch * rows .. of F ([n][slots][wd], in the sweep's order) and the line
// values of the rows that enter the solver's window 'ahead' rows after them.  Returns false when a wait expired.
template <typename T, bool FWD>
__device__ __forceinline__ bool y_produce(const YRing<T>& rg, const T* F, int n, int slots, int wd, int ahead,
                                          RowPtr<T> rp, bool live, int lane, int& it) {
  const int nch = (n + rg.rows - 1) / rg.rows;
  int next = 0;  // rp stands on row 'next' of the sweep
  for (int ch = 0; ch < nch; ++ch, ++it) {
    const int st = it % kYStages, r0 = ch * rg.rows, cnt = min(rg.rows, n - r0);
    if (it >= kYStages && !__all_sync(0xffffffffu, mbar_wait(rg.empty + 8 * st, ((uint32_t)(it / kYStages) & 1u) ^ 1u)))
      return false;
    T* dst = rg.stage(st);
    const uint32_t bar = rg.full + 8 * st;
    if (lane == 0) {
      const uint32_t bytes = (uint32_t)(cnt * slots * wd * (int)sizeof(T));
      mbar_expect_tx(bar, bytes);
      bulk_load((uint32_t)__cvta_generic_to_shared(dst), F + (int64_t)r0 * slots * wd, bytes, bar);
    }
    while (next < r0 + ahead && next < n) {  // first chunk only: the rows the solver loads itself
      if (FWD) rp.next();
      else rp.prev();
      ++next;
    }
    T* line = dst + rg.fstride + lane;
    for (int q = 0; q < cnt && next < n; ++q, ++next) {
      if (live) {
        const uint32_t d = (uint32_t)__cvta_generic_to_shared(line + q * 32);
        if (sizeof(T) == 8) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(rp.p + lane) : "memory");
        else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(rp.p + lane) : "memory");
      }
      if (FWD) rp.next();
      else rp.prev();
    }
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
  }
  return true;
}

// The solver's sweeps.  Forward: z_r = the pivot row's entry of the window, w <- (swapped, shifted) w - L_r z_r.
// Backward: x_r = s_0 / pivot, s <- (shifted) s - U_r x_r with U_r[d] the coefficient of x_r in row r - d.
template <typename T, int KL, int STEP, bool FWD>
__device__ __forceinline__ bool y_sweep(const YRing<T>& rg, int n, int wd, int lane, int lf, bool live, RowPtr<T> rp, T* first,
                                        int& it) {
  constexpr int NW = FWD ? KL + 1 : 2 * KL;  // window
  constexpr int SL = FWD ? KL + 1 : 2 * KL + 1;
  T w[NW];
#pragma unroll
  for (int i = 0; i < NW; ++i) w[i] = first[i];
  const int nch = (n + rg.rows - 1) / rg.rows;
  for (int ch = 0; ch < nch; ++ch, ++it) {
    const int st = it % kYStages, r0 = ch * rg.rows, cnt = min(rg.rows, n - r0);
    if (!__all_sync(0xffffffffu, mbar_wait(rg.full + 8 * st, (uint32_t)(it / kYStages) & 1u))) return false;
    const T* f = rg.stage(st) + lf;
    const T* line = rg.stage(st) + rg.fstride + lane;
#pragma unroll 2
    for (int q = 0; q < cnt; ++q, f += SL * wd) {
      const T in = (r0 + q + NW < n) ? line[q * 32] : (T)0;
      if (FWD) {
        const int p = pivot_of(f[0]);
        const T w0 = w[0];
        T x = w0;
#pragma unroll
        for (int i = STEP; i <= KL; i += STEP)
          if (p == i) x = w[i];
#pragma unroll
        for (int i = 0; i < KL; ++i) {
          T src = w[i + 1];
          if ((i + 1) % STEP == 0 && p == i + 1) src = w0;
          w[i] = fma(-f[(i + 1) * wd], x, src);
        }
        w[KL] = in;
        if (live) rp.p[lane] = x;
        rp.next();
      } else {
        const T x = w[0] * f[0];
#pragma unroll
        for (int i = 0; i + 1 < NW; ++i) w[i] = fma(-f[(i + 1) * wd], x, w[i + 1]);
        w[NW - 1] = fma(-f[NW * wd], x, in);
        if (live) rp.p[lane] = x;
        rp.prev();
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(rg.empty + 8 * st);
  }
  return true;
}

// the instantiation of a chain: band half-width and pivot step (the wide bands only with step 1)
#define FM_Y_SWITCH(GO)                              \
  switch (kl * 16 + (step == 1 ? 1 : step)) {        \
    case 2 * 16 + 1: GO(2, 1) break;                 \
    case 4 * 16 + 1: GO(4, 1) break;                 \
    case 5 * 16 + 1: GO(5, 1) break;                 \
    case 5 * 16 + 2: GO(5, 2) break;                 \
    case 7 * 16 + 1: GO(7, 1) break;                 \
    case 7 * 16 + 3: GO(7, 3) break;                 \
    case 9 * 16 + 1: GO(9, 1) break;                 \
    case 9 * 16 + 2: GO(9, 2) break;                 \
    case 9 * 16 + 4: GO(9, 4) break;                 \
    case 11 * 16 + 1: GO(11, 1) break;               \
    case 11 * 16 + 5: GO(11, 5) break;               \
    case 13 * 16 + 1: GO(13, 1) break;               \
    case 13 * 16 + 3: GO(13, 3) break;               \
    case 15 * 16 + 1: GO(15, 1) break;               \
    case 17 * 16 + 1: GO(17, 1) break;               \
    case 17 * 16 + 4: GO(17, 4) break;               \
    case 19 * 16 + 1: GO(19, 1) break;               \
    case 21 * 16 + 1: GO(21, 1) break;               \
    case 23 * 16 + 1: GO(23, 1) break;               \
    default: GO(25, 1) break;                        \
  }

// the components of one launch (blockIdx.z selects one)
template <typename T>
struct YBatch {
  YArgs a[3];
  const T* U[3];
  const T* L[3];
  int* err;
};

template <typename T>
__global__ void __launch_bounds__(64) k_ysolve(const __grid_constant__ YBatch<T> yb, int rows, int slots_max, T* __restrict__ t) {
  extern __shared__ __align__(128) unsigned char smraw_y[];
  __shared__ __align__(8) uint64_t bars[2 * kYStages];
  __shared__ int failed;
  const YArgs& a = yb.a[blockIdx.z];
  const int il = blockIdx.y, ix0 = blockIdx.x * 32;
  if (il >= a.nl || ix0 >= a.nx) return;  // grid sized for the largest component (uniform per CTA)
  const int nc = a.chain_n[il], lo = a.chain_lo[il], n = nc * a.ny;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int valid = min(32, a.nx - ix0), wd = (valid + 3) & ~3;  // lines of the block, and as stored
  const bool live = lane < valid;
  const int lf = min(lane, wd - 1);
  const int kl = (nc == 1) ? a.kq : a.kq * nc + 1;  // band half-width of this chain (band_kl on the host)
  const int64_t blk = (int64_t)ix0 * n;             // full blocks before this one hold 32 lines each
  const T* Lb = yb.L[blockIdx.z] + a.lmul_off[il] + blk * (kl + 1);
  const T* Ub = yb.U[blockIdx.z] + a.band_off[il] + blk * (2 * kl + 1);
  RowPtr<T> rp0;
  rp0.p = t + a.comp_off + ((int64_t)lo * a.nz + (il - lo)) * a.ny * a.nx + ix0;  // (iM, k) = (lo, l - M0 - lo), j = 0
  rp0.c = 0;
  rp0.nc = nc;
  rp0.dc = (int64_t)(a.nz - 1) * a.ny * a.nx;  // (iM + 1, k - 1) from (iM, k): row r + 1 within one j
  rp0.nx = a.nx;
  RowPtr<T> rpe = rp0;  // row n - 1
  rpe.p += (int64_t)(a.ny - 1) * a.nx + (int64_t)(nc - 1) * rp0.dc;
  rpe.c = nc - 1;
  YRing<T> rg;
  rg.buf = reinterpret_cast<T*>(smraw_y);
  rg.full = (uint32_t)__cvta_generic_to_shared(bars);
  rg.empty = rg.full + 8 * kYStages;
  rg.rows = rows;
  rg.fstride = rows * slots_max * 32;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kYStages; ++s) {
      mbar_init(rg.full + 8 * s, 33);  // the bulk copy's expect and the 32 lanes' cp.async
      mbar_init(rg.empty + 8 * s, 1);
    }
    failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  int it = 0;
  bool ok = true;
  if (warp == 1) {
    ok = y_produce<T, true>(rg, Lb, n, kl + 1, wd, kl + 1, rp0, live, lane, it);
  } else {
    T first[fmi::kMaxBandKL + 1];
    const int step = a.pstep[il];
#define FM_YF(KLV, ST)                                                                              \
  {                                                                                                 \
    RowPtr<T> rw = rp0;                                                                             \
    _Pragma("unroll") for (int i = 0; i <= KLV; ++i) {                                              \
      first[i] = (live && i < n) ? rw.p[lane] : (T)0;                                               \
      rw.next();                                                                                    \
    }                                                                                               \
    ok = y_sweep<T, KLV, ST, true>(rg, n, wd, lane, lf, live, rp0, first, it);                      \
  }
    FM_Y_SWITCH(FM_YF)
#undef FM_YF
  }
  if (!ok) failed = 1;
  // the forward results must be in memory before the backward sweep reads them
  __threadfence();
  __syncthreads();
  if (!failed) {
    if (warp == 1) {
      ok = y_produce<T, false>(rg, Ub, n, 2 * kl + 1, wd, 2 * kl, rpe, live, lane, it);
    } else {
      T first[2 * fmi::kMaxBandKL];
      const int step = 1;
#define FM_YB(KLV, ST)                                                                              \
  {                                                                                                 \
    RowPtr<T> rw = rpe;                                                                             \
    _Pragma("unroll") for (int i = 0; i < 2 * KLV; ++i) {                                           \
      first[i] = (live && i < n) ? rw.p[lane] : (T)0;                                               \
      rw.prev();                                                                                    \
    }                                                                                               \
    ok = y_sweep<T, KLV, 1, false>(rg, n, wd, lane, lf, live, rpe, first, it);                      \
  }
      FM_Y_SWITCH(FM_YB)
#undef FM_YB
    }
    if (!ok) failed = 1;
  }
  __syncthreads();
  if (failed) {  // a wait expired: let the copies in flight land, then nothing of these lines may pass for a result
    if (warp == 1) {
      asm volatile("cp.async.wait_all;" ::: "memory");
      for (int s = 0; s < kYStages && s < it; ++s) (void)mbar_wait(rg.full + 8 * ((it - 1 - s) % kYStages), (uint32_t)((it - 1 - s) / kYStages) & 1u);
      if (lane == 0 && yb.err) atomicExch(yb.err, 1);
    } else if (live) {
      RowPtr<T> rw = rp0;
      for (int r = 0; r < n; ++r) {
        rw.p[lane] = (T)__int_as_float(0x7FC00000);
        rw.next();
      }
    }
  }
}

}  // namespace

namespace fmi {

// Banded y solves (Eq. prec-2 y stage with the M' chain) of the given components in one launch,
// in place on u[slab][j][i].
template <typename T>
int ysolve_banded(fm_ctx* c, const std::vector<fmi::Comp*>& comps, T* u) {
  if (comps.empty()) return FM_OK;
  if (comps.size() > 3) return FM_ERR_ARG;
  const double ts = (double)sizeof(T);
  double yfl = 0.0, yby = 0.0;  // per line 2n(kl + ku + kl) + n flops; factor and vector bytes
  YBatch<T> yb;
  std::memset(&yb, 0, sizeof(yb));
  yb.err = c->tc_err;
  int slots = 5, gx = 1, gy = 1, ctas = 0;
  for (size_t q = 0; q < comps.size(); ++q) {
    const fmi::Comp& cp = *comps[q];
    for (int il = 0; il < cp.nl; ++il) {
      const int nc = cp.chain_n[il], n = nc * cp.ny, kl = band_kl(cp.ay, nc);
      yfl += (double)cp.nx * (2.0 * n * (3.0 * kl) + n);
      yby += (double)cp.nx * ((double)n * (3.0 * kl + 2.0) * ts + 2.0 * n * ts);
      slots = std::max(slots, 2 * kl + 1);
    }
    YArgs& ya = yb.a[q];
    ya.nx = cp.nx; ya.ny = cp.ny; ya.nz = cp.nz; ya.M0 = c->M0; ya.nl = cp.nl; ya.comp_off = cp.off;
    ya.kq = band_kq(cp.ay);
    ya.chain_lo = (const int*)cp.d_chain_lo; ya.chain_n = (const int*)cp.d_chain_n;
    ya.pstep = cp.d_pstep;
    ya.band_off = cp.d_band_off; ya.lmul_off = cp.d_lmul_off;
    yb.U[q] = std::is_same<T, double>::value ? (const T*)cp.yU : (const T*)cp.yU32;
    yb.L[q] = std::is_same<T, double>::value ? (const T*)cp.yL : (const T*)cp.yL32;
    gx = std::max(gx, (cp.nx + 31) / 32);
    gy = std::max(gy, cp.nl);
    ctas += ((cp.nx + 31) / 32) * cp.nl;
  }
  // Rows per stage: as many CTAs per SM as the grid gives it (up to 8) share 220 KB; 2 to 16 rows a stage
  const size_t per_row = (size_t)(slots + 1) * 32 * sizeof(T);
  const int per_sm = std::max(1, std::min(8, (ctas + 151) / 152));
  const int rows = (int)std::max<size_t>(2, std::min<size_t>(16, (220 * 1024 / per_sm - 1024) / (kYStages * per_row)));
  const size_t sm = kYStages * rows * per_row;
  const int tk_ = prof_begin(c, FM_KERNEL_YSOLVE);
  k_ysolve<T><<<dim3(gx, gy, (unsigned)comps.size()), 64, sm, c->stream>>>(yb, rows, slots, u);
  prof_end(c, tk_, yfl, yby);
  c->launches++;
  FM_CUDA(cudaGetLastError());
  return FM_OK;
}

template int ysolve_banded<double>(fm_ctx*, const std::vector<Comp*>&, double*);
template int ysolve_banded<float>(fm_ctx*, const std::vector<Comp*>&, float*);

int ysolve_init() {
  FM_CUDA(cudaFuncSetAttribute(k_ysolve<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024));
  FM_CUDA(cudaFuncSetAttribute(k_ysolve<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024));
  return FM_OK;
}

}  // namespace fmi
