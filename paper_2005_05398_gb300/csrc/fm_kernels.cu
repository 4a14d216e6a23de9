// CUDA kernels of libfm (sm_103a).
//
//  * operator apply y = (H - E S) x (Eq. FM-lin; H from Eq. FM-pre, storage idea of
//    Eq. l-form): sum-factorised banded contractions in y, x and z with the pointwise
//    coefficients and the M' +- 1 couplings, one kernel that walks the z planes;
//    (the V^(s) coupling term of Eqs. r-form, s-rot is in fm_coupling.cuh);
//  * the tensor-trick preconditioner (Eq. prec-2): its chain and the CUDA-core z and x
//    mode products (the banded y solves that replace the y eigen-transforms and the
//    tridiagonal M' chains, the same operator factorised by banded LU, are in fm_ysolve.cu);
//  * deterministic Krylov reductions (fixed grid, fixed reduction order).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cstring>
#include <type_traits>
#include <vector>

#include "fm_apply.h"
#include "fm_internal.h"

namespace {

// ---------------------------------------------------------------------------
// The local part of the operator, y = (L - E S) c (or S c).  At a collocation point (zeta, xi, eta) of component M'
//   y = (W - E) U + q Z - D + (n_M > 1) iy2 [T+ psi_{M'+1} + T- psi_{M'-1}],   q = 1/x^2 + 1/y^2,
//   U = S_z P,  Z = [2 (M'+1) z D1_z - (1 - z^2) D2_z] P,  D = S_z Q,
//   P = S_x S_y c,  Q = (D2_x S_y + S_x D2_y) c,
// with the z contractions' taps combined on the host (cp.zt), so that a point takes 8 (y, times the halo) + 12 (x)
// + 12 (z) + 3 multiply-adds for r = 4 and n_M = 1 (five separate z contractions and three planes took 45).
//
// float32, one pass over the coefficients: a CTA owns a tile of 16 x 16 (x, y) points and a chunk of z intervals
// and walks the z planes; an interval's planes (with their halo, all M') stream into shared memory by cp.async while
// the previous ones are contracted in y (shared memory) and x (registers), and every thread keeps the last r planes
// of P and Q of its point in registers, from which it forms the z outputs of each interval.  The planes never go to
// memory: 47 us an application at 3.7 M unknowns against 95 us of two kernels (He L = 0, 96 x 96 x 24).
// ---------------------------------------------------------------------------
constexpr int kLX = 16, kLY = 16, kLThreads = kLX * kLY;  // tile (points)

struct LocalComp {
  const float* x;
  float* y;
  const float *W, *Sx, *D2x, *Sy, *D2y, *zt, *qx, *iy2;
  const int *bx, *by, *zf;   // tap bases; first z point of each z interval [nint + 1]
  int nx, ny, nz;
  int rows, cols;            // coefficients a tile reads in x and y
  int tiles_x, tiles_y, nint, q, ipc;  // tiles; z intervals, functions per node, intervals per chunk
  int first;                 // first block of the component
};
struct LocalArgs {
  LocalComp c[3];
  int ncomp;
  float E;
  int only_S;
};

template <int B>
__device__ __forceinline__ void cp_async_elem(void* dst, const void* src, bool ok) {  // zero-filled when !ok
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(d), "l"(src), "n"(B), "r"(ok ? B : 0) : "memory");
}

template <int R, int NM>
__global__ void __launch_bounds__(kLThreads, R * NM <= 8 ? 4 : (R * NM <= 12 ? 3 : 2))
    k_apply_local(const __grid_constant__ LocalArgs a) {
  using T = float;
  constexpr int PS = R / 2, kAhead = 2;  // planes per step (an interval); z points whose W is loaded ahead
  extern __shared__ __align__(16) unsigned char smraw_l[];
  int ci = 0;
  while (ci + 1 < a.ncomp && (int)blockIdx.x >= a.c[ci + 1].first) ++ci;
  const LocalComp& c = a.c[ci];
  const int rows = c.rows, ld = c.cols + 1, tiles = c.tiles_x * c.tiles_y;
  T* tab = reinterpret_cast<T*>(smraw_l);       // S_y, D2_y [R][kLY]; S_x, D2_x [R][kLX]
  T* cs = tab + 2 * R * (kLX + kLY);            // [2][PS][NM][rows][ld]
  T* As = cs + 2 * PS * NM * rows * ld;         // [PS][NM][rows][kLY]  S_y c
  T* Bs = As + PS * NM * rows * kLY;            //                      D2_y c
  const int b = (int)blockIdx.x - c.first, chunk = b / tiles, tile = b - chunk * tiles;
  const int xi0 = (tile / c.tiles_y) * kLX, eta0 = (tile % c.tiles_y) * kLY;
  const int tid = threadIdx.x, tx = tid / kLY, ty = tid % kLY;
  const int xi = xi0 + tx, eta = eta0 + ty;
  const bool live = xi < c.nx && eta < c.ny;
  const int xc = min(xi, c.nx - 1), ec = min(eta, c.ny - 1);
  const int r0 = c.bx[xi0], c0 = c.by[eta0];
  const int lr = c.bx[xc] - r0, lc = c.by[ec] - c0;
  for (int e = tid; e < R * (kLX + kLY); e += kLThreads) {
    const bool isx = e >= R * kLY;
    const int q = isx ? e - R * kLY : e, n = isx ? kLX : kLY, t = q / n, g = q - t * n;
    const int at = isx ? min(xi0 + g, c.nx - 1) : min(eta0 + g, c.ny - 1);
    T* d = tab + (isx ? 2 * R * kLY : 0) + q;
    d[0] = (isx ? c.Sx : c.Sy)[at * R + t];
    d[R * n] = (isx ? c.D2x : c.D2y)[at * R + t];
  }
  const T* ys = tab + ty;
  const T* xs = tab + 2 * R * kLY + tx;
  const T iy2 = c.iy2[ec], q = c.qx[xc] + iy2;
  const int64_t nxy = (int64_t)c.nx * c.ny, npts = nxy * c.nz;
  const int m0 = chunk * c.ipc, m1 = min(c.nint, m0 + c.ipc);
  const int k0 = c.q * m0, k1 = c.q * (m1 - 1) + R - 1;  // planes of the chunk (their number is a multiple of PS)
  // rows of PS planes' tiles (all M'), 32 lanes a row
  auto fetch = [&](int k, int buf) {
    T* dst = cs + buf * PS * NM * rows * ld;
    constexpr int LN = 2 * kLY;
    const int ln = tid % LN;
    if (ln < c.cols) {
      const int col = c0 + ln;
      for (int rr = tid / LN; rr < PS * NM * rows; rr += kLThreads / LN) {
        const int pm = PS * NM == 1 ? 0 : rr / rows, ps = pm / NM, M = pm - ps * NM, r = r0 + rr - pm * rows;
        const bool ok = r >= 0 && r < c.nx && col >= 0 && col < c.ny;
        const T* src = ok ? c.x + ((int64_t)M * c.nz + k + ps) * nxy + (int64_t)r * c.ny + col : c.x;
        cp_async_elem<sizeof(T)>(dst + rr * ld + ln, src, ok);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  T P[NM][R], Q[NM][R];
#pragma unroll
  for (int M = 0; M < NM; ++M)
#pragma unroll
    for (int t = 0; t < R; ++t) P[M][t] = Q[M][t] = (T)0;
  int m = m0;
  fetch(k0, 0);
  const int64_t oxy = (int64_t)xc * c.ny + ec;
  T wq[kAhead + 1][NM];  // W of the next z points
  if (!a.only_S) {
#pragma unroll
    for (int h = 0; h < kAhead; ++h)
#pragma unroll
      for (int M = 0; M < NM; ++M) wq[h][M] = c.W[M * npts + min(c.zf[m0] + h, c.nz - 1) * nxy + oxy];
  }
  for (int k = k0, buf = 0; k <= k1; k += PS, buf ^= 1) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // these planes are in shared memory; the previous ones' x pass is done
    if (k + PS <= k1) fetch(k + PS, buf ^ 1);
    const T* cb = cs + buf * PS * NM * rows * ld;
    for (int rr = tx; rr < PS * NM * rows; rr += kLX) {
      const T* v = cb + rr * ld + lc;
      T s = ys[0] * v[0], d = ys[R * kLY] * v[0];
#pragma unroll
      for (int t = 1; t < R; ++t) {
        s = fma(ys[t * kLY], v[t], s);
        d = fma(ys[(R + t) * kLY], v[t], d);
      }
      As[rr * kLY + ty] = s;
      Bs[rr * kLY + ty] = d;
    }
    __syncthreads();
#pragma unroll
    for (int M = 0; M < NM; ++M) {
#pragma unroll
      for (int t = 0; t + PS < R; ++t) {
        P[M][t] = P[M][t + PS];
        Q[M][t] = Q[M][t + PS];
      }
#pragma unroll
      for (int ps = 0; ps < PS; ++ps) {
        const T* pa = As + ((ps * NM + M) * rows + lr) * kLY + ty;
        const T* pb = Bs + ((ps * NM + M) * rows + lr) * kLY + ty;
        T p = (T)0, d = (T)0;
#pragma unroll
        for (int t = 0; t < R; ++t) {
          const T av = pa[t * kLY], sx = xs[t * kLX];
          p = fma(sx, av, p);
          d = fma(xs[(R + t) * kLX], av, fma(sx, pb[t * kLY], d));
        }
        P[M][R - PS + ps] = p;
        Q[M][R - PS + ps] = d;
      }
    }
    if (k + PS - R != c.q * m) continue;
    // planes q m .. q m + r - 1 are at hand: the z points of interval m
    const int z1 = c.zf[m + 1];
    for (int zeta = c.zf[m]; zeta < z1; ++zeta) {
      const int64_t o = (int64_t)zeta * nxy + oxy;
      T w[NM];
      if (!a.only_S) {
        const int64_t on = min(zeta + kAhead, c.nz - 1) * nxy + oxy;
#pragma unroll
        for (int M = 0; M < NM; ++M) {
          wq[kAhead][M] = c.W[M * npts + on];
          w[M] = wq[0][M];
#pragma unroll
          for (int h = 0; h < kAhead; ++h) wq[h][M] = wq[h + 1][M];
        }
      }
      const T* zt = c.zt + (int64_t)zeta * (1 + 3 * NM) * R;  // S_z, then per M': Z, T+, T- taps
      T out[NM];
#pragma unroll
      for (int M = 0; M < NM; ++M) {
        T U = zt[0] * P[M][0];
#pragma unroll
        for (int t = 1; t < R; ++t) U = fma(zt[t], P[M][t], U);
        if (a.only_S) {
          out[M] = U;
          continue;
        }
        const T* zm = zt + (1 + 3 * M) * R;
        T L = (T)0, D = (T)0;
#pragma unroll
        for (int t = 0; t < R; ++t) {
          L = fma(zm[t], P[M][t], L);
          D = fma(zt[t], Q[M][t], D);
        }
        T v = fma(w[M] - a.E, U, fma(q, L, -D));
        if (NM > 1) {
          T e = (T)0;
          if (M + 1 < NM) {
#pragma unroll
            for (int t = 0; t < R; ++t) e = fma(zm[R + t], P[M + 1 < NM ? M + 1 : M][t], e);
          }
          if (M > 0) {
#pragma unroll
            for (int t = 0; t < R; ++t) e = fma(zm[2 * R + t], P[M > 0 ? M - 1 : M][t], e);
          }
          v = fma(iy2, e, v);
        }
        out[M] = v;
      }
      if (live) {
#pragma unroll
        for (int M = 0; M < NM; ++M) c.y[M * npts + o] = out[M];
      }
    }
    ++m;
  }
}

// The two-pass form: float64 (bound by its pipe, so what counts is an even spread of the work: k_apply_local's
// tiles and z chunks cost 5 .. 25 % of it on grids that do not fill them) and n_M beyond the instantiations of
// k_apply_local.
// Pass 1: for one (component, M', z-dof k) plane c[i][j] and a tile of 16 x 32 points, the planes
// P = (S_x (x) S_y) c and Q = (D2_x (x) S_y + S_x (x) D2_y) c.
constexpr int kPX = 16, kPY = 32;
template <typename T>
struct PlaneComp {
  const T* x;
  T *P, *Q, *y;
  const T *W, *Sx, *D2x, *Sy, *D2y, *zt, *qx, *iy2;
  const int *bx, *by, *bz;
  int nx, ny, nz, rows, cols, tiles_x, tiles_y;
  int first_xy, first_z;     // first blocks of the component in the two passes
};
template <typename T>
struct PlaneArgs {
  PlaneComp<T> c[3];
  int ncomp, nM;
  T E;
  int only_S;
};

template <int R, typename T>
__global__ void __launch_bounds__(256) k_apply_xy(const __grid_constant__ PlaneArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smraw_xy[];
  int ci = 0;
  while (ci + 1 < a.ncomp && (int)blockIdx.x >= a.c[ci + 1].first_xy) ++ci;
  const PlaneComp<T>& c = a.c[ci];
  const int rows = c.rows, ld = c.cols + 1;
  T* cs = reinterpret_cast<T*>(smraw_xy);  // [rows][ld]
  T* As = cs + rows * ld;                  // [rows][kPY]  S_y c
  T* Bs = As + rows * kPY;                 //              D2_y c
  const int tiles = c.tiles_x * c.tiles_y, b = (int)blockIdx.x - c.first_xy, pl = b / tiles, tile = b - pl * tiles;
  const int64_t plane = (int64_t)pl * c.nx * c.ny;
  const int xi0 = (tile / c.tiles_y) * kPX, eta0 = (tile % c.tiles_y) * kPY;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int eta = eta0 + lane, ec = min(eta, c.ny - 1);
  const int r0 = c.bx[xi0], c0 = c.by[eta0], lc = c.by[ec] - c0;
  for (int rr = warp; rr < rows; rr += 8) {
    const int r = r0 + rr;
    for (int cc = lane; cc < c.cols; cc += 32) {
      const int col = c0 + cc;
      cs[rr * ld + cc] = (r >= 0 && r < c.nx && col >= 0 && col < c.ny) ? c.x[plane + (int64_t)r * c.ny + col] : (T)0;
    }
  }
  T sy[R], dy[R];
#pragma unroll
  for (int t = 0; t < R; ++t) {
    sy[t] = c.Sy[ec * R + t];
    dy[t] = c.D2y[ec * R + t];
  }
  __syncthreads();
  const int last = min(rows, c.bx[min(xi0 + kPX, c.nx) - 1] + R - r0);  // rows the tile's points read
  for (int rr = warp; rr < last; rr += 8) {
    const T* v = cs + rr * ld + lc;
    T s = sy[0] * v[0], d = dy[0] * v[0];
#pragma unroll
    for (int t = 1; t < R; ++t) {
      s = fma(sy[t], v[t], s);
      d = fma(dy[t], v[t], d);
    }
    As[rr * kPY + lane] = s;
    Bs[rr * kPY + lane] = d;
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < kPX / 8; ++h) {
    const int xi = xi0 + warp + 8 * h;
    if (xi >= c.nx) break;
    const int lr = c.bx[xi] - r0;
    T p = 0, q = 0;
#pragma unroll
    for (int t = 0; t < R; ++t) {
      const T av = As[(lr + t) * kPY + lane], sx = c.Sx[xi * R + t];
      p = fma(sx, av, p);
      q = fma(c.D2x[xi * R + t], av, fma(sx, Bs[(lr + t) * kPY + lane], q));
    }
    if (eta < c.ny) {
      const int64_t o = plane + (int64_t)xi * c.ny + eta;
      c.P[o] = p;
      if (!a.only_S) c.Q[o] = q;
    }
  }
}

// Pass 2: one thread per output point (M', zeta, xi, eta) (R taps in z).
template <int R, typename T>
__global__ void __launch_bounds__(256) k_apply_z(const __grid_constant__ PlaneArgs<T> a) {
  int ci = 0;
  while (ci + 1 < a.ncomp && (int)blockIdx.x >= a.c[ci + 1].first_z) ++ci;
  const PlaneComp<T>& c = a.c[ci];
  const int nxy = c.nx * c.ny, chunks = (nxy + 255) / 256, b = (int)blockIdx.x - c.first_z;
  const int pl = b / chunks, iM = pl / c.nz, zeta = pl - iM * c.nz;
  const int xy = (b - pl * chunks) * 256 + threadIdx.x;
  if (xy >= nxy) return;
  const int64_t npts = (int64_t)c.nz * nxy;
  const T* zt = c.zt + (int64_t)zeta * (1 + 3 * a.nM) * R;
  const T* zm = zt + (1 + 3 * iM) * R;
  const int64_t o = (int64_t)iM * npts + (int64_t)c.bz[zeta] * nxy + xy;  // the z basis keeps all its functions
  const int64_t out = (int64_t)pl * nxy + xy;
  T U = 0, L = 0, D = 0, e = 0;
  if (a.only_S) {
#pragma unroll
    for (int t = 0; t < R; ++t) U = fma(zt[t], c.P[o + (int64_t)t * nxy], U);
    c.y[out] = U;
    return;
  }
  const T w = c.W[out];
#pragma unroll
  for (int t = 0; t < R; ++t) {
    const T p = c.P[o + (int64_t)t * nxy];
    U = fma(zt[t], p, U);
    L = fma(zm[t], p, L);
    D = fma(zt[t], c.Q[o + (int64_t)t * nxy], D);
  }
  if (iM + 1 < a.nM) {
#pragma unroll
    for (int t = 0; t < R; ++t) e = fma(zm[R + t], c.P[o + npts + (int64_t)t * nxy], e);
  }
  if (iM >= 1) {
#pragma unroll
    for (int t = 0; t < R; ++t) e = fma(zm[2 * R + t], c.P[o - npts + (int64_t)t * nxy], e);
  }
  const int ix = xy / c.ny;
  const T iy2 = c.iy2[xy - ix * c.ny], q = c.qx[ix] + iy2;
  T v = fma(w - a.E, U, fma(q, L, -D));
  if (a.nM > 1) v = fma(iy2, e, v);
  c.y[out] = v;
}

// ---------------------------------------------------------------------------
// preconditioner: z mode product  out[l][p] = sum_k W[l][k] in[k][p] for one (component, M').
// A CTA stages W (n_z x n_z) and an n_z x 128 column tile of the input in shared memory;
// each thread produces the n_z outputs of its column.
// ---------------------------------------------------------------------------
template <typename TI, typename TO, typename TW>
__global__ void __launch_bounds__(128) k_zmix(const TW* __restrict__ Wall, const TI* __restrict__ in,
                                              TO* __restrict__ out, int nz, int64_t nxy, int64_t comp_off) {
  extern __shared__ unsigned char smraw[];
  TW* Ws = reinterpret_cast<TW*>(smraw);  // [nz][nz]
  TW* Vs = Ws + nz * nz;                  // [nz][128]
  const int iM = blockIdx.y;
  const TW* W = Wall + (int64_t)iM * nz * nz;
  for (int i = threadIdx.x; i < nz * nz; i += blockDim.x) Ws[i] = W[i];
  const int64_t p0 = (int64_t)blockIdx.x * 128;
  const int64_t base = comp_off + (int64_t)iM * nz * nxy + p0;
  const int cols = (int)min((int64_t)128, nxy - p0);
  for (int k = 0; k < nz; ++k)
    Vs[k * 128 + threadIdx.x] = (threadIdx.x < cols) ? (TW)in[base + (int64_t)k * nxy + threadIdx.x] : (TW)0;
  __syncthreads();
  if ((int)threadIdx.x >= cols) return;
  constexpr int CH = 10;
  for (int l0 = 0; l0 < nz; l0 += CH) {
    TW acc[CH];
#pragma unroll
    for (int u = 0; u < CH; ++u) acc[u] = 0;
    for (int k = 0; k < nz; ++k) {
      const TW v = Vs[k * 128 + threadIdx.x];
#pragma unroll
      for (int u = 0; u < CH; ++u)
        if (l0 + u < nz) acc[u] = fma(Ws[(l0 + u) * nz + k], v, acc[u]);
    }
#pragma unroll
    for (int u = 0; u < CH; ++u)
      if (l0 + u < nz) out[base + (int64_t)(l0 + u) * nxy + threadIdx.x] = (TO)acc[u];
  }
}

// Mode product on every (M', z-mode) slab of a component, slab l = M' + k:
//   out[r][c] = sum_r' W^{l}[r][r'] in[r'][c]   (R x R matrix per l, slabs of R x C)
// x stage: R = n_x, C = n_y; y stage on transposed slabs: R = n_y, C = n_x.  TIN / TOUT read /
// write the slab transposed ([c][r]); SCALE divides the result by lamR[l][r] + lamC[l][c]
// (the diagonal of the tensor-trick inverse).  64x64 output tiles, 256 threads, 4x4 outputs per
// thread, K in steps of 16.
template <typename T, bool TIN, bool TOUT, bool SCALE>
__global__ void __launch_bounds__(256) k_mix(const T* __restrict__ Wall, const T* __restrict__ in, T* __restrict__ out,
                                             int R, int C, int nz, int64_t comp_off, int M0,
                                             const T* __restrict__ lamR, const T* __restrict__ lamC) {
  constexpr int BT = 64, BK = 16;
  __shared__ T smem[BT * (BT + 1) > 2 * BK * (BT + 1) ? BT * (BT + 1) : 2 * BK * (BT + 1)];
  T (*As)[BT + 1] = reinterpret_cast<T (*)[BT + 1]>(smem);
  T (*Bs)[BT + 1] = reinterpret_cast<T (*)[BT + 1]>(smem + BK * (BT + 1));
  const int slab = blockIdx.z;  // iM * nz + k
  const int iM = slab / nz, k = slab % nz;
  const int il = iM + k;        // l - M0
  const T* W = Wall + (int64_t)il * R * R;
  const int64_t so = comp_off + (int64_t)slab * R * C;
  const int row0 = blockIdx.y * BT, col0 = blockIdx.x * BT;
  const int tr = threadIdx.x / 16, tc = threadIdx.x % 16;
  T acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0;
  for (int k0 = 0; k0 < R; k0 += BK) {
    for (int e = threadIdx.x; e < BK * BT; e += 256) {
      const int kk = e % BK, rr = e / BK;  // A tile: W[row0+rr][k0+kk]
      const int gr = row0 + rr, gk = k0 + kk;
      As[kk][rr] = (gr < R && gk < R) ? W[(int64_t)gr * R + gk] : (T)0;
      if (TIN) {  // in stored [c][r']: consecutive threads walk r'
        const int kb = e % BK, cc = e / BK;
        const int gk2 = k0 + kb, gc = col0 + cc;
        Bs[kb][cc] = (gk2 < R && gc < C) ? in[so + (int64_t)gc * R + gk2] : (T)0;
      } else {
        const int cc = e % BT, kb = e / BT;
        const int gk2 = k0 + kb, gc = col0 + cc;
        Bs[kb][cc] = (gk2 < R && gc < C) ? in[so + (int64_t)gk2 * C + gc] : (T)0;
      }
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      T a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][tr + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tc + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
  if (SCALE) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int gr = row0 + tr + 16 * i, gc = col0 + tc + 16 * j;
        if (gr < R && gc < C) acc[i][j] = acc[i][j] / (lamR[(int64_t)il * R + gr] + lamC[(int64_t)il * C + gc]);
      }
  }
  if (!TOUT) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int gr = row0 + tr + 16 * i, gc = col0 + tc + 16 * j;
        if (gr < R && gc < C) out[so + (int64_t)gr * C + gc] = acc[i][j];
      }
  } else {  // stage the tile, then store [c][r] with consecutive threads along r
    T (*Cs)[BT + 1] = reinterpret_cast<T (*)[BT + 1]>(smem);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) Cs[tc + 16 * j][tr + 16 * i] = acc[i][j];
    __syncthreads();
    for (int e = threadIdx.x; e < BT * BT; e += 256) {
      const int rr = e % BT, cc = e / BT;
      const int gr = row0 + rr, gc = col0 + cc;
      if (gr < R && gc < C) out[so + (int64_t)gc * R + gr] = Cs[cc][rr];
    }
  }
}

// ---------------------------------------------------------------------------
// Krylov helpers
// ---------------------------------------------------------------------------
// A warp's float64 instruction holds the SM's FP64 pipe for 16 cycles, so what a reduction costs is its adds
// and how many SMs share them.  With 608 blocks of 256 threads, a shuffle tree per vector and the last block's
// partial sums added by few warps, the tail of a multi-dot took 10 us per eight vectors and the update's last
// block (2432 partial sums in one warp) 19 us: 49 and 26 us a launch on vectors of 83 k elements, 16 vectors.
constexpr int kRedThreads = 512;
constexpr int kGsMaxVec = 264;  // basis vectors one Gram-Schmidt pass takes (restart length <= 256)
// gsd layout: [0, kGsMaxVec) first-pass coefficients, [kGsMaxVec, 2 kGsMaxVec) second pass, [3 kGsMaxVec, +4)
// scalars, [kGsFlag] the tensor-core kernels' wait flag (an int), read back with every Gram-Schmidt result
constexpr int kGsFlag = 3 * kGsMaxVec + 8;
constexpr int kGsRead = kGsFlag + 1;

__device__ __forceinline__ double block_sum(double v, double* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) r += sh[i];
  __syncthreads();
  return r;
}

// Called by every thread of every block at the end of a reduction kernel, after each block has
// written its partial[j * nb + b] (j < nv, nb = gridDim.x): the block that arrives last sums the
// partials in a fixed order (lane-strided, then a shuffle tree) into out[j] and resets the
// counter, so the reduction needs neither a second kernel nor a host round trip.
__device__ void last_block_reduce(const double* partial, int nv, unsigned* counter, double* out) {
  __shared__ unsigned ticket;
  const int nb = (int)gridDim.x;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) ticket = atomicAdd(counter, 1u);
  __syncthreads();
  if (ticket != gridDim.x * gridDim.y - 1u) return;
  __threadfence();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
  for (int j = wid; j < nv; j += nw) {
    const double* pj = partial + (int64_t)j * nb;
    double s = 0.0;
    int b = lane;
    for (; b + 96 < nb; b += 128) {  // four loads in flight
      const double p0 = __ldcg(&pj[b]), p1 = __ldcg(&pj[b + 32]), p2 = __ldcg(&pj[b + 64]), p3 = __ldcg(&pj[b + 96]);
      s += (p0 + p1) + (p2 + p3);
    }
    for (; b < nb; b += 32) s += __ldcg(&pj[b]);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) out[j] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0) *counter = 0u;
}

__device__ __forceinline__ double lane_xor(double v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }
__device__ __forceinline__ fmi::dd lane_xor(fmi::dd v, int m) {
  return fmi::dd(__shfl_xor_sync(0xffffffffu, v.hi, m), __shfl_xor_sync(0xffffffffu, v.lo, m));
}
__device__ __forceinline__ double wide(double v) { return v; }
__device__ __forceinline__ double wide(fmi::dd v) { return (double)v.hi + (double)v.lo; }

// Sums eight values over the warp's lanes, each lane keeping half of its values at every exchange: nine adds
// instead of the 40 of eight shuffle trees.  Lane 4 u (in the bit order below) returns the sum of v[u].
// S: double, or pairs of floats (48 bits) for float32 sums: twenty instructions of the FP32 pipe an add, where a
// conversion or an add in float64 holds its pipe as long as 64 of them.
template <typename S>
__device__ __forceinline__ S warp_sum8(S (&v)[8], int lane) {
#pragma unroll
  for (int h = 4; h >= 1; h >>= 1) {
    const bool up = (lane & (4 * h)) != 0;
#pragma unroll
    for (int u = 0; u < h; ++u) {
      const S send = up ? v[u] : v[u + h];
      const S keep = up ? v[u + h] : v[u];
      v[u] = keep + lane_xor(send, 4 * h);
    }
  }
  v[0] += lane_xor(v[0], 2);
  v[0] += lane_xor(v[0], 1);
  return v[0];  // of vector lane >> 2
}

// |c|^2 of a coefficient vector, by the 32 lanes of one warp (the sum is lane 0's)
__device__ __forceinline__ double warp_norm2(const double* c, int n, int lane) {
  double s = 0.0;
  for (int j = lane; j < n; j += 32) s = fma(c[j], c[j], s);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  return s;
}

// The block's sums of eight vectors from its threads' values, added in warp order: thread j < nj writes out[j * ldo].
template <typename S>
__device__ __forceinline__ void block_sum8(S (&v)[8], int nj, double (*sh)[kRedThreads / 32], double* out, int64_t ldo) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const S s = warp_sum8(v, lane);
  if ((lane & 3) == 0) sh[lane >> 2][wid] = wide(s);
  __syncthreads();
  if ((int)threadIdx.x < nj) {
    double r = 0.0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) r += sh[threadIdx.x][q];
    out[(int64_t)threadIdx.x * ldo] = r;
  }
  __syncthreads();
}

// The float with the sign, the exponent and the 20 leading mantissa bits of a double (truncated;
// 0 below the float range), built with integer operations so that no FP64 instruction is issued.
__device__ __forceinline__ float f64_lead_f32(double d) {
  const unsigned hi = (unsigned)((unsigned long long)__double_as_longlong(d) >> 32);
  const unsigned fe = ((hi >> 20) & 0x7FFu) - 896u;  // float exponent (wraps below the float range)
  const unsigned sign = hi & 0x80000000u;
  return __uint_as_float((fe - 1u < 254u) ? (sign | (fe << 23) | ((hi & 0xFFFFFu) << 3)) : sign);
}

// a float64 value truncated to float32 by integer operations (1 + 23 significand bits; relative error < 2^-23),
// without the FP64 pipe; values outside float32's normal range become signed zero
__device__ __forceinline__ float f64_trunc_f32(double d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
  const unsigned fe = ((hi >> 20) & 0x7FFu) - 896u;  // float exponent (wraps below the float range)
  const unsigned sign = hi & 0x80000000u;
  const unsigned mant = ((hi & 0xFFFFFu) << 3) | (lo >> 29);
  return __uint_as_float((fe - 1u < 254u) ? (sign | (fe << 23) | mant) : sign);
}

// partial[j][block] = sum over this block's slice of V[j] . w  (j < nv), and for j = nv, when
// 'extra' is given, extra . w; the last block reduces the partials into out[j].  The vectors are read
// as 16-byte element pairs (n even, 16-byte aligned vectors), eight vectors and two pairs per thread
// and iteration with every load issued before the FMAs, so that a thread keeps 18 loads of 16 bytes
// in flight: the kernel is bound by memory latency otherwise.
// LOWP: products and per-thread sums in float32 from the leading bits of the operands (relative
// accuracy about 1e-6 of sum |V_j| |w|), for the first Gram-Schmidt pass only.
__device__ __forceinline__ double dot2(double2 a, double2 b, double acc) { return fma(a.y, b.y, fma(a.x, b.x, acc)); }
__device__ __forceinline__ void dot2f(double2 a, double2 b, float& x, float& y) {
  x = fmaf(f64_lead_f32(a.x), f64_lead_f32(b.x), x);
  y = fmaf(f64_lead_f32(a.y), f64_lead_f32(b.y), y);
}
// four float32 sums as one pair of floats (exact to 48 bits)
__device__ __forceinline__ fmi::dd sum4f(float a, float b, float c, float d) {
  return (fmi::dd(a, 0.f) + fmi::dd(b, 0.f)) + (fmi::dd(c, 0.f) + fmi::dd(d, 0.f));
}

template <bool LOWP>
__global__ void __launch_bounds__(kRedThreads) k_dot_many(const double* __restrict__ V, int64_t ldv, int nv,
                                                         const double* __restrict__ w, int64_t n,
                                                         double* __restrict__ partial, const double* __restrict__ extra,
                                                         unsigned* counter, double* __restrict__ out) {
  constexpr int JT = 8;
  __shared__ double sh[JT][kRedThreads / 32];
  const int64_t npair = n / 2;
  const int64_t chunk = (npair + gridDim.x - 1) / gridDim.x;
  const int64_t lo = (int64_t)blockIdx.x * chunk;
  const int64_t hi = min(npair, lo + chunk);
  const int nt = nv + (extra ? 1 : 0);
  const double2* w2 = reinterpret_cast<const double2*>(w);
  const int64_t bs = blockDim.x;
  for (int j0 = (int)blockIdx.y * JT; j0 < nt; j0 += JT * (int)gridDim.y) {
    const int nj = min(JT, nt - j0);
    const double2* vp[JT];
#pragma unroll
    for (int u = 0; u < JT; ++u) {
      const int j = j0 + min(u, nj - 1);
      vp[u] = reinterpret_cast<const double2*>((j < nv) ? V + (int64_t)j * ldv : extra);
    }
    double acc[JT];
    float accf[4][JT];
#pragma unroll
    for (int u = 0; u < JT; ++u) {
      acc[u] = 0.0;
      accf[0][u] = accf[1][u] = accf[2][u] = accf[3][u] = 0.f;
    }
    int64_t p = lo + threadIdx.x;
    for (; p + bs < hi; p += 2 * bs) {
      const double2 wa = w2[p], wb = w2[p + bs];
      double2 va[JT], vb[JT];
#pragma unroll
      for (int u = 0; u < JT; ++u)
        if (u < nj) {
          va[u] = vp[u][p];
          vb[u] = vp[u][p + bs];
        }
#pragma unroll
      for (int u = 0; u < JT; ++u)
        if (u < nj) {
          if (LOWP) {
            dot2f(va[u], wa, accf[0][u], accf[1][u]);
            dot2f(vb[u], wb, accf[2][u], accf[3][u]);
          } else {
            acc[u] = dot2(vb[u], wb, dot2(va[u], wa, acc[u]));
          }
        }
    }
    for (; p < hi; p += bs) {
      const double2 wa = w2[p];
#pragma unroll
      for (int u = 0; u < JT; ++u)
        if (u < nj) {
          if (LOWP) dot2f(vp[u][p], wa, accf[0][u], accf[1][u]);
          else acc[u] = dot2(vp[u][p], wa, acc[u]);
        }
    }
    if ((n & 1) && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {  // odd length: the last element
      const int64_t e = n - 1;
#pragma unroll
      for (int u = 0; u < JT; ++u)
        if (u < nj) {
          const double* vv = reinterpret_cast<const double*>(vp[u]);
          if (LOWP) accf[3][u] = fmaf(f64_lead_f32(vv[e]), f64_lead_f32(w[e]), accf[3][u]);
          else acc[u] = fma(vv[e], w[e], acc[u]);
        }
    }
    double* out8 = partial + (int64_t)j0 * gridDim.x + blockIdx.x;
    if constexpr (LOWP) {
      fmi::dd both[JT];
#pragma unroll
      for (int u = 0; u < JT; ++u) both[u] = sum4f(accf[0][u], accf[1][u], accf[2][u], accf[3][u]);
      block_sum8(both, nj, sh, out8, gridDim.x);
    } else {
      block_sum8(acc, nj, sh, out8, gridDim.x);
    }
  }
  last_block_reduce(partial, nt, counter, out);
}

// k_dot_many with scalar loads: for vectors that do not all start on 16-byte boundaries (odd strides)
template <bool LOWP>
__global__ void __launch_bounds__(kRedThreads) k_dot_many_s(const double* __restrict__ V, int64_t ldv, int nv,
                                                           const double* __restrict__ w, int64_t n,
                                                           double* __restrict__ partial, const double* __restrict__ extra,
                                                           unsigned* counter, double* __restrict__ out) {
  constexpr int JT = 8;
  __shared__ double sh[JT][kRedThreads / 32];
  const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const int64_t lo = (int64_t)blockIdx.x * chunk;
  const int64_t hi = min(n, lo + chunk);
  const int nt = nv + (extra ? 1 : 0);
  for (int j0 = (int)blockIdx.y * JT; j0 < nt; j0 += JT * (int)gridDim.y) {
    const int nj = min(JT, nt - j0);
    const double* vp[JT];
#pragma unroll
    for (int u = 0; u < JT; ++u) {
      const int j = j0 + min(u, nj - 1);
      vp[u] = (j < nv) ? V + (int64_t)j * ldv : extra;
    }
    double acc[JT];
    float accf[4][JT];
#pragma unroll
    for (int u = 0; u < JT; ++u) {
      acc[u] = 0.0;
      accf[0][u] = accf[1][u] = accf[2][u] = accf[3][u] = 0.f;
    }
    const int64_t bs = blockDim.x;
    for (int64_t i = lo + threadIdx.x; i < hi; i += 4 * bs) {
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        if (i + t * bs >= hi) break;
        const double wi = w[i + t * bs];
#pragma unroll
        for (int u = 0; u < JT; ++u)
          if (u < nj) {
            if (LOWP) accf[t][u] = fmaf(f64_lead_f32(vp[u][i + t * bs]), f64_lead_f32(wi), accf[t][u]);
            else acc[u] = fma(vp[u][i + t * bs], wi, acc[u]);
          }
      }
    }
    double* out8 = partial + (int64_t)j0 * gridDim.x + blockIdx.x;
    if constexpr (LOWP) {
      fmi::dd both[JT];
#pragma unroll
      for (int u = 0; u < JT; ++u) both[u] = sum4f(accf[0][u], accf[1][u], accf[2][u], accf[3][u]);
      block_sum8(both, nj, sh, out8, gridDim.x);
    } else {
      block_sum8(acc, nj, sh, out8, gridDim.x);
    }
  }
  last_block_reduce(partial, nt, counter, out);
}

// float32 vectors: partial[j][block] (float64) = V[j] . w over the block's slice (eight vectors per pass)
__global__ void __launch_bounds__(kRedThreads) k_dot_many32(const float* __restrict__ V, int64_t ldv, int nv,
                                                           const float* __restrict__ w, int64_t n,
                                                           double* __restrict__ partial, unsigned* counter,
                                                           double* __restrict__ out) {
  constexpr int JT = 8;
  __shared__ double sh[JT][kRedThreads / 32];
  const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const int64_t lo = (int64_t)blockIdx.x * chunk;
  const int64_t hi = min(n, lo + chunk);
  for (int j0 = (int)blockIdx.y * JT; j0 < nv; j0 += JT * (int)gridDim.y) {
    const int nj = min(JT, nv - j0);
    float acc[4][JT];
#pragma unroll
    for (int u = 0; u < JT; ++u) acc[0][u] = acc[1][u] = acc[2][u] = acc[3][u] = 0.0f;
    const int64_t bs = blockDim.x;
    for (int64_t i = lo + threadIdx.x; i < hi; i += 4 * bs) {
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        if (i + t * bs >= hi) break;
        const float wi = w[i + t * bs];
#pragma unroll
        for (int u = 0; u < JT; ++u)
          if (u < nj) acc[t][u] = fmaf(V[(int64_t)(j0 + u) * ldv + i + t * bs], wi, acc[t][u]);
      }
    }
    fmi::dd accd[JT];
#pragma unroll
    for (int u = 0; u < JT; ++u) accd[u] = sum4f(acc[0][u], acc[1][u], acc[2][u], acc[3][u]);
    block_sum8(accd, nj, sh, partial + (int64_t)j0 * gridDim.x + blockIdx.x, gridDim.x);
  }
  last_block_reduce(partial, nv, counter, out);
}

// float32: w += sign * sum_j h[j] V[j]; with 'out', partial[block] = sum of the new w^2 (float64)
__global__ void __launch_bounds__(kRedThreads) k_axpy_many_norm32(const float* __restrict__ V, int64_t ldv, int nv,
                                                                 const float* __restrict__ h, float sign,
                                                                 float* __restrict__ w, int64_t n,
                                                                 double* __restrict__ partial, unsigned* counter,
                                                                 double* __restrict__ out) {
  __shared__ double sh[32];
  double acc = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f, s3 = 0.0f;
    int j = 0;
    for (; j + 3 < nv; j += 4) {
      s0 = fmaf(h[j], V[(int64_t)j * ldv + i], s0);
      s1 = fmaf(h[j + 1], V[(int64_t)(j + 1) * ldv + i], s1);
      s2 = fmaf(h[j + 2], V[(int64_t)(j + 2) * ldv + i], s2);
      s3 = fmaf(h[j + 3], V[(int64_t)(j + 3) * ldv + i], s3);
    }
    for (; j < nv; ++j) s0 = fmaf(h[j], V[(int64_t)j * ldv + i], s0);
    const float v = fmaf(sign, (s0 + s1) + (s2 + s3), w[i]);
    w[i] = v;
    if (out) acc = fma((double)v, (double)v, acc);
  }
  if (!out) return;
  const double a = block_sum(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = a;
  last_block_reduce(partial, 1, counter, out);
}

// y32 = (float)(a * x64)
__global__ void k_to32(const double* __restrict__ x, double a, float* __restrict__ y, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = (float)(a * x[i]);
}

// x64 += a * (double)y32
__global__ void k_add32(const float* __restrict__ y, double a, double* __restrict__ x, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    x[i] = fma(a, (double)y[i], x[i]);
}

// float32 y = a x + b y
__global__ void k_axpby32(float a, const float* __restrict__ x, float b, float* __restrict__ y, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = a * x[i] + (b == 0.0f ? 0.0f : b * y[i]);
}

// One pass of classical Gram-Schmidt with the coefficients on the device:
//   w' = w - sum_j c_j V_j,  c = h, or c = G a (G k x k row-major, a of length k) when G is given.
// MODE 0: w <- w', out[0] = ||w'||^2.
// MODE 1 (closing pass): nu^2 = nrm2_prev - |c|^2 (the norm of w' by Pythagoras, V orthonormal and
// c = V^T w), vout <- w' / nu (0 when nu^2 <= 0), out[0] = ||vout||^2 (1 up to rounding), out[1] = nu.
// MODE 2 (single pass with the DGKS test): as MODE 1 when nu^2 >= nrm2_prev / 2 (little cancellation: one
// float64 projection is enough), out[2] = 0; otherwise as MODE 0 (w <- w', out[0] = ||w'||^2) with
// out[2] = 1, and the caller re-orthogonalises.  Every block takes the same decision from the same values.
// PAIRS: the vectors are read as 16-byte element pairs (every vector on a 16-byte boundary).
template <int MODE, bool PAIRS>
__global__ void __launch_bounds__(kRedThreads, 2) k_gs_axpy(const double* __restrict__ V, int64_t ldv, int nv,
                                                        const double* __restrict__ h, const double* __restrict__ G,
                                                        const double* __restrict__ a, double* w, double* vout,
                                                        int64_t n, double* __restrict__ partial, unsigned* counter,
                                                        double* __restrict__ out, const double* __restrict__ nrm2_prev) {
  __shared__ double cs[kGsMaxVec];
  __shared__ double sh[32];
  __shared__ double inv_nu;
  __shared__ int reorth;
  __shared__ int corr32;
  for (int j = threadIdx.x; j < nv; j += blockDim.x) {
    double cj;
    if (G) {
      cj = 0.0;
      for (int q = 0; q < nv; ++q) cj = fma(G[(int64_t)j * nv + q], a[q], cj);
    } else {
      cj = h[j];
    }
    cs[j] = cj;
  }
  __syncthreads();
  if (MODE >= 1 && threadIdx.x < 32) {
    const double c2 = warp_norm2(cs, nv, threadIdx.x);
    if (threadIdx.x == 0) {
      const double nu2 = *nrm2_prev - c2;
      const double nu = nu2 > 0.0 ? sqrt(nu2) : 0.0;
      inv_nu = nu > 0.0 ? 1.0 / nu : 0.0;
      reorth = (MODE == 2 && !(nu2 >= 0.5 * *nrm2_prev)) ? 1 : 0;
      // closing update on the FP32 pipe only while |h| <= 1e-5 |w'| (its float32 error, ~1e-7 |V h|, then stays
      // below 1e-12 |w'|); with heavier cancellation the float64 path below
      corr32 = (MODE == 1 && c2 <= 1e-10 * *nrm2_prev) ? 1 : 0;
      if (blockIdx.x == 0) {
        out[1] = nu;
        if (MODE == 2) out[2] = (double)reorth;
      }
    }
  }
  __syncthreads();
  const bool write_w = MODE == 0 || (MODE == 2 && reorth);
  double acc = 0.0;
  if (MODE == 1 && corr32) {
    // the closing update of CGS2: its coefficients are the second projection, of relative size ~1e-6 (the
    // error of the first, FP32-pipe projection), so V h is summed on the FP32 pipe from 24-bit truncations
    // (error ~1e-7 of a term <= 1e-5 |w'|) and only w - corr, the scaling and the norm run in float64
    __shared__ float csf[kGsMaxVec];
    for (int j = threadIdx.x; j < nv; j += blockDim.x) csf[j] = (float)cs[j];
    __syncthreads();
    const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, st = (int64_t)gridDim.x * blockDim.x;
    int64_t tail = 0;
    if (PAIRS) {
      const int64_t npair = n / 2, ldp = ldv / 2;
      tail = 2 * npair;
      const double2* V2 = reinterpret_cast<const double2*>(V);
      for (int64_t p = i0; p < npair; p += st) {
        float ca = 0.f, cb = 0.f, ca1 = 0.f, cb1 = 0.f;  // even and odd basis vectors
        int j = 0;
        for (; j + 7 < nv; j += 8) {
          double2 t[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) t[u] = V2[(int64_t)(j + u) * ldp + p];
#pragma unroll
          for (int u = 0; u < 8; u += 2) {
            ca = fmaf(csf[j + u], f64_trunc_f32(t[u].x), ca);
            cb = fmaf(csf[j + u], f64_trunc_f32(t[u].y), cb);
            ca1 = fmaf(csf[j + u + 1], f64_trunc_f32(t[u + 1].x), ca1);
            cb1 = fmaf(csf[j + u + 1], f64_trunc_f32(t[u + 1].y), cb1);
          }
        }
        for (; j < nv; ++j) {
          const double2 t = V2[(int64_t)j * ldp + p];
          ca = fmaf(csf[j], f64_trunc_f32(t.x), ca);
          cb = fmaf(csf[j], f64_trunc_f32(t.y), cb);
        }
        const double2 wp = reinterpret_cast<const double2*>(w)[p];
        const double oa = (wp.x - (double)(ca + ca1)) * inv_nu, ob = (wp.y - (double)(cb + cb1)) * inv_nu;
        reinterpret_cast<double2*>(vout)[p] = make_double2(oa, ob);
        acc = fma(ob, ob, fma(oa, oa, acc));
      }
    }
    for (int64_t i = tail + i0; i < n; i += st) {
      float c0 = 0.f, c1 = 0.f;
      int j = 0;
      for (; j + 1 < nv; j += 2) {
        c0 = fmaf(csf[j], f64_trunc_f32(V[(int64_t)j * ldv + i]), c0);
        c1 = fmaf(csf[j + 1], f64_trunc_f32(V[(int64_t)(j + 1) * ldv + i]), c1);
      }
      if (j < nv) c0 = fmaf(csf[j], f64_trunc_f32(V[(int64_t)j * ldv + i]), c0);
      const double o = (w[i] - (double)(c0 + c1)) * inv_nu;
      vout[i] = o;
      acc = fma(o, o, acc);
    }
    acc = block_sum(acc, sh);
    if (threadIdx.x == 0) partial[blockIdx.x] = acc;
    last_block_reduce(partial, 1, counter, out);
    return;
  }
  // one FMA per basis vector and element on a single chain (no partial sums to add: FP64 issue is the bound);
  // eight 16-byte loads ahead of their FMAs
  const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, st = (int64_t)gridDim.x * blockDim.x;
  int64_t tail = 0;
  if (PAIRS) {
    const int64_t npair = n / 2, ldp = ldv / 2;
    tail = 2 * npair;
    const double2* V2 = reinterpret_cast<const double2*>(V);
    for (int64_t p = i0; p < npair; p += st) {
      double2 v = reinterpret_cast<const double2*>(w)[p];
      int j = 0;
      for (; j + 7 < nv; j += 8) {
        double2 t[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) t[u] = V2[(int64_t)(j + u) * ldp + p];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          v.x = fma(-cs[j + u], t[u].x, v.x);
          v.y = fma(-cs[j + u], t[u].y, v.y);
        }
      }
      for (; j < nv; ++j) {
        const double2 t = V2[(int64_t)j * ldp + p];
        v.x = fma(-cs[j], t.x, v.x);
        v.y = fma(-cs[j], t.y, v.y);
      }
      if (!write_w) {
        v.x *= inv_nu;
        v.y *= inv_nu;
      }
      reinterpret_cast<double2*>(write_w ? w : vout)[p] = v;
      acc = fma(v.y, v.y, fma(v.x, v.x, acc));
    }
  }
  for (int64_t i = tail + i0; i < n; i += st) {
    double v = w[i];
    for (int j = 0; j < nv; ++j) v = fma(-cs[j], V[(int64_t)j * ldv + i], v);
    if (!write_w) v *= inv_nu;
    (write_w ? w : vout)[i] = v;
    acc = fma(v, v, acc);
  }
  acc = block_sum(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = acc;
  last_block_reduce(partial, 1, counter, out);
}

// float32 counterparts of the Gram-Schmidt kernels (MIXED precision inner solves): vectors of
// float32, coefficients, norms and reductions in float64.
// Multi-dot: partial[j][block] of V[j] . w over 16-byte quads (n a multiple of 4, 16-byte aligned
// vectors), eight vectors and two quads per thread and iteration, loads issued before the FMAs.
// (a quad's products are summed by themselves: fewer roundings than one chain over the quads of a thread)
__device__ __forceinline__ float dot4f(float4 a, float4 b, float acc) {
  return acc + (fmaf(a.y, b.y, a.x * b.x) + fmaf(a.w, b.w, a.z * b.z));
}

__global__ void __launch_bounds__(kRedThreads) k_dot_many32v(const float* __restrict__ V, int64_t ldv, int nv,
                                                            const float* __restrict__ w, int64_t n,
                                                            double* __restrict__ partial, unsigned* counter,
                                                            double* __restrict__ out) {
  constexpr int JT = 8;
  __shared__ double sh[JT][kRedThreads / 32];
  const int64_t nq = n / 4;
  const int64_t chunk = (nq + gridDim.x - 1) / gridDim.x;
  const int64_t lo = (int64_t)blockIdx.x * chunk;
  const int64_t hi = min(nq, lo + chunk);
  const float4* w4 = reinterpret_cast<const float4*>(w);
  const int64_t bs = blockDim.x;
  for (int j0 = (int)blockIdx.y * JT; j0 < nv; j0 += JT * (int)gridDim.y) {
    const int nj = min(JT, nv - j0);
    const float4* vp[JT];
#pragma unroll
    for (int u = 0; u < JT; ++u) vp[u] = reinterpret_cast<const float4*>(V + (int64_t)(j0 + min(u, nj - 1)) * ldv);
    float acc[2][JT];
#pragma unroll
    for (int u = 0; u < JT; ++u) acc[0][u] = acc[1][u] = 0.f;
    int64_t p = lo + threadIdx.x;
    for (; p + bs < hi; p += 2 * bs) {
      const float4 wa = w4[p], wb = w4[p + bs];
      float4 va[JT], vb[JT];
#pragma unroll
      for (int u = 0; u < JT; ++u)
        if (u < nj) {
          va[u] = vp[u][p];
          vb[u] = vp[u][p + bs];
        }
#pragma unroll
      for (int u = 0; u < JT; ++u)
        if (u < nj) {
          acc[0][u] = dot4f(va[u], wa, acc[0][u]);
          acc[1][u] = dot4f(vb[u], wb, acc[1][u]);
        }
    }
    for (; p < hi; p += bs) {
      const float4 wa = w4[p];
#pragma unroll
      for (int u = 0; u < JT; ++u)
        if (u < nj) acc[0][u] = dot4f(vp[u][p], wa, acc[0][u]);
    }
    fmi::dd accd[JT];
#pragma unroll
    for (int u = 0; u < JT; ++u) accd[u] = fmi::dd(acc[0][u], 0.f) + fmi::dd(acc[1][u], 0.f);
    block_sum8(accd, nj, sh, partial + (int64_t)j0 * gridDim.x + blockIdx.x, gridDim.x);
  }
  last_block_reduce(partial, nv, counter, out);
}

// w' = w - sum_j h_j V_j (float32, h from the device); MODE 0: w <- w', out[0] = ||w'||^2;
// MODE 1: vout = w' / nu with nu^2 = nrm2_prev - |h|^2, out[0] = ||vout||^2, out[1] = nu.
// QUADS: 16-byte quads (n a multiple of 4, 16-byte aligned vectors), eight in flight per thread.
__device__ __forceinline__ void sub4(float4& v, float c, const float4& t) {
  v.x = fmaf(-c, t.x, v.x);
  v.y = fmaf(-c, t.y, v.y);
  v.z = fmaf(-c, t.z, v.z);
  v.w = fmaf(-c, t.w, v.w);
}

template <int MODE, bool QUADS>
__global__ void __launch_bounds__(kRedThreads, 2) k_gs_axpy32(const float* __restrict__ V, int64_t ldv, int nv,
                                                          const double* __restrict__ h, float* w, float* vout,
                                                          int64_t n, double* __restrict__ partial, unsigned* counter,
                                                          double* __restrict__ out,
                                                          const double* __restrict__ nrm2_prev) {
  __shared__ float cs[kGsMaxVec];
  __shared__ double sh[32];
  __shared__ float inv_nu;
  for (int j = threadIdx.x; j < nv; j += blockDim.x) cs[j] = (float)h[j];
  __syncthreads();
  if (MODE == 1 && threadIdx.x < 32) {
    const double c2 = warp_norm2(h, nv, threadIdx.x);
    if (threadIdx.x == 0) {
      const double nu2 = *nrm2_prev - c2;
      const double nu = nu2 > 0.0 ? sqrt(nu2) : 0.0;
      inv_nu = nu > 0.0 ? (float)(1.0 / nu) : 0.f;
      if (blockIdx.x == 0) out[1] = nu;
    }
  }
  __syncthreads();
  double acc = 0.0;
  const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, st = (int64_t)gridDim.x * blockDim.x;
  if (QUADS) {
    const int64_t nq = n / 4, ldq = ldv / 4;
    const float4* V4 = reinterpret_cast<const float4*>(V);
    for (int64_t p = i0; p < nq; p += st) {
      float4 v = reinterpret_cast<const float4*>(w)[p];
      int j = 0;
      for (; j + 7 < nv; j += 8) {
        float4 t[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) t[u] = V4[(int64_t)(j + u) * ldq + p];
#pragma unroll
        for (int u = 0; u < 8; ++u) sub4(v, cs[j + u], t[u]);
      }
      for (; j < nv; ++j) sub4(v, cs[j], V4[(int64_t)j * ldq + p]);
      if (MODE == 1) v = make_float4(v.x * inv_nu, v.y * inv_nu, v.z * inv_nu, v.w * inv_nu);
      reinterpret_cast<float4*>(MODE == 1 ? vout : w)[p] = v;
      acc = fma((double)v.x, (double)v.x, acc);
      acc = fma((double)v.y, (double)v.y, acc);
      acc = fma((double)v.z, (double)v.z, acc);
      acc = fma((double)v.w, (double)v.w, acc);
    }
  } else {
    for (int64_t i = i0; i < n; i += st) {
      float v = w[i];
      for (int j = 0; j < nv; ++j) v = fmaf(-cs[j], V[(int64_t)j * ldv + i], v);
      if (MODE == 1) v *= inv_nu;
      (MODE == 1 ? vout : w)[i] = v;
      acc = fma((double)v, (double)v, acc);
    }
  }
  acc = block_sum(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = acc;
  last_block_reduce(partial, 1, counter, out);
}

// w += sign * sum_j h[j] V[j]
__global__ void __launch_bounds__(256) k_axpy_many(const double* __restrict__ V, int64_t ldv, int nv,
                                                   const double* __restrict__ h, double sign, double* __restrict__ w,
                                                   int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    int j = 0;
    for (; j + 3 < nv; j += 4) {
      s0 = fma(h[j], V[(int64_t)j * ldv + i], s0);
      s1 = fma(h[j + 1], V[(int64_t)(j + 1) * ldv + i], s1);
      s2 = fma(h[j + 2], V[(int64_t)(j + 2) * ldv + i], s2);
      s3 = fma(h[j + 3], V[(int64_t)(j + 3) * ldv + i], s3);
    }
    for (; j < nv; ++j) s0 = fma(h[j], V[(int64_t)j * ldv + i], s0);
    w[i] = fma(sign, (s0 + s1) + (s2 + s3), w[i]);
  }
}

__global__ void k_axpby(double a, const double* __restrict__ x, double b, double* __restrict__ y, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = a * x[i] + (b == 0.0 ? 0.0 : b * y[i]);
}

// counter-based normal deviates: splitmix64 -> two uniforms -> Box-Muller
__device__ __forceinline__ uint64_t splitmix64(uint64_t z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__global__ void k_fill_normal(double* x, int64_t n, uint64_t seed) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t a = splitmix64(seed ^ (2 * (uint64_t)i)), b = splitmix64(seed ^ (2 * (uint64_t)i + 1));
    const double u1 = ((a >> 11) + 1.0) * (1.0 / 9007199254740993.0);
    const double u2 = (b >> 11) * (1.0 / 9007199254740992.0);
    x[i] = sqrt(-2.0 * log(u1)) * cospi(2.0 * u2);
  }
}

// out[c][i] = sum_j V[j][i] Q[j][c]  (Q row-major nv x nc on the device)
__global__ void __launch_bounds__(256) k_combine(const double* __restrict__ V, int64_t ldv, int nv,
                                                 const double* __restrict__ Qm, int nc, double* __restrict__ out,
                                                 int64_t ldo, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    for (int cc = 0; cc < nc; ++cc) {
      double s = 0.0;
      for (int j = 0; j < nv; ++j) s = fma(V[(int64_t)j * ldv + i], Qm[j * nc + cc], s);
      out[(int64_t)cc * ldo + i] = s;
    }
  }
}

// per block: the entry of largest magnitude (value), first index on ties
__global__ void __launch_bounds__(256) k_absmax(const double* __restrict__ x, int64_t n, double* __restrict__ pval,
                                                long long* __restrict__ pidx) {
  __shared__ double sv[256];
  __shared__ long long si[256];
  double best = 0.0;
  long long bi = -1;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double v = x[i];
    if (bi < 0 || fabs(v) > fabs(best)) { best = v; bi = i; }
  }
  sv[threadIdx.x] = best;
  si[threadIdx.x] = bi;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) {
      const double a = sv[threadIdx.x], b = sv[threadIdx.x + o];
      const long long ia = si[threadIdx.x], ib = si[threadIdx.x + o];
      if (ia < 0 || (ib >= 0 && (fabs(b) > fabs(a) || (fabs(b) == fabs(a) && ib < ia)))) {
        sv[threadIdx.x] = b;
        si[threadIdx.x] = ib;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    pval[blockIdx.x] = sv[0];
    pidx[blockIdx.x] = si[0];
  }
}

// ---------------------------------------------------------------------------
// Double-float Krylov kernels (mixed_scheme 2 inner solves): vectors of dd, reductions summed in dd per
// thread and in float64 across threads (fixed order, deterministic).
// ---------------------------------------------------------------------------
using fmi::dd;

__device__ __forceinline__ double dd_d(dd v) { return (double)v.hi + (double)v.lo; }

// y = dd(a x)
__global__ void k_to_dd(const double* __restrict__ x, double a, dd* __restrict__ y, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = dd(a * x[i]);
}
// x += a y
__global__ void k_add_dd(const dd* __restrict__ y, double a, double* __restrict__ x, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    x[i] = fma(a, dd_d(y[i]), x[i]);
}
// leading parts as float32 (the tensor preconditioner's input), and back (its output, lo = 0)
__global__ void k_dd_hi(const dd* __restrict__ x, float* __restrict__ y, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = x[i].hi;
}
__global__ void k_f_to_dd(const float* __restrict__ x, dd* __restrict__ y, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = dd(x[i], 0.f);
}
// y = a x + b y (y is not read when b = 0)
__global__ void k_axpby_dd(dd a, const dd* x, dd b, bool b_zero, dd* y, int64_t n) {  // x may be y
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = b_zero ? a * x[i] : fma(a, x[i], b * y[i]);
}

// out[j] = V_j . w for j < nv (eight vectors per pass)
__global__ void __launch_bounds__(kRedThreads) k_dot_many_dd(const dd* __restrict__ V, int64_t ldv, int nv,
                                                            const dd* __restrict__ w, int64_t n,
                                                            double* __restrict__ partial, unsigned* counter,
                                                            double* __restrict__ out) {
  constexpr int JT = 8;
  __shared__ double sh[JT][kRedThreads / 32];
  for (int j0 = (int)blockIdx.y * JT; j0 < nv; j0 += JT * (int)gridDim.y) {
    const int nj = min(JT, nv - j0);
    dd acc[JT];
#pragma unroll
    for (int u = 0; u < JT; ++u) acc[u] = dd(0.f, 0.f);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
      const dd wi = w[i];
#pragma unroll
      for (int u = 0; u < JT; ++u)
        if (u < nj) acc[u] = fma(V[(int64_t)(j0 + u) * ldv + i], wi, acc[u]);
    }
    double accd[JT];
#pragma unroll
    for (int u = 0; u < JT; ++u) accd[u] = dd_d(acc[u]);
    block_sum8(accd, nj, sh, partial + (int64_t)j0 * gridDim.x + blockIdx.x, gridDim.x);
  }
  last_block_reduce(partial, nv, counter, out);
}

// w' = w - sum_j h_j V_j in dd (h from the device); MODE 0: w <- w', out[0] = ||w'||^2; MODE 1:
// vout = w' / nu with nu^2 = nrm2_prev - |h|^2, out[0] = ||vout||^2, out[1] = nu.  MODE 2: w <- w + sum_j
// h_j V_j (sign +, no norm).
template <int MODE>
__global__ void __launch_bounds__(kRedThreads) k_gs_axpy_dd(const dd* __restrict__ V, int64_t ldv, int nv,
                                                           const double* __restrict__ h, dd* w, dd* vout, int64_t n,
                                                           double* __restrict__ partial, unsigned* counter,
                                                           double* __restrict__ out,
                                                           const double* __restrict__ nrm2_prev) {
  __shared__ dd cs[kGsMaxVec];
  __shared__ double sh[32];
  __shared__ dd inv_nu;
  for (int j = threadIdx.x; j < nv; j += blockDim.x) cs[j] = MODE == 2 ? dd(h[j]) : dd(-h[j]);
  if (MODE == 1 && threadIdx.x < 32) {
    const double c2 = warp_norm2(h, nv, threadIdx.x);
    if (threadIdx.x == 0) {
      const double nu2 = *nrm2_prev - c2;
      const double nu = nu2 > 0.0 ? sqrt(nu2) : 0.0;
      inv_nu = nu > 0.0 ? dd(1.0 / nu) : dd(0.f, 0.f);
      if (blockIdx.x == 0) out[1] = nu;
    }
  }
  __syncthreads();
  dd acc(0.f, 0.f);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    dd v = w[i];
    for (int j = 0; j < nv; ++j) v = fma(cs[j], V[(int64_t)j * ldv + i], v);
    if (MODE == 1) {
      v = v * inv_nu;
      vout[i] = v;
    } else {
      w[i] = v;
    }
    if (MODE != 2) acc = fma(v, v, acc);
  }
  if (MODE == 2) return;
  const double a = block_sum(dd_d(acc), sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = a;
  last_block_reduce(partial, 1, counter, out);
}

inline int grid_for(int64_t n, int threads, int cap = 152 * 16) {
  int64_t g = (n + threads - 1) / threads;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return (int)g;
}

// Launch shapes of the Gram-Schmidt kernels, n = work items (elements, pairs or quads) per vector.
// Long vectors: one block of 512 threads per SM for the multi-dots (fewest adds; 18 16-byte loads in flight per
// thread are enough), two per SM for the updates (8 in flight).  Measured at 3.7 M float64 elements and 30
// vectors: multi-dot 228 us (252 with two blocks per SM, 294 with four), update 212 us (260 with one, 220 with
// four).  Short vectors: 256 threads, one pass over the items, and the groups of eight vectors side by side in
// blockIdx.y (83 k elements, 30 vectors: 16 us; 27 with the groups in turn).
// Float32 sums: a thread has four (two over quads, each summed by itself first), so that no sum takes more roundings
// than one of ceil(n / 155,648) items, also between the two lengths.
struct RedShape {
  dim3 grid;
  int threads;
};
inline RedShape dot_shape(int64_t n, int nv) {
  if (n >= 152 * 512 * 4) return {dim3(152), 512};
  const int nb = (int)std::max<int64_t>(1, std::min<int64_t>((n + 511) / 512, 152));
  return {dim3(nb, std::max(1, std::min((nv + 7) / 8, (304 + nb - 1) / nb))), 256};
}
inline RedShape upd_shape(int64_t n) {
  if (n >= 152 * 512 * 2) return {dim3(304), 512};
  return {dim3((int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 304))), 256};
}
// Double-float: bound by the latency of its multiply-adds (twenty dependent instructions each), so on long vectors
// more warps: 3.7 M elements, a solve of 48 steps, multi-dots 17 ms (152 blocks of 512 threads 30 ms), updates 10.6 ms
// (304 blocks of 512 threads 15.7 ms).
inline RedShape dot_shape_dd(int64_t n, int nv) {
  if (n >= 152 * 512 * 4) return {dim3(608), 256};
  return dot_shape(n, nv);
}
inline RedShape upd_shape_dd(int64_t n) {
  if (n >= 152 * 512 * 6) return {dim3((int)std::min<int64_t>((n + 255) / 256, 2432)), 256};
  return upd_shape(n);
}

}  // namespace

namespace fmi {

// The local part of the operator on every component in float32, one launch (k_apply_local).
static int apply_local32(fm_ctx* c, double E, const float* x, float* y, bool only_S, bool timed) {
  LocalArgs a;
  std::memset(&a, 0, sizeof(a));
  a.ncomp = (int)c->comps.size();
  a.E = (float)E;
  a.only_S = only_S ? 1 : 0;
  const int r = c->comps[0].r, q = c->comps[0].az.q;
  int tiles = 0, nintmax = 1, smem_elems = 0;
  double fl = 0.0, by = 0.0;
  for (int k = 0; k < a.ncomp; ++k) {
    const Comp& cp = c->comps[k];
    const ApplyTabs<float> tb = tabs_of<float>(cp);
    LocalComp& f = a.c[k];
    f.x = x + cp.off; f.y = y + cp.off; f.W = tb.W; f.Sx = tb.Sx; f.D2x = tb.D2x; f.Sy = tb.Sy; f.D2y = tb.D2y;
    f.zt = tb.zt; f.qx = tb.qx; f.iy2 = tb.iy2; f.bx = cp.dx.base; f.by = cp.dy.base; f.zf = cp.zf;
    f.nx = cp.nx; f.ny = cp.ny; f.nz = cp.nz; f.rows = cp.ax.tile_rows(kLX); f.cols = cp.ay.tile_rows(kLY);
    f.tiles_x = (cp.nx + kLX - 1) / kLX; f.tiles_y = (cp.ny + kLY - 1) / kLY;
    f.nint = cp.az.nint; f.q = q;
    tiles += f.tiles_x * f.tiles_y;
    nintmax = std::max(nintmax, f.nint);
    smem_elems = std::max(smem_elems, 2 * r * (kLX + kLY) + q * c->nM * f.rows * (2 * (f.cols + 1) + 2 * kLY));
    const double tot = (double)cp.npts * c->nM;
    fl += tot * (only_S ? 6.0 * r : (c->nM > 1 ? 20.0 : 16.0) * r + 6.0);
    by += tot * (only_S ? 2.0 : 3.0) * sizeof(float);
  }
  // z chunks: a CTA of n intervals walks q n + r - q planes; the split with the fewest planes on the SM that gets the
  // most CTAs, counting at least four (fewer leave the latency of a plane uncovered)
  int ipc = 1;
  double cost = 1e300;
  for (int n = 1; n <= nintmax; ++n) {
    const int per_cta = (nintmax + n - 1) / n;
    const int ctas = tiles * ((nintmax + per_cta - 1) / per_cta);
    const double cst = std::max(4, (ctas + 151) / 152) * (double)(q * per_cta + r - q);
    if (cst < cost) {
      cost = cst;
      ipc = per_cta;
    }
  }
  int grid = 0;
  for (int k = 0; k < a.ncomp; ++k) {
    LocalComp& f = a.c[k];
    f.ipc = std::min(ipc, f.nint);
    f.first = grid;
    grid += f.tiles_x * f.tiles_y * ((f.nint + f.ipc - 1) / f.ipc);
  }
  const size_t smem = (size_t)smem_elems * sizeof(float);
  const int tk_ = timed ? prof_begin(c, FM_KERNEL_APPLY_XY) : -1;
  switch ((r == 6 ? 16 : 0) + c->nM) {
    case 1: k_apply_local<4, 1><<<grid, kLThreads, smem, c->stream>>>(a); break;
    case 2: k_apply_local<4, 2><<<grid, kLThreads, smem, c->stream>>>(a); break;
    case 3: k_apply_local<4, 3><<<grid, kLThreads, smem, c->stream>>>(a); break;
    case 4: k_apply_local<4, 4><<<grid, kLThreads, smem, c->stream>>>(a); break;
    case 5: k_apply_local<4, 5><<<grid, kLThreads, smem, c->stream>>>(a); break;
    case 17: k_apply_local<6, 1><<<grid, kLThreads, smem, c->stream>>>(a); break;
    case 18: k_apply_local<6, 2><<<grid, kLThreads, smem, c->stream>>>(a); break;
    case 19: k_apply_local<6, 3><<<grid, kLThreads, smem, c->stream>>>(a); break;
    default: return FM_ERR_ARG;
  }
  prof_end(c, tk_, fl, by);
  c->launches++;
  FM_CUDA(cudaGetLastError());
  return FM_OK;
}

// The local part of the operator in two passes (scratch planes P and Q), every component in each launch.
template <typename T>
static int apply_planes(fm_ctx* c, double E, const T* x, T* y, bool only_S, T* P, T* Q, bool timed) {
  PlaneArgs<T> a;
  std::memset(&a, 0, sizeof(a));
  a.ncomp = (int)c->comps.size();
  a.nM = c->nM;
  a.E = (T)E;
  a.only_S = only_S ? 1 : 0;
  const int r = c->comps[0].r;
  int64_t gxy = 0, gz = 0;
  size_t elems = 0;
  double tot = 0.0;
  for (int k = 0; k < a.ncomp; ++k) {
    const Comp& cp = c->comps[k];
    const ApplyTabs<T> tb = tabs_of<T>(cp);
    PlaneComp<T>& f = a.c[k];
    f.x = x + cp.off; f.P = P + cp.off; f.Q = Q + cp.off; f.y = y + cp.off; f.W = tb.W; f.Sx = tb.Sx; f.D2x = tb.D2x;
    f.Sy = tb.Sy; f.D2y = tb.D2y; f.zt = tb.zt; f.qx = tb.qx; f.iy2 = tb.iy2;
    f.bx = cp.dx.base; f.by = cp.dy.base; f.bz = cp.dz.base;
    f.nx = cp.nx; f.ny = cp.ny; f.nz = cp.nz; f.rows = cp.ax.tile_rows(kPX); f.cols = cp.ay.tile_rows(kPY);
    f.tiles_x = (cp.nx + kPX - 1) / kPX; f.tiles_y = (cp.ny + kPY - 1) / kPY;
    f.first_xy = (int)gxy;
    f.first_z = (int)gz;
    const int64_t planes = (int64_t)c->nM * cp.nz;
    gxy += planes * f.tiles_x * f.tiles_y;
    gz += planes * (((int64_t)cp.nx * cp.ny + 255) / 256);
    elems = std::max(elems, (size_t)f.rows * (f.cols + 1 + 2 * kPY));
    tot += (double)cp.npts * c->nM;
  }
  if (gxy > 0x7FFFFFFF || gz > 0x7FFFFFFF) return FM_ERR_ARG;
  {
    const int tk_ = timed ? prof_begin(c, FM_KERNEL_APPLY_XY) : -1;
    if (r == 6) k_apply_xy<6, T><<<(unsigned)gxy, 256, elems * sizeof(T), c->stream>>>(a);
    else k_apply_xy<4, T><<<(unsigned)gxy, 256, elems * sizeof(T), c->stream>>>(a);
    prof_end(c, tk_, tot * r * (only_S ? 4.0 : 10.0), tot * (only_S ? 2.0 : 3.0) * sizeof(T));
  }
  {
    const int tk_ = timed ? prof_begin(c, FM_KERNEL_APPLY_Z) : -1;
    if (r == 6) k_apply_z<6, T><<<(unsigned)gz, 256, 0, c->stream>>>(a);
    else k_apply_z<4, T><<<(unsigned)gz, 256, 0, c->stream>>>(a);
    prof_end(c, tk_, tot * (only_S ? 2.0 * r : (c->nM > 1 ? 10.0 : 6.0) * r + 6.0),
             tot * (only_S ? 2.0 : 4.0) * sizeof(T));
  }
  c->launches += 2;
  FM_CUDA(cudaGetLastError());
  return FM_OK;
}

// y = (H - E S) x (only_S: y = S x) in the element type T; scratch planes P and Q for the two-pass local form.
template <typename T>
static int apply_t(fm_ctx* c, double E, const T* x, T* y, bool only_S, T* P, T* Q, bool timed) {
  int rc;
  bool one_pass = false;
  if constexpr (std::is_same<T, float>::value) {
    one_pass = local_one_pass(c->nM, c->comps[0].r);
    if (one_pass && (rc = apply_local32(c, E, x, y, only_S, timed))) return rc;
  }
  if (!one_pass && (rc = apply_planes<T>(c, E, x, y, only_S, P, Q, timed))) return rc;
  return only_S ? FM_OK : apply_coupling<T>(c, x, y, timed);
}

int launch_apply(fm_ctx* c, double E, const double* x, double* y, bool only_S) {
  return apply_t<double>(c, E, x, y, only_S, c->P, c->Q, true);
}

int launch_apply32(fm_ctx* c, double E, const float* x, float* y, bool only_S) {
  return apply_t<float>(c, E, x, y, only_S, c->P32, c->Q32, true);
}

// The operator apply with caller-chosen scratch planes (used by the entry point that allocates
// nothing, whose planes live in a fixed device array).  Same kernels and launch shapes as
// launch_apply; no per-kernel timing.
int launch_apply_scratch(fm_ctx* c, double E, const double* x, double* y, double* P, double* Q) {
  return apply_t<double>(c, E, x, y, false, P, Q, false);
}

// y = P^{-1} x (Eq. prec-2), stage-major over the components: every component's z and x forward
// stages (and the diagonalised y stage for n_M = 1), then one launch with the banded y solves of
// all components that need them, then every component's x and z inverse stages.
template <typename T, typename TIO>
static int precond_impl(fm_ctx* c, const TIO* x, TIO* y, T* t) {
  const bool is32 = std::is_same<T, float>::value;
  const bool tc = is32 && c->tc_active;
  T* u = is32 ? (T*)c->u32 : (T*)c->u64;
  std::vector<fmi::Comp*> banded;
  int rc;
  // float64 on the tensor cores: z forward, x forward here, x inverse, z inverse below, all components per launch
  const bool f64 = !is32 && c->f64_tc;
  if constexpr (std::is_same<T, double>::value && std::is_same<TIO, double>::value) {
    if (f64 && ((rc = f64_stage(c, 0, x, t)) || (rc = f64_stage(c, 2, t, u)))) return rc;
  }
  if (tc) {  // z, x and y stages on the tensor cores
    if ((rc = fmi::precond_tc_front<TIO>(c, x, &banded))) return rc;
    if ((rc = ysolve_banded<T>(c, banded, u))) return rc;
    if ((rc = fmi::precond_tc_back<TIO>(c, y))) return rc;
    FM_CUDA(cudaGetLastError());
    return FM_OK;
  }
  for (auto& cp : c->comps) {
    const bool ymda = cp.ydiag_ok && (c->opts.y_solver == 2 || (c->opts.y_solver == 0 && is32));
    if (!ymda) banded.push_back(&cp);
    const int64_t nxy = (int64_t)cp.nx * cp.ny;
    const T* Wzb = std::is_same<T, double>::value ? (const T*)cp.Wzb : (const T*)cp.Wzb32;
    const T* Wxb = std::is_same<T, double>::value ? (const T*)cp.Wxb : (const T*)cp.Wxb32;
    const double ncomp = (double)nxy * cp.nz * c->nM;  // unknowns of this component
    const double ts = (double)sizeof(T);
    if (!f64) {
      dim3 gz((unsigned)((nxy + 127) / 128), c->nM);
      const size_t smz = ((size_t)cp.nz * cp.nz + (size_t)cp.nz * 128) * sizeof(T);
      {
        const int tk_ = prof_begin(c, FM_KERNEL_ZMIX);
        k_zmix<TIO, T, T><<<gz, 128, smz, c->stream>>>(Wzb, x, t, cp.nz, nxy, cp.off);
        prof_end(c, tk_, 2.0 * cp.nz * ncomp, ncomp * (8.0 + ts));
      }
      dim3 gx((cp.ny + 63) / 64, (cp.nx + 63) / 64, c->nM * cp.nz);
      {
        const int tk_ = prof_begin(c, FM_KERNEL_XMIX);
        k_mix<T, false, true, false><<<gx, 256, 0, c->stream>>>(Wxb, t, u, cp.nx, cp.ny, cp.nz, cp.off, c->M0, nullptr, nullptr);
        prof_end(c, tk_, 2.0 * cp.nx * ncomp, 2.0 * ncomp * ts);
      }
      c->launches += 2;
    }
    if (ymda) {
      // n_M = 1: per-l diagonalisation of (A_l, S_y): W_y (Lambda_y + lambda_x)^{-1} W-bar_y on transposed slabs
      const T* Wyb = is32 ? (const T*)cp.Wyb32 : (const T*)cp.Wyb64;
      const T* Wy = is32 ? (const T*)cp.Wy32 : (const T*)cp.Wy64;
      const T* dLy = is32 ? (const T*)cp.dLy32 : (const T*)cp.dLy64;
      const T* dLx = is32 ? (const T*)cp.dLx32 : (const T*)cp.dLx64;
      dim3 gyy((cp.nx + 63) / 64, (cp.ny + 63) / 64, c->nM * cp.nz);
      {
        const int tk_ = prof_begin(c, FM_KERNEL_YSOLVE);
        k_mix<T, false, false, true><<<gyy, 256, 0, c->stream>>>(Wyb, u, t, cp.ny, cp.nx, cp.nz, cp.off, c->M0, dLy, dLx);
        prof_end(c, tk_, 2.0 * cp.ny * ncomp, 2.0 * ncomp * ts);
      }
      {
        const int tk_ = prof_begin(c, FM_KERNEL_YSOLVE);
        k_mix<T, false, false, false><<<gyy, 256, 0, c->stream>>>(Wy, t, u, cp.ny, cp.nx, cp.nz, cp.off, c->M0, nullptr, nullptr);
        prof_end(c, tk_, 2.0 * cp.ny * ncomp, 2.0 * ncomp * ts);
      }
      c->launches += 2;
    }
  }
  if ((rc = ysolve_banded<T>(c, banded, u))) return rc;
  if constexpr (std::is_same<T, double>::value && std::is_same<TIO, double>::value) {
    if (f64) {
      if ((rc = f64_stage(c, 3, u, t))) return rc;
      return f64_stage(c, 1, t, y);
    }
  }
  for (auto& cp : c->comps) {
    const int64_t nxy = (int64_t)cp.nx * cp.ny;
    const T* Wz = std::is_same<T, double>::value ? (const T*)cp.Wz : (const T*)cp.Wz32;
    const T* Wx = std::is_same<T, double>::value ? (const T*)cp.Wx : (const T*)cp.Wx32;
    const double ncomp = (double)nxy * cp.nz * c->nM;
    const double ts = (double)sizeof(T);
    dim3 gz((unsigned)((nxy + 127) / 128), c->nM);
    const size_t smz = ((size_t)cp.nz * cp.nz + (size_t)cp.nz * 128) * sizeof(T);
    dim3 gx((cp.ny + 63) / 64, (cp.nx + 63) / 64, c->nM * cp.nz);
    {
      const int tk_ = prof_begin(c, FM_KERNEL_XMIX);
      k_mix<T, true, false, false><<<gx, 256, 0, c->stream>>>(Wx, u, t, cp.nx, cp.ny, cp.nz, cp.off, c->M0, nullptr, nullptr);
      prof_end(c, tk_, 2.0 * cp.nx * ncomp, 2.0 * ncomp * ts);
    }
    {
      const int tk_ = prof_begin(c, FM_KERNEL_ZMIX);
      k_zmix<T, TIO, T><<<gz, 128, smz, c->stream>>>(Wz, t, y, cp.nz, nxy, cp.off);
      prof_end(c, tk_, 2.0 * cp.nz * ncomp, ncomp * (8.0 + ts));
    }
    c->launches += 2;
  }
  FM_CUDA(cudaGetLastError());
  return FM_OK;
}

int launch_precond(fm_ctx* c, const double* x, double* y) {
  if (c->opts.precision != FM_PREC_FP64) return precond_impl<float, double>(c, x, y, c->t32);
  return precond_impl<double, double>(c, x, y, c->t64);
}

int launch_precond32(fm_ctx* c, const float* x, float* y) { return precond_impl<float, float>(c, x, y, c->t32); }

int dot_many(fm_ctx* c, const double* V, int64_t ldv, int nv, const double* w, double* h_host) {
  return dot_many_x(c, V, ldv, nv, w, nullptr, h_host);
}

int dot_many_x(fm_ctx* c, const double* V, int64_t ldv, int nv, const double* w, const double* extra, double* h_host) {
  const int nt = nv + (extra ? 1 : 0);
  int rc;
  if ((rc = dot_many_dev(c, V, ldv, nv, w, extra, c->gsd))) return rc;
  FM_CUDA(cudaMemcpyAsync(c->red_host, c->gsd, nt * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  FM_CUDA(cudaStreamSynchronize(c->stream));
  std::memcpy(h_host, c->red_host, nt * sizeof(double));
  return prof_harvest(c);
}

// h_dev[j] = V[j] . w (j < nv), h_dev[nv] = extra . w when extra is given; stays on the device
int dot_many_dev(fm_ctx* c, const double* V, int64_t ldv, int nv, const double* w, const double* extra, double* h_dev,
                 bool lowp) {
  const int nt = nv + (extra ? 1 : 0);
  if (nt > kGsMaxVec) return FM_ERR_ARG;
  // 16-byte element pairs when every vector starts on a 16-byte boundary, scalar loads otherwise (an odd
  // vector length puts every other basis vector on an 8-byte boundary)
  const uintptr_t al = reinterpret_cast<uintptr_t>(V) | reinterpret_cast<uintptr_t>(w) |
                       reinterpret_cast<uintptr_t>(extra) | (uintptr_t)(ldv * 8);
  const bool pairs = (al & 15u) == 0;
  const RedShape sh = dot_shape(pairs ? c->N / 2 : c->N, nt);
  const int tk_ = prof_begin(c, FM_KERNEL_DOT);
  if (pairs && lowp) k_dot_many<true><<<sh.grid, sh.threads, 0, c->stream>>>(V, ldv, nv, w, c->N, c->red, extra, c->gs_cnt, h_dev);
  else if (pairs) k_dot_many<false><<<sh.grid, sh.threads, 0, c->stream>>>(V, ldv, nv, w, c->N, c->red, extra, c->gs_cnt, h_dev);
  else if (lowp) k_dot_many_s<true><<<sh.grid, sh.threads, 0, c->stream>>>(V, ldv, nv, w, c->N, c->red, extra, c->gs_cnt, h_dev);
  else k_dot_many_s<false><<<sh.grid, sh.threads, 0, c->stream>>>(V, ldv, nv, w, c->N, c->red, extra, c->gs_cnt, h_dev);
  prof_end(c, tk_, 2.0 * nt * (double)c->N, (nt + 1.0) * 8.0 * (double)c->N);
  c->launches++;
  FM_CUDA(cudaGetLastError());
  return FM_OK;
}

int axpy_many(fm_ctx* c, const double* V, int64_t ldv, int nv, const double* h_host, double* w, double sign) {
  double* hd = c->red + (int64_t)c->red_blocks * 256 + 512;
  FM_CUDA(cudaMemcpyAsync(hd, h_host, nv * sizeof(double), cudaMemcpyHostToDevice, c->stream));
  {
    const int tk_ = prof_begin(c, FM_KERNEL_AXPY);
    k_axpy_many<<<grid_for(c->N, 256), 256, 0, c->stream>>>(V, ldv, nv, hd, sign, w, c->N);
    prof_end(c, tk_, 2.0 * nv * (double)c->N, (nv + 2.0) * 8.0 * (double)c->N);
  }
  c->launches++;
  FM_CUDA(cudaGetLastError());
  return FM_OK;
}

// One launch of k_gs_axpy on vectors of stride N: 16-byte pairs when N is even and every buffer allows them.
template <int MODE>
static void gs_update(fm_ctx* c, const double* V, int nv, const double* h, const double* G, const double* a, double* w,
                      double* vout, double* out, const double* nrm2_prev) {
  const uintptr_t al = reinterpret_cast<uintptr_t>(V) | reinterpret_cast<uintptr_t>(w) |
                       reinterpret_cast<uintptr_t>(vout) | (uintptr_t)(c->N * 8);
  const bool pairs = (al & 15u) == 0;
  const RedShape sh = upd_shape(pairs ? c->N / 2 : c->N);
  if (pairs)
    k_gs_axpy<MODE, true><<<sh.grid, sh.threads, 0, c->stream>>>(V, c->N, nv, h, G, a, w, vout, c->N, c->red, c->gs_cnt,
                                                                 out, nrm2_prev);
  else
    k_gs_axpy<MODE, false><<<sh.grid, sh.threads, 0, c->stream>>>(V, c->N, nv, h, G, a, w, vout, c->N, c->red, c->gs_cnt,
                                                                  out, nrm2_prev);
}

// Classical Gram-Schmidt with one re-orthogonalisation (CGS2) of w against the orthonormal
// V[0..nv), all coefficients kept on the device:
//   h1 = V^T w;  w' = w - V h1;  h2 = V^T w';  vout = (w' - V h2) / nu,  nu^2 = ||w'||^2 - |h2|^2.
// Four launches and one host synchronisation.  On return h = h1 + h2 and *hn = ||w' - V h2||
// (nu times the measured norm of vout, which is renormalised if it is not 1 to rounding);
// *hn = 0 when w lies in span V to rounding (vout is then 0).  w is overwritten; vout may be w.
int gs_cgs2(fm_ctx* c, const double* V, int nv, double* w, double* vout, double* h, double* hn) {
  if (nv < 1 || nv > kGsMaxVec) return FM_ERR_ARG;
  const int64_t N = c->N;
  double* h1 = c->gsd;
  double* h2 = c->gsd + kGsMaxVec;
  double* sc = c->gsd + 3 * kGsMaxVec;  // [0] ||w'||^2, [1] ||vout||^2, [2] nu
  int rc;
  // first pass: projections to about 1e-6, on the FP32 pipe; the float64 second pass removes what it leaves
  if ((rc = dot_many_dev(c, V, N, nv, w, nullptr, h1, true))) return rc;
  {
    const int tk_ = prof_begin(c, FM_KERNEL_AXPY);
    gs_update<0>(c, V, nv, h1, nullptr, nullptr, w, nullptr, sc, nullptr);
    prof_end(c, tk_, (2.0 * nv + 2.0) * (double)N, (nv + 2.0) * 8.0 * (double)N);
  }
  if ((rc = dot_many_dev(c, V, N, nv, w, nullptr, h2))) return rc;
  {
    const int tk_ = prof_begin(c, FM_KERNEL_AXPY);
    gs_update<1>(c, V, nv, h2, nullptr, nullptr, w, vout, sc + 1, sc);
    prof_end(c, tk_, (2.0 * nv + 2.0) * (double)N, (nv + 2.0) * 8.0 * (double)N);
  }
  c->launches += 2;
  FM_CUDA(cudaGetLastError());
  // one read-back: h1, h2 and the three scalars
  FM_CUDA(cudaMemcpyAsync(c->red_host, c->gsd, kGsRead * sizeof(double), cudaMemcpyDeviceToHost,
                          c->stream));
  FM_CUDA(cudaStreamSynchronize(c->stream));
  const double* hh = c->red_host;
  if (c->tc_err && reinterpret_cast<const int*>(hh + kGsFlag)[0] != 0) return FM_ERR_TIMEOUT;
  for (int i = 0; i < nv; ++i) h[i] = hh[i] + hh[kGsMaxVec + i];
  const double vn2 = hh[3 * kGsMaxVec + 1], nu = hh[3 * kGsMaxVec + 2];
  if (!(nu > 0.0) || !(vn2 > 0.0)) {
    *hn = std::isfinite(nu) && std::isfinite(vn2) ? 0.0 : nu + vn2;
    return prof_harvest(c);
  }
  const double vn = std::sqrt(vn2);
  *hn = nu * vn;
  if (std::fabs(vn - 1.0) > 1e-12)  // Pythagoras lost digits: rescale to unit norm
    if ((rc = scale_copy(c, vout, 1.0 / vn, vout))) return rc;
  return prof_harvest(c);
}

// Single-pass classical Gram-Schmidt in float64 with the DGKS re-orthogonalisation test: one multi-dot (with
// |w|^2 from the same pass), one update that normalises directly when |w - V h| >= |w| / sqrt(2); otherwise
// it keeps w - V h and a second float64 pass (multi-dot, closing update) follows.  One host synchronisation
// when no re-orthogonalisation is needed, two otherwise.  Same results as gs_cgs2 to rounding.
int gs_cgs1(fm_ctx* c, const double* V, int nv, double* w, double* vout, double* h, double* hn) {
  if (nv < 1 || nv + 1 > kGsMaxVec) return FM_ERR_ARG;
  const int64_t N = c->N;
  double* h1 = c->gsd;                  // [nv] V^T w, [nv] |w|^2
  double* h2 = c->gsd + kGsMaxVec;
  double* sc = c->gsd + 3 * kGsMaxVec;  // [1] |out|^2, [2] nu, [3] re-orthogonalise
  int rc;
  if ((rc = dot_many_dev(c, V, N, nv, w, w, h1))) return rc;
  {
    const int tk_ = prof_begin(c, FM_KERNEL_AXPY);
    gs_update<2>(c, V, nv, h1, nullptr, nullptr, w, vout, sc + 1, h1 + nv);
    prof_end(c, tk_, (2.0 * nv + 2.0) * (double)N, (nv + 2.0) * 8.0 * (double)N);
  }
  c->launches++;
  FM_CUDA(cudaGetLastError());
  FM_CUDA(cudaMemcpyAsync(c->red_host, c->gsd, kGsRead * sizeof(double), cudaMemcpyDeviceToHost,
                          c->stream));
  FM_CUDA(cudaStreamSynchronize(c->stream));
  const double* hh = c->red_host;
  if (c->tc_err && reinterpret_cast<const int*>(hh + kGsFlag)[0] != 0) return FM_ERR_TIMEOUT;
  for (int i = 0; i < nv; ++i) h[i] = hh[i];
  if (hh[3 * kGsMaxVec + 3] != 0.0) {  // cancellation: second float64 pass on w - V h
    if ((rc = dot_many_dev(c, V, N, nv, w, nullptr, h2))) return rc;
    {
      const int tk_ = prof_begin(c, FM_KERNEL_AXPY);
      gs_update<1>(c, V, nv, h2, nullptr, nullptr, w, vout, sc + 1, sc + 1);
      prof_end(c, tk_, (2.0 * nv + 2.0) * (double)N, (nv + 2.0) * 8.0 * (double)N);
    }
    c->launches++;
    FM_CUDA(cudaGetLastError());
    FM_CUDA(cudaMemcpyAsync(c->red_host, c->gsd, kGsRead * sizeof(double), cudaMemcpyDeviceToHost,
                            c->stream));
    FM_CUDA(cudaStreamSynchronize(c->stream));
    if (c->tc_err && reinterpret_cast<const int*>(hh + kGsFlag)[0] != 0) return FM_ERR_TIMEOUT;
    for (int i = 0; i < nv; ++i) h[i] += hh[kGsMaxVec + i];
  }
  const double vn2 = hh[3 * kGsMaxVec + 1], nu = hh[3 * kGsMaxVec + 2];
  if (!(nu > 0.0) || !(vn2 > 0.0)) {
    *hn = std::isfinite(nu) && std::isfinite(vn2) ? 0.0 : nu + vn2;
    return prof_harvest(c);
  }
  const double vn = std::sqrt(vn2);
  *hn = nu * vn;
  if (std::fabs(vn - 1.0) > 1e-12)  // Pythagoras lost digits: rescale to unit norm
    if ((rc = scale_copy(c, vout, 1.0 / vn, vout))) return rc;
  return prof_harvest(c);
}

// float32 CGS2 (MIXED precision inner solves): as gs_cgs2 on float32 vectors, coefficients and norms
// in float64, one host synchronisation.
int gs_cgs2_32(fm_ctx* c, const float* V, int nv, float* w, float* vout, double* h, double* hn) {
  if (nv < 1 || nv > kGsMaxVec) return FM_ERR_ARG;
  const int64_t N = c->N;
  // 16-byte quads when every vector starts on a 16-byte boundary (N a multiple of 4), scalar loads otherwise
  const uintptr_t al = reinterpret_cast<uintptr_t>(V) | reinterpret_cast<uintptr_t>(w) | (uintptr_t)(N * 4);
  const bool quads = (al & 15u) == 0;
  double* h1 = c->gsd;
  double* h2 = c->gsd + kGsMaxVec;
  double* sc = c->gsd + 3 * kGsMaxVec;
  const RedShape sd = dot_shape(quads ? N / 4 : N, nv), su = upd_shape(quads ? N / 4 : N);
  {
    const int tk_ = prof_begin(c, FM_KERNEL_DOT);
    if (quads) k_dot_many32v<<<sd.grid, sd.threads, 0, c->stream>>>(V, N, nv, w, N, c->red, c->gs_cnt, h1);
    else k_dot_many32<<<sd.grid, sd.threads, 0, c->stream>>>(V, N, nv, w, N, c->red, c->gs_cnt, h1);
    prof_end(c, tk_, 2.0 * nv * (double)N, (nv + 1.0) * 4.0 * (double)N);
  }
  {
    const int tk_ = prof_begin(c, FM_KERNEL_AXPY);
    if (quads) k_gs_axpy32<0, true><<<su.grid, su.threads, 0, c->stream>>>(V, N, nv, h1, w, nullptr, N, c->red, c->gs_cnt, sc, nullptr);
    else k_gs_axpy32<0, false><<<su.grid, su.threads, 0, c->stream>>>(V, N, nv, h1, w, nullptr, N, c->red, c->gs_cnt, sc, nullptr);
    prof_end(c, tk_, (2.0 * nv + 2.0) * (double)N, (nv + 2.0) * 4.0 * (double)N);
  }
  {
    const int tk_ = prof_begin(c, FM_KERNEL_DOT);
    if (quads) k_dot_many32v<<<sd.grid, sd.threads, 0, c->stream>>>(V, N, nv, w, N, c->red, c->gs_cnt, h2);
    else k_dot_many32<<<sd.grid, sd.threads, 0, c->stream>>>(V, N, nv, w, N, c->red, c->gs_cnt, h2);
    prof_end(c, tk_, 2.0 * nv * (double)N, (nv + 1.0) * 4.0 * (double)N);
  }
  {
    const int tk_ = prof_begin(c, FM_KERNEL_AXPY);
    if (quads) k_gs_axpy32<1, true><<<su.grid, su.threads, 0, c->stream>>>(V, N, nv, h2, w, vout, N, c->red, c->gs_cnt, sc + 1, sc);
    else k_gs_axpy32<1, false><<<su.grid, su.threads, 0, c->stream>>>(V, N, nv, h2, w, vout, N, c->red, c->gs_cnt, sc + 1, sc);
    prof_end(c, tk_, (2.0 * nv + 2.0) * (double)N, (nv + 2.0) * 4.0 * (double)N);
  }
  c->launches += 4;
  FM_CUDA(cudaGetLastError());
  FM_CUDA(cudaMemcpyAsync(c->red_host, c->gsd, kGsRead * sizeof(double), cudaMemcpyDeviceToHost,
                          c->stream));
  FM_CUDA(cudaStreamSynchronize(c->stream));
  const double* hh = c->red_host;
  if (c->tc_err && reinterpret_cast<const int*>(hh + kGsFlag)[0] != 0) return FM_ERR_TIMEOUT;
  for (int i = 0; i < nv; ++i) h[i] = hh[i] + hh[kGsMaxVec + i];
  const double vn2 = hh[3 * kGsMaxVec + 1], nu = hh[3 * kGsMaxVec + 2];
  if (!(nu > 0.0) || !(vn2 > 0.0)) {
    *hn = std::isfinite(nu) && std::isfinite(vn2) ? 0.0 : nu + vn2;
    return prof_harvest(c);
  }
  const double vn = std::sqrt(vn2);
  *hn = nu * vn;
  int rc;
  if (std::fabs(vn - 1.0) > 1e-6)  // float32 vector: renormalise when Pythagoras lost digits
    if ((rc = axpby32(c, (float)(1.0 / vn), vout, 0.0f, vout))) return rc;
  return prof_harvest(c);
}

// z <- z - (W - U) G (U^T z) for the tuned preconditioner, G = (U^T W)^{-1} (k x k, on the device);
// no host synchronisation
int tuning_correct(fm_ctx* c, const double* U, const double* WmU, const double* Gdev, int k, double* z) {
  if (k <= 0) return FM_OK;
  if (k > kGsMaxVec) return FM_ERR_ARG;
  double* a = c->gsd + 2 * kGsMaxVec;
  int rc;
  if ((rc = dot_many_dev(c, U, c->N, k, z, nullptr, a))) return rc;
  const int tk_ = prof_begin(c, FM_KERNEL_AXPY);
  gs_update<0>(c, WmU, k, nullptr, Gdev, a, z, nullptr, c->gsd + 3 * kGsMaxVec + 4, nullptr);
  prof_end(c, tk_, 2.0 * k * (double)c->N, (k + 2.0) * 8.0 * (double)c->N);
  c->launches++;
  FM_CUDA(cudaGetLastError());
  return FM_OK;
}

int scale_copy(fm_ctx* c, const double* x, double a, double* y) {
  {
    const int tk_ = prof_begin(c, FM_KERNEL_OTHER);
    k_axpby<<<grid_for(c->N, 256), 256, 0, c->stream>>>(a, x, 0.0, y, c->N);
    prof_end(c, tk_, 0.0, 0.0);
  }
  c->launches++;
  FM_CUDA(cudaGetLastError());
  return FM_OK;
}

int axpby(fm_ctx* c, double a, const double* x, double b, double* y) {
  {
    const int tk_ = prof_begin(c, FM_KERNEL_OTHER);
    k_axpby<<<grid_for(c->N, 256), 256, 0, c->stream>>>(a, x, b, y, c->N);
    prof_end(c, tk_, 0.0, 0.0);
  }
  c->launches++;
  FM_CUDA(cudaGetLastError());
  return FM_OK;
}

int combine(fm_ctx* c, const double* V, int64_t ldv, int nv, const double* Q_host, int nc, double* out, int64_t ldo) {
  double* qd = c->red + (int64_t)c->red_blocks * 256 + 512;
  if (nv * nc > 7680) return FM_ERR_ARG;
  FM_CUDA(cudaMemcpyAsync(qd, Q_host, (size_t)nv * nc * sizeof(double), cudaMemcpyHostToDevice, c->stream));
  {
    const int tk_ = prof_begin(c, FM_KERNEL_OTHER);
    k_combine<<<grid_for(c->N, 256), 256, 0, c->stream>>>(V, ldv, nv, qd, nc, out, ldo, c->N);
    prof_end(c, tk_, 0.0, 0.0);
  }
  c->launches++;
  FM_CUDA(cudaGetLastError());
  FM_CUDA(cudaStreamSynchronize(c->stream));
  return FM_OK;
}

int absmax(fm_ctx* c, const double* x, double* val) {
  const int nb = c->red_blocks;
  double* pv = c->red;
  long long* pi = (long long*)(c->red + nb);
  {
    const int tk_ = prof_begin(c, FM_KERNEL_OTHER);
    k_absmax<<<nb, 256, 0, c->stream>>>(x, c->N, pv, pi);
    prof_end(c, tk_, 0.0, 0.0);
  }
  c->launches++;
  std::vector<double> hv(nb);
  std::vector<long long> hi(nb);
  FM_CUDA(cudaMemcpyAsync(hv.data(), pv, nb * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  FM_CUDA(cudaMemcpyAsync(hi.data(), pi, nb * sizeof(long long), cudaMemcpyDeviceToHost, c->stream));
  FM_CUDA(cudaStreamSynchronize(c->stream));
  double best = 0.0;
  long long bi = -1;
  for (int b = 0; b < nb; ++b) {
    if (hi[b] < 0) continue;
    if (bi < 0 || fabs(hv[b]) > fabs(best) || (fabs(hv[b]) == fabs(best) && hi[b] < bi)) { best = hv[b]; bi = hi[b]; }
  }
  *val = best;
  return FM_OK;
}

int prof_begin(fm_ctx* c, int cls) {
  if (!c->prof) return -1;
  cudaEvent_t a, b;
  for (cudaEvent_t* e : {&a, &b}) {
    if (!c->ev_free.empty()) {
      *e = c->ev_free.back();
      c->ev_free.pop_back();
    } else if (cudaEventCreate(e) != cudaSuccess) {
      return -1;
    }
  }
  cudaEventRecord(a, c->stream);
  c->recs.push_back({cls, a, b});
  return (int)c->recs.size() - 1;
}

void prof_end(fm_ctx* c, int token, double flops, double bytes) {
  if (token < 0 || token >= (int)c->recs.size()) return;
  cudaEventRecord(c->recs[token].b, c->stream);
  c->prof_flops[c->recs[token].cls] += flops;
  c->prof_bytes[c->recs[token].cls] += bytes;
}

int prof_harvest(fm_ctx* c) {
  if (c->recs.empty()) return FM_OK;
  std::vector<fm_ctx::ProfRec> keep;
  for (auto& r : c->recs) {
    if (cudaEventQuery(r.b) != cudaSuccess) {
      cudaGetLastError();
      keep.push_back(r);
      continue;
    }
    float ms = 0.0f;
    if (cudaEventElapsedTime(&ms, r.a, r.b) == cudaSuccess) {
      c->prof_ms[r.cls] += ms;
      c->prof_n[r.cls] += 1;
    } else {
      cudaGetLastError();
    }
    c->ev_free.push_back(r.a);
    c->ev_free.push_back(r.b);
  }
  c->recs.swap(keep);
  return FM_OK;
}

int dot_many32(fm_ctx* c, const float* V, int64_t ldv, int nv, const float* w, double* h_host) {
  if (nv > kGsMaxVec) return FM_ERR_ARG;
  const RedShape sh = dot_shape(c->N, nv);
  {
    const int tk_ = prof_begin(c, FM_KERNEL_DOT);
    k_dot_many32<<<sh.grid, sh.threads, 0, c->stream>>>(V, ldv, nv, w, c->N, c->red, c->gs_cnt, c->gsd);
    prof_end(c, tk_, 2.0 * nv * (double)c->N, (nv + 1.0) * 4.0 * (double)c->N);
  }
  c->launches++;
  FM_CUDA(cudaGetLastError());
  FM_CUDA(cudaMemcpyAsync(c->red_host, c->gsd, nv * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  FM_CUDA(cudaStreamSynchronize(c->stream));
  std::memcpy(h_host, c->red_host, nv * sizeof(double));
  return prof_harvest(c);
}

int axpy_many_norm32(fm_ctx* c, const float* V, int64_t ldv, int nv, const double* h_host, float sign, float* w,
                     double* nrm2_out) {
  std::vector<float> hf(h_host, h_host + nv);
  float* hd = reinterpret_cast<float*>(c->red + (int64_t)c->red_blocks * 256 + 512);
  FM_CUDA(cudaMemcpyAsync(hd, hf.data(), nv * sizeof(float), cudaMemcpyHostToDevice, c->stream));
  const RedShape sh = upd_shape(c->N);
  {
    const int tk_ = prof_begin(c, FM_KERNEL_AXPY);
    k_axpy_many_norm32<<<sh.grid, sh.threads, 0, c->stream>>>(V, ldv, nv, hd, sign, w, c->N, c->red, c->gs_cnt,
                                                              nrm2_out ? c->gsd + 3 * kGsMaxVec : nullptr);
    prof_end(c, tk_, (2.0 * nv + 2.0) * (double)c->N, (nv + 2.0) * 4.0 * (double)c->N);
  }
  c->launches++;
  FM_CUDA(cudaGetLastError());
  if (nrm2_out) {
    FM_CUDA(cudaMemcpyAsync(c->red_host, c->gsd + 3 * kGsMaxVec, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    FM_CUDA(cudaStreamSynchronize(c->stream));
    *nrm2_out = c->red_host[0];
    return prof_harvest(c);
  }
  return FM_OK;
}

int to32(fm_ctx* c, const double* x, double a, float* y) {
  const int tk_ = prof_begin(c, FM_KERNEL_OTHER);
  k_to32<<<grid_for(c->N, 256), 256, 0, c->stream>>>(x, a, y, c->N);
  prof_end(c, tk_, 0.0, 0.0);
  c->launches++;
  FM_CUDA(cudaGetLastError());
  return FM_OK;
}

int add32(fm_ctx* c, const float* y, double a, double* x) {
  const int tk_ = prof_begin(c, FM_KERNEL_OTHER);
  k_add32<<<grid_for(c->N, 256), 256, 0, c->stream>>>(y, a, x, c->N);
  prof_end(c, tk_, 0.0, 0.0);
  c->launches++;
  FM_CUDA(cudaGetLastError());
  return FM_OK;
}

int axpby32(fm_ctx* c, float a, const float* x, float b, float* y) {
  const int tk_ = prof_begin(c, FM_KERNEL_OTHER);
  k_axpby32<<<grid_for(c->N, 256), 256, 0, c->stream>>>(a, x, b, y, c->N);
  prof_end(c, tk_, 0.0, 0.0);
  c->launches++;
  FM_CUDA(cudaGetLastError());
  return FM_OK;
}

// ---------------------------------------------------------------------------
// double-float inner solves (mixed_scheme 2)
// ---------------------------------------------------------------------------
int launch_apply_dd(fm_ctx* c, double E, const dd* x, dd* y, bool only_S) {
  // the float64 scratch planes, read as dd (the same 8 bytes per element; the float64 and dd applies never
  // overlap)
  return apply_t<dd>(c, E, x, y, only_S, reinterpret_cast<dd*>(c->P), reinterpret_cast<dd*>(c->Q),
                     true);
}

int launch_precond_dd(fm_ctx* c, const dd* x, dd* y) {
  int rc;
  {
    const int tk_ = prof_begin(c, FM_KERNEL_OTHER);
    k_dd_hi<<<grid_for(c->N, 256), 256, 0, c->stream>>>(x, c->d32, c->N);
    prof_end(c, tk_, 0.0, 12.0 * (double)c->N);
  }
  if ((rc = launch_precond32(c, c->d32, c->e32))) return rc;
  {
    const int tk_ = prof_begin(c, FM_KERNEL_OTHER);
    k_f_to_dd<<<grid_for(c->N, 256), 256, 0, c->stream>>>(c->e32, y, c->N);
    prof_end(c, tk_, 0.0, 12.0 * (double)c->N);
  }
  c->launches += 2;
  FM_CUDA(cudaGetLastError());
  return FM_OK;
}

int to_dd(fm_ctx* c, const double* x, double a, dd* y) {
  const int tk_ = prof_begin(c, FM_KERNEL_OTHER);
  k_to_dd<<<grid_for(c->N, 256), 256, 0, c->stream>>>(x, a, y, c->N);
  prof_end(c, tk_, 0.0, 16.0 * (double)c->N);
  c->launches++;
  FM_CUDA(cudaGetLastError());
  return FM_OK;
}

int add_dd(fm_ctx* c, const dd* y, double a, double* x) {
  const int tk_ = prof_begin(c, FM_KERNEL_OTHER);
  k_add_dd<<<grid_for(c->N, 256), 256, 0, c->stream>>>(y, a, x, c->N);
  prof_end(c, tk_, 0.0, 24.0 * (double)c->N);
  c->launches++;
  FM_CUDA(cudaGetLastError());
  return FM_OK;
}

int axpby_dd(fm_ctx* c, double a, const dd* x, double b, dd* y) {
  const int tk_ = prof_begin(c, FM_KERNEL_OTHER);
  k_axpby_dd<<<grid_for(c->N, 256), 256, 0, c->stream>>>(dd(a), x, dd(b), b == 0.0, y, c->N);
  prof_end(c, tk_, 0.0, 24.0 * (double)c->N);
  c->launches++;
  FM_CUDA(cudaGetLastError());
  return FM_OK;
}

int dot_many_dd(fm_ctx* c, const dd* V, int64_t ldv, int nv, const dd* w, double* h_host) {
  if (nv < 1 || nv > kGsMaxVec) return FM_ERR_ARG;
  const RedShape sh = dot_shape_dd(c->N, nv);
  {
    const int tk_ = prof_begin(c, FM_KERNEL_DOT);
    k_dot_many_dd<<<sh.grid, sh.threads, 0, c->stream>>>(V, ldv, nv, w, c->N, c->red, c->gs_cnt, c->gsd);
    prof_end(c, tk_, 2.0 * nv * (double)c->N, (nv + 1.0) * 8.0 * (double)c->N);
  }
  c->launches++;
  FM_CUDA(cudaGetLastError());
  FM_CUDA(cudaMemcpyAsync(c->red_host, c->gsd, nv * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  FM_CUDA(cudaStreamSynchronize(c->stream));
  std::memcpy(h_host, c->red_host, nv * sizeof(double));
  return prof_harvest(c);
}

int axpy_many_dd(fm_ctx* c, const dd* V, int64_t ldv, int nv, const double* h_host, dd* w) {
  if (nv < 1 || nv > kGsMaxVec) return FM_ERR_ARG;
  double* hd = c->red + (int64_t)c->red_blocks * 256 + 512;
  FM_CUDA(cudaMemcpyAsync(hd, h_host, nv * sizeof(double), cudaMemcpyHostToDevice, c->stream));
  const RedShape sh = upd_shape_dd(c->N);
  {
    const int tk_ = prof_begin(c, FM_KERNEL_AXPY);
    k_gs_axpy_dd<2><<<sh.grid, sh.threads, 0, c->stream>>>(V, ldv, nv, hd, w, nullptr, c->N, nullptr, nullptr, nullptr,
                                                           nullptr);
    prof_end(c, tk_, 2.0 * nv * (double)c->N, (nv + 2.0) * 8.0 * (double)c->N);
  }
  c->launches++;
  FM_CUDA(cudaGetLastError());
  return FM_OK;  // the next copy into hd is ordered after this kernel on the stream
}

// Two classical Gram-Schmidt passes in dd (dot products and updates accumulated in dd): w <- w - V h,
// vout = w / hn, as gs_cgs2_32 does in float32.
int gs_cgs2_dd(fm_ctx* c, const dd* V, int nv, dd* w, dd* vout, double* h, double* hn) {
  if (nv < 1 || nv > kGsMaxVec) return FM_ERR_ARG;
  const int64_t N = c->N;
  double* h1 = c->gsd;
  double* h2 = c->gsd + kGsMaxVec;
  double* sc = c->gsd + 3 * kGsMaxVec;
  const RedShape sd = dot_shape_dd(N, nv), su = upd_shape_dd(N);
  {
    const int tk_ = prof_begin(c, FM_KERNEL_DOT);
    k_dot_many_dd<<<sd.grid, sd.threads, 0, c->stream>>>(V, N, nv, w, N, c->red, c->gs_cnt, h1);
    prof_end(c, tk_, 2.0 * nv * (double)N, (nv + 1.0) * 8.0 * (double)N);
  }
  {
    const int tk_ = prof_begin(c, FM_KERNEL_AXPY);
    k_gs_axpy_dd<0><<<su.grid, su.threads, 0, c->stream>>>(V, N, nv, h1, w, nullptr, N, c->red, c->gs_cnt, sc, nullptr);
    prof_end(c, tk_, (2.0 * nv + 2.0) * (double)N, (nv + 2.0) * 8.0 * (double)N);
  }
  {
    const int tk_ = prof_begin(c, FM_KERNEL_DOT);
    k_dot_many_dd<<<sd.grid, sd.threads, 0, c->stream>>>(V, N, nv, w, N, c->red, c->gs_cnt, h2);
    prof_end(c, tk_, 2.0 * nv * (double)N, (nv + 1.0) * 8.0 * (double)N);
  }
  {
    const int tk_ = prof_begin(c, FM_KERNEL_AXPY);
    k_gs_axpy_dd<1><<<su.grid, su.threads, 0, c->stream>>>(V, N, nv, h2, w, vout, N, c->red, c->gs_cnt, sc + 1, sc);
    prof_end(c, tk_, (2.0 * nv + 2.0) * (double)N, (nv + 2.0) * 8.0 * (double)N);
  }
  c->launches += 4;
  FM_CUDA(cudaGetLastError());
  FM_CUDA(cudaMemcpyAsync(c->red_host, c->gsd, kGsRead * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  FM_CUDA(cudaStreamSynchronize(c->stream));
  const double* hh = c->red_host;
  if (c->tc_err && reinterpret_cast<const int*>(hh + kGsFlag)[0] != 0) return FM_ERR_TIMEOUT;
  for (int i = 0; i < nv; ++i) h[i] = hh[i] + hh[kGsMaxVec + i];
  const double vn2 = hh[3 * kGsMaxVec + 1], nu = hh[3 * kGsMaxVec + 2];
  if (!(nu > 0.0) || !(vn2 > 0.0)) {
    *hn = std::isfinite(nu) && std::isfinite(vn2) ? 0.0 : nu + vn2;
    return prof_harvest(c);
  }
  const double vn = std::sqrt(vn2);
  *hn = nu * vn;
  int rc;
  if (std::fabs(vn - 1.0) > 1e-12)  // renormalise when Pythagoras lost digits
    if ((rc = axpby_dd(c, 1.0 / vn, vout, 0.0, vout))) return rc;
  return prof_harvest(c);
}

int* tc_flag_slot(fm_ctx* c) { return reinterpret_cast<int*>(c->gsd + kGsFlag); }

int kernels_init(fm_ctx* c) {
  (void)c;
  const int most = 200 * 1024;
  FM_CUDA(cudaFuncSetAttribute(k_apply_local<4, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
  FM_CUDA(cudaFuncSetAttribute(k_apply_local<4, 5>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
  FM_CUDA(cudaFuncSetAttribute(k_apply_local<6, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
  FM_CUDA(cudaFuncSetAttribute(k_apply_local<6, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
  FM_CUDA(cudaFuncSetAttribute(k_apply_local<6, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
  FM_CUDA(cudaFuncSetAttribute(k_zmix<double, double, double>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  FM_CUDA(cudaFuncSetAttribute(k_zmix<double, float, float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  FM_CUDA(cudaFuncSetAttribute(k_zmix<float, double, float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  FM_CUDA(cudaFuncSetAttribute(k_zmix<float, float, float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  int rc = ysolve_init();
  return rc ? rc : tc_kernels_init();
}

int fill_normal(fm_ctx* c, double* x, uint64_t seed) {
  {
    const int tk_ = prof_begin(c, FM_KERNEL_OTHER);
    k_fill_normal<<<grid_for(c->N, 256), 256, 0, c->stream>>>(x, c->N, seed);
    prof_end(c, tk_, 0.0, 0.0);
  }
  c->launches++;
  FM_CUDA(cudaGetLastError());
  return FM_OK;
}

}  // namespace fmi
