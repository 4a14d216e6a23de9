// V^(s) coupling of the operator: kernels and their launch, for one element type per translation unit.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "fm_apply.h"
#include "fm_internal.h"

namespace fmcpl {  // (outside fmi, whose fma would hide the float and double ones)

using fmi::kMaxM;

// ---------------------------------------------------------------------------
// V^(s) coupling (Eqs. r-form, s-rot): every active collocation point adds the other components' expansions at its
// rotated position, r x r x r taps per source and M''.  One launch serves every component; bound by the FP64 pipe
// (r^3 + r^2 + r multiply-adds per point, source and M''), in float32 by L1.
//   * A (point, source) pair whose rotated position lies outside the source's box (z base -1) is passed over: the
//     expansion is zero there.  With boxes of different sizes most pairs of the wide component are outside.
//   * With an identical pair both sources of the third component are the same expansion, and on a z grid symmetric
//     about 0 source 2 at (x, y, z) is source 1 at (x, y, -z) (the rotations of an exchanged pair differ in the
//     sign of s alone).  Its points are then taken in pairs (zeta, n_z - 1 - zeta) that share two evaluations
//     instead of four.
// He L = 0 96 x 96 x 24: 463 -> 342 us (0.95 of the FP64 pipe); J = 2..4 on mid-size grids 1.4 .. 2.1x (the sums over
// M' in registers: their count is a template argument up to five components, six in the quintic basis, the longest
// chains its y solves take).
// ---------------------------------------------------------------------------
template <typename T>
struct CplSource {
  const int* base;      // [3][n_act] (z, x, y) tap bases
  const T* val;         // [3 R][n_act]
  const T* w;           // [nM * nM][n_act]
  const T* src;         // the source component's coefficients
  const T* stage;       // float32: y coefficients regrouped by y interval, [nM][nz][nx][nint_y][R]
  int64_t npts;
  int nx, ny, nz, nint;
};
template <typename T>
struct CplComp {
  CplSource<T> s[3];
  T* y;
  const int* act_pt;
  int64_t npts;
  int n_act, ns;
  int mirror, nz, nxy;  // mirrored pairs of sources 0 and 1: z points, active points per z plane
  int first;            // first block
};
template <typename T>
struct CplArgs {
  CplComp<T> c[3];
  int ncomp, nM;
  int sdir, sq;         // float32: interval of a y base = (base + sdir) / sq
};

// The source's expansion of every M'' at point p: ahead(M''), then take(M'', value); false outside its box.  UN: M''
// unrolled (bodies of r^3 taps); UNZ: z taps unrolled.
template <int R, int UN, int UNZ, typename T, typename A, typename F>
__device__ __forceinline__ bool cpl_eval(const CplSource<T>& s, int p, int n_act, int nM, int sdir, int sq, A ahead, F take) {
  const int bz = s.base[p];
  if (bz < 0) return false;
  const int bx = s.base[n_act + p], by = s.base[2 * n_act + p];
  T vz[R], vx[R], vy[R];
  int ix[R];
#pragma unroll
  for (int t = 0; t < R; ++t) {
    if (UNZ == R) vz[t] = s.val[(0 * R + t) * (int64_t)n_act + p];
    vx[t] = s.val[(1 * R + t) * (int64_t)n_act + p];
    vy[t] = s.val[(2 * R + t) * (int64_t)n_act + p];
    ix[t] = min(max(bx + t, 0), s.nx - 1);
  }
  auto zval = [&](int t) { return UNZ == R ? vz[t] : s.val[t * (int64_t)n_act + p]; };
  if constexpr (std::is_same<T, float>::value) {
    // regrouped by y interval: a source row's R taps are one aligned vector load
    const int my = min(max((by + sdir) / sq, 0), s.nint - 1);
#pragma unroll UN
    for (int jM = 0; jM < nM; ++jM) {
      ahead(jM);
      const float* tb = s.stage + (int64_t)jM * s.nz * s.nx * s.nint * R;
      float sz = 0.f;
#pragma unroll UNZ
      for (int tz = 0; tz < R; ++tz) {
        const int64_t rz = (int64_t)(bz + tz) * s.nx;
        float sx = 0.f;
#pragma unroll
        for (int tx = 0; tx < R; ++tx) {
          const float* row = tb + ((rz + ix[tx]) * s.nint + my) * R;
          float sy = 0.f;
          if constexpr (R == 4) {
            const float4 c4 = __ldg(reinterpret_cast<const float4*>(row));
            sy = fmaf(vy[3], c4.w, fmaf(vy[2], c4.z, fmaf(vy[1], c4.y, vy[0] * c4.x)));
          } else {
#pragma unroll
            for (int t = 0; t < R; t += 2) {
              const float2 c2 = __ldg(reinterpret_cast<const float2*>(row + t));
              sy = fmaf(vy[t + 1], c2.y, fmaf(vy[t], c2.x, sy));
            }
          }
          sx = fmaf(vx[tx], sy, sx);
        }
        sz = fmaf(zval(tz), sx, sz);
      }
      take(jM, sz);
    }
  } else {
    int iy[R];
#pragma unroll
    for (int t = 0; t < R; ++t) iy[t] = min(max(by + t, 0), s.ny - 1);
#pragma unroll UN
    for (int jM = 0; jM < nM; ++jM) {
      ahead(jM);
      const T* cb = s.src + (int64_t)jM * s.npts;
      T sz = 0;
#pragma unroll UNZ
      for (int tz = 0; tz < R; ++tz) {
        T sx = 0;
#pragma unroll
        for (int tx = 0; tx < R; ++tx) {
          const T* row = cb + ((int64_t)(bz + tz) * s.nx + ix[tx]) * s.ny;
          T sy = vy[0] * row[iy[0]];
#pragma unroll
          for (int ty = 1; ty < R; ++ty) sy = fma(vy[ty], row[iy[ty]], sy);
          sx = fma(vx[tx], sy, sx);
        }
        sz = fma(zval(tz), sx, sz);
      }
      take(jM, sz);
    }
  }
  return true;
}

// acc[iM] += sum_jM w[iM][jM](p) E[jM]
template <int NM, typename T>
__device__ __forceinline__ void cpl_add(const T* w, int p, int n_act, const T* E, T* acc) {
#pragma unroll
  for (int iM = 0; iM < NM; ++iM)
#pragma unroll
    for (int jM = 0; jM < NM; ++jM) acc[iM] = fma(w[(int64_t)(iM * NM + jM) * n_act + p], E[jM], acc[iM]);
}

template <int R, int NM, typename T>
__global__ void __launch_bounds__(128) k_apply_coupling(const __grid_constant__ CplArgs<T> a) {
  int ci = 0;
  while (ci + 1 < a.ncomp && (int)blockIdx.x >= a.c[ci + 1].first) ++ci;
  const CplComp<T>& c = a.c[ci];
  const int item = ((int)blockIdx.x - c.first) * blockDim.x + threadIdx.x;
  T acc[NM], E[NM];
  auto eval = [&](const CplSource<T>& s, int p) {
    return cpl_eval<R, NM, R, T>(s, p, c.n_act, NM, a.sdir, a.sq, [](int) {}, [&](int jM, T v) { E[jM] = v; });
  };
#pragma unroll
  for (int m = 0; m < NM; ++m) acc[m] = (T)0;
  if (!c.mirror) {
    if (item >= c.n_act) return;
    bool any = false;
    for (int s = 0; s < c.ns; ++s) {
      if (!eval(c.s[s], item)) continue;
      cpl_add<NM, T>(c.s[s].w, item, c.n_act, E, acc);
      any = true;
    }
    if (!any) return;
    T* y = c.y + c.act_pt[item];
#pragma unroll
    for (int iM = 0; iM < NM; ++iM) y[(int64_t)iM * c.npts] += acc[iM];
    return;
  }
  // planes zeta and n_z - 1 - zeta
  const int zeta = item / c.nxy;
  if (2 * zeta >= c.nz) return;
  const int p = item, pm = item + (c.nz - 1 - 2 * zeta) * c.nxy;
  T accm[NM];
#pragma unroll
  for (int m = 0; m < NM; ++m) accm[m] = (T)0;
  bool any = false;
  if (eval(c.s[0], p)) {
    cpl_add<NM, T>(c.s[0].w, p, c.n_act, E, acc);
    cpl_add<NM, T>(c.s[1].w, pm, c.n_act, E, accm);
    any = true;
  }
  if (eval(c.s[0], pm)) {
    cpl_add<NM, T>(c.s[0].w, pm, c.n_act, E, accm);
    cpl_add<NM, T>(c.s[1].w, p, c.n_act, E, acc);
    any = true;
  }
  if (!any) return;
  T *y = c.y + c.act_pt[p], *ym = c.y + c.act_pt[pm];
#pragma unroll
  for (int iM = 0; iM < NM; ++iM) {
    y[(int64_t)iM * c.npts] += acc[iM];
    ym[(int64_t)iM * c.npts] += accm[iM];
  }
}

// The same with n_M known at run time (NA = 12; more bodies take the compiler minutes) or in double-float: one body of
// taps, each value going straight into the sums of every M'.  Bound by latency at 128 .. 255 registers, so
//   * the weights of an M'' are loaded before its taps (predicated, not branched over: the loads have to be in flight
//     together);
//   * the two points of a mirrored pair are two threads of a block: each evaluates its own position, adds it with its
//     own weights and hands what it is worth at the other point over in shared memory.
// Against one thread for both points with kept values and a weight loop unrolled to 12 x 12: float64 He J = 5 / 7 / 10
// on 40 x 40 x 8 (whole application) 358 / 495 / 713 -> 322 / 434 / 610 us, He J = 10 on 58 x 58 x 6 525 -> 433 us;
// float32 J = 8 155 -> 106 us; double-float He L = 0 96 x 96 x 24 362 -> 220 us, Ps- L = 2 242 -> 193 us, J = 6 on
// 30 x 30 x 6 118 -> 102 us.  float64 takes the z taps in a loop (unrolled: J = 10 723 us), float32 and double-float
// unrolled (in a loop: float32 J = 8 142 us).
template <int R, int NA, typename T>
__global__ void __launch_bounds__(128) k_apply_coupling_any(const __grid_constant__ CplArgs<T> a) {
  constexpr int kUnZ = std::is_same<T, double>::value ? 1 : R;
  __shared__ T give[NA][128];
  __shared__ int hit[128];
  int ci = 0;
  while (ci + 1 < a.ncomp && (int)blockIdx.x >= a.c[ci + 1].first) ++ci;
  const CplComp<T>& c = a.c[ci];
  const int blk = (int)blockIdx.x - c.first, tid = threadIdx.x, nM = NA < kMaxM ? NA : a.nM;
  int q, r = 0;  // this thread's point, the mirrored one
  bool live;
  if (c.mirror) {
    const int i = blk * 64 + (tid & 63), zeta = i / c.nxy, im = i + (c.nz - 1 - 2 * zeta) * c.nxy;
    live = 2 * zeta < c.nz;
    q = tid < 64 ? i : im;
    r = tid < 64 ? im : i;
  } else {
    q = blk * 128 + tid;
    live = q < c.n_act;
  }
  T own[NA], oth[NA];
#pragma unroll
  for (int m = 0; m < NA; ++m) own[m] = oth[m] = (T)0;
  bool any = false;
  if (live) {
    const int ns = c.mirror ? 1 : c.ns;
    for (int s = 0; s < ns; ++s) {
      const T *wq = c.s[s].w + q, *wr = c.s[1].w + r;
      const int64_t row = (int64_t)nM * c.n_act;
      T w0[NA], w1[NA];
      any |= cpl_eval<R, 1, kUnZ, T>(
          c.s[s], q, c.n_act, nM, a.sdir, a.sq,
          [&](int jM) {
#pragma unroll
            for (int m = 0; m < NA; ++m)
              if (m < nM) {
                w0[m] = wq[m * row + (int64_t)jM * c.n_act];
                if (c.mirror) w1[m] = wr[m * row + (int64_t)jM * c.n_act];
              }
          },
          [&](int jM, T v) {
#pragma unroll
            for (int m = 0; m < NA; ++m)
              if (m < nM) {
                own[m] = fma(w0[m], v, own[m]);
                if (c.mirror) oth[m] = fma(w1[m], v, oth[m]);
              }
          });
    }
  }
  if (c.mirror) {
    hit[tid] = any;
#pragma unroll
    for (int m = 0; m < NA; ++m)
      if (m < nM) give[m][tid] = oth[m];
    __syncthreads();
    any = any || hit[tid ^ 64];
#pragma unroll
    for (int m = 0; m < NA; ++m)
      if (m < nM) own[m] = own[m] + give[m][tid ^ 64];
  }
  if (!live || !any) return;
  T* y = c.y + c.act_pt[q];
#pragma unroll
  for (int m = 0; m < NA; ++m)
    if (m < nM) y[(int64_t)m * c.npts] += own[m];
}

// The y coefficients of a component regrouped by y interval: T[row][m][t] = c[row][q m - d + t] for every
// (M', k, i) row, interval m and tap t (0 outside the basis), so that the R taps a point of interval m
// reads are contiguous and aligned.  One thread per (row, interval); blockIdx.y = component.
struct StageArgs {
  const float* c[3];
  float* T[3];
  int64_t rows[3];
  int ny[3], nint[3];
  int q, d;
};
template <int R>
__global__ void __launch_bounds__(256) k_stage_ytaps(const StageArgs a) {
  const int cq = blockIdx.y, nint = a.nint[cq], ny = a.ny[cq];
  const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= a.rows[cq] * nint) return;
  const int64_t row = gid / nint;
  const int m = (int)(gid - row * nint);
  const float* cr = a.c[cq] + row * ny;
  float v[R];
#pragma unroll
  for (int t = 0; t < R; ++t) {
    const int j = a.q * m - a.d + t;
    v[t] = (j >= 0 && j < ny) ? cr[j] : 0.f;
  }
  float* o = a.T[cq] + gid * R;
  if constexpr (R == 4) {
    *reinterpret_cast<float4*>(o) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int t = 0; t < R; t += 2) *reinterpret_cast<float2*>(o + t) = make_float2(v[t], v[t + 1]);
  }
}

template <int R, int NM, typename T>
void run_coupling(const CplArgs<T>& a, int grid, cudaStream_t stream) {
  k_apply_coupling<R, NM, T><<<grid, 128, 0, stream>>>(a);
}
// (25 to 50 s of the compiler each: in files of their own)
extern template void run_coupling<6, 4, double>(const CplArgs<double>&, int, cudaStream_t);
extern template void run_coupling<6, 5, double>(const CplArgs<double>&, int, cudaStream_t);
extern template void run_coupling<6, 6, double>(const CplArgs<double>&, int, cudaStream_t);

}  // namespace fmcpl

namespace fmi {

using namespace fmcpl;

// y += the V^(s) coupling of x, every component in one launch (float32: on sources regrouped by y interval first).
template <typename T>
int apply_coupling(fm_ctx* c, const T* x, T* y, bool timed) {
  const int RT = c->comps[0].r;
  if constexpr (std::is_same<T, float>::value) {
    StageArgs st;
    std::memset(&st, 0, sizeof(st));
    int64_t most = 0;
    double bytes = 0.0;
    for (size_t k = 0; k < c->comps.size(); ++k) {
      const Comp& cp = c->comps[k];
      st.c[k] = x + cp.off;
      st.T[k] = c->ystage32 + cp.ystage_off;
      st.rows[k] = (int64_t)c->nM * cp.nz * cp.nx;
      st.ny[k] = cp.ny;
      st.nint[k] = cp.ay.nint;
      most = std::max(most, st.rows[k] * cp.ay.nint);
      bytes += 4.0 * (double)st.rows[k] * (cp.ny + (double)cp.ay.nint * RT);
    }
    st.q = c->comps[0].ay.q;
    st.d = 1;
    const dim3 g((unsigned)((most + 255) / 256), (unsigned)c->comps.size());
    const int tk_ = timed ? prof_begin(c, FM_KERNEL_COUPLING) : -1;
    if (RT == 6) k_stage_ytaps<6><<<g, 256, 0, c->stream>>>(st);
    else k_stage_ytaps<4><<<g, 256, 0, c->stream>>>(st);
    prof_end(c, tk_, 0.0, bytes);
    c->launches++;
  }
  const bool any_nM = std::is_same<T, dd>::value || c->nM > (RT == 6 ? 6 : 5);
  CplArgs<T> a;
  std::memset(&a, 0, sizeof(a));
  a.nM = c->nM;
  a.sdir = 1;
  a.sq = c->comps[0].ay.q;
  int grid = 0;
  double fl = 0.0, by = 0.0;
  for (auto& cp : c->comps) {
    if (cp.n_act == 0 || cp.sources.empty()) continue;
    const ApplyTabs<T> tb = tabs_of<T>(cp);
    CplComp<T>& f = a.c[a.ncomp++];
    f.y = y + cp.off; f.npts = cp.npts; f.n_act = cp.n_act; f.act_pt = cp.act_pt; f.ns = (int)cp.sources.size();
    f.mirror = cp.cpl_mirror ? 1 : 0; f.nz = cp.nz; f.nxy = cp.n_act / cp.nz; f.first = grid;
    for (int s = 0; s < f.ns; ++s) {
      const Comp& src = c->comps[cp.sources[s].src];
      CplSource<T>& q = f.s[s];
      const int tab = cp.cpl_mirror ? 0 : s;  // mirrored: source 0's taps serve both
      q.base = cp.cpl_base + (int64_t)tab * 3 * cp.n_act;
      q.val = tb.cval + (int64_t)tab * 3 * RT * cp.n_act;
      q.w = tb.cw + (int64_t)s * c->nM * c->nM * cp.n_act;
      q.src = x + src.off; q.npts = src.npts; q.nx = src.nx; q.ny = src.ny; q.nz = src.nz; q.nint = src.ay.nint;
      if constexpr (std::is_same<T, float>::value) q.stage = c->ystage32 + src.ystage_off;
    }
    const int64_t items = cp.cpl_mirror ? (int64_t)(cp.nz / 2) * f.nxy * (any_nM ? 2 : 1) : cp.n_act;
    grid += (int)((items + 127) / 128);
    // per evaluation 2 (R^3 + R^2 + R) flops per M'', per point and source 2 n_M^2 for the weights
    const double cfl = 2.0 * (RT * RT * RT + RT * RT + RT) * c->nM;
    fl += (double)cp.n_act * (cfl * (cp.cpl_mirror ? 1 : f.ns) + 2.0 * f.ns * c->nM * c->nM);
    by += (double)cp.n_act * (4.0 + 2.0 * c->nM * sizeof(T) +
                              (cp.cpl_mirror ? 1 : f.ns) * (12.0 + 3.0 * RT * sizeof(T)) + f.ns * c->nM * c->nM * sizeof(T));
  }
  if (grid == 0) return FM_OK;
  const int tk_ = timed ? prof_begin(c, FM_KERNEL_COUPLING) : -1;
  const int key = (RT == 6 ? 16 : 0) + c->nM;
  if constexpr (std::is_same<T, dd>::value) {
    switch (key) {
      case 1: k_apply_coupling_any<4, 1, T><<<grid, 128, 0, c->stream>>>(a); break;
      case 2: k_apply_coupling_any<4, 2, T><<<grid, 128, 0, c->stream>>>(a); break;
      case 3: k_apply_coupling_any<4, 3, T><<<grid, 128, 0, c->stream>>>(a); break;
      case 4: k_apply_coupling_any<4, 4, T><<<grid, 128, 0, c->stream>>>(a); break;
      case 5: k_apply_coupling_any<4, 5, T><<<grid, 128, 0, c->stream>>>(a); break;
      case 17: k_apply_coupling_any<6, 1, T><<<grid, 128, 0, c->stream>>>(a); break;
      case 18: k_apply_coupling_any<6, 2, T><<<grid, 128, 0, c->stream>>>(a); break;
      case 19: k_apply_coupling_any<6, 3, T><<<grid, 128, 0, c->stream>>>(a); break;
      case 20: k_apply_coupling_any<6, 4, T><<<grid, 128, 0, c->stream>>>(a); break;
      case 21: k_apply_coupling_any<6, 5, T><<<grid, 128, 0, c->stream>>>(a); break;
      case 22: k_apply_coupling_any<6, 6, T><<<grid, 128, 0, c->stream>>>(a); break;
      default:
        if (RT == 6) k_apply_coupling_any<6, kMaxM, T><<<grid, 128, 0, c->stream>>>(a);
        else k_apply_coupling_any<4, kMaxM, T><<<grid, 128, 0, c->stream>>>(a);
    }
  } else {
    switch (key) {
      case 1: run_coupling<4, 1, T>(a, grid, c->stream); break;
      case 2: run_coupling<4, 2, T>(a, grid, c->stream); break;
      case 3: run_coupling<4, 3, T>(a, grid, c->stream); break;
      case 4: run_coupling<4, 4, T>(a, grid, c->stream); break;
      case 5: run_coupling<4, 5, T>(a, grid, c->stream); break;
      case 17: run_coupling<6, 1, T>(a, grid, c->stream); break;
      case 18: run_coupling<6, 2, T>(a, grid, c->stream); break;
      case 19: run_coupling<6, 3, T>(a, grid, c->stream); break;
      case 20: run_coupling<6, 4, T>(a, grid, c->stream); break;
      case 21: run_coupling<6, 5, T>(a, grid, c->stream); break;
      case 22: run_coupling<6, 6, T>(a, grid, c->stream); break;
      default:
        if (RT == 6) k_apply_coupling_any<6, kMaxM, T><<<grid, 128, 0, c->stream>>>(a);
        else k_apply_coupling_any<4, kMaxM, T><<<grid, 128, 0, c->stream>>>(a);
    }
  }
  prof_end(c, tk_, fl, by);
  c->launches++;
  FM_CUDA(cudaGetLastError());
  return FM_OK;
}

}  // namespace fmi
