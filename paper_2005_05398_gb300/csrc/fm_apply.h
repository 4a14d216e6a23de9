// The operator's device tables in one element type, and the parts of the application and of the preconditioner that
// stand in files of their own: the coupling (fm_coupling.cuh, a translation unit per element type, since its unrolled
// bodies take the compiler longest) and the banded y solves (fm_ysolve.cu).
#pragma once
#include <type_traits>
#include <vector>

#include "fm_internal.h"

namespace fmi {

constexpr int kMaxM = 12;  // largest n_M (J <= 11 for tau = +1)

template <typename T>
struct ApplyTabs {
  const T *Sx, *D2x, *Sy, *D2y, *zt, *qx, *W, *iy2, *cval, *cw;
};

template <typename T>
inline ApplyTabs<T> tabs_of(const Comp& cp);

template <>
inline ApplyTabs<double> tabs_of<double>(const Comp& cp) {
  return {cp.dx.S, cp.dx.D2, cp.dy.S, cp.dy.D2, cp.zt, cp.qx, cp.W, cp.iy2, cp.cpl_val, cp.cpl_w};
}

template <>
inline ApplyTabs<float> tabs_of<float>(const Comp& cp) {
  return {cp.f32.Sx, cp.f32.D2x, cp.f32.Sy, cp.f32.D2y, cp.f32.zt, cp.f32.qx, cp.f32.W, cp.f32.iy2, cp.f32.cval, cp.f32.cw};
}

template <>
inline ApplyTabs<dd> tabs_of<dd>(const Comp& cp) {
  return {cp.tdd.Sx, cp.tdd.D2x, cp.tdd.Sy, cp.tdd.D2y, cp.tdd.zt, cp.tdd.qx, cp.tdd.W, cp.tdd.iy2, cp.tdd.cval, cp.tdd.cw};
}

// y += the V^(s) coupling of x
template <typename T>
int apply_coupling(fm_ctx* c, const T* x, T* y, bool timed);

// Banded y solves of the given components, in place on u[slab][j][i]
template <typename T>
int ysolve_banded(fm_ctx* c, const std::vector<Comp*>& comps, T* u);
int ysolve_init();

}  // namespace fmi
