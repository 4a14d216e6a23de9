#include "fm_coupling.cuh"

namespace fmi {
template int apply_coupling<double>(fm_ctx*, const double*, double*, bool);
}  // namespace fmi
