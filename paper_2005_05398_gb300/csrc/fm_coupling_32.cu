#include "fm_coupling.cuh"

namespace fmi {
template int apply_coupling<float>(fm_ctx*, const float*, float*, bool);
}  // namespace fmi
