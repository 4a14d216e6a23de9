#include "fm_coupling.cuh"

namespace fmi {
template int apply_coupling<dd>(fm_ctx*, const dd*, dd*, bool);
}  // namespace fmi
