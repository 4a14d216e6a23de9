#include "fm_coupling.cuh"

namespace fmcpl {
template void run_coupling<6, 5, double>(const CplArgs<double>&, int, cudaStream_t);
}  // namespace fmcpl
