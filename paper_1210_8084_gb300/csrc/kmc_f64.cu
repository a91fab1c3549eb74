// kmc_f64.cu -- binary64-state instantiation of the step kernels.
#include "kmc_filter.cuh"

namespace kmc {
KMC_INSTANTIATE(double)
}  // namespace kmc
