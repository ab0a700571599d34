// FP32 basket kernels, widths 48 and 56, Euler.
#define GBMC_BASKET_IMPL
#include "k_basket.cuh"

namespace gbmc {
GBMC_INSTANTIATE_BASKET(48, MC_EULER)
GBMC_INSTANTIATE_BASKET(56, MC_EULER)
}  // namespace gbmc
