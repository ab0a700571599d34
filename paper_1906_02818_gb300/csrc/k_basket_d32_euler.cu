// FP32 basket kernels, widths 32 and 40, Euler.
#define GBMC_BASKET_IMPL
#include "k_basket.cuh"

namespace gbmc {
GBMC_INSTANTIATE_BASKET(32, MC_EULER)
GBMC_INSTANTIATE_BASKET(40, MC_EULER)
}  // namespace gbmc
