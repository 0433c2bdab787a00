// Column-resident Cartesian kernels, lengths PP_CART_D (see pp_cart_cols.cuh).
#include "pp_cart_cols.cuh"

namespace pp {
PP_CART_UNIT(d, PP_CART_D)
}  // namespace pp
