// Column-resident Cartesian kernels, lengths PP_CART_A (see pp_cart_cols.cuh).
#include "pp_cart_cols.cuh"

namespace pp {
PP_CART_UNIT(a, PP_CART_A)
}  // namespace pp
