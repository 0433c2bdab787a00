// Column-resident Cartesian kernels, lengths PP_CART_C (see pp_cart_cols.cuh).
#include "pp_cart_cols.cuh"

namespace pp {
PP_CART_UNIT(c, PP_CART_C)
}  // namespace pp
