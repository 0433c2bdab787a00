// Column-resident Cartesian kernels, lengths PP_CART_B (see pp_cart_cols.cuh).
#include "pp_cart_cols.cuh"

namespace pp {
PP_CART_UNIT(b, PP_CART_B)
}  // namespace pp
