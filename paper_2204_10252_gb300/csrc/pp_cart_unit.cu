// Column-resident Cartesian kernels of one length (see pp_lines_lengths.h); the build
// gives N1 and N2.
#ifdef PP_N1
#include "pp_cart_cols.cuh"

namespace pp {
template cudaError_t cart_cols_launch<PP_N1, PP_N2>(const CartLaunch&, const float2*, const CartChain&, cudaStream_t);
}  // namespace pp
#endif
