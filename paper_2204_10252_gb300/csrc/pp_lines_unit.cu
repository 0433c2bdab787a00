// Row and column FFT stages of one length (see pp_lines_lengths.h); the build gives N1
// and N2.
#ifdef PP_N1
#include "pp_lines.cuh"

namespace pp {
template cudaError_t line_launch<PP_N1, PP_N2>(LineOp, const LineUnion&, dim3, cudaStream_t);
}  // namespace pp
#endif
