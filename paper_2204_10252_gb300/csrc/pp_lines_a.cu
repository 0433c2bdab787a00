// Row and column FFT stages, lengths PP_LINES_A (see pp_lines.cuh).
#include "pp_lines.cuh"

namespace pp {
PP_LINES_UNIT(a, PP_LINES_A)
}  // namespace pp
