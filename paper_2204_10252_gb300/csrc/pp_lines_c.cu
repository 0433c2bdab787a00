// Row and column FFT stages, lengths PP_LINES_C (see pp_lines.cuh).
#include "pp_lines.cuh"

namespace pp {
PP_LINES_UNIT(c, PP_LINES_C)
}  // namespace pp
