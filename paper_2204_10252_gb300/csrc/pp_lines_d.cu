// Row and column FFT stages, lengths PP_LINES_D (see pp_lines.cuh).
#include "pp_lines.cuh"

namespace pp {
PP_LINES_UNIT(d, PP_LINES_D)
}  // namespace pp
