// Row and column FFT stages, lengths PP_LINES_B (see pp_lines.cuh).
#include "pp_lines.cuh"

namespace pp {
PP_LINES_UNIT(b, PP_LINES_B)
}  // namespace pp
