// passes_x_f64.cu - the x passes of the FP64 path (passes_fx.cuh); a translation
// unit of its own so that the passes compile in parallel.
#include "passes_fx.cuh"

namespace scfft {

INST_PASSES_X(double)

}  // namespace scfft
