// FFT passes instantiated for transform length 180 (box transforms).
#include "passes.cuh"

namespace csngf {
CSNGF_INSTANTIATE_PASSES(180)
}  // namespace csngf
