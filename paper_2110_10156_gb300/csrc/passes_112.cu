// FFT passes instantiated for transform length 112 (box transforms).
#include "passes.cuh"

namespace csngf {
CSNGF_INSTANTIATE_PASSES(112)
}  // namespace csngf
