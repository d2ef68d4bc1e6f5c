// FFT passes instantiated for transform length 56 (box transforms).
#include "passes.cuh"

namespace csngf {
CSNGF_INSTANTIATE_PASSES(56)
}  // namespace csngf
