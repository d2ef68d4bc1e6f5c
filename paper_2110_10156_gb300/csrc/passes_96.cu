// FFT passes instantiated for transform length 96 (box transforms).
#include "passes.cuh"

namespace csngf {
CSNGF_INSTANTIATE_PASSES(96)
}  // namespace csngf
