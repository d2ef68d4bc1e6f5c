// FFT passes instantiated for transform length 24 (box transforms).
#include "passes.cuh"

namespace csngf {
CSNGF_INSTANTIATE_PASSES(24)
}  // namespace csngf
