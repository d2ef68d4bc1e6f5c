// FFT passes instantiated for transform length 72 (box transforms).
#include "passes.cuh"

namespace csngf {
CSNGF_INSTANTIATE_PASSES(72)
}  // namespace csngf
