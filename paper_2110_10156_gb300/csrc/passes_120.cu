// FFT passes instantiated for transform length 120 (box transforms).
#include "passes.cuh"

namespace csngf {
CSNGF_INSTANTIATE_PASSES(120)
}  // namespace csngf
