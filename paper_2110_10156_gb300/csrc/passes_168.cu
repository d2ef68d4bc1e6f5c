// FFT passes instantiated for transform length 168 (box transforms).
#include "passes.cuh"

namespace csngf {
CSNGF_INSTANTIATE_PASSES(168)
}  // namespace csngf
