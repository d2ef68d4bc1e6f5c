// FFT passes instantiated for transform length 48 (box transforms).
#include "passes.cuh"

namespace csngf {
CSNGF_INSTANTIATE_PASSES(48)
}  // namespace csngf
