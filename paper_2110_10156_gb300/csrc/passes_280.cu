// FFT passes instantiated for transform length 280 (box transforms).
#include "passes.cuh"

namespace csngf {
CSNGF_INSTANTIATE_PASSES(280)
}  // namespace csngf
