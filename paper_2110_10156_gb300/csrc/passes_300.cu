// FFT passes instantiated for transform length 300 (box transforms).
#include "passes.cuh"

namespace csngf {
CSNGF_INSTANTIATE_PASSES(300)
}  // namespace csngf
