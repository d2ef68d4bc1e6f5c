// FFT passes instantiated for transform length 144 (box transforms).
#include "passes.cuh"

namespace csngf {
CSNGF_INSTANTIATE_PASSES(144)
}  // namespace csngf
