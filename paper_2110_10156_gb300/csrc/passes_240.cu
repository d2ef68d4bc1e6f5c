// FFT passes instantiated for transform length 240 (box transforms).
#include "passes.cuh"

namespace csngf {
CSNGF_INSTANTIATE_PASSES(240)
}  // namespace csngf
