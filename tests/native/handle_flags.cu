// Raises the flag of a handle's fixed spectra, as a pass whose wait ran out does.
#include "handle.h"

extern "C" int raise_spectra_flag(cs_ngf_fixed* f) {
  const int one = 1;
  if (cudaError_t e = cudaDeviceSynchronize()) return e;
  return cudaMemcpy(f->g.wait_err - 1, &one, sizeof(int), cudaMemcpyHostToDevice);
}
