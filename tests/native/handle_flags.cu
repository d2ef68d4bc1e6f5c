// Raises the flag of a handle's fixed spectra, as a pass whose wait ran out does.
#include "handle.h"

extern "C" int raise_spectra_flag(cs_ngf_fixed* f) {
  const int one = 1;
  if (cudaError_t e = cudaDeviceSynchronize()) return e;
  return cudaMemcpy(f->g.wait_err - 1, &one, sizeof(int), cudaMemcpyHostToDevice);
}

// The floating mask's cell box as the next call finds it.
extern "C" int read_mask_box(cs_ngf_fixed* f, int* box) {
  if (cudaError_t e = cudaDeviceSynchronize()) return e;
  return cudaMemcpy(box, f->mbox, 6 * sizeof(int), cudaMemcpyDeviceToHost);
}

// Preloaded: every handle that the library itself prepares comes with the flag raised.
#include <dlfcn.h>
#include <cstdlib>
extern "C" cs_ngf_status cs_ngf_prepare_fixed(const float* A, const uint8_t* maskA, const int32_t dims[3],
                                              const cs_ngf_config* cfg, void* stream, cs_ngf_fixed** out) {
  void* lib = dlopen(getenv("CS_NGF_LIB"), RTLD_NOLOAD | RTLD_NOW);
  if (!lib) return CS_NGF_EUNSUPPORTED;
  auto real = reinterpret_cast<decltype(&cs_ngf_prepare_fixed)>(dlsym(lib, "cs_ngf_prepare_fixed"));
  if (cs_ngf_status s = real(A, maskA, dims, cfg, stream, out)) return s;
  return raise_spectra_flag(*out) ? CS_NGF_EINVAL : CS_NGF_OK;
}
