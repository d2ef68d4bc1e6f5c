// The allocation-free entry point at 16-point lengths (dims up to 8) with one bulk
// copy left out; see wait_limits.h.
#include "wait_limits.h"

namespace csngf {
void set_last_error(const std::string&) {}
#define NO_LENGTH(P)                                                                                       \
  template <> void launch_fwd_x<P>(const float*, const uint8_t*, void*, const RotIn*, Geo, int, cudaStream_t, int) {} \
  template <> void launch_fwd_y<P>(const void*, void*, Geo, int, cudaStream_t, int) {}                     \
  template <> void launch_zmac<P>(const void*, const float2*, float2*, Geo, int, const RotIn*, cudaStream_t, int) {} \
  template <> void launch_prep_z<P>(const float2*, float2*, Geo, cudaStream_t) {}                          \
  template <> void launch_inv_y<P>(const float2*, float2*, Geo, int, const RotIn*, cudaStream_t, int) {}   \
  template <> void launch_inv_x<P>(const float2*, unsigned long long*, float*, Geo, int, const RotIn*, cudaStream_t, int) {}
NO_LENGTH(32)
NO_LENGTH(64)
}  // namespace csngf
#include "noalloc.cu"

// the number of the copy to leave out (-1: none); copies issued since the last call
extern "C" int set_drop(int drop, int* copies) {
  cudaDeviceSynchronize();
  int zero = 0;
  cudaMemcpyFromSymbol(copies, csngf::tc::g_copies, sizeof(int));
  cudaMemcpyToSymbol(csngf::tc::g_copies, &zero, sizeof(int));
  cudaMemcpyToSymbol(csngf::tc::g_drop, &drop, sizeof(int));
  return cudaGetLastError();
}
