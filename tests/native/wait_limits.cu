// The y and z passes with one bulk copy left out; see wait_limits.h.
#include "wait_limits.h"

using namespace csngf;

// pass 0: k_fwd_y, four groups of four planes a block; pass 1: k_zpass, two sets
// of rotations a block.  Returns the CUDA error; *flag: the error flag.
extern "C" int run_pass(int pass, int drop, int* flag) {
  constexpr int P = 16, R = 8;
  Geo g{};
  g.nz = 16; g.ny = g.nx = 8;
  g.Pz = pass ? 32 : 16; g.Py = g.Px = P;
  g.vz = 31; g.vy = g.vx = 15;
  g.ez = 16; g.ey = g.ex = 8;
  g.wz = g.vz; g.wy = g.vy;
  g.nch = 3; g.nf = 4;
  for (int j = 0; j < 4; ++j) g.scale0[j] = g.scale1[j] = 1.0f;
  const size_t n0 = (size_t)R * 4 * g.ez * P * ky_total(P);           // F0, F1 values at most
  const size_t n2 = (size_t)R * P * g.wz * ky_total(P), nuv = (size_t)7 * (P / 2 + 1) * ky_total(P) * 32;
  float2 *F0 = nullptr, *F1 = nullptr, *F2 = nullptr, *UV = nullptr;
  RotIn* rot = nullptr;
  int* err = nullptr;                               // [spectra, group]
  const int zero = 0;
  cudaMalloc(&F0, n0 * sizeof(float2));
  cudaMalloc(&F1, n0 * sizeof(float2));
  cudaMalloc(&F2, n2 * sizeof(float2));
  cudaMalloc(&UV, nuv * sizeof(float2));
  cudaMalloc(&rot, R * sizeof(RotIn));
  cudaMalloc(&err, 2 * sizeof(int));
  if (cudaError_t e = cudaGetLastError()) return e;
  cudaMemset(F0, 0, n0 * sizeof(float2));
  cudaMemset(F1, 0, n0 * sizeof(float2));
  cudaMemset(UV, 0, nuv * sizeof(float2));
  cudaMemset(rot, 0, R * sizeof(RotIn));            // window of one slot
  cudaMemset(err, 0, 2 * sizeof(int));
  cudaMemcpyToSymbol(tc::g_copies, &zero, sizeof(int));
  cudaMemcpyToSymbol(tc::g_drop, &drop, sizeof(int));
  g.wait_err = err + 1;
  if (pass == 0) {
    using C = FwdYCfg<P, 0>;
    k_fwd_y<P, kStoreF32, true, 0><<<dim3(P / 4, 1, R * g.nf), C::NT, C::smem_bytes(g.ey)>>>(F0, F1, g, 4);
  } else {
    using C = ZCfg<32, 0, kZFull>;
    const int q = std::min(C::Q, C::fit(g.ez));
    const size_t smem = C::smem_bytes(q, g.ez);
    set_smem<k_zpass<32, kStoreF32, true, 0, kZFull>>(smem);
    k_zpass<32, kStoreF32, true, 0, kZFull><<<dim3(ky_total(P) / 4, P / 2 + 1, 1), q * C::W * C::N1, smem>>>(
        F1, UV, nullptr, F2, g, R, R, rot);
  }
  cudaError_t e = cudaGetLastError();
  if (!e) e = cudaDeviceSynchronize();
  if (!e) e = cudaMemcpy(flag, err + 1, sizeof(int), cudaMemcpyDeviceToHost);
  cudaFree(F0); cudaFree(F1); cudaFree(F2); cudaFree(UV); cudaFree(rot); cudaFree(err);
  return e;
}
