// Internal view of the library's handle, shared by its translation units
// (the C ABI only exposes it as an opaque pointer).
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <string>
#include <vector>

#include "../../include/cs_ngf.h"
#include "kernels.cuh"

struct cs_ngf_fixed {
  using Geo = csngf::Geo;
  using RotIn = csngf::RotIn;
  using RotBounds = csngf::RotBounds;
  using FixedBox = csngf::FixedBox;
  int device = 0;
  Geo g{};
  float eps = 1e-5f, gamma = 0.5f;
  int batch = 1;               // rotations the workspace holds at the longest lengths
  int group_cap = 1;           // most rotations of a launch group: B_hat, M_hat and keys are sized for them
  int sumA = 0;
  // FFT lengths the buffers are sized for (the automatic or requested ones);
  // g.Pz/Py/Px are the lengths in use, which bound-limited padding
  // (pad_mode CS_NGF_PAD_BOUND) lowers per call
  int alloc_pad[3] = {0, 0, 0};
  int pad_mode = 0;
  float* A_keep = nullptr;     // copies of A and M_A: the fixed spectra are
  uint8_t* MA_keep = nullptr;  // recomputed when the lengths in use change
  RotIn* boxA = nullptr;       // device: the fixed volume's box (origin)
  int extA[3] = {0, 0, 0};     // its extents in use, and the slabs [a0, a1] its mask holds
  int a0[3] = {0, 0, 0}, a1[3] = {-1, -1, -1};
  // per-rotation mask counts and bounds of a call and its rotations regrouped
  // by FFT lengths (bound-limited padding), grown on demand to the call's R
  int* allm = nullptr;         // device, of up to kCountRotations: sums, then slab counts [nz + ny + nx]
  RotBounds* allb_h = nullptr; // [R], pinned host memory the bounds kernel writes to
  int* perm_d = nullptr;       // device: original index of each regrouped rotation
  float* perm_score = nullptr; // device results in regrouped order
  int32_t* perm_shift = nullptr;
  int allb_cap = 0, allm_cap = 0;
  // lengths the overlap rule gives (n + max(-lo, hi)): those of the last class
  // reported, the sets of the last scoring call and their rotation counts
  int rule_pad[3] = {0, 0, 0};
  int length_sets = 1;
  std::vector<int> last_pads, last_counts;
  // transform lengths of the last scoring call's launch classes (see
  // csngf::detail::ClassGeom) and their rotation counts
  std::vector<int> run_pads, run_counts;
  // transforms take only the masks' boxes, at lengths as short as those allow
  // (the FP32 form with bound-limited padding and the built-in splits)
  bool boxed = false;
  bool spectra_ok = false;     // UV holds A's spectra at g.Pz, Py, Px
  // split variant of each FFT pass at the lengths in use (fwd_x, fwd_y, zmac,
  // inv_y, inv_x): 0 unless autotuning chose the alternative (autotune 1) or
  // the alternatives are requested outright (autotune 2)
  int autotune = 0;
  int vars[5] = {0, 0, 0, 0, 0};
  size_t f02_elems = 0, f13_elems = 0, zx_elems = 0;   // per rotation at the longest lengths
  float2* UV = nullptr;
  float* Bh = nullptr;
  uint8_t* Mh = nullptr;
  float4* BQ = nullptr;        // x-pairs of rows y, y+1 (B[i], B[i+1], B[i+sy], B[i+sy+1]) of the current call
  uint8_t* C8 = nullptr;       // corner codes of M_B of the current call
  uint8_t* N8 = nullptr;       // cells near its mask, and a scratch volume before them [2][nvox]
  int* mbox = nullptr;         // its mask's cell box (k_pack_floating)
  bool near = false;           // N8 holds the current call's
  float2* F02 = nullptr;
  float2* F13 = nullptr;
  int* msum = nullptr;
  int* margA = nullptr;        // slab counts of M_A per axis [nz | ny | nx]
  int* margB = nullptr;        // the same for each rotated mask of a batch
  RotBounds* bounds = nullptr; // per rotation of a batch (full padding)
  unsigned long long* keys = nullptr;   // per rotation; Geo::wait_err[-1, 0] is the entry before them
  int* wait_h = nullptr;       // pinned: [0] the last call whose passes' waits ran out, [1] spectra among them
  int call_id = 0;             // number of the last call staged
  FixedBox* fbox_h = nullptr;  // pinned host memory k_fixed_box writes to
  float2* zx = nullptr;        // X of the tensor-core z pass (reduced-precision forms), per launch group
  // rotations: pinned host memory, copied to the device by a kernel, grown on demand
  RotIn* rot_h = nullptr;
  RotIn* rot_d = nullptr;
  int rot_cap = 0;
  cudaEvent_t rot_ev = nullptr;
  // host-buffer entry point staging
  float* stage_B = nullptr;
  uint8_t* stage_M = nullptr;
  float* res_score = nullptr;  // pinned host memory the last kernel writes results to
  int32_t* res_shift = nullptr;
  int res_cap = 0;
  size_t fixed_bytes = 0, workspace_bytes = 0;
  // per-stage CUDA-event timing (cs_ngf_set_profiling)
  bool profiling = false;
  struct Span { int stage; cudaEvent_t a, b; };
  std::vector<Span> spans;
  // one call at a time: set while a host thread is inside a call on this
  // handle (a second thread gets CS_NGF_EBUSY)
  std::atomic<int> busy{0};
  // recorded on the caller's stream at the end of every call; the next call
  // waits for it on its own stream, so calls on different streams do not
  // overlap on the workspace
  cudaEvent_t order_ev = nullptr;
};

namespace csngf {
namespace detail {

// record the calling thread's error detail (cs_ngf_last_error) and return s
cs_ngf_status fail(cs_ngf_status s, const std::string& msg);
// a call's floating volume and rotations on the device: (B, M_B) -> f->BQ, f->C8,
// host FP64 quaternions -> FP32 matrices in f->rot_h[0..R) and f->rot_d[0..R)
cs_ngf_status stage_call(cs_ngf_fixed* f, const float* B, const uint8_t* MB, const double* quats, int R,
                         cudaStream_t st);
// Rotations scored together: FFT lengths, box extents and shift windows per
// axis (z, y, x), and the end of the class in the call's regrouped order.
struct ClassGeom { int pad[3], ext[3], win[3], end; };
struct Plan {
  std::vector<int> perm;         // original index of the i-th regrouped rotation (empty: unchanged)
  std::vector<ClassGeom> cls;
};
// Bound-limited padding (pad_mode CS_NGF_PAD_BOUND): the R uploaded
// rotations of the floating volume packed by stage_call, grouped into
// classes by the FFT lengths their admitted shifts need, their boxes uploaded
// in class order.  Synchronises `st`.  In full mode: one class with the
// lengths in use.
cs_ngf_status plan_classes(cs_ngf_fixed* f, int R, cudaStream_t st, Plan& plan);
// switch the handle to a class's geometry (recomputing the fixed spectra if
// the FFT lengths change)
cs_ngf_status set_class(cs_ngf_fixed* f, const ClassGeom& c, cudaStream_t st);
// score rotations [r0, r0 + n) of the uploaded set into best_score / best_shift
// (device, indexed from r0), in launch groups of f->batch
cs_ngf_status score_range(cs_ngf_fixed* f, int r0, int n, float* best_score, int32_t* best_shift,
                          cudaStream_t st);
// ECUDA if a wait of the last call's passes ran out; the caller has
// synchronised its stream
cs_ngf_status wait_status(const cs_ngf_fixed* f);
// validate dims / cfg and return the FFT lengths; EINVAL / EUNSUPPORTED on error
cs_ngf_status resolve_pads(const int32_t dims[3], const cs_ngf_config& cfg, int pad[3]);
// the automatic launch group: what a third of the free device memory holds, 1 .. most
int auto_batch(const int32_t dims[3], const int pad[3], int measure, int precision, int tensor_cores, int most);
// device bytes a handle of these dims, FFT lengths and batch allocates
size_t handle_bytes(const int32_t dims[3], const int pad[3], int batch, int measure, int precision,
                    int tensor_cores);

}  // namespace detail
}  // namespace csngf
