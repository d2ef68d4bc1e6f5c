// FFT passes of the all-shift NGF correlation (Cross-Sim-NGF Eq. 6-8).
// Included by one translation unit per FFT length (passes_<P>.cu).
#pragma once

#include "kernels.cuh"

namespace csngf {

// Output index m of a length-P circular correlation sums the linear
// correlation over every shift of its residue class mod P.  With the fixed
// mask on slabs [a0, a1] and the rotated one on [b0, b1] the linear
// correlation lives on chi in [b0 - a1, b1 - a0], so a slot in the admitted
// range [lo, hi] holds its one shift whenever
// P >= max(b1 - a0 - chi_lo, chi_hi - (b0 - a1)) + 1, which the caller
// guarantees (for masks that fill the volume that is n + max(-chi_lo, chi_hi),
// and for every shift 2n - 1).

// Forward-transform inputs: box extents e are zero padded to P.  When
// e <= P/2 the upper half of every step-1 sequence is zero and step 1 is the
// pruned form (FourStep::step1_half); otherwise all N1 inputs are read.
template <class FS, bool HALF>
struct FwdIn {
  static constexpr int NI = HALF ? FS::N1 / 2 : FS::N1;   // step-1 inputs per thread
  template <int S, bool TS = false>
  __device__ __forceinline__ static void step1(float2 (&v)[NI], float2* ex_seq, int n2,
                                               const float2* __restrict__ twN) {
    if constexpr (HALF) FS::template step1_half<S, TS>(v, ex_seq, n2, twN);
    else FS::template step1<S, TS>(v, ex_seq, n2, twN);
  }
  // the same to an exchange whose elements lie W apart, twiddles in shared memory
  template <int S, int W>
  __device__ __forceinline__ static void step1w(float2 (&v)[NI], float2* ex_row, int n2, const float2* tws) {
    if constexpr (HALF) FS::template step1_half<S, true, W>(v, ex_row - n2 * FS::RS * W, n2, tws);
    else FS::template step1<S, true, W>(v, ex_row - n2 * FS::RS * W, n2, tws);
  }
};

// calls f with the storage form of the channel fields as a compile-time constant
template <int P, class F>
static void by_store(int store, F&& f) {
  if constexpr (box_only(P)) f(std::integral_constant<int, kStoreF32>{});
  else if (store == kStoreBF16) f(std::integral_constant<int, kStoreBF16>{});
  else if (store == kStoreF16) f(std::integral_constant<int, kStoreF16>{});
  else f(std::integral_constant<int, kStoreF32>{});
}

// calls f with split variant v of length P (0 where P has no second split)
template <int P, class F>
static void by_split(int v, F&& f) {
  if constexpr (has_alt_split(P)) {
    if (v == 1) {
      f(std::integral_constant<int, 1>{});
      return;
    }
  }
  f(std::integral_constant<int, 0>{});
}

// calls f with whether a box extent e fills at most half the length (where the
// split's first factor is even, so that the pruned first step exists)
template <int P, int V, class F>
static void by_half(int e, F&& f) {
  if constexpr (SplitV<P, V>::N1 % 2 == 0 && !box_only(P)) {
    if (2 * e <= P) {
      f(std::true_type{});
      return;
    }
  }
  f(std::false_type{});
}

template <class K>
static void set_smem(K kern, size_t bytes) {
  if (bytes > 48 * 1024)
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// ---------------------------------------------------------------------------
// fwd_x: Eq. 1 NGF of the resampled volume, the Eq. 6 channels packed in four
// complex fields, and the x-axis FFT of every row (zero padded to Px).
// Block: ROWS rows of one slab; thread (row, n2) gathers x = N2*n1 + n2.
// ---------------------------------------------------------------------------
// A thread keeps the NGF (x, y, z, mask) of its step-1 inputs across the
// four fields: in registers for half-length inputs, in its own slots of
// shared memory [NI][NT] (float4) for full-length ones, which would spill.
template <int P, bool HALF, int V>
struct FwdXCfg {
  static constexpr int N2 = SplitV<P, V>::N2;
  static constexpr int ROWS = (256 / N2) > 0 ? (256 / N2) : 1;
  static constexpr int NT = ROWS * N2;
  static constexpr int NI = FwdIn<FourStep<P, true, V>, HALF>::NI;
  static constexpr size_t ex_bytes = ((size_t)ROWS * FourStep<P, true, V>::CS * sizeof(float2) + 15) / 16 * 16;
  static constexpr size_t smem_bytes = ex_bytes + (HALF ? 0 : (size_t)NI * NT * sizeof(float4));
  // three blocks per SM (at most 80 registers per thread): the gradient
  // gathers and the per-field barriers leave the pass latency-bound, and the
  // extra resident warps hide more of it than the few spilled registers cost
  // (measured: 200-point lengths 2.13 -> 1.67 ms per 32 rotations, 320-point
  // half-input lengths 72 -> 65 ms per 1000 rotations; 400 and 320 unchanged)
  static constexpr int MIN_BLOCKS = 3;
};

template <int P, int ROWS, int ST, bool HALF, int V>
__global__ void __launch_bounds__(ROWS * SplitV<P, V>::N2, FwdXCfg<P, HALF, V>::MIN_BLOCKS)
k_fwd_x(const float* __restrict__ Bh, const uint8_t* __restrict__ Mh, void* __restrict__ F0,
        const RotIn* __restrict__ rot, Geo g, long long nrows) {
  const float2* __restrict__ tw = kTw<P>.w;
  using FS = FourStep<P, true, V>;
  using FI = FwdIn<FS, HALF>;
  constexpr int N1 = FS::N1, N2 = FS::N2, CS = FS::CS, H = FI::NI;
  extern __shared__ float2 ex[];
  const int t = threadIdx.x;
  const int lrow = t / N2, n2 = t - lrow * N2;
  const long long grow = (long long)blockIdx.x * ROWS + lrow;
  const bool row_ok = grow < nrows;
  const long long rz = row_ok ? grow / g.ey : 0;
  const int yb = row_ok ? (int)(grow - rz * g.ey) : 0;
  const int r = (int)(rz / g.ez), zb = (int)(rz - (long long)r * g.ez);
  const RotBox& bx = rot[r].b;
  const int z = zb + bx.org[0], y = yb + bx.org[1], ox = bx.org[2];   // voxel of box index (zb, yb, 0)

  // x = org + N2*n1 + n2 over ex voxels: with ex <= P/2 only n1 < N1/2 can hold data
  constexpr bool NS = !HALF;                  // NGF staged in shared memory
  constexpr int HR = NS ? 1 : H;
  float vx[HR], vy[HR], vz[HR], mm[HR];
  float4* ngs = reinterpret_cast<float4*>(reinterpret_cast<char*>(ex) + FwdXCfg<P, HALF, V>::ex_bytes);
  const int NTX = ROWS * N2;
  const float* Vol = Bh + (long long)r * g.nvox;
  const uint8_t* M = Mh + (long long)r * g.nvox;
  const long long sy = g.nx, sz = (long long)g.nx * g.ny;
  const int ym = max(y - 1, 0), yp = min(y + 1, g.ny - 1);
  const int zm = max(z - 1, 0), zp = min(z + 1, g.nz - 1);
  const long long base = (long long)z * sz + (long long)y * sy;
  const long long rows_per_field = (long long)g.ez * g.ey;
  const int nrot = (int)(nrows / rows_per_field);
  const bool has_partner = !(r & 1) && r + 1 < nrot;
  // the partner's mask in its own box: offset of its row from M, and its x origin
  long long pbase = 0;
  int pox = 0, pnx = 0;
  if (has_partner) {
    const RotBox& pb = rot[r + 1].b;
    const int pz = zb + pb.org[0], py = yb + pb.org[1];
    pox = pb.org[2];
    pnx = (pz < g.nz && py < g.ny) ? min(g.ex, g.nx - pox) : 0;
    pbase = g.nvox + (long long)pz * sz + (long long)py * sy + pox;
  }
  const bool in_vol = row_ok && z < g.nz && y < g.ny;
  // per element: the NGF times the mask (m^2 = m, so every Eq. 6 product of
  // two masked components equals the product times m, bit for bit) and the
  // mask pair of the mask field coded as m + 2 m2 (m2: the next rotation's mask)
#pragma unroll
  for (int n1 = 0; n1 < H; ++n1) {
    const int xb = N2 * n1 + n2, x = xb + ox;
    float4 q = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    const float m2 = xb < pnx && M[pbase + xb] ? 2.0f : 0.0f;
    q.w = m2;
    if (in_vol && xb < g.ex && x < g.nx) {
      const int xm = max(x - 1, 0), xp = min(x + 1, g.nx - 1);
      const float gx = 0.5f * (__ldg(&Vol[base + xp]) - __ldg(&Vol[base + xm]));
      const float gy = 0.5f * (__ldg(&Vol[(long long)z * sz + (long long)yp * sy + x]) -
                               __ldg(&Vol[(long long)z * sz + (long long)ym * sy + x]));
      const float gz = 0.5f * (__ldg(&Vol[(long long)zp * sz + (long long)y * sy + x]) -
                               __ldg(&Vol[(long long)zm * sz + (long long)y * sy + x]));
      const float inv = rsqrtf(gx * gx + gy * gy + gz * gz + g.eps2);
      const float m = M[base + x] ? 1.0f : 0.0f;
      q = make_float4(m * (gx * inv), m * (gy * inv), m * (gz * inv), m + m2);
    }
    if constexpr (NS) {
      ngs[n1 * NTX + t] = q;
    } else {
      vx[n1] = q.x;
      vy[n1] = q.y;
      vz[n1] = q.z;
      mm[n1] = q.w;
    }
  }
  // Masks are paired across consecutive rotations: the even rotation's mask
  // field carries (M_r, M_{r+1}); an odd rotation has no mask field of its own.
  const bool odd_block = ((blockIdx.x * (long long)ROWS) / rows_per_field & 1) &&
                         (blockIdx.x * (long long)ROWS) / rows_per_field ==
                             (min(blockIdx.x * (long long)ROWS + ROWS, nrows) - 1) / rows_per_field;
#pragma unroll 1
  for (int j = 0; j < g.nf; ++j) {
    if (j == g.nch && odd_block) break;          // uniform over the block
    // Eq. 6 products (squared measure) or Eq. 3 components (unsquared); the
    // mask field comes last
    const int code = j == g.nch ? 3 : (g.nch == 3 ? j : 4 + j);
    float2 v[H];
    // this field's inputs, with the field's product chosen at compile time
    auto inputs = [&](auto cc) {
      constexpr int CODE = decltype(cc)::value;
#pragma unroll
      for (int n1 = 0; n1 < H; ++n1) {
        float X, Y, Z, w;
        if constexpr (NS) {
          const float4 q = ngs[n1 * NTX + t];   // this thread's own slot
          X = q.x; Y = q.y; Z = q.z; w = q.w;
        } else {
          X = vx[n1 < HR ? n1 : 0]; Y = vy[n1 < HR ? n1 : 0]; Z = vz[n1 < HR ? n1 : 0];
          w = mm[n1 < HR ? n1 : 0];
        }
        if constexpr (CODE == 0) v[n1] = make_float2(X * X, Y * Y);
        else if constexpr (CODE == 1) v[n1] = make_float2(Z * Z, X * Y);
        else if constexpr (CODE == 2) v[n1] = make_float2(X * Z, Y * Z);
        else if constexpr (CODE == 4) v[n1] = make_float2(X, Y);
        else if constexpr (CODE == 5) v[n1] = make_float2(Z, 0.0f);
        else {                                   // mask pair (M_r, M_{r+1}); w = m + 2 m2
          const float m2 = w >= 2.0f ? 1.0f : 0.0f;
          v[n1] = (r & 1) ? make_float2(0.0f, 0.0f) : make_float2(w - 2.0f * m2, m2);
        }
      }
    };
    switch (code) {
      case 0: inputs(std::integral_constant<int, 0>{}); break;
      case 1: inputs(std::integral_constant<int, 1>{}); break;
      case 2: inputs(std::integral_constant<int, 2>{}); break;
      case 4: inputs(std::integral_constant<int, 4>{}); break;
      case 5: inputs(std::integral_constant<int, 5>{}); break;
      default: inputs(std::integral_constant<int, 3>{}); break;
    }
    FI::template step1<-1>(v, ex + lrow * CS, n2, tw);
    __syncthreads();
    if (t < ROWS * N1) {
      const int lr = t / N1, k1 = t - lr * N1;
      const long long gr = (long long)blockIdx.x * ROWS + lr;
      const bool skip_row = j == g.nch && ((gr / rows_per_field) & 1);   // odd rotation: no mask field
      if (gr < nrows && !skip_row) {
        float2 u[N2];
        FS::template step2<-1>(u, ex + lr * CS, k1);
        const long long rz2 = gr / g.ey;
        const int y2 = (int)(gr - rz2 * g.ey);
        const int r2 = (int)(rz2 / g.ez), z2 = (int)(rz2 - (long long)r2 * g.ez);
        char* fld = Fields<ST>::field(F0, g, rows_per_field * P, r2, j);
        const long long row = ((long long)z2 * g.ey + y2) * P;
        const float sc = field_scale(g.scale0, j);
        if (j == g.nch) {
#pragma unroll
          for (int k2 = 0; k2 < N2; ++k2) Fields<ST>::put(fld, row + k1 + N1 * k2, u[k2], true, sc);
        } else {
#pragma unroll
          for (int k2 = 0; k2 < N2; ++k2) Fields<ST>::put(fld, row + k1 + N1 * k2, u[k2], false, sc);
        }
      }
    }
    __syncthreads();
  }
}

template <int P, bool HALF, int V>
void launch_fwd_x_t(const float* Bh, const uint8_t* Mh, void* F0, const RotIn* rot, Geo g, int nrot,
                    cudaStream_t st) {
  constexpr int N2 = SplitV<P, V>::N2;
  constexpr int ROWS = FwdXCfg<P, HALF, V>::ROWS;
  const long long nrows = (long long)nrot * g.ez * g.ey;
  const size_t smem = FwdXCfg<P, HALF, V>::smem_bytes;
  const unsigned blocks = (unsigned)((nrows + ROWS - 1) / ROWS);
  auto go = [&](auto kern) {
    set_smem(kern, smem);
    kern<<<blocks, ROWS * N2, smem, st>>>(Bh, Mh, F0, rot, g, nrows);
  };
  by_store<P>(g.store, [&](auto st) { go(k_fwd_x<P, ROWS, decltype(st)::value, HALF, V>); });
}

template <int P>
void launch_fwd_x(const float* Bh, const uint8_t* Mh, void* F0, const RotIn* rot, Geo g, int nrot,
                  cudaStream_t st, int v) {
  by_split<P>(v, [&](auto vc) {
    constexpr int V = decltype(vc)::value;
    by_half<P, V>(g.ex, [&](auto hc) {
      launch_fwd_x_t<P, decltype(hc)::value, V>(Bh, Mh, F0, rot, g, nrot, st);
    });
  });
}

// ---------------------------------------------------------------------------
// fwd_y: y-axis FFT of every column of F0 (rows y >= ey are zero); the output
// is transposed so that ky is contiguous for the z pass.
// Block: W consecutive kx of one (r, j, z) plane.
// ---------------------------------------------------------------------------
// Blocks per SM for the single-transform passes: as many as keep at least
// MINR registers per thread (each of the SM's four sub-partitions holds 16384
// registers for the warps placed on it) and fit in shared memory.
constexpr int pass_blocks(int threads, size_t smem, int minr) {
  int best = 1;
  for (int b = 2; b <= 8; ++b) {
    const int per_sub = (b * ((threads + 31) / 32) + 3) / 4;
    const int regs = (16384 / (32 * per_sub)) / 8 * 8;
    if (regs >= minr && (size_t)b * (smem + 1024) <= 228 * 1024) best = b;
  }
  return best;
}
template <int P, int V> struct FwdYCfg {
  // 16 columns per block; 8 where the second stage is longer than 20 points
  // (more registers per thread: smaller blocks keep several per SM)
  static constexpr int W = SplitV<P, V>::N2 > 20 ? 8 : 16;
  static constexpr int NT = W * SplitV<P, V>::N2;
  static constexpr size_t smem_bytes = (size_t)W * FourStep<P, true, V>::CS * sizeof(float2);
  // the 25- and 32-point second stages need more registers than 16- or 20-point ones
  static constexpr int MIN_BLOCKS = pass_blocks(NT, smem_bytes, SplitV<P, V>::N2 > 20 ? 80 : 48);
};

template <int P, int W, int ST, bool HALF, int V>
__global__ void __launch_bounds__(W * SplitV<P, V>::N2, FwdYCfg<P, V>::MIN_BLOCKS)
k_fwd_y(const void* __restrict__ F0, void* __restrict__ F1, Geo g) {
  const float2* __restrict__ tw = kTw<P>.w;
  using FS = FourStep<P, true, V>;
  using FI = FwdIn<FS, HALF>;
  constexpr int N1 = FS::N1, N2 = FS::N2, CS = FS::CS;
  extern __shared__ float2 ex[];
  const int t = threadIdx.x;
  // kx tiles run fastest over the grid, so the blocks that read the two halves
  // of a 128-byte line of F0 run together and the second one hits in L2
  const long long plane = blockIdx.y;                // ((r * nf) + j) * ez + z
  const long long rj = plane / g.ez;
  const int z = (int)(plane - rj * g.ez);
  const int r = (int)(rj / g.nf), j = (int)(rj - (long long)r * g.nf);
  const bool is_mask = j == g.nch;
  if (is_mask && (r & 1)) return;                    // paired into the even rotation's mask field
  const int kx0 = blockIdx.x * W;
  {
    const int col = t % W, n2 = t / W;
    const int kx = kx0 + col;
    const char* src = Fields<ST>::field(F0, g, (long long)g.ez * g.ey * g.Px, r, j);
    const float isc = 1.0f / field_scale(g.scale0, j);
    const long long zoff = (long long)z * g.ey * g.Px;
    float2 v[FI::NI];                     // y < ey: with ey <= P/2 the upper half is zero
    if (is_mask) {
#pragma unroll
      for (int n1 = 0; n1 < FI::NI; ++n1) {
        const int y = N2 * n1 + n2;
        v[n1] = (y < g.ey && kx < g.Px) ? Fields<ST>::get(src, zoff + (long long)y * g.Px + kx, true, isc)
                                        : make_float2(0.f, 0.f);
      }
    } else {
#pragma unroll
      for (int n1 = 0; n1 < FI::NI; ++n1) {
        const int y = N2 * n1 + n2;
        v[n1] = (y < g.ey && kx < g.Px) ? Fields<ST>::get(src, zoff + (long long)y * g.Px + kx, false, isc)
                                        : make_float2(0.f, 0.f);
      }
    }
    FI::template step1<-1>(v, ex + col * CS, n2, tw);
  }
  __syncthreads();
  if (t < W * N1) {
    const int col = t / N1, k1 = t - col * N1;
    const int kx = kx0 + col;
    if (kx < g.Px) {
      float2 u[N2];
      FS::template step2<-1>(u, ex + col * CS, k1);
      char* dst = Fields<ST>::field(F1, g, (long long)g.ez * g.Px * P, r, j);
      const long long row = ((long long)kx * g.ez + z) * P;       // [kx][z][ky]
      const float sc = field_scale(g.scale1, j);
      if (is_mask) {
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) Fields<ST>::put(dst, row + k1 + N1 * k2, u[k2], true, sc);
      } else {
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) Fields<ST>::put(dst, row + k1 + N1 * k2, u[k2], false, sc);
      }
    }
  }
}

template <int P, int V>
void launch_fwd_y_t(const void* F0, void* F1, Geo g, int nrot, cudaStream_t st) {
  constexpr int W = FwdYCfg<P, V>::W, N2 = SplitV<P, V>::N2;
  const size_t smem = FwdYCfg<P, V>::smem_bytes;
  dim3 grid((unsigned)((g.Px + W - 1) / W), (unsigned)(nrot * g.nf * g.ez));   // y: at most 32 * 4 * 256
  auto go = [&](auto kern) {
    set_smem(kern, smem);
    kern<<<grid, W * N2, smem, st>>>(F0, F1, g);
  };
  by_store<P>(g.store, [&](auto sf) {
    constexpr int ST = decltype(sf)::value;
    by_half<P, V>(g.ey, [&](auto hc) { go(k_fwd_y<P, W, ST, decltype(hc)::value, V>); });
  });
}

template <int P>
void launch_fwd_y(const void* F0, void* F1, Geo g, int nrot, cudaStream_t st, int v) {
  by_split<P>(v, [&](auto vc) { launch_fwd_y_t<P, decltype(vc)::value>(F0, F1, g, nrot, st); });
}

}  // namespace csngf

#include "zpass.cuh"
#include "zmac_tc.cuh"

namespace csngf {

template <int P>
void launch_zmac(const void* F1, const float2* UV, float2* F2, Geo g, int nrot, const RotIn* rot,
                 cudaStream_t st, int v) {
  float2* W = const_cast<float2*>(UV);            // written in the prepare mode only
  by_split<P>(v, [&](auto vc) {
    constexpr int V = decltype(vc)::value;
    by_store<P>(g.store, [&](auto sf) {
      constexpr int ST = decltype(sf)::value;
      by_half<P, V>(g.ez, [&](auto hc) {
        constexpr bool HALF = decltype(hc)::value;
        // reduced-precision forms: the channels' z DFT on the tensor cores
        if constexpr (ST != kStoreF32) {
          if (g.tc && launch_zx_tc<P, ST>(F1, UV, g, nrot, st)) {
            launch_zpass_t<P, ST, HALF, V, kZFromX>(F1, W, g.zx, F2, g, nrot, rot, st);
            return;
          }
        }
        launch_zpass_t<P, ST, HALF, V, kZFull>(F1, W, nullptr, F2, g, nrot, rot, st);
      });
    });
  });
}

template <int P>
void launch_prep_z(const float2* F1, float2* UV, Geo g, cudaStream_t st) {
  by_half<P, 0>(g.ez, [&](auto hc) {
    launch_zpass_t<P, kStoreF32, decltype(hc)::value, 0, kZPrep>(F1, UV, nullptr, nullptr, g, 1, nullptr, st);
  });
}

// ---------------------------------------------------------------------------
// inv_y: y-axis inverse FFT of every (dz, kx) row of F2, keeping the window's
// shift rows, transposed so kx is contiguous.  Block: W consecutive kx rows.
// ---------------------------------------------------------------------------
template <int P, int W, int V>
__global__ void __launch_bounds__(W * SplitV<P, V>::N2)
k_inv_y(const float2* __restrict__ F2, float2* __restrict__ F3, Geo g, const RotIn* __restrict__ rot) {
  const float2* __restrict__ tw = kTw<P>.w;
  using FS = FourStep<P, true, V>;
  constexpr int N1 = FS::N1, N2 = FS::N2, CS = FS::CS;
  extern __shared__ float2 ex[];
  const int t = threadIdx.x;
  const long long plane = blockIdx.x;               // r * wz + dz
  const int kx0 = blockIdx.y * W;
  const int r = (int)(plane / g.wz), dz = (int)(plane - (long long)r * g.wz);
  const RotBox& b = rot[r].b;
  if (dz > b.hi[0] - b.lo[0]) return;                // past this rotation's window
  const int m0 = b.m0[1], last = b.hi[1] - b.lo[1];
  {
    const int row = t / N2, n2 = t - row * N2;
    const int kx = kx0 + row;
    float2 v[N1];
    const float2* src = F2 + (((long long)r * g.Px + kx) * g.wz + dz) * (long long)P;   // [r][kx][dz][ky]
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1)
      v[n1] = (kx < g.Px) ? src[N2 * n1 + n2] : make_float2(0.f, 0.f);
    FS::template step1<1>(v, ex + row * CS, n2, tw);
  }
  __syncthreads();
  if (t < W * N1) {
    const int col = t % W, k1 = t / W;
    const int kx = kx0 + col;
    if (kx < g.Px) {
      float2 u[N2];
      FS::template step2<1>(u, ex + col * CS, k1);
      float2* dst = F3 + plane * (long long)g.wy * g.Px + kx;
#pragma unroll
      for (int k2 = 0; k2 < N2; ++k2) {
        const int dy = window_index(k1 + N1 * k2, m0, P);
        if (dy <= last) dst[(long long)dy * g.Px] = u[k2];
      }
    }
  }
}

template <int P>
void launch_inv_y(const float2* F2, float2* F3, Geo g, int nrot, const RotIn* rot, cudaStream_t st,
                  int v) {
  by_split<P>(v, [&](auto vc) {
    constexpr int V = decltype(vc)::value;
    constexpr int W = 16, N2 = SplitV<P, V>::N2;
    const size_t smem = (size_t)W * FourStep<P, true, V>::CS * sizeof(float2);
    set_smem(k_inv_y<P, W, V>, smem);
    dim3 grid((unsigned)(nrot * g.wz), (unsigned)((g.Px + W - 1) / W));
    k_inv_y<P, W, V><<<grid, W * N2, smem, st>>>(F2, F3, g, rot);
  });
}

// ---------------------------------------------------------------------------
// inv_x: x-axis inverse FFT of every (dz, dy) row of F3; at each valid shift
// s = X / N (Eq. 5) where N >= the minimum overlap, and the block's argmax is
// folded into the rotation's key with one atomicMax.  Optionally writes the
// score map (-inf where invalid).  Block: ROWS consecutive dy of one plane.
// ---------------------------------------------------------------------------
template <int P, int ROWS, int V>
__global__ void __launch_bounds__((ROWS * SplitV<P, V>::N2 + 31) / 32 * 32)
k_inv_x(const float2* __restrict__ F3, unsigned long long* __restrict__ keys, float* __restrict__ map,
        Geo g, const RotIn* __restrict__ rot) {
  const float2* __restrict__ tw = kTw<P>.w;
  using FS = FourStep<P, true, V>;
  constexpr int N1 = FS::N1, N2 = FS::N2, CS = FS::CS, NT = (ROWS * N2 + 31) / 32 * 32;
  extern __shared__ float2 ex[];
  __shared__ unsigned long long red[NT / 32];
  const int t = threadIdx.x;
  const int plane = blockIdx.y;                       // r * wz + dz
  const int r = plane / g.wz, dz = plane - r * g.wz;
  const int dy0 = blockIdx.x * ROWS;
  const RotBox& b = rot[r].b;
  const int ny_w = b.hi[1] - b.lo[1] + 1, last = b.hi[2] - b.lo[2], m0 = b.m0[2];
  if (dz > b.hi[0] - b.lo[0] || dy0 >= ny_w) return;   // past this rotation's window
  if (t < ROWS * N2) {
    const int lrow = t / N2, n2 = t - lrow * N2;
    const int dy = dy0 + lrow;
    const float2* src = F3 + ((long long)plane * g.wy + dy) * P;
    float2 v[N1];
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1)
      v[n1] = (dy < ny_w) ? src[N2 * n1 + n2] : make_float2(0.f, 0.f);
    FS::template step1<1>(v, ex + lrow * CS, n2, tw);
  }
  __syncthreads();
  unsigned long long best = 0ull;
  if (t < ROWS * N1) {
    const int lr = t / N1, k1 = t - lr * N1;
    const int dy = dy0 + lr;
    if (dy < ny_w) {
      float2 u[N2];
      FS::template step2<1>(u, ex + lr * CS, k1);
      const float th = b.thr;
      const unsigned row_lin = ((unsigned)(b.lo[0] + dz) * (unsigned)g.vy + (unsigned)(b.lo[1] + dy)) *
                                   (unsigned)g.vx + (unsigned)b.lo[2];
#pragma unroll
      for (int k2 = 0; k2 < N2; ++k2) {
        const int dx = window_index(k1 + N1 * k2, m0, P);
        if (dx <= last) {
          const float2 zz = u[k2];
          float s = __int_as_float(0xff800000);
          if (zz.y >= th) {
            s = __fdiv_rn(zz.x, zz.y);
            const unsigned long long key = make_key(s, row_lin + (unsigned)dx);
            best = key > best ? key : best;
          }
          if (map) map[(long long)row_lin + dx] = s;
        }
      }
    }
  }
  // block max
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const unsigned long long o = __shfl_xor_sync(0xffffffffu, best, off);
    best = o > best ? o : best;
  }
  if ((t & 31) == 0) red[t >> 5] = best;
  __syncthreads();
  if (t == 0) {
    unsigned long long top = 0ull;
    for (int w = 0; w < NT / 32; ++w) top = red[w] > top ? red[w] : top;
    if (top) atomicMax(&keys[r], top);
  }
}

template <int P>
void launch_inv_x(const float2* F3, unsigned long long* keys, float* map, Geo g, int nrot, const RotIn* rot,
                  cudaStream_t st, int v) {
  by_split<P>(v, [&](auto vc) {
    constexpr int V = decltype(vc)::value;
    constexpr int N2 = SplitV<P, V>::N2;
    constexpr int ROWS = (256 / N2) > 0 ? (256 / N2) : 1;
    const size_t smem = (size_t)ROWS * FourStep<P, true, V>::CS * sizeof(float2);
    set_smem(k_inv_x<P, ROWS, V>, smem);
    dim3 grid((unsigned)((g.wy + ROWS - 1) / ROWS), (unsigned)(nrot * g.wz));
    k_inv_x<P, ROWS, V><<<grid, (ROWS * N2 + 31) / 32 * 32, smem, st>>>(F3, keys, map, g, rot);
  });
}

#define CSNGF_INSTANTIATE_PASSES(P)                                                              \
  template void launch_fwd_x<P>(const float*, const uint8_t*, void*, const RotIn*, Geo, int,     \
                                cudaStream_t, int);                                              \
  template void launch_fwd_y<P>(const void*, void*, Geo, int, cudaStream_t, int);                \
  template void launch_zmac<P>(const void*, const float2*, float2*, Geo, int, const RotIn*,      \
                               cudaStream_t, int);                                               \
  template void launch_prep_z<P>(const float2*, float2*, Geo, cudaStream_t);                     \
  template void launch_inv_y<P>(const float2*, float2*, Geo, int, const RotIn*, cudaStream_t,    \
                                int);                                                            \
  template void launch_inv_x<P>(const float2*, unsigned long long*, float*, Geo, int,            \
                                const RotIn*, cudaStream_t, int);

}  // namespace csngf
