// z pass of the all-shift NGF correlation (Cross-Sim-NGF Eq. 7-8), included by
// passes.cuh.
//
// A packed field holds two real channels a, b in one complex value.  Their own
// (kx, ky, z) columns follow at each z from the column h and its mirror
// h' = h(-kx, -ky): a' = 2a = h + conj h', b' = 2b = -i (h - conj h').  So the
// channels are separated before the z transform, at the load, and everything
// after it happens at one (kx, ky, kz): the products with the fixed volume's
// weights are summed in the registers that hold the second transform step's
// outputs, X for the channels and Y for the mask, and the inverse starts from
// those registers.  Each transform crosses shared memory once.
//
// After the inverse, x and y are columns of the numerator's and the overlap
// count's half spectra (kx <= Px/2); F2 gets x + iy at (kx, ky) and
// conj x + i conj y at (-kx, -ky), whose y and x inverses have the numerator as
// real and the count as imaginary part.
//
// Weights (UV): [kx <= Px/2][ky / 8][channel 2 nch + 1][kz][ky % 8].
#pragma once

namespace csngf {

constexpr int kZW = 8;                            // ky columns per block: 64-byte rows of F1

enum { kZFull = 0, kZFromX = 1, kZPrep = 2 };     // see k_zpass

// Q: rotations a block transforms side by side.  Two share each weight tile,
// and the mask field that carries both their masks; above 16 points in the
// second step a thread's X and transform registers no longer leave room for
// two blocks of two rotations on an SM, and one rotation per block fits three.
template <int P, int V, int MODE>
struct ZCfg {
  using FS = FourStep<P, true, V>;                // odd row stride: conflict-free for 8-column rows
  static constexpr int N1 = FS::N1, N2 = FS::N2, W = kZW;
  static constexpr int Q = (MODE == kZPrep || N2 > 16) ? 1 : 2;
  static constexpr int NT = Q * W * N2;
  static constexpr int SEQ = N2 * FS::RS * W;     // one transform per column in exchange, 2 per rotation
  static constexpr int NWT = MODE == kZFull ? 2 : MODE == kZFromX ? 1 : 0;   // weight tiles held
  static constexpr size_t smem_bytes = ((size_t)Q * 2 * SEQ + (size_t)NWT * W * P + P) * sizeof(float2);
  static constexpr int warps = (NT + 31) / 32;
  // registers a thread needs: X and the transform (2 N2 each) and about 56 more
  static constexpr int regs = (4 * N2 + 56 + 7) / 8 * 8;
  static constexpr int fit_regs = 65536 / (warps * 32 * (regs < 255 ? regs : 255));
  static constexpr int fit_smem = (int)(228 * 1024 / (smem_bytes + 1024));
  static constexpr int fit = fit_regs < fit_smem ? fit_regs : fit_smem;
  static constexpr int MIN_BLOCKS = fit < 1 ? 1 : fit > 6 ? 6 : fit;
};

__device__ __forceinline__ void cmac(float2& x, float2 w, float2 u) {
  x.x = fmaf(w.x, u.x, x.x);
  x.y = fmaf(w.x, u.y, x.y);
  x.x = fmaf(-w.y, u.y, x.x);
  x.y = fmaf(w.y, u.x, x.y);
}

// MODE kZFull: the pass of a launch group: forward transforms, X and Y, the
// inverse, the window's planes to F2.  kZFromX: the same with X read from the
// tensor-core half (Xg, laid out as one weight channel).  kZPrep: the fixed
// volume: the weights w/4 conj(a'), w the Eq. 6 (Eq. 3) weight of the channel,
// 1 for the mask (1/4: both sides carry a factor 2).
// Block: 8 ky columns of one kx, the rotations [blockIdx.z * rpb, + rpb).
template <int P, int ST, bool HALF, int V, int MODE>
__global__ void __launch_bounds__(ZCfg<P, V, MODE>::NT, ZCfg<P, V, MODE>::MIN_BLOCKS)
k_zpass(const void* __restrict__ F1, float2* __restrict__ UV, const float2* __restrict__ Xg,
        float2* __restrict__ F2, Geo g, int nrot, int rpb, const RotIn* __restrict__ rot) {
  using C = ZCfg<P, V, MODE>;
  using FS = typename C::FS;
  using FI = FwdIn<FS, HALF>;
  constexpr int N1 = FS::N1, N2 = FS::N2, RS = FS::RS, W = C::W, Q = C::Q, NT = C::NT, SEQ = C::SEQ;
  constexpr int NI = FI::NI;
  extern __shared__ __align__(16) float2 zsm[];
  float2* ex = zsm;                               // [Q][2][N2][RS][W]
  float2* ws = ex + Q * 2 * SEQ;                  // [NWT][P][W]
  float2* tws = ws + C::NWT * W * P;              // [P]
  const int t = threadIdx.x;
  const int kx = blockIdx.y, ky0 = blockIdx.x * W;
  const int mkx = kx == 0 ? 0 : g.Px - kx;
  const int c = t % W, ky = ky0 + c;
  const bool col_ok = ky < g.Py;
  const int mky = ky == 0 ? 0 : g.Py - ky;
  const int q1 = t / (W * N2), n2 = t / W - q1 * N2;   // first-step role
  const int q2 = t / (W * N1), k1 = t / W - q2 * N1;   // second-step role
  const bool has2 = t < Q * W * N1;
  const int nchan = 2 * g.nch + 1;
  float2* wt = UV + ((long long)kx * gridDim.x + blockIdx.x) * nchan * (P * W);
  const long long E = (long long)g.ez * g.Px * g.Py;   // F1 is [r][j][kx][z][ky]
  const long long off_h = (long long)kx * g.ez * g.Py + ky, off_m = (long long)mkx * g.ez * g.Py + mky;
  for (int i = t; i < P; i += NT) tws[i] = kTw<P>.w[i];
  // (the first barrier of the loop orders these writes before their reads)

  float2* e1 = ex + (q1 * 2) * SEQ + n2 * RS * W + c;
  float2* e2 = ex + (q2 * 2) * SEQ + k1 * W + c;
  float2 X[N2], u[N2];

  auto load = [&](float2 (&h)[NI], float2 (&m)[NI], int r, int j) {
    const bool mask = ST == kStoreF32 || j == g.nch;
    const char* f = Fields<ST>::field(F1, g, E, r, j);
    const float isc = 1.0f / field_scale(g.scale1, j);
    const bool ok = col_ok && r < nrot;
    if (mask) {
#pragma unroll
      for (int n1 = 0; n1 < NI; ++n1) {
        const int z = N2 * n1 + n2;
        h[n1] = m[n1] = make_float2(0.f, 0.f);
        if (ok && z < g.ez) {
          h[n1] = Fields<ST>::get(f, off_h + (long long)z * g.Py, true, isc);
          m[n1] = Fields<ST>::get(f, off_m + (long long)z * g.Py, true, isc);
        }
      }
    } else {
#pragma unroll
      for (int n1 = 0; n1 < NI; ++n1) {
        const int z = N2 * n1 + n2;
        h[n1] = m[n1] = make_float2(0.f, 0.f);
        if (ok && z < g.ez) {
          h[n1] = Fields<ST>::get(f, off_h + (long long)z * g.Py, false, isc);
          m[n1] = Fields<ST>::get(f, off_m + (long long)z * g.Py, false, isc);
        }
      }
    }
  };
  auto step2 = [&](const float2* e) {             // u[k2] = transform at k1 + N1 k2
#pragma unroll
    for (int i = 0; i < N2; ++i) u[i] = e[i * RS * W];
    Dft<N2, -1>::run(u);
  };
  auto fetch_weights = [&](int ch, int n) {       // n channels from ch
    const float2* src = wt + (long long)ch * P * W;
    for (int i = t; i < n * P * W / 2; i += NT) cp_async16(ws + 2 * i, src + 2 * i);
    cp_async_commit();
  };
  auto inv1 = [&](float2 (&v)[N2], float2* e) {   // over k2, twiddle, to the exchange
    Dft<N2, 1>::run(v);
#pragma unroll
    for (int i = 0; i < N2; ++i) {
      const float2 w = tws[i * k1];
      e[i * RS * W] = i == 0 ? v[i] : cmul(v[i], make_float2(w.x, -w.y));
    }
  };

  const int rend = min(nrot, ((int)blockIdx.z + 1) * rpb);
#pragma unroll 1
  for (int r0 = (int)blockIdx.z * rpb; r0 < rend; r0 += Q) {
#pragma unroll
    for (int i = 0; i < N2; ++i) X[i] = make_float2(0.f, 0.f);
    const int r2 = r0 + q2;                       // this thread's rotation in the second step
    if constexpr (MODE == kZFromX) {
      if (has2 && r2 < nrot) {
        const float2* xs = Xg + (((long long)r2 * gridDim.y + kx) * gridDim.x + blockIdx.x) * (P * W) + k1 * W + c;
#pragma unroll
        for (int i = 0; i < N2; ++i) X[i] = __ldg(&xs[i * N1 * W]);
      }
    }
#pragma unroll 1
    for (int j = MODE == kZFromX ? g.nch : 0; j <= g.nch; ++j) {
      const bool mask = j == g.nch;
      const bool two = !mask && !(g.nch == 2 && j == 1);   // Eq. 3: (z, 0) holds one channel
      __syncthreads();                            // the previous reads of ex and ws are done
      if constexpr (MODE != kZPrep) fetch_weights(2 * j, MODE == kZFull && two ? 2 : 1);
      {
        float2 h[NI], m[NI];
        // a mask field carries rotations 2k and 2k + 1 as its a and b
        load(h, m, mask ? (r0 + q1) & ~1 : r0 + q1, j);
#pragma unroll
        for (int i = 0; i < NI; ++i) {
          const float2 s = make_float2(h[i].x + m[i].x, h[i].y - m[i].y);
          const float2 d = make_float2(h[i].y + m[i].y, m[i].x - h[i].x);
          h[i] = s;
          m[i] = d;
        }
        if (!mask || !((r0 + q1) & 1)) FI::template step1w<-1, W>(h, e1 + (mask ? SEQ : 0), n2, tws);
        if (two || (mask && ((r0 + q1) & 1))) FI::template step1w<-1, W>(m, e1 + SEQ, n2, tws);
      }
      if constexpr (MODE != kZPrep) cp_async_wait_all();
      __syncthreads();
      if (!has2) continue;
      if constexpr (MODE == kZPrep) {
        float wa = 0.25f, wb = 0.25f;             // Eq. 6: (1, 1), (1, 2), (2, 2); Eq. 3: (1, 1), (1, 0)
        if (!mask && g.nch == 3) { wa = j == 2 ? 0.5f : 0.25f; wb = j == 0 ? 0.25f : 0.5f; }
        for (int s = 0; s < (mask ? 1 : 2); ++s) {
          float2* o = wt + (long long)(2 * j + s) * P * W + k1 * W + c;
          const float w = s ? wb : wa;
          if (s == 1 && !two) {
#pragma unroll
            for (int i = 0; i < N2; ++i) o[i * N1 * W] = make_float2(0.f, 0.f);
            continue;
          }
          step2(e2 + (mask || s ? SEQ : 0));
#pragma unroll
          for (int i = 0; i < N2; ++i) o[i * N1 * W] = make_float2(w * u[i].x, -w * u[i].y);
        }
      } else if (!mask) {
        step2(e2);
#pragma unroll
        for (int i = 0; i < N2; ++i) cmac(X[i], ws[(k1 + N1 * i) * W + c], u[i]);
        if (two) {
          step2(e2 + SEQ);
#pragma unroll
          for (int i = 0; i < N2; ++i) cmac(X[i], ws[(P + k1 + N1 * i) * W + c], u[i]);
        }
      } else {
        // the second step read this thread's own slots only, and the channels'
        // exchange is free: both inverses start in place
        step2(e2 + SEQ);
#pragma unroll
        for (int i = 0; i < N2; ++i) u[i] = cmul(ws[(k1 + N1 * i) * W + c], u[i]);
        inv1(u, e2 + SEQ);
        inv1(X, e2);
      }
    }
    if constexpr (MODE == kZPrep) continue;
    __syncthreads();
    const int r1 = r0 + q1;
    if (r1 < nrot && col_ok) {
      float2 x[N1], y[N1];
#pragma unroll
      for (int i = 0; i < N1; ++i) {
        x[i] = e1[i * W];
        y[i] = e1[SEQ + i * W];
      }
      Dft<N1, 1>::run(x);
      Dft<N1, 1>::run(y);
      const int m0 = rot[r1].b.m0[0], last = rot[r1].b.hi[0] - rot[r1].b.lo[0];
      float2* d = F2 + ((long long)r1 * g.Px + kx) * g.wz * g.Py + ky;      // [r][kx][dz][ky]
      float2* dm = F2 + ((long long)r1 * g.Px + mkx) * g.wz * g.Py + mky;
      const bool self = mkx == kx;                // its mirrors are columns of this kx
#pragma unroll
      for (int i = 0; i < N1; ++i) {
        const int dz = window_index(N2 * i + n2, m0, P);
        if (dz <= last) {
          d[(long long)dz * g.Py] = make_float2(x[i].x - y[i].y, x[i].y + y[i].x);
          if (!self) dm[(long long)dz * g.Py] = make_float2(x[i].x + y[i].y, y[i].x - x[i].y);
        }
      }
    }
  }
}

template <int P, int ST, bool HALF, int V, int MODE>
void launch_zpass_t(const void* F1, float2* UV, const float2* Xg, float2* F2, Geo g, int nrot, const RotIn* rot,
                    cudaStream_t st) {
  using C = ZCfg<P, V, MODE>;
  const unsigned tiles = (unsigned)((g.Py + C::W - 1) / C::W), nkx = (unsigned)(g.Px / 2 + 1);
  // rotations per block: few enough that the blocks fill the SMs many times
  // over (a short last wave), more where there are blocks to spare (the weights
  // then come from L2)
  const long long cols = (long long)tiles * nkx;
  int rpb = 2;
  while (rpb < 8 && cols * ((nrot + 2 * rpb - 1) / (2 * rpb)) >= 152 * C::MIN_BLOCKS * 16) rpb *= 2;
  set_smem(k_zpass<P, ST, HALF, V, MODE>, C::smem_bytes);
  k_zpass<P, ST, HALF, V, MODE><<<dim3(tiles, nkx, (unsigned)((nrot + rpb - 1) / rpb)), C::NT, C::smem_bytes, st>>>(
      F1, UV, Xg, F2, g, nrot, rpb, rot);
}

}  // namespace csngf
