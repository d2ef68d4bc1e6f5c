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
// The two channels of a field travel side by side (c2) through the transform;
// so do X and Y through the inverse.
//
// What bounds it: with inputs and weights read where they were needed, the pass
// waited on memory whatever its arithmetic (45 us per rotation at 150^3 with
// the transforms, 50 without).  So a tile's inputs and weights arrive by bulk
// copies one field ahead, issued by one thread: no registers, no address
// arithmetic, no load instructions in the other warps.
//
// Weights (UV): [kx <= Px/2][p / 4] tiles of per field [kz][p % 4][a, b] and
// the mask's [kz][p % 4].
#pragma once

#include <algorithm>

#include "tc.cuh"

namespace csngf {

constexpr int kZW = 4;                            // columns per block: one tile of F1

enum { kZFull = 0, kZFromX = 1, kZPrep = 2 };     // see k_zpass

// A block transforms a tile of up to four rotations side by side: they share the
// weights, and pairs the mask field that carries both their masks.
//
// The z transform takes the split's larger factor first (N1 >= N2): X, which
// stays in registers through all fields, has N2 values per thread, the pair of
// transforms 2 N1 in the first step and 2 N2 in the second, so that 128
// registers hold both (10 x 16 with the larger factor last: 168 and spills).
template <int P, int V, int MODE>
struct ZCfg {
  static constexpr int A = SplitV<P, V>::N1, B = SplitV<P, V>::N2;
  static constexpr int N1 = A > B ? A : B, N2 = A > B ? B : A, W = kZW, QMAX = MODE == kZPrep ? 1 : 4;
  // exchange [Q][N2][N1 (odd)][W] of pairs: 8 lanes take four columns of two
  // rows, which an odd row length puts in different banks
  static constexpr int RS = N1 | 1, SEQ = N2 * RS * W;
  static constexpr int NWT = MODE == kZFull ? 2 : MODE == kZFromX ? 1 : 0;   // weights: values per column
  static constexpr size_t wbytes = (size_t)NWT * W * P * sizeof(float2);     // of one buffer, two are held
  // q rotations of ez planes: exchange, inputs [q][column, mirror][ez][W], weights
  static constexpr size_t smem_bytes(int q, int ez) {
    return (size_t)(q * SEQ + P) * sizeof(c2) + (size_t)q * 2 * ez * W * sizeof(float2) + 2 * wbytes + 64;
  }
  // registers a thread needs: in the first step the pair of transforms, with X
  // beside it where the fields are summed here (with 40 more instead of 24 there:
  // 96x128x128 19.2 -> 20.1 us per rotation; with 24 in the other modes: 150^3 BF16
  // 84.9 -> 90.4)
  static constexpr int regs0 = (4 * N1 + (MODE == kZFull ? 2 * N2 : 0) > 6 * N2 ? 4 * N1 + (MODE == kZFull ? 2 * N2 : 0) : 6 * N2) + (MODE == kZFull ? 24 : 40);
  static constexpr int regs = regs0 < 248 ? regs0 : 248;
  static constexpr int blocks(int q, int ez) { return pass_blocks(q * W * N1, smem_bytes(q, ez), regs); }
  // rotations side by side: the most, unless fewer put a fifth more threads on an
  // SM (at 96 points one rotation per block counted two warps for its 48 threads
  // and took 1.4 times as long as four)
  static constexpr int fit(int ez) {
    int best = 1, threads = 0;
    for (int q = QMAX; q >= 1; q /= 2) {
      if (smem_bytes(q, ez) > 227 * 1024) continue;
      const int n = blocks(q, ez) * q * W * N1;
      if (5 * n > 6 * threads) { threads = n; best = q; }
    }
    return best;
  }
  static constexpr int Q = fit(2 * P / 3);        // what the registers are bounded for: typical boxes
  static constexpr int MIN_BLOCKS = blocks(Q, 2 * P / 3);
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
// Block: one tile of one kx, the rotations [blockIdx.z * rpb, + rpb).
template <int P, int ST, bool HALF, int V, int MODE>
__global__ void __launch_bounds__(ZCfg<P, V, MODE>::Q * kZW * ZCfg<P, V, MODE>::N1,
                                          ZCfg<P, V, MODE>::MIN_BLOCKS)
k_zpass(const void* __restrict__ F1, float2* __restrict__ UV, const float2* __restrict__ Xg,
        float2* __restrict__ F2, Geo g, int nrot, int rpb, const RotIn* __restrict__ rot) {
  using C = ZCfg<P, V, MODE>;
  constexpr int N1 = C::N1, N2 = C::N2, W = C::W, RS = C::RS, SEQ = C::SEQ;
  constexpr int NI = HALF ? N1 / 2 : N1;
  constexpr bool kMaskOnly = MODE == kZFromX, kWeights = MODE != kZPrep;
  const int Q = blockDim.x / (W * N1);            // rotations side by side
  const int t = threadIdx.x;
  extern __shared__ __align__(128) c2 zsm[];
  c2* ex = zsm;                                   // [Q][N2][RS][W]
  c2* tw2 = ex + Q * SEQ;                         // [P]
  float2* ws = reinterpret_cast<float2*>(tw2 + P);                      // [2][P][W][a, b], or the mask's [P][W]
  float2* stg = ws + 2 * C::wbytes / sizeof(float2);                    // [Q][column, mirror][ez][W]
  uint64_t* bar = reinterpret_cast<uint64_t*>(stg + Q * 2 * g.ez * W);  // inputs, weights per buffer
  const int kx = blockIdx.y, mkx = kx == 0 ? 0 : g.Px - kx;
  const int ntile = gridDim.x, half = ntile / 2, tile = blockIdx.x;
  const int mtile = tile < half ? tile + half : tile - half;
  const bool own = tile == 0 || tile == half;     // column 0 is ky = 0 or P/2: its own mirror
  const int c = t % W, pos = tile * W + c;
  const int q1 = t / (W * N2), n2 = t / W - q1 * N2;   // first-step role
  const int q2 = t / (W * N1), k1 = t / W - q2 * N1;   // second-step role
  const int nchan = 2 * g.nch + 1;
  float2* wt = UV + ((long long)kx * ntile + tile) * nchan * (P * W);
  const long long E = (long long)g.ez * g.Px * W * ntile;              // F1 is [r][j][kx][p/4][z][p%4]
  const long long tz = (long long)g.ez * W;                            // values of a tile
  const long long off_h = ((long long)kx * ntile + tile) * tz, off_m = ((long long)mkx * ntile + mtile) * tz;

  auto fetch_inputs = [&](int r0, int j) {        // one thread: field j of rotations r0 .. r0 + Q - 1
    const int b = (ST == kStoreF32 || j == g.nch) ? 8 : 4;
    const uint32_t bytes = (uint32_t)tz * b;
    int n = 0;
    for (int q = 0; q < Q; ++q) {
      const int r = j == g.nch ? (r0 + q) & ~1 : r0 + q;   // a mask field carries rotations 2k and 2k + 1
      if (r < nrot) ++n;
    }
    tc::mbar_expect(&bar[0], 2 * n * bytes);
    for (int q = 0; q < Q; ++q) {
      const int r = j == g.nch ? (r0 + q) & ~1 : r0 + q;
      if (r >= nrot) continue;
      const char* f = Fields<ST>::field(F1, g, E, r, j);
      tc::bulk_load(stg + 2 * q * tz, f + off_h * b, bytes, &bar[0]);
      tc::bulk_load(stg + (2 * q + 1) * tz, f + off_m * b, bytes, &bar[0]);
    }
  };
  auto fetch_weights = [&](int j, int s) {        // one thread: field j's weights
    const uint32_t bytes = (j == g.nch ? 1 : 2) * P * W * sizeof(float2);
    tc::mbar_expect(&bar[1 + s], bytes);
    tc::bulk_load(reinterpret_cast<char*>(ws) + s * C::wbytes, wt + (long long)2 * j * P * W, bytes, &bar[1 + s]);
  };

  const int rbeg = (int)blockIdx.z * rpb, rend = min(nrot, rbeg + rpb);
  const int jbeg = kMaskOnly ? g.nch : 0;
  if (t == 0) {
    for (int i = 0; i < 3; ++i) tc::mbar_init(&bar[i], 1);
    tc::mbar_init_fence();
    fetch_inputs(rbeg, jbeg);
    if (kWeights) fetch_weights(jbeg, 0);
  }
  for (int i = t; i < P; i += blockDim.x) tw2[i] = {dup(kTw<P>.w[i].x), dup(kTw<P>.w[i].y)};
  __syncthreads();                                // the barriers are initialised

  float2 X[N2];
  int f = 0;                                      // fields so far: buffers and phases of the barriers
  int dead = -1;                                  // 2 field + (inputs: 0, weights: 1) of a wait that ran out: no more
                                                  // waits, results invalid
  auto wait = [&](int b, int phase) {
    if (dead < 0 && !tc::mbar_wait(&bar[b], phase & 1, kTcWaitNs)) dead = 2 * f + (b > 0);
  };
  // channels a', b' at this thread's z; zero past the box
  auto load = [&](c2 (&v)[NI], const float2* s, int r, int j) {
    const float isc = 1.0f / field_scale(g.scale1, j);
    auto rows = [&](auto mc) {
      constexpr bool wide = decltype(mc)::value;
#pragma unroll
      for (int n1 = 0; n1 < NI; ++n1) {
        const int i = (N2 * n1 + n2) * W + c;
        float2 h = make_float2(0.f, 0.f), m = h;
        if (i < (int)tz) {
          h = Fields<ST>::get(reinterpret_cast<const char*>(s), i, wide, isc);
          m = Fields<ST>::get(reinterpret_cast<const char*>(s + tz), i, wide, isc);
        }
        v[n1] = {h, m};
      }
      if (own && c == 0) {                        // the column's own mirror: the same tile of -kx
        const char* fld = Fields<ST>::field(F1, g, E, j == g.nch ? r & ~1 : r, j);
        const long long o = ((long long)mkx * ntile + tile) * tz;
#pragma unroll
        for (int n1 = 0; n1 < NI; ++n1) {
          const int i = (N2 * n1 + n2) * W;
          v[n1].y = make_float2(0.f, 0.f);
          if (r < nrot && i < (int)tz) v[n1].y = Fields<ST>::get(fld, o + i, wide, isc);
        }
      }
#pragma unroll
      for (int n1 = 0; n1 < NI; ++n1) {
        const float2 h = v[n1].x, m = v[n1].y;
        v[n1] = {cadd(h, m), make_float2(h.y - m.y, m.x - h.x)};
      }
    };
    if (ST == kStoreF32 || j == g.nch) rows(std::true_type{});
    else rows(std::false_type{});
  };

#pragma unroll 1
  for (int r0 = rbeg; r0 < rend; r0 += Q) {
    if constexpr (MODE == kZFull) {
#pragma unroll
      for (int i = 0; i < N2; ++i) X[i] = make_float2(0.f, 0.f);
    }
    const int r2 = r0 + q2;                       // this thread's rotation in the second step
    // a first-step role; the empty slots of a short last set have none, and load and
    // transform nothing (five rotations of 90x100x84 with full padding take eight slots:
    // 789 -> 747 us, of 130x128x140 in the FP16 form 2891 -> 2769 us; more rotations as before)
    const bool has1 = t < min(Q, nrot - r0) * W * N2;
#pragma unroll 1
    for (int j = jbeg; j <= g.nch; ++j, ++f) {
      const bool mask = j == g.nch;
      wait(0, f);
      __syncthreads();                            // the previous reads of ex are done
      if (has1) {
        c2 in[NI];
        load(in, stg + 2 * q1 * tz, r0 + q1, j);
        c2* e = ex + (q1 * N2 + n2) * RS * W + c; // this thread's row [k1]
        c2 v[N1];
        if constexpr (HALF) {                     // zero for n1 >= N1/2: two N1/2-point transforms
          dft_half<N1, -1>(in, v);
        } else {
#pragma unroll
          for (int i = 0; i < N1; ++i) v[i] = in[i];
          Dft<N1, -1>::run(v);
        }
#pragma unroll
        for (int k = 0; k < N1; ++k) e[k * W] = k == 0 ? v[k] : cmul(v[k], tw2[n2 * k]);
      }
      __syncthreads();
      // the inputs have been read, the other weights' products summed (dead: a phase
      // is still open, and a second arrival on it would be undefined)
      if (t == 0 && dead < 0) {
        const int nr = mask ? r0 + Q : r0, nj = mask ? jbeg : j + 1;
        if (nr < rend) {
          fetch_inputs(nr, nj);
          if (kWeights) fetch_weights(nj, (f + 1) & 1);
        }
      }
      if constexpr (MODE == kZFromX) {
        if (r2 < nrot) {
          const float2* xs = Xg + (((long long)r2 * gridDim.y + kx) * ntile + tile) * (P * W) + k1 * W + c;
#pragma unroll
          for (int i = 0; i < N2; ++i) X[i] = __ldg(&xs[i * N1 * W]);
        }
      }
      c2* e = ex + (q2 * N2 * RS + k1) * W + c;   // its column [n2] in the second step
      c2 u[N2];
#pragma unroll
      for (int i = 0; i < N2; ++i) u[i] = e[i * RS * W];
      if (kWeights) wait(1 + (f & 1), f >> 1);
      Dft<N2, -1>::run(u);                        // at kz = k1 + N1 i
      if constexpr (MODE == kZPrep) {
        float wa = 0.25f, wb = 0.25f;             // Eq. 6: (1, 1), (1, 2), (2, 2); Eq. 3: (1, 1), (1, 0)
        if (!mask && g.nch == 3) { wa = j == 2 ? 0.5f : 0.25f; wb = j == 0 ? 0.25f : 0.5f; }
        if (!mask && g.nch == 2 && j == 1) wb = 0.0f;
        if (mask) {
          float2* o = wt + (long long)(2 * j) * P * W + k1 * W + c;
#pragma unroll
          for (int i = 0; i < N2; ++i) o[i * N1 * W] = make_float2(wa * u[i].x.x, -wa * u[i].y.x);
        } else {
          float4* o = reinterpret_cast<float4*>(wt + (long long)(2 * j) * P * W) + k1 * W + c;
#pragma unroll
          for (int i = 0; i < N2; ++i)
            o[i * N1 * W] = make_float4(wa * u[i].x.x, -wa * u[i].y.x, wb * u[i].x.y, -wb * u[i].y.y);
        }
        continue;
      }
      const char* wb = reinterpret_cast<const char*>(ws) + (f & 1) * C::wbytes;
      if (!mask) {
        const float4* w4 = reinterpret_cast<const float4*>(wb) + k1 * W + c;
#pragma unroll
        for (int i = 0; i < N2; ++i) {
          const float4 w = w4[i * N1 * W];
          cmac(X[i], make_float2(w.x, w.y), make_float2(u[i].x.x, u[i].y.x));
          cmac(X[i], make_float2(w.z, w.w), make_float2(u[i].x.y, u[i].y.y));
        }
      } else {
        // Y from this rotation's mask, then X and Y side by side into the
        // inverse: over k2, twiddle, back to the slots this thread has read
        const float2* wm = reinterpret_cast<const float2*>(wb) + k1 * W + c;
        const bool odd = r2 & 1;
#pragma unroll
        for (int i = 0; i < N2; ++i) {
          const float2 Y = cmul(wm[i * N1 * W], odd ? make_float2(u[i].x.y, u[i].y.y) : make_float2(u[i].x.x, u[i].y.x));
          u[i] = {make_float2(X[i].x, Y.x), make_float2(X[i].y, Y.y)};
        }
        Dft<N2, 1>::run(u);
#pragma unroll
        for (int i = 0; i < N2; ++i) {
          c2 w = tw2[i * k1];
          w.y = make_float2(-w.y.x, -w.y.y);
          e[i * RS * W] = i == 0 ? u[i] : cmul(u[i], w);
        }
      }
    }
    if constexpr (MODE == kZPrep) continue;
    __syncthreads();
    const int r1 = r0 + q1;
    if (has1) {                                   // (padded positions hold what nobody reads)
      const c2* e = ex + (q1 * N2 + n2) * RS * W + c;
      c2 v[N1];
#pragma unroll
      for (int i = 0; i < N1; ++i) v[i] = e[i * W];
      Dft<N1, 1>::run(v);
      const int m0 = rot[r1].b.m0[0], last = rot[r1].b.hi[0] - rot[r1].b.lo[0];
      const int pp = W * ntile, mpos = own && c == 0 ? pos : mtile * W + c;
      float2* d = F2 + ((long long)r1 * g.Px + kx) * g.wz * pp + pos;       // [r][kx][dz][p]
      float2* dm = F2 + ((long long)r1 * g.Px + mkx) * g.wz * pp + mpos;
      const bool self = mkx == kx;                // its mirrors are columns of this kx
#pragma unroll
      for (int i = 0; i < N1; ++i) {
        const int dz = window_index(N2 * i + n2, m0, P);
        if (dz <= last) {                         // x + iy, and conj x + i conj y
          d[dz * pp] = make_float2(v[i].x.x - v[i].y.y, v[i].y.x + v[i].x.y);
          if (!self) dm[dz * pp] = make_float2(v[i].x.x + v[i].y.y, v[i].x.y - v[i].y.x);
        }
      }
    }
  }
  if (dead >= 0) {
    atomicExch(g.wait_err, 1);
    if (t == 0) {                                 // the copies still in flight end before the block does: inputs and
      const int d = dead >> 1;                    // weights of field d, or its weights and all of field d + 1
      const bool in = !(dead & 1);
      tc::mbar_wait(&bar[0], (in ? d : d + 1) & 1, kTcWaitNs / 4);
      if (kWeights)
        for (int l = d; l <= d + !in; ++l) tc::mbar_wait(&bar[1 + (l & 1)], (l >> 1) & 1, kTcWaitNs / 4);
    }
  }
}

template <int P, int ST, bool HALF, int V, int MODE>
void launch_zpass_t(const void* F1, float2* UV, const float2* Xg, float2* F2, Geo g, int nrot, const RotIn* rot,
                    cudaStream_t st) {
  using C = ZCfg<P, V, MODE>;
  const unsigned tiles = (unsigned)(ky_total(g.Py) / C::W), nkx = (unsigned)(g.Px / 2 + 1);
  int q = std::min(C::Q, C::fit(g.ez));           // large boxes leave room for fewer
  while (q > 1 && q >= 2 * nrot) q /= 2;
  // rotations per block: few enough that the blocks fill the SMs many times
  // over (a short last wave), more where there are blocks to spare (the weights
  // then come from L2)
  const long long cols = (long long)tiles * nkx;
  int rpb = q;
  while (rpb < 16 && cols * ((nrot + 2 * rpb - 1) / (2 * rpb)) >= 152 * C::MIN_BLOCKS * 16) rpb *= 2;
  const size_t smem = C::smem_bytes(q, g.ez);
  set_smem<k_zpass<P, ST, HALF, V, MODE>>(smem);
  k_zpass<P, ST, HALF, V, MODE><<<dim3(tiles, nkx, (unsigned)((nrot + rpb - 1) / rpb)), q * C::W * C::N1, smem, st>>>(
      F1, UV, Xg, F2, g, nrot, rpb, rot);
}

}  // namespace csngf
