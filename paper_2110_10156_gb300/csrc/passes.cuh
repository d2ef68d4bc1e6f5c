// FFT passes of the all-shift NGF correlation (Cross-Sim-NGF Eq. 6-8).
// Included by one translation unit per FFT length (passes_<P>.cu).
#pragma once

#include <atomic>
#include <mutex>

#include "kernels.cuh"
#include "tc.cuh"

namespace csngf {

// Output index m of a length-P circular correlation sums the linear
// correlation over every shift of its residue class mod P.  With the fixed
// mask on slabs [a0, a1] and the rotated one on [b0, b1] the linear
// correlation lives on chi in [b0 - a1, b1 - a0], so a slot in the admitted
// range [lo, hi] holds its one shift whenever
// P >= max(b1 - a0 - chi_lo, chi_hi - (b0 - a1)) + 1, which the caller
// guarantees (for masks that fill the volume that is n + max(-chi_lo, chi_hi),
// and for every shift 2n - 1).

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

// calls f with whether a box extent e fills at most half the length: the upper
// half of every first-step sequence is then zero and the step is pruned
// (dft_half; where the split's first factor is even)
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

// the same for the z pass, whose first step takes the larger factor
template <int P, int V, class F>
static void by_half_z(int e, F&& f) {
  if constexpr (SplitV<P, V>::N2 % 2 == 0 && !box_only(P)) {
    if (2 * e <= P) {
      f(std::true_type{});
      return;
    }
  }
  f(std::false_type{});
}

// Kernel K may take `bytes` of dynamic shared memory on the current device.  The
// limit is the kernel's own, shared by every handle and host thread, and sizes
// follow the boxes: it is only ever raised, under a lock, or a launch that needs
// more would fail between another thread's setting and its own.
template <auto K>
static void set_smem(size_t bytes) {
  if (bytes <= 48 * 1024) return;
  constexpr int kDevices = 64;
  static std::atomic<size_t> high[kDevices];
  static std::mutex mu;
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= kDevices) {                             // not remembered: the most a block can have
    cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    return;
  }
  if (bytes <= high[dev].load(std::memory_order_acquire)) return;
  std::lock_guard<std::mutex> lk(mu);
  if (bytes <= high[dev].load(std::memory_order_relaxed)) return;
  if (cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess)
    high[dev].store(bytes, std::memory_order_release);
}

// Offsets of a second step's outputs in a tiled axis: tiles of four consecutive
// indices, each with L entries per index ([i / 4][L][i % 4]).  Index k + N1 m for
// compile-time m advances by N1 L every PER = 4 / gcd(4, N1) steps, so a thread
// computes PER offsets once.
__device__ __forceinline__ int tile_off(int i, int L) { return (i >> 2) * 4 * L + (i & 3); }
template <int N1>
struct TileRun {
  static constexpr int PER = N1 % 4 == 0 ? 1 : N1 % 2 == 0 ? 2 : 4;
  int b[PER], step;
  __device__ __forceinline__ TileRun(int k, int L) : step(N1 * PER * L) {
#pragma unroll
    for (int e = 0; e < PER; ++e) b[e] = tile_off(k + N1 * e, L);
  }
  __device__ __forceinline__ int at(int m) const { return b[m % PER] + m / PER * step; }
};
// the same for ky = k1 + N1 k2 in the order of ky_pos
template <int P, int N1, int N2>
struct KyRun {
  TileRun<N1> up, down;
  int k1, L;
  __device__ __forceinline__ KyRun(int k1_, int L_) : up(k1_, L_), down(N1 - k1_, L_), k1(k1_), L(L_) {}
  __device__ __forceinline__ int at(int k2) const {
    if (N1 * (k2 + 1) <= P / 2) return up.at(k2);                       // first half for every k1
    const int second = ky_half(P) * L + down.at(N2 - 1 - k2);           // P - ky = N1 (N2 - 1 - k2) + N1 - k1
    if (N1 * k2 > P / 2) return second;
    const int ky2 = 2 * (k1 + N1 * k2);
    return ky2 < P ? up.at(k2) : ky2 == P ? ky_half(P) * L : second;
  }
};

// Blocks per SM for the passes: as many as keep at least
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

// ---------------------------------------------------------------------------
// fwd_x: Eq. 1 NGF of the resampled volume, the Eq. 6 channels packed in four
// complex fields, and the x-axis FFT of every row of the box (zero padded to
// Px).  Block: ROWS rows; thread (row, n2) gathers x = N2*n1 + n2.
// ---------------------------------------------------------------------------
// Two fields travel side by side (c2): (j = 0, 1), then (j = 2, mask), half the
// instructions and half the barriers of one after the other.  The second
// pair's inputs wait in the thread's own shared-memory slots [NI][NT].
// What bounds it: the gradient's gathers through L1 (68 % of its throughput
// before) and their latency.  Most voxels of a box lie outside the mask (two
// thirds at 150^3), so the masks are read first and a masked-out voxel's
// gathers go to its row's first voxel, one sector per warp.
template <int P, bool HALF, int V>
struct FwdXCfg {
  static constexpr int N1 = SplitV<P, V>::N1, N2 = SplitV<P, V>::N2;
  static constexpr int ROWS = 128 / N2 > 0 ? 128 / N2 : 1;
  static constexpr int NT = ROWS * N2;
  static constexpr int NI = HALF ? N1 / 2 : N1;
  // exchange [row][n2][k1] of pairs: odd row length, and rows N1 apart (mod 8),
  // put eight consecutive lanes of either step in different 16-byte banks
  static constexpr int RS = N1 | 1, CS0 = N2 * RS, CS = CS0 + ((N1 - CS0) % 8 + 8) % 8;
  static constexpr size_t smem_bytes = ((size_t)ROWS * CS + (size_t)NI * NT) * sizeof(c2);
  // registers: the larger step's pair of values and the gather's addresses, fewer
  // where half of the inputs are zero (320 points: 51.4 -> 48.2 us per rotation of
  // 120x144x132 with full padding; whole inputs at 160 and 300 spill with as few,
  // 150^3 25.4 -> 30.3, 256^3 149 -> 166)
  static constexpr int regs0 = 4 * (N1 > N2 ? N1 : N2) + (HALF ? 40 : 56), regs = regs0 < 248 ? regs0 : 248;
  static constexpr int MIN_BLOCKS = pass_blocks(NT, smem_bytes, regs);
};

template <int P, int ST, bool HALF, int V>
__global__ void __launch_bounds__(FwdXCfg<P, HALF, V>::NT, FwdXCfg<P, HALF, V>::MIN_BLOCKS)
k_fwd_x(const float* __restrict__ Bh, const uint8_t* __restrict__ Mh, void* __restrict__ F0,
        const RotIn* __restrict__ rot, Geo g) {
  using C = FwdXCfg<P, HALF, V>;
  constexpr int N1 = C::N1, N2 = C::N2, RS = C::RS, CS = C::CS, NI = C::NI, ROWS = C::ROWS, NT = C::NT;
  extern __shared__ __align__(16) c2 xsm[];
  c2* ex = xsm;
  c2* slot = ex + ROWS * CS + threadIdx.x;
  const int t = threadIdx.x;
  const int lrow = t / N2, n2 = t - lrow * N2;
  // rows [row0, row0 + ROWS) of one plane of one rotation
  const int r = blockIdx.z, zb = blockIdx.y, row0 = blockIdx.x * ROWS;
  const bool even = !(r & 1);

  c2 v[N1];
  {
    const int yb = row0 + lrow;
    const RotBox& bx = rot[r].b;
    const int z = zb + bx.org[0], y = yb + bx.org[1], ox = bx.org[2];   // voxel of box index (zb, yb, 0)
    // byte offsets into a rotation's volume fit 32 bits (2^24 voxels)
    const char* Vol = reinterpret_cast<const char*>(Bh + r * g.nvox);
    const uint8_t* M = Mh + r * g.nvox;
    const int sy = g.nx, sz = g.nx * g.ny;
    const bool row_in = yb < g.ey && z < g.nz && y < g.ny;
    const int nx_ok = row_in ? min(g.ex, g.nx - ox) : 0;
    const unsigned row = row_in ? z * sz + y * sy : 0u;
    const unsigned oc = 4 * row, oym = oc - (row_in && y > 0 ? 4 * sy : 0), oyp = oc + (row_in && y + 1 < g.ny ? 4 * sy : 0);
    const unsigned ozm = oc - (row_in && z > 0 ? 4 * sz : 0), ozp = oc + (row_in && z + 1 < g.nz ? 4 * sz : 0);
    auto vol = [&](unsigned o) { return __ldg(reinterpret_cast<const float*>(Vol + o)); };
    // masks are paired across consecutive rotations: the even rotation's mask
    // field carries (M_r, M_{r+1}), the partner's in its own box
    unsigned prow = 0;
    int pnx = 0;
    if (even && r + 1 < (int)gridDim.z && yb < g.ey) {
      const RotBox& pb = rot[r + 1].b;
      const int pz = zb + pb.org[0], py = yb + pb.org[1];
      if (pz < g.nz && py < g.ny) {
        pnx = min(g.ex, g.nx - pb.org[2]);
        prow = (unsigned)g.nvox + pz * sz + py * sy + pb.org[2];
      }
    }
    unsigned mb = 0, pb = 0;
#pragma unroll
    for (int n1 = 0; n1 < NI; ++n1) {
      const int x = N2 * n1 + n2;                 // box index
      if (x < nx_ok && M[row + ox + x]) mb |= 1u << n1;
      if (x < pnx && M[prow + x]) pb |= 1u << n1;
    }
    // the first NA inputs gathered, the others zero: one branch, so that the
    // gathers of all inputs are in flight together
    auto gather = [&](auto na) {
      constexpr int NA = decltype(na)::value;
#pragma unroll
      for (int n1 = 0; n1 < NI; ++n1) {
        if (n1 >= NA) {
          v[n1] = slot[n1 * NT] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
          continue;
        }
        const bool in = mb >> n1 & 1;
        const int xo = in ? 4 * (ox + N2 * n1 + n2) : 0;
        const float gx = 0.5f * (vol(oc + min(xo + 4, 4 * g.nx - 4)) - vol(oc + max(xo - 4, 0)));
        const float gy = 0.5f * (vol(oyp + xo) - vol(oym + xo));
        const float gz = 0.5f * (vol(ozp + xo) - vol(ozm + xo));
        const float inv = rsqrtf(gx * gx + gy * gy + gz * gz + g.eps2);
        // the NGF times the mask (m^2 = m: every product of two masked components
        // equals the product times m, bit for bit)
        const float X = in ? gx * inv : 0.0f, Y = in ? gy * inv : 0.0f, Z = in ? gz * inv : 0.0f;
        const float m = even && in ? 1.0f : 0.0f, m2 = pb >> n1 & 1 ? 1.0f : 0.0f;
        // Eq. 6 products (squared measure): (xx, yy) and (zz, xy), then (xz, yz) and
        // the mask pair; Eq. 3 (unsquared): (x, y) and (z, 0), then the mask pair
        if (g.nch == 3) {
          v[n1] = {make_float2(X * X, Z * Z), make_float2(Y * Y, X * Y)};
          slot[n1 * NT] = {make_float2(X * Z, m), make_float2(Y * Z, m2)};
        } else {
          v[n1] = {make_float2(X, Z), make_float2(Y, 0.0f)};
          slot[n1 * NT] = {make_float2(0.0f, m), make_float2(0.0f, m2)};
        }
      }
    };
    constexpr int NA = (3 * NI + 3) / 4;          // boxes of 3/4 of the length are typical
    if (N2 * NA >= g.ex) gather(std::integral_constant<int, NA>{});
    else gather(std::integral_constant<int, NI>{});
  }
#pragma unroll 1
  for (int pair = 0; pair < 2; ++pair) {
    if (pair) {
      __syncthreads();                            // the first pair has left the exchange
#pragma unroll
      for (int n1 = 0; n1 < NI; ++n1) v[n1] = slot[n1 * NT];
    }
    if constexpr (HALF) {
      c2 h[NI];
#pragma unroll
      for (int n1 = 0; n1 < NI; ++n1) h[n1] = v[n1];
      dft_half<N1, -1>(h, v);
    } else {
      Dft<N1, -1>::run(v);
    }
    c2* e = ex + lrow * CS + n2 * RS;
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) {
      const float2 w = __ldg(&kTwStep<P, N1, N2>.w[k1 * N2 + n2]);
      e[k1] = k1 == 0 ? v[k1] : cmul(v[k1], c2{dup(w.x), dup(w.y)});
    }
    __syncthreads();
    const int lr = t / N1, k1 = t - lr * N1;
    // the fields of this pair that exist: (0, 1), then (2 if nch == 3, the mask if
    // the rotation is even)
    const bool lo = pair == 0 || g.nch == 3, hi = pair == 0 || even;
    if (t < ROWS * N1 && row0 + lr < g.ey && (lo || hi)) {
      c2 u[N2];
      const c2* s = ex + lr * CS + k1;
#pragma unroll
      for (int i = 0; i < N2; ++i) u[i] = s[i * RS];
      Dft<N2, -1>::run(u);
      const long long E = (long long)g.ez * g.ey * P;
      const int j0 = 2 * pair, j1 = pair ? g.nch : 1;
      const int o = zb * P * g.ey + 4 * (row0 + lr);       // [z][kx/4][y][kx%4]
      const TileRun<N1> run(k1, g.ey);
      if (lo) {
        char* f0 = Fields<ST>::field(F0, g, E, r, j0);
        const float s0 = field_scale(g.scale0, j0);
#pragma unroll
        for (int i = 0; i < N2; ++i) Fields<ST>::put(f0, o + run.at(i), make_float2(u[i].x.x, u[i].y.x), false, s0);
      }
      if (hi) {
        char* f1 = Fields<ST>::field(F0, g, E, r, j1);
        const float s1 = field_scale(g.scale0, j1);
        if (pair == 0) {
#pragma unroll
          for (int i = 0; i < N2; ++i) Fields<ST>::put(f1, o + run.at(i), make_float2(u[i].x.y, u[i].y.y), false, s1);
        } else {
#pragma unroll
          for (int i = 0; i < N2; ++i) Fields<ST>::put(f1, o + run.at(i), make_float2(u[i].x.y, u[i].y.y), true, s1);
        }
      }
    }
  }
}

template <int P, bool HALF, int V>
void launch_fwd_x_t(const float* Bh, const uint8_t* Mh, void* F0, const RotIn* rot, Geo g, int nrot,
                    cudaStream_t st) {
  using C = FwdXCfg<P, HALF, V>;
  const dim3 grid((unsigned)((g.ey + C::ROWS - 1) / C::ROWS), (unsigned)g.ez, (unsigned)nrot);
  by_store<P>(g.store, [&](auto sf) {
    constexpr int ST = decltype(sf)::value;
    set_smem<k_fwd_x<P, ST, HALF, V>>(C::smem_bytes);
    k_fwd_x<P, ST, HALF, V><<<grid, C::NT, C::smem_bytes, st>>>(Bh, Mh, F0, rot, g);
  });
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
// fwd_y: y-axis FFT of every column of F0 (rows y >= ey are zero), to the z
// pass's tiles.  Block: one tile of four kx in four z planes of one (r, j).
// ---------------------------------------------------------------------------
// F0's tiles of four kx are contiguous over y, so a plane's columns arrive as
// one bulk copy, and four planes make 128-byte pieces of F1's tiles
// [kx][p/4][z][p%4] (one plane: 32-byte pieces, 31 us per rotation at 150^3
// against 29).  A block takes several groups of four planes, the copies of the
// next under the current one: a block of one group waited for its copy a third
// of its life.
template <int P, int V> struct FwdYCfg {
  static constexpr int N1 = SplitV<P, V>::N1, N2 = SplitV<P, V>::N2, W = 16;
  static constexpr int NT = W * N2;
  // exchange [column][n2][k1]: odd rows, and columns 4 rows apart (mod 16), put
  // four columns of four rows in different banks
  static constexpr int RS = N1 | 1, CS0 = N2 * RS, CS = CS0 + ((4 * RS - CS0) % 16 + 16) % 16;
  static constexpr size_t smem_bytes(int ey) { return ((size_t)W * CS + (size_t)2 * W * ey) * sizeof(float2) + 16; }
  static constexpr int MIN_BLOCKS = pass_blocks(NT, smem_bytes(3 * P / 4), N2 > 20 ? 80 : 64);
};

template <int P, int ST, bool HALF, int V>
__global__ void __launch_bounds__(FwdYCfg<P, V>::NT, FwdYCfg<P, V>::MIN_BLOCKS)
k_fwd_y(const void* __restrict__ F0, void* __restrict__ F1, Geo g, int groups) {
  using C = FwdYCfg<P, V>;
  constexpr int N1 = C::N1, N2 = C::N2, W = C::W, RS = C::RS, CS = C::CS, NI = HALF ? N1 / 2 : N1;
  extern __shared__ __align__(128) float2 ysm[];
  float2* in = ysm;                                  // [2][4 z][ey][4 kx] (4-byte values in the 16-bit forms)
  float2* ex = in + 2 * W * g.ey;                    // [W][CS]
  uint64_t* bar = reinterpret_cast<uint64_t*>(ex + W * CS);
  const int t = threadIdx.x;
  const int rj = blockIdx.z;                         // r * nf + j
  const int r = g.nf == 4 ? rj >> 2 : rj / 3, j = rj - r * g.nf;
  const bool is_mask = j == g.nch;
  if (is_mask && (r & 1)) return;                    // paired into the even rotation's mask field
  const bool wide = ST == kStoreF32 || is_mask;
  const uint32_t bytes = (uint32_t)g.ey * 4 * (wide ? 8 : 4);   // of one plane's tile
  const int zbeg = 4 * groups * blockIdx.y, zend = min(g.ez, zbeg + 4 * groups);
  auto fetch = [&](int z0, int s) {                  // one thread: planes z0 .. z0 + 3
    if (z0 >= zend) return;
    const int nz = min(4, zend - z0);
    const char* src = Fields<ST>::field(F0, g, (long long)g.ez * g.ey * g.Px, r, j);
    tc::mbar_expect(&bar[s], nz * bytes);
    for (int z = 0; z < nz; ++z)
      tc::bulk_load(reinterpret_cast<char*>(in + s * W * g.ey) + z * bytes,
                    src + ((long long)(z0 + z) * (g.Px / 4) + blockIdx.x) * bytes, bytes, &bar[s]);
  };
  if (t == 0) {
    tc::mbar_init(&bar[0], 1);
    tc::mbar_init(&bar[1], 1);
    tc::mbar_init_fence();
    fetch(zbeg, 0);
    fetch(zbeg + 4, 1);
  }
  __syncthreads();                                   // the barriers are initialised
  int dead = -1;                                     // the group whose wait ran out: no more waits, results invalid
  int it = 0;
#pragma unroll 1
  for (int z0 = zbeg; z0 < zend; z0 += 4, ++it) {
    const int nz = min(4, zend - z0);
    const float2* src = in + (it & 1) * W * g.ey;
    if (dead < 0 && !tc::mbar_wait(&bar[it & 1], (it >> 1) & 1, kTcWaitNs)) dead = it;
    {
      const int kxi = t & 3, n2 = (t >> 2) % N2, zz = t / (4 * N2);
      const float isc = 1.0f / field_scale(g.scale0, j);
      const int o = (zz * g.ey + n2) * 4 + kxi;
      float2 v[NI];                                  // y < ey: with ey <= P/2 the upper half is zero
      auto rows = [&](auto mc) {
#pragma unroll
        for (int n1 = 0; n1 < NI; ++n1)
          v[n1] = N2 * n1 + n2 < g.ey && zz < nz
                      ? Fields<ST>::get(reinterpret_cast<const char*>(src), o + 4 * N2 * n1, decltype(mc)::value, isc)
                      : make_float2(0.f, 0.f);
      };
      if (wide) rows(std::true_type{});
      else rows(std::false_type{});
      float2* e = ex + (zz * 4 + kxi) * CS + n2 * RS;
      float2 a[N1];
      if constexpr (HALF) {
        dft_half<N1, -1>(v, a);
      } else {
#pragma unroll
        for (int i = 0; i < N1; ++i) a[i] = v[i];
        Dft<N1, -1>::run(a);
      }
#pragma unroll
      for (int k1 = 0; k1 < N1; ++k1) {
        const float2 w = __ldg(&kTwStep<P, N1, N2>.w[k1 * N2 + n2]);
        e[k1] = k1 == 0 ? a[k1] : cmul(a[k1], w);
      }
    }
    __syncthreads();
    // this group's inputs have been read (dead: its phase is still open, and a
    // second arrival on it would be undefined)
    if (t == 0 && dead < 0) fetch(z0 + 8, it & 1);
    if (t < W * N1) {
      const int k1 = t % N1, kxi = t / N1 & 3, zz = t / (4 * N1);
      if (zz < nz) {
        float2 u[N2];
        const float2* s = ex + (zz * 4 + kxi) * CS + k1;
#pragma unroll
        for (int i = 0; i < N2; ++i) u[i] = s[i * RS];
        Dft<N2, -1>::run(u);
        char* dst = Fields<ST>::field(F1, g, (long long)g.ez * g.Px * ky_total(P), r, j);
        const int row = (4 * blockIdx.x + kxi) * ky_total(P) * g.ez + 4 * (z0 + zz);
        const KyRun<P, N1, N2> run(k1, g.ez);
        const float sc = field_scale(g.scale1, j);
        if (is_mask) {
#pragma unroll
          for (int k2 = 0; k2 < N2; ++k2) Fields<ST>::put(dst, row + run.at(k2), u[k2], true, sc);
        } else {
#pragma unroll
          for (int k2 = 0; k2 < N2; ++k2) Fields<ST>::put(dst, row + run.at(k2), u[k2], false, sc);
        }
      }
    }
    __syncthreads();
  }
  if (dead >= 0) {                                   // the copies still in flight end before the block does
    atomicExch(g.wait_err, 1);
    if (t == 0)
      for (int l = dead; l < it && l < dead + 2; ++l) tc::mbar_wait(&bar[l & 1], (l >> 1) & 1, kTcWaitNs / 4);
  }
}

template <int P, int V>
void launch_fwd_y_t(const void* F0, void* F1, Geo g, int nrot, cudaStream_t st) {
  using C = FwdYCfg<P, V>;
  const size_t smem = C::smem_bytes(g.ey);
  // groups of four planes per block: more where there are blocks to spare
  const int quads = (g.ez + 3) / 4;
  int groups = 1;
  while (groups < 4 && (long long)(g.Px / 4) * nrot * g.nf * (quads / (2 * groups)) >= 152 * C::MIN_BLOCKS * 8) groups *= 2;
  const dim3 grid((unsigned)(g.Px / 4), (unsigned)((quads + groups - 1) / groups), (unsigned)(nrot * g.nf));
  by_store<P>(g.store, [&](auto sf) {
    constexpr int ST = decltype(sf)::value;
    by_half<P, V>(g.ey, [&](auto hc) {
      constexpr bool HALF = decltype(hc)::value;
      set_smem<k_fwd_y<P, ST, HALF, V>>(smem);
      k_fwd_y<P, ST, HALF, V><<<grid, C::NT, smem, st>>>(F0, F1, g, groups);
    });
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
      by_half_z<P, V>(g.ez, [&](auto hc) {
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
  by_half_z<P, 0>(g.ez, [&](auto hc) {
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
    const float2* src = F2 + (((long long)r * g.Px + kx) * g.wz + dz) * (long long)ky_total(P);   // [r][kx][dz][p]
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1)
      v[n1] = (kx < g.Px) ? src[ky_pos(N2 * n1 + n2, P)] : make_float2(0.f, 0.f);
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
    set_smem<k_inv_y<P, W, V>>(smem);
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
    set_smem<k_inv_x<P, ROWS, V>>(smem);
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
