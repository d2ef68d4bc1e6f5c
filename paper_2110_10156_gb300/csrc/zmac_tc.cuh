// The channel fields' half of the z pass in the reduced-precision forms: their
// forward z-axis DFT on the tensor cores (tcgen05, FP32 accumulation in tensor
// memory) and the Eq. 7-8 sum X, written to HBM.  Included by passes.cuh;
// k_zpass (kZFromX) reads X, transforms the mask field in FP32 and runs the
// inverse.
//
// The dense DFT: for a column b(z), z < nz, of a packed complex field and
// kz in [0, P/2]
//     C[kz][z] = cos(2 pi kz z / P),  S[kz][z] = sin(2 pi kz z / P)
//     H(kz)     = (C.re b + S.im b) + i (C.im b - S.re b)
//     H(P - kz) = (C.re b - S.im b) + i (C.im b + S.re b)
// so two M = 128 products (C and S, rows kz, K = z padded to a multiple of
// 16) give every frequency of every column.  The B operand is a tile of the
// 16-bit field values as they lie in F1 ([kx][p/4][z][p%4] with (re, im) pairs):
// N-major, its columns (field, primary / mirror, column, re / im), so that
// a tile of it is a bulk copy.  Tensor memory lane
// kz then holds H at kz and P - kz of a column and of its mirror column
// (-kx, -ky), which is all the multiply-accumulate of that frequency pair
// needs.  The mask field (the overlap count N) and the inverse stay on the
// FP32 CUDA-core transforms, so N(chi) keeps FP32 accuracy.
#pragma once

#include <algorithm>

#include "tc.cuh"

namespace csngf {

template <int ST>
__device__ __forceinline__ void store16(unsigned char* p, float v) {
  if constexpr (ST == kStoreBF16) *reinterpret_cast<__nv_bfloat16*>(p) = __float2bfloat16_rn(v);
  else *reinterpret_cast<__half*>(p) = __float2half_rn(v);
}

// ---------------------------------------------------------------------------
// X costs one write and one read of a half spectrum of complex values per
// rotation; in exchange the tensor-core kernel double-buffers its operands and
// keeps no CUDA-core transform in its per-rotation chain.
// X layout: [r][kx <= P/2][p/4][kz][p%4].
//
// k_zx_tc, per block: one kx, W = 8 columns (two tiles) and their mirrors, every
// rotation of the launch; the cos / sin tiles and the block's weights stay
// in shared memory.  Rotation r + 1's MMAs run while rotation r's products
// are summed; rotation r + 2's operand is copied (twelve bulk copies) as soon as
// rotation r's MMAs are done.  16 warps, four per tensor-memory lane quarter.
// ---------------------------------------------------------------------------
template <int P>
struct ZxTcCfg {
  static constexpr int W = 8;                          // primary columns per block
  static constexpr int NT = 512;                       // 16 warps: 4 per tensor-memory lane quarter,
                                                       // each summing two primary columns
  static constexpr int HF = P / 2;
  static constexpr bool OK = HF + 1 <= 128;
  static constexpr uint32_t TMEM_COLS = 512;           // 2 buffers x (C, S) x N <= 512 columns
  static constexpr size_t bytes(int kp, int nb, int nuv) {
    return (size_t)2 * 128 * kp * 2 + (size_t)2 * nb * kp * 2 + (size_t)nuv * W * P * 8 + 64;
  }
};

template <int P, int ST>
__global__ void __launch_bounds__(ZxTcCfg<P>::NT, 1)
k_zx_tc(const void* __restrict__ F1, const float2* __restrict__ UV, float2* __restrict__ Xg,
        Geo g, int nrot, int KP) {
  const float2* __restrict__ tw = kTw<P>.w;
  using C = ZxTcCfg<P>;
  constexpr int W = C::W, NT = C::NT, TILE = W * P, HF = C::HF;
  const int NB = g.nch * 4 * W;                    // MMA N: (field, primary/mirror, column, re/im)
  const int NUV = 2 * g.nch;                       // weight channels
  extern __shared__ __align__(128) unsigned char smem_raw[];
  unsigned char* As = smem_raw;                    // [cos | sin][128][KP], K-major
  const uint32_t tileA = 128u * (uint32_t)KP * 2u;
  const uint32_t sbo = (uint32_t)KP * 16u;
  unsigned char* Bs = As + 2 * tileA;              // [2][KP][NB], N-major
  const uint32_t stageB = (uint32_t)NB * (uint32_t)KP * 2u;
  float2* uvs = reinterpret_cast<float2*>(Bs + 2 * stageB);   // [NUV][W][P]
  uint64_t* mbar = reinterpret_cast<uint64_t*>(uvs + (size_t)NUV * TILE);   // products of each buffer
  uint64_t* bar = mbar + 2;                        // operands of each stage
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 2);

  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int kx = blockIdx.y;
  const int mkx = (g.Px - kx) % g.Px;
  const int ntile = 2 * gridDim.x, half = ky_half(g.Py) / 4;   // tiles of four columns
  const long long E = (long long)g.ez * g.Px * 4 * ntile;

  // operand rows past the box stay zero
  for (int q = t; q < 2 * (NB / 8) * (KP - g.ez); q += NT) {
    const int n8 = q / (KP - g.ez), k = g.ez + q - n8 * (KP - g.ez);
    reinterpret_cast<uint4*>(Bs)[n8 * KP + k] = make_uint4(0u, 0u, 0u, 0u);
  }
  // the block's weights, [tile][field][kz][column][a, b] in HBM, transposed so that
  // kz runs over the lanes
  for (int q = t; q < NUV * TILE; q += NT) {
    const int i = q % (NUV * TILE / 2), h = q / (NUV * TILE / 2);   // entry of the block's tile h
    const int j = i / TILE, k = i % TILE / 8, c = 4 * h + i % 8 / 2, s = i & 1;
    cp_async8(uvs + (2 * j + s) * TILE + c * P + k,
              UV + ((long long)kx * ntile + 2 * blockIdx.x + h) * (NUV + 1) * 4 * P + i);
  }
  for (int m = warp; m < 128; m += NT / 32) {
    int e = m * lane % P;                          // m k mod P
    const int step = 32 * m % P;
    for (int k = lane; k < KP; k += 32, e = e + step >= P ? e + step - P : e + step) {
      float cv = 0.f, sv = 0.f;
      if (m <= HF && k < g.ez) {
        const float2 w = __ldg(&tw[e]);             // exp(-2 pi i m k / P)
        cv = w.x;
        sv = -w.y;
      }
      const uint32_t off = (uint32_t)(m / 8) * sbo + (uint32_t)(k / 8) * 128u + (m % 8) * 16 + (k % 8) * 2;
      store16<ST>(As + off, cv);
      store16<ST>(As + tileA + off, sv);
    }
  }
  if (t == 0) {
    for (int i = 0; i < 4; ++i) tc::mbar_init(&mbar[i], 1);
    tc::mbar_init_fence();
  }
  if (warp == 0) tc::alloc(tslot, C::TMEM_COLS);

  // A tile's columns are N-major operand rows as they lie in F1 (16 bytes per z),
  // so a field takes four bulk copies: the block's two tiles and the two of their
  // mirrors.  Where a tile's first column is ky = 0 or P/2, its own mirror, that
  // column is filled in by the threads (own_h: the tile, or -1).
  const int own_h = blockIdx.x == 0 ? 0 : half / 2 == (int)blockIdx.x ? half & 1 : -1;
  const long long tz = 4LL * g.ez;                 // values per tile
  auto fetch_b = [&](int r, int s) {               // one thread
    if (r >= nrot) return;
    const uint32_t bytes = (uint32_t)g.ez * 16;
    tc::mbar_expect(&bar[s], 4 * g.nch * bytes);
    for (int j = 0; j < g.nch; ++j) {
      const char* src = Fields<ST>::field(F1, g, E, r, j);
      unsigned char* d = Bs + (size_t)s * stageB + (uint32_t)(4 * j) * sbo;
      for (int h = 0; h < 2; ++h) {
        const int tile = 2 * blockIdx.x + h, mtile = tile < half ? tile + half : tile - half;
        tc::bulk_load(d + h * sbo, src + ((long long)kx * ntile + tile) * tz * 4, bytes, &bar[s]);
        tc::bulk_load(d + (2 + h) * sbo, src + ((long long)mkx * ntile + mtile) * tz * 4, bytes, &bar[s]);
      }
    }
  };
  auto patch_b = [&](int r, int s) {               // all threads, after the copies
    const long long o = ((long long)mkx * ntile + 2 * blockIdx.x + own_h) * tz;
    for (int q = t; q < g.nch * g.ez; q += NT) {
      const int j = q / g.ez, z = q - j * g.ez;
      *reinterpret_cast<uint32_t*>(Bs + (size_t)s * stageB + (uint32_t)(4 * j + 2 + own_h) * sbo + z * 16) =
          reinterpret_cast<const uint32_t*>(Fields<ST>::field(F1, g, E, r, j))[o + 4 * z];
    }
    tc::fence_async_smem();
  };
  const uint32_t idesc = tc::idesc_f16(ST == kStoreBF16, 0, 1, 128, NB);
  auto issue = [&](uint32_t tmem, int s) {         // operand stage s -> tensor-memory buffer s
    tc::fence_after_sync();
    const uint32_t a0 = tc::smem_addr(As), b0 = tc::smem_addr(Bs + (size_t)s * stageB);
    const uint32_t d0 = tmem + (uint32_t)(s * 2 * NB);
    for (int q = 0; q < KP / 16; ++q) {
      const uint64_t bd = tc::desc(b0 + q * 256, 128, sbo);
      tc::mma_f16(d0, tc::desc(a0 + q * 256, 128, sbo), bd, idesc, q > 0);
      tc::mma_f16(d0 + NB, tc::desc(a0 + tileA + q * 256, 128, sbo), bd, idesc, q > 0);
    }
    tc::commit(&mbar[s]);
  };

  cp_async_wait_all();                             // the weights
  tc::fence_async_smem();                          // the tables and zero rows, for the tensor core and the copies
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tslot;
  if (t == 0) {
    fetch_b(0, 0);
    fetch_b(1, 1);
  }
  // rotation r's operand has landed (and is completed): its products start
  auto start = [&](int r) {
    if (own_h >= 0) {
      if (tc::mbar_wait(&bar[r & 1], (uint32_t)((r >> 1) & 1), kTcWaitNs)) patch_b(r, r & 1);
      __syncthreads();
    }
    if (t == 0 && tc::mbar_wait(&bar[r & 1], (uint32_t)((r >> 1) & 1), kTcWaitNs)) issue(tmem, r & 1);
  };
  start(0);

  bool failed = false;
  int fail_buf = 0, fail_next = -1;
  uint32_t fail_par = 0;
  const int lq = warp & 3, cg = warp >> 2;         // lane quarter, column pair
  const int kz = lq * 32 + lane;
  const bool kz_ok = kz <= HF;
  const int kzm = kz == 0 ? 0 : P - kz;
#pragma unroll 1
  for (int r = 0; r < nrot; ++r) {
    const int s = r & 1;
    // (1) rotation r's products are done; its operand stage takes rotation r + 2
    const bool ok = tc::mbar_wait(&mbar[s], (uint32_t)((r >> 1) & 1), kTcWaitNs);
    if (__syncthreads_or(!ok)) {
      failed = true;
      fail_buf = s;
      fail_par = (uint32_t)((r >> 1) & 1);
      fail_next = r + 1 < nrot ? r + 1 : r;
      break;
    }
    tc::fence_after_sync();
    if (t == 0) fetch_b(r + 2, s);
    // (2) rotation r + 1's products (the barrier above also orders rotation
    // r - 1's tensor-memory reads of that buffer)
    if (r + 1 < nrot) start(r + 1);
    // (3) Eq. 7-8: X at kz and P - kz of this thread's four primary columns
    const uint32_t trow = tmem + ((uint32_t)(lq * 32) << 16) + (uint32_t)(s * 2 * NB);
    float2* Xr = Xg + (((long long)r * gridDim.y + kx) * ntile + 2 * blockIdx.x + (cg >> 1)) * 4 * P + 2 * (cg & 1);
    {
      const int ch = cg;                           // primary columns 2 ch, 2 ch + 1
      uint32_t rc[3][4], rs[3][4], rcm[3][4], rsm[3][4];
#pragma unroll
      for (int j = 0; j < 3; ++j)
        if (j < g.nch) {
          const uint32_t col = (uint32_t)(j * 4 * W + 4 * ch);
          tc::ld4(trow + col, rc[j]);
          tc::ld4(trow + NB + col, rs[j]);
          tc::ld4(trow + 16 + col, rcm[j]);
          tc::ld4(trow + NB + 16 + col, rsm[j]);
        }
      tc::wait_ld();
      if (kz_ok) {
        float2 Xa[2], Xb[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int c = 2 * ch + i;
          Xa[i] = Xb[i] = make_float2(0.f, 0.f);
#pragma unroll
          for (int j = 0; j < 3; ++j)
            if (j < g.nch) {
              const float isc = ST == kStoreF16 ? 1.0f / field_scale(g.scale1, j) : 1.0f;
              const float Cr = __uint_as_float(rc[j][2 * i]) * isc, Ci = __uint_as_float(rc[j][2 * i + 1]) * isc;
              const float Cmr = __uint_as_float(rcm[j][2 * i]) * isc;
              const float Cmi = __uint_as_float(rcm[j][2 * i + 1]) * isc;
              const float Sr = __uint_as_float(rs[j][2 * i]) * isc, Si = __uint_as_float(rs[j][2 * i + 1]) * isc;
              const float Smr = __uint_as_float(rsm[j][2 * i]) * isc;
              const float Smi = __uint_as_float(rsm[j][2 * i + 1]) * isc;
              // H = (Cr + Si, Ci - Sr) at kz and (Cr - Si, Ci + Sr) at P - kz, its mirror H'
              // likewise; channels a = H + conj H', b = -i (H - conj H') at both
              const float p = Cr + Cmr, q = Cr - Cmr, u = Si - Smi, v = Si + Smi;
              const float e = Ci - Cmi, f = Ci + Cmi, g1 = Sr + Smr, h = Sr - Smr;
              const float2* Wa = uvs + (2 * j) * TILE + c * P;
              const float2* Wb = Wa + TILE;
              cmac(Xa[i], Wa[kz], make_float2(p + u, e - g1));
              cmac(Xa[i], Wb[kz], make_float2(f - h, -q - v));
              cmac(Xb[i], Wa[kzm], make_float2(p - u, e + g1));
              cmac(Xb[i], Wb[kzm], make_float2(f + h, v - q));
            }
        }
        *reinterpret_cast<float4*>(Xr + kz * 4) = make_float4(Xa[0].x, Xa[0].y, Xa[1].x, Xa[1].y);
        if (kzm != kz)
          *reinterpret_cast<float4*>(Xr + kzm * 4) = make_float4(Xb[0].x, Xb[0].y, Xb[1].x, Xb[1].y);
      }
    }
    tc::fence_before_sync();
  }
  if (failed) {                                    // its copies and products, and the next rotation's copies
    if (t == 0) atomicExch(g.wait_err, 1);
    tc::mbar_wait(&bar[fail_buf], fail_par, kTcWaitNs / 4);
    tc::mbar_wait(&mbar[fail_buf], fail_par, kTcWaitNs / 4);
    if (fail_next >= 0) tc::mbar_wait(&bar[fail_next & 1], (uint32_t)((fail_next >> 1) & 1), kTcWaitNs / 4);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::dealloc(tmem, C::TMEM_COLS);
}

// the channel sum X into g.zx when the length, precision form and shared memory
// allow it; false otherwise
template <int P, int ST>
bool launch_zx_tc(const void* F1, const float2* UV, Geo g, int nrot, cudaStream_t st) {
  using C1 = ZxTcCfg<P>;
  if constexpr (!C1::OK) {
    return false;
  } else {
    if (!g.zx) return false;
    const int KP = (g.ez + 15) / 16 * 16;
    const int NB = g.nch * 4 * C1::W;
    if (NB > 128 || NB % 16 != 0) return false;
    if (C1::bytes((g.nz + 15) / 16 * 16, NB, 2 * g.nch) > 232448) return false;
    const size_t s1 = std::max<size_t>(C1::bytes(KP, NB, 2 * g.nch), 120 * 1024);   // one block per SM: all of its tensor memory
    set_smem<k_zx_tc<P, ST>>(s1);
    dim3 grid((unsigned)(ky_total(g.Py) / C1::W), (unsigned)(g.Px / 2 + 1));
    k_zx_tc<P, ST><<<grid, C1::NT, s1, st>>>(F1, UV, g.zx, g, nrot, KP);
    return true;
  }
}

}  // namespace csngf
