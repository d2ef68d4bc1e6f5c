// Register-level DFTs and the two-level (four-step) block FFT used by every
// transform pass of the all-shift NGF correlation (Eq. 7-8: the channel and
// mask correlations are evaluated in the frequency domain).
//
// Conventions: forward transforms use S = -1, X[k] = sum_n x[n] exp(-2 pi i nk/N);
// inverse transforms use S = +1 and are unnormalised.
//
// A length N = N1 * N2 transform is split as n = N2*n1 + n2, k = k1 + N1*k2:
//   step 1: for each n2, an N1-point DFT over n1 in registers, then the
//           twiddle exp(S 2 pi i n2 k1 / N), then a store to shared memory;
//   step 2: for each k1, an N2-point DFT over n2 in registers; its k2-th
//           output is X[k1 + N1*k2].
// One shared-memory exchange per transform; the caller decides where the
// step-1 inputs come from and where the step-2 outputs go.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <utility>
#include <type_traits>

namespace csngf {

// ---------------------------------------------------------------- twiddles
// Compile-time cos/sin of 2*pi*e/R from their Maclaurin series after an exact
// quadrant reduction done in integers, so quarter-turn twiddles are exact.
namespace ctw {
constexpr double kPi = 3.141592653589793238462643383279502884;
constexpr double sin_series(double a) {
  double a2 = a * a, term = a, sum = a;
  for (int k = 1; k <= 14; ++k) { term *= -a2 / ((2.0 * k) * (2.0 * k + 1.0)); sum += term; }
  return sum;
}
constexpr double cos_series(double a) {
  double a2 = a * a, term = 1.0, sum = 1.0;
  for (int k = 1; k <= 14; ++k) { term *= -a2 / ((2.0 * k - 1.0) * (2.0 * k)); sum += term; }
  return sum;
}
// angle = 2*pi*e/R = q*(pi/2) + (pi/2)*rem/R with rem in [0, R)
constexpr double cos2pi(long e, long R) {
  e %= R; if (e < 0) e += R;
  long q = (4 * e) / R, rem = 4 * e - q * R;
  double a = (kPi / 2.0) * (double)rem / (double)R;
  double c = cos_series(a), s = sin_series(a);
  return (q & 3) == 0 ? c : (q & 3) == 1 ? -s : (q & 3) == 2 ? -c : s;
}
constexpr double sin2pi(long e, long R) {
  e %= R; if (e < 0) e += R;
  long q = (4 * e) / R, rem = 4 * e - q * R;
  double a = (kPi / 2.0) * (double)rem / (double)R;
  double c = cos_series(a), s = sin_series(a);
  return (q & 3) == 0 ? s : (q & 3) == 1 ? c : (q & 3) == 2 ? -s : -c;
}
}  // namespace ctw

// exp(-2 pi i m / P), m < P, as a constant table of the module (rounded from
// FP64), so that a change of FFT length uploads nothing and waits for nothing
template <int P>
struct TwTable { float2 w[P]; };
template <int P>
constexpr TwTable<P> make_twiddles() {
  TwTable<P> t{};
  for (int m = 0; m < P; ++m) {
    t.w[m].x = (float)ctw::cos2pi(m, P);
    t.w[m].y = (float)(-ctw::sin2pi(m, P));
  }
  return t;
}
template <int P>
__device__ const TwTable<P> kTw = make_twiddles<P>();
// the first step's twiddles exp(-2 pi i k1 n2 / P) as [k1][n2]: lanes over n2 read
// consecutive entries
template <int P, int N1, int N2>
constexpr TwTable<P> make_step_twiddles() {
  TwTable<P> t{};
  for (int k = 0; k < N1; ++k)
    for (int n = 0; n < N2; ++n) {
      t.w[k * N2 + n].x = (float)ctw::cos2pi((long)k * n, P);
      t.w[k * N2 + n].y = (float)(-ctw::sin2pi((long)k * n, P));
    }
  return t;
}
template <int P, int N1, int N2>
__device__ const TwTable<P> kTwStep = make_step_twiddles<P, N1, N2>();

// ---------------------------------------------------------------- complex
// Complex add and subtract as one paired FP32 instruction (add/sub.rn.f32x2:
// each lane rounds exactly as a scalar add), half the issue slots of two adds.
__device__ __forceinline__ float2 cadd(float2 a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 pa, pb, pr;\n\tmov.b64 pa, {%2, %3};\n\tmov.b64 pb, {%4, %5};\n\t"
      "add.rn.f32x2 pr, pa, pb;\n\tmov.b64 {%0, %1}, pr;\n\t}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 pa, pb, pr;\n\tmov.b64 pa, {%2, %3};\n\tmov.b64 pb, {%4, %5};\n\t"
      "sub.rn.f32x2 pr, pa, pb;\n\tmov.b64 {%0, %1}, pr;\n\t}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// asynchronous global -> shared copies (cp.async, L1-allocating); the copies a
// thread issued are visible to that thread after cp_async_wait_all()
__device__ __forceinline__ void cp_async8(void* smem_dst, const void* gsrc) {
  const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(gsrc) : "memory");
}
// (wait_group 0 would not wait for copies that no commit_group closed)
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
// a * (S i)
template <int S>
__device__ __forceinline__ float2 mul_si(float2 a) {
  return S < 0 ? make_float2(a.y, -a.x) : make_float2(-a.y, a.x);
}

// static for-loop with compile-time index
template <class F, int... I>
__device__ __forceinline__ void sfor_impl(F&& f, std::integer_sequence<int, I...>) {
  (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void sfor(F&& f) {
  sfor_impl(f, std::make_integer_sequence<int, N>{});
}

// multiply by exp(S 2 pi i E / R), E a compile-time constant
template <int R, int S, int E>
__device__ __forceinline__ float2 tw_mul(float2 x) {
  constexpr int e = ((E % R) + R) % R;
  if constexpr (e == 0) {
    return x;
  } else if constexpr (2 * e == R) {
    return make_float2(-x.x, -x.y);
  } else if constexpr (4 * e == R) {
    return mul_si<S>(x);
  } else if constexpr (4 * e == 3 * R) {
    return mul_si<-S>(x);
  } else {
    constexpr float c = (float)ctw::cos2pi(e, R);
    constexpr float s = (float)(S * ctw::sin2pi(e, R));
    return make_float2(x.x * c - x.y * s, x.x * s + x.y * c);
  }
}
// a + S i d, a - S i d; a + c t, c t
template <int S> __device__ __forceinline__ float2 add_si(float2 a, float2 d) { return cadd(a, mul_si<S>(d)); }
template <int S> __device__ __forceinline__ float2 sub_si(float2 a, float2 d) { return csub(a, mul_si<S>(d)); }
__device__ __forceinline__ float2 cmad(float2 a, float2 t, float c) { return make_float2(a.x + c * t.x, a.y + c * t.y); }

// Two complex values side by side, x their real and y their imaginary parts:
// every step of two transforms at once is paired FP32 instructions without
// moves between lanes, half the issue slots (the z pass: 30 M warp
// instructions per rotation with one value per step, issue-bound latency at
// 16 warps per SM).
struct __align__(16) c2 { float2 x, y; };
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 pa, pb, pr;\n\tmov.b64 pa, {%2, %3};\n\tmov.b64 pb, {%4, %5};\n\t"
      "mul.rn.f32x2 pr, pa, pb;\n\tmov.b64 {%0, %1}, pr;\n\t}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 r;
  asm("{\n\t.reg .b64 pa, pb, pc, pr;\n\tmov.b64 pa, {%2, %3};\n\tmov.b64 pb, {%4, %5};\n\t"
      "mov.b64 pc, {%6, %7};\n\tfma.rn.f32x2 pr, pa, pb, pc;\n\tmov.b64 {%0, %1}, pr;\n\t}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return r;
}
__device__ __forceinline__ float2 dup(float s) { return make_float2(s, s); }
__device__ __forceinline__ c2 cadd(c2 a, c2 b) { return {cadd(a.x, b.x), cadd(a.y, b.y)}; }
__device__ __forceinline__ c2 csub(c2 a, c2 b) { return {csub(a.x, b.x), csub(a.y, b.y)}; }
__device__ __forceinline__ c2 cscale(c2 a, float s) { return {mul2(a.x, dup(s)), mul2(a.y, dup(s))}; }
__device__ __forceinline__ c2 cmad(c2 a, c2 t, float c) { return {fma2(t.x, dup(c), a.x), fma2(t.y, dup(c), a.y)}; }
template <int S> __device__ __forceinline__ c2 add_si(c2 a, c2 d) {
  return S < 0 ? c2{cadd(a.x, d.y), csub(a.y, d.x)} : c2{csub(a.x, d.y), cadd(a.y, d.x)};
}
template <int S> __device__ __forceinline__ c2 sub_si(c2 a, c2 d) { return add_si<-S>(a, d); }
// both values times w = (wx, wx), (wy, wy)
__device__ __forceinline__ c2 cmul(c2 v, c2 w) {
  const float2 n = make_float2(-w.y.x, -w.y.y);
  return {fma2(v.y, n, mul2(v.x, w.x)), fma2(v.x, w.y, mul2(v.y, w.x))};
}
template <int R, int S, int E>
__device__ __forceinline__ c2 tw_mul(c2 v) {
  constexpr int e = ((E % R) + R) % R;
  if constexpr (e == 0) {
    return v;
  } else {
    constexpr float c = (float)ctw::cos2pi(e, R);
    constexpr float s = (float)(S * ctw::sin2pi(e, R));
    if constexpr (2 * e == R) return {mul2(v.x, dup(-1.0f)), mul2(v.y, dup(-1.0f))};
    else if constexpr (4 * e == R || 4 * e == 3 * R)
      return s < 0 ? c2{v.y, mul2(v.x, dup(-1.0f))} : c2{mul2(v.y, dup(-1.0f)), v.x};
    else return {fma2(v.y, dup(-s), mul2(v.x, dup(c))), fma2(v.x, dup(s), mul2(v.y, dup(c)))};
  }
}

// ---------------------------------------------------------------- DFTs
// of R values of T (float2: one complex value, c2: two side by side)
template <int R, int S>
struct Dft;

template <int S>
struct Dft<1, S> {
  template <class T>
  __device__ __forceinline__ static void run(T (&)[1]) {}
};

template <int S>
struct Dft<2, S> {
  template <class T>
  __device__ __forceinline__ static void run(T (&v)[2]) {
    T a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  }
};

template <int S>
struct Dft<3, S> {
  template <class T>
  __device__ __forceinline__ static void run(T (&v)[3]) {
    constexpr float c1 = (float)ctw::cos2pi(1, 3), s1 = (float)ctw::sin2pi(1, 3);
    const T t = cadd(v[1], v[2]), d = csub(v[1], v[2]);
    const T x0 = v[0];
    v[0] = cadd(x0, t);
    const T a = cmad(x0, t, c1), b = cscale(d, s1);
    v[1] = add_si<S>(a, b);                      // a + S i sin(2 pi/3) (x1 - x2)
    v[2] = sub_si<S>(a, b);
  }
};

template <int S>
struct Dft<4, S> {
  template <class T>
  __device__ __forceinline__ static void run(T (&v)[4]) {
    T a0 = cadd(v[0], v[2]), a1 = csub(v[0], v[2]);
    T b0 = cadd(v[1], v[3]), b1 = csub(v[1], v[3]);
    v[0] = cadd(a0, b0);
    v[2] = csub(a0, b0);
    v[1] = add_si<S>(a1, b1);
    v[3] = sub_si<S>(a1, b1);
  }
};

template <int S>
struct Dft<5, S> {
  template <class T>
  __device__ __forceinline__ static void run(T (&v)[5]) {
    constexpr float c1 = (float)ctw::cos2pi(1, 5), c2_ = (float)ctw::cos2pi(2, 5);
    constexpr float s1 = (float)ctw::sin2pi(1, 5), s2 = (float)ctw::sin2pi(2, 5);
    T t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]);
    T t3 = csub(v[1], v[4]), t4 = csub(v[2], v[3]);
    T x0 = v[0];
    v[0] = cadd(x0, cadd(t1, t2));
    const T a1 = cmad(cmad(x0, t1, c1), t2, c2_), a2 = cmad(cmad(x0, t1, c2_), t2, c1);
    const T b1 = cmad(cscale(t3, s1), t4, s2), b2 = cmad(cscale(t3, s2), t4, -s1);
    // X1 = a1 + S i b1, X4 = a1 - S i b1, X2 = a2 + S i b2, X3 = a2 - S i b2
    v[1] = add_si<S>(a1, b1);
    v[4] = sub_si<S>(a1, b1);
    v[2] = add_si<S>(a2, b2);
    v[3] = sub_si<S>(a2, b2);
  }
};

template <int S>
struct Dft<7, S> {
  template <class T>
  __device__ __forceinline__ static void run(T (&v)[7]) {
    constexpr float c[3] = {(float)ctw::cos2pi(1, 7), (float)ctw::cos2pi(2, 7), (float)ctw::cos2pi(3, 7)};
    constexpr float s[3] = {(float)ctw::sin2pi(1, 7), (float)ctw::sin2pi(2, 7), (float)ctw::sin2pi(3, 7)};
    const T x0 = v[0];
    T t[3], d[3];
    sfor<3>([&](auto ic) { constexpr int i = decltype(ic)::value; t[i] = cadd(v[i + 1], v[6 - i]); d[i] = csub(v[i + 1], v[6 - i]); });
    v[0] = cadd(cadd(x0, t[0]), cadd(t[1], t[2]));
    sfor<3>([&](auto kc) {                       // X_k = a + S i b, X_{7-k} = a - S i b
      constexpr int k = decltype(kc)::value + 1;
      T a = x0, b;
      sfor<3>([&](auto ic) {
        constexpr int i = decltype(ic)::value, e = (i + 1) * k % 7;
        constexpr float ce = c[(e <= 3 ? e : 7 - e) - 1], se = e <= 3 ? s[e - 1] : -s[6 - e];
        a = cmad(a, t[i], ce);
        if constexpr (i == 0) b = cscale(d[i], se);
        else b = cmad(b, d[i], se);
      });
      v[k] = add_si<S>(a, b);
      v[7 - k] = sub_si<S>(a, b);
    });
  }
};

constexpr int first_factor(int R) {
  return (R % 4 == 0 && R != 4) ? 4
         : (R % 2 == 0 && R != 2) ? 2
         : (R % 5 == 0 && R != 5) ? 5
         : (R % 3 == 0 && R != 3) ? 3
         : (R % 7 == 0 && R != 7) ? 7
                                  : R;
}

// composite R = A * B in registers (same split as the block four-step)
template <int R, int S>
struct Dft {
  static constexpr int A = first_factor(R);
  static constexpr int B = R / A;
  static_assert(A * B == R && A > 1 && B > 1, "unsupported DFT length");
  template <class T>
  __device__ __forceinline__ static void run(T (&v)[R]) {
    T t[B][A];
    sfor<B>([&](auto bc) {
      constexpr int b = decltype(bc)::value;
      T s[A];
      sfor<A>([&](auto ac) { constexpr int a = decltype(ac)::value; s[a] = v[B * a + b]; });
      Dft<A, S>::run(s);
      sfor<A>([&](auto kc) {
        constexpr int ka = decltype(kc)::value;
        t[b][ka] = tw_mul<R, S, b * ka>(s[ka]);
      });
    });
    sfor<A>([&](auto kc) {
      constexpr int ka = decltype(kc)::value;
      T u[B];
      sfor<B>([&](auto bc) { constexpr int b = decltype(bc)::value; u[b] = t[b][ka]; });
      Dft<B, S>::run(u);
      sfor<B>([&](auto kb) { constexpr int k = decltype(kb)::value; v[ka + A * k] = u[k]; });
    });
  }
};

// R-point transform of R/2 values and R/2 zeros: two R/2-point ones,
// X[2m] = DFT(x)[m], X[2m+1] = DFT(x W_R^n)[m]
template <int R, int S, class T>
__device__ __forceinline__ void dft_half(T (&x)[R / 2], T (&v)[R]) {
  static_assert(R % 2 == 0);
  T o[R / 2];
  sfor<R / 2>([&](auto nc) { constexpr int n = decltype(nc)::value; o[n] = tw_mul<R, S, n>(x[n]); });
  Dft<R / 2, S>::run(x);
  Dft<R / 2, S>::run(o);
#pragma unroll
  for (int m = 0; m < R / 2; ++m) {
    v[2 * m] = x[m];
    v[2 * m + 1] = o[m];
  }
}

// ---------------------------------------------------------------- four-step
// N = N1 * N2 with N1 <= N2 (step 2 then has at most one item per thread).
// Split variant V = 0 is the built-in choice; V = 1, where a length has one,
// is the alternative the autotuner times against it.
template <int N, int V>
struct SplitV;
template <> struct SplitV<16, 0>  { static constexpr int N1 = 4,  N2 = 4; };
template <> struct SplitV<32, 0>  { static constexpr int N1 = 4,  N2 = 8; };
template <> struct SplitV<40, 0>  { static constexpr int N1 = 5,  N2 = 8; };
template <> struct SplitV<64, 0>  { static constexpr int N1 = 8,  N2 = 8; };
template <> struct SplitV<80, 0>  { static constexpr int N1 = 8,  N2 = 10; };
template <> struct SplitV<100, 0> { static constexpr int N1 = 10, N2 = 10; };
template <> struct SplitV<128, 0> { static constexpr int N1 = 8,  N2 = 16; };
template <> struct SplitV<160, 0> { static constexpr int N1 = 8,  N2 = 20; };
template <> struct SplitV<192, 0> { static constexpr int N1 = 12, N2 = 16; };
template <> struct SplitV<200, 0> { static constexpr int N1 = 10, N2 = 20; };
template <> struct SplitV<216, 0> { static constexpr int N1 = 12, N2 = 18; };
template <> struct SplitV<256, 0> { static constexpr int N1 = 16, N2 = 16; };
template <> struct SplitV<320, 0> { static constexpr int N1 = 16, N2 = 20; };
template <> struct SplitV<360, 0> { static constexpr int N1 = 18, N2 = 20; };
template <> struct SplitV<400, 0> { static constexpr int N1 = 16, N2 = 25; };
template <> struct SplitV<512, 0> { static constexpr int N1 = 16, N2 = 32; };
template <> struct SplitV<24, 0>  { static constexpr int N1 = 4,  N2 = 6; };
template <> struct SplitV<48, 0>  { static constexpr int N1 = 6,  N2 = 8; };
template <> struct SplitV<56, 0>  { static constexpr int N1 = 7,  N2 = 8; };
template <> struct SplitV<72, 0>  { static constexpr int N1 = 8,  N2 = 9; };
template <> struct SplitV<96, 0>  { static constexpr int N1 = 8,  N2 = 12; };
template <> struct SplitV<112, 0> { static constexpr int N1 = 8,  N2 = 14; };
template <> struct SplitV<120, 0> { static constexpr int N1 = 10, N2 = 12; };
template <> struct SplitV<144, 0> { static constexpr int N1 = 12, N2 = 12; };
template <> struct SplitV<168, 0> { static constexpr int N1 = 12, N2 = 14; };
template <> struct SplitV<180, 0> { static constexpr int N1 = 12, N2 = 15; };
template <> struct SplitV<240, 0> { static constexpr int N1 = 15, N2 = 16; };
template <> struct SplitV<280, 0> { static constexpr int N1 = 14, N2 = 20; };
template <> struct SplitV<300, 0> { static constexpr int N1 = 15, N2 = 20; };
template <> struct SplitV<64, 1>  { static constexpr int N1 = 4,  N2 = 16; };
template <> struct SplitV<80, 1>  { static constexpr int N1 = 4,  N2 = 20; };
template <> struct SplitV<128, 1> { static constexpr int N1 = 4,  N2 = 32; };
template <> struct SplitV<160, 1> { static constexpr int N1 = 10, N2 = 16; };
template <> struct SplitV<192, 1> { static constexpr int N1 = 8,  N2 = 24; };
template <> struct SplitV<200, 1> { static constexpr int N1 = 8,  N2 = 25; };
template <> struct SplitV<216, 1> { static constexpr int N1 = 8,  N2 = 27; };
template <> struct SplitV<256, 1> { static constexpr int N1 = 8,  N2 = 32; };
template <> struct SplitV<320, 1> { static constexpr int N1 = 10, N2 = 32; };
template <> struct SplitV<400, 1> { static constexpr int N1 = 20, N2 = 20; };
// lengths with a second split
constexpr bool has_alt_split(int N) {
  return N == 64 || N == 80 || N == 128 || N == 160 || N == 192 || N == 200 || N == 216 || N == 256 ||
         N == 320 || N == 400;
}
// lengths that only box transforms use (FP32, built-in split): steps of about
// 1/8 between the lengths the ABI offers.  At 150^3 the boxes need 138..164
// points, which 144, 160 and 168 cover with 0.8 of the volume 160 and 192 take.
constexpr bool box_only(int N) {
  return N == 24 || N == 48 || N == 56 || N == 72 || N == 96 || N == 112 || N == 120 || N == 144 ||
         N == 168 || N == 180 || N == 240 || N == 280 || N == 300;
}

template <int N, bool PAD_ROWS = true, int V = 0>
struct FourStep {
  static constexpr int N1 = SplitV<N, V>::N1;
  static constexpr int N2 = SplitV<N, V>::N2;
  // exchange layout per sequence: [n2][k1] with padded strides (odd strides keep
  // 16 consecutive lanes on distinct bank pairs for either lane ordering).
  // Without row padding (RS = N1) a transformed sequence is in natural order;
  // that suits callers whose lanes run over sequences (the odd CS spreads them).
  static constexpr int RS = (PAD_ROWS && N1 % 2 == 0) ? N1 + 1 : N1;
  static constexpr int CS0 = N2 * RS;
  static constexpr int CS = (CS0 % 2 == 0) ? CS0 + 1 : CS0;
  static_assert(CS >= N, "sequence stride must hold N natural-order values");

  // v holds x[N2*n1 + n2] for n1 = 0..N1-1; writes twiddled N1-point outputs
  template <int S>
  __device__ __forceinline__ static void step1(float2 (&v)[N1], float2* ex_seq, int n2,
                                               const float2* __restrict__ twN) {
    Dft<N1, S>::run(v);
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) {
      float2 w = __ldg(&twN[n2 * k1]);
      if (S > 0) w.y = -w.y;
      ex_seq[n2 * RS + k1] = (k1 == 0) ? v[k1] : cmul(v[k1], w);
    }
  }

  // u[k2] = X[k1 + N1*k2]
  template <int S>
  __device__ __forceinline__ static void step2(float2 (&u)[N2], const float2* ex_seq, int k1) {
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) u[n2] = ex_seq[n2 * RS + k1];
    Dft<N2, S>::run(u);
  }
};

}  // namespace csngf
