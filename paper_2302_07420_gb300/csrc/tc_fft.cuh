// Register-resident mixed-radix DFT codelets and CTA-level 3D FFT passes.
//
// One thread transforms whole pencils held in registers; a CTA transforms a
// full n^3 volume held in shared memory, one axis per pass.  Layout of a
// shared-memory volume: element (i1, i2, i3) at (i1 * n + i2) * P + i3 with
// P = n | 1 (odd row pitch, so the row-per-thread axis-3 pass is free of bank
// conflicts).  Global fields use the unpadded layout (i1 * n + i2) * n + i3.
//
// Conventions (periodic transform of Sec. 2.2 on the grid): the forward
// transform computes sum_r f(r) e^{-2 pi i m.r/n} (SIGN = -1, unnormalised;
// callers fold the 1/N of FT into their kernel factors) and the inverse
// computes sum_m F(m) e^{+2 pi i m.r/n} (SIGN = +1).
#pragma once
#include <cuda_runtime.h>

#include <cmath>

namespace tc {

template <typename T> struct cplx { T x, y; };

template <typename T> __device__ __forceinline__ cplx<T> mk(T a, T b) { return {a, b}; }
template <typename T> __device__ __forceinline__ cplx<T> operator+(cplx<T> a, cplx<T> b) { return {a.x + b.x, a.y + b.y}; }
template <typename T> __device__ __forceinline__ cplx<T> operator-(cplx<T> a, cplx<T> b) { return {a.x - b.x, a.y - b.y}; }
template <typename T> __device__ __forceinline__ cplx<T> operator*(cplx<T> a, cplx<T> b) {
  return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <typename T> __device__ __forceinline__ cplx<T> operator*(T s, cplx<T> a) { return {s * a.x, s * a.y}; }
template <typename T> __device__ __forceinline__ cplx<T> conjg(cplx<T> a) { return {a.x, -a.y}; }
// a * (s i) for s = +-1
template <typename T, int S> __device__ __forceinline__ cplx<T> mul_si(cplx<T> a) {
  return S > 0 ? cplx<T>{-a.y, a.x} : cplx<T>{a.y, -a.x};
}
// Read-only (non-coherent) load of a complex value: lets the compiler hoist it
// above stores to other arrays.
template <typename T> __device__ __forceinline__ cplx<T> ldg(const cplx<T>* p) {
  if constexpr (sizeof(T) == 4) {
    const float2 v = __ldg(reinterpret_cast<const float2*>(p));
    return {v.x, v.y};
  } else {
    const double2 v = __ldg(reinterpret_cast<const double2*>(p));
    return {v.x, v.y};
  }
}
// a * conj(b)
template <typename T> __device__ __forceinline__ cplx<T> mulc(cplx<T> a, cplx<T> b) {
  return {a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y};
}

// ---------------------------------------------------------------------------
// Twiddle tables: exp(-2 pi i j / N), j < N, computed on the host in FP64
// (glibc sin/cos) and stored in constant memory per supported length.
constexpr int kTwLens[] = {2, 3, 4, 5, 6, 8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48};
constexpr int kNumTwLens = sizeof(kTwLens) / sizeof(int);
__host__ __device__ constexpr int tw_offset(int N) {
  int off = 0;
  for (int i = 0; i < kNumTwLens; ++i) {
    if (kTwLens[i] == N) return off;
    off += kTwLens[i];
  }
  return -1;
}
constexpr int kTwTotal = tw_offset(48) + 48;

// One copy per translation unit (internal linkage); each instantiation unit
// uploads its own copy in prepare_kernels.
static __constant__ double c_tw64[2 * kTwTotal];
static __constant__ float c_tw32[2 * kTwTotal];
static __constant__ long long c_twfx[2 * kTwTotal];   // 2^62 w as two signed digits (fx_digits), fixed-point transforms

// Products in fixed point go by signed 32-bit digits and are rounded to nearest.  A product that is cut off
// instead is half a unit low in every pencil alike, and over the following passes such errors add up at
// one point of the volume (inverse transform at 24^3, 17 nonzero values per axis falling off as
// exp(-0.2 m^2): 981 units at the worst point, 4.3e-15 of the result's root mean square, where FP64
// arithmetic is off by 7.2e-16; rounded, 69 units and 3.0e-16, in the same time: a 24-point codelet with the
// shift before it takes 12.6 clocks per thread and SM, with products cut off by __mul64hi 12.5).
struct Digits {   // x = h 2^32 + l, l in [-2^31, 2^31)
  int h, l;
};
// (h from the upper word and the lower one's top bit; from x + 2^31 the 3x3x3 FP64 apply takes 236 ms, not 225)
__host__ __device__ constexpr Digits fx_digits(long long x) {
  return {(int)(x >> 32) + (int)((unsigned)x >> 31), (int)(unsigned)x};
}
// The entry of exp(-2 pi i j / L) in c_twfx, in long double; quarter turns are never loaded.
inline void fx_twiddle(int j, int L, long long* w) {
  const long double a = -2.0L * 3.14159265358979323846264338327950288L * j / L, c[2] = {std::cos(a), std::sin(a)};
  for (int i = 0; i < 2; ++i) {
    const Digits d = fx_digits((4 * j) % L == 0 ? 0 : (long long)std::nearbyint(c[i] * 4611686018427387904.0L));
    w[i] = (long long)d.h * (1ll << 32) + (long long)(unsigned)d.l;
  }
}

template <typename T> __device__ __forceinline__ cplx<T> tw_load(int idx);
template <> __device__ __forceinline__ cplx<double> tw_load<double>(int idx) { return {c_tw64[2 * idx], c_tw64[2 * idx + 1]}; }
template <> __device__ __forceinline__ cplx<float> tw_load<float>(int idx) { return {c_tw32[2 * idx], c_tw32[2 * idx + 1]}; }

// Real factors K of the butterflies, by name: 1/2, sqrt(3)/2, sqrt(1/2), cos(2 pi/5), -cos(4 pi/5),
// sin(2 pi/5), sin(4 pi/5)/sin(2 pi/5); floating and as round(K 2^64) for the fixed-point transforms.
enum { KH, KS3, KR8, KC1, KC2, KS1, KRHO };
template <int K> __device__ __forceinline__ long long fxmul(long long x);

// v * exp(S 2 pi i e / N)
template <typename T, int N, int S> __device__ __forceinline__ cplx<T> twiddle(int e, cplx<T> v) {
  e %= N;
  if (e == 0) return v;
  if ((4 * e) % N == 0) {
    const int q = (4 * e) / N;              // quarter turns
    if (q == 2) return cplx<T>{-v.x, -v.y};
    return (q == 1) ? mul_si<T, S>(v) : mul_si<T, -S>(v);
  }
  if constexpr (T(0.5) == T(0)) {
    if ((8 * e) % N == 0) {   // odd multiples of pi / 4: sqrt(1/2) (x -+ y, y +- x) and quarter turns
      const int q = (8 * e) / N;
      const cplx<T> u = S > 0 ? cplx<T>{v.x - v.y, v.y + v.x} : cplx<T>{v.x + v.y, v.y - v.x};
      const cplx<T> r = {fxmul<KR8>(u.x), fxmul<KR8>(u.y)};
      if (q == 1) return r;
      if (q == 5) return cplx<T>{-r.x, -r.y};
      return (q == 3) ? mul_si<T, S>(r) : mul_si<T, -S>(r);
    }
    const int i = tw_offset(N) + e;
    const long long pr = c_twfx[2 * i], pi = c_twfx[2 * i + 1];
    const Digits x = fx_digits(v.x), y = fx_digits(v.y), wr = {(int)(pr >> 32), (int)pr};
    const Digits wi = {S > 0 ? -(int)(pi >> 32) : (int)(pi >> 32), S > 0 ? -(int)pi : (int)pi};
    // |v| <= 2^62 and |w| = 1: the sums of middle products stay below 2^63
    auto mul = [](int a, int b) { return (long long)a * b; };
    constexpr long long half = 1ll << 29;
    const long long mr = half + (mul(x.l, wr.h) + mul(x.h, wr.l)) - (mul(y.l, wi.h) + mul(y.h, wi.l)) +
                         ((mul(x.l, wr.l) - mul(y.l, wi.l)) >> 32);
    const long long mi = half + (mul(x.l, wi.h) + mul(x.h, wi.l)) + (mul(y.l, wr.h) + mul(y.h, wr.l)) +
                         ((mul(x.l, wi.l) + mul(y.l, wr.l)) >> 32);
    return {4 * (mul(x.h, wr.h) - mul(y.h, wi.h)) + (mr >> 30), 4 * (mul(x.h, wi.h) + mul(y.h, wr.h)) + (mi >> 30)};
  } else {
    cplx<T> w = tw_load<T>(tw_offset(N) + e);   // exp(-2 pi i e/N)
    if (S > 0) w.y = -w.y;
    return v * w;
  }
}

// ---------------------------------------------------------------------------
// Codelets.  Every transform takes the set IN of its nonzero inputs (bit i: input i) at compile
// time: the pruned passes feed 17 of 24 (or 13 of 16, ...) values, and IEEE arithmetic keeps
// x + 0, so a zero that the code does not name costs its additions.  Outputs that nobody reads
// fall to dead-code elimination.
//
// What bounds them: in FP64 the FP64 pipe (1.6 operations per clock and SM), in FP32 the issue
// slots of the kernels around them.  Measured on one GB300 (3x3x3 FP64 apply / 4x4x4 FP32 apply of
// the silicon-like cell, 24^3): mixed radix 4 x 3 x 2 with twiddles, zeros unnamed, scalar FP32:
// 607 / 143.9 ms; as below 501 / 128.1 ms; as below with scalar FP32: - / 136 ms.
using InSet = unsigned long long;
template <int N> __host__ __device__ constexpr InSet all_in() { return (N >= 64 ? ~0ull : (1ull << N) - 1ull); }

// FP32 sums of complex values as one packed instruction for both halves (add / fma .f32x2): the
// lanes do no more per clock (127 against 124 additions per clock and SM measured), but half the
// instructions are issued
__device__ __forceinline__ cplx<float> operator+(cplx<float> a, cplx<float> b) {
  const float2 r = __fadd2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y));
  return {r.x, r.y};
}
__device__ __forceinline__ cplx<float> operator-(cplx<float> a, cplx<float> b) {
  const float2 r = __ffma2_rn(make_float2(b.x, b.y), make_float2(-1.f, -1.f), make_float2(a.x, a.y));
  return {r.x, r.y};
}
// Transforms run in float, double or in 64-bit fixed point (T = long long, told by T(0.5) == 0; its
// scaling is in tc_fixed.cuh).
__host__ __device__ constexpr double kval(int k) {
  constexpr double v[] = {0.5,
                          0.86602540378443864676372317075294,
                          0.70710678118654752440084436210485,
                          0.30901699437494742410229341718282,
                          0.80901699437494742410229341718282,
                          0.95105651629515357211643933337938,
                          0.61803398874989484820458683436564};
  return v[k];
}
__host__ __device__ constexpr unsigned long long kfix(int k) {
  constexpr unsigned long long v[] = {0x8000000000000000ull, 0xddb3d742c265539eull, 0xb504f333f9de6484ull,
                                      0x4f1bbcdcbfa53e0bull, 0xcf1bbcdcbfa53e0bull, 0xf378709a22a7faf3ull,
                                      0x9e3779b97f4a7c16ull};
  return v[k];
}
// x K in fixed point, to nearest; a K above 1/2 as K - 1, plus x.  K = 1/2: a half goes up or down by bit 32
// of x.  Else by digits: the product of the low ones, below a quarter of a unit and of either sign, is left out.
template <int K> __device__ __forceinline__ long long fxmul(long long x) {
  if constexpr (K == KH) {
    return (x >> 1) + ((int)(unsigned)x & (int)(x >> 32) & 1);
  } else {
    constexpr Digits k = fx_digits((long long)kfix(K));
    const Digits d = fx_digits(x);
    const long long m = (long long)d.l * k.h + 0x80000000ll + (long long)d.h * k.l;   // |x| <= sqrt(2) 2^62: < 2^63
    const long long r = (long long)d.h * k.h + (m >> 32);
    return (kfix(K) >> 63) ? r + x : r;
  }
}
// s K b
template <int K, int SG, typename T> __device__ __forceinline__ cplx<T> scalek(cplx<T> b) {
  if constexpr (sizeof(cplx<T>) == 16 && T(0.5) == T(0)) {
    const cplx<T> m = {fxmul<K>(b.x), fxmul<K>(b.y)};
    return SG > 0 ? m : cplx<T>{-m.x, -m.y};
  } else {
    constexpr T s = T(SG * kval(K));
    return {s * b.x, s * b.y};
  }
}
// a + s K b
template <int K, int SG, typename T> __device__ __forceinline__ cplx<T> axpy(cplx<T> b, cplx<T> a) {
  if constexpr (sizeof(T) == 4) {
    constexpr float s = float(SG * kval(K));
    const float2 r = __ffma2_rn(make_float2(b.x, b.y), make_float2(s, s), make_float2(a.x, a.y));
    return {r.x, r.y};
  } else if constexpr (T(0.5) == T(0)) {
    const cplx<T> m = {fxmul<K>(b.x), fxmul<K>(b.y)};
    return SG > 0 ? cplx<T>{a.x + m.x, a.y + m.y} : cplx<T>{a.x - m.x, a.y - m.y};
  } else {
    constexpr T s = T(SG * kval(K));
    return {fma(s, b.x, a.x), fma(s, b.y, a.y)};
  }
}
// a + s K i b
template <int K, int SG, typename T> __device__ __forceinline__ cplx<T> axpy_i(cplx<T> b, cplx<T> a) {
  if constexpr (T(0.5) == T(0)) {
    const cplx<T> m = {fxmul<K>(b.x), fxmul<K>(b.y)};
    return SG > 0 ? cplx<T>{a.x - m.y, a.y + m.x} : cplx<T>{a.x + m.y, a.y - m.x};
  } else {
    constexpr T s = T(SG * kval(K));
    return {fma(-s, b.y, a.x), fma(s, b.x, a.y)};
  }
}
// p = a + K b, m = a - K b (one product in fixed point)
template <int K, typename T> __device__ __forceinline__ void both(cplx<T> b, cplx<T> a, cplx<T>& p, cplx<T>& m) {
  if constexpr (T(0.5) == T(0)) {
    const cplx<T> t = {fxmul<K>(b.x), fxmul<K>(b.y)};
    p = {a.x + t.x, a.y + t.y};
    m = {a.x - t.x, a.y - t.y};
  } else {
    p = axpy<K, 1>(b, a);
    m = axpy<K, -1>(b, a);
  }
}
// p = a + S K i b, m = a - S K i b
template <int K, int S, typename T> __device__ __forceinline__ void rot2(cplx<T> b, cplx<T> a, cplx<T>& p, cplx<T>& m) {
  if constexpr (T(0.5) == T(0)) {
    const cplx<T> t = {fxmul<K>(b.x), fxmul<K>(b.y)};
    const cplx<T> u = {a.x - t.y, a.y + t.x}, v = {a.x + t.y, a.y - t.x};
    p = S > 0 ? u : v;
    m = S > 0 ? v : u;
  } else {
    p = axpy_i<K, S>(b, a);
    m = axpy_i<K, -S>(b, a);
  }
}
// sum and difference of values that may be known zeros
template <bool ZA, bool ZB, typename T> __device__ __forceinline__ cplx<T> addz(cplx<T> a, cplx<T> b) {
  if constexpr (ZA && ZB) return a + b;
  else if constexpr (ZA) return a;
  else if constexpr (ZB) return b;
  else return cplx<T>{0, 0};
}
template <bool ZA, bool ZB, typename T> __device__ __forceinline__ cplx<T> subz(cplx<T> a, cplx<T> b) {
  if constexpr (ZA && ZB) return a - b;
  else if constexpr (ZA) return a;
  else if constexpr (ZB) return cplx<T>{-b.x, -b.y};
  else return cplx<T>{0, 0};
}

// Small butterflies (in place, natural order), exponent sign S, nonzero inputs IN.  The rotations
// by i and by the real factors of the radix-3, -5 and -8 butterflies are folded into the closing
// additions as fused multiply-adds: 12, 32 and 52 operations for 3, 5 and 8 points.
template <typename T, int R, int S> struct Small;

template <typename T, int S> struct Small<T, 2, S> {
  template <InSet IN> static __device__ __forceinline__ void run(cplx<T>* z) {
    constexpr bool A = IN & 1, B = IN & 2;
    const cplx<T> a = z[0], b = z[1];
    z[0] = addz<A, B>(a, b);
    z[1] = subz<A, B>(a, b);
  }
};

template <typename T, int S> struct Small<T, 3, S> {
  template <InSet IN> static __device__ __forceinline__ void run(cplx<T>* z) {
    constexpr bool A = IN & 1, B = IN & 2, C = IN & 4;
    const cplx<T> a = z[0];
    if constexpr (!B && !C) {
      z[1] = a;
      z[2] = a;
    } else {
      const cplx<T> t1 = addz<B, C>(z[1], z[2]), t2 = subz<B, C>(z[1], z[2]);
      cplx<T> m;
      if constexpr (A) m = axpy<KH, -1>(t1, a);
      else m = scalek<KH, -1>(t1);
      z[0] = addz<A, true>(a, t1);
      rot2<KS3, S>(t2, m, z[1], z[2]);
    }
  }
};

template <typename T, int S> struct Small<T, 4, S> {
  template <InSet IN> static __device__ __forceinline__ void run(cplx<T>* z) {
    constexpr bool A = IN & 1, B = IN & 2, C = IN & 4, D = IN & 8, E = A || C, O = B || D;
    const cplx<T> a = addz<A, C>(z[0], z[2]), b = subz<A, C>(z[0], z[2]), c = addz<B, D>(z[1], z[3]),
                  d = mul_si<T, S>(subz<B, D>(z[1], z[3]));
    z[0] = addz<E, O>(a, c);
    z[2] = subz<E, O>(a, c);
    if constexpr (E && O) {   // the rotated difference by halves: no pair to pack
      z[1] = cplx<T>{b.x + d.x, b.y + d.y};
      z[3] = cplx<T>{b.x - d.x, b.y - d.y};
    } else {
      z[1] = addz<E, O>(b, d);
      z[3] = subz<E, O>(b, d);
    }
  }
};

template <typename T, int S> struct Small<T, 5, S> {
  template <InSet IN> static __device__ __forceinline__ void run(cplx<T>* z) {
    constexpr bool A = IN & 1, B1 = IN & 2, B2 = IN & 4, B3 = IN & 8, B4 = IN & 16, P = B1 || B4, Q = B2 || B3;
    const cplx<T> x0 = A ? z[0] : cplx<T>{0, 0};
    if constexpr (!P && !Q) {
      z[1] = z[2] = z[3] = z[4] = x0;
    } else {
      const cplx<T> t1 = addz<B1, B4>(z[1], z[4]), t2 = addz<B2, B3>(z[2], z[3]), t3 = subz<B1, B4>(z[1], z[4]),
                    t4 = subz<B2, B3>(z[2], z[3]);
      cplx<T> a1 = x0, a2 = x0, b1, b2;
      if constexpr (P) {
        a1 = axpy<KC1, 1>(t1, a1);
        a2 = axpy<KC2, -1>(t1, a2);
      }
      if constexpr (Q) {
        a1 = axpy<KC2, -1>(t2, a1);
        a2 = axpy<KC1, 1>(t2, a2);
      }
      // sin parts over sin(2 pi/5): t3 + r t4 and r t3 - t4
      if constexpr (P && Q) {
        b1 = axpy<KRHO, 1>(t4, t3);
        b2 = axpy<KRHO, 1>(t3, cplx<T>{-t4.x, -t4.y});
      } else if constexpr (P) {
        b1 = t3;
        b2 = scalek<KRHO, 1>(t3);
      } else {
        b1 = scalek<KRHO, 1>(t4);
        b2 = cplx<T>{-t4.x, -t4.y};
      }
      z[0] = addz<A, true>(x0, addz<P, Q>(t1, t2));
      rot2<KS1, S>(b1, a1, z[1], z[4]);
      rot2<KS1, S>(b2, a2, z[2], z[3]);
    }
  }
};

template <typename T, int S> struct Small<T, 8, S> {
  template <InSet IN> static __device__ __forceinline__ void run(cplx<T>* z) {
    constexpr InSet EV = (IN & 1) | ((IN >> 1) & 2) | ((IN >> 2) & 4) | ((IN >> 3) & 8);
    constexpr InSet OD = ((IN >> 1) & 1) | ((IN >> 2) & 2) | ((IN >> 3) & 4) | ((IN >> 4) & 8);
    cplx<T> e[4] = {z[0], z[2], z[4], z[6]}, o[4] = {z[1], z[3], z[5], z[7]};
    if constexpr (EV != 0) Small<T, 4, S>::template run<EV>(e);
    else e[0] = e[1] = e[2] = e[3] = cplx<T>{0, 0};
    if constexpr (OD == 0) {
#pragma unroll
      for (int k = 0; k < 4; ++k) z[k] = z[k + 4] = e[k];
    } else {
      Small<T, 4, S>::template run<OD>(o);
      constexpr bool E = EV != 0;
      z[0] = addz<E, true>(e[0], o[0]);
      z[4] = subz<E, true>(e[0], o[0]);
      const cplx<T> q = mul_si<T, S>(o[2]);
      z[2] = cplx<T>{e[2].x + q.x, e[2].y + q.y};
      z[6] = cplx<T>{e[2].x - q.x, e[2].y - q.y};
      // exp(S i pi/4) o = r u1 and exp(S 3 i pi/4) o = -r u3
      const cplx<T> u1 = S > 0 ? cplx<T>{o[1].x - o[1].y, o[1].y + o[1].x} : cplx<T>{o[1].x + o[1].y, o[1].y - o[1].x};
      const cplx<T> u3 = S > 0 ? cplx<T>{o[3].x + o[3].y, o[3].y - o[3].x} : cplx<T>{o[3].x - o[3].y, o[3].y + o[3].x};
      both<KR8>(u1, e[1], z[1], z[5]);
      both<KR8>(u3, e[3], z[7], z[3]);
    }
  }
};

// Split N = P Q of the codelet for N points.  Coprime factors (the power of 2, of 3 or of 5 taken
// out first) need no twiddles (Good-Thomas); prime powers beyond the butterflies split by radix 4,
// 3 or 5 with twiddles.  24 points cost 252 operations this way (3 x 52 + 8 x 12) against 332 for
// the mixed-radix decimation 4 x 3 x 2 with twiddles.
__host__ __device__ constexpr bool small_radix(int n) { return n == 2 || n == 3 || n == 4 || n == 5 || n == 8; }
__host__ __device__ constexpr int coprime_part(int n) {
  int p = 1;
  for (int f : {2, 3, 5}) {
    int q = 1, m = n;
    for (; m % f == 0; m /= f) q *= f;
    if (q > 1 && q < n) {
      p = q;
      break;
    }
  }
  return p;   // 1: n is a prime power
}
__host__ __device__ constexpr int pick_radix(int n) { return n % 4 == 0 ? 4 : (n % 3 == 0 ? 3 : (n % 5 == 0 ? 5 : 2)); }
__host__ __device__ constexpr int inv_mod(int a, int m) {
  for (int i = 1; i < m; ++i)
    if ((a * i) % m == 1) return i;
  return 1;   // m = 1
}

template <typename T, int N, int S> struct Codelet {
  template <InSet IN = all_in<N>()> static __device__ __forceinline__ void run(cplx<T>* x) {
    if constexpr (small_radix(N)) {
      Small<T, N, S>::template run<IN>(x);
    } else if constexpr (coprime_part(N) > 1) {
      // x[(Q a + P b) mod N], transformed over b (Q points) for each a, then over a (P points);
      // output (a', b') is X[(Q qi a' + P pi b') mod N] with Q qi = 1 mod P, P pi = 1 mod Q
      constexpr int P = coprime_part(N), Q = N / P;
      cplx<T> y[N];
      outer<P, Q, IN, 0>(x, y);
      inner<P, Q, IN, 0>(y, x);
    } else {
      // decimation in time: X[k + M s] = sum_r W_R^{rs} (W_N^{rk} Y_r[k]), Y_r = DFT_M of x[r::R]
      constexpr int R = pick_radix(N), M = N / R;
      cplx<T> y[N];
      split<R, M, IN, 0>(x, y);
#pragma unroll
      for (int k = 0; k < M; ++k) {
        cplx<T> z[R];
#pragma unroll
        for (int r = 0; r < R; ++r) z[r] = twiddle<T, N, S>(r * k, y[r * M + k]);
        Small<T, R, S>::template run<some<R, M, R, 1, IN>()>(z);
#pragma unroll
        for (int s = 0; s < R; ++s) x[k + M * s] = z[s];
      }
    }
  }

 private:
  // nonzero set of the sub-transform over m < M of x[(off + m step) mod N]
  template <int M, int step, int off, InSet IN> static constexpr InSet sub_in() {
    InSet s = 0;
    for (int m = 0; m < M; ++m)
      if ((IN >> ((off + m * step) % N)) & 1) s |= 1ull << m;
    return s;
  }
  // set of the a < A whose sub-transform (M points, step, offset a off) has any nonzero input
  template <int A, int M, int step, int off, InSet IN> static constexpr InSet some() {
    InSet s = 0;
    for (int a = 0; a < A; ++a)
      for (int m = 0; m < M; ++m)
        if ((IN >> ((a * off + m * step) % N)) & 1) s |= 1ull << a;
    return s;
  }
  template <int P, int Q, InSet IN, int A> static __device__ __forceinline__ void outer(const cplx<T>* x, cplx<T>* y) {
    if constexpr (A < P) {
      constexpr InSet in = sub_in<Q, P, Q * A, IN>();
      cplx<T> t[Q];
#pragma unroll
      for (int b = 0; b < Q; ++b) t[b] = (in >> b) & 1 ? x[(Q * A + P * b) % N] : cplx<T>{0, 0};
      if constexpr (in != 0) Codelet<T, Q, S>::template run<in>(t);
#pragma unroll
      for (int b = 0; b < Q; ++b) y[A * Q + b] = t[b];
      outer<P, Q, IN, A + 1>(x, y);
    }
  }
  template <int P, int Q, InSet IN, int B> static __device__ __forceinline__ void inner(const cplx<T>* y, cplx<T>* x) {
    if constexpr (B < Q) {
      constexpr InSet in = some<P, Q, P, Q, IN>();
      cplx<T> t[P];
#pragma unroll
      for (int a = 0; a < P; ++a) t[a] = y[a * Q + B];
      Codelet<T, P, S>::template run<in>(t);
#pragma unroll
      for (int a = 0; a < P; ++a) x[(Q * inv_mod(Q, P) * a + P * inv_mod(P, Q) * B) % N] = t[a];
      inner<P, Q, IN, B + 1>(y, x);
    }
  }
  template <int R, int M, InSet IN, int A> static __device__ __forceinline__ void split(const cplx<T>* x, cplx<T>* y) {
    if constexpr (A < R) {
      constexpr InSet in = sub_in<M, R, A, IN>();
      cplx<T> t[M];
#pragma unroll
      for (int m = 0; m < M; ++m) t[m] = (in >> m) & 1 ? x[m * R + A] : cplx<T>{0, 0};
      if constexpr (in != 0) Codelet<T, M, S>::template run<in>(t);
#pragma unroll
      for (int m = 0; m < M; ++m) y[A * M + m] = t[m];
      split<R, M, IN, A + 1>(x, y);
    }
  }
};

// ---------------------------------------------------------------------------
// CTA-level passes over an n^3 volume.  Pencil index p enumerates the n^2
// pencils of the pass; each thread takes p = tid, tid + blockDim.x, ...
//
//   axis 1: pencil (i2, i3), elements i1 = 0..n-1
//   axis 2: pencil (i1, i3), elements i2
//   axis 3: pencil (i1, i2), elements i3
//
// load(i1, i2, i3) -> cplx<T>;  store(i1, i2, i3, value).  Both are called
// with the element's coordinates; the pass performs the 1D DFT in between.
template <int N> struct Geo {
  static constexpr int n = N;
  static constexpr int P = N | 1;                 // shared-memory row pitch
  static constexpr int vol = N * N * P;           // shared-memory complex elements
  static constexpr int nn = N * N * N;            // global (unpadded) elements
  static __device__ __forceinline__ int sidx(int i1, int i2, int i3) { return (i1 * N + i2) * P + i3; }
  static __device__ __forceinline__ int gidx(int i1, int i2, int i3) { return (i1 * N + i2) * N + i3; }
};

template <typename T, int N, int S, int AXIS, typename Load, typename Store>
__device__ __forceinline__ void fft_pass(Load load, Store store) {
  for (int p = threadIdx.x; p < N * N; p += blockDim.x) {
    const int a = p / N, b = p % N;
    cplx<T> v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      if (AXIS == 1) v[i] = load(i, a, b);
      else if (AXIS == 2) v[i] = load(a, i, b);
      else v[i] = load(a, b, i);
    }
    Codelet<T, N, S>::run(v);
#pragma unroll
    for (int i = 0; i < N; ++i) {
      if (AXIS == 1) store(i, a, b, v[i]);
      else if (AXIS == 2) store(a, i, b, v[i]);
      else store(a, b, i, v[i]);
    }
  }
}

// Full 3D transforms through a shared-memory work volume W.  Global memory is
// touched only in axis-1 and axis-2 passes, whose pencils put consecutive
// threads on consecutive i3 (coalesced); the axis-3 pass stays in shared memory.
//   forward  (SIGN -1): axes 1, 3, 2   load = real-space input, emit = spectrum
//   inverse  (SIGN +1): axes 2, 3, 1   load = spectrum,         emit = real-space output
// The caller synchronises after emit when it reuses W.
template <typename T, int N, typename Load, typename Emit>
__device__ __forceinline__ void fwd3d(cplx<T>* W, Load load, Emit emit) {
  using G = Geo<N>;
  fft_pass<T, N, -1, 1>(load, [&](int a, int b, int c, cplx<T> v) { W[G::sidx(a, b, c)] = v; });
  __syncthreads();
  fft_pass<T, N, -1, 3>([&](int a, int b, int c) { return W[G::sidx(a, b, c)]; },
                        [&](int a, int b, int c, cplx<T> v) { W[G::sidx(a, b, c)] = v; });
  __syncthreads();
  fft_pass<T, N, -1, 2>([&](int a, int b, int c) { return W[G::sidx(a, b, c)]; }, emit);
}

template <typename T, int N, typename Load, typename Emit>
__device__ __forceinline__ void inv3d(cplx<T>* W, Load load, Emit emit) {
  using G = Geo<N>;
  fft_pass<T, N, +1, 2>(load, [&](int a, int b, int c, cplx<T> v) { W[G::sidx(a, b, c)] = v; });
  __syncthreads();
  fft_pass<T, N, +1, 3>([&](int a, int b, int c) { return W[G::sidx(a, b, c)]; },
                        [&](int a, int b, int c, cplx<T> v) { W[G::sidx(a, b, c)] = v; });
  __syncthreads();
  fft_pass<T, N, +1, 1>([&](int a, int b, int c) { return W[G::sidx(a, b, c)]; }, emit);
}

// A pass whose store needs per-element data from global memory: after the
// transform of a pencil, pre(i1, i2, i3) is evaluated for a chunk of CH
// elements before store(i1, i2, i3, v, pre_value) runs on any of them, so the
// loads of a chunk are in flight together (each store through a generic
// pointer would otherwise hold back every later load).
template <typename T, int N, int S, int AXIS, int CH, typename Load, typename Pre, typename Store>
__device__ __forceinline__ void fft_pass_pre(Load load, Pre pre, Store store) {
  for (int p = threadIdx.x; p < N * N; p += blockDim.x) {
    const int a = p / N, b = p % N;
    cplx<T> v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      if (AXIS == 1) v[i] = load(i, a, b);
      else if (AXIS == 2) v[i] = load(a, i, b);
      else v[i] = load(a, b, i);
    }
    Codelet<T, N, S>::run(v);
#pragma unroll
    for (int c0 = 0; c0 < N; c0 += CH) {
      decltype(pre(0, 0, 0)) o[CH];
#pragma unroll
      for (int u = 0; u < CH; ++u) {
        const int i = c0 + u;
        if (i >= N) continue;
        if (AXIS == 1) o[u] = pre(i, a, b);
        else if (AXIS == 2) o[u] = pre(a, i, b);
        else o[u] = pre(a, b, i);
      }
#pragma unroll
      for (int u = 0; u < CH; ++u) {
        const int i = c0 + u;
        if (i >= N) continue;
        if (AXIS == 1) store(i, a, b, v[i], o[u]);
        else if (AXIS == 2) store(a, i, b, v[i], o[u]);
        else store(a, b, i, v[i], o[u]);
      }
    }
  }
}

// Forward transform whose emit needs per-element global data (see fft_pass_pre).
template <typename T, int N, int CH, typename Load, typename Pre, typename Emit>
__device__ __forceinline__ void fwd3d_pre(cplx<T>* W, Load load, Pre pre, Emit emit) {
  using G = Geo<N>;
  fft_pass<T, N, -1, 1>(load, [&](int a, int b, int c, cplx<T> v) { W[G::sidx(a, b, c)] = v; });
  __syncthreads();
  fft_pass<T, N, -1, 3>([&](int a, int b, int c) { return W[G::sidx(a, b, c)]; },
                        [&](int a, int b, int c, cplx<T> v) { W[G::sidx(a, b, c)] = v; });
  __syncthreads();
  fft_pass_pre<T, N, -1, 2, CH>([&](int a, int b, int c) { return W[G::sidx(a, b, c)]; }, pre, emit);
}

// Last (axis-1) pass of an inverse transform that feeds a read-modify-write of
// global arrays.  Per pencil and chunk of CH elements, pre(i1, i2, i3) loads
// every old value first and post(i1, i2, i3, v, old) then computes and stores,
// so the loads of a chunk are in flight together instead of one at a time.
template <typename T, int N, int CH, typename Pre, typename Post>
__device__ __forceinline__ void inv_axis1_rmw(cplx<T>* W, Pre pre, Post post) {
  using G = Geo<N>;
  for (int p = threadIdx.x; p < N * N; p += blockDim.x) {
    const int a = p / N, b = p % N;
    cplx<T> v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = W[G::sidx(i, a, b)];
    Codelet<T, N, +1>::run(v);
#pragma unroll
    for (int c0 = 0; c0 < N; c0 += CH) {
      decltype(pre(0, 0, 0)) o[CH];
#pragma unroll
      for (int u = 0; u < CH; ++u)
        if (c0 + u < N) o[u] = pre(c0 + u, a, b);
#pragma unroll
      for (int u = 0; u < CH; ++u)
        if (c0 + u < N) post(c0 + u, a, b, v[c0 + u], o[u]);
    }
  }
}

template <typename T, int N, int CH, typename Load, typename Pre, typename Post>
__device__ __forceinline__ void inv3d_rmw(cplx<T>* W, Load load, Pre pre, Post post) {
  using G = Geo<N>;
  fft_pass<T, N, +1, 2>(load, [&](int a, int b, int c, cplx<T> v) { W[G::sidx(a, b, c)] = v; });
  __syncthreads();
  fft_pass<T, N, +1, 3>([&](int a, int b, int c) { return W[G::sidx(a, b, c)]; },
                        [&](int a, int b, int c, cplx<T> v) { W[G::sidx(a, b, c)] = v; });
  __syncthreads();
  inv_axis1_rmw<T, N, CH>(W, pre, post);
}

// Pass on a pencil without a transform (pointwise work in the same thread mapping).
template <typename T, int N, int AXIS, typename Body>
__device__ __forceinline__ void pointwise_pass(Body body) {
  for (int p = threadIdx.x; p < N * N; p += blockDim.x) {
    const int a = p / N, b = p % N;
#pragma unroll 4
    for (int i = 0; i < N; ++i) {
      if (AXIS == 1) body(i, a, b);
      else if (AXIS == 2) body(a, i, b);
      else body(a, b, i);
    }
  }
}

}  // namespace tc
