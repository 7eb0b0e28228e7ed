// 64-bit fixed-point transforms for the FP64 pair kernels.
//
// The FP64 pipe of GB300 gives 1.6 additions or fused multiply-adds per clock and SM, the integer
// pipe 57 64-bit additions and 5.8 64-bit high products (measured, 1024 threads): a 24-point codelet
// (252 operations, 28 of them products by constants) takes 157 clocks per thread and SM in FP64
// and about 12 in integers.  So the work volumes of the FP64 pruned kernels hold integers
// v 2^(62 - e), with one exponent e per transform and pass; the products in real space, the spectral
// multiplications and every accumulator stay in FP64, and FP32 kernels use none of this.
//
// Scaling.  An integer transform neither overflows nor loses bits when e follows from a bound: with
// |v| <= b0 for every nonzero input and sum |v| <= bt, every partial sum of the first, second and
// third pass over len values is at most b_k = min(len^k b0, bt), and every intermediate of a codelet
// is a combination of its inputs with weights of modulus at most 1, taken apart into x +- y at most
// once (a factor sqrt(2)).  With e_k = ceil(log2 b_k) the magnitudes stay below sqrt(2) 2^62 < 2^63.
// Values are converted at e_1 and shifted right, rounded, by e_2 - e_1 and e_3 - e_2 before the second
// and third pass.  Every product and shift is rounded to nearest, so that the errors of a pass add up like
// independent ones: a result is off by 1 to 26 units of 2^(e_3 - 62) in the root mean square and by up to
// 120 at the worst point, before its conversion to FP64 (boxes of 9^3 to 24^3, both directions, spectra flat
// and falling off; on the CPU against long double).  With e_3 from bounds as tight as below, that is 0.1e-16
// to 2.4e-16 of the results' root mean square and 0.7e-16 to 9e-16 at the worst point; the same codelets in
// FP64 are off by 1.6e-16 to 3.2e-16 and 6e-16 to 42e-16.  (3x3x3 apply, 24^3: 222 ms with them in integers, 499 in
// FP64 arithmetic; 2x2x2 gradient 147 and 324.)  (Values that are the same in every pencil are
// rounded the same way in every pencil: such a coefficient, where only the two ends of the spheres meet, may
// be off by N^2 / 2 units.)  Bounds come from the 2- and max norms of the real-space factors (k_norms;
// |sum a b| <= |a|_2 |b|_2) and, for spectra, from sums of upper-rounded floats over the spectrum; factors
// that barely overlap in space leave |a|_2 |b|_2, and with it the unit, far above the size of their product.
// Bounds are kept as a scaled value and an exponent until they are whole, so that they hold for values between
// 2^-950 and 2^1000: results are multiples of at least 2^-1012, and a bound beyond 2^1000 or not finite (an
// infinity or NaN among the inputs) poisons the transform, all of whose results are then NaN, as a
// floating-point transform of a volume with such a value gives.
#pragma once
#include "tc_kernels.cuh"

namespace tc {

// Element type of a work volume: fixed point for FP64 kernels.
template <typename T> struct Work { using type = cplx<T>; };
template <> struct Work<double> { using type = cplx<long long>; };
template <typename T> using WorkT = typename Work<T>::type;

// Scale of one transform (empty in FP32).
template <typename T> struct Scale {};
template <> struct Scale<double> {
  int k_in;        // inputs are converted as v 2^k_in
  int s2, s3;      // right shifts before the second and third pass
  int hi_out;      // exponent field added to results (e_3 - 62, shifted into the high word)
  int poison;      // bits set in the high word of every result: NaN when a bound is not finite
};

// Smallest e with b < 2^e (b >= 0; an infinity or NaN: 1025), clamped to where a zero is still shifted out
// (to_fx) and every result's exponent is that of a normal number (from_fx).
__device__ __forceinline__ int fx_exp(double b) {
  const int e = ((__double2hiint(b) >> 20) & 0x7ff) - 1022;
  return e < -950 ? -950 : e;
}
constexpr int ceil_log2(long long v) { return v <= 1 ? 0 : 1 + ceil_log2((v + 1) / 2); }

// Scale of a transform over LEN nonzero values per axis with |v| <= b0 and sum |v| <= bt.
template <typename T, int LEN> __device__ __forceinline__ Scale<T> fx_scale(double b0, double bt) {
  Scale<T> s;
  if constexpr (sizeof(T) == 8) {
    constexpr int l1 = ceil_log2(LEN), l2 = ceil_log2((long long)LEN * LEN), l3 = ceil_log2((long long)LEN * LEN * LEN);
    // the norms themselves are rounded: one part in 10^6 on top
    const int x0 = fx_exp(b0 * 1.000001), xt = fx_exp(bt * 1.000001);
    const int e3 = min(x0 + l3, xt), e1 = min(x0 + l1, e3), e2 = min(x0 + l2, e3);
    s.k_in = 62 - e1;
    s.s2 = e2 - e1;
    s.s3 = e3 - e2;
    s.hi_out = (e3 - 62) * (1 << 20);
    s.poison = (xt < 1000 && x0 < 1000) ? 0 : 0x7ff80000;
  }
  return s;
}

// v 2^k to the nearest integer, in integer instructions (the conversion instruction runs at the FP64
// pipe's rate).  |v| 2^k < sqrt(2) 2^62 by the bound, so the shift is not negative; a shift beyond 63
// (zero among the values) gives 0.
__device__ __forceinline__ long long to_fx(double v, int k) {
  const int hi = __double2hiint(v), lo = __double2loint(v);
  unsigned long long m = ((unsigned long long)((unsigned)(hi & 0xfffff) | 0x100000u) << 32 | (unsigned)lo) << 11;
  const int t = 1085 - k - ((hi >> 20) & 0x7ff);
  // twice the magnitude; the instruction clamps the shift
#ifdef __CUDA_ARCH__
  asm("shr.u64 %0, %1, %2;" : "=l"(m) : "l"(m), "r"(t));
#else
  m = t < 64 ? m >> t : 0;
#endif
  const long long r = (long long)((m + 1) >> 1), s = (long long)(hi >> 31);
  return (r ^ s) - s;
}
__device__ __forceinline__ cplx<long long> to_work(cplx<double> v, const Scale<double>& s) {
  return {to_fx(v.x, s.k_in), to_fx(v.y, s.k_in)};
}
__device__ __forceinline__ cplx<float> to_work(cplx<float> v, const Scale<float>&) { return v; }
// v 2^(e_3 - 62), rounded to nearest, in integer instructions
__device__ __forceinline__ double from_fx(long long v, const Scale<double>& s) {
  const long long sg = v >> 63;
  const unsigned long long a = (unsigned long long)((v ^ sg) - sg);
  const int lz = __clzll((long long)a);
  unsigned long long m = a << (lz & 63);
  m = (m >> 11) + ((m >> 10) & 1);                       // 53 bits, the leading one among them
  int hi = (int)(m >> 32) + ((1022 + 63 - lz) << 20) + s.hi_out;   // the leading one adds to the exponent
  hi = a == 0 ? 0 : hi;
  return __hiloint2double(hi | ((int)(sg) & 0x80000000) | s.poison, (int)m);
}
__device__ __forceinline__ cplx<double> from_work(cplx<long long> v, const Scale<double>& s) {
  return {from_fx(v.x, s), from_fx(v.y, s)};
}
__device__ __forceinline__ cplx<float> from_work(cplx<float> v, const Scale<float>&) { return v; }
// v / 2^s to nearest, for the values i of pencil p of a pass.  A half goes up or down by the parity of the
// bits set in p and in i: always up, shifts by one and two bits would add a quarter and an eighth of a unit to
// every value.  (To even instead: 15.5 clocks per thread and SM for a 24-point codelet, not 12.6.)
template <typename T> struct PassShift {
  __device__ __forceinline__ cplx<T> operator()(cplx<T> v, int) const { return v; }
};
template <> struct PassShift<double> {
  long long add[2];
  int s;
  __device__ __forceinline__ cplx<long long> operator()(cplx<long long> v, int i) const {
    const long long a = add[(i ^ (i >> 1) ^ (i >> 2) ^ (i >> 3) ^ (i >> 4) ^ (i >> 5)) & 1];
    return {(v.x + a) >> s, (v.y + a) >> s};
  }
};
__device__ __forceinline__ PassShift<double> pass_shift(int s, int p) {
  const long long up = (1ll << s) >> 1, down = s > 0 ? up - 1 : 0;
  return (__popc(p) & 1) ? PassShift<double>{{down, up}, s} : PassShift<double>{{up, down}, s};
}
// before the second and before the third pass
__device__ __forceinline__ PassShift<double> pass2(const Scale<double>& s, int p) { return pass_shift(s.s2, p); }
__device__ __forceinline__ PassShift<double> pass3(const Scale<double>& s, int p) { return pass_shift(s.s3, p); }
__device__ __forceinline__ PassShift<float> pass2(const Scale<float>&, int) { return {}; }
__device__ __forceinline__ PassShift<float> pass3(const Scale<float>&, int) { return {}; }

// v 2^-x from above, as a float (x: exponent of a bound on |v|, so that nothing overflows; the
// conversion rounds up, so that nothing is lost at the other end).
__device__ __forceinline__ float fx_float(double v, int x) {
  const int hi = __double2hiint(v) & 0x7fffffff;
  const int xh = x * (1 << 20), h = hi >= 0x7ff00000 ? hi : (hi > max(0, xh) || x < 0) && hi != 0 ? hi - xh : 0;
  return __double2float_ru(__hiloint2double(h, __double2loint(v)));
}
// a 2^x for |x| <= 2000, in two steps
__device__ __forceinline__ double fx_unscale(double a, int x) {
  const int h = x / 2;
  return a * __hiloint2double((h + 1023) << 20, 0) * __hiloint2double((x - h + 1023) << 20, 0);
}

// Bounds of a spectrum: the largest modulus and the sum of the moduli of the values added, in floats
// scaled by 2^-x.
struct SpecBound {
  float m = 0.f, s = 0.f;
  // |v| w, w >= 0 from above
  __device__ __forceinline__ void add(cplx<double> v, float w, int x) {
    const float a = __fmul_ru(__fadd_ru(fx_float(v.x, x), fx_float(v.y, x)), w);
    m = (a <= m) ? m : a;   // (a NaN stays in the sum)
    s = __fadd_ru(s, a);
  }
};
constexpr int kBoundBuf = 8 * 32;   // floats of shared memory for block_bounds of up to 4 bounds

// Block-wide maxima and sums, returned to every thread.
template <int NB> __device__ __forceinline__ void block_bounds(SpecBound (&b)[NB], float* buf) {
  static_assert(2 * NB * 32 <= kBoundBuf, "bound buffer");
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    for (int o = 16; o > 0; o >>= 1) {
      const float m = __shfl_xor_sync(0xffffffffu, b[i].m, o), s = __shfl_xor_sync(0xffffffffu, b[i].s, o);
      b[i].m = (m <= b[i].m) ? b[i].m : m;
      b[i].s = __fadd_ru(b[i].s, s);
    }
  }
  __syncthreads();   // buf may still be read from the previous use
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      buf[(2 * i) * 32 + wid] = b[i].m;
      buf[(2 * i + 1) * 32 + wid] = b[i].s;
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    float m = 0.f, s = 0.f;
    for (int w = 0; w < nw; ++w) {
      const float x = buf[(2 * i) * 32 + w];
      m = (x <= m) ? m : x;
      s = __fadd_ru(s, buf[(2 * i + 1) * 32 + w]);
    }
    b[i].m = m;
    b[i].s = s;
  }
}

// Scale of the inverse transform of a spectrum given by value(c), c < n, as the work volume's scale
// for LEN nonzero values per axis: the exponent of the largest component first, then the sum.
template <typename T, int LEN, typename Value>
__device__ __forceinline__ Scale<T> spectrum_scale(int n, Value value, float* buf) {
  if constexpr (sizeof(T) == 8) {
    int h = 0;
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
      const cplx<double> v = value(c);
      h = max(h, max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff));
    }
    h = __reduce_max_sync(0xffffffffu, h);
    int* ib = reinterpret_cast<int*>(buf);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0) ib[wid] = h;
    __syncthreads();
    h = 0;
    for (int w = 0; w < nw; ++w) h = max(h, ib[w]);
    const int x = (h >> 20) - 1022 + 1;   // modulus below 2^x (two components)
    SpecBound b[1];
    for (int c = threadIdx.x; c < n; c += blockDim.x) b[0].add(value(c), 1.f, x);
    block_bounds<1>(b, buf);
    return fx_scale<T, LEN>(fx_unscale(b[0].m, x), fx_unscale(b[0].s, x));
  } else {
    return Scale<T>{};
  }
}

// |u p| 2^-x from above at compact index (c1, c2, c3), u a kernel-table value, 2^x a bound on its table
struct PBound {
  float c[3], b[3][3], slop;
};
template <typename T> __device__ __forceinline__ PBound pbound_setup(const Params<T>& P, const T* dl) {
  PBound q;
  q.slop = 0.f;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    q.c[d] = (float)dl[d];
    float t = fabsf(q.c[d]);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      q.b[a][d] = (float)P.Bm[a][d];
      t += 24.f * fabsf(q.b[a][d]);
    }
    q.slop += t;
  }
  q.slop *= 1e-6f;   // float rounding of the components, against cancellation at small |p|
  return q;
}
__device__ __forceinline__ float pbound(const PBound& q, double u, int x, float m1, float m2, float m3) {
  float p2 = 0.f;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float p = q.c[d] + m1 * q.b[0][d] + m2 * q.b[1][d] + m3 * q.b[2][d];
    p2 = fmaf(p, p, p2);
  }
  return __fmul_ru(fx_float(u, x), sqrtf(p2) * 1.00001f + q.slop);
}

// 3D transforms of one volume per CTA (fwd3d, inv3d of tc_fft.cuh; same arguments) in fixed point where
// the FP64 volume is in shared memory: their latency is that of one CTA on one SM's FP64 pipe
// otherwise.  The values go into the volume first and the scale is taken from there: a load may be 25 FP64
// operations, which are done once.  buf: kBoundBuf floats.
template <typename T, int N> constexpr bool kFxVolume = sizeof(T) == 8 && (size_t)Geo<N>::vol * sizeof(cplx<T>) + 1024 <= (size_t)kSmemLimit;

template <typename T, int N, bool FWD, typename Load, typename Emit>
__device__ __forceinline__ void volume3d(cplx<T>* V, Load load, Emit emit, float* buf) {
  using G = Geo<N>;
  if constexpr (kFxVolume<T, N>) {
    using I = long long;
    constexpr int S = FWD ? -1 : +1, A1 = FWD ? 1 : 2, A3 = FWD ? 2 : 1;
    auto at = [](int c) { return G::sidx(c / (N * N), (c / N) % N, c % N); };
#pragma unroll 2
    for (int c = threadIdx.x; c < G::nn; c += blockDim.x) V[at(c)] = load(c / (N * N), (c / N) % N, c % N);
    // (each thread takes the maximum and the sum over the points that it stored itself)
    const Scale<T> sc = spectrum_scale<T, N>(G::nn, [&](int c) { return V[at(c)]; }, buf);
    cplx<I>* W = reinterpret_cast<cplx<I>*>(V);
    auto put = [&](int a, int b, int c, cplx<I> v) { W[G::sidx(a, b, c)] = v; };
    fft_pass<I, N, S, A1>([&](int a, int b, int c) { return to_work(V[G::sidx(a, b, c)], sc); }, put);
    __syncthreads();
    fft_pass<I, N, S, 3>([&](int a, int b, int c) { return pass2(sc, a * N + b)(W[G::sidx(a, b, c)], c); }, put);
    __syncthreads();
    fft_pass<I, N, S, A3>([&](int a, int b, int c) { return FWD ? pass3(sc, a * N + c)(W[G::sidx(a, b, c)], b) : pass3(sc, b * N + c)(W[G::sidx(a, b, c)], a); },
                          [&](int a, int b, int c, cplx<I> v) { emit(a, b, c, from_work(v, sc)); });
  } else if constexpr (FWD) {
    fwd3d<T, N>(V, load, emit);
  } else {
    inv3d<T, N>(V, load, emit);
  }
}

// Norms of the volumes a[v], v < count (blockIdx.x), into out: the 2-norm over the grid points and the
// largest modulus, from above (parts in 10^6).  The largest component's exponent first: the squares are of values
// scaled by it, which neither overflow nor vanish (2-norms from squares as they are: infinite from 2^512, 0
// below 2^-538).  The scaled values are floats made of the upper word, as the FP64 pipe would take 27 us for a
// 24^3 volume; the words stay in registers between the two (27 points per thread at 24^3).
template <int N> __global__ void __launch_bounds__(512) k_norms(const cplx<double>* a, const cplx<double>* b, Norm* na, Norm* nb) {
  constexpr int W = 512 / 32, M = (N * N * N + 511) / 512;
  const cplx<double>* v = (blockIdx.y == 0 ? a : b) + (size_t)blockIdx.x * N * N * N;
  __shared__ float ss[W];
  __shared__ int sh[W];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int u[2 * M], h = 0;
#pragma unroll
  for (int i = 0; i < M; ++i) {
    const int r = threadIdx.x + 512 * i;
    const cplx<double> t = r < N * N * N ? v[r] : cplx<double>{0, 0};
    u[2 * i] = __double2hiint(t.x) & 0x7fffffff;
    u[2 * i + 1] = __double2hiint(t.y) & 0x7fffffff;
  }
#pragma unroll
  for (int i = 0; i < 2 * M; ++i) h = max(h, u[i]);
  h = __reduce_max_sync(0xffffffffu, h);
  if (lane == 0) sh[wid] = h;
  __syncthreads();
  for (int w = 0; w < W; ++w) h = max(h, sh[w]);
  const int x = (h >> 20) - 1023, shift = (896 + x) * (1 << 20);   // the largest in [1, 2), exponent field 127
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < 2 * M; ++i) {
    const float f = __int_as_float(max(0, u[i] + 1 - shift) << 3);
    s = __fmaf_ru(f, f, s);
  }
  for (int o = 16; o > 0; o >>= 1) s = __fadd_ru(s, __shfl_xor_sync(0xffffffffu, s, o));
  if (lane == 0) ss[wid] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < W; ++w) s = __fadd_ru(s, ss[w]);
    const double inf = __hiloint2double(0x7ff00000, 0);   // (an infinity or NaN among the values)
    Norm n = {h < 0x7ff00000 ? fx_unscale(sqrt((double)s), x) : inf,
              h < 0x7ff00000 ? fx_unscale(1.4143 * __hiloint2double((h & 0xfffff) + 1 + 0x3ff00000, 0), x) : inf};
    (blockIdx.y == 0 ? na : nb)[blockIdx.x] = n;
  }
}

}  // namespace tc
