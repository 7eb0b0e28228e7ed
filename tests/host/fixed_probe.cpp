// Test probe: the fixed-point transforms of the FP64 pair kernels and the same codelets in FP64, against
// long double, on the CPU (tests/host/cuda stands in for the CUDA names).  Prints, per box, direction and
// input, "<dir> <N> <L> <input> <rms> <max> <unit> <fp64 rms> <fp64 max>": errors over the outputs and the
// fixed-point unit, all relative to the root mean square of the outputs (fixed point: beyond the half ulp that the
// conversion of each result to FP64 is allowed).
#include <complex>
#include <cstdio>
#include <random>
#include <vector>

#include "tc_pruned.cuh"

using namespace tc;
using cl = std::complex<long double>;
using vol = std::vector<cl>;
static const long double kTwoPi = 2.0L * 3.14159265358979323846264338327950288L;

static void twiddles() {   // as prepare_kernels uploads them
  for (int i = 0, off = 0; i < kNumTwLens; off += kTwLens[i++])
    for (int j = 0; j < kTwLens[i]; ++j) {
      const int L = kTwLens[i];
      const double a = -2.0 * 3.14159265358979323846 * j / L;
      c_tw64[2 * (off + j)] = std::cos(a);
      c_tw64[2 * (off + j) + 1] = std::sin(a);
      fx_twiddle(j, L, c_twfx + 2 * (off + j));
    }
}

static void dft3(vol& v, int n, int sign) {
  std::vector<cl> w(n), t(n);
  for (int k = 0; k < n; ++k) w[k] = std::polar(1.0L, sign * kTwoPi * k / n);
  for (int st : {n * n, n, 1})
    for (int b = 0; b < n * n * n; ++b) {
      if ((b / st) % n) continue;
      for (int k = 0; k < n; ++k) {
        t[k] = 0;
        for (int j = 0; j < n; ++j) t[k] += v[b + j * st] * w[j * k % n];
      }
      for (int k = 0; k < n; ++k) v[b + k * st] = t[k];
    }
}

static void report(const char* dir, int N, int L, const char* kind, const vol& ref, const std::vector<cplx<double>>& fx,
                   const std::vector<cplx<double>>& fp, const Scale<double>& sc) {
  long double r = 0, e[2] = {0, 0}, m[2] = {0, 0};
  for (size_t i = 0; i < ref.size(); ++i) {
    r += std::norm(ref[i]);
    for (int k = 0; k < 2; ++k) {
      const cplx<double> v = k ? fp[i] : fx[i];
      long double d = std::abs(cl(v.x, v.y) - ref[i]);
      if (k == 0) d = std::max(0.0L, d - std::abs(ref[i]) * std::ldexp(1.0L, -53));   // the conversion of the result
      e[k] += d * d;
      m[k] = std::max(m[k], d);
    }
  }
  const long double rms = std::sqrt(r / ref.size());
  std::printf("%s %d %d %s %.6Le %.6Le %.6Le %.6Le %.6Le\n", dir, N, L, kind, std::sqrt(e[0] / ref.size()) / rms, m[0] / rms,
              std::ldexp(1.0L, sc.hi_out / (1 << 20)) / rms, std::sqrt(e[1] / ref.size()) / rms, m[1] / rms);
}

template <int N, int L> static void box() {
  using S = Sup<N, L>;
  using G = Geo<N>;
  std::mt19937_64 rng(100 * N + L);
  std::normal_distribution<double> nd;
  const char* kinds[] = {"flat", "gauss", "exponential"};
  for (int kind = 0; kind < 3; ++kind) {
    auto weight = [&](double m2) { return kind == 0 ? 1.0 : kind == 1 ? std::exp(-0.2 * m2) : 0x1p-60 * std::exp(-0.5 * std::sqrt(m2)); };
    auto random_spectrum = [&](std::vector<cplx<double>>& A, vol& v) {
      A.resize(S::cvol);
      v.assign(G::nn, cl(0));
      for (int c = 0; c < S::cvol; ++c) {
        const int c1 = c / (L * L), c2 = c / L % L, c3 = c % L;
        const double a = S::mil(c1), b = S::mil(c2), d = S::mil(c3), w = weight(a * a + b * b + d * d);
        A[c] = {w * nd(rng), w * nd(rng)};
        v[gidx_c<N, L>(c1, c2, c3)] = cl(A[c].x, A[c].y);
      }
    };
    std::vector<cplx<double>> A, fx(G::nn), fp(G::nn), V(G::vol), R(G::nn);
    std::vector<cplx<long long>> B(S::bvol);
    static float buf[kBoundBuf];
    // inverse, the support's spectrum to the grid
    vol x, y;
    random_spectrum(A, x);
    Scale<double> sc = spectrum_scale<double, L>(S::cvol, [&](int c) { return A[c]; }, buf);
    pinv_23<double, N, L>(B.data(), [&](int a, int b, int c) { return A[S::cidx(a, b, c)]; }, sc);
    pass_axis1<double, N, L, true>(B.data(), [](int, int, int) { return cplx<double>{0, 0}; },
                                   [&](int i2, int i3, cplx<double>(&v)[N]) {
                                     for (int i = 0; i < N; ++i) fx[G::gidx(i, i2, i3)] = v[i];
                                   },
                                   false, sc, sc);
    inv3d<double, N>(V.data(), [&](int a, int b, int c) { const cl v = x[G::gidx(a, b, c)]; return cplx<double>{(double)v.real(), (double)v.imag()}; },
                     [&](int a, int b, int c, cplx<double> v) { fp[G::gidx(a, b, c)] = v; });
    dft3(x, N, 1);
    report("inv", N, L, kinds[kind], x, fx, fp, sc);
    // forward, a product of two such fields on the grid to the support
    random_spectrum(A, y);
    dft3(y, N, 1);
    double xi = 0, yi = 0, x2 = 0, y2 = 0;
    for (int i = 0; i < G::nn; ++i) {
      const double a = std::abs(x[i]), b = std::abs(y[i]);
      R[i] = cplx<double>{(double)(x[i] * std::conj(y[i])).real(), (double)(x[i] * std::conj(y[i])).imag()};
      xi = std::max(xi, a);
      yi = std::max(yi, b);
      x2 += a * a;
      y2 += b * b;
    }
    auto load = [&](int a, int b, int c) { return R[G::gidx(a, b, c)]; };
    sc = fx_scale<double, N>(xi * yi, std::sqrt(x2) * std::sqrt(y2));
    pass_axis1<double, N, L, false>(B.data(), load, [](int, int, cplx<double>(&)[N]) {}, true, sc, sc);
    fx.resize(S::cvol);
    fp.resize(S::cvol);
    pfwd_32<double, N, L>(B.data(), [&](int a, int b, int c, cplx<double> v) { fx[S::cidx(a, b, c)] = v; }, sc);
    std::vector<cplx<double>> F(G::nn);
    fwd3d<double, N>(V.data(), load, [&](int a, int b, int c, cplx<double> v) { F[G::gidx(a, b, c)] = v; });
    for (int i = 0; i < G::nn; ++i) x[i] = cl(R[i].x, R[i].y);
    dft3(x, N, -1);
    for (int c = 0; c < S::cvol; ++c) {
      const int g = gidx_c<N, L>(c / (L * L), c / L % L, c % L);
      fp[c] = F[g];
      x[c] = x[g];   // (g >= c: not yet overwritten)
    }
    x.resize(S::cvol);
    report("fwd", N, L, kinds[kind], x, fx, fp, sc);
  }
}

int main() {
  twiddles();
  box<24, 17>();
  box<20, 17>();
  box<18, 17>();
  box<16, 13>();
  box<16, 16>();
  box<15, 15>();
  box<12, 12>();
  box<9, 9>();
  return 0;
}
