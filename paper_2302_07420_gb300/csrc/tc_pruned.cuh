// Pair chains with pruned transforms (templated on precision T, box size N and support length L).
//
// Every transform of a pair chain has its spectrum on the support of the pair densities: the
// forward transform of a pair density chi_q^* phi_j has nonzero coefficients only at m_j - m_q
// (sphere Miller vectors, cyclic on the box), and every spectral accumulator of the chain is
// consumed only through ket_q FT^{-1}[.], whose projection onto the sphere of k_j reads it at those
// same indices.  When the Miller span s of all spheres satisfies 2 s + 1 <= L, the support per axis
// lies in the L box indices {0 .. (L-1)/2} U {N - (L-1)/2 .. N-1}, so
//   * an inverse transform reads L^3 spectral values: the axis-2 pass runs over L^2 pencils with
//     L nonzero inputs each, the axis-3 pass over L N pencils with L nonzero inputs, and only the
//     axis-1 pass produces the full N^3 real-space values;
//   * a forward transform keeps L outputs per pencil in the same passes in reverse order;
//   * the pair spectrum A and the spectral accumulator C are stored compactly ([L]^3), next to the
//     work volume [L][N][N|1] (first index: compact axis-1 index) in shared memory.
// This is exact for the discrete operator (the dropped coefficients are zero there).  Compact
// index c maps to box index box(c) = c for c < (L+1)/2 and c + N - L otherwise; L = N means no
// pruning (box(c) = c).
#pragma once
#include "tc_kernels_impl.cuh"
#include "tc_fixed.cuh"

namespace tc {

template <int N, int L> struct Sup {
  static_assert(L <= N, "support longer than the box");
  static constexpr int H = (L == N) ? N : (L + 1) / 2;
  static constexpr int P = N | 1;              // row pitch of the work volume
  static constexpr int bvol = L * N * P;       // work volume [L][N][P]
  static constexpr int cvol = L * L * L;       // compact spectrum [L][L][L]
  static __host__ __device__ constexpr int box(int c) { return c < H ? c : c + N - L; }
  // Miller integer of compact index c
  static __host__ __device__ constexpr int mil(int c) {
    return (L == N) ? (c <= (N - 1) / 2 ? c : c - N) : (c < H ? c : c - L);
  }
  // box indices on the support (the nonzero inputs of an inverse pencil)
  static __host__ __device__ constexpr InSet on() {
    InSet m = 0;
    for (int c = 0; c < L; ++c) m |= 1ull << box(c);
    return m;
  }
  // compact index of the negated Miller integer (L < N: the support is symmetric and clear of the
  // Nyquist index, so -m is again on the support)
  static __host__ __device__ constexpr int refl(int c) { return c == 0 ? 0 : L - c; }
  static __device__ __forceinline__ int bidx(int c1, int i2, int i3) { return (c1 * N + i2) * P + i3; }
  static __device__ __forceinline__ int cidx(int c1, int c2, int c3) { return (c1 * L + c2) * L + c3; }
};

// Support length of the pruned kernels compiled for box size N (N: not compiled pruned): 17 at 24^3
// (the silicon-like 4x4x4 cell's spheres) and the supports 4 floor((N-1)/4) + 1 of the batched HEG
// cells' spheres at 16^3, 18^3 and 20^3.
template <int N> constexpr int kPruneL = (N == 16) ? 13 : (N == 18 || N == 20 || N == 24) ? 17 : N;

// Small boxes whose pair densities do not fit that support run these kernels on the full support
// (L = N): their volumes and spectra fit one CTA's shared memory in FP64 too, and FP64 takes the
// fixed-point transforms (14-electron gas, FP64 16^3: pair kernels of the full transforms 1.9 ms).
template <int N> constexpr bool kFullPr = N <= 16;

// Threads per CTA of the pruned kernels: one axis-1 pencil per thread, in FP64 at most 384 threads (a
// pencil of N double-complex values takes 4 N registers; 12 warps leave 168 each, as 9 would).
template <typename T, int N> struct PrCfg {
  static constexpr int one = ((N * N + 31) / 32) * 32;
  static constexpr int threads = sizeof(T) == 8 && one > 384 ? 384 : one;
  // CTAs per SM that the registers are cut for: two of a small FP32 box (16 warps of 128 registers)
  static constexpr int minb = sizeof(T) == 4 && N <= 16 ? 2 : 1;
};

// Shared-memory plan: work volume B first; the compact spectra A and C and the three kernel tables
// of the current Delta (U_pp, U_ap, V on the support) follow when they fit, else A and C live in a
// per-CTA slice of the global scratch and the tables are read from the full-box tables.
template <typename T, int N, int L, int NSPEC, int NTAB> struct PrSmem {
  using S = Sup<N, L>;
  static constexpr size_t bB = (size_t)S::bvol * sizeof(cplx<T>);
  static constexpr size_t bC = (size_t)S::cvol * sizeof(cplx<T>);
  static constexpr size_t bT = (size_t)S::cvol * sizeof(T);
  static constexpr size_t lim = (size_t)kSmemLimit - 1024;
  static constexpr bool spec = bB + NSPEC * bC <= lim;
  // (tables only where the CTAs per SM that the launch bounds ask for still fit: 233,472 bytes per SM,
  // 1 KB of them per CTA reserved; two 16^3 CTAs without tables beat one with, see PrCfg)
  static constexpr bool tab = spec && bB + NSPEC * bC + NTAB * bT <= lim &&
                              PrCfg<T, N>::minb * (bB + NSPEC * bC + NTAB * bT + 2048) <= 233472;
  static constexpr size_t bytes = bB + (spec ? NSPEC * bC : 0) + (tab ? NTAB * bT : 0);
};

// *p += v in L2 without a return value; FP32 complex as one vector reduction.
__device__ __forceinline__ void red_add_v(cplx<float>* p, cplx<float> v) {
  asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void red_add_v(cplx<double>* p, cplx<double> v) {
  atomicAdd(&p->x, v.x);
  atomicAdd(&p->y, v.y);
}

// Load from L2, where red_add_v adds.
__device__ __forceinline__ cplx<float> ld_l2(const cplx<float>* p) {
  const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
  return {v.x, v.y};
}
__device__ __forceinline__ cplx<double> ld_l2(const cplx<double>* p) {
  const double2 v = __ldcg(reinterpret_cast<const double2*>(p));
  return {v.x, v.y};
}

// Inverse transform, axes 2 and 3, of a compact spectrum spec(c1, c2, c3) into the work volume.
template <typename T, int N, int L, typename Spec>
__device__ __forceinline__ void pinv_23(WorkT<T>* B, Spec spec, const Scale<T>& sc) {
  using W = WorkT<T>;
  using CT = decltype(W().x);
  using S = Sup<N, L>;
  for (int p = threadIdx.x; p < L * L; p += blockDim.x) {
    const int c1 = p / L, c3 = p % L;
    W v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = W{0, 0};
#pragma unroll
    for (int c2 = 0; c2 < L; ++c2) v[S::box(c2)] = to_work(spec(c1, c2, c3), sc);
    Codelet<CT, N, +1>::template run<S::on()>(v);
#pragma unroll
    for (int i2 = 0; i2 < N; ++i2) B[S::bidx(c1, i2, c3)] = v[i2];
  }
  __syncthreads();
  for (int p = threadIdx.x; p < L * N; p += blockDim.x) {
    const int c1 = p / N, i2 = p % N;
    const auto shift = pass2(sc, p);
    W v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = W{0, 0};
#pragma unroll
    for (int c3 = 0; c3 < L; ++c3) v[S::box(c3)] = shift(B[S::bidx(c1, i2, c3)], c3);
    Codelet<CT, N, +1>::template run<S::on()>(v);
#pragma unroll
    for (int i3 = 0; i3 < N; ++i3) B[S::bidx(c1, i2, i3)] = v[i3];
  }
  __syncthreads();
}

// Axis-1 pass over the N^2 pencils (i2, i3).  FROM_B: the pencil's L spectral values are read from
// the work volume and inverse-transformed (else load(i1, i2, i3) supplies N real-space values);
// body(i2, i3, v) then works on the N real-space values; with fwd the pencil is forward-transformed
// and its L support values are written back into the work volume.  si, sf: the scales of the inverse
// and of the forward transform.
template <typename T, int N, int L, bool FROM_B, typename Load, typename Body>
__device__ __forceinline__ void pass_axis1(WorkT<T>* B, Load load, Body body, bool fwd, const Scale<T>& si,
                                           const Scale<T>& sf) {
  using S = Sup<N, L>;
  using W = WorkT<T>;
  using CT = decltype(W().x);
  for (int p = threadIdx.x; p < N * N; p += blockDim.x) {
    const int i2 = p / N, i3 = p % N;
    cplx<T> v[N];
    if constexpr (FROM_B) {
      const auto shift = pass3(si, p);
      W u[N];
#pragma unroll
      for (int i = 0; i < N; ++i) u[i] = W{0, 0};
#pragma unroll
      for (int c1 = 0; c1 < L; ++c1) u[S::box(c1)] = shift(B[S::bidx(c1, i2, i3)], c1);
      Codelet<CT, N, +1>::template run<S::on()>(u);
#pragma unroll
      for (int i = 0; i < N; ++i) v[i] = from_work(u[i], si);
    } else {
#pragma unroll
      for (int i = 0; i < N; ++i) v[i] = load(i, i2, i3);
    }
    body(i2, i3, v);
    if (fwd) {
      W u[N];
#pragma unroll
      for (int i = 0; i < N; ++i) u[i] = to_work(v[i], sf);
      Codelet<CT, N, -1>::run(u);
#pragma unroll
      for (int c1 = 0; c1 < L; ++c1) B[S::bidx(c1, i2, i3)] = u[S::box(c1)];
    }
  }
  __syncthreads();
}

// Forward transform, axes 3 and 2, of the work volume (axis 1 done, L x N x N values) onto the
// support; emit(c1, c2, c3, value) receives each of the L^3 outputs once, from the thread that owns
// the compact pencil (c1, c3) -- the same thread that reads it in pinv_23.
template <typename T, int N, int L, typename Emit>
__device__ __forceinline__ void pfwd_32(WorkT<T>* B, Emit emit, const Scale<T>& sc) {
  using S = Sup<N, L>;
  using W = WorkT<T>;
  using CT = decltype(W().x);
  for (int p = threadIdx.x; p < L * N; p += blockDim.x) {
    const int c1 = p / N, i2 = p % N;
    const auto shift = pass2(sc, p);
    W v[N];
#pragma unroll
    for (int i3 = 0; i3 < N; ++i3) v[i3] = shift(B[S::bidx(c1, i2, i3)], i3);
    Codelet<CT, N, -1>::run(v);
#pragma unroll
    for (int c3 = 0; c3 < L; ++c3) B[S::bidx(c1, i2, c3)] = v[S::box(c3)];
  }
  __syncthreads();
  for (int p = threadIdx.x; p < L * L; p += blockDim.x) {
    const int c1 = p / L, c3 = p % L;
    const auto shift = pass3(sc, p);
    W v[N];
#pragma unroll
    for (int i2 = 0; i2 < N; ++i2) v[i2] = shift(B[S::bidx(c1, i2, c3)], i2);
    Codelet<CT, N, -1>::run(v);
#pragma unroll
    for (int c2 = 0; c2 < L; ++c2) emit(c1, c2, c3, from_work(v[S::box(c2)], sc));
  }
  __syncthreads();
}

// p_d = Delta_d + G_d at compact index (c1, c2, c3)
template <typename T, int N, int L>
__device__ __forceinline__ T pcomp_c(const PComp<T>& q, int c1, int c2, int c3) {
  using S = Sup<N, L>;
  // c2 runs along a pencil: its term last, the rest once per pencil
  return (q.c0 + (T)S::mil(c1) * q.b1 + (T)S::mil(c3) * q.b3) + (T)S::mil(c2) * q.b2;
}

template <int N, int L> __device__ __forceinline__ int gidx_c(int c1, int c2, int c3) {
  using S = Sup<N, L>;
  return (S::box(c1) * N + S::box(c2)) * N + S::box(c3);
}

// Whether every term group of the pair chains' parallel-spin pass is on (the kernels' ALL).
template <typename T> inline bool all_terms(const Params<T>& P) {
  const T* t = P.tw;
  return (t[T3A3] != T(0) || t[T3B4] != T(0)) && (t[T2BX1] != T(0) || t[T3A4] != T(0)) &&
         (t[T3B3] != T(0) || t[T2BX2] != T(0)) && t[T3B5] != T(0) && t[T3B6] != T(0);
}

// Fused pair chains, pruned (same work, grid and accumulators as k_pair_chain):
//   A  = FT[conj(bra_q) ket_j]                                          on the support
//   for d: b = FT^{-1}[U^pp_d A];  acc += f Z(q)_d b;  w_d += f ket_q b   (2bx1, 3a4, 3a3's w_j)
//          F = conj(bra_q) Y(j)_d - tw3b5 ket_j h3b(q)_d + tw3b6 n b;  C += -U^pp_d FT[F]
//   for d: b = FT^{-1}[U^ap_d A];  C += -U^ap_d FT[tw3b6 n b]             (3b6, antiparallel)
//   acc += ket_q FT^{-1}[f (C - tw2ax V A)]                               (3b3, 2bx2, 3b5, 3b6, 2ax)
// (Algs. 2, 5, 6, 9, 11, 12 and the 2bx terms of Sec. 2.6.3.)  Z comes with f, Y and n over tw3b5, which
// C takes back: 22 operations per grid point and component instead of 28.
//
// What bounds it.  FP64: no single pipe; the products of the parallel-spin pass keep the FP64 pipe busy half
// of the time (the transforms run in integers, tc_fixed.cuh), and the warps wait for instructions (unrolled
// pencils of 64-bit code), for that pipe's results and at barriers: 3x3x3 apply, 24^3, 270.6 -> 129 ms.  FP32: the
// latency of that pass's loads, seven per grid point (one point ahead, 18 warps): 4x4x4 88.4 -> 71 ms.
//
// Mirrored two-sided launches (P.mirror; Eq. BITCSCFconj).  The left pair density of (output q,
// partner j) is conj(phi_j^* chi_q) -- the complex conjugate of the right pair density of (output j,
// partner q) -- and the left side's kernel momentum is -(k_j - k_q + G), so on a support symmetric
// under G -> -G its compact spectrum is A_L(c) = conj(A_R(refl c)).  With u~ real and even,
// U_d(-p) = conj(U_d(p)), so FT^{-1}[U^ap_d A_L] = conj(FT^{-1}[U^ap_d A_R]); the left density is
// conj of the right one, so the antiparallel 3b6 spectrum is C_ap,L(c) = conj(C_ap,R(refl c)) too.
// mirror = 1 (right launch): a CTA whose output j is itself a partner (band < no) stores both
// reflections for the left pair (q, j), the antiparallel one summed over d as it is emitted;
// mirror = 2 (left launch, after it): such a pair loads them as its A and initial C and skips its
// own pair-density transform and antiparallel loop (7 of its 14 transforms).  Left outputs whose
// right counterpart was skipped for a zero occupation compute their own.  The parallel-spin loop
// and the final transform stay per side: their partner fields (Y, Z, h3b, V) have no such
// relation.  Built for FP64; in FP32 the parallel-spin
// passes' loads dominate and the mirror code is compiled out.
// ALL: every term group of the parallel-spin pass is on (all_terms): the pass then has no tests, and the
// kernel not the other form of it beside it, which alone costs 7 % (4x4x4 FP32: 71.6 against 76.8 ms,
// by the registers and the order of the loads that the compiler gives the pass).  FP32 only: FP64, bound
// by its products, gains nothing and keeps both forms in one kernel (ALL = false).
template <typename T, int N, int L, bool ALL>
__global__ void __launch_bounds__(PrCfg<T, N>::threads, PrCfg<T, N>::minb) k_pair_chain_pr(Params<T> P) {
  using G = Geo<N>;
  using S = Sup<N, L>;
  using SM = PrSmem<T, N, L, 2, 3>;
  // what the pointwise pass reads per grid point; in FP32 the next point's loads are issued before this
  // one's work (4x4x4 chains: 71.6 ms; without the explicit next point 77.8 to 86.2 by the compiler's
  // order, 81.4 with the terms tested per point; FP64 has no registers for it)
  struct Elem { cplx<T> z, k, y, b, j, h, n; };
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ T red[32];
  __shared__ float bbuf[sizeof(T) == 8 ? kBoundBuf : 1];   // bounds of the fixed-point transforms
  constexpr bool FX = sizeof(T) == 8;
  const SideArgs<T>& SD = P.side[P.side0 + blockIdx.y];
  const int jitem = blockIdx.x / P.sc, chunk = blockIdx.x % P.sc;
  const int jo = out_item(P, jitem), j = P.j0 + jo, kj = j / P.nb;
  const int M = P.Nk * P.no, nj = P.nj_out;
  // mirrored launches (FP64 only: the FP32 kernel is bound by the loads of its parallel-spin
  // passes, which both sides keep, and gains nothing from them): output j as a partner index; write
  // (right) or read (left) the reflections
  constexpr bool MIR = sizeof(T) == 8;
  const int jocc = kj * P.no + j % P.nb;
  const bool mw = MIR && P.mirror == 1 && j % P.nb < P.no;
  // (the right CTA of output q skipped its pair with j when f_j, in the compute precision, was 0)
  const bool mr = MIR && P.mirror == 2 && j % P.nb < P.no && weight(P, j) != T(0);
  const int qi_begin = (int)((long long)chunk * M / P.sc), qi_end = (int)((long long)(chunk + 1) * M / P.sc);
  WorkT<T>* B = reinterpret_cast<WorkT<T>*>(smraw);
  cplx<T>* A;
  if constexpr (SM::spec) {
    A = reinterpret_cast<cplx<T>*>(B + S::bvol);
  } else {
    const size_t cta = (size_t)blockIdx.y * gridDim.x + blockIdx.x;
    A = P.scratch + cta * 2 * (size_t)S::cvol;
  }
  cplx<T>* C = A + S::cvol;
  T* tU = SM::tab ? reinterpret_cast<T*>(reinterpret_cast<unsigned char*>(smraw) + SM::bB + 2 * SM::bC) : nullptr;
  const size_t NN = G::nn;
  const cplx<T>* ketj = SD.ket + (size_t)j * NN;
  const cplx<T>* Yj = SD.Y + (size_t)jo * 3 * NN;
  cplx<T>* acc = SD.acc + ((size_t)chunk * nj + jo) * NN;
  cplx<T>* w = SD.w + ((size_t)chunk * nj + jo) * 3 * NN;
  const T* tw = P.tw;
  const bool need_w = ALL || tw[T3A3] != T(0) || tw[T3B4] != T(0);
  const bool need_z = ALL || tw[T2BX1] != T(0) || tw[T3A4] != T(0);
  const bool need_y = ALL || tw[T3B3] != T(0) || tw[T2BX2] != T(0);
  const bool need_pp = need_w || need_z || tw[T3B6] != T(0);
  const bool need_F = need_y || tw[T3B5] != T(0) || tw[T3B6] != T(0);
  const bool need_ap = tw[T3B6] != T(0) && !P.no_ap;
  const T t3b5 = tw[T3B5], t3b6 = tw[T3B6], t2ax = tw[T2AX];
  const bool all = need_z && need_w && need_y && t3b5 != T(0) && t3b6 != T(0);
  const T g35 = t3b5 != T(0) ? t3b5 : T(1);   // Y and tn are held over g35 (k_prep_zy, k_vloc), C takes it back
  for (int r = threadIdx.x; r < (int)NN; r += blockDim.x) {
    acc[r] = cplx<T>{0, 0};
    for (int d = 0; d < 3; ++d) w[d * NN + r] = cplx<T>{0, 0};
  }
  int staged = -1;   // Delta whose kernel tables are in shared memory
  for (int qi = qi_begin; qi < qi_end; ++qi) {
    const int kq = qi / P.no, mu = qi % P.no;
    const int q = kq * P.nb + mu;
    const T f = weight(P, q);
    if (f == T(0)) continue;
    const T ft2ax = f * t2ax;
    const int did = P.delta_id[kj * P.kstride + kq];
    const T* dl = P.delta + did * 3;
    const T* Vt = SD.tabV + ((size_t)did * 2 + SD.side) * NN;
    const T* Upp = P.tabU + ((size_t)did * 2 + 0) * NN;
    const T* Uap = P.tabU + ((size_t)did * 2 + 1) * NN;
    if constexpr (SM::tab) {
      if (did != staged) {
        // the previous pair's last reads of the tables ended before its closing barrier
        for (int c = threadIdx.x; c < S::cvol; c += blockDim.x) {
          const int g = gidx_c<N, L>(c / (L * L), (c / L) % L, c % L);
          tU[c] = Upp[g];
          tU[S::cvol + c] = Uap[g];
          tU[2 * S::cvol + c] = Vt[g];
        }
        staged = did;   // first read after the barriers of the forward transform below
      }
    }
    auto tab = [&](int which, int c1, int c2, int c3) -> T {
      if constexpr (SM::tab) {
        return tU[which * S::cvol + S::cidx(c1, c2, c3)];
      } else {
        const T* t = which == 0 ? Upp : (which == 1 ? Uap : Vt);
        return __ldg(t + gidx_c<N, L>(c1, c2, c3));   // read-only: not held back by the stores of C
      }
    };
    const cplx<T>* braq = SD.bra + (size_t)q * NN;
    const cplx<T>* ketq = SD.ket + (size_t)q * NN;
    const cplx<T>* Zq = SD.Z + ((size_t)(kq * P.no + mu) * 3) * NN;
    const cplx<T>* h3bq = SD.h3b + ((size_t)(kq * P.no + mu) * 3) * NN;
    // the reflections of this pair: [A][C_ap] of the left pair (q, j) (write) or of this one (read)
    cplx<T>* MA = (mw || mr) ? P.mir + ((size_t)(mw ? qi : jocc) * M + (mw ? jocc : qi)) * 2 * S::cvol : nullptr;
    // scales of the fixed-point transforms: the pair density, then per spin channel the bounds of
    // u_s |p| A (sb) and the inverse transforms' scales
    Scale<T> s_rho, s_inv[2];
    SpecBound sb[2];
    double b_inf[2] = {0, 0}, b_two[2] = {0, 0};   // max norm and 2-norm of FT^{-1}[U_d A] on the grid
    PBound pb;
    int xa = 0;   // |A| < 2^xa; the bounds of u_s |p| A are in units of 2^(xa + P.u_exp[s])
    if constexpr (FX) {
      const double two = SD.nket[j].two * SD.nbra[q].two;
      s_rho = fx_scale<T, N>(SD.nket[j].inf * SD.nbra[q].inf, two);
      xa = fx_exp(two * (double)P.invN * 1.000001) + 1;
      pb = pbound_setup<T>(P, dl);
    }
    auto bound_A = [&](int c1, int c2, int c3, cplx<T> a) {
      if constexpr (FX) {
        const int g = gidx_c<N, L>(c1, c2, c3);
        const float m1 = S::mil(c1), m2 = S::mil(c2), m3 = S::mil(c3);
        sb[0].add(a, pbound(pb, __ldg(Upp + g), P.u_exp[0], m1, m2, m3), xa);
        if (need_ap) sb[1].add(a, pbound(pb, __ldg(Uap + g), P.u_exp[1], m1, m2, m3), xa);
      }
    };
    if (mr) {
      for (int c = threadIdx.x; c < S::cvol; c += blockDim.x) {
        A[c] = MA[c];
        bound_A(c / (L * L), (c / L) % L, c % L, A[c]);
        C[c] = need_ap ? MA[S::cvol + c] : cplx<T>{0, 0};
      }
      __syncthreads();
    } else {
      // A = FT[conj(bra_q) ket_j] on the support
      pass_axis1<T, N, L, false>(
          B, [&](int a, int b, int c) { const int g = G::gidx(a, b, c); return mulc(ldg(ketj + g), ldg(braq + g)); },
          [&](int, int, cplx<T>(&)[N]) {}, true, s_rho, s_rho);
      pfwd_32<T, N, L>(B, [&](int c1, int c2, int c3, cplx<T> v) {
        const cplx<T> a = P.invN * v;
        A[S::cidx(c1, c2, c3)] = a;
        bound_A(c1, c2, c3, a);
        if (mw) MA[S::cidx(S::refl(c1), S::refl(c2), S::refl(c3))] = conjg(a);
      }, s_rho);
    }
    if constexpr (FX) {
      block_bounds<2>(sb, bbuf);
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const double m = sb[s].m, t = sb[s].s;
        const int xb = xa + P.u_exp[s];
        b_inf[s] = fx_unscale(t, xb);
        b_two[s] = fx_unscale(sqrt((double)G::nn * m * t), xb);   // N sum |x|^2 <= N max|x| sum|x|
        s_inv[s] = fx_scale<T, L>(fx_unscale(m, xb), b_inf[s]);
      }
    }
    if (P.div && kq == kj && t3b6 != T(0)) {
      // O_qj = A(0) and X_s = sum_{G != 0} u~_s(G) A(G) n~(-G) for the 3b6 corrections
      for (int s = 0; s < 2; ++s) {
        T xr = 0, xi = 0;
        for (int c = threadIdx.x; c < S::cvol; c += blockDim.x) {
          const int c1 = c / (L * L), c2 = (c / L) % L, c3 = c % L;
          const int a = S::box(c1), b = S::box(c2), e = S::box(c3);
          const int gn = G::gidx((N - a) % N, (N - b) % N, (N - e) % N);
          const cplx<T> t = P.hartUs[(size_t)s * NN + G::gidx(a, b, e)] * (A[c] * SD.nt[gn]);
          xr += t.x;
          xi += t.y;
        }
        const T sr = block_sum<T>(xr, red);
        const T si = block_sum<T>(xi, red);
        if (threadIdx.x == 0) {
          double* cs = SD.cs + ((size_t)jo * P.no + mu) * 6;
          cs[2 + 2 * s] = sr;
          cs[3 + 2 * s] = si;
          if (s == 0) { cs[0] = A[0].x; cs[1] = A[0].y; }
        }
      }
      __syncthreads();
    }
    // spin channels: parallel then antiparallel (a reading mirrored CTA has the antiparallel
    // spectrum in C already; a writing one also sums it, reflected, into the left pair's slot)
    for (int sp = 0; sp < 2; ++sp) {
      if (sp == 0 && !(need_pp || need_F)) continue;
      if (sp == 1 && (!need_ap || mr)) continue;
      for (int d = 0; d < 3; ++d) {
        const bool first_C = sp == 0 && d == 0 && !mr;
        const PComp<T> qd = pcomp_setup<T>(P, dl, d);
        // b = FT^{-1}[U_d A]
        const PComp<T> qf = scaled(qd, g35 * P.invN);
        pinv_23<T, N, L>(B, [&](int c1, int c2, int c3) {
          return mul_si<T, 1>((pcomp_c<T, N, L>(qd, c1, c2, c3) * tab(sp, c1, c2, c3)) * A[S::cidx(c1, c2, c3)]);
        }, s_inv[sp]);
        Scale<T> s_F;
        if constexpr (FX) {
          // F from the norms of its factors
          const Norm nn = *SD.nn;
          double f0 = nn.inf * b_inf[sp], ft = nn.two * b_two[sp];
          if (sp == 0) {
            const Norm nY = SD.nY[jo * 3 + d], nh = SD.nh3b[(kq * P.no + mu) * 3 + d], nk = SD.nket[j], nbq = SD.nbra[q];
            if (need_y) {
              f0 += nbq.inf * nY.inf;
              ft += nbq.two * nY.two;
            }
            if (t3b5 != T(0)) {
              f0 += nk.inf * nh.inf;
              ft += nk.two * nh.two;
            }
          }
          s_F = fx_scale<T, N>(f0, ft);
        }
        const bool fwd = sp == 1 || need_F;
        pass_axis1<T, N, L, true>(
            B, [&](int, int, int) { return cplx<T>{0, 0}; },
            [&](int i2, int i3, cplx<T>(&v)[N]) {
              if (sp == 0) {
                if (ALL || (FX && all)) {
                  auto load = [&](int i) {
                    const int g = G::gidx(i, i2, i3);
                    return Elem{ldg(Zq + d * NN + g),  ldg(ketq + g), ldg(Yj + d * NN + g), ldg(braq + g),
                                ldg(ketj + g), ldg(h3bq + d * NN + g), ldg(SD.tn + g)};
                  };
                  Elem cur{};
                  if (!FX) cur = load(0);
#pragma unroll
                  for (int i = 0; i < N; ++i) {
                    Elem nxt{};
                    if (FX) cur = load(i);
                    else if (i + 1 < N) nxt = load(i + 1);
                    const int g = G::gidx(i, i2, i3);
                    const cplx<T> bv = v[i];
                    red_add_v(&acc[g], cur.z * bv);
                    red_add_v(&w[d * NN + g], f * (cur.k * bv));
                    v[i] = cur.n * bv + mulc(cur.y, cur.b) - cur.j * cur.h;   // F / g35
                    if (!FX) cur = nxt;
                  }
                } else {   // some of the terms are off
#pragma unroll
                  for (int i = 0; i < N; ++i) {
                    const int g = G::gidx(i, i2, i3);
                    const cplx<T> bv = v[i];
                    if (need_z) red_add_v(&acc[g], ldg(Zq + d * NN + g) * bv);
                    if (need_w) red_add_v(&w[d * NN + g], f * (ldg(ketq + g) * bv));
                    cplx<T> F = {0, 0};
                    if (t3b6 != T(0)) F = ldg(SD.tn + g) * bv;
                    if (need_y) F = F + mulc(ldg(Yj + d * NN + g), ldg(braq + g));
                    if (t3b5 != T(0)) F = F - ldg(ketj + g) * ldg(h3bq + d * NN + g);
                    v[i] = F;
                  }
                }
              } else {
#pragma unroll
                for (int i = 0; i < N; ++i) v[i] = ldg(SD.tn + G::gidx(i, i2, i3)) * v[i];
              }
            },
            fwd, s_inv[sp], s_F);
        if (!fwd) continue;
        // C += -U_d FT[F] = -i p_d u FT[F]
        pfwd_32<T, N, L>(B, [&](int c1, int c2, int c3, cplx<T> v) {
          const T k = pcomp_c<T, N, L>(qf, c1, c2, c3) * tab(sp, c1, c2, c3);
          const int s = S::cidx(c1, c2, c3);
          const cplx<T> c0 = first_C ? cplx<T>{0, 0} : C[s];
          C[s] = cplx<T>{fma(k, v.y, c0.x), fma(-k, v.x, c0.y)};   // C -= i k v
          if (sp == 1 && mw) {
            const cplx<T> t = mul_si<T, -1>(k * v);
            // the thread that emits an index emits it for every d
            cplx<T>* mc = MA + S::cvol + S::cidx(S::refl(c1), S::refl(c2), S::refl(c3));
            *mc = d == 0 ? conjg(t) : *mc + conjg(t);
          }
        }, s_F);
      }
    }
    const bool has_C = need_F || need_ap;
    if (has_C || t2ax != T(0)) {
      // f (C - V A): in fixed point summed into C first, for its bounds
      auto total = [&](int c1, int c2, int c3) {
        const int s = S::cidx(c1, c2, c3);
        cplx<T> v = has_C ? f * C[s] : cplx<T>{0, 0};
        if (t2ax != T(0)) v = v - (ft2ax * tab(2, c1, c2, c3)) * A[s];
        return v;
      };
      if constexpr (FX) {
#pragma unroll 4
        for (int c = threadIdx.x; c < S::cvol; c += blockDim.x) C[c] = total(c / (L * L), (c / L) % L, c % L);
      }
      const Scale<T> s_C = spectrum_scale<T, L>(S::cvol, [&](int c) { return C[c]; }, bbuf);
      pinv_23<T, N, L>(
          B,
          [&](int c1, int c2, int c3) {
            if constexpr (FX) return C[S::cidx(c1, c2, c3)];
            else return total(c1, c2, c3);
          },
          s_C);
      pass_axis1<T, N, L, true>(
          B, [&](int, int, int) { return cplx<T>{0, 0}; },
          [&](int i2, int i3, cplx<T>(&v)[N]) {
#pragma unroll
            for (int c0 = 0; c0 < N; c0 += 4) {
              cplx<T> lk[4];
#pragma unroll
              for (int u = 0; u < 4; ++u)
                if (c0 + u < N) lk[u] = ldg(ketq + G::gidx(c0 + u, i2, i3));
#pragma unroll
              for (int u = 0; u < 4; ++u)
                if (c0 + u < N) red_add_v(&acc[G::gidx(c0 + u, i2, i3)], lk[u] * v[c0 + u]);
            }
          },
          false, s_C, s_C);
    }
  }
}

// Pass 2 for 3b4 (Alg. 10), pruned: acc += tw3b4 f ket_q FT^{-1}[-U^pp . FT[-conj(bra_q) w_j]]
// (same grid and accumulators as k_pair_3b4).
template <typename T, int N, int L>
__global__ void __launch_bounds__(PrCfg<T, N>::threads, PrCfg<T, N>::minb) k_pair_3b4_pr(Params<T> P) {
  using G = Geo<N>;
  using S = Sup<N, L>;
  using SM = PrSmem<T, N, L, 1, 1>;
  extern __shared__ __align__(16) unsigned char smraw[];
  const SideArgs<T>& SD = P.side[blockIdx.y];
  __shared__ float bbuf[sizeof(T) == 8 ? kBoundBuf : 1];
  const int jitem = blockIdx.x / P.sc, chunk = blockIdx.x % P.sc;
  const int jo = out_item(P, jitem), j = P.j0 + jo, kj = j / P.nb;
  const int M = P.Nk * P.no, nj = P.nj_out;
  const int qi_begin = (int)((long long)chunk * M / P.sc), qi_end = (int)((long long)(chunk + 1) * M / P.sc);
  WorkT<T>* B = reinterpret_cast<WorkT<T>*>(smraw);
  cplx<T>* A;
  if constexpr (SM::spec) {
    A = reinterpret_cast<cplx<T>*>(B + S::bvol);
  } else {
    const size_t cta = (size_t)blockIdx.y * gridDim.x + blockIdx.x;
    A = P.scratch + cta * (size_t)S::cvol;
  }
  T* tU = SM::tab ? reinterpret_cast<T*>(reinterpret_cast<unsigned char*>(smraw) + SM::bB + SM::bC) : nullptr;
  const size_t NN = G::nn;
  cplx<T>* acc = SD.acc + ((size_t)chunk * nj + jo) * NN;
  const cplx<T>* w = SD.w + (size_t)jo * 3 * NN;
  const T t3b4 = P.tw[T3B4];
  if (t3b4 == T(0)) return;
  if (chunk > 0) {
    for (int r = threadIdx.x; r < (int)NN; r += blockDim.x) acc[r] = cplx<T>{0, 0};
    __syncthreads();
  }
  int staged = -1;
  for (int qi = qi_begin; qi < qi_end; ++qi) {
    const int kq = qi / P.no, mu = qi % P.no;
    const int q = kq * P.nb + mu;
    const T f = weight(P, q);
    if (f == T(0)) continue;
    const int did = P.delta_id[kj * P.kstride + kq];
    const T* dl = P.delta + did * 3;
    const T* Upp = P.tabU + ((size_t)did * 2 + 0) * NN;
    if constexpr (SM::tab) {
      if (did != staged) {
        for (int c = threadIdx.x; c < S::cvol; c += blockDim.x)
          tU[c] = Upp[gidx_c<N, L>(c / (L * L), (c / L) % L, c % L)];
        staged = did;
      }
    }
    auto tab = [&](int c1, int c2, int c3) -> T {
      if constexpr (SM::tab) return tU[S::cidx(c1, c2, c3)];
      else return __ldg(Upp + gidx_c<N, L>(c1, c2, c3));
    };
    const cplx<T>* braq = SD.bra + (size_t)q * NN;
    const cplx<T>* ketq = SD.ket + (size_t)q * NN;
    const T fw = t3b4 * f;
    for (int d = 0; d < 3; ++d) {
      const PComp<T> qd = scaled(pcomp_setup<T>(P, dl, d), fw * P.invN);
      Scale<T> s_w;
      if constexpr (sizeof(T) == 8) {
        const Norm nw = SD.nw[jo * 3 + d], nbq = SD.nbra[q];
        s_w = fx_scale<T, N>(nw.inf * nbq.inf, nw.two * nbq.two);
      }
      pass_axis1<T, N, L, false>(
          B, [&](int a, int b, int c) { const int g = G::gidx(a, b, c); return mulc(ldg(w + d * NN + g), ldg(braq + g)); },
          [&](int, int, cplx<T>(&)[N]) {}, true, s_w, s_w);
      // -U_d FT[-conj(bra_q) w_d] = +i p_d u FT[conj(bra_q) w_d]
      pfwd_32<T, N, L>(B, [&](int c1, int c2, int c3, cplx<T> v) {
        const T k = pcomp_c<T, N, L>(qd, c1, c2, c3) * tab(c1, c2, c3);
        const int s = S::cidx(c1, c2, c3);
        const cplx<T> a0 = d == 0 ? cplx<T>{0, 0} : A[s];
        A[s] = cplx<T>{fma(-k, v.y, a0.x), fma(k, v.x, a0.y)};   // A += i k v
      }, s_w);
    }
    const Scale<T> s_A = spectrum_scale<T, L>(S::cvol, [&](int c) { return A[c]; }, bbuf);
    pinv_23<T, N, L>(B, [&](int c1, int c2, int c3) { return A[S::cidx(c1, c2, c3)]; }, s_A);
    pass_axis1<T, N, L, true>(
        B, [&](int, int, int) { return cplx<T>{0, 0}; },
        [&](int i2, int i3, cplx<T>(&v)[N]) {
#pragma unroll
          for (int c0 = 0; c0 < N; c0 += 4) {
            cplx<T> lk[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (c0 + u < N) lk[u] = ldg(ketq + G::gidx(c0 + u, i2, i3));
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (c0 + u < N) red_add_v(&acc[G::gidx(c0 + u, i2, i3)], lk[u] * v[c0 + u]);
          }
        },
        false, s_A, s_A);
  }
}

// Occupied-pair stage, pruned (same grid, outputs and per-CTA h6 part as k_occ_pairs; Algs. 4, 6, 8,
// 11 and the 3a2 corrections of Eqs. divcor_3a2_first/second in the general-overlap form):
//   A1 = FT[conj(bra_q2) ket_q1], A2 = FT[conj(bra_q1) ket_q2]                      on the support
//   B1 = P^s_d(q2, q1) = FT^{-1}[U^s_d(k1 - k2 + G) A1]   (real space, in shared memory)
//   B2 = P^s_d(q1, q2) = FT^{-1}[U^s_d(k2 - k1 + G) A2]   (its last pass fused with the products)
//   h6 += w f1 f2 B1 . B2;  h3a4(q2)_d += f1 B2 ket_q1;  h3b(q2)_d += f1 B1 conj(bra_q1)   (s = pp)
// Shared memory (FP32): B1 as a real-space volume [N][N][N|1] (rows c1 < L serve as its inverse work
// area), then the work volume of B2 [L][N][N|1].  FP64, where both do not fit: one work volume for
// both, B1 in the CTA's L2-resident scratch slice (slot 3, written and read once by the same thread; the
// other way round, the work volume of B2 in L2, costs three passes over it: 73.7 ms against 64.2 of a
// 3x3x3 apply).  The compact spectra A1, A2 and the 3a2 spectrum F_ab live in the CTA's scratch slice
// (slots 0, 1, 2; slot 4 is the h6 part that k_reduce_a4 sums, as for k_occ_pairs).
template <typename T, int N, int L> struct OccSmem {
  using S = Sup<N, L>;
  static constexpr size_t bR = (size_t)Geo<N>::vol * sizeof(cplx<T>);
  static constexpr size_t bW = (size_t)S::bvol * sizeof(cplx<T>);
  static constexpr size_t lim = (size_t)kSmemLimit - 1024;
  static constexpr bool w_smem = bR + bW <= lim;
  static constexpr size_t bytes = w_smem ? bR + bW : bW;
};

template <typename T, int N, int L>
__global__ void __launch_bounds__(PrCfg<T, N>::threads, PrCfg<T, N>::minb) k_occ_pairs_pr(Params<T> P) {
  using G = Geo<N>;
  using S = Sup<N, L>;
  using SM = OccSmem<T, N, L>;
  static_assert(S::bvol <= G::vol && S::cvol <= G::vol, "slots hold a full volume");
  constexpr int NS = 6;
  constexpr int CH = sizeof(T) == 4 ? 2 : 1;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ double sO[2][2];
  __shared__ double sF0[2];
  __shared__ float bbuf[sizeof(T) == 8 ? kBoundBuf : 1];
  constexpr bool FX = sizeof(T) == 8;
  const SideArgs<T>& SD = P.side[blockIdx.y];
  const int M = P.Nk * P.no;
  const int item = blockIdx.x / P.so, chunk = blockIdx.x % P.so;
  const int i2 = P.sym ? P.irr[item / P.no] * P.no + item % P.no : P.i2_0 + item;
  const int k2 = i2 / P.no, mu2 = i2 % P.no;
  const int q2 = k2 * P.nb + mu2;
  const int i1_begin = (int)((long long)chunk * M / P.so), i1_end = (int)((long long)(chunk + 1) * M / P.so);
  const size_t cta = (size_t)blockIdx.y * gridDim.x + blockIdx.x;
  cplx<T>* slice = P.scratch + cta * NS * (size_t)G::vol;
  // (the inverse work area W1 of B1 shares R1: a pencil's L spectral values are read before its N
  // real-space values are written by the same thread)
  cplx<T>* R1 = SM::w_smem ? reinterpret_cast<cplx<T>*>(smraw) : slice + 3 * (size_t)G::vol;
  WorkT<T>* W1 = reinterpret_cast<WorkT<T>*>(smraw);
  WorkT<T>* W2 = SM::w_smem ? reinterpret_cast<WorkT<T>*>(R1 + G::vol) : W1;
  cplx<T>* A1 = slice;
  cplx<T>* A2 = slice + G::vol;
  cplx<T>* FAB = slice + 2 * (size_t)G::vol;
  cplx<T>* H6 = slice + 4 * (size_t)G::vol;
  auto ridx = [](int i, int a2, int a3) { return SM::w_smem ? G::sidx(i, a2, a3) : G::gidx(i, a2, a3); };
  const size_t NN = G::nn;
  const T f2 = weight(P, q2);
  cplx<T>* h3a4 = SD.h3a4 + ((size_t)chunk * P.nq2 + (i2 - P.i2_0)) * 3 * NN;
  cplx<T>* h3b = SD.h3b + ((size_t)chunk * P.nq2 + (i2 - P.i2_0)) * 3 * NN;
  const cplx<T>* bra2 = SD.bra + (size_t)q2 * NN;
  const cplx<T>* ket2 = SD.ket + (size_t)q2 * NN;
  for (int r = threadIdx.x; r < S::cvol; r += blockDim.x) FAB[r] = cplx<T>{0, 0};
  for (int r = threadIdx.x; r < (int)NN; r += blockDim.x) {
    H6[r] = cplx<T>{0, 0};
    for (int d = 0; d < 3; ++d) {
      h3a4[d * NN + r] = cplx<T>{0, 0};
      h3b[d * NN + r] = cplx<T>{0, 0};
    }
  }
  if (threadIdx.x == 0) { sF0[0] = 0.0; sF0[1] = 0.0; }
  __syncthreads();
  for (int i1 = i1_begin; i1 < i1_end; ++i1) {
    const int k1 = i1 / P.no, mu1 = i1 % P.no;
    const int q1 = k1 * P.nb + mu1;
    const T f1 = weight(P, q1);
    if (f1 == T(0) || f2 == T(0)) continue;
    const int id12 = P.delta_id[k2 * P.kstride + k1];   // Delta = k2 - k1 -> for P(q1,q2)
    const int id21 = P.delta_id[k1 * P.kstride + k2];   // Delta = k1 - k2 -> for P(q2,q1)
    const T* d12 = P.delta + id12 * 3;
    const T* d21 = P.delta + id21 * 3;
    const cplx<T>* bra1 = SD.bra + (size_t)q1 * NN;
    const cplx<T>* ket1 = SD.ket + (size_t)q1 * NN;
    // A1 = FT[conj(bra_q2) ket_q1], A2 = FT[conj(bra_q1) ket_q2] (work area: the rows of R1)
    // and, in fixed point, the scales of both and of the inverse transforms of u_s |p| A1 and A2
    Scale<T> s1, s2, s_inv[4];   // s_inv: (A1, pp), (A1, ap), (A2, pp), (A2, ap)
    SpecBound sb[4];
    PBound pb1, pb2;
    int x1 = 0, x2 = 0;
    if constexpr (FX) {
      const double t1 = SD.nket[q1].two * SD.nbra[q2].two, t2 = SD.nket[q2].two * SD.nbra[q1].two;
      s1 = fx_scale<T, N>(SD.nket[q1].inf * SD.nbra[q2].inf, t1);
      s2 = fx_scale<T, N>(SD.nket[q2].inf * SD.nbra[q1].inf, t2);
      x1 = fx_exp(t1 * (double)P.invN * 1.000001) + 1;
      x2 = fx_exp(t2 * (double)P.invN * 1.000001) + 1;
      pb1 = pbound_setup<T>(P, d21);
      pb2 = pbound_setup<T>(P, d12);
    }
    auto bound = [&](int c1, int c2, int c3, cplx<T> a, int which) {
      if constexpr (FX) {
        const int g = gidx_c<N, L>(c1, c2, c3);
        const float m1 = S::mil(c1), m2 = S::mil(c2), m3 = S::mil(c3);
        const T* U = P.tabU + ((size_t)(which ? id12 : id21) * 2) * NN;
#pragma unroll
        for (int s = 0; s < 2; ++s)
          (which ? sb[2 + s] : sb[s]).add(a, pbound(which ? pb2 : pb1, __ldg(U + s * NN + g), P.u_exp[s], m1, m2, m3), which ? x2 : x1);
      }
    };
    pass_axis1<T, N, L, false>(
        W1, [&](int a, int b, int c) { const int g = G::gidx(a, b, c); return mulc(ldg(ket1 + g), ldg(bra2 + g)); },
        [&](int, int, cplx<T>(&)[N]) {}, true, s1, s1);
    pfwd_32<T, N, L>(W1, [&](int c1, int c2, int c3, cplx<T> v) {
      const cplx<T> a = P.invN * v;
      A1[S::cidx(c1, c2, c3)] = a;
      bound(c1, c2, c3, a, 0);
    }, s1);
    pass_axis1<T, N, L, false>(
        W1, [&](int a, int b, int c) { const int g = G::gidx(a, b, c); return mulc(ldg(ket2 + g), ldg(bra1 + g)); },
        [&](int, int, cplx<T>(&)[N]) {}, true, s2, s2);
    pfwd_32<T, N, L>(W1, [&](int c1, int c2, int c3, cplx<T> v) {
      const cplx<T> a = P.invN * v;
      A2[S::cidx(c1, c2, c3)] = a;
      bound(c1, c2, c3, a, 1);
    }, s2);
    if constexpr (FX) {
      block_bounds<4>(sb, bbuf);
#pragma unroll
      for (int i = 0; i < 4; ++i)
      {
        const double fi = i < 2 ? 1.0 : i == 2 ? (double)f1 : 2.0 * (double)f1;
        const int x = (i < 2 ? x1 : x2) + P.u_exp[i & 1];
        s_inv[i] = fx_scale<T, L>(fx_unscale(fi * sb[i].m, x), fx_unscale(fi * sb[i].s, x));
      }
    }
    // 3a2 correction pieces for pairs at the same k (Eqs. divcor_3a2_*_density_matrix_mixing)
    if (P.div && k1 == k2) {
      if (threadIdx.x == 0) {
        const cplx<T> o21 = A1[0], o12 = A2[0];   // <bra_q2|ket_q1>, <bra_q1|ket_q2>
        sO[0][0] = o21.x; sO[0][1] = o21.y; sO[1][0] = o12.x; sO[1][1] = o12.y;
        const double fq = P.occ[q1];
        sF0[0] += fq * ((double)o21.x * o12.x - (double)o21.y * o12.y);
        sF0[1] += fq * ((double)o21.x * o12.y + (double)o21.y * o12.x);
      }
      __syncthreads();
      const cplx<T> o21 = {(T)sO[0][0], (T)sO[0][1]}, o12 = {(T)sO[1][0], (T)sO[1][1]};
      const T fq = (T)P.occ[q1];
      for (int r = threadIdx.x; r < S::cvol; r += blockDim.x) FAB[r] = FAB[r] + fq * (o12 * A1[r] + o21 * A2[r]);
      __syncthreads();
    }
    // antiparallel channel: each unordered pair once (see k_occ_pairs)
    const int cyc = (i1 - i2 + M) % M;
    const bool ap_here = P.sym || cyc == 0 || 2 * cyc < M || (2 * cyc == M && i2 < i1);
    const T ap_w = (P.sym || cyc == 0) ? T(1) : T(2);
    for (int sp = 0; sp < 2; ++sp) {
      if (sp == 1 && (!ap_here || P.h3_only || P.no_ap)) continue;
      const T w12 = (sp == 1 ? ap_w : T(1)) * f1;
      const T* U21 = P.tabU + ((size_t)id21 * 2 + sp) * NN;
      const T* U12 = P.tabU + ((size_t)id12 * 2 + sp) * NN;
      for (int d = 0; d < 3; ++d) {
        // B2 carries f1 (and the antiparallel weight): h6 / f2 and h3a4 then take it as it is
        const PComp<T> q21 = pcomp_setup<T>(P, d21, d), q12 = scaled(pcomp_setup<T>(P, d12, d), w12);
        // B1 = P^s_d(q2, q1), real space in R1
        pinv_23<T, N, L>(W1, [&](int c1, int c2, int c3) {
          const int s = S::cidx(c1, c2, c3);
          return mul_si<T, 1>((pcomp_c<T, N, L>(q21, c1, c2, c3) * __ldg(U21 + gidx_c<N, L>(c1, c2, c3))) * A1[s]);
        }, s_inv[sp]);
        pass_axis1<T, N, L, true>(
            W1, [&](int, int, int) { return cplx<T>{0, 0}; },
            [&](int a2, int a3, cplx<T>(&v)[N]) {
#pragma unroll
              for (int i = 0; i < N; ++i) R1[ridx(i, a2, a3)] = v[i];
            },
            false, s_inv[sp], s_inv[sp]);
        // B2 = P^s_d(q1, q2); its axis-1 pass forms the products with B1
        pinv_23<T, N, L>(W2, [&](int c1, int c2, int c3) {
          const int s = S::cidx(c1, c2, c3);
          return mul_si<T, 1>((pcomp_c<T, N, L>(q12, c1, c2, c3) * __ldg(U12 + gidx_c<N, L>(c1, c2, c3))) * A2[s]);
        }, s_inv[2 + sp]);
        pass_axis1<T, N, L, true>(
            W2, [&](int, int, int) { return cplx<T>{0, 0}; },
            [&](int a2, int a3, cplx<T>(&v)[N]) {
#pragma unroll
              for (int c0 = 0; c0 < N; c0 += CH) {
                cplx<T> lb1[CH], lk[CH], lr[CH];
#pragma unroll
                for (int u = 0; u < CH; ++u) {
                  if (c0 + u >= N) continue;
                  const int g = G::gidx(c0 + u, a2, a3);
                  lb1[u] = R1[ridx(c0 + u, a2, a3)];
                  if (sp == 0) {
                    lk[u] = ldg(ket1 + g);
                    lr[u] = ldg(bra1 + g);
                  }
                }
#pragma unroll
                for (int u = 0; u < CH; ++u) {
                  if (c0 + u >= N) continue;
                  const int g = G::gidx(c0 + u, a2, a3);
                  const cplx<T> b2 = v[c0 + u];
                  red_add_v(&H6[g], lb1[u] * b2);
                  if (sp == 0) {
                    red_add_v(&h3a4[d * NN + g], b2 * lk[u]);
                    red_add_v(&h3b[d * NN + g], f1 * mulc(lb1[u], lr[u]));
                  }
                }
              }
            },
            false, s_inv[2 + sp], s_inv[2 + sp]);
      }
    }
  }
  // 3a2 corrections of this q2: (f2/Nk)/Omega^2 sum_s [c_s F0 + (4 pi A_s/Nk) FT^{-1}[u~_s F_ab]]
  if (P.div && f2 != T(0) && !P.h3_only) {
    const T pref = (T)P.invOm2;   // (times f2 below)
    const T c0 = (T)(P.corr_c[0] + P.corr_c[1]);
    const cplx<T> cF0 = {(T)(c0 * sF0[0]), (T)(c0 * sF0[1])};
    const T a0 = (T)(4.0 * 3.14159265358979323846 * P.A[0] / P.Nk), a1 = (T)(4.0 * 3.14159265358979323846 * P.A[1] / P.Nk);
    auto field = [&](int c1, int c2, int c3) {
      const int g = gidx_c<N, L>(c1, c2, c3);
      const T u = a0 * P.hartUs[g] + a1 * P.hartUs[NN + g];
      return u * FAB[S::cidx(c1, c2, c3)];
    };
    const Scale<T> s_f = spectrum_scale<T, L>(
        S::cvol, [&](int c) { return field(c / (L * L), (c / L) % L, c % L); }, bbuf);
    pinv_23<T, N, L>(W2, field, s_f);
    pass_axis1<T, N, L, true>(
        W2, [&](int, int, int) { return cplx<T>{0, 0}; },
        [&](int a2, int a3, cplx<T>(&v)[N]) {
#pragma unroll
          for (int i = 0; i < N; ++i) red_add_v(&H6[G::gidx(i, a2, a3)], pref * (v[i] + cF0));
        },
        false, s_f, s_f);
  }
  if (f2 != T(0) && !P.h3_only) {
    // h6 so far without f2: the factor once per item, by the thread that added to the element
    __threadfence();
    for (int t = threadIdx.x; t < N * N; t += blockDim.x)
      for (int i = 0; i < N; ++i) {
        cplx<T>* h = H6 + G::gidx(i, t / N, t % N);
        *h = f2 * ld_l2(h);
      }
  }
}

}  // namespace tc
