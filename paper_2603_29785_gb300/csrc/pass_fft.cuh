// FFT of M = product of compile-time passes inside one block, NB transforms side
// by side: each pass is one butterfly per thread and one exchange through shared
// memory.  The row kernels (rows_any.cuh) and the passes of the long FFT
// (kernels_long_any.cu) are built on it.
#pragma once

#include "fft_core.cuh"

namespace qtam {
namespace {

// One pass over shared memory: a butterfly of R = r_0 r_1 ... points.  A single
// radix runs as Dft<R>; several run as that many Stockham stages in registers,
// each with its own twiddles and in the order and arithmetic of separate
// stages: the twiddles cost the same loads and multiplies as one R-point stage.
template <int... Rs> struct Pass {
  static constexpr int R = (Rs * ...);
  static constexpr int n = sizeof...(Rs);
  // radix of stage s, product of the radices before it
  __host__ __device__ static constexpr int radix(int s) {
    const int r[n] = {Rs...};
    return r[s];
  }
  __host__ __device__ static constexpr int before(int s) { return s == 0 ? 1 : before(s - 1) * radix(s - 1); }
  // After s stages the registers hold before(s) runs; run number q (digits of
  // the stages so far, the first most significant) belongs to this output digit
  // (the first least significant).
  __host__ __device__ static constexpr int digit(int s, int q) {
    return s == 0 ? 0 : digit(s - 1, q / radix(s - 1)) + before(s - 1) * (q % radix(s - 1));
  }
};

__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// Stages of pass P at span NS on the inputs a[]; t points at the first stage's
// table plus the butterfly's k = j mod NS (tables [i][k] per stage, one after
// another; the first pass, NS = 1, has none for its first stage).
template <class P, int SIGN, int NS, typename V> struct PassRun {
  template <int S, int Q, int... I> __device__ __forceinline__ static void run_of(const V* __restrict__ t, V* a, std::integer_sequence<int, I...>) {
    constexpr int DONE = P::before(S), REM = P::R / DONE, R = P::radix(S), STEP = REM / R;
    constexpr int D = P::digit(S, Q);
#pragma unroll
    for (int m = 0; m < STEP; ++m) {
      V v[R];
      ((v[I] = a[Q * REM + m + I * STEP]), ...);
      if constexpr (NS == 1) {
        (twiddle_fixed<I * D, DONE * R>(v[I]), ...);
      } else {
        (twiddle_by<(I * DONE + D) * NS, I>(t, v[I]), ...);
      }
      Dft<R, SIGN>::run(v);
      ((a[Q * REM + m + I * STEP] = v[I]), ...);
    }
  }
  // the first pass's inner twiddles are constants; products and sums round as
  // in twiddle_by, whose cosine products go into the fused multiply-adds
  template <int E, int L> __device__ __forceinline__ static void twiddle_fixed(V& x) {
    using T = decltype(V::x);
    if constexpr (E % L == 0 || (4 * (E % L)) % L == 0) {
      twiddle_const<E, L, SIGN>(x);
    } else {
      constexpr T c = (T)ce_cos2pi(E % L, L), s = (T)(SIGN * ce_sin2pi(E % L, L));
      const T p = mul_rn(x.y, s), q = mul_rn(x.x, s);
      x = mk<V>(fma(x.x, c, -p), fma(x.y, c, q));
    }
  }
  template <int E, int I> __device__ __forceinline__ static void twiddle_by(const V* __restrict__ t, V& x) {
    if constexpr (I > 0) {
      V w = __ldg(&t[E]);
      if (SIGN > 0) w.y = -w.y;
      x = cmul(x, w);
    }
  }
  template <int S, int... Q> __device__ __forceinline__ static void stage(const V* __restrict__ t, V* a, std::integer_sequence<int, Q...>) {
    (run_of<S, Q>(t, a, std::make_integer_sequence<int, P::radix(S)>{}), ...);
    if constexpr (S + 1 < P::n)
      stage<S + 1>(t + NS * P::before(S + 1), a, std::make_integer_sequence<int, P::before(S + 1)>{});
  }
  template <int... Q> __device__ __forceinline__ static void order(V* a, std::integer_sequence<int, Q...>) {
    V b[P::R];
    ((b[P::digit(P::n, Q)] = a[Q]), ...);
    ((a[Q] = b[Q]), ...);
  }
  __device__ __forceinline__ static void run(const V* __restrict__ t, V* a) {
    stage<0>(t, a, std::make_integer_sequence<int, 1>{});
    if constexpr (P::n > 1) order(a, std::make_integer_sequence<int, P::R>{});
  }
};

// M, rows per block, threads, blocks per SM the registers must allow, passes
template <int M_, int NB_, int NT_, int MINB_, class... Ps> struct RowShape {
  static constexpr int M = M_, NB = NB_, NT = NT_, MINB = MINB_;
  static constexpr int npass = sizeof...(Ps);
  static constexpr int nrad = (Ps::n + ...);
  static_assert((Ps::R * ...) == M_, "the passes make up the length");
  static_assert(M_ <= 8192, "bisquare weights in FP32 need h < 4096");
  __host__ __device__ static constexpr int points(int p) {   // R of pass p
    const int r[npass] = {Ps::R...};
    return r[p];
  }
  static constexpr int R0 = points(0), RL = points(npass - 1);
  __host__ __device__ static constexpr int span(int p) { return p == 0 ? 1 : span(p - 1) * points(p - 1); }
  // Exchange p (between passes p and p + 1): element e lies at
  // e + (e / block(p)) * gap(p).  Exchange 0 pads every R0 elements when R0 is
  // even, so that the writers' stride R0 + 1 is odd; the later ones shift every
  // block of span(p + 1) elements so that the next block's writers go on at the
  // bank where these ended (span(p + 1) + gap = span(p) mod 16, the number of
  // 8-byte banks): both the writes and the reads of a half-warp hit 16 banks.
  __host__ __device__ static constexpr int block(int p) { return span(p + 1); }
  __host__ __device__ static constexpr int gap(int p) {
    return p == 0 ? (R0 % 2 == 0 ? 1 : 0) : (((span(p) - span(p + 1)) % 16) + 16) % 16;
  }
  template <int S> __host__ __device__ __forceinline__ static constexpr int at(int e) {
    constexpr int g = gap(S), len = block(S);
    return g != 0 ? e + (e / len) * g : e;
  }
  static constexpr int extent(int p) { return (M_ / block(p)) * (block(p) + gap(p)); }
  static constexpr int pitch_from(int p) {
    return p + 1 >= npass ? 0 : (extent(p) > pitch_from(p + 1) ? extent(p) : pitch_from(p + 1));
  }
  static constexpr int PITCH = pitch_from(0);   // elements from one row of the block to the next
  static constexpr size_t smem_elems() { return (size_t)NB * PITCH; }
  // flat radix sequence, for the stage tables
  template <class Q> static void append(int* r, int& n) {
    for (int i = 0; i < Q::n; ++i) r[n++] = Q::radix(i);
  }
  static int sequence(int* r) {
    int n = 0;
    (append<Ps>(r, n), ...);
    return n;
  }
};

// The passes of a shape.  ld(b, j, a) fills the R0 inputs of butterfly j of
// row b, st(b, j, a) takes the outputs of the last pass.  Consecutive threads
// take consecutive butterflies of a row, in the passes of ACROSS consecutive rows.
enum { ACROSS_FIRST = 1, ACROSS_LATER = 2, ACROSS_LAST = 4 };
template <class Sh, int SIGN, typename T, class Load, class Store, int ACROSS = 0> struct AnyFft {
  using V = cplx<T>;
  static constexpr int M = Sh::M, NB = Sh::NB, NT = Sh::NT;

  template <int R, int WHEN> __device__ __forceinline__ static void locate(int w, int& b, int& j) {
    constexpr int MR = M / R;
    if constexpr ((ACROSS & WHEN) != 0) {
      b = w % NB;
      j = w / NB;
    } else {
      b = NB == 1 ? 0 : w / MR;
      j = NB == 1 ? w : w - b * MR;
    }
  }
  // butterfly of pass S >= 1 from shared memory (exchange S - 1; every stride
  // M / R is a multiple of that exchange's block, so slot i is a constant away)
  template <int S, int NS, class P> __device__ __forceinline__ static void gather(const V* sm, const V* tws, int b, int j, V* a) {
    constexpr int R = P::R;
    static_assert((M / R) % Sh::block(S - 1) == 0, "");
    const V* p = sm + b * Sh::PITCH + Sh::template at<S - 1>(j);
#pragma unroll
    for (int i = 0; i < R; ++i) a[i] = p[Sh::template at<S - 1>(i * (M / R))];
    PassRun<P, SIGN, NS, V>::run(tws + j % NS, a);
  }
  // outputs of pass S into exchange S: the butterfly's R outputs share a block
  template <int S, int NS, int R> __device__ __forceinline__ static void scatter(V* sm, int b, int j, const V* a) {
    constexpr int LEN = NS * R + Sh::gap(S);
    V* p = sm + b * Sh::PITCH + (j / NS) * LEN + j % NS;
#pragma unroll
    for (int i = 0; i < R; ++i) p[i * NS] = a[i];
  }
  // entries of a pass's stage tables (the very first stage has none)
  template <int NS, class P> __host__ __device__ static constexpr int table_size() {
    int n = 0;
    for (int s = 0; s < P::n; ++s)
      if (NS * P::before(s) > 1) n += NS * P::before(s + 1);
    return n;
  }

  template <int S, int NS, class P> __device__ __forceinline__ static void later(V* sm, const V* tws, const Load&, const Store& st) {
    constexpr int R = P::R, ITEMS = NB * (M / R), IPT = (ITEMS + NT - 1) / NT;
#pragma unroll
    for (int q = 0; q < IPT; ++q) {
      const int w = threadIdx.x + q * NT;
      if (ITEMS % NT == 0 || w < ITEMS) {
        int b, j;
        locate<R, ACROSS_LAST>(w, b, j);
        V a[R];
        gather<S, NS, P>(sm, tws, b, j, a);
        st(b, j, a);
      }
    }
  }
  template <int S, int NS, class P, class P2, class... Rest>
  __device__ __forceinline__ static void later(V* sm, const V* tws, const Load& ld, const Store& st) {
    constexpr int R = P::R, ITEMS = NB * (M / R), IPT = (ITEMS + NT - 1) / NT;
    V a[IPT][R];
#pragma unroll
    for (int q = 0; q < IPT; ++q) {
      const int w = threadIdx.x + q * NT;
      if (ITEMS % NT == 0 || w < ITEMS) {
        int b, j;
        locate<R, ACROSS_LATER>(w, b, j);
        gather<S, NS, P>(sm, tws, b, j, a[q]);
      }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < IPT; ++q) {
      const int w = threadIdx.x + q * NT;
      if (ITEMS % NT == 0 || w < ITEMS) {
        int b, j;
        locate<R, ACROSS_LATER>(w, b, j);
        scatter<S, NS, R>(sm, b, j, a[q]);
      }
    }
    __syncthreads();
    constexpr int SKIP = table_size<NS, P>();
    later<S + 1, NS * R, P2, Rest...>(sm, tws + SKIP, ld, st);
  }
  template <class P, class... Rest> __device__ __forceinline__ static void first(V* sm, const V* tws, const Load& ld, const Store& st) {
    constexpr int R = P::R, ITEMS = NB * (M / R), IPT = (ITEMS + NT - 1) / NT;
#pragma unroll
    for (int q = 0; q < IPT; ++q) {
      const int w = threadIdx.x + q * NT;
      if (ITEMS % NT == 0 || w < ITEMS) {
        int b, j;
        locate<R, ACROSS_FIRST>(w, b, j);
        V a[R];
        ld(b, j, a);
        PassRun<P, SIGN, 1, V>::run(tws, a);
        if constexpr (sizeof...(Rest) == 0) st(b, j, a);
        else scatter<0, 1, R>(sm, b, j, a);
      }
    }
    if constexpr (sizeof...(Rest) > 0) {
      __syncthreads();
      constexpr int SKIP = table_size<1, P>();
      later<1, R, Rest...>(sm, tws + SKIP, ld, st);
    }
  }
  template <int M_, int NB_, int NT_, int MINB_, class... Ps>
  __device__ __forceinline__ static void start(RowShape<M_, NB_, NT_, MINB_, Ps...>, V* sm, const V* tws, const Load& ld,
                                               const Store& st) {
    first<Ps...>(sm, tws, ld, st);
  }
  __device__ __forceinline__ static void run(V* sm, const V* tws, const Load& ld, const Store& st) {
    start(Sh(), sm, tws, ld, st);
  }
};

}  // namespace
}  // namespace qtam
