// Row kernels with the whole launch shape fixed at compile time and the plan's
// options chosen at run time: one forward and one inverse kernel per envelope
// length serve every storage type, window family and dense-mode option.
//
// A block transforms NB rows that lie side by side in shared memory (row b at
// b * PITCH): item w of a stage is butterfly j = w mod (M / R) of row
// b = w / (M / R), so a warp's global accesses run along a row (and on into the
// next one) whatever the length.  Each exchange through shared memory has
// its own padding (RowShape::at), chosen so that neither its writers nor its
// readers hit a bank twice and every offset within a butterfly is a
// compile-time constant.
//
// The baseband position e = j + i M/R of a first-stage (forward) or last-stage
// (inverse) element holds offset d = e or d = e - M.  With |d| <= h <= (M-1)/2
// the unrolled slot i alone decides which, except the middle slot of an odd
// radix, so a slot costs one comparison and one predicated access.
#pragma once
#include "rows_common.cuh"

namespace qtam {
namespace {

// n / f.d for n < 2^31
__device__ __forceinline__ uint32_t div_by(uint32_t n, FastDiv f) {
  return f.d == 1 ? n : __umulhi(n, f.m) >> f.s;
}

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

// One row as the band loads and accumulations see it.
template <typename T> struct AnyRow {
  int kc, h, dhi, mlo;
  T kw, h2;
  int64_t base;    // element offset of the row's segment in X / A
  const T* wt;
  T cw, ew;
  bool valid;
};
template <int MODE, typename T>
__device__ __forceinline__ AnyRow<T> any_row(const AnyArgs<T>& a, uint32_t unit, int M, bool inv, int& row,
                                             uint32_t& seg) {
  AnyRow<T> r;
  r.valid = unit < a.n_units;
  seg = r.valid ? div_by(unit, a.sel) : 0;
  row = r.valid ? (int)(unit - seg * a.sel.d) : 0;
  if (inv) row = a.row_list[row];
  const RowDev<T>& rd = a.rows[row];
  const int nhalf = (int)(a.Nr - 1);
  r.kc = rd.kc;
  r.h = rd.h;
  r.kw = inv ? rd.kw_inv : rd.kw_fwd;
  r.h2 = (T)rd.h * (T)rd.h;
  r.base = (int64_t)seg * a.Nr;
  r.wt = nullptr;
  r.cw = r.ew = (T)0;
  if constexpr (MODE != ANY_BISQUARE) {
    if (a.wtab && rd.woff >= 0) {
      r.wt = a.wtab + rd.woff;
      r.cw = inv ? rd.c_inv : rd.c_fwd;
    }
    r.ew = inv ? rd.eps_inv : rd.eps_fwd;
  }
  r.dhi = max(-1, min(rd.hb, nhalf - rd.kc));
  r.mlo = M + max(-rd.hb, -rd.kc);
  if (!r.valid) {
    r.dhi = -1;
    r.mlo = M;
  }
  return r;
}
// bisquare weight at offset d (exact in T: |d|, h < 4096 for FP32)
template <typename T> __device__ __forceinline__ T bisq_weight(const AnyRow<T>& r, T d) {
  const T u = (r.h2 - d * d) * r.kw;
  return u * u;
}
// window table at |d| <= h
template <typename T> __device__ __forceinline__ T table_weight(const AnyRow<T>& r, int a) { return r.cw * __ldg(&r.wt[a]); }

// Where slot i of an R-point butterfly at position j + i MR lies: 1 below the
// middle (d = e), 2 above it (d = e - M), 3 either (middle slot, odd R).
template <int M, int MR> __host__ __device__ constexpr int slot_side(int i) {
  return (i + 1) * MR - 1 < (M + 1) / 2 ? 1 : (i * MR > (M - 1) / 2 ? 2 : 3);
}

// The usable offsets of butterfly j: slot i is in the lower band when
// below >= i MR, in the upper one when above >= -i MR.
template <typename T> struct BandRange {
  int below, above;
  __device__ __forceinline__ BandRange(const AnyRow<T>& r, int j) : below(r.dhi - j), above(j - r.mlo) {}
  template <int M, int MR> __device__ __forceinline__ bool lower(int i) const {
    return (slot_side<M, MR>(i) & 1) != 0 && below >= i * MR;
  }
  template <int M, int MR> __device__ __forceinline__ bool upper(int i) const {
    return (slot_side<M, MR>(i) & 2) != 0 && above >= -i * MR;
  }
};

// Weight of the dense placements at offset d: the window inside its support,
// its floor outside (the formula is exact as bisq_weight wherever it counts).
template <bool TAB, typename T> __device__ __forceinline__ T dense_weight(const AnyRow<T>& r, int d) {
  if constexpr (TAB) {
    const int a = d < 0 ? -d : d;
    return a <= r.h ? r.cw * __ldg(&r.wt[a]) : r.ew;
  } else {
    const T df = (T)d, v = r.h2 - df * df, u = v * r.kw;
    return v > (T)0 ? u * u : r.ew;
  }
}
// bin and offset of position e of a dense tile, at baseband or (ABS) at its own; false: none
template <int MODE, typename T>
__device__ __forceinline__ bool dense_place(const AnyRow<T>& r, int M, int nhalf, int e, int& bin, int& d) {
  if constexpr (MODE == ANY_ABS) {
    bin = e;
    d = e - r.kc;
    return e <= nhalf;
  } else {
    const bool below = e <= r.dhi;
    d = below ? e : e - M;
    bin = r.kc + d;
    return below || e >= r.mlo;
  }
}
template <class Sh, int R, typename T, int MODE, bool TAB>
__device__ __forceinline__ void load_dense(const AnyArgs<T>& g, const AnyRow<T>& r, int j, cplx<T>* a) {
  using V = cplx<T>;
  constexpr int M = Sh::M, MR = M / R;
  const int nhalf = r.valid ? (int)(g.Nr - 1) : -1;
  const V* Xs = g.X + r.base;
#pragma unroll
  for (int i = 0; i < R; ++i) {
    int bin, d;
    const bool in = dense_place<MODE>(r, M, nhalf, j + i * MR, bin, d);
    V x = mk<V>((T)0, (T)0);
    if (in) x = Xs[bin];
    a[i] = cscale(x, dense_weight<TAB>(r, d));
  }
}
template <class Sh, int R, typename T, int MODE, bool TAB>
__device__ __forceinline__ void store_dense(const AnyArgs<T>& g, const AnyRow<T>& r, int j, const cplx<T>* a) {
  using V = cplx<T>;
  constexpr int M = Sh::M, MR = M / R;
  const int nhalf = r.valid ? (int)(g.Nr - 1) : -1;
  V* As = g.A + r.base;
  if (g.divide) {
#pragma unroll
    for (int i = 0; i < R; ++i) {
      int bin, d;
      if (dense_place<MODE>(r, M, nhalf, j + i * MR, bin, d)) As[bin] = cscale(a[i], g.scale / dense_weight<TAB>(r, d));
    }
  } else {
#pragma unroll
    for (int i = 0; i < R; ++i) {
      int bin, d;
      const bool in = dense_place<MODE>(r, M, nhalf, j + i * MR, bin, d);
      add_if(As + bin, cscale(a[i], dense_weight<TAB>(r, d)), in);
    }
  }
}

// first stage, forward: a[i] = weight x spectrum at baseband position j + i MR
template <class Sh, int R, typename T, int MODE>
__device__ __forceinline__ void load_band(const AnyArgs<T>& g, const AnyRow<T>& r, int j, cplx<T>* a) {
  using V = cplx<T>;
  constexpr int M = Sh::M, MR = M / R;
  if constexpr (MODE >= ANY_DENSE) {
    if (g.wtab) load_dense<Sh, R, T, MODE, true>(g, r, j, a);
    else load_dense<Sh, R, T, MODE, false>(g, r, j, a);
  } else {
    const V* lo = g.X + (r.base + r.kc + j);
    const V* hi = lo - M;
    const BandRange<T> in(r, j);
    const T jf = (T)j;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const bool l = in.template lower<M, MR>(i), h = in.template upper<M, MR>(i);
      const int sd = slot_side<M, MR>(i);
      V x = mk<V>((T)0, (T)0);
      if (l) x = lo[i * MR];
      if (h && !(sd == 3 && l)) x = hi[i * MR];
      if constexpr (MODE == ANY_BISQUARE) {
        const T d = jf + (sd == 1 || (sd == 3 && l) ? (T)(i * MR) : (T)(i * MR - M));
        a[i] = cscale(x, bisq_weight(r, d));
      } else {
        T w = (T)0;
        if (l || h) w = table_weight(r, sd == 1 || (sd == 3 && l) ? j + i * MR : M - j - i * MR);
        a[i] = cscale(x, w);
      }
    }
  }
}

// *(p + OFF) += v when `on`: the offset goes into the instruction
template <int OFF> __device__ __forceinline__ void add_at(float2* p, float2 v, bool on) {
  asm volatile("{ .reg .pred q; setp.ne.b32 q, %3, 0; @q red.global.add.v2.f32 [%0 + %4], {%1, %2}; }"
               :: "l"(p), "f"(v.x), "f"(v.y), "r"((int)on), "n"(OFF * 8));
}
template <int OFF> __device__ __forceinline__ void add_at(double2* p, double2 v, bool on) { add_if(p + OFF, v, on); }

template <class Sh, int R, typename T, int MODE, int I>
__device__ __forceinline__ void store_slot(const AnyRow<T>& r, const BandRange<T>& in, cplx<T>* lo, cplx<T>* hi, int j, T jf,
                                           cplx<T> v) {
  constexpr int M = Sh::M, MR = M / R, sd = slot_side<M, MR>(I);
  const bool l = in.template lower<M, MR>(I), h = in.template upper<M, MR>(I);
  const bool low = sd == 1 || (sd == 3 && l);
  cplx<T>* p = low ? lo : hi;
  // Above M = 4096 a slot spans many warps and is mostly wholly inside or outside
  // the band: branching around it took 193 against 197 us at M = 4800 and 226
  // against 228 at 6000 (80 M points); below, the predicated reduction is faster
  // or equal (165.7 against 170.6 us at 1200, 156 against 162 at 1536).
  if constexpr (MODE == ANY_BISQUARE && M > 4096) {
    if (l || h) add_at<I * MR>(p, cscale(v, bisq_weight(r, jf + (low ? (T)(I * MR) : (T)(I * MR - M)))), true);
  } else if constexpr (MODE == ANY_BISQUARE) {
    add_at<I * MR>(p, cscale(v, bisq_weight(r, jf + (low ? (T)(I * MR) : (T)(I * MR - M)))), l || h);
  } else if (l || h) {
    add_at<I * MR>(p, cscale(v, table_weight(r, low ? j + I * MR : M - j - I * MR)), true);
  }
}
template <class Sh, int R, typename T, int MODE, int... I>
__device__ __forceinline__ void store_slots(const AnyArgs<T>& g, const AnyRow<T>& r, int j, const cplx<T>* a,
                                            std::integer_sequence<int, I...>) {
  cplx<T>* lo = g.A + (r.base + r.kc + j);
  cplx<T>* hi = lo - Sh::M;
  const BandRange<T> in(r, j);
  (store_slot<Sh, R, T, MODE, I>(r, in, lo, hi, j, (T)j, a[I]), ...);
}

// last stage, inverse: A[k_c + d] += weight x value at position j + i MR
template <class Sh, int R, typename T, int MODE>
__device__ __forceinline__ void store_band(const AnyArgs<T>& g, const AnyRow<T>& r, int j, const cplx<T>* a) {
  if constexpr (MODE >= ANY_DENSE) {
    if (g.wtab) store_dense<Sh, R, T, MODE, true>(g, r, j, a);
    else store_dense<Sh, R, T, MODE, false>(g, r, j, a);
  } else {
    store_slots<Sh, R, T, MODE>(g, r, j, a, std::make_integer_sequence<int, R>{});
  }
}

// envelope element `e0 + i MR` of a stage, i < R, as EnvKind E (run time when E < 0)
template <int R, int MR, typename T, int E>
__device__ __forceinline__ void store_env(const AnyArgs<T>& g, int64_t e0, const cplx<T>* a) {
  if constexpr (sizeof(T) == 8) {
    double2* p = static_cast<double2*>(g.y) + e0;
#pragma unroll
    for (int i = 0; i < R; ++i) stream_store(p + i * MR, a[i]);
  } else {
    const int env = E >= 0 ? E : g.env;
    if (env == ENV_F32) {
      float2* p = static_cast<float2*>(g.y) + e0;
#pragma unroll
      for (int i = 0; i < R; ++i) stream_store(p + i * MR, a[i]);
    } else if (env == ENV_BF16) {
      __nv_bfloat162* p = static_cast<__nv_bfloat162*>(g.y) + e0;
#pragma unroll
      for (int i = 0; i < R; ++i) stream_store(p + i * MR, Env<float2, ENV_BF16>::to(a[i]));
    } else {
      __half2* p = static_cast<__half2*>(g.y) + e0;
#pragma unroll
      for (int i = 0; i < R; ++i) stream_store(p + i * MR, Env<float2, ENV_F16>::to(a[i]));
    }
  }
}
template <int R, int MR, typename T, int E>
__device__ __forceinline__ void load_env(const AnyArgs<T>& g, int64_t e0, cplx<T>* a) {
  if constexpr (sizeof(T) == 8) {
    const double2* p = static_cast<const double2*>(g.y) + e0;
#pragma unroll
    for (int i = 0; i < R; ++i) a[i] = stream_load(p + i * MR);
  } else {
    const int env = E >= 0 ? E : g.env;
    if (env == ENV_F32) {
      const float2* p = static_cast<const float2*>(g.y) + e0;
#pragma unroll
      for (int i = 0; i < R; ++i) a[i] = stream_load(p + i * MR);
    } else if (env == ENV_BF16) {
      const __nv_bfloat162* p = static_cast<const __nv_bfloat162*>(g.y) + e0;
#pragma unroll
      for (int i = 0; i < R; ++i) a[i] = Env<float2, ENV_BF16>::from(stream_load(p + i * MR));
    } else {
      const __half2* p = static_cast<const __half2*>(g.y) + e0;
#pragma unroll
      for (int i = 0; i < R; ++i) a[i] = Env<float2, ENV_F16>::from(stream_load(p + i * MR));
    }
  }
}

// The passes of a shape.  ld(b, j, a) fills the R0 inputs of butterfly j of
// row b, st(b, j, a) takes the outputs of the last pass.
template <class Sh, int SIGN, typename T, class Load, class Store> struct AnyFft {
  using V = cplx<T>;
  static constexpr int M = Sh::M, NB = Sh::NB, NT = Sh::NT;

  template <int R> __device__ __forceinline__ static void locate(int w, int& b, int& j) {
    constexpr int MR = M / R;
    b = NB == 1 ? 0 : w / MR;
    j = NB == 1 ? w : w - b * MR;
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
        locate<R>(w, b, j);
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
        locate<R>(w, b, j);
        gather<S, NS, P>(sm, tws, b, j, a[q]);
      }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < IPT; ++q) {
      const int w = threadIdx.x + q * NT;
      if (ITEMS % NT == 0 || w < ITEMS) {
        int b, j;
        locate<R>(w, b, j);
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
        locate<R>(w, b, j);
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
template <class Sh, int SIGN, typename T, class Load, class Store>
__device__ __forceinline__ void any_fft(cplx<T>* sm, const cplx<T>* tws, const Load& ld, const Store& st) {
  AnyFft<Sh, SIGN, T, Load, Store>::run(sm, tws, ld, st);
}

// e^{+2 pi i k_c n / M} (or its conjugate) on the elements n = j + i MR
template <int R, int MR, typename T>
__device__ __forceinline__ void apply_carrier(const AnyArgs<T>& g, int kc, int M, int j, bool conj, cplx<T>* a) {
  const int kcm = kc % M;
#pragma unroll
  for (int i = 0; i < R; ++i) a[i] = carrier_rot(a[i], g.twM, kcm, j + i * MR, M, conj);
}

// Where a streaming launch stores (forward) or finds (inverse) a row's columns.
// Forward: columns Gm .. Gm + Hn - 1 of the chunk, times the chunk's phase, go
// to the map.  Inverse: chunk column n is history column n (n < split) or new
// column n - split, times the conjugate phase; both bases are those of row 0
// for rows past the last unit.
template <typename T> struct StreamRow {
  cplx<T>* out;
  const cplx<T>*hist, *fresh;
  int split;
  cplx<T> ph;
};
template <typename T>
__device__ __forceinline__ StreamRow<T> stream_row(const AnyArgs<T>& g, int row, uint32_t seg, bool inv) {
  StreamRow<T> r;
  const int64_t c0 = (int64_t)seg * g.Hn;
  r.ph = g.phase[(int64_t)seg * g.n_rows + row];
  r.out = static_cast<cplx<T>*>(g.y) + row * g.pitch + c0 - g.Gm;
  if (inv) {
    r.hist = g.hist + (int64_t)row * g.hcols + c0;
    r.fresh = static_cast<const cplx<T>*>(g.y) + row * g.pitch + max((int64_t)0, c0 - g.hcols);
    r.split = (int)max((int64_t)0, g.hcols - c0);
  }
  return r;
}
template <int R, int MR, typename T>
__device__ __forceinline__ void store_crop(const AnyArgs<T>& g, const StreamRow<T>& s, int j, const cplx<T>* a) {
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int n = j + i * MR;
    if ((unsigned)(n - g.Gm) < (unsigned)g.Hn) stream_store(s.out + n, cmul(a[i], s.ph));
  }
}
// unconditional loads, so that a butterfly's loads issue back to back, and
// default-cached: the neighbouring chunk reads each column again within the L2
template <int R, int MR, typename T>
__device__ __forceinline__ void load_chunk(const StreamRow<T>& s, int j, cplx<T>* a) {
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int n = j + i * MR;
    a[i] = cmul(*(n < s.split ? s.hist + n : s.fresh + (n - s.split)), s.ph);
  }
}

// E: the storage type, or -1: g.env.  MODE: AnyMode.  STREAM: overlap-save columns
// in place of whole envelopes (FP32).  Kernels with E < 0 also take the carrier.
template <class Sh, typename T, int E, int MODE, bool STREAM>
__global__ void __launch_bounds__(Sh::NT, Sh::MINB) k_rows_forward_any(const __grid_constant__ AnyArgs<T> g) {
  using V = cplx<T>;
  extern __shared__ __align__(16) unsigned char smraw[];
  V* sm = reinterpret_cast<V*>(smraw);
  constexpr int NB = Sh::NB, RL = Sh::RL, MR = Sh::M / RL;
  const uint32_t unit0 = blockIdx.x * NB;
  auto store = [&](uint32_t unit, int kc, const StreamRow<T>& s, int j, V* a) {
    if constexpr (STREAM) {
      store_crop<RL, MR>(g, s, j, a);
    } else {
      if (E < 0 && g.carrier) apply_carrier<RL, MR>(g, kc, Sh::M, j, false, a);
      store_env<RL, MR, T, E>(g, (int64_t)unit * Sh::M + j, a);
    }
  };
  if constexpr (NB == 1) {
    int row;
    uint32_t seg;
    const AnyRow<T> r = any_row<MODE>(g, unit0, Sh::M, false, row, seg);
    StreamRow<T> s;
    if constexpr (STREAM) s = stream_row(g, row, seg, false);
    any_fft<Sh, +1, T>(
        sm, g.tws, [&](int, int j, V* a) { load_band<Sh, Sh::R0, T, MODE>(g, r, j, a); },
        [&](int, int j, V* a) { store(unit0, r.kc, s, j, a); });
  } else {
    __shared__ AnyRow<T> rs[NB];
    __shared__ StreamRow<T> ss[STREAM ? NB : 1];
    if (threadIdx.x < NB) {
      int row;
      uint32_t seg;
      rs[threadIdx.x] = any_row<MODE>(g, unit0 + threadIdx.x, Sh::M, false, row, seg);
      if constexpr (STREAM) ss[threadIdx.x] = stream_row(g, row, seg, false);
    }
    __syncthreads();
    any_fft<Sh, +1, T>(
        sm, g.tws, [&](int b, int j, V* a) { load_band<Sh, Sh::R0, T, MODE>(g, rs[b], j, a); },
        [&](int b, int j, V* a) {
          if (unit0 + b < g.n_units) store(unit0 + b, rs[b].kc, ss[STREAM ? b : 0], j, a);
        });
  }
}

template <class Sh, typename T, int E, int MODE, bool STREAM>
__global__ void __launch_bounds__(Sh::NT, Sh::MINB) k_rows_inverse_any(const __grid_constant__ AnyArgs<T> g) {
  using V = cplx<T>;
  extern __shared__ __align__(16) unsigned char smraw[];
  V* sm = reinterpret_cast<V*>(smraw);
  constexpr int NB = Sh::NB, R0 = Sh::R0, RL = Sh::RL, MR0 = Sh::M / R0;
  const uint32_t unit0 = blockIdx.x * NB;
  // rows past the last unit read row 0's envelope; nothing of them is stored
  auto load = [&](int64_t y0, int kc, const StreamRow<T>& s, int j, V* a) {
    if constexpr (STREAM) {
      load_chunk<R0, MR0>(s, j, a);
    } else {
      load_env<R0, MR0, T, E>(g, y0 + j, a);
      if (E < 0 && g.carrier) apply_carrier<R0, MR0>(g, kc, Sh::M, j, true, a);
    }
  };
  if constexpr (NB == 1) {
    int row;
    uint32_t seg;
    const AnyRow<T> r = any_row<MODE>(g, unit0, Sh::M, true, row, seg);
    const int64_t y0 = ((int64_t)seg * g.n_rows + row) * Sh::M;
    StreamRow<T> s;
    if constexpr (STREAM) s = stream_row(g, row, seg, true);
    any_fft<Sh, -1, T>(
        sm, g.tws, [&](int, int j, V* a) { load(y0, r.kc, s, j, a); },
        [&](int, int j, V* a) { store_band<Sh, RL, T, MODE>(g, r, j, a); });
  } else {
    __shared__ AnyRow<T> rs[NB];
    __shared__ int64_t ys[NB];
    __shared__ StreamRow<T> ss[STREAM ? NB : 1];
    if (threadIdx.x < NB) {
      int row;
      uint32_t seg;
      rs[threadIdx.x] = any_row<MODE>(g, unit0 + threadIdx.x, Sh::M, true, row, seg);
      ys[threadIdx.x] = ((int64_t)seg * g.n_rows + row) * Sh::M;
      if constexpr (STREAM) ss[threadIdx.x] = stream_row(g, row, seg, true);
    }
    __syncthreads();
    any_fft<Sh, -1, T>(
        sm, g.tws, [&](int b, int j, V* a) { load(ys[b], rs[b].kc, ss[STREAM ? b : 0], j, a); },
        [&](int b, int j, V* a) { store_band<Sh, RL, T, MODE>(g, rs[b], j, a); });
  }
}

template <class Sh, typename T, int E, int MODE, bool STREAM = false>
cudaError_t launch_any_fwd(const AnyArgs<T>& g, cudaStream_t st) {
  const size_t smem = Sh::smem_elems() * sizeof(cplx<T>);
  cudaError_t e = allow_smem((const void*)k_rows_forward_any<Sh, T, E, MODE, STREAM>, smem);
  if (e != cudaSuccess) return e;
  const unsigned blocks = (g.n_units + Sh::NB - 1) / Sh::NB;
  k_rows_forward_any<Sh, T, E, MODE, STREAM><<<blocks, Sh::NT, smem, st>>>(g);
  return cudaGetLastError();
}
template <class Sh, typename T, int E, int MODE, bool STREAM = false>
cudaError_t launch_any_inv(const AnyArgs<T>& g, cudaStream_t st) {
  const size_t smem = Sh::smem_elems() * sizeof(cplx<T>);
  cudaError_t e = allow_smem((const void*)k_rows_inverse_any<Sh, T, E, MODE, STREAM>, smem);
  if (e != cudaSuccess) return e;
  const unsigned blocks = (g.n_units + Sh::NB - 1) / Sh::NB;
  k_rows_inverse_any<Sh, T, E, MODE, STREAM><<<blocks, Sh::NT, smem, st>>>(g);
  return cudaGetLastError();
}

}  // namespace
}  // namespace qtam
