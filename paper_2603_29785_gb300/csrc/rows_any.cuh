// Row kernels with the whole launch shape fixed at compile time.  Each envelope
// length has a pair of kernels (forward, inverse) per AnyMode, which takes every
// storage type and the carrier at run time, one pair for FP32 envelopes and bisquare
// bands, and one pair for overlap-save columns.
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
#include "pass_fft.cuh"
#include "rows_common.cuh"

namespace qtam {
namespace {

// n / f.d for n < 2^31
__device__ __forceinline__ uint32_t div_by(uint32_t n, FastDiv f) {
  return f.d == 1 ? n : __umulhi(n, f.m) >> f.s;
}

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
    const AnyRow<T> r = any_row<MODE>(g, unit0, Sh::M, false, row, seg);   // tables of the plan
    after_previous();
    StreamRow<T> s;
    if constexpr (STREAM) s = stream_row(g, row, seg, false);
    any_fft<Sh, +1, T>(
        sm, g.tws, [&](int, int j, V* a) { load_band<Sh, Sh::R0, T, MODE>(g, r, j, a); },
        [&](int, int j, V* a) { store(unit0, r.kc, s, j, a); });
  } else {
    __shared__ AnyRow<T> rs[NB];
    __shared__ StreamRow<T> ss[STREAM ? NB : 1];
    if constexpr (STREAM) after_previous();
    if (threadIdx.x < NB) {
      int row;
      uint32_t seg;
      rs[threadIdx.x] = any_row<MODE>(g, unit0 + threadIdx.x, Sh::M, false, row, seg);
      if constexpr (STREAM) ss[threadIdx.x] = stream_row(g, row, seg, false);
    }
    __syncthreads();
    if constexpr (!STREAM) after_previous();
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
    after_previous();
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
    if constexpr (STREAM) after_previous();
    if (threadIdx.x < NB) {
      int row;
      uint32_t seg;
      rs[threadIdx.x] = any_row<MODE>(g, unit0 + threadIdx.x, Sh::M, true, row, seg);
      ys[threadIdx.x] = ((int64_t)seg * g.n_rows + row) * Sh::M;
      if constexpr (STREAM) ss[threadIdx.x] = stream_row(g, row, seg, true);
    }
    __syncthreads();
    if constexpr (!STREAM) after_previous();
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
  return launch_next(k_rows_forward_any<Sh, T, E, MODE, STREAM>, dim3(blocks), Sh::NT, smem, st, g);
}
template <class Sh, typename T, int E, int MODE, bool STREAM = false>
cudaError_t launch_any_inv(const AnyArgs<T>& g, cudaStream_t st) {
  const size_t smem = Sh::smem_elems() * sizeof(cplx<T>);
  cudaError_t e = allow_smem((const void*)k_rows_inverse_any<Sh, T, E, MODE, STREAM>, smem);
  if (e != cudaSuccess) return e;
  const unsigned blocks = (g.n_units + Sh::NB - 1) / Sh::NB;
  return launch_next(k_rows_inverse_any<Sh, T, E, MODE, STREAM>, dim3(blocks), Sh::NT, smem, st, g);
}

}  // namespace
}  // namespace qtam
