// Long real FFT of each segment (step a1) and its inverse with the dual-frame
// normaliser fused in (step a7).
//
// A real segment x of N = 2n samples is read as n complex values
// z[m] = x[2m] + i x[2m+1] and transformed as an n = n1 * n2 four-step FFT:
//   column pass:  U[k1][m2] = w_n^(m2 k1) sum_m1 z[m1 n2 + m2] w_n1^(m1 k1)
//   row pass:     Z[k1 + n1 k2] = sum_m2 U[k1][m2] w_n2^(m2 k2)
// followed by the real-to-complex untangle
//   X[k] = (Z[k] + Z*[n-k]) / 2 - (i/2) w_N^k (Z[k] - Z*[n-k]),  k = 0..n
// which gives the one-sided spectrum X[f] = sum_n x[n] exp(-2 pi i f n / N)
// of App. C.  The inverse runs the same steps backwards: the untangle's
// inverse (with X_hat = A / P read through the plan's 1/P table and the DC
// and Nyquist bins taken real) feeds the row pass, then the column pass
// writes x_hat[2m] + i x_hat[2m+1] directly.
#include "fft_static.cuh"
#include "qtam_internal.h"

namespace qtam {

namespace {

// FFT engines for the four-step passes: the runtime engine takes any
// 2^a 3^b 5^c length and interleave count; the static engines fix both.
struct GenLong {
  RadixPlan rp;
  int nbs;
  static constexpr int NT = kMaxBlock;
  static constexpr int MINB = 1;
  __device__ __forceinline__ int m() const { return rp.m; }
  __host__ __device__ __forceinline__ int nb_shift() const { return nbs; }
  template <int S, typename V, class L, class St>
  __device__ __forceinline__ void run(V* sm, const V* tw, int twstride, const L& ld, const St& st) const {
    block_fft<S>(rp, nbs, sm, tw, twstride, ld, st);
  }
};
constexpr int kLongColsLog2 = 4;   // columns a block of the static column engines, log2
template <int M_, int... Rs> struct StatLong {
  static constexpr int NBS = kLongColsLog2;
  static constexpr int nrad = sizeof...(Rs);
  static constexpr int radices[nrad] = {Rs...};
  static constexpr int NT = StaticThreads<M_, NBS, Rs...>::value;   // the widest stage's items
  static constexpr int MINB = NT >= 512 ? 1 : 512 / NT;             // at least 512 threads per SM
  __device__ __forceinline__ int m() const { return M_; }
  __host__ __device__ __forceinline__ int nb_shift() const { return NBS; }
  template <int S, typename V, class L, class St>
  __device__ __forceinline__ void run(V* sm, const V* tws, int, const L& ld, const St& st) const {
    StaticFFT<S, M_, NT, NBS, Rs...>::run(sm, tws, ld, st);
  }
  static size_t smem_bytes(size_t elem) { return StaticFFT<1, M_, NT, NBS, Rs...>::smem_elems() * elem; }
};

template <typename V> struct LoadColumns {
  const V* zs; int n2; int c0;
  __device__ __forceinline__ V get(int b, int m1) const { return zs[(int64_t)m1 * n2 + c0 + b]; }
};
// tw4[k1 * n2 + c] = w_n^(c k1): the four-step twiddles in the layout of U,
// so a warp's loads are as contiguous as its stores.
template <typename V> struct StoreColumnsTwiddled {
  V* Us; const V* tw4; int n2; int c0;
  __device__ __forceinline__ void put(int b, int k1, V v) const {
    const int64_t e = (int64_t)k1 * n2 + c0 + b;
    Us[e] = cmul(v, __ldg(&tw4[e]));
  }
};
template <typename V> struct LoadRows {
  const V* Us; int n2; int r0;
  __device__ __forceinline__ V get(int b, int m2) const { return Us[(int64_t)(r0 + b) * n2 + m2]; }
};
template <typename V> struct StoreRowsTransposed {
  V* Zs; int n1; int r0;
  __device__ __forceinline__ void put(int b, int k2, V v) const { Zs[(int64_t)k2 * n1 + r0 + b] = v; }
};

template <class Eng, typename T>
__global__ void __launch_bounds__(Eng::NT, Eng::MINB) k_col_forward(Eng eng, int n, int n2, const cplx<T>* z,
                                                          cplx<T>* U, const cplx<T>* __restrict__ tw4,
                                                          const cplx<T>* __restrict__ ftw) {
  using V = cplx<T>;
  extern __shared__ __align__(16) unsigned char smraw[];
  V* sm = reinterpret_cast<V*>(smraw);
  after_previous();
  const int64_t seg = blockIdx.y;
  const int c0 = blockIdx.x << eng.nb_shift();
  LoadColumns<V> ld{z + seg * n, n2, c0};
  StoreColumnsTwiddled<V> stv{U + seg * n, tw4, n2, c0};
  eng.template run<-1>(sm, ftw, n / eng.m(), ld, stv);
}

template <class Eng, typename T>
__global__ void __launch_bounds__(Eng::NT, Eng::MINB) k_row_forward(Eng eng, int n, int n1, const cplx<T>* U,
                                                          cplx<T>* Z, const cplx<T>* __restrict__ ftw) {
  using V = cplx<T>;
  extern __shared__ __align__(16) unsigned char smraw[];
  V* sm = reinterpret_cast<V*>(smraw);
  after_previous();
  const int64_t seg = blockIdx.y;
  const int r0 = blockIdx.x << eng.nb_shift();
  LoadRows<V> ld{U + seg * n, eng.m(), r0};
  StoreRowsTransposed<V> stv{Z + seg * n, n1, r0};
  eng.template run<-1>(sm, ftw, n / eng.m(), ld, stv);
}

// w_N^k for k in [0, n]: table holds k <= n/2; w_N^(n-k) = -conj(w_N^k)
template <typename V> __device__ __forceinline__ V wN(const V* twN, int n, int k) {
  if (k <= (n >> 1)) return __ldg(&twN[k]);
  V t = __ldg(&twN[n - k]);
  return mk<V>(-t.x, t.y);
}

// (k, n-k) pairs a thread and threads a block.  FP32: four, for memory-level
// parallelism: all loaded before the first is stored, for the kernel may not claim that
// its input and its output never alias (launch_next).  FP64: one, in small blocks,
// because the FP64 pipe (2 lanes a cycle and SM) bounds it and 1024 pairs a block left
// all but five SMs idle at n = 8192 (8.4 us).
template <typename T> struct Untangle {
  static constexpr int PAIRS = sizeof(T) == 8 ? 1 : 4, NT = sizeof(T) == 8 ? 64 : 256;
  static dim3 grid(int n, int64_t nb) { return dim3((unsigned)((n / 2 + 1 + NT * PAIRS - 1) / (NT * PAIRS)), (unsigned)nb); }
};

template <typename T>
__global__ void k_untangle_forward(int n, const cplx<T>* Z, cplx<T>* X, const cplx<T>* __restrict__ twN) {
  using V = cplx<T>;
  after_previous();
  const int64_t seg = blockIdx.y;
  const V* Zs = Z + seg * n;
  V* Xs = X + seg * (int64_t)(n + 1);
  const T half = (T)0.5;
  constexpr int PAIRS = Untangle<T>::PAIRS;
  const int base = blockIdx.x * blockDim.x * PAIRS + threadIdx.x;
  V zk[PAIRS], zm[PAIRS];
#pragma unroll
  for (int u = 0; u < PAIRS; ++u) {
    const int k = base + u * blockDim.x, kk = n - k;   // partner bin, in [n/2, n]
    if (k > (n >> 1)) break;
    zk[u] = Zs[k];
    zm[u] = Zs[kk == n ? 0 : kk];
  }
#pragma unroll
  for (int u = 0; u < PAIRS; ++u) {
    const int k = base + u * blockDim.x, kk = n - k;
    if (k > (n >> 1)) break;
    {
      const V a = zk[u], b = cconj(zm[u]);
      const V s = a + b, d = a - b;
      const V t = cmul(__ldg(&twN[k]), d);    // w^k (a - b)
      Xs[k] = mk<V>(half * (s.x + t.y), half * (s.y - t.x));   // s/2 - (i/2) t
    }
    if (kk != k) {
      const V a = zm[u], b = cconj(zk[u]);
      const V s = a + b, d = a - b;
      const V t = cmul(wN(twN, n, kk), d);
      Xs[kk] = mk<V>(half * (s.x + t.y), half * (s.y - t.x));
    }
  }
}

// Inverse untangle with the dual-frame normaliser: for the pair (k, n-k),
//   Xh = A * (1/P) (DC and Nyquist taken real),
//   Zi[k] = scale (E[k] + i O[k]),  E = (Xh[k] + conj Xh[n-k]) / 2,
//   O = (Xh[k] - conj Xh[n-k]) / 2 * w_N^(-k),
// written in natural order; coalesced reads and writes, pairs per thread.
template <typename T>
__device__ __forceinline__ cplx<T> zi_value(cplx<T> xk, cplx<T> xm, cplx<T> wk, T hs) {
  using V = cplx<T>;
  const V e = xk + cconj(xm);
  const V o = cmul(xk - cconj(xm), cconj(wk));
  return mk<V>(hs * (e.x - o.y), hs * (e.y + o.x));    // scale/2 (e + i o)
}

template <typename T>
__global__ void k_untangle_inverse(int n, const cplx<T>* A, const T* __restrict__ invP, cplx<T>* Zi,
                                   const cplx<T>* __restrict__ twN, T scale) {
  using V = cplx<T>;
  after_previous();
  const int64_t seg = blockIdx.y;
  const V* As = A + seg * (int64_t)(n + 1);
  V* Zs = Zi + seg * n;
  const T hs = (T)0.5 * scale;
  constexpr int PAIRS = Untangle<T>::PAIRS;
  const int base = blockIdx.x * blockDim.x * PAIRS + threadIdx.x;
  V ak[PAIRS], am[PAIRS];
#pragma unroll
  for (int u = 0; u < PAIRS; ++u) {
    const int k = base + u * blockDim.x, kk = n - k;   // kk in [n/2, n]
    if (k > (n >> 1)) break;
    ak[u] = As[k];
    am[u] = As[kk];
  }
#pragma unroll
  for (int u = 0; u < PAIRS; ++u) {
    const int k = base + u * blockDim.x, kk = n - k;
    if (k > (n >> 1)) break;
    V xk = cscale(ak[u], __ldg(&invP[k]));
    V xm = cscale(am[u], __ldg(&invP[kk]));
    if (k == 0) xk.y = (T)0;
    if (kk == n) xm.y = (T)0;
    const V wk = __ldg(&twN[k]);
    Zs[k] = zi_value<T>(xk, xm, wk, hs);
    if (kk != k && kk != n) Zs[kk] = zi_value<T>(xm, xk, mk<V>(-wk.x, wk.y), hs);   // w^(n-k) = -conj(w^k)
  }
}

// row pass of the inverse: rows k1 of Zi, read with stride n1
template <typename V> struct LoadRowsTransposed {
  const V* Zs; int n1; int r0;
  __device__ __forceinline__ V get(int b, int k2) const { return Zs[(int64_t)k2 * n1 + r0 + b]; }
};
template <typename V> struct StoreRowsTwiddledConj {
  V* Vs; const V* tw4; int n2; int r0;
  __device__ __forceinline__ void put(int b, int m2, V v) const {
    const int64_t e = (int64_t)(r0 + b) * n2 + m2;
    Vs[e] = cmul(v, cconj(__ldg(&tw4[e])));
  }
};
template <typename V> struct StoreColumns {
  V* xs; int n2; int c0;
  __device__ __forceinline__ void put(int b, int m1, V v) const { xs[(int64_t)m1 * n2 + c0 + b] = v; }
};

template <class Eng, typename T>
__global__ void __launch_bounds__(Eng::NT, Eng::MINB) k_row_inverse(Eng eng, int n, int n1, const cplx<T>* Zi,
                                                          cplx<T>* Vb, const cplx<T>* __restrict__ tw4,
                                                          const cplx<T>* __restrict__ ftw) {
  using V = cplx<T>;
  extern __shared__ __align__(16) unsigned char smraw[];
  V* sm = reinterpret_cast<V*>(smraw);
  after_previous();
  const int64_t seg = blockIdx.y;
  const int r0 = blockIdx.x << eng.nb_shift();
  LoadRowsTransposed<V> ld{Zi + seg * n, n1, r0};
  StoreRowsTwiddledConj<V> stv{Vb + seg * n, tw4, eng.m(), r0};
  eng.template run<+1>(sm, ftw, n / eng.m(), ld, stv);
}

template <class Eng, typename T>
__global__ void __launch_bounds__(Eng::NT, Eng::MINB) k_col_inverse(Eng eng, int n, int n2, const cplx<T>* Vb,
                                                          cplx<T>* xout, const cplx<T>* __restrict__ ftw) {
  using V = cplx<T>;
  extern __shared__ __align__(16) unsigned char smraw[];
  V* sm = reinterpret_cast<V*>(smraw);
  after_previous();
  const int64_t seg = blockIdx.y;
  const int c0 = blockIdx.x << eng.nb_shift();
  LoadColumns<V> ld{Vb + seg * n, n2, c0};
  StoreColumns<V> stv{xout + seg * n, n2, c0};
  eng.template run<+1>(sm, ftw, n / eng.m(), ld, stv);
}

constexpr int64_t kMaxGridY = 65535;

// Static engines of the column pass at power-of-two lengths (FP32), 16 columns
// interleaved: 29.4 and 22.5 us forward and inverse for 64 segments of 131072
// points, where the pass engine (kernels_long_any.cu), whose exchange is padded for
// rows, takes 33.4 and 22.6.  Rows of every length run on the pass engine.
#define QTAM_LONG_CASES(X) \
  X(32, 8, 4)              \
  X(64, 16, 4)             \
  X(128, 16, 8)            \
  X(256, 16, 16)           \
  X(512, 16, 32)           \
  X(1024, 32, 32)

template <class Eng> unsigned pass_threads(const Eng&) { return Eng::NT; }
// The runtime engine runs a stage's items in rounds over whatever threads there are.
unsigned pass_threads(const GenLong& eng) { return (unsigned)spread_threads(eng.rp, eng.nbs); }
template <class Eng, class K, class... Args>
cudaError_t launch_pass(K kernel, const Eng& eng, size_t smem, dim3 g, cudaStream_t st, Args... args) {
  const cudaError_t e = allow_smem((const void*)kernel, smem);
  return e == cudaSuccess ? launch_next(kernel, g, pass_threads(eng), smem, st, eng, args...) : e;
}
// Transforms per block of a runtime pass over `count` of them: as many as the plan
// allows for coalescing, fewer while the grid leaves SMs without a block.
int gen_nbs(int nbs, int64_t count, int64_t batch) {
  while (nbs > 0 && (count >> nbs) * batch < 2 * 152) --nbs;
  return nbs;
}

#define QTAM_CASE(M, ...)                                              \
  case M: {                                                            \
    using E = StatLong<M, __VA_ARGS__>;                                \
    return f(E(), E::smem_bytes(sizeof(float2)), (const cplx<T>*)stw); \
  }

// The result of f(engine, smem bytes, engine twiddles): the static column engine where the
// plan built its tables (stw), else the runtime engine with the length-n table.
template <typename T, class F>
cudaError_t with_engine(const RadixPlan& rp, int nbs, size_t gen_smem, const void* stw, const cplx<T>* twn, int count, int64_t batch,
                 F&& f) {
  if constexpr (sizeof(T) == 4) {
    if (stw) {
      switch (rp.m) { QTAM_LONG_CASES(QTAM_CASE) default: break; }
    }
  }
  return f(GenLong{rp, gen_nbs(nbs, count, batch)}, gen_smem, twn);
}
#undef QTAM_CASE

#define QTAM_RADICES(M, ...)                                \
  case M: {                                                 \
    using E = StatLong<M, __VA_ARGS__>;                     \
    *nst = E::nrad;                                         \
    for (int i = 0; i < E::nrad; ++i) r[i] = E::radices[i]; \
    return true;                                            \
  }

// one pass of a batch through its compile-time shape
template <typename T>
cudaError_t launch_shape(LongFn f, const LongCfg& c, bool cols, const cplx<T>* in, cplx<T>* out, int64_t nb, cudaStream_t st) {
  return f(LongPass{c.n, cols ? c.n2 : c.n1, in, out, c.tw4, cols ? c.stw_col : c.stw_row}, (unsigned)nb, st);
}

}  // namespace

#define QTAM_PARTS32(X) X(0) X(1) X(2) X(3)
#define QTAM_PARTS64(X) X(0) X(1) X(2) X(3) X(4) X(5)
#define QTAM_DECL(k) const LongShapeFns* long_shapes_##k(int* count);
QTAM_PARTS32(QTAM_DECL)
#undef QTAM_DECL
#define QTAM_DECL(k) const LongShapeFns* f64_long_##k(int* count);
QTAM_PARTS64(QTAM_DECL)
#undef QTAM_DECL
namespace {
using LongPart = const LongShapeFns* (*)(int*);
template <size_t N> const LongShapeFns* find_length(const LongPart (&parts)[N], int M) {
  for (LongPart part : parts) {
    int n = 0;
    const LongShapeFns* s = part(&n);
    for (int i = 0; i < n; ++i)
      if (s[i].M == M) return &s[i];
  }
  return nullptr;
}
}  // namespace
const LongShapeFns* long_shape(int M, bool f64) {
#define QTAM_NAME(k) long_shapes_##k,
  static const LongPart p32[] = {QTAM_PARTS32(QTAM_NAME)};
#undef QTAM_NAME
#define QTAM_NAME(k) f64_long_##k,
  static const LongPart p64[] = {QTAM_PARTS64(QTAM_NAME)};
#undef QTAM_NAME
  return f64 ? find_length(p64, M) : find_length(p32, M);
}

bool long_static_radices(int m, int nbs, int* r, int* nst) {
  if (nbs != kLongColsLog2) return false;
  switch (m) { QTAM_LONG_CASES(QTAM_RADICES) default: break; }
  return false;
}
#undef QTAM_RADICES

template <typename T>
cudaError_t launch_spectrum(const LongCfg& c, const cplx<T>* z, cplx<T>* U, cplx<T>* Z, cplx<T>* X, int64_t B,
                            const cplx<T>* twn, const cplx<T>* twN, cudaStream_t st) {
  const cplx<T>* tw4 = static_cast<const cplx<T>*>(c.tw4);
  for (int64_t s0 = 0; s0 < B; s0 += kMaxGridY) {
    const int64_t nb = (B - s0) < kMaxGridY ? (B - s0) : kMaxGridY;
    const int64_t off = s0 * c.n;
    if (c.cols) {
      const cudaError_t e = launch_shape<T>(c.cols->col_fwd, c, true, z + off, U + off, nb, st);
      if (e != cudaSuccess) return e;
    } else {
      const cudaError_t e = with_engine<T>(c.rp1, c.col_nbs, c.col_smem, c.stw_col, twn, c.n2, nb,
                                              [&](auto eng, size_t smem, const cplx<T>* ftw) {
        using E = decltype(eng);
        dim3 g(c.n2 >> eng.nb_shift(), (unsigned)nb);
        return launch_pass(k_col_forward<E, T>, eng, smem, g, st, c.n, c.n2, z + off, U + off, tw4, ftw);
      });
      if (e != cudaSuccess) return e;
    }
    if (c.rows) {
      const cudaError_t e = launch_shape<T>(c.rows->row_fwd, c, false, (const cplx<T>*)(U + off), Z + off, nb, st);
      if (e != cudaSuccess) return e;
    } else {
      const cudaError_t e = with_engine<T>(c.rp2, c.row_nbs, c.row_smem, nullptr, twn, c.n1, nb,
                                              [&](auto eng, size_t smem, const cplx<T>* ftw) {
        using E = decltype(eng);
        dim3 g(c.n1 >> eng.nb_shift(), (unsigned)nb);
        return launch_pass(k_row_forward<E, T>, eng, smem, g, st, c.n, c.n1, (const cplx<T>*)(U + off), Z + off, ftw);
      });
      if (e != cudaSuccess) return e;
    }
    const cudaError_t e = launch_next(k_untangle_forward<T>, Untangle<T>::grid(c.n, nb), Untangle<T>::NT, 0, st, c.n, Z + off,
                                      X + s0 * (int64_t)(c.n + 1), twN);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <typename T>
cudaError_t launch_synthesis(const LongCfg& c, const cplx<T>* A, const T* invP, cplx<T>* Zi, cplx<T>* Vb,
                             cplx<T>* xout, int64_t B, const cplx<T>* twn, const cplx<T>* twN, cudaStream_t st) {
  const cplx<T>* tw4 = static_cast<const cplx<T>*>(c.tw4);
  for (int64_t s0 = 0; s0 < B; s0 += kMaxGridY) {
    const int64_t nb = (B - s0) < kMaxGridY ? (B - s0) : kMaxGridY;
    const int64_t off = s0 * c.n;
    const cudaError_t e0 = launch_next(k_untangle_inverse<T>, Untangle<T>::grid(c.n, nb), Untangle<T>::NT, 0, st, c.n,
                                       A + s0 * (int64_t)(c.n + 1), invP, Zi + off, twN, (T)1 / (T)c.n);
    if (e0 != cudaSuccess) return e0;
    if (c.rows) {
      const cudaError_t e = launch_shape<T>(c.rows->row_inv, c, false, (const cplx<T>*)(Zi + off), Vb + off, nb, st);
      if (e != cudaSuccess) return e;
    } else {
      const cudaError_t e = with_engine<T>(c.rp2, c.row_nbs, c.row_smem, nullptr, twn, c.n1, nb,
                                              [&](auto eng, size_t smem, const cplx<T>* ftw) {
        using E = decltype(eng);
        dim3 g(c.n1 >> eng.nb_shift(), (unsigned)nb);
        return launch_pass(k_row_inverse<E, T>, eng, smem, g, st, c.n, c.n1, (const cplx<T>*)(Zi + off), Vb + off, tw4, ftw);
      });
      if (e != cudaSuccess) return e;
    }
    if (c.cols) {
      const cudaError_t e = launch_shape<T>(c.cols->col_inv, c, true, (const cplx<T>*)(Vb + off), xout + off, nb, st);
      if (e != cudaSuccess) return e;
    } else {
      const cudaError_t e = with_engine<T>(c.rp1, c.col_nbs, c.col_smem, c.stw_col, twn, c.n2, nb,
                                              [&](auto eng, size_t smem, const cplx<T>* ftw) {
        using E = decltype(eng);
        dim3 g(c.n2 >> eng.nb_shift(), (unsigned)nb);
        return launch_pass(k_col_inverse<E, T>, eng, smem, g, st, c.n, c.n2, (const cplx<T>*)(Vb + off), xout + off, ftw);
      });
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

template cudaError_t launch_spectrum<float>(const LongCfg&, const float2*, float2*, float2*, float2*, int64_t,
                                            const float2*, const float2*, cudaStream_t);
template cudaError_t launch_spectrum<double>(const LongCfg&, const double2*, double2*, double2*, double2*, int64_t,
                                             const double2*, const double2*, cudaStream_t);
template cudaError_t launch_synthesis<float>(const LongCfg&, const float2*, const float*, float2*, float2*, float2*,
                                             int64_t, const float2*, const float2*, cudaStream_t);
template cudaError_t launch_synthesis<double>(const LongCfg&, const double2*, const double*, double2*, double2*,
                                              double2*, int64_t, const double2*, const double2*, cudaStream_t);

}  // namespace qtam
