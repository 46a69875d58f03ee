// Per-row kernels of the QTAM transform pair: each thread block transforms
// 2^NBS (segment, plane/row) windows.
//
// Forward (steps a2-a4; Sec. III demodulation, App. A): the first FFT stage
// gathers the row's band straight from the L2-resident spectrum, applies the
// bisquare window (Eq. gwpy_window_formula) on the fly and places offset d at
// baseband position d mod M (the roll by -k_c, crop and symmetric zero-pad);
// the short inverse FFT of length M runs in shared memory; the last stage
// writes the envelope row to HBM with unit stride, scaled by
// c_k / sqrt(M N) = c_k * sqrt(M/N) * (1/M).
//
// Inverse (steps a5-a6; Eq. qtam_canonical_inverse, App. C synthesis): the
// first stage reads the envelope row, the short forward FFT runs in shared
// memory, and the last stage keeps only the band offsets |d| <= h, re-scales
// by sqrt(N/M), weights by c_k W'(d) and adds the result into the spectrum
// accumulator A[k_c + d] with vector atomics (A stays L2-resident).
//
// FP32 plans run compile-time FFTs: the length's own shape (kernels_any.cu:
// every length a plan can have, with every window, storage type and dense-mode
// option), or a variant registered below once qtam_plan_set_variant chose it.
// The own shapes are the default because they were faster than the best
// registered variant, forward + inverse on a GB300: M = 4800 (64 segments x 640
// rows) 450 + 490 against 488 + 483 us; 2400 (55 x 384) 111 + 123 against 115 +
// 141; 1200 (48 x 384) 55 + 58 against 57 + 65; 600 (96 x 384) 47 + 55 against 51
// + 60; 300 (128 x 384) 35 + 41 against 35 + 47; 150 (200 x 384) 29 + 35 against
// 33 + 45; 75 (400 x 384) 45 + 37 against 49 + 62; 8192 (16 x 640) 248 + 201
// against 252 + 230.  FP64 plans run kernels_f64.cu for bisquare bands and the runtime
// mixed-radix engine for window tables and dense tiles.
#include "rows_common.cuh"

namespace qtam {
namespace {

// StaticEngine<M, log2 rows per block, min blocks per SM, radices...>.
// QTAM_VT: also built for window tables.
#define QTAM_V(M, NBS, MINB, ...) \
  make_variant<StaticEngine<M, NBS, MINB, __VA_ARGS__>>(#M ":" #__VA_ARGS__ " rows/blk 2^" #NBS " minblk " #MINB)
#define QTAM_VT(M, NBS, MINB, ...) \
  make_variant_tab<StaticEngine<M, NBS, MINB, __VA_ARGS__>>(#M ":" #__VA_ARGS__ " rows/blk 2^" #NBS " minblk " #MINB)
const RowVariant kVariants[] = {
    QTAM_VT(4800, 0, 4, 16, 20, 15),
    QTAM_V(4800, 0, 3, 16, 20, 15),
    QTAM_V(4800, 0, 3, 16, 15, 20),
    QTAM_V(4800, 0, 2, 16, 20, 15),
    QTAM_V(4800, 0, 3, 8, 6, 10, 10),
    QTAM_V(4800, 0, 2, 16, 12, 25),
    QTAM_VT(2400, 0, 3, 16, 10, 15),
    QTAM_V(2400, 1, 2, 16, 10, 15),
    QTAM_V(2400, 0, 4, 16, 10, 15),
    QTAM_VT(1200, 1, 2, 16, 15, 5),
    QTAM_V(1200, 2, 2, 16, 3, 25),
    QTAM_VT(600, 3, 2, 8, 3, 25),
    QTAM_V(600, 2, 2, 8, 15, 5),
    QTAM_VT(500, 3, 2, 4, 5, 25),
    QTAM_VT(300, 3, 2, 12, 25),
    QTAM_V(300, 4, 2, 4, 3, 25),
    QTAM_VT(150, 4, 2, 6, 25),
    QTAM_VT(75, 5, 2, 3, 25),
    QTAM_VT(8192, 0, 1, 16, 16, 32),
    QTAM_V(8192, 0, 1, 32, 16, 16),
    QTAM_V(8192, 0, 1, 16, 32, 16),
};
#undef QTAM_V
#undef QTAM_VT

template <typename V, int E>
__global__ void k_scale_rows(typename Env<V, E>::S* y, const float* gain, int64_t n_rows, int M) {
  // one block-stride loop per row; rows with gain 1 are left untouched
  after_previous();
  for (int64_t r = blockIdx.x; r < n_rows; r += gridDim.x) {
    const float g = gain[r];
    if (g == 1.0f) continue;
    typename Env<V, E>::S* row = y + r * M;
    for (int i = threadIdx.x; i < M; i += blockDim.x) {
      V v = Env<V, E>::from(row[i]);
      v.x *= g;
      v.y *= g;
      row[i] = Env<V, E>::to(v);
    }
  }
}

// Zeroes 8-byte words.  A kernel, not a memset node, so that it is set up while the
// kernel before drains and the accumulation while it drains; 16-byte stores between an
// odd first and last word.  Pair of one 64 s segment 47 -> 43.5 us, uneven graph 276 -> 270.
__global__ void __launch_bounds__(256) k_zero(uint2* p, int64_t words) {
  after_previous();
  const int64_t head = (reinterpret_cast<uintptr_t>(p) & 8) && words > 0 ? 1 : 0, quads = (words - head) / 2;
  uint4* q = reinterpret_cast<uint4*>(p + head);
  const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x, stride = (int64_t)gridDim.x * 256;
  if (t == 0) {
    if (head) p[0] = make_uint2(0u, 0u);
    if (head + 2 * quads < words) p[words - 1] = make_uint2(0u, 0u);
  }
  for (int64_t i = t; i < quads; i += stride) q[i] = make_uint4(0u, 0u, 0u, 0u);
}

// Per (segment, plane) pair: energy = sum |Y|^2 and peak = max |Y|^2 over
// the K*M envelope values (App. A optimal-plane selection).  FP32 envelopes are
// squared in FP32 and summed in FP32 partials of at most 8 terms (relative
// error <= ~5e-7) before FP64 accumulation; FP64 envelopes stay in FP64.  The
// partials are those of 64 parts a pair, element i of a part in partial
// (i / 2048, i mod 256), however the parts are spread over blocks: another
// grouping would move the energies by more than their FP64 sums resolve.
// Blocks combine with a double atomicAdd and an integer atomicMax on the
// (non-negative) float bits; both outputs are zeroed by the launcher first.
//
// The FP64 pipe (2 lanes a cycle and SM) bounds the reduction, not the read: one
// block per part spent 48 FP64 instructions on two or three elements a thread (128 x 5
// planes of 62 x 675: 186 us, 14 % of HBM).  A block takes `parts` consecutive parts, as
// many as leave several waves, and reduces once, in one warp from shared memory (13 FP64
// instructions, not 48); a partial widens to FP64 in the integer pipe.  Joining the parts
// took the kernel from 186 to 61 us, the one-warp reduction a scan of those planes from
// 145 to 137 us.  A NaN makes the energy NaN and is left out of the peak (fmaxf).
constexpr int kMetricParts = 64;

// (double)x of a sum of squares; normal numbers by moving exponent and fraction
__device__ __forceinline__ double widen(float x) {
  const uint32_t u = __float_as_uint(x);
  if (u - 0x00800000u >= 0x7f000000u) return (double)x;   // zero, subnormal, infinite, NaN, negative
  return __hiloint2double((int)((u >> 3) + 0x38000000u), (int)(u << 29));
}
__device__ __forceinline__ double widen(double x) { return x; }

template <typename V, int E>
__global__ void __launch_bounds__(256) k_plane_metrics(const typename Env<V, E>::S* y, int64_t per_plane, int parts, double* energy,
                                                       float* peak) {
  using R = decltype(V().x);
  after_previous();
  const int64_t pair = blockIdx.x;
  const int64_t len = (per_plane + kMetricParts - 1) / kMetricParts;
  const typename Env<V, E>::S* p = y + pair * per_plane;
  double e = 0.0;
  float mx = 0.0f;
  for (int part = blockIdx.y * parts; part < (int)(blockIdx.y + 1) * parts; ++part) {
    const int64_t b0 = part * len, b1 = min(per_plane, b0 + len);
    for (int64_t i0 = b0 + threadIdx.x; i0 < b1; i0 += 8 * (int64_t)256) {
      R es = (R)0;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int64_t i = i0 + u * 256;
        if (i < b1) {
          const V v = Env<V, E>::from(stream_load(&p[i]));
          const R a2 = v.x * v.x + v.y * v.y;
          es += a2;
          mx = fmaxf(mx, (float)a2);
        }
      }
      e += widen(es);
    }
  }
  __shared__ double se[256];
  __shared__ float sm[256];
  se[threadIdx.x] = e;
  sm[threadIdx.x] = mx;
  __syncthreads();
  if (threadIdx.x >= 32) return;
#pragma unroll
  for (int k = 1; k < 8; ++k) {
    e += se[threadIdx.x + 32 * k];
    mx = fmaxf(mx, sm[threadIdx.x + 32 * k]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    e += __shfl_xor_sync(0xffffffffu, e, o);
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  if (threadIdx.x == 0) {
    atomicAdd(&energy[pair], e);
    atomicMax(reinterpret_cast<int*>(&peak[pair]), __float_as_int(mx));
  }
}

__global__ void __launch_bounds__(256) k_clear_metrics(double* energy, float* peak, int64_t pairs) {
  after_previous();
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i < pairs) {
    energy[i] = 0.0;
    peak[i] = 0.0f;
  }
}

// One thread per segment and metric over the segment's few planes: both choices in
// one launch of the latency of a single load chain (2 us; two general arg-max
// reductions took 7.4 + 3.5 us for 128 x 5 planes).
template <typename T> __device__ __forceinline__ int64_t first_largest(const T* v, int n) {
  int best = 0;
  T m = v[0];
  for (int i = 1; i < n; ++i) {
    const T x = v[i];
    if (x > m || (x != x && m == m)) {
      m = x;
      best = i;
    }
  }
  return best;
}
__global__ void __launch_bounds__(64) k_best_planes(const double* energy, const float* peak, int64_t B, int P,
                                                    int64_t* best_energy, int64_t* best_peak) {
  after_previous();
  const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  if (blockIdx.y == 0) best_energy[b] = first_largest(energy + b * P, P);
  else best_peak[b] = first_largest(peak + b * P, P);
}

}  // namespace

cudaError_t launch_zero(void* p, size_t bytes, cudaStream_t st) {
  if (bytes == 0) return cudaSuccess;
  const int64_t words = (int64_t)(bytes / 8), blocks = (words + 2047) / 2048;   // four 16-byte stores a thread
  return launch_next(k_zero, dim3((unsigned)(blocks < 152 * 64 ? blocks : 152 * 64)), 256, 0, st, static_cast<uint2*>(p), words);
}

cudaError_t launch_best_planes(const double* energy, const float* peak, int64_t B, int P, int64_t* best_energy,
                               int64_t* best_peak, cudaStream_t st) {
  if (B == 0) return cudaSuccess;
  return launch_next(k_best_planes, dim3((unsigned)((B + 63) / 64), 2), 64, 0, st, energy, peak, B, P, best_energy, best_peak);
}

cudaError_t launch_plane_metrics(const void* y, int env, int64_t pairs, int64_t per_plane, double* energy, float* peak,
                                 cudaStream_t st) {
  if (pairs == 0) return cudaSuccess;
  const cudaError_t e0 = launch_next(k_clear_metrics, dim3((unsigned)((pairs + 255) / 256)), 256, 0, st, energy, peak, pairs);
  if (e0 != cudaSuccess) return e0;
  // a power of two, so that it divides the 64; 1216 = 8 blocks on each of 152 SMs, and
  // at least four such waves, so that a ragged last one costs little
  int parts = 1;
  while (parts < kMetricParts && pairs * (kMetricParts / parts) >= 8 * 1216) parts *= 2;
  const dim3 grid((unsigned)pairs, (unsigned)(kMetricParts / parts));
  const auto launch = [&](auto kernel, const auto* p) {
    return launch_next(kernel, grid, 256, 0, st, p, per_plane, parts, energy, peak);
  };
  switch (env) {
    case ENV_F64: return launch(k_plane_metrics<double2, ENV_F64>, static_cast<const double2*>(y));
    case ENV_BF16: return launch(k_plane_metrics<float2, ENV_BF16>, static_cast<const __nv_bfloat162*>(y));
    case ENV_F16: return launch(k_plane_metrics<float2, ENV_F16>, static_cast<const __half2*>(y));
    default: return launch(k_plane_metrics<float2, ENV_F32>, static_cast<const float2*>(y));
  }
}

cudaError_t launch_scale_rows(void* y, int env, const float* gain, int64_t n_rows, int M, cudaStream_t st) {
  if (n_rows == 0) return cudaSuccess;
  const dim3 blocks((unsigned)(n_rows < 65535 ? n_rows : 65535));
  switch (env) {
    case ENV_F64: return launch_next(k_scale_rows<double2, ENV_F64>, blocks, 256, 0, st, static_cast<double2*>(y), gain, n_rows, M);
    case ENV_BF16:
      return launch_next(k_scale_rows<float2, ENV_BF16>, blocks, 256, 0, st, static_cast<__nv_bfloat162*>(y), gain, n_rows, M);
    case ENV_F16:
      return launch_next(k_scale_rows<float2, ENV_F16>, blocks, 256, 0, st, static_cast<__half2*>(y), gain, n_rows, M);
    default: return launch_next(k_scale_rows<float2, ENV_F32>, blocks, 256, 0, st, static_cast<float2*>(y), gain, n_rows, M);
  }
}

// the dense-mode variants follow the ones registered here
// and the row-pair variants follow those
constexpr int kMainVariants = (int)(sizeof(kVariants) / sizeof(kVariants[0]));
int row_variant_count() {
  return kMainVariants + dense_row_variant_count() + pair_row_variant_count() + tuned_row_variant_count();
}
const RowVariant* row_variant(int i) {
  if (i < 0) return nullptr;
  if (i < kMainVariants) return &kVariants[i];
  i -= kMainVariants;
  if (i < dense_row_variant_count()) return dense_row_variant(i);
  i -= dense_row_variant_count();
  if (i < pair_row_variant_count()) return pair_row_variant(i);
  return tuned_row_variant(i - pair_row_variant_count());
}

#define QTAM_PARTS(X) X(0) X(1) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9) X(10) X(11) X(12) X(13) X(14) X(15)
#define QTAM_DECL(k) const AnyShape* any_shapes_##k(int* count);
QTAM_PARTS(QTAM_DECL)
#undef QTAM_DECL
const AnyShape* any_shape(int M) {
  using Part = const AnyShape* (*)(int*);
#define QTAM_NAME(k) any_shapes_##k,
  static const Part parts[] = {QTAM_PARTS(QTAM_NAME)};
#undef QTAM_NAME
  for (Part part : parts) {
    int n = 0;
    const AnyShape* s = part(&n);
    for (int i = 0; i < n; ++i)
      if (s[i].M == M) return &s[i];
  }
  return nullptr;
}
#undef QTAM_PARTS

#define QTAM_PARTS(X) X(0) X(1) X(2) X(3) X(4) X(5)
#define QTAM_DECL(k) const F64Rows* f64_rows_##k(int* count);
QTAM_PARTS(QTAM_DECL)
#undef QTAM_DECL
const F64Rows* f64_rows(int M) {
  using Part = const F64Rows* (*)(int*);
#define QTAM_NAME(k) f64_rows_##k,
  static const Part parts[] = {QTAM_PARTS(QTAM_NAME)};
#undef QTAM_NAME
  for (Part part : parts) {
    int n = 0;
    const F64Rows* s = part(&n);
    for (int i = 0; i < n; ++i)
      if (s[i].M == M) return &s[i];
  }
  return nullptr;
}
#undef QTAM_PARTS

namespace {
// what forward and inverse launches of the length's own kernels share
template <typename T>
AnyArgs<T> any_args(const RowCfg& c, const RowDev<T>* rows, int n_rows, int n_sel, int64_t Nr, int env, int64_t B,
                    const cplx<T>* twM, const T* wtab) {
  AnyArgs<T> g{};
  g.rows = rows;
  g.sel = fast_div((uint32_t)n_sel);
  g.n_rows = n_rows;
  g.n_units = (uint32_t)(B * n_sel);
  g.Nr = Nr;
  g.tws = static_cast<const cplx<T>*>(c.any_tw);
  g.wtab = wtab;
  g.twM = twM;
  g.env = env;
  g.mode = c.floor ? (c.remod ? ANY_ABS : ANY_DENSE) : wtab ? ANY_TABLE : ANY_BISQUARE;
  g.carrier = c.remod && g.mode != ANY_ABS;
  return g;
}
// Threads of a runtime-engine row: one per item of the widest stage while every row
// has an SM to itself (64 rows of 250: 22.8 -> 13.9 us), else as few as hold its
// rounds, for the FP64 pipe is then full and more warps only wait for it (3162 rows of
// 1125: 363 us against 460).
int runtime_threads(const RowCfg& c, int64_t units) { return units <= 152 ? spread_threads(c.rp, 0) : c.threads; }
// the kernels built for FP32 envelopes and bisquare bands serve the launch
bool plain(const AnyArgs<float>& g) { return g.env == ENV_F32 && g.mode == ANY_BISQUARE && !g.carrier && !g.divide; }
}  // namespace

template <typename T>
cudaError_t launch_rows_forward(const RowCfg& c, const RowDev<T>* rows, int n_rows, int64_t Nr, const cplx<T>* X,
                                void* y, int env, int64_t B, const cplx<T>* twM, cudaStream_t st, const T* wtab) {
  const int64_t units = B * n_rows;
  if (units == 0) return cudaSuccess;
  if constexpr (sizeof(T) == 4) {
    if (const RowVariant* v = c.chosen ? row_variant(c.variant) : nullptr) {
      const float2* stw = static_cast<const float2*>(c.stw);
      if (c.dense) {
        if (v->fwd_dense)
          return v->fwd_dense(rows, n_rows, Nr, X, y, B, stw, st, wtab, twM, c.dense == 2 ? 2 : c.remod, env);
      } else {
        if (!wtab) return v->fwd[env](rows, n_rows, Nr, X, y, B, stw, st);
        if (env == ENV_F32 && v->fwd_tab) return v->fwd_tab(rows, n_rows, Nr, X, y, B, stw, st, wtab);
      }
    }
    AnyArgs<float> g = any_args(c, rows, n_rows, n_rows, Nr, env, B, twM, wtab);
    g.X = X;
    g.y = y;
    if (!plain(g)) return c.any->fwd[g.mode](g, st);
    g.tws = static_cast<const float2*>(c.any_tw_plain);
    return c.any->fwd_plain(g, st);
  } else {
    if (c.f64) {
      AnyArgs<T> g = any_args<T>(c, rows, n_rows, n_rows, Nr, env, B, twM, wtab);
      g.X = X;
      g.y = y;
      return c.f64->fwd(g, st);
    }
    GenericEngine eng{c.rp};
    DenseArgs<T> da;
    da.remod = c.remod;
    const cudaError_t e = allow_smem((const void*)k_rows_forward<T, ENV_F64>, c.smem);
    if (e != cudaSuccess) return e;
    return launch_next(k_rows_forward<T, ENV_F64>, dim3((unsigned)units), runtime_threads(c, units), c.smem, st, eng, rows,
                       n_rows, Nr, X, static_cast<double2*>(y), units, twM, wtab, da);
  }
}

template <typename T>
cudaError_t launch_rows_inverse(const RowCfg& c, const RowDev<T>* rows, const int* row_list, int n_sel, int n_rows,
                                int64_t Nr, const void* y, int env, cplx<T>* A, int64_t B, const cplx<T>* twM,
                                cudaStream_t st, const T* wtab, DenseArgs<T> da) {
  const int64_t units = B * n_sel;
  da.remod = c.remod;
  if (units == 0) return cudaSuccess;
  if constexpr (sizeof(T) == 4) {
    if (const RowVariant* v = c.chosen && !da.divide ? row_variant(c.variant) : nullptr) {
      const float2* stw = static_cast<const float2*>(c.stw);
      if (c.dense) {
        if (v->inv_dense)
          return v->inv_dense(rows, row_list, n_sel, n_rows, Nr, y, A, B, stw, st, wtab, twM, c.dense == 2 ? 2 : c.remod,
                              env);
      } else {
        if (!wtab) return v->inv[env](rows, row_list, n_sel, n_rows, Nr, y, A, B, stw, st);
        if (env == ENV_F32 && v->inv_tab) return v->inv_tab(rows, row_list, n_sel, n_rows, Nr, y, A, B, stw, st, wtab);
      }
    }
    AnyArgs<float> g = any_args(c, rows, n_rows, n_sel, Nr, env, B, twM, wtab);
    g.row_list = row_list;
    g.A = A;
    g.y = const_cast<void*>(y);
    g.divide = da.divide;
    g.scale = da.scale;
    return plain(g) ? c.any->inv_plain(g, st) : c.any->inv[g.mode](g, st);
  } else {
    if (c.f64 && !da.divide) {
      AnyArgs<T> g = any_args<T>(c, rows, n_rows, n_sel, Nr, env, B, twM, wtab);
      g.row_list = row_list;
      g.A = A;
      g.y = const_cast<void*>(y);
      return c.f64->inv(g, st);
    }
    GenericEngine eng{c.rp};
    const cudaError_t e = allow_smem((const void*)k_rows_inverse<T, ENV_F64>, c.smem);
    if (e != cudaSuccess) return e;
    return launch_next(k_rows_inverse<T, ENV_F64>, dim3((unsigned)units), runtime_threads(c, units), c.smem, st, eng, rows,
                       row_list, n_sel, n_rows, Nr, static_cast<const double2*>(y), A, units, twM, wtab, da);
  }
}

cudaError_t launch_rows_stream_forward(const RowCfg& c, const RowDev<float>* rows, int n_rows, int64_t Nr, const float2* X,
                                       float2* y, int64_t pitch, int Gm, int Hn, const float2* phase, int64_t B,
                                       cudaStream_t st) {
  if (B * n_rows == 0) return cudaSuccess;
  AnyArgs<float> g = any_args<float>(c, rows, n_rows, n_rows, Nr, ENV_F32, B, nullptr, nullptr);
  g.X = X;
  g.y = y;
  g.pitch = pitch;
  g.Gm = Gm;
  g.Hn = Hn;
  g.phase = phase;
  return c.any->fwd_stream(g, st);
}
cudaError_t launch_rows_stream_inverse(const RowCfg& c, const RowDev<float>* rows, const int* row_list, int n_sel,
                                       int n_rows, int64_t Nr, const float2* hist, int hcols, const float2* ynew,
                                       int64_t pitch, int Hn, const float2* phase, float2* A, int64_t B,
                                       cudaStream_t st) {
  if (B * n_sel == 0) return cudaSuccess;
  AnyArgs<float> g = any_args<float>(c, rows, n_rows, n_sel, Nr, ENV_F32, B, nullptr, nullptr);
  g.row_list = row_list;
  g.A = A;
  g.y = const_cast<float2*>(ynew);
  g.hist = hist;
  g.hcols = hcols;
  g.pitch = pitch;
  g.Hn = Hn;
  g.phase = phase;
  return c.any->inv_stream(g, st);
}

template cudaError_t launch_rows_forward<float>(const RowCfg&, const RowDev<float>*, int, int64_t, const float2*, void*,
                                                int, int64_t, const float2*, cudaStream_t, const float*);
template cudaError_t launch_rows_forward<double>(const RowCfg&, const RowDev<double>*, int, int64_t, const double2*,
                                                 void*, int, int64_t, const double2*, cudaStream_t, const double*);
template cudaError_t launch_rows_inverse<float>(const RowCfg&, const RowDev<float>*, const int*, int, int, int64_t,
                                                const void*, int, float2*, int64_t, const float2*, cudaStream_t,
                                                const float*, DenseArgs<float>);
template cudaError_t launch_rows_inverse<double>(const RowCfg&, const RowDev<double>*, const int*, int, int, int64_t,
                                                 const void*, int, double2*, int64_t, const double2*, cudaStream_t,
                                                 const double*, DenseArgs<double>);

}  // namespace qtam
