// The two passes of the long FFT (kernels_long.cu) at compile-time sub-lengths.
//
// What bounds them is the L2/HBM traffic of 16 bytes a point and pass; the runtime
// engine that served the lengths that are no power of two was 10 to 40 times above
// that, with its four to six stages through shared memory, a division and strided
// twiddle loads per element, and as few as one column a block where 16 did not
// divide the row.  Here a length is two passes in registers (three for a few), and
// a block always takes 16 columns, or 4 to 16 rows, with the last block ragged.
// Neighbouring threads follow whichever index is contiguous in memory: the columns
// in the column pass; along the row on the untransposed side of the row pass and
// across the block's rows on the transposed one, whose runs are then 32 to 128
// bytes.  Measured on a GB300 against the runtime engine: rows of 192 (128 segments
// of 12288 points) 93 -> 5.1 us, 354 segments of 12000 points 175 + 1200 -> 17 + 11,
// 34 of 36000 48 + 112 -> 7.5 + 5.1 (2.6 and 3.8 TB/s), 32 of 51200 54 + 65 -> 6.3 + 5.7.
#pragma once
#include "pass_fft.cuh"
#include "qtam_internal.h"

namespace qtam {
namespace {

// A RowShape whose transforms lie PITCH elements apart with PITCH = (16 / NB) x odd:
// the NB transforms of neighbouring threads then start 16 / NB banks apart (of 16
// 8-byte ones) and their 16 / NB neighbouring butterflies fill the banks between.
template <int M_, int NB_, int NT_, int MINB_, class... Ps> struct LongShape : RowShape<M_, NB_, NT_, MINB_, Ps...> {
  using Base = RowShape<M_, NB_, NT_, MINB_, Ps...>;
  static_assert(16 % NB_ == 0, "");
  static constexpr int STEP = 16 / NB_;
  static constexpr int PITCH = ((Base::PITCH + STEP - 1) / STEP | 1) * STEP;
  static constexpr size_t smem_elems() { return Base::npass > 1 ? (size_t)NB_ * PITCH : 0; }
};

template <class Sh, int SIGN, typename T>
__global__ void __launch_bounds__(Sh::NT, Sh::MINB) k_long_columns(const __grid_constant__ LongPass g) {
  using V = cplx<T>;
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int NB = Sh::NB, M = Sh::M, R0 = Sh::R0, RL = Sh::RL;
  const int64_t seg = (int64_t)blockIdx.y * g.n;
  const int c0 = blockIdx.x * NB, n2 = g.other;
  const V* in = static_cast<const V*>(g.in) + seg + c0;
  V* out = static_cast<V*>(g.out) + seg + c0;
  const V* tw4 = static_cast<const V*>(g.tw4) + c0;
  const int cols = n2 - c0;
  after_previous();
  auto ld = [&](int b, int j, V* a) {
    if (b < cols) {
      const V* p = in + (int64_t)j * n2 + b;
#pragma unroll
      for (int i = 0; i < R0; ++i) a[i] = p[i * (M / R0) * n2];
    } else {
#pragma unroll
      for (int i = 0; i < R0; ++i) a[i] = mk<V>((T)0, (T)0);
    }
  };
  auto st = [&](int b, int j, const V* a) {
    if (b < cols) {
      const int e = j * n2 + b;
#pragma unroll
      for (int i = 0; i < RL; ++i) {
        const int o = e + i * (M / RL) * n2;
        out[o] = SIGN < 0 ? cmul(a[i], __ldg(&tw4[o])) : a[i];
      }
    }
  };
  AnyFft<Sh, SIGN, T, decltype(ld), decltype(st), ACROSS_FIRST | ACROSS_LATER | ACROSS_LAST>::run(
      reinterpret_cast<V*>(smraw), static_cast<const V*>(g.tws), ld, st);
}

template <class Sh, int SIGN, typename T>
__global__ void __launch_bounds__(Sh::NT, Sh::MINB) k_long_rows(const __grid_constant__ LongPass g) {
  using V = cplx<T>;
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int NB = Sh::NB, M = Sh::M, R0 = Sh::R0, RL = Sh::RL;
  const int64_t seg = (int64_t)blockIdx.y * g.n;
  const int r0 = blockIdx.x * NB, n1 = g.other;
  const int rows = n1 - r0;
  const V* in = static_cast<const V*>(g.in) + seg;
  V* out = static_cast<V*>(g.out) + seg;
  after_previous();
  // natural: row r0 + b of [n1][M]; transposed: column r0 + b of [M][n1]
  auto ld = [&](int b, int j, V* a) {
    if (b < rows) {
      if constexpr (SIGN < 0) {
        const V* p = in + (int64_t)(r0 + b) * M + j;
#pragma unroll
        for (int i = 0; i < R0; ++i) a[i] = p[i * (M / R0)];
      } else {
        const V* p = in + (int64_t)j * n1 + (r0 + b);
#pragma unroll
        for (int i = 0; i < R0; ++i) a[i] = p[i * (M / R0) * n1];
      }
    } else {
#pragma unroll
      for (int i = 0; i < R0; ++i) a[i] = mk<V>((T)0, (T)0);
    }
  };
  auto st = [&](int b, int j, const V* a) {
    if (b < rows) {
      if constexpr (SIGN < 0) {
        V* p = out + (int64_t)j * n1 + (r0 + b);
#pragma unroll
        for (int i = 0; i < RL; ++i) p[i * (M / RL) * n1] = a[i];
      } else {
        const int e = (r0 + b) * M + j;
        V* p = out + e;
#pragma unroll
        for (int i = 0; i < RL; ++i) p[i * (M / RL)] = cmul(a[i], cconj(__ldg(&static_cast<const V*>(g.tw4)[e + i * (M / RL)])));
      }
    }
  };
  AnyFft<Sh, SIGN, T, decltype(ld), decltype(st), SIGN < 0 ? ACROSS_LAST : ACROSS_FIRST>::run(
      reinterpret_cast<V*>(smraw), static_cast<const V*>(g.tws), ld, st);
}

template <class Sh, bool COLS, int SIGN, typename T> cudaError_t launch_long(const LongPass& g, unsigned B, cudaStream_t st) {
  const auto kernel = COLS ? k_long_columns<Sh, SIGN, T> : k_long_rows<Sh, SIGN, T>;
  const size_t smem = Sh::smem_elems() * sizeof(cplx<T>);
  const cudaError_t e = allow_smem((const void*)kernel, smem);
  if (e != cudaSuccess) return e;
  return launch_next(kernel, dim3((unsigned)((g.other + Sh::NB - 1) / Sh::NB), B), Sh::NT, smem, st, g);
}

template <typename T, class Sh> LongShapeFns rows_only() {
  LongShapeFns f{};
  f.M = Sh::M;
  f.nst = Sh::sequence(f.r);
  f.row_fwd = launch_long<Sh, false, -1, T>;
  f.row_inv = launch_long<Sh, false, +1, T>;
  return f;
}
template <typename T, class Col, class Row> LongShapeFns both() {
  static_assert(Col::M == Row::M, "");
  LongShapeFns f = rows_only<T, Row>();
  f.col_fwd = launch_long<Col, true, -1, T>;
  f.col_inv = launch_long<Col, true, +1, T>;
  return f;
}

}  // namespace
}  // namespace qtam
