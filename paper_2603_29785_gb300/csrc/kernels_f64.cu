// FP64 rows (bisquare bands at baseband) of every envelope length and FP64 passes of
// the long FFT (f64_shapes.inc), compiled once per part.  The other FP64 plans' rows
// and lengths past the lists run the runtime engine.
//
// One 4 s pair (n = 8192, 64 rows of 250): 79 -> 50 us, its latency in chains of FP64
// instructions that issue one warp in 16 cycles or more; 17 segments of 18000 points,
// 3162 rows of 1125: 1027 -> 901 us, of which the rows' 2 x 350 us are the FP64 pipe's
// time for about 45 operations a point.
#include "long_any.cuh"
#include "rows_any.cuh"

#ifndef QTAM_F64_PART
#error "QTAM_F64_PART selects the lengths of this object"
#endif

namespace qtam {
namespace {

template <class Sh> F64Rows make_rows() {
  F64Rows s{};
  s.M = Sh::M;
  s.nst = Sh::sequence(s.r);
  s.fwd = launch_any_fwd<Sh, double, ENV_F64, ANY_BISQUARE>;
  s.inv = launch_any_inv<Sh, double, ENV_F64, ANY_BISQUARE>;
  return s;
}
#define QTAM_F64_ROWS(...) make_rows<__VA_ARGS__>(),
const F64Rows kRows[] = {
#include "f64_shapes.inc"
};
#undef QTAM_F64_ROWS
#define QTAM_F64_LONG(...) both<double, __VA_ARGS__, __VA_ARGS__>(),
#define QTAM_F64_LONG_ROWS(...) rows_only<double, __VA_ARGS__>(),
const LongShapeFns kLong[] = {
#include "f64_shapes.inc"
};

}  // namespace

#define QTAM_PASTE_(a, b) a##b
#define QTAM_PASTE(a, b) QTAM_PASTE_(a, b)
const F64Rows* QTAM_PASTE(f64_rows_, QTAM_F64_PART)(int* count) {
  *count = (int)(sizeof(kRows) / sizeof(kRows[0]));
  return kRows;
}
const LongShapeFns* QTAM_PASTE(f64_long_, QTAM_F64_PART)(int* count) {
  *count = (int)(sizeof(kLong) / sizeof(kLong[0]));
  return kLong;
}

}  // namespace qtam
