// The row kernels of every envelope length a plan can have (rows_any.cuh
// instantiated over row_shapes.inc).  Compiled once per part, so the parts
// build in parallel.
#include "rows_any.cuh"

#ifndef QTAM_PART
#error "QTAM_PART selects the lengths of this object"
#endif

namespace qtam {
namespace {

// Plain: forward rows of FP32 envelopes and bisquare bands; Sh: the others
template <class Plain, class Sh> AnyShape make_shape() {
  static_assert(Plain::M == Sh::M, "");
  AnyShape s{};
  s.M = Sh::M;
  s.nst_plain = Plain::sequence(s.r_plain);
  s.nst = Sh::sequence(s.r);
  s.fwd_plain = launch_any_fwd<Plain, float, ENV_F32, ANY_BISQUARE>;
  s.inv_plain = launch_any_inv<Sh, float, ENV_F32, ANY_BISQUARE>;
  s.fwd_stream = launch_any_fwd<Sh, float, ENV_F32, ANY_BISQUARE, true>;
  s.inv_stream = launch_any_inv<Sh, float, ENV_F32, ANY_BISQUARE, true>;
  s.fwd[0] = launch_any_fwd<Sh, float, -1, ANY_BISQUARE>;
  s.inv[0] = launch_any_inv<Sh, float, -1, ANY_BISQUARE>;
  s.fwd[1] = launch_any_fwd<Sh, float, -1, ANY_TABLE>;
  s.inv[1] = launch_any_inv<Sh, float, -1, ANY_TABLE>;
  s.fwd[2] = launch_any_fwd<Sh, float, -1, ANY_DENSE>;
  s.inv[2] = launch_any_inv<Sh, float, -1, ANY_DENSE>;
  s.fwd[3] = launch_any_fwd<Sh, float, -1, ANY_ABS>;
  s.inv[3] = launch_any_inv<Sh, float, -1, ANY_ABS>;
  return s;
}
#define QTAM_SHAPE(...) make_shape<__VA_ARGS__>(),
const AnyShape kShapes[] = {
#include "row_shapes.inc"
};
#undef QTAM_SHAPE

}  // namespace

#define QTAM_PASTE_(a, b) a##b
#define QTAM_PASTE(a, b) QTAM_PASTE_(a, b)
const AnyShape* QTAM_PASTE(any_shapes_, QTAM_PART)(int* count) {
  *count = (int)(sizeof(kShapes) / sizeof(kShapes[0]));
  return kShapes;
}

}  // namespace qtam
