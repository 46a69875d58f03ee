// The passes of the long FFT in FP32 at every sub-length of long_shapes.inc, compiled
// once per part.
#include "long_any.cuh"

#ifndef QTAM_LONG_PART
#error "QTAM_LONG_PART selects the lengths of this object"
#endif

namespace qtam {
namespace {

#define QTAM_LONG(...) both<float, __VA_ARGS__>(),
#define QTAM_LONG_ROWS(...) rows_only<float, __VA_ARGS__>(),
const LongShapeFns kShapes[] = {
#include "long_shapes.inc"
};
#undef QTAM_LONG
#undef QTAM_LONG_ROWS

}  // namespace

#define QTAM_PASTE_(a, b) a##b
#define QTAM_PASTE(a, b) QTAM_PASTE_(a, b)
const LongShapeFns* QTAM_PASTE(long_shapes_, QTAM_LONG_PART)(int* count) {
  *count = (int)(sizeof(kShapes) / sizeof(kShapes[0]));
  return kShapes;
}

}  // namespace qtam
