// 2D and 3D periodic passes with FP64 transforms on mixed-precision storage
// (start and read-out of mixed contexts): see periodic2d.cuh.
#include "periodic2d.cuh"

namespace tdse {
TDSE_PASSES(f64r32, double2, float2)
}  // namespace tdse
