// 2D and 3D periodic passes with FP32 transforms (mixed-precision steps): see periodic2d.cuh.
#include "periodic2d.cuh"

namespace tdse {
TDSE_PASSES(f32, float2, float2)
}  // namespace tdse
