// 2D and 3D periodic passes: dispatch, and the FP64 instantiation
// (periodic2d.cuh has the kernels; periodic2d_f32.cu, periodic2d_mix.cu the others).
#include "periodic2d.cuh"

namespace tdse {

#define TDSE_DECLARE(NAME)                                                 \
    cudaError_t run2d_##NAME(const KArgs& a, cudaStream_t s);             \
    cudaError_t part2d_##NAME(const KArgs& a, int part, cudaStream_t s);  \
    cudaError_t run3d_##NAME(const KArgs& a, cudaStream_t s);             \
    cudaError_t part3d_##NAME(const KArgs& a, int part, cudaStream_t s);
TDSE_DECLARE(f32)
TDSE_DECLARE(f64r32)
TDSE_PASSES(f64, double2, double2)

bool periodic3d_supported(int n0, int n1, int n2) {
    auto ok = [](int n, int hi) { return n >= 8 && n <= hi && (n & (n - 1)) == 0; };
    return ok(n0, 1024) && ok(n1, 256) && ok(n2, 1024) && (long long)n0 * n1 * n2 <= (1LL << 24);
}

cudaError_t launch_periodic3d(const KArgs& a, int combo, cudaStream_t s) {
    if (!periodic3d_supported(a.tn0, a.tn1, a.tn2)) return cudaErrorInvalidValue;
    switch (combo) {
        case COMBO_F64: return run3d_f64(a, s);
        case COMBO_F32: return run3d_f32(a, s);
        case COMBO_F64_R32: return run3d_f64r32(a, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_periodic3d_part(const KArgs& a, int combo, int part, cudaStream_t s) {
    if (!periodic3d_supported(a.tn0, a.tn1, a.tn2)) return cudaErrorInvalidValue;
    switch (combo) {
        case COMBO_F64: return part3d_f64(a, part, s);
        case COMBO_F32: return part3d_f32(a, part, s);
        case COMBO_F64_R32: return part3d_f64r32(a, part, s);
        default: return cudaErrorInvalidValue;
    }
}

bool periodic2d_supported(int n0, int n1) {
    auto ok = [](int n) { return n >= 8 && n <= 1024 && (n & (n - 1)) == 0; };
    return ok(n0) && ok(n1);
}

cudaError_t launch_periodic2d(const KArgs& a, int combo, cudaStream_t s) {
    if (!periodic2d_supported(a.n0, a.n1)) return cudaErrorInvalidValue;
    switch (combo) {
        case COMBO_F64: return run2d_f64(a, s);
        case COMBO_F32: return run2d_f32(a, s);
        case COMBO_F64_R32: return run2d_f64r32(a, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_periodic2d_part(const KArgs& a, int combo, int part, cudaStream_t s) {
    if (!periodic2d_supported(a.n0, a.n1)) return cudaErrorInvalidValue;
    switch (combo) {
        case COMBO_F64: return part2d_f64(a, part, s);
        case COMBO_F32: return part2d_f32(a, part, s);
        case COMBO_F64_R32: return part2d_f64r32(a, part, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace tdse
