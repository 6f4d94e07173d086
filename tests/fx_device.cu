// Device functions of csrc/step_common.cuh and csrc/fx.cuh against CUDA's own
// division and conversions.  `fx_device recip`: 1/d of recip_ge1, prints the largest
// error in ulps of 1.0 / d over random d in 1..2^1022, the largest relative error
// of the estimate that it starts from, and the number of wrong results of recip_any
// beyond (d up to infinity, NaN).  `fx_device float`: conversions between FP32 and FP64, prints
// the number of results that are not nearest, for widening and for narrowing.
#include <cmath>
#include <cstdio>
#include <cstring>

#include "step_common.cuh"

using namespace tdse;

struct Out {
    double ulps, estimate;
    int wrong, widen, narrow;
};

__device__ unsigned long long mix(unsigned long long z) {        // splitmix64
    z += 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}
__device__ void put_max(double* p, double v) {                   // v >= 0: ordered as its bits
    atomicMax(reinterpret_cast<unsigned long long*>(p), (unsigned long long)__double_as_longlong(v));
}

__global__ void k_recip(Out* o, int n) {
    double ulps = 0.0, est = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const unsigned long long b = mix(i);
        // a quarter next to a power of two
        unsigned long long m = b & 0xfffffffffffffull;
        if (i % 4 == 0) m = i % 8 == 0 ? (b & 7) : 0xfffffffffffffull - (b & 7);
        const double d = __longlong_as_double((long long)((1023 + (b >> 53) % 1022) << 52 | m));
        const double x = 1.0 / d, r = recip_ge1(d);
        const double ulp = __longlong_as_double(__double_as_longlong(x) & 0x7ff0000000000000ll) * 0x1p-52;
        ulps = fmax(ulps, ulp > 0.0 ? fabs(r - x) / ulp : (r == x ? 0.0 : 1e9));
        double e;
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(e) : "d"(d));
        est = fmax(est, fabs(fma(-d, e, 1.0)));
    }
    put_max(&o->ulps, ulps);
    put_max(&o->estimate, est);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const double inf = __longlong_as_double(0x7ff0000000000000ll), nan = __longlong_as_double(0x7ff8000000000000ll);
        const double big[] = {0x1p1022, 0x1.5555555555555p1022, 0x1.fffffffffffffp1022, 0x1p1023, 0x1.fffffffffffffp1023, inf};
        for (double d : big)
            if (recip_any(d) != 1.0 / d) atomicAdd(&o->wrong, 1);
        if (recip_any(nan) == recip_any(nan) || recip_any(-nan) == recip_any(-nan)) atomicAdd(&o->wrong, 1);
    }
}

__global__ void k_float(Out* o, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const unsigned long long b = mix(i);
        unsigned f = (unsigned)b;                                // any FP32 value; a quarter subnormal or zero
        if (i % 4 == 0) f = (f & 0x80000000u) | ((f & 0x7fffffu) >> (b >> 60));
        if (i % 64 == 1) f = (f & 0x80000000u) | 0x7f800000u;
        const float x = __uint_as_float(f);
        const float x2 = __uint_as_float((unsigned)(b >> 32));    // any neighbour
        const double w = FX_WIDEN * (i & 1 ? fx_widen(make_float2(x, x2)).x : fx_widen(make_float2(x2, x)).y), t = (double)x;
        // a pair as integers and back, the second component within 2^34 of the first
        if (x == x && isfinite(x)) {
            int E;
            const float y = ldexpf(1.0f + (float)(b >> 59), max(-149, min(120, ilogbf(x == 0.0f ? 1e-30f : x) - 20 + (int)((b >> 40) % 40))));
            const longlong2 v = fx_from_float(make_float2(x, y), E);
            const float2 z = fx_to_float(v, E);
            if (z.x != x || z.y != y) atomicAdd(&o->widen, 1);
        }
        if (x == x ? __double_as_longlong(w) != __double_as_longlong(t) : w == w) atomicAdd(&o->widen, 1);
        // FP64 values over FP32's range and a little beyond it on both sides
        const unsigned long long e = 1023 - 155 + (b >> 54) % 290;
        double v = __longlong_as_double((long long)((b << 63) | e << 52 | (mix(b) & 0xfffffffffffffull)));
        if (i % 64 == 2) v = 0.0;
        if (i % 64 == 3) v = __longlong_as_double(0x7ff0000000000000ll | (long long)(b << 63));
        if (i % 64 == 4) v = __longlong_as_double(0x7ff0000000000001ll);
        const double v2 = __longlong_as_double((long long)mix(b + 1));
        const float got = i & 1 ? fx_to_float(make_double2(v, v2)).x : fx_to_float(make_double2(v2, v)).y, want = (float)v;
        // nearest, ties either way; subnormal results: rounded to 24 bits, then to their step
        const bool sub = fabs(v) < 0x1p-126;
        const double off = fabs((double)got - v);
        if (v != v ? got == got : (got != want && (sub ? off > 0x1p-150 + fabs(v) * 0x1p-24 : off != fabs((double)want - v)))) atomicAdd(&o->narrow, 1);
        if (v == v && signbit(got) != signbit(want)) atomicAdd(&o->narrow, 1);
    }
}

int main(int argc, char** argv) {
    Out* o = nullptr;
    Out h{};
    if (argc < 2 || cudaMalloc(&o, sizeof(Out)) != cudaSuccess || cudaMemset(o, 0, sizeof(Out)) != cudaSuccess) return 2;
    if (!std::strcmp(argv[1], "recip")) k_recip<<<512, 256>>>(o, 1 << 26);
    else k_float<<<512, 256>>>(o, 1 << 26);
    if (cudaGetLastError() != cudaSuccess || cudaMemcpy(&h, o, sizeof(Out), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    if (!std::strcmp(argv[1], "recip")) std::printf("%.4f %.6e %d\n", h.ulps, h.estimate, h.wrong);
    else std::printf("%d %d\n", h.widen, h.narrow);
    return 0;
}
