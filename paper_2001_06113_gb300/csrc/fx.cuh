// FP64 transforms in 64-bit fixed point.
//
// GB300 issues FP64 at 1/64 of its FP32 rate: an FP64 instruction holds an
// SM's scheduler partition for 64 cycles per warp, an IADD for 1 and a
// 32 x 32 + 64-bit multiply-add for 2 (measured: 1.6 FP64, 91 IADD, 49 wide
// multiply-add lanes per SM and cycle, launch included).  A radix-8 butterfly
// with its twiddles is 84 FP64 instructions = 5376 cycles, and about 375
// cycles in the form below.
//
// A transform takes FP64 inputs, finds the largest exponent E of the line, and
// holds x 2^(S + 1022 - E), S = 62 - log2(first radix), as 64-bit
// integers: components below 2^S, so that after the first butterfly the
// modulus is at most 2^62.5.  Every later pass of radix R multiplies by the
// twiddle and by 1/R in the same 128-bit product and adds up R terms, which
// keeps that bound; the power of two is put back into the exponent when the
// results are rounded to FP64.  Quantisation of the input is below 2^-58 of
// the line's largest component, each product is rounded at 2^-59.5 / R of
// the full scale.  Lines of 2048 points and more are scaled up again before each
// middle pass (FxPass::rescales).  Relative L2 error of a transform, FP64 passes in
// brackets: input spread over the line 7e-17 (4e-16) at any n; one nonzero value
// 7.5e-17 (3e-16) at n = 512, 1.6e-16 (3.5e-16) at 1024, 9e-17 (4e-16) at 8192, where
// without the scaling it was 1.4e-15 (tests/test_fx_cpu.py, test_fx_long_cpu.py compare
// both with long double).  Measured: 100 steps of 4 x 512^2 in FP64 90.4 -> 51.4 ms,
// 60 steps of the 256^2 free-space workload 328 -> 216 ms.
//
// A table factor w (|w| <= 1) is an int4 {ch, cl, sh, sl}: cos = ch 2^32 + cl in
// units of 2^-61, cl signed (likewise sin), so that signed 32-bit
// multiply-adds form every product: with a = xh 2^32 + xl (xl signed too)
//   a w / 2^64 = (xh ch) + (xh cl + xl ch) / 2^32 + (dropped) xl cl / 2^64,
// and for complex factors the four cross products of one component stay
// below 2^63 when |a| <= 2^62.5.
//
// NaN or infinity anywhere in a line gives NaN everywhere in it (an FP64
// transform spreads them over the whole line).  A line is held to 2^-1017 at best:
// magnitudes below 2^-958 lose low bits and those below 2^-1022 become 0.  (Keeping
// them costs three more instructions in every conversion: 4 x 512^2 in FP64 31.6 ->
// 33.9 ms.)
#pragma once
#include <cuda_runtime.h>

namespace tdse {

#define FX_HD __host__ __device__ __forceinline__

FX_HD longlong2 operator+(longlong2 a, longlong2 b) { return make_longlong2(a.x + b.x, a.y + b.y); }
FX_HD longlong2 operator-(longlong2 a, longlong2 b) { return make_longlong2(a.x - b.x, a.y - b.y); }

// Exponent of a block from the largest high word (sign bit cleared) of its
// values: E, at least 64 so that the shifts below stay in range.
FX_HD int fx_exponent(unsigned max_hi) {
    const int e = (int)(max_hi >> 20);
    return e < 64 ? 64 : e;
}
constexpr int FX_NAN = 1 << 20;     // output exponent of a block with a NaN or an infinity

// v 2^(S + 1022 - E), truncated towards zero (S <= 61, E >= the exponent of v).
FX_HD long long fx_from_bits(int hi, unsigned lo, int S, int E) {
    const unsigned long long mant = ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32 | lo) << 10;
    int sh = 63 - S + E - ((hi >> 20) & 0x7ff);
    sh = sh > 63 ? 63 : sh;
    const long long t = (long long)(mant >> (sh & 63));
    return hi < 0 ? -t : t;
}

// v 2^X rounded to FP64, as its bits.
FX_HD unsigned long long fx_to_bits(long long v, int X) {
    const unsigned long long sign = (unsigned long long)v & 0x8000000000000000ull;
    const unsigned long long u = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
#ifdef __CUDA_ARCH__
    const int lz = __clzll((long long)u);
#else
    const int lz = u ? __builtin_clzll(u) : 64;
#endif
    const unsigned long long t = u << (lz & 63);
    const int e = X - lz + 1085;
    if (u == 0 || (unsigned)e >= 2046u) {
        if (X >= FX_NAN / 2) return 0x7ff8000000000000ull;
        return sign | (u == 0 || e < 0 ? 0ull : 0x7ff0000000000000ull);
    }
    return sign | (((unsigned long long)(unsigned)e << 52) + (t >> 11) + ((t >> 10) & 1));
}

// a w 2^K / 2^64 (w in units of 2^-61: K = 3 multiplies by w, K = 3 - log2 R by w / R;
// K may be negative), |a| <= 2^62.5 and the result likewise.
template <bool CONJ, int K>
FX_HD longlong2 fx_mul(longlong2 a, int4 w) {
    const int xl = (int)a.x, yl = (int)a.y;
    const int xh = (int)(a.x >> 32) + (int)((unsigned)xl >> 31), yh = (int)(a.y >> 32) + (int)((unsigned)yl >> 31);
    const int sh = CONJ ? -w.z : w.z, sl = CONJ ? -w.w : w.w, nsh = CONJ ? w.z : -w.z, nsl = CONJ ? w.w : -w.w;
    const long long half = K < 0 ? 1ll << 31 : 1ll << (31 - K);
    long long re = (long long)xh * w.x + (long long)yh * nsh;
    long long im = (long long)xh * sh + (long long)yh * w.x;
    const long long cr = (long long)xl * w.x + ((long long)yl * nsh + ((long long)xh * w.y + ((long long)yh * nsl + half)));
    const long long ci = (long long)xl * sh + ((long long)yl * w.x + ((long long)xh * sl + ((long long)yh * w.y + half)));
    if constexpr (K >= 0) {
        re = (long long)((unsigned long long)re << K) + (cr >> (32 - K));
        im = (long long)((unsigned long long)im << K) + (ci >> (32 - K));
    } else {
        re = (re + (cr >> 32) + (1ll << (-K - 1))) >> -K;
        im = (im + (ci >> 32) + (1ll << (-K - 1))) >> -K;
    }
    return make_longlong2(re, im);
}

// v / sqrt 2 for |v| <= 2^62.5, as v - (1 - 1/sqrt 2) v; 1 - 1/sqrt 2 =
// (CH 2^32 + CL) / 2^64.
FX_HD long long fx_times_rsqrt2(long long v) {
    constexpr int CH = 0x4AFB0CCC, CL = 0x06219B7C;
    const unsigned lo = (unsigned)v;
    const int hi = (int)(v >> 32);
    const long long cr = (long long)((unsigned long long)lo * (unsigned)CH) + ((long long)hi * CL + (1ll << 31));
    return v - ((long long)hi * CH + (cr >> 32));
}

// v w 2^K / 2^64 for a real factor w = h 2^32 + l (units of 2^-61, as fx_mul).
template <int K>
FX_HD long long fx_mul_real(long long v, int2 w) {
    const int vl = (int)v, vh = (int)(v >> 32) + (int)((unsigned)vl >> 31);
    const long long hi = (long long)vh * w.x;
    const long long cr = (long long)vl * w.x + ((long long)vh * w.y + (1ll << (31 - K)));
    return (long long)((unsigned long long)hi << K) + (cr >> (32 - K));
}

// Table factors as 2^61 values, and such a value (a product of factors) as a
// factor again; its low bit is set so that the low limb can be negated.
FX_HD longlong2 fx_value(int4 w) {
    return make_longlong2(((long long)w.x << 32) + w.y, ((long long)w.z << 32) + w.w);
}
FX_HD int4 fx_as_factor(longlong2 v) {
    const int xl = (int)v.x | 1, yl = (int)v.y | 1;
    return make_int4((int)(v.x >> 32) + (int)((unsigned)xl >> 31), xl, (int)(v.y >> 32) + (int)((unsigned)yl >> 31), yl);
}

// The two limbs of a table factor's component v (units of 2^-61).
FX_HD void fx_limbs(long long v, int& h, int& l) {
    l = (int)v;
    if (l == (int)0x80000000) v += 1, l = (int)v;      // -l has to be representable
    h = (int)((v - (long long)l) >> 32);
}

// Table load (read-only cache on the device).
FX_HD int4 fx_ldg(const int4* p) {
#ifdef __CUDA_ARCH__
    return __ldg(p);
#else
    return *p;
#endif
}

// Factor of fx_widen's results.
constexpr double FX_WIDEN = 0x1p896;

// ---- device side
#ifdef __CUDACC__
__device__ __forceinline__ unsigned fx_hi(double2 v) {
    const unsigned a = (unsigned)__double2hiint(v.x) & 0x7fffffffu, b = (unsigned)__double2hiint(v.y) & 0x7fffffffu;
    return a > b ? a : b;
}
__device__ __forceinline__ longlong2 fx_from(double2 v, int S, int E) {
    return make_longlong2(fx_from_bits(__double2hiint(v.x), (unsigned)__double2loint(v.x), S, E),
                          fx_from_bits(__double2hiint(v.y), (unsigned)__double2loint(v.y), S, E));
}
__device__ __forceinline__ double2 fx_to(longlong2 v, int X) {
    return make_double2(__longlong_as_double((long long)fx_to_bits(v.x, X)),
                        __longlong_as_double((long long)fx_to_bits(v.y, X)));
}
__device__ __forceinline__ int4 fx_factor(double c, double s) {
    int4 w;
    fx_limbs(__double2ll_rn(c * 2305843009213693952.0), w.x, w.y);
    fx_limbs(__double2ll_rn(s * 2305843009213693952.0), w.z, w.w);
    return w;
}
__device__ __forceinline__ double2 fx_factor_to_d(int4 w) {
    const double u = 1.0 / 536870912.0, l = 1.0 / 2305843009213693952.0;
    return make_double2(fma((double)w.y, l, (double)w.x * u), fma((double)w.w, l, (double)w.z * u));
}
// FP64 -> FP32, rounded to nearest (ties away), in integer arithmetic: small
// values as v 2^64 and an FP32 product with 2^-64, which gives the subnormals
// (rounded twice).  A branch to the conversion instruction for them instead cost the
// 256^2 free-space step 1 % (FP64 conversions are issued at 1/64 of the FP32 rate).
__device__ __forceinline__ float fx_to_float(double v) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const int e0 = (int)((hi >> 20) & 0x7ff) - 896, k = e0 < 64 ? 64 : 0, e = e0 + k;
    unsigned f = ((unsigned)e << 23 | (hi & 0xfffffu) << 3 | lo >> 29) + ((lo >> 28) & 1);
    if (e <= 0) f = 0;
    if (e >= 255) f = 0x7f800000u + (e == 1151 && ((hi & 0xfffffu) | lo) ? 0x400000u : 0);
    return __uint_as_float(f | (hi & 0x80000000u)) * (k ? 0x1p-64f : 1.0f);
}
__device__ __forceinline__ float2 fx_to_float(double2 v) { return make_float2(fx_to_float(v.x), fx_to_float(v.y)); }
// FP32 -> FP64 times 1 / FX_WIDEN in integer arithmetic: with the exponent field
// as it is, zeros, subnormals and normal numbers move alike.  What multiplies
// the result takes the factor FX_WIDEN, which changes no rounding.
__device__ __forceinline__ double2 fx_widen(float2 v) {
    auto one = [](float f) {
        const unsigned x = __float_as_uint(f), a = x & 0x7fffffffu;
        return __hiloint2double((int)((a >> 3) + (a >= 0x7f800000u ? 0x70000000u : 0u) | (x & 0x80000000u)), (int)(x << 29));
    };
    return make_double2(one(v.x), one(v.y));
}
// An FP32 pair as integers: components v 2^(59 + 126 - E), E the larger exponent field
// (1 at least), and back from such integers.
__device__ __forceinline__ longlong2 fx_from_float(float2 v, int& E) {
    const unsigned a = __float_as_uint(v.x), b = __float_as_uint(v.y);
    const int ea = max((int)((a >> 23) & 0xff), 1), eb = max((int)((b >> 23) & 0xff), 1);
    E = max(ea, eb);
    auto one = [E](unsigned x, int e) {
        const unsigned m = (x & 0x7fffffu) | ((x & 0x7f800000u) ? 0x800000u : 0u);
        const long long t = (long long)((unsigned long long)m << 35 >> min(E - e, 63));
        return (int)x < 0 ? -t : t;
    };
    return make_longlong2(one(a, ea), one(b, eb));
}
__device__ __forceinline__ float2 fx_to_float(longlong2 v, int E) {
    const float s = __uint_as_float((unsigned)E << 23);          // 2^(E - 127); infinite for a pair with an infinity or a NaN
    return make_float2(__ll2float_rn(v.x) * 0x1p-58f * s, __ll2float_rn(v.y) * 0x1p-58f * s);
}
// Largest value of v over the T threads of a CTA (all of them call it).
template <int T>
__device__ __forceinline__ unsigned fx_cta_max(unsigned v) {
    v = __reduce_max_sync(0xffffffffu, v);
    if constexpr (T > 32) {
        __shared__ unsigned mx[T / 32];
        if ((threadIdx.x & 31) == 0) mx[threadIdx.x >> 5] = v;
        __syncthreads();
        v = __reduce_max_sync(0xffffffffu, mx[(threadIdx.x & 31) % (T / 32)]);
    }
    return v;
}
// The same per line, L lines interleaved over the threads (thread t works on line t % L).
template <int T, int L>
__device__ __forceinline__ unsigned fx_line_max(unsigned v) {
    static_assert(L <= 32 && 32 % L == 0 && T % 32 == 0, "a warp holds whole sets of lines");
    if constexpr (L == 1) {
        return fx_cta_max<T>(v);
    } else {
        auto fold = [](unsigned x) {
#pragma unroll
            for (int o = 16; o >= L; o >>= 1) x = max(x, __shfl_xor_sync(0xffffffffu, x, o));
            return x;
        };
        v = fold(v);
        if constexpr (T > 32) {
            __shared__ unsigned mx[T / 32 * L];
            const int lane = threadIdx.x & 31;
            if (lane < L) mx[(threadIdx.x >> 5) * L + lane] = v;
            __syncthreads();
            v = 0;
#pragma unroll
            for (int w = 0; w < T / 32; w += 32 / L)
                if (w + lane / L < T / 32) v = max(v, mx[(w + lane / L) * L + lane % L]);
            v = fold(v);
        }
        return v;
    }
}
#endif  // __CUDACC__

}  // namespace tdse
