// Host-side check of the conversions of csrc/fx.cuh at the ends of the FP64 range:
// values down to the smallest subnormal, alone and in a transform.  Prints the
// number of failures of each kind, then n and the transform's error.
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstring>
#include <vector>

#include "cplx.cuh"

using namespace tdse;

static unsigned long long lcg = 88172645463325252ull;
static unsigned long long rnd() {
    lcg ^= lcg << 13; lcg ^= lcg >> 7; lcg ^= lcg << 17;
    return lcg;
}
static unsigned long long bits(double x) { unsigned long long b; std::memcpy(&b, &x, 8); return b; }
static double value(unsigned long long b) { double x; std::memcpy(&x, &b, 8); return x; }
static unsigned high(double x) { return (unsigned)(bits(x) >> 32) & 0x7fffffffu; }
static long long from(double x, int S, int E) { return fx_from_bits((int)(bits(x) >> 32), (unsigned)bits(x), S, E); }

template <int N, int S> static void pass(std::vector<longlong2>& x, const int4* tw) {
    using P = FftPlan<N, false>;
    if constexpr (S < P::NPASS) {
        constexpr int R = P::radix(S), Ns = P::ns(S), NB = N / R;
        std::vector<longlong2> y(N);
        for (int j = 0; j < NB; ++j) {
            longlong2 v[R];
            for (int r = 0; r < R; ++r) v[r] = x[j + r * NB];
            FxPass<N, false>::template butterfly<S>(v, j, tw);
            const int k = j & (Ns - 1);
            for (int r = 0; r < R; ++r) y[(j - k) * R + k + r * Ns] = v[r];
        }
        x = y;
        pass<N, S + 1>(x, tw);
    }
}

// One transform of values of about 2^lg against the same one of about 1.
template <int N> static double scaled(int lg) {
    using Fx = FxPass<N, false>;
    std::vector<int4> tw(N);
    for (int m = 0; m < N; ++m) {
        fx_limbs(llround(std::cos(2 * M_PI * m / N) * 0x1p61), tw[m].x, tw[m].y);
        fx_limbs(llround(-std::sin(2 * M_PI * m / N) * 0x1p61), tw[m].z, tw[m].w);
    }
    std::vector<std::complex<double>> out[2];
    std::vector<double> re(N), im(N);
    for (int j = 0; j < N; ++j) {
        re[j] = (double)(int)(rnd() >> 40) * 0x1p-24;      // 24 bits: exact at 2^lg too
        im[j] = (double)(int)(rnd() >> 40) * 0x1p-24;
    }
    for (int c = 0; c < 2; ++c) {
        unsigned mx = 0;
        for (int j = 0; j < N; ++j) mx = std::max(mx, std::max(high(std::ldexp(re[j], c ? lg : 0)), high(std::ldexp(im[j], c ? lg : 0))));
        const int E = fx_exponent(mx), X = Fx::out_exp(mx, E, 0);
        std::vector<longlong2> v(N);
        for (int j = 0; j < N; ++j) v[j] = make_longlong2(from(std::ldexp(re[j], c ? lg : 0), Fx::S0, E), from(std::ldexp(im[j], c ? lg : 0), Fx::S0, E));
        pass<N, 0>(v, tw.data());
        for (auto& z : v) out[c].push_back({value(fx_to_bits(z.x, X)), value(fx_to_bits(z.y, X))});
    }
    double worst = 0.0;                                    // in units of the smallest FP64 step at 2^lg, or of 2^-52
    for (int k = 0; k < N; ++k) {
        const double a = std::abs(std::ldexp(1.0, lg)) * std::abs(out[0][k]);
        const double unit = std::fmax(0x1p-1074, a * 0x1p-52);
        worst = std::fmax(worst, std::fabs(out[1][k].real() - std::ldexp(out[0][k].real(), lg)) / unit);
        worst = std::fmax(worst, std::fabs(out[1][k].imag() - std::ldexp(out[0][k].imag(), lg)) / unit);
    }
    return worst;
}

int main() {
    int trip = 0, beside = 0, step = 0;
    for (int i = 0; i < 200000; ++i) {
        // round trips: subnormals and the smallest normal numbers, each its own block
        const unsigned long long b = (rnd() >> 12 >> (rnd() % 52)) | ((rnd() % 70) << 52) | (rnd() & 1) << 63;
        const double x = value(b);
        const int E = fx_exponent(high(x));
        if (value(fx_to_bits(from(x, 59, E), E - 1022 - 59)) != x) ++trip;
        // beside a larger value of the block: truncated at 2^-59 of its scale
        const int lead = 1 + (int)(rnd() % 60);
        const long long v = from(x, 59, E + lead);
        const long double exact = ldexpl((long double)x, 1022 + 59 - (E + lead));
        if (fabsl((long double)v - exact) >= 1.0L) ++beside;
        // rounding of results into the subnormal range
        const long long w = (long long)(rnd() >> 2) * (rnd() & 1 ? 1 : -1);
        const int X = -1074 - (int)(rnd() % 62);
        const long double want = ldexpl((long double)w, X);
        if (fabsl((long double)value(fx_to_bits(w, X)) - want) > fmaxl(0x1p-1075L, fabsl(want) * 0x1p-53L)) ++step;
    }
    std::printf("%d %d %d\n", trip, beside, step);
    for (int lg : {-900, -950, -990, -1000, -1020, -1040}) std::printf("%d %.3f\n", lg, scaled<64>(lg));
}
