// Host-side check of the fixed-point transforms (csrc/fx.cuh, FxPass of
// csrc/cplx.cuh): the same passes as the kernels', on the CPU, against long
// double sums.  Prints one line per transform: n, direction, scale of the
// input, error of the fixed-point transform and of the same passes in FP64.
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstring>
#include <vector>

#include "cplx.cuh"

using namespace tdse;
typedef std::complex<long double> cl;
typedef std::complex<double> cd;

static unsigned long long lcg = 88172645463325252ull;
static double rnd() {
    lcg ^= lcg << 13; lcg ^= lcg >> 7; lcg ^= lcg << 17;
    return (double)(lcg >> 11) / 9007199254740992.0 * 2.0 - 1.0;
}
static unsigned long long bits(double x) { unsigned long long b; std::memcpy(&b, &x, 8); return b; }
static double value(unsigned long long b) { double x; std::memcpy(&x, &b, 8); return x; }

template <int N, bool INV, int S> static void pass(std::vector<longlong2>& x, const int4* tw) {
    using P = FftPlan<N, INV>;
    if constexpr (S < P::NPASS) {
        constexpr int R = P::radix(S), Ns = P::ns(S), NB = N / R;
        std::vector<longlong2> y(N);
        for (int j = 0; j < NB; ++j) {
            longlong2 v[R];
            for (int r = 0; r < R; ++r) v[r] = x[j + r * NB];
            FxPass<N, INV>::template butterfly<S>(v, j, tw);
            const int k = j & (Ns - 1);
            for (int r = 0; r < R; ++r) y[(j - k) * R + k + r * Ns] = v[r];
        }
        x = y;
        pass<N, INV, S + 1>(x, tw);
    }
}

// radix-2 FP64 Stockham transform, the precision to beat
static std::vector<cd> fft64(std::vector<cd> x, bool inv) {
    const int n = (int)x.size();
    for (int ns = 1; ns < n; ns *= 2) {
        std::vector<cd> y(n);
        for (int j = 0; j < n / 2; ++j) {
            const int k = j % ns;
            const double th = (inv ? 1 : -1) * M_PI * k / ns;
            const cd a = x[j], b = x[j + n / 2] * cd(std::cos(th), std::sin(th));
            y[(j - k) * 2 + k] = a + b;
            y[(j - k) * 2 + k + ns] = a - b;
        }
        x = y;
    }
    return x;
}

template <int N, bool INV> static void check(int kind, double scale) {
    const long double pi = 3.141592653589793238462643383279502884L;
    std::vector<int4> tw(N);
    std::vector<cl> w(N);
    for (int m = 0; m < N; ++m) {
        const double c = (double)cosl(2 * pi * m / N), s = (double)-sinl(2 * pi * m / N);
        fx_limbs((long long)(c * 0x1p61), tw[m].x, tw[m].y);
        fx_limbs((long long)(s * 0x1p61), tw[m].z, tw[m].w);
        w[m] = cl(cosl(2 * pi * m / N), (INV ? 1 : -1) * sinl(2 * pi * m / N));
    }
    std::vector<cd> x(N);
    for (int j = 0; j < N; ++j) {
        const double g = kind == 0 ? 1.0 : kind == 1 ? std::exp(-0.5 * std::pow((j - N / 3.0) / (0.06 * N), 2)) : std::pow(2.0, -60.0 * j / N);
        x[j] = scale * g * (kind == 2 ? cd(1.0, -0.5) : cd(rnd(), rnd()));
    }
    unsigned mx = 0;
    for (auto& v : x) {
        mx = std::max(mx, (unsigned)(bits(v.real()) >> 32) & 0x7fffffffu);
        mx = std::max(mx, (unsigned)(bits(v.imag()) >> 32) & 0x7fffffffu);
    }
    using Fx = FxPass<N, INV>;
    const int E = fx_exponent(mx), X = Fx::out_exp(mx, E, 0);
    std::vector<longlong2> v(N);
    auto from = [&](double d) { return fx_from_bits((int)(bits(d) >> 32), (unsigned)bits(d), Fx::S0, E); };
    for (int j = 0; j < N; ++j) v[j] = make_longlong2(from(x[j].real()), from(x[j].imag()));
    pass<N, INV, 0>(v, tw.data());
    const std::vector<cd> y64 = fft64(x, INV);
    long double e = 0, e64 = 0, n2 = 0;
    for (int k = 0; k < N; ++k) {
        cl s = 0;
        for (int j = 0; j < N; ++j) s += cl(x[j].real(), x[j].imag()) * w[(long long)j * k % N];
        const cl got(value(fx_to_bits(v[k].x, X)), value(fx_to_bits(v[k].y, X)));
        e += std::norm(got - s);
        e64 += std::norm(cl(y64[k].real(), y64[k].imag()) - s);
        n2 += std::norm(s);
    }
    std::printf("%d %d %d %g %.3Le %.3Le\n", N, (int)INV, kind, scale, sqrtl(e / n2), sqrtl(e64 / n2));
}

template <int N> static void both() {
    for (int kind = 0; kind < 3; ++kind) {
        check<N, false>(kind, 1.0);
        check<N, true>(kind, 1.0);
    }
    check<N, false>(1, 1e-200);
    check<N, true>(0, 1e+200);
}

int main() {
    // conversions: exact round trips, zeros, extremes
    int bad = 0;
    for (int i = 0; i < 20000; ++i) {
        const double x = rnd() * std::pow(2.0, (int)(rnd() * 900));
        const unsigned long long b = bits(x);
        const int E = fx_exponent((unsigned)(b >> 32) & 0x7fffffffu);
        const long long v = fx_from_bits((int)(b >> 32), (unsigned)b, 59, E);
        if (value(fx_to_bits(v, E - 1022 - 59)) != x) ++bad;
    }
    if (fx_to_bits(0, 5) != 0) ++bad;
    if (fx_from_bits(0, 0, 59, 64) != 0 || fx_from_bits((int)0x80000000, 0, 59, 1023) != 0) ++bad;
    if (!std::isnan(value(fx_to_bits(1, FX_NAN))) || !std::isnan(value(fx_to_bits(0, FX_NAN)))) ++bad;
    if (!std::isinf(value(fx_to_bits(1ll << 60, 1000)))) ++bad;
    if (value(fx_to_bits(1ll << 40, -1200)) != 0.0) ++bad;
    // products at the edge of their range
    for (int i = 0; i < 200000; ++i) {
        const double r = std::pow(2.0, 62.5), ph = M_PI * rnd(), q = M_PI * rnd();
        const longlong2 a = make_longlong2((long long)(r * std::cos(ph)), (long long)(r * std::sin(ph)));
        int4 w;
        fx_limbs(llroundl(cosl(q) * 0x1p61L), w.x, w.y);
        fx_limbs(llroundl(sinl(q) * 0x1p61L), w.z, w.w);
        const longlong2 p = fx_mul<false, 0>(a, w);
        const __int128 wc = ((__int128)w.x << 32) + w.y, ws = ((__int128)w.z << 32) + w.w;
        const long long re = (long long)((a.x * wc - a.y * ws) >> 64), im = (long long)((a.x * ws + a.y * wc) >> 64);
        if (llabs(p.x - re) > 2 || llabs(p.y - im) > 2) ++bad;
        const long long u = fx_times_rsqrt2(a.x);
        if (fabsl((long double)u - (long double)a.x * sqrtl(0.5L)) > 2.0L) ++bad;
    }
    std::printf("bad %d\n", bad);
    both<8>();
    both<16>();
    both<32>();
    both<64>();
    both<128>();
    both<256>();
    both<512>();
    both<1024>();
    both<4096>();
    return bad != 0;
}
