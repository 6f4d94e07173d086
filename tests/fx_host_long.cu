// Host-side check of the fixed-point transforms (csrc/fx.cuh, FxPass of
// csrc/cplx.cuh) on inputs that sit in few places of the line, as the modes of a
// smooth state on a fine grid and a narrow state do: one nonzero value, and
// Gaussians a few points to a tenth of the line wide.  The kernels' passes on the
// CPU, long lines scaled up before their middle passes, against long double sums.
// Prints n, direction, plan (8: radix 8, 4: radix 4), input, error of the
// fixed-point transform and of an FP64 transform (radix 2).
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstring>
#include <vector>

#include "cplx.cuh"

using namespace tdse;
typedef std::complex<long double> cl;
typedef std::complex<double> cd;

static unsigned long long bits(double x) { unsigned long long b; std::memcpy(&b, &x, 8); return b; }
static double value(unsigned long long b) { double x; std::memcpy(&x, &b, 8); return x; }

template <int N, bool INV, class P, int S> static int pass(std::vector<longlong2>& x, const int4* tw) {
    using Fx = FxPass<N, INV, P>;
    if constexpr (S < P::NPASS) {
        constexpr int R = P::radix(S), Ns = P::ns(S), NB = N / R;
        std::vector<longlong2> y(N);
        int up = 0;
        if (Fx::rescales(S)) {
            unsigned m = 0;
            for (auto& v : x) m = std::max(m, Fx::magnitude(v));
            up = Fx::headroom(m);
            for (auto& v : x) v = Fx::up(v, up);
        }
        for (int j = 0; j < NB; ++j) {
            longlong2 v[R];
            for (int r = 0; r < R; ++r) v[r] = x[j + r * NB];
            Fx::template butterfly<S>(v, j, tw);
            const int k = j & (Ns - 1);
            for (int r = 0; r < R; ++r) y[(j - k) * R + k + r * Ns] = v[r];
        }
        x = y;
        return up + pass<N, INV, P, S + 1>(x, tw);
    }
    return 0;
}

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

template <int N, bool INV, class P> static void check(int plan, int kind) {
    using Fx = FxPass<N, INV, P>;
    std::vector<int4> tw(N);
    std::vector<cl> w(N);
    for (int m = 0; m < N; ++m) {
        const long double t = 2 * 3.141592653589793238462643383279502884L * m / N;
        fx_limbs((long long)((double)cosl(t) * 0x1p61), tw[m].x, tw[m].y);
        fx_limbs((long long)((double)-sinl(t) * 0x1p61), tw[m].z, tw[m].w);
        w[m] = cl(cosl(t), (INV ? 1 : -1) * sinl(t));
    }
    const double width = kind == 1 ? 5.0 : kind == 2 ? 40.0 : 0.1 * N;
    std::vector<cd> x(N);
    for (int j = 0; j < N; ++j)
        x[j] = kind == 0 ? (j == N / 3 ? cd(0.7, -0.3) : cd(0.0, 0.0))
                         : std::exp(-0.5 * std::pow((j - N / 3.0) / width, 2)) * cd(std::cos(0.37 * j), std::sin(0.11 * j * j));
    unsigned mx = 0;
    for (auto& v : x)
        for (double c : {v.real(), v.imag()}) mx = std::max(mx, (unsigned)(bits(c) >> 32) & 0x7fffffffu);
    const int E = fx_exponent(mx);
    std::vector<longlong2> v(N);
    auto from = [&](double d) { return fx_from_bits((int)(bits(d) >> 32), (unsigned)bits(d), Fx::S0, E); };
    for (int j = 0; j < N; ++j) v[j] = make_longlong2(from(x[j].real()), from(x[j].imag()));
    const int X = Fx::out_exp(mx, E, 0) - pass<N, INV, P, 0>(v, tw.data());
    const std::vector<cd> y64 = fft64(x, INV);
    std::vector<cl> s(N, cl(0));
    for (int j = 0; j < N; ++j)
        if (std::abs(x[j]) > 1e-25)
            for (int k = 0; k < N; ++k) s[k] += cl(x[j].real(), x[j].imag()) * w[(long long)j * k % N];
    long double e = 0, e64 = 0, n2 = 0;
    for (int k = 0; k < N; ++k) {
        e += std::norm(cl(value(fx_to_bits(v[k].x, X)), value(fx_to_bits(v[k].y, X))) - s[k]);
        e64 += std::norm(cl(y64[k].real(), y64[k].imag()) - s[k]);
        n2 += std::norm(s[k]);
    }
    std::printf("%d %d %d %d %.3Le %.3Le\n", N, (int)INV, plan, kind, sqrtl(e / n2), sqrtl(e64 / n2));
}

template <int N, bool INV> static void kinds() {
    for (int kind = 0; kind < 4; ++kind) {
        check<N, INV, FftPlan<N, INV>>(8, kind);
        if constexpr (N <= 1024) check<N, INV, FftPlan4<N, INV>>(4, kind);
    }
}
template <int N> static void both() {
    kinds<N, false>();
    kinds<N, true>();
}

int main() {
    both<128>();
    both<512>();
    both<1024>();
    both<2048>();
    both<4096>();
    both<8192>();
}
