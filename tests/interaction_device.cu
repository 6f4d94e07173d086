// The change of a state's history to the interaction picture (csrc/tables.cu,
// launch_to_interaction) against long double arithmetic: ring values z conj(E) R,
// FP32 roundings of products whose phases are held in more.  Prints, for a 2D and
// a 3D grid, the largest distance from the exact product beyond half an FP32 ulp
// of the component, relative to the product.
#include <cmath>
#include <complex>
#include <cstdio>
#include <vector>

#include "kargs.h"

using namespace tdse;
typedef std::complex<long double> cl;

static unsigned long long lcg = 88172645463325252ull;
static float rnd() {
    lcg ^= lcg << 13; lcg ^= lcg >> 7; lcg ^= lcg << 17;
    return (float)((double)(lcg >> 11) / 9007199254740992.0 * 2.0 - 1.0);
}

static double excess(int n0, int n1, int n2) {
    const int B = 2, RS = 4, nsteps = 40, ntf = 8 * nsteps + 1, inner = n1 * (n2 ? n2 : 1), len = n0 + n1 + n2;
    const size_t NP = (size_t)n0 * inner;
    const double dt = 1.25e-3;
    const int steps[8] = {5, 2, 3, 4, -1, -1, -1, -1};
    float z[16];
    for (int q = 0; q < 8; ++q) z[2 * q] = std::cos(0.7f * q), z[2 * q + 1] = std::sin(0.7f * q);
    std::vector<float2> ring(B * RS * NP), out(B * RS * NP);
    for (auto& r : ring) r = make_float2(rnd(), rnd());
    void *uhat, *dring, *phi, *scratch;
    if (cudaMalloc(&uhat, B * NP * 16) != cudaSuccess || cudaMalloc(&dring, ring.size() * 8) != cudaSuccess ||
        cudaMalloc(&phi, (size_t)B * 3 * ntf * 8) != cudaSuccess || cudaMalloc(&scratch, (size_t)B * 9 * len * 16) != cudaSuccess)
        return 1e9;
    cudaMemset(uhat, 0, B * NP * 16);
    cudaMemset(phi, 0, (size_t)B * 3 * ntf * 8);
    cudaMemcpy(dring, ring.data(), ring.size() * 8, cudaMemcpyHostToDevice);
    KArgs a{};
    a.B = B;
    a.n0 = a.tn0 = n0;
    a.n1 = a.tn1 = n1;
    a.tn2 = n2;
    a.uhat = uhat;
    a.ring = dring;
    a.ring_slots = RS;
    a.phi = static_cast<double*>(phi);
    a.ntf = ntf;
    a.dt = dt;
    if (launch_to_interaction(a, 5, steps, z, RS, scratch, 0) != cudaSuccess) return 1e9;
    if (cudaMemcpy(out.data(), dring, out.size() * 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 1e9;
    auto phase = [&](int m, int n, int step) -> cl {     // conj(E) of one axis, A = 0
        const double k = m < n / 2 ? m : m - n, arg = -(k * k) * ((double)step * dt);
        return cl(cosl((long double)arg), -sinl((long double)arg));
    };
    long double worst = 0;
    for (int b = 0; b < B; ++b)
        for (int q = 0; q < RS; ++q)
            for (size_t i = 0; i < NP; ++i) {
                const int m0 = (int)(i / inner), rem = (int)(i % inner), m1 = n2 ? rem / n2 : rem;
                cl v = cl(z[2 * q], z[2 * q + 1]) * phase(m0, n0, steps[q]) * phase(m1, n1, steps[q]);
                if (n2) v *= phase(rem % n2, n2, steps[q]);
                const size_t at = ((size_t)b * RS + q) * NP + i;
                v *= cl(ring[at].x, ring[at].y);
                auto over = [&](float got, long double want) {
                    const float w = (float)fabsl(want);
                    const long double ulp = std::nextafterf(w, 4.0f) - w;
                    return (fabsl(got - want) - 0.5L * ulp) / std::abs(v);
                };
                worst = std::max(worst, std::max(over(out[at].x, v.real()), over(out[at].y, v.imag())));
            }
    cudaFree(uhat);
    cudaFree(dring);
    cudaFree(phi);
    cudaFree(scratch);
    return (double)worst;
}

int main() {
    std::printf("%.4e %.4e\n", excess(256, 128, 0), excess(64, 32, 64));
    return 0;
}
